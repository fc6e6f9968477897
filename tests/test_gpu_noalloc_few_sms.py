"""The allocation-free CSR solve in the forms of a device of few SMs: up to 16 chunks of 32 rows per
block (four a thread), up to 64 (sixteen a thread), and a system beyond them."""
import numpy as np
import pytest

ss = pytest.importorskip("paper_1808_06381_gb300")
torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


def _system(n, seed):
    """A ring with random second neighbours, diagonally dominant."""
    rng = np.random.default_rng(seed)
    i = np.arange(n)
    pairs = np.unique(np.sort(np.concatenate([np.stack([i, (i + 1) % n], 1), rng.integers(0, n, (2 * n, 2))]), 1), axis=0)
    pairs = pairs[pairs[:, 0] != pairs[:, 1]]
    w = rng.random(len(pairs)) + 0.01
    rows, cols = np.concatenate([pairs[:, 0], pairs[:, 1]]), np.concatenate([pairs[:, 1], pairs[:, 0]])
    order = np.lexsort((cols, rows))
    rows, cols, ww = rows[order], cols[order], np.concatenate([w, w])[order]
    ptr = np.concatenate([[0], np.cumsum(np.bincount(rows, minlength=n))]).astype(np.int32)
    return ptr, cols.astype(np.int32), ww, rows, 1.0 + 2.0 * np.bincount(rows, weights=ww, minlength=n), rng.standard_normal((3, n))


# (rows, SMs): 11 and 16 chunks a block; 17, 64; one chunk too many
@pytest.mark.parametrize("n,sms,ok", [(3500, 10, True), (5120, 10, True), (5121, 10, True), (20480, 10, True),
                                      (32768, 16, True), (20481, 10, False)])
def test_solve_on_few_sms(n, sms, ok, monkeypatch):
    monkeypatch.setenv("SHEARSIM_NOALLOC_SMS", str(sms))
    ptr, col, w, rows, diag, b = _system(n, n)
    dev = torch.device("cuda", 0)
    t = [torch.from_numpy(a).to(dev) for a in (ptr, col, w, diag, b)]
    x = torch.zeros((3, n), dtype=torch.float64, device=dev)
    info = ss.solve_csr_noalloc(n, *(a.data_ptr() for a in t[:4]), 1.0, t[4].data_ptr(), x.data_ptr(), tol=1e-12,
                                max_iter=2000, stream=torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    if not ok:
        assert info["status"] != 0 and "too few SMs" in info["error"], info
        return
    assert info["status"] == 0 and info["residual"] <= 1e-12, info
    x = x.cpu().numpy()
    r = np.stack([b[c] - diag * x[c] + np.bincount(rows, weights=w * x[c][col], minlength=n) for c in range(3)])
    # numpy's residual rounds the terms of a row (2^-53 of the diagonal's part)
    assert np.linalg.norm(r) <= (1e-12 + 1e-14) * np.linalg.norm(b)

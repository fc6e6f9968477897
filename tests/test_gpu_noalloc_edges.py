"""The allocation-free CSR solve at the edges of its launch shapes, on rows in any order of
columns and of any length, and the refusal of a decreasing row_ptr."""
import numpy as np
import pytest

ss = pytest.importorskip("paper_1808_06381_gb300")
torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


def _random_system(n, seed, dense_rows):
    """A symmetric pattern without self-coupling, ~6 entries a row, the first dense_rows rows
    coupled to all others; the columns of a row in random order; diagonally dominant."""
    rng = np.random.default_rng(seed)
    i = rng.integers(0, n, 3 * n)
    j = rng.integers(0, n, 3 * n)
    for d in range(min(dense_rows, n)):
        i = np.concatenate([i, np.full(n, d)])
        j = np.concatenate([j, np.arange(n)])
    lo, hi = np.minimum(i, j), np.maximum(i, j)
    pairs = np.unique(np.stack([lo, hi], 1)[lo != hi], axis=0)
    w = rng.random(len(pairs)) + 0.01
    rows, cols = np.concatenate([pairs[:, 0], pairs[:, 1]]), np.concatenate([pairs[:, 1], pairs[:, 0]])
    ww = np.concatenate([w, w])
    order = np.lexsort((rng.random(len(rows)), rows))
    rows, cols, ww = rows[order], cols[order], ww[order]
    row_ptr = np.concatenate([[0], np.cumsum(np.bincount(rows, minlength=n))]).astype(np.int32)
    diag = 1.0 + 2.0 * np.bincount(rows, weights=ww, minlength=n)
    return row_ptr, cols.astype(np.int32), ww, rows, diag, rng.standard_normal((3, n))


# chunks of 32 rows per SM on 152 SMs: 1 up to 4,864 rows, 5 up to 24,320 (one component a
# thread), 7 up to 32,768 (two); a row coupled to all others is longer than its chunk's share of
# shared memory.
@pytest.mark.parametrize("n,dense_rows", [(1, 0), (2, 0), (33, 0), (4864, 0), (4865, 0), (24320, 0), (24321, 0),
                                          (32768, 0), (700, 3), (30001, 1)])
def test_solution_meets_the_tolerance_on_the_callers_arrays(n, dense_rows):
    row_ptr, col, w, rows, diag, b = _random_system(n, n, dense_rows)
    dev = torch.device("cuda", 0)
    pad = lambda a: torch.from_numpy(a if len(a) else np.zeros(1, a.dtype)).to(dev)
    t = [pad(a) for a in (row_ptr, col, w, diag)]
    tb = torch.from_numpy(b).to(dev)
    tx = torch.full((3, n), float("nan"), dtype=torch.float64, device=dev)
    info = ss.solve_csr_noalloc(n, *(a.data_ptr() for a in t), 1.0, tb.data_ptr(), tx.data_ptr(), tol=1e-12,
                                max_iter=2000, stream=torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    assert info["status"] == 0 and info["residual"] <= 1e-12, info
    x = tx.cpu().numpy()
    r = np.stack([b[c] - diag * x[c] + np.bincount(rows, weights=w * x[c][col], minlength=n) for c in range(3)])
    # numpy's residual rounds each of a row's terms (2^-53 of the diagonal's part, up to ~4 times ||b||'s share)
    assert np.linalg.norm(r) <= (1e-12 + 1e-14 * np.sqrt(1 + dense_rows * n / 10)) * np.linalg.norm(b)


def test_a_decreasing_row_ptr_is_refused():
    dev = torch.device("cuda", 0)
    for n, at in ((40, 3), (5000, 4097)):
        rp = torch.zeros(n + 1, dtype=torch.int32)
        rp[1:] = 2
        rp[at] = 1                     # row at - 1 runs from 2 to 1
        rp = rp.to(dev)
        col = torch.tensor([1, 1], dtype=torch.int32, device=dev)
        w = torch.full((2,), 0.1, dtype=torch.float64, device=dev)
        diag = torch.ones(n, dtype=torch.float64, device=dev)
        b = torch.ones(3, n, dtype=torch.float64, device=dev)
        x = torch.zeros(3, n, dtype=torch.float64, device=dev)
        info = ss.solve_csr_noalloc(n, rp.data_ptr(), col.data_ptr(), w.data_ptr(), diag.data_ptr(), 1.0,
                                    b.data_ptr(), x.data_ptr(), tol=1e-12, max_iter=100,
                                    stream=torch.cuda.current_stream().cuda_stream)
        torch.cuda.synchronize()
        assert info["status"] == ss.SP_ERR_INVALID_ARG and "row_ptr" in info["error"], info

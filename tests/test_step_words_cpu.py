"""noise_step (the step whose normals are drawn) is written by k_row_normals while the pair search
runs beside it: no other code may store to it then, not even the value it has read.  A race cannot
be provoked safely, so the stores are checked in the source."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1808_06381_gb300", "csrc")


def test_only_the_normals_kernel_stores_noise_step_beside_the_search():
    stores = []
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        for line in open(path, encoding="utf-8"):
            code = line.split("//")[0]
            if re.search(r"->noise_step\s*=[^=]", code):
                stores.append((os.path.basename(path), code.strip()))
    device = [c for f, c in stores if f == "neighbors.cu"]
    assert sorted(device) == ["if (draw_noise != 2) st->noise_step = draw_noise ? st->step : -1;",
                              "if (i == 0) st->noise_step = st->step;"], device
    # the host sets it once, before any launch
    assert [(f, c) for f, c in stores if f != "neighbors.cu"] == [("sim.cu", "s->st_host->noise_step = -1;")]

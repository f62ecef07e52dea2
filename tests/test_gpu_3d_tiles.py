"""The 3-D kernels where their tiles end: rows that do not fill a tile or a
warp's pair of rows, x extents beside the 128 columns of a box and beside the
rounding to four, and z extents of few planes per block, against the FP64
oracle (the fields at the required relative L2)."""
import numpy as np
import pytest

import workloads as W
from rtm_cases import TOL, case_3d, gpu_shot, oracle_shot, rel

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

# interior (nx, ny, nz), boundary cells: padded ny = 9 (one row beyond a tile), 16, 17, 23; nx = 33, 128, 131, 257
GRIDS = [(25, 1, 30, 4), (120, 8, 1, 4), (123, 9, 12, 4), (249, 15, 5, 4)]


@pytest.mark.parametrize("grid", GRIDS, ids=lambda g: "x".join(map(str, g)))
def test_edges_of_the_tiles_match_the_oracle(grid):
    import paper_2204_03380_gb300 as R
    nx, ny, nz, nb = grid
    nt = 60
    w, v, src, _, _ = case_3d("tiles", nx, ny, nz, nb, nt, seed=nx)
    wav = W.ricker(nt + 90, w.dt, w.f_peak)[90:]   # from near the peak: short records carry signal
    NX, NY, NZ = nx + 2 * nb, ny + 2 * nb, nz + 2 * nb
    src = np.array([min(NX - 1, 128), min(NY - 1, 8), NZ // 2], np.int32)
    rec = np.array([[x, y, z] for x in sorted({0, NX // 2, min(127, NX - 1), NX - 1})
                    for y in sorted({0, 7, 8, NY - 2, NY - 1}) for z in (0, nb + 1, NZ - 1)], np.int32)
    g, o = gpu_shot(R, torch, w, v, src, rec, wav), oracle_shot(w, v, src, rec, wav)
    for k in ("seis", "prev", "last", "num", "den"):
        assert rel(g[k], o[k]) <= TOL, k

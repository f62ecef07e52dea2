"""Low and tall tiles of the denoiser's convolutions: a batch that fills the
SMs runs 8-row tiles, its images alone 4-row tiles.  An output's products are
summed in the same order in both, so the results are the same bits; gradients
add fp32 partial sums in another order (two sums of n terms with random signs
differ by about eps sqrt(n) of the terms' root sum of squares, n = 10^6
pixels: 1e-4; the bound leaves a factor of 3)."""
import numpy as np
import pytest

from oracle import cnn
from rtm_cases import rel

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _run(R, P, X, dY):
    Y, Yi, G = torch.empty_like(X), torch.full_like(X, float("nan")), torch.zeros_like(P)
    ws = torch.empty(R.rbc_cnn_workspace_bytes(*X.shape), dtype=torch.uint8, device="cuda")
    R.rbc_cnn_infer(P, X, Yi, ws)
    R.rbc_cnn_forward(P, X, Y, ws)
    R.rbc_cnn_backward(P, dY, G, ws)
    torch.cuda.synchronize()
    assert torch.equal(Y, Yi)
    return Y, G


# (images, rows, columns): ragged in both tile heights and the 126-column width
@pytest.mark.parametrize("shape", [(400, 17, 130), (700, 9, 127), (300, 24, 252)])
def test_batch_equals_its_images_alone(shape):
    import paper_2204_03380_gb300 as R
    n, H, W = shape
    g = torch.Generator(device="cuda").manual_seed(n)
    P = torch.tensor(cnn.init_params(6), dtype=torch.float32, device="cuda")
    P += 0.05 * torch.randn(P.shape, device="cuda", generator=g)
    X = torch.randn(shape, device="cuda", generator=g)
    dY = torch.randn(shape, device="cuda", generator=g)
    Y, G = _run(R, P, X, dY)
    Gs = torch.zeros_like(P, dtype=torch.float64)
    for i in range(n):
        y, gi = _run(R, P, X[i:i + 1].contiguous(), dY[i:i + 1].contiguous())
        assert torch.equal(Y[i:i + 1], y), i
        Gs += gi.double()
    assert rel(G.cpu().numpy(), Gs.cpu().numpy()) <= 3e-4


# memory orders of a volume (nz, ny, nx): row major, z and y swapped, x not
# innermost, a window of a larger volume, a slice repeated along y; slabs that
# leave a remainder, a single row and a single column
@pytest.mark.parametrize("order", ["rows", "swapped", "x_outer", "window", "repeated"])
@pytest.mark.parametrize("shape,slab", [((19, 7, 131), 3), ((1, 5, 1), 64), ((40, 3, 64), 1)])
def test_volume_in_place_equals_its_slices(order, shape, slab):
    from paper_2204_03380_gb300 import denoise as D
    nz, ny, nx = shape
    g = torch.Generator(device="cuda").manual_seed(nz)
    v = torch.randn(shape, device="cuda", generator=g)
    if order == "swapped":
        v = v.transpose(0, 1).contiguous().transpose(0, 1)
    elif order == "x_outer":
        v = v.permute(2, 0, 1).contiguous().permute(1, 2, 0)
    elif order == "window":
        v = torch.randn((nz + 2, ny + 3, nx + 5), device="cuda", generator=g)[1:nz + 1, 2:ny + 2, 3:nx + 3]
    elif order == "repeated":
        v = v[:, :1].expand(nz, ny, nx)
    net = D.Denoiser(seed=2)
    out = net.denoise_volume(v, slab=slab)
    ref = net(v.permute(1, 0, 2).contiguous()).permute(1, 0, 2)
    assert torch.equal(out, ref)

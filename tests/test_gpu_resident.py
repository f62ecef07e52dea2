"""The resident 2-D time loops (one launch per phase, fields on the chip)
against the one-launch-per-step path and the FP64 oracle, over every tile
shape: ragged grids, short last tiles, grids narrower than a tile, a source on
a tile corner, receivers on tile edges, in the pad, repeated, and more of them
in one warp's rows than it keeps in registers; even and odd record lengths."""
import numpy as np
import pytest

import workloads as W
from rtm_cases import TOL, case_2d, gpu_build, oracle_shot, rel

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

# (kernel variant by rows per warp: 1, 2, 4, 7, 10; warps per block), None: the plan's own choice
TILES = [None, "0,4", "0,8", "0,16", "1,3", "1,8", "1,16", "2,1", "2,3", "3,2", "4,2"]
GRIDS = [("ragged", 150, 37, 9, 301), ("narrow", 1, 30, 4, 200), ("flat", 261, 1, 4, 150), ("edge", 120, 24, 4, 250)]


def _run(R, monkeypatch, w, v, src, rec, wav, env):
    for k in ("RBC_RESIDENT", "RBC_RES_TILE"):
        monkeypatch.delenv(k, raising=False)
    for k, val in env.items():
        monkeypatch.setenv(k, val)
    g, a, _ = gpu_build(R, torch, w, v)
    wt = torch.tensor(np.asarray(wav, np.float32), device="cuda")
    seis = torch.zeros((len(rec), w.nt + 1), device="cuda")
    prev, last = torch.zeros(g.padded, device="cuda"), torch.zeros(g.padded, device="cuda")
    num, den = torch.ones(g.interior, device="cuda"), torch.ones(g.interior, device="cuda")
    ctx = R.rbc_create(g, a)
    try:
        R.rbc_model(ctx, src, wt, rec, seis)
        R.rbc_get_panels(ctx, prev, last)
        R.rbc_rtm_shot(ctx, src, wt, rec, seis, R.RBC_REINJECT_SOURCE, num, den)                      # += onto ones
        num1, den1 = torch.empty_like(num), torch.empty_like(den)
        R.rbc_rtm_shot(ctx, src, wt, rec, seis, R.RBC_REINJECT_SOURCE | R.RBC_ZERO_FIRST, num1, den1)  # overwrite
        torch.cuda.synchronize()
    finally:
        R.rbc_destroy(ctx)
    assert rel((num - 1).cpu(), num1.cpu()) <= TOL and rel((den - 1).cpu(), den1.cpu()) <= TOL
    return dict(seis=seis.cpu().numpy(), prev=prev.cpu().numpy(), last=last.cpu().numpy(), num=num1.cpu().numpy(),
                den=den1.cpu().numpy())


@pytest.mark.parametrize("grid", GRIDS, ids=lambda c: c[0])
def test_every_tile_shape_matches_the_step_path_and_the_oracle(grid, monkeypatch):
    import paper_2204_03380_gb300 as R
    name, nx, nz, nb, nt = grid
    w, v, _, _, _ = case_2d(name, nx, nz, nb, nt, seed=3, layered=False)
    wav = W.ricker(nt + 90, w.dt, w.f_peak)[90:]   # from near the peak: short records carry signal
    NX, NZ = w.nx + 2 * w.nb, w.nz + 2 * w.nb
    src = np.array([min(128, NX - 1), 0, min(8, NZ - 1)], np.int32)
    xs, zs = np.arange(NX), np.arange(0, NZ, 3)
    rows = [np.stack([xs, 0 * xs, np.full_like(xs, min(z, NZ - 1))], 1) for z in (0, 7, 8)]
    cols = [np.stack([np.full_like(zs, min(x, NX - 1)), 0 * zs, zs], 1) for x in (0, 127, 128, NX - 1)]
    rec = np.concatenate(rows + cols + rows[1:2]).astype(np.int32)
    o = oracle_shot(w, v, src, rec, wav)
    ref = _run(R, monkeypatch, w, v, src, rec, wav, {"RBC_RESIDENT": "0"})
    for k in ref:
        assert rel(ref[k], o[k]) <= TOL, k
    for tile in TILES:
        got = _run(R, monkeypatch, w, v, src, rec, wav, {} if tile is None else {"RBC_RES_TILE": tile})
        for k in ref:
            assert rel(got[k], o[k]) <= TOL, (tile, k)


def test_a_shared_device_gives_the_same_results():
    import paper_2204_03380_gb300 as R
    w, v, src, rec, wav = case_2d("share", 300, 120, 10, 150)
    g, a, _ = gpu_build(R, torch, w, v)
    wt = torch.tensor(np.asarray(wav, np.float32), device="cuda")
    ctx = R.rbc_create(g, a)
    try:
        recs = []
        for n in (1, 4, 1):
            R.rbc_set_share(ctx, n)
            seis = torch.zeros((len(rec), w.nt + 1), device="cuda")
            R.rbc_model(ctx, src, wt, rec, seis)
            recs.append(seis.cpu())
        assert torch.equal(recs[0], recs[1]) and torch.equal(recs[0], recs[2])
        with pytest.raises(R.RBCError):
            R.rbc_set_share(ctx, 0)
    finally:
        R.rbc_destroy(ctx)


def test_loops_of_several_streams_that_do_not_fit_together():
    # three loops of 114 blocks and two of a few, each on its own stream, queued at once and twice over: on 152 SMs
    # the large ones have to follow one another, whichever of them the small ones run beside (a cooperative launch
    # starts as a whole or not at all, so that none of them waits half resident)
    import paper_2204_03380_gb300 as R
    runs = []
    for k, (n, nt) in enumerate([(280, 700), (280, 300), (40, 900), (280, 500), (90, 200)]):
        w, v, src, rec, wav = case_2d(f"flight{k}", n, n, 10, nt, seed=k)
        g, a, _ = gpu_build(R, torch, w, v)
        wt = torch.tensor(np.asarray(wav, np.float32), device="cuda")
        runs.append((R.rbc_create(g, a), src, wt, rec, [torch.zeros((len(rec), nt + 1), device="cuda") for _ in range(3)],
                     torch.cuda.Stream()))
    try:
        for c, src, wt, rec, out, _ in runs:
            R.rbc_model(c, src, wt, rec, out[0])
        torch.cuda.synchronize()
        for i in (1, 2):
            for c, src, wt, rec, out, s in runs:
                R.rbc_model(c, src, wt, rec, out[i], stream=s)
        torch.cuda.synchronize()
        for c, src, wt, rec, out, _ in runs:
            R.rbc_model(c, src, wt, rec, torch.empty_like(out[0]))   # (an earlier wait that ran out would be reported)
            assert torch.equal(out[0], out[1]) and torch.equal(out[0], out[2])
    finally:
        torch.cuda.synchronize()
        for r in runs:
            R.rbc_destroy(r[0])


def test_a_capturing_stream_is_refused():
    import paper_2204_03380_gb300 as R
    w, v, src, rec, wav = case_2d("capture", 60, 40, 8, 20)
    g, a, _ = gpu_build(R, torch, w, v)
    wt = torch.tensor(np.asarray(wav, np.float32), device="cuda")
    seis = torch.zeros((len(rec), w.nt + 1), device="cuda")
    ctx = R.rbc_create(g, a)
    try:
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            with pytest.raises(R.RBCError) as e:
                R.rbc_model(ctx, src, wt, rec, seis)
        assert e.value.code == 4
    finally:
        R.rbc_destroy(ctx)

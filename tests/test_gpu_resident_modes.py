"""The resident loops' other modes -- storage RTM, the FWI gradient, batches --
over the tile shapes (registers and tensor memory, several warps per quarter,
short last tiles), and the same calls by one launch per step, against the FP64
oracle.  The launch count tells which path ran."""
import numpy as np
import pytest

import oracle
import test_gpu_batch as tb
import workloads as W
from rtm_cases import TOL, case_2d, f32, gpu_build, oracle_a, rel

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

# "variant,warps" (rows per warp 1, 2, 4, 7, 10) that the grid's 55 / 233 rows can take; "step": one launch per step
LOW = ["step", None, "0,4", "0,16", "1,3", "1,16", "2,1", "2,5", "3,2", "4,2"]
TALL = [None, "2,9", "2,16", "3,9", "3,13", "3,15", "3,16", "4,9", "4,11"]
NO_REVERSE = ("step", "3,16")   # (112 rows in four buffers are more than an SM's shared memory: that adjoint runs by steps)
CASES = [("low", 150, 37, 9, 201, t) for t in LOW] + [("tall", 120, 215, 9, 200, t) for t in TALL]


def _case(name, nx, nz, nb, nt):
    w, v, _, _, _ = case_2d(name, nx, nz, nb, nt, seed=5, layered=False)
    wav = W.ricker(nt + 90, w.dt, w.f_peak)[90:]   # from near the peak: short records carry signal
    NX, NZ = w.nx + 2 * w.nb, w.nz + 2 * w.nb
    src = np.array([min(128, NX - 1), 0, NZ // 2], np.int32)
    xs, zs = np.arange(0, NX, 2), np.arange(0, NZ, 3)
    rows = [np.stack([xs, 0 * xs, np.full_like(xs, z)], 1) for z in (0, 8, NZ - 1)]
    cols = [np.stack([np.full_like(zs, x), 0 * zs, zs], 1) for x in (127, NX - 1)]
    return w, v, src, np.concatenate(rows + cols).astype(np.int32), wav


def _env(monkeypatch, tile):
    for k in ("RBC_RESIDENT", "RBC_RES_TILE"):
        monkeypatch.delenv(k, raising=False)
    if tile == "step":
        monkeypatch.setenv("RBC_RESIDENT", "0")
    elif tile is not None:
        monkeypatch.setenv("RBC_RES_TILE", tile)


@pytest.mark.parametrize("case", CASES, ids=lambda c: f"{c[0]}-{c[5]}")
def test_storage_and_gradient_match_the_oracle(case, monkeypatch):
    import paper_2204_03380_gb300 as R
    *dims, tile = case
    w, v, src, rec, wav = _case(*dims)
    _env(monkeypatch, tile)
    g, a, _ = gpu_build(R, torch, w, v)
    a64 = oracle_a(w, v)[1].astype(np.float64)
    wt = torch.tensor(np.asarray(wav, np.float32), device="cuda")
    seis = torch.zeros((len(rec), w.nt + 1), device="cuda")
    ctx = R.rbc_create(g, a)
    try:
        R.rbc_model(ctx, src, wt, rec, seis)
        d = seis.cpu().numpy()
        for k in (3, 1):
            store = torch.full((R.rbc_storage_bytes(g, k) // 4,), float("nan"), device="cuda")
            num, den = torch.empty(g.interior, device="cuda"), torch.empty(g.interior, device="cuda")
            R.rbc_launch_count(True)
            R.rbc_rtm_storage(ctx, src, wt, rec, seis, k, store, R.RBC_ZERO_FIRST, num, den)
            torch.cuda.synchronize()
            assert (R.rbc_launch_count() > w.nt) == (tile == "step")
            o = oracle.rtm_storage(a64, w.h, w.nt, src, f32(wav), rec, f32(d), w.nb, (w.nx, 1, w.nz), k, keep_store=True)
            assert rel(store.view((w.nt // k + 1,) + g.interior).cpu(), np.asarray(o["store"])) <= TOL
            assert rel(num.cpu(), o["num"]) <= TOL and rel(den.cpu(), o["den"]) <= TOL
        misfit = torch.zeros(1, dtype=torch.float64, device="cuda")
        resid, grad = torch.empty_like(seis), torch.zeros(g.interior, device="cuda")
        R.rbc_launch_count(True)
        R.rbc_fwi_forward(ctx, src, wt, rec, torch.zeros_like(seis), resid, misfit)
        R.rbc_fwi_backward(ctx, src, wt, rec, resid, None, grad)
        torch.cuda.synchronize()
        assert (R.rbc_launch_count() > w.nt) == (tile in NO_REVERSE)
        J, go = oracle.fwi_grad(a64, w.h, w.dt, w.nt, src, f32(wav), rec, np.zeros_like(d, dtype=np.float64), w.nb,
                                (w.nx, 1, w.nz))
        assert float(misfit) == pytest.approx(J, rel=TOL)
        assert rel(grad.cpu(), go) <= TOL
    finally:
        R.rbc_destroy(ctx)


@pytest.mark.parametrize("tile", [None, "2,9", "3,9", "4,9", "step"])
def test_batches_of_several_widths_match_single_shots(tile, monkeypatch):
    import paper_2204_03380_gb300 as R
    w, v, _, _, wav = _case("batch", 330, 215, 9, 120)
    wt = torch.tensor(np.asarray(wav, np.float32), device="cuda")
    wins = [(0, 330), (40, 90), (100, 230), (5, 1)]
    shots, coefs, grids = [], [], []
    for off, nx in wins:
        g, a, _ = gpu_build(R, torch, W.dataclasses.replace(w, nx=nx), v[:, off:off + nx])
        src = np.array([nx // 2 + w.nb, 0, 100], np.int32)
        xs = np.arange(0, nx, 3) + w.nb
        rec = np.stack([xs, 0 * xs, 12 + xs % 5], 1).astype(np.int32)
        seis = torch.randn((len(rec), w.nt + 1), generator=torch.Generator().manual_seed(nx)).cuda()
        shots.append(dict(src=src, rec=rec, seis=seis, off_x=off))
        coefs.append(a)
        grids.append(g)
    survey = R.make_grid(2, w.nx, 1, w.nz, w.nb, w.h, w.dt, w.nt)
    single = torch.zeros(survey.interior, device="cuda")
    monkeypatch.setenv("RBC_RESIDENT", "0")
    for sh, a, g in zip(shots, coefs, grids):
        ctx = R.rbc_create(g, a)
        num, den = torch.empty(g.interior, device="cuda"), torch.empty(g.interior, device="cuda")
        R.rbc_rtm_shot(ctx, sh["src"], wt, sh["rec"], sh["seis"], R.RBC_REINJECT_SOURCE | R.RBC_ZERO_FIRST, num, den)
        R.rbc_image_stack(g, num, den, 1e-2, sh["off_x"], 0, survey, single)
        R.rbc_destroy(ctx)
    _env(monkeypatch, tile)
    b = R.rbc_batch_create(R.make_grid(2, 1, 1, w.nz, w.nb, w.h, w.dt, w.nt), [nx for _, nx in wins], coefs)
    try:
        for _ in range(2):
            img = torch.zeros_like(single)
            R.rbc_launch_count(True)
            R.rbc_batch_rtm(b, shots, wt, R.RBC_REINJECT_SOURCE, 1e-2, img)
            torch.cuda.synchronize()
            assert (R.rbc_launch_count() > w.nt) == (tile == "step")
            assert rel(img.cpu(), single.cpu()) <= 1e-5   # the bound of the batch and single-shot paths elsewhere
    finally:
        R.rbc_batch_destroy(b)


@pytest.mark.parametrize("l2mb,groups", [(None, 1), ("0.3", 5)])
def test_the_step_path_of_a_batch_is_tuned_and_matches(l2mb, groups, monkeypatch):
    import paper_2204_03380_gb300 as R
    monkeypatch.setenv("RBC_RESIDENT", "0")
    seen = []
    info = R.rbc_batch_info
    monkeypatch.setattr(R, "rbc_batch_info", lambda b: seen.append(info(b)) or seen[-1])
    tb.test_batch_matches_single_shots_and_oracle(None, l2mb, groups, monkeypatch)
    assert any(t > 0 for t in seen[0]["tune_us"].values())   # the tuner timed its candidates


@pytest.mark.parametrize("case", [c for c in CASES if c[5] in (None, "0,4", "1,16", "2,5", "2,16", "3,9", "4,11")],
                         ids=lambda c: f"{c[0]}-{c[5]}")
def test_a_loop_in_parts_gives_the_same_bits(case, monkeypatch):
    # fields, sums, receivers, the source and the exchange words carried from part to part: every step a part of its
    # own, and parts that cut the record unevenly
    import paper_2204_03380_gb300 as R
    *dims, tile = case
    w, v, src, rec, wav = _case(*dims)
    rec = np.unique(rec, axis=0)   # (a repeated receiver's adds have no fixed order)
    _env(monkeypatch, tile)
    wt = torch.tensor(np.asarray(wav, np.float32), device="cuda")
    outs, counts = [], []
    for steps in (None, "1", "23"):
        monkeypatch.delenv("RBC_RES_STEPS", raising=False)
        if steps:
            monkeypatch.setenv("RBC_RES_STEPS", steps)
        g, a, _ = gpu_build(R, torch, w, v)
        seis = torch.zeros((len(rec), w.nt + 1), device="cuda")
        z = [torch.ones(g.interior, device="cuda") for _ in range(5)]
        store = torch.empty(R.rbc_storage_bytes(g, 3) // 4, device="cuda")
        panels = [torch.empty(g.padded, device="cuda") for _ in range(4)]
        misfit, resid = torch.zeros(1, dtype=torch.float64, device="cuda"), torch.empty_like(seis)
        R.rbc_launch_count(True)
        ctx = R.rbc_create(g, a)
        try:
            R.rbc_model(ctx, src, wt, rec, seis)
            R.rbc_get_panels(ctx, *panels[:2])
            R.rbc_rtm_shot(ctx, src, wt, rec, seis, R.RBC_REINJECT_SOURCE, *z[:2])     # += onto ones
            R.rbc_rtm_storage(ctx, src, wt, rec, seis, 3, store, R.RBC_ZERO_FIRST, *z[2:4])
            R.rbc_get_panels(ctx, *panels[2:])                                             # the forward loop's, kept
            R.rbc_fwi_forward(ctx, src, wt, rec, torch.zeros_like(seis), resid, misfit)
            R.rbc_fwi_backward(ctx, src, wt, rec, resid, None, z[4])
            torch.cuda.synchronize()
        finally:
            R.rbc_destroy(ctx)
        counts.append(R.rbc_launch_count())
        outs.append([t.cpu() for t in [seis, store, resid, *z, *panels]])
    assert counts[0] < 40 and counts[1] > 6 * w.nt > counts[2] > counts[0]
    for o in outs[1:]:
        for k, (x, y) in enumerate(zip(outs[0], o)):
            assert torch.equal(x, y), k
    assert all(float(x.abs().max()) > 0 for x in outs[0])


def test_a_batch_in_parts_gives_the_same_bits(monkeypatch):
    import paper_2204_03380_gb300 as R
    w, v, src, rec, wav = _case("bparts", 150, 37, 9, 201)
    rec = np.unique(rec, axis=0)
    wt = torch.tensor(np.asarray(wav, np.float32), device="cuda")
    g, a, _ = gpu_build(R, torch, w, v)
    seis = torch.randn((len(rec), w.nt + 1), generator=torch.Generator().manual_seed(1)).cuda()
    imgs = []
    for steps in (None, "1", "23"):
        if steps:
            monkeypatch.setenv("RBC_RES_STEPS", steps)
        b = R.rbc_batch_create(g, [150, 150], [a, a])
        try:
            for _ in range(2):
                img = torch.zeros((w.nz, 300), device="cuda")
                R.rbc_batch_rtm(b, [dict(src=src, rec=rec, seis=seis, off_x=150 * k) for k in range(2)], wt,
                                R.RBC_REINJECT_SOURCE, 1e-2, img)
                torch.cuda.synchronize()
                imgs.append(img)
        finally:
            R.rbc_batch_destroy(b)
    assert all(torch.equal(imgs[0], i) for i in imgs) and float(imgs[0].abs().max()) > 0
    assert torch.equal(imgs[0][:, :150], imgs[0][:, 150:])


@pytest.mark.parametrize("tile,every,steps", [("2,9", 1, True), ("2,9", 4, False), ("0,8", 1, False)])
def test_records_of_most_nodes_match_whichever_path_takes_them(tile, every, steps, monkeypatch):
    # more receivers than a warp's turns are worth go by launches: 4 rows per warp hold 32 and take 64 more
    import paper_2204_03380_gb300 as R
    w, v, src, _, wav = _case("dense", 120, 215, 9, 60)
    X, Z = np.meshgrid(np.arange(0, w.nx + 2 * w.nb, every), np.arange(w.nz + 2 * w.nb))
    rec = np.stack([X.ravel(), 0 * X.ravel(), Z.ravel()], 1).astype(np.int32)
    wt = torch.tensor(np.asarray(wav, np.float32), device="cuda")
    out = []
    for t in ("step", tile):
        _env(monkeypatch, t)
        g, a, _ = gpu_build(R, torch, w, v)
        seis = torch.zeros((len(rec), w.nt + 1), device="cuda")
        ctx = R.rbc_create(g, a)
        try:
            R.rbc_launch_count(True)
            R.rbc_model(ctx, src, wt, rec, seis)
            torch.cuda.synchronize()
            assert (R.rbc_launch_count() > w.nt) == (steps or t == "step")
        finally:
            R.rbc_destroy(ctx)
        out.append(seis.cpu())
    assert torch.equal(*out) and float(out[0].abs().max()) > 0

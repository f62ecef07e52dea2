"""Contexts that share the device: rbc_set_share, and contexts or batches
whose loops' tables find no memory."""
import numpy as np
import pytest

from rtm_cases import case_2d, gpu_build

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _ctx(R, name, nx, nz, nb, nt, seed=0):
    w, v, src, rec, wav = case_2d(name, nx, nz, nb, nt, seed=seed)
    g, a, _ = gpu_build(R, torch, w, v)
    wt = torch.tensor(np.asarray(wav, np.float32), device="cuda")
    return R.rbc_create(g, a), g, a, src, rec, wt, torch.zeros((len(rec), nt + 1), device="cuda")


def test_a_change_of_share_waits_for_nothing_and_allocates_nothing():
    import paper_2204_03380_gb300 as R
    long, _, _, src, rec, wt, out = _ctx(R, "long", 300, 300, 50, 30000)   # some 50 ms
    other, _, _, src2, rec2, wt2, out2 = _ctx(R, "other", 400, 300, 50, 60)
    try:
        R.rbc_model(long, src, wt, rec, out)
        for n in (2, 5, 3):   # (kernels are loaded at their first launch)
            R.rbc_set_share(other, n)
            R.rbc_model(other, src2, wt2, rec2, out2)
        torch.cuda.synchronize()
        free = torch.cuda.mem_get_info()[0]
        R.rbc_model(long, src, wt, rec, out)
        done = torch.cuda.Event()
        done.record()
        for n in (2, 5, 1, 3):
            R.rbc_set_share(other, n)
        assert not done.query()                       # the loop is still running: nothing waited for it
        R.rbc_model(other, src2, wt2, rec2, out2)     # with tables of another share
        torch.cuda.synchronize()
        assert torch.cuda.mem_get_info()[0] == free
    finally:
        torch.cuda.synchronize()
        R.rbc_destroy(long)
        R.rbc_destroy(other)


def test_a_context_whose_tables_find_no_memory_steps():
    import paper_2204_03380_gb300 as R
    runs = []
    for mode in (0, 3):
        R.rbc_inject_fault(None, mode)
        ctx, _, _, src, rec, wt, out = _ctx(R, "nomem", 150, 60, 10, 120)
        try:
            for n in (1, 4):
                R.rbc_set_share(ctx, n)
                R.rbc_launch_count(True)
                R.rbc_model(ctx, src, wt, rec, out)
                torch.cuda.synchronize()
                assert (R.rbc_launch_count() > 120) == (mode == 3)
        finally:
            R.rbc_destroy(ctx)
        runs.append(out.cpu())
    assert torch.equal(*runs) and float(runs[0].abs().max()) > 0


def test_a_batch_whose_tables_find_no_memory_steps():
    import paper_2204_03380_gb300 as R
    c0, g, a, src, rec, wt, seis = _ctx(R, "bnomem", 150, 60, 10, 120)
    R.rbc_model(c0, src, wt, rec, seis)
    R.rbc_destroy(c0)
    imgs = []
    for mode in (0, 3):
        R.rbc_inject_fault(None, mode)
        b = R.rbc_batch_create(g, [150], [a])
        try:
            img = torch.zeros(g.interior, device="cuda")
            R.rbc_launch_count(True)
            R.rbc_batch_rtm(b, [dict(src=src, rec=rec, seis=seis, off_x=0)], wt, R.RBC_REINJECT_SOURCE, 1e-2, img)
            torch.cuda.synchronize()
            assert (R.rbc_launch_count() > 120) == (mode == 3)
        finally:
            R.rbc_batch_destroy(b)
        imgs.append(img)
    assert float((imgs[0] - imgs[1]).norm()) <= 1e-5 * float(imgs[0].norm()) and float(imgs[0].norm()) > 0


@pytest.mark.parametrize("nx,nz,nb,share", [(300, 300, 50, 40), (1000, 600, 50, 2), (1000, 600, 50, 3), (2301, 751, 60, 2)])
def test_any_share_gives_the_same_record(nx, nz, nb, share):
    # side by side, in turn, or by launches
    import paper_2204_03380_gb300 as R
    ctx, _, _, src, rec, wt, out = _ctx(R, "many", nx, nz, nb, 60)
    try:
        recs = []
        for n in (1, share, 1):
            R.rbc_set_share(ctx, n)
            R.rbc_model(ctx, src, wt, rec, out)
            recs.append(out.cpu())
        assert torch.equal(recs[0], recs[1]) and torch.equal(recs[0], recs[2]) and float(recs[0].abs().max()) > 0
    finally:
        R.rbc_destroy(ctx)


def test_contexts_on_streams_of_their_own_run_side_by_side():
    # four contexts of 400 x 400 padded nodes, no rbc_set_share: with the whole device for each loop they would take
    # four times as long as one; side by side they take some 1.5 times (one launch per step: 2.2 times)
    import paper_2204_03380_gb300 as R
    runs = [_ctx(R, f"own{k}", 300, 300, 50, 4000, seed=k) for k in range(4)]
    streams = [torch.cuda.Stream() for _ in runs]
    try:
        def timed(n):
            t = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
            main = torch.cuda.current_stream()
            t[0].record(main)
            for (ctx, _, _, src, rec, wt, out), s in zip(runs[:n], streams):
                s.wait_event(t[0])
                R.rbc_model(ctx, src, wt, rec, out, stream=s)
                main.wait_stream(s)
            t[1].record(main)
            torch.cuda.synchronize()
            return t[0].elapsed_time(t[1])

        first = [None] * len(runs)
        timed(4)
        for k, r in enumerate(runs):
            first[k] = r[-1].clone()
        together = min(timed(4) for _ in range(3))
        alone = min(timed(1) for _ in range(4))   # (the first of these still counts the others)
        assert together < 0.6 * 4 * alone, (together, alone)
        for k, r in enumerate(runs):
            assert torch.equal(r[-1], first[k])
    finally:
        torch.cuda.synchronize()
        for r in runs:
            R.rbc_destroy(r[0])


def test_a_kernel_on_another_stream_runs_before_a_long_loop_ends():
    # the loop takes every SM's shared memory for some 40 ms in all, and the denoiser's kernels need most of an SM's
    import paper_2204_03380_gb300 as R
    from paper_2204_03380_gb300.denoise import Denoiser
    ctx, _, _, src, rec, wt, out = _ctx(R, "survey", 2301, 751, 60, 12000)
    net, x = Denoiser(seed=1), torch.randn((1, 200, 200), device="cuda")
    loop, side = torch.cuda.Stream(), torch.cuda.Stream()
    try:
        ref = net(x)
        R.rbc_model(ctx, src, wt, rec, out, stream=loop)
        torch.cuda.synchronize()
        R.rbc_model(ctx, src, wt, rec, out, stream=loop)
        done = torch.cuda.Event()
        done.record(loop)
        with torch.cuda.stream(side):
            y = net(x)
            ready = torch.cuda.Event()
            ready.record(side)
        ready.synchronize()
        assert not done.query()
        torch.cuda.synchronize()
        assert torch.equal(y, ref)
    finally:
        torch.cuda.synchronize()
        R.rbc_destroy(ctx)


def test_batches_on_streams_of_their_own_run_side_by_side():
    # four batches of one shot of 300 x 300 padded nodes: one after the other they would take four times as long as
    # one; side by side some 1.5 times (one launch per step: 2.1 times)
    import paper_2204_03380_gb300 as R
    c0, g, a, src, rec, wt, seis = _ctx(R, "bown", 200, 200, 50, 3000)
    R.rbc_model(c0, src, wt, rec, seis)
    torch.cuda.synchronize()
    R.rbc_destroy(c0)
    batches = [R.rbc_batch_create(g, [200], [a]) for _ in range(4)]
    imgs = [torch.zeros(g.interior, device="cuda") for _ in batches]
    streams = [torch.cuda.Stream() for _ in batches]
    shot = dict(src=src, rec=rec, seis=seis, off_x=0)
    try:
        def timed(n):
            t = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
            main = torch.cuda.current_stream()
            for i in imgs:
                i.zero_()
            t[0].record(main)
            for b, i, s in zip(batches[:n], imgs, streams):
                s.wait_event(t[0])
                R.rbc_batch_rtm(b, [shot], wt, R.RBC_REINJECT_SOURCE, 1e-2, i, stream=s)
                main.wait_stream(s)
            t[1].record(main)
            torch.cuda.synchronize()
            return t[0].elapsed_time(t[1])

        timed(4)
        together = min(timed(4) for _ in range(3))
        assert all(torch.equal(i, imgs[0]) for i in imgs) and float(imgs[0].abs().max()) > 0
        beside = imgs[0].clone()
        alone = min(timed(1) for _ in range(4))
        assert together < 0.6 * 4 * alone, (together, alone)
        assert torch.equal(beside, imgs[0])
    finally:
        torch.cuda.synchronize()
        for b in batches:
            R.rbc_batch_destroy(b)


def test_loops_with_tensor_memory_in_flight_together(monkeypatch):
    # reverse loops of low tiles, whose fields take little of an SM: 4, 7 and 10 rows per warp hold 256, 512 and 512
    # tensor-memory columns, which must not meet on an SM
    import paper_2204_03380_gb300 as R
    runs = []
    for k, tile in enumerate(("2,3", "3,2", "4,1", "2,5")):
        monkeypatch.setenv("RBC_RES_TILE", tile)
        ctx, g, _, src, rec, wt, seis = _ctx(R, f"tm{k}", 500, 250, 20, 300, seed=k)
        num = [torch.empty(g.interior, device="cuda") for _ in range(3)]
        runs.append((ctx, src, wt, rec, seis, num, torch.cuda.Stream()))
    flags = R.RBC_REINJECT_SOURCE | R.RBC_ZERO_FIRST
    R.rbc_launch_count(True)
    try:
        for n in range(2):   # one by one, then in flight together and several times over
            for _ in range(1 + 3 * n):
                for ctx, src, wt, rec, seis, num, s in runs:
                    R.rbc_set_share(ctx, 1)
                    if n == 0:
                        R.rbc_model(ctx, src, wt, rec, seis)
                    R.rbc_rtm_shot(ctx, src, wt, rec, seis, flags, num[n], num[2], stream=s if n else None)
            torch.cuda.synchronize()
        assert R.rbc_launch_count() < 300
        for ctx, src, wt, rec, seis, num, _ in runs:
            assert torch.equal(*num[:2]) and float(num[0].abs().max()) > 0
            R.rbc_model(ctx, src, wt, rec, seis)   # (an earlier wait that ran out would be reported)
    finally:
        torch.cuda.synchronize()
        for r in runs:
            R.rbc_destroy(r[0])


def test_contexts_of_several_host_threads():
    # every thread makes, uses and destroys contexts of its own on a stream of its own while the others do; the counts
    # and so the plans change from call to call, the records do not
    import threading

    import paper_2204_03380_gb300 as R
    cases = [_ctx(R, f"thr{k}", 120 + 90 * k, 80 + 40 * k, 10, 120, seed=k) for k in range(5)]
    want = []
    for ctx, _, _, src, rec, wt, out in cases:
        R.rbc_model(ctx, src, wt, rec, out)
        torch.cuda.synchronize()
        want.append(out.clone())
        R.rbc_destroy(ctx)
    errors = []

    def work(k):
        try:
            _, g, a, src, rec, wt, _ = cases[k]
            s = torch.cuda.Stream()
            with torch.cuda.stream(s):
                for _ in range(3):
                    ctx = R.rbc_create(g, a)
                    try:
                        for _ in range(6):
                            got = torch.zeros_like(want[k])
                            R.rbc_model(ctx, src, wt, rec, got, stream=s)
                            s.synchronize()
                            assert torch.equal(got, want[k])
                    finally:
                        R.rbc_destroy(ctx)
        except BaseException as e:   # reported by the main thread
            errors.append((k, e))

    threads = [threading.Thread(target=work, args=(k,)) for k in range(len(cases))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors

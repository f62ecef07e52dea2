"""A resident loop whose blocks wait for edges that never come: every wait
ends, the next call reports it, and the loop's later parts do not wait again.
The edges are missing because the host withheld the part that sends them."""
import time

import numpy as np
import pytest

from rtm_cases import case_2d, gpu_build

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_a_wait_that_runs_out_is_reported_by_the_next_call(monkeypatch):
    import paper_2204_03380_gb300 as R
    monkeypatch.setenv("RBC_RES_STEPS", "5")
    w, v, src, rec, wav = case_2d("wait", 200, 60, 8, 100)
    g, a, _ = gpu_build(R, torch, w, v)
    wt = torch.tensor(np.asarray(wav, np.float32), device="cuda")
    clean, seis = (torch.zeros((len(rec), w.nt + 1), device="cuda") for _ in range(2))
    ctx = R.rbc_create(g, a)
    try:
        R.rbc_model(ctx, src, wt, rec, clean)
        R.rbc_inject_fault(ctx, 2)
        R.rbc_launch_count(True)
        t0 = time.perf_counter()
        R.rbc_model(ctx, src, wt, rec, seis)              # 19 of its 20 parts
        torch.cuda.synchronize()                          # the device finished
        took = time.perf_counter() - t0
        assert R.rbc_launch_count() == 20                 # 19 parts and the record's transposition
        assert 0.1 < took < 30                            # one wait, not nineteen
        with pytest.raises(R.RBCError) as e:
            R.rbc_model(ctx, src, wt, rec, seis)
        assert e.value.code == 5                          # RBC_ETIMEOUT, reported once
        R.rbc_model(ctx, src, wt, rec, seis)
        torch.cuda.synchronize()
        assert torch.equal(seis, clean) and float(clean.abs().max()) > 0
    finally:
        R.rbc_destroy(ctx)

"""A limit reached while other warps have parked their packets for the next
round of the peeling-ray buffer: every packet that was started has its status
written, and those that had ended have their results, as in a run without
limits.  The limits run out on purpose with small values; nothing faults."""
import numpy as np
import pytest

import synth
from gpu_util import context, gpu_run

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("limit", [5, 7, 9, 12, 16, 24])
def test_started_packets_are_all_written(limit):
    import torch
    import paper_2001_11252_gb300 as rg
    n = 250_000
    wl = synth.sphere(tau0=1e4, T=1e4, tau_dust=1.0, n_packets=n, base=3, max_level=4)
    wl.detector.dirs = np.array([[0.0, 0.0, 1.0]])
    wl.physics.max_scatt = 3
    ctx = context(wl)
    ctx.set_peel_capacity(1)   # the least that the launch shape allows
    ref, st = gpu_run(ctx, wl.packets)
    assert st["packets"] == n
    dev = torch.device("cuda:0")
    pk = wl.packets
    t = lambda a, dt: torch.as_tensor(np.ascontiguousarray(a)).to(dev, dt)
    args = (t(pk.pos, torch.float64), t(pk.dir, torch.float64), t(pk.nu, torch.float64),
            t(pk.ids.view(np.int64), torch.int64))
    out = {"status": torch.full((n,), -1, dtype=torch.int32, device=dev),
           "nscatt": torch.full((n,), -1, dtype=torch.int64, device=dev)}
    ctx.set_limits(max_iterations=limit)
    try:
        ctx.propagate(*args, out=out)   # the larger limits may be enough
    except rg.RascasError as e:
        assert "E_TIMEOUT" in str(e)
    status, nscatt = out["status"].cpu().numpy(), out["nscatt"].cpu().numpy()
    started = np.flatnonzero(status != -1)
    # packets leave the queue in order: those started are the first of the list
    assert len(started) == started.max() + 1, (len(started), started.max() + 1)
    ended = started[status[started] != rg.PK_ACTIVE]
    print(limit, "started", len(started), "ended", len(ended))
    assert (status[ended] == ref["status"][ended]).all() and (nscatt[ended] == ref["nscatt"][ended]).all()
    # no limit again: the whole run, as before
    ctx.set_limits(0, 0.0)
    again, st = gpu_run(ctx, pk)
    assert st["packets"] == n
    for k in ref:
        assert again[k].tobytes() == ref[k].tobytes(), k

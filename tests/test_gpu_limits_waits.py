"""max_iterations counts the walk steps of a thread, not the iterations in which
it waits for others: a launch that fills every thread with one packet of 64
steps completes with a budget of a few more, and gives up with one of fewer."""
import numpy as np
import pytest

import synth
from gpu_util import context, gpu_run

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("peel", [False, True])
def test_waiting_spends_nothing(peel):
    import torch
    import paper_2001_11252_gb300 as rg
    n = 512 * torch.cuda.get_device_properties(0).multi_processor_count
    wl = synth.sphere(tau0=1e6, T=1e4, n_packets=n, base=3, max_level=5)
    if peel:
        wl.detector.dirs = np.array([[0.0, 0.0, 1.0]])
    wl.physics.max_steps = 64
    ctx = context(wl)
    ref, st = gpu_run(ctx, wl.packets)
    assert st["capped"] == n   # 64 steps each
    ctx.set_limits(max_iterations=72)
    got, st = gpu_run(ctx, wl.packets)
    assert st["capped"] == n
    for k in ref:
        assert got[k].tobytes() == ref[k].tobytes(), k
    ctx.set_limits(max_iterations=60)
    with pytest.raises(rg.RascasError) as e:
        gpu_run(ctx, wl.packets)
    assert "E_TIMEOUT" in str(e.value)

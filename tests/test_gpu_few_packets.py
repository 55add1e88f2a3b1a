"""Launches of few packets give some lanes of each warp no work: a packet's
results are the same, bit for bit, for every number of packets around the
limits of that rule (lanes, warps and one more or less)."""
import numpy as np
import pytest

import synth
from gpu_util import context, gpu_run

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("peel", [False, True])
def test_results_do_not_depend_on_the_number_of_packets(peel):
    import torch
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    warps = 8 * sms
    n = 32 * warps + 1
    kw = dict(N_HI=2e15, tau_dust=0.3, v_max_kms=50.0, n_packets=n, base=3, max_level=4, npix=4, nchan=8)
    wl = synth.expanding_sphere(**kw) if peel else synth.sphere(tau0=100.0, T=1e4, n_packets=n, base=3, max_level=4)
    ctx = context(wl)
    pk = wl.packets
    g, st = gpu_run(ctx, pk)
    assert st["packets"] == n
    for m in (1, 2, 31, 33, warps - 1, warps, warps + 1, 2 * warps + 1, 31 * warps + 1, 32 * warps):
        r, st = gpu_run(ctx, synth.Packets(pk.pos[:m], pk.dir[:m], pk.nu[:m], pk.ids[:m]))
        assert st["packets"] == m
        for k in r:
            assert r[k].tobytes() == g[k][:m].tobytes(), (k, m)

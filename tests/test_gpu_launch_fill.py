"""Launches around the number of resident threads, where lanes begin to wait for
company, and spreads of few packets over warps by each branch of that rule:
a packet's results are those of the same packet in a small launch, bit for bit,
with one and several lines, in gas at rest and in a fast wind, and with peeling
rays parked and drained many times over."""
import numpy as np
import pytest

import synth
from gpu_util import context, gpu_run

pytestmark = pytest.mark.gpu


def _sms():
    import torch
    return torch.cuda.get_device_properties(0).multi_processor_count


def _workload(which, n):
    if which == "rest":
        return synth.sphere(tau0=100.0, T=1e4, n_packets=n, base=3, max_level=4)
    if which == "lines":
        wl = synth.sphere(tau0=100.0, T=1e4, tau_dust=0.5, n_packets=n, base=3, max_level=4)
        wl.lines = wl.lines + [synth.d_lya(0.3)]
        return wl
    if which == "wind":
        wl = synth.expanding_sphere(N_HI=2e13, T=1e3, v_max_kms=300.0, n_packets=n, base=3, max_level=4)
        wl.detector.dirs = wl.detector.dirs[:0]
        wl.detector.npix = wl.detector.cube = 0
        return wl
    return synth.expanding_sphere(N_HI=2e15, tau_dust=0.3, v_max_kms=50.0, n_packets=n, base=3, max_level=4, npix=4,
                                  nchan=8)


def _check(ctx, pk, ref, a, b):
    r, st = gpu_run(ctx, synth.Packets(pk.pos[a:b], pk.dir[a:b], pk.nu[a:b], pk.ids[a:b]))
    assert st["packets"] == b - a
    for k in r:
        assert r[k].tobytes() == ref[k][a:b].tobytes(), (k, a, b)


@pytest.mark.parametrize("which", ["rest", "lines", "wind", "peel"])
def test_results_do_not_depend_on_the_fill(which):
    sms = _sms()
    full = 512 * sms      # resident threads
    wl = _workload(which, full + 1)
    ctx = context(wl)
    if which == "peel":
        ctx.set_peel_capacity(1)   # the least that the launch shape allows: many rounds
    pk = wl.packets
    ref, st = gpu_run(ctx, pk)   # lanes wait
    assert st["packets"] == full + 1
    for n in (full - 1, full):
        _check(ctx, pk, ref, 0, n)
    # pieces of the list, spread over warps by each of the shares
    for a, n in ((0, 1), (7, sms), (99, sms + 1), (1000, 3 * sms), (5000, 3 * sms + 1), (9000, 8 * sms), (20000, 8 * sms + 1),
                 (0, 32 * sms), (123, 32 * sms + 1), (1, 96 * sms + 1), (2, 256 * sms), (3, 256 * sms + 1)):
        _check(ctx, pk, ref, a, a + n)

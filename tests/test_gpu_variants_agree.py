"""A packet's history is the same, bit for bit, in the plain kernel, the one
that peels and the one of batches, for either H(a, x), for one to four lines
of comparable strength (one of them fluorescent) and over temperatures from
0.1 to 1e5 K: no rounding on its path is left to the compiler's choice in one
kernel or the other."""
import numpy as np
import pytest

import synth
from gpu_util import gpu_run

pytestmark = pytest.mark.gpu

KEYS = ("status", "nscatt", "nu", "pos", "dir", "path")


def _workload(nline, voigt, n):
    wl = synth.expanding_sphere(N_HI=2e14, tau_dust=0.5, v_max_kms=20.0, n_packets=n, base=3, max_level=4, npix=4,
                                nchan=8)
    H = synth.MP_CGS
    others = [synth.Line("B", 1215.34, 6.265e8, 0.416, 2 * H, density=2, abundance=0.6),
              synth.Line("C", 1215.5, 6.265e8, 0.416, 2.5 * H, density=2, abundance=0.5),
              synth.Line("D", 1215.8, 6.265e8, 0.416, 3.5 * H, density=2, abundance=0.4, phase=1,
                         channels=[(3e8, 1300.0)])]
    wl.lines = wl.lines + others[4 - nline:]   # the fluorescent one wherever there are two
    rng = np.random.default_rng(11)
    wl.medium.T = (10 ** rng.uniform(-1, 5, len(wl.medium.T))).astype(np.float32)
    wl.medium.n_HI = (wl.medium.n_HI * np.sqrt(wl.medium.T / 1e4)).astype(np.float32)
    wl.physics.voigt = voigt
    wl.physics.max_scatt = 16
    return wl


@pytest.mark.parametrize("voigt", [0, 1])
@pytest.mark.parametrize("nline", [1, 2, 3, 4])
def test_plain_peeling_and_batch_histories(nline, voigt):
    import paper_2001_11252_gb300 as rg
    wl = _workload(nline, voigt, 60000)
    ctx = rg.Context(0)
    ctx.setup(wl)
    peel, st = gpu_run(ctx, wl.packets)
    assert st["npeel_rays"] > 0 and st["nscatt_line"] > wl.packets.n
    wl.detector.dirs = wl.detector.dirs[:0]
    wl.detector.npix = wl.detector.cube = 0
    ctx.setup(wl)
    plain, _ = gpu_run(ctx, wl.packets)
    ctx.load_batch([wl], nbin=8)
    batch, _ = ctx.propagate_batch_packets()
    for k in KEYS:
        assert peel[k].tobytes() == plain[k].tobytes(), ("peel", k, int((peel[k] != plain[k]).sum()))
        assert batch[k].tobytes() == plain[k].tobytes(), ("batch", k, int((batch[k] != plain[k]).sum()))

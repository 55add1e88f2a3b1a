"""Steps that draw as many words as a step can (a decay channel, several
rejection trials, core-skipping) take the words of the packet's stream: each
event replayed by the oracle from the GPU's state draws the same number and
ends in the same place, within the FP32 sampling tolerances of the other
replays."""
import pytest

import synth
from gpu_util import replay_steps

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("core_skip", [0.0, 2.0])
@pytest.mark.parametrize("nline", [1, 3])
def test_steps_with_every_draw(core_skip, nline):
    # a second channel that is hardly ever taken: its draw is made at every
    # scattering; a is large where it is cold, and trials fail often
    wl = synth.sphere(tau0=1e5, T=1e2, tau_dust=0.5, n_packets=64, base=3, max_level=5)
    wl.lines[0].channels = [(1e5, 1300.0)]
    wl.lines = wl.lines + [synth.d_lya(0.2), synth.d_lya(0.1)][:nline - 1]
    wl.physics.core_skip = core_skip
    st = replay_steps(wl, 64, 200)
    print(core_skip, nline, st)
    assert st["steps"] > 1000
    assert st["mismatch"] <= 0.002 * st["steps"] + 2
    assert st["pos"] < 1e-6 and st["dir"] < 1e-6 and st["x"] < 3e-5

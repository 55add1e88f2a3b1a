"""The per-temperature constants a lane keeps from leaf to leaf, and from one
packet to the next (Doppler widths, Voigt parameters, u0 coefficients): a
packet's results must be the same, bit for bit, whether its lane ran other
packets before it (a launch of more packets than lanes) or started with none
(a launch of that packet alone), in media where neighbouring leaves share a
temperature, alternate between two, or all differ."""
import numpy as np
import pytest

import synth
from gpu_util import context, gpu_run

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("temps", ["one", "two", "all"])
@pytest.mark.parametrize("lines,v_kms", [("lya", 0.0), ("deuterium", 40.0)])
def test_results_do_not_depend_on_the_lane(temps, lines, v_kms):
    n = 120_000
    wl = synth.sphere(tau0=100.0, T=1e4, n_packets=n, base=3, max_level=4)
    if lines == "deuterium":
        wl.lines = wl.lines + [synth.d_lya()]
    med = wl.medium
    if temps == "two":
        med.T[:] = np.where(med.tree.leaf_ijk.sum(1) % 2 == 0, 1e4, 2.5e4)
    elif temps == "all":
        med.T[:] = 10.0 ** np.random.default_rng(11).uniform(3.0, 5.0, med.tree.nleaf)
    v = (v_kms * 1e5 / wl.domain.size) * (med.tree.leaf_centres() - 0.5)
    med.vx, med.vy, med.vz = (v[:, i].astype(np.float32) for i in range(3))
    ctx = context(wl)
    pk = wl.packets
    g, _ = gpu_run(ctx, pk)
    assert (g["status"] == 1).all()
    for i in list(range(4)) + list(np.random.default_rng(3).integers(0, n, 60)):
        one = synth.Packets(pk.pos[i:i + 1], pk.dir[i:i + 1], pk.nu[i:i + 1], pk.ids[i:i + 1])
        r, _ = gpu_run(ctx, one)
        for k in r:
            assert r[k].tobytes() == g[k][i:i + 1].tobytes(), (k, int(i))

"""Set-up calls on a context whose stream is a non-blocking one: the tree, its
face links and the leaf records are complete and those of the last call, also
where smaller and larger trees replace each other in the same buffers."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu


def _sphere(level, dust):
    return synth.sphere(tau0=1e3, T=1e4, tau_dust=dust, n_packets=1, base=2, max_level=level)


def test_trees_reloaded_on_a_side_stream():
    import torch
    import paper_2001_11252_gb300 as rg
    rng = np.random.default_rng(3)
    n = 64
    pos = 0.5 + rng.uniform(-0.15, 0.15, (n, 3))
    d = rng.normal(size=(n, 3))
    d /= np.linalg.norm(d, axis=1)[:, None]
    ctx = rg.Context(0)
    side = torch.cuda.Stream()
    ctx.set_stream(side)
    for level, dust in ((5, 0.5), (3, 1.0), (6, 0.25), (4, 2.0), (6, 0.5)):
        wl = _sphere(level, dust)
        nu = np.full(n, synth.nu_of(wl.lines[0].lambda_A) * (1.0 + 1e-4))
        ctx.setup(wl)
        tau, cells, lens, ncell = ctx.ray_tau(pos, d, nu, cap=512)
        o = oracle.Oracle(wl)
        for i in range(n):
            _, c_o, l_o, n_o = o.ray_tau(pos[i], d[i], nu[i], cap=512)
            assert ncell[i] == n_o and (cells[i, :n_o] == c_o).all(), (level, i)
            assert lens[i, :n_o].tobytes() == l_o[:n_o].tobytes(), (level, i)
        # the domain alone, then the fields alone: both rewrite the records
        wl.domain.size = 0.3
        ctx.set_domain(wl.domain.kind, wl.domain.centre, wl.domain.size)
        m = wl.medium
        m.n_dust = (m.n_dust * 3).astype(np.float32)
        ctx.update_fields(m.n_HI, m.vx, m.vy, m.vz, m.T, m.n_dust)
        tau, _, _, ncell = ctx.ray_tau(pos, d, nu)
        o = oracle.Oracle(wl)
        for i in range(n):
            t_o, _, _, n_o = o.ray_tau(pos[i], d[i], nu[i], cap=512)
            # tau within 1e-6 of the oracle, as in the other ray tests
            assert ncell[i] == n_o and abs(tau[i] - t_o) <= 1e-6 * abs(t_o), (level, i)
    ctx.close()

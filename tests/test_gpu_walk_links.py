"""The ray walks by face links with the exit face chosen in FP32: the leaves
and FP64 path lengths must be the oracle's, bit for bit, on trees where the
general search is needed (levels that jump by more than one, a one-level
tree, a periodic slab) and on rays where the FP32 choice cannot tell (ties
between axes, directions along axes and with components next to zero, starts
on faces, edges and corners); and a ray's result must not depend on how many
rays share the launch."""
import numpy as np
import pytest

import oracle
import synth
from gpu_util import context

pytestmark = pytest.mark.gpu


def _workload(which):
    wl = synth.sphere(tau0=1e3, T=1e4, tau_dust=0.5, n_packets=1, base=2, max_level=3)
    if which == "slab":
        wl = synth.slab(tau0=1e3, n_packets=1, level=3)
    elif which == "root":
        wl.medium = synth.uniform_medium(synth.uniform_octree(1), wl.medium.box_cm, 1e-3, 1e4, 1e-3)
        wl.domain = synth.Domain(2, (0.5, 0.5, 0.5), 0.5)
    elif which == "jumps":
        # one corner refined to level 12 next to leaves of level 2, the
        # opposite corner to level 7
        def refine(l, i, j, k):
            n = (1 << l) - 1
            return (l < 2) | ((i + j + k) == 0) | ((l < 7) & (i == n) & (j == n) & (k == n))
        tree = synth.build_octree(refine, 12)
        wl.medium = synth.uniform_medium(tree, wl.medium.box_cm, 1e-3, 1e4, 1e-3)
        wl.domain = synth.Domain(2, (0.5, 0.5, 0.5), 0.5)
    return wl


def _rays(n, seed):
    rng = np.random.default_rng(seed)
    pos = rng.uniform(0.0, 1.0, (n, 3))
    d = rng.normal(size=(n, 3))
    q = n // 8
    pos[:q] = np.floor(pos[:q] * 16) / 16                      # faces, edges, corners
    pos[q:2 * q] *= 2.0 ** -rng.integers(1, 11, (q, 1))         # towards the refined corner
    d[:q:2] = np.sign(d[:q:2])                                  # diagonals: ties between axes
    d[1:q:4, 0] = 0.0
    d[q:2 * q:5] = np.eye(3)[rng.integers(0, 3, len(d[q:2 * q:5]))] * np.where(rng.random((len(d[q:2 * q:5]), 1)) < 0.5, -1, 1)
    d[2 * q:3 * q, 1] *= 10.0 ** -rng.uniform(5, 300, q)       # next to zero
    d[3 * q:4 * q, 2] = d[3 * q:4 * q, 0] * (1.0 + 2.0 ** -rng.uniform(15, 52, q))   # nearly tied
    d /= np.linalg.norm(d, axis=1)[:, None]
    return pos, d


@pytest.mark.parametrize("which", ["sphere", "slab", "root", "jumps"])
def test_leaves_and_lengths_equal_the_oracle(which):
    wl = _workload(which)
    ctx = context(wl)
    o = oracle.Oracle(wl)
    pos, d = _rays(800, 5)
    if which == "slab":
        d[:, 2] = np.where(np.abs(d[:, 2]) < 0.05, 0.05, d[:, 2])   # a ray in the plane never ends
    nu = np.full(len(pos), synth.nu_of(wl.lines[0].lambda_A) * (1.0 + 1e-4))
    cap = 2048
    tau, cells, lens, ncell = ctx.ray_tau(pos, d, nu, cap=cap)
    cols, _, nc = ctx.ray_columns(pos, d)
    assert (nc == ncell).all()
    for i in range(len(pos)):
        t_o, c_o, l_o, n_o = o.ray_tau(pos[i], d[i], nu[i], cap=cap)
        assert ncell[i] == n_o, i
        m = min(n_o, cap)
        assert (cells[i, :m] == c_o[:m]).all() and lens[i, :m].tobytes() == l_o[:m].tobytes(), i
        # tau within 1e-6 of the oracle, as in the other ray tests
        assert abs(tau[i] - t_o) <= 1e-6 * abs(t_o) + 1e-300, i


def test_rays_do_not_depend_on_their_number():
    import torch
    warps = 8 * torch.cuda.get_device_properties(0).multi_processor_count
    n = 32 * warps + 1
    wl = _workload("jumps")
    ctx = context(wl)
    pos, d = _rays(n, 6)
    nu = np.full(n, synth.nu_of(wl.lines[0].lambda_A))
    tau, _, _, ncell = ctx.ray_tau(pos, d, nu)
    cols, _, _ = ctx.ray_columns(pos, d)
    for m in (1, 33, warps, warps + 1, 31 * warps + 1, 32 * warps):
        t, _, _, c = ctx.ray_tau(pos[:m], d[:m], nu[:m])
        q, _, _ = ctx.ray_columns(pos[:m], d[:m])
        assert t.tobytes() == tau[:m].tobytes() and (c == ncell[:m]).all() and q.tobytes() == cols[:m].tobytes(), m

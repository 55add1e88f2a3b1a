"""The reads that a run's statistics count for a peeling ray are those of the
general neighbour search, which the scattering kernel counts for a packet: a
packet and a peeling ray that cross the same leaves of a medium without opacity
add the same numbers, on trees and directions where the ray's face links do not
hold as well."""
import numpy as np
import pytest

import synth
from gpu_util import gpu_run
from test_gpu_walk_links import _workload

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("direction", [(1, 1, 1), (-1, 1, -1), (1, 1, 0), (0, 0, 1), (0.3, -0.5, 0.7), (1, 1 + 2e-16, 1 - 3e-16)])
@pytest.mark.parametrize("which", ["sphere", "slab", "root", "jumps"])
def test_rays_count_what_packets_count(which, direction):
    import paper_2001_11252_gb300 as rg
    wl = _workload(which)
    if which == "slab" and direction[2] == 0:
        direction = (1, 1, 0.05)   # a packet in the plane never ends
    med = wl.medium
    med.n_HI, med.n_dust = np.zeros_like(med.n_HI), np.zeros_like(med.n_dust)
    n = 3000
    rng = np.random.default_rng(7)
    pos = rng.uniform(0.2, 0.8, (n, 3))
    pos[:n // 2] = np.floor(pos[:n // 2] * 16) / 16              # faces, edges, corners
    pos[n // 3:n // 2] = 0.5 + (pos[n // 3:n // 2] - 0.5) / 512
    if which == "jumps":
        pos[n // 2:2 * n // 3] *= 2.0 ** -rng.integers(1, 11, (2 * n // 3 - n // 2, 1))
    d = np.array(direction, dtype=np.float64)
    d = d / np.sqrt(d[0] * d[0] + d[1] * d[1] + d[2] * d[2])
    nu = np.full(n, synth.nu_of(wl.lines[0].lambda_A))
    pk = synth.Packets(pos, np.tile(d, (n, 1)), nu, np.arange(n, dtype=np.uint64))
    counts = {}
    for ndir in (0, 1):
        wl.detector.dirs = np.array([direction], dtype=np.float64)[:ndir]
        ctx = rg.Context(0)
        ctx.setup(wl)
        out, st = gpu_run(ctx, pk)
        assert (out["status"] == rg.PK_ESCAPED).all()
        counts[ndir] = st
        ctx.close()
    # a packet also looks up its first leaf: one read of the top grid (level 6 at
    # most), one of a son for each level below
    first = 0
    t = med.tree
    top = min(t.max_level, 6)
    o = np.zeros(n, dtype=np.int64)
    lev = np.zeros(n, dtype=np.int64)
    live = np.ones(n, dtype=bool)
    fine = 1 << t.max_level
    cell = np.where(d < 0, np.ceil(pos * fine) - 1, np.floor(pos * fine)).astype(np.int64)
    son = np.asarray(t.son, dtype=np.int64).reshape(-1, 8)
    for m in range(1, t.max_level + 1):
        b = (cell >> (t.max_level - m)) & 1
        v = son[o, b[:, 0] | b[:, 1] << 1 | b[:, 2] << 2]
        lev = np.where(live, m, lev)
        live &= v > 0
        o = np.where(live, v, o)
    first = int((1 + np.maximum(lev - top, 0)).sum())
    for k, extra in (("son_loads", first), ("nbor_loads", 0)):
        assert counts[1][k] - counts[0][k] == counts[0][k] - extra, (k, counts[0][k], counts[1][k], extra)

"""Blocks of every size that a batch launch may have give the same results, bit
for bit, for one to four lines."""
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nline", [1, 2, 3, 4])
def test_results_do_not_depend_on_the_block_size(nline):
    import paper_2001_11252_gb300 as rg
    wl = synth.sphere(tau0=50.0, T=1e4, tau_dust=0.5, n_packets=3001, base=2, max_level=3)
    wl.lines = wl.lines + [synth.d_lya(0.3), synth.d_lya(0.2), synth.d_lya(0.1)][:nline - 1]
    ctx = rg.Context(0)
    ctx.setup(wl)
    ctx.load_batch([wl], nbin=8)
    ref, _ = ctx.propagate_batch_packets()
    for block in (32, 64, 96, 128):
        ctx.set_batch_launch(block, 0, 1)
        got, st = ctx.propagate_batch_packets()
        assert st["packets"] == wl.packets.n
        for k in ref:
            assert got[k].tobytes() == ref[k].tobytes(), (block, k)

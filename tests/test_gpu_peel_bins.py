"""Detector bins of peeled contributions where FP32 cannot decide them: an
empty medium, so that every packet leaves one contribution of 1/4pi per
direction, with frequencies and projected positions on, next to and between
the edges of channels and pixels, inside and outside the detector; the counts
per bin equal those of the plain FP64 definition exactly."""
import math

import numpy as np
import pytest

import oracle
import synth
from gpu_util import context

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("npix,nbin,fov", [(8, 24, 0.5), (100, 200, 0.9), (37, 1001, 0.3), (1, 1, 1.3)])
def test_bins_equal_the_plain_definition(npix, nbin, fov):
    n = 20000
    wl = synth.expanding_sphere(N_HI=0.0, v_max_kms=0.0, tau_dust=0.0, n_packets=n, npix=npix, nchan=nbin, base=2,
                                max_level=3)
    det = wl.detector
    det.dirs = np.array([[0.0, 0.0, 1.0], [1.0, 1.0, 1.0]])
    det.fov = fov
    det.centre = (0.5, 0.5, 0.5)
    rng = np.random.default_rng(npix)
    pk = wl.packets
    v = rng.normal(size=(n, 3))
    pk.pos = 0.5 + 0.4 * v / np.linalg.norm(v, axis=1)[:, None] * rng.random((n, 1)) ** (1 / 3)
    q = n // 4
    edge = lambda k: fov * (rng.integers(-1, npix + 2, k) / npix - 0.5)
    pk.pos[:q, 0] = 0.5 + np.clip(edge(q), -0.25, 0.25)
    pk.pos[q:2 * q, 1] = 0.5 + np.clip(edge(q), -0.25, 0.25)
    pk.pos[q // 2:q, 0] = np.nextafter(pk.pos[q // 2:q, 0], rng.integers(0, 2, q - q // 2))
    inside = np.linalg.norm(pk.pos - 0.5, axis=1) < 0.44
    pk.pos[~inside] = 0.5
    width = det.nu_hi - det.nu_lo
    pk.nu = det.nu_lo + width * rng.uniform(-0.1, 1.1, n)
    pk.nu[::3] = det.nu_lo + width * (rng.integers(-1, nbin + 2, len(pk.nu[::3])) / nbin)
    pk.nu[::6] = np.nextafter(pk.nu[::6], 0.0)
    ctx = context(wl)
    one = 1.0 / (4.0 * math.pi)
    # 200 packets at a time: a bin then holds at most 200 equal FP32 terms, whose
    # sum is within 200 x half an ulp of 16 = 2e-4 of the exact one, 0.0024 counts
    counts = [0, 0, 0]
    for lo in range(0, n, 200):
        ctx.zero_tallies()
        w = slice(lo, lo + 200)
        ctx.propagate(pk.pos[w], pk.dir[w], pk.nu[w], pk.ids[w], stats=True)
        for j, kind in enumerate((1, 2, 3)):
            c = ctx.get_tally(kind).astype(np.float64) / one
            assert np.abs(c - np.rint(c)).max() < 0.0025
            counts[j] = counts[j] + np.rint(c).astype(np.int64)
    spec, img, cube = counts
    fb = np.floor((pk.nu - det.nu_lo) / width * nbin)
    ch = np.where((fb >= 0) & (fb < nbin), fb, -1).astype(np.int64)
    for d, k in enumerate(det.dirs):
        eu, ev = oracle.onb(k / math.sqrt(float((k * k).sum())))
        r = pk.pos - np.array(det.centre)
        u = (r[:, 0] * eu[0] + r[:, 1] * eu[1]) + r[:, 2] * eu[2]
        w = (r[:, 0] * ev[0] + r[:, 1] * ev[1]) + r[:, 2] * ev[2]
        fu, fv = np.floor((u / fov + 0.5) * npix), np.floor((w / fov + 0.5) * npix)
        ok = (fu >= 0) & (fu < npix) & (fv >= 0) & (fv < npix)
        px = np.where(ok, fv * npix + fu, -1).astype(np.int64)
        s = np.bincount(ch[ch >= 0], minlength=nbin)
        i = np.bincount(px[px >= 0], minlength=npix * npix)
        both = (ch >= 0) & (px >= 0)
        c = np.bincount(px[both] * nbin + ch[both], minlength=npix * npix * nbin)
        assert (spec[d] == s).all() and (img[d].ravel() == i).all() and (cube[d].ravel() == c).all()

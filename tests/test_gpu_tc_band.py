"""N^-1 of an FP64 TOD on the tensor cores (exact integer digits, FP64 FMA chain for the tiles they do not
take) against an extended-precision direct sum, at the edges of tiles, bands and of the rule that
chooses between the two.

Bound per element: |got - ref| <= 127 u (|N^-1| |x|) with u = 2^-53, the standard bound of the 127-term
FP64 FMA chain, which the digits must stay within wherever they are used.
"""
import numpy as np
import pytest
import torch

import synth
from parity import rel

pytestmark = pytest.mark.gpu

BOUND = 127 * 2.0 ** -53


def _ref(x, taps):
    x, t = x.astype(np.longdouble), taps.astype(np.longdouble)
    y = t[:, :1] * x
    for j in range(1, min(taps.shape[1], x.shape[1])):
        y[:, j:] += t[:, j:j + 1] * x[:, :-j]
        y[:, :-j] += t[:, j:j + 1] * x[:, j:]
    return y


def _apply(fx, dev, x, taps):
    nd, ns = x.shape
    o = synth.Observation(4, synth.satellite_scan(ns), synth.hex_focal_plane(nd))
    P = fx.Pointing.from_observations([o], mode="cache_f64", device=dev)
    N = fx.Noise.banded(P, taps)
    return N.inv_apply(torch.as_tensor(x.ravel(), device=dev)).cpu().numpy().reshape(nd, ns)


def _check(fx, dev, x, taps):
    got = _apply(fx, dev, x, taps)
    scale = _ref(np.abs(x), np.abs(taps))
    assert np.all(np.abs(got - _ref(x, taps)) <= BOUND * scale), float(np.max(np.abs(got - _ref(x, taps)) / scale))


@pytest.mark.parametrize("ns", [1, 15, 17, 64, 127, 4095, 4096, 4097, 4159, 8193])
@pytest.mark.parametrize("ntaps", [1, 2, 33, 64])
def test_tile_and_band_edges(fx, dev, ns, ntaps):
    g = np.random.default_rng(ns * 100 + ntaps)
    taps = g.normal(size=(3, ntaps)) * 10.0 ** np.array([[0.0], [-7.0], [5.0]])
    _check(fx, dev, g.normal(0, 100, (3, ns)), taps)


@pytest.mark.parametrize("r", [0, 6, 8, 9, 10, 12, 30])
def test_dynamic_range_within_a_tile(fx, dev, r):
    """Loud and quiet stretches 2^r apart, and one loud sample: both sides of the rule."""
    g = np.random.default_rng(r)
    x = g.normal(size=(4, 9000))
    x[0, 2000:2500] *= 2.0 ** r
    x[1, 5000] *= 2.0 ** r
    x[2, ::7] *= 2.0 ** -r
    x[3, :4000] = 0.0
    x[3, 4000:4100] *= 2.0 ** r
    _check(fx, dev, x, np.tile(synth.inverse_noise_taps(), (4, 1)))


@pytest.mark.parametrize("scale", [1e-300, 2.0 ** -1000, 1e-30, 2.0 ** 40, 1e290])
def test_extreme_exponents_and_digits(fx, dev, scale):
    """Samples and taps whose digits are all at their largest, and exponents at the ends of FP64."""
    x = np.full((3, 4200), 1.0 - 2.0 ** -53)
    x[1, ::2] *= -1.0
    x[2] = -1.0
    taps = np.full((3, 64), 1.0 - 2.0 ** -53)
    taps[1, 1::2] *= -1.0
    _check(fx, dev, x * scale, taps)


def test_infinities_and_nans_stay_where_they_act(fx, dev):
    g = np.random.default_rng(5)
    x = g.normal(size=(2, 9000))
    clean = x.copy()
    x[0, 3000], x[1, 6000] = np.inf, np.nan
    clean[0, 3000] = clean[1, 6000] = 0.0
    taps = np.tile(synth.inverse_noise_taps(), (2, 1))
    got = _apply(fx, dev, x, taps)
    ref, scale = _ref(clean, taps), _ref(np.abs(clean), np.abs(taps))
    for d, t in ((0, 3000), (1, 6000)):
        hit = np.zeros(9000, bool)
        hit[t - 63:t + 64] = True
        assert not np.isfinite(got[d][hit]).any()
        assert np.all(np.abs(got[d][~hit] - ref[d][~hit]) <= BOUND * scale[d][~hit])
    taps[0, 3] = np.nan
    assert np.isnan(_apply(fx, dev, clean, taps)[0][100:-100]).all()


@pytest.mark.parametrize("mode", ["cache_f64", "cache_mixed", "on_the_fly"])
def test_operators_with_tiles_of_both_kinds(fx, dev, orc, mode):
    """Right-hand side and normal operator on data and maps whose range within a tile exceeds the digits' (a
    glitch, a zeroed stretch, bright pixels), in both FP64-accurate precisions, against the oracle to the
    1e-12 that these paths are held to elsewhere."""
    nd, ns, nside = 3, 13000, 16
    o = synth.Observation(nside, synth.satellite_scan(ns), synth.hex_focal_plane(nd))
    P = fx.Pointing.from_observations([o], mode=mode, device=dev)
    taps = np.tile(synth.inverse_noise_taps(), (nd, 1))
    N = fx.Noise.banded(P, taps)
    pix, c, s, _ = orc.pointing(nside, o.q_bore, o.q_det)
    g = np.random.default_rng(11)
    d = g.normal(0, 10, (nd, ns)).astype(np.float32)
    d[0, 6000] = 1e6
    d[1, 2000:2300] = 0.0
    every = np.ones(o.npix, bool)
    ref = orc.rhs(o.npix, pix, c, s, orc.Noise(taps=taps), every, d.astype(np.float64))
    got = fx.rhs(P, N, torch.as_tensor(d.ravel(), device=dev)).cpu().numpy()
    assert rel(got, ref) < 1e-12
    x = synth.gaussian_sky(nside, g)
    x[pix[0, 5000]] *= 1e5
    ref = orc.apply_ata(o.npix, pix, c, s, orc.Noise(taps=taps), every, x)
    for precision in ("f64", "f32x2"):
        got = fx.ptnp_apply(P, N, torch.as_tensor(x, device=dev), precision=precision).cpu().numpy()
        assert rel(got, ref) < 1e-12, precision


@pytest.mark.parametrize("what", ["project", "chi2", "normal"])
def test_first_call_inside_a_stream_capture(fx, dev, what):
    """The workspaces of a handle's first call are allocated without disturbing a capture in progress."""
    nd, ns = 4, 20000
    o = synth.Observation(8, synth.satellite_scan(ns), synth.hex_focal_plane(nd))
    taps = np.tile(synth.inverse_noise_taps(), (nd, 1))
    m = torch.as_tensor(synth.gaussian_sky(8, np.random.default_rng(2)), device=dev)

    def call(P, N, d, m):
        if what == "project":
            return P.apply(m)
        if what == "chi2":
            return fx.chi2_grad(P, N, d, m)[1]
        return fx.ptnp_apply(P, N, m, precision="f64")

    make = lambda: fx.Pointing.from_observations([o], mode="cache_f64", device=dev)  # noqa: E731
    P0 = make()
    N = fx.Noise.banded(P0, taps)
    d = P0.apply(m) + 1.0
    ref = call(P0, N, d, m)
    P = make()
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        got = call(P, N, d, m)
    graph.replay()
    torch.cuda.synchronize()
    assert rel(got, ref.cpu().numpy()) < 1e-13

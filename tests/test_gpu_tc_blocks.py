"""Which outputs the tensor-core band product forms in integer digits: single loud samples among quiet ones, bands that
reach little, loud stretches of every length, ends of streams.

FP64 products are held per output to 127 u |N^-1| |x| (u = 2^-53), the bound of the 127-term FP64 FMA chain, against an
extended-precision direct sum.
"""
import numpy as np
import pytest
import torch

import synth
from test_gpu_tc_band import _apply, _check, _ref

pytestmark = pytest.mark.gpu


def _bands():
    k = synth.inverse_noise_taps()
    return {
        "inverse64": k,
        "short8": synth.inverse_noise_taps(8),
        "short9": synth.inverse_noise_taps(9),
        "short15": synth.inverse_noise_taps(15),
        "short17": synth.inverse_noise_taps(17),
        "tridiagonal in 64": np.r_[1.25, -0.5, np.zeros(62)],
        "decay": 2.0 ** -np.arange(64.0),
        "first and last": np.r_[1.0, np.zeros(62), 0.3],
        "zero diagonal": np.r_[0.0, np.full(63, 0.5)],
        "zero crossing": np.cos(np.arange(64) * np.pi / 20) * (1 - np.arange(64) / 64),
    }


@pytest.mark.parametrize("band", list(_bands()))
@pytest.mark.parametrize("r", [0, 6, 10, 20, 40])
def test_quiet_samples_between_loud_ones(fx, dev, band, r):
    """Every 32nd (8th) sample 2^r louder than the others, and pairs of loud and quiet halves of a block."""
    c = _bands()[band]
    g = np.random.default_rng(r)
    x = g.normal(size=(4, 5000))
    x[0, ::32] *= 2.0 ** r
    x[1, 3::8] *= 2.0 ** r
    x[2, :4090] *= 2.0 ** r
    x[3, 4099:] *= 2.0 ** r
    _check(fx, dev, x, np.tile(c, (4, 1)))


@pytest.mark.parametrize("length", [1, 8, 30, 250, 1000, 3100, 4000])
@pytest.mark.parametrize("r", [7, 10, 13, 25])
def test_loud_stretches_of_every_length(fx, dev, length, r):
    """From a few blocks formed again one by one to tiles that take the chain for all; zeros beside them."""
    g = np.random.default_rng(length)
    x = g.normal(size=(3, 8300))
    x[0, 17:17 + length] *= 2.0 ** r
    x[1] *= 2.0 ** -r
    x[1, 4000:4000 + length] *= 2.0 ** r
    x[2, 100:100 + length] = 0.0
    x[2, 100 + length:] *= 2.0 ** -r
    _check(fx, dev, x, np.tile(synth.inverse_noise_taps(), (3, 1)))


@pytest.mark.parametrize("ns", [5, 31, 33, 70, 4100, 4127])
def test_quiet_ends_of_short_streams(fx, dev, ns):
    """Streams whose last or first samples, less than a block or a group of 32, are far below the others."""
    g = np.random.default_rng(ns)
    x = g.normal(size=(3, ns))
    x[0, -4:] *= 2.0 ** -30
    x[1, :4] *= 2.0 ** -30
    x[2, ns // 2:] *= 2.0 ** -30
    for ntaps in (9, 64):
        _check(fx, dev, x, np.tile(synth.inverse_noise_taps(ntaps), (3, 1)))


@pytest.mark.parametrize("ns", [4096, 9001])
def test_error_on_ordinary_noise(fx, dev, ns):
    """Gaussian samples: one rounding (u) per output and the dropped weights, 2^-59.7 X C rms where X <= 8 sigma, C <= 2
    c_0 and an output is of the order c_0 sigma: 2^-55.7. Together less than 2 u in the 2-norm (the chain: 2 u alone; one
    weight less: above 2^6 u)."""
    g = np.random.default_rng(1)
    x, taps = g.normal(0, 100, (4, ns)), np.tile(synth.inverse_noise_taps(), (4, 1))
    got, ref = _apply(fx, dev, x, taps), _ref(x, taps)
    assert float(np.sqrt(((got - ref) ** 2).sum() / (ref ** 2).sum())) <= 2 * 2.0 ** -53


def test_compensated_product_between_loud_samples(fx, dev, orc):
    """The right-hand side of data with one sample of 2^20 in every tile, all of whose other outputs take the compensated
    double-FP32 product: per pixel (254 2^-24)^2 |P|^T |N^-1| |d|, the bound of algorithm Dot2 without its final rounding."""
    nd, ns, nside = 3, 12288, 32
    o = synth.Observation(nside, synth.satellite_scan(ns), synth.hex_focal_plane(nd))
    P = fx.Pointing.from_observations([o], mode="cache_f64", device=dev)
    taps = np.tile(synth.inverse_noise_taps(), (nd, 1))
    pix, c, s, _ = orc.pointing(nside, o.q_bore, o.q_det)
    d = np.random.default_rng(3).normal(size=(nd, ns))
    d[:, 2048::4096] *= 2.0 ** 20
    got = fx.rhs(P, fx.Noise.banded(P, taps), torch.as_tensor(d.ravel(), device=dev)).cpu().numpy()
    ref, scale = np.zeros((2, o.npix, 3), np.longdouble)
    y, a = _ref(d, taps), _ref(np.abs(d), np.abs(taps))
    for k, w in enumerate((np.ones_like(c), c, s)):
        np.add.at(ref[:, k], pix.ravel(), (y * w).ravel())
        np.add.at(scale[:, k], pix.ravel(), (a * np.abs(w)).ravel())
    assert np.all(np.abs(got - ref) <= (254 * 2.0 ** -24) ** 2 * scale)


def test_compensated_product_of_fp32_data(fx, dev, orc):
    """The same from FP32 data (no low words), every second half tile 2^16 louder, so that half of every tile takes it."""
    nd, ns, nside = 3, 12288, 32
    o = synth.Observation(nside, synth.satellite_scan(ns), synth.hex_focal_plane(nd))
    P = fx.Pointing.from_observations([o], mode="cache_f64", device=dev)
    taps = np.tile(synth.inverse_noise_taps(), (nd, 1))
    pix, c, s, _ = orc.pointing(nside, o.q_bore, o.q_det)
    d = np.random.default_rng(4).normal(size=(nd, ns)).astype(np.float32)
    d[:, np.arange(ns) // 2048 % 2 == 1] *= np.float32(2.0 ** 16)
    got = fx.rhs(P, fx.Noise.banded(P, taps), torch.as_tensor(d.ravel(), device=dev)).cpu().numpy()
    ref, scale = np.zeros((2, o.npix, 3), np.longdouble)
    y, a = _ref(d, taps), _ref(np.abs(d), np.abs(taps))
    for k, w in enumerate((np.ones_like(c), c, s)):
        np.add.at(ref[:, k], pix.ravel(), (y * w).ravel())
        np.add.at(scale[:, k], pix.ravel(), (a * np.abs(w)).ravel())
    assert np.all(np.abs(got - ref) <= (254 * 2.0 ** -24) ** 2 * scale)


@pytest.mark.parametrize("n", [1, 11, 12, 13, 60])
@pytest.mark.parametrize("loud", [2.0 ** 10, 2.0 ** 40, 1e300, np.inf, np.nan])
def test_loud_samples_around_the_number_left_out(fx, dev, n, loud):
    """Up to 12 groups of 32 samples of a tile may hold samples that stay out of the digits: both sides of that number,
    with samples that are not finite acting only where their band reaches."""
    ns = 4096
    g = np.random.default_rng(n)
    x = g.normal(size=(3, ns))
    at = 32 * (g.permutation(ns // 32)[:n]) + g.integers(0, 32, n)
    x[:2, at] *= loud
    x[1, :] *= 2.0 ** -100
    taps = np.tile(synth.inverse_noise_taps(), (3, 1))
    if np.isfinite(loud):
        _check(fx, dev, x, taps)
        return
    got, clean = _apply(fx, dev, x, taps), np.where(np.isfinite(x), x, 0.0)
    ref, scale = _ref(clean, taps), _ref(np.abs(clean), np.abs(taps))
    reach = _ref((~np.isfinite(x)).astype(float), np.ones((3, 64))) > 0
    assert not np.isfinite(got[reach]).any()
    assert np.all(np.abs(got[~reach] - ref[~reach]) <= 127 * 2.0 ** -53 * scale[~reach])

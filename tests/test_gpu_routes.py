"""Routes that a rule on the arguments or sizes chooses, each against the general one: FP64 sums taken straight
into the output, the chunks of the on-the-fly operator, pixel tiles of the PCG.

Two routes that add the same terms in another order differ per pixel by at most 2 h u sum|terms| <= 2 h^2 u max|term|,
with h the pixel's hits and u = 2^-53.
"""
import numpy as np
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu

U = 2.0 ** -53


def _problem(fx, dev, mode, nside=16, nd=3, ns=9001, ntaps=64, seed=3):
    o = synth.Observation(nside, synth.satellite_scan(ns), synth.hex_focal_plane(nd))
    P = fx.Pointing.from_observations([o], mode=mode, device=dev)
    taps = np.zeros((nd, ntaps))
    k = synth.inverse_noise_taps()
    taps[:, :min(ntaps, k.size)] = k[:ntaps]
    N = fx.Noise.banded(P, taps)
    g = np.random.default_rng(seed)
    x = torch.as_tensor(synth.gaussian_sky(nside, g), device=dev)
    d = torch.as_tensor(g.normal(0, 10, nd * ns), device=dev)
    return P, N, x, d


def _reorder_bound(P, tod):
    hits = int(P.transpose(tod, hits=True)[1].max())
    return 2 * hits * hits * U * float(tod.abs().max())


def _odd(t):
    """A copy that starts 8 bytes past a 16-byte boundary."""
    return torch.cat([t.new_zeros(1), t.reshape(-1)])[1:].view(t.shape)


@pytest.mark.parametrize("ntaps", [64, 65])
@pytest.mark.parametrize("mode,precision", [("cache_f32", "f32"), ("on_the_fly", "f32"), ("cache_f64", "f64"),
                                            ("cache_mixed", "f32x2")])
def test_sums_straight_into_the_output(fx, dev, mode, precision, ntaps):
    P, N, x, d = _problem(fx, dev, mode, ntaps=ntaps)
    every = torch.ones(x.shape[0], dtype=torch.uint8, device=dev)
    # the operator: FP32 terms are the same in both routes, so only the order of the FP64 sums differs
    tol = _reorder_bound(P, 1.01 * N.inv_apply(P.apply(x)))
    ref = fx.ptnp_apply(P, N, x, valid=every, precision=precision, acc="f64")
    out = _odd(torch.full_like(ref, float("nan")))
    fx.ptnp_apply(P, N, x, precision=precision, acc="f64", out=out)
    assert float((out - ref).abs().max()) <= tol
    # the right-hand side, from both data types
    tol = _reorder_bound(P, 1.01 * N.inv_apply(d))
    for t in (d, d.float()):
        assert float((fx.rhs(P, N, t) - fx.rhs(P, N, t, valid=every)).abs().max()) <= tol
    # P^T: a new map against one added to zeros; and a map that is added to
    tol = _reorder_bound(P, d)
    zero = torch.zeros_like(x)
    ref = P.transpose(d, out=zero.clone(), accumulate=True)
    out = _odd(torch.full_like(x, float("nan")))
    assert float((P.transpose(d, out=out) - ref).abs().max()) <= tol
    two = P.transpose(d, out=ref.clone(), accumulate=True)
    assert float((two - 2 * ref).abs().max()) <= 2 * tol


def test_on_the_fly_in_several_chunks(fx, dev):
    """More tiles than one chunk of the expansion holds (32 per SM), the last one short."""
    nd = 33 * torch.cuda.get_device_properties(dev).multi_processor_count + 5
    P, N, x, _ = _problem(fx, dev, "on_the_fly", nd=nd, ns=150)
    C = fx.Pointing.from_observations([synth.Observation(16, synth.satellite_scan(150), synth.hex_focal_plane(nd))],
                                      mode="cache_f32", device=dev)
    tol = _reorder_bound(P, 1.01 * N.inv_apply(P.apply(x)))
    got = fx.ptnp_apply(P, N, x, precision="f32", acc="f64")
    ref = fx.ptnp_apply(C, N, x, precision="f32", acc="f64")
    assert float((got - ref).abs().max()) <= tol


@pytest.mark.parametrize("precision", ["f64", "f32"])
def test_solution_does_not_depend_on_the_pixel_tiles(fx, dev, precision):
    """One small map alone (256-pixel tiles, the white operator and the vectors split over several blocks) and in
    a batch with a map of 786432 pixels (1024-pixel tiles): residuals of 1e-10 and a preconditioned condition
    number below 1e4 leave 2e-6 between the solutions."""
    nd, ns = 3, 9001
    small = synth.Observation(16, synth.satellite_scan(ns), synth.hex_focal_plane(nd))
    large = synth.Observation(256, synth.satellite_scan(ns), synth.hex_focal_plane(nd))
    mode = "cache_f64" if precision == "f64" else "cache_mixed"
    d = np.random.default_rng(9).normal(0, 10, (nd, ns))
    maps = []
    for obs in ([small], [small, large]):
        P = fx.Pointing.from_observations(obs, mode=mode, device=dev)
        N = fx.Noise.white(P, np.full(nd * len(obs), 2.0))
        m, _, info = fx.mapmaker_cg(P, N, torch.as_tensor(np.tile(d.ravel(), len(obs)), device=dev), maxiter=200, tol=1e-10,
                                 precision=precision)
        assert info.converged
        maps.append(m[:small.npix].clone())
    assert float((maps[0] - maps[1]).norm()) <= 2e-6 * float(maps[0].norm())


@pytest.mark.parametrize("ntaps", [4, 16, 17, 64])
def test_short_bands_agree_in_either_precision(fx, dev, ntaps):
    """Bands on both sides of the rules that choose among digits, FMA chain and compensated product, to the 1e-12
    that the FP64-accurate paths are held to elsewhere."""
    P, N, x, d = _problem(fx, dev, "cache_mixed", ntaps=ntaps)
    f64 = fx.ptnp_apply(P, N, x, precision="f64")
    assert float((fx.ptnp_apply(P, N, x, precision="f32x2") - f64).norm()) <= 1e-12 * float(f64.norm())
    ref = P.transpose(N.inv_apply(d))
    assert float((fx.rhs(P, N, d) - ref).norm()) <= 1e-12 * float(ref.norm())


@pytest.mark.parametrize("per_sm,ns", [(17, 150), (0, 9001)])
def test_on_the_fly_fp64_pointing_is_kept_for_the_scatter(fx, dev, per_sm, ns):
    """Several chunks (16 tiles per SM), and tiles of full length with both halos."""
    nd = per_sm * torch.cuda.get_device_properties(dev).multi_processor_count + 3
    P, N, x, d = _problem(fx, dev, "on_the_fly", nd=nd, ns=ns)
    C, M, _, _ = _problem(fx, dev, "cache_f64", nd=nd, ns=ns)
    tol = _reorder_bound(C, 1.01 * M.inv_apply(C.apply(x)))
    got, ref = (fx.ptnp_apply(p, n, x, precision="f64") for p, n in ((P, N), (C, M)))
    assert float((got - ref).abs().max()) <= tol
    got, ref = (fx.chi2_grad(p, n, d, x) for p, n in ((P, N), (C, M)))
    tol = 2 * _reorder_bound(C, 1.01 * M.inv_apply(d - C.apply(x)))
    assert float((got[1] - ref[1]).abs().max()) <= tol

"""GPU soft-binarisation iterations (Alg. 1 step 3, Sec. 4.1) against the FP64 oracle."""
import numpy as np
import pytest
import torch

import oracle
from paper_2212_08058_gb300 import synth

pytestmark = pytest.mark.gpu

TOL = 1e-5   # FP32 storage, on values in (0, 1)


@pytest.fixture(scope="module")
def sf():
    from paper_2212_08058_gb300 import build, sfseg
    build.build()
    oracle.build()
    return sfseg


def _check(x, mask, xo, margin):
    """x within TOL of the oracle; the mask is x > 1/2 of the GPU's own x, bit for bit, and
    equals the oracle's mask wherever the oracle's x is farther than `margin` from 1/2."""
    err = np.abs(x - xo).max()
    assert err < TOL, err
    np.testing.assert_array_equal(mask, (x > 0.5).astype(np.uint8))
    clear = np.abs(xo - 0.5) > margin
    np.testing.assert_array_equal(mask[clear], (xo[clear] > 0.5).astype(np.uint8))


@pytest.mark.parametrize("shape,radius,iters,gain,center", [
    ((8, 64, 64), (1, 3, 3), 3, 10.0, 0.5),     # TMA kernel
    ((5, 37, 70), (2, 7, 7), 2, 6.0, 0.35),     # TMA kernel, ragged tiles
    ((4, 20, 33), (1, 2, 3), 3, 12.0, 0.5),     # radius without a TMA kernel: generic stencil
    ((1, 1, 1), (1, 3, 3), 2, 4.0, 0.5),        # one voxel
])
def test_soft_binarize_matches_oracle(sf, shape, radius, iters, gain, center):
    T, H, W = shape
    if shape == (1, 1, 1):
        V = np.full((1, 1, 1, 1), 0.7, np.float32)
    else:
        V = synth.drifting_blob(T, H, W, seed=7100 + T)
    f = V[0].astype(np.float64)
    # the continuous solution both sides start from: 10 oracle iterations, rounded to float32
    xc, _ = oracle.power_filter(f, f, 0.3, 1.0, radius, np.ones(f.shape), 10)
    x0 = xc.astype(np.float32)
    with sf.PowerIteration(1, T, H, W, p=0.3) as h:
        h.set_features(torch.from_numpy(V).cuda())
        x, mask = h.soft_binarize(torch.from_numpy(x0).cuda(), radius, iters=iters, gain=gain, center=center)
        x, mask = x.cpu().numpy().astype(np.float64), mask.cpu().numpy()
    xo, _ = oracle.soft_binarize(f, f, 0.3, 1.0, radius, x0.astype(np.float64), iters, gain, center)
    _check(x, mask, xo, margin=1e-4)


def test_segment_end_to_end(sf):
    """Alg. 1 with C = 8 channels: 40 continuous iterations, then 4 soft-binarisation steps;
    against the oracle run from the oracle's own continuous solution."""
    V, gt, w = synth.multichannel(8, 48, 64, C=8, seed=7200)
    radius = (1, 3, 3)
    with sf.PowerIteration(8, 8, 48, 64) as h:
        x, mask = h.segment(torch.from_numpy(V).cuda(), w, 0.0, radius, n_iter=44, n_cont=40, gain=8.0)
        x, mask = x.cpu().numpy().astype(np.float64), mask.cpu().numpy()
    f = oracle.combine(V.astype(np.float64), w, 0.0)
    xc, _ = oracle.power_filter(f, f, 0.1, 1.0, radius, np.ones(f.shape), 40)
    xo, mo = oracle.soft_binarize(f, f, 0.1, 1.0, radius, xc, 4, 8.0, 0.5)
    _check(x, mask, xo, margin=1e-4)
    assert 0 < mask.sum() < mask.size


def test_soft_binarize_errors(sf):
    with sf.PowerIteration(1, 2, 8, 8) as h:
        x = torch.ones((2, 8, 8), device="cuda")
        with pytest.raises(sf.SFSegError) as e:
            h.soft_binarize(x, (1, 3, 3))
        assert e.value.status == "STATE"
        h.set_features(torch.rand((1, 2, 8, 8), device="cuda") + 0.1)
        for kw in ({"iters": 0}, {"gain": -1.0}, {"gain": float("inf")}, {"center": float("nan")}):
            with pytest.raises(sf.SFSegError):
                h.soft_binarize(x, (1, 3, 3), **kw)
        # features all zero: A x = 0, max(A x) = 0 -> ZERO_NORM, reported not hidden
        h.set_features(torch.zeros((1, 2, 8, 8), device="cuda"))
        with pytest.raises(sf.SFSegError) as e:
            h.soft_binarize(x, (1, 3, 3))
        assert e.value.status == "ZERO_NORM"
        # the handle stays usable
        h.set_features(torch.rand((1, 2, 8, 8), device="cuda") + 0.1)
        xs, m = h.soft_binarize(x, (1, 3, 3), iters=2)
        assert bool(((xs > 0) & (xs < 1)).all())


@pytest.mark.parametrize("bad", [float("nan"), float("inf")])
@pytest.mark.parametrize("T,H,W", [(4, 40, 70), (40, 200, 300)])
@pytest.mark.parametrize("radius", [(1, 6, 6), (0, 1, 1), (3, 1, 2)])
def test_non_finite_x_stops_the_step(sf, radius, T, H, W, bad):
    """A NaN or Inf in the caller's x makes the maximum of A x a NaN for a radius without a kernel of its
    own, whichever kernel runs it: the call says so, and x stays."""
    g = torch.Generator(device="cuda").manual_seed(8)
    V = torch.rand((1, T, H, W), device="cuda", generator=g) + 0.1
    x = torch.rand((T, H, W), device="cuda", generator=g)
    x[T // 2, H // 3, W // 2] = bad
    with sf.PowerIteration(1, T, H, W) as h:
        h.set_features(V)
        x0 = x.clone()
        with pytest.raises(sf.SFSegError) as e:
            h.soft_binarize(x, radius, iters=3, inplace=True)
        assert e.value.status == "ZERO_NORM"
        assert torch.equal(x.view(torch.int32), x0.view(torch.int32))
        xs, _ = h.soft_binarize(torch.rand((T, H, W), device="cuda", generator=g), radius, iters=2)
        assert bool(((xs > 0) & (xs < 1)).all())


@pytest.mark.parametrize("separate", [False, True])
@pytest.mark.parametrize("radius", [(1, 3, 3), (1, 6, 6), (3, 1, 2)])
@pytest.mark.parametrize("T,H,W", [(3, 17, 40), (40, 200, 300)])
def test_stop_at_a_later_step_keeps_the_step_before(sf, T, H, W, radius, separate):
    """With centre 2 and gain 200 the sigmoid is at most e^-200 = 0 in float32, so A x of the second
    step is 0 and that step stops: x is what the first step left, as a call of one step gives it."""
    g = torch.Generator(device="cuda").manual_seed(9)
    V = torch.rand((2, T, H, W), device="cuda", generator=g)
    x = torch.rand((T, H, W), device="cuda", generator=g)
    w = [0.7, 0.4]
    with sf.PowerIteration(2, T, H, W) as h:
        if separate:
            h.set_features_sf(V, w, 0.1, V, w, 0.0)
        else:
            h.set_features(V, w, 0.0)
        one, _ = h.soft_binarize(x, radius, iters=1, gain=200.0, center=2.0)
        assert float(one.max()) == 0.0
        y = x.clone()
        with pytest.raises(sf.SFSegError) as e:
            h.soft_binarize(y, radius, iters=4, gain=200.0, center=2.0, inplace=True)
        assert e.value.status == "ZERO_NORM"
        assert torch.equal(y, one)


@pytest.mark.parametrize("shape,radius", [((5, 30, 40), (3, 1, 2)), ((6, 20, 33), (4, 3, 2)), ((9, 40, 150), (1, 6, 6)),
                                          ((24, 325, 449), (1, 3, 3)), ((24, 325, 449), (2, 7, 7))])
def test_soft_binarize_on_every_kernel(sf, shape, radius):
    """The generic stencil (rt = 3, 4), a padded radius, and the streaming kernel with the maximum taken
    in the step, three steps each, against the oracle."""
    T, H, W = shape
    V = synth.drifting_blob(T, H, W, seed=7300 + T)
    f = V[0].astype(np.float64)
    rng = np.random.default_rng(T)
    x0 = rng.random(shape).astype(np.float32)
    with sf.PowerIteration(1, T, H, W, p=0.3) as h:
        h.set_features(torch.from_numpy(V).cuda())
        x, mask = h.soft_binarize(torch.from_numpy(x0).cuda(), radius, iters=3, gain=6.0, center=0.4)
        x, mask = x.cpu().numpy().astype(np.float64), mask.cpu().numpy()
    xo, _ = oracle.soft_binarize(f, f, 0.3, 1.0, radius, x0.astype(np.float64), 3, 6.0, 0.4)
    _check(x, mask, xo, margin=1e-4)

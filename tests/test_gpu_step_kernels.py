"""The two kernels of the Eq. 7 step (csrc/iter_stream.cuh and, for small and short volumes,
csrc/iter_tile.cuh) and the radii that run on a wider radius's kernel with
zero taps, at the sizes where they can go wrong: one row, column or frame past a tile, fewer tiles than
SMs and more, tiles cut in time, both sides of the line between the kernels.

Reference: the FP64 oracle.  Bound: an iterate of K steps is K times (2 rt + 1) + (2 rh + 1) + (2 rw + 1)
+ 12 roundings of positive float32 sums away from it, each 2^-24 of max x: 4 steps at (2,7,7) 4 * 47 *
2^-24 = 1.1e-5 of max x."""
import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sf():
    from paper_2212_08058_gb300 import build, sfseg
    build.build()
    oracle.build()
    return sfseg


def _check(sf, T, H, W, radius, seed, iters=4, bf16=0, init="uniform"):
    rng = np.random.default_rng(seed)
    V = rng.random((1, T, H, W)).astype(np.float32)
    with sf.PowerIteration(1, T, H, W) as h:
        x, nu = h.power_iterate(torch.from_numpy(V).cuda(), radius=radius, iters=iters, iters_bf16=bf16, init=init,
                                return_norms=True)
    f = V[0].astype(np.float64)
    xo, nuo = oracle.power_filter(f, f, 0.1, 1.0, radius, f if init == "smap" else np.ones(f.shape), iters)
    tol = 2e-2 if bf16 else iters * (2 * sum(radius) + 3 + 12) * 2.0 ** -24
    assert np.abs(x.cpu().numpy() - xo).max() <= tol * xo.max(), (T, H, W, radius)
    np.testing.assert_allclose(nu, nuo, rtol=tol)


# tiles of 18 x 112 on 152 SMs, one column, row or frame past a tile
@pytest.mark.parametrize("T,H,W", [
    (60, 342, 560), (61, 343, 561),                  # fewer tiles than SMs, cut in time
    (40, 325, 1009),                                 # 190 tiles: whole ones and a rest that is cut
    (40, 144, 2128), (17, 306, 2241),                # 152 tiles: whole ones only; 357: two each and a rest
    (2000, 17, 113), (2000, 1, 300),                 # long and flat
    (6, 342, 336), (5, 342, 1008), (13, 152, 58),    # the small-volume kernel's
])
@pytest.mark.parametrize("radius", [(1, 3, 3), (2, 7, 7)])
def test_stream_and_tile_kernels(sf, T, H, W, radius):
    _check(sf, T, H, W, radius, seed=T + H + W)


@pytest.mark.parametrize("radius", [(0, 0, 0), (0, 1, 1), (1, 1, 1), (1, 6, 6), (2, 4, 4), (2, 2, 5), (0, 8, 0),
                                    (1, 8, 8), (2, 8, 8), (2, 0, 8)])
@pytest.mark.parametrize("T,H,W", [(7, 20, 113), (61, 343, 561)])
def test_padded_radii(sf, radius, T, H, W):
    _check(sf, T, H, W, radius, seed=17, init="smap")
    assert sf.iterate_kernel_stats()[2].startswith("stream_stencil")


def test_bf16_storage_in_the_stream_kernel(sf):
    _check(sf, 61, 343, 561, (2, 7, 7), seed=3, iters=3, bf16=2)


@pytest.mark.parametrize("T,H,W", [(7, 20, 113), (40, 325, 561)])
def test_padded_radius_adjoint(sf, T, H, W):
    """The adjoint of a padded radius: the directional derivative of a linear loss along a random
    weight direction against central differences of the FP64 iteration (step 1e-4: truncation below
    1e-6 of the derivative, float32 roundings of 3 steps below 1e-5)."""
    rng = np.random.default_rng(5)
    V = rng.random((2, T, H, W)).astype(np.float32)
    c = rng.normal(size=(T, H, W)).astype(np.float32)
    w = np.array([0.8, -0.5], dtype=np.float32)
    r = (1, 6, 6)
    with sf.PowerIteration(2, T, H, W) as h:
        h.power_iterate(torch.from_numpy(V).cuda(), w, 0.1, r, iters=3, record_every=2)
        gw, gb = h.backward(torch.from_numpy(c).cuda(), r)
    d = np.array([0.6, 0.8, -0.5])                   # direction in (w0, w1, b)

    def loss(t):
        f = oracle.combine(V.astype(np.float64), w.astype(np.float64) + t * d[:2], 0.1 + t * d[2])
        x, _ = oracle.power_filter(f, f, 0.1, 1.0, r, np.ones(f.shape), 3)
        return float((x * c).sum())

    num = (loss(1e-4) - loss(-1e-4)) / 2e-4
    scale = float(np.abs(np.append(gw, gb)).max())
    assert abs(gw[0] * d[0] + gw[1] * d[1] + gb * d[2] - num) <= 1e-4 * scale


@pytest.mark.parametrize("radius", [(0, 0, 0), (1, 1, 1), (0, 2, 1), (1, 6, 6), (1, 3, 3)])
def test_apply_keeps_inf_in_its_neighbourhood(sf, radius):
    """An Inf in x reaches the outputs of its own neighbourhood and no others: those are what they are
    with a zero in its place, bit for bit (a zero adds exactly nothing)."""
    T, H, W = 5, 30, 40
    g = torch.Generator(device="cuda").manual_seed(6)
    V = torch.rand((1, T, H, W), device="cuda", generator=g) + 0.1
    x = torch.rand((T, H, W), device="cuda", generator=g)
    at = (2, 14, 21)
    x[at] = 0.0
    with sf.PowerIteration(1, T, H, W) as h:
        h.set_features(V)
        y0 = h.apply(x, radius).clone()
        x[at] = float("inf")
        y1 = h.apply(x, radius)
    inside = torch.zeros((T, H, W), dtype=torch.bool, device="cuda")
    inside[tuple(slice(max(c - r, 0), c + r + 1) for c, r in zip(at, radius))] = True
    assert not torch.isfinite(y1[inside]).any()
    assert torch.equal(y1[~inside], y0[~inside])


def test_norm_of_many_equal_voxels(sf):
    """The Eq. 8 norm of a volume of 4000 tiles (26 per SM) with one feature value: a thread adds 80
    equal squares per tile in float32, each addition 2^-24 of the sum away at most, so the root of the
    sum 80 * 2^-25 = 2.4e-6.  One float32 sum over a thread's 26 tiles is up to 1.5e-5 away."""
    T, H, W, r = 20, 1800, 4480, (1, 3, 3)
    with sf.PowerIteration(1, T, H, W) as h:
        V = torch.full((1, T, H, W), 0.6, device="cuda")
        _, nu = h.power_iterate(V, radius=r, iters=1, return_norms=True)
        x0 = torch.full((T, H, W), (T * H * W) ** -0.5, device="cuda")
        y = h.apply(x0, r)
    assert abs(float(nu[0]) / float(y.double().norm()) - 1.0) <= 2.4e-6


def test_exact_operator_in_the_stream_kernel(sf):
    """The exact (Eq. 1) operator on a volume of the streaming kernel, with the centred series, against
    the same operator on a crop that the small-volume kernel runs, with the series in f, at voxels
    whose whole neighbourhood lies in the crop.  Bound: both truncate at 2^-24 of the sum and sum 9 and
    16 terms of 35 taps each in float32: (9 + 16) * 35 * 2^-24 = 5.2e-5 of max y at most."""
    T, H, W, r = 40, 325, 561, (1, 3, 3)
    g = torch.Generator(device="cuda").manual_seed(4)
    V = torch.rand((1, T, H, W), device="cuda", generator=g)
    x = torch.rand((T, H, W), device="cuda", generator=g)
    with sf.PowerIteration(1, T, H, W) as h:
        h.set_features(V)
        y = h.apply_exact(x, r)
    h0, w0, n = 200, 300, 90
    crop = (slice(None), slice(h0, h0 + n), slice(w0, w0 + n))
    with sf.PowerIteration(1, T, n, n) as h:
        h.set_features(V[:, :, h0:h0 + n, w0:w0 + n].contiguous())
        yc = h.apply_exact(x[crop].contiguous(), r, n_terms=16)
    a, b = y[crop][:, 3:-3, 3:-3], yc[:, 3:-3, 3:-3]
    assert float((a - b).abs().max()) <= 5.2e-5 * float(b.abs().max())


def test_exact_refusals_stay(sf):
    """A feature range whose series in f is too long is refused, although the centred one is short."""
    V = torch.rand((1, 4, 20, 30), device="cuda") * 0.1 + 6.0        # 2 alpha f^2 = 74
    with sf.PowerIteration(1, 4, 20, 30) as h:
        h.set_features(V)
        with pytest.raises(sf.SFSegError) as e:
            h.apply_exact(torch.rand((4, 20, 30), device="cuda"), (1, 3, 3))
        assert e.value.status == "UNSUPPORTED"


def test_norm_of_many_frames(sf):
    """The Eq. 8 norm of 500 equal frames of 152 tiles, one run of 500 frames per SM: at most 32 frames
    go into one float32 sum of 128 equal squares per lane, each addition 2^-24 of the sum away at most,
    so the root of the sum 128 * 2^-25 = 3.8e-6."""
    T, H, W, r = 500, 342, 896, (1, 3, 3)
    with sf.PowerIteration(1, T, H, W) as h:
        V = torch.full((1, T, H, W), 0.37, device="cuda")
        _, nu = h.power_iterate(V, radius=r, iters=1, return_norms=True)
        x0 = torch.full((T, H, W), (T * H * W) ** -0.5, device="cuda")
        y = h.apply(x0, r)
    assert abs(float(nu[0]) / float(y.double().norm()) - 1.0) <= 3.8e-6


@pytest.mark.parametrize("T,H,W,radius,maps,bf16,kernel", [
    (24, 325, 449, (2, 7, 7), 1, 0, "iter_stream<2,7,7,float,x~>"),
    (24, 325, 449, (1, 6, 6), 1, 0, "iter_stream<1,7,7,float,x~> for radius 1,6,6"),
    (24, 325, 449, (1, 3, 3), 2, 0, "iter_stream<1,3,3,float,caller x,separate maps>"),
    (24, 325, 449, (1, 3, 3), 1, 2, "iter_stream<1,3,3,bf16,caller x>"),
    (5, 40, 70, (2, 7, 7), 1, 0, "iter_tile<2,7,7,float,x~>"),
    (5, 40, 70, (0, 1, 1), 1, 0, "iter_tile<1,2,2,float,x~> for radius 0,1,1"),
    (4, 24, 33, (0, 0, 8), 1, 0, "iter_tile<2,8,8,float,x~> for radius 0,0,8"),
    (5, 40, 70, (1, 6, 6), 2, 0, "iter_tile<1,7,7,float,caller x,separate maps> for radius 1,6,6"),
    (5, 40, 70, (3, 5, 5), 1, 0, "stream_stencil<3,5,5,float,caller x>"),
    (5, 40, 70, (1, 3, 3), 2, 2, "stream_stencil<1,3,3,bf16,caller x,separate maps>"),
])
def test_step_kernels_says_what_ran(sf, T, H, W, radius, maps, bf16, kernel):
    g = torch.Generator(device="cuda").manual_seed(2)
    V = torch.rand((1, T, H, W), device="cuda", generator=g)
    with sf.PowerIteration(1, T, H, W) as h:
        if maps == 2:
            h.set_features_sf(V, None, 0.0, V.flip(1).contiguous())
        else:
            h.set_features(V)
        n0 = sf.step_kernels()
        h.power_iterate(None, radius=radius, iters=2, iters_bf16=bf16)
        n1 = sf.step_kernels()
    at = ("iter_stream", "iter_tile", "stream_stencil").index(kernel.split("<")[0])
    assert [b - a for a, b in zip(n0[:3], n1[:3])] == [2 * (i == at) for i in range(3)]
    assert n1[3] == kernel
    label = sf.iterate_kernel_stats()[2]
    assert label in ("iter_fast: " + kernel, "stream_stencil: " + kernel)


@pytest.mark.parametrize("radius", [(1, 3, 3), (2, 7, 7), (1, 6, 6), (3, 1, 2)])
@pytest.mark.parametrize("T,H,W", [(1, 1, 2), (4, 30, 40), (3, 37, 230), (40, 325, 561)])
def test_unary_below_the_normal_range(sf, radius, T, H, W):
    """u = s^9.6 is 10^-38.4 = 4e-39, a subnormal float32, where s = 1e-4, and 1 elsewhere; the outputs
    there are ordinary numbers again for x = 1e6.  u's relative error: the product p log2 s = 128 and the
    logarithm are rounded to 2^-22, so 128 * 2^-21 * ln 2 = 4.2e-5, the rest far below."""
    f = np.ones((T, H, W), np.float32)
    at = (T // 2, H // 2, W // 2)
    f[at] = 1e-4
    x = np.full((T, H, W), 1e6, np.float32)
    with sf.PowerIteration(1, T, H, W, p=9.6) as h:
        h.set_features(torch.from_numpy(f[None]).cuda())
        y = h.apply(torch.from_numpy(x).cuda(), radius).cpu().numpy()
        xi, nu = h.power_iterate(None, radius=radius, iters=3, return_norms=True)
        xi = xi.cpu().numpy()
    f64 = f.astype(np.float64)
    yo = oracle.filter_apply(f64, f64, 9.6, 1.0, radius, x.astype(np.float64))
    assert np.abs(y / yo - 1.0).max() <= 5e-5
    xo, nuo = oracle.power_filter(f64, f64, 9.6, 1.0, radius, np.ones(f.shape), 3)
    assert np.abs(xi - xo).max() <= 3 * (2 * sum(radius) + 3 + 12) * 2.0 ** -24 * xo.max()
    np.testing.assert_allclose(nu, nuo, rtol=1e-5)


@pytest.mark.parametrize("r", [(1, 3, 3), (2, 7, 7), (2, 4, 4)])
def test_adjoint_on_the_streaming_kernel(sf, r):
    """The recording, recomputing and reverse steps of the streaming kernel on radii of its own and a
    padded one: as test_padded_radius_adjoint, four steps in two segments."""
    T, H, W = 40, 325, 561
    rng = np.random.default_rng(5)
    V = rng.random((2, T, H, W)).astype(np.float32)
    c = rng.normal(size=(T, H, W)).astype(np.float32)
    w = np.array([0.8, -0.5], dtype=np.float32)
    with sf.PowerIteration(2, T, H, W) as h:
        h.power_iterate(torch.from_numpy(V).cuda(), w, 0.1, r, iters=4, record_every=2)
        gw, gb = h.backward(torch.from_numpy(c).cuda(), r)
    d = np.array([0.6, 0.8, -0.5])

    def loss(t):
        f = oracle.combine(V.astype(np.float64), w.astype(np.float64) + t * d[:2], 0.1 + t * d[2])
        x, _ = oracle.power_filter(f, f, 0.1, 1.0, r, np.ones(f.shape), 4)
        return float((x * c).sum())

    num = (loss(1e-4) - loss(-1e-4)) / 2e-4
    scale = float(np.abs(np.append(gw, gb)).max())
    assert abs(gw[0] * d[0] + gw[1] * d[1] + gb * d[2] - num) <= 1e-4 * scale

"""GPU exact (Eq. 1) kernel, the diagnostic of the first-order approximation (Sec. 4.3), against
the FP64 oracle's explicit Eq. 1 matrix (oracle.affinity(..., exact=True))."""
import math

import numpy as np
import pytest
import torch

import oracle
from paper_2212_08058_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sf():
    from paper_2212_08058_gb300 import build, sfseg
    build.build()
    oracle.build()
    return sfseg


@pytest.mark.parametrize("T,H,W,radius,alpha,p", [
    (5, 37, 70, (1, 3, 3), 1.0, 0.1),     # ragged tiles
    (4, 20, 40, (2, 7, 7), 0.5, 0.2),
    (6, 16, 33, (1, 2, 2), 2.0, 0.1),     # a longer series (larger alpha)
    (3, 30, 64, (1, 4, 4), 0.25, 0.3),
])
def test_apply_exact_matches_oracle(sf, T, H, W, radius, alpha, p):
    V = synth.drifting_blob(T, H, W, seed=7600 + T)
    f = V[0].astype(np.float64)
    rng = np.random.default_rng(T)
    x = rng.random((T, H, W)).astype(np.float32)
    Me = oracle.affinity(f, f, p, alpha, radius, exact=True)
    yo = (Me @ x.astype(np.float64).ravel()).reshape(T, H, W) / alpha
    with sf.PowerIteration(1, T, H, W, alpha=alpha, p=p) as h:
        h.set_features(torch.from_numpy(V).cuda())
        y = h.apply_exact(torch.from_numpy(x).cuda(), radius).cpu().numpy().astype(np.float64)
    assert np.abs(y - yo).max() <= 2e-6 * np.abs(yo).max()


def test_power_iterate_exact_matches_oracle(sf):
    """Eq. 4 + Eq. 8 on the Eq. 1 matrix: 15 normalised steps from the uniform start."""
    T, H, W, r, K = 6, 30, 45, (1, 3, 3), 15
    V = synth.drifting_blob(T, H, W, seed=7650)
    f = V[0].astype(np.float64)
    Me = oracle.affinity(f, f, 0.1, 1.0, r, exact=True)
    xo, nuo = oracle.power_csr(Me, np.ones(T * H * W), K)
    with sf.PowerIteration(1, T, H, W) as h:
        h.set_features(torch.from_numpy(V).cuda())
        x, nu = h.power_iterate_exact(r, iters=K, return_norms=True)
    assert np.abs(x.cpu().numpy().ravel() - xo).max() < 1e-5
    np.testing.assert_allclose(nu, np.asarray(nuo)[:K], rtol=1e-5)


def test_series_length(sf):
    """The automatic series length reaches the result of the longest series (120 terms), and a
    single term is the n = 0 kernel (1/a) u_i e^{-a f_i^2} G_ij u_j e^{-a f_j^2}: the oracle's
    Eq. 7 operator with the pairwise term off (f = 0) and the unary map u e^{-a f^2}."""
    T, H, W, r, alpha, p = 4, 24, 40, (1, 3, 3), 2.0, 0.1
    V = synth.drifting_blob(T, H, W, seed=7660)
    x = torch.rand((T, H, W), device="cuda")
    with sf.PowerIteration(1, T, H, W, alpha=alpha, p=p) as h:
        h.set_features(torch.from_numpy(V).cuda())
        ya = h.apply_exact(x, r)
        yl = h.apply_exact(x, r, n_terms=120)
        y1 = h.apply_exact(x, r, n_terms=1).cpu().numpy().astype(np.float64)
    assert float((ya - yl).abs().max()) <= 1e-6 * float(yl.abs().max())
    f = V[0].astype(np.float64)
    s_eff = (f ** p * np.exp(-alpha * f * f)) ** (1.0 / p)     # s_eff^p = u e^{-a f^2}
    yo = oracle.filter_apply(s_eff, np.zeros_like(f), p, alpha, r, x.cpu().numpy().astype(np.float64))
    assert np.abs(y1 - yo).max() <= 2e-6 * np.abs(yo).max()


def _angle_deg(a, b):
    """Angle between two vectors, well conditioned for small angles (2 asin(|a - b| / 2) of the
    unit vectors)."""
    a = a / np.linalg.norm(a)
    b = b / np.linalg.norm(b)
    return np.degrees(2 * np.arcsin(min(1.0, np.linalg.norm(a - b) / 2)))


def test_exact_approaches_taylor(sf):
    """The Fig. 4 comparison on the GPU, on the oracle's own test volume: the GPU's exact-kernel
    eigenvector equals the oracle's (dense eigh of the Eq. 1 matrix), and the angle between the
    exact and the first-order eigenvectors is the oracle's (dense eigh of both matrices), which
    shrinks like alpha^2 (0.093, 0.022, 0.0055 degrees)."""
    f = synth.drifting_blob(4, 10, 12, seed=7)
    T, H, W = f.shape[1:]
    f64 = f[0].astype(np.float64)
    r, K = (1, 2, 2), 3000
    angles = []
    for alpha in (0.4, 0.2, 0.1):
        Me = oracle.affinity(f64, f64, 0.1, alpha, r, exact=True)
        Mt = oracle.affinity(f64, f64, 0.1, alpha, r)
        xo = np.linalg.eigh(Me.toarray())[1][:, -1]
        xo *= np.sign(xo.sum())
        xto = np.linalg.eigh(Mt.toarray())[1][:, -1]
        xto *= np.sign(xto.sum())
        with sf.PowerIteration(1, T, H, W, alpha=alpha) as h:
            h.set_features(torch.from_numpy(f).cuda())
            xt = h.power_iterate(None, radius=r, iters=K).double().cpu().numpy().ravel()
            xe = h.power_iterate_exact(r, iters=K).double().cpu().numpy().ravel()
        assert _angle_deg(xe, xo) < 2e-4
        a, ao = _angle_deg(xt, xe), _angle_deg(xto, xo)
        assert abs(a - ao) <= 0.05 * ao + 2e-4, (alpha, a, ao)
        angles.append(a)
    assert angles[0] > angles[1] > angles[2]
    assert 3.0 < angles[1] / angles[2] < 5.0, angles


def test_exact_errors(sf):
    T, H, W = 3, 16, 16
    V = synth.drifting_blob(T, H, W, seed=7680)
    x = torch.rand((T, H, W), device="cuda")
    with sf.PowerIteration(1, T, H, W) as h:
        with pytest.raises(sf.SFSegError) as e:
            h.apply_exact(x, (1, 3, 3))
        assert e.value.status == "STATE"
        h.set_features(torch.from_numpy(V).cuda())
        with pytest.raises(sf.SFSegError) as e:
            h.apply_exact(x, (1, 1, 2))
        assert e.value.status == "UNSUPPORTED"
        with pytest.raises(sf.SFSegError) as e:
            h.apply_exact(x, (1, 3, 3), n_terms=121)
        assert e.value.status == "INVALID_ARG"
    Vs, _, ws = synth.multichannel(T, H, W, C=2, seed=7681)
    with sf.PowerIteration(2, T, H, W) as h:
        h.set_features_sf(torch.from_numpy(Vs).cuda(), ws, 0.0, torch.from_numpy(Vs).cuda(), ws, 0.0)
        with pytest.raises(sf.SFSegError) as e:
            h.power_iterate_exact((1, 3, 3), iters=2)
        assert e.value.status == "UNSUPPORTED"


@pytest.mark.parametrize("alpha", [0.5, 1.0, 2.0, 4.0, 8.0, 12.0])
def test_every_output_keeps_its_digits(sf, alpha):
    """Each output's own relative error, not only the largest output's: half of the voxels at the dark
    end of f's range and half at its bright end, the dark ones' x a millionth of the bright ones', so
    that a dark voxel's output is a sum over pairs at opposite ends of the range, e^{-alpha} small.

    Bound, in roundings of 2^-24: a series of N terms whose products g_i g_j are of one sign is a sum of
    positive numbers, each off by the taps of the three filters, one multiplication per power of g on
    either side (2 N), 12 for u, e^{-alpha g^2} and the combination, and 4 alpha range^2 for the rounded
    exponents of the two exponentials.  A centre between the two ends multiplies that by e^{alpha range^2}
    at most, which is admitted up to alpha range^2 = 1: a factor of e."""
    T, H, W, r = 4, 20, 60, (1, 3, 3)
    rng = np.random.default_rng(77)
    bright = rng.random((T, H, W)) < 0.5
    f32 = np.where(bright, rng.uniform(0.95, 1.0, (T, H, W)), rng.uniform(0.01, 0.05, (T, H, W))).astype(np.float32)
    x = np.where(bright, 1.0, 1e-6).astype(np.float32)
    f = f32.astype(np.float64)
    Me = oracle.affinity(f, f, 0.1, alpha, r, exact=True)
    yo = (Me @ x.astype(np.float64).ravel()).reshape(T, H, W) / alpha
    with sf.PowerIteration(1, T, H, W, alpha=alpha) as h:
        h.set_features(torch.from_numpy(f32[None]).cuda())
        y = h.apply_exact(torch.from_numpy(x).cuda(), r).cpu().numpy().astype(np.float64)
    q, terms = 2.0 * alpha * f.max() ** 2, 1
    tail = q * math.exp(q)
    while tail > 2.0 ** -24:
        tail *= q / (terms + 1)
        terms += 1
    bound = (2 * sum(r) + 3 + 2 * terms + 12 + 4 * alpha) * 2.0 ** -24 * (math.e if alpha <= 1.0 else 1.0)
    assert (np.abs(y - yo) / yo).max() <= bound


@pytest.mark.parametrize("T,H,W", [(1, 1, 1), (3, 17, 41), (2, 480, 854)])
def test_no_exact_steps_is_the_normalised_start(sf, T, H, W):
    """iters = 0: the uniform vector of norm 1 (each component a rounded N^-1/2), or the caller's x over
    its norm (2 roundings), and a zero x is reported."""
    V = torch.rand((1, T, H, W), device="cuda") + 0.1
    x = torch.rand((T, H, W), device="cuda") + 0.1
    with sf.PowerIteration(1, T, H, W) as h:
        h.set_features(V)
        u = h.power_iterate_exact((1, 3, 3), iters=0)
        assert float((u.double() * (T * H * W) ** 0.5 - 1.0).abs().max()) <= 2.0 ** -24
        n0 = sf.kernel_launches()
        h.power_iterate_exact((1, 3, 3), iters=0, x=u)
        assert sf.kernel_launches() - n0 == 2          # f's range, and the vector
        y = h.power_iterate_exact((1, 3, 3), iters=0, x=x.clone(), init="user").double()
        assert float((y / (x.double() / x.double().norm()) - 1.0).abs().max()) <= 4 * 2.0 ** -24
        with pytest.raises(sf.SFSegError) as e:
            h.power_iterate_exact((1, 3, 3), iters=0, x=torch.zeros_like(x), init="user", return_norms=True)
        assert e.value.status == "ZERO_NORM"


def test_exact_norm_of_many_equal_voxels(sf):
    """The norms of the exact operator on 120x1080x1920 equal voxels.  A thread's sum carries its own
    roundings, 2 of 2^-24 in all, and the outputs' own (17 taps, two equal sides of an edge, 8 for u, the
    exponential and the combination) are common to the reference: (2 + 8) / 2 * 2^-24 = 3e-7, and as much
    for the float32 reciprocal norm of each step."""
    T, H, W, r = 120, 1080, 1920, (1, 3, 3)
    with sf.PowerIteration(1, T, H, W) as h:
        h.set_features(torch.full((1, T, H, W), 0.6, device="cuda"))
        _, nu = h.power_iterate_exact(r, iters=2, return_norms=True)
        y = h.apply_exact(torch.full((T, H, W), (T * H * W) ** -0.5, device="cuda"), r)
        n1 = float(y.double().norm())
        y.mul_(1.0 / n1)
        n2 = float(h.apply_exact(y, r).double().norm())
    assert abs(nu[0] / n1 - 1.0) <= 6e-7 and abs(nu[1] / n2 - 1.0) <= 6e-7

"""Calls with little device memory left: what fits is done, what does not is reported once, and the next
call works."""
import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu

MB = 1 << 20


@pytest.fixture(scope="module")
def sf():
    from paper_2212_08058_gb300 import build, sfseg
    build.build()
    oracle.build()
    return sfseg


class _Full:
    """All device memory but `leave` bytes taken while it is entered."""

    def __init__(self, leave):
        self.leave = leave

    def __enter__(self):
        torch.cuda.synchronize()
        torch.cuda.empty_cache()
        self.blocks = []
        step = torch.cuda.mem_get_info()[0] - self.leave
        while step >= 20 * MB:       # one block, or smaller ones where the free memory is in pieces
            try:
                self.blocks.append(torch.empty(step, device="cuda", dtype=torch.uint8))
            except torch.OutOfMemoryError:
                step //= 2
            step = min(step, torch.cuda.mem_get_info()[0] - self.leave)

    def __exit__(self, *exc):
        del self.blocks
        torch.cuda.empty_cache()


def test_a_call_after_an_allocation_failed(sf):
    """The failure belongs to the call that met it: the next call of another handle works."""
    V = torch.rand((1, 4, 16, 16), device="cuda") + 0.1
    with sf.PowerIteration(1, 4, 16, 16) as h:
        x0 = h.power_iterate(V, radius=(1, 3, 3), iters=2).clone()
        with _Full(100 * MB):
            with pytest.raises(sf.SFSegError) as e:
                sf.PowerIteration(1, 64, 512, 512)       # three volumes of 64 MB
            assert e.value.status == "OOM"
        x1 = h.power_iterate(V, radius=(1, 3, 3), iters=2)
    assert float((x0 - x1).abs().max()) <= 1e-6


@pytest.mark.parametrize("n_terms", [0, 16])
def test_exact_operator_in_little_memory(sf, n_terms):
    """Volumes of 32 MB, room for one: the exact operator's own workspace needs no more, whether the
    series' length is the caller's or not.  Same result as with room, to the roundings of two series:
    (9 + 16) * 17 * 2^-24 = 2.5e-5 of the largest output."""
    T, H, W, r = 32, 512, 512, (1, 3, 3)
    g = torch.Generator(device="cuda").manual_seed(32)
    V = torch.rand((1, T, H, W), device="cuda", generator=g)
    x = torch.rand((T, H, W), device="cuda", generator=g)
    with sf.PowerIteration(1, T, H, W) as h:
        h.set_features(V)
        ref = h.apply_exact(x, r, n_terms=n_terms)
    with sf.PowerIteration(1, T, H, W) as h:
        h.set_features(V)
        with _Full((32 + 32 + 24) * MB):     # the output, one volume, and less than another
            y = h.apply_exact(x, r, n_terms=n_terms)
    assert float((y - ref).abs_().max()) <= 2.5e-5 * float(ref.max())


def test_reverse_pass_of_a_padded_radius_in_little_memory(sf):
    """30 steps recorded as one segment, volumes of 8 MB.  With room for the segment's iterates and the
    three gradient volumes (272 MB), not for the Q of every step that the stencil kernels' form keeps
    (264 MB more), a radius without a kernel of its own takes the form that needs none.  Same gradient:
    roundings of 30 steps of float32, 30 * (2 (1 + 6 + 6) + 3 + 12) * 2^-24 = 7.3e-5 of the largest,
    twice for the pass back."""
    T, H, W, r = 8, 512, 512, (1, 6, 6)
    g = torch.Generator(device="cuda").manual_seed(31)
    V = torch.rand((2, T, H, W), device="cuda", generator=g)
    c = torch.randn((T, H, W), device="cuda", generator=g)
    w = [0.8, -0.5]
    out = []
    for leave in (None, 272 * MB + 100 * MB):
        with sf.PowerIteration(2, T, H, W) as h:
            x = h.power_iterate(V, w, 0.1, r, iters=30, record_every=30)
            if leave is None:
                gw, gb = h.backward(c, r)
            else:
                with _Full(leave):
                    gw, gb = h.backward(c, r)
                    gw2, gb2 = h.backward(c, r)
                    np.testing.assert_allclose(np.append(gw2, gb2), np.append(gw, gb), rtol=1e-6)
            del x
            out.append(np.append(gw, gb).astype(np.float64))
    assert np.abs(out[0] - out[1]).max() <= 1.5e-4 * np.abs(out[0]).max()


@pytest.mark.parametrize("leave", [100 * MB, 240 * MB])
def test_training_after_an_allocation_failed(sf, leave):
    """A training call that runs out of memory part of the way (2M voxels: z and x0 of 8 MB each, then
    128 + 64 + 128 + 128 MB) reports it, holds on to nothing twice when it is called again, and works
    once there is room, with the gradients of a network that never ran short."""
    T, H, W = 8, 512, 512
    g = torch.Generator(device="cuda").manual_seed(33)
    feats = torch.rand((3, T, H, W), device="cuda", generator=g).to(torch.bfloat16)
    target = torch.rand((T, H, W), device="cuda", generator=g)
    ref = sf.WarmStartNet(3, seed=5)
    loss0, g0 = ref.backward(feats, target, want_grads=True)
    ref.close()
    net = sf.WarmStartNet(3, seed=5)
    net.forward(feats)
    with _Full(leave):
        free = []
        for _ in range(3):
            with pytest.raises(sf.SFSegError) as e:
                net.backward(feats, target)
            assert e.value.status == "OOM"
            free.append(torch.cuda.mem_get_info()[0])
        assert free[0] == free[1] == free[2]
    loss1, g1 = net.backward(feats, target, want_grads=True)
    net.close()
    assert abs(loss1 - loss0) <= 1e-6 and np.array_equal(g0, g1)


def test_network_on_a_smaller_volume_after_an_allocation_failed(sf):
    """A forward pass that does not fit reports it, and a smaller one still works."""
    g = torch.Generator(device="cuda").manual_seed(34)
    small = torch.rand((3, 4, 64, 64), device="cuda", generator=g)
    large = torch.rand((3, 8, 512, 512), device="cuda", generator=g)
    net = sf.WarmStartNet(3, seed=5)
    with _Full(200 * MB):                    # 64 + 128 + 128 MB of activations and the result's 8
        with pytest.raises(sf.SFSegError) as e:
            net.forward(large)
        assert e.value.status == "OOM"
        x0 = net.forward(small).clone()
    ref = sf.WarmStartNet(3, seed=5)
    assert torch.equal(x0, ref.forward(small))
    assert bool(torch.isfinite(net.forward(large)).all())
    net.close()
    ref.close()

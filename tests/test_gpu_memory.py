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
        self.block = torch.empty(torch.cuda.mem_get_info()[0] - self.leave, device="cuda", dtype=torch.uint8)

    def __exit__(self, *exc):
        del self.block
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

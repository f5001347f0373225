"""Grids in device memory that start at an odd element: every entry point takes them, whatever the
width of its kernels' loads and stores, and gives what it gives for arrays of its own.

Tolerances: the fluid update has a fixed order, so its bits agree.  Spreading and the adjoint add
with atomics: a node or blob sums at most a few hundred terms in any order, so FP32 sums agree to
1e-5 and FP64 ones to 1e-12.  The directional derivative is a central difference with step 1e-6 of
values of order one: 1e-6.
"""
import numpy as np
import pytest

from helpers import rel_l2, to_np

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("CUDA device required", allow_module_level=True)

import paper_1407_5600_gb300 as mb  # noqa: E402
from paper_1407_5600_gb300 import workloads as wl  # noqa: E402


def _odd(shape, dtype, off, values=None):
    """A contiguous tensor that starts `off` elements into an allocation, and the allocation."""
    n = int(np.prod(shape))
    store = torch.full((n + 8,), 7.0, dtype=dtype, device="cuda")
    t = store[off:off + n].view(shape)
    if values is not None:
        t.copy_(values)
    return t, store


def _untouched(store, off, n):
    return bool((store[:off] == 7.0).all()) and bool((store[off + n:] == 7.0).all())


@pytest.mark.parametrize("off", [1, 2, 3])
@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("n,nblobs", [((4, 8, 16), 5), ((32, 16, 8), 5000), ((16, 16, 16), 0)])
def test_spread_into_an_odd_offset(n, nblobs, prec, off):
    rng = np.random.default_rng(nblobs)
    pos = torch.as_tensor(rng.random((nblobs, 3)) * n, device="cuda")
    F = torch.as_tensor(rng.normal(size=(nblobs, 3)), device="cuda")
    d = mb.GridDesc(*n, precision=prec)
    with mb.Multiblob(d) as sim:
        want = sim.spread(pos, F)
        out, store = _odd(want.shape, want.dtype, off)
        mb.spread(sim.ctx, pos, F, out)
    assert rel_l2(to_np(out), to_np(want)) < (1e-12 if prec else 1e-5)
    assert _untouched(store, off, out.numel())

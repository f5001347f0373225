"""The five-pass fluid update (a side above 128) at the edges of its block rules: the 256-point
line layouts along each axis with short, middle and long other sides, partial column chunks, both
precisions, with the convective stress joined to its right-hand side, against the FP64 oracle.

Tolerances: FP64 sums of 16 + 16 terms a line in three directions and back stay within 100 ulps
(1e-13 allows ten times that); FP32 values of the same solve are a few 1e-7 off, held to 2e-6.
"""
import numpy as np
import pytest

import oracle
from helpers import rel_l2, to_np

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("CUDA device required", allow_module_level=True)

import paper_1407_5600_gb300 as mb  # noqa: E402
from paper_1407_5600_gb300 import workloads as wl  # noqa: E402


@pytest.mark.parametrize("prec,tol", [(1, 1e-13), (0, 2e-6)])
@pytest.mark.parametrize("advection", [0, 1])
@pytest.mark.parametrize("n", [(256, 4, 4), (4, 256, 8), (8, 4, 256), (256, 64, 16), (16, 256, 256),
                               (64, 128, 256), (256, 256, 4), (32, 16, 256)])
def test_fluid_update_five_pass(n, advection, prec, tol):
    nx, ny, nz = n
    kw = dict(h=0.8, rho=1.2, eta=0.7, dt=0.1)
    d = mb.GridDesc(nx, ny, nz, precision=prec, advection=advection, **kw)
    v = (0.1 * wl.random_field((nz, ny, nx), 51)).astype(d.grid_dtype).astype(np.float64)
    f = wl.random_field((nz, ny, nx), 52, scale=0.3).astype(d.grid_dtype).astype(np.float64)
    body = (0.3, 1, 0, 2)
    with mb.Multiblob(d) as sim:
        got = to_np(sim.fluid_update(v, f, body_force=body))[0]
    g = oracle.Grid(nx, ny, nz, advection=advection, **kw)
    assert rel_l2(got, oracle.fluid_update(g, v, f, body=body)) < tol

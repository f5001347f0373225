"""The three-pass fluid update of FP64 grids (packed double-float transforms) at every parity of
log2 of its sides, from the smallest to the largest side it takes, against the FP64 oracle.

Tolerance: a value passes 2 (log2 nx + log2 ny + log2 nz) <= 42 butterfly levels, each with an
addition and at most one twiddle product, of about 2^-48 each, and a dozen operations in the
right-hand side and the solve: (2 * 42 + 12) 2^-48 = 3.4e-13, held to 1e-12.
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


@pytest.mark.parametrize("n", [(4, 4, 4), (8, 4, 128), (4, 8, 16), (32, 128, 8), (128, 16, 4),
                               (64, 64, 64), (16, 32, 64), (128, 128, 32)])
@pytest.mark.parametrize("mean_mode,body", [(0, None), (1, (0.3, 1, 0, 2))])
def test_fluid_update_fp64_sides(n, mean_mode, body):
    nx, ny, nz = n
    d = mb.GridDesc(nx, ny, nz, h=0.8, rho=1.2, eta=0.7, dt=0.1, precision=1, mean_mode=mean_mode)
    v, f = wl.random_field((nz, ny, nx), 41), wl.random_field((nz, ny, nx), 42, scale=0.3)
    with mb.Multiblob(d) as sim:
        got = to_np(sim.fluid_update(v, f, body_force=body))[0]
    g = oracle.Grid(nx, ny, nz, h=0.8, rho=1.2, eta=0.7, dt=0.1, mean_mode=mean_mode)
    assert rel_l2(got, oracle.fluid_update(g, v, f, body=body)) < 1e-12

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


def _particles(n, seed):
    """Two icosahedra at random places of a box of sides n."""
    rng = np.random.default_rng(seed)
    L = np.array(n, dtype=np.float64)
    return wl.build_particles(rng.random((2, 3)) * L, 0.9, rng, L), rng


@pytest.mark.parametrize("off", [1, 2, 3])
@pytest.mark.parametrize("n", [(8, 8, 256), (256, 4, 8), (16, 8, 32)])
def test_step_adjoint_on_odd_offsets(n, off):
    """Velocity and gradients at an odd element (the field behind the positions in one flat state,
    say), with five FFT passes and with three, against arrays of their own; and that gradient
    against central differences of the step."""
    s, rng = _particles(n, off)
    shape = (1, 3, n[2], n[1], n[0])
    body = (1e-3, 0, 2, 1)

    def dev(x):
        return torch.as_tensor(x, device="cuda")

    q, ext = dev(s.pos), dev(rng.normal(scale=1e-3, size=s.pos.shape))
    v = dev(rng.normal(scale=1e-3, size=shape))
    cq, cv = dev(rng.normal(size=s.pos.shape)), dev(rng.normal(size=shape))
    L = dev(np.array(n, dtype=np.float64))
    with mb.Multiblob(mb.GridDesc(*n, precision=1, dt=0.05)) as sim:
        sim.set_particles(0, s.pos, s.pid, s.bonds, s.rest, 100.0)
        gq, gv, gk = cq.clone(), cv.clone(), torch.zeros(1, dtype=torch.float64, device="cuda")
        mb.adjoint_step(sim.ctx, q, v, ext, body, gq, gv, gk)
        vo, _ = _odd(shape, torch.float64, off, v)
        qo, _ = _odd(s.pos.shape, torch.float64, off, q)
        go, store = _odd(shape, torch.float64, off, cv)
        gqo, qstore = _odd(s.pos.shape, torch.float64, off, cq)
        gko = torch.zeros(1, dtype=torch.float64, device="cuda")
        mb.adjoint_step(sim.ctx, qo, vo, ext, body, gqo, go, gko)
        for a, b in ((gqo, gq), (go, gv), (gko, gk)):
            assert rel_l2(to_np(a), to_np(b)) < 1e-12
        assert _untouched(store, off, v.numel()) and _untouched(qstore, off, q.numel())
        assert torch.equal(vo, v) and torch.equal(qo, q)

        def loss(qq, vv):
            sim.set_positions(qq)
            sim.set_velocity_field(vv)
            sim.step(1, ext_blob_force=ext, body_force=body)
            dq = sim.blob_positions() - q
            dq -= torch.round(dq / L) * L
            return float((cq * dq).sum() + (cv * sim.velocity_field()).sum())

        eps = 1e-6
        for dq, dv, g in ((dev(rng.normal(size=s.pos.shape)), 0.0 * v, gq),
                          (0.0 * q, dev(rng.normal(size=shape)), gv)):
            fd = (loss(q + eps * dq, v + eps * dv) - loss(q - eps * dq, v - eps * dv)) / (2 * eps)
            an = float((g * (dv if g is gv else dq)).sum())
            assert abs(an - fd) < 1e-6 * max(1.0, abs(fd)), (an, fd)


@pytest.mark.parametrize("off", [1, 2, 3])
@pytest.mark.parametrize("prec,n", [(0, (16, 8, 32)), (0, (32, 64, 4)), (0, (8, 8, 256)),
                                    (1, (16, 8, 32)), (1, (256, 8, 4))])
@pytest.mark.parametrize("advection", [0, 1])
def test_fluid_update_on_odd_offsets(prec, n, advection, off):
    dt = torch.float64 if prec else torch.float32
    shape = (1, 3, n[2], n[1], n[0])
    g = torch.Generator(device="cuda").manual_seed(off)
    v, f = (torch.randn(shape, generator=g, device="cuda", dtype=dt) for _ in range(2))
    with mb.Multiblob(mb.GridDesc(*n, precision=prec, advection=advection)) as sim:
        want = sim.fluid_update(v, f)
        (vo, _), (fo, _), (out, store) = (_odd(shape, dt, off, x) for x in (v, f, None))
        mb.fluid_update(sim.ctx, vo, fo, out)
        assert torch.equal(out, want) and _untouched(store, off, v.numel())
        assert torch.equal(vo, v) and torch.equal(fo, f)
        mb.fluid_update(sim.ctx, vo, None, vo)             # in place, without a force
        assert torch.equal(vo, sim.fluid_update(v))

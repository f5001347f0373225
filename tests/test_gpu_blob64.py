"""The FP64 blob kernels at the edges of their launch rules (a thread per blob and component up
to 4096 blobs, small blocks up to 16384), positions outside the box and at exact midpoints of
nodes, graph replays of FP64 steps, and the adjoint's in-place arrays.

Tolerances: an interpolated value or a node sum is a handful of terms of weights good to a few
ulps, so 1e-13 (FP64) and 2e-6 (FP32: 27 products and sums of 2^-24 each) in relative L2.
"""
import numpy as np
import pytest

import oracle
from helpers import assert_positions, rel_l2, to_np

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("CUDA device required", allow_module_level=True)

import paper_1407_5600_gb300 as mb  # noqa: E402
from paper_1407_5600_gb300 import workloads as wl  # noqa: E402

TOL = {0: 2e-6, 1: 1e-13}


@pytest.mark.parametrize("prec", [1, 0])
@pytest.mark.parametrize("n", [1, 31, 33, 4096, 4097, 16384, 16385])
def test_operators_at_launch_edges(prec, n):
    shape, h = (8, 32, 16), 0.7
    d = mb.GridDesc(16, 32, 8, h=h, precision=prec)
    g = oracle.Grid(16, 32, 8, h=h)
    q, F, _ = wl.random_blobs(n, shape, seed=n, h=h)
    rng = np.random.default_rng(n)
    k = max(1, n // 3)                              # a third at midpoints of nodes and on nodes
    q[:k] = np.round(2 * q[:k] / h) * h / 2
    q = np.mod(q, g.L)
    out = q + rng.integers(-3, 4, size=q.shape) * g.L          # the same blobs, outside the box
    v = wl.random_field(shape, seed=n + 1).astype(d.grid_dtype).astype(np.float64)
    with mb.Multiblob(d) as sim:
        f = to_np(sim.spread(out, F))[0]
        u = to_np(sim.interp(out, v[None]))
    assert rel_l2(f, oracle.spread(g, q, F)) < TOL[prec] + 1e-14 * 4
    assert rel_l2(u, oracle.interp(g, q, v)) < TOL[prec] + 1e-14 * 4


@pytest.mark.parametrize("det,integrator", [(1, 0), (0, 0), (0, 1)])
def test_fp64_graph_replays(monkeypatch, det, integrator):
    """Seven steps (two direct, the rest replayed) with the body force's axis changed between
    them, against the oracle; deterministic steps give the bits of direct launches."""
    spec, s = wl.dense_suspension(n=16, a=2.2, phi=0.2, seed=3, mc_sweeps=1)
    ext = np.random.default_rng(4).normal(scale=1e-3, size=s.pos.shape)
    bodies = [((1e-3, 0, 2, 1), 4), ((1e-3, 1, 0, 1), 3)]
    got = []
    for no_graph in ("1", "0"):
        monkeypatch.setenv("MB_NO_GRAPH", no_graph)
        d = mb.GridDesc(16, 16, 16, dt=spec.dt, precision=1, deterministic=det, mean_mode=1,
                        integrator=integrator)
        with mb.Multiblob(d) as sim:
            sim.set_particles(0, s.pos, s.pid, s.bonds, s.rest, s.k_spring, s.k_rep, s.r_cut)
            for body, n in bodies:
                sim.step(n, ext_blob_force=ext, body_force=body)
            got.append((to_np(sim.blob_positions()), to_np(sim.velocity_field())[0]))
    g = oracle.Grid(16, 16, 16, dt=spec.dt, mean_mode=1)
    q, v = s.pos, g.zeros()
    for body, n in bodies:
        args = (s.pid, s.bonds, s.rest, s.k_spring, s.k_rep, s.r_cut)
        q, v = (oracle.stokes_step(g, n, q, *args, ext=ext, body=body) if integrator else
                oracle.step(g, n, q, v, *args, ext=ext, body=body))
    for q_gpu, v_gpu in got:
        assert_positions(q_gpu, q, s.pos, g.L, 7, 1e-10)
        assert rel_l2(v_gpu, v) < 1e-10
    if det:
        assert np.array_equal(got[0][0], got[1][0]) and np.array_equal(got[0][1], got[1][1])


@pytest.mark.parametrize("k_rep", [0.0, 50.0])
def test_adjoint_arrays_in_place_and_staged(k_rep):
    """The adjoint of a step from device arrays (used in place), host arrays and gradients that
    share memory with the inputs gives the same results."""
    spec, s = wl.dense_suspension(n=16, a=2.2, phi=0.2, seed=3, mc_sweeps=1)
    rng = np.random.default_rng(6)
    d = mb.GridDesc(16, 16, 16, precision=1, dt=spec.dt)
    v0 = wl.random_field((16, 16, 16), 7, scale=1e-2)[None]
    cq, cv, body = rng.normal(size=s.pos.shape), rng.normal(size=v0.shape), (1e-3, 0, 2, 1)
    dev = lambda x: torch.tensor(x, device="cuda")  # noqa: E731
    res = []
    with mb.Multiblob(d) as sim:
        sim.set_particles(0, s.pos, s.pid, s.bonds, s.rest, s.k_spring, k_rep, 1.0)
        gq, gv, gk = dev(cq), dev(cv), torch.zeros(1, dtype=torch.float64, device="cuda")
        mb.adjoint_step(sim.ctx, dev(s.pos), dev(v0), dev(cq), body, gq, gv, gk)
        res.append((to_np(gq), to_np(gv), to_np(gk)))
        gq, gv, gk = cq.copy(), cv.copy(), np.zeros(1)
        mb.adjoint_step(sim.ctx, s.pos, v0, cq, body, gq, gv, gk)
        res.append((gq, gv, gk))
        both = dev(cq)                             # the external forces and dL/dq in one array
        gv, gk = dev(cv), torch.zeros(1, dtype=torch.float64, device="cuda")
        mb.adjoint_step(sim.ctx, dev(s.pos), dev(v0), both, body, both, gv, gk)
        res.append((to_np(both), to_np(gv), to_np(gk)))
    for r in res[1:]:
        for a, b in zip(r, res[0]):
            assert rel_l2(a, b) < 1e-10


@pytest.mark.parametrize("prec", [1, 0])
def test_state_arrays_are_free_on_return(prec):
    """Page-locked host arrays given to set_positions and set_velocity_field behind a queue of
    steps may be overwritten as soon as the calls return; so may a device array by another
    stream's work."""
    d = mb.GridDesc(32, 32, 32, precision=prec, mean_mode=1, dt=0.01)
    rng = np.random.default_rng(5)
    none = (np.zeros((0, 2), np.int32), np.zeros(0))
    q0 = rng.random((200, 3)) * 32
    v0 = wl.random_field((32, 32, 32), 6).astype(d.grid_dtype)[None]
    dev = torch.tensor(q0, device="cuda")
    other = torch.cuda.Stream()
    torch.cuda.synchronize()
    with mb.Multiblob(d) as sim:
        sim.set_particles(0, rng.random((200, 3)) * 32, np.arange(200, dtype=np.int32), *none, 0.0)
        for kind in ("pinned", "device"):
            sim.step(200, body_force=(0.1, 0, 1, 1))
            if kind == "pinned":
                q, v = torch.tensor(q0).pin_memory(), torch.tensor(v0).pin_memory()
                mb.set_positions(sim.ctx, q.numpy())
                q.zero_()
                sim.step(200)
                mb.set_velocity_field(sim.ctx, v.numpy())
                v.zero_()
                assert np.array_equal(to_np(sim.velocity_field()), v0)
                sim.step(200)
                mb.set_positions(sim.ctx, torch.tensor(q0).pin_memory().numpy())
            else:
                mb.set_positions(sim.ctx, dev)
                with torch.cuda.stream(other):
                    dev.zero_()
            assert np.max(np.abs(to_np(sim.blob_positions()) - q0)) < 1e-12


@pytest.mark.parametrize("pattern", [True, False])
def test_springs_of_blobs_that_move_by_more_than_the_box(pattern):
    """A field under which half a step carries the ends of a bond several boxes apart: the spring is
    that of the nearest images, as for any two positions (1e-9: the differences of positions of up
    to ten boxes are rounded at 1e-15 of them, the spring multiplies the bond's by a few)."""
    n, L = 8, 8.0
    pos = np.array([[1.0, 1.0, 1.0], [1.8, 5.5, 1.5], [4.0, 2.0, 6.0], [4.9, 6.0, 6.5]])
    pid, bonds = np.array([0, 0, 1, 1], np.int32), np.array([[0, 1], [2, 3]], np.int32)
    rest = np.array([3.0, 3.0 if pattern else 3.1])
    v = np.zeros((1, 3, n, n, n))
    v[0, 0, :, 4:, :] = 900.0                     # 2.8 boxes in half a step, in half of the box
    d = mb.GridDesc(n, n, n, precision=1, dt=0.05)
    with mb.Multiblob(d) as sim:
        sim.set_particles(0, pos, pid, bonds, rest, 40.0)
        sim.set_velocity_field(v)
        sim.step(1)
        F, qh = (to_np(x) for x in sim.last_forces())
    assert np.min(np.max(np.abs(qh[bonds[:, 0]] - qh[bonds[:, 1]]), axis=1)) > 1.5 * L
    F_ref = oracle.bond_forces(oracle.Grid(n, n, n, dt=0.05), qh, bonds, rest, 40.0)
    assert rel_l2(F, F_ref) < 1e-9

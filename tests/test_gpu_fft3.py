"""The FP32 three-pass fluid update on every line layout it chooses from (sides of 32, 64 and 128
at compile-time offsets, shorter ones at run-time offsets), steps whose blobs leave most planes of
the force grid untouched, and steps at the edges of the few-blob kernels (three blobs a warp, up
to 24,576 blobs), against the FP64 oracle.

Tolerances: FP32 line transforms of up to 128 points in three directions and back are a few 1e-7
off in relative L2, held to 2e-6.  A step adds at most that to the velocity, so 24 steps are held
to 5e-5 and three to 6e-6; a plane of forces or a blob lost or kept would be off by far more.
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


@pytest.mark.parametrize("advection", [0, 1])
@pytest.mark.parametrize("n", [(32, 32, 32), (64, 32, 4), (128, 32, 16), (32, 64, 64), (64, 64, 64),
                               (128, 64, 8), (32, 128, 128), (64, 128, 32), (128, 128, 64),
                               (16, 64, 32), (64, 16, 128), (8, 4, 64), (4, 8, 32)])
def test_fluid_update_three_pass_fp32(n, advection):
    nx, ny, nz = n
    kw = dict(h=0.8, rho=1.2, eta=0.7, dt=0.1)
    d = mb.GridDesc(nx, ny, nz, precision=0, advection=advection, **kw)
    v = (0.1 * wl.random_field((nz, ny, nx), 51)).astype(np.float32).astype(np.float64)
    f = wl.random_field((nz, ny, nx), 52, scale=0.3).astype(np.float32).astype(np.float64)
    body = (0.3, 1, 0, 2)
    with mb.Multiblob(d) as sim:
        got = to_np(sim.fluid_update(v, f, body_force=body))[0]
    g = oracle.Grid(nx, ny, nz, advection=advection, **kw)
    assert rel_l2(got, oracle.fluid_update(g, v, f, body=body)) < 2e-6


@pytest.mark.parametrize("nblobs,nz", [(3, 64), (3, 16), (700, 32)])
def test_fp32_steps_with_few_planes_spread_into(nblobs, nz):
    """Free blobs driven along z through about a plane a step, two boxes of different forces, the
    blobs set anew elsewhere half-way (from few blobs to one for every 32 nodes, where the
    corrector reads the summed velocity)."""
    g = oracle.Grid(32, 16, nz, dt=0.5, mean_mode=1)
    d = mb.GridDesc(32, 16, nz, dt=0.5, precision=0, mean_mode=1, batch=2)
    rng = np.random.default_rng(nblobs + nz)
    none = (np.zeros((0, 2), np.int32), np.zeros(0))
    pid = np.arange(nblobs, dtype=np.int32)
    F = rng.normal(size=(2, nblobs, 3)) * [1.0, 1.0, 4.0]
    F[:, :, 2] += 300.0 / nblobs
    q0 = rng.random((2, 2, nblobs, 3)) * [32, 16, 3]
    q0[1, :, :, 2] += 7
    with mb.Multiblob(d) as sim:
        for half in range(2):
            for b in range(2):
                sim.set_particles(b, q0[half, b], pid, *none, 0.0)
            sim.step(5, ext_blob_force=F.reshape(-1, 3))
            sim.step(7, ext_blob_force=F.reshape(-1, 3))
        got = to_np(sim.velocity_field())
    for b in range(2):
        v = g.zeros()
        for half in range(2):
            _, v = oracle.step(g, 12, q0[half, b], v, pid, *none, 0.0, 0.0, 0.0, ext=F[b])
        assert rel_l2(got[b], v) < 5e-5


@pytest.mark.parametrize("mean_mode", [0, 1])
@pytest.mark.parametrize("nblobs", [1, 2, 4, 11, 13, 4099, 24576, 24577])
def test_fp32_steps_at_the_edges_of_the_few_blob_kernels(nblobs, mean_mode):
    """Two boxes that share the blobs out unevenly, three steps."""
    g = oracle.Grid(32, 16, 64, dt=0.2, mean_mode=mean_mode)
    d = mb.GridDesc(32, 16, 64, dt=0.2, precision=0, mean_mode=mean_mode, batch=2)
    rng = np.random.default_rng(nblobs)
    none = (np.zeros((0, 2), np.int32), np.zeros(0))
    n = [nblobs // 3, nblobs - nblobs // 3]
    q0 = [rng.random((k, 3)) * [32, 16, 64] for k in n]
    F = [rng.normal(size=(k, 3)) for k in n]
    with mb.Multiblob(d) as sim:
        for b in range(2):
            sim.set_particles(b, q0[b], np.arange(n[b], dtype=np.int32), *none, 0.0)
        sim.step(3, ext_blob_force=np.concatenate(F))
        v, q = to_np(sim.velocity_field()), to_np(sim.blob_positions())
    for b, lo in ((0, 0), (1, n[0])):
        if n[b] == 0:
            continue
        q_ref, v_ref = oracle.step(g, 3, q0[b], g.zeros(), np.arange(n[b], dtype=np.int32), *none,
                                   0.0, 0.0, 0.0, ext=F[b])
        assert rel_l2(v[b], v_ref) < 6e-6
        assert_positions(q[lo:lo + n[b]], q_ref, q0[b], g.L, 3, 2e-5)


@pytest.mark.parametrize("nblobs", [1, 4, 13, 24576, 24577])
def test_fp32_stokes_steps_at_the_edges_of_the_few_blob_kernels(nblobs):
    """Two boxes, a direct step, then graph replays that clear the force grid as they read it."""
    g = oracle.Grid(32, 16, 64, dt=0.05, mean_mode=1)
    d = mb.GridDesc(32, 16, 64, dt=0.05, precision=0, mean_mode=1, integrator=1, batch=2)
    rng = np.random.default_rng(nblobs)
    none = (np.zeros((0, 2), np.int32), np.zeros(0))
    n = [nblobs // 3, nblobs - nblobs // 3]
    q0 = [rng.random((k, 3)) * [32, 16, 64] for k in n]
    F = [rng.normal(size=(k, 3)) for k in n]
    with mb.Multiblob(d) as sim:
        for b in range(2):
            sim.set_particles(b, q0[b], np.arange(n[b], dtype=np.int32), *none, 0.0)
        sim.step(4, ext_blob_force=np.concatenate(F))
        v, q = to_np(sim.velocity_field()), to_np(sim.blob_positions())
    for b, lo in ((0, 0), (1, n[0])):
        if n[b] == 0:
            continue
        q_ref, v_ref = oracle.stokes_step(g, 4, q0[b], np.arange(n[b], dtype=np.int32), *none,
                                          0.0, 0.0, 0.0, ext=F[b])
        assert rel_l2(v[b], v_ref) < 1e-5            # the repository's bound for FP32 Stokes steps
        assert_positions(q[lo:lo + n[b]], q_ref, q0[b], g.L, 4, 2e-5)


@pytest.mark.parametrize("n", [(8, 256, 8), (16, 16, 64)])
def test_fp32_stokes_replays_after_the_tile_timing(n):
    """Stokes steps in both numbers of passes whose first, direct step times the spreading tiles
    and leaves the force grid cleared: the replays after it clear it themselves where due."""
    g = oracle.Grid(*n, dt=0.3, mean_mode=1)
    d = mb.GridDesc(*n, dt=0.3, precision=0, mean_mode=1, integrator=1)
    rng = np.random.default_rng(n[1])
    none = (np.zeros((0, 2), np.int32), np.zeros(0))
    for nblobs in (7, 19):                    # a tile choice of their own each
        q0, F = rng.random((nblobs, 3)) * n, rng.normal(size=(nblobs, 3))
        F -= F.mean(0)
        pid = np.arange(nblobs, dtype=np.int32)
        with mb.Multiblob(d) as sim:
            sim.set_particles(0, q0, pid, *none, 0.0)
            sim.step(5, ext_blob_force=F)
            v, q = to_np(sim.velocity_field())[0], to_np(sim.blob_positions())
        q_ref, v_ref = oracle.stokes_step(g, 5, q0, pid, *none, 0.0, 0.0, 0.0, ext=F)
        assert rel_l2(v, v_ref) < 1e-5
        assert_positions(q, q_ref, q0, g.L, 5, 2e-5)


@pytest.mark.parametrize("integrator", [0, 1])
@pytest.mark.parametrize("nblobs", [10240, 10241, 16512, 16513])
def test_fp32_steps_at_the_edges_of_the_few_blob_rules(nblobs, integrator):
    """32^3 cells: nine lanes a blob up to 10240 (spreading) and 16384 + cells / 256
    (interpolation) blobs."""
    g = oracle.Grid(32, 32, 32, dt=0.1, mean_mode=1)
    d = mb.GridDesc(32, 32, 32, dt=0.1, precision=0, mean_mode=1, integrator=integrator)
    rng = np.random.default_rng(nblobs)
    none = (np.zeros((0, 2), np.int32), np.zeros(0))
    q0, F = rng.random((nblobs, 3)) * 32, rng.normal(size=(nblobs, 3))
    F -= F.mean(0)
    pid = np.arange(nblobs, dtype=np.int32)
    with mb.Multiblob(d) as sim:
        sim.set_particles(0, q0, pid, *none, 0.0)
        sim.step(3, ext_blob_force=F)
        v, q = to_np(sim.velocity_field())[0], to_np(sim.blob_positions())
    if integrator:
        q_ref, v_ref = oracle.stokes_step(g, 3, q0, pid, *none, 0.0, 0.0, 0.0, ext=F)
    else:
        q_ref, v_ref = oracle.step(g, 3, q0, g.zeros(), pid, *none, 0.0, 0.0, 0.0, ext=F)
    assert rel_l2(v, v_ref) < (1e-5 if integrator else 6e-6)
    assert_positions(q, q_ref, q0, g.L, 3, 2e-5)


@pytest.mark.parametrize("integrator,nblobs,timed", [(0, 13, False), (0, 10240, False), (0, 10241, True),
                                                     (1, 13, True)])
def test_tiles_are_timed_where_they_are_used(integrator, nblobs, timed):
    """Inertial steps of few blobs spread without tiles, and none is timed then (32,768 cells: up to
    10,240 blobs).  Grid and blob counts of no other test, whose choice would be taken over."""
    rng = np.random.default_rng(nblobs)
    none = (np.zeros((0, 2), np.int32), np.zeros(0))
    d = mb.GridDesc(16, 64, 32, dt=0.05, mean_mode=1, integrator=integrator)
    with mb.Multiblob(d) as sim:
        sim.set_particles(0, rng.random((nblobs, 3)) * [16, 64, 32], np.arange(nblobs, dtype=np.int32), *none, 0.0)
        sim.step(4, ext_blob_force=rng.normal(size=(nblobs, 3)))
        tile, ms = mb.get_tuning(sim.ctx)
    assert len(tile) == 3 and (ms > 0.0) == timed

"""Steps and CUDA graphs.

FP64 steps captured into a caller's CUDA graph: accepted before any step and after the library
has graphs of its own, replayed any number of times, with the library's own steps before, between
and after; the same states as steps taken one by one.

Tolerance: deterministic steps agree to the bit; the others add with atomics in any order, 1e-12
over a dozen steps (the forces differ by the rounding of at most a few hundred terms a node).
"""
import numpy as np
import pytest

from helpers import assert_positions, rel_l2, to_np

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("CUDA device required", allow_module_level=True)

import paper_1407_5600_gb300 as mb  # noqa: E402
from paper_1407_5600_gb300 import workloads as wl  # noqa: E402


@pytest.mark.parametrize("integrator,deterministic,n", [(0, 0, (16, 16, 16)), (0, 1, (16, 16, 16)),
                                                        (1, 0, (16, 16, 16)), (0, 0, (8, 8, 256))])
@pytest.mark.parametrize("warm", [1, 2, 7])
def test_steps_in_a_callers_graph(integrator, deterministic, n, warm):
    rng = np.random.default_rng(warm)
    s = wl.build_particles(rng.random((2, 3)) * n, 1.0, rng, n)
    ext = torch.as_tensor(rng.normal(scale=1e-2, size=s.pos.shape), device="cuda")
    stream = torch.cuda.Stream()
    stream.wait_stream(torch.cuda.current_stream())
    d = mb.GridDesc(*n, precision=1, integrator=integrator, mean_mode=integrator,
                    deterministic=deterministic)
    with torch.cuda.stream(stream), mb.Multiblob(d, stream=stream) as a, mb.Multiblob(d, stream=stream) as b:
        for sim in (a, b):
            sim.set_particles(0, s.pos, s.pid, s.bonds, s.rest, 20.0, 10.0, 1.0)
            sim.step(warm, ext_blob_force=ext)
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream, capture_error_mode="thread_local"):
            a.step(2, ext_blob_force=ext)
        graph.replay()
        a.step(2, ext_blob_force=ext)
        graph.replay()
        graph.replay()
        a.step(2, ext_blob_force=ext)
        b.step(10, ext_blob_force=ext)
        for x, y in ((a.blob_positions(), b.blob_positions()), (a.velocity_field(), b.velocity_field())):
            assert rel_l2(to_np(x), to_np(y)) < 1e-12
        if deterministic:
            assert torch.equal(a.last_forces()[0], b.last_forces()[0])
            assert torch.equal(a.blob_positions(), b.blob_positions())
            assert torch.equal(a.velocity_field(), b.velocity_field())


@pytest.mark.parametrize("prec,integrator", [(0, 0), (0, 1), (1, 0), (1, 1)])
def test_steps_that_alternate_in_their_forces(prec, integrator, monkeypatch):
    """Calls with and without external forces and with body forces along different axes in turn,
    each from the captured step of its own kind, against direct launches.  The same kernels in the
    same order: FP64 1e-12 (atomics in any order), FP32 1e-5 (the repository's bound)."""
    n = 16
    rng = np.random.default_rng(31)
    s = wl.build_particles(rng.random((2, 3)) * n, 1.5, rng, (n, n, n))
    ext = torch.as_tensor(rng.normal(scale=1e-2, size=s.pos.shape), device="cuda")
    d = mb.GridDesc(n, n, n, precision=prec, integrator=integrator, mean_mode=integrator)
    kinds = [(e, b) for e in (None, ext) for b in (None, (1e-2, 0, 2, 1), (2e-2, 1, 0, 1), (1e-2, 0, 1, 2))]

    def run():
        with mb.Multiblob(d) as sim:
            sim.set_particles(0, s.pos, s.pid, s.bonds, s.rest, 20.0, 10.0, 1.0)
            for i in range(40):
                e, b = kinds[(5 * i) % len(kinds)]
                sim.step(1 + i % 3, ext_blob_force=e, body_force=b)
            return to_np(sim.blob_positions()), to_np(sim.velocity_field())

    q, v = run()
    monkeypatch.setenv("MB_NO_GRAPH", "1")
    q_ref, v_ref = run()
    tol = 1e-12 if prec else 1e-5
    assert rel_l2(v, v_ref) < tol
    assert_positions(q, q_ref, s.pos, (n, n, n), 80, tol)

"""The fluid update leaves smooth flows their amplitude: a cellular flow (the discrete curl of
sin sin along two axes) is divergence-free and an eigenmode of the discrete update, so that after
m updates it is f^m of itself, f = (rho/dt - eta lambda/2) / (rho/dt + eta lambda/2).  At large
theta = eta dt / (rho h^2) the weights of the stencil are 3 theta times larger than what is left of
them on such a flow, so a rounding of theirs that does not cancel shows in every update, the same
way each time.

Tolerance per update, in ulps of 2^-23 (FP32), 2^-52 (FP64, five passes) and 2^-47 (double-float,
three passes): every level of the two axes' transforms, log2 n there and back, may scale the mode by
the rounding of its twiddles' modulus, half an ulp; the solve adds the rounding of the symbol, the
sum and the reciprocal, three ulps; the rounding of a node's terms, 3 theta ulps, is random over
the nodes of a plane.
"""
import math

import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("CUDA device required", allow_module_level=True)

import paper_1407_5600_gb300 as mb  # noqa: E402


def _cellular(n, axes):
    """[3, nz, ny, nx]: wave number one along both axes, phases off the nodes' symmetries."""
    a, b = axes
    x = [2 * math.pi * (torch.arange(k, dtype=torch.float64) + 0.3) / k for k in n]
    view = [(1, 1, -1), (1, -1, 1), (-1, 1, 1)]
    psi = torch.sin(x[a]).view(view[a]) * torch.sin(x[b]).view(view[b])
    psi = psi.expand(n[2], n[1], n[0])
    v = torch.zeros((3, n[2], n[1], n[0]), dtype=torch.float64)
    v[a] = torch.roll(psi, -1, 2 - b) - psi
    v[b] = psi - torch.roll(psi, -1, 2 - a)
    return v


@pytest.mark.parametrize("prec,n,ulp", [
    (0, (256, 128, 8), 2.0 ** -23), (0, (8, 256, 128), 2.0 ** -23), (0, (128, 8, 256), 2.0 ** -23),
    (0, (128, 128, 8), 2.0 ** -23),
    (1, (256, 128, 8), 2.0 ** -52), (1, (8, 256, 128), 2.0 ** -52), (1, (128, 8, 256), 2.0 ** -52),
    (1, (128, 128, 8), 2.0 ** -47), (1, (8, 128, 128), 2.0 ** -47), (1, (128, 8, 128), 2.0 ** -47)])
@pytest.mark.parametrize("rho,eta,h,dt", [
    (1.0, 10.1, 0.7, 1.0), (1.13, 97.3, 0.71, 1.07), (0.83, 31.7, 0.6, 0.91), (1.9, 1.3, 0.9, 0.031)])
def test_cellular_flow_keeps_its_amplitude(prec, n, ulp, rho, eta, h, dt):
    a, b = (d for d in range(3) if n[d] > 8)
    lam = sum(4.0 / h ** 2 * math.sin(math.pi / n[d]) ** 2 for d in (a, b))
    theta = eta * dt / (rho * h ** 2)
    updates = max(1, min(20, int(1.0 / (theta * lam * h ** 2))))
    with mb.Multiblob(mb.GridDesc(*n, rho=rho, eta=eta, h=h, dt=dt, precision=prec)) as sim:
        v = _cellular(n, (a, b))[None].to(device="cuda", dtype=sim.grid_dtype)
        u = v
        for _ in range(updates):
            u = sim.fluid_update(u)
        u, v = u.double(), v.double()
        got = float((u * v).sum() / (v * v).sum())
    f = (rho / dt - 0.5 * eta * lam) / (rho / dt + 0.5 * eta * lam)
    tol = (math.log2(n[a] * n[b]) + 3 + 3 * theta / math.sqrt(n[a] * n[b])) * ulp
    assert abs(got / f ** updates - 1.0) < updates * tol, (got / f ** updates - 1.0, updates * tol)

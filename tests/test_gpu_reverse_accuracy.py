"""Rounding of the residual's gradient, with dissipation: its relative L2 distance
from a reference whose own rounding is averaged out -- the residual scales with
the state (r(a u) = a r(u)) and inversely with the mesh, so the gradient is the
same for every scaling, while the roundings of the plain torch form (perf/cases.py)
differ; the mean over K scalings carries 1/sqrt(K) of them.

Bounds: the distance of the float64 kernels that took a division for every
reciprocal, 2.75e-15 (triangles) and 2.45e-15 (tetrahedra), plus the
reference's share at K = 12 (0.5e-15, in squares) and 2 % for another state:
2.85e-15 and 2.55e-15."""
import copy
import random

import pytest
import torch

pytestmark = pytest.mark.gpu

K = 12


@pytest.mark.parametrize("grid,n,bound", [("tri", 40, 2.85e-15), ("tet", 6, 2.55e-15)])
def test_gradient_rounding(grid, n, bound):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from perf import cases
    case = dict(call="adjoint", grid=grid, p=1, n=n, scheme="split", precision="fp64", dissipation=True, viscous=False)
    st = cases.prepare(case, 1)
    g = cases.run(st)["grad"]
    op, m, u = cases._inputs(case, 1)
    cot = st["cot"].transpose(1, 2)
    rng, ref = random.Random(7), torch.zeros_like(g)
    for k in range(K):
        a, b, h = (rng.uniform(1.0, 2.0) for _ in range(3))
        ms = copy.copy(m)
        ms.nu, ms.Lam, ms.J = m.nu * b, m.Lam * b, m.J * h     # residual times b / h
        x = torch.as_tensor(u * a, device=g.device).transpose(1, 2).contiguous().requires_grad_(True)
        (gk,) = torch.autograd.grad(cases._Exact(case, op, ms, g.device).residual(x), x, cot)
        ref += gk.transpose(1, 2) * (h / b / K)
    st["solver"].close()
    err = float((g - ref).norm() / ref.norm())
    print(f"gradient, {grid}: {err:.3e}")
    assert err <= bound

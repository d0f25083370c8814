"""Accuracy of the tensor-core contraction against the summands of each node
itself (test_gpu_tensor_contraction.py bounds it by those of the element): a
state with one node per element whose conservative variables are larger than
the others' by a factor, up to which the digits resolve the small entries as a
float64 sum does (csrc/tc64.cuh: rounding of an operand 2^-60 or, above 32
nodes, 2^-63 of the largest entry).  The factors keep that rounding, 2^-60 times
30 or 2^-63 times 300 over n_p entries, below 2^-52 of a node's summands on rows
whose products reach 2^-3 of the largest one's.

Bound: ROUNDING_C eps times the node's summands, as for the other float64 parity
tests, at the interior nodes (the volume term alone), against the same term in
extended precision: the float64 oracle itself reaches 9 eps of them here."""
import numpy as np
import pytest
import torch

from esplit_inputs import tri_operator, tet_operator, periodic_tri_mesh, states
from esplit_inputs.mesh import periodic_tet_mesh
from parity_bounds import EPS, ROUNDING_C, summand_scale

pytestmark = pytest.mark.gpu


def _volume_term(op, m, u, e, gam=1.4, beta=2.5):
    """-sum_i [beta D_i f_i + A~_i D_i w] / (beta + 1) of element e (Eq. (100)
    without its facet part) in np.longdouble: 113 bits on aarch64, 64 on x86."""
    X = np.longdouble
    gam, beta = X(gam), X(beta)
    al, d, n_p = -gam - beta * (gam - 1), op.d, op.n_p
    Q, lam = op.Q.reshape(d, n_p, n_p).astype(X), m.Lam[e].reshape(d, d, n_p).astype(X)
    nu, H = m.nu[e].reshape(-1, d).astype(X), op.H.astype(X) * m.J[e].astype(X)
    U = u[e].astype(X)
    rho, V, E = U[0], U[1:-1] / U[0], U[-1]
    v2 = (V * V).sum(0)
    p = (gam - 1) * (E - rho * v2 / 2)
    q = (rho / p) * (p * rho ** (-gam)) ** (1 / (al + gam))
    a, th, aq, bq = -al / (gam - 1), p / rho, al / (al + gam), (1 - al - gam) / (al + gam)
    W = np.concatenate([[q * (a * th - v2 / 2)], q * V, [-q]])
    res = np.zeros_like(U)
    for i in range(d):
        S = sum((lam[i, j][:, None] * Q[j] - Q[j].T * lam[i, j][None, :]) / 2 for j in range(d))
        for s, n in enumerate(op.facet_nodes.reshape(-1)):
            S[n, n] += nu[s, i] / 2
        D = S / H[:, None]
        F = np.concatenate([[rho * V[i]], rho * V[i] * V, [(E + p) * V[i]]])
        F[1 + i] += p
        g, f = W @ D.T, F @ D.T
        dq = -g[-1]
        dV = (g[1:-1] - dq * V) / q
        vdv = (V * dV).sum(0)
        dth = ((g[0] - dq * (a * th - v2 / 2)) / q + vdv) / a
        drho = rho / (aq + bq) * (dq / q - bq * dth / th)
        dp = drho * th + rho * dth
        mom = (drho * V[i] + rho * dV[i]) * V + rho * V[i] * dV
        mom[i] += dp
        dE = dp / (gam - 1) + drho * v2 / 2 + rho * vdv
        dF = np.concatenate([[drho * V[i] + rho * dV[i]], mom, [(dE + dp) * V[i] + (E + p) * dV[i]]])
        res -= (beta * f + dF) / (beta + 1)
    return res


@pytest.mark.parametrize("d,p,factor", [(2, 2, 30.0), (2, 3, 30.0), (2, 4, 30.0), (3, 2, 30.0), (3, 3, 300.0),
                                        (3, 4, 300.0)])
def test_one_large_node(d, p, factor):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2305_07181_gb300 as es
    from oracle.physics import Params as OP
    if d == 2:
        op = tri_operator(p)
        m = periodic_tri_mesh(op, 6, 10.0, 0.05)
    else:
        op = tet_operator(p)
        m = periodic_tet_mesh(op, 2, 2 * np.pi, 0.02)
    u = states.random_positive_state(m.n_e, d, op.n_p, seed=5, vel=(-0.5, 0.5))
    node = np.random.default_rng(6).integers(op.n_p, size=m.n_e)
    u[np.arange(m.n_e), :, node] *= factor
    s = es.Solver(op, m, es.Params())
    r = s.residual(s.to_device(u)).cpu().numpy()
    assert s.status() == 0
    s.close()
    ro = np.stack([_volume_term(op, m, u, e) for e in range(m.n_e)])
    sc = summand_scale(u, op, m, np.arange(m.n_e), "split", OP(), dissipation=False)
    inner = np.setdiff1d(np.arange(op.n_p), op.facet_nodes.reshape(-1))
    ratio = (np.abs(r - ro) / (EPS * sc))[:, :, inner].max()
    print(f"d = {d}, p = {p}: {ratio:.2f} eps of the node's summands")
    assert ratio <= ROUNDING_C

"""Two-point flux and dissipation where the exponential average switches
(Eq. (47): fixed-point series below a relative jump of 0.05, quotient above):
element-wise constant states whose jumps are zero, at round-off, tiny, and on
both sides of the switch, with either sign, in density and pressure, against
the oracle.  Bound: ROUNDING_C eps times the largest summand of the element,
as for the other float64 parity tests."""
import numpy as np
import pytest
import torch

from esplit_inputs import tri_operator, tet_operator, periodic_tri_mesh, states
from esplit_inputs.mesh import periodic_tet_mesh
from parity_bounds import EPS, ROUNDING_C, summand_scale

pytestmark = pytest.mark.gpu

JUMPS = np.array([0.0, 1e-15, -1e-15, 1e-8, -1e-8, 1e-3, -1e-3, 0.0499999, -0.0499999, 0.05, -0.05, 0.0500001, 0.051])


@pytest.mark.parametrize("scheme", ["split", "hadamard"])
@pytest.mark.parametrize("d,p", [(2, 1), (2, 3), (3, 2)])
def test_jumps_across_the_series_switch(d, p, scheme):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2305_07181_gb300 as es
    from oracle import residual as R
    from oracle.physics import Params as OP
    if d == 2:
        op = tri_operator(p)
        m = periodic_tri_mesh(op, 5, 10.0, 0.05)
    else:
        op = tet_operator(p)
        m = periodic_tet_mesh(op, 2, 2 * np.pi, 0.02)
    rng = np.random.default_rng(11)
    rho = np.repeat(1.3 * (1.0 + rng.choice(JUMPS, m.n_e))[:, None], op.n_p, 1)
    pr = np.repeat(0.9 * (1.0 + rng.choice(JUMPS, m.n_e))[:, None], op.n_p, 1)
    V = np.repeat(rng.uniform(-0.4, 0.4, (d, m.n_e))[:, :, None], op.n_p, 2)
    u = np.ascontiguousarray(np.moveaxis(states.prim_to_cons(rho, V, pr), 0, 1))
    s = es.Solver(op, m, es.Params(scheme=scheme, dissipation=True))
    r = s.residual(s.to_device(u)).cpu().numpy()
    assert s.status() == 0
    s.close()
    ro = R.residual(u, op, m, OP(), scheme=scheme, dissipation=True).numpy()
    sc = summand_scale(u, op, m, np.arange(m.n_e), scheme, OP()).max(axis=2, keepdims=True)
    assert np.all(np.abs(r - ro) <= ROUNDING_C * EPS * sc)

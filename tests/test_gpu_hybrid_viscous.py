"""Relaxation step of the hybrid scheme with viscous terms and mixed flags: the
entropy of u_n covers the elements of both forms, so g, the entropy before the
step, the stage productions and the state equal the oracle's, one step at a
time and recorded as a graph.  Bounds as for the other relaxation parity tests
(g 1e-10, states 1e-12)."""
import numpy as np
import pytest
import torch

from esplit_inputs import tri_operator, tet_operator, periodic_tri_mesh, states
from esplit_inputs.mesh import periodic_tet_mesh

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,p,every", [(2, 1, 2), (2, 3, 5), (3, 1, 3), (3, 2, 2)])
def test_rrk_step(d, p, every):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2305_07181_gb300 as es
    from oracle import residual as R, rrk
    from oracle.physics import Params as OP
    if d == 2:
        op = tri_operator(p)
        m = periodic_tri_mesh(op, 5, 10.0, 0.05)
        u0 = states.add_uniform_noise(states.isentropic_vortex(m), 1e-2, 3)
    else:
        op = tet_operator(p)
        m = periodic_tet_mesh(op, 2, 2 * np.pi, 0.02)
        u0 = states.add_uniform_noise(states.taylor_green(m), 1e-2, 3)
    flags = (np.arange(m.n_e) % every == 0).astype(np.uint8)   # split list shorter than the mesh, and ragged
    mu = 1.0 / 50.0
    dt = states.cfl_timestep(m, u0, 0.05)
    s = es.Solver(op, m, es.Params(scheme="hybrid", dissipation=True, viscous=True, mu=mu))
    s.set_hybrid_flags(flags)
    ud = s.to_device(u0)
    uo = torch.as_tensor(u0)
    prm = OP(mu=mu)
    rhs = lambda x: R.residual(x, op, m, prm, scheme="hybrid", dissipation=True, viscous=True, hybrid_flags=flags)
    for _ in range(2):
        g, info = s.rrk_step(ud, dt)
        uo, io = rrk.rrk4_step(uo, dt, rhs, op, m, prm)
        assert abs(g - io.g) <= 1e-10
        assert abs(info.S_before - io.S_before) <= 1e-12 * abs(io.S_before)
        for a, b in zip(info.stage_rate, io.stage_production):
            assert abs(a - b) <= 1e-9 * abs(b)
        un = uo.numpy()
        assert np.abs(ud.cpu().numpy() - un).max() <= 1e-12 * np.abs(un).max()
    v = s.to_device(u0)
    s.rrk_steps(v, dt, 2)
    assert torch.equal(v, ud)
    s.close()

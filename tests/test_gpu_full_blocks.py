"""The split volume kernel and its reverse with blocks of several elements, which
take over where short blocks (as many elements as fill one warp) would be more
than four per SM: meshes just above that line for every operator, whose element
list leaves the last block ragged (58 and 78 nodes, two elements per block and
even meshes: through the list of the hybrid scheme).  Here the results of one
element go over the digits of the one before it (25, 58 and 78 nodes).

Residual: against the oracle at sampled elements, among them the first and the
last blocks, bounds as in test_gpu_tensor_contraction.py and
test_gpu_parity.py.  Gradient: against plain float64 torch (perf/cases.py); both
are within 3e-15 of the exact gradient in relative L2, so 1e-14 in L2 and, with
a factor of 10 for the largest of a million entries, 1e-13 in the maximum norm.
Step: bounds of the other relaxation parity tests."""
import numpy as np
import pytest
import torch

from esplit_inputs import tri_operator, tet_operator, periodic_tri_mesh, states
from esplit_inputs.mesh import periodic_tet_mesh
from parity_bounds import EPS, ROUNDING_C, summand_scale

pytestmark = pytest.mark.gpu

SHORT_MOST = 4 * 152
# d, p, nodes, elements per full block, cells per side
CASES = [(2, 1, 7, 18, 35), (2, 2, 12, 10, 26), (2, 3, 18, 7, 19), (2, 4, 27, 7, 19), (3, 1, 12, 10, 6),
         (3, 2, 25, 5, 6), (3, 3, 58, 2, 5), (3, 4, 78, 2, 5)]


def _setup(d, p, n_p, eb, n):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    if d == 2:
        op = tri_operator(p)
        m = periodic_tri_mesh(op, n, 10.0, 0.05)
    else:
        op = tet_operator(p)
        m = periodic_tet_mesh(op, n, 2 * np.pi, 0.02)
    assert op.n_p == n_p
    flags = np.zeros(m.n_e, dtype=np.uint8)
    if m.n_e % eb == 0:
        flags[m.n_e // 3] = 1          # one Hadamard-form element: an odd list
    n_split = m.n_e - int(flags.sum())
    assert -(-n_split // max(1, 32 // n_p)) > SHORT_MOST and n_split % eb != 0
    return op, m, flags


def _state(kind, m, d, n_p):
    u = states.random_positive_state(m.n_e, d, n_p, seed=5, vel=(-0.5, 0.5))
    if kind == "at_rest":
        u[:, -1] -= 0.5 * np.sum(u[:, 1:-1] ** 2, axis=1) / u[:, 0]
        u[:, 1:-1] = 0.0
    elif kind == "wide":
        u *= 10.0 ** np.random.default_rng(6).uniform(-3.0, 3.0, size=(m.n_e, 1, n_p))
    return u


@pytest.mark.parametrize("kind", ["ordinary", "at_rest", "wide"])
@pytest.mark.parametrize("d,p,n_p,eb,n", CASES)
def test_residual(d, p, n_p, eb, n, kind):
    op, m, flags = _setup(d, p, n_p, eb, n)
    import paper_2305_07181_gb300 as es
    from oracle import residual as R
    from oracle.physics import Params as OP
    u = _state(kind, m, d, op.n_p)
    scheme = "hybrid" if flags.any() else "split"
    s = es.Solver(op, m, es.Params(scheme=scheme))
    if flags.any():
        s.set_hybrid_flags(flags)
    r = s.residual(s.to_device(u)).cpu().numpy()
    assert s.status() == 0
    s.close()
    el = np.concatenate([np.arange(eb), np.random.default_rng(7).choice(m.n_e, 16, replace=False),
                         np.arange(m.n_e - 2 * eb, m.n_e)])
    el = np.unique(el[flags[el] == 0])
    ro = R.residual(u, op, m, OP(), scheme=scheme, hybrid_flags=flags if flags.any() else None, elems=el).numpy()
    sc = summand_scale(u, op, m, el, "split", OP(), dissipation=False).max(axis=2, keepdims=True)
    nodes = np.arange(op.n_p)
    if kind != "ordinary":             # facet nodes: conditioning of the means between very different states
        nodes = np.setdiff1d(nodes, op.facet_nodes.reshape(-1))
    if len(nodes):                     # 12-node tetrahedra have no interior node
        assert np.all((np.abs(r[el] - ro) <= ROUNDING_C * EPS * sc)[:, :, nodes])
    assert np.isfinite(r).all()


@pytest.mark.parametrize("d,p,n_p,eb,n", CASES)
def test_gradient(d, p, n_p, eb, n):
    _setup(d, p, n_p, eb, n)
    from perf import cases
    case = dict(call="adjoint", grid="tri" if d == 2 else "tet", p=p, n=n, scheme="split", precision="fp64",
                dissipation=True, viscous=False)
    st = cases.prepare(case, 3)
    g = cases.run(st)["grad"]
    ref = cases.exact(case, 3)["grad"]
    st["solver"].close()
    assert float((g - ref).norm()) <= 1e-14 * float(ref.norm())
    assert float((g - ref).abs().max()) <= 1e-13 * float(ref.abs().max())


@pytest.mark.parametrize("d,p,n_p,eb,n", [CASES[1], CASES[3], CASES[4], CASES[5]])
def test_relaxation_step(d, p, n_p, eb, n):
    op, m, _ = _setup(d, p, n_p, eb, n)
    import paper_2305_07181_gb300 as es
    from oracle import residual as R, rrk
    from oracle.physics import Params as OP
    u = states.isentropic_vortex(m) if d == 2 else states.taylor_green(m)
    u = states.add_uniform_noise(u, 1e-2, 3)
    dt = states.cfl_timestep(m, u, 0.1)
    s = es.Solver(op, m, es.Params(dissipation=True))
    ud = s.to_device(u)
    g, _ = s.rrk_step(ud, dt)
    s.close()
    uo, io = rrk.rrk4_step(torch.as_tensor(u), dt, lambda x: R.residual(x, op, m, OP(), dissipation=True), op, m, OP())
    uo = uo.numpy()
    assert abs(g - io.g) <= 1e-10
    assert np.abs(ud.cpu().numpy() - uo).max() <= 1e-12 * np.abs(uo).max()

"""The entropy-split residual where the tensor-core contraction (fixed-point
operator rows and columns cut into fp16 digits, csrc/tc64.cuh) could go wrong:
every operator size (padding of the 8- and 16-wide tiles, both digit widths),
element counts that leave the last block ragged, columns that are zero, and
states whose entries span six orders of magnitude inside an element.

Bound: ROUNDING_C eps times the largest summand of the element (the digits
are relative to the largest entry of a row or column), ROUNDING_C as for the
other float64 parity tests.  Compared at the interior nodes, whose residual is
the volume term alone: at a facet node the conditioning of the two-point
averages between very different states adds to the error of either side.
"""
import numpy as np
import pytest
import torch

from esplit_inputs import tri_operator, tet_operator, periodic_tri_mesh, states
from esplit_inputs.mesh import periodic_tet_mesh
from parity_bounds import EPS, ROUNDING_C, summand_scale

pytestmark = pytest.mark.gpu


def _mesh(d, p):
    if d == 2:
        op = tri_operator(p)
        return op, periodic_tri_mesh(op, 3, 10.0, 0.05)
    op = tet_operator(p)
    return op, periodic_tet_mesh(op, 2, 2 * np.pi, 0.02)


def _state(kind, m, d, n_p):
    u = states.random_positive_state(m.n_e, d, n_p, seed=5, vel=(-0.5, 0.5))
    if kind == "at_rest":      # zero momentum: whole columns of f_i and w are zero
        u[:, -1] -= 0.5 * np.sum(u[:, 1:-1] ** 2, axis=1) / u[:, 0]
        u[:, 1:-1] = 0.0
    elif kind == "wide":       # density and pressure scaled by 1e-3 .. 1e3, node by node
        u *= 10.0 ** np.random.default_rng(6).uniform(-3.0, 3.0, size=(m.n_e, 1, n_p))
    return u


@pytest.mark.parametrize("kind", ["ordinary", "at_rest", "wide"])
@pytest.mark.parametrize("d,p", [(2, 1), (2, 2), (2, 3), (2, 4), (3, 2), (3, 3), (3, 4)])  # (3, 1): no interior node
def test_split_residual_digits(d, p, kind):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2305_07181_gb300 as es
    from oracle import residual as R
    from oracle.physics import Params as OP
    op, m = _mesh(d, p)
    u = _state(kind, m, d, op.n_p)
    s = es.Solver(op, m, es.Params())
    r = s.residual(s.to_device(u)).cpu().numpy()
    assert s.status() == 0
    s.close()
    ro = R.residual(u, op, m, OP()).numpy()
    sc = summand_scale(u, op, m, np.arange(m.n_e), "split", OP(), dissipation=False).max(axis=2, keepdims=True)
    inner = np.setdiff1d(np.arange(op.n_p), op.facet_nodes.reshape(-1))
    assert np.all((np.abs(r - ro) <= ROUNDING_C * EPS * sc)[:, :, inner])


@pytest.mark.parametrize("d,p", [(2, 3), (3, 3)])
def test_non_finite_column_stays_visible(d, p):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2305_07181_gb300 as es
    op, m = _mesh(d, p)
    u = _state("ordinary", m, d, op.n_p)
    u[1, -1, 0] = np.nan
    s = es.Solver(op, m, es.Params())
    r = s.residual(s.to_device(u)).cpu().numpy()
    assert s.status() == -4
    s.close()
    assert not np.isfinite(r[1]).any()          # every node of the element takes part in its contractions
    assert np.isfinite(r[0, :, op.n_p - 1]).all()

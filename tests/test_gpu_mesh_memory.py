"""Device memory of a mesh: the arrays that the kernels of its operator read, no
packed tensor-core operators for the 7-node triangles, whose kernels contract
in float64 loops."""
import pytest
import torch

from esplit_inputs import tri_operator, periodic_tri_mesh

pytestmark = pytest.mark.gpu


def test_seven_node_triangles():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2305_07181_gb300 as es
    op = tri_operator(1)
    es.Solver(op, periodic_tri_mesh(op, 2, 10.0, 0.05)).close()   # the library's own set-up
    m = periodic_tri_mesh(op, 256, 10.0, 0.05)
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    s = es.Solver(op, m)
    torch.cuda.synchronize()
    used = before - torch.cuda.mem_get_info()[0]
    s.close()
    d, n_p, n_s, n_c = 2, 7, 6, 4
    f64 = n_p + n_s * d + d * d * n_p + d * n_p * n_p + n_c * n_s + (d + 9) * n_s + n_p + n_s * (d + 1) \
        + 8 + 8 * n_p / 256     # J, nu, Lambda, D_i, facet scratch, facet cache, 1/(H J), |nu| and nu/|nu|, partial sums
    f32 = d * n_p * n_p + d * n_p * 12 + n_p   # D_i, its padded copy for the float32 path, 1/(H J)
    i32 = n_s * 2 + n_s
    assert used <= 1.08 * m.n_e * (8 * f64 + 4 * f32 + 4 * i32)

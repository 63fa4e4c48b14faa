"""Mixed solves of one column on both sides of the lattice sizes at which they change from the red-black to the
whole-lattice cycles: the FP64 residual of the solution meets the tolerance, from a zero and from a poor start vector, and
the workspace is the one the header gives for each side."""
import ctypes

import pytest

pytestmark = pytest.mark.gpu


def _al(n):
    return (n + 255) // 256 * 256


@pytest.mark.parametrize("graph", [True, False])
@pytest.mark.parametrize("solver,dims,redblack", [("mixed_bf16", (16, 16, 16, 14), True),
                                                  ("mixed_bf16", (16, 16, 16, 16), False),
                                                  ("mixed_f16", (24, 16, 32, 30), True),
                                                  ("mixed_f16", (24, 16, 32, 32), False),
                                                  ("mixed_f32", (32, 32, 32, 30), True),
                                                  ("mixed_f32", (32, 32, 32, 32), False)])
def test_one_column_on_both_sides_of_the_rule(solver, dims, redblack, graph):
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_1603_05988_gb300 import dtr
    lat, m0 = dtr.make_lattice(dims), -0.75
    g = dtr.make_gauge(lat, 0.8, 5)
    p = dtr.solve_params(tol=1e-10, solver=solver, graph=graph)
    z = dtr.gen_noise(lat, 9, 0, 1, False, 0, 1)
    for y0 in (None, 3.0 * dtr.gen_noise(lat, 9, 1, 1, False, 0, 1)):
        y, _ = dtr.solve_batch(g, m0, z, y0=y0, params=p)
        assert float((z - dtr.dslash(g, m0, y)).norm() / z.norm()) <= 1.001e-10
    p2 = dtr.solve_params(solver="f64")
    vec64, vec32, half = _al(12 * lat.V * 16), _al(12 * lat.V * 8), _al(lat.V // 2 * 12 * 2 * 8)
    fixed = dtr._lib.dtr_solve_workspace_bytes(lat._h, 1, ctypes.byref(p2)) - 6 * vec64
    assert dtr._lib.dtr_solve_workspace_bytes(lat._h, 1, ctypes.byref(p)) == fixed + (12 * half if redblack
                                                                                      else vec64 + 7 * vec32)

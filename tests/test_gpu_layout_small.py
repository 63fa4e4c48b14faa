"""Layout conversions at the stencils' boundary on both sides of the size at which they change kernels (2^18 values), with
padded columns and partial groups: the stencil of a block equals, bit for bit, the stencil of its columns one by one."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["f64", "f32", "df32", "bf16", "f16"])
@pytest.mark.parametrize("dims,nrhs", [((2, 2, 2, 2), 3), ((8, 8, 8, 8), 3), ((8, 8, 8, 8), 5), ((6, 6, 6, 10), 9),
                                       ((6, 6, 6, 10), 11), ((4, 4, 4, 4), 64)])
def test_block_equals_columns(dims, nrhs, prec):
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_1603_05988_gb300 import dtr
    lat = dtr.make_lattice(dims)
    gauge = dtr.make_gauge(lat, 0.5, 7)
    rng = np.random.default_rng(nrhs)
    x = torch.from_numpy(rng.standard_normal((nrhs, lat.N)) + 1j * rng.standard_normal((nrhs, lat.N))).cuda()
    y = dtr.dslash(gauge, -0.4, x, prec=prec)
    for j in range(nrhs):
        assert torch.equal(y[j], dtr.dslash(gauge, -0.4, x[j:j + 1].contiguous(), prec=prec)[0])

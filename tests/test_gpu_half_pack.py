"""Packing of FP64 fields into half storage, at full and partial groups of 32 (site, column) items: the stencil of a field
equals, bit for bit, the stencil of that field already rounded (to FP32 and then to the storage type, as packing does)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["bf16", "f16"])
@pytest.mark.parametrize("dims,nrhs", [((2, 2, 2, 2), 1), ((2, 2, 2, 2), 3), ((4, 2, 6, 2), 5), ((8, 8, 8, 8), 1)])
def test_half_pack_rounds_once(dims, nrhs, prec):
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_1603_05988_gb300 import dtr
    lat = dtr.make_lattice(dims)
    gauge = dtr.make_gauge(lat, 0.5, 7)
    rng = np.random.default_rng(nrhs)
    x = torch.from_numpy(rng.standard_normal((nrhs, lat.N)) + 1j * rng.standard_normal((nrhs, lat.N))).cuda()
    half = {"bf16": torch.bfloat16, "f16": torch.float16}[prec]
    rounded = torch.view_as_complex(torch.view_as_real(x).to(torch.float32).to(half).to(torch.float64).contiguous())
    assert not torch.equal(x, rounded)
    y = dtr.dslash(gauge, -0.4, x, prec=prec)
    assert bool(torch.isfinite(torch.view_as_real(y)).all()) and float(torch.view_as_real(y).abs().max()) > 0
    assert torch.equal(y, dtr.dslash(gauge, -0.4, rounded, prec=prec))

"""The conversions between user and internal fields: block remainders, batches, and buffers of doubles that are
8-byte but not 16-byte aligned."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import oracle
import paper_1206_5214_gb300 as mdwf
import synthetic as sy
from _gpu import Ctx, rel_err

pytestmark = pytest.mark.gpu
F64, F32, F16N = mdwf.MDWF_F64, mdwf.MDWF_F32, mdwf.MDWF_F16N
SHAPES = [((2, 2, 2, 2), 2), ((2, 2, 2, 2), 32), ((6, 2, 2, 4), 10), ((4, 6, 2, 4), 16)]


def doubles(n, offset):
    """n doubles on the device, `offset` doubles behind a 256-byte boundary."""
    return torch.empty(n + offset, dtype=torch.float64, device="cuda")[offset:]


@pytest.mark.parametrize("offset", [0, 1])
@pytest.mark.parametrize("nrhs", [1, 3])
@pytest.mark.parametrize("dims,Ls", SHAPES)
def test_odd_fields(dims, Ls, nrhs, offset):
    """FP64 comes back bit for bit, FP32 rounded once, FP16+norm within 2^-11 of each site's largest component."""
    with Ctx(dims, Ls, 1.8, 1.5, 0.5, 0.02, sy.unit_gauge(dims)) as c:
        n = nrhs * Ls * c.Vh * 24
        src = doubles(n, offset)
        src.copy_(torch.from_numpy(np.random.default_rng(7).standard_normal(n)))
        for prec in (F64, F32, F16N):
            buf, back = c.alloc(prec, nrhs), doubles(n, offset)
            mdwf.mdwf_field_import(c.h, buf, src, prec, nrhs)
            mdwf.mdwf_field_export(c.h, back, buf, prec, nrhs)
            torch.cuda.synchronize()
            if prec == F64:
                assert torch.equal(back, src)
            elif prec == F32:
                assert torch.equal(back, src.float().double())
            else:
                a, b = src.reshape(-1, 24), back.reshape(-1, 24)
                assert ((a - b).abs().amax(1) <= 2.0 ** -11 * a.abs().amax(1) * 1.001).all()


@pytest.mark.parametrize("dims,Ls", SHAPES[2:])
def test_full_fields_unaligned(dims, Ls):
    """D_DW on full fields gives the same bits from and into unaligned buffers (split and join of both parities)."""
    x, y, z, t = dims
    n = 2 * Ls * x * y * z * t * 24
    vals = torch.from_numpy(np.random.default_rng(8).standard_normal(n))
    with Ctx(dims, Ls, 1.8, 1.5, 0.5, 0.02, sy.gauge_field(dims, 0.3, 1501)) as c:
        outs = []
        for offset in (0, 1):
            src, out = doubles(n, offset), doubles(n, offset)
            src.copy_(vals)
            mdwf.mdwf_apply_full(c.h, out, src, 2)
            torch.cuda.synchronize()
            outs.append(out)
        assert torch.equal(*outs)


@pytest.mark.parametrize("offset", [0, 1])
@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (2, 2, 2, 6), (6, 4, 2, 4), (4, 2, 6, 10)])
def test_links(dims, offset):
    """Links loaded from aligned and unaligned buffers, with whole and partial blocks of sites: M in every precision
    against the oracle (each precision reads a copy of its own)."""
    U = sy.gauge_field(dims, 0.5, 1502)
    buf = doubles(U.size * 2, offset)
    buf.copy_(torch.from_numpy(U.reshape(-1).view(np.float64)))
    odd = oracle.split(sy.gaussian_field(dims, 4, 2502), dims)[1]
    ref = oracle.m(odd, U, oracle.Params(dims, 4, 1.8, 1.5, 0.5, 0.02))
    with Ctx(dims, 4, 1.8, 1.5, 0.5, 0.02, sy.unit_gauge(dims)) as c:
        mdwf.mdwf_load_gauge(c.h, buf)
        for prec, tol in ((F64, 1e-12), (F32, 1e-5), (F16N, 1e-2)):
            assert rel_err(c.apply(odd, prec)[0], ref)[0] <= tol

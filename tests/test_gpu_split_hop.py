"""The hop kernels with four or two threads per column (small lattices) against the ordinary block shape, which a tuned
shape selects: the same bits in M, M^dag and the fused CG iterations."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import oracle
import paper_1206_5214_gb300 as mdwf
import synthetic as sy
from _gpu import Ctx

pytestmark = pytest.mark.gpu
F64, F32 = mdwf.MDWF_F64, mdwf.MDWF_F32
# the smallest field, columns that fill a warp, leave it ragged (10, 20, 24), exceed half of it, an odd last block
SHAPES = [((2, 2, 2, 2), 2), ((4, 2, 2, 2), 8), ((6, 2, 2, 4), 10), ((4, 4, 2, 4), 16), ((2, 2, 2, 6), 16),
          ((4, 2, 2, 4), 20), ((2, 4, 2, 4), 24), ((4, 2, 2, 2), 32),
          # FP64 with two threads: 65 to 228 ordinary blocks
          ((8, 8, 4, 8), 10), ((4, 4, 6, 8), 24), ((4, 4, 4, 10), 32), ((8, 8, 8, 4), 16)]


@pytest.mark.parametrize("dense", [False, True])
@pytest.mark.parametrize("prec", [F64, F32])
@pytest.mark.parametrize("dims,Ls", SHAPES)
def test_apply_same_bits(dims, Ls, prec, dense):
    U = sy.gauge_field(dims, 0.4, 1601)
    odd = np.stack([oracle.split(sy.gaussian_field(dims, Ls, 2601 + r), dims)[1] for r in range(2)])
    with Ctx(dims, Ls, 1.8, 1.5, 0.5, 0.03, U, dense_s=dense) as c:
        for dagger in (False, True):
            for mu in (0.0, 0.3, -1.7):  # the time terms take a factor of their own
                mdwf.mdwf_set_chemical_potential(c.h, mu)
                split = c.apply(odd, prec, dagger, 2, [0.01, 0.2])
                mdwf.mdwf_set_tuning(c.h, prec, 2, 128 // Ls)
                plain = c.apply(odd, prec, dagger, 2, [0.01, 0.2])
                mdwf.mdwf_set_tuning(c.h, prec, 2, 0)
                assert np.array_equal(split, plain), mu


@pytest.mark.parametrize("prec", [F64, F32])
@pytest.mark.parametrize("dims,Ls", [((4, 4, 2, 4), 16), ((6, 2, 2, 4), 10), ((4, 2, 2, 4), 20), ((4, 4, 6, 8), 24)])
def test_iterations_agree(dims, Ls, prec):
    """Eight iterations of the fused CG: the vectors follow the same arithmetic, but the partial sums of the CG
    scalars are grouped by block, so their last bits may differ (FP32 within a warp)."""
    U = sy.gauge_field(dims, 0.4, 1602)
    b = torch.from_numpy(sy.gaussian_field(dims, Ls, 2602)).cuda()
    with Ctx(dims, Ls, 1.8, 1.5, 0.5, 0.03, U) as c:
        xs = []
        for sites in (0, 128 // Ls):
            mdwf.mdwf_set_tuning(c.h, prec, 1, sites)
            x = torch.empty_like(b)
            mdwf.mdwf_cgne(c.h, x, b, maxiter=8, inner_prec=prec, raise_on_error=False)
            xs.append(x)
        rel = float((xs[0] - xs[1]).norm() / xs[1].norm())
    assert rel <= (1e-11 if prec == F64 else 1e-5), rel


@pytest.mark.parametrize("prec,dims,Ls,threads", [(F32, (4, 4, 4, 4), 8, 4), (F64, (4, 4, 4, 4), 8, 4),
                                                  (F64, (6, 10, 4, 14), 10, 2)])
def test_autotuner_finds_the_split_form(prec, dims, Ls, threads):
    """The default form is one of the tuner's candidates, and the fastest on small lattices: by 13.5 against 16.4 us in
    FP32 and 31 against 47 and 45 against 54 in FP64. Its number of sites per block selects it again."""
    U = sy.gauge_field(dims, 0.4, 1603)
    odd = oracle.split(sy.gaussian_field(dims, Ls, 2603), dims)[1]
    sites = 128 // threads // Ls
    with Ctx(dims, Ls, 1.8, 1.5, 0.5, 0.03, U) as c:
        assert mdwf.mdwf_get_tuning(c.h, prec, 1) == sites
        before = c.apply(odd, prec)
        assert mdwf.mdwf_autotune(c.h, prec, 1) == sites
        assert mdwf.mdwf_get_tuning(c.h, prec, 1) == sites
        assert np.array_equal(c.apply(odd, prec), before)
        mdwf.mdwf_set_tuning(c.h, prec, 1, 128 // Ls)
        assert mdwf.mdwf_get_tuning(c.h, prec, 1) == 128 // Ls

"""Coefficients with b5 zero or small beside c5, for which M_phi and K keep their factor (the others fold b5 into a
later coefficient): M, M^dag, the full operator and a mixed solve against the oracle."""
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
# all with |M-/M+| <= 1: the oracle's elimination amplifies rounding by |M-/M+|^Ls, 5.6^16 = 1e12 for (-0.5, 0.2)
COEF = [(0.0, 0.5), (1e-300, 0.5), (4e-4, 0.5), (6e-4, 0.5), (-1.5, 0.5), (0.0, 0.0)]
TOL = {mdwf.MDWF_F64: 1e-12, mdwf.MDWF_F32: 1e-5}


@pytest.mark.parametrize("b5,c5", COEF)
@pytest.mark.parametrize("dims,Ls", [((4, 4, 2, 4), 16), ((4, 2, 2, 4), 8), ((2, 4, 2, 4), 6)])
def test_operator(dims, Ls, b5, c5):
    U = sy.gauge_field(dims, 0.3, 1701)
    psi = sy.gaussian_field(dims, Ls, 2701)
    odd = oracle.split(psi, dims)[1]
    p = oracle.Params(dims, Ls, 1.8, b5, c5, 0.05)
    with Ctx(dims, Ls, 1.8, b5, c5, 0.05, U) as c:
        for dagger in (False, True):
            ref = oracle.m(odd, U, p, dagger=dagger)
            for prec, tol in TOL.items():
                assert rel_err(c.apply(odd, prec, dagger)[0], ref)[0] <= tol
            out = torch.empty(psi.shape, dtype=torch.complex128, device="cuda")
            mdwf.mdwf_apply_full(c.h, out, torch.from_numpy(psi).cuda(), dagger=dagger)
            assert rel_err(out.cpu().numpy(), oracle.ddw(psi, U, p, dagger=dagger))[0] <= 1e-12


@pytest.mark.parametrize("b5,c5", [(0.0, 0.5), (4e-4, 0.5)])
@pytest.mark.parametrize("Ls", [16, 8])
def test_mixed_solve(Ls, b5, c5):
    dims = (4, 4, 2, 4)
    U = sy.gauge_field(dims, 0.3, 1702)
    b = sy.gaussian_field(dims, Ls, 2702)
    p = oracle.Params(dims, Ls, 1.8, b5, c5, 0.05)
    with Ctx(dims, Ls, 1.8, b5, c5, 0.05, U) as c:
        x = torch.zeros(b.shape, dtype=torch.complex128, device="cuda")
        _, info = mdwf.mdwf_cgne(c.h, x, torch.from_numpy(b).cuda(), inner_prec=mdwf.MDWF_F32, tol=1e-10)
    assert info[0].true_res <= 1e-10
    xs = x.cpu().numpy()
    bp = oracle.prepare(b, U, p)
    src = oracle.m(bp, U, p, dagger=True)
    xo = oracle.split(xs, dims)[1]
    assert np.linalg.norm(src - oracle.mdagm(xo, U, p)) <= 1.05e-10 * np.linalg.norm(src)

"""The FP64 operator's fixed-point hops (csrc/fx.cuh) where their format could go wrong: shared exponents far
apart between neighbours and links, the ends of the FP64 range, zeros, non-finite values, the time factors."""
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
F64 = mdwf.MDWF_F64
DIMS, LS = (4, 6, 2, 4), 6


def setup(seed=1):
    U = sy.gauge_field(DIMS, 0.7, 1400 + seed)
    odd = oracle.split(sy.gaussian_field(DIMS, LS, 2400 + seed), DIMS)[1]
    return U, odd, oracle.Params(DIMS, LS, 1.8, 1.5, 0.5, 0.02)


@pytest.mark.parametrize("dagger", [False, True])
@pytest.mark.parametrize("what", ["sites", "slices", "links"])
def test_exponents_far_apart(what, dagger):
    """Magnitudes spread over many decades between sites, slices or links. The result is within 1e-12 of the
    largest element as everywhere, and each site within 1e-12 of the largest input that reaches it in M: for
    "sites" that is the largest of its two-hop neighbourhood, so the bound is checked on the whole field only."""
    U, odd, p = setup()
    rng = np.random.default_rng(5)
    if what == "sites":
        odd = odd * np.exp(8 * rng.standard_normal(odd.shape[1]))[None, :, None, None]
    elif what == "slices":
        odd = odd * np.exp(-3.0 * np.arange(LS))[:, None, None, None]
    else:
        U = U * np.exp(2 * rng.standard_normal(U.shape[:-2]))[..., None, None]
    with Ctx(DIMS, LS, 1.8, 1.5, 0.5, 0.02, U) as c:
        emax, el2 = rel_err(c.apply(odd, F64, dagger)[0], oracle.m(odd, U, p, dagger=dagger))
    assert emax <= 1e-12 and el2 <= 1e-12, (emax, el2)


@pytest.mark.parametrize("k", [-950, -700, 700, 950])
def test_powers_of_two_commute(k):
    """M(2^k psi) = 2^k M psi to the last bit while nothing under- or overflows: the exponents carry the scale."""
    U, odd, _ = setup(2)
    with Ctx(DIMS, LS, 1.8, 1.5, 0.5, 0.02, U) as c:
        one = c.apply(odd, F64)[0]
        two = c.apply(odd * 2.0 ** k, F64)[0]
    assert np.array_equal(two, one * 2.0 ** k)


@pytest.mark.parametrize("scale", [2.0 ** -1060, 2.0 ** 1010])
def test_ends_of_the_range(scale):
    """Subnormal fields keep the accuracy that subnormals have (2^-1074 a rounding, under 400 of them a site);
    large ones stay finite."""
    U, odd, p = setup(3)
    psi = odd * scale
    with Ctx(DIMS, LS, 1.8, 1.5, 0.5, 0.02, U) as c:
        got = c.apply(psi, F64)[0]
    ref = oracle.m(odd, U, p)
    assert np.isfinite(got).all()
    bound = 400 * 2.0 ** -1074 / scale + 1e-12 * np.abs(ref).max()
    # (numpy's complex division by a subnormal overflows: real by real)
    assert np.abs(got.view(np.float64) / scale - ref.view(np.float64)).max() <= bound


def test_zero_field_and_zero_links():
    U, odd, p = setup(4)
    with Ctx(DIMS, LS, 1.8, 1.5, 0.5, 0.02, U) as c:
        assert not c.apply(np.zeros_like(odd), F64)[0].any()
    U = U.copy()
    U[1] = 0
    with Ctx(DIMS, LS, 1.8, 1.5, 0.5, 0.02, U) as c:
        emax, _ = rel_err(c.apply(odd, F64)[0], oracle.m(odd, U, p))
    assert emax <= 1e-12


@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf])
@pytest.mark.parametrize("where", ["field", "link"])
def test_nonfinite_spreads_as_in_fp64(where, bad):
    """A non-finite entry makes the same sites non-finite as FP64 arithmetic (the oracle) does and leaves the
    others as they are without it."""
    dims = (8, 4, 4, 8)
    U = sy.gauge_field(dims, 0.3, 1405)
    odd = oracle.split(sy.gaussian_field(dims, LS, 2405), dims)[1]
    p = oracle.Params(dims, LS, 1.8, 1.5, 0.5, 0.02)
    with Ctx(dims, LS, 1.8, 1.5, 0.5, 0.02, U) as c:
        clean = c.apply(odd, F64)[0]
    if where == "field":
        odd = odd.copy()
        odd[2, 37, 1, 2] = bad
    else:
        U = U.copy()
        U[3, 1, 2, 5, 1, 0, 2] = bad
    with Ctx(dims, LS, 1.8, 1.5, 0.5, 0.02, U) as c:
        got = c.apply(odd, F64)[0]
    ref = oracle.m(odd, U, p)
    hit = ~np.isfinite(got).all(axis=(0, 2, 3))
    assert np.array_equal(hit, ~np.isfinite(ref).all(axis=(0, 2, 3)))
    assert hit.any() and not hit.all()
    assert np.array_equal(got[:, ~hit], clean[:, ~hit])


@pytest.mark.parametrize("mu", [-10.0, -0.3, 3.0, 10.0])
@pytest.mark.parametrize("dagger", [False, True])
def test_time_factors(mu, dagger):
    U, odd, _ = setup(6)
    p = oracle.Params(DIMS, LS, 1.8, 1.5, 0.5, 0.02, mu=mu)
    with Ctx(DIMS, LS, 1.8, 1.5, 0.5, 0.02, U) as c:
        mdwf.mdwf_set_chemical_potential(c.h, mu)
        emax, _ = rel_err(c.apply(odd, F64, dagger)[0], oracle.m(odd, U, p, dagger=dagger))
    assert emax <= 1e-12

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


# the FP64 kernels: four threads a column, two, and one (a tuned number of sites selects it)
FORMS = [((4, 6, 2, 4), 6, 0), ((8, 8, 4, 8), 10, 0), ((4, 6, 2, 4), 6, 21)]
forms = pytest.mark.parametrize("dims,Ls,sites", FORMS, ids=["four", "two", "one"])


def setup(dims, Ls, seed=1):
    U = sy.gauge_field(dims, 0.7, 1400 + seed)
    odd = oracle.split(sy.gaussian_field(dims, Ls, 2400 + seed), dims)[1]
    return U, odd, oracle.Params(dims, Ls, 1.8, 1.5, 0.5, 0.02)


def ctx(dims, Ls, sites, U):
    c = Ctx(dims, Ls, 1.8, 1.5, 0.5, 0.02, U)
    mdwf.mdwf_set_tuning(c.h, F64, 1, sites)
    return c


@forms
@pytest.mark.parametrize("dagger", [False, True])
def test_error_in_the_norm(dims, Ls, sites, dagger):
    """Gaussian fields: M is 1.2e-16 from long double, the oracle's FP64 1.6e-16: 2e-16 apart, and 4e-16 a bit more."""
    U, odd, p = setup(dims, Ls, 7)
    with ctx(dims, Ls, sites, U) as c:
        _, el2 = rel_err(c.apply(odd, F64, dagger)[0], oracle.m(odd, U, p, dagger=dagger))
    assert el2 <= 4e-16, el2


def largest_within_two_hops(odd, dims):
    """For each odd site the largest element of odd among the odd sites that reach it through M."""
    mask = oracle.parity_mask(dims)
    f = np.zeros(mask.shape)
    f[mask == 1] = np.abs(odd).max(axis=(0, 2, 3))
    for _ in range(2):
        f = np.max([f] + [np.roll(f, d, a) for a in range(4) for d in (1, -1)], axis=0)
    return f[mask == 1]


@forms
@pytest.mark.parametrize("dagger", [False, True])
@pytest.mark.parametrize("what", ["sites", "slices", "links"])
def test_exponents_far_apart(what, dims, Ls, sites, dagger):
    """Magnitudes spread over many decades between sites, slices or links: within 1e-12 of the largest element as
    everywhere, and (sites, slices) each site within 2e-13 of the largest input that reaches it. A hop adds 8 x 6
    products whose sizes sum to at most 28 times the largest neighbour, the s-operators at most double a column, so
    M's terms sum to 0.25 x 28 x 28 x 2 = 400 times the input, and each of the two hops rounds them about twice:
    1600 x 2^-53."""
    U, odd, p = setup(dims, Ls)
    rng = np.random.default_rng(5)
    if what == "sites":
        odd = odd * np.exp(8 * rng.standard_normal(odd.shape[1]))[None, :, None, None]
    elif what == "slices":
        odd = odd * np.exp(-3.0 * np.arange(Ls))[:, None, None, None]
    else:
        U = U * np.exp(2 * rng.standard_normal(U.shape[:-2]))[..., None, None]
    ref = oracle.m(odd, U, p, dagger=dagger)
    with ctx(dims, Ls, sites, U) as c:
        got = c.apply(odd, F64, dagger)[0]
    emax, el2 = rel_err(got, ref)
    assert emax <= 1e-12 and el2 <= 1e-12, (emax, el2)
    if what != "links":
        err = np.abs(got - ref).max(axis=(0, 2, 3))
        assert (err <= 2e-13 * largest_within_two_hops(odd, dims)).all()


@forms
@pytest.mark.parametrize("k", [-950, -700, 700, 950])
def test_powers_of_two_commute(k, dims, Ls, sites):
    """M(2^k psi) = 2^k M psi to the last bit while nothing under- or overflows: the exponents carry the scale."""
    U, odd, _ = setup(dims, Ls, 2)
    with ctx(dims, Ls, sites, U) as c:
        one = c.apply(odd, F64)[0]
        two = c.apply(odd * 2.0 ** k, F64)[0]
    assert np.array_equal(two, one * 2.0 ** k)


@forms
@pytest.mark.parametrize("scale", [2.0 ** -1060, 2.0 ** 1010])
def test_ends_of_the_range(scale, dims, Ls, sites):
    """Subnormal fields keep the accuracy that subnormals have (2^-1074 a rounding, under 400 of them a site);
    large ones stay finite."""
    U, odd, p = setup(dims, Ls, 3)
    psi = odd * scale
    with ctx(dims, Ls, sites, U) as c:
        got = c.apply(psi, F64)[0]
    ref = oracle.m(odd, U, p)
    assert np.isfinite(got).all()
    bound = 400 * 2.0 ** -1074 / scale + 1e-12 * np.abs(ref).max()
    # (numpy's complex division by a subnormal overflows: real by real)
    assert np.abs(got.view(np.float64) / scale - ref.view(np.float64)).max() <= bound


@forms
def test_zero_field_and_zero_links(dims, Ls, sites):
    U, odd, p = setup(dims, Ls, 4)
    with ctx(dims, Ls, sites, U) as c:
        assert not c.apply(np.zeros_like(odd), F64)[0].any()
    U = U.copy()
    U[1] = 0
    with ctx(dims, Ls, sites, U) as c:
        emax, _ = rel_err(c.apply(odd, F64)[0], oracle.m(odd, U, p))
    assert emax <= 1e-12


@pytest.mark.parametrize("dims,Ls,sites", [((8, 4, 4, 8), 6, 0), ((8, 8, 4, 8), 10, 0), ((8, 4, 4, 8), 6, 21)],
                         ids=["four", "two", "one"])
@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf])
@pytest.mark.parametrize("where", ["field", "link"])
def test_nonfinite_spreads_as_in_fp64(where, bad, dims, Ls, sites):
    """A non-finite entry makes the same sites non-finite as FP64 arithmetic (the oracle) does and leaves the
    others as they are without it."""
    U = sy.gauge_field(dims, 0.3, 1405)
    odd = oracle.split(sy.gaussian_field(dims, Ls, 2405), dims)[1]
    p = oracle.Params(dims, Ls, 1.8, 1.5, 0.5, 0.02)
    with ctx(dims, Ls, sites, U) as c:
        clean = c.apply(odd, F64)[0]
    if where == "field":
        odd = odd.copy()
        odd[2, 37, 1, 2] = bad
    else:
        U = U.copy()
        U[3, 1, 2, 5, 1, 0, 2] = bad
    with ctx(dims, Ls, sites, U) as c:
        got = c.apply(odd, F64)[0]
    ref = oracle.m(odd, U, p)
    hit = ~np.isfinite(got).all(axis=(0, 2, 3))
    assert np.array_equal(hit, ~np.isfinite(ref).all(axis=(0, 2, 3)))
    assert hit.any() and not hit.all()
    assert np.array_equal(got[:, ~hit], clean[:, ~hit])


@forms
@pytest.mark.parametrize("mu", [-10.0, -0.3, 3.0, 10.0])
@pytest.mark.parametrize("dagger", [False, True])
def test_time_factors(mu, dims, Ls, sites, dagger):
    U, odd, _ = setup(dims, Ls, 6)
    p = oracle.Params(dims, Ls, 1.8, 1.5, 0.5, 0.02, mu=mu)
    with ctx(dims, Ls, sites, U) as c:
        mdwf.mdwf_set_chemical_potential(c.h, mu)
        emax, _ = rel_err(c.apply(odd, F64, dagger)[0], oracle.m(odd, U, p, dagger=dagger))
    assert emax <= 1e-12


def far_apart(odd, k, part):
    """odd with its colours, or its spins, 1, 2^-k and 2^-2k (a fourth spin: zero) in size."""
    f = 2.0 ** (-k * np.arange(3.0))
    return odd * f if part == "colours" else odd * np.append(f, 0.0)[:, None]


def assert_each_part(got, ref, tol):
    """Every (spin, colour) component within tol of its own largest element of the field."""
    err = np.abs(got - ref).reshape(-1, 12).max(0)
    top = np.abs(ref).reshape(-1, 12).max(0)
    assert (err <= tol * top).all(), err / top


# FP64 arithmetic: about 200 roundings a component and hop, 2e-14 at worst. Fixed point, where it is taken: 1.5 units of
# the last place in the root mean square, six times that over the components of a field, against terms that add
# up to 2^(54 - 8) units (a part 2^-8 of the largest component) times a link entry of 0.57: 2.3e-13 at the edge.
PARTS_TOL = 3e-13


@pytest.mark.parametrize("dagger", [False, True])
@pytest.mark.parametrize("k", [1, 4, 7, 9, 20, 40])
@pytest.mark.parametrize("shape", [0, 1])
def test_colours_that_do_not_mix(shape, k, dagger):
    """Links diagonal in colour (free fields, Abelian backgrounds) never add one colour to another in M, so a small
    colour keeps its relative accuracy beside a large one."""
    dims, Ls = [(DIMS, LS), ((8, 8, 4, 8), 10)][shape]
    rng = np.random.default_rng(11)
    ph = rng.uniform(-np.pi, np.pi, (*dims[::-1], 4, 2))
    ph = np.concatenate([ph, -ph.sum(-1, keepdims=True)], -1)
    U = np.exp(1j * ph)[..., None] * np.eye(3)
    odd = far_apart(oracle.split(sy.gaussian_field(dims, Ls, 2411), dims)[1], k, "colours")
    p = oracle.Params(dims, Ls, 1.8, 1.5, 0.5, 0.02)
    ref = oracle.m(odd, U, p, dagger=dagger)
    with Ctx(dims, Ls, 1.8, 1.5, 0.5, 0.02, U) as c:
        for sites in (0, 128 // Ls):
            mdwf.mdwf_set_tuning(c.h, F64, 1, sites)
            assert_each_part(c.apply(odd, F64, dagger)[0], ref, PARTS_TOL)


@pytest.mark.parametrize("k", [7, 9, 20, 40])
def test_one_colour_a_site(k):
    """Each site holds one colour only, of a size of its own: the neighbours of a site differ in both."""
    rng = np.random.default_rng(12)
    U = np.broadcast_to(np.eye(3), (*DIMS[::-1], 4, 3, 3)).astype(complex)
    odd = far_apart(oracle.split(sy.gaussian_field(DIMS, LS, 2412), DIMS)[1], k, "colours")
    odd = odd * (rng.integers(0, 3, odd.shape[1])[:, None] == np.arange(3))[:, None, :]
    with Ctx(DIMS, LS, 1.8, 1.5, 0.5, 0.02, U) as c:
        got = c.apply(odd, F64)[0]
    assert_each_part(got, oracle.m(odd, U, oracle.Params(DIMS, LS, 1.8, 1.5, 0.5, 0.02)), PARTS_TOL)


@pytest.mark.parametrize("dagger", [False, True])
@pytest.mark.parametrize("k", [7, 9, 20, 40])
def test_spins_that_do_not_mix(k, dagger):
    """One hop adds to the upper spins only themselves and the lower ones: with the field on the even sites alone,
    D_DW on the odd sites is one hop, and its small upper spins keep their accuracy."""
    U = sy.gauge_field(DIMS, 0.7, 1413)
    psi = sy.gaussian_field(DIMS, LS, 2413)
    odd = oracle.split(psi, DIMS)[1]
    psi = oracle.join(far_apart(oracle.split(psi, DIMS)[0], k, "spins"), 0 * odd, DIMS)
    p = oracle.Params(DIMS, LS, 1.8, 1.5, 0.5, 0.02)
    ref = oracle.ddw(psi, U, p, dagger=dagger)
    out = torch.empty(psi.shape, dtype=torch.complex128, device="cuda")
    with Ctx(DIMS, LS, 1.8, 1.5, 0.5, 0.02, U) as c:
        mdwf.mdwf_apply_full(c.h, out, torch.from_numpy(psi).cuda(), dagger=dagger)
        torch.cuda.synchronize()
    got, ref = (oracle.split(f, DIMS)[1] for f in (out.cpu().numpy(), ref))
    assert_each_part(got, ref, PARTS_TOL)


@pytest.mark.parametrize("dagger", [False, True])
@pytest.mark.parametrize("k", [2, 7, 20, 40])
def test_links_with_small_rows(k, dagger):
    """Links that are not unitary, diagonal in colour with entries 1, 2^-k and 2^-2k."""
    U = np.broadcast_to(np.diag(2.0 ** (-k * np.arange(3.0))), (*DIMS[::-1], 4, 3, 3)).astype(complex)
    psi = sy.gaussian_field(DIMS, LS, 2414)
    psi = oracle.join(oracle.split(psi, DIMS)[0], 0 * oracle.split(psi, DIMS)[1], DIMS)
    p = oracle.Params(DIMS, LS, 1.8, 1.5, 0.5, 0.02)
    ref = oracle.ddw(psi, U, p, dagger=dagger)
    out = torch.empty(psi.shape, dtype=torch.complex128, device="cuda")
    with Ctx(DIMS, LS, 1.8, 1.5, 0.5, 0.02, U) as c:
        mdwf.mdwf_apply_full(c.h, out, torch.from_numpy(psi).cuda(), dagger=dagger)
        torch.cuda.synchronize()
    got, ref = (oracle.split(f, DIMS)[1] for f in (out.cpu().numpy(), ref))
    assert_each_part(got, ref, PARTS_TOL)


def test_links_without_a_fixed_point_copy():
    """With little device memory free the links are held without the fixed-point copy (228 instead of 372 B each),
    and the FP64 operator runs in FP64 arithmetic."""
    dims, Ls, nlink = (16, 16, 16, 16), 32, 4 * 16 ** 4
    field = dims[0] ** 4 // 2 * Ls * 192
    U = sy.gauge_field(dims, 0.3, 1415)
    odd = oracle.split(sy.gaussian_field(dims, Ls, 2415), dims)[1]
    outs, taken = [], []
    for short in (False, True):
        torch.cuda.empty_cache()
        with Ctx((4, 4, 2, 2), 4, 1.8, 1.5, 0.5, 0.02, sy.unit_gauge((4, 4, 2, 2))) as c:  # loads the kernels
            c.apply(np.zeros((4, 32, 4, 3), complex), F64)
        Ud = torch.from_numpy(U).cuda()
        h = mdwf.mdwf_create(dims, Ls, 1.8, 1.5, 0.5, 0.02)
        try:
            src, dst = (torch.empty(field, dtype=torch.uint8, device="cuda") for _ in range(2))
            mdwf.mdwf_field_import(h, src, torch.from_numpy(odd).cuda(), F64, 1)
            torch.cuda.synchronize()
            torch.cuda.empty_cache()
            free = torch.cuda.mem_get_info()[0]
            filler = torch.empty(free - 7 * field // 2, dtype=torch.uint8, device="cuda") if short else None
            free = torch.cuda.mem_get_info()[0]
            mdwf.mdwf_load_gauge(h, Ud)
            taken.append(free - torch.cuda.mem_get_info()[0])
            mdwf.mdwf_apply(h, dst, src, F64, 1)
            torch.cuda.synchronize()
            del filler
            torch.cuda.empty_cache()
            out = torch.empty((1, Ls, 8 * 16 ** 3, 4, 3), dtype=torch.complex128, device="cuda")
            mdwf.mdwf_field_export(h, out, dst, F64, 1)
            outs.append(out.cpu().numpy()[0])
        finally:
            mdwf.mdwf_destroy(h)
    page = 4 << 20   # the driver's granularity
    assert taken[0] > 372 * nlink - page and taken[1] < 228 * nlink + page, taken
    ref = oracle.m(odd, U, oracle.Params(dims, Ls, 1.8, 1.5, 0.5, 0.02))
    assert all(rel_err(o, ref)[0] <= 1e-12 for o in outs)

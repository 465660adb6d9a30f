"""The fixed-point solve of the FP64 plans (csrc/lens.cuh, solve_point_fixed and
factor_fixed; csrc/xi_table.cu's integer table) on the host, through the lens
kernel's whole per-tile path, against the same path in FP64 and the oracle: every
stencil size the host driver builds, spin 0, 1 and 2, from the smallest skies the
form accepts (r^2 just below 2^-5 for spin 1 and 2) to Nside 16384.

Tolerances: sums carry 2^-57 and the rounding of S is that of FP64, so the values
stay within the FP64 path's own parity tolerance of the oracle (1e-9 of the map's
rms), and within 1e-10 of the FP64 form on realisations of the field.  Maps that are
not realisations (white noise, 1e5 and 1e-200 in size) amplify both forms' rounding:
there the two agree to a few times the FP64 form's distance from the oracle."""
import numpy as np
import pytest

from oracle import kriging as kr
from oracle import xi
from tests import host_compile as hc
from tests import test_lens_host as T

FIXED = """    std::vector<CoefFx> cfx(n);
    for (int k = 0; k < n; ++k) {
        threadIdx.x = k;
        fixed_table_kernel(c64.data(), n, cfx.data());
    }
    a.tab.cfx = cfx.data();
    a.two_r = 2.0 * tg.r;
    a.inv_2r = 0.5 / tg.r;
    a.tabm = a.tab;"""


@pytest.fixture(scope="module")
def both(tmp_path_factory):
    if hc.compiler() is None:
        pytest.skip("no host C++ compiler")
    plain, saved = T._build(tmp_path_factory.mktemp("plain")), T.DRIVER
    try:
        T.DRIVER = saved.replace("    a.tabm = a.tab;", FIXED, 1)
        assert T.DRIVER != saved
        fixed = T._build(tmp_path_factory.mktemp("fixed"), sanitize="address")
    finally:
        T.DRIVER = saved
    return plain, fixed


CASES = [(0, 64, 16, 128, 100.0, 20_000), (0, 4, 16, 8, 5.0, 0), (0, 2048, 32, 4096, 2500.0, 25_000_000),
         (0, 16384, 32, 2048, 1250.0, 3_200_000_000), (1, 64, 32, 128, 80.0, 30_000), (1, 2048, 32, 2048, 1250.0, 40_000_000),
         (2, 32, 32, 64, 40.0, 3_000), (2, 32, 16, 64, 40.0, 0), (2, 64, 48, 128, 78.0, 20_000),
         (2, 1024, 48, 2048, 1250.0, 6_000_000), (2, 4096, 32, 4096, 2500.0, 8_390_000)]


@pytest.mark.parametrize("values", ["field", "white", "huge", "tiny"])
@pytest.mark.parametrize("case", CASES, ids=lambda c: f"spin{c[0]}-nside{c[1]}-K{c[2]}")
def test_fixed_point_against_fp64_and_the_oracle(case, values, both):
    spin, N, K, lmax, ld, first = case
    if values != "field" and case not in (CASES[2], CASES[6], CASES[9]):
        pytest.skip("one case per spin and stencil shape for maps that are not realisations")
    n = 16
    cl, bb, defl, pix, vals = T._inputs(spin, N, lmax, ld, first, n, seed=N + K + spin)
    if values != "field":
        vals = np.random.default_rng(N).normal(size=vals.shape) * {"white": 1.0, "huge": 1e150, "tiny": 1e-200}[values]
    t_max, m = xi.grid_rule(np.abs(cl), K, N)
    tab, x0 = (xi.spin0_table(cl, t_max, m) if spin == 0
               else (xi.spin1_tables if spin == 1 else xi.spin2_tables)(cl, bb, t_max, m)[::2])
    ref = kr.lens(N, K, spin, T._Band(pix, vals), defl, np.arange(first, first + n), tab, x0)
    (_, s0, v0, q0), (_, s1, v1, q1) = (r(spin, K, 0, N, cl, bb, first, defl, pix, vals) for r in both)
    assert np.array_equal(s0, s1) and not s1.any()
    scale = np.max(np.abs(ref.value))
    off, off0, apart = (np.max(np.abs(a - b)) / scale for a, b in ((v1, ref.value), (v0, ref.value), (v1, v0)))
    if values == "field":
        assert off <= 1e-9 and apart <= 1e-10
    else:
        assert apart <= 8 * off0 + 1e-12
    assert np.max(np.abs(q1 - ref.variance)) <= 1e-13 * x0 and not np.array_equal(v0, v1)


def test_a_value_that_is_not_finite_takes_the_fp64_form(both):
    spin, N, K, lmax, ld, first = CASES[6]
    cl, bb, defl, pix, vals = T._inputs(spin, N, lmax, ld, first, 8, seed=3)
    vals = vals.copy()
    vals[np.searchsorted(pix, first + 3)] = np.inf
    (x0, s0, v0, q0), (_, s1, v1, q1) = (r(spin, K, 0, N, cl, bb, first, defl, pix, vals) for r in both)
    bad = ~np.isfinite(v0)
    assert bad.any() and np.array_equal(bad, ~np.isfinite(v1)) and np.array_equal(s0, s1)
    assert np.max(np.abs(q0 - q1)) <= 1e-13 * x0  # as above

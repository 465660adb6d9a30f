"""Map data at the ends of the FP64 range in the fixed-point solve of the FP64 plans
(csrc/lens.cuh, solve_point_fixed), through the lens kernel's per-tile path on the
host: maps of zeros (a masked region) give zeros, exactly; maps of subnormal values
and maps whose largest values are near the smallest normal number give what the FP64
form gives, to the rounding of numbers of that size."""
import numpy as np
import pytest

from tests import test_fixed_point_host as F
from tests import test_lens_host as T

both = F.both
CASES = [F.CASES[k] for k in (0, 4, 7)]  # K = 16 at spin 0, spin 1, spin 2


@pytest.mark.parametrize("case", CASES, ids=lambda c: f"spin{c[0]}")
def test_zero_maps_give_zeros(case, both):
    spin, N, K, lmax, ld, first = case
    cl, bb, defl, pix, vals = T._inputs(spin, N, lmax, ld, first, 8, seed=3)
    x0, s, v, q = both[1](spin, K, 0, N, cl, bb, first, defl, pix, 0.0 * vals)
    assert np.all(v == 0) and not s.any()
    assert np.array_equal(q, both[1](spin, K, 0, N, cl, bb, first, defl, pix, vals)[3])


@pytest.mark.parametrize("size", [2.0 ** -1060, 2.0 ** -1022, 2.0 ** -1000, 2.0 ** -960])
@pytest.mark.parametrize("case", CASES, ids=lambda c: f"spin{c[0]}")
def test_tiny_values_are_kept(case, size, both):
    spin, N, K, lmax, ld, first = case
    cl, bb, defl, pix, vals = T._inputs(spin, N, lmax, ld, first, 8, seed=3)
    vals = vals * (size / np.max(np.abs(vals)))
    (_, s0, v0, q0), (x0, s1, v1, q1) = (r(spin, K, 0, N, cl, bb, first, defl, pix, vals) for r in both)
    assert np.array_equal(s0, s1) and np.max(np.abs(q0 - q1)) <= 1e-13 * x0
    # 1e-10 between the forms as on maps of ordinary size; below it subnormal results, whose
    # K products are each rounded to 2^-1074
    assert np.max(np.abs(v1 - v0)) <= 1e-10 * np.max(np.abs(v0)) + 2 * K * 5e-324

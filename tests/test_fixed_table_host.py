"""The integer correlation table of the fixed-point solves (csrc/xi_table.cu,
fixed_table_kernel) on the host: every coefficient is the nearest multiple of 2^-59,
over the sizes that fixed_table_ok admits and both signs."""
from fractions import Fraction

import numpy as np
import pytest

from tests import host_compile as hc
from tests import test_lens_host as T

DRIVER = r"""
using namespace flints;
int main() {
    Coef64 c;
    while (scanf("%la %la %la %la", &c.f, &c.m, &c.c2, &c.c3) == 4) {
        CoefFx x;
        fixed_table_kernel(&c, 1, &x);
        printf("%lld %lld %lld %lld\n", (long long)x.f, (long long)x.m, (long long)x.c2, (long long)x.c3);
    }
    return 0;
}
"""


def test_coefficients_are_rounded_to_the_nearest_unit(tmp_path):
    if hc.compiler() is None:
        pytest.skip("no host C++ compiler")
    text = (hc.LENS_SHIM + T.KERNEL_SHIM + "namespace flints {\n"
            + hc.cut("common.cuh", "constexpr unsigned FULL", "// Host-side launchers (lens_spin0.cu", False)
            + hc.cut("xi_table.cu", "__global__ void fixed_table_kernel", "cudaError_t launch_xi_table(", False)
            + "\n}\n" + DRIVER)
    exe = hc.build(tmp_path, "table", text, warp="threads")
    rng = np.random.default_rng(5)
    c = rng.normal(size=(500, 4)) * 2.0 ** rng.uniform(-70, 0, (500, 4))
    c = np.concatenate([np.clip(c, -1.99, 1.99), [[0.0, 1.0, -1.0, 1.0 + 2.0 ** -52], [2.0 ** -60, -2.0 ** -60, 1.5 * 2.0 ** -59, 5e-324]]])
    out = hc.run(exe, "\n".join(" ".join(float(v).hex() for v in r) for r in c) + "\n").split()
    for v, k in zip(c.ravel(), map(int, out), strict=True):
        assert abs(Fraction(float(v)) * 2 ** 59 - k) <= Fraction(1, 2), (v, k)

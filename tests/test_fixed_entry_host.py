"""Entries of L^-1 as the fixed-point apply kernel loads them (csrc/paper.cu, fx_entry) on
the host: within one unit of 2^(e - 57) of the entry, either sign and conjugated, and
exactly 0 for zeros (pads and entries past the diagonal)."""
from fractions import Fraction

import numpy as np
import pytest

from tests import host_compile as hc
from tests import test_lens_host as T

DRIVER = r"""
using namespace flints;
int main() {
    double v;
    int e, flip;
    while (scanf("%la %d %d", &v, &e, &flip) == 3) printf("%lld\n", (long long)fx_val(fx_entry(v, e, flip ? 0x80000000u : 0u)));
    return 0;
}
"""


def test_entries(tmp_path):
    if hc.compiler() is None:
        pytest.skip("no host C++ compiler")
    text = (hc.LENS_SHIM + T.KERNEL_SHIM + "namespace flints {\n"
            + hc.cut("common.cuh", "constexpr unsigned FULL", "// Host-side launchers (lens_spin0.cu", False)
            + hc.cut("paper.cu", "__device__ __forceinline__ fx fx_entry(", "// Sum of products of L^-1 entries", False)
            + "\n}\n" + DRIVER)
    exe = hc.build(tmp_path, "entry", text, warp="threads")
    rng = np.random.default_rng(6)
    rows = [(s * 0.0, e, f) for s in (1.0, -1.0) for e in (-6, 0, 16) for f in (0, 1)]
    for e in (-6, 0, 9, 16):
        for v in np.concatenate([rng.uniform(0.5, 1, 50) * 2.0 ** rng.integers(-70, 1, 50), [2.0 ** -1, 1 - 2.0 ** -53]]):
            rows += [(s * v * 2.0 ** e, e, f) for s in (1, -1) for f in (0, 1)]
    out = hc.run(exe, "\n".join(f"{float(v).hex()} {e} {f}" for v, e, f in rows) + "\n").split()
    for (v, e, f), k in zip(rows, map(int, out), strict=True):
        x = Fraction(v) * (-1 if f else 1) / Fraction(2) ** (e - 57)
        assert k == 0 if v == 0 else abs(k - x) <= 1, (v, e, f, k)

"""The recurrence tables of a mixed synthesis plan (csrc/synth.cu, synth_order_kernel and
synth_coef_kernel) on the host, for stretches of one and of several pairs per thread and
chains of every remainder: with alpha_l from the table of alpha_l N_l, one step of the
recurrence has C_l alpha_{l-1} / alpha_{l+1} = 1, a_l and b_l are the FP64 coefficients
times alpha_l / alpha_{l+1}, and alpha is 1 at the two largest l.  Tolerances: a few FP64
roundings (alpha_l: one product and two factors per step of a chain, 16 where a stretch
meets the next), the integers' half units (2^-55 for a, 2^-60 for b) besides."""
import numpy as np
import pytest

from tests import cuda_host as ch
from tests import host_compile as hc

DRIVER = r"""
int main() {
    int lmax, spin;
    while (scanf("%d %d", &lmax, &spin) == 2) {
        flints_synth_t h = nullptr;
        if (flints_synth_plan(&h, 1, lmax, spin, 1, nullptr)) return 3;
        for (int m = 0; m <= lmax; ++m)
            for (int l = m > spin ? m : spin; l <= lmax; ++l) {
                const SynthStep &c = h->d_steps[tri_row(lmax, m) + l];
                printf("%lld %lld %a\n", (long long)flints::fx_val(c.a), c.b, h->d_na[tri_row(lmax, m) + l]);
            }
        flints_synth_free(h);
    }
    return 0;
}
"""


@pytest.mark.parametrize("spin", [0, 1, 2])
def test_tables(spin, tmp_path):
    if hc.compiler() is None:
        pytest.skip("no host C++ compiler")
    if np.finfo(np.longdouble).eps > 2.0 ** -60:
        pytest.skip("no extended long double")
    L, eps = np.longdouble, 2.0 ** -53
    exe = ch.build(tmp_path, "coef", ["common.cuh", "synth.cu"], DRIVER)
    sizes = [spin, spin + 1, spin + 2, spin + 3, 40, 530 + spin]
    rows = iter(hc.run(exe, " ".join(f"{n} {spin}" for n in sizes) + "\n").splitlines())
    for lmax in sizes:
        for m in range(lmax + 1):
            l0 = max(m, spin)
            t = [next(rows).split() for _ in range(l0, lmax + 1)]
            a, b = (np.array([int(r[k]) for r in t], dtype=L) / L(2) ** e for k, e in ((0, 54), (1, 59)))
            l = np.arange(l0, lmax + 1, dtype=L)
            alpha = np.array([float.fromhex(r[2]) for r in t], dtype=L) / np.sqrt((2 * l + 1) / (4 * L(np.pi)))
            assert np.all(np.abs(alpha[-2:] - 1) <= 4 * eps)
            q = np.sqrt((l * l - m * m) * (l * l - spin * spin)) / np.maximum(l, 1)  # q_l; C_l = q_l / q_{l+1}
            if len(l) > 2:
                c = q[1:-1] / q[2:] * alpha[:-2] / alpha[2:]
                assert np.max(np.abs(c - 1)) <= 16 * eps, (lmax, m)
            if len(l) > 1:
                r = (2 * l[:-1] + 1) / q[1:] * alpha[:-1] / alpha[1:]
                assert np.max(np.abs(a[:-1] - r) / r) <= 16 * eps and np.all(a[:-1] < 256)
                rb = r * m * spin / np.maximum(l[:-1] * (l[:-1] + 1), 1)
                assert np.max(np.abs(b[:-1] - rb)) <= 2.0 ** -60 + 16 * eps * np.max(rb)

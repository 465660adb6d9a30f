"""The fixed-point apply kernel of the tabulated route (csrc/paper.cu, apply_kernel_fx)
on the host, through the C API, against the FP64 kernel of the same plan.

Rows of L^-1 that no positive covariance has (a class's entries scaled up after the plan
is made; spectra with negative multipoles are accepted, so plans can hold such rows) give
what the FP64 kernel gives.  Tolerance: the two forms hold c to 2^-54 and 2^-58, and sums
of 36 products of rows up to 2^14 in size, each rounded at 2^-53, agree to 36 2^-39 of the
largest; values and variances are compared at 1e-9 of their largest."""
import numpy as np
import pytest

import workloads as wl
from oracle import healpix as hp
from oracle import sht
from tests import cuda_host as ch
from tests import host_compile as hc

DRIVER = r"""
namespace flints {
int device_sm_count() { return 152; }
size_t device_smem_optin() { return 232448; }
}
static double rd() { char b[64]; if (scanf("%63s", b) != 1) exit(2); return strtod(b, nullptr); }
// row `row` of every class's L^-1 times 2^k, and its exponent as the plan's kernel forms it
static void scale_row(flints_paper_t p, int row, int k) {
    const int comp = p->spin == 0 ? 1 : 2;
    for (int64_t sl = 0; sl < p->nslot; ++sl) {
        double *blk = p->d_linv + sl * flints::paper::linv_len(36) * comp;
        int ex = 0;
        for (int col = 0; col <= row; ++col)
            for (int c = 0; c < comp; ++c) {
                double &v = blk[flints::paper::lanestep_index(row, col) * comp + c];
                v = std::ldexp(v, k);
                ex = std::max(ex, flints::paper::expo_of(v));
            }
        p->d_row_exp[sl * 36 + row] = flints::paper::row_exponent(ex);
    }
}
int main() {
    long long nside, first, count;
    int lmax, spin, row, k;
    while (scanf("%lld %d %d %lld %lld %d %d", &nside, &lmax, &spin, &first, &count, &row, &k) == 7) {
        const int comp = spin == 0 ? 1 : 2;
        const long long npix = 12 * nside * nside;
        std::vector<double> cl(lmax + 1), map(npix * comp), defl(2 * count);
        for (double &v : cl) v = rd();
        for (double &v : map) v = rd();
        for (double &v : defl) v = rd();
        flints_paper_t h = nullptr;
        if (flints_paper_plan(&h, nside, lmax, cl.data(), nullptr, 2, spin, 0, 0, nullptr) || !h->fixed) return 3;
        if (k) scale_row(h, row, k);
        for (int form = 0; form < 2; ++form) {  // the FP64 kernel, the fixed-point kernel
            h->fixed = form == 1;
            std::vector<double> out(count * comp), var(count);
            std::vector<uint8_t> st(count);
            if (flints_paper_lens(h, first, count, map.data(), defl.data(), out.data(), var.data(), st.data(), nullptr)) return 4;
            for (long long p = 0; p < count; ++p)
                printf("%d %a %a %a\n", (int)st[p], out[p * comp], comp == 2 ? out[2 * p + 1] : 0.0, var[p]);
        }
        flints_paper_free(h);
    }
    return 0;
}
"""


@pytest.fixture(scope="module")
def call(tmp_path_factory):
    """(status, values, variances) of the FP64 and of the fixed-point kernel."""
    if hc.compiler() is None:
        pytest.skip("no host C++ compiler")
    exe = ch.build(tmp_path_factory.mktemp("paper_fx"), "paper_fx", ["common.cuh", "lens.cuh", "paper_geom.cuh", "xi_table.cu", "paper.cu"],
                   DRIVER, sanitize="address")

    def run(nside, spin, cl, m, first, defl, row=0, k=0):
        vals = np.concatenate([cl, np.ravel(m), np.ravel(defl)])
        line = f"{nside} {cl.size - 1} {spin} {first} {len(defl)} {row} {k} " + " ".join(float(x).hex() for x in vals)
        o = np.array([[float.fromhex(t) for t in ln.split()] for ln in hc.run(exe, line + "\n").splitlines()])
        o = o.reshape(2, len(defl), 4)
        return [(r[:, 0].astype(int), r[:, 1] + 1j * r[:, 2], r[:, 3]) for r in o]

    return run


def _inputs(spin, nside, n):
    lmax = 2 * nside
    cl = wl.cl_tt(lmax, 0.7 * lmax)
    m = sht.synth_map(nside, lmax, wl.draw_alm(cl, 41))
    npix = hp.npix(nside)
    return cl, m, wl.random_deflection(n, 42, rms=0.5 * np.sqrt(4 * np.pi / npix))


def _agree(a, b, tol):
    (s0, v0, q0), (s1, v1, q1) = a, b
    assert np.array_equal(s0, s1)
    assert np.max(np.abs(v1 - v0)) <= tol * np.max(np.abs(v0)), np.max(np.abs(v1 - v0)) / np.max(np.abs(v0))
    assert np.max(np.abs(q1 - q0)) <= tol * np.max(np.abs(q0)), np.max(np.abs(q1 - q0)) / np.max(np.abs(q0))


@pytest.mark.parametrize("row", [0, 20, 35])
@pytest.mark.parametrize("k", [30, 400])
def test_rows_beyond_the_kernels_range_take_the_fp64_form(row, k, call):
    cl, m, defl = _inputs(0, 16, 40)
    _agree(*call(16, 0, cl, m, 700, defl, row, k), 1e-9)


@pytest.mark.parametrize("row", [0, 16, 35])
@pytest.mark.parametrize("k", [3, 6, 11])
def test_target_covariances_of_any_length(row, k, call):
    """|L^-1 c|^2 beyond 1, through 32 (where the kernel's sums wrap), up to 2^22."""
    cl, m, defl = _inputs(0, 16, 40)
    _agree(*call(16, 0, cl, m, 700, defl, row, k), 1e-9)


def test_zero_maps_give_zeros(call):
    cl, m, defl = _inputs(0, 16, 40)
    (_, v, q), (_, v0, q0) = call(16, 0, cl, 0.0 * m, 700, defl)[1], call(16, 0, cl, m, 700, defl)[1]
    assert np.all(v == 0) and np.array_equal(q, q0)


@pytest.mark.parametrize("size", [2.0 ** -1022, 2.0 ** -960])
def test_tiny_values_are_kept(size, call):
    """Maps whose values are subnormal in part or whole, to 1e-9 of the largest and, below
    that, the rounding of the 36 x 36 products to 2^-1074 carried through L^-1 (2^13)."""
    cl, m, defl = _inputs(0, 16, 40)
    (s0, v0, _), (s1, v1, _) = call(16, 0, cl, m * (size / np.max(np.abs(m))), 700, defl)
    assert np.array_equal(s0, s1)
    assert np.max(np.abs(v1 - v0)) <= 1e-9 * np.max(np.abs(v0)) + 36 * 2 ** 13 * 5e-324

"""Bounds of the fixed-point solve (csrc/lens.cuh) on covariances that are not
positive, where its sums (modulo 32) could wrap into acceptable numbers: a matrix row
whose squared length passes 32 before its own pivot, and a target covariance c with
|L^-1 c|^2 beyond 32.  Both are declined (the caller's FP64 form decides), whatever
the length, from just above the bound (1.5) to the longest that entries below 1.9 can
make; rows of unit length pass."""
import numpy as np
import pytest

from oracle import kriging as kr
from tests import host_compile as hc
from tests import test_lens_host as T

DRIVER = r"""
using namespace flints;
static double rd() { char b[64]; if (scanf("%63s", b) != 1) exit(2); return strtod(b, nullptr); }
// S = I but for row `row`, whose first `cnt` entries are v (spin 2: v + iv)
template <int K, class E> static void factor(int row, int cnt, double v) {
    std::vector<E> mat(K * (K + 1) / 2 + 2 * K);
    auto put = [](E &e, double re, double im) {
        if constexpr (std::is_same<E, fx>::value) e = fx_split(fx_of(re, FXB));
        else e = E{fx_split(fx_of(re, FXB)), fx_split(fx_of(im, FXB))};
    };
    for (int i = 0; i < K; ++i)
        for (int j = 0; j <= i; ++j) put(mat[tri<K>(i, j)], i == j ? 1.0 : (i == row && j < cnt ? v : 0.0), i == row && j < cnt ? v : 0.0);
    for (int k = 0; k < K; ++k) {
        put(mat[tri<K>(K, k)], 0.0, 0.0);
        put(mat[tri<K>(K + 1, k)], 0.0, 0.0);
    }
    bool ok = false;
    run_warp([&](int lane) {
        int ey = 0;
        const bool r = factor_fixed<K, 2>(mat.data(), lane, ey);
        if (lane == 0) ok = r;
    });
    printf("%d\n", ok ? 1 : 0);
}
// neighbours so far apart that S = I, and c = v for `cnt` of them, 0 for the rest
template <int K, int SPIN> static void solve(int cnt, double v) {
    static WarpSmem<K, SPIN, double> sm;
    const int n = 64;
    std::vector<Coef64> c64(n, Coef64{0.0, 0.0, 0.0, 0.0});
    c64[0].f = v;
    std::vector<CoefFx> cfx(n);
    for (int k = 0; k < n; ++k) {
        threadIdx.x = k;
        fixed_table_kernel(c64.data(), n, cfx.data());
    }
    LensArgs a{};
    a.tab.c64 = c64.data();
    a.tab.cfx = cfx.data();
    a.tab.n = n;
    const double r = 0.125;
    a.r2 = r * r;
    a.two_r = 2.0 * r;
    a.inv_2r = 0.5 / r;
    a.tab.t_max = 4.0 * a.r2;
    a.tab.inv_h = n / a.tab.t_max;
    PointA P{};
    P.s = P.cph = 1.0;
    double vre = 0.0, vim = 0.0, var = 0.0;
    bool ok = false;
    run_warp([&](int lane) {
        double keyd[Shape<K>::RPL], yre[Shape<K>::RPL], yim[Shape<K>::RPL];
        for (int q = 0; q < Shape<K>::RPL; ++q) {
            const int i = lane + 32 * q;
            keyd[q] = i < cnt ? 0.0 : 0.2 * a.tab.t_max;  // inside the disc
            yre[q] = 1.0;
            yim[q] = 0.0;
            if (i < K) {  // a 4 x 4 x 4 grid of spacing r / 2: chords beyond t_max / 64
                sm.gx[i] = (i % 4 - 1.5) * 0.5 * r;
                sm.gy[i] = (i / 4 % 4 - 1.5) * 0.5 * r;
                sm.gz[i] = (i / 16 - 1.5) * 0.5 * r;
                sm.gnz[i] = sm.gnsn[i] = 0.0;
                sm.gns[i] = sm.gnc[i] = 1.0;
            }
        }
        __syncwarp();
        double x, y, z;
        const bool g = solve_point_fixed<K, SPIN>(sm, P, lane, a, keyd, yre, yim, x, y, z);
        if (lane == 0) {
            ok = g;
            var = z;
        }
    });
    printf("%d %a\n", ok ? 1 : 0, var);
}
int main() {
    char op[16];
    int K, spin, row, cnt;
    while (scanf("%15s %d %d %d %d", op, &K, &spin, &row, &cnt) == 5) {
        const double v = rd();
        if (op[0] == 'f') {
            if (K == 48 && spin == 0) factor<48, fx>(row, cnt, v);
            else if (K == 48) factor<48, fxc>(row, cnt, v);
            else if (spin == 0) factor<16, fx>(row, cnt, v);
            else factor<16, fxc>(row, cnt, v);
        } else if (K == 48) {
            if (spin == 0) solve<48, 0>(cnt, v);
            else solve<48, 2>(cnt, v);
        } else if (spin == 0) {
            solve<16, 0>(cnt, v);
        } else {
            solve<16, 2>(cnt, v);
        }
    }
    return 0;
}
"""


@pytest.fixture(scope="module")
def call(tmp_path_factory):
    if hc.compiler() is None:
        pytest.skip("no host C++ compiler")
    text = (hc.LENS_SHIM + T.KERNEL_SHIM + '#include "' + hc.ROOT + '/include/flints.h"\nnamespace flints {\n'
            + hc.cut("common.cuh", "constexpr unsigned FULL", "// Host-side launchers (lens_spin0.cu", False)
            + hc.cut("xi_table.cu", "__global__ void fixed_table_kernel", "cudaError_t launch_xi_table(", False)
            + hc.cut("lens.cuh", "template <class T>\nstruct Cx {", "// Single-launch kernel", False) + "\n}\n" + DRIVER)
    exe = hc.build(tmp_path_factory.mktemp("bounds"), "bounds", text, warp="threads", sanitize="address")
    return lambda *a: [float.fromhex(t) for t in hc.run(exe, " ".join(str(x) for x in a[:-1]) + f" {float(a[-1]).hex()}\n").split()]


# squared lengths: below 1 (accepted), around 1.5, around 32 (a wrap would make the pivot 1 - 32 + 32), beyond
@pytest.mark.parametrize("spin", [0, 2])
@pytest.mark.parametrize("K", [16, 48])
@pytest.mark.parametrize("length", [0.5, 0.99, 1.2, 1.6, 12.0, 31.2, 31.99, 32.5, 33.5, 64.4])
def test_rows_longer_than_a_positive_matrix_allows_are_declined(K, spin, length, call):
    parts = 2 if spin else 1
    for row in (K - 5, K - 4, K - 1):
        v = np.sqrt(length / (row * parts))
        if v >= 1.9 or row * parts * 1.9 ** 2 < length:
            continue
        assert call("factor", K, spin, row, row, v)[0] == (1.0 if length < 1 else 0.0), row


@pytest.mark.parametrize("spin", [0, 2])
@pytest.mark.parametrize("K,cnt", [(16, 16), (16, 9), (48, 48), (48, 40)])
@pytest.mark.parametrize("length", [0.9, 2.0, 31.5, 32.4, 64.3, 100.0])
def test_target_covariances_longer_than_the_bound_are_declined(K, cnt, spin, length, call):
    v = np.sqrt(length / cnt)
    if v >= 1.9:
        pytest.skip("no such entries")
    ok, var = call("solve", K, spin, 0, cnt, v)
    assert ok == (1.0 if length < 1 else 0.0)
    if ok:
        assert abs(var - (1.0 - length / (1 + kr.EPS_NUGGET))) <= 1e-14 * K

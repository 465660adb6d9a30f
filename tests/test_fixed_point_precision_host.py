"""Rounding of the fixed-point solve of the FP64 plans (csrc/lens.cuh,
solve_point_fixed): the lens kernel's per-tile path runs on the host with the
fixed-point and with the FP64 form, and both are compared with a long double solve
(64-bit significands) of the same systems -- offsets, frames, squared chords and
data as the kernel holds them in FP64, written out at the point of the solve.  The
fixed-point form may be no further from it than the FP64 form, in value (rms over
the targets) and variance, on realisations of the field and on the same maps with
an offset of a hundred times their size, where the data's own rounding decides."""
import os

import numpy as np
import pytest

from oracle import kriging as kr
from tests import host_compile as hc
from tests import test_fixed_point_host as F
from tests import test_lens_host as T

HOOK = "            if constexpr (!MIXED && SPIN != SPIN2_AUG) {\n                if (a.tab.cfx) {"
# per solved target: z, sin(theta), cos(phi), sin(phi) of n'; the neighbour arrays; (t, y_re, y_im) per member
DUMP = r"""            if constexpr (!MIXED && SPIN != SPIN2_AUG) {
                static double rows[K][3];
                for (int r = 0; r < RPL; ++r)
                    if (lane + 32 * r < K) {
                        rows[lane + 32 * r][0] = keyd[r];
                        rows[lane + 32 * r][1] = yre[r];
                        rows[lane + 32 * r][2] = yim[r];
                    }
                __syncwarp();
                if (lane == 0) {
                    FILE *fp = fopen("DIR/systems", "ab");
                    const double h[4] = {P.z, P.s, P.cph, P.sph};
                    fwrite(h, 8, 4, fp);
                    for (const double *g : {sm.gx, sm.gy, sm.gz, sm.gnz, sm.gns, sm.gnc, sm.gnsn}) fwrite(g, 8, K, fp);
                    fwrite(rows, 8, 3 * K, fp);
                    fclose(fp);
                }
                __syncwarp();
            }
"""
TABLE = r"""    {
        FILE *fp = fopen("DIR/table", "wb");
        fwrite(&tg.inv_h, 8, 1, fp);
        fwrite(c64.data(), sizeof(Coef64), n, fp);
        fclose(fp);
    }
    a.tabm = a.tab;"""


@pytest.fixture(scope="module")
def forms(tmp_path_factory):
    """The FP64 form (which writes its systems to the returned directory) and the fixed-point form."""
    if hc.compiler() is None:
        pytest.skip("no host C++ compiler")
    if np.finfo(np.longdouble).eps > 2.0 ** -60:
        pytest.skip("no extended long double")
    d, driver, cut = tmp_path_factory.mktemp("systems"), T.DRIVER, hc.cut

    def cut_with_dump(path, *args):
        text = cut(path, *args)
        if path != "lens.cuh":
            return text
        assert HOOK in text
        return text.replace(HOOK, DUMP.replace("DIR", str(d)) + HOOK)

    try:
        T.DRIVER = driver.replace("    a.tabm = a.tab;", F.FIXED, 1)
        fixed = T._build(tmp_path_factory.mktemp("fixed"))
        T.DRIVER = driver.replace("    a.tabm = a.tab;", TABLE.replace("DIR", str(d)), 1)
        hc.cut = cut_with_dump
        plain = T._build(tmp_path_factory.mktemp("plain"))
    finally:
        T.DRIVER, hc.cut = driver, cut
    return plain, fixed, d


def _solve(d, spin, K):
    """Values and relative variances of the systems written to d, in long double."""
    L = np.longdouble
    t = np.fromfile(d / "table")
    inv_h, C = L(t[0]), t[1:].reshape(-1, 4).astype(L)
    S = np.fromfile(d / "systems").reshape(-1, 4 + 10 * K).astype(L)
    z, s, cph, sph = (S[:, k:k + 1] for k in range(4))
    gx, gy, gz, nz, ns, nc, nsn = (S[:, 4 + k * K:4 + (k + 1) * K] for k in range(7))
    t0, yre, yim = (S[:, 4 + 7 * K:].reshape(-1, K, 3)[..., k] for k in range(3))

    def xi_of(t):
        x = t * inv_h
        k = np.clip(np.floor(x).astype(int), 0, len(C) - 1)
        u, c = x - k, C[k]
        return c[..., 0] + u * (c[..., 1] + u * (c[..., 2] + u * c[..., 3]))

    def phase(dx, dy, dz, zi, si, ci, sni, zj, sj, cj, snj):
        a = zi * (dx * ci + dy * sni) - si * dz + 1j * (dy * ci - dx * sni)
        b = zj * (dx * cj + dy * snj) - sj * dz - 1j * (dy * cj - dx * snj)
        q = a * b
        with np.errstate(invalid="ignore"):
            return np.where(q == 0, 1, q / np.abs(q)) ** spin

    i, j = (lambda a: a[:, :, None]), (lambda a: a[:, None, :])
    dx, dy, dz = j(gx) - i(gx), j(gy) - i(gy), j(gz) - i(gz)
    A = xi_of(dx * dx + dy * dy + dz * dz).astype(np.clongdouble)
    c, y = xi_of(t0).astype(np.clongdouble), yre + 1j * yim
    if spin:
        A = A * phase(dx, dy, dz, i(nz), i(ns), i(nc), i(nsn), j(nz), j(ns), j(nc), j(nsn))
        c = c * phase(gx, gy, gz, z, s, cph, sph, nz, ns, nc, nsn)
    k = np.arange(K)
    A[:, k, k] = L(1.0 + kr.EPS_NUGGET)
    M = np.concatenate([A, c[:, None, :], np.conj(y)[:, None, :]], 1)  # bordered factor, as the kernel's
    for j in range(K):
        for r in range(j, K + 2):
            M[:, r, j] -= (M[:, r, :j] * np.conj(M[:, j, :j])).sum(-1)
        M[:, j:, j] /= np.sqrt(M[:, j, j].real)[:, None]
    return (M[:, K] * np.conj(M[:, K + 1])).sum(-1), L(1) - (np.abs(M[:, K]) ** 2).sum(-1)


@pytest.mark.parametrize("offset", [0.0, 100.0], ids=["field", "offset"])
@pytest.mark.parametrize("case", [F.CASES[k] for k in (0, 2, 3, 4, 9, 10)], ids=lambda c: f"spin{c[0]}-nside{c[1]}-K{c[2]}")
def test_no_further_from_long_double_than_the_fp64_form(case, offset, forms):
    plain, fixed, d = forms
    spin, N, K, lmax, ld, first = case
    cl, bb, defl, pix, vals = T._inputs(spin, N, lmax, ld, first, 64, seed=N + K + spin)
    vals = vals + offset * np.max(np.abs(vals))
    if os.path.exists(d / "systems"):
        os.unlink(d / "systems")
    x0, s0, v0, q0 = plain(spin, K, 0, N, cl, bb, first, defl, pix, vals)
    _, s1, v1, q1 = fixed(spin, K, 0, N, cl, bb, first, defl, pix, vals)
    value, var = _solve(d, spin, K)
    assert not s0.any() and not s1.any() and len(value) == len(v0)
    rms = lambda e: float(np.sqrt(np.mean(np.abs(e) ** 2)))
    assert rms(v1 - value) <= rms(v0 - value)
    assert rms(q1 / x0 - var) <= rms(q0 / x0 - var)

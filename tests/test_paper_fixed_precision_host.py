"""Rounding of the fixed-point apply kernel of the tabulated route (csrc/paper.cu,
apply_kernel_fx), spin 0, 1 and 2, run on the host through the C API under the address
sanitizer at Nside 64, the smallest sky it takes for spin 1 and 2: value and variance of
this kernel and of the FP64 kernel of the same plan against long double sums (64-bit
significands) of the plan's own L^-1, table, member frames and targets.  The fixed-point
kernel may be no further from them than the FP64 kernel (rms over the targets), on
realisations of the field, on the same maps with an offset of a hundred times their size
(the rows of L^-1 cancel there, which the kernel's scaling must not pay for) and on white
noise.  Targets on both sides of the equator: the southern classes are mirrored."""
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
static std::vector<double> rd(FILE *f, size_t n) {
    std::vector<double> v(n);
    if (fread(v.data(), 8, n, f) != n) exit(2);
    return v;
}
int main(int, char **arg) {
    FILE *in = fopen(arg[1], "rb"), *out = fopen(arg[2], "wb");
    const std::vector<double> head = rd(in, 6);
    const long long nside = (long long)head[0], first = (long long)head[3], count = (long long)head[4];
    const int lmax = (int)head[1], spin = (int)head[2], nmap = (int)head[5], comp = spin == 0 ? 1 : 2;
    const size_t nval = (size_t)12 * nside * nside * comp;
    const std::vector<double> cl = rd(in, lmax + 1), defl = rd(in, 2 * count);
    flints_paper_t h = nullptr;
    if (flints_paper_plan(&h, nside, lmax, cl.data(), nullptr, 2, spin, 0, 0, nullptr) || !h->fixed) return 3;
    const double info[3] = {h->xi0, h->n / h->t_max, (double)h->n};
    fwrite(info, 8, 3, out);
    fwrite(h->d_c64, 32, h->n, out);
    flints::paper::ApplyArgs a{};
    a.N = nside;
    a.Nc = h->nside_c;
    a.first = first;
    a.count = count;
    a.defl = defl.data();
    for (long long p = 0; p < count; ++p) {  // target, mirrored or not; members' pixels and frames; L^-1 by rows
        double t[4] = {0.0, 0.0, 1.0, 0.0};
        int64_t c = 0;
        flints::paper::target_of(a, p, t[0], t[1], t[2], c);
        t[3] = spin != 0 && c >= 6 * a.Nc * a.Nc + 2 * a.Nc;
        const int64_t sl = h->d_slot[c];
        fwrite(t, 8, 4, out);
        for (int j = 0; j < 36; ++j) {
            const int m = h->d_members[c * 36 + j];
            double v[5] = {(double)m, 0.0, 0.0, 0.0, 0.0};
            if (m >= 0) std::memcpy(v + 1, h->d_pv + 2 * (size_t)m, 32);
            fwrite(v, 8, 5, out);
        }
        for (int i = 0; i < 36; ++i)
            for (int j = 0; j < 36; ++j) {
                double v[2] = {0.0, 0.0};
                for (int q = 0; q < comp && j <= i; ++q)
                    v[q] = h->d_linv[(sl * flints::paper::linv_len(36) + flints::paper::lanestep_index(i, j)) * comp + q];
                fwrite(v, 8, 2, out);
            }
    }
    for (int k = 0; k < nmap; ++k) {
        const std::vector<double> map = rd(in, nval);
        for (int form = 0; form < 2; ++form) {  // the FP64 kernel, the fixed-point kernel
            h->fixed = form == 1;
            std::vector<double> o(count * comp), var(count);
            std::vector<uint8_t> st(count);
            if (flints_paper_lens(h, first, count, map.data(), defl.data(), o.data(), var.data(), st.data(), nullptr)) return 4;
            for (long long p = 0; p < count; ++p) {
                const double v[4] = {(double)st[p], o[p * comp], comp == 2 ? o[2 * p + 1] : 0.0, var[p]};
                fwrite(v, 8, 4, out);
            }
        }
    }
    flints_paper_free(h);
    fclose(out);
    return 0;
}
"""


@pytest.fixture(scope="module")
def exe(tmp_path_factory):
    if hc.compiler() is None:
        pytest.skip("no host C++ compiler")
    if np.finfo(np.longdouble).eps > 2.0 ** -60:
        pytest.skip("no extended long double")
    return ch.build(tmp_path_factory.mktemp("paper_fx"), "paper_fx", ["common.cuh", "lens.cuh", "paper_geom.cuh", "xi_table.cu", "paper.cu"],
                    DRIVER, sanitize="address")


@pytest.mark.parametrize("spin", [0, 1, 2])
def test_no_further_from_long_double_than_the_fp64_kernel(spin, exe, tmp_path):
    import subprocess

    L, nside, n = np.longdouble, 64, 64
    lmax, npix, comp = 2 * nside, hp.npix(nside), 1 if spin == 0 else 2
    ell = np.arange(lmax + 1.0)
    cl = {0: wl.cl_tt(lmax, 0.7 * lmax), 1: ell * (ell + 1) * wl.cl_phiphi(lmax), 2: wl.cl_ee(lmax, 0.7 * lmax)}[spin]
    m = sht.synth_map(nside, lmax, wl.draw_alm(wl.cl_phiphi(lmax) if spin == 1 else cl, 31), spin=2 if spin == 2 else 0, gradient=spin == 1)
    m = (np.stack([m.real, m.imag], 1) if spin == 2 else np.asarray(m)).reshape(npix, comp)
    maps = [m, m + 100 * np.max(np.abs(m)), np.random.default_rng(3).normal(size=m.shape)]
    defl = wl.random_deflection(n, 5, rms=0.5 * np.sqrt(4 * np.pi / npix))
    first = npix // 2 + 2 * nside - n // 2  # across the last ring of the northern classes
    np.concatenate([[nside, lmax, spin, first, n, len(maps)], cl, defl.ravel(), *(v.ravel() for v in maps)]).tofile(tmp_path / "in")
    r = subprocess.run([exe, str(tmp_path / "in"), str(tmp_path / "out")], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    o = np.fromfile(tmp_path / "out")
    x0, inv_h, nt = o[0], L(o[1]), int(o[2])
    C, o = o[3:3 + 4 * nt].reshape(-1, 4).astype(L), o[3 + 4 * nt:]
    rec = 4 + 36 * 5 + 36 * 36 * 2
    T, res = o[:n * rec].reshape(n, rec), o[n * rec:].reshape(len(maps), 2, n, 4)
    tx, ty, tz, mirrored = (T[:, k:k + 1].astype(L) for k in range(4))
    assert spin == 0 or 0 < mirrored.sum() < n
    mem = T[:, 4:184].reshape(n, 36, 5)
    idx, (p0, p1, p2, p3) = mem[..., 0].astype(int), (mem[..., k].astype(L) for k in (1, 2, 3, 4))
    Li = T[:, 184:].reshape(n, 36, 36, 2).astype(L)
    Li = Li[..., 0] + 1j * np.where(mirrored[..., None] > 0, -Li[..., 1], Li[..., 1])
    # members: (x, y), (z, 0) at spin 0; (cos phi, sin phi), (z, sin theta) at spin 1 and 2
    mx, my, mz = (p0, p1, p2) if spin == 0 else (p3 * p0, p3 * p1, p2)
    dx, dy, dz = mx - tx, my - ty, mz - tz
    x = (dx * dx + dy * dy + dz * dz) * inv_h
    k = np.clip(np.floor(x).astype(int), 0, nt - 1)
    u, c4 = x - k, C[k]
    c = (c4[..., 0] + u * (c4[..., 1] + u * (c4[..., 2] + u * c4[..., 3]))).astype(np.clongdouble)
    if spin:  # transport phase from the direction of the chord in both frames
        s = np.sqrt(tx * tx + ty * ty)
        a = tz * (dx * tx + dy * ty) / s - s * dz + 1j * (dy * tx - dx * ty) / s
        b = p2 * (dx * p0 + dy * p1) - p3 * dz - 1j * (dy * p0 - dx * p1)
        c = c * (a * b / np.abs(a * b)) ** spin
    c = np.where(idx >= 0, c, 0)
    zc = (Li * np.conj(c)[:, None]).sum(-1)
    var = L(1) - (np.abs(zc) ** 2).sum(-1)
    rms = lambda e: float(np.sqrt(np.mean(np.abs(e) ** 2)))
    assert not res[..., 0].any()
    for name, mp, (f64, fx) in zip(("field", "offset", "white"), maps, res):
        y = np.where(idx >= 0, (mp[idx] @ ([1] if comp == 1 else [1, 1j])).astype(np.clongdouble), 0)
        value = (np.conj(zc) * (Li * y[:, None]).sum(-1)).sum(-1)
        off = [rms(q[:, 1] + 1j * q[:, 2] - value) for q in (f64, fx)]
        assert off[1] <= off[0], (name, off)
        off = [rms(q[:, 3] / x0 - var) for q in (f64, fx)]
        assert off[1] <= off[0], (name, "variance", off)

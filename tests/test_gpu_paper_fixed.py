"""The y = 2 FP64 plans of the tabulated route on the integer pipe (apply_kernel_fx), from
the smallest sky it takes for spin 1 and 2 (Nside 64): against the oracle's class route on
targets of every zone (tolerance: the route's FP64 parity, 1e-9 of the map's rms), ranges
of every remainder of its 8-target groups and 32-target tiles bit for bit equal to the
whole sky, and a value that is not finite touching only the targets whose stencil holds it."""
import numpy as np
import pytest

import workloads as wl
from oracle import faces as fc
from oracle import sht
from oracle import xi
from tests.gpu_common import require_gpu

pytestmark = pytest.mark.gpu
NSIDE, NPIX, LMAX = 64, 12 * 64 * 64, 128


@pytest.fixture(scope="module")
def fl():
    return require_gpu()


@pytest.mark.parametrize("spin", [0, 1, 2])
def test_fixed_point_apply(fl, spin):
    import torch

    ell = np.arange(LMAX + 1.0)
    cl = {0: wl.cl_tt(LMAX, 78.0), 1: ell * (ell + 1) * wl.cl_phiphi(LMAX), 2: wl.cl_ee(LMAX, 78.0)}[spin]
    alm = wl.draw_alm(wl.cl_phiphi(LMAX) if spin == 1 else cl, 31)
    m = sht.synth_map(NSIDE, LMAX, alm, spin=2 if spin == 2 else 0, gradient=spin == 1)
    m = np.ascontiguousarray(np.stack([m.real, m.imag], 1) if spin == 2 else m)
    d = wl.random_deflection(NPIX, 32) * 16
    t_max, n = fc.paper_grid_rule(cl, NSIDE, 2)
    tab, x0 = (xi.spin0_table(cl, t_max, n) if spin == 0
               else (xi.spin1_tables if spin == 1 else xi.spin2_tables)(cl, None, t_max, n)[::2])
    pix = np.unique(np.r_[:12, 8000:8012, 24500:24512, 41000:41012, NPIX - 12:NPIX, wl.sample_pixels(NPIX, 60, 33)])
    ref = fc.paper_lens(NSIDE, 2, m, d[pix], pix, tab, x0, classes=True, **({"spin": spin} if spin else {}))
    dm, dd = torch.from_numpy(m).cuda(), torch.from_numpy(d).cuda()
    plan = fl.PaperPlan(NSIDE, cl, 2, spin=spin)
    st = torch.empty(NPIX, dtype=torch.uint8, device="cuda")
    out, var = plan.lens(dm, dd, status=st)
    v = out.cpu().numpy()[pix]
    v = v if spin == 0 else v[:, 0] + 1j * v[:, 1]
    assert not st.any()
    assert np.max(np.abs(v - ref[0])) <= 1e-9 * np.sqrt(np.mean(np.abs(ref[0]) ** 2))
    assert np.max(np.abs(var.cpu().numpy()[pix] - ref[1])) <= 1e-9 * x0
    for first, count in [(0, 1), (3, 7), (100, 8), (77, 9), (5, 31), (12000, 33), (40000, 97)]:
        o, q = plan.lens(dm, dd[first:first + count].contiguous(), first, count)
        assert torch.equal(o, out[first:first + count]) and torch.equal(q, var[first:first + count])
    dm[20000] = float("inf")
    o, q = plan.lens(dm, dd)
    bad = ~torch.isfinite(o).reshape(NPIX, -1).all(1)
    assert 4 <= int(bad.sum()) <= 200 and torch.equal(o[~bad], out[~bad])
    assert float((q - var).abs().max()) <= 1e-12 * x0
    plan.close()

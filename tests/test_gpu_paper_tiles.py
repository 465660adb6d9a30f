"""Launch shapes of the tabulated route chosen from the number of targets: ranges of every
tile size of the fixed-point kernel (y = 2, FP64; one target to full tiles), and ranges on
both sides of the line between the two forms for nine members at spin 0, have the values of
the same range inside the whole-sky call, bit for bit."""
import pytest

import workloads as wl
from tests.gpu_common import require_gpu

pytestmark = pytest.mark.gpu
NSIDE, NPIX = 128, 12 * 128 * 128


@pytest.fixture(scope="module")
def fl():
    return require_gpu()


def _ranges_equal_the_whole_sky(fl, spin, y, precision, counts):
    import torch

    cl = wl.cl_tt(256, 180.0) if spin == 0 else wl.cl_ee(256, 180.0)
    m = torch.from_numpy(wl.white_map(NPIX, 1 if spin == 0 else 2, 51)).cuda()
    d = torch.from_numpy(wl.random_deflection(NPIX, 52) * 8).cuda()
    plan = fl.PaperPlan(NSIDE, cl, y, spin=spin, precision=precision)
    buf = lambda n: torch.empty(n, dtype=torch.uint8, device="cuda")
    s = buf(NPIX)
    out, var = plan.lens(m, d, status=s)
    for k, count in enumerate(counts):
        first = (977 * k * k + 13 * k) % (NPIX - count + 1)
        sl, t = slice(first, first + count), buf(count)
        o, q = plan.lens(m, d[sl].contiguous(), first, count, status=t)
        assert torch.equal(o, out[sl]) and torch.equal(q, var[sl]) and torch.equal(t, s[sl]), (first, count)
    plan.close()


@pytest.mark.parametrize("spin", [0, 1, 2])
def test_fixed_point_tiles(fl, spin):
    import torch

    warps = torch.cuda.get_device_properties(0).multi_processor_count * 16  # 1, 2, 8, 9 -> 16, 24, 32 targets a tile
    _ranges_equal_the_whole_sky(fl, spin, 2, "fp64", [1, 2, 31, warps, warps + 1, 8 * warps - 3, 8 * warps + 1, 17 * warps, 24 * warps + 5])


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_nine_members(fl, precision):
    import torch

    line = torch.cuda.get_device_properties(0).multi_processor_count * 8
    _ranges_equal_the_whole_sky(fl, 0, 1, precision, [1, 2, 3, 7, 8, 9, 101, line - 1, line, line + 1, 3 * line])

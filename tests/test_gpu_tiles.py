"""Launch shapes chosen from the number of targets: a range lensed on its own has the
values of the same range inside the whole-sky call, bit for bit (every target's
arithmetic is its own; only the split into warp tiles and blocks differs), from one
target up past the size where full tiles are used."""
import numpy as np
import pytest

import workloads as wl
from tests.gpu_common import require_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def fl():
    return require_gpu()


@pytest.mark.parametrize("spin,K,flags", [(0, 16, 0), (2, 24, 0), (1, 16, 0), (2, 16, 1)])
@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_ranges_equal_the_whole_sky(fl, spin, K, flags, precision):
    import torch

    nside, npix = 64, 12 * 64 * 64
    cl = wl.cl_tt(128, 100.0) if spin == 0 else wl.cl_ee(128, 100.0)
    m = torch.from_numpy(wl.white_map(npix, 1 if spin == 0 else 2, 21)).cuda()
    d = torch.from_numpy(wl.random_deflection(npix, 22) * 4).cuda()
    plan = fl.Plan(nside, cl, spin=spin, K=K, precision=precision, flags=flags)
    buf = lambda n: (torch.empty(n, dtype=torch.float64, device="cuda"), torch.empty(n, dtype=torch.uint8, device="cuda"))
    var, st = buf(npix)
    out, _, _ = plan.lens(m, d, var=var, status=st)
    for first, count in [(0, 1), (5, 15), (1000, 17), (77, 151), (20000, 153), (3, 1009), (12345, 2433), (1, 38913)]:
        v, s = buf(count)
        o, _, _ = plan.lens(m, d[first:first + count].contiguous(), var=v, status=s, first=first, count=count)
        sl = slice(first, first + count)
        assert torch.equal(o, out[sl]) and torch.equal(v, var[sl]) and torch.equal(s, st[sl]), (first, count)
    plan.close()

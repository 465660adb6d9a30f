"""Tile sizes that a batch chooses (csrc/api.cu, flints_batch_stage) on the host: per class
the size that balances that class's targets over the warps which its kernel keeps
resident (the stand-in's occupancy: two blocks per SM of the warps that fit), as plan
calls choose it; a tile size of the caller's is taken as it is."""
import numpy as np
import pytest

import workloads as wl
from tests import cuda_host as ch
from tests import host_compile as hc
from tests import test_api_host as A

DRIVER = r"""
int main() {
    int lmax, tile;
    long long count;
    if (scanf("%d", &lmax) != 1) return 2;
    std::vector<double> cl(lmax + 1);
    for (double &v : cl) if (scanf("%la", &v) != 1) return 2;
    alignas(16) static double buf[2 * 12 * 16 * 16];
    const int kinds[3][3] = {{0, 16, 0}, {2, 48, 0}, {2, 32, 1}};  // spin, K, precision
    flints_plan_t p[3];
    for (int k = 0; k < 3; ++k)
        if (flints_plan(&p[k], 16, lmax, cl.data(), nullptr, kinds[k][0], kinds[k][1], kinds[k][2], 0, nullptr)) return 3;
    flints_batch_t b = nullptr;
    if (flints_batch_create(&b, 64)) return 4;
    while (scanf("%lld %d", &count, &tile) == 2) {
        int64_t own[BATCH_CLASSES] = {0};
        std::vector<flints_job> jobs;  // `count` targets in jobs of at most a sky, plans in turn
        for (long long left = count; left > 0; left -= jobs.back().count) {
            flints_job j{};
            j.plan = p[jobs.size() % 3];
            j.map = j.defl = buf;
            j.out = buf;
            j.count = left < 3072 ? left : 3072;
            jobs.push_back(j);
            const int *k = kinds[(jobs.size() - 1) % 3];
            own[8 * k[2] + (k[0] == 2 ? 4 : 0) + batch_k_index(k[1])] += j.count;
        }
        if (flints_batch_stage(b, jobs.data(), (int)jobs.size(), tile)) return 5;
        for (int cls = 0; cls < BATCH_CLASSES; ++cls)
            printf("%d %d\n", hdr_of(b->h_buf)->tile_pts[cls],
                   tile ? tile : auto_tile_points(own[cls], (int64_t)152 * 2 * b->wpb[cls]));
    }
    flints_batch_free(b);
    for (flints_plan_t q : p) flints_free(q);
    return 0;
}
"""


def test_tile_sizes(tmp_path):
    if hc.compiler() is None:
        pytest.skip("no host C++ compiler")
    exe = ch.build(tmp_path, "tiles", A.FILES, "using namespace flints;\n" + DRIVER)
    cl = wl.cl_ee(32, 22.0)
    cases = [(1, 0), (1000, 0), (1500, 0), (5000, 0), (20000, 0), (60000, 0), (180000, 0), (5000, 7)]
    out = hc.run(exe, f"32 {' '.join(x.hex() for x in cl)} " + " ".join(f"{c} {t}" for c, t in cases) + "\n").split()
    got = np.array(out, dtype=int).reshape(len(cases), -1, 2)
    assert np.array_equal(got[..., 0], got[..., 1])
    assert len(np.unique(got[..., 0])) > 4  # the rule's whole range

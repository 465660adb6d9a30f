"""The fork and join of a batch's class kernels (csrc/api.cu, ClassStreams) on a recording
stand-in for CUDA's streams and events, whose happens-before order is followed through
every record and wait: each kernel sees what the caller's stream held before the launch,
the caller's stream holds every kernel afterwards, side streams have the caller's
priority, a capture creates no stream, and a freed batch leaves no stream or event."""
import os

import pytest

from tests import host_compile as hc

RUNTIME = r"""
#include <algorithm>
#include <set>
typedef int cudaError_t;
enum { cudaSuccess = 0 };
struct Stream { int priority; std::set<int> seen; };
struct Event { std::set<int> seen; };
typedef Stream *cudaStream_t;
typedef Event *cudaEvent_t;
enum { cudaEventDisableTiming = 2, cudaStreamNonBlocking = 1 };
enum cudaStreamCaptureStatus { cudaStreamCaptureStatusNone, cudaStreamCaptureStatusActive };
static int g_live = 0, g_streams_made = 0;
static Stream g_default{0, {}};
static Stream &at(cudaStream_t s) { return s ? *s : g_default; }
static cudaError_t cudaDeviceGetStreamPriorityRange(int *least, int *greatest) { *least = 0; *greatest = -5; return 0; }
static cudaError_t cudaStreamCreateWithPriority(cudaStream_t *s, unsigned, int p) {
    ++g_live;
    ++g_streams_made;
    *s = new Stream{std::max(-5, std::min(0, p)), {}};
    return 0;
}
static cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, unsigned f) { return cudaStreamCreateWithPriority(s, f, 0); }
static cudaError_t cudaStreamDestroy(cudaStream_t s) { --g_live; delete s; return 0; }
static cudaError_t cudaStreamGetPriority(cudaStream_t s, int *p) { *p = at(s).priority; return 0; }
static cudaError_t cudaEventCreateWithFlags(cudaEvent_t *e, unsigned) { ++g_live; *e = new Event; return 0; }
static cudaError_t cudaEventDestroy(cudaEvent_t e) { --g_live; delete e; return 0; }
static cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t s) { e->seen = at(s).seen; return 0; }
static cudaError_t cudaStreamWaitEvent(cudaStream_t s, cudaEvent_t e, unsigned) {
    at(s).seen.insert(e->seen.begin(), e->seen.end());
    return 0;
}
static cudaError_t cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus *c) { *c = cudaStreamCaptureStatusNone; return 0; }
"""

DRIVER = r"""
#define CHECK(x) if (!(x)) { fprintf(stderr, "line %d: %s\n", __LINE__, #x); return 1; }
int main() {
    ClassStreams cs;
    std::memset(&cs, 0, sizeof cs);
    CHECK(cs.create() == 0);
    Stream low{0, {}}, high{-5, {}}, mid{-2, {}};
    int op = 0;
    auto launch = [&](cudaStream_t st, int kernels, bool capture, bool spread) -> int {
        const int made = g_streams_made, before = ++op, priority = at(st).priority;
        at(st).seen.insert(before);
        CHECK(cs.fork(st, kernels, capture) == 0);
        std::set<cudaStream_t> used;
        for (int q = 0; q < kernels; ++q) {
            const cudaStream_t s = cs.of(st, q);
            CHECK(at(s).seen.count(before) == 1);
            CHECK(at(s).priority == priority);
            at(s).seen.insert(++op);
            used.insert(s);
        }
        CHECK(cs.join(st) == 0);
        for (int k = before; k <= op; ++k) CHECK(at(st).seen.count(k) == 1);
        CHECK(!capture || g_streams_made == made);
        CHECK((int)used.size() == (spread ? std::min(kernels, BATCH_SIDE + 1) : (kernels > 0)));
        return 0;
    };
    for (int kernels : {0, 1, 2, 3, 4, 5, 16}) {
        CHECK(launch(nullptr, kernels, false, true) == 0);
        CHECK(launch(&low, kernels, true, true) == 0);  // the default priority's streams come with the batch
    }
    CHECK(launch(&high, 16, true, false) == 0);  // a priority without streams, in a capture: one stream
    CHECK(launch(&high, 7, false, true) == 0);
    CHECK(launch(&high, 16, true, true) == 0);
    CHECK(launch(&mid, 3, false, true) == 0);
    CHECK(launch(&low, 7, false, true) == 0);
    const int made = g_streams_made;
    CHECK(launch(&high, 7, false, true) == 0 && g_streams_made == made);  // kept, not made again
    cs.release();
    CHECK(g_live == 0);
    return 0;
}
"""


def test_fork_and_join(tmp_path):
    if hc.compiler() is None:
        pytest.skip("no host C++ compiler")
    src = open(os.path.join(hc.CSRC, "api.cu")).read()
    a = src.index("constexpr int BATCH_SIDE")
    text = src[a:src.index("struct flints_batch_s {", a)].replace("#ifdef __CUDACC__", "#if 1")
    hc.run(hc.build(tmp_path, "streams", RUNTIME + text + DRIVER, warp="none", sanitize="address"), "")

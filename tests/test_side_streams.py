"""Side streams of a count call, with the CUDA runtime's calls replaced by the
test's: their priority is the caller's stream's, sets are kept by device and
priority and bounded, and an error between fork and join waits for the sides."""
from host_check import run_host_program

PROGRAM = r"""
#include <cstdio>
#include <cstdlib>
#include <map>
#include <memory>
#include <set>
#include <vector>
#include "tg_side.hpp"

static int device = 0, live_events = 0, synced = 0, records = 0, fail_record = -1;
static std::map<cudaStream_t, int> live;                     // stream -> priority
static std::map<cudaStream_t, int> callers;
static uintptr_t next_handle = 1000;

extern "C" {
cudaError_t cudaGetDevice(int *d) { *d = device; return cudaSuccess; }
cudaError_t cudaStreamGetPriority(cudaStream_t s, int *p) {
    if (callers.count(s)) { *p = callers[s]; return cudaSuccess; }
    return cudaErrorInvalidResourceHandle;
}
cudaError_t cudaStreamCreateWithPriority(cudaStream_t *s, unsigned flags, int p) {
    if (flags != cudaStreamNonBlocking) return cudaErrorInvalidValue;
    *s = (cudaStream_t)(next_handle++);
    live[*s] = p;
    return cudaSuccess;
}
cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, unsigned flags) { return cudaStreamCreateWithPriority(s, flags, 0); }
cudaError_t cudaStreamDestroy(cudaStream_t s) { live.erase(s); return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { ++synced; return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t *e, unsigned) {
    *e = (cudaEvent_t)(next_handle++);
    ++live_events;
    return cudaSuccess;
}
cudaError_t cudaEventDestroy(cudaEvent_t) { --live_events; return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) {
    return records++ == fail_record ? cudaErrorUnknown : cudaSuccess;
}
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
const char *cudaGetErrorString(cudaError_t) { return "error"; }
}

#define CHECK(x) do { if (!(x)) { std::printf("line %d: %s\n", __LINE__, #x); std::exit(1); } } while (0)
using tg::SideStreams;

static std::set<cudaStream_t> call(cudaStream_t main, int priority) {
    SideStreams s(main);
    s.fork();
    s.after_main(0);
    s.join();
    std::set<cudaStream_t> used;
    for (int k = 0; k < SideStreams::kSides; ++k) {
        used.insert(s.side(k));
        CHECK(live.count(s.side(k)) && live[s.side(k)] == priority);
    }
    return used;
}

int main() {
    cudaStream_t ordinary = (cudaStream_t)1, high = (cudaStream_t)2, unknown = (cudaStream_t)3;
    callers = {{ordinary, 0}, {high, -5}};
    const auto a = call(ordinary, 0), b = call(high, -5);
    CHECK(call(ordinary, 0) == a && call(high, -5) == b);    // kept by priority
    CHECK(call(unknown, 0) == a);                            // a stream without one
    device = 1;
    const auto c = call(ordinary, 0);
    CHECK(c != a && call(ordinary, 0) == c);                 // and by device
    device = 0;
    {                                                        // twenty calls at once, eight sets kept
        std::vector<std::unique_ptr<SideStreams>> at_once;
        for (int k = 0; k < 20; ++k) at_once.push_back(std::make_unique<SideStreams>(ordinary));
    }
    CHECK((int)live.size() == SideStreams::kSides * (8 + 1 + 1));
    const size_t streams = live.size();
    const int events = live_events;
    for (int at = 0; at < 5; ++at) {                         // an error at any record from the fork on
        records = 0, fail_record = at, synced = 0;
        bool thrown = false;
        try {
            call(high, -5);
        } catch (const tg::Error &) {
            thrown = true;
        }
        CHECK(thrown && synced == SideStreams::kSides);
        CHECK(live.size() == streams - SideStreams::kSides && live_events == events - (2 + SideStreams::kSides));
        fail_record = -1;
        call(high, -5);                                      // a set in its place
        CHECK(live.size() == streams && live_events == events);
    }
    std::printf("ok\n");
    return 0;
}
"""


def test_side_streams(tmp_path):
    assert run_host_program(PROGRAM, tmp_path).strip() == "ok"

// Runs the canonicaliser's 32 lanes on the host.  Each lane is a coroutine that runs
// from one warp-wide call to the next; the lanes take their turns in an order of the
// caller's choice, so a lane may be a whole step ahead of another wherever no barrier
// stands between them, as independent thread scheduling allows.
#include <ucontext.h>

#include <cstring>
#include <vector>

#include "pt_internal.h"

namespace {
constexpr int kLanes = 32;
enum Kind { kDone, kSync, kVote, kShuffle };
ucontext_t g_main, g_lane[kLanes];
std::vector<char> g_stack[kLanes];
int g_cur, g_kind[kLanes];
unsigned g_calls[kLanes];
unsigned long long g_val[2][kLanes];  // by the parity of a lane's calls: no lane is more than one ahead

unsigned long long* arrive(Kind kind, unsigned long long x) {
    unsigned long long* v = g_val[g_calls[g_cur]++ & 1];
    v[g_cur] = x;
    g_kind[g_cur] = kind;
    swapcontext(&g_lane[g_cur], &g_main);
    return v;
}
void __syncwarp() { arrive(kSync, 0); }
bool __all_sync(unsigned, bool p) {
    const unsigned long long* v = arrive(kVote, p);
    bool all = true;
    for (int l = 0; l < kLanes; ++l) all = all && v[l];
    return all;
}
unsigned long long __shfl_down_sync(unsigned, unsigned long long x, int d) {
    const unsigned long long* v = arrive(kShuffle, x);
    return v[g_cur + d < kLanes ? g_cur + d : g_cur];
}
int atomicAdd(int* p, int x) { const int old = *p; *p += x; return old; }
int atomicCAS(int* p, int want, int x) { const int old = *p; if (old == want) *p = x; return old; }
}  // namespace

#include "pt_canon.h"

namespace {
struct Job {
    int n;
    const int32_t* edges;
    const double* lengths;
    pt::TreeSet ts;
    int32_t* err;
    pt::CanonSmem s;
} g_job;
void lane_main() {
    pt::canon_tree(g_job.n, 0, g_cur, g_job.edges, g_job.lengths, g_job.ts, g_job.err, g_job.s);
    g_kind[g_cur] = kDone;
}
}  // namespace

// order: 0 lanes upwards, 1 downwards, else a new order after every call, from that seed.
// Returns 0, or 1 when the lanes met at different calls (a hang or worse on a GPU).
extern "C" int canon_lanes(int n, const int32_t* edges, const double* lengths, unsigned order, int32_t* up, int32_t* ch,
                           double* len, uint64_t* bits, int32_t* erank, int32_t* sched, uint64_t* key, int32_t* emap,
                           int32_t* err) {
    g_job.n = n;
    g_job.edges = edges;
    g_job.lengths = lengths;
    g_job.ts = pt::TreeSet{n, 1, up, ch, len, bits, erank, sched, key, emap};
    g_job.err = err;
    std::memset(&g_job.s, 0x55, sizeof g_job.s);  // shared memory starts with anything in it
    int turn[kLanes];
    for (int l = 0; l < kLanes; ++l) {
        turn[l] = order == 1 ? kLanes - 1 - l : l;
        g_stack[l].resize(1 << 16);
        g_calls[l] = 0;
        getcontext(&g_lane[l]);
        g_lane[l].uc_stack.ss_sp = g_stack[l].data();
        g_lane[l].uc_stack.ss_size = g_stack[l].size();
        g_lane[l].uc_link = &g_main;
        makecontext(&g_lane[l], lane_main, 0);
    }
    unsigned rnd = order;
    do {
        if (order > 1)
            for (int l = kLanes - 1; l > 0; --l) {
                rnd = rnd * 1664525u + 1013904223u;
                std::swap(turn[l], turn[(rnd >> 8) % (l + 1)]);
            }
        for (int l = 0; l < kLanes; ++l) {
            g_cur = turn[l];
            swapcontext(&g_main, &g_lane[g_cur]);
        }
        for (int l = 1; l < kLanes; ++l)
            if (g_kind[l] != g_kind[0]) return 1;
    } while (g_kind[0] != kDone);
    return 0;
}

// Runs the Newton exchange of one CTA of a cluster on the host.  Each thread is a coroutine
// that runs until a barrier, a warp vote or a wait stops it; whenever it can, the thread of
// the first warp of the caller's order runs, so one warp may be as far ahead of another as
// the barriers allow.  The other CTAs' sums come with every exchange but those from `drop`
// on, which never do.  starve: the last warp of the order only runs when a wait has run out
// or nothing else can run.
#include <ucontext.h>

#include <algorithm>
#include <vector>

#include "pt_internal.h"

namespace {
constexpr int kMaxThreads = 512;
enum State { kReady, kSpin, kVote, kBarrier, kDone };
ucontext_t g_main, g_thread[kMaxThreads];
std::vector<char> g_stack[kMaxThreads];
State g_state[kMaxThreads];
bool g_vote[kMaxThreads], g_any[kMaxThreads];
int g_cur, g_threads, g_nw, g_drop, g_armed, g_broken;
long long g_clock;  // moves when only waits are left

void stop(State s) {
    g_state[g_cur] = s;
    swapcontext(&g_thread[g_cur], &g_main);
}
// An mbarrier of nw + 1 arrivals and the bytes still to come.
struct Bar {
    int arrived, phase;
    long long bytes;
} g_bar[2];
struct Smem {
    alignas(16) float cxr[2][pt::kMaxTeamWarps][4];
    unsigned long long mbx[2];
    int abort_, done;
} g_ns;
Bar& bar_of(unsigned long long* b) { return g_bar[b - g_ns.mbx]; }
void complete(Bar& b) {
    if (b.arrived > g_nw + 1) g_broken = 1;  // more arrivals than the phase takes
    if (b.arrived == g_nw + 1 && b.bytes == 0) b.arrived = 0, ++b.phase;
}
}  // namespace

namespace pt {
void mbar_arrive(unsigned long long* b) { ++bar_of(b).arrived, complete(bar_of(b)); }
void mbar_arrive_expect(unsigned long long* b, unsigned bytes) {
    if (g_armed++ >= g_drop) bar_of(b).bytes += bytes;
    mbar_arrive(b);
}
bool mbar_test_wait(unsigned long long* b, unsigned parity) {
    if ((bar_of(b).phase & 1) != (int)parity) return true;
    stop(kSpin);
    return (bar_of(b).phase & 1) != (int)parity;
}
void cluster_push16(float*, unsigned long long*, unsigned, float4) {}
long long clock64() { return g_clock; }
void __syncthreads() { stop(kBarrier); }
bool __any_sync(unsigned, bool p) {
    g_vote[g_cur] = p;
    stop(kVote);
    return g_any[g_cur];
}
}  // namespace pt

#include "pt_exchange.h"

namespace {
int g_solves, g_steps, g_maxit, g_ld, *g_evals;
void thread_main() {
    const int id = g_cur, w = id / 32, lane = id % 32;
    pt::Team tm{2, 0, 0, 0};
    for (int s = 0; s < g_solves; ++s) {
        pt::__syncthreads();
        int n = 0;
        g_evals[s * g_threads + id] = pt::newton_evaluations<true>(
            g_maxit, w, lane, g_nw, g_ld, g_ns, tm, [] { return make_float4(0, 0, 0, 0); },
            [&](int, bool last) { return ++n == g_steps || last ? 1 : 0; });
    }
    g_state[id] = kDone;
}
}  // namespace

// `solves` solves that end at their `steps`-th evaluation, by nw warps led by warp ld, which
// run in the order `turn`; exchanges from number `drop` on never complete.  evals: [solve][thread].
// Returns 0; 1 when no thread can go on (a hang on a GPU); 2 when a barrier took too many arrivals.
extern "C" int exchange_warps(int nw, int ld, const int* turn, int solves, int steps, int maxit, int drop, int starve,
                              int* evals, int* gave_up) {
    g_threads = 32 * nw;
    g_nw = nw, g_ld = ld, g_solves = solves, g_steps = steps, g_maxit = maxit, g_drop = drop, g_evals = evals;
    g_armed = g_broken = 0, g_clock = 0;
    g_ns = Smem{}, g_bar[0] = g_bar[1] = Bar{};
    for (int t = 0; t < g_threads; ++t) {
        g_stack[t].resize(1 << 15);
        g_state[t] = kReady;
        getcontext(&g_thread[t]);
        g_thread[t].uc_stack.ss_sp = g_stack[t].data();
        g_thread[t].uc_stack.ss_size = g_stack[t].size();
        g_thread[t].uc_link = &g_main;
        makecontext(&g_thread[t], thread_main, 0);
    }
    auto all = [&](int from, int to, State s) {
        return std::all_of(g_state + from, g_state + to, [=](State x) { return x == s; });
    };
    while (!all(0, g_threads, kDone)) {
        int next = -1, spin = -1;
        for (int k = 0; k < nw && next < 0; ++k)
            for (int l = 0; l < 32 && next < 0; ++l) {
                const int t = 32 * turn[k] + l;
                if (g_state[t] == kSpin && spin < 0) spin = t;
                if (g_state[t] == kReady && !(starve && spin >= 0 && k == nw - 1)) next = t;
            }
        if (next < 0 && all(0, g_threads, kBarrier)) {
            std::fill(g_state, g_state + g_threads, kReady);
            continue;
        }
        for (int w = 0; w < nw && next < 0; ++w)
            if (all(32 * w, 32 * w + 32, kVote)) {
                const bool any = std::any_of(g_vote + 32 * w, g_vote + 32 * w + 32, [](bool x) { return x; });
                std::fill(g_any + 32 * w, g_any + 32 * w + 32, any);
                std::fill(g_state + 32 * w, g_state + 32 * w + 32, kReady);
                next = 32 * w;
            }
        if (next < 0 && spin < 0) return 1;
        if (next < 0) {  // only waits are left: they go on until they run out
            g_clock += pt::kExchangeWaitCycles / 2;
            next = spin;
            for (int t = 0; t < g_threads; ++t)
                if (g_state[t] == kSpin) g_state[t] = kReady;
        }
        g_cur = next;
        swapcontext(&g_main, &g_thread[next]);
        if (g_broken) return 2;
    }
    *gave_up = g_ns.abort_;
    return 0;
}

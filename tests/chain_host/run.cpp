// The chain kernel's control flow on the host: its own source (chain.inc is csrc/pf_chain.cu, with the few instructions that matter here
// redirected), every thread of a CTA a coroutine, its mbarriers and named barriers modelled, its data not.  Shows whether every CTA ends
// by itself when waits run out: `run CONFIG [WARP N] [copy M]`, in which the N-th wait of that warp gives up at once and the M-th copy never lands.
// Other bounded waits run out only when nothing else can go on, the longest one first.  Prints the status word; exit code 0: every CTA
// ended, 1: one hangs, 2: a barrier was used wrongly.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <float.h>
#include <math.h>
#include <stdint.h>
#include <stdio.h>
#include <stdlib.h>
#include <string.h>
#include <ucontext.h>
#include <unistd.h>

#include <algorithm>
#include <atomic>
#include <map>
#include <set>
#include <string>
#include <vector>

namespace host {
enum State { READY, MBAR, NAMED, DONE };
struct Thread {
    ucontext_t ctx;
    State state;
    uint32_t bar;           // MBAR: which, and the parity waited for
    int id, parity, waits;
    long since;
    bool gave_up;
};
struct Mbar { int count, pending, phase; };
struct Named {
    int n = 0, arrived = 0;
    std::set<int> who;
    std::vector<int> waiting;
};
std::vector<Thread> threads;
std::map<uint32_t, Mbar> mbars;
std::map<int, Named> named_bars;
ucontext_t scheduler;
int self, give_up_warp = -1, give_up_wait = -1, lost_copy = -1, copies;
long now;

int lane() { return self & 31; }
void fail(int code, const char* what, int id) {
    printf("%s: barrier %d, thread %d (warp %d)\n", what, id, self, self / 32);
    fflush(stdout);
    _exit(code);                        // (this may be a coroutine, on a stack that exit would free)
}
void yield() { swapcontext(&threads[self].ctx, &scheduler); }
void mbar_init(uint32_t bar, int count) { mbars[bar] = {count, count, 0}; }
void mbar_arrive(uint32_t bar) {
    if (!mbars.count(bar)) fail(2, "no such mbarrier", (int)bar);
    Mbar& m = mbars[bar];
    if (--m.pending > 0) return;
    m.pending = m.count;
    m.phase ^= 1;
    for (Thread& t : threads)
        if (t.state == MBAR && t.bar == bar && t.parity != m.phase) t.state = READY;
}
void landed(uint32_t bar) {
    if (copies++ != lost_copy) mbar_arrive(bar);
}
// (the phase with parity p is complete when the present one has the other)
bool mbar_wait(uint32_t bar, int parity, bool patient) {
    Thread& t = threads[self];
    if (self / 32 == give_up_warp && t.waits++ == give_up_wait) return false;
    if (!mbars.count(bar)) fail(2, "no such mbarrier", (int)bar);
    if (mbars[bar].phase != parity) return true;
    if (!patient) return false;
    t.state = MBAR; t.bar = bar; t.parity = parity; t.since = now++; t.gave_up = false;
    yield();
    return !threads[self].gave_up;
}
void named(int id, int n, bool wait) {
    Named& b = named_bars[id];
    if (b.arrived == 0) b.n = n;
    if (b.n != n) fail(2, "another number of threads is expected", id);
    if (!b.who.insert(self).second) fail(2, "arrived at twice by one thread", id);
    if (++b.arrived == n) {
        b.arrived = 0;
        b.who.clear();
        for (int t : b.waiting) threads[t].state = READY;
        b.waiting.clear();
        return;
    }
    if (!wait) return;
    b.waiting.push_back(self);
    threads[self].state = NAMED; threads[self].id = id;
    yield();
}
long long clock64() { static long long t = 0; return t += 600000000ll; }
}  // namespace host

struct Dim { unsigned x, y; };
static Dim threadIdx, blockIdx, gridDim;
alignas(1024) static uint8_t host_smem[228 * 1024];
#undef __shared__
#undef __global__
#undef __device__
#undef __host__
#undef __forceinline__
#undef __noinline__
#undef __launch_bounds__
#undef __grid_constant__
#define __shared__ static
#define __global__
#define __device__
#define __host__
#define __forceinline__ inline
#define __launch_bounds__(...)
#define __grid_constant__
#define __syncthreads() host::named(0, pf::host_threads, true)
#define __syncwarp() ((void)0)
#define __threadfence() ((void)0)
#define __shfl_xor_sync(m, x, o) (x)
#define __all_sync(m, x) (x)
#define clock64() host::clock64()
template <class T> T atomicCAS(T* p, T a, T b) { const T old = *p; if (old == a) *p = b; return old; }
template <class T> T atomicAdd(T* p, T b) { const T old = *p; *p += b; return old; }
template <class T> T atomicOr(T* p, T b) { const T old = *p; *p |= b; return old; }
static float __uint_as_float(uint32_t x) { float y; memcpy(&y, &x, 4); return y; }
static uint32_t __float_as_uint(float x) { uint32_t y; memcpy(&y, &x, 4); return y; }
using std::max;
using std::min;
namespace pf { static int host_threads; }
#define asm
#define volatile(...)
#include "chain.inc"
#undef volatile
#undef asm

using namespace pf;

static void (*body)();
static void entry() {
    body();
    host::threads[host::self].state = host::DONE;
    host::yield();
}
static void run_cta(int threads) {
    using namespace host;
    host_threads = threads;
    host::threads.assign(threads, Thread{});
    mbars.clear();
    named_bars.clear();
    static std::vector<char> stacks;
    constexpr size_t STACK = 48 << 10;
    stacks.resize(threads * STACK);
    for (int t = 0; t < threads; ++t) {
        Thread& x = host::threads[t];
        getcontext(&x.ctx);
        x.ctx.uc_stack.ss_sp = stacks.data() + t * STACK;
        x.ctx.uc_stack.ss_size = STACK;
        x.ctx.uc_link = nullptr;
        makecontext(&x.ctx, entry, 0);
    }
    for (;;) {
        bool ran = false;
        for (int t = 0; t < threads; ++t)
            if (host::threads[t].state == READY) {
                ran = true;
                self = t;
                threadIdx.x = (unsigned)t;
                swapcontext(&scheduler, &host::threads[t].ctx);
            }
        if (ran) continue;
        int first = -1, open = 0;
        for (int t = 0; t < threads; ++t) {
            const Thread& x = host::threads[t];
            open += x.state != DONE;
            if (x.state == MBAR && (first < 0 || x.since < host::threads[first].since)) first = t;
        }
        if (!open) return;
        if (first < 0) {
            for (int t = 0; t < threads; t += 32)
                if (host::threads[t].state == NAMED) printf("warp %d waits at named barrier %d\n", t / 32, host::threads[t].id);
            fail(1, "hangs", -1);
        }
        for (int t = first & ~31; t < (first | 31) + 1; ++t)            // (a warp gives up as a whole)
            if (host::threads[t].state == MBAR && host::threads[t].bar == host::threads[first].bar) {
                host::threads[t].state = READY;
                host::threads[t].gave_up = true;
            }
    }
}

static ChainMaps maps;
static ChainGeo geo;
static ChainSeg segs;
static std::vector<float> out, state, hand;
static std::vector<uint16_t> in;
static std::vector<int> flags;
static int status_word;

// nseq sequences of nblk blocks; MODE SHARED: over `ctas` CTAs, which run one after another (who waits for another's state has the higher index)
template <int DK, int R, int DV, int MODE>
static void run_walks(int nseq, int nblk, int ctas) {
    const int L = nblk * (NB / R) - 1;
    in.assign((size_t)nseq * L * R * 128, 0);
    out.assign((size_t)nseq * L * DV, 0.f);
    state.assign((size_t)nseq * DK * DV, 0.f);
    hand.assign((size_t)ctas * DK * DV, 0.f);
    flags.assign(2 * ctas, 0);
    geo = {};
    geo.L = L; geo.d_v = DV; geo.nblk = geo.seg_blk = geo.first_blk = nblk; geo.nseg = 1; geo.rm = R;
    geo.total = nseq * nblk; geo.share = (geo.total + ctas - 1) / ctas;
    geo.hand = hand.data(); geo.handed = flags.data(); geo.finished = flags.data() + ctas;
    geo.q = geo.k = geo.v = geo.beta = (const __nv_bfloat16*)in.data();
    geo.S0 = state.data(); geo.O = out.data(); geo.S_final = state.data();
    gridDim.x = (unsigned)ctas;
    body = [] { chain_kernel<DK, R, DV, MODE>(maps, geo.beta, geo.S0, geo.O, geo.S_final, &status_word, geo, segs); };
    for (int x = 0; x < ctas; ++x) {
        blockIdx.x = (unsigned)x;
        run_cta(CHAIN_THREADS);
    }
}
static void run_config(int c) {
    switch (c) {
        case 0: return run_walks<128, 2, 128, WHOLE>(1, 5, 1);
        case 1: return run_walks<64, 1, 64, WHOLE>(1, 7, 1);
        case 2: return run_walks<128, 3, 64, WHOLE>(1, 6, 1);
        case 3: return run_walks<128, 1, 128, SHARED>(3, 4, 2);
        case 4: return run_walks<64, 4, 64, SHARED>(3, 5, 2);
        default: exit(3);
    }
}

int main(int argc, char** argv) {
    for (int x = 2; x + 1 < argc; x += 2) {
        if (!strcmp(argv[x], "copy")) host::lost_copy = atoi(argv[x + 1]);
        else { host::give_up_warp = atoi(argv[x]); host::give_up_wait = atoi(argv[x + 1]); }
    }
    run_config(atoi(argv[1]));
    printf("status %d\n", status_word);
    return 0;
}

// One CTA of the persistent wide batch kernel on the CPU (test support only):
// the kernel's own text (KERNEL_TEXT, cut out of csrc/qs_wide.cu) is compiled
// with one host thread per CUDA thread.  __shared__ variables are statics, and
// the barrier names the line it is called from, so threads that meet at
// different barriers are seen.  After every barrier all threads but the first
// are held up for a while: what they then still read of the shared item has to
// survive thread 0 running ahead to the next barrier.  The items' bodies are
// replaced by records of what each thread was asked to run.
#include <atomic>
#include <chrono>
#include <condition_variable>
#include <cstdio>
#include <cstdlib>
#include <mutex>
#include <random>
#include <thread>
#include <vector>

#include "../paper_1608_00263_gb300/csrc/qs_internal.h"

using namespace qs;

struct float2 { float x, y; };
struct float4 { float x, y, z, w; };
static float4 make_float4(float x, float y, float z, float w) { return {x, y, z, w}; }
static const int kStatAcc = 12, kWideThreads = 16;
struct WideSmem {};
struct WideFoldSmem {};
struct Index { unsigned x; };
static thread_local Index threadIdx;
static const Index blockDim = {kWideThreads};

static void fail(const char *what, int a, int b)
{
    std::printf("%s: %d, %d\n", what, a, b);
    std::fflush(stdout);
    std::_Exit(1);
}

static void cta_barrier(int line)
{
    static std::mutex mu;
    static std::condition_variable cv;
    static int arrived = 0, at = 0, generation = 0;
    static thread_local std::mt19937 rng(threadIdx.x + 1);
    {
        std::unique_lock<std::mutex> lock(mu);
        if (arrived == 0) at = line;
        if (at != line) fail("threads at different barriers, lines", at, line);
        if (++arrived == kWideThreads) {
            arrived = 0;
            ++generation;
            cv.notify_all();
        } else {
            const int mine = generation;
            cv.wait(lock, [&] { return generation != mine; });
        }
    }
    if (threadIdx.x) std::this_thread::sleep_for(std::chrono::microseconds(rng() % 400));
}

struct Ran { uint32_t kind_pass, lo, hi; };
static std::vector<Ran> ran[kWideThreads];

static uint32_t atomicAdd(uint32_t *p, uint32_t v) { return __atomic_fetch_add(p, v, __ATOMIC_SEQ_CST); }
static void atomicExch(uint32_t *p, uint32_t v) { __atomic_store_n(p, v, __ATOMIC_SEQ_CST); }
static void __threadfence() { std::atomic_thread_fence(std::memory_order_seq_cst); }
static double __ldcg(const double *p) { return *p; }
// (one CTA takes the items in order, so an item's dependencies are complete)
static int flag_wait_bounded(const uint32_t *count, uint32_t target, const uint32_t *, uint64_t)
{
    return __atomic_load_n(count, __ATOMIC_SEQ_CST) >= target ? 0 : 1;
}

static const WidePass *pass_base;
template <int THREADS, bool BATCHED>
static void batch_stats_chunk(const float2 *, uint64_t cnt, float, double *dst)
{
    ran[threadIdx.x].push_back({kPersistStats, (uint32_t)cnt, 0});
    cta_barrier(-1);
    if (threadIdx.x < (unsigned)kStatAcc) dst[threadIdx.x] = (double)cnt * (threadIdx.x + 1);
}
template <int KIND, int FOLD, int GROUPED>
static void wide_pass_body(float2 *, const WidePass *pass, const WideOp *, const uint8_t *, uint32_t lo, uint32_t hi,
                           WideSmem &, WideFoldSmem *, unsigned char *, uint64_t, const FoldArgs *)
{
    ran[threadIdx.x].push_back({1000u + (uint32_t)(pass - pass_base), lo, hi});
    cta_barrier(-2);
}

#define __global__ static
#define __device__ static
#define __forceinline__ inline
#define __restrict__
#define __launch_bounds__(...)
#define __shared__ static
#define __syncthreads() cta_barrier(__LINE__)
#include KERNEL_TEXT

int main()
{
    // per instance: an initial chunk, passes, statistics chunks; an instance's
    // items wait for its earlier ones
    const int kInst = 6;
    std::vector<PersistItem> items;
    std::vector<uint32_t> before(kInst, 0);
    std::vector<double> want(kInst * kStatAcc, 0.0);
    std::vector<float2> amps(64 * kInst);
    uint32_t slots = 0, passes = 0;
    auto add = [&](uint32_t kind, int i) -> PersistItem & {
        PersistItem w{};
        w.kind = kind;
        w.inst = (uint32_t)i;
        w.amp_off = 64u * (uint32_t)i;
        w.need = before[i];
        w.lo = 16;
        items.push_back(w);
        return items.back();
    };
    for (int i = 0; i < kInst; ++i) {
        const size_t first = items.size();
        const uint32_t slot0 = slots, npass = 1 + (uint32_t)i % 3, nstat = i == 4 ? 35 : 1 + (uint32_t)i % 2;
        add(kPersistInit, i);
        ++before[i];
        for (uint32_t p = 0; p < npass; ++p) {
            PersistItem &w = add(p & 1 ? kPersistPassFull : kPersistPass, i);
            w.pass = passes++;
            w.lo = p;
            w.hi = p + 5;
            ++before[i];
        }
        for (uint32_t p = 0; p < nstat; ++p) {
            PersistItem &w = add(kPersistStats, i);
            w.lo = 3 + p + (uint32_t)i;
            w.pass = slots++;
            w.hi = slot0;
            w.nslots = nstat;
            for (int k = 0; k < kStatAcc; ++k) want[i * kStatAcc + k] += (double)w.lo * (k + 1);
        }
        for (size_t j = first; j < items.size(); ++j) items[j].total = (uint32_t)(items.size() - first);
    }
    std::vector<WidePass> pass(passes);
    pass_base = pass.data();
    std::vector<double> part(slots * kStatAcc), sums(kInst * kStatAcc);
    std::vector<uint32_t> done(kInst);
    PersistCtl ctl{};
    std::vector<std::thread> threads;
    for (int t = 0; t < kWideThreads; ++t)
        threads.emplace_back([&, t] {
            threadIdx.x = (unsigned)t;
            k_batch_persistent_wide<true, 2>(amps.data(), items.data(), (int)items.size(), pass.data(), nullptr, nullptr,
                                             nullptr, done.data(), &ctl, part.data(), sums.data(), 0);
        });
    for (std::thread &t : threads) t.join();
    if (ctl.err || ctl.abort) fail("a wait ran out", (int)ctl.err, (int)ctl.abort);
    for (int t = 0; t < kWideThreads; ++t) {
        size_t k = 0;
        for (const PersistItem &w : items) {
            if (w.kind == kPersistInit) continue;
            if (k >= ran[t].size()) fail("items left out by thread", t, (int)k);
            const Ran &r = ran[t][k++];
            const bool same = w.kind == kPersistStats ? r.kind_pass == kPersistStats && r.lo == w.lo
                                                      : r.kind_pass == 1000u + w.pass && r.lo == w.lo && r.hi == w.hi;
            if (!same) fail("another item run by thread", t, (int)k - 1);
        }
        if (k != ran[t].size()) fail("items too many for thread", t, (int)ran[t].size());
    }
    for (size_t k = 0; k < want.size(); ++k)
        if (sums[k] != want[k]) fail("sum", (int)k, (int)sums[k]);
    std::printf("ok\n");
    return 0;
}

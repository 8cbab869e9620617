// core.cu -- core ordering (Algorithm OrdCore, Sec. III) computed in synchronous peeling rounds.
//
// Each round first raises the level to the smallest remaining degree (the level never falls),
// then removes every remaining vertex whose remaining degree is at most the level, all together,
// and only then lowers the remaining degrees of their neighbours.  rank orders the vertices by
// (removal round, id).  A vertex's later neighbours were all present when its round began, so its
// out-degree is at most that round's level and the maximum out-degree is the degeneracy -- the
// property the paper wants from the core ordering (Sec. III, Table II) -- while the rounds run in
// parallel instead of one vertex per step.
//
// One cooperative persistent kernel runs every round, one block per SM.  What bounds it is the
// latency of a round (R-MAT 20: 670 rounds of about 1.6 k vertices and 47 k arcs each): the grid
// barriers and the chains of dependent L2 accesses between them, so a round does as few of both as
// it can.
//   - The frontier is kept as two lists in one array, rows of at most kLongRow arcs from the front and
//     longer ones from the back.  A warp takes one or more short rows and walks their arcs as one
//     sequence; a long row is cut into units of kLongRow arcs over the warps of the block (of the
//     whole grid when there are few).  One warp per vertex left a hub's row to a single warp.
//   - A neighbour whose degree falls from level + 1 to level joins the next frontier (only one
//     decrement can make that step, so it is pushed exactly once).
//   - A round that leaves no frontier raises the level.  The smallest remaining degree is then above
//     the level, nearly always level + 1, so one pass over the remaining vertices collects those of
//     degree level + 1 and, for the case that there are none, finds the smallest degree.
//   - The remaining vertices are a list that is compacted whenever half of it is gone, and blocks
//     leave when the list no longer needs them: fewer blocks make cheaper barriers.
// Rounds are separated by a grid barrier whose wait is bounded in time.  The ranks then come from
// the stable radix sort of the ids by round (sort.cu).
// R-MAT 20 (655 rounds): 18.5 ms with one warp per vertex, three barriers and two passes over all
// vertices per level raise; 9.2 ms with the above (8, 16 and 48 blocks to the end: 9.7, 9.2, 9.0), 7.9 ms
// with the barrier's round trips cut.  Chung-Lu 1M (1,367 rounds): 42.5 -> 14.4 ms.
#include <cuda/atomic>
#include <cuda_runtime.h>
#include <stdint.h>

#include "common.cuh"

namespace citron {

// round_of[] of a vertex not removed yet: its row has at most kLongRow arcs, or more
constexpr uint32_t kPresent = 0xffffffffu, kPresentLong = 0xfffffffeu;
__device__ __forceinline__ bool present(uint32_t r) { return r >= kPresentLong; }
constexpr int kCoreThreads = 1024;
constexpr uint32_t kLongRow = 256;      // arcs of a unit; longer rows are cut
constexpr uint32_t kCoreMinBlocks = 16;  // blocks that stay to the end
constexpr unsigned long long kGridWaitNs = 4000000000ull;  // 4 s per barrier at most

struct CoreState {
    unsigned int arrived;  // blocks that arrived at a barrier, over all barriers
    unsigned int pad;
    unsigned int cnt[3];  // short rows of the frontier, ring over rounds (round t's in cnt[t % 3])
    unsigned int lng[3];  // long rows of the frontier, likewise
    unsigned int raised[2], raised_lng[2];  // frontier of a level raise's first pass, by turns
    unsigned int alive[2];  // vertices in the compacted list being written, likewise
    unsigned int gmin[2];   // smallest remaining degree, likewise
    unsigned int rounds;
    unsigned int level;
};

__device__ __forceinline__ uint32_t load_relaxed(unsigned int *p)
{
    cuda::atomic_ref<unsigned int, cuda::thread_scope_device> r(*p);
    return r.load(cuda::memory_order_relaxed);
}

// Barrier over the first `blocks` blocks of a cooperative launch (all of them resident); `due` counts
// the arrivals up to it.  Returns false on every thread of the block when the wait (at most wait_ns)
// gave up or some block has reported an error, so that the kernel can return; the other blocks then
// give up at their next barrier.  The thread that waited also reads the words p[0..N) that the
// round needs next, in the same round trip as the error word, for the whole block.
template <int N>
__device__ bool grid_barrier(CoreState *s, uint32_t blocks, uint32_t &due, uint32_t *err,
                             unsigned long long wait_ns, unsigned int *const (&p)[N], uint32_t (&out)[N])
{
    __shared__ int s_ok;
    __shared__ uint32_t s_out[N];
    due += blocks;
    __syncthreads();
    if (threadIdx.x == 0) {
        cuda::atomic_ref<unsigned int, cuda::thread_scope_device> arrived(s->arrived);
        __threadfence();
        int ok = 1;
        arrived.fetch_add(1u, cuda::memory_order_acq_rel);
        const unsigned long long t0 = global_ns();
        uint32_t spins = 0;
        while ((int32_t)(arrived.load(cuda::memory_order_acquire) - due) < 0) {
            if ((++spins & 63u) == 0 && global_ns() - t0 > wait_ns) {
                set_error(err, kDevTimeout);
                ok = 0;
                break;
            }
        }
        __threadfence();
        const uint32_t e = load_relaxed(err);
        uint32_t v[N];
#pragma unroll
        for (int i = 0; i < N; i++) v[i] = load_relaxed(p[i]);
        if (e) ok = 0;
        s_ok = ok;
#pragma unroll
        for (int i = 0; i < N; i++) s_out[i] = v[i];
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < N; i++) out[i] = s_out[i];
    return s_ok != 0;
}

// Frontier lists of one round in one array of n entries: short rows from the front, long from the
// back (a vertex is in one of them once, so they never meet).
struct Frontier {
    uint32_t *v;
    unsigned int *cnt, *lng;
};

// Adds the vertices of the lanes with take set (the whole warp calls this).
__device__ __forceinline__ void push(const Frontier &f, uint32_t n, bool take, uint32_t v, bool is_long, int lane)
{
    const uint32_t any = __ballot_sync(kFull, take);
    if (!any) return;
    const bool lng = take && is_long;
    const uint32_t lm = __ballot_sync(kFull, lng), sm = any & ~lm;
    uint32_t base = 0;
    if (lane == 0 && sm) base = atomicAdd(f.cnt, (unsigned)__popc(sm));
    if (lane == 1 && lm) base = atomicAdd(f.lng, (unsigned)__popc(lm));
    const uint32_t sb = __shfl_sync(kFull, base, 0), lb = __shfl_sync(kFull, base, 1);
    if (take && !lng) __stcg(f.v + sb + __popc(sm & lanemask_lt()), v);
    if (lng) __stcg(f.v + (n - 1 - (lb + __popc(lm & lanemask_lt()))), v);
}

__global__ __launch_bounds__(kCoreThreads) void k_core_peel(
    uint32_t n, uint64_t arcs, const uint64_t *__restrict__ off, const uint32_t *__restrict__ cols,
    uint32_t *cur, uint32_t *round_of, uint32_t *fa, uint32_t *fb, uint32_t *la, uint32_t *lb, CoreState *s,
    uint32_t *err, unsigned long long wait_ns, uint32_t absent_block)
{
    // injected fault (tests only): this block never arrives at the first barrier, so that the
    // other blocks' bounded wait there must run out
    if (blockIdx.x == absent_block) return;
    uint32_t blocks = gridDim.x;
    const uint32_t tid = blockIdx.x * blockDim.x + threadIdx.x;
    const uint32_t lane = threadIdx.x & 31, w = threadIdx.x >> 5, gwarp = tid >> 5;
    constexpr uint32_t kWarps = kCoreThreads / 32;
    const bool leader = blockIdx.x == 0 && threadIdx.x == 0;

    for (uint32_t v = tid; v < n; v += blocks * kCoreThreads) {
        const uint64_t a = off[v], b = off[v + 1];
        if (b < a || b > arcs) set_error(err, kDevBadInput);
        const uint32_t d = b >= a ? (uint32_t)(b - a) : 0u;
        cur[v] = d;
        round_of[v] = d > kLongRow ? kPresentLong : kPresent;
    }
    if (leader) s->gmin[0] = s->gmin[1] = kPresent;
    uint32_t due = 0;
    {
        unsigned int *const p[1] = {&s->rounds};
        uint32_t out[1];
        if (!grid_barrier(s, blocks, due, err, wait_ns, p, out)) return;
    }

    uint32_t t = 0, level = 0, removed = 0, f = 0, fl = 0, turn = 0;
    uint32_t *F = fa, *N = fb;
    // the remaining vertices are among list[0 .. len) (NULL: all ids)
    uint32_t *list = nullptr, *spare = la;
    uint32_t len = n;
    while (removed < n) {
        if (f + fl == 0) {
            // The smallest remaining degree is above the level (only in round 0 it can be the
            // level itself): take the vertices of the next degree, and in a second pass, if there
            // are none, those of the smallest.
            uint32_t want = t == 0 ? level : level + 1;
            const bool pack = n - removed <= len / 2;
            for (int pass = 0; pass < 2; pass++) {
                // (counters of their own for either pass: a block may still be reading the first's
                // when another is in the second)
                const Frontier now = {F, pass ? &s->cnt[t % 3] : &s->raised[turn],
                                      pass ? &s->lng[t % 3] : &s->raised_lng[turn]};
                uint32_t least = kPresent;
                for (uint32_t i0 = tid - lane; i0 < len; i0 += blocks * kCoreThreads) {
                    const uint32_t i = i0 + lane;
                    bool take = false, stay = false;
                    uint32_t v = 0, r = 0;
                    if (i < len) {
                        v = list ? __ldcg(list + i) : i;
                        r = __ldcg(round_of + v);
                        const uint32_t c = __ldcg(cur + v);
                        if (present(r)) {
                            take = c <= want;
                            stay = !take;
                            if (stay) least = min(least, c);
                        }
                    }
                    push(now, n, take, v, r == kPresentLong, lane);
                    if (take) __stcg(round_of + v, t);
                    if (pack && pass == 0) {  // (pass 0 takes none when there is a second pass)
                        const uint32_t mask = __ballot_sync(kFull, stay);
                        uint32_t base = 0;
                        if (lane == 0 && mask) base = atomicAdd(&s->alive[turn], (unsigned)__popc(mask));
                        base = __shfl_sync(kFull, base, 0);
                        if (stay) __stcg(spare + base + __popc(mask & lanemask_lt()), v);
                    }
                }
                if (pass == 0) {
                    least = __reduce_min_sync(kFull, least);
                    if (lane == 0 && least < load_relaxed(&s->gmin[turn])) atomicMin(&s->gmin[turn], least);
                }
                unsigned int *const p[4] = {now.cnt, now.lng, &s->alive[turn], &s->gmin[turn]};
                uint32_t out[4];
                if (!grid_barrier(s, blocks, due, err, wait_ns, p, out)) return;
                f = out[0];
                fl = out[1];
                if (pass == 0 && pack) {
                    len = out[2];
                    uint32_t *was = list;
                    list = spare;
                    spare = was ? was : lb;
                }
                if (f + fl != 0) break;
                want = out[3];
                if (pass == 1 || want == kPresent) {  // nothing left although removed < n: bad input
                    set_error(err, kDevBadInput);
                    return;
                }
            }
            level = max(level, want);
            turn ^= 1;
            if (leader) {  // the next raise's words: last read two raises ago
                s->gmin[turn] = kPresent;
                s->alive[turn] = s->raised[turn] = s->raised_lng[turn] = 0;
            }
            if (f + fl > n - removed) {
                set_error(err, kDevBadInput);
                return;
            }
        }
        // Remove the frontier: lower the degrees of the neighbours still present.
        if (leader) {
            s->cnt[(t + 2) % 3] = 0;  // last read at the start of round t - 1
            s->lng[(t + 2) % 3] = 0;
        }
        const Frontier nxt = {N, &s->cnt[(t + 1) % 3], &s->lng[(t + 1) % 3]};
        // four neighbours per lane (in: which of them are arcs)
        auto drop = [&](const uint32_t (&x)[4], const bool (&in)[4]) {
            uint32_t r[4];
#pragma unroll
            for (int h = 0; h < 4; h++) {
                r[h] = 0;
                if (in[h]) {
                    if (x[h] < n) r[h] = __ldcg(round_of + x[h]);
                    else set_error(err, kDevBadInput);
                }
            }
            bool hit[4];
#pragma unroll
            for (int h = 0; h < 4; h++) hit[h] = present(r[h]) && atomicSub(cur + x[h], 1u) == level + 1;
#pragma unroll
            for (int h = 0; h < 4; h++) {
                push(nxt, n, hit[h], x[h], r[h] == kPresentLong, lane);
                if (hit[h]) __stcg(round_of + x[h], t + 1);
            }
        };
        // short rows: as many per warp as it takes (one while there are warps enough, at most 32), as one
        // sequence of arcs, four arcs per lane in flight
        const uint32_t per = min(max(f / (blocks * kWarps), 1u), 32u);
        // (one row per warp needs no sequence: rounds of a few vertices, of which a path has n / 2, are
        // all latency; a path of 4,000 7.7 -> 7.2 ms, R-MAT 18 3.9 -> 3.8)
        for (uint32_t i = gwarp; per == 1 && i < f; i += blocks * kWarps) {
            const uint32_t v = __ldcg(F + i);
            const uint64_t a = off[v];
            const uint32_t d = (uint32_t)(min(off[v + 1], arcs) - a);
            for (uint32_t e0 = 0; e0 < d; e0 += 128) {
                uint32_t x[4];
                bool in[4];
#pragma unroll
                for (int h = 0; h < 4; h++) {
                    const uint32_t e = e0 + 32 * h + lane;
                    in[h] = e < d;
                    x[h] = in[h] ? cols[a + e] : 0u;
                }
                drop(x, in);
            }
        }
        for (uint32_t i0 = per == 1 ? f : gwarp * per; i0 < f; i0 += blocks * kWarps * per) {
            uint64_t a = 0;
            uint32_t d = 0;
            if (lane < per && i0 + lane < f) {
                const uint32_t v = __ldcg(F + i0 + lane);
                a = off[v];
                d = (uint32_t)(min(off[v + 1], arcs) - a);
            }
            const uint32_t incl = warp_incl_scan(d), excl = incl - d, total = __shfl_sync(kFull, incl, 31);
            for (uint32_t e0 = 0; e0 < total; e0 += 128) {
                uint32_t x[4];
                bool in[4];
#pragma unroll
                for (int h = 0; h < 4; h++) {
                    const uint32_t e = e0 + 32 * h + lane;
                    uint32_t o = 0;  // the last lane whose sequence starts at or before e
#pragma unroll
                    for (uint32_t step = 16; step > 0; step >>= 1)
                        if (__shfl_sync(kFull, excl, o + step) <= e) o += step;
                    const uint64_t ao = __shfl_sync(kFull, a, o);
                    const uint32_t eo = __shfl_sync(kFull, excl, o);
                    in[h] = e < total;
                    x[h] = in[h] ? cols[ao + (e - eo)] : 0u;
                }
                drop(x, in);
            }
        }
        // long rows: units of kLongRow arcs over the block's warps, or over all when they are few
        const bool few = fl <= 64;
        for (uint32_t i0 = few ? 0u : blockIdx.x * 32; i0 < fl; i0 += few ? 32u : blocks * 32) {
            uint64_t a = 0;
            uint32_t d = 0;
            if (i0 + lane < fl) {
                const uint32_t v = __ldcg(F + (n - 1 - (i0 + lane)));
                a = off[v];
                d = (uint32_t)(min(off[v + 1], arcs) - a);
            }
            const uint32_t units = (d + kLongRow - 1) / kLongRow;
            const uint32_t incl = warp_incl_scan(units), excl = incl - units, total = __shfl_sync(kFull, incl, 31);
            for (uint32_t u = few ? gwarp : w; u < total; u += few ? blocks * kWarps : kWarps) {
                const int o = __popc(__ballot_sync(kFull, incl <= u));
                const uint64_t ao = __shfl_sync(kFull, a, o);
                const uint32_t e0 = (u - __shfl_sync(kFull, excl, o)) * kLongRow, len_o = __shfl_sync(kFull, d, o);
#pragma unroll
                for (uint32_t q = 0; q < kLongRow; q += 128) {
                    uint32_t x[4];
                    bool in[4];
#pragma unroll
                    for (int h = 0; h < 4; h++) {
                        const uint32_t e = e0 + q + 32 * h + lane;
                        in[h] = e < len_o;
                        x[h] = in[h] ? cols[ao + e] : 0u;
                    }
                    drop(x, in);
                }
            }
        }
        removed += f + fl;
        t++;
        {
            unsigned int *const p[2] = {&s->cnt[t % 3], &s->lng[t % 3]};
            uint32_t out[2];
            if (!grid_barrier(s, blocks, due, err, wait_ns, p, out)) return;
            f = out[0];
            fl = out[1];
        }
        if (f + fl > n - removed) {
            set_error(err, kDevBadInput);
            return;
        }
        uint32_t *tmp = F;
        F = N;
        N = tmp;
        // blocks that the remaining vertices do not need leave
        const uint32_t need = max(kCoreMinBlocks, (n - removed + kCoreThreads - 1) / kCoreThreads);
        if (need <= blocks / 2) {
            blocks = need;
            if (blockIdx.x >= blocks) return;
        }
    }
    if (leader) {
        s->rounds = t;
        s->level = level;
    }
}

}  // namespace citron

namespace citron_host {

using namespace citron;

cudaError_t launch_rank_by_key(uint32_t n, const uint32_t *keys, uint32_t key_bound, uint32_t *rank,
                               uint32_t *perm, uint32_t *err, Carver &c, cudaStream_t st);
size_t order_ws_bytes(uint32_t n);

size_t core_ws_bytes(uint32_t n)
{
    Sizer s;
    s.take<CoreState>(1);
    for (int i = 0; i < 4; i++) s.take<uint32_t>((size_t)n + 1);  // cur, round_of, two frontiers
    return s.used + order_ws_bytes(n);
}

// Synchronous: the round count sizes the radix sort.  Device errors land in err.
cudaError_t launch_core_order(uint32_t n, uint64_t arcs, const uint64_t *off, const uint32_t *cols,
                              uint32_t *rank, uint32_t *perm, uint32_t *h_level,
                              uint32_t *h_rounds, uint32_t *err, Carver &c, cudaStream_t st,
                              int num_sms)
{
    CoreState *state = c.take<CoreState>(1);
    uint32_t *cur = c.take<uint32_t>((size_t)n + 1);
    uint32_t *round_of = c.take<uint32_t>((size_t)n + 1);
    uint32_t *fa = c.take<uint32_t>((size_t)n + 1);
    uint32_t *fb = c.take<uint32_t>((size_t)n + 1);
    // the lists of remaining vertices lie where the radix sort will keep its ids afterwards
    Carver later = c;
    uint32_t *la = later.take<uint32_t>(n), *lb = later.take<uint32_t>(n);
    if (!c.ok || !later.ok) return cudaErrorMemoryAllocation;
    if (h_level) *h_level = 0;
    if (h_rounds) *h_rounds = 0;
    if (n == 0) return cudaSuccess;
    int dev = 0, coop = 0, per_sm = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (!e) e = cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev);
    if (!e && !coop) return cudaErrorNotSupported;
    if (!e) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_core_peel, kCoreThreads, 0);
    if (!e && per_sm < 1) return cudaErrorLaunchOutOfResources;
    if (!e) e = cudaMemsetAsync(state, 0, sizeof(CoreState), st);
    if (e) return e;
    // One thread per vertex and one block per SM at most (fewer blocks make cheaper barriers), all
    // blocks resident.
    uint32_t grid = (n + kCoreThreads - 1) / kCoreThreads;
    if (grid > (uint32_t)num_sms) grid = (uint32_t)num_sms;
    const citron_faults f = injected_faults();
    unsigned long long wait_ns = f.barrier_wait_ns ? f.barrier_wait_ns : kGridWaitNs;
    uint32_t absent = f.barrier_absent_block ? f.barrier_absent_block - 1 : 0xffffffffu;
    void *args[] = {&n, &arcs, &off, &cols, &cur, &round_of, &fa, &fb, &la, &lb, &state, &err, &wait_ns, &absent};
    e = cudaLaunchCooperativeKernel((const void *)k_core_peel, dim3(grid), dim3(kCoreThreads), args,
                                    0, st);
    note_launches(1);
    if (e) return e;
    CoreState hs = {};
    uint32_t code = 0;
    e = cudaMemcpyAsync(&hs, state, sizeof(hs), cudaMemcpyDeviceToHost, st);
    if (!e) e = cudaMemcpyAsync(&code, err, sizeof(code), cudaMemcpyDeviceToHost, st);
    if (!e) e = cudaStreamSynchronize(st);
    if (e) return e;
    if (code) return cudaSuccess;  // reported from the error word by the caller
    if (h_level) *h_level = hs.level;
    if (h_rounds) *h_rounds = hs.rounds;
    return launch_rank_by_key(n, round_of, hs.rounds, rank, perm, err, c, st);
}

}  // namespace citron_host

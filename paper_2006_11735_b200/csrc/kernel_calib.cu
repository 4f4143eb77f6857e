// The n-sigma bound of Section 3.2.2 on the GPU: the smallest value among the largest
// `fraction` of an int32 feature map Y, i.e. its k-th largest element with
// k = max(1, ceil(count * fraction)), clamped to at least 1 (a BReLU bound is positive).
// It is the step right before the hot path: the bound h_ri it returns feeds Eq. 9-13
// (`iq_brelu_params`), which give the layer's mul, shift and h_i.
//
// Exact selection without sorting, Y read ONCE:
//   1. bracket   8192 keys at hashed positions; two order statistics of the sample, 4.5 standard
//                deviations around the rank, bracket the k-th largest of Y: [lo, hi], about 0.4 % of Y
//                at the usual fraction.
//   2. collect   one pass over Y: counts what lies above hi, at hi or above and at lo or above (so a value
//                that fills a bracket's end by itself, as a clamped map's bound, costs nothing) and keeps
//                what lies between.
//   3. settle    a radix select over the kept keys by one cluster of blocks.
// The result is exact because the ranks are counted, not estimated.  A sample that misled (the rank
// is outside the bracket, or more keys in it than the scratch keeps) is noticed, and a
// most-significant-byte radix select does the call instead: four passes, any input.
// The three launches overlap (programmatic dependent launch): while the bracket is being taken the pass has its first
// values on their way, the next ones as far as the L2 cache.
//
// 51.4 M normal values (206 MB), whole call: 63 us (100.5 before its parts were rebuilt, four radix passes 297).  Reading
// the tensor alone takes 37 to 39 us here, whatever the loads (4 or 8 vectors a thread, 296 to 592 blocks; bulk copies to shared memory 45).
// Kernel by kernel (apart, caches cold) the bracket takes 12 us (it was 21), the pass 41 (60), the settling 14 (11).
// Where the bracket misses, the call pays for it and the pass before the radix select.  Sorted values, of which a few blocks keep all that lies in
// the bracket, and a rank near the smallest of a large tensor (fraction 0.9) are 2 to 15 % slower than before, all else is faster.
#include <cmath>
#include <cstddef>
#include <mutex>

#include "plan.h"

namespace iconv {

namespace {

constexpr int CALIB_THREADS = 512;
constexpr int CALIB_WARPS = CALIB_THREADS / 32;
constexpr int SAMPLE = 8192;                     // keys sampled; a tensor no larger is selected from directly
constexpr int COLLECT_BLOCKS = 148 * 3;          // three blocks of 512 threads are resident on an SM: one wave
constexpr unsigned KEEP_BLOCK = 6144;            // keys of the bracket that a block keeps at most
constexpr int AHEAD = 3;                         // rounds of the pass that are asked for before the bracket is known (14.5 MB each, all blocks)
constexpr int COARSE_BITS = 9;                   // of a kept key: the histogram that a block of the pass takes
constexpr int COARSE = 1 << COARSE_BITS;
constexpr int BIN_BITS = 11;
constexpr int BINS = 1 << BIN_BITS;
// bracket and settle: one cluster of blocks
constexpr int CLUSTER = 8;
constexpr int CLUSTER_THREADS = 1024;
constexpr int CLUSTER_WARPS = CLUSTER_THREADS / 32;
static_assert(SAMPLE == CLUSTER * CLUSTER_THREADS, "");

enum { CALIB_DONE = 1, CALIB_MISS = 2 };

struct SelectOut {                               // in pinned host memory
    int result, status;
};

// Scratch of one call.  hist is zero between calls.
struct SelectState {
    unsigned long long hist[256];                // radix: keys of the prefix by their next byte
    unsigned long long k;                        // radix: rank (from the top, 1-based) still to find inside the prefix
    unsigned prefix, mask;                       // radix: key bits fixed so far
    unsigned lo, hi;                             // the bracket
    uint4 counts[COLLECT_BLOCKS];                // by each block of the pass: keys > hi, >= hi, >= lo; kept (more than KEEP_BLOCK: not all)
    unsigned coarse[COLLECT_BLOCKS][COARSE / 2]; // by each block: kept keys by their upper bits, two 16-bit counts a word
    unsigned keep[COLLECT_BLOCKS][KEEP_BLOCK];
};

__device__ __forceinline__ unsigned key_of(int32_t v) { return (unsigned)v ^ 0x80000000u; }     // order-preserving
__device__ __forceinline__ int bound_of(unsigned key)
{
    const int v = (int)(key ^ 0x80000000u);
    return v < 1 ? 1 : v;
}
__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ unsigned cluster_rank() { unsigned r; asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r)); return r; }
__device__ __forceinline__ void cluster_sync()
{
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// the word at p in the shared memory of block `rank` of the cluster
__device__ __forceinline__ unsigned ld_cluster(const void *p, unsigned rank)
{
    unsigned v;
    asm volatile("{ .reg .b32 a; mapa.shared::cluster.u32 a, %1, %2; ld.shared::cluster.u32 %0, [a]; }" : "=r"(v) : "r"(smem_u32(p)), "r"(rank) : "memory");
    return v;
}
__device__ __forceinline__ void st_cluster(void *p, unsigned rank, unsigned v)
{
    asm volatile("{ .reg .b32 a; mapa.shared::cluster.u32 a, %0, %1; st.shared::cluster.u32 [a], %2; }" ::"r"(smem_u32(p)), "r"(rank), "r"(v) : "memory");
}

// What a block needs to find the bin that holds a rank.
struct Finder {
    unsigned warp[CLUSTER_WARPS];
    unsigned bin, rank;
};
// The bin of `total` (from the top) that holds rank `want`, and the rank inside it: a thread adds up two neighbouring bins, a
// scan over the warp and the warps' sums gives what lies above them.  Whole block, in step before.
__device__ __forceinline__ void pick_bin(Finder &f, const unsigned *total, unsigned want, unsigned &bin, unsigned &rank)
{
    static_assert(BINS == 2 * CLUSTER_THREADS, "");
    const unsigned warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const unsigned top = BINS - 1 - 2 * threadIdx.x;
    const uint2 c = *(const uint2 *)&total[top - 1];               // (.y: the upper bin)
    const unsigned sum = c.x + c.y;
    unsigned inc = sum;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const unsigned o = __shfl_up_sync(0xffffffffu, inc, d);
        if (lane >= d) inc += o;
    }
    if (lane == 31) f.warp[warp] = inc;
    __syncthreads();
    const unsigned above = __reduce_add_sync(0xffffffffu, lane < warp ? f.warp[lane] : 0u) + inc - sum;
    if (above < want && want <= above + sum) {
        const bool upper = want <= above + c.y;
        f.bin = upper ? top : top - 1;
        f.rank = want - above - (upper ? 0u : c.y);
    }
    __syncthreads();
    bin = f.bin;
    rank = f.rank;
}

// Draws the sample and finds the bracket; with `whole` (no more keys than the sample holds) the sample is Y itself and
// its k-th largest key the answer.  One cluster draws, a key per thread (one block alone needs three times as long for the
// 8192 reads); its first block has the keys in its shared memory and goes on alone.  Ranks up to 32: each of its 32 warps
// has a key at least as large as the least of the warps' largest, so what is below that (99 keys in 100) is left out and the
// rest compared with one another.  Other ranks: a histogram of eleven bits a round.  12 us with cold caches; with a barrier
// for each bit instead, 21.
__global__ void __cluster_dims__(CLUSTER, 1, 1) __launch_bounds__(CLUSTER_THREADS)
bracket_kernel(const int32_t *__restrict__ y, unsigned long long count, unsigned long long k, int whole, unsigned rank_hi, unsigned rank_lo,
               SelectState *st, SelectOut *out)
{
    constexpr unsigned FEW = 512;
    __shared__ __align__(8) unsigned sample[SAMPLE];
    unsigned (*hist)[BINS] = (unsigned (*)[BINS])sample;       // once the keys are in registers: of the keys under either prefix, or the few that matter
    __shared__ Finder f;
    __shared__ unsigned s_warp[CLUSTER_WARPS], s_least, s_most, s_few, s_found[2];
    grid_dep_launch();
    const unsigned block = cluster_rank(), lane = threadIdx.x & 31;
    const unsigned n = whole ? (unsigned)count : (unsigned)SAMPLE;
    {
        const unsigned i = block * CLUSTER_THREADS + threadIdx.x;
        unsigned long long at = i;
        if (!whole) {
            unsigned h = (i + 1u) * 0x9E3779B9u;                     // (hashed: no stride of the tensor's layout shows in the sample)
            h ^= h >> 16; h *= 0x85EBCA6Bu; h ^= h >> 13; h *= 0xC2B2AE35u; h ^= h >> 16;
            at = (unsigned long long)(((unsigned __int128)count * h) >> 32);
        }
        const unsigned key = i < n ? key_of(y[at]) : 0u;
        cluster_sync();                                              // (the first block is there)
        st_cluster(&sample[i], 0, key);
        cluster_sync();
    }
    if (block != 0) return;
    auto there = [&](int j) { return (unsigned)j * CLUSTER_THREADS + threadIdx.x < n; };
    unsigned key[CLUSTER];                                           // (a missing key: 0)
    unsigned least = 0xffffffffu, most = 0;
#pragma unroll
    for (int j = 0; j < CLUSTER; ++j) {
        key[j] = sample[j * CLUSTER_THREADS + threadIdx.x];
        if (there(j)) least = min(least, key[j]);
        most = max(most, key[j]);
    }
    if (threadIdx.x == 0) { s_least = 0xffffffffu; s_most = 0; s_few = 0; }
    least = __reduce_min_sync(0xffffffffu, least);
    most = __reduce_max_sync(0xffffffffu, most);
    if (lane == 0) s_warp[threadIdx.x >> 5] = most;
    __syncthreads();
    const unsigned rank_of[2] = {whole ? (unsigned)k : max(1u, rank_hi), whole ? (unsigned)k : min(n, rank_lo)};
    unsigned found[2] = {0, 0};
    bool done = false;
    if (rank_of[1] <= CLUSTER_WARPS && rank_of[0] <= rank_of[1] && n == SAMPLE) {
        const unsigned floor = __reduce_min_sync(0xffffffffu, s_warp[lane]);
        unsigned *few = hist[0];
#pragma unroll
        for (int j = 0; j < CLUSTER; ++j)
            if (key[j] >= floor) {
                const unsigned at = atomicAdd(&s_few, 1u);
                if (at < FEW) few[at] = key[j];
            }
        __syncthreads();
        const unsigned m = s_few;
        done = m <= FEW;                                             // (more: a value that many keys share)
        if (done) {
            if (threadIdx.x < m) {
                const unsigned mine = few[threadIdx.x];
                unsigned above = 0, from = 0;
#pragma unroll 8
                for (unsigned j = 0; j < m; ++j) {
                    const unsigned v = few[j];
                    above += v > mine;
                    from += v >= mine;
                }
                if (above < rank_of[0] && rank_of[0] <= from) s_found[0] = mine;      // (equal keys write the same)
                if (above < rank_of[1] && rank_of[1] <= from) s_found[1] = mine;
            }
            __syncthreads();
            found[0] = s_found[0];
            found[1] = s_found[1];
        }
    }
    if (!done) {
        if (lane == 0) { atomicMin(&s_least, least); atomicMax(&s_most, most); }
        __syncthreads();
        // the bits in which the sample's keys differ, what the found keys begin with, and the ranks among the keys that begin so
        const unsigned diff = s_least ^ s_most;
        int left = diff ? 32 - __clz((int)diff) : 0;
        found[0] = found[1] = left >= 32 ? 0u : s_most & ~((1u << left) - 1u);
        unsigned rank[2] = {rank_of[0], rank_of[1]};
        while (left > 0) {
            const int w = min(left, BIN_BITS), s = left - w;
            const bool apart = found[0] != found[1];
            for (int b = (int)threadIdx.x; b < 2 * BINS; b += CLUSTER_THREADS) hist[0][b] = 0;
            __syncthreads();
#pragma unroll
            for (int j = 0; j < CLUSTER; ++j) {
                const unsigned d0 = key[j] ^ found[0], d1 = key[j] ^ found[1];       // (the prefixes' open bits are zero)
                if (there(j) && (left >= 32 || (d0 >> left) == 0)) atomicAdd(&hist[0][d0 >> s], 1u);
                if (there(j) && apart && (d1 >> left) == 0) atomicAdd(&hist[1][d1 >> s], 1u);
            }
            __syncthreads();
            unsigned bin[2];
            pick_bin(f, hist[0], rank[0], bin[0], rank[0]);
            __syncthreads();
            pick_bin(f, hist[apart ? 1 : 0], rank[1], bin[1], rank[1]);
            found[0] |= bin[0] << s;
            found[1] |= bin[1] << s;
            left = s;
        }
    }
    if (threadIdx.x == 0) {
        if (whole) {
            out->result = bound_of(found[0]);
            out->status = CALIB_DONE;
        } else {
            st->hi = rank_hi < 1 ? 0xffffffffu : found[0];
            st->lo = rank_lo > n ? 0u : found[1];
        }
    }
}

// Bits below the bin of a kept key (they are 0 ... inside - 1) in the blocks' histograms.
__device__ __forceinline__ int coarse_shift(unsigned inside) { return inside > 1 ? max(0, 32 - __clz((int)(inside - 1u)) - COARSE_BITS) : 0; }

// The one pass over Y, bound by its read where the tensor is large.  Nothing below the bracket matters, so four
// values cost a maximum and a vote.  Where a lane says yes (four votes in ten at the usual fraction, 1.3 lanes of the 32) its four
// values go to a queue of the warp's in shared memory, and only when 32 such lanes have come together are the values
// compared one by one: handled on the spot, with all lanes at every hit, they were five sixths of this kernel's
// instructions (101 per warp and four values, issue slots 70 % busy; now 31 and 35 %).
// What a block keeps goes to places of its own in global memory, its counts and a histogram of the keys' upper bits with it: no
// global atomics (180 000 single additions to 8 KB of bins took 19 us), no fence, no block that ends last.
__global__ void __launch_bounds__(CALIB_THREADS, 3) collect_kernel(const int32_t *__restrict__ y, long long count, SelectState *st)
{
    static_assert(COARSE / 2 <= CALIB_THREADS && KEEP_BLOCK < 65536, "");
    __shared__ int4 queue[CALIB_WARPS][64];                        // (31 that wait and 32 more at most)
    __shared__ unsigned coarse[COARSE / 2];
    __shared__ unsigned s_count[4];                                // keys > hi, >= hi, >= lo; kept
    const int warp = (int)threadIdx.x >> 5, lane = (int)threadIdx.x & 31;
    const unsigned tid = blockIdx.x * CALIB_THREADS + threadIdx.x, step = gridDim.x * CALIB_THREADS;
    // 16-byte loads over the aligned middle, scalar loads at the ragged ends
    const long long head = min(count, (long long)((16 - ((uintptr_t)y & 15)) & 15) / 4);
    const long long vecs = (count - head) / 4;
    const int4 *p = (const int4 *)(y + head) + tid;
    const long long trips = vecs / (4ll * step);                   // of the whole grid, four vectors per thread each
    grid_dep_launch();
    int4 v[4];
    if (trips > 0) {
#pragma unroll
        for (int j = 0; j < 4; ++j) v[j] = __ldcs(p + j * (size_t)step);
        // the memory would idle until the bracket is there: the next rounds' values on their way to the L2 cache
        if (threadIdx.x < 4 * AHEAD && 1 + threadIdx.x / 4 < trips)
            asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(p - threadIdx.x + (4 + threadIdx.x) * (size_t)step), "r"(CALIB_THREADS * 16) : "memory");
    }
    if (threadIdx.x < COARSE / 2) coarse[threadIdx.x] = 0;
    if (threadIdx.x < 4) s_count[threadIdx.x] = 0;
    __syncthreads();
    grid_dep_wait();                                                    // the bracket
    const unsigned lo = __ldcg(&st->lo), hi = __ldcg(&st->hi);
    const unsigned inside = hi > lo ? hi - lo - 1u : 0u;            // keys lo + 1 ... lo + inside are kept, as 0 ... inside - 1
    const int hi_v = (int)(hi ^ 0x80000000u), lo_v = (int)(lo ^ 0x80000000u);
    const unsigned off = 0x80000000u - lo - 1u;                    // key - lo - 1 = v + off (mod 2^32)
    const int sh = coarse_shift(inside);
    unsigned n_above = 0, n_hi = 0, n_lo = 0;
    unsigned n_queue = 0;                                          // the warp's, the same in every lane
    const unsigned below = (1u << lane) - 1u;
    unsigned *const keep = st->keep[blockIdx.x];
    int4 *const q = queue[warp];
    auto take4 = [&](const int4 &x, unsigned has) {                // (whole warp; has: bit j for value j)
        const int v4[4] = {x.x, x.y, x.z, x.w};
        unsigned m[4], n = 0;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            m[j] = __ballot_sync(0xffffffffu, (has >> j & 1u) && (unsigned)v4[j] + off < inside);
            n += (unsigned)__popc(m[j]);
            if (has >> j & 1u) { n_above += v4[j] > hi_v; n_hi += v4[j] >= hi_v; n_lo += v4[j] >= lo_v; }
        }
        unsigned at = 0;
        if (lane == 0) at = atomicAdd(&s_count[3], n);
        at = __shfl_sync(0xffffffffu, at, 0);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const unsigned d = (unsigned)v4[j] + off, to = at + (unsigned)__popc(m[j] & below);
            if ((m[j] >> lane & 1u) && to < KEEP_BLOCK) {
                const unsigned b = d >> sh;
                keep[to] = d;
                atomicAdd(&coarse[b >> 1], 1u << (16 * (b & 1u)));
            }
            at += (unsigned)__popc(m[j]);
        }
    };
    auto take = [&](unsigned n) {                                  // the queue's last n vectors, one per lane
        __syncwarp();
        const bool there = (unsigned)lane < n;
        n_queue -= n;
        const int4 x = there ? q[n_queue + (unsigned)lane] : make_int4(0, 0, 0, 0);
        take4(x, there ? 15u : 0u);
        __syncwarp();
    };
    auto offer = [&](const int4 &x, bool there) {
        const bool hit = there && max(max(x.x, x.y), max(x.z, x.w)) >= lo_v;
        const unsigned m = __ballot_sync(0xffffffffu, hit);
        if (m) {
            if (hit) q[n_queue + (unsigned)__popc(m & below)] = x;
            n_queue += (unsigned)__popc(m);
            if (n_queue >= 32) take(32);
        }
    };
    for (long long t = 0; t < trips; ++t) {
#pragma unroll
        for (int j = 0; j < 4; ++j) offer(v[j], true);
        p += 4 * (size_t)step;
        if (t + 1 < trips) {
#pragma unroll
            for (int j = 0; j < 4; ++j) v[j] = __ldcs(p + j * (size_t)step);
        }
    }
    for (long long i = trips * 4 * step + tid - lane; i < vecs; i += step, p += step) {       // (the same trips for the whole warp)
        const bool there = i + lane < vecs;
        offer(there ? __ldcs(p) : make_int4(0, 0, 0, 0), there);
    }
    if (n_queue) take(n_queue);
    if (blockIdx.x == 0 && warp == 0) {                            // at most three values at either end
        const long long tail = head + vecs * 4;
        const long long e = lane < 4 ? (lane < head ? (long long)lane : -1) : (lane < 8 && tail + lane - 4 < count ? tail + lane - 4 : -1);
        take4(make_int4(e >= 0 ? y[e] : 0, 0, 0, 0), e >= 0 ? 1u : 0u);
    }
    n_above = __reduce_add_sync(0xffffffffu, n_above);
    n_hi = __reduce_add_sync(0xffffffffu, n_hi);
    n_lo = __reduce_add_sync(0xffffffffu, n_lo);
    if (lane == 0) {
        if (n_above) atomicAdd(&s_count[0], n_above);
        if (n_hi) atomicAdd(&s_count[1], n_hi);
        if (n_lo) atomicAdd(&s_count[2], n_lo);
    }
    __syncthreads();
    if (threadIdx.x < COARSE / 2) st->coarse[blockIdx.x][threadIdx.x] = coarse[threadIdx.x];
    if (threadIdx.x == 0) st->counts[blockIdx.x] = make_uint4(s_count[0], s_count[1], s_count[2], s_count[3]);
}

// Adds up the blocks' histograms `hist` (the same place in every block's shared memory; complete, and the cluster in step): a
// block takes an eighth of the bins and hands the sums to all.  The cluster is in step again afterwards.
__device__ __forceinline__ void cluster_total(const unsigned *hist, unsigned *total, unsigned block)
{
    constexpr unsigned SHARE = BINS / CLUSTER;
    if (threadIdx.x < SHARE) {
        const unsigned b = block * SHARE + threadIdx.x;
        unsigned sum = 0;
#pragma unroll
        for (unsigned r = 0; r < CLUSTER; ++r) sum += ld_cluster(&hist[b], r);
#pragma unroll
        for (unsigned r = 0; r < CLUSTER; ++r) st_cluster(&total[b], r, sum);
    }
    cluster_sync();
}

// The answer from what the pass counted and kept, by one cluster.  The blocks' histograms, added up, give the bin of the
// key's upper nine bits; the bits below it come from the kept keys in that bin (each block has an eighth of the lists), eleven a
// round.  A list is read by sixteen threads, which hold its first 480 keys.  14 us with cold
// caches, half of it the first reads; it replaces a last block's work in the pass as well (19 us there).
__global__ void __cluster_dims__(CLUSTER, 1, 1) __launch_bounds__(CLUSTER_THREADS, 1)
settle_kernel(SelectState *st, unsigned n_blocks, unsigned long long k, SelectOut *out)
{
    constexpr unsigned READERS = 16, EACH = 30;
    static_assert(COLLECT_BLOCKS <= CLUSTER_THREADS && COLLECT_BLOCKS <= CLUSTER * CLUSTER_THREADS / READERS, "");
    __shared__ __align__(8) unsigned hist[BINS], total[BINS];
    __shared__ Finder f;
    __shared__ uint4 s_part[CLUSTER_WARPS];            // the warps' sums: keys > hi, >= hi, >= lo; kept
    __shared__ unsigned long long s_sum[4];
    const unsigned block = cluster_rank(), warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    hist[2 * threadIdx.x] = hist[2 * threadIdx.x + 1] = 0;
    __syncthreads();
    grid_dep_wait();
    const unsigned lo = __ldcg(&st->lo), hi = __ldcg(&st->hi);
    // this thread's list and its place in it
    const unsigned of = block + CLUSTER * (threadIdx.x / READERS), sub = threadIdx.x % READERS;
    const unsigned len = of < n_blocks ? min(__ldcg(&st->counts[of].w), KEEP_BLOCK) : 0u;
    const unsigned *list = st->keep[of < n_blocks ? of : 0];
    uint4 c = make_uint4(0, 0, 0, 0);                              // (every block needs all counts)
    if (threadIdx.x < n_blocks) c = __ldcg(&st->counts[threadIdx.x]);
    // the histograms of this block's share of the pass's blocks
    constexpr unsigned WORDS = COARSE / 2, ROWS = CLUSTER * CLUSTER_THREADS / WORDS, ROUNDS = (COLLECT_BLOCKS + ROWS - 1) / ROWS;
    const unsigned word = threadIdx.x % WORDS;
    unsigned even = 0, odd = 0;
#pragma unroll
    for (unsigned i = 0; i < ROUNDS; ++i) {
        const unsigned b = block + CLUSTER * (threadIdx.x / WORDS) + i * ROWS, two = b < n_blocks ? __ldcg(&st->coarse[b][word]) : 0u;
        even += two & 0xffffu;
        odd += two >> 16;
    }
    if (even) atomicAdd(&hist[2 * word], even);
    if (odd) atomicAdd(&hist[2 * word + 1], odd);
    unsigned key[EACH];
#pragma unroll
    for (unsigned i = 0; i < EACH; ++i) key[i] = sub + READERS * i < len ? __ldcg(list + sub + READERS * i) : 0u;
    // (the sums of a warp's 32 blocks fit 32 bits, those of all need not)
    const unsigned p0 = __reduce_add_sync(0xffffffffu, c.x), p1 = __reduce_add_sync(0xffffffffu, c.y);
    const unsigned p2 = __reduce_add_sync(0xffffffffu, c.z), p3 = __reduce_add_sync(0xffffffffu, c.w);
    if (lane == 0) s_part[warp] = make_uint4(p0, p1, p2, p3);
    const bool over = __syncthreads_or(c.w > KEEP_BLOCK);
    if (warp == 0) {
        const uint4 p = s_part[lane];
        const unsigned v[4] = {p.x, p.y, p.z, p.w};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const unsigned l = __reduce_add_sync(0xffffffffu, v[i] & 0xffffu), h = __reduce_add_sync(0xffffffffu, v[i] >> 16);
            if (lane == 0) s_sum[i] = l + ((unsigned long long)h << 16);
        }
    }
    cluster_sync();
    const unsigned long long above = s_sum[0], from_hi = s_sum[1], from_lo = s_sum[2], kept = s_sum[3];
    // k in (above, from_hi]: hi itself; up to as many more as were kept: a kept key; from there to from_lo: lo itself
    const bool at_hi = k <= from_hi;
    const bool at_lo = !at_hi && !over && k > from_hi + kept;
    const bool miss = k <= above || k > from_lo || (!at_hi && over);
    if (miss || at_hi || at_lo) {                                  // (the same in every block of the cluster, which has read nothing of another's yet)
        if (block == 0 && threadIdx.x == 0) {
            out->result = bound_of(at_hi ? hi : lo);
            out->status = miss ? CALIB_MISS : CALIB_DONE;
        }
        return;
    }
    int left = coarse_shift(hi - lo - 1u);
    unsigned found, want;
    cluster_total(hist, total, block);
    pick_bin(f, total, (unsigned)(k - from_hi), found, want);      // (at most all that is kept)
    found <<= left;
    while (left > 0) {
        const int w = min(left, BIN_BITS), s = left - w;
        __syncthreads();
        hist[2 * threadIdx.x] = hist[2 * threadIdx.x + 1] = 0;
        __syncthreads();
        auto add = [&](unsigned d) {
            d ^= found;                                            // (its open bits are zero)
            if ((d >> left) == 0) atomicAdd(&hist[d >> s], 1u);
        };
#pragma unroll
        for (unsigned i = 0; i < EACH; ++i)
            if (sub + READERS * i < len) add(key[i]);
#pragma unroll 4
        for (unsigned e = sub + READERS * EACH; e < len; e += READERS) add(__ldcg(list + e));
        cluster_sync();
        cluster_total(hist, total, block);
        unsigned bin;
        pick_bin(f, total, want, bin, want);
        found |= bin << s;
        left = s;
        // (the next round writes what others read only behind a barrier of the cluster that all reach after these reads)
    }
    if (block == 0 && threadIdx.x == 0) {
        out->result = bound_of(lo + 1u + found);
        out->status = CALIB_DONE;
    }
    cluster_sync();                                                // no block leaves while another may read its shared memory
}

// ---------------------------------------------------------------- radix select (where the sample misled)
__global__ void select_init_kernel(SelectState *st, unsigned long long k)
{
    if (threadIdx.x == 0) { st->k = k; st->prefix = 0; st->mask = 0; }
}

// Counts one key into the block's histogram if it lies under the prefix.  A feature map's keys
// crowd into a few bins of the upper bytes, so a thread keeps the count of its current bin
// in a register and touches shared memory only when the bin changes.
__device__ __forceinline__ void tally(unsigned key, unsigned prefix, unsigned mask, int shift, unsigned *sh, unsigned &cur, unsigned &cnt)
{
    if ((key & mask) != prefix) return;
    const unsigned bin = (key >> shift) & 255u;
    if (bin == cur) { ++cnt; return; }
    if (cnt) atomicAdd(&sh[cur], cnt);
    cur = bin;
    cnt = 1;
}

// One pass: the byte at `shift` of every key under the current prefix.
__global__ void __launch_bounds__(CALIB_THREADS) select_hist_kernel(const int32_t *__restrict__ y, long long count, int shift, SelectState *st)
{
    __shared__ unsigned sh[256];
    if (threadIdx.x < 256) sh[threadIdx.x] = 0;
    __syncthreads();
    const unsigned prefix = st->prefix, mask = st->mask;
    unsigned cur = 0, cnt = 0;
    const long long tid = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const long long step = (long long)gridDim.x * blockDim.x;
    // 16-byte loads over the aligned middle, scalar loads at the ragged ends
    const long long head = min(count, (long long)((16 - ((uintptr_t)y & 15)) & 15) / 4);
    const long long vecs = (count - head) / 4;
    const int4 *yv = (const int4 *)(y + head);
    for (long long i = tid; i < vecs; i += step) {
        const int4 v = __ldg(yv + i);
        tally(key_of(v.x), prefix, mask, shift, sh, cur, cnt);
        tally(key_of(v.y), prefix, mask, shift, sh, cur, cnt);
        tally(key_of(v.z), prefix, mask, shift, sh, cur, cnt);
        tally(key_of(v.w), prefix, mask, shift, sh, cur, cnt);
    }
    for (long long e = tid; e < head; e += step) tally(key_of(y[e]), prefix, mask, shift, sh, cur, cnt);
    for (long long e = head + vecs * 4 + tid; e < count; e += step) tally(key_of(y[e]), prefix, mask, shift, sh, cur, cnt);
    if (cnt) atomicAdd(&sh[cur], cnt);
    __syncthreads();
    if (threadIdx.x < 256 && sh[threadIdx.x]) atomicAdd(&st->hist[threadIdx.x], (unsigned long long)sh[threadIdx.x]);
}

// Picks the bin that holds the k-th largest key, fixes it in the prefix, clears the histogram.
__global__ void select_step_kernel(SelectState *st, int shift, int last, SelectOut *out)
{
    __shared__ unsigned long long hist[256];
    hist[threadIdx.x] = st->hist[threadIdx.x];
    st->hist[threadIdx.x] = 0;
    __syncthreads();
    if (threadIdx.x == 0) {
        unsigned long long k = st->k, above = 0;
        int b = 255;
        for (; b > 0; --b) {
            if (above + hist[b] >= k) break;
            above += hist[b];
        }
        st->k = k - above;
        st->prefix |= (unsigned)b << shift;
        st->mask |= 255u << shift;
        if (last) { out->result = bound_of(st->prefix); out->status = CALIB_DONE; }
    }
}

static_assert(offsetof(SelectState, counts) % 16 == 0, "");

// ---------------------------------------------------------------- host side
// A call holds one scratch from its first launch until it has seen its result, so calls of several
// threads and streams never share one.  Scratches that are not in use are kept, at most KEEP_FREE per
// device, until iq_release_scratch gives them back; one more than that is released when its call ends.
// Where the 11 MB with the places for the bracket's keys are not to be had, the first 2 KB do, with the radix select.
struct Scratch {
    SelectState *state = nullptr;
    SelectOut *out = nullptr, *out_dev = nullptr;      // pinned host memory and its device address
    bool small = false;                                // nothing from `counts` on
};
constexpr int KEEP_FREE = 4;
struct FreeList {
    Scratch s[KEEP_FREE];
    int n = 0;
};
std::mutex g_free_mutex;
FreeList g_free[MAX_DEVICES];

void scratch_release(const Scratch &s)
{
    cudaFree(s.state);
    cudaFreeHost(s.out);
}

int scratch_take(int dev, Scratch &s)
{
    {
        std::lock_guard<std::mutex> lock(g_free_mutex);
        if (g_free[dev].n) {
            s = g_free[dev].s[--g_free[dev].n];
            return ICONV_OK;
        }
    }
    Scratch f;
    cudaError_t e = cudaMalloc((void **)&f.state, sizeof(SelectState));
    if (e == cudaErrorMemoryAllocation) {
        cudaGetLastError();
        f.small = true;
        e = cudaMalloc((void **)&f.state, offsetof(SelectState, counts));
    }
    if (e == cudaSuccess) e = cudaHostAlloc((void **)&f.out, sizeof(SelectOut), cudaHostAllocMapped);
    if (e == cudaSuccess) e = cudaHostGetDevicePointer((void **)&f.out_dev, f.out, 0);
    if (e == cudaSuccess) e = cudaMemset(f.state, 0, offsetof(SelectState, counts));
    if (e == cudaSuccess) e = cudaStreamSynchronize(cudaStreamLegacy);      // before a launch on a stream that does not wait for the legacy one
    if (e != cudaSuccess) { scratch_release(f); return cuda_fail(e, "iq_sigma_bound: scratch"); }
    s = f;
    return ICONV_OK;
}

// Was the launch refused because a part of a GPU has no room for a cluster of eight blocks?
bool no_room(cudaError_t e) { return e == cudaErrorInvalidClusterSize || e == cudaErrorLaunchOutOfResources || e == cudaErrorInvalidConfiguration; }

int select_run(const Scratch &s, const int32_t *y, long long count, unsigned long long k, cudaStream_t stream, int *bound)
{
    long long blocks = (count / 4 + CALIB_THREADS - 1) / CALIB_THREADS;
    if (blocks < 1) blocks = 1;
    if (blocks > COLLECT_BLOCKS) blocks = COLLECT_BLOCKS;
    const bool whole = count <= SAMPLE;
    // ranks in the sample: the k-th largest of Y is near the (k * SAMPLE / count)-th of the sample, with the
    // deviation of a binomial count
    const double p = (double)k / (double)count, mid = p * SAMPLE, dev = 4.5 * sqrt(mid * (1.0 - p)) + 2.0;
    // (an end without bound leaves the histogram's bins too wide to tell keys apart, so the sample's largest key
    // stands in where the rank is very likely below it: e^-8 at most that it is not)
    const double r_hi = mid >= 8.0 ? fmax(1.0, floor(mid - dev)) : 0.0, r_lo = ceil(mid + dev) + 1.0;
    s.out->status = 0;
    // more in the bracket than is kept (a rank near the middle of a large tensor): the radix select right away
    bool radix = !whole && (s.small || (fmin(r_lo, (double)SAMPLE) - r_hi) / SAMPLE * (double)count > 0.8 * (double)KEEP_BLOCK * (double)blocks);
    if (!radix) {
        cudaError_t e = launch_kernel(bracket_kernel, false, CLUSTER, CLUSTER_THREADS, 0, stream, y, (unsigned long long)count, k, (int)whole,
                               r_hi < 1.0 ? 0u : (unsigned)r_hi, (unsigned)r_lo, s.state, s.out_dev);
        if (e == cudaSuccess && !whole) {
            e = launch_kernel(collect_kernel, true, (unsigned)blocks, CALIB_THREADS, 0, stream, y, count, s.state);
            if (e == cudaSuccess) e = launch_kernel(settle_kernel, true, CLUSTER, CLUSTER_THREADS, 0, stream, s.state, (unsigned)blocks, k, s.out_dev);
        }
        if (no_room(e)) {
            cudaGetLastError();
            radix = true;
        } else {
            ICONV_CUDA_TRY(e);
        }
    }
    if (!radix) ICONV_CUDA_TRY(cudaStreamSynchronize(stream));
    if (((volatile SelectOut *)s.out)->status != CALIB_DONE) {
        select_init_kernel<<<1, 32, 0, stream>>>(s.state, k);
        for (int pass = 3; pass >= 0; --pass) {
            select_hist_kernel<<<(unsigned)blocks, CALIB_THREADS, 0, stream>>>(y, count, 8 * pass, s.state);
            select_step_kernel<<<1, 256, 0, stream>>>(s.state, 8 * pass, pass == 0, s.out_dev);
        }
        ICONV_CUDA_TRY(cudaGetLastError());
        ICONV_CUDA_TRY(cudaStreamSynchronize(stream));
    }
    *bound = ((volatile SelectOut *)s.out)->result;
    return ICONV_OK;
}

}  // namespace

}  // namespace iconv

using namespace iconv;

extern "C" int iq_sigma_bound(const int32_t *y, int64_t count, double fraction, int32_t *bound, void *cuda_stream)
{
    if (!bound || count < 0 || !(fraction > 0.0) || fraction > 1.0 || (count > 0 && !y)) {
        set_error("iq_sigma_bound: needs a device tensor, 0 < fraction <= 1 and a place for the result");
        return ICONV_ERR_ARG;
    }
    if ((uintptr_t)y % 4) { set_error("iq_sigma_bound: the tensor must be 4-byte aligned"); return ICONV_ERR_ALIGN; }
    if (count == 0) { *bound = 1; return ICONV_OK; }       // an empty map bounds nothing: the smallest legal bound
    const int dev = current_device_slot();
    if (dev < 0) { set_error("iq_sigma_bound: no current device, or its index is beyond %d", MAX_DEVICES - 1); return ICONV_ERR_ARG; }
    // (the wait for the result would end a capture, and a scratch cannot be freed inside one)
    cudaStreamCaptureStatus capture;
    ICONV_CUDA_TRY(cudaStreamIsCapturing((cudaStream_t)cuda_stream, &capture));
    if (capture != cudaStreamCaptureStatusNone) { set_error("iq_sigma_bound: the stream is capturing"); return ICONV_ERR_CUDA; }
    double kd = ceil((double)count * fraction);
    unsigned long long k = kd < 1.0 ? 1ull : (unsigned long long)kd;
    if (k > (unsigned long long)count) k = (unsigned long long)count;
    Scratch s;
    int rc = scratch_take(dev, s);
    if (rc != ICONV_OK) return rc;
    int result = 0;
    rc = select_run(s, y, (long long)count, k, (cudaStream_t)cuda_stream, &result);
    bool kept = false;
    if (rc == ICONV_OK) {                                  // (after an error the scratch may not be zero: it is not used again)
        std::lock_guard<std::mutex> lock(g_free_mutex);
        if (!s.small && g_free[dev].n < KEEP_FREE) { g_free[dev].s[g_free[dev].n++] = s; kept = true; }
    }
    if (!kept) scratch_release(s);
    if (rc == ICONV_OK) *bound = result;
    return rc;
}

extern "C" int iq_release_scratch(void)
{
    const int dev = current_device_slot();
    if (dev < 0) { set_error("iq_release_scratch: no current device, or its index is beyond %d", MAX_DEVICES - 1); return ICONV_ERR_ARG; }
    FreeList unused;
    {
        std::lock_guard<std::mutex> lock(g_free_mutex);
        unused = g_free[dev];
        g_free[dev].n = 0;
    }
    for (int i = 0; i < unused.n; ++i) scratch_release(unused.s[i]);
    return ICONV_OK;
}

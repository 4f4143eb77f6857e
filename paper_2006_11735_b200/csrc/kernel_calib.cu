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
//                that fills a bracket's end by itself, as a clamped map's bound, costs nothing), keeps
//                what lies between and histograms its upper bits; the block that ends last picks the bin.
//   3. settle    the kept keys of that bin (about a hundred) and their order.
// The result is exact because the ranks are counted, not estimated.  A sample that misled (the rank
// is outside the bracket, or more keys in it than the scratch keeps) is noticed, and a
// most-significant-byte radix select does the call instead: four passes, any input.
//
// 51.4 M normal values (206 MB), whole call: 100 us; four radix passes took 297.  Kernel by kernel (apart, caches cold) the
// bracket takes 20 (one block finds the two order statistics, a barrier per bit), the pass 61 to 64 (the read alone
// would take 32 at the copy rate, the kept keys about 16), the settling 13.  Where the bracket misses, the call pays for it and
// the pass before the radix select.
#include <cmath>
#include <cstddef>
#include <mutex>

#include "plan.h"

namespace iconv {

namespace {

constexpr int CALIB_THREADS = 512;
constexpr int SAMPLE = 8192;                     // keys sampled; a tensor no larger is selected from directly
constexpr int SAMPLE_THREADS = 1024;
constexpr int SAMPLE_BLOCKS = SAMPLE / SAMPLE_THREADS;
constexpr int COLLECT_BLOCKS = 148 * 3;          // three blocks of 512 threads are resident on an SM: one wave
constexpr unsigned KEEP_WARP = 384;              // keys of the bracket that a warp keeps at most
constexpr unsigned KEEP_BLOCK = KEEP_WARP * (CALIB_THREADS / 32);
constexpr unsigned KEEP_MAX = KEEP_BLOCK * COLLECT_BLOCKS;
constexpr int BIN_BITS = 11;
constexpr int BINS = 1 << BIN_BITS;

constexpr int LIST = 2048;                       // keys of one bin that are ordered by comparing all with all
constexpr int SETTLE_BLOCKS = 148;

enum { CALIB_DONE = 1, CALIB_MISS = 2 };

struct SelectOut {                               // in pinned host memory
    int result, status;
};

// Scratch of one call.  hist, the counts, overflow and the tickets are zero between calls.
struct SelectState {
    unsigned long long hist[BINS];               // keys of the bracket (collect), or of the prefix (radix), by bin
    unsigned long long above, from_hi, from_lo;  // keys > hi, >= hi, >= lo
    unsigned kept, overflow;
    unsigned ticket_sample, ticket_collect, ticket_settle;
    unsigned listed;                             // settle: kept keys of the bin
    unsigned found;                              // collect: the bin's first key (as kept), `left` lower bits open, the rank inside it
    int left;
    unsigned long long rank;
    unsigned lo, hi;                             // the bracket
    unsigned long long k;                        // radix: rank (from the top, 1-based) still to find inside the prefix
    unsigned prefix, mask;                       // radix: key bits fixed so far
    unsigned list[LIST];
    unsigned sample[SAMPLE];
    alignas(16) unsigned keep[KEEP_MAX];         // (read in 16-byte vectors)
};

__device__ __forceinline__ unsigned key_of(int32_t v) { return (unsigned)v ^ 0x80000000u; }     // order-preserving
__device__ __forceinline__ int bound_of(unsigned key)
{
    const int v = (int)(key ^ 0x80000000u);
    return v < 1 ? 1 : v;
}

// Two order statistics of the block's keys at once, bit by bit from `top` (above it `base`, which all keys
// share): the largest value that at least `rank` keys reach.  One barrier per bit: the warps' counts (both in one
// word: at most 2^15 keys) go through one of two arrays in turn, and every warp adds them up for itself.
__device__ __forceinline__ void block_ranks(const unsigned (&key)[SAMPLE / SAMPLE_THREADS], unsigned base, int top, unsigned rank_a, unsigned rank_b,
                                            unsigned (&sh)[2][32], unsigned &pa, unsigned &pb)
{
    static_assert(SAMPLE_THREADS == 1024 && SAMPLE <= 32768, "");
    pa = pb = base;
    for (int bit = top; bit >= 0; --bit) {
        const unsigned ca = pa | (1u << bit), cb = pb | (1u << bit);
        unsigned n = 0;
#pragma unroll
        for (int j = 0; j < SAMPLE / SAMPLE_THREADS; ++j) n += (key[j] >= ca ? 1u : 0u) + (key[j] >= cb ? 0x10000u : 0u);
        n = __reduce_add_sync(0xffffffffu, n);
        if ((threadIdx.x & 31) == 0) sh[bit & 1][threadIdx.x >> 5] = n;
        __syncthreads();
        n = __reduce_add_sync(0xffffffffu, sh[bit & 1][threadIdx.x & 31]);
        if ((n & 0xffffu) >= rank_a) pa = ca;
        if ((n >> 16) >= rank_b) pb = cb;
    }
}

// Draws the sample, and in the block that ends last finds the bracket; with `whole` (no more keys than
// the sample holds) the sample is Y itself and its k-th largest key the answer.
__global__ void __launch_bounds__(SAMPLE_THREADS) bracket_kernel(const int32_t *__restrict__ y, unsigned long long count, unsigned long long k, int whole,
                                                                 unsigned rank_hi, unsigned rank_lo, SelectState *st, SelectOut *out)
{
    __shared__ unsigned sh[2][32];
    __shared__ unsigned s_least, s_most;
    __shared__ bool last;
    const unsigned i = blockIdx.x * SAMPLE_THREADS + threadIdx.x;
    const unsigned n = whole ? (unsigned)count : (unsigned)SAMPLE;
    if (i < n) {
        unsigned long long at = i;
        if (!whole) {
            unsigned h = (i + 1u) * 0x9E3779B9u;                     // (hashed: no stride of the tensor's layout shows in the sample)
            h ^= h >> 16; h *= 0x85EBCA6Bu; h ^= h >> 13; h *= 0xC2B2AE35u; h ^= h >> 16;
            at = (unsigned long long)(((unsigned __int128)count * h) >> 32);
        }
        st->sample[i] = key_of(y[at]);
    }
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) {
        last = atomicAdd(&st->ticket_sample, 1u) == gridDim.x - 1;
        s_least = 0xffffffffu;
        s_most = 0;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    unsigned key[SAMPLE / SAMPLE_THREADS];             // (a missing key is 0, which no prefix with a bit set counts)
    unsigned least = 0xffffffffu, most = 0;
#pragma unroll
    for (int j = 0; j < SAMPLE / SAMPLE_THREADS; ++j) {
        const unsigned e = (unsigned)j * SAMPLE_THREADS + threadIdx.x;
        key[j] = e < n ? __ldcg(st->sample + e) : 0u;
        if (e < n) {
            least = min(least, key[j]);
            most = max(most, key[j]);
        }
    }
    // the bits in which the sample's keys differ
    least = __reduce_min_sync(0xffffffffu, least);
    most = __reduce_max_sync(0xffffffffu, most);
    if ((threadIdx.x & 31) == 0) { atomicMin(&s_least, least); atomicMax(&s_most, most); }
    __syncthreads();
    const unsigned diff = s_least ^ s_most;
    const int top = diff ? 31 - __clz((int)diff) : -1;
    const unsigned base = top >= 31 ? 0u : top < 0 ? s_most : s_most & ~((2u << top) - 1u);
    if (whole) {
        unsigned v, same;
        block_ranks(key, base, top, (unsigned)k, (unsigned)k, sh, v, same);
        if (threadIdx.x == 0) {
            out->result = bound_of(v);
            out->status = CALIB_DONE;
            st->ticket_sample = 0;
        }
        return;
    }
    unsigned lo, hi;
    block_ranks(key, base, top, rank_hi, rank_lo, sh, hi, lo);
    if (threadIdx.x == 0) {
        st->hi = rank_hi < 1 ? 0xffffffffu : hi;
        st->lo = rank_lo > n ? 0u : lo;
        st->ticket_sample = 0;
    }
}

// The bin (of n_bins <= BINS, from the top) that holds rank `k`, and the rank inside it.  Whole block of
// CALIB_THREADS; hist in shared memory.  A thread adds up four neighbouring bins, a scan over the warp and the
// warps' sums gives what lies above them.
__device__ __forceinline__ void pick_bin(const unsigned *hist, int n_bins, unsigned long long k, int &bin, unsigned long long &rank_in)
{
    static_assert(BINS == 4 * CALIB_THREADS, "");
    __shared__ unsigned s_warp[CALIB_THREADS / 32];
    __shared__ int s_bin;
    __shared__ unsigned long long s_rank;
    const int warp = (int)threadIdx.x >> 5, lane = (int)threadIdx.x & 31;
    const int top = n_bins - 1 - 4 * (int)threadIdx.x;             // this thread's topmost bin
    unsigned c[4], sum = 0;                                        // (all counts together are below 2^32: keys that were kept)
#pragma unroll
    for (int j = 0; j < 4; ++j) { c[j] = top - j >= 0 ? hist[top - j] : 0u; sum += c[j]; }
    unsigned inc = sum;
    for (int d = 1; d < 32; d <<= 1) {
        const unsigned o = __shfl_up_sync(0xffffffffu, inc, d);
        if (lane >= d) inc += o;
    }
    if (lane == 31) s_warp[warp] = inc;
    __syncthreads();
    unsigned long long above = inc - sum;
    for (int w = 0; w < warp; ++w) above += s_warp[w];
    if (above < k && k <= above + sum) {
        int j = 0;
        while (k > above + c[j]) above += c[j++];
        s_bin = top - j;
        s_rank = k - above;
    }
    __syncthreads();
    bin = s_bin;
    rank_in = s_rank;
    __syncthreads();
}

// The one pass over Y, bound by its read where the tensor is large.  Nothing below the bracket matters, so four
// values cost a maximum and a vote, and only where a lane says yes (a third of the votes) the counts, and a
// place in a list of the warp's own for what lies inside; ballots give the places (shared-memory atomics
// with their results cost 40 us here).
__global__ void __launch_bounds__(CALIB_THREADS, 3) collect_kernel(const int32_t *__restrict__ y, long long count, unsigned long long k, SelectState *st,
                                                                   SelectOut *out)
{
    __shared__ unsigned buf[KEEP_BLOCK];
    __shared__ unsigned hist[BINS];
    __shared__ unsigned n_warp[CALIB_THREADS / 32], base_buf;
    __shared__ bool last;
    const int warp = (int)threadIdx.x >> 5, lane = (int)threadIdx.x & 31;
    for (int b = (int)threadIdx.x; b < BINS; b += CALIB_THREADS) hist[b] = 0;
    const unsigned lo = st->lo, hi = st->hi;
    const unsigned inside = hi > lo ? hi - lo - 1u : 0u;            // keys lo + 1 ... lo + inside are kept, as 0 ... inside - 1
    const int hi_v = (int)(hi ^ 0x80000000u), lo_v = (int)(lo ^ 0x80000000u);
    const unsigned off = 0x80000000u - lo - 1u;                    // key - lo - 1 = v + off (mod 2^32)
    const int bits = inside > 1 ? 32 - __clz((int)(inside - 1u)) : 0;
    const int sh = max(0, bits - BIN_BITS);
    unsigned n_above = 0, n_hi = 0, n_lo = 0, n_kept = 0;          // n_kept: the warp's, the same in every lane
    unsigned *mine = buf + warp * KEEP_WARP;
    auto take1 = [&](int v, bool there) {                          // (whole warp)
        const unsigned d = (unsigned)v + off;
        const bool in = there && d < inside;
        const unsigned m = __ballot_sync(0xffffffffu, in);
        const unsigned at = n_kept + (unsigned)__popc(m & ((1u << lane) - 1u));
        if (in && at < KEEP_WARP) mine[at] = d;
        n_kept += (unsigned)__popc(m);
        if (there) { n_above += v > hi_v; n_hi += v >= hi_v; n_lo += v >= lo_v; }
    };
    const long long tid = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const long long step = (long long)gridDim.x * blockDim.x;
    // 16-byte loads over the aligned middle, scalar loads at the ragged ends
    const long long head = min(count, (long long)((16 - ((uintptr_t)y & 15)) & 15) / 4);
    const long long vecs = (count - head) / 4;
    const int4 *yv = (const int4 *)(y + head);
    for (long long i0 = tid - lane; i0 < vecs; i0 += 4 * step) {    // (the same trips for the whole warp; four loads in flight per lane)
        int4 v[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const long long i = i0 + lane + j * step;
            v[j] = i < vecs ? __ldcs(yv + i) : make_int4(0, 0, 0, 0);
        }
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const bool there = i0 + lane + j * step < vecs;
            if (!__any_sync(0xffffffffu, there && max(max(v[j].x, v[j].y), max(v[j].z, v[j].w)) >= lo_v)) continue;
            take1(v[j].x, there); take1(v[j].y, there); take1(v[j].z, there); take1(v[j].w, there);
        }
    }
    if (blockIdx.x == 0 && warp == 0) {                            // at most three values at either end
        const long long tail = head + vecs * 4;
        const long long e = lane < 4 ? (lane < head ? (long long)lane : -1) : (lane < 8 && tail + lane - 4 < count ? tail + lane - 4 : -1);
        take1(e >= 0 ? y[e] : 0, e >= 0);
    }
    n_above = __reduce_add_sync(0xffffffffu, n_above);
    n_hi = __reduce_add_sync(0xffffffffu, n_hi);
    n_lo = __reduce_add_sync(0xffffffffu, n_lo);
    if (lane == 0) {
        if (n_above) atomicAdd(&st->above, (unsigned long long)n_above);
        if (n_hi) atomicAdd(&st->from_hi, (unsigned long long)n_hi);
        if (n_lo) atomicAdd(&st->from_lo, (unsigned long long)n_lo);
        n_warp[warp] = min(n_kept, KEEP_WARP);
        if (n_kept > KEEP_WARP) st->overflow = 1;
    }
    __syncthreads();
    // the warps' lists to global memory, one after another, and into the block's histogram
    unsigned before = 0, all = 0;
    for (int w = 0; w < CALIB_THREADS / 32; ++w) {
        if (w == warp) before = all;
        all += n_warp[w];
    }
    if (threadIdx.x == 0) base_buf = all ? atomicAdd(&st->kept, all) : 0u;
    __syncthreads();
    for (unsigned e = lane; e < n_warp[warp]; e += 32) {
        const unsigned d = mine[e];
        st->keep[base_buf + before + e] = d;
        atomicAdd(&hist[d >> sh], 1u);
    }
    __syncthreads();
    for (int b = (int)threadIdx.x; b < BINS; b += CALIB_THREADS)
        if (hist[b]) atomicAdd(&st->hist[b], (unsigned long long)hist[b]);
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) last = atomicAdd(&st->ticket_collect, 1u) == gridDim.x - 1;
    __syncthreads();
    if (!last) return;
    __threadfence();

    // the block that ends last: the bin; and the scratch back to zero
    for (int b = (int)threadIdx.x; b < BINS; b += CALIB_THREADS) {
        hist[b] = (unsigned)__ldcg(&st->hist[b]);                  // (at most KEEP_MAX)
        st->hist[b] = 0;
    }
    __syncthreads();
    const unsigned long long above = __ldcg(&st->above), from_hi = __ldcg(&st->from_hi), from_lo = __ldcg(&st->from_lo);
    const unsigned kept = __ldcg(&st->kept);
    const bool over = __ldcg(&st->overflow) != 0;
    // k in (above, from_hi]: hi itself; up to `kept` more: a kept key; from there to from_lo: lo itself
    const bool at_hi = k <= from_hi;
    const bool at_lo = !at_hi && !over && k > from_hi + kept;
    const bool miss = k <= above || k > from_lo || (!at_hi && over);
    int bin = 0;
    unsigned long long rank = 0;
    const bool search = !miss && !at_hi && !at_lo;
    if (search) pick_bin(hist, BINS, k - from_hi, bin, rank);
    __syncthreads();
    if (threadIdx.x == 0) {
        const bool open = search && sh > 0;                        // the bin holds several values: settle_kernel
        out->result = bound_of(at_hi ? hi : at_lo ? lo : lo + 1u + (unsigned)bin);
        out->status = miss ? CALIB_MISS : open ? 0 : CALIB_DONE;
        st->found = (unsigned)bin << sh;
        st->left = open ? sh : 0;
        st->rank = rank;
        st->above = st->from_hi = st->from_lo = 0;
        st->overflow = 0;
        st->ticket_collect = 0;
        if (!open) st->kept = 0;
    }
}

// The kept keys of the bin, and the one of rank `rank` among them.
__global__ void __launch_bounds__(CALIB_THREADS) settle_kernel(SelectState *st, SelectOut *out)
{
    __shared__ unsigned hist[BINS];
    __shared__ unsigned key[LIST];
    __shared__ bool last;
    int left = st->left;
    if (left == 0) return;
    const unsigned kept = st->kept, lo = st->lo;
    unsigned found = st->found;
    unsigned long long rank = st->rank;
    auto list1 = [&](unsigned d) {
        if ((d >> left) != (found >> left)) return;
        const unsigned at = atomicAdd(&st->listed, 1u);
        if (at < LIST) st->list[at] = d;
    };
    const unsigned step = gridDim.x * CALIB_THREADS;
    const uint4 *q = (const uint4 *)st->keep;
    for (unsigned e = blockIdx.x * CALIB_THREADS + threadIdx.x; e < kept / 4; e += step) {
        const uint4 v = __ldcg(q + e);
        list1(v.x); list1(v.y); list1(v.z); list1(v.w);
    }
    if (blockIdx.x == 0 && threadIdx.x < kept % 4) list1(__ldcg(st->keep + kept / 4 * 4 + threadIdx.x));
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) last = atomicAdd(&st->ticket_settle, 1u) == gridDim.x - 1;
    __syncthreads();
    if (!last) return;
    __threadfence();
    const unsigned n = __ldcg(&st->listed);
    if (n <= LIST) {
        for (unsigned e = threadIdx.x; e < n; e += CALIB_THREADS) key[e] = __ldcg(st->list + e);
        __syncthreads();
        for (unsigned e = threadIdx.x; e < n; e += CALIB_THREADS) {
            unsigned above = 0, same = 0;
            for (unsigned j = 0; j < n; ++j) { above += key[j] > key[e]; same += key[j] == key[e]; }
            if (above < rank && rank <= above + same) out->result = bound_of(lo + 1u + key[e]);      // (equal keys write the same)
        }
    } else {
        // a crowded bin: the remaining bits by histograms over the kept keys, by this block alone
        while (left > 0) {
            const int w = min(left, BIN_BITS), s = left - w;
            for (int b = (int)threadIdx.x; b < BINS; b += CALIB_THREADS) hist[b] = 0;
            __syncthreads();
            for (unsigned e = threadIdx.x; e < kept; e += CALIB_THREADS) {
                const unsigned d = __ldcg(st->keep + e);
                if ((d >> left) == (found >> left)) atomicAdd(&hist[(d >> s) & ((1u << w) - 1u)], 1u);
            }
            __syncthreads();
            int bin;
            pick_bin(hist, 1 << w, rank, bin, rank);
            found |= (unsigned)bin << s;
            left = s;
        }
        if (threadIdx.x == 0) out->result = bound_of(lo + 1u + found);
    }
    if (threadIdx.x == 0) {
        out->status = CALIB_DONE;
        st->kept = 0;
        st->listed = 0;
        st->left = 0;
        st->ticket_settle = 0;
    }
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

static_assert(offsetof(SelectState, keep) % 16 == 0, "");

// ---------------------------------------------------------------- host side
// A call holds one scratch from its first launch until it has seen its result, so calls of several
// threads and streams never share one.  Scratches that are not in use are kept, at most KEEP_FREE per
// device, until iq_release_scratch gives them back; one more than that is released when its call ends.
// Where the 11 MB with the places for the bracket's keys are not to be had, the first 58 KB do, with the radix select.
struct Scratch {
    SelectState *state = nullptr;
    SelectOut *out = nullptr, *out_dev = nullptr;      // pinned host memory and its device address
    bool small = false;                                // no `keep`
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
        e = cudaMalloc((void **)&f.state, offsetof(SelectState, keep));
    }
    if (e == cudaSuccess) e = cudaHostAlloc((void **)&f.out, sizeof(SelectOut), cudaHostAllocMapped);
    if (e == cudaSuccess) e = cudaHostGetDevicePointer((void **)&f.out_dev, f.out, 0);
    if (e == cudaSuccess) e = cudaMemset(f.state, 0, offsetof(SelectState, list));
    if (e == cudaSuccess) e = cudaStreamSynchronize(cudaStreamLegacy);      // before a launch on a stream that does not wait for the legacy one
    if (e != cudaSuccess) { scratch_release(f); return cuda_fail(e, "iq_sigma_bound: scratch"); }
    s = f;
    return ICONV_OK;
}

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
    const bool radix = !whole && (s.small || (fmin(r_lo, (double)SAMPLE) - r_hi) / SAMPLE * (double)count > 0.8 * (double)KEEP_BLOCK * (double)blocks);
    if (!radix) bracket_kernel<<<whole ? (unsigned)((count + SAMPLE_THREADS - 1) / SAMPLE_THREADS) : SAMPLE_BLOCKS, SAMPLE_THREADS, 0, stream>>>(
        y, (unsigned long long)count, k, whole, r_hi < 1.0 ? 0u : (unsigned)r_hi, (unsigned)r_lo, s.state, s.out_dev);
    if (!whole && !radix) {
        collect_kernel<<<(unsigned)blocks, CALIB_THREADS, 0, stream>>>(y, count, k, s.state, s.out_dev);
        settle_kernel<<<SETTLE_BLOCKS, CALIB_THREADS, 0, stream>>>(s.state, s.out_dev);
    }
    ICONV_CUDA_TRY(cudaGetLastError());
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

// The n-sigma bound of Section 3.2.2 on the GPU: the smallest value among the largest
// `fraction` of an int32 feature map Y, i.e. its k-th largest element with
// k = max(1, ceil(count * fraction)), clamped to at least 1 (a BReLU bound is positive).
// It is the step right before the hot path: the bound h_ri it returns feeds Eq. 9-13
// (`iq_brelu_params`), which give the layer's mul, shift and h_i.
//
// Exact selection without sorting, Y read ONCE:
//   1. bracket   16384 keys at hashed positions; two order statistics of the sample, 4.5 standard
//                deviations around the rank, bracket the k-th largest of Y: [lo, hi], about 0.3 % of Y
//                at the usual fraction.
//   2. collect   one pass over Y: counts what lies above hi, keeps what lies in the bracket and
//                histograms its upper bits; the block that ends last picks the bin, then the
//                remaining bits among the kept keys.
// The result is exact because the ranks are counted, not estimated.  A sample that misled (the rank
// is outside the bracket, or more keys in it than the scratch keeps) is noticed, and a
// most-significant-byte radix select does the call instead: four passes, any input.
//
// What bounds it: the read of Y, see collect_kernel.
#include <cmath>
#include <cstddef>
#include <mutex>
#include <vector>

#include "plan.h"

namespace iconv {

namespace {

constexpr int CALIB_THREADS = 512;
constexpr int SAMPLE = 16384;                    // keys sampled; a tensor no larger is selected from directly
constexpr int SAMPLE_THREADS = 1024;
constexpr int SAMPLE_BLOCKS = SAMPLE / SAMPLE_THREADS;
constexpr int SAMPLE_BITS = 18;                  // bits of the sampled range that the bracket resolves
constexpr int COLLECT_BLOCKS = 148 * 4;          // four blocks of 512 threads fill an SM
constexpr unsigned KEEP_BLOCK = 4096;            // keys of the bracket that a block keeps at most
constexpr unsigned KEEP_MAX = KEEP_BLOCK * COLLECT_BLOCKS;
constexpr int BIN_BITS = 11;
constexpr int BINS = 1 << BIN_BITS;

enum { CALIB_DONE = 1, CALIB_MISS = 2 };

struct SelectOut {                               // in pinned host memory
    int result, status;
};

// Scratch of one call.  hist, above, kept, overflow and the tickets are zero between calls.
struct SelectState {
    unsigned long long hist[BINS];               // keys of the bracket (collect), or of the prefix (radix), by bin
    unsigned long long above;                    // keys above the bracket
    unsigned kept, overflow;
    unsigned ticket_sample, ticket_collect;
    unsigned lo, hi;                             // the bracket
    unsigned long long k;                        // radix: rank (from the top, 1-based) still to find inside the prefix
    unsigned prefix, mask;                       // radix: key bits fixed so far
    unsigned sample[SAMPLE];
    unsigned keep[KEEP_MAX];
};

__device__ __forceinline__ unsigned key_of(int32_t v) { return (unsigned)v ^ 0x80000000u; }     // order-preserving
__device__ __forceinline__ int bound_of(unsigned key)
{
    const int v = (int)(key ^ 0x80000000u);
    return v < 1 ? 1 : v;
}

// Two order statistics of the block's keys at once, bit by bit: for each rank the largest prefix (bits
// top .. low; above them `base`, which all keys share) that at least `rank` keys reach, i.e. the
// rank-th largest key with its lower bits cleared.  One barrier per bit: the warps' counts (both in one
// word: at most 2^15 keys) go through one of two arrays in turn, and every warp adds them up for itself.
__device__ __forceinline__ void block_ranks(const unsigned (&key)[SAMPLE / SAMPLE_THREADS], unsigned base, int top, int low, unsigned rank_a, unsigned rank_b,
                                            unsigned (&sh)[2][32], unsigned &pa, unsigned &pb)
{
    static_assert(SAMPLE_THREADS == 1024 && SAMPLE <= 32768, "");
    pa = pb = base;
    for (int bit = top; bit >= low; --bit) {
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
        block_ranks(key, base, top, 0, (unsigned)k, (unsigned)k, sh, v, same);
        if (threadIdx.x == 0) {
            out->result = bound_of(v);
            out->status = CALIB_DONE;
            st->ticket_sample = 0;
        }
        return;
    }
    const int low = max(0, top - SAMPLE_BITS + 1);
    unsigned lo, hi;
    block_ranks(key, base, top, low, rank_hi, rank_lo, sh, hi, lo);
    if (threadIdx.x == 0) {
        st->hi = rank_hi < 1 ? 0xffffffffu : hi | ((1u << low) - 1u);
        st->lo = rank_lo > n ? 0u : lo;
        st->ticket_sample = 0;
    }
}

// The bin (of n_bins, a multiple of 32 or fewer than that, from the top) that holds rank `k`, and the rank inside
// it.  Whole block; hist in shared memory.
__device__ __forceinline__ void pick_bin(const unsigned *hist, int n_bins, unsigned long long k, int &bin, unsigned long long &rank_in)
{
    __shared__ int s_bin;
    __shared__ unsigned long long s_rank;
    if (threadIdx.x < 32) {                       // one warp: 32 bins per step from the top
        const int lane = threadIdx.x;
        unsigned long long above = 0;
        for (int b0 = n_bins - 32; b0 > -32; b0 -= 32) {
            const int b = b0 + 31 - lane;         // lane 0: the topmost
            unsigned long long c = b >= 0 ? hist[b] : 0ull, inc = c;
            for (int d = 1; d < 32; d <<= 1) {
                const unsigned long long o = __shfl_up_sync(0xffffffffu, inc, d);
                if (lane >= d) inc += o;
            }
            const unsigned hit = __ballot_sync(0xffffffffu, above + inc >= k);
            if (hit) {
                if (lane == __ffs((int)hit) - 1) { s_bin = b; s_rank = k - (above + inc - c); }
                break;
            }
            above += __shfl_sync(0xffffffffu, inc, 31);
        }
    }
    __syncthreads();
    bin = s_bin;
    rank_in = s_rank;
    __syncthreads();
}

// The one pass over Y.  Nearly every vector misses the bracket: its four values are compared with both
// ends without a branch (four instructions a value), eight vectors in flight per thread.
__global__ void __launch_bounds__(CALIB_THREADS) collect_kernel(const int32_t *__restrict__ y, long long count, unsigned long long k, SelectState *st,
                                                                SelectOut *out)
{
    __shared__ unsigned buf[KEEP_BLOCK];
    __shared__ unsigned hist[BINS];
    __shared__ unsigned n_buf, base_buf;
    __shared__ unsigned long long s_total;
    __shared__ bool last;
    for (int b = (int)threadIdx.x; b < BINS; b += CALIB_THREADS) hist[b] = 0;
    if (threadIdx.x == 0) { n_buf = 0; s_total = 0; }
    __syncthreads();
    const unsigned lo = st->lo, hi = st->hi, span = hi - lo;
    const int hi_v = (int)(hi ^ 0x80000000u);
    const unsigned off = 0x80000000u - lo;                         // key - lo = v + off (mod 2^32)
    const int bits = span ? 32 - __clz((int)span) : 0;             // bits of (key - lo)
    const int sh = max(0, bits - BIN_BITS);
    unsigned n_above = 0;
    auto keep = [&](int v) {
        const unsigned d = (unsigned)v + off;
        if (d > span) return;
        atomicAdd(&hist[d >> sh], 1u);
        if (!sh || *(volatile unsigned *)&n_buf >= KEEP_BLOCK) return;      // every bin a single value: nothing to keep; or too many
        const unsigned at = atomicAdd(&n_buf, 1u);
        if (at < KEEP_BLOCK) buf[at] = d;
    };
    auto take = [&](int v) { n_above += v > hi_v; keep(v); };
    auto take4 = [&](const int4 &v) {
        n_above += (v.x > hi_v) + (v.y > hi_v) + (v.z > hi_v) + (v.w > hi_v);
        if (((unsigned)v.x + off <= span) | ((unsigned)v.y + off <= span) | ((unsigned)v.z + off <= span) | ((unsigned)v.w + off <= span)) {
            keep(v.x); keep(v.y); keep(v.z); keep(v.w);
        }
    };
    const long long tid = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const long long step = (long long)gridDim.x * blockDim.x;
    // 16-byte loads over the aligned middle, scalar loads at the ragged ends
    const long long head = min(count, (long long)((16 - ((uintptr_t)y & 15)) & 15) / 4);
    const long long vecs = (count - head) / 4;
    const int4 *yv = (const int4 *)(y + head);
    long long i = tid;
    for (; i + 7 * step < vecs; i += 8 * step) {
        int4 v[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) v[j] = __ldcs(yv + i + j * step);
#pragma unroll
        for (int j = 0; j < 8; ++j) take4(v[j]);
    }
    for (; i < vecs; i += step) take4(__ldcs(yv + i));
    for (long long e = tid; e < head; e += step) take(y[e]);
    for (long long e = head + vecs * 4 + tid; e < count; e += step) take(y[e]);
    n_above = __reduce_add_sync(0xffffffffu, n_above);
    if ((threadIdx.x & 31) == 0 && n_above) atomicAdd(&st->above, (unsigned long long)n_above);
    __syncthreads();
    const unsigned mine = min(n_buf, KEEP_BLOCK);
    if (threadIdx.x == 0) {
        base_buf = mine ? atomicAdd(&st->kept, mine) : 0u;
        if (n_buf >= KEEP_BLOCK) st->overflow = 1;
    }
    __syncthreads();
    for (unsigned e = threadIdx.x; e < mine; e += CALIB_THREADS) st->keep[base_buf + e] = buf[e];
    for (int b = (int)threadIdx.x; b < BINS; b += CALIB_THREADS)
        if (hist[b]) atomicAdd(&st->hist[b], (unsigned long long)hist[b]);
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) last = atomicAdd(&st->ticket_collect, 1u) == gridDim.x - 1;
    __syncthreads();
    if (!last) return;
    __threadfence();

    // the block that ends last: rank, bin, remaining bits; and the scratch back to zero
    unsigned long long total = 0;
    bool wide = false;                                             // a count beyond 32 bits: the radix select
    for (int b = (int)threadIdx.x; b < BINS; b += CALIB_THREADS) {
        const unsigned long long c = __ldcg(&st->hist[b]);
        hist[b] = (unsigned)c;
        wide |= (c >> 32) != 0;
        total += c;
        st->hist[b] = 0;
    }
    atomicAdd(&s_total, total);
    wide = __syncthreads_or(wide) != 0;
    const unsigned long long above = __ldcg(&st->above);
    const unsigned kept = __ldcg(&st->kept);
    const bool miss = wide || k <= above || k > above + s_total || __ldcg(&st->overflow) != 0;
    unsigned found = 0;
    if (!miss) {
        int bin;
        unsigned long long rank;
        pick_bin(hist, BINS, k - above, bin, rank);
        found = (unsigned)bin << sh;                               // key - lo so far; `left` lower bits to find
        int left = sh;
        while (left > 0) {
            const int w = min(left, BIN_BITS), s = left - w;
            for (int b = (int)threadIdx.x; b < BINS; b += CALIB_THREADS) hist[b] = 0;
            __syncthreads();
            const uint4 *q = (const uint4 *)st->keep;
            auto see = [&](unsigned d) { if ((d >> left) == (found >> left)) atomicAdd(&hist[(d >> s) & ((1u << w) - 1u)], 1u); };
            unsigned e4 = threadIdx.x;
            for (; e4 + 7 * CALIB_THREADS < kept / 4; e4 += 8 * CALIB_THREADS) {      // (one block reads them all: eight loads in flight)
                uint4 v[8];
#pragma unroll
                for (int j = 0; j < 8; ++j) v[j] = __ldcg(q + e4 + j * CALIB_THREADS);
#pragma unroll
                for (int j = 0; j < 8; ++j) { see(v[j].x); see(v[j].y); see(v[j].z); see(v[j].w); }
            }
            for (; e4 < kept / 4; e4 += CALIB_THREADS) {
                const uint4 v = __ldcg(q + e4);
                see(v.x); see(v.y); see(v.z); see(v.w);
            }
            for (unsigned e = kept / 4 * 4 + threadIdx.x; e < kept; e += CALIB_THREADS) see(__ldcg(st->keep + e));
            __syncthreads();
            pick_bin(hist, 1 << w, rank, bin, rank);
            found |= (unsigned)bin << s;
            left = s;
        }
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        out->result = bound_of(lo + found);
        out->status = miss ? CALIB_MISS : CALIB_DONE;
        st->above = 0;
        st->kept = 0;
        st->overflow = 0;
        st->ticket_collect = 0;
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

// ---------------------------------------------------------------- host side
// A call holds one scratch from its first launch until it has seen its result, so calls of several
// threads and streams never share one.  Scratches that are not in use are kept, at most KEEP_FREE per
// device; one more than that is released when its call ends.
struct Scratch {
    SelectState *state = nullptr;
    SelectOut *out = nullptr, *out_dev = nullptr;      // pinned host memory and its device address
};
constexpr size_t KEEP_FREE = 4;
std::mutex g_free_mutex;
std::vector<Scratch> g_free[MAX_DEVICES];

void scratch_release(const Scratch &s)
{
    cudaFree(s.state);
    cudaFreeHost(s.out);
}

int scratch_take(int dev, Scratch &s)
{
    {
        std::lock_guard<std::mutex> lock(g_free_mutex);
        if (!g_free[dev].empty()) {
            s = g_free[dev].back();
            g_free[dev].pop_back();
            return ICONV_OK;
        }
    }
    Scratch f;
    cudaError_t e = cudaMalloc((void **)&f.state, sizeof(SelectState));
    if (e == cudaSuccess) e = cudaHostAlloc((void **)&f.out, sizeof(SelectOut), cudaHostAllocMapped);
    if (e == cudaSuccess) e = cudaHostGetDevicePointer((void **)&f.out_dev, f.out, 0);
    if (e == cudaSuccess) e = cudaMemset(f.state, 0, offsetof(SelectState, sample));
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
    const double r_hi = floor(mid - dev), r_lo = ceil(mid + dev) + 1.0;
    s.out->status = 0;
    bracket_kernel<<<whole ? (unsigned)((count + SAMPLE_THREADS - 1) / SAMPLE_THREADS) : SAMPLE_BLOCKS, SAMPLE_THREADS, 0, stream>>>(
        y, (unsigned long long)count, k, whole, r_hi < 1.0 ? 0u : (unsigned)r_hi, (unsigned)r_lo, s.state, s.out_dev);
    if (!whole) collect_kernel<<<(unsigned)blocks, CALIB_THREADS, 0, stream>>>(y, count, k, s.state, s.out_dev);
    ICONV_CUDA_TRY(cudaGetLastError());
    ICONV_CUDA_TRY(cudaStreamSynchronize(stream));
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
        if (g_free[dev].size() < KEEP_FREE) { g_free[dev].push_back(s); kept = true; }
    }
    if (!kept) scratch_release(s);
    if (rc == ICONV_OK) *bound = result;
    return rc;
}

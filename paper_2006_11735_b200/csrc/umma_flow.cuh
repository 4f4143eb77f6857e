// A run of different layers in ONE launch: 1x1 and k x k convolutions of any stride with everything the
// im2col kernel fuses into them (BReLU and Eq. 4, an 8-bit skip, a projection), each reading what earlier
// layers of the run wrote.  The bottleneck and basic blocks of the ResNets.
//
// What it is for: launched one by one these layers are short (10 to 30 us at batch 256, 8 at batch 1) and
// pay 5 to 7 us each for set-up, an empty pipeline, a last wave that leaves SMs idle and a drain.  Here
// the tiles of ALL layers are one sequence; CTA pair c takes tiles c, c + pairs, ... of it.  A tile's loads
// wait for the units (a tile's pixels, 256 as a rule, with all channels) of earlier layers that it reads, nothing else: the pipeline
// runs on across layers, waves of different layers fill one another's gaps, and the weights of a tile are
// on their way while its activations are still being computed.
//
// The math per tile is the CTA-pair form of the im2col kernel (umma_device.cuh): 256 pixels x block_n
// channels, each CTA loads its 128 pixel rows and half of the B tile, the leader issues M = 256
// instructions.  Different here:
//   - 1x1 layers over dense pixels load A by plain tiled copies (52 to 58 B/clk per SM against 41 in im2col mode).
//   - block_n, and the pixel rows a CTA takes (128, or 64 or 32 of which the loads are shorter; the instruction
//     still spans 128, whose other rows nobody reads), are chosen per layer so that small grids spread over the SMs.
//   - An output tile is staged as whole 128-row pieces; the skip arrives in the same buffer before, and every
//     16 bytes of it are replaced in place by the outputs they went into.  One warp loads (skip, constants),
//     another stores and, once the stores are complete, counts the tile for its unit.
//
// Order between CTAs: the storing thread waits until its bulk stores are complete, fences, and adds to the
// unit's counter in global memory; in every CTA one warp follows the counters (acquire) and keeps the length
// of the finished prefix of the sequence of units in shared memory, where the loading warps find it; what
// follows is fenced against their bulk-asynchronous reads.  A tile only reads units of earlier layers and
// every CTA pair takes its tiles in order, so the launch cannot lock up as long as all its CTAs are
// resident (cooperative launch).  All waits are bounded as in the other kernels.
#pragma once

#include "umma_device.cuh"

namespace iconv {

constexpr int FLOW_MAX_LAYERS = 50;              // the layers travel as kernel arguments (at most 32764 bytes)
constexpr int FLOW_STAGES = 5;                   // 32 KB each: 128 rows of A, up to 128 rows of B
constexpr int FLOW_SLOT = 32768;
constexpr int FLOW_STAGING = 32768;              // one output tile of 128 rows x 256 channels; two of them
constexpr int FLOW_SYNC_WORDS = 32;              // words before the units' counters; word 0: CTAs that are done
constexpr int FLOW_A_WARP = 0, FLOW_B_WARP = 1, FLOW_READY_WARP = 2, FLOW_MMA_WARP = 3;
constexpr int FLOW_SKIP_WARP = EPI_WARP0 + EPI_WARPS_MAX, FLOW_STORE_WARP = FLOW_SKIP_WARP + 1;
constexpr int FLOW_STORE_WARPS = 2;              // one per staged tile: a tile's stores are on their way while the one before is being counted
constexpr int FLOW_A_WARP2 = FLOW_STORE_WARP + FLOW_STORE_WARPS, FLOW_B_WARP2 = FLOW_A_WARP2 + 1;
constexpr int FLOW_THREADS = 32 * (FLOW_B_WARP2 + 1);

enum { FLOW_FAST = 0, FLOW_FAST_SKIP8 = 1, FLOW_SAFE = 2, FLOW_SAFE_SKIP8 = 3, FLOW_PROJ_FAST = 4, FLOW_PROJ_SAFE = 5 };

struct FlowLayer {
    CUtensorMap x;                  // A operand: rows of a dense tensor (box {kc, rows}) or im2col
    CUtensorMap w;                  // packed weights, box {kc, block_n / 2}
    CUtensorMap out;                // output rows, box {piece, rows}
    CUtensorMap aux;                // skip rows (the box of `out`), or the projection's input (as x)
    const int32_t *c_a;             // the variant's per-channel constants
    int m_total, tiles, units, unit0;            // pixels; tiles; units of the layer; index of its first unit in the sequence of units
    int src_unit, aux_unit;         // first unit of the layers that write x and aux, or -1: not of this run
    int q_mul, q_h, skip_mul;
    unsigned nt_mul, w_mul, hw_mul;              // exact division by n_tiles, w_out, h_out * w_out (fast_div)
    unsigned short block_n, n_tiles, k_iters, p_iters;
    unsigned short h_out, w_out, h_in, w_in, h_aux, w_aux;
    unsigned char nt_shr, w_shr, hw_shr, q_shift, skip_shift, skip_signed;
    unsigned char kc, epi, cchunks, kh, kw, stride, pad, dense;
    unsigned char p_cchunks, p_k, p_stride, p_pad, p_dense;
    unsigned char rows, shift, src_shift, aux_shift;      // pixel rows per CTA; log2 of the pixels per unit: here, and of x's and aux's writers
};
struct FlowArgs {
    FlowLayer l[FLOW_MAX_LAYERS];
    unsigned *sync;                 // FLOW_SYNC_WORDS + units words, zero before and after every launch
    int *status;
    int n_layers, units;
};
static_assert(sizeof(FlowLayer) == 640 && sizeof(FlowArgs) <= 32764, "kernel arguments");

struct FlowShared {
    int consts[2][256];             // the staged tiles' per-channel constants (16-byte aligned: bulk copies)
    unsigned long long full[FLOW_STAGES], empty[FLOW_STAGES];
    unsigned long long tmem_full[2], tmem_empty[2];
    unsigned long long stg_full[2], stg_empty[2], out_ready[2];
    unsigned long long drain;
    int want;                       // unit the A warp waits for: whoever waits for a later layer asks less often
    int ready;                      // units of the sequence known to be stored by everybody: a prefix
    uint32_t tmem_base;
    volatile int abort_flag;
    int last_cta;
};

__device__ __forceinline__ void flow_give_up(FlowShared *sh, int *status, int code)
{
    sh->abort_flag = 1;
    atomicCAS(status, 0, code);
}

// A CTA pair's walk over its tiles.
struct FlowWalk {
    int layer, tile, t;             // layer, tile of the layer, index among the pair's tiles
    __device__ __forceinline__ FlowWalk(const FlowArgs &f, int first) : layer(0), tile(first), t(0) { settle(f); }
    __device__ __forceinline__ void settle(const FlowArgs &f)
    {
        while (layer < f.n_layers && tile >= f.l[layer].tiles) { tile -= f.l[layer].tiles; ++layer; }
    }
    __device__ __forceinline__ void next(const FlowArgs &f, int step)
    {
        tile += step;
        ++t;
        settle(f);
    }
};

// Last output pixel of a unit, and the last pixel of the input (h x w pixels per image) that a k x k / stride filter
// reads for it.
__device__ __forceinline__ int flow_last(const FlowLayer &L, int unit) { return min((unit + 1) << L.shift, L.m_total) - 1; }
__device__ __forceinline__ int flow_need(const FlowLayer &L, int unit, int k, int stride, int pad, int h, int w)
{
    const unsigned last = (unsigned)flow_last(L, unit);
    const unsigned img = fast_div(last, L.hw_mul, L.hw_shr);
    const unsigned p = fast_div(last - img * (unsigned)L.h_out * (unsigned)L.w_out, L.w_mul, L.w_shr);
    const int row = min((int)p * stride - pad + k - 1, h - 1);
    return (int)((img * (unsigned)h + (unsigned)row) * (unsigned)w + (unsigned)w - 1u);
}

// Wait of a loading warp until unit `need` of the sequence is stored; `ready` is the prefix it last saw.
__device__ __forceinline__ bool flow_wait_unit(FlowShared *sh, int need, int &ready)
{
    if (ready > need) return true;
    long long t0 = 0;
    for (unsigned spin = 1;; ++spin) {
        ready = ld_acquire_cta_shared(&sh->ready);
        if (__all_sync(0xffffffffu, ready > need)) break;
        if ((spin & 63u) == 0) {
            bool stop = sh->abort_flag != 0;
            const long long now = clock64();
            if (t0 == 0) t0 = now;
            else if (now - t0 > WAIT_LIMIT_CYCLES) stop = true;
            if (__any_sync(0xffffffffu, stop)) return false;
        }
    }
    ready = __reduce_min_sync(0xffffffffu, ready);   // (a lane may have seen more than another; this every lane has acquired)
    fence_async_proxy();                             // what the others stored, before this warp's bulk-asynchronous reads
    return true;
}

// A value that is to be in a register from here on.  What a role works out for a tile it works out BEFORE it waits for it: the layers'
// parameters come through the constant cache, which a new layer always misses, and a chain of such reads and divisions
// behind the wait would be part of every layer's latency: 800 cycles from a unit's arrival to the first load of it, 370 from a staged
// tile to its store (ResNet-50 of one image 258 -> 241 us, ResNet-18 of seven 142 -> 132, ResNet-152 of fifty 1112 -> 1068).
__device__ __forceinline__ void pin(int &v) { asm volatile("" : "+r"(v)); }
__device__ __forceinline__ void pin(uint32_t &v) { asm volatile("" : "+r"(v)); }

// One epilogue warp's part of a tile: groups of 16 columns from c0 on.  st: address of this lane's row in the
// staged tile's first piece; a column's 16 bytes are at piece (c / piece), chunk (c % piece) / 16 swizzled.
template <int EPI, int PROJ32>
__device__ __forceinline__ void flow_groups(uint32_t t_row, uint32_t consts, uint32_t st, uint32_t piece, uint32_t swz16, int c0, int groups, int block_n,
                                            EpiScalars es)
{
    constexpr bool SKIP8 = (EPI == EPI_FAST_SKIP8 || EPI == EPI_SAFE_SKIP8);
    es.proj32 = PROJ32;
    ConvArgs a = {};
    UmmaArgs u = {};
    const uint32_t mask = piece - 1u;
#pragma unroll 1
    for (int g = 0; g < groups; ++g) {
        const uint32_t c = (uint32_t)(c0 + (g << 4));
        const uint32_t at = st + (c & ~mask) * (uint32_t)BLOCK_M + ((c & mask) ^ swz16);
        int4 ca[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const uint4 v = lds128(consts + 4u * c + 16u * (uint32_t)k);
            ca[k] = make_int4((int)v.x, (int)v.y, (int)v.z, (int)v.w);
        }
        uint4 sk = make_uint4(0, 0, 0, 0);
        if (SKIP8) sk = lds128(at);
        int acc[16], accp[16], V[16];
        if (EPI == EPI_PROJ) tmem_ld16(t_row + (uint32_t)block_n + c, accp);
        tmem_ld16_sync(t_row + c, acc);
        epilogue16_pc<EPI, false>(acc, accp, V, ca, 0, 0, false, sk, es, a, u);
        uint4 o;
        o.x = pack4_sat<false>(V[0], V[1], V[2], V[3]); o.y = pack4_sat<false>(V[4], V[5], V[6], V[7]);
        o.z = pack4_sat<false>(V[8], V[9], V[10], V[11]); o.w = pack4_sat<false>(V[12], V[13], V[14], V[15]);
        sts128(at, o);
    }
}

__global__ void __launch_bounds__(FLOW_THREADS, 1) umma_flow_kernel(const __grid_constant__ FlowArgs f)
{
    // (all of shared memory is used: no room to align by hand; without static arrays the base is 1024-byte aligned)
    extern __shared__ __align__(1024) uint8_t smem_flow[];
    uint8_t *slots = smem_flow;
    if (smem_u32(slots) & 1023u) {
        if (threadIdx.x == 0) atomicCAS(f.status, 0, 7);
        return;
    }
    uint8_t *staging = slots + FLOW_STAGES * FLOW_SLOT;
    FlowShared *sh = (FlowShared *)(staging + 2 * FLOW_STAGING);
    const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0);
    const int lane = threadIdx.x & 31;
    const int rank = __shfl_sync(0xffffffffu, (int)cluster_rank(), 0);
    const int pair = (int)(blockIdx.x >> 1), step = (int)(gridDim.x >> 1);

    if (threadIdx.x == 0) {
        for (int s = 0; s < FLOW_STAGES; ++s) {
            mbar_init(smem_u32(&sh->full[s]), 2);                // the A and the B warp of the leader arm it
            mbar_init(smem_u32(&sh->empty[s]), 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(smem_u32(&sh->tmem_full[b]), 1);
            mbar_init(smem_u32(&sh->tmem_empty[b]), 2 * EPI_WARPS_MAX);      // both CTAs' epilogue warps, at the leader
            mbar_init(smem_u32(&sh->stg_full[b]), 1);
            mbar_init(smem_u32(&sh->stg_empty[b]), 1);
            mbar_init(smem_u32(&sh->out_ready[b]), EPI_WARPS_MAX);
        }
        mbar_init(smem_u32(&sh->drain), 1);
        sh->ready = 0;
        sh->want = 0;
        sh->abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == FLOW_MMA_WARP) tmem_alloc_pair(smem_u32(&sh->tmem_base), 512u);
    tc_fence_before();
    __syncthreads();
    cluster_sync_all();                          // the peer's barriers exist before anything arrives at them
    tc_fence_after();
    const uint32_t tmem_base = sh->tmem_base;
    const uint32_t full0 = smem_u32(&sh->full[0]), empty0 = smem_u32(&sh->empty[0]);
    const uint32_t slots0 = smem_u32(slots), staging0 = smem_u32(staging);

    if (warp == FLOW_A_WARP || warp == FLOW_A_WARP2) {
        // ---------------------------------------------------------------- activations
        // (two warps take the k-iterations in turn, and two those of the weights: a warp needs 300 to 400 cycles per
        // load, and a short tile's k-iteration is less than that)
        int turn = warp == FLOW_A_WARP ? 0 : 1;      // 0: the next k-iteration is this warp's
        int stage = 0, ready = 0;
        uint32_t parity = 0;
        bool ok = true, have = false;                // have: the next stage is known to be free
        // one k-iteration's 128 rows: waits for the stage, arms it (leader), loads
        auto load = [&](const CUtensorMap *map, bool dense, int bytes, int c, int x, int y, int img, int s, int r) {
            if (turn == 0) {
                if (!have && !mbar_wait_warp(empty0 + 8u * (uint32_t)stage, parity ^ 1u, &sh->abort_flag, lane)) {
                    flow_give_up(sh, f.status, 1);
                    ok = false;
                    return;
                }
                have = false;
                if (elect_one()) {
                    const uint32_t bar = full0 + 8u * (uint32_t)stage, dst = slots0 + (uint32_t)(stage * FLOW_SLOT);
                    if (rank == 0) mbar_expect_tx(bar, (uint32_t)(2 * bytes));
                    if (dense) tma_load_2d_pair(dst, map, bar & PEER_MASK, c, x);
                    else tma_load_im2col_4d_pair(dst, map, bar & PEER_MASK, c, x, y, img, (unsigned short)s, (unsigned short)r);
                }
                __syncwarp();
            }
            turn ^= 1;
            if (++stage == FLOW_STAGES) { stage = 0; parity ^= 1u; }
        };
        for (FlowWalk w(f, pair); ok && w.layer < f.n_layers; w.next(f, step)) {
            const FlowLayer &L = f.l[w.layer];
            const int unit = (int)fast_div((unsigned)w.tile, L.nt_mul, L.nt_shr);
            const int m0 = (unit << L.shift) + rank * L.rows;
            int need = -1;
            if (L.src_unit >= 0) need = L.src_unit + ((L.dense ? flow_last(L, unit) : flow_need(L, unit, L.kh, L.stride, L.pad, L.h_in, L.w_in)) >> L.src_shift);
            if (L.p_iters && L.aux_unit >= 0) 
                need = max(need, L.aux_unit + ((L.p_dense ? flow_last(L, unit) : flow_need(L, unit, L.p_k, L.p_stride, L.p_pad, L.h_aux, L.w_aux)) >> L.aux_shift));
            if (lane == 0) {
                if (warp == FLOW_A_WARP) *(volatile int *)&sh->want = need;
                prefetch_tensormap(&L.x);            // (the descriptor fetch would otherwise follow the wait)
                if (L.p_iters) prefetch_tensormap(&L.aux);
            }
            __syncwarp();
            int img = (int)fast_div((unsigned)m0, L.hw_mul, L.hw_shr);
            const int rem = m0 - img * (int)L.h_out * (int)L.w_out;
            const int p = (int)fast_div((unsigned)rem, L.w_mul, L.w_shr), q = rem - p * (int)L.w_out;
            int kc = L.kc, bytes = L.rows * kc, taps_h = L.kh, taps_w = L.kw, chunks = L.cchunks, dense = L.dense;
            int x = dense ? m0 : q * L.stride - L.pad, y = p * L.stride - L.pad;
            const int p_iters = L.p_iters;
            int p_taps = 0, p_chunks = 0, p_dense = 0, px = 0, py = 0;
            if (p_iters) {
                p_taps = L.p_k;
                p_chunks = L.p_cchunks;
                p_dense = L.p_dense;
                px = p_dense ? m0 : q * L.p_stride - L.p_pad;
                py = p * L.p_stride - L.p_pad;
            }
            pin(img); pin(kc); pin(bytes); pin(taps_h); pin(taps_w); pin(chunks); pin(dense); pin(x); pin(y);
            pin(p_taps); pin(p_chunks); pin(p_dense); pin(px); pin(py);
            if (turn == 0) {
                if (!mbar_wait_warp(empty0 + 8u * (uint32_t)stage, parity ^ 1u, &sh->abort_flag, lane)) {
                    flow_give_up(sh, f.status, 1);
                    break;
                }
                have = true;
            }
            if (!flow_wait_unit(sh, need, ready)) {
                flow_give_up(sh, f.status, 1);
                break;
            }
            for (int r = 0; r < p_taps && ok; ++r)
                for (int s = 0; s < p_taps && ok; ++s)
                    for (int cc = 0; cc < p_chunks && ok; ++cc) load(&L.aux, p_dense != 0, bytes, cc * kc, px, py, img, s, r);
            for (int r = 0; r < taps_h && ok; ++r)
                for (int s = 0; s < taps_w && ok; ++s)
                    for (int cc = 0; cc < chunks && ok; ++cc) load(&L.x, dense != 0, bytes, cc * kc, x, y, img, s, r);
        }
    } else if (warp == FLOW_B_WARP || warp == FLOW_B_WARP2) {
        // ---------------------------------------------------------------- weights (nothing to wait for but the stage)
        int turn = warp == FLOW_B_WARP ? 0 : 1;
        int stage = 0;
        uint32_t parity = 0;
        bool ok = true;
        for (FlowWalk w(f, pair); ok && w.layer < f.n_layers; w.next(f, step)) {
            const FlowLayer &L = f.l[w.layer];
            const int unit = (int)fast_div((unsigned)w.tile, L.nt_mul, L.nt_shr);
            const int half = L.block_n >> 1, row = (w.tile - unit * L.n_tiles) * L.block_n + rank * half;
            for (int ki = 0; ki < L.k_iters; ++ki, turn ^= 1) {
                if (turn) {
                    if (++stage == FLOW_STAGES) { stage = 0; parity ^= 1u; }
                    continue;
                }
                if (!mbar_wait_warp(empty0 + 8u * (uint32_t)stage, parity ^ 1u, &sh->abort_flag, lane)) {
                    flow_give_up(sh, f.status, 1);
                    ok = false;
                    break;
                }
                if (elect_one()) {
                    const uint32_t bar = full0 + 8u * (uint32_t)stage;
                    if (rank == 0) mbar_expect_tx(bar, (uint32_t)(2 * half * L.kc));
                    tma_load_2d_pair(slots0 + (uint32_t)(stage * FLOW_SLOT + FLOW_SLOT / 2), &L.w, bar & PEER_MASK, ki * L.kc, row);
                }
                __syncwarp();
                if (++stage == FLOW_STAGES) { stage = 0; parity ^= 1u; }
            }
        }
    } else if (warp == FLOW_READY_WARP) {
        // ---------------------------------------------------------------- counters -> ready (whole warp; a round stays inside a layer)
        int unit = 0, layer = 0;
        long long t0 = clock64();
        const int last = f.n_layers - 1;                  // (nobody waits for the last layer)
        while (layer < last) {
            const FlowLayer &L = f.l[layer];
            const int end = L.unit0 + L.units;
            bool full = false;
            if (unit + lane < end) full = ld_acquire_gpu(f.sync + FLOW_SYNC_WORDS + unit + lane) >= 2u * L.n_tiles;
            const unsigned open = __ballot_sync(0xffffffffu, !full);
            const int n = open ? __ffs((int)open) - 1 : 32;
            if (n) {
                unit += n;
                __syncwarp();                             // what the lanes acquired, before the release of one of them (votes order no memory)
                if (lane == 0) st_release_cta_shared(&sh->ready, unit);
                __syncwarp();
                if (unit == end) ++layer;
                t0 = clock64();
            } else {
                if (__any_sync(0xffffffffu, sh->abort_flag != 0 || clock64() - t0 > WAIT_LIMIT_CYCLES)) break;
                if (*(volatile int *)&sh->want >= end) __nanosleep(200);
            }
        }
    } else if (warp == FLOW_MMA_WARP) {
        // ---------------------------------------------------------------- MMA issuer (the leader's; whole warp, an elected lane issues)
        if (rank == 0) {
            int stage = 0;
            uint32_t parity = 0;
            bool ok = true;
            for (FlowWalk w(f, pair); ok && w.layer < f.n_layers; w.next(f, step)) {
                const FlowLayer &L = f.l[w.layer];
                const int buf = w.t & 1;
                if (!mbar_wait_warp(smem_u32(&sh->tmem_empty[buf]), (uint32_t)(((w.t >> 1) & 1) ^ 1), &sh->abort_flag, lane)) {
                    flow_give_up(sh, f.status, 2);
                    break;
                }
                tc_fence_after();
                // D = s32, A = u8, B = s8, both K-major, N / 8, M / 16 (both CTAs' rows)
                const uint32_t idesc = (2u << 4) | (1u << 10) | ((uint32_t)(L.block_n >> 3) << 17) | ((uint32_t)((2 * BLOCK_M) >> 4) << 24);
                // 8-row groups 8 * kc bytes apart, descriptor version 1, swizzle of kc bytes (128: 2, 64: 4)
                const uint32_t desc_hi = ((uint32_t)(8 * L.kc) >> 4) | (1u << 14) | ((L.kc == 128 ? 2u : 4u) << 29);
                const uint32_t d_tmem = tmem_base + (uint32_t)(buf * 256);
                const int k_iters = L.k_iters, p_iters = L.p_iters;
                const bool wide = L.kc == 128;
                for (int ki = 0; ki < k_iters; ++ki) {
                    if (!mbar_wait_warp(full0 + 8u * (uint32_t)stage, parity, &sh->abort_flag, lane)) {
                        flow_give_up(sh, f.status, 3);
                        ok = false;
                        break;
                    }
                    if (elect_one()) {
                        const uint32_t a_lo = (((slots0 + (uint32_t)(stage * FLOW_SLOT)) & 0x3FFFFu) >> 4) | (1u << 16);
                        const uint32_t b_lo = a_lo + (FLOW_SLOT / 2 >> 4);
                        const uint32_t d = ki < p_iters ? d_tmem + (uint32_t)L.block_n : d_tmem;       // a projection has its own accumulator
                        umma_i8_pair(d, a_lo, b_lo, desc_hi, idesc, (uint32_t)(ki != 0 && ki != p_iters));
                        umma_i8_pair(d, a_lo + 2u, b_lo + 2u, desc_hi, idesc, 1u);
                        if (wide) {
                            umma_i8_pair(d, a_lo + 4u, b_lo + 4u, desc_hi, idesc, 1u);
                            umma_i8_pair(d, a_lo + 6u, b_lo + 6u, desc_hi, idesc, 1u);
                        }
                        umma_commit_pair(empty0 + 8u * (uint32_t)stage);
                        if (ki == k_iters - 1) umma_commit_pair(smem_u32(&sh->tmem_full[buf]));
                    }
                    __syncwarp();
                    if (++stage == FLOW_STAGES) { stage = 0; parity ^= 1u; }
                }
            }
        }
    } else if (warp == FLOW_SKIP_WARP) {
        // ---------------------------------------------------------------- constants and skip of the next tiles
        int ready = 0;
        for (FlowWalk w(f, pair); w.layer < f.n_layers; w.next(f, step)) {
            const FlowLayer &L = f.l[w.layer];
            const int s = w.t & 1;
            if (!mbar_wait_warp(smem_u32(&sh->stg_empty[s]), (uint32_t)(((w.t >> 1) & 1) ^ 1), &sh->abort_flag, lane)) {
                flow_give_up(sh, f.status, 5);
                break;
            }
            const int unit = (int)fast_div((unsigned)w.tile, L.nt_mul, L.nt_shr);
            const int n0 = (w.tile - unit * L.n_tiles) * L.block_n, m0 = (unit << L.shift) + rank * L.rows;
            const bool skip = L.epi == FLOW_FAST_SKIP8 || L.epi == FLOW_SAFE_SKIP8;
            if (skip && lane == 0) prefetch_tensormap(&L.aux);
            __syncwarp();
            if (skip && L.aux_unit >= 0 && !flow_wait_unit(sh, L.aux_unit + (flow_last(L, unit) >> L.aux_shift), ready)) {
                flow_give_up(sh, f.status, 5);
                break;
            }
            if (elect_one()) {
                const uint32_t bar = smem_u32(&sh->stg_full[s]);
                mbar_expect_tx(bar, (uint32_t)L.block_n * (skip ? 4u + L.rows : 4u));
                bulk_load(smem_u32(&sh->consts[s][0]), L.c_a + n0, (uint32_t)L.block_n * 4u, bar);
                if (skip) {
                    const int piece = min((int)L.block_n, 64);
                    for (int c = 0; c < L.block_n; c += piece)
                        tma_load_2d(staging0 + (uint32_t)(s * FLOW_STAGING + c * BLOCK_M), &L.aux, bar, n0 + c, m0);
                }
            }
            __syncwarp();
        }
    } else if (warp >= FLOW_STORE_WARP && warp < FLOW_STORE_WARP + FLOW_STORE_WARPS) {
        // ---------------------------------------------------------------- staged tiles -> memory -> counters (one lane: its bulk groups)
        if (lane == 0) {
            for (FlowWalk w(f, pair); w.layer < f.n_layers; w.next(f, step)) {
                if ((w.t & 1) != warp - FLOW_STORE_WARP) continue;
                const FlowLayer &L = f.l[w.layer];
                const int s = w.t & 1;
                prefetch_tensormap(&L.out);
                int unit = (int)fast_div((unsigned)w.tile, L.nt_mul, L.nt_shr);
                int n0 = (w.tile - unit * L.n_tiles) * L.block_n, m0 = (unit << L.shift) + rank * L.rows;
                int piece = min((int)L.block_n, 64), columns = m0 < L.m_total ? (int)L.block_n : 0;
                unit += L.unit0;
                pin(unit); pin(n0); pin(m0); pin(piece); pin(columns);
                if (!mbar_wait(smem_u32(&sh->out_ready[s]), (uint32_t)((w.t >> 1) & 1), &sh->abort_flag)) {
                    flow_give_up(sh, f.status, 4);
                    break;
                }
                for (int c = 0; c < columns; c += piece)
                        asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.bulk_group [%0, {%2, %3}], [%1];"
                                     ::"l"(&L.out), "r"(staging0 + (uint32_t)(s * FLOW_STAGING + c * BLOCK_M)), "r"(n0 + c), "r"(m0)
                                     : "memory");
                asm volatile("cp.async.bulk.commit_group;" ::: "memory");
                asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
                mbar_arrive(smem_u32(&sh->stg_empty[s]));
                asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
                fence_async_proxy();
                fence_acq_rel_gpu();
                red_relaxed_gpu(f.sync + FLOW_SYNC_WORDS + unit, 1u);
            }
        }
        __syncwarp();
    } else {
        // ---------------------------------------------------------------- epilogue
        const int quad = warp & 3, part = (warp - EPI_WARP0) >> 2;
        const uint32_t t_quad = tmem_base + ((uint32_t)(quad * 32) << 16);
        for (FlowWalk w(f, pair); w.layer < f.n_layers; w.next(f, step)) {
            const FlowLayer &L = f.l[w.layer];
            const int s = w.t & 1;
            const uint32_t phase = (uint32_t)((w.t >> 1) & 1);
            int block_n = L.block_n, rows = L.rows, epi = L.epi;
            EpiScalars es = {};
            es.q_mul = L.q_mul; es.q_shift = L.q_shift; es.q_h = L.q_h; es.q_half = 1 << (L.q_shift - 1);
            es.skip_mul = L.skip_mul; es.skip_shift = L.skip_shift; es.skip_xor = L.skip_signed ? 0x80808080u : 0u;
            pin(block_n); pin(rows); pin(epi); pin(es.q_mul); pin(es.q_shift); pin(es.q_h); pin(es.q_half); pin(es.skip_mul); pin(es.skip_shift); pin(es.skip_xor);
            if (!mbar_wait_warp(smem_u32(&sh->stg_full[s]), phase, &sh->abort_flag, lane)) {
                flow_give_up(sh, f.status, 5);
                break;
            }
            if (!mbar_wait_warp(smem_u32(&sh->tmem_full[s]), phase, &sh->abort_flag, lane)) {
                flow_give_up(sh, f.status, 4);
                break;
            }
            tc_fence_after();
            // sixteen-column groups: a quarter of the tile's per part (parts 2 and 3 have none in a 32-column tile)
            const int groups = quad * 32 >= rows ? 0 : block_n >= 64 ? block_n >> 6 : (part < 2 ? 1 : 0);
            const int c0 = part * (block_n >= 64 ? block_n >> 2 : 16);
            const uint32_t piece = (uint32_t)min(block_n, 64);
            const unsigned row = (unsigned)(quad * 32 + lane);
            const uint32_t st = staging0 + (uint32_t)(s * FLOW_STAGING) + row * piece;
            const uint32_t swz16 = piece == 64 ? ((row >> 1) & 3u) << 4 : ((row >> 2) & 1u) << 4;
            const uint32_t t_row = t_quad + (uint32_t)(s * 256), consts = smem_u32(&sh->consts[s][0]);
            switch (epi) {
            case FLOW_FAST: flow_groups<EPI_FAST, 0>(t_row, consts, st, piece, swz16, c0, groups, block_n, es); break;
            case FLOW_FAST_SKIP8: flow_groups<EPI_FAST_SKIP8, 0>(t_row, consts, st, piece, swz16, c0, groups, block_n, es); break;
            case FLOW_SAFE: flow_groups<EPI_SAFE, 0>(t_row, consts, st, piece, swz16, c0, groups, block_n, es); break;
            case FLOW_SAFE_SKIP8: flow_groups<EPI_SAFE_SKIP8, 0>(t_row, consts, st, piece, swz16, c0, groups, block_n, es); break;
            case FLOW_PROJ_FAST: flow_groups<EPI_PROJ, 2>(t_row, consts, st, piece, swz16, c0, groups, block_n, es); break;
            default: flow_groups<EPI_PROJ, 1>(t_row, consts, st, piece, swz16, c0, groups, block_n, es); break;
            }
            tc_fence_before();
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            __syncwarp();
            if (lane == 0) {
                mbar_arrive_leader(smem_u32(&sh->tmem_empty[s]));
                mbar_arrive(smem_u32(&sh->out_ready[s]));
            }
        }
    }

    // ---------------------------------------------------------------- teardown
    if (threadIdx.x == 0) grid_dep_launch();         // the kernel after this one may come up while the last CTAs finish
    __syncwarp();
    tc_fence_before();
    __syncthreads();
    if (sh->abort_flag) {
        // something gave up: whatever was handed to the TMA unit has landed long before this spin ends, then the MMAs
        const long long t0 = clock64();
        while (clock64() - t0 < 2000000) {}
        if (warp == FLOW_MMA_WARP && lane == 0 && rank == 0) {
            volatile int never = 0;
            umma_commit_pair(smem_u32(&sh->drain));
            mbar_wait(smem_u32(&sh->drain), 0, &never);
        }
        __syncthreads();
    }
    // neither CTA may leave (or give back its TMEM) while the other can still reach it
    cluster_sync_all();
    if (warp == FLOW_MMA_WARP) {
        tc_fence_after();
        tmem_dealloc_pair(tmem_base, 512u);
    }
    // the last CTA to get here leaves the counters as it found them
    if (threadIdx.x == 0) {
        __threadfence();
        sh->last_cta = atomicAdd(f.sync, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (sh->last_cta)
        for (int i = (int)threadIdx.x; i < FLOW_SYNC_WORDS + f.units; i += FLOW_THREADS) f.sync[i] = 0u;
}

}  // namespace iconv

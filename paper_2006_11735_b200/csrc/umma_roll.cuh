// Stride-1 filters over few channels, several filter rows per instruction.
//
// A K = 32 instruction reads its 128 rows of A from shared memory whatever its width, and that takes 48 cycles
// for 64 output channels where the arithmetic takes 32 (measured: N = 16 39 cycles, 48 44, 64 48, 128 64,
// 192 96, 240 120).  So a layer of 64 channels in the window kernel, one filter tap per instruction, can use
// two thirds of the tensor pipe and one of 48 half of it.  Here one instruction covers ALL kh filter rows of
// a tap column: input row i of a strip of 128 pixels contributes to output rows i - pad ... i + pad, whose
// accumulators lie side by side in tensor memory; the filter bank is packed so that the kh taps of a column
// are neighbouring rows of B in the order of the output rows they go to:
//
//   D[rows i - pad ... i + pad][128 pixels x kh * block_n] += A[input row i, shifted by s] x B[s]
//
// The accumulators of consecutive output rows form a ring in tensor memory (8 rows, 10 under a 5x5 filter); a range
// that wraps is two instructions, and a row's first contribution is an instruction of its own that does not
// accumulate.  3x3 of 64 channels: 592 cycles per input row against 18 x 48 = 864 for the taps one by one; 5x5
// of 48: 1220 against 50 x 44 = 2200.
//
// What this relies on: instructions of one issuing thread add to an accumulator in the order of their issue also where
// their N, and so the ranges of accumulators that they cover, differ (a row is opened by an instruction of BN columns
// that does not accumulate, and the next ones, of up to kh * BN columns at another first column, add to it).  The PTX
// ISA promises the order for the same accumulator and shape only, and a commit and a wait between the others would
// cost what the form gains.  The tensor core takes a CTA's instructions one after another whatever their N: every
// filter size and width (all but 3x3 of 48 and 64 columns also with explicit clamps) is compared bit for bit with the
// integer oracle over tens of rows per CTA (tests/test_gpu_layers.py), where one lost partial sum would show.
//
// A tile is a strip of 128 pixels x up to `rows` output rows; its rows + kh - 1 input rows stream through a
// ring of single-row stages (one TMA copy each, zero outside the image), as many as there are accumulator
// rows.  EVERY input row opens an output row and closes one: the last kh - 1 rows that a tile opens are not
// outputs (what the next tile adds to them is nobody's), the epilogue passes over them.  So all rows are
// alike, the issuing warp's loop is unrolled over the ring, and every address in it is an immediate.
// That warp is what bounds the kernel when it does more than issue: the tensor pipe queues hardly more than an
// instruction, a barrier that is already complete costs a warp 140 cycles to look at, a commit 60 to 100, and with
// the bookkeeping of open and closed rows done at run time its own instructions took 1200 cycles a row.  So another
// warp (the gate) waits for a row's pixels and accumulators and raises a count in shared memory, which the
// issuer looks at when it has used up the rows it knows of; and one commit per row tells the loader that the stage,
// and the epilogue that the row closed kh - 1 rows ago, is done.  16 epilogue warps take the finished rows in turn, 32 pixels of a row
// each, with the window kernel's epilogue.
#pragma once

#include "umma_stack.cuh"         // stack_wait_ready

namespace iconv {

constexpr int ROLL_MAX_SLOTS = 10;
__host__ __device__ constexpr int roll_slots(int kh) { return kh == 5 ? 10 : 8; }        // accumulator rows, and stages
constexpr int ROLL_GATE_WARP = 1;
constexpr int ROLL_GROUPS = 4;           // epilogue warps per lane quadrant: they take the rows in turn

struct RollArgs {
    int tiles;
    int strips, rows, bands;             // strips per image row; output rows per tile; tiles per strip of an image
    int h, w, pad;
    int stage_bytes, tmem_cols;
    unsigned idesc;                      // without N
    unsigned div_strips_mul, div_strips_shr, div_bands_mul, div_bands_shr;
    int *status;
};

struct RollShared {
    unsigned long long full[ROLL_MAX_SLOTS], done[ROLL_MAX_SLOTS];       // a stage's row is there; its MMAs are done
    unsigned long long tmem_empty[ROLL_MAX_SLOTS];                      // an accumulator row may be opened again
    unsigned long long b_full;
    unsigned long long drain;
    int go;                              // input rows whose pixels and accumulators are ready
    uint32_t tmem_base;
    volatile int abort_flag;
};

__device__ __forceinline__ void roll_give_up(RollShared *sh, int *status, int code)
{
    sh->abort_flag = 1;
    atomicCAS(status, 0, code);
}

// A CTA's walk over its tiles: first pixel, output rows.
struct RollWalk {
    int tile, img, x0, y0, rows;
    __device__ __forceinline__ RollWalk(const RollArgs &u, int first) : tile(first) { locate(u); }
    __device__ __forceinline__ void locate(const RollArgs &u)
    {
        const unsigned line = fast_div((unsigned)tile, u.div_strips_mul, u.div_strips_shr);       // image * bands + band
        img = (int)fast_div(line, u.div_bands_mul, u.div_bands_shr);
        x0 = (tile - (int)line * u.strips) * BLOCK_M;
        y0 = ((int)line - img * u.bands) * u.rows;
        rows = min(u.rows, u.h - y0);
    }
    __device__ __forceinline__ void next(const RollArgs &u, int step)
    {
        tile += step;
        locate(u);
    }
};

template <bool FIRST, typename A, typename B> struct RollPick { using type = A; };
template <typename A, typename B> struct RollPick<false, A, B> { using type = B; };

template <int EPI, int KH, int BN>
__global__ void __launch_bounds__(NUM_THREADS, 1)
umma_roll_kernel(const __grid_constant__ CUtensorMap map_x, const __grid_constant__ CUtensorMap map_w, const __grid_constant__ RollArgs u, const __grid_constant__ ConvArgs a, const __grid_constant__ UmmaArgs ua)
{
    constexpr int KW = KH, KJ = 2, KC = 64;                                // K = 32 steps of a pixel, its bytes
    constexpr int S = roll_slots(KH);                                      // accumulator rows = stages
    constexpr int TAP = BN * KC, BANK = TAP * KH * KW;                     // bytes of a tap's and of the whole filter bank
    constexpr int STAGE = ((BLOCK_M + KW - 1) * KC + 1023) / 1024 * 1024;
    static_assert(KH * BN <= 256 && S * BN <= 512 && TAP % 512 == 0, "");
    extern __shared__ uint8_t smem_raw[];
    uint8_t *stages = (uint8_t *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    uint8_t *banks = stages + S * STAGE;
    RollShared *sh = (RollShared *)(banks + BANK);
    const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0);
    const int lane = threadIdx.x & 31;
    const int G = (int)gridDim.x;

    if (threadIdx.x == 0) {
        for (int s = 0; s < S; ++s) {
            mbar_init(smem_u32(&sh->full[s]), 1);
            mbar_init(smem_u32(&sh->done[s]), 1);
            mbar_init(smem_u32(&sh->tmem_empty[s]), 4);
        }
        mbar_init(smem_u32(&sh->b_full), 1);
        mbar_init(smem_u32(&sh->drain), 1);
        sh->go = 0;
        sh->abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        grid_dep_launch();
    }
    if (threadIdx.x == 32) {
        prefetch_tensormap(&map_x);
        prefetch_tensormap(&map_w);
    }
    if (warp == MMA_WARP) tmem_alloc(smem_u32(&sh->tmem_base), (uint32_t)u.tmem_cols);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = sh->tmem_base;

    int last_stage = -1;
    bool b_issued = false;
    uint32_t last_parity = 0;

    if (warp == 0) {
        // ---------------------------------------------------------------- TMA producer (whole warp; an elected lane issues)
        // Tap (r, s) becomes row block kh - 1 - r of column s: the order of the output rows that an input row contributes to.
        if ((int)blockIdx.x < u.tiles) {
            if (elect_one()) {
                const uint32_t bf = smem_u32(&sh->b_full), dst = smem_u32(banks);
                mbar_expect_tx(bf, (uint32_t)BANK);
                for (int r = 0; r < KH; ++r)
                    for (int s = 0; s < KW; ++s)
                        tma_load_2d(dst + (uint32_t)((s * KH + KH - 1 - r) * TAP), &map_w, bf, (r * KW + s) * KC, 0);
            }
            __syncwarp();
            b_issued = true;
        }
        int stage = 0;
        uint32_t parity = 0;
        const uint32_t tx = (uint32_t)(KC * (BLOCK_M + KW - 1));
        bool ok = true;
        grid_dep_wait();                                // the activations may come from the kernel before this one
        for (RollWalk w(u, (int)blockIdx.x); ok && w.tile < u.tiles; w.next(u, G)) {
            for (int e = 0; e < w.rows + KH - 1; ++e) {
                if (!mbar_wait_warp(smem_u32(&sh->done[stage]), parity ^ 1u, &sh->abort_flag, lane)) {
                    roll_give_up(sh, u.status, 1);
                    ok = false;
                    break;
                }
                if (elect_one()) {
                    const uint32_t full = smem_u32(&sh->full[stage]);
                    mbar_expect_tx(full, tx);
                    tma_load_tile_4d(smem_u32(stages) + (uint32_t)(stage * STAGE), &map_x, full, 0, w.x0 - u.pad, w.y0 - u.pad + e, w.img);
                }
                __syncwarp();
                last_stage = stage;
                last_parity = parity;
                if (++stage == S) { stage = 0; parity ^= 1u; }
            }
        }
        __syncwarp();
    } else if (warp == MMA_WARP) {
        // ---------------------------------------------------------------- MMA issuer (whole warp; an elected lane issues)
        const uint32_t a_lo0 = ((smem_u32(stages) & 0x3FFFFu) >> 4) | (1u << 16);
        const uint32_t bank = ((smem_u32(banks) & 0x3FFFFu) >> 4) | (1u << 16);
        const uint32_t done0 = smem_u32(&sh->done[0]);
        constexpr uint32_t HI = (uint32_t)((8 * KC) >> 4) | (1u << 14) | (4u << 29);           // 8-row groups 512 bytes apart, version 1, 64-byte swizzle
        constexpr uint32_t UNIT = (uint32_t)(BN >> 3) << 17;                                   // a row's share of the instruction descriptor's N
        RollWalk w(u, (int)blockIdx.x);
        int left = w.rows + KH - 1;                       // input rows left of the tile
        int issued = 0, known = 0, budget = 0;            // rows issued; rows the gate has let through; rows to issue without a look at either
        bool ok = true, bank_there = false;
        auto refill = [&]() -> bool {                     // false: nothing left to issue, or a wait gave up
            if (left == 0) {
                w.next(u, G);
                left = w.rows + KH - 1;
            }
            if (w.tile >= u.tiles) return false;
            if (!bank_there) {
                if (!mbar_wait_warp(smem_u32(&sh->b_full), 0u, &sh->abort_flag, lane)) {
                    roll_give_up(sh, u.status, 6);
                    return false;
                }
                bank_there = true;
            }
            if (issued >= known) {
                if (!stack_wait_ready(&sh->go, issued, known, &sh->abort_flag)) {
                    roll_give_up(sh, u.status, 3);
                    return false;
                }
            }
            tc_fence_after();
            budget = min(left, known - issued);
            left -= budget;
            issued += budget;
            return true;
        };
        while (ok) {
#pragma unroll
            for (int s = 0; s < S; ++s) {
                if (budget == 0 && !(ok = refill())) break;
                --budget;
                if (elect_one()) {
                    // the open rows: slots s - KH + 1 ... s, of which the first W wrap to the ring's end
                    const int W = s < KH - 1 ? KH - 1 - s : 0, n = KH - W;
                    const uint32_t d_wrap = tmem_base + (uint32_t)((S - W) * BN), d_row = tmem_base + (uint32_t)((W ? 0 : s - KH + 1) * BN);
                    const uint32_t a_row = a_lo0 + (uint32_t)((s * STAGE) >> 4);
#pragma unroll
                    for (int k = 0; k < KW * KJ; ++k) {
                        // K step k: A shifted by k / KJ pixels, B's column k / KJ
                        const uint32_t ka = a_row + (uint32_t)((k / KJ) * (KC >> 4) + 2 * (k % KJ)), kb = bank + (uint32_t)(((k / KJ) * KH * TAP) >> 4) + 2u * (uint32_t)(k % KJ);
                        const uint32_t kb_row = kb + (uint32_t)((W * TAP) >> 4);
                        if (W) umma_i8_split(d_wrap, ka, kb, HI, u.idesc + (uint32_t)W * UNIT, 1u);
                        if (k) {
                            umma_i8_split(d_row, ka, kb_row, HI, u.idesc + (uint32_t)n * UNIT, 1u);
                        } else {                          // the last of them opens: its first instruction does not accumulate
                            if (n > 1) umma_i8_split(d_row, ka, kb_row, HI, u.idesc + (uint32_t)(n - 1) * UNIT, 1u);
                            umma_i8_split(d_row + (uint32_t)((n - 1) * BN), ka, kb_row + (uint32_t)(((n - 1) * TAP) >> 4), HI, u.idesc + UNIT, 0u);
                        }
                    }
                    umma_commit(done0 + 8u * s);
                }
            }
        }
        __syncwarp();
    } else if (warp == ROLL_GATE_WARP) {
        // ---------------------------------------------------------------- gate: pixels and accumulators of a row -> count
        int s = 0, rows = 0;
        uint32_t parity = 0;
        bool ok = true;
        for (RollWalk w(u, (int)blockIdx.x); ok && w.tile < u.tiles; w.next(u, G)) {
            for (int e = 0; e < w.rows + KH - 1; ++e) {
                if (!mbar_wait_warp(smem_u32(&sh->tmem_empty[s]), parity ^ 1u, &sh->abort_flag, lane)) {
                    roll_give_up(sh, u.status, 2);
                    ok = false;
                    break;
                }
                if (!mbar_wait_warp(smem_u32(&sh->full[s]), parity, &sh->abort_flag, lane)) {
                    roll_give_up(sh, u.status, 3);
                    ok = false;
                    break;
                }
                tc_fence_after();
                __syncwarp();
                if (lane == 0) st_release_cta_shared(&sh->go, ++rows);
                if (++s == S) { s = 0; parity ^= 1u; }
            }
        }
        __syncwarp();
    } else if (warp >= EPI_WARP0 && warp < EPI_WARP0 + EPI_WARPS_MAX) {
        // ---------------------------------------------------------------- epilogue: group `turn` takes every fourth opened row
        grid_dep_wait();                                // the skip operand may come from the kernel before this one
        const int ew = warp - EPI_WARP0;
        const int quad = warp & 3, turn = ew >> 2;
        const EpiScalars es = epi_scalars(a, ua);
        struct None { __device__ None(const UmmaArgs &) {} };
        const typename RollPick<EPI == EPI_NARROW, NarrowOne, None>::type one(ua);
        uint8_t *out = (uint8_t *)a.out + a.out_c_offset;
        int row = turn, slot = turn;                    // row of the tile; its accumulators' slot
        int closer = turn + KH - 1;                     // the stage of the row that closes it
        uint32_t parity = 0;
        if (closer >= S) { closer -= S; parity ^= 1u; }
        for (RollWalk w(u, (int)blockIdx.x); w.tile < u.tiles;) {
            if (row >= w.rows + KH - 1) {
                row -= w.rows + KH - 1;
                w.next(u, G);
                continue;
            }
            // (the last rows that the CTA opens are never closed, and nobody opens their slots again)
            if (row >= w.rows && w.tile + G >= u.tiles) break;
            const int x = w.x0 + quad * 32 + lane, y = w.y0 + row;
            const bool valid = x < u.w && row < w.rows;
            const long long mpix = ((long long)w.img * u.h + y) * u.w + x;
            int sk_one = 0;
            if constexpr (EPI == EPI_NARROW) sk_one = a.c_out == 1 ? one.skip(valid, mpix, a) : 0;
            if (!mbar_wait_warp(smem_u32(&sh->done[closer]), parity, &sh->abort_flag, lane)) {
                roll_give_up(sh, u.status, 4);
                break;
            }
            tc_fence_after();
            if (row < w.rows) {
                uint8_t *ocol = out + mpix * a.out_c_total;
                const uint32_t t_row = tmem_base + ((uint32_t)(quad * 32) << 16) + (uint32_t)(slot * BN);
                constexpr int NG = BN / 16;
                int accA[16];
                if constexpr (EPI == EPI_NARROW) {
                    if (a.c_out == 1) one.store(t_row, ocol, valid, sk_one, a);
                    else window_narrow(t_row, ocol, valid, 0, NG, mpix, accA, a, ua);
                } else {
                    const int4 *cap = (const int4 *)ua.c_a;
                    if (es.group_uniform) window_groups<EPI, NG, true>(t_row, cap, ocol, nullptr, valid, 0, NG, accA, es, a, ua);
                    else window_groups<EPI, NG, false>(t_row, cap, ocol, nullptr, valid, 0, NG, accA, es, a, ua);
                }
                tc_fence_before();
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&sh->tmem_empty[slot]));
            row += ROLL_GROUPS;
            slot += ROLL_GROUPS;
            if (slot >= S) slot -= S;
            closer += ROLL_GROUPS;
            if (closer >= S) { closer -= S; parity ^= 1u; }
        }
    }

    // ---------------------------------------------------------------- teardown
    __syncwarp();
    tc_fence_before();
    __syncthreads();
    if (sh->abort_flag) {
        volatile int never = 0;
        if (warp == 0 && lane == 0) {
            if (b_issued) mbar_wait(smem_u32(&sh->b_full), 0, &never);
            if (last_stage >= 0) mbar_wait(smem_u32(&sh->full[last_stage]), last_parity, &never);
            const long long t0 = clock64();
            while (clock64() - t0 < 2000000) {}
        }
        if (warp == MMA_WARP && lane == 0) {
            umma_commit(smem_u32(&sh->drain));
            mbar_wait(smem_u32(&sh->drain), 0, &never);
        }
        __syncthreads();
    }
    if (warp == MMA_WARP) {
        tc_fence_after();
        tmem_dealloc(tmem_base, (uint32_t)u.tmem_cols);
    }
}

}  // namespace iconv

// A stack of equal stride-1 layers in ONE launch: consecutive convolutions of the same geometry, each
// reading what the one before wrote (Section 3.1: V_i is the input of layer i + 1; the twenty 3x3
// layers of the VDSR-shaped network).
//
// What it is for: launched one by one, such layers each pay a set-up, an empty pipeline, a last wave
// that leaves SMs idle and a drain around their loop.  Here a CTA walks the tiles of ALL layers as one
// sequence (g = layer * tiles + tile, CTA c takes g = c, c + grid, ...), so the pipeline never empties
// and the remainders of the layers' waves add up to one.  A tile may start when the tiles of the layer
// before that its patch touches are stored; the next layer's filter bank is fetched while this one runs
// (two banks in shared memory).  Whole forwards of the VDSR shape when this came: 16 x 256 x 256 from 773 to
// 711 us, 1 x 481 x 321 from 170 to 147 us (682 and 129 since, with the fences below for global memory only and
// other first and last layers).
// What bounds it now: at 16 x 256 x 256 the tensor pipe (878 cycles per tile of 18 instructions at 48
// cycles, the rate for 64 columns) at the clock the power limit leaves; at 481 x 321 the memory system
// under reads of lines just written (10 100 cycles per layer without any waiting for tiles, 7 700 with
// the stores or the reads taken out) and the way from a store to the tile that waits for it (3 000).
//
// The order between CTAs: an epilogue warp, after its stores, raises its progress word in shared memory;
// one warp that does nothing else turns progress into tiles, fences once for all that are new and adds
// them to the counters of their chunks (STACK_CHUNK consecutive tiles of a layer).  (A device-scope
// fence waits for the SM's stores in flight, some thousand cycles here: with one by every epilogue warp
// and tile a layer of 16 x 256 x 256 took 46.9 us instead of 33.5 launched alone.)  Another
// warp follows the counters (acquire, 32 at a time) and keeps the prefix of the sequence that is
// stored in shared memory, where the loading warp finds it (polling from the loading warp itself took
// it half of its time: 28 600 of 64 600 cycles per layer).  A change of the prefix is fenced against
// the bulk-asynchronous reads that follow.  A CTA takes its tiles in order
// and a tile only depends on tiles with a smaller g, so the launch cannot lock up as long as all CTAs
// are resident: one per SM, launched cooperatively.  Waits are bounded as everywhere.
//
// Everything else (patch per tile, taps as shifted views, issuing warps, epilogue) is the window
// kernel's, see umma_device.cuh.
#pragma once

#include "umma_device.cuh"

namespace iconv {

constexpr int STACK_CHUNK = 16;          // tiles per counter
constexpr int STACK_ISSUERS = 2;         // (two divide the accumulator buffers, and leave a warp for the counters)
constexpr int STACK_READY_WARP = 2;
constexpr int STACK_SIGNAL_WARP = EPI_WARP0 + EPI_WARPS_MAX;
constexpr int STACK_THREADS = NUM_THREADS + 32;
constexpr int STACK_SYNC_WORDS = 32;     // words before the counters; word 0: CTAs that are done

constexpr int STACK_MAX_LAYERS = 32;     // the layers travel as kernel arguments (a tensor map in device memory would cost fences)

struct StackLayer {
    CUtensorMap x;                  // patch map over the layer's input
    CUtensorMap w;                  // 3-D map over its packed weights: one box is the whole filter bank
    const int32_t *c_a;             // [block_n] b * mul + 2^(shift-1)
    uint8_t *out;                   // output slice (channel offset applied)
    int out_c_total, q_mul, q_shift, pad_[9];
};
struct StackLayers {
    StackLayer l[STACK_MAX_LAYERS];
};

struct StackArgs {
    int n_layers, tiles;            // tiles per layer
    int chunks;                     // counters per layer
    int fwd;                        // a tile needs the tiles of the layer before up to its own index + fwd (inside its image)
    int h, w, c_out, pad;
    int block_n, kc, stages, stage_bytes, b_tile_bytes, tmem_cols, nbuf, lg_nbuf, cs, bi, part_n, epi_warps;
    int vw, bw, bh, full_width, blocks, tpi;      // tiling of an image, as in UmmaArgs
    unsigned idesc, desc_hi_a, desc_hi_b;
    unsigned div_tpi_mul, div_tpi_shr, div_vw_mul, div_vw_shr;
    unsigned *sync;                 // STACK_SYNC_WORDS + n_layers * chunks words, zero before and after every launch
    int *status;
};

struct StackShared {
    unsigned long long full[MAX_STAGES], empty[MAX_STAGES];
    unsigned long long tmem_full[MAX_TMEM_BUFS], tmem_empty[MAX_TMEM_BUFS];
    unsigned long long b_full[2], b_empty[2];
    unsigned long long drain;
    int ready;                           // tiles of the sequence (layer * tiles + tile) known to be stored by everybody: a prefix
    int progress[EPI_WARPS_MAX];         // per epilogue warp: 1 + the CTA's tile index it stored last
    uint32_t tmem_base;
    volatile int abort_flag;
    int last_cta;
};

__device__ __forceinline__ void stack_give_up(StackShared *sh, int *status, int code)
{
    sh->abort_flag = 1;
    atomicCAS(status, 0, code);
}
// Wait of a warp for the prefix to pass `need`; `ready` receives what every lane has seen (a lane may have seen more
// than another, and callers branch on the value around votes of the whole warp).
__device__ __forceinline__ bool stack_wait_ready(const int *word, int need, int &ready, volatile int *abort_flag)
{
    long long t0 = 0;
    for (unsigned spin = 1;; ++spin) {
        ready = ld_acquire_cta_shared(word);
        if (__all_sync(0xffffffffu, ready > need)) {
            ready = __reduce_min_sync(0xffffffffu, ready);
            return true;
        }
        if ((spin & 63u) == 0) {
            bool stop = *abort_flag != 0;
            const long long now = clock64();
            if (t0 == 0) t0 = now;
            else if (now - t0 > WAIT_LIMIT_CYCLES) stop = true;
            if (__any_sync(0xffffffffu, stop)) return false;
        }
    }
}
// The whole bank of a layer in one copy: box {KC, block_n, taps}.
__device__ __forceinline__ void tma_load_3d(uint32_t dst, const CUtensorMap *map, uint32_t bar, int x, int y, int z)
{
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
        " [%0], [%1, {%3, %4, %5}], [%2];"
        ::"r"(dst), "l"(map), "r"(bar), "r"(x), "r"(y), "r"(z)
        : "memory");
}

template <int KH, int KW, int KJ>
__global__ void __launch_bounds__(STACK_THREADS, 1)
umma_stack_kernel(const __grid_constant__ StackLayers layers, const __grid_constant__ StackArgs u, const __grid_constant__ ConvArgs a, const __grid_constant__ UmmaArgs ua)
{
    extern __shared__ uint8_t smem_raw[];
    uint8_t *tiles = (uint8_t *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    uint8_t *b_res = tiles + (size_t)u.stages * u.stage_bytes;             // two filter banks
    const int bank_bytes = u.b_tile_bytes * KH * KW;
    // the layers' additive constants: from global memory they would miss L1 after every acquire, which empties it
    const uint32_t ca_s = smem_u32(b_res + 2 * (size_t)bank_bytes);            // [n_layers][block_n] int32
    StackShared *sh = (StackShared *)(b_res + 2 * (size_t)bank_bytes + (size_t)u.n_layers * u.block_n * 4);
    const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0);
    const int lane = threadIdx.x & 31;
    const int G = (int)gridDim.x;                                          // <= u.tiles: every CTA has a tile in every layer

    if (threadIdx.x == 0) {
        for (int s = 0; s < u.stages; ++s) {
            mbar_init(smem_u32(&sh->full[s]), 1);
            mbar_init(smem_u32(&sh->empty[s]), 1);
        }
        for (int b = 0; b < u.nbuf; ++b) {
            mbar_init(smem_u32(&sh->tmem_full[b]), 1);
            mbar_init(smem_u32(&sh->tmem_empty[b]), (uint32_t)(4 * u.cs));
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(smem_u32(&sh->b_full[b]), 1);
            mbar_init(smem_u32(&sh->b_empty[b]), (uint32_t)STACK_ISSUERS);
        }
        mbar_init(smem_u32(&sh->drain), STACK_ISSUERS);
        for (int w = 0; w < EPI_WARPS_MAX; ++w) sh->progress[w] = 0;
        sh->ready = 0;
        sh->abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    for (int i = (int)threadIdx.x; i < u.n_layers * (u.block_n >> 2); i += STACK_THREADS) {
        const int l = i / (u.block_n >> 2), k = i - l * (u.block_n >> 2);
        sts128(ca_s + 16u * (uint32_t)i, __ldg((const uint4 *)layers.l[l].c_a + k));
    }
    if (warp == MMA_WARP) tmem_alloc(smem_u32(&sh->tmem_base), (uint32_t)u.tmem_cols);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = sh->tmem_base;

    int last_stage = -1, bank_next = 0;
    uint32_t last_parity = 0;

    if (warp == 0) {
        // ---------------------------------------------------------------- TMA producer (whole warp; an elected lane issues)
        // Bank l goes to half l & 1 once the MMAs of layer l - 2 are done.
        auto load_bank = [&]() -> bool {
            const int l = bank_next;
            if (l >= 2 && !mbar_wait_warp(smem_u32(&sh->b_empty[l & 1]), (uint32_t)(((l >> 1) & 1) ^ 1), &sh->abort_flag, lane)) {
                stack_give_up(sh, u.status, 1);
                return false;
            }
            if (elect_one()) {
                const uint32_t bf = smem_u32(&sh->b_full[l & 1]);
                mbar_expect_tx(bf, (uint32_t)bank_bytes);
                tma_load_3d(smem_u32(b_res + (size_t)(l & 1) * bank_bytes), &layers.l[l].w, bf, 0, 0, 0);
            }
            __syncwarp();
            ++bank_next;
            return true;
        };
        // the bank of the layer after this one is fetched once this layer is under way (not at its first tile: the
        // wait for the layer before would let the patch ring run dry)
        const int bank_at = min(u.stages, u.tiles / G);
        int layer = 0, tile = (int)blockIdx.x, in_layer = 0, ready = 0, seq0 = -u.tiles, stage = 0;      // seq0: first tile of the layer before, in the sequence
        uint32_t parity = 0;
        const uint32_t tx = (uint32_t)(u.kc * u.bw * u.bh);
        bool ok = load_bank();
        while (ok && layer < u.n_layers) {
            const int img = (int)fast_div((unsigned)tile, u.div_tpi_mul, u.div_tpi_shr);
            const unsigned rem = (unsigned)(tile - img * u.tpi);
            int cx, cy;                                   // first output pixel of the tile
            if (u.blocks) {
                const int by = (int)fast_div(rem, u.div_vw_mul, u.div_vw_shr);
                cx = ((int)rem - by * u.vw) * 8;
                cy = by * 16;
            } else {
                const unsigned i0 = rem * BLOCK_M;
                cy = (int)fast_div(i0, u.div_vw_mul, u.div_vw_shr);
                cx = u.full_width ? 0 : (int)i0 - cy * u.vw;
            }
            if (layer > 0) {
                const int need = min(tile + u.fwd, (img + 1) * u.tpi - 1);
                if (ready <= seq0 + need) {
                    if (!stack_wait_ready(&sh->ready, seq0 + need, ready, &sh->abort_flag)) {
                        stack_give_up(sh, u.status, 1);
                        break;
                    }
                    fence_async_proxy();         // what the others stored, before this thread's bulk-asynchronous reads
                }
            }
            if (!mbar_wait_warp(smem_u32(&sh->empty[stage]), parity ^ 1u, &sh->abort_flag, lane)) {
                stack_give_up(sh, u.status, 1);
                break;
            }
            if (elect_one()) {
                const uint32_t full = smem_u32(&sh->full[stage]);
                mbar_expect_tx(full, tx);
                tma_load_tile_4d(smem_u32(tiles + (size_t)stage * u.stage_bytes), &layers.l[layer].x, full, 0, cx - u.pad, cy - u.pad, img);
            }
            __syncwarp();
            last_stage = stage;
            last_parity = parity;
            if (++stage == u.stages) { stage = 0; parity ^= 1u; }
            if (++in_layer == bank_at && bank_next == layer + 1 && bank_next < u.n_layers) ok = load_bank();
            tile += G;
            if (tile >= u.tiles) { tile -= u.tiles; ++layer; in_layer = 0; seq0 += u.tiles; }
        }
        __syncwarp();
    } else if (warp == STACK_READY_WARP) {
        // ---------------------------------------------------------------- counters -> ready (whole warp)
        // Follows the chunks of all layers but the last one in order, 32 counters per round.
        const int total = (u.n_layers - 1) * u.chunks;
        int chunk = 0, layer = 0, in = 0;                 // next chunk not known to be full: overall, its layer, its index in the layer
        long long t0 = clock64();
        while (chunk < total) {
            const int left = min(u.chunks - in, 32);      // (a round stays inside a layer)
            bool full = false;
            if (lane < left) {
                const int c = in + lane;
                full = ld_acquire_gpu(u.sync + STACK_SYNC_WORDS + chunk + lane) >= (unsigned)min(STACK_CHUNK, u.tiles - c * STACK_CHUNK);
            }
            const unsigned open = __ballot_sync(0xffffffffu, !full);
            const int n = open ? __ffs((int)open) - 1 : 32;
            if (n) {
                chunk += n;
                in += n;
                __syncwarp();                             // what the lanes acquired, before the release of one of them (votes order no memory)
                if (lane == 0) st_release_cta_shared(&sh->ready, layer * u.tiles + min(in * STACK_CHUNK, u.tiles));
                __syncwarp();
                if (in == u.chunks) { in = 0; ++layer; }
                t0 = clock64();
            } else {
                if (__any_sync(0xffffffffu, sh->abort_flag != 0 || clock64() - t0 > WAIT_LIMIT_CYCLES)) break;
                __nanosleep(100);
            }
        }
    } else if (warp == MMA_WARP || warp == MMA_WARP2) {
        // ---------------------------------------------------------------- MMA issuers (as in the window kernel)
        const int which = warp == MMA_WARP ? 0 : 1;
        {
            int t = which, stage = which % u.stages, layer = 0, tile = (int)blockIdx.x + which * G, cur = -1;
            uint32_t parity = (uint32_t)((which / u.stages) & 1);
            bool ok = true;
            const uint32_t a_lo0 = ((smem_u32(tiles) & 0x3FFFFu) >> 4) | (1u << 16);
            const uint32_t b_lo0 = ((smem_u32(b_res) & 0x3FFFFu) >> 4) | (1u << 16);
            const uint32_t stage_step = (uint32_t)u.stage_bytes >> 4, row_step = (uint32_t)u.kc >> 4;
            const uint32_t b_step = (uint32_t)u.b_tile_bytes >> 4;
            const uint32_t line_step = (uint32_t)u.bw * row_step;
            // passes on to layer l: gives the banks of the layers left behind back (every issuer arrives once per
            // layer, with or without a tile in it), waits for the new ones
            auto enter = [&](int l) -> bool {
                while (cur < l) {
                    if (cur >= 0 && elect_one()) umma_commit(smem_u32(&sh->b_empty[cur & 1]));
                    __syncwarp();
                    ++cur;
                    if (!mbar_wait_warp(smem_u32(&sh->b_full[cur & 1]), (uint32_t)((cur >> 1) & 1), &sh->abort_flag, lane)) {
                        stack_give_up(sh, u.status, 6);
                        return false;
                    }
                }
                return true;
            };
            while (tile >= u.tiles) { tile -= u.tiles; ++layer; }
            while (layer < u.n_layers) {
                if (!(ok = enter(layer))) break;
                const int buf = t & (u.nbuf - 1);
                uint32_t off0 = 0;
                if (u.full_width) {
                    const int img = (int)fast_div((unsigned)tile, u.div_tpi_mul, u.div_tpi_shr);
                    const unsigned i0 = (unsigned)(tile - img * u.tpi) * BLOCK_M;
                    off0 = i0 - fast_div(i0, u.div_vw_mul, u.div_vw_shr) * (unsigned)u.vw;
                }
                // (the patch before the buffer: see the window kernel)
                if (!mbar_wait_warp(smem_u32(&sh->full[stage]), parity, &sh->abort_flag, lane)) {
                    stack_give_up(sh, u.status, 3);
                    ok = false;
                    break;
                }
                if (!mbar_wait_warp(smem_u32(&sh->tmem_empty[buf]), (uint32_t)(((t >> u.lg_nbuf) & 1) ^ 1), &sh->abort_flag, lane)) {
                    stack_give_up(sh, u.status, 2);
                    ok = false;
                    break;
                }
                tc_fence_after();
                const uint32_t d_tmem = tmem_base + (uint32_t)(buf * u.block_n);
                uint32_t a_line = a_lo0 + (uint32_t)stage * stage_step + off0 * row_step;
                const uint32_t b_lo = b_lo0 + (uint32_t)(layer & 1) * ((uint32_t)bank_bytes >> 4);
                if (elect_one()) {
#pragma unroll
                    for (int r = 0; r < KH; ++r) {
#pragma unroll
                        for (int sx = 0; sx < KW; ++sx)
                            umma_slot2<KJ>(d_tmem, a_line + (uint32_t)sx * row_step, u.desc_hi_a, b_lo + (uint32_t)(r * KW + sx) * b_step, u.desc_hi_b,
                                           u.idesc, (uint32_t)((r | sx) != 0));
                        a_line += line_step;
                    }
                    umma_commit(smem_u32(&sh->empty[stage]));
                    umma_commit(smem_u32(&sh->tmem_full[buf]));
                }
                __syncwarp();
                stage += STACK_ISSUERS;
                if (stage >= u.stages) { stage -= u.stages; parity ^= 1u; }
                t += STACK_ISSUERS;
                tile += STACK_ISSUERS * G;
                while (tile >= u.tiles) { tile -= u.tiles; ++layer; }
            }
            if (ok) enter(u.n_layers - 1);
        }
        __syncwarp();
    } else if (warp >= EPI_WARP0 && warp < EPI_WARP0 + u.epi_warps) {
        // ---------------------------------------------------------------- epilogue
        const int ew = warp - EPI_WARP0;
        const int quad = warp & 3;
        const int slot = ew >> 2;
        const int part = slot % u.cs;
        const int turn = slot / u.cs;
        const int col_lo = part * u.part_n;
        const int ngroups = min(u.block_n - col_lo, u.part_n) >> 4;
        EpiScalars es = epi_scalars(a, ua);
        uint32_t cap_s = 0;
        uint8_t *out = nullptr;
        int out_c_total = 0, cur = -1;
        int layer = 0, tile = (int)blockIdx.x + turn * G;
        while (tile >= u.tiles) { tile -= u.tiles; ++layer; }
        for (int t = turn; layer < u.n_layers; t += u.bi) {
            if (layer != cur) {
                const StackLayer *L = &layers.l[layer];
                cap_s = ca_s + 4u * (uint32_t)(layer * u.block_n + col_lo); out = L->out + col_lo; out_c_total = L->out_c_total; es.q_mul = L->q_mul; es.q_shift = L->q_shift;
                cur = layer;
            }
            const int buf = t & (u.nbuf - 1);
            const int img = (int)fast_div((unsigned)tile, u.div_tpi_mul, u.div_tpi_shr);
            const unsigned rem = (unsigned)(tile - img * u.tpi);
            int y, xq;                                        // this lane's (virtual) output pixel
            if (u.blocks) {
                const int by = (int)fast_div(rem, u.div_vw_mul, u.div_vw_shr);
                const int mm = quad * 32 + lane;
                y = by * 16 + (mm >> 3);
                xq = ((int)rem - by * u.vw) * 8 + (mm & 7);
            } else {
                const unsigned i = rem * BLOCK_M + (unsigned)(quad * 32 + lane);
                y = (int)fast_div(i, u.div_vw_mul, u.div_vw_shr);
                xq = (int)i - y * u.vw;
            }
            const bool valid = xq < u.w && y < u.h;
            uint8_t *ocol = out + (((long long)img * u.h + y) * u.w + xq) * out_c_total;
            if (!mbar_wait_warp(smem_u32(&sh->tmem_full[buf]), (uint32_t)((t >> u.lg_nbuf) & 1), &sh->abort_flag, lane)) {
                stack_give_up(sh, u.status, 4);
                break;
            }
            tc_fence_after();
            const uint32_t t_row = tmem_base + ((uint32_t)(quad * 32) << 16) + (uint32_t)(buf * u.block_n + col_lo);
            int accA[16];
            if (ngroups == 4) window_groups<EPI_FAST, 4, false, true>(t_row, nullptr, ocol, nullptr, valid, col_lo, ngroups, accA, es, a, ua, cap_s);
            else window_groups<EPI_FAST, 0, false, true>(t_row, nullptr, ocol, nullptr, valid, col_lo, ngroups, accA, es, a, ua, cap_s);
            tc_fence_before();
            __syncwarp();
            if (lane == 0) {
                mbar_arrive(smem_u32(&sh->tmem_empty[buf]));
                st_release_cta_shared(&sh->progress[ew], t + 1);
            }
            tile += u.bi * G;
            while (tile >= u.tiles) { tile -= u.tiles; ++layer; }
        }
    } else if (warp == STACK_SIGNAL_WARP) {
        // ---------------------------------------------------------------- tiles stored -> counters
        const int total = (u.n_layers * u.tiles - (int)blockIdx.x + G - 1) / G;      // tiles of this CTA
        const int per_group = 4 * u.cs;                                              // warps that share a tile
        long long t0 = clock64();
        int next = 0;                                                                // first tile not yet counted
        while (next < total) {
            const int mine = lane < u.epi_warps ? ld_acquire_cta_shared(&sh->progress[lane]) : 0x7fffffff;
            // the slowest warp of every group (a group's warps are 4 * cs neighbours); lane g holds group g's
            int slow = mine;
            for (int d = 1; d < per_group; d <<= 1) slow = min(slow, __shfl_xor_sync(0xffffffffu, slow, d));
            const int t = next + lane;
            const int group_progress = __shfl_sync(0xffffffffu, slow, (t % u.bi) * per_group);
            const unsigned open = __ballot_sync(0xffffffffu, t >= total || group_progress <= t);
            const int n = open ? __ffs((int)open) - 1 : 32;
            if (n) {
                __syncwarp();                                    // what other lanes acquired (votes and shuffles order no memory)
                fence_acq_rel_gpu();
                if (lane < n) {
                    const int g = (int)blockIdx.x + t * G;
                    const int l = g / u.tiles;
                    red_relaxed_gpu(u.sync + STACK_SYNC_WORDS + l * u.chunks + (g - l * u.tiles) / STACK_CHUNK, 1u);
                }
                __syncwarp();
                next += n;
                t0 = clock64();
            } else {
                if (__any_sync(0xffffffffu, sh->abort_flag != 0 || clock64() - t0 > WAIT_LIMIT_CYCLES)) break;
                __nanosleep(64);
            }
        }
    }

    // ---------------------------------------------------------------- teardown
    if (threadIdx.x == 0) grid_dep_launch();         // the kernel after this one may come up while the last CTAs finish
    tc_fence_before();
    __syncthreads();
    if (sh->abort_flag) {
        volatile int never = 0;
        if (warp == 0 && lane == 0) {
            for (int l = max(0, bank_next - 2); l < bank_next; ++l) mbar_wait(smem_u32(&sh->b_full[l & 1]), (uint32_t)((l >> 1) & 1), &never);
            if (last_stage >= 0) mbar_wait(smem_u32(&sh->full[last_stage]), last_parity, &never);
            const long long t0 = clock64();
            while (clock64() - t0 < 2000000) {}
        }
        if ((warp == MMA_WARP || warp == MMA_WARP2) && lane == 0) {
            umma_commit(smem_u32(&sh->drain));
            mbar_wait(smem_u32(&sh->drain), 0, &never);
        }
        __syncthreads();
    }
    if (warp == MMA_WARP) {
        tc_fence_after();
        tmem_dealloc(tmem_base, (uint32_t)u.tmem_cols);
    }
    // the last CTA to get here leaves the counters as it found them
    if (threadIdx.x == 0) {
        __threadfence();
        sh->last_cta = atomicAdd(u.sync, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (sh->last_cta)
        for (int i = (int)threadIdx.x; i < STACK_SYNC_WORDS + u.n_layers * u.chunks; i += STACK_THREADS) u.sync[i] = 0u;
}

}  // namespace iconv

// The 7x7/2 first layer over three channels and the 3x3/2 max-pool behind it as ONE kernel (after the repack that
// rearranges the image, kernel_stem.cu): the layer's own output, four times the pooled one, is never written.
//
// The pool takes the maximum of the requantised bytes, so the result is that of the two operations apart.  What makes it cheap is
// the order of the GEMM's rows: a row of A is a POOLED column px, and the accumulators beside one another are the four
// convolution outputs that belong to it (rows 2 py and 2 py + 1, columns 2 px and 2 px + 1):
//
//   - A window's lower row and right column come with it; its upper row is the lower one of the step before (a warp walks
//     down a strip of the image, and keeps it), its left column the right one of the lane before (one shuffle of packed bytes).
//   - The repacked image holds 16 bytes a position (2 x 2 pixels x 3 channels); pooled column px needs positions 2 px
//     ... 2 px + 4, that is the pairs px, px + 1 and px + 2, which are the same operand read one and two rows further on.  So
//     a K = 32 instruction takes a pair of positions of one row, and N covers all outputs that need it: 64 ... 256 columns.
//     16 instructions, 1312 cycles for 512 convolution outputs x 64 channels (the layer alone: 32 of 48 = 1536).
//
// A tile: 2 images x 2 strips of 32 lanes, of which 29 are outputs (lane 0 is the column to the left, and the last two read
// beyond their strip).  A CTA works on two tiles in turn ("streams"), each with half of tensor memory, and walks each down a band of rows; a band begins one step early, for the row above it.  One 5-D TMA copy brings a
// step's five rows of all four strips.  A row of the repacked image is its even positions, then its odd ones: so the copy is of
// 512-byte runs, and they are the operand as it is (no swizzle: eight rows of 16 bytes, each half of K in a plane of its
// own); pairs as 32-byte rows under a 32-byte swizzle are 640 rows a step.
//
// 256 images of 224 x 224, repack included: 83 us (the layer and the pool apart 114 + 57).  A step's instructions take 1391 of about 2300
// cycles: bound by the epilogue's.
#include <cuda.h>

#include <atomic>
#include <cstring>
#include <vector>

#include "plan.h"
#include "umma_inst.h"

namespace iconv {

namespace {

constexpr int POOL_N = 64;                        // channels
constexpr int POOL_LANES = 32, POOL_OUT = 29;     // lanes of a strip, outputs of it
constexpr int POOL_ROWS = 5;                      // rows of positions that a step reads
constexpr int POOL_ROW_BYTES = 4 * POOL_LANES * 32;                  // one such row of the tile's four strips: 4096
constexpr int POOL_PLANE = POOL_ROW_BYTES / 2;                       // even positions, odd positions
constexpr int POOL_STAGE = POOL_ROWS * POOL_ROW_BYTES;               // 20480
constexpr int POOL_STAGES = 6;
constexpr int POOL_LOAD_WARP = 0, POOL_MMA_WARP = 1, POOL_EPI_WARP0 = 2;
constexpr int POOL_EPI_WARPS = 16, POOL_THREADS = 32 * (POOL_EPI_WARP0 + POOL_EPI_WARPS);
// the bank: row blocks of 64 columns x 32 bytes, in the order of the instructions (pool_bank)
constexpr int POOL_BLOCK = POOL_N * 32;
constexpr int POOL_BLOCKS = 40;
constexpr int POOL_BANK = POOL_BLOCKS * POOL_BLOCK;                  // 81920

// One instruction: row t of positions, pair j (the operand's rows shifted by j), the first of its 64-column accumulators and their
// number, the bank's block, and whether it adds.  Accumulators: even column of the upper row, odd of the upper, odd of the
// lower, even of the lower, so that what one pair is needed for lies side by side.
struct PoolStep {
    int t, j, first, count, block, add;
};
#define POOL_STEP_LIST \
    {0, 0, 0, 2, 0, 0}, {0, 1, 0, 2, 2, 1}, {0, 2, 1, 1, 4, 1}, \
    {1, 0, 0, 2, 5, 1}, {1, 0, 2, 2, 7, 0}, {1, 1, 0, 4, 9, 1}, {1, 2, 1, 2, 13, 1}, \
    {2, 0, 0, 4, 15, 1}, {2, 1, 0, 4, 19, 1}, {2, 2, 1, 2, 23, 1}, \
    {3, 0, 0, 4, 25, 1}, {3, 1, 0, 4, 29, 1}, {3, 2, 1, 2, 33, 1}, \
    {4, 0, 2, 2, 35, 1}, {4, 1, 2, 2, 37, 1}, {4, 2, 2, 1, 39, 1},
constexpr PoolStep POOL_STEPS[] = {POOL_STEP_LIST};
constexpr int POOL_NSTEPS = sizeof(POOL_STEPS) / sizeof(POOL_STEPS[0]);

struct PoolArgs {
    const int32_t *c_a;              // [64] the layer's additive constants (EPI_FAST)
    uint8_t *out;
    int n, h_conv, w_conv, h_out, w_out;
    int items, strip_pairs, bands, rows;             // tiles' walks; pairs of strips per image row, bands per image, pooled rows per band
    int q_mul, q_shift;
    unsigned idesc;                                  // without N
    int *status;
};

struct PoolShared {
    unsigned long long full[POOL_STAGES], empty[POOL_STAGES];
    unsigned long long tmem_full[2], tmem_empty[2];
    unsigned long long b_full, drain;
    int c_a[POOL_N];
    uint32_t tmem_base;
    volatile int abort_flag;
};
constexpr size_t POOL_SMEM = 1024 + (size_t)POOL_STAGES * POOL_STAGE + POOL_BANK + sizeof(PoolShared);
static_assert(POOL_SMEM <= (size_t)MAX_SMEM, "");

__device__ __forceinline__ void pool_give_up(PoolShared *sh, int *status, int code)
{
    sh->abort_flag = 1;
    atomicCAS(status, 0, code);
}

// Item i: band, pair of strips, pair of images.
struct PoolItem {
    int img, strip, row;             // first image, first strip, first pooled row
    __device__ __forceinline__ PoolItem(const PoolArgs &u, int i)
    {
        const int band = i % u.bands, k = i / u.bands;
        strip = 2 * (k % u.strip_pairs);
        img = 2 * (k / u.strip_pairs);
        row = band * u.rows;
    }
};

__device__ __forceinline__ void tma_load_5d(uint32_t dst, const CUtensorMap *map, uint32_t bar, int a, int b, int c, int d, int e)
{
    asm volatile(
        "cp.async.bulk.tensor.5d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
        " [%0], [%1, {%3, %4, %5, %6, %7}], [%2];"
        ::"r"(dst), "l"(map), "r"(bar), "r"(a), "r"(b), "r"(c), "r"(d), "r"(e)
        : "memory");
}

// Two values, saturated to 16 bits, in one word (lo in the low half); the maxima are taken of such words, two channels an instruction
// (with the byte-wise maximum, which is several: 14.1 M instructions for 64 images, now 11.5), and the bytes'
// saturation comes after the last of them.
// SHIFT16: the shift is 16 (what iq_mul_shift yields unless the multiplier is small), and the two results are the upper halves: one
// byte permutation where two shifts and a conversion were (256 images, repack included: 85.8 -> 82.7 us).
template <bool SHIFT16>
__device__ __forceinline__ uint32_t pool_pack2(int lo, int hi, int shift)
{
    if (SHIFT16) return __byte_perm((unsigned)lo, (unsigned)hi, 0x7632);
    uint32_t d;
    asm("cvt.pack.sat.s16.s32 %0, %1, %2;" : "=r"(d) : "r"(hi >> shift), "r"(lo >> shift));
    return d;
}
// The wait for both loads; the values pass through it, so that nothing uses them before.
__device__ __forceinline__ void tmem_ld16_ready(int (&a)[16], int (&b)[16])
{
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+r"(a[0]), "+r"(a[1]), "+r"(a[2]), "+r"(a[3]), "+r"(a[4]), "+r"(a[5]), "+r"(a[6]), "+r"(a[7]), "+r"(a[8]), "+r"(a[9]), "+r"(a[10]),
                   "+r"(a[11]), "+r"(a[12]), "+r"(a[13]), "+r"(a[14]), "+r"(a[15])
                 :
                 : "memory");
    asm volatile("" : "+r"(b[0]), "+r"(b[1]), "+r"(b[2]), "+r"(b[3]), "+r"(b[4]), "+r"(b[5]), "+r"(b[6]), "+r"(b[7]), "+r"(b[8]), "+r"(b[9]), "+r"(b[10]),
                       "+r"(b[11]), "+r"(b[12]), "+r"(b[13]), "+r"(b[14]), "+r"(b[15])::"memory");
}

// map_x: the strip's positions of one plane, strips, images, planes, rows of positions.  The CTA's walks: item blockIdx.x + gridDim.x *
// (2 * k + stream); a step of stream 0, the same of stream 1, the next.
template <bool SHIFT16>
__global__ void __launch_bounds__(POOL_THREADS, 1)
stem_pool_kernel(const __grid_constant__ CUtensorMap map_x, const __grid_constant__ CUtensorMap map_w, const __grid_constant__ PoolArgs u)
{
    extern __shared__ uint8_t smem_raw[];
    uint8_t *stages = (uint8_t *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    uint8_t *bank = stages + POOL_STAGES * POOL_STAGE;
    PoolShared *sh = (PoolShared *)(bank + POOL_BANK);
    const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0);
    const int lane = threadIdx.x & 31;
    const int G = (int)gridDim.x, steps = u.rows + 1;
    const int rounds = (u.items - (int)blockIdx.x + 2 * G - 1) / (2 * G);        // of stream 0's items (every CTA has one)

    if (threadIdx.x == 0) {
        for (int s = 0; s < POOL_STAGES; ++s) {
            mbar_init(smem_u32(&sh->full[s]), 1);
            mbar_init(smem_u32(&sh->empty[s]), 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(smem_u32(&sh->tmem_full[b]), 1);
            mbar_init(smem_u32(&sh->tmem_empty[b]), POOL_EPI_WARPS);
        }
        mbar_init(smem_u32(&sh->b_full), 1);
        mbar_init(smem_u32(&sh->drain), 1);
        sh->abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        grid_dep_launch();
    }
    if (threadIdx.x < POOL_N) sh->c_a[threadIdx.x] = __ldg(u.c_a + threadIdx.x);
    if (warp == POOL_MMA_WARP) tmem_alloc(smem_u32(&sh->tmem_base), 512u);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = sh->tmem_base;
    int last_stage = -1;
    uint32_t last_parity = 0;

    if (warp == POOL_LOAD_WARP) {
        // ---------------------------------------------------------------- loads (whole warp; an elected lane issues)
        if (elect_one()) {
            const uint32_t bf = smem_u32(&sh->b_full), dst = smem_u32(bank);
            mbar_expect_tx(bf, (uint32_t)POOL_BANK);
            for (int i = 0; i < POOL_BANK / 8192; ++i) tma_load_2d(dst + (uint32_t)(i * 8192), &map_w, bf, 0, i * 256);
        }
        __syncwarp();
        grid_dep_wait();                                 // the repacked image comes from the kernel before this one
        int stage = 0;
        uint32_t parity = 0;
        bool ok = true;
        for (int k = 0; ok && k < rounds; ++k) {
            const int i0 = (int)blockIdx.x + G * 2 * k, i1 = i0 + G;
            const PoolItem w0(u, i0), w1(u, i1);
            const int streams = i1 < u.items ? 2 : 1;
            for (int s = 0; ok && s < steps; ++s)
                for (int b = 0; b < streams; ++b) {
                    if (!mbar_wait_warp(smem_u32(&sh->empty[stage]), parity ^ 1u, &sh->abort_flag, lane)) {
                        pool_give_up(sh, u.status, 1);
                        ok = false;
                        break;
                    }
                    if (elect_one()) {
                        const uint32_t full = smem_u32(&sh->full[stage]);
                        mbar_expect_tx(full, (uint32_t)POOL_STAGE);
                        // (the first row of a step: position row 2 (row - 1 + s); above the image it is negative, zeros)
                        tma_load_5d(smem_u32(stages) + (uint32_t)(stage * POOL_STAGE), &map_x, full, 0, b ? w1.strip : w0.strip, b ? w1.img : w0.img, 0,
                                    2 * ((b ? w1.row : w0.row) - 1 + s));
                    }
                    __syncwarp();
                    last_stage = stage;
                    last_parity = parity;
                    if (++stage == POOL_STAGES) { stage = 0; parity ^= 1u; }
                }
        }
        __syncwarp();
    } else if (warp == POOL_MMA_WARP) {
        // ---------------------------------------------------------------- MMA issuer (whole warp; an elected lane issues)
        constexpr uint32_t HI_A = (uint32_t)(128 >> 4) | (1u << 14);                      // 8-row groups 128 bytes apart, version 1, no swizzle
        constexpr uint32_t HI_B = (uint32_t)((8 * 32) >> 4) | (1u << 14) | (6u << 29);    // ... 256 bytes apart, 32-byte swizzle
        const uint32_t a_lo0 = ((smem_u32(stages) & 0x3FFFFu) >> 4) | ((uint32_t)(POOL_PLANE >> 4) << 16), b_lo0 = ((smem_u32(bank) & 0x3FFFFu) >> 4) | (1u << 16);
        int stage = 0, t = 0;                            // t: steps of a stream so far
        uint32_t parity = 0;
        bool ok = mbar_wait_warp(smem_u32(&sh->b_full), 0u, &sh->abort_flag, lane);
        if (!ok) pool_give_up(sh, u.status, 6);
        int t1 = 0;
        constexpr PoolStep STEPS[] = {POOL_STEP_LIST};   // (an array outside has no device copy)
        for (int k = 0; ok && k < rounds; ++k) {
            const int streams = (int)blockIdx.x + G * (2 * k + 1) < u.items ? 2 : 1;
            for (int s = 0; ok && s < steps; ++s)
                for (int b = 0; b < streams; ++b) {
                    int &n = b ? t1 : t;
                    if (!mbar_wait_warp(smem_u32(&sh->tmem_empty[b]), (uint32_t)((n & 1) ^ 1), &sh->abort_flag, lane)) {
                        pool_give_up(sh, u.status, 2);
                        ok = false;
                        break;
                    }
                    if (!mbar_wait_warp(smem_u32(&sh->full[stage]), parity, &sh->abort_flag, lane)) {
                        pool_give_up(sh, u.status, 3);
                        ok = false;
                        break;
                    }
                    tc_fence_after();
                    ++n;
                    if (elect_one()) {
                        const uint32_t d0 = tmem_base + (uint32_t)(b * 4 * POOL_N), a0 = a_lo0 + (uint32_t)((stage * POOL_STAGE) >> 4);
#pragma unroll
                        for (int i = 0; i < POOL_NSTEPS; ++i) {
                            const PoolStep st = STEPS[i];
                            umma_i8_split2(d0 + (uint32_t)(st.first * POOL_N), a0 + (uint32_t)((st.t * POOL_ROW_BYTES + st.j * 16) >> 4), HI_A,
                                           b_lo0 + (uint32_t)((st.block * POOL_BLOCK) >> 4), HI_B, u.idesc | ((uint32_t)(st.count * POOL_N >> 3) << 17), (uint32_t)st.add);
                        }
                        umma_commit(smem_u32(&sh->empty[stage]));
                        umma_commit(smem_u32(&sh->tmem_full[b]));
                    }
                    __syncwarp();
                    if (++stage == POOL_STAGES) { stage = 0; parity ^= 1u; }
                }
        }
        __syncwarp();
    } else {
        // ---------------------------------------------------------------- epilogue: every warp a strip and 16 channels, the streams in turn
        // (with half of the warps for either stream a step's 32 channels took a warp 2000 cycles by itself and 3300 beside the other
        // stream's, and the stream's next instructions wait for it: 256 images 109 us, now 93, repack included)
        grid_dep_wait();                                 // `out` may still be read by the kernel before this one
        const int quad = warp & 3, part = (warp - POOL_EPI_WARP0) >> 2;
        const int q_mul = u.q_mul, q_shift = u.q_shift;
        const uint32_t t_base = tmem_base + ((uint32_t)(quad * 32) << 16) + (uint32_t)(part * 16);
        int ca[16];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const uint4 v = lds128(smem_u32(&sh->c_a[part * 16 + q * 4]));
            ca[4 * q] = (int)v.x; ca[4 * q + 1] = (int)v.y; ca[4 * q + 2] = (int)v.z; ca[4 * q + 3] = (int)v.w;
        }
        uint32_t phase[2] = {0, 0};
        bool ok = true;
        for (int k = 0; ok && k < rounds; ++k) {
            const int i0 = (int)blockIdx.x + G * 2 * k, streams = i0 + G < u.items ? 2 : 1;
            uint32_t up_even[2][8], up_odd[2][8];        // the streams' row above: two channels a word
            uint32_t odd_ok[2];
            uint8_t *to[2];
            bool mine[2];
            int row[2];
#pragma unroll
            for (int b = 0; b < 2; ++b) {
                const PoolItem w(u, i0 + G * b);
                const int img = w.img + (quad >> 1), px = (w.strip + (quad & 1)) * POOL_OUT + lane - 1;
                mine[b] = img < u.n && lane >= 1 && lane <= POOL_OUT && px < u.w_out;
                odd_ok[b] = px >= 0 && 2 * px + 1 < u.w_conv ? 0xffffffffu : 0u;
                row[b] = w.row;
                to[b] = u.out + (((size_t)img * u.h_out + w.row) * u.w_out + px) * POOL_N + part * 16;
#pragma unroll
                for (int q = 0; q < 8; ++q) up_even[b][q] = up_odd[b][q] = 0;
            }
            for (int s = 0; ok && s < steps; ++s)
#pragma unroll
                for (int b = 0; b < 2; ++b) {
                    if (b >= streams || !ok) continue;
                    const int py = row[b] - 1 + s;
                    const uint32_t low_ok = py >= 0 && 2 * py + 1 < u.h_conv ? 0xffffffffu : 0u;
                    if (!mbar_wait_warp(smem_u32(&sh->tmem_full[b]), phase[b], &sh->abort_flag, lane)) {
                        pool_give_up(sh, u.status, 4);
                        ok = false;
                        continue;
                    }
                    phase[b] ^= 1u;
                    tc_fence_after();
                    // a column of the four outputs: its upper and lower row, the largest with the row above (a row below the image: 0,
                    // which no maximum of the clamped values falls under)
                    auto column = [&](int upper, int lower, uint32_t (&up)[8], uint32_t (&most)[8]) {
                        int au[16], al[16];
                        tmem_ld16(t_base + (uint32_t)((4 * b + upper) * POOL_N), au);
                        tmem_ld16(t_base + (uint32_t)((4 * b + lower) * POOL_N), al);
                        tmem_ld16_ready(au, al);
#pragma unroll
                        for (int q = 0; q < 8; ++q) {
                            const uint32_t pu = pool_pack2<SHIFT16>(au[2 * q] * q_mul + ca[2 * q], au[2 * q + 1] * q_mul + ca[2 * q + 1], q_shift);
                            const uint32_t pl = pool_pack2<SHIFT16>(al[2 * q] * q_mul + ca[2 * q], al[2 * q + 1] * q_mul + ca[2 * q + 1], q_shift) & low_ok;
                            most[q] = __vimax3_s16x2(up[q], pu, pl);
                            up[q] = pl;
                        }
                    };
                    uint32_t even[8], odd[8], o[4];
                    column(0, 3, up_even[b], even);
                    column(1, 2, up_odd[b], odd);
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(smem_u32(&sh->tmem_empty[b]));
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        uint32_t m[2];
#pragma unroll
                        for (int i = 0; i < 2; ++i) {
                            const uint32_t right = odd[2 * q + i] & odd_ok[b];
                            m[i] = __vimin_s16x2_relu(__vimax3_s16x2(even[2 * q + i], right, __shfl_up_sync(0xffffffffu, right, 1)), 0x00ff00ffu);
                        }
                        o[q] = __byte_perm(m[0], m[1], 0x6420);
                    }
                    if (s > 0) {
                        if (mine[b] && py < u.h_out) *(uint4 *)to[b] = make_uint4(o[0], o[1], o[2], o[3]);
                        to[b] += (size_t)u.w_out * POOL_N;
                    }
                }
        }
    }

    // ---------------------------------------------------------------- teardown
    __syncwarp();
    tc_fence_before();
    __syncthreads();
    if (sh->abort_flag) {
        volatile int never = 0;
        if (warp == POOL_LOAD_WARP && lane == 0) {
            mbar_wait(smem_u32(&sh->b_full), 0, &never);
            if (last_stage >= 0) mbar_wait(smem_u32(&sh->full[last_stage]), last_parity, &never);
            const long long t0 = clock64();
            while (clock64() - t0 < 2000000) {}
        }
        if (warp == POOL_MMA_WARP && lane == 0) {
            umma_commit(smem_u32(&sh->drain));
            mbar_wait(smem_u32(&sh->drain), 0, &never);
        }
        __syncthreads();
    }
    if (warp == POOL_MMA_WARP) {
        tc_fence_after();
        tmem_dealloc(tmem_base, 512u);
    }
}

// The bank's rows: for every instruction its accumulators' 64 channels of 32 bytes, the taps of two positions.  w2: the repacked
// layer's weights [64][4][4][16].  Accumulator c is row c / 2 (of 0, 0, 1, 1) and column 0, 1, 1, 0 of the four outputs.
std::vector<int8_t> pool_bank(const int8_t *w2)
{
    static const int ROW[4] = {0, 0, 1, 1}, ODD[4] = {0, 1, 1, 0};
    std::vector<int8_t> bank((size_t)POOL_BANK, 0);
    for (const PoolStep &st : POOL_STEPS)
        for (int i = 0; i < st.count; ++i) {
            const int c = st.first + i, r = st.t - ROW[c];
            for (int co = 0; co < POOL_N; ++co)
                for (int h = 0; h < 2; ++h) {
                    const int s = 2 * st.j + h - ODD[c];
                    if (r < 0 || r > 3 || s < 0 || s > 3) continue;
                    memcpy(&bank[((size_t)(st.block + i) * POOL_N + co) * 32 + h * 16], &w2[(((size_t)co * 4 + r) * 4 + s) * 16], 16);
                }
        }
    return bank;
}

}  // namespace

// Positions of a row of the repacked image, for a layer w_conv wide: two more on the left, a multiple of four (see stem_repack_wide_kernel;
// network.py finds the images in it again).
int pool_row_positions(int w_conv) { return (w_conv + 3 + 2 + 3) / 4 * 4; }
// ... and the bytes of it all, with what the last strips read beyond the last row.
static size_t pool_workspace(int n, int h_conv, int w_conv) { return ((size_t)n * (h_conv + 3) * pool_row_positions(w_conv) + 4 * POOL_LANES * 2) * 16; }

static int pool_strip_pairs(const iconv_plan_t *p) { return (((p->w_out - 1) / 2 + 1 + POOL_OUT - 1) / POOL_OUT + 1) / 2; }

// Can the layer behind p (its repacked form is p->inner) and the pool behind it be one kernel?  If so, packs the bank and divides the images into bands.
int pool_setup(iconv_plan_t *p, const int8_t *w2)
{
    const iconv_desc &d = p->d;
    const iconv_plan_t *in = p->inner;
    // (EPI_FAST also stands for parameters that are equal within groups of 16 channels: the window kernel reads a group's, this
    // one has a single multiplier and shift)
    bool one = true;
    for (int co = 1; d.per_channel && co < d.c_out; ++co) one = one && d.mul[co] == d.mul[0] && d.shift[co] == d.shift[0];
    if (d.c_out != POOL_N || d.out_c_total != POOL_N || d.out_c_offset || d.out_dtype != ICONV_U8 || d.skip_dtype >= 0 || in->epi != EPI_FAST ||
        in->c_out_pad != POOL_N || !one) {
        set_error("first layer and max-pool in one kernel: 64 channels of unsigned bytes, their whole tensor, with layer-wide parameters that need no clamp");
        return ICONV_ERR_UNSUPPORTED;
    }
    const int rc = umma_init_once();
    if (rc != ICONV_OK) return rc;
    const int dev = current_device_slot(), sms = dev < 0 ? 0 : umma_device_ready(dev);
    if (sms <= 0) { set_error("iconv_plan_stem_pool: no current device, or its index is beyond %d", MAX_DEVICES - 1); return ICONV_ERR_ARG; }
    // bands of an image: as many as make the longest CTA's walk shortest, a step early included
    const int h_pool = (p->h_out - 1) / 2 + 1;
    const long long columns = (long long)pool_strip_pairs(p) * (((long long)d.n + 1) / 2);
    long long best = -1;
    for (int bands = 1; bands <= h_pool; ++bands) {
        const int rows = (h_pool + bands - 1) / bands;
        const long long walks = (columns * bands + 2 * sms - 1) / (2 * sms), cost = walks * (rows + 1);
        if (best < 0 || cost < best) { best = cost; p->pool_rows = rows; }
    }
    if (columns * ((h_pool + p->pool_rows - 1) / p->pool_rows) >= (1ll << 30) ||
        (long long)d.n * (p->h_out + 3) * pool_row_positions(p->w_out) >= (1ll << 31)) {
        set_error("first layer and max-pool in one kernel: too many tiles, or more than 2^31 positions");
        return ICONV_ERR_UNSUPPORTED;
    }
    const std::vector<int8_t> bank = pool_bank(w2);
    ICONV_CUDA_TRY(cudaMalloc((void **)&p->w_packed, bank.size()));
    ICONV_CUDA_TRY(cudaMemcpy(p->w_packed, bank.data(), bank.size(), cudaMemcpyHostToDevice));
    p->workspace_bytes = pool_workspace(d.n, p->h_out, p->w_out);
    return umma_encode_2d(&p->tmap_w, p->w_packed, 32, POOL_BLOCKS * POOL_N, 32, 32, 256, 32);
}

// T: where the repacked image goes, rows of pool_row_positions positions.  Whatever may be refused is refused before the first launch.
int launch_pool(const iconv_plan_t *p, const ConvArgs &a, void *T, cudaStream_t stream)
{
    const iconv_desc &d = p->d;
    const iconv_plan_t *in = p->inner;
    if ((uintptr_t)a.out % 16) { set_error("iconv_forward: the pooled output must be 16-byte aligned"); return ICONV_ERR_ALIGN; }
    int rc = umma_init_once();
    if (rc != ICONV_OK) return rc;
    UmmaArgs ua;
    rc = umma_args(in, ua);
    if (rc != ICONV_OK) return rc;
    const int dev = current_device_slot();
    if (dev < 0) { set_error("iconv_forward: no current device, or its index is beyond %d", MAX_DEVICES - 1); return ICONV_ERR_ARG; }
    const int sms = umma_device_ready(dev);
    static std::atomic<int> opted[MAX_DEVICES];
    if (!opted[dev].load(std::memory_order_acquire)) {
        ICONV_CUDA_TRY(cudaFuncSetAttribute(stem_pool_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, MAX_SMEM));
        ICONV_CUDA_TRY(cudaFuncSetAttribute(stem_pool_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, MAX_SMEM));
        opted[dev].store(1, std::memory_order_release);
    }
    PoolArgs u;
    memset(&u, 0, sizeof(u));
    u.n = d.n;
    u.h_conv = p->h_out; u.w_conv = p->w_out;
    u.h_out = (p->h_out - 1) / 2 + 1; u.w_out = (p->w_out - 1) / 2 + 1;
    u.strip_pairs = pool_strip_pairs(p);
    u.rows = p->pool_rows;
    u.bands = (u.h_out + u.rows - 1) / u.rows;
    u.items = u.strip_pairs * ((d.n + 1) / 2) * u.bands;
    u.c_a = ua.c_a;
    u.out = (uint8_t *)a.out;
    u.q_mul = ua.q_mul; u.q_shift = ua.q_shift;
    u.idesc = ua.idesc & ~(0x3Fu << 17);
    u.status = ua.status;
    CUtensorMap mx;
    const int pitch = pool_row_positions(p->w_out);
    rc = umma_encode_strips(&mx, T, POOL_LANES, POOL_OUT, 2 * u.strip_pairs, d.n, p->h_out + 3, pitch, POOL_ROWS);
    if (rc != ICONV_OK) return rc;
    rc = launch_repack(p, a, T, stream);
    if (rc != ICONV_OK) return rc;
    ICONV_CUDA_TRY(launch_kernel(u.q_shift == 16 ? stem_pool_kernel<true> : stem_pool_kernel<false>, true, (unsigned)(u.items < sms ? u.items : sms), POOL_THREADS, POOL_SMEM, stream, mx, p->tmap_w, u));
    return ICONV_OK;
}

}  // namespace iconv

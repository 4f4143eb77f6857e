// The first layer over a grey picture (one channel, stride 1, 3x3 or 5x5) without a repacked copy of the picture.
//
// One pixel's whole neighbourhood is at most 25 bytes: a single K = 32 step.  Builder warps read it straight from the picture
// (two aligned words per filter row and pixel, neighbouring lanes share them), line the bytes up in registers and
// write one 32-byte row of the A operand per output pixel to shared memory; one instruction per tile of 128 pixels
// then does the arithmetic, where the repacked form had one per filter row and moved sixteen bytes per pixel out to
// memory and back.  Output pixels are numbered through rows and images, so only the last tile is ragged.
// Order of the bytes of an A (and B) row: the first four of every filter row as one word, then the fifth ones.
//
// What bounds it is the epilogue's arithmetic (64 columns: about 500 issue cycles per tile and scheduler, builders
// included) and the output's way to memory.  Four builder groups of four warps, a tile each, hide the way of the
// picture's words (the next tile's are under way while a tile is lined up): 1x1600x2560, 5x5, 64 channels with two groups
// 93 us, three 74, four 69; the repacked form took 109.  A group's first warp issues its tile's instruction
// itself: the group meets at a named barrier anyway, and an issuing warp of its own would add two waits to every
// tile.  A slot of A has its accumulators' number: free again once the epilogue has read those.
#include <cstring>
#include <vector>

#include "plan.h"
#include "umma_inst.h"

namespace iconv {

namespace {

constexpr int PIC_SLOTS = 8;
constexpr int PIC_GROUPS = 4;                                  // builder groups of four warps
constexpr int PIC_EPI_WARP0 = 4 * PIC_GROUPS;
constexpr int PIC_THREADS = 32 * (PIC_EPI_WARP0 + EPI_WARPS_MAX);
constexpr int PIC_MAX_N = 64;

struct PicArgs {
    const uint8_t *x;
    const int8_t *w;                                           // [block_n][32]
    int h, w_, pad, w_out, total;                              // total: bytes of x
    int m_total, tiles, tmem_cols;
    unsigned flip, idesc;                                      // flip: 0x80 in every byte that is stored biased
    unsigned div_w_mul, div_w_shr, div_hw_mul, div_hw_shr, hw;
    int *status;
};

struct PicShared {
    unsigned long long done[PIC_SLOTS], empty[PIC_SLOTS];      // a tile's MMA is done; its accumulators are read
    unsigned long long drain;
    uint32_t tmem_base;
    volatile int abort_flag;
};

__device__ __forceinline__ void pic_give_up(PicShared *sh, int *status, int code)
{
    sh->abort_flag = 1;
    atomicCAS(status, 0, code);
}

// A barrier of a builder group that also tells whether any of its threads gave up: all leave together or none does.
__device__ __forceinline__ bool pic_group_sync(int id, bool failed)
{
    unsigned any;
    __syncwarp();
    asm volatile("{\n\t.reg .pred p, q;\n\tsetp.ne.u32 p, %1, 0;\n\tbarrier.cta.red.or.aligned.pred q, %2, 128, p;\n\tselp.u32 %0, 1, 0, q;\n\t}"
                 : "=r"(any)
                 : "r"((unsigned)failed), "r"(id)
                 : "memory");
    return any != 0;
}

// The bytes of a picture behind its last whole word, and no more: what follows may be another tensor's.
__device__ __forceinline__ unsigned pic_rest(const uint8_t *x, int whole, int total)
{
    unsigned v = x[whole];
    if (total - whole > 1) v |= (unsigned)x[whole + 1] << 8;
    if (total - whole > 2) v |= (unsigned)x[whole + 2] << 16;
    return v;
}

// The words that hold one output pixel's neighbourhood, and what lines them up.  A warp whose pixels all lie inside the picture
// with their neighbourhoods (nearly every one) needs no masks: what a word holds beyond the filter's width meets weights of zero.
// REST: the picture's size is no multiple of 4.
template <int K, bool REST>
struct PicPixel {
    unsigned w0[K], w1[K];
    int at;                        // offset of the first row's first byte
    unsigned m_lo, m_hi, rows;     // bytes inside the picture; filter rows inside it
    bool inner;

    __device__ __forceinline__ void load(const PicArgs &u, int m)
    {
        const unsigned img = fast_div((unsigned)m, u.div_hw_mul, u.div_hw_shr), in = (unsigned)m - img * u.hw;
        const int y = (int)fast_div(in, u.div_w_mul, u.div_w_shr), x = (int)in - y * u.w_out;
        const int x0 = x - u.pad, y0 = y - u.pad;
        at = ((int)img * u.h + y0) * u.w_ + x0;
        inner = __all_sync(0xffffffffu, m < u.m_total && x0 >= 0 && x0 + K <= u.w_ && y0 >= 0 && y0 + K <= u.h && at + (K - 1) * u.w_ + 8 <= u.total);
        if (inner) {
#pragma unroll
            for (int r = 0; r < K; ++r) {
                const unsigned *w = (const unsigned *)(u.x + (unsigned)((at + r * u.w_) & ~3));
                w0[r] = ld_tensor(w);
                w1[r] = ld_tensor(w + 1);
            }
            return;
        }
        const bool real = m < u.m_total;
        const int left = -x0, have = u.w_ - x0;                        // bytes of a row before the picture; up to its end
        const unsigned from = left >= 4 ? 0u : left > 0 ? 0xFFFFFFFFu << (8 * left) : 0xFFFFFFFFu;
        const unsigned upto = have >= 4 ? 0xFFFFFFFFu : have > 0 ? (1u << (8 * have)) - 1u : 0u;
        m_lo = from & upto;
        m_hi = left <= 4 && have > 4 ? 0xFFu : 0u;
        rows = 0;
        // (loads without a branch between them, so that all are in flight together; the last bytes of a picture whose size is no
        // multiple of 4 come afterwards: asked for word by word they cost 1 us of 5 on 481 x 321, like this 0.1, and an instance without
        // them leaves 1600 x 2560 at 65 us instead of 67)
        const int whole = REST ? u.total & ~3 : u.total;
#pragma unroll
        for (int r = 0; r < K; ++r) {
            const int iy = y0 + r, a = (at + r * u.w_) & ~3;
            const bool in_row = real && iy >= 0 && iy < u.h;
            w0[r] = in_row && (unsigned)a < (unsigned)whole ? ld_tensor((const unsigned *)(u.x + a)) : 0u;
            w1[r] = in_row && (unsigned)(a + 4) < (unsigned)whole ? ld_tensor((const unsigned *)(u.x + a + 4)) : 0u;
            if (in_row) rows |= 1u << r;
        }
        if (REST && real && at + (K - 1) * u.w_ + 8 > whole) {
            const unsigned rest = pic_rest(u.x, whole, u.total);
#pragma unroll
            for (int r = 0; r < K; ++r) {
                const int a = (at + r * u.w_) & ~3;
                if ((rows >> r) & 1u) {
                    if (a == whole) w0[r] = rest;
                    if (a + 4 == whole) w1[r] = rest;
                }
            }
        }
    }

    // out: the 32 bytes of the operand row
    __device__ __forceinline__ void line_up(const PicArgs &u, uint4 &lo, uint4 &hi) const
    {
        unsigned a[K], b[K];
#pragma unroll
        for (int r = 0; r < K; ++r) {
            const int s = 8 * (at + r * u.w_);                         // (the shift takes it modulo 32)
            a[r] = __funnelshift_r(w0[r], w1[r], s) ^ u.flip;
            b[r] = K == 5 ? __funnelshift_r(w1[r], 0u, s) ^ u.flip : 0u;
        }
        if (!inner) {
#pragma unroll
            for (int r = 0; r < K; ++r) {
                a[r] &= (rows >> r) & 1u ? m_lo : 0u;
                b[r] &= (rows >> r) & 1u ? m_hi : 0u;
            }
        }
        if constexpr (K == 3) {
            lo = make_uint4(a[0], a[1], a[2], 0u);
            hi = make_uint4(0u, 0u, 0u, 0u);
        } else {
            lo = make_uint4(a[0], a[1], a[2], a[3]);
            hi = make_uint4(a[4], __byte_perm(__byte_perm(b[0], b[1], 0x0040), __byte_perm(b[2], b[3], 0x0040), 0x5410), b[4], 0u);
        }
    }
};

// byte of an operand row that holds tap (r, s)
constexpr int pic_byte(int k, int r, int s) { return s < 4 ? 4 * r + s : 4 * k + r; }

// NG: groups of 16 columns when known at compile time (0: from ua)
template <int EPI, int K, int NG, bool REST>
__global__ void __launch_bounds__(PIC_THREADS, 1)
picture_kernel(const __grid_constant__ PicArgs u, const __grid_constant__ ConvArgs a, const __grid_constant__ UmmaArgs ua)
{
    __shared__ __align__(1024) uint8_t slots[PIC_SLOTS][BLOCK_M * 32];
    __shared__ __align__(1024) uint8_t bank[PIC_MAX_N * 32];
    __shared__ __align__(16) int consts[PIC_MAX_N];
    __shared__ PicShared shared;
    PicShared *sh = &shared;
    const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0);
    const int lane = threadIdx.x & 31;
    const int G = (int)gridDim.x, bn = NG ? 16 * NG : ua.block_n;

    if (threadIdx.x == 0) {
        for (int s = 0; s < PIC_SLOTS; ++s) {
            mbar_init(smem_u32(&sh->done[s]), 1);
            mbar_init(smem_u32(&sh->empty[s]), 4);
        }
        mbar_init(smem_u32(&sh->drain), PIC_GROUPS);
        sh->abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        grid_dep_launch();
    }
    // operand rows of 32 bytes, 32-byte swizzle: the halves of rows 4 to 7 of every eight change places
    if ((int)threadIdx.x < 2 * bn) {
        const int row = (int)threadIdx.x >> 1, c = (int)threadIdx.x & 1;
        sts128(smem_u32(bank) + (uint32_t)(row * 32 + ((c ^ ((row >> 2) & 1)) << 4)), __ldg((const uint4 *)u.w + threadIdx.x));
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if ((int)threadIdx.x < bn) consts[threadIdx.x] = __ldg(ua.c_a + threadIdx.x);
    if (warp == 0) tmem_alloc(smem_u32(&sh->tmem_base), (uint32_t)u.tmem_cols);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = sh->tmem_base;
    grid_dep_wait();               // the picture may come from, and the output may still be read by, the kernel before this one

    if (warp < PIC_EPI_WARP0) {
        // ---------------------------------------------------------------- builders
        const int group = warp >> 2, row = (warp & 3) * 32 + lane;
        const uint32_t at = (uint32_t)(row * 32), swap = (uint32_t)((row >> 2) & 1) << 4;
        const uint32_t b_lo = ((smem_u32(bank) & 0x3FFFFu) >> 4) | (1u << 16);
        constexpr uint32_t HI = (uint32_t)((8 * 32) >> 4) | (1u << 14) | (6u << 29);        // 8-row groups 256 bytes apart, version 1, 32-byte swizzle
        int slot = group;
        uint32_t parity = 0;
        int tile = (int)blockIdx.x + group * G;
        PicPixel<K, REST> px;
        if (tile < u.tiles) px.load(u, tile * BLOCK_M + row);
        for (; tile < u.tiles; tile += PIC_GROUPS * G) {
            uint4 lo, hi;
            px.line_up(u, lo, hi);
            if (tile + PIC_GROUPS * G < u.tiles) px.load(u, (tile + PIC_GROUPS * G) * BLOCK_M + row);
            const bool ok = mbar_wait_warp(smem_u32(&sh->empty[slot]), parity ^ 1u, &sh->abort_flag, lane);
            if (!ok) pic_give_up(sh, u.status, 2);
            const uint32_t s = smem_u32(slots[slot]);
            if (ok) {
                sts128(s + at + swap, lo);
                sts128(s + at + (swap ^ 16u), hi);
            }
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            if (pic_group_sync(1 + group, !ok)) break;
            if ((warp & 3) == 0) {
                tc_fence_after();
                if (elect_one()) {
                    umma_i8_split(tmem_base + (uint32_t)(slot * bn), ((s & 0x3FFFFu) >> 4) | (1u << 16), b_lo, HI, u.idesc, 0u);
                    umma_commit(smem_u32(&sh->done[slot]));
                }
                __syncwarp();
            }
            slot += PIC_GROUPS;
            if (slot >= PIC_SLOTS) { slot -= PIC_SLOTS; parity ^= 1u; }
        }
    } else {
        // ---------------------------------------------------------------- epilogue: group `turn` takes every fourth tile
        const int quad = warp & 3, turn = (warp - PIC_EPI_WARP0) >> 2;
        const EpiScalars es = epi_scalars(a, ua);
        const uint32_t cap_s = smem_u32(consts);
        uint8_t *out = (uint8_t *)a.out + a.out_c_offset;
        int slot = turn;
        uint32_t parity = 0;
        for (int tile = (int)blockIdx.x + turn * G; tile < u.tiles; tile += (EPI_WARPS_MAX / 4) * G) {
            const int m = tile * BLOCK_M + quad * 32 + lane;
            if (!mbar_wait_warp(smem_u32(&sh->done[slot]), parity, &sh->abort_flag, lane)) {
                pic_give_up(sh, u.status, 4);
                break;
            }
            tc_fence_after();
            int acc[16];
            const uint32_t t_row = tmem_base + ((uint32_t)(quad * 32) << 16) + (uint32_t)(slot * bn);
            uint8_t *ocol = out + (long long)m * a.out_c_total;
            if (es.group_uniform) window_groups<EPI, NG, true, true>(t_row, nullptr, ocol, nullptr, m < u.m_total, 0, bn / 16, acc, es, a, ua, cap_s);
            else window_groups<EPI, NG, false, true>(t_row, nullptr, ocol, nullptr, m < u.m_total, 0, bn / 16, acc, es, a, ua, cap_s);
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&sh->empty[slot]));
            slot += EPI_WARPS_MAX / 4;
            if (slot >= PIC_SLOTS) { slot -= PIC_SLOTS; parity ^= 1u; }
        }
    }

    // ---------------------------------------------------------------- teardown
    __syncwarp();
    tc_fence_before();
    __syncthreads();
    if (sh->abort_flag) {
        // something gave up: wait (bounded) for the MMAs still in flight before TMEM and shared memory go
        volatile int never = 0;
        if (warp < PIC_EPI_WARP0 && (warp & 3) == 0 && elect_one()) {
            umma_commit(smem_u32(&sh->drain));
            mbar_wait(smem_u32(&sh->drain), 0, &never);
        }
        __syncthreads();
    }
    if (warp == 0) {
        tc_fence_after();
        tmem_dealloc(tmem_base, (uint32_t)u.tmem_cols);
    }
}

template <int EPI, int K, int NG>
cudaError_t pic_launch(const PicArgs &u, const ConvArgs &a, const UmmaArgs &ua, unsigned grid, cudaStream_t stream)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(PIC_THREADS);
    cfg.stream = stream;
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    return u.total % 4 ? cudaLaunchKernelEx(&cfg, picture_kernel<EPI, K, NG, true>, u, a, ua) : cudaLaunchKernelEx(&cfg, picture_kernel<EPI, K, NG, false>, u, a, ua);
}

template <int EPI, int K>
cudaError_t pic_launch_n(const PicArgs &u, const ConvArgs &a, const UmmaArgs &ua, unsigned grid, cudaStream_t stream)
{
    return ua.block_n == 64 ? pic_launch<EPI, K, 4>(u, a, ua, grid, stream) : pic_launch<EPI, K, 0>(u, a, ua, grid, stream);
}

template <int EPI>
cudaError_t pic_launch_k(int k, const PicArgs &u, const ConvArgs &a, const UmmaArgs &ua, unsigned grid, cudaStream_t stream)
{
    return k == 3 ? pic_launch_n<EPI, 3>(u, a, ua, grid, stream) : pic_launch_n<EPI, 5>(u, a, ua, grid, stream);
}

}  // namespace

// The filter bank of a layer this kernel takes (p->inner is the repacked form's plan, whose epilogue and geometry it shares);
// without one the layer is left to the repacked form.
int picture_setup(iconv_plan_t *p)
{
    const iconv_desc &d = p->d;
    const iconv_plan_t *in = p->inner;
    if (d.kh != d.kw || (d.kh != 3 && d.kh != 5) || in->block_n > PIC_MAX_N || in->c_out_pad != in->block_n ||
        (in->epi != umma_epilogue_fast() && in->epi != umma_epilogue_safe()))
        return ICONV_OK;
    // (offsets into the picture and pixel numbers are 32-bit)
    if ((long long)d.n * d.h * d.w >= (1ll << 31) - (long long)d.w * d.kh - 64 || (long long)d.n * p->h_out * p->w_out >= (1ll << 31) - 2 * 148 * BLOCK_M * PIC_GROUPS)
        return ICONV_OK;
    std::vector<int8_t> packed((size_t)in->block_n * 32, 0);
    for (int co = 0; co < d.c_out; ++co)
        for (int r = 0; r < d.kh; ++r)
            for (int s = 0; s < d.kw; ++s) packed[(size_t)co * 32 + pic_byte(d.kh, r, s)] = d.weights[((size_t)co * d.kh + r) * d.kw + s];
    ICONV_CUDA_TRY(cudaMalloc((void **)&p->w_packed, packed.size()));
    ICONV_CUDA_TRY(cudaMemcpy(p->w_packed, packed.data(), packed.size(), cudaMemcpyHostToDevice));
    return ICONV_OK;
}

int launch_picture(const iconv_plan_t *p, const ConvArgs &a, cudaStream_t stream)
{
    const iconv_desc &d = p->d;
    const iconv_plan_t *in = p->inner;
    if ((uintptr_t)a.out % 16) {              // (launch_stem sends no unaligned picture here)
        set_error("iconv_forward: tensor pointers must be 16-byte aligned");
        return ICONV_ERR_ALIGN;
    }
    int rc = umma_init_once();
    if (rc != ICONV_OK) return rc;
    UmmaArgs ua;
    rc = umma_args(in, ua);
    if (rc != ICONV_OK) return rc;
    PicArgs u;
    memset(&u, 0, sizeof(u));
    u.x = (const uint8_t *)a.x;
    u.w = p->w_packed;
    u.h = d.h; u.w_ = d.w; u.pad = d.pad; u.w_out = p->w_out;
    u.total = d.n * d.h * d.w;
    u.m_total = d.n * p->h_out * p->w_out;
    u.tiles = (u.m_total + BLOCK_M - 1) / BLOCK_M;
    u.tmem_cols = 32;
    while (u.tmem_cols < PIC_SLOTS * in->block_n) u.tmem_cols *= 2;
    u.flip = d.in_dtype == ICONV_U8_RAW128 ? 0x80808080u : 0u;
    u.idesc = ua.idesc;
    u.hw = (unsigned)(p->h_out * p->w_out);
    u.div_w_mul = ua.div_w_mul; u.div_w_shr = ua.div_w_shr; u.div_hw_mul = ua.div_hw_mul; u.div_hw_shr = ua.div_hw_shr;
    u.status = ua.status;
    const int sms = umma_device_ready(current_device_slot());
    const unsigned grid = (unsigned)(u.tiles < sms ? u.tiles : sms);
    ICONV_CUDA_TRY(in->epi == EPI_FAST ? pic_launch_k<EPI_FAST>(d.kh, u, a, ua, grid, stream) : pic_launch_k<EPI_SAFE>(d.kh, u, a, ua, grid, stream));
    return ICONV_OK;
}

}  // namespace iconv

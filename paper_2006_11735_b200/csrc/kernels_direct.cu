// CUDA-core kernels: the any-shape direct convolution (the path of last resort and the
// home of shapes no faster kernel takes), the stand-alone add-rescale, and the pooling
// layers of the ResNet-shaped networks.
#include "common.cuh"

namespace iconv {

__device__ __forceinline__ int dp4a_u8s8(unsigned a, int b, int c)
{
    int d;
    asm("dp4a.u32.s32 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(c));
    return d;
}
__device__ __forceinline__ int dp4a_s8s8(int a, int b, int c)
{
    int d;
    asm("dp4a.s32.s32 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(c));
    return d;
}

// One thread per output element (pixel-major, channel fastest).  VEC: the channel slice of
// every pixel starts on a 4-byte boundary and c_in is a multiple of 4, so the reduction
// runs on dp4a; otherwise byte by byte.
template <int IN_DTYPE, bool VEC>
__global__ void __launch_bounds__(256) direct_conv_kernel(const __grid_constant__ ConvArgs a)
{
    const long long total = (long long)a.n * a.h_out * a.w_out * a.c_out;
    for (long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x; e < total;
         e += (long long)gridDim.x * blockDim.x) {
        const int co = (int)(e % a.c_out);
        const long long pix = e / a.c_out;
        const int ow = (int)(pix % a.w_out);
        const int oh = (int)((pix / a.w_out) % a.h_out);
        const int n = (int)(pix / ((long long)a.w_out * a.h_out));
        int U = 0;
        for (int r = 0; r < a.kh; ++r) {
            const int ih = oh * a.stride - a.pad + r;
            if (ih < 0 || ih >= a.h) continue;
            for (int s = 0; s < a.kw; ++s) {
                const int iw = ow * a.stride - a.pad + s;
                if (iw < 0 || iw >= a.w_) continue;
                const long long xb = (((long long)n * a.h + ih) * a.w_ + iw) * a.in_c_total + a.in_c_offset;
                const long long wb = (((long long)co * a.kh + r) * a.kw + s) * a.c_in;
                if (VEC) {
                    const unsigned *xp = (const unsigned *)((const uint8_t *)a.x + xb);
                    const int *wp = (const int *)(a.w + wb);
                    for (int c4 = 0; c4 < a.c_in / 4; ++c4) {
                        unsigned xv = __ldg(xp + c4);
                        const int wv = __ldg(wp + c4);
                        if (IN_DTYPE == ICONV_U8) {
                            U = dp4a_u8s8(xv, wv, U);
                        } else {
                            if (IN_DTYPE == ICONV_U8_RAW128) xv ^= 0x80808080u;   // u8 - 128 as s8
                            U = dp4a_s8s8((int)xv, wv, U);
                        }
                    }
                } else {
                    for (int ci = 0; ci < a.c_in; ++ci) {
                        int xv;
                        if (IN_DTYPE == ICONV_S8) xv = ((const int8_t *)a.x)[xb + ci];
                        else xv = (int)((const uint8_t *)a.x)[xb + ci] - (IN_DTYPE == ICONV_U8_RAW128 ? 128 : 0);
                        U += xv * (int)a.w[wb + ci];
                    }
                }
            }
        }
        long long Y = (long long)U + a.bias[co];
        if (a.skip_dtype >= 0) {
            const int sv = load_skip(a.skip, pix * a.skip_c_total + a.skip_c_offset + co, a.skip_dtype);
            Y += round_shift64((long long)sv * a.skip_mul, a.skip_shift);
        }
        const long long oi = pix * a.out_c_total + a.out_c_offset + co;
        if (a.out_dtype == ICONV_I32) {
            ((int32_t *)a.out)[oi] = (int32_t)Y;
        } else {
            const int q = a.per_channel ? co : 0;
            const int V = requant_tail(Y, a.brelu, a.h_i[q], a.mul[q], a.shift[q], a.out_zero, a.out_lo, a.out_hi);
            if (a.out_dtype == ICONV_U8) ((uint8_t *)a.out)[oi] = (uint8_t)V;
            else ((int8_t *)a.out)[oi] = (int8_t)V;
        }
    }
}

int launch_direct(const ConvArgs &a, cudaStream_t stream)
{
    const long long total = (long long)a.n * a.h_out * a.w_out * a.c_out;
    if (total == 0) return ICONV_OK;
    const bool vec = (a.c_in % 4 == 0) && (a.in_c_total % 4 == 0) && (a.in_c_offset % 4 == 0) &&
                     (((uintptr_t)a.x) % 4 == 0) && (((uintptr_t)a.w) % 4 == 0);
    long long blocks = (total + 255) / 256;
    const long long cap = 148ll * 8 * 16;
    if (blocks > cap) blocks = cap;
#define LAUNCH(DT)                                                                         \
    if (vec) direct_conv_kernel<DT, true><<<(unsigned)blocks, 256, 0, stream>>>(a);        \
    else direct_conv_kernel<DT, false><<<(unsigned)blocks, 256, 0, stream>>>(a)
    switch (a.in_dtype) {
    case ICONV_U8: LAUNCH(ICONV_U8); break;
    case ICONV_S8: LAUNCH(ICONV_S8); break;
    default: LAUNCH(ICONV_U8_RAW128); break;
    }
#undef LAUNCH
    ICONV_CUDA_TRY(cudaGetLastError());
    return ICONV_OK;
}

// ---------------------------------------------------------------- add-rescale
__device__ __forceinline__ int load_elem(const void *p, long long i, int dtype)
{
    if (dtype == ICONV_U8) return ((const uint8_t *)p)[i];
    if (dtype == ICONV_S8) return ((const int8_t *)p)[i];
    return ((const int32_t *)p)[i];
}

// Loads 16 consecutive elements starting at i (a multiple of 16) with 16-byte accesses.
__device__ __forceinline__ void load16(const void *p, long long i, int dtype, int (&v)[16])
{
    if (dtype == ICONV_I32) {
        const int4 *q = (const int4 *)((const int32_t *)p + i);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int4 t = __ldg(q + k);
            v[4 * k] = t.x; v[4 * k + 1] = t.y; v[4 * k + 2] = t.z; v[4 * k + 3] = t.w;
        }
    } else {
        const uint4 t = __ldg((const uint4 *)((const uint8_t *)p + i));
        const unsigned wds[4] = {t.x, t.y, t.z, t.w};
#pragma unroll
        for (int k = 0; k < 16; ++k) {
            const unsigned b = (wds[k >> 2] >> (8 * (k & 3))) & 0xffu;
            v[k] = dtype == ICONV_U8 ? (int)b : (int)(int8_t)b;
        }
    }
}

__device__ __forceinline__ int add_one(const iadd_desc &d, int av, int bv)
{
    const long long Y = round_shift64((long long)(av - d.a_zero) * d.mul_a, d.sh_a) +
                        round_shift64((long long)(bv - d.b_zero) * d.mul_b, d.sh_b);
    return requant_tail(Y, d.brelu, d.h_i, d.mul, d.shift, d.out_zero, d.out_lo, d.out_hi);
}

__global__ void __launch_bounds__(256) add_requant_kernel(const __grid_constant__ iadd_desc d, const void *A,
                                                          const void *B, void *out, int vec_ok)
{
    const long long groups = d.n_elems / 16;
    const long long tid = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const long long nthreads = (long long)gridDim.x * blockDim.x;
    if (vec_ok) {
        for (long long g = tid; g < groups; g += nthreads) {
            int av[16], bv[16], ov[16];
            load16(A, g * 16, d.a_dtype, av);
            load16(B, g * 16, d.b_dtype, bv);
#pragma unroll
            for (int k = 0; k < 16; ++k) ov[k] = add_one(d, av[k], bv[k]);
            if (d.out_dtype == ICONV_I32) {
#pragma unroll
                for (int k = 0; k < 4; ++k)
                    ((int4 *)((int32_t *)out + g * 16))[k] = make_int4(ov[4 * k], ov[4 * k + 1], ov[4 * k + 2], ov[4 * k + 3]);
            } else {
                unsigned wds[4];
#pragma unroll
                for (int k = 0; k < 4; ++k)
                    wds[k] = (ov[4 * k] & 0xff) | ((ov[4 * k + 1] & 0xff) << 8) | ((ov[4 * k + 2] & 0xff) << 16) |
                             ((unsigned)(ov[4 * k + 3] & 0xff) << 24);
                *(uint4 *)((uint8_t *)out + g * 16) = make_uint4(wds[0], wds[1], wds[2], wds[3]);
            }
        }
    }
    // ragged tail (or everything when the pointers are not 16-byte aligned)
    for (long long i = (vec_ok ? groups * 16 : 0) + tid; i < d.n_elems; i += nthreads) {
        const int V = add_one(d, load_elem(A, i, d.a_dtype), load_elem(B, i, d.b_dtype));
        if (d.out_dtype == ICONV_I32) ((int32_t *)out)[i] = V;
        else if (d.out_dtype == ICONV_U8) ((uint8_t *)out)[i] = (uint8_t)V;
        else ((int8_t *)out)[i] = (int8_t)V;
    }
}

// The usual case in 32-bit arithmetic: 8-bit operands, an 8-bit result, and bounds (checked on the
// host from the descriptor alone) under which every product and sum below stays inside int32:
//   a' = (A * mul_a + ca) >> sh_a   with ca = 2^(sh_a-1) - a_zero * mul_a   (the zero point folded in)
//   b' likewise,  Y = a' + b',  clamp, V = (Y * mul + 2^(shift-1)) >> shift, zero point, saturation.
struct AddFast {
    int mul_a, ca, sh_a, mul_b, cb, sh_b;
    int y_lo, y_hi;          // BReLU's clamp, or the (unreachable) bounds of Y when there is none
    int mul, half, shift, out_zero, out_lo, out_hi;
    unsigned xor_a, xor_b;   // 0x80808080 turns int8 bytes into offset-binary (the offset rides in ca / cb)
    int form;                // ADD_*
};

// Forms of the 32-bit kernel.  ADD_CLAMP takes every descriptor whose products fit; the others are what
// the u8 saturation at the end makes of it when it stands for every clamp (out_zero = 0, the full
// range, and BReLU's bound, if any, already maps to 255), and are issue-bound no longer:
// 7 instructions an output instead of 17.
enum {
    ADD_CLAMP = 0,
    ADD_FREE = 1,            // V = sat_u8((Y * mul + half) >> shift)
    ADD_FREE_ID = 2,         // ... and A is at the target ratio already (mul_a = 1, sh_a = 0): its zero point rides in cb
    ADD_FREE_ID8 = 3         // ... and sh_b = 8, what iq_skip_sync yields unless B is scaled down a lot: shift and add are one instruction
};

__device__ __forceinline__ unsigned add_pack4(int v0, int v1, int v2, int v3)      // four values saturated to u8
{
    unsigned hi, d;
    asm("cvt.pack.sat.u8.s32.b32 %0, %1, %2, %3;" : "=r"(hi) : "r"(v3), "r"(v2), "r"(0));
    asm("cvt.pack.sat.u8.s32.b32 %0, %1, %2, %3;" : "=r"(d) : "r"(v1), "r"(v0), "r"(hi));
    return d;
}

template <int FORM>
__device__ __forceinline__ unsigned add_fast4(const AddFast &f, unsigned wa, unsigned wb)
{
    int V[4];
    wa ^= f.xor_a;
    wb ^= f.xor_b;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const int av = (int)__byte_perm(wa, 0, 0x4440 + k);
        const int bv = (int)__byte_perm(wb, 0, 0x4440 + k);
        const int b = (bv * f.mul_b + f.cb) >> (FORM == ADD_FREE_ID8 ? 8 : f.sh_b);
        int y = (FORM >= ADD_FREE_ID ? av : (av * f.mul_a + f.ca) >> f.sh_a) + b;
        if (FORM == ADD_CLAMP) {
            y = min(max(y, f.y_lo), f.y_hi);
            const int v = ((y * f.mul + f.half) >> f.shift) + f.out_zero;
            V[k] = min(max(v, f.out_lo), f.out_hi) & 0xff;
        } else {
            V[k] = (y * f.mul + f.half) >> f.shift;
        }
    }
    return add_pack4(V[0], V[1], V[2], V[3]);
}

// A block takes 1024 neighbouring groups of 16 elements, four to a thread with all eight loads in flight.
// Bound by memory: 51.4 M elements (154 MB) in 25.7 us, 6.0 TB/s, where the operands come from memory (27.6 before a launch could
// come up under the tail of the one before; on the same operands again and again, part of them in L2, 22.6 and 25.1); one wave
// of blocks that strides over the whole tensor takes 29.6, and the form with every clamp (ADD_CLAMP) is issue-bound at 41.  The
// fewer than 16 elements behind the last group are the last block's (a launch of their own cost 4 us).
constexpr int ADD_THREADS = 256, ADD_UNROLL = 4;
template <int FORM, bool RESIDENT>
__global__ void __launch_bounds__(ADD_THREADS, 4) add_requant_fast_kernel(const __grid_constant__ AddFast f, const uint4 *A, const uint4 *B, uint4 *out,
                                                                          long long n_elems)
{
    const long long groups = n_elems / 16, g = (long long)blockIdx.x * (ADD_THREADS * ADD_UNROLL) + threadIdx.x;
    // RESIDENT: a grid that is resident as a whole lets the next one come up only when it runs itself: before its wait, a third and a fourth come up
    // under it as well and take places unevenly (4.2 M elements again and again 5.7 us instead of 4.6, 2.1 M 4.3 instead of 2.9).  A
    // larger one has its last blocks running by then, and what comes up sooner is ready sooner (51.4 M: 25.9, behind the wait 26.0).
    if (!RESIDENT) grid_dep_launch();
    grid_dep_wait();                                // the operands may come from, and `out` still be read by, the kernel before this one
    if (RESIDENT) grid_dep_launch();
    uint4 a[ADD_UNROLL], b[ADD_UNROLL];
#pragma unroll
    for (int j = 0; j < ADD_UNROLL; ++j)
        if (g + j * ADD_THREADS < groups) { a[j] = __ldcs(A + g + j * ADD_THREADS); b[j] = __ldcs(B + g + j * ADD_THREADS); }
#pragma unroll
    for (int j = 0; j < ADD_UNROLL; ++j)
        if (g + j * ADD_THREADS < groups)
            __stcs(out + g + j * ADD_THREADS, make_uint4(add_fast4<FORM>(f, a[j].x, b[j].x), add_fast4<FORM>(f, a[j].y, b[j].y),
                                                         add_fast4<FORM>(f, a[j].z, b[j].z), add_fast4<FORM>(f, a[j].w, b[j].w)));
    const long long e = groups * 16 + threadIdx.x;
    if (blockIdx.x == gridDim.x - 1 && e < n_elems)
        ((uint8_t *)out)[e] = (uint8_t)add_fast4<FORM>(f, ((const uint8_t *)A)[e], ((const uint8_t *)B)[e]);
}

// Fills `f` and returns true when the 32-bit form is exact for every possible operand value.
static bool add_fast_plan(const iadd_desc &d, AddFast &f)
{
    const auto eight = [](int t) { return t == ICONV_U8 || t == ICONV_S8; };
    if (!eight(d.a_dtype) || !eight(d.b_dtype) || !eight(d.out_dtype)) return false;
    if (d.sh_a > 30 || d.sh_b > 30 || d.shift > 30) return false;
    const long long LIM = 1ll << 31;
    // stored byte as an unsigned number sv in [0, 255]; value = sv - z with z = zero (u8) or zero + 128 (offset-binary int8)
    const long long za = d.a_zero + (d.a_dtype == ICONV_S8 ? 128 : 0), zb = d.b_zero + (d.b_dtype == ICONV_S8 ? 128 : 0);
    const long long half_a = d.sh_a ? 1ll << (d.sh_a - 1) : 0, half_b = d.sh_b ? 1ll << (d.sh_b - 1) : 0, half = d.shift ? 1ll << (d.shift - 1) : 0;
    const long long ca = half_a - za * d.mul_a, cb = half_b - zb * d.mul_b;
    const auto mag = [](long long v) { return v < 0 ? -v : v; };
    if (mag(ca) + 255ll * d.mul_a >= LIM || mag(cb) + 255ll * d.mul_b >= LIM) return false;
    const long long a_lo = ca >> d.sh_a, a_hi = (255ll * d.mul_a + ca) >> d.sh_a, b_lo = cb >> d.sh_b, b_hi = (255ll * d.mul_b + cb) >> d.sh_b;
    long long y_lo = a_lo + b_lo, y_hi = a_hi + b_hi;
    if (d.brelu) { y_lo = 0; y_hi = d.h_i; }
    if (mag(y_lo) >= LIM || mag(y_hi) >= LIM) return false;
    if (mag(y_lo) * d.mul + half >= LIM || mag(y_hi) * d.mul + half >= LIM) return false;
    if (mag((long long)d.out_zero) >= (1ll << 30)) return false;
    f.mul_a = d.mul_a; f.ca = (int)ca; f.sh_a = d.sh_a; f.mul_b = d.mul_b; f.cb = (int)cb; f.sh_b = d.sh_b;
    f.y_lo = (int)y_lo; f.y_hi = (int)y_hi;
    f.mul = d.mul; f.half = (int)half; f.shift = d.shift; f.out_zero = d.out_zero; f.out_lo = d.out_lo; f.out_hi = d.out_hi;
    f.xor_a = d.a_dtype == ICONV_S8 ? 0x80808080u : 0u; f.xor_b = d.b_dtype == ICONV_S8 ? 0x80808080u : 0u;
    // the clamp-free forms: the range of Y without BReLU's clamp must fit as well
    f.form = ADD_CLAMP;
    const long long w_lo = a_lo + b_lo, w_hi = a_hi + b_hi;
    const bool bound_maps = !d.brelu || ((long long)d.h_i * d.mul + half) >> d.shift >= 255;
    if (d.out_dtype == ICONV_U8 && d.out_zero == 0 && d.out_lo == 0 && d.out_hi == 255 && bound_maps && mag(w_lo) * d.mul + half < LIM &&
        mag(w_hi) * d.mul + half < LIM) {
        f.form = ADD_FREE;
        const long long cz = cb - (za << d.sh_b);
        if (d.mul_a == 1 && d.sh_a == 0 && mag(za) < (1ll << 30) && mag(cz) + 255ll * d.mul_b < LIM) {
            f.form = d.sh_b == 8 ? ADD_FREE_ID8 : ADD_FREE_ID;
            f.cb = (int)cz;
        }
    }
    return true;
}

int launch_add_requant(const iadd_desc &d, const void *a, const void *b, void *out, cudaStream_t stream)
{
    if (d.n_elems == 0) return ICONV_OK;
    const int vec_ok = ((uintptr_t)a % 16 == 0) && ((uintptr_t)b % 16 == 0) && ((uintptr_t)out % 16 == 0);
    AddFast f;
    iadd_desc e = d;
    if (d.mul_b == 1 && d.sh_b == 0 && !(d.mul_a == 1 && d.sh_a == 0)) {      // the sum commutes: the operand at the target ratio is A
        e.a_dtype = d.b_dtype; e.a_zero = d.b_zero; e.mul_a = d.mul_b; e.sh_a = d.sh_b;
        e.b_dtype = d.a_dtype; e.b_zero = d.a_zero; e.mul_b = d.mul_a; e.sh_b = d.sh_a;
    }
    if (vec_ok && d.n_elems >= 16 && d.n_elems < (1ll << 44) && add_fast_plan(e, f)) {      // (the grid's x extent)
        const unsigned fblocks = (unsigned)((d.n_elems / 16 + ADD_THREADS * ADD_UNROLL - 1) / (ADD_THREADS * ADD_UNROLL));
        const bool swapped = e.mul_a != d.mul_a || e.sh_a != d.sh_a;
        const uint4 *A = (const uint4 *)(swapped ? b : a), *B = (const uint4 *)(swapped ? a : b);
        uint4 *o = (uint4 *)out;
        const bool resident = fblocks <= 4 * 148;
        switch (f.form) {
        case ADD_FREE_ID8: ICONV_CUDA_TRY(launch_kernel(resident ? add_requant_fast_kernel<ADD_FREE_ID8, true> : add_requant_fast_kernel<ADD_FREE_ID8, false>, true, fblocks, ADD_THREADS, 0, stream, f, A, B, o, (long long)d.n_elems)); break;
        case ADD_FREE_ID: ICONV_CUDA_TRY(launch_kernel(resident ? add_requant_fast_kernel<ADD_FREE_ID, true> : add_requant_fast_kernel<ADD_FREE_ID, false>, true, fblocks, ADD_THREADS, 0, stream, f, A, B, o, (long long)d.n_elems)); break;
        case ADD_FREE: ICONV_CUDA_TRY(launch_kernel(resident ? add_requant_fast_kernel<ADD_FREE, true> : add_requant_fast_kernel<ADD_FREE, false>, true, fblocks, ADD_THREADS, 0, stream, f, A, B, o, (long long)d.n_elems)); break;
        default: ICONV_CUDA_TRY(launch_kernel(resident ? add_requant_fast_kernel<ADD_CLAMP, true> : add_requant_fast_kernel<ADD_CLAMP, false>, true, fblocks, ADD_THREADS, 0, stream, f, A, B, o, (long long)d.n_elems)); break;
        }
        return ICONV_OK;
    }
    long long blocks = (d.n_elems / 16 + 255) / 256 + 1;
    if (blocks > 148ll * 32) blocks = 148ll * 32;
    add_requant_kernel<<<(unsigned)blocks, 256, 0, stream>>>(d, a, b, out, vec_ok);
    ICONV_CUDA_TRY(cudaGetLastError());
    return ICONV_OK;
}

// ---------------------------------------------------------------- pooling
// One thread per (output pixel, group of 16 channels): 16-byte loads, byte-wise unsigned max.
__global__ void __launch_bounds__(256) maxpool_kernel(const uint8_t *x, uint8_t *out, int n, int h, int w, int c,
                                                      int k, int stride, int pad, int h_out, int w_out)
{
    const int cg = c / 16;
    const long long total = (long long)n * h_out * w_out * cg;
    for (long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x; e < total;
         e += (long long)gridDim.x * blockDim.x) {
        const int g = (int)(e % cg);
        const long long pix = e / cg;
        const int ow = (int)(pix % w_out);
        const int oh = (int)((pix / w_out) % h_out);
        const int in = (int)(pix / ((long long)w_out * h_out));
        uint4 m = make_uint4(0, 0, 0, 0);
        for (int r = 0; r < k; ++r) {
            const int ih = oh * stride - pad + r;
            if (ih < 0 || ih >= h) continue;
            for (int s = 0; s < k; ++s) {
                const int iw = ow * stride - pad + s;
                if (iw < 0 || iw >= w) continue;
                const uint4 v = __ldg((const uint4 *)(x + (((long long)in * h + ih) * w + iw) * c) + g);
                m.x = __vmaxu4(m.x, v.x); m.y = __vmaxu4(m.y, v.y);
                m.z = __vmaxu4(m.z, v.z); m.w = __vmaxu4(m.w, v.w);
            }
        }
        *((uint4 *)(out + pix * c) + g) = m;
    }
}

// The 3x3 stride-2 pad-1 pooling of the ResNet-shaped networks: the nine loads carry no branch
// (a tap outside the image re-reads the nearest row or column inside it, which the window
// holds anyway, so the maximum is unchanged) and are all in flight together; one thread per
// (output pixel, group of 16 channels), 32-bit index arithmetic.
__global__ void __launch_bounds__(256) maxpool_3x3s2_kernel(const uint8_t *x, uint8_t *out, unsigned total,
                                                            int h, int w, int cg, int h_out, int w_out)
{
    const unsigned e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= total) return;
    const unsigned pix = e / (unsigned)cg;
    const int g = (int)(e - pix * (unsigned)cg);
    const unsigned row = pix / (unsigned)w_out;               // image * h_out + oh
    const int ow = (int)(pix - row * (unsigned)w_out);
    const unsigned in = row / (unsigned)h_out;
    const int oh = (int)(row - in * (unsigned)h_out);
    const uint4 *base = (const uint4 *)x + (size_t)in * h * w * cg + g;
    grid_dep_wait();                                          // x may come from, and `out` still be read by, the kernel before this one
    grid_dep_launch();
    uint4 v[9];
#pragma unroll
    for (int r = 0; r < 3; ++r) {
        const int ih = min(max(2 * oh - 1 + r, 0), h - 1);
#pragma unroll
        for (int s = 0; s < 3; ++s) {
            const int iw = min(max(2 * ow - 1 + s, 0), w - 1);
            v[r * 3 + s] = base[(size_t)(ih * w + iw) * cg];
        }
    }
    uint4 m = v[0];
#pragma unroll
    for (int t = 1; t < 9; ++t) {
        m.x = __vmaxu4(m.x, v[t].x); m.y = __vmaxu4(m.y, v[t].y);
        m.z = __vmaxu4(m.z, v[t].z); m.w = __vmaxu4(m.w, v[t].w);
    }
    ((uint4 *)out)[e] = m;
}

// The same with 32 channels per thread (32-byte loads and one 32-byte store: half the memory
// instructions, every store a whole sector), for channel counts that are multiples of 32 and
// 32-byte aligned tensors.
struct Bytes32 {
    unsigned v[8];
};
__device__ __forceinline__ Bytes32 ld_global_32(const void *p)
{
    Bytes32 r;
    asm volatile("ld.global.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(r.v[0]), "=r"(r.v[1]), "=r"(r.v[2]), "=r"(r.v[3]), "=r"(r.v[4]), "=r"(r.v[5]), "=r"(r.v[6]), "=r"(r.v[7])
                 : "l"(p));
    return r;
}
__device__ __forceinline__ void st_global_32(void *p, const Bytes32 &m)
{
    asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(p), "r"(m.v[0]), "r"(m.v[1]), "r"(m.v[2]), "r"(m.v[3]), "r"(m.v[4]),
                 "r"(m.v[5]), "r"(m.v[6]), "r"(m.v[7])
                 : "memory");
}
// ROWS output rows per thread, one below the other: the input row that two of them share is read once (its maximum stays), so
// that an output costs 6.75 loads at four rows instead of nine.  The loads are what the kernel is bound by: 256 x 112 x 112
// x 64 (256 MB) in 46.8 us, 5.5 TB/s; one row a thread takes 50.9, two 48.7, seven (too few threads in flight) 61.9.
// One row, where four would leave too few threads, has arithmetic of its own: as the general form with ROWS = 1 it is 3 to 5 % slower (32 x 56
// x 56 x 256: 7.9 us without early launches, 8.25, like this 7.4).  The next kernel may come up when this one runs, not before: with
// the signal ahead of the wait maps of 200 to 600 blocks, again and again, took 5.2 us for 3.4 and 5.6 for 5.4.
template <int ROWS>
__global__ void __launch_bounds__(256) maxpool_3x3s2_wide_kernel(const uint8_t *x, uint8_t *out, unsigned total,
                                                                 int h, int w, int cg, int h_out, int w_out, int bands)
{
    const unsigned e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= total) return;
    if (ROWS == 1) {
        const unsigned pix = e / (unsigned)cg;
        const int g = (int)(e - pix * (unsigned)cg);
        const unsigned row = pix / (unsigned)w_out;           // image * h_out + oh
        const int ow = (int)(pix - row * (unsigned)w_out);
        const unsigned in = row / (unsigned)h_out;
        const int oh = (int)(row - in * (unsigned)h_out);
        const uint8_t *base = x + ((size_t)in * h * w * cg + g) * 32;
        Bytes32 v[9];
        grid_dep_wait();                                      // x may come from, and `out` still be read by, the kernel before this one
        grid_dep_launch();
#pragma unroll
        for (int r = 0; r < 3; ++r) {
            const int ih = min(max(2 * oh - 1 + r, 0), h - 1);
#pragma unroll
            for (int s = 0; s < 3; ++s) {
                const int iw = min(max(2 * ow - 1 + s, 0), w - 1);
                v[r * 3 + s] = ld_global_32(base + (size_t)(ih * w + iw) * cg * 32);
            }
        }
#pragma unroll
        for (int t = 1; t < 9; ++t)
#pragma unroll
            for (int k = 0; k < 8; ++k) v[0].v[k] = __vmaxu4(v[0].v[k], v[t].v[k]);
        st_global_32(out + (size_t)e * 32, v[0]);
        return;
    }
    const unsigned col = e / (unsigned)cg;
    const int g = (int)(e - col * (unsigned)cg);
    const unsigned band = col / (unsigned)w_out;              // image * bands + band of ROWS output rows
    const int ow = (int)(col - band * (unsigned)w_out);
    const unsigned in = band / (unsigned)bands;
    const int oh0 = (int)(band - in * (unsigned)bands) * ROWS, rows = min(ROWS, h_out - oh0);
    const uint8_t *base = x + ((size_t)in * h * w * cg + g) * 32;
    uint8_t *to = out + (((size_t)in * h_out + oh0) * w_out + ow) * cg * 32 + (size_t)g * 32;
    size_t at[3];                                             // the window's three columns (outside the image: the nearest inside, which the window holds)
#pragma unroll
    for (int s = 0; s < 3; ++s) at[s] = (size_t)min(max(2 * ow - 1 + s, 0), w - 1) * cg * 32;
    auto load = [&](int ih, Bytes32 (&v)[3]) {
        const uint8_t *line = base + (size_t)min(max(ih, 0), h - 1) * w * cg * 32;
#pragma unroll
        for (int s = 0; s < 3; ++s) v[s] = ld_global_32(line + at[s]);
    };
    auto most = [](const Bytes32 &a, const Bytes32 &b) {
        Bytes32 m;
#pragma unroll
        for (int k = 0; k < 8; ++k) m.v[k] = __vmaxu4(a.v[k], b.v[k]);
        return m;
    };
    grid_dep_wait();                                          // x may come from, and `out` still be read by, the kernel before this one
    grid_dep_launch();
    Bytes32 shared_row;
#pragma unroll
    for (int r = 0; r < ROWS; ++r) {
        if (r >= rows) break;
        Bytes32 a[3], b[3], c[3];
        const int ih = 2 * (oh0 + r);
        if (r == 0) load(ih - 1, c);
        load(ih, a);
        load(ih + 1, b);
        if (r == 0) shared_row = most(most(c[0], c[1]), c[2]);
        const Bytes32 low = most(most(b[0], b[1]), b[2]);
        const Bytes32 m = most(most(most(a[0], a[1]), a[2]), most(shared_row, low));
        shared_row = low;
        st_global_32(to, m);
        to += (size_t)w_out * cg * 32;
    }
}

int launch_maxpool(const void *x, void *out, int n, int h, int w, int c, int k, int stride, int pad,
                   cudaStream_t stream)
{
    const int h_out = (h + 2 * pad - k) / stride + 1, w_out = (w + 2 * pad - k) / stride + 1;
    const long long total = (long long)n * h_out * w_out * (c / 16);
    if (total == 0) return ICONV_OK;
    if (k == 3 && stride == 2 && pad == 1 && c % 32 == 0 && ((uintptr_t)x % 32) == 0 && ((uintptr_t)out % 32) == 0 && total < (1ll << 31) &&
        (long long)n * h * w * (c / 16) < (1ll << 31)) {
        // four rows a thread while that leaves enough threads to fill the GPU twice
        const bool four = total / 2 >= 4ll * 2 * 148 * 768;
        const int bands = four ? (h_out + 3) / 4 : h_out;
        const unsigned threads = (unsigned)((long long)n * bands * w_out * (c / 32));
        ICONV_CUDA_TRY(launch_kernel(four ? maxpool_3x3s2_wide_kernel<4> : maxpool_3x3s2_wide_kernel<1>, true, (threads + 255) / 256, 256, 0, stream,
                                     (const uint8_t *)x, (uint8_t *)out, threads, h, w, c / 32, h_out, w_out, bands));
        return ICONV_OK;
    }
    if (k == 3 && stride == 2 && pad == 1 && total < (1ll << 31) && (long long)n * h * w * (c / 16) < (1ll << 31)) {
        ICONV_CUDA_TRY(launch_kernel(maxpool_3x3s2_kernel, true, (unsigned)((total + 255) / 256), 256, 0, stream, (const uint8_t *)x, (uint8_t *)out, (unsigned)total,
                                     h, w, c / 16, h_out, w_out));
        return ICONV_OK;
    }
    long long blocks = (total + 255) / 256;
    if (blocks > 148ll * 64) blocks = 148ll * 64;
    maxpool_kernel<<<(unsigned)blocks, 256, 0, stream>>>((const uint8_t *)x, (uint8_t *)out, n, h, w, c, k, stride,
                                                         pad, h_out, w_out);
    ICONV_CUDA_TRY(cudaGetLastError());
    return ICONV_OK;
}

// One thread per (image, channel); consecutive threads take consecutive channels, so every
// pixel row is read coalesced.  Sum, then Eq. 4 and a clamp to [0, max_int].
__global__ void __launch_bounds__(256) avgpool_kernel(const uint8_t *x, uint8_t *out, int n, int hw, int c, int mul,
                                                      int shift, int max_int)
{
    const long long total = (long long)n * c;
    for (long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x; e < total;
         e += (long long)gridDim.x * blockDim.x) {
        const int ch = (int)(e % c);
        const long long in = e / c;
        const uint8_t *p = x + in * hw * c + ch;
        long long sum = 0;
        for (int i = 0; i < hw; ++i) sum += p[(long long)i * c];
        long long V = round_shift64(sum * mul, shift);
        V = V < 0 ? 0 : (V > max_int ? max_int : V);
        out[e] = (uint8_t)V;
    }
}

// Sixteen channels per thread (16-byte loads), the pixels of an image shared out over PARTS threads whose sums meet
// in shared memory: one thread per image and 16 channels is a chain of loads that takes 6 us for a 7 x 7 map
// whatever the batch.  For channel counts that are multiples of 16 and 16-byte aligned tensors.  The sums stay far
// inside int32 (at most hw * 255).
template <int PARTS>
__global__ void __launch_bounds__(256) avgpool16_kernel(const uint8_t *x, uint8_t *out, int n, int hw, int cg, int mul, int shift,
                                                        int max_int)
{
    constexpr int AVG_GROUPS = 256 / PARTS, AVG_PARTS = PARTS;
    __shared__ int sums[AVG_PARTS][AVG_GROUPS][17];                        // (17: a part's threads fall on different banks)
    const int part = (int)threadIdx.x / AVG_GROUPS, slot = (int)threadIdx.x % AVG_GROUPS;
    const int e = blockIdx.x * AVG_GROUPS + slot;
    int sum[16];
#pragma unroll
    for (int k = 0; k < 16; ++k) sum[k] = 0;
    grid_dep_launch();
    grid_dep_wait();                                                       // x may come from, and `out` still be read by, the kernel before this one
    if (e < n * cg) {
        const int img = e / cg, g = e - img * cg;
        const uint4 *p = (const uint4 *)x + (size_t)img * hw * cg + g;
#pragma unroll 4
        for (int i = part; i < hw; i += AVG_PARTS) {
            const uint4 v = p[(size_t)i * cg];
            const unsigned wds[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
            for (int k = 0; k < 16; ++k) sum[k] += (int)((wds[k >> 2] >> (8 * (k & 3))) & 0xffu);
        }
    }
#pragma unroll
    for (int k = 0; k < 16; ++k) sums[part][slot][k] = sum[k];
    __syncthreads();
    // output bytes
    for (int b = (int)threadIdx.x; b < AVG_GROUPS * 16; b += 256) {
        const int o_slot = b / 16, k = b % 16, o = blockIdx.x * AVG_GROUPS + o_slot;
        if (o >= n * cg) break;
        int total = 0;
#pragma unroll
        for (int q = 0; q < AVG_PARTS; ++q) total += sums[q][o_slot][k];
        long long V = round_shift64((long long)total * mul, shift);
        V = V < 0 ? 0 : (V > max_int ? max_int : V);
        out[(size_t)o * 16 + k] = (uint8_t)V;
    }
}

int launch_avgpool(const void *x, void *out, int n, int h, int w, int c, int mul, int shift, int max_int,
                   cudaStream_t stream)
{
    const long long total = (long long)n * c;
    if (total == 0) return ICONV_OK;
    if (c % 16 == 0 && (uintptr_t)x % 16 == 0 && (uintptr_t)out % 16 == 0 && total / 16 < (1ll << 31) && max_int <= 255 &&
        (long long)h * w * 255 < (1ll << 31)) {
        const int groups = (int)(total / 16);
        // 16 threads per 16 channels while that does not fill the GPU (7 x 7 x 2048: one image 6.0 -> 2.6 us, 50 images 6.6
        // -> 3.6), four beyond (256 images: 7.1, and 9.4 with 16)
        if (groups <= 148 * 64)
            ICONV_CUDA_TRY(launch_kernel(avgpool16_kernel<16>, true, (unsigned)((groups + 15) / 16), 256, 0, stream, (const uint8_t *)x, (uint8_t *)out, n, h * w,
                                         c / 16, mul, shift, max_int));
        else
            ICONV_CUDA_TRY(launch_kernel(avgpool16_kernel<4>, true, (unsigned)((groups + 63) / 64), 256, 0, stream, (const uint8_t *)x, (uint8_t *)out, n, h * w,
                                         c / 16, mul, shift, max_int));
        return ICONV_OK;
    }
    long long blocks = (total + 255) / 256;
    avgpool_kernel<<<(unsigned)blocks, 256, 0, stream>>>((const uint8_t *)x, (uint8_t *)out, n, h * w, c, mul, shift,
                                                         max_int);
    ICONV_CUDA_TRY(cudaGetLastError());
    return ICONV_OK;
}

}  // namespace iconv

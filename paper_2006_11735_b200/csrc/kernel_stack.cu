// Host side of the stacked layers (umma_stack.cuh): which runs of layers it takes, on which tensors, the launch
// (the layers travel as kernel arguments) and what runs where it is refused.
#include <cuda.h>

#include <atomic>
#include <cstdio>
#include <cstring>
#include <new>
#include <vector>

#include "flow.h"
#include "umma_inst.h"
#include "umma_stack.cuh"

struct iconv_stack_s {
    std::vector<iconv_stack_layer> tensors; // one per layer (without its descriptor)
    std::vector<iconv_plan_t *> plans;      // one per layer: packed weights and epilogue constants
    iconv::StackLayers layers;
    iconv::StackArgs u;
    iconv::ConvArgs a;
    iconv::UmmaArgs ua;
    size_t smem = 0;
    iconv_flow_s *flow = nullptr;           // the general form, in place of all of the above
    ~iconv_stack_s()
    {
        iconv::flow_destroy(flow);
        for (iconv_plan_t *p : plans) iconv_plan_destroy(p);
    }
};

namespace iconv {

namespace {

const char *stack_refusal(const iconv_stack_layer *ls, int n)
{
    const iconv_desc &a = *ls[0].desc;
    if (a.kh != 3 || a.kw != 3 || a.stride != 1 || a.pad != 1) return "3x3 layers of stride 1 and pad 1 only";
    if (a.in_dtype != ICONV_U8 || a.out_dtype != ICONV_U8) return "8-bit unsigned activations only";
    if (a.c_in <= 32 || a.c_in > 64 || a.c_out > 64) return "33 to 64 input channels and at most 64 output channels";
    for (int i = 0; i < n; ++i) {
        const iconv_desc &d = *ls[i].desc;
        if (d.n != a.n || d.h != a.h || d.w != a.w || d.c_in != a.c_in || d.c_out != a.c_out || d.kh != a.kh || d.kw != a.kw || d.stride != a.stride ||
            d.pad != a.pad || d.in_dtype != a.in_dtype || d.out_dtype != a.out_dtype)
            return "the layers' geometries differ";
        if (d.skip_dtype >= 0 || d.proj_weights || d.per_channel) return "no skip, no per-channel parameters";
        if (i && (ls[i].x != ls[i - 1].out || d.in_c_total != ls[i - 1].desc->out_c_total || d.in_c_offset != ls[i - 1].desc->out_c_offset))
            return "every layer must read exactly the output slice of the one before";
    }
    return nullptr;
}

// A channel slice of a tensor: `pixels` rows of `width` bytes, `stride` bytes apart.
struct Slice {
    long long base, pixels, stride, width;
};

Slice slice(const void *tensor, int n, int h, int w, int c_total, int c_offset, int c)
{
    return {(long long)(uintptr_t)tensor + c_offset, (long long)n * h * w, c_total, c};
}

// Do two slices share a byte?  (Of different strides: may they?)
bool overlap(const Slice &a, const Slice &b)
{
    if (a.pixels < 1 || b.pixels < 1) return false;
    if (a.base + (a.pixels - 1) * a.stride + a.width <= b.base || b.base + (b.pixels - 1) * b.stride + b.width <= a.base) return false;
    if (a.stride != b.stride || a.stride < 1) return true;
    const long long d = ((b.base - a.base) % a.stride + a.stride) % a.stride;      // where b's rows begin between a's
    return d < a.width || d + b.width > a.stride;
}

}  // namespace

const char *stack_aliases(const iconv_stack_layer *ls, int n)
{
    constexpr int MOST = 64;                              // (more than any form takes: refused for their number)
    if (n > MOST) return nullptr;
    Slice in[MOST], aux[MOST], out[MOST];
    // (an equal stack may read fewer or more channels than are written; the flow kernel's writer_of wants the very slice)
    auto same = [](const Slice &a, const Slice &b) { return a.base == b.base && a.pixels == b.pixels && a.stride == b.stride; };
    auto shared = [](const Slice &a, const Slice &b, const void *p, const void *q) { return p == q || overlap(a, b); };
    for (int i = 0; i < n; ++i) {
        const iconv_desc &d = *ls[i].desc;
        if (d.stride < 1) return nullptr;                 // (no layer: planning it says so)
        const int ho = (d.h + 2 * d.pad - d.kh) / d.stride + 1, wo = (d.w + 2 * d.pad - d.kw) / d.stride + 1;
        in[i] = slice(ls[i].x, d.n, d.h, d.w, d.in_c_total, d.in_c_offset, d.c_in);
        out[i] = slice(ls[i].out, d.n, ho, wo, d.out_c_total, d.out_c_offset, d.c_out);
        aux[i] = {0, 0, 0, 0};
        if (d.skip_dtype >= 0 && d.proj_weights) aux[i] = slice(ls[i].skip, d.n, d.proj_h, d.proj_w, d.proj_c_total, d.proj_c_offset, d.proj_c_in);
        else if (d.skip_dtype >= 0) aux[i] = slice(ls[i].skip, d.n, ho, wo, d.skip_c_total, d.skip_c_offset, d.c_out);
        for (int j = 0; j <= i; ++j) {
            const bool aux_j = aux[j].pixels > 0;
            if (j < i) {
                if (overlap(in[i], out[j]) && !(ls[i].x == ls[j].out && same(in[i], out[j]))) return "reads part of another layer's output";
                if (overlap(aux[i], out[j]) && !(ls[i].skip == ls[j].out && same(aux[i], out[j]))) return "reads part of another layer's output";
                if (shared(out[i], out[j], ls[i].out, ls[j].out)) return "writes a tensor that an earlier layer writes";
            }
            if (shared(out[i], in[j], ls[i].out, ls[j].x) || (aux_j && shared(out[i], aux[j], ls[i].out, ls[j].skip)))
                return "writes a tensor that it or an earlier layer reads";
        }
    }
    return nullptr;
}

int stack_layer_refused(int rc, int i)
{
    if (rc == ICONV_ERR_UNSUPPORTED) {
        char why[400];
        snprintf(why, sizeof(why), "%s", iconv_last_error());
        set_error("iconv_plan_stack: layer %d: %s", i, why);
    }
    return rc;
}

namespace {

// Tile sequence, shared memory and pipeline of the stack, from the first layer's plan.
int stack_geometry(iconv_stack_t *s)
{
    const iconv_plan_t *p = s->plans[0];
    const iconv_desc &d = p->d;
    StackArgs &u = s->u;
    memset(&u, 0, sizeof(u));
    u.n_layers = (int)s->plans.size();
    u.tiles = p->win_tpi * d.n;
    u.chunks = (u.tiles + STACK_CHUNK - 1) / STACK_CHUNK;
    if ((long long)u.tiles * u.n_layers >= (1ll << 31) - 4096 || (long long)u.chunks * u.n_layers >= (1ll << 24)) {
        set_error("iconv_plan_stack: too many tiles");
        return ICONV_ERR_UNSUPPORTED;
    }
    // the patch of a tile reaches pad rows below its last pixel
    u.fwd = p->win_blocks ? p->win_vw + 1 : ((d.pad + 1) * p->win_vw + BLOCK_M - 1) / BLOCK_M + 1;
    u.h = d.h; u.w = d.w; u.c_out = d.c_out; u.pad = d.pad;
    u.block_n = p->block_n; u.kc = p->kc;
    u.b_tile_bytes = p->block_n * p->kc;                   // (the bank arrives as one box, tap after tap)
    if (u.b_tile_bytes % 1024) { set_error("iconv_plan_stack: a tap of the filter bank is no whole swizzle pattern"); return ICONV_ERR_UNSUPPORTED; }
    const int bank = u.b_tile_bytes * d.kh * d.kw;
    const int fixed = 1024 + (int)sizeof(StackShared) + 2 * bank + u.n_layers * u.block_n * 4;
    const int room = MAX_SMEM - fixed;
    u.stage_bytes = p->win_patch_bytes;
    u.stages = room / u.stage_bytes;
    u.nbuf = p->win_nbuf; u.lg_nbuf = u.nbuf == 8 ? 3 : u.nbuf == 4 ? 2 : 1;
    u.stages = u.stages < 6 ? u.stages / 2 * 2 : 6;        // issuers divide stages, as in the window kernel
    if (u.stages < 2) { set_error("iconv_plan_stack: two filter banks and the patches do not fit shared memory"); return ICONV_ERR_UNSUPPORTED; }
    int cols = 32;
    while (cols < u.nbuf * u.block_n) cols *= 2;
    u.tmem_cols = cols;
    u.cs = p->cs; u.bi = p->bi; u.part_n = p->half_n; u.epi_warps = p->epi_warps;
    u.vw = p->win_vw; u.bw = p->win_bw; u.bh = p->win_bh; u.full_width = p->win_full_width; u.blocks = p->win_blocks; u.tpi = p->win_tpi;
    u.idesc = (2u << 4) | (1u << 10) | ((unsigned)(p->block_n >> 3) << 17) | ((unsigned)(BLOCK_M >> 4) << 24);
    const unsigned long long layout = p->kc == 128 ? 2ull : (p->kc == 64 ? 4ull : 6ull);
    u.desc_hi_b = (unsigned)((((unsigned long long)((8 * p->kc) >> 4) << 32) | (1ull << 46) | (layout << 61)) >> 32);
    u.desc_hi_a = p->win_blocks ? (unsigned)((((unsigned long long)((p->win_bw * p->kc) >> 4) << 32) | (1ull << 46) | (layout << 61)) >> 32) : u.desc_hi_b;
    umma_find_divisor((unsigned)u.tpi, u.div_tpi_mul, u.div_tpi_shr);
    umma_find_divisor((unsigned)u.vw, u.div_vw_mul, u.div_vw_shr);
    s->smem = (size_t)fixed + (size_t)u.stages * u.stage_bytes;
    // what the shared epilogue reads of the single-layer kernels' arguments
    memset(&s->a, 0, sizeof(s->a));
    memset(&s->ua, 0, sizeof(s->ua));
    s->a.c_out = d.c_out; s->a.out_dtype = ICONV_U8; s->a.skip_dtype = -1;
    return ICONV_OK;
}

int stack_opt_in()
{
    static std::atomic<int> done[MAX_DEVICES];
    int rc = umma_init_once();
    if (rc != ICONV_OK) return rc;
    const int dev = current_device_slot();
    if (dev < 0) return ICONV_ERR_UNSUPPORTED;
    if (!done[dev].load(std::memory_order_acquire)) {
        ICONV_CUDA_TRY(cudaFuncSetAttribute(umma_stack_kernel<3, 3, 2>, cudaFuncAttributeMaxDynamicSharedMemorySize, MAX_SMEM));
        done[dev].store(1, std::memory_order_release);
    }
    return ICONV_OK;
}

int stack_build(iconv_stack_t *s, const iconv_stack_layer *ls, int n)
{
    int rc = stack_opt_in();
    if (rc != ICONV_OK) return rc;
    if (n > STACK_MAX_LAYERS) { set_error("iconv_plan_stack: more than %d layers", STACK_MAX_LAYERS); return ICONV_ERR_UNSUPPORTED; }
    memset(&s->layers, 0, sizeof(s->layers));
    for (int i = 0; i < n; ++i) {
        iconv_plan_t *p = nullptr;
        rc = iconv_plan(ls[i].desc, &p);
        if (rc != ICONV_OK) return stack_layer_refused(rc, i);
        s->plans.push_back(p);
        if (p->kernel != ICONV_KERNEL_UMMA || !p->window || p->epi != EPI_FAST || p->kc != 64 || p->group_uniform) {
            set_error("iconv_plan_stack: layer %d does not run in window mode with the clamp-free epilogue", i);
            return ICONV_ERR_UNSUPPORTED;
        }
        StackLayer &t = s->layers.l[i];
        rc = umma_encode_patch(p, ls[i].x, &t.x);
        if (rc != ICONV_OK) return rc;
        rc = umma_encode_bank(p, &t.w);
        if (rc != ICONV_OK) return rc;
        t.c_a = p->params_packed;
        t.out = (uint8_t *)ls[i].out + ls[i].desc->out_c_offset;
        t.out_c_total = ls[i].desc->out_c_total;
        t.q_mul = p->q_mul;
        t.q_shift = p->q_shift;
    }
    return stack_geometry(s);
}

}  // namespace

}  // namespace iconv

using namespace iconv;

extern "C" int iconv_stack_destroy(iconv_stack_t *s)
{
    delete s;
    return ICONV_OK;
}

extern "C" int iconv_plan_stack(const iconv_stack_layer *layers, int32_t n_layers, iconv_stack_t **stack_out)
{
    if (!layers || !stack_out || n_layers < 1) { set_error("iconv_plan_stack: null argument or no layers"); return ICONV_ERR_ARG; }
    *stack_out = nullptr;
    for (int i = 0; i < n_layers; ++i)        // (an empty batch's tensors may have no address)
        if (layers[i].desc && layers[i].desc->n == 0) { set_error("iconv_plan_stack: empty batch"); return ICONV_ERR_UNSUPPORTED; }
    for (int i = 0; i < n_layers; ++i) {
        if (!layers[i].desc || !layers[i].x || !layers[i].out) { set_error("iconv_plan_stack: layer %d has a null pointer", i); return ICONV_ERR_ARG; }
        if (((uintptr_t)layers[i].x % 16) || ((uintptr_t)layers[i].out % 16)) { set_error("iconv_plan_stack: tensor pointers must be 16-byte aligned"); return ICONV_ERR_ALIGN; }
        if (layers[i].desc->n < 1) { set_error("iconv_plan_stack: empty batch"); return ICONV_ERR_UNSUPPORTED; }
    }
    if (n_layers < 2) { set_error("iconv_plan_stack: a stack has at least two layers"); return ICONV_ERR_UNSUPPORTED; }
    if (const char *why = stack_aliases(layers, n_layers)) { set_error("iconv_plan_stack: a layer %s", why); return ICONV_ERR_UNSUPPORTED; }
    iconv_stack_t *s = new (std::nothrow) iconv_stack_s();
    if (!s) { set_error("iconv_plan_stack: out of host memory"); return ICONV_ERR_ARG; }
    // equal 3x3 layers of few channels read patches (umma_stack.cuh); anything else is the flow kernel's
    int rc = ICONV_ERR_UNSUPPORTED;
    if (!stack_refusal(layers, n_layers)) rc = stack_build(s, layers, n_layers);
    else rc = flow_plan(layers, n_layers, &s->flow);
    if (rc != ICONV_OK) { iconv_stack_destroy(s); return rc; }
    s->tensors.assign(layers, layers + n_layers);
    for (iconv_stack_layer &t : s->tensors) t.desc = nullptr;
    *stack_out = s;
    return ICONV_OK;
}

extern "C" size_t iconv_stack_sync_bytes(const iconv_stack_t *s)
{
    if (s && s->flow) return flow_sync_bytes(s->flow);
    return s ? sizeof(unsigned) * ((size_t)STACK_SYNC_WORDS + (size_t)s->u.n_layers * s->u.chunks) : 0;
}

int iconv::cooperative_launch_status(cudaError_t e, const char *what)
{
    if (e == cudaSuccess) return ICONV_OK;
    if (e != cudaErrorCooperativeLaunchTooLarge) return cuda_fail(e, what);
    cudaGetLastError();                                   // (nothing is enqueued; the next call is not to find this error)
    set_error("%s: not all of its CTAs can be resident here", what);
    return ICONV_ERR_UNSUPPORTED;
}

namespace {

int launch_stack(const iconv_stack_t *s, void *sync, cudaStream_t stream)
{
    int rc = stack_opt_in();
    if (rc != ICONV_OK) return rc;
    const int sms = umma_device_ready(current_device_slot());
    StackArgs u = s->u;
    u.sync = (unsigned *)sync;
    u.status = device_status_ptr();
    if (!u.status || sms < 1) { set_error("iconv_forward_stack: device not initialised"); return ICONV_ERR_CUDA; }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(u.tiles < sms ? u.tiles : sms));
    cfg.blockDim = dim3(STACK_THREADS);
    cfg.dynamicSmemBytes = s->smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;      // the CTAs wait on one another: all resident, or the launch is refused
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cooperative_launch_status(cudaLaunchKernelEx(&cfg, umma_stack_kernel<3, 3, 2>, s->layers, u, s->a, s->ua), "the stack kernel");
}

// The layers one after another, for a part of a GPU that does not hold all CTAs of the one launch.
int forward_apart(const iconv_stack_t *s, void *stream)
{
    for (size_t i = 0; i < s->tensors.size(); ++i) {
        const iconv_stack_layer &t = s->tensors[i];
        const int rc = iconv_forward(s->flow ? flow_layer(s->flow, (int)i) : s->plans[i], t.x, t.skip, t.out, nullptr, stream);
        if (rc != ICONV_OK) return rc;
    }
    return ICONV_OK;
}

}  // namespace

extern "C" int iconv_forward_stack(const iconv_stack_t *s, void *sync, void *cuda_stream)
{
    if (!s || !sync) { set_error("iconv_forward_stack: null argument"); return ICONV_ERR_ARG; }
    if ((uintptr_t)sync % 16) { set_error("iconv_forward_stack: the counters must be 16-byte aligned"); return ICONV_ERR_ALIGN; }
    const int rc = s->flow ? flow_forward(s->flow, sync, (cudaStream_t)cuda_stream) : launch_stack(s, sync, (cudaStream_t)cuda_stream);
    return rc == ICONV_ERR_UNSUPPORTED ? forward_apart(s, cuda_stream) : rc;
}

extern "C" int iconv_selftest_stack_apart(const iconv_stack_t *s, void *cuda_stream)
{
    if (!s) { set_error("iconv_selftest_stack_apart: null stack"); return ICONV_ERR_ARG; }
    return forward_apart(s, cuda_stream);
}

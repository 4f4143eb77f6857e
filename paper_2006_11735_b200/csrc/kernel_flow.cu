// Host side of a run of different layers in one launch (umma_flow.cuh): which runs it takes, the tile
// shapes, the dependencies between the layers, the launch.
#include <cuda.h>

#include <atomic>
#include <cstring>
#include <new>
#include <vector>

#include "flow.h"
#include "umma_flow.cuh"
#include "umma_inst.h"

struct iconv_flow_s {
    std::vector<iconv_plan_t *> plans;      // one per layer: packed weights and epilogue constants
    iconv::FlowArgs f;
    ~iconv_flow_s()
    {
        for (iconv_plan_t *p : plans) iconv_plan_destroy(p);
    }
};

namespace iconv {

namespace {

constexpr size_t FLOW_SMEM = (size_t)FLOW_STAGES * FLOW_SLOT + 2 * FLOW_STAGING + sizeof(FlowShared);
static_assert(FLOW_SMEM <= (size_t)MAX_SMEM, "shared memory of the flow kernel");

std::atomic<int> g_flow_pairs[MAX_DEVICES];      // CTA pairs that are resident at a time (0: not asked yet)

int flow_opt_in(int *pairs)
{
    const int rc = umma_init_once();
    if (rc != ICONV_OK) return rc;
    const int dev = current_device_slot();
    if (dev < 0) return ICONV_ERR_UNSUPPORTED;
    int n = g_flow_pairs[dev].load(std::memory_order_acquire);
    if (!n) {
        ICONV_CUDA_TRY(cudaFuncSetAttribute(umma_flow_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, MAX_SMEM));
        cudaLaunchConfig_t cfg = {};
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = 2;
        attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
        cfg.gridDim = dim3(2u * (unsigned)(umma_device_ready(dev) / 2));
        cfg.blockDim = dim3(FLOW_THREADS);
        cfg.dynamicSmemBytes = FLOW_SMEM;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        ICONV_CUDA_TRY(cudaOccupancyMaxActiveClusters(&n, umma_flow_kernel, &cfg));
        if (n > umma_device_ready(dev) / 2) n = umma_device_ready(dev) / 2;
        if (n < 1) { set_error("iconv_plan_stack: no CTA pair of the flow kernel is resident on this device"); return ICONV_ERR_UNSUPPORTED; }
        g_flow_pairs[dev].store(n, std::memory_order_release);
    }
    *pairs = n;
    return ICONV_OK;
}

const char *flow_refusal(const iconv_stack_layer &l)
{
    const iconv_desc &d = *l.desc;
    if (d.in_dtype != ICONV_U8 || d.out_dtype != ICONV_U8) return "8-bit unsigned activations only";
    if (d.c_in % 64 || d.c_out % 64 || d.in_c_total % 16 || d.in_c_offset % 16 || d.out_c_total % 16 || d.out_c_offset % 16) return "channels must be multiples of 64, strides and offsets of 16";
    if (d.kh != d.kw || d.kh > 15 || d.pad >= d.kh || d.stride > 8) return "square filters of at most 15, padded by less than their size, strides up to 8";
    if (d.per_channel) return "per-layer mul / shift / h_i only";
    if (d.h > 32767 || d.w > 32767 || (long long)d.n * d.h * d.w >= (1ll << 31) - 512) return "more pixels than 32-bit indices hold";
    if (d.proj_weights) {
        if (d.skip_dtype != ICONV_U8 || d.proj_c_in % 64 || d.proj_c_total % 16 || d.proj_c_offset % 16) return "a projection reads unsigned 8-bit channels in multiples of 64";
        if (d.proj_k > 15 || d.proj_pad >= d.proj_k || d.proj_stride > 8 || d.proj_h > 32767 || d.proj_w > 32767) return "projection filter, padding, stride or input too large";
        if ((long long)d.n * d.proj_h * d.proj_w >= (1ll << 31) - 512) return "more pixels than 32-bit indices hold";
    } else if (d.skip_dtype >= 0) {
        if (d.skip_dtype == ICONV_I32 || d.skip_c_total % 16 || d.skip_c_offset % 16) return "8-bit skips at channel strides and offsets of 16 only";
    }
    if (d.skip_dtype >= 0 && !l.skip) return "a layer with a skip needs its tensor";
    return nullptr;
}

// Index of the layer that writes the tensor at `ptr` (the latest before `i`), -1: none of the run (stack_aliases has
// seen to tensors that overlap at other addresses).  Its output slice must be exactly what is read.
int writer_of(const iconv_stack_layer *ls, int i, const void *ptr, int n, int h, int w, int c, int c_total, int c_offset, bool *fits)
{
    for (int j = i - 1; j >= 0; --j) {
        if (ls[j].out != ptr) continue;
        const iconv_desc &d = *ls[j].desc;
        const int ho = (d.h + 2 * d.pad - d.kh) / d.stride + 1, wo = (d.w + 2 * d.pad - d.kw) / d.stride + 1;
        if (d.n != n || ho != h || wo != w || d.c_out != c || d.out_c_total != c_total || d.out_c_offset != c_offset) *fits = false;
        return j;
    }
    return -1;
}

// Tile of a layer: columns and pixel rows per CTA, powers of two for which the layer takes least, by a model of
// one pass.  A CTA pulls its operands at about 45 bytes per clock, a K = 32 step takes block_n / 2 clocks (48
// at least) whatever the rows, the epilogue about 11 clocks per column with a skip and 7 without; and no layer
// is shorter than one tile.  So a large layer gets 256 columns and 128 rows, a small one as many tiles as
// there are CTA pairs.
void choose_tile(const iconv_plan_t *p, int k_iters, long long m_total, int pairs, bool proj, bool skip, int *block_n, int *rows)
{
    double best = 0;
    *block_n = 0;
    for (int r = BLOCK_M; r >= 32; r /= 2) {
        const double units = (double)((m_total + 2 * r - 1) / (2 * r));
        for (int n = proj ? 128 : 256; n >= 32; n /= 2) {
            if (p->d.c_out % n) continue;
            const double mma = (p->kc / 32) * (n / 2 > 48 ? n / 2 : 48), tma = (r + n / 2) * (double)p->kc / 45.0;
            const double loop = k_iters * (mma > tma ? mma : tma), epi = n * (proj ? 13.0 : skip ? 11.0 : 7.0);
            const double waves = units * (p->d.c_out / n) / pairs;
            const double cost = waves > 1.0 ? waves * (loop > epi ? loop : epi) : loop + epi;
            if (!*block_n || cost < 0.97 * best) { *block_n = n; *rows = r; best = cost; }
        }
    }
}

int flow_build(iconv_flow_s *s, const iconv_stack_layer *ls, int n, int pairs)
{
    FlowArgs &f = s->f;
    int units = 0;
    std::vector<int> unit0((size_t)n);
    for (int i = 0; i < n; ++i) {
        iconv_desc d = *ls[i].desc;
        d.kernel = ICONV_KERNEL_UMMA_IM2COL;
        iconv_plan_t *p = nullptr;
        int rc = iconv_plan(&d, &p);
        if (rc != ICONV_OK) return stack_layer_refused(rc, i);
        s->plans.push_back(p);
        const bool proj = d.proj_weights != nullptr, skip = d.skip_dtype >= 0 && !proj;
        FlowLayer &L = f.l[i];
        switch (p->epi) {
        case EPI_FAST: L.epi = FLOW_FAST; break;
        case EPI_FAST_SKIP8: L.epi = FLOW_FAST_SKIP8; break;
        case EPI_SAFE: L.epi = FLOW_SAFE; break;
        case EPI_SAFE_SKIP8: L.epi = FLOW_SAFE_SKIP8; break;
        default: L.epi = p->epi == EPI_PROJ && p->proj32 ? (p->proj32 == 2 ? FLOW_PROJ_FAST : FLOW_PROJ_SAFE) : 255;
        }
        const bool clamps = L.epi == FLOW_SAFE || L.epi == FLOW_SAFE_SKIP8 || L.epi == FLOW_PROJ_FAST || L.epi == FLOW_PROJ_SAFE;
        if (p->kernel != ICONV_KERNEL_UMMA || L.epi == 255 || (clamps && p->tail) || p->kc < 64 || p->c_in_pad != d.c_in || (proj && p->proj_c_in_pad != d.proj_c_in)) {
            set_error("iconv_plan_stack: layer %d needs an epilogue or a padding that a run of layers does not have", i);
            return ICONV_ERR_UNSUPPORTED;
        }
        bool fits = true;
        const int xw = writer_of(ls, i, ls[i].x, d.n, d.h, d.w, d.c_in, d.in_c_total, d.in_c_offset, &fits);
        int aw = -1;
        if (proj) aw = writer_of(ls, i, ls[i].skip, d.n, d.proj_h, d.proj_w, d.proj_c_in, d.proj_c_total, d.proj_c_offset, &fits);
        else if (skip) aw = writer_of(ls, i, ls[i].skip, d.n, p->h_out, p->w_out, d.c_out, d.skip_c_total, d.skip_c_offset, &fits);
        if (!fits) {
            set_error("iconv_plan_stack: a layer reads part of another layer's output");
            return ICONV_ERR_UNSUPPORTED;
        }
        const long long m_total = (long long)d.n * p->h_out * p->w_out;
        const int taps = d.kh * d.kw, ptaps = proj ? d.proj_k * d.proj_k : 0;
        L.cchunks = (unsigned char)(d.c_in / p->kc);
        L.p_cchunks = proj ? (unsigned char)(d.proj_c_in / p->kc) : 0;
        L.p_iters = (unsigned short)(ptaps * L.p_cchunks);
        const int k_iters = L.p_iters + taps * L.cchunks;
        if (d.c_in / p->kc > 255 || (proj && d.proj_c_in / p->kc > 255) || k_iters > 65535 || m_total >= (1ll << 31) - 512) {
            set_error("iconv_plan_stack: layer %d is too large", i);
            return ICONV_ERR_UNSUPPORTED;
        }
        L.k_iters = (unsigned short)k_iters;
        L.c_a = p->params_packed;
        L.m_total = (int)m_total;
        int block_n = 0, rows = 0;
        choose_tile(p, k_iters, m_total, pairs, proj, skip, &block_n, &rows);
        L.block_n = (unsigned short)block_n;
        L.rows = (unsigned char)rows;
        L.shift = rows == 128 ? 8 : rows == 64 ? 7 : 6;
        L.units = (int)((m_total + 2 * rows - 1) / (2 * rows));
        L.n_tiles = (unsigned short)(d.c_out / L.block_n);
        if ((long long)L.units * L.n_tiles >= (1ll << 30) || (long long)units + L.units >= (1ll << 26)) {
            set_error("iconv_plan_stack: too many tiles");
            return ICONV_ERR_UNSUPPORTED;
        }
        L.tiles = L.units * L.n_tiles;
        L.unit0 = unit0[(size_t)i] = units;
        units += L.units;
        L.src_unit = xw < 0 ? -1 : unit0[(size_t)xw];
        L.aux_unit = aw < 0 ? -1 : unit0[(size_t)aw];
        L.src_shift = xw < 0 ? 0 : f.l[xw].shift;
        L.aux_shift = aw < 0 ? 0 : f.l[aw].shift;
        L.q_mul = p->q_mul; L.q_shift = (unsigned char)p->q_shift; L.q_h = p->q_h;
        L.skip_mul = d.skip_mul; L.skip_shift = (unsigned char)d.skip_shift; L.skip_signed = d.skip_dtype == ICONV_S8;
        unsigned shr;
        umma_find_divisor((unsigned)L.n_tiles, L.nt_mul, shr); L.nt_shr = (unsigned char)shr;
        umma_find_divisor((unsigned)p->w_out, L.w_mul, shr); L.w_shr = (unsigned char)shr;
        umma_find_divisor((unsigned)(p->h_out * p->w_out), L.hw_mul, shr); L.hw_shr = (unsigned char)shr;
        L.h_out = (unsigned short)p->h_out; L.w_out = (unsigned short)p->w_out; L.h_in = (unsigned short)d.h; L.w_in = (unsigned short)d.w;
        L.kc = (unsigned char)p->kc;
        L.kh = (unsigned char)d.kh; L.kw = (unsigned char)d.kw; L.stride = (unsigned char)d.stride; L.pad = (unsigned char)d.pad;
        L.dense = d.kh == 1 && d.stride == 1 && d.pad == 0;
        // maps: activations, weights (half of a B tile per CTA), output pieces of 128 rows, skip pieces or the projection's input
        if (L.dense) rc = umma_encode_2d(&L.x, (const uint8_t *)ls[i].x + d.in_c_offset, d.c_in, m_total, d.in_c_total, p->kc, rows, p->kc);
        else rc = umma_encode_im2col(p, ls[i].x, rows, &L.x);
        if (rc != ICONV_OK) return rc;
        const long long k_pad = (long long)k_iters * p->kc;
        rc = umma_encode_2d(&L.w, p->w_packed, k_pad, p->c_out_pad, k_pad, p->kc, L.block_n / 2, p->kc);
        if (rc != ICONV_OK) return rc;
        const int piece = L.block_n < 64 ? L.block_n : 64;
        rc = umma_encode_2d(&L.out, (uint8_t *)ls[i].out + d.out_c_offset, d.c_out, m_total, d.out_c_total, piece, rows, piece);
        if (rc != ICONV_OK) return rc;
        if (proj) {
            L.h_aux = (unsigned short)d.proj_h; L.w_aux = (unsigned short)d.proj_w;
            L.p_k = (unsigned char)d.proj_k; L.p_stride = (unsigned char)d.proj_stride; L.p_pad = (unsigned char)d.proj_pad;
            L.p_dense = d.proj_k == 1 && d.proj_stride == 1 && d.proj_pad == 0;
            if (L.p_dense) rc = umma_encode_2d(&L.aux, (const uint8_t *)ls[i].skip + d.proj_c_offset, d.proj_c_in, m_total, d.proj_c_total, p->kc, rows, p->kc);
            else rc = umma_encode_projection(p, ls[i].skip, rows, &L.aux);
        } else if (skip) {
            rc = umma_encode_2d(&L.aux, (const uint8_t *)ls[i].skip + d.skip_c_offset, d.c_out, m_total, d.skip_c_total, piece, rows, piece);
        }
        if (rc != ICONV_OK) return rc;
    }
    f.n_layers = n;
    f.units = units;
    return ICONV_OK;
}

}  // namespace

int flow_plan(const iconv_stack_layer *layers, int n, iconv_flow_s **out)
{
    *out = nullptr;
    if (n > FLOW_MAX_LAYERS) { set_error("iconv_plan_stack: more than %d layers", FLOW_MAX_LAYERS); return ICONV_ERR_UNSUPPORTED; }
    for (int i = 0; i < n; ++i)
        if (const char *why = flow_refusal(layers[i])) { set_error("iconv_plan_stack: layer %d: %s", i, why); return ICONV_ERR_UNSUPPORTED; }
    int pairs = 0;
    int rc = flow_opt_in(&pairs);
    if (rc != ICONV_OK) return rc;
    iconv_flow_s *s = new (std::nothrow) iconv_flow_s();
    if (!s) { set_error("iconv_plan_stack: out of host memory"); return ICONV_ERR_ARG; }
    memset(&s->f, 0, sizeof(s->f));
    rc = flow_build(s, layers, n, pairs);
    if (rc != ICONV_OK) { delete s; return rc; }
    *out = s;
    return ICONV_OK;
}

void flow_destroy(iconv_flow_s *s) { delete s; }

size_t flow_sync_bytes(const iconv_flow_s *s) { return sizeof(unsigned) * ((size_t)FLOW_SYNC_WORDS + (size_t)s->f.units); }

int flow_forward(const iconv_flow_s *s, void *sync, cudaStream_t stream)
{
    int pairs = 0;
    const int rc = flow_opt_in(&pairs);
    if (rc != ICONV_OK) return rc;
    FlowArgs f = s->f;
    f.sync = (unsigned *)sync;
    f.status = device_status_ptr();
    if (!f.status) { set_error("device status word not available"); return ICONV_ERR_CUDA; }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(2u * (unsigned)pairs);
    cfg.blockDim = dim3(FLOW_THREADS);
    cfg.dynamicSmemBytes = FLOW_SMEM;
    cfg.stream = stream;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 2;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeCooperative;      // the CTAs wait on one another: all resident, or the launch is refused
    attr[1].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    return cooperative_launch_status(cudaLaunchKernelEx(&cfg, umma_flow_kernel, f), "the flow kernel");
}

const iconv_plan_t *flow_layer(const iconv_flow_s *s, int i) { return s->plans[(size_t)i]; }

}  // namespace iconv

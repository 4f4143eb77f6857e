// Body of one translation unit of the rolling window kernel: define ICONV_INST_EPI (2, 4 or 8) before including.
#include "umma_inst.h"
#include "umma_roll.cuh"

namespace iconv {

#define ICONV_CAT2(a, b) a##b
#define ICONV_CAT(a, b) ICONV_CAT2(a, b)

namespace {

constexpr int E = ICONV_INST_EPI;
constexpr bool MORE = E != EPI_NARROW;          // the narrow variant has sixteen columns only

template <typename F>
cudaError_t for_instance(int k, int n, F &&f)
{
    if (MORE && k == 3 && n == 64) return f(umma_roll_kernel<E, 3, MORE ? 64 : 16>);
    if (MORE && k == 3 && n == 48) return f(umma_roll_kernel<E, 3, MORE ? 48 : 16>);
    if (MORE && k == 3 && n == 32) return f(umma_roll_kernel<E, 3, MORE ? 32 : 16>);
    if (k == 3 && n == 16) return f(umma_roll_kernel<E, 3, 16>);
    if (MORE && k == 5 && n == 48) return f(umma_roll_kernel<E, 5, MORE ? 48 : 16>);
    if (MORE && k == 5 && n == 32) return f(umma_roll_kernel<E, 5, MORE ? 32 : 16>);
    if (k == 5 && n == 16) return f(umma_roll_kernel<E, 5, 16>);
    return cudaErrorInvalidValue;
}

}  // namespace

cudaError_t ICONV_CAT(umma_roll_launch_, ICONV_INST_EPI)(int k, int n, const UmmaLaunch &l, const RollArgs &r)
{
    return for_instance(k, n, [&](auto kernel) { return umma_launch_pdl(kernel, l, *l.tmap_x, *l.tmap_w, r, *l.a, *l.u); });
}

cudaError_t ICONV_CAT(umma_roll_opt_in_, ICONV_INST_EPI)()
{
    cudaError_t e = cudaSuccess;
    for (int k : {3, 5})
        for (int n : {16, 32, 48, 64})
            if (e == cudaSuccess && n * k <= 256 && (MORE || n == 16))
                e = for_instance(k, n, [](auto kernel) { return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, MAX_SMEM); });
    return e;
}

}  // namespace iconv

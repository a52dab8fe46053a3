// The encoder kernels of one element format: ZC_ENC_FMT selects it (1: BF16, 2: FP8, 3: scale bytes, 4: FP4), one object
// each, so that a build compiles the formats side by side.
#include "zc_encode.cuh"

namespace zc {

template <int F>
cudaError_t enc_launch_t(int shape, uint32_t grid, uint32_t threads, size_t smem, cudaStream_t st, const EncParams& P, const EncRanges& R)
{
    cudaError_t e = cudaSuccess;
    auto launch = [&](auto kern) {
        e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return;
#if ZC_DEBUG_CHECKS
        dbg_set_ranges(st, R.in, R.in_bytes, R.out, R.out_bytes, R.ws, R.ws_bytes);
#else
        (void)R;
#endif
        kern<<<grid, threads, smem, st>>>(P);
        e = cudaGetLastError();
    };
    const bool h0 = P.mode[0] == ZC_MODE_HUFF, h1 = P.mode[1] == ZC_MODE_HUFF;
#define ZC_ENC_CASE(SHAPE)                                                   \
    if (h0 && h1) launch(encode_kernel<F, true, true, SHAPE>);              \
    else if (h0) launch(encode_kernel<F, true, false, SHAPE>);              \
    else if (h1) launch(encode_kernel<F, false, true, SHAPE>);              \
    else launch(encode_kernel<F, false, false, SHAPE>);
    if (shape == kEncSolo) { ZC_ENC_CASE(kEncSolo) }
    else if (shape == kEncTeam) { ZC_ENC_CASE(kEncTeam) }
    else if (shape == kEncAny) { ZC_ENC_CASE(kEncAny) }
    else if (shape == kEncAny48) { ZC_ENC_CASE(kEncAny48) }
    else if (shape == kEncBig) { ZC_ENC_CASE(kEncBig) }
    else if (shape == kEncUnit) { ZC_ENC_CASE(kEncUnit) }
#undef ZC_ENC_CASE
#define ZC_ENC_CASE(SHAPE)                                                   \
    if (h0) launch(encode_kernel<F, true, false, SHAPE>);                   \
    else launch(encode_kernel<F, false, true, SHAPE>);
    else if (shape == kEncSolo80) { ZC_ENC_CASE(kEncSolo80) }                // one coded stream only (see enc_shape)
    else if (shape == kEncSolo96) { ZC_ENC_CASE(kEncSolo96) }
    else { ZC_ENC_CASE(kEncSolo112) }
#undef ZC_ENC_CASE
    return e;
}

#if ZC_DEBUG_CHECKS
#define ZC_ENC_COUNTS(out) dbg_read_counts(out)
#else
#define ZC_ENC_COUNTS(out) (void)(out)
#endif
#define ZC_ENC_DEFINE(NAME, F)                                                                                            \
    cudaError_t enc_launch_##NAME(int shape, uint32_t grid, uint32_t threads, size_t smem, cudaStream_t st,               \
                                  const EncParams& P, const EncRanges& R)                                                 \
    { return enc_launch_t<F>(shape, grid, threads, smem, st, P, R); }                                                     \
    void enc_debug_counts_##NAME(uint32_t out[2]) { ZC_ENC_COUNTS(out); }
#if ZC_ENC_FMT == 1
ZC_ENC_DEFINE(bf16, ZC_FMT_BF16)
#elif ZC_ENC_FMT == 2
ZC_ENC_DEFINE(fp8, ZC_FMT_FP8_E4M3)
#elif ZC_ENC_FMT == 3
ZC_ENC_DEFINE(scale, ZC_FMT_SCALE_U8)
#else
ZC_ENC_DEFINE(fp4, ZC_FMT_FP4_E2M1)
#endif

}  // namespace zc

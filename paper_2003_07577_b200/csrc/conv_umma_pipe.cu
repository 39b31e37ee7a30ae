// Dispatch over the activation bit count for the persistent pipeline kernel, and its host-side geometry check.
#include "conv_umma_pipe.cuh"

namespace ebs {

#define EBS_DECLARE_PIPE(AB)                                         \
    const ConvVariant* conv_umma_pipe_variant_a##AB(int variant);    \
    unsigned long long conv_umma_pipe_timeouts_a##AB();
EBS_DECLARE_PIPE(0) EBS_DECLARE_PIPE(1) EBS_DECLARE_PIPE(2) EBS_DECLARE_PIPE(3) EBS_DECLARE_PIPE(4)
EBS_DECLARE_PIPE(5) EBS_DECLARE_PIPE(6) EBS_DECLARE_PIPE(7) EBS_DECLARE_PIPE(8)
#undef EBS_DECLARE_PIPE

int pipe_sm_count() {
    int dev = 0, n = 148;
    if (cudaGetDevice(&dev) == cudaSuccess) cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
    return n > 0 ? n : 148;
}

bool pipe_words_map(const ConvParams& p, const PipeGeom& g, CUtensorMap* map) {
    if ((p.test_flags & 4) != 0) return false;
    using Encode = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*, const cuuint32_t*,
                                const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
    static const Encode encode = [] {
        void* fn = nullptr;
        cudaDriverEntryPointQueryResult found;
        return cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &found) == cudaSuccess &&
                       found == cudaDriverEntryPointSuccess
                   ? reinterpret_cast<Encode>(fn)
                   : nullptr;
    }();
    if (!encode) return false;
    const cuuint64_t dims[2] = {(cuuint64_t)p.CW * p.x_words, (cuuint64_t)p.N * p.H * p.W}, strides[1] = {dims[0] * 4};
    const cuuint32_t box[2] = {(cuuint32_t)(g.raw_words * p.x_words), (cuuint32_t)(g.tile_pix < 256 ? g.tile_pix : 256)}, one[2] = {1, 1};
    return encode(map, CU_TENSOR_MAP_DATA_TYPE_UINT32, 2, const_cast<uint32_t*>(p.x), dims, strides, box, one, CU_TENSOR_MAP_INTERLEAVE_NONE,
                  CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

const ConvVariant* conv_umma_pipe_variant(int a_bits, int variant) {
    switch (a_bits) {
        case 0: return conv_umma_pipe_variant_a0(variant);      // activations as byte codes
        case 1: return conv_umma_pipe_variant_a1(variant);
        case 2: return conv_umma_pipe_variant_a2(variant);
        case 3: return conv_umma_pipe_variant_a3(variant);
        case 4: return conv_umma_pipe_variant_a4(variant);
        case 5: return conv_umma_pipe_variant_a5(variant);
        case 6: return conv_umma_pipe_variant_a6(variant);
        case 7: return conv_umma_pipe_variant_a7(variant);
        case 8: return conv_umma_pipe_variant_a8(variant);
        default: return nullptr;
    }
}

bool conv_umma_pipe_applies(const ConvParams& p, int variant) {
    if (variant == 3) return pipe_pair_request_ok(p) && pipe_geometry(p, 256, pipe_sm_count(), p.pipe_m_sub, true).ok;
    return variant >= 0 && variant < 3 && pipe_geometry(p, 64 << variant, pipe_sm_count(), p.pipe_m_sub).ok;
}

bool conv_umma_pipe_copies(const ConvParams& p, int variant) {
    if (variant < 0 || variant > 2) return false;
    const PipeGeom g = pipe_geometry(p, 64 << variant, pipe_sm_count(), p.pipe_m_sub);
    return g.ok && g.tma;
}

void conv_umma_pipe_route(const ConvParams& p, int variant, int* route) {
    const PipeGeom g = pipe_geometry(p, variant == 3 ? 256 : 64 << variant, pipe_sm_count(), p.pipe_m_sub, variant == 3);
    const int values[] = {g.tma, g.m_sub, g.ks, g.kss, g.n_stages, g.b_resident, g.raw_slots, g.b_slots, g.n_ptiles * g.n_ctiles};
    for (int v : values) *route++ = v;
}

unsigned long long conv_umma_pipe_timeouts() {
    return conv_umma_pipe_timeouts_a0() + conv_umma_pipe_timeouts_a1() + conv_umma_pipe_timeouts_a2() + conv_umma_pipe_timeouts_a3() +
           conv_umma_pipe_timeouts_a4() + conv_umma_pipe_timeouts_a5() + conv_umma_pipe_timeouts_a6() +
           conv_umma_pipe_timeouts_a7() + conv_umma_pipe_timeouts_a8();
}

}  // namespace ebs

// Dispatch over the activation bit count for the tile kernel, and its host-side geometry.
#include "conv_umma_tile.cuh"

namespace ebs {

#define EBS_EACH_AB(X) X(1) X(2) X(3) X(4) X(5) X(6) X(7) X(8)
#define EBS_DECLARE_TILE(AB)                                    \
    const ConvVariant* conv_umma_variant_a##AB(int variant);    \
    unsigned long long conv_umma_timeouts_a##AB();
EBS_EACH_AB(EBS_DECLARE_TILE)

int tile_sm_count() {
    static int cached[64] = {};
    int dev = 0, n = 148;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return n;
    if (!cached[dev]) {
        cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
        cached[dev] = n > 0 ? n : 148;
    }
    return cached[dev];
}

const ConvVariant* conv_umma_variant(int a_bits, int variant) {
    switch (a_bits) {
#define EBS_TILE_CASE(AB) case AB: return conv_umma_variant_a##AB(variant);
        EBS_EACH_AB(EBS_TILE_CASE)
        default: return nullptr;
    }
}

bool conv_umma_applies(const ConvParams& p, int variant) {
    return variant >= 0 && variant < NUM_TILE_VARIANTS && tile_geometry(p, 16 << variant, tile_sm_count(), p.tile_split).ok;
}

float conv_umma_cost(const ConvParams& p, int variant) {
    const TileGeom g = tile_geometry(p, 16 << variant, tile_sm_count(), p.tile_split);
    return g.ok ? g.cost : -1.0f;
}

bool conv_umma_tap_form(const ConvParams& p) {
    FrameGeom g{};
    return tile_tap_form(p, g);
}

unsigned long long conv_umma_tile_timeouts() {
    unsigned long long v = 0;
#define EBS_TILE_SUM(AB) v += conv_umma_timeouts_a##AB();
    EBS_EACH_AB(EBS_TILE_SUM)
    return v;
}

}  // namespace ebs

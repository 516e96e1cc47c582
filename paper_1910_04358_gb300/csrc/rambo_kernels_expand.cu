// rambo_kernels_expand.cu -- row-by-row expansion of bucket masks (Algorithm
// 2's union and intersection): per repetition, the OR of the document bitmaps
// of the passing buckets; then the AND over the R repetitions, written as a
// K-bit mask.  It serves the geometries that the answer kernels' 16-bit slots
// do not reach (R * B of 16,384 and more).  Also the OR table it and the
// persistent fused query use.
#include "rambo_query_common.cuh"

namespace rgpu {
namespace {

// C answer words a lane: as many as the answer has for it, up to 8 (lanes with
// 8 words of an answer that has 16 in all: 515 us for 1,000 k-mers over 500
// documents, R = 4, B = 4,096, and 209 with one).
template <int C>
__global__ void __launch_bounds__(EXPAND_THREADS) k_expand(ExpandArgs a) {
    const int lane = threadIdx.x & 31;
    const uint64_t warp = (uint64_t)blockIdx.x * (EXPAND_THREADS / 32) + threadIdx.x / 32;
    const uint64_t nwarps = (uint64_t)gridDim.x * (EXPAND_THREADS / 32);
    const uint32_t chunks = (a.W + 32 * C - 1) / (32 * C);
    const uint64_t units = a.n * chunks;
    for (uint64_t u = warp; u < units; u += nwarps) {
        const uint64_t q = chunks == 1 ? u : u / chunks;
        expand_one<C>(a, a.acc + q * a.Gw, q, (uint32_t)(u - q * chunks) * 32 * C + lane, lane);
    }
}

// Byte table: tab[((r*NJ + j)*256 + v)*W + w] = OR over set bits i of v
// (8j+i < B) of DocBits[r][8j+i][w].
__global__ void k_build_bytetab(const uint32_t *docbits, uint32_t B, uint32_t R, uint32_t W,
                                uint32_t *tab) {
    const uint32_t NJ = (B + 7) / 8;
    const uint64_t total = (uint64_t)R * NJ * 256 * W;
    for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < total;
         i += (uint64_t)gridDim.x * blockDim.x) {
        const uint32_t w = (uint32_t)(i % W);
        const uint64_t rest = i / W;
        const uint32_t v = (uint32_t)(rest % 256);
        const uint64_t rj = rest / 256;
        const uint32_t j = (uint32_t)(rj % NJ), r = (uint32_t)(rj / NJ);
        uint32_t o = 0;
        for (uint32_t t = 0; t < 8; ++t) {
            const uint32_t b = 8 * j + t;
            if (((v >> t) & 1u) && b < B) o |= docbits[((uint64_t)r * B + b) * W + w];
        }
        tab[i] = o;
    }
}

}  // namespace

template <int C>
cudaError_t launch_expand_c(const ExpandArgs &a, int max_blocks, cudaStream_t s) {
    const uint64_t units = a.n * ((a.W + 32 * C - 1) / (32 * C));
    uint64_t blocks = (units + EXPAND_THREADS / 32 - 1) / (EXPAND_THREADS / 32);
    if (blocks > (uint64_t)max_blocks) blocks = (uint64_t)max_blocks;
    k_expand<C><<<(unsigned)blocks, EXPAND_THREADS, 0, s>>>(a);
    return cudaGetLastError();
}

cudaError_t launch_expand(const ExpandArgs &a, int max_blocks, cudaStream_t s) {
    if (a.n == 0) return cudaSuccess;
    const uint32_t words = (a.W + 31) / 32;  // of a lane
    if (words >= 8) return launch_expand_c<8>(a, max_blocks, s);
    if (words >= 4) return launch_expand_c<4>(a, max_blocks, s);
    if (words >= 2) return launch_expand_c<2>(a, max_blocks, s);
    return launch_expand_c<1>(a, max_blocks, s);
}

uint64_t bytetab_words(uint32_t B, uint32_t R, uint32_t W) {
    return (uint64_t)R * ((B + 7) / 8) * 256 * W;
}

cudaError_t launch_build_bytetab(const uint32_t *docbits, uint32_t B, uint32_t R, uint32_t W,
                                 uint32_t *tab, int sm_count, cudaStream_t s) {
    k_build_bytetab<<<sm_count * 8, 256, 0, s>>>(docbits, B, R, W, tab);
    return cudaGetLastError();
}

}  // namespace rgpu

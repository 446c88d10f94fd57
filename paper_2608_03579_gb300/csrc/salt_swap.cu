// Residual swap-in of a batch (Section "Multi-Tenant Serving": only the
// ultra-low-rank residual moves host -> device): one launch reads every blob
// from page-locked host memory over the host link and writes it into its
// slot, in place of one copy per blob.
//
// Bound by the host link.  A copy engine pays about 2 us between two copies
// (64 blobs of 1.31 MB: 535 us one by one, 400 us as one copy); this kernel
// takes 416 us.  Its CTAs (128 threads, at most 48 registers, no shared memory,
// the same shared-memory split) fit on an SM beside one CTA of the apply or
// base kernels, so a swap on a side stream runs beside a step's applies: those
// have 384 threads of 145 to 151 registers, handed out in eights, and 152 * 384
// + 48 * 128 is within the SM's 65,536 (their shared memory is asserted where
// they are).  An 8B decode step of four layers with that swap: 538 us by
// copies, 458 with 20 CTAs, 545 with 12 (518 us alone), 481 with 28 and 588
// with 64 (405 alone, but they hold up the applies).
#include "salt_internal.cuh"

#include <algorithm>

namespace salt {
namespace {

constexpr int SWAP_THREADS = 128;
constexpr int SWAP_CTAS_PER_SM = 10;                        // caps the registers: 65,536 / 1,280 threads, in eights
static_assert(65536 / (SWAP_CTAS_PER_SM * SWAP_THREADS) / 8 * 8 * SWAP_THREADS + 152 * APPLY_THREADS <= 65536,
              "registers beside a CTA of the apply or base kernels");
constexpr int SWAP_UNROLL = 8;                              // 16-byte loads a thread has in flight
constexpr int SWAP_PIECE = SWAP_THREADS * SWAP_UNROLL;      // 16-byte units a CTA moves at a time
constexpr int SWAP_CTAS = 20;                               // 0.33 MB in flight (above)
constexpr int SWAP_MAX = 256;                               // blobs per launch (the parameter block)

struct SwapParams {
    const uint4 *src[SWAP_MAX];
    uint4 *dst[SWAP_MAX];
    uint32_t n16[SWAP_MAX];      // 16-byte units of the blob
    uint32_t piece0[SWAP_MAX + 1];  // first piece of the blob, then the total
    int32_t n;
};

__global__ void __launch_bounds__(SWAP_THREADS, SWAP_CTAS_PER_SM) salt_swap_kernel(const __grid_constant__ SwapParams p)
{
    int e = 0;
    for (uint32_t piece = blockIdx.x; piece < p.piece0[p.n]; piece += gridDim.x) {
        while (piece >= p.piece0[e + 1]) ++e;
        const uint4 *src = p.src[e];
        uint4 *dst = p.dst[e];
        const uint32_t n16 = p.n16[e], first = (piece - p.piece0[e]) * SWAP_PIECE + threadIdx.x;
        uint4 v[SWAP_UNROLL];
#pragma unroll
        for (int k = 0; k < SWAP_UNROLL; ++k)
            if (first + k * SWAP_THREADS < n16) v[k] = __ldcs(src + first + k * SWAP_THREADS);
#pragma unroll
        for (int k = 0; k < SWAP_UNROLL; ++k)
            if (first + k * SWAP_THREADS < n16) dst[first + k * SWAP_THREADS] = v[k];
    }
}

}  // namespace

cudaError_t swap_prepare()
{
    // the shared-memory split of the kernels it runs beside: an SM does not
    // hold CTAs of two splits at once
    return cudaFuncSetAttribute(salt_swap_kernel, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
}

cudaError_t launch_swap(int n, const void *const *src, void *const *dst, const uint64_t *bytes, cudaStream_t stream)
{
    for (int at = 0; at < n; at += SWAP_MAX) {
        SwapParams p;
        p.n = std::min(SWAP_MAX, n - at);
        uint32_t pieces = 0;
        for (int i = 0; i < p.n; ++i) {
            p.src[i] = static_cast<const uint4 *>(src[at + i]);
            p.dst[i] = static_cast<uint4 *>(dst[at + i]);
            p.n16[i] = (uint32_t)(bytes[at + i] / 16);
            p.piece0[i] = pieces;
            pieces += (p.n16[i] + SWAP_PIECE - 1) / SWAP_PIECE;
        }
        p.piece0[p.n] = pieces;
        salt_swap_kernel<<<std::min<uint32_t>(SWAP_CTAS, pieces), SWAP_THREADS, 0, stream>>>(p);
        const cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

}  // namespace salt

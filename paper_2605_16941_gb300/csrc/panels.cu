// panels.cu -- the LM head's panel layout (wino_lm_head_panels): Wp[k][v][c] = W[v][64k + c].
//
// The score kernel reads W in copies of bn/2 vocabulary rows x one 64-wide K slice.  In row-major W such a
// copy is bn/2 pieces of 128 B, 2*d bytes apart; in the panel copy it is one contiguous block.
//
// The copy is bound by HBM (each byte read and written once, 2.07 GB at d = 4096, V = 126464).  One CTA copies a tile of
// 32 vocabulary rows x 8 panels, all of a thread's loads in flight at once: runs of 1 KB are read and of 4 KB written,
// against 128 B and one piece in flight per thread in a grid-stride loop over the pieces of Wp (343 us; here 301 us,
// 6.88 TB/s, the copy rate; the same tiles in a loop of 8 CTAs per SM 321 us).  d = 2048, V = 10001: 16.4 -> 14.6 us.
// Heads of fewer than 8 panels take 256 rows x 1 panel.
#include <cstdint>

#include "internal.h"

namespace wino {
namespace {

constexpr int kThreads = 256;
constexpr int kPieces = 8;  // 16-byte pieces per thread: a tile has kRows * kPanels = 256 runs of 128 bytes

template <int kRows, int kPanels>
__global__ void __launch_bounds__(kThreads) panels_kernel(const uint4 *__restrict__ W, uint4 *__restrict__ Wp,
                                                          int32_t V, int32_t n_kb, int32_t row_tiles)
{
    static_assert(kRows * kPanels * 8 == kPieces * kThreads, "tile size");
    const int32_t kt = (int32_t)blockIdx.x / row_tiles;
    const int32_t v0 = ((int32_t)blockIdx.x - kt * row_tiles) * kRows, k0 = kt * kPanels;
    // piece p of the tile: 16 bytes c8 (of 8) of row r in panel k, p = (k * kRows + r) * 8 + c8; consecutive threads
    // write consecutive pieces
    uint4 x[kPieces];
#pragma unroll
    for (int i = 0; i < kPieces; ++i) {
        const int p = i * kThreads + (int)threadIdx.x, c8 = p & 7, r = (p >> 3) % kRows, k = (p >> 3) / kRows;
        if (v0 + r < V && k0 + k < n_kb)
            x[i] = __ldcs(W + ((int64_t)(v0 + r) * n_kb + k0 + k) * 8 + c8);
    }
#pragma unroll
    for (int i = 0; i < kPieces; ++i) {
        const int p = i * kThreads + (int)threadIdx.x, c8 = p & 7, r = (p >> 3) % kRows, k = (p >> 3) / kRows;
        if (v0 + r < V && k0 + k < n_kb)
            __stcs(Wp + ((int64_t)(k0 + k) * V + v0 + r) * 8 + c8, x[i]);
    }
}

template <int kRows, int kPanels>
void launch(const uint16_t *W, uint16_t *Wp, int32_t n_kb, int32_t V, cudaStream_t stream)
{
    const int32_t row_tiles = (V + kRows - 1) / kRows;
    const int64_t tiles = (int64_t)row_tiles * ((n_kb + kPanels - 1) / kPanels);  // n_kb * V <= 2^30: fits an int
    panels_kernel<kRows, kPanels><<<(unsigned)tiles, kThreads, 0, stream>>>(
        reinterpret_cast<const uint4 *>(W), reinterpret_cast<uint4 *>(Wp), V, n_kb, row_tiles);
}

}  // namespace

cudaError_t launch_panels(const uint16_t *W, uint16_t *Wp, int64_t d, int64_t V, cudaStream_t stream)
{
    const int32_t n_kb = (int32_t)(d / 64);
    if (n_kb >= 8)
        launch<32, 8>(W, Wp, n_kb, (int32_t)V, stream);
    else
        launch<256, 1>(W, Wp, n_kb, (int32_t)V, stream);
    return cudaGetLastError();
}

}  // namespace wino

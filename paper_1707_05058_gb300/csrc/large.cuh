// PSD projection of large clique blocks (order > 128) on the tensor cores.
//
// The projection of Section 4.1.2 (Eq. XkUpdate) needs only
//   P(W) = V max(Lambda, 0) V^T = (W + W sign(W)) / 2,
// where sign(W) = V sign(Lambda) V^T.  For blocks of order 129 .. a few
// thousand (the cliques of a minimum-degree extension of a sparse random
// graph) the sign is computed by an odd polynomial (Newton-Schulz) iteration
// on X_0 = W / ||W||_F, whose eigenvalues lie in [-1, 1]:
//   phase 1 (range growth), N1 steps of  X <- a X + b X^3 + c X^5,
//            a = 3.30, b = -3.66, c = 1.36: p(1) = 1, p maps [0, 1.3] into
//            itself, every x >= 0.22 into [0.7, 1.3], and small x grow by
//            3.3 per step (coefficients found by a grid search under those
//            constraints);
//   phase 2 (convergence), N2 steps of  X <- 1.5 X - 0.5 X^3  (Newton-Schulz;
//            quadratic convergence from [0.7, 1.3]);
// then P = (W + W X) / 2.  With N1 = 16 and N2 = 5 every eigenvalue with
// |lambda| >= 1e-8 ||W||_F reaches |sign| within float32 rounding of 1; an
// eigenvalue below that contributes at most |lambda| / 2 to the error of P.
// Every step is a product of two symmetric matrices that commute (powers of
// W), so only the lower tiles of each product are computed and mirrored.
//
// Products run in float32 accuracy as three float16 products (Ootomo and
// Yokota, 2022): 2^12 x = x_hi + 2^-11 x_lo with x_hi = half(2^12 x) and x_lo =
// half(2^11 (2^12 x - x_hi)), 22 bits and a sign; A B ~ A_hi B_hi + 2^-11 (A_hi
// B_lo + A_lo B_hi), both sums accumulated in float32, each in its own columns of
// tensor memory.  Every operand is a power of X_0 or a polynomial of it with
// eigenvalues below 4, so 2^12 x stays below the float16 range, and an entry
// keeps its 22 bits down to 1.5e-8 (an absolute 2^-48 below that).
// Every such matrix is stored as its (hi, lo) pair, row-major, block k at a
// 256-byte aligned offset with row pitch S_k = ceil(s_k / 128) * 128 (zero
// padding stays zero under odd polynomials); W itself and P stay float32.
// Before, the pairs were TF32 ones (float32 words): twice the bytes, of which
// an SM takes in about 45 a clock, and half the tensor rate.  TF32 products
// also cut x_lo to 11 bits instead of rounding it: replayed in float64 over
// orders 150..900 the rounding of the operands alone puts P off by 2.7e-7 (rms,
// N(0, 1) entries) with TF32 pairs and 2.2e-7 with float16 pairs; measured, with
// the float32 accumulation in tensor memory (half as many steps as for TF32, and
// the small terms by themselves), 2.3e-5 -> 1.6e-5 relative at order 1500, 1.5e-5 ->
// 1.0e-5 at 900 and 4.9e-6 -> 3.0e-6 at 300.  Blocks of order 129..1500 (four of
// them): 3.93 -> 3.27 ms a projection.
#pragma once

#include <cuda.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

namespace cdsdp_large {

constexpr int kTile = 128;         // rows of an output tile, one CTA each
// Columns of an output tile: 128, 64 or 32, chosen block by block (choose_tiles).
// A K step of 64 costs 0.50 us at 128 columns and 0.42 us at 64 and 32 (shared
// memory: the operands are written once and read by two MMAs a 16-wide step), a
// launch with its first loads and its epilogue 11, 8.7 and 8.0 us: narrow tiles
// are less efficient but finish sooner while SMs would stand idle otherwise.
// (A_hi B_hi, A_hi B_lo and A_lo B_hi as three MMAs read A_hi twice: 0.65, 0.64
// and 0.61 us a K step.)  Every entry is the same sum in the same order at each
// width.
constexpr int kWidths = 3;
__host__ __device__ constexpr int width_of(int w) { return kTile >> w; }
constexpr int kChunk = 64;         // K halves per stage: one 128-byte swizzle row
constexpr int kTileBytes = kTile * kChunk * 2;       // 16 KB per operand tile of 128 rows
__host__ __device__ constexpr int stage_bytes(int cols) { return 2 * kTileBytes + 2 * cols * kChunk * 2; }  // A_hi, A_lo, B_hi, B_lo
// Stages of the operand ring: about 192 KB in flight at every width.
__host__ __device__ constexpr int stages(int cols) { return cols == 128 ? 3 : (cols == 64 ? 4 : 5); }
constexpr int kRingBytes = 5 * stage_bytes(32);      // the largest of the three rings
constexpr int kGemmSmem = kRingBytes + 1024 + 256;
static_assert(kRingBytes >= 3 * stage_bytes(128) && kRingBytes >= 4 * stage_bytes(64), "ring");
constexpr int kGemmThreads = 256;  // producer, MMA issuer; all warps read the accumulator

// Phase-1 polynomial and the iteration counts.
constexpr float kPa = 3.30f, kPb = -3.66f, kPc = 1.36f;
constexpr int kPhase1 = 16, kPhase2 = 5;

// One output tile of block `blk`: rows 128 ti .., columns width_of(w) tj ..; it
// reaches into the lower triangle.
struct Tile { int blk, ti, tj, w; };

// Dense layout of one block in every buffer: float offset and padded order.
struct Block { long long off; int S, s; };

// The (hi, lo) buffers of the iteration.  X_0 keeps its own: the last product
// takes it in the place of W.  P (float32) overlays the pair of X^2.
enum { BUF_X0 = 0, BUF_XA = 1, BUF_XB = 2, BUF_X2 = 3, BUF_B = 4, NBUF = 5 };

// 2^12 x as a (hi, lo) pair of float16.
constexpr float kPairScale = 4096.f, kLoScale = 2048.f;
__device__ __forceinline__ void pair_split(float x, __half& hi, __half& lo) {
    const float y = x * kPairScale;
    hi = __float2half_rn(y);
    lo = __float2half_rn((y - __half2float(hi)) * kLoScale);
}
__device__ __forceinline__ float pair_value(__half hi, __half lo) {
    return (__half2float(hi) + __half2float(lo) * (1.f / kLoScale)) * (1.f / kPairScale);
}

// Epilogue of one product over the lower tiles: D = alpha A B + beta C, all
// (hi, lo) pairs; or, with P set, P = (W + |W|_F A B) / 2 in float32.
struct GemmArgs {
    const CUtensorMap* maps[kWidths];  // per box height width_of(w): [buffer][hi, lo][block]
    int a, b, c, nb;                   // operands' buffers (c < 0: no C), number of blocks
    __half* D_hi; __half* D_lo;
    const float* W; float* P;
    const double* scale;                        // |W|_F per block
    const Block* blocks;
    const Tile* tiles;
    int ntiles;
    float alpha, beta;
    int* err;                                   // set on a timed-out wait (kernel returns early)
};

// (a, b), a >= b, of packed (lower, column-major) element f of an s x s block:
// the column from an exact integer radicand and a float32 root (a float64 root
// costs some forty operations of the slow float64 pipe), then exact.
__device__ __forceinline__ void packed_rc(long long f, int s, int& a, int& b) {
    const long long t = 2LL * s + 1;
    int bb = (int)(((float)t - sqrtf((float)(t * t - 8 * f))) * 0.5f);
    bb = max(0, min(bb, s - 1));
    while (bb > 0 && (long long)bb * (2 * s - bb + 1) / 2 > f) --bb;
    while (bb + 1 < s && (long long)(bb + 1) * (2 * s - bb) / 2 <= f) ++bb;
    b = bb;
    a = bb + (int)(f - (long long)bb * (2 * s - bb + 1) / 2);
}

}  // namespace cdsdp_large

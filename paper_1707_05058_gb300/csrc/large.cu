// Large-order PSD projection (order 129 and above) by the Newton-Schulz sign
// iteration on the tensor cores (see large.cuh for the method), and the C ABI
// entry point that projects a batch of packed blocks this way.
//
// Product kernel (one CTA of 256 threads per output tile of 128 rows and 128,
// 64 or 32 columns):
//  * thread 0 of warp 0 streams 64-half wide tiles of A_hi, A_lo, B_hi, B_lo
//    into a shared-memory ring of 3 to 5 stages with TMA (cp.async.bulk.tensor, 128-byte
//    swizzle), one mbarrier per stage with the transaction byte count, and after
//    them the tile of C as one more stage;
//  * thread 0 of warp 1 issues tcgen05.mma kind::f16 (M = 128, K = 16):
//    two a K step, A_hi [B_hi; B_lo] into two float32 accumulators in tensor
//    memory (hi hi; hi lo) and A_lo B_hi into the second, and frees a stage with tcgen05.commit on that stage's "empty" mbarrier;
//  * the warps read the accumulator back (tcgen05.ld 32x32b, one row per
//    thread, the columns split between the two groups of four warps), apply
//    D = alpha acc + beta C, split D into its (hi, lo) pair and lay the tile and
//    its mirror (the products are symmetric) out in the free stages, from which
//    they go to global memory in whole lines.  Stored from the accumulator's
//    layout instead (16 bytes a lane and row, 2 bytes a lane and column, and C
//    read likewise) the epilogue took 26 of 48 us a product at order 1500, 15 of
//    32 us at order 903 and 11 of 22 us at order 300.
// Every wait is bounded (about a second of clock cycles): on a timeout the
// kernel records an error code, lets its in-flight copies land (bounded
// again), frees its tensor memory and returns; the host reports
// CDSDP_ERR_TIMEOUT.
#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <functional>
#include <map>
#include <mutex>
#include <vector>

#include "cdsdp_internal.h"
#include "large.cuh"
#include "large_launch.h"

namespace cdsdp_large {
namespace {

constexpr int kSMs = 152;
constexpr long long kSpinCycles = 2000000000LL;  // ~1 s at 2 GHz

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ bool mbar_try(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}

// Bounded wait for the phase of `parity` to complete; false on timeout.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity) {
    const long long t0 = clock64();
    while (!mbar_try(bar, parity))
        if (clock64() - t0 > kSpinCycles) return false;
    return true;
}

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}

__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}

__device__ __forceinline__ void tma_load_2d(uint32_t dst, const void* tmap, int x, int y, uint32_t bar) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
        ::"r"(dst), "l"(tmap), "r"(x), "r"(y), "r"(bar)
        : "memory");
}

// Shared-memory matrix descriptor of a K-major operand tile written by TMA with
// the 128-byte swizzle: rows of 128 bytes, 8-row groups 1024 bytes apart.
__device__ __forceinline__ uint64_t sdesc(uint32_t saddr) {
    uint64_t d = 0;
    d |= (uint64_t)((saddr >> 4) & 0x3FFFu);
    // leading byte offset 0: one swizzle atom spans the whole K extent of a tile
    d |= (uint64_t)(1024u >> 4) << 32;   // stride byte offset: next 8-row group
    d |= (uint64_t)1u << 46;             // descriptor version of the tcgen05 family
    d |= (uint64_t)2u << 61;             // 128-byte swizzle
    return d;
}

// Instruction descriptor: D float32, A and B float16, both K-major, M = 128, N = cols.
__host__ __device__ constexpr uint32_t idesc(int cols) {
    return (1u << 4) | ((uint32_t)(cols >> 3) << 17) | ((uint32_t)(kTile >> 4) << 24);
}

__device__ __forceinline__ void mma_f16(uint32_t tmem, uint64_t a, uint64_t b, uint32_t desc, uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
        ::"r"(tmem), "l"(a), "l"(b), "r"(desc), "r"(accumulate)
        : "memory");
}

__device__ __forceinline__ void mma_commit(uint32_t bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}

__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t (&v)[32]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
        "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
        : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
          "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15]),
          "=r"(v[16]), "=r"(v[17]), "=r"(v[18]), "=r"(v[19]), "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]),
          "=r"(v[24]), "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]), "=r"(v[30]), "=r"(v[31])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

__device__ __forceinline__ void prefetch_map(const CUtensorMap* m) {
    asm volatile("prefetch.tensormap [%0];" ::"l"(m) : "memory");
}

// 32 columns of this thread's row of A B, from the two accumulators (of operands
// scaled by kPairScale each).
__device__ __forceinline__ void load_acc(uint32_t taddr, int N, float (&v)[32]) {
    uint32_t a[32], b[32];
    tmem_ld32(taddr, a);
    tmem_ld32(taddr + (uint32_t)N, b);
    constexpr float s = 1.f / (kPairScale * kPairScale);
#pragma unroll
    for (int j = 0; j < 32; ++j) v[j] = s * fmaf(1.f / kLoScale, __uint_as_float(b[j]), __uint_as_float(a[j]));
}

__device__ __forceinline__ uint4 pack8(const __half* h) {
    uint32_t w[4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
        w[i] = (uint32_t)__half_as_ushort(h[2 * i]) | ((uint32_t)__half_as_ushort(h[2 * i + 1]) << 16);
    return make_uint4(w[0], w[1], w[2], w[3]);
}

__global__ void __launch_bounds__(kGemmThreads, 1) k_f16x3_sym(const __grid_constant__ GemmArgs g) {
    const Tile t = g.tiles[blockIdx.x];
    const int N = width_of(t.w);
    const int kStages = stages(N), kStageBytes = stage_bytes(N), kColBytes = N * kChunk * 2;
    extern __shared__ unsigned char smem_raw[];
    unsigned char* smem = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                                           ~static_cast<uintptr_t>(1023));
    uint64_t* bars = reinterpret_cast<uint64_t*>(smem + kRingBytes);  // full[kStages], empty[kStages], done
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2 * kStages + 1);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
    int* issued_slot = reinterpret_cast<int*>(tmem_slot + 2);

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const Block B = g.blocks[t.blk];
    const int nk = B.S / kChunk;
    const CUtensorMap* mAh = g.maps[0] + 2 * g.a * g.nb + t.blk;
    const CUtensorMap* mAl = mAh + g.nb;
    const CUtensorMap* mBh = g.maps[t.w] + 2 * g.b * g.nb + t.blk;
    const CUtensorMap* mBl = mBh + g.nb;
    const bool has_c = g.c >= 0;
    const CUtensorMap* mCh = g.maps[t.w] + 2 * max(g.c, 0) * g.nb + t.blk;
    const CUtensorMap* mCl = mCh + g.nb;
    const uint32_t full0 = smem_u32(bars), empty0 = smem_u32(bars + kStages), done = smem_u32(bars + 2 * kStages);

    if (tid == 0) {
        for (int s = 0; s < kStages; ++s) {
            mbar_init(full0 + 8 * s, 1);
            mbar_init(empty0 + 8 * s, 1);
        }
        mbar_init(done, 1);
        *abort_flag = 0;
        *issued_slot = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (tid == 32) {  // the descriptors come from global memory, once per SM and launch
        prefetch_map(mAh);
        prefetch_map(mAl);
        prefetch_map(mBh);
        prefetch_map(mBl);
        if (has_c) {
            prefetch_map(mCh);
            prefetch_map(mCl);
        }
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                     "r"(2 * kTile)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = *tmem_slot;
    // Launched while the previous product still ran (launch_gemm): let the next
    // one be launched, and wait for the previous one's results.
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");

    if (warp == 0 && lane == 0) {  // TMA producer
        int issued = 0;
        uint32_t lap = 0;  // kc / kStages
        for (int kc = 0, s = 0; kc < nk + (has_c ? 1 : 0); ++kc, s = s + 1 == kStages ? (++lap, 0) : s + 1) {
            if (kc >= kStages && !mbar_wait(empty0 + 8 * s, (lap - 1) & 1)) {
                *abort_flag = 1;
                atomicExch(g.err, 1);
                break;
            }
            if (*abort_flag) break;
            const uint32_t base = smem_u32(smem + s * kStageBytes);
            if (kc == nk) {  // C by its symmetric entries (tj, ti): two boxes of 64 columns each, hi then lo
                mbar_expect_tx(full0 + 8 * s, 4 * kColBytes);
                for (int q = 0; q < 2; ++q) {
                    tma_load_2d(base + q * kColBytes, mCh, t.ti * kTile + q * kChunk, t.tj * N, full0 + 8 * s);
                    tma_load_2d(base + (2 + q) * kColBytes, mCl, t.ti * kTile + q * kChunk, t.tj * N, full0 + 8 * s);
                }
                ++issued;
                break;
            }
            mbar_expect_tx(full0 + 8 * s, kStageBytes);
            const int x = kc * kChunk;
            tma_load_2d(base, mAh, x, t.ti * kTile, full0 + 8 * s);
            tma_load_2d(base + kTileBytes, mAl, x, t.ti * kTile, full0 + 8 * s);
            tma_load_2d(base + 2 * kTileBytes, mBh, x, t.tj * N, full0 + 8 * s);
            tma_load_2d(base + 2 * kTileBytes + kColBytes, mBl, x, t.tj * N, full0 + 8 * s);
            ++issued;
        }
        *issued_slot = issued;
    } else if (warp == 1 && lane == 0) {  // MMA issuer
        const uint32_t desc = idesc(N), desc2 = idesc(2 * N);
        uint32_t lap = 0;
        for (int kc = 0, s = 0; kc < nk; ++kc, s = s + 1 == kStages ? (++lap, 0) : s + 1) {
            if (!mbar_wait(full0 + 8 * s, lap & 1)) {
                *abort_flag = 1;
                atomicExch(g.err, 2);
                break;
            }
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const uint32_t base = smem_u32(smem + s * kStageBytes);
#pragma unroll
            for (int k = 0; k < kChunk / 16; ++k) {
                const uint64_t ah = sdesc(base + 32 * k), al = sdesc(base + kTileBytes + 32 * k);
                const uint64_t bh = sdesc(base + 2 * kTileBytes + 32 * k);
                // B_lo lies behind B_hi, and so do the accumulators: A_hi [B_hi; B_lo]
                // is one product of 2 N columns, which reads A_hi once
                mma_f16(tmem, ah, bh, desc2, (kc | k) != 0 ? 1u : 0u);
                mma_f16(tmem + N, al, bh, desc, 1u);
            }
            mma_commit(empty0 + 8 * s);
        }
        mma_commit(done);  // completes once every MMA issued above has finished
    }
    __syncwarp();

    // epilogue: thread (warp w, lane l) owns row 32 (w mod 4) + l of the tile
    const int c_slot = nk % kStages;
    bool ok = mbar_wait(done, 0);
    if (ok && has_c && !*abort_flag) ok = mbar_wait(full0 + 8 * c_slot, (nk / kStages) & 1);
    if (!ok) atomicExch(g.err, 3);
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    if (__syncthreads_and(ok && !*abort_flag)) {
        // Every stored matrix is kept exactly symmetric: an off-diagonal tile is
        // stored with its mirror, a diagonal tile only from its lower triangle
        // (mirrored).  The products are symmetric only up to rounding, and the
        // B operand enters transposed, so an antisymmetric remainder left in an
        // iterate would be amplified by the sign iteration near eigenvalue 0.
        const int S = B.S;
        const int wr = warp & 3, half = warp >> 2;
        const int r = 32 * wr + lane;
        // A tile that reaches the diagonal holds columns c0 .. c0 + N - 1 of its
        // 128 x 128 diagonal block: rows above c0 belong to the mirrors of other
        // tiles, rows c0 .. c0 + N - 1 are a symmetric square, the rest lies below.
        const int c0 = t.tj * N - t.ti * kTile;
        const bool diag = c0 >= 0;
        const uint32_t row = tmem + ((uint32_t)(32 * wr) << 16);
        if (g.P) {  // P = (W + |W|_F A B) / 2; |W|_F in two floats, so that its rounding does not scale W sign(W)
            const long long gr = (long long)t.ti * kTile + r;
            const double nrm = g.scale[t.blk];
            const float up = nrm > 1e30 ? 16777216.f : 1.f;  // |W|_F itself may pass the float32 range
            const float nh = (float)(nrm / up), nl = (float)(nrm / up - (double)nh);
            const float* Wk = g.W + B.off;
            float* P = g.P + B.off;
#pragma unroll 1
            for (int cc = half; cc < N / 32; cc += 2) {
                float v[32];
                load_acc(row + (uint32_t)(32 * cc), N, v);
                const long long gc0 = (long long)t.tj * N + 32 * cc;
#pragma unroll
                for (int j = 0; j < 32; ++j) {
                    // W is symmetric: read its entry (gc, gr), consecutive over the warp's rows
                    const float w = Wk[(gc0 + j) * S + gr];
                    v[j] = 0.5f * fmaf(v[j] * up, nh, fmaf(v[j] * up, nl, w));
                }
#pragma unroll
                for (int j = 0; j < 32; ++j) {
                    if (diag && gc0 + j > gr) continue;  // upper triangle: written as the mirror of (gc, gr)
                    P[gr * S + gc0 + j] = v[j];
                    P[(gc0 + j) * S + gr] = v[j];
                }
            }
        } else {
            // tile (rows of N halves, 16-byte units permuted within a row so that
            // eight rows' units fall into different banks) and mirror (N rows of 128)
            unsigned char* tile = smem + ((c_slot + 1) % kStages) * kStageBytes;
            unsigned char* mirr = smem + ((c_slot + 2) % kStages) * kStageBytes;
            const int kOut = kTile * N * 2;  // bytes of one of hi, lo
            auto perm = [&](int rr) { return N >= 64 ? (rr & 7) : ((rr >> 1) & 3); };
            auto tile_at = [&](int rr, int col) { return rr * (2 * N) + ((((col >> 3) ^ perm(rr)) << 4) | ((col & 7) << 1)); };
            // C (gc, gr): row gc of box r / 64, its 16-byte units permuted by the TMA swizzle
            const unsigned char* cbase = smem + c_slot * kStageBytes + (r >> 6) * kColBytes + ((r & 7) << 1);
            const int cq = (r & 63) >> 3;
            const int lc = r - c0;  // own column within the diagonal square
            const bool square = diag && lc >= 0 && lc < N;
#pragma unroll 1
            for (int cc = half; cc < N / 32; cc += 2) {
                float v[32];
                load_acc(row + (uint32_t)(32 * cc), N, v);
                __half hi[32], lo[32];
#pragma unroll
                for (int j = 0; j < 32; ++j) {
                    float c = 0.f;
                    if (has_c) {
                        const unsigned char* pc = cbase + (32 * cc + j) * 128 + ((cq ^ (j & 7)) << 4);
                        c = pair_value(*reinterpret_cast<const __half*>(pc),
                                       *reinterpret_cast<const __half*>(pc + 2 * kColBytes));
                    }
                    pair_split(g.alpha * v[j] + g.beta * c, hi[j], lo[j]);
                }
                if (!square) {
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        const int at = tile_at(r, 32 * cc + 8 * q);
                        *reinterpret_cast<uint4*>(tile + at) = pack8(hi + 8 * q);
                        *reinterpret_cast<uint4*>(tile + kOut + at) = pack8(lo + 8 * q);
                    }
#pragma unroll
                    for (int j = 0; j < 32; ++j) {
                        const int at = (32 * cc + j) * (2 * kTile) + 2 * r;
                        *reinterpret_cast<__half*>(mirr + at) = hi[j];
                        *reinterpret_cast<__half*>(mirr + kOut + at) = lo[j];
                    }
                } else {
#pragma unroll
                    for (int j = 0; j < 32; ++j) {
                        const int col = 32 * cc + j;
                        if (col > lc) continue;
                        const int at = tile_at(r, col), am = tile_at(c0 + col, lc);
                        *reinterpret_cast<__half*>(tile + at) = hi[j];
                        *reinterpret_cast<__half*>(tile + kOut + at) = lo[j];
                        *reinterpret_cast<__half*>(tile + am) = hi[j];
                        *reinterpret_cast<__half*>(tile + kOut + am) = lo[j];
                    }
                }
            }
            __syncthreads();
            __half* Dh = g.D_hi + B.off;
            __half* Dl = g.D_lo + B.off;
            const int r0 = diag ? c0 : 0;
            const int lg = 4 - t.w;  // units of a row: N / 8 = 2^lg
            for (int i = tid; i < ((kTile - r0) << lg); i += kGemmThreads) {
                const int rr = r0 + (i >> lg), q = i & ((1 << lg) - 1);
                const int at = tile_at(rr, 8 * q);
                const long long to = ((long long)t.ti * kTile + rr) * S + (long long)t.tj * N + 8 * q;
                *reinterpret_cast<uint4*>(Dh + to) = *reinterpret_cast<const uint4*>(tile + at);
                *reinterpret_cast<uint4*>(Dl + to) = *reinterpret_cast<const uint4*>(tile + kOut + at);
            }
            const int m0 = diag ? c0 + N : 0, nv = (kTile - m0) / 8;
            for (int i = tid; i < N * nv; i += kGemmThreads) {
                const int gc = i / nv, q = m0 / 8 + i - gc * nv;
                const int at = gc * (2 * kTile) + 16 * q;
                const long long to = ((long long)t.tj * N + gc) * S + (long long)t.ti * kTile + 8 * q;
                *reinterpret_cast<uint4*>(Dh + to) = *reinterpret_cast<const uint4*>(mirr + at);
                *reinterpret_cast<uint4*>(Dl + to) = *reinterpret_cast<const uint4*>(mirr + kOut + at);
            }
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    // after an abort, let the copies already issued land before the CTA exits
    if (*abort_flag && warp == 0 && lane == 0) {
        const int issued = *issued_slot;  // the chunks, then C
        for (int kc = max(0, issued - kStages); kc < issued; ++kc)
            (void)mbar_wait(full0 + 8 * (kc % kStages), (kc / kStages) & 1);
    }
    __syncthreads();
    if (warp == 0) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(2 * kTile) : "memory");
    }
}

// ---- element-wise kernels ---------------------------------------------------

// Dense symmetric W of block k from its packed lower values (grid.y = block).
__global__ void k_dense_from_packed(const Block* __restrict__ blocks, const long long* __restrict__ poff,
                                    const float* __restrict__ Wp, float* W) {
    const int k = blockIdx.y;
    const Block B = blocks[k];
    const long long npk = (long long)B.s * (B.s + 1) / 2;
    for (long long f = blockIdx.x * (long long)blockDim.x + threadIdx.x; f < npk; f += (long long)gridDim.x * blockDim.x) {
        int a, b;
        packed_rc(f, B.s, a, b);
        const float w = Wp[poff[k] + f];
        W[B.off + (long long)a * B.S + b] = w;
        W[B.off + (long long)b * B.S + a] = w;
    }
}

// Partial sums of ||W||_F^2 over fixed chunks of each block's dense rows
// (deterministic: one partial per (block, chunk), summed in order below).
constexpr int kNormChunkRows = 8;  // 190 thread blocks at order 1500
__global__ void k_norm_partials(const Block* __restrict__ blocks, const int* __restrict__ chunk_off,
                                const float* __restrict__ W, double* partial) {
    const int k = blockIdx.y;
    const Block B = blocks[k];
    const int nchunk = chunk_off[k + 1] - chunk_off[k];
    if ((int)blockIdx.x >= nchunk) return;
    const long long r0 = (long long)blockIdx.x * kNormChunkRows;
    const long long e0 = B.off + r0 * B.S;
    const long long ne = (long long)min((long long)kNormChunkRows, B.S - r0) * B.S;
    double acc = 0.0;
    for (long long e = threadIdx.x; e < ne; e += blockDim.x) {
        const double w = (double)W[e0 + e];
        acc += w * w;
    }
    __shared__ double sh[32];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x == 0) {
        double s = 0.0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) s += sh[w];
        partial[chunk_off[k] + blockIdx.x] = s;
    }
}

// X_0 = W / ||W||_F as (hi, lo); scale[k] = ||W||_F as rounded for that (grid.y = block).
__global__ void k_scale_start(const Block* __restrict__ blocks, const int* __restrict__ chunk_off,
                              const double* __restrict__ partial, const float* __restrict__ W, __half* Xh, __half* Xl,
                              double* scale) {
    const int k = blockIdx.y;
    const Block B = blocks[k];
    // one warp adds the partial sums for its block (every thread did: 93 us of
    // float64 additions at order 1500)
    __shared__ float s_inv;
    if (threadIdx.x < 32) {
        double s2 = 0.0;
        for (int c = chunk_off[k] + threadIdx.x; c < chunk_off[k + 1]; c += 32) s2 += partial[c];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) s2 += __shfl_xor_sync(0xffffffffu, s2, o);
        if (threadIdx.x == 0) {
            const double nrm = sqrt(s2);
            s_inv = nrm > 0.0 ? (float)(1.0 / nrm) : 0.f;
            if (blockIdx.x == 0) scale[k] = s_inv > 0.f ? 1.0 / (double)s_inv : 0.0;  // what X_0 was divided by
        }
    }
    __syncthreads();
    const float inv = s_inv;
    const long long nq = (long long)B.S * B.S / 4;  // S is a multiple of 128
    const float4* W4 = reinterpret_cast<const float4*>(W + B.off);
    uint2* Xh4 = reinterpret_cast<uint2*>(Xh + B.off);
    uint2* Xl4 = reinterpret_cast<uint2*>(Xl + B.off);
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < nq; e += (long long)gridDim.x * blockDim.x) {
        const float4 w = W4[e];
        const float x[4] = {w.x * inv, w.y * inv, w.z * inv, w.w * inv};
        __half h[4], l[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) pair_split(x[i], h[i], l[i]);
        auto pack2 = [](const __half* p) {
            return (uint32_t)__half_as_ushort(p[0]) | ((uint32_t)__half_as_ushort(p[1]) << 16);
        };
        Xh4[e] = make_uint2(pack2(h), pack2(h + 2));
        Xl4[e] = make_uint2(pack2(l), pack2(l + 2));
    }
}

// Packed lower values of the dense P (grid.y = block).
__global__ void k_packed_from_dense(const Block* __restrict__ blocks, const long long* __restrict__ poff,
                                    const float* __restrict__ P, float* Xp) {
    const int k = blockIdx.y;
    const Block B = blocks[k];
    const long long npk = (long long)B.s * (B.s + 1) / 2;
    for (long long f = blockIdx.x * (long long)blockDim.x + threadIdx.x; f < npk; f += (long long)gridDim.x * blockDim.x) {
        int a, b;
        packed_rc(f, B.s, a, b);
        Xp[poff[k] + f] = P[B.off + (long long)a * B.S + b];
    }
}

// ---- host side ----------------------------------------------------------------

std::mutex g_encode_mutex;
PFN_cuTensorMapEncodeTiled_v12000 g_encode = nullptr;

bool get_encode() {
    std::lock_guard<std::mutex> lock(g_encode_mutex);
    if (g_encode) return true;
    void* fn = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &q) != cudaSuccess ||
        q != cudaDriverEntryPointSuccess || !fn) {
        cudaGetLastError();
        return false;
    }
    g_encode = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(fn);
    return true;
}

bool encode_map(CUtensorMap* m, const __half* base, int S, int rows) {
    const cuuint64_t dims[2] = {(cuuint64_t)S, (cuuint64_t)S};
    const cuuint64_t strides[1] = {(cuuint64_t)S * 2};
    const cuuint32_t box[2] = {(cuuint32_t)kChunk, (cuuint32_t)rows};
    const cuuint32_t estr[2] = {1, 1};
    return g_encode(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2, const_cast<__half*>(base), dims, strides, box, estr,
                    CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                    CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// Time an SM spends on a tile of width w and nk K steps, in us (fitted to single
// blocks of order 300..1500 at each width).
double tile_cost(int w, int nk) {
    constexpr double step[kWidths] = {0.50, 0.42, 0.42}, rest[kWidths] = {6.0, 3.7, 3.0};
    return rest[w] + step[w] * nk;
}

// Blocks of one padded order: their count and, with a width, their tiles.
struct Group { int S, count; };
long long tiles_of(const Group& g, int w) {
    const long long T = g.S / kTile;
    return (g.count * T * (T + 1) / 2) << w;
}

// Time until 152 SMs, each taking the longest tile left, are through; the groups
// before `cut` have tiles of width a, the others of width b.
double makespan(const std::vector<Group>& gs, int cut, int a, int b) {
    std::vector<std::pair<double, long long>> jobs;  // cost, count
    for (int i = 0; i < (int)gs.size(); ++i) {
        const int w = i < cut ? a : b;
        jobs.push_back({tile_cost(w, gs[i].S / kChunk), tiles_of(gs[i], w)});
    }
    std::stable_sort(jobs.begin(), jobs.end(), [](const auto& x, const auto& y) { return x.first > y.first; });
    std::map<double, long long> load;  // busy until -> SMs
    load[0.0] = kSMs;
    for (auto [cost, n] : jobs)
        while (n > 0) {
            const auto it = load.begin();
            const double at = it->first;
            const long long k = std::min(n, it->second);
            if (k == it->second) load.erase(it);
            else it->second -= k;
            load[at + cost] += k;
            n -= k;
        }
    return load.rbegin()->first;
}

// The output tiles of every block.  Batches whose 32-column (64-column) tiles
// fit the SMs at once take those; up to four waves of 128-column tiles, the
// widths are one for the larger blocks and one for the smaller ones, whichever
// pair and cut end first (four blocks of order 1500, 1052, 943 and 245: 162
// tiles of 128 columns took 34.3 us a product, with these 32.4); beyond that 128.
// The longest tiles come first, so that the last ones taken are short.
void choose_tiles(NsLayout& L) {
    std::vector<Group> gs;
    std::map<int, int, std::greater<int>> by_order;
    for (const Block& b : L.blocks) ++by_order[b.S];
    long long wide = 0;
    for (auto [S, n] : by_order) {
        gs.push_back({S, n});
        wide += tiles_of(gs.back(), 0);
    }
    int a = 0, b = 0, cut = 0;
    if (wide * 4 <= kSMs) {
        a = b = 2;
    } else if (wide * 2 <= kSMs) {
        a = b = 1;
    } else if (wide <= 4 * kSMs && gs.size() <= 16) {
        double best = 1e300;
        for (int w0 = 0; w0 < kWidths; ++w0)
            for (int w1 = w0; w1 < kWidths; ++w1)
                for (int c = w0 == w1 ? (int)gs.size() : 1; c <= (int)gs.size(); ++c) {
                    const double t = makespan(gs, c, w0, w1);
                    if (t < best - 1e-9) { best = t; a = w0; b = w1; cut = c; }
                }
    }
    const int small = cut < (int)gs.size() && !gs.empty() ? gs[cut].S : 0;  // orders up to it: width b
    for (int k = 0; k < L.nb; ++k) {
        const int w = L.blocks[k].S > small ? a : b;
        L.widths[w] = true;
        for (int i = 0; i < L.blocks[k].S / kTile; ++i)
            for (int j = 0; j * width_of(w) < (i + 1) * kTile; ++j) L.tiles.push_back(Tile{k, i, j, w});
    }
    std::stable_sort(L.tiles.begin(), L.tiles.end(), [&](const Tile& x, const Tile& y) {
        return tile_cost(x.w, L.blocks[x.blk].S / kChunk) > tile_cost(y.w, L.blocks[y.blk].S / kChunk);
    });
}

inline size_t up256(size_t x) { return (x + 255) & ~size_t(255); }

}  // namespace

// ---- layout of the iteration's device memory ------------------------------------

NsLayout ns_layout(const std::vector<int>& sizes) {
    NsLayout L;
    L.nb = (int)sizes.size();
    long long off = 0;
    int chunks = 0;
    L.chunk_off.push_back(0);
    for (int s : sizes) {
        Block b;
        b.s = s;
        b.S = (s + kTile - 1) / kTile * kTile;
        b.off = off;
        off += (long long)b.S * b.S;
        L.blocks.push_back(b);
        chunks += (b.S + kNormChunkRows - 1) / kNormChunkRows;
        L.chunk_off.push_back(chunks);
        L.max_S = std::max(L.max_S, b.S);
        const int nu = (int)(((long long)s * (s + 1) / 2 + kUpdChunk - 1) / kUpdChunk);
        if (L.upd_off.empty()) L.upd_off.push_back(0);
        L.upd_off.push_back(L.upd_off.back() + nu);
        L.max_upd = std::max(L.max_upd, nu);
    }
    if (L.upd_off.empty()) L.upd_off.push_back(0);
    choose_tiles(L);
    L.elems = off;
    size_t o = 0;
    L.o_err = o; o = up256(o + 16);
    // operand A's boxes are 128 rows high, B's and C's as high as a tile is wide
    for (int w = 0; w < kWidths; ++w) {
        L.o_maps[w] = o;
        if (w == 0 || L.widths[w]) o = up256(o + sizeof(CUtensorMap) * 2 * NBUF * (size_t)std::max(1, L.nb));
    }
    L.o_tiles = o; o = up256(o + sizeof(Tile) * std::max<size_t>(1, L.tiles.size()));
    L.o_blocks = o; o = up256(o + sizeof(Block) * std::max(1, L.nb));
    L.o_chunk = o; o = up256(o + sizeof(int) * (L.nb + 1));
    L.o_partial = o; o = up256(o + sizeof(double) * std::max(1, chunks));
    L.o_scale = o; o = up256(o + sizeof(double) * std::max(1, L.nb));
    L.o_poff = o; o = up256(o + sizeof(long long) * std::max(1, L.nb));
    L.o_list = o; o = up256(o + sizeof(int) * std::max(1, L.nb));
    L.o_upd = o; o = up256(o + sizeof(int) * (L.nb + 1));
    L.o_updpart = o; o = up256(o + sizeof(double) * 8 * std::max(1, L.upd_off.back()));
    L.o_w = o; o = up256(o + (size_t)off * sizeof(float));
    // off is a multiple of 128 x 128: a pair's two buffers are adjacent
    for (int b = 0; b < 2 * NBUF; ++b) {
        L.o_buf[b] = o;
        o = up256(o + (size_t)off * sizeof(__half));
    }
    L.bytes = o;
    return L;
}

// Host image of the tables (tensor maps, tiles, blocks, chunk offsets, packed
// offsets) for device memory at `base`; false when the tensor-map encoder is
// unavailable or refuses a map.
bool ns_tables(const NsLayout& L, unsigned char* base, const std::vector<long long>& poff,
               const std::vector<int>& list, std::vector<unsigned char>& img) {
    if (!get_encode()) return false;
    img.assign(L.o_w, 0);
    for (int w = 0; w < kWidths; ++w) {
        if (w > 0 && !L.widths[w]) continue;
        CUtensorMap* maps = reinterpret_cast<CUtensorMap*>(img.data() + L.o_maps[w]);
        for (int buf = 0; buf < 2 * NBUF; ++buf)
            for (int k = 0; k < L.nb; ++k) {
                const __half* p = reinterpret_cast<const __half*>(base + L.o_buf[buf]) + L.blocks[k].off;
                if (!encode_map(&maps[buf * L.nb + k], p, L.blocks[k].S, width_of(w))) return false;
            }
    }
    std::memcpy(img.data() + L.o_tiles, L.tiles.data(), sizeof(Tile) * L.tiles.size());
    std::memcpy(img.data() + L.o_blocks, L.blocks.data(), sizeof(Block) * L.blocks.size());
    std::memcpy(img.data() + L.o_chunk, L.chunk_off.data(), sizeof(int) * L.chunk_off.size());
    std::memcpy(img.data() + L.o_poff, poff.data(), sizeof(long long) * poff.size());
    std::memcpy(img.data() + L.o_list, list.data(), sizeof(int) * list.size());
    std::memcpy(img.data() + L.o_upd, L.upd_off.data(), sizeof(int) * L.upd_off.size());
    return true;
}

namespace {

cudaError_t launch_gemm(const GemmArgs& g, cudaStream_t st) {
    static bool attr = false;
    if (!attr) {
        cudaError_t e = cudaFuncSetAttribute(k_f16x3_sym, cudaFuncAttributeMaxDynamicSharedMemorySize, kGemmSmem);
        if (e != cudaSuccess) return e;
        attr = true;
    }
    cudaLaunchAttribute at;
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(g.ntiles);
    cfg.blockDim = dim3(kGemmThreads);
    cfg.dynamicSmemBytes = kGemmSmem;
    cfg.stream = st;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, k_f16x3_sym, g);
}

// D = alpha A B + beta C on pairs; with d < 0 the last product, P = (W + |W|_F A B) / 2.
cudaError_t gemm(const NsLayout& L, unsigned char* base, int a, int bsrc, int c, int d, float alpha, float beta,
                 cudaStream_t st) {
    auto half_buf = [&](int i) { return reinterpret_cast<__half*>(base + L.o_buf[i]); };
    GemmArgs g;
    for (int w = 0; w < kWidths; ++w) g.maps[w] = reinterpret_cast<const CUtensorMap*>(base + L.o_maps[w]);
    g.a = a;
    g.b = bsrc;
    g.c = c;
    g.nb = L.nb;
    g.D_hi = d >= 0 ? half_buf(2 * d) : nullptr;
    g.D_lo = d >= 0 ? half_buf(2 * d + 1) : nullptr;
    g.W = reinterpret_cast<const float*>(base + L.o_w);
    g.P = d >= 0 ? nullptr : reinterpret_cast<float*>(base + L.o_p());
    g.scale = reinterpret_cast<const double*>(base + L.o_scale);
    g.blocks = reinterpret_cast<const Block*>(base + L.o_blocks);
    g.tiles = reinterpret_cast<const Tile*>(base + L.o_tiles);
    g.ntiles = (int)L.tiles.size();
    g.alpha = alpha;
    g.beta = beta;
    g.err = reinterpret_cast<int*>(base + L.o_err);
    return launch_gemm(g, st);
}

}  // namespace

// The sign iteration and P = (W + W X) / 2 on buffers already holding W and
// X_0.
cudaError_t ns_iterate(const NsLayout& L, unsigned char* base, cudaStream_t st) {
    cudaError_t e = cudaSuccess;
    int x = BUF_X0, xn = BUF_XA;
    auto next = [&] {
        x = xn;
        xn = x == BUF_XA ? BUF_XB : BUF_XA;
    };
    for (int i = 0; i < kPhase1 && e == cudaSuccess; ++i) {  // X <- a X + b X^3 + c X^5
        e = gemm(L, base, x, x, -1, BUF_X2, 1.f, 0.f, st);                          // X2 = X X
        if (e == cudaSuccess) e = gemm(L, base, BUF_X2, BUF_X2, BUF_X2, BUF_B, kPc, kPb, st);  // c X2 X2 + b X2
        if (e == cudaSuccess) e = gemm(L, base, x, BUF_B, x, xn, 1.f, kPa, st);     // X B + a X
        next();
    }
    for (int i = 0; i < kPhase2 && e == cudaSuccess; ++i) {  // X <- 1.5 X - 0.5 X^3
        e = gemm(L, base, x, x, -1, BUF_X2, 1.f, 0.f, st);
        if (e == cudaSuccess) e = gemm(L, base, x, BUF_X2, x, xn, -0.5f, 1.5f, st);
        next();
    }
    if (e == cudaSuccess) e = gemm(L, base, BUF_X0, x, -1, -1, 0.f, 0.f, st);  // P
    return e;
}

cudaError_t ns_scale_and_iterate(const NsLayout& L, unsigned char* base, cudaStream_t st) {
    const Block* blocks = reinterpret_cast<const Block*>(base + L.o_blocks);
    const int* chunk = reinterpret_cast<const int*>(base + L.o_chunk);
    const float* W = reinterpret_cast<const float*>(base + L.o_w);
    __half* Xh = reinterpret_cast<__half*>(base + L.o_buf[2 * BUF_X0]);
    __half* Xl = reinterpret_cast<__half*>(base + L.o_buf[2 * BUF_X0 + 1]);
    const int gx = std::min(1024, std::max(1, (int)(((long long)L.max_S * L.max_S / 2 + 255) / 256)));
    const int maxchunk = (L.max_S + kNormChunkRows - 1) / kNormChunkRows;
    k_norm_partials<<<dim3(maxchunk, L.nb), 256, 0, st>>>(blocks, chunk, W,
                                                         reinterpret_cast<double*>(base + L.o_partial));
    k_scale_start<<<dim3(gx, L.nb), 256, 0, st>>>(blocks, chunk, reinterpret_cast<const double*>(base + L.o_partial),
                                                  W, Xh, Xl, reinterpret_cast<double*>(base + L.o_scale));
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess) e = ns_iterate(L, base, st);
    return e;
}

cudaError_t ns_from_packed(const NsLayout& L, unsigned char* base, const float* Wp, cudaStream_t st) {
    const Block* blocks = reinterpret_cast<const Block*>(base + L.o_blocks);
    const long long* poff = reinterpret_cast<const long long*>(base + L.o_poff);
    float* W = reinterpret_cast<float*>(base + L.o_w);
    cudaError_t e = cudaMemsetAsync(W, 0, (size_t)L.elems * sizeof(float), st);
    if (e != cudaSuccess) return e;
    const int gx = std::min(1024, std::max(1, (int)(((long long)L.max_S * L.max_S / 2 + 255) / 256)));
    k_dense_from_packed<<<dim3(gx, L.nb), 256, 0, st>>>(blocks, poff, Wp, W);
    return cudaGetLastError();
}

cudaError_t ns_to_packed(const NsLayout& L, unsigned char* base, float* Xp, cudaStream_t st) {
    const int gx = std::min(1024, std::max(1, (int)(((long long)L.max_S * L.max_S / 2 + 255) / 256)));
    k_packed_from_dense<<<dim3(gx, L.nb), 256, 0, st>>>(reinterpret_cast<const Block*>(base + L.o_blocks),
                                                        reinterpret_cast<const long long*>(base + L.o_poff),
                                                        reinterpret_cast<const float*>(base + L.o_p()),
                                                        Xp);
    return cudaGetLastError();
}

}  // namespace cdsdp_large

using namespace cdsdp_large;

extern "C" {

int cdsdp_psd_project_large_bytes(int p, const int* h_size, size_t* bytes) {
    if (p < 1 || !h_size || !bytes) return CDSDP_ERR_ARG;
    std::vector<int> sizes(h_size, h_size + p);
    for (int s : sizes)
        if (s < 1 || s > kMaxLargeOrder) return CDSDP_ERR_ARG;
    *bytes = ns_layout(sizes).bytes;
    return CDSDP_SOLVED;
}

int cdsdp_psd_project_large(int p, const int* h_size, const long long* h_off, const float* d_W, float* d_X,
                            void* d_scratch, size_t scratch_bytes, void* stream) {
    if (p < 1 || !h_size || !h_off || !d_W || !d_X || !d_scratch) return CDSDP_ERR_ARG;
    if (reinterpret_cast<uintptr_t>(d_scratch) % 256) return CDSDP_ERR_ARG;
    std::vector<int> sizes(h_size, h_size + p);
    for (int s : sizes)
        if (s < 1 || s > kMaxLargeOrder) return CDSDP_ERR_ARG;
    for (int k = 0; k < p; ++k)
        if (h_off[k] < 0) return CDSDP_ERR_ARG;
    try {
        const NsLayout L = ns_layout(sizes);
        if (scratch_bytes < L.bytes) return CDSDP_ERR_NOMEM;
        unsigned char* base = static_cast<unsigned char*>(d_scratch);
        std::vector<long long> poff(h_off, h_off + p);
        std::vector<int> list(p);
        for (int k = 0; k < p; ++k) list[k] = k;
        std::vector<unsigned char> img;
        if (!ns_tables(L, base, poff, list, img)) return CDSDP_ERR_CUDA;
        cudaStream_t st = static_cast<cudaStream_t>(stream);
        if (cudaMemcpyAsync(base, img.data(), img.size(), cudaMemcpyHostToDevice, st) != cudaSuccess ||
            cudaStreamSynchronize(st) != cudaSuccess) {
            cudaGetLastError();
            return CDSDP_ERR_CUDA;
        }
        cudaError_t e = ns_from_packed(L, base, d_W, st);
        if (e == cudaSuccess) e = ns_scale_and_iterate(L, base, st);
        if (e == cudaSuccess) e = ns_to_packed(L, base, d_X, st);
        if (e != cudaSuccess) {
            cudaGetLastError();
            return CDSDP_ERR_CUDA;
        }
        int err = 0;
        if (cudaMemcpyAsync(&err, base + L.o_err, sizeof(int), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
            cudaStreamSynchronize(st) != cudaSuccess) {
            cudaGetLastError();
            return CDSDP_ERR_CUDA;
        }
        return err ? CDSDP_ERR_TIMEOUT : CDSDP_SOLVED;
    } catch (const std::exception&) {
        return CDSDP_ERR_NOMEM;
    }
}

}  // extern "C"

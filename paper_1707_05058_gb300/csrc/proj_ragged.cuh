// Standalone projection (cdsdp_psd_project) of a batch whose block orders
// differ: the orders are device data, so the choice of kernel per order that
// the solver makes on the host is made here by each thread block or warp.
//
// Orders <= 32 (k_project_ragged): a thread block takes a run of consecutive
// batch entries, sorts them by padded order (steps of 4) with warp ballots and
// lets its four warps draw work items, largest orders first: one block per
// warp above order 16, two at orders 9..16 and four up to 8 (BLJacobi's lane
// groups).  Before, every block of the batch ran at the padded order of the
// largest one, a whole warp each: 4096 blocks of orders 1..32 (log-uniform)
// took a pass of 412 us, 202 us now.  Bound: the rounds of the largest orders (a
// cold order-32 block runs six sweeps of 31 dependent rounds).
//
// Orders 33..64 (k_project_cta_ragged): one thread block per batch entry,
// solved at its own padded order by CTAJacobiReg (600 blocks of orders 33..64:
// a pass of 0.90 ms at padded order 64 throughout, 0.72 ms now).
#pragma once

#include "jacobi_cta.cuh"

namespace cdsdp_dev {

constexpr int kRaggedWarps = 4;

template <typename T, int SMAX>
__host__ __device__ constexpr size_t ragged_warp_bytes() {
    const size_t a = 4 * BLJacobi<T, 8, 8>::bytes, b = 2 * BLJacobi<T, 16, 16>::bytes;
    const size_t c = SMAX > 16 ? BLJacobi<T, 32>::bytes : 0;
    return a > b ? (a > c ? a : c) : (b > c ? b : c);
}

// Up to 32 / LW blocks, one per group of LW lanes: group g takes entry ks[g].
template <typename T, int S>
__device__ __noinline__ void project_item(int smem_at, const int* ks, int count, const int* __restrict__ off_arr,
                                          const int* __restrict__ size_arr, const T* W, T* X, double tolrel,
                                          int max_sweeps) {
    constexpr int LW = proj_lanes(S);
    using J = BLJacobi<T, S, LW>;
    extern __shared__ __align__(16) unsigned char smem[];
    const int lane = (threadIdx.x & 31) % LW, grp = (threadIdx.x & 31) / LW;
    J jac;
    jac.bind(smem + smem_at + grp * J::bytes, lane);
    const bool active = grp < count;
    const int k = ks[active ? grp : 0];
    const int off = off_arr[k], s = active ? size_arr[k] : 0, npk = s * (s + 1) / 2;
    T w[J::MAXE];
#pragma unroll
    for (int e = 0; e < J::MAXE; ++e) w[e] = lane + LW * e < npk ? W[off + lane + LW * e] : T(0);
    jac.clear(lane, s);
    T nrm = T(0);
#pragma unroll
    for (int e = 0; e < J::MAXE; ++e) {
        const int f = lane + LW * e;
        if (f < npk) {
            const int ab = packed_ab(f, s), a = ab >> 8, b = ab & 255;
            jac.put(a, b, w[e]);
            nrm += (a == b ? T(1) : T(2)) * w[e] * w[e];
        }
    }
    nrm = group_sum(nrm, LW);
    __syncwarp();
    jac.run(tolrel, nrm, max_sweeps, lane, float(kThetaSolve * tolrel), false, active);
    jac.project(lane);
    for (int f = lane; f < npk; f += LW) {
        const int ab = packed_ab(f, s), a = ab >> 8, b = ab & 255;
        X[off + f] = jac.projected(a, b);
    }
    __syncwarp();
}

// `run` consecutive entries (at most 32) per thread block; orders outside
// 1..limit are left alone.
template <typename T, int SMAX>
__global__ void __launch_bounds__(32 * kRaggedWarps) k_project_ragged(int p, int run, int limit,
                                                                      const int* __restrict__ off_arr,
                                                                      const int* __restrict__ size_arr, const T* W,
                                                                      T* X, double tolrel, int max_sweeps) {
    __shared__ int entry[32], item_cls[32], item_pos[32], item_n[32];
    __shared__ int n_items, next;
    batch_begin();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (warp == 0) {
        const int k = blockIdx.x * run + lane;
        const int s = lane < run && k < p ? size_arr[k] : 0;
        // padded order 4 cls; in double order 2 by itself (0), whose rotation is exact (jacobi.cuh)
        const int cls = s < 1 || s > limit ? -1 : (sizeof(T) == 8 && s <= 2 ? 0 : (s + 3) / 4);
        int pos0 = 0, it0 = 0;
#pragma unroll
        for (int c = SMAX / 4; c >= (sizeof(T) == 8 ? 0 : 1); --c) {
            const unsigned mask = __ballot_sync(0xffffffffu, cls == c);
            const int n = __popc(mask), G = 32 / proj_lanes(c ? 4 * c : 2);
            if (cls == c) {
                const int r = __popc(mask & ((1u << lane) - 1u));
                entry[pos0 + r] = k;
                if (r % G == 0) {
                    const int it = it0 + r / G;
                    item_cls[it] = c;
                    item_pos[it] = pos0 + r;
                    item_n[it] = min(G, n - r);
                }
            }
            pos0 += n;
            it0 += (n + G - 1) / G;
        }
        if (lane == 0) { n_items = it0; next = 0; }
    }
    __syncthreads();
    const int ws = warp * (int)ragged_warp_bytes<T, SMAX>();
    while (true) {
        int it = 0;
        if (lane == 0) it = atomicAdd(&next, 1);
        it = __shfl_sync(0xffffffffu, it, 0);
        if (it >= n_items) break;
        const int* ks = entry + item_pos[it];
        const int n = item_n[it];
#define CDSDP_ITEM(C) \
    case C: project_item<T, 4 * C>(ws, ks, n, off_arr, size_arr, W, X, tolrel, max_sweeps); break;
        if constexpr (SMAX > 16) {
            switch (item_cls[it]) {
                CDSDP_ITEM(5) CDSDP_ITEM(6) CDSDP_ITEM(7) CDSDP_ITEM(8)
            }
        }
        switch (item_cls[it]) {
            case 0: if constexpr (sizeof(T) == 8) project_item<T, 2>(ws, ks, n, off_arr, size_arr, W, X, tolrel, max_sweeps); break;
            CDSDP_ITEM(1) CDSDP_ITEM(2) CDSDP_ITEM(3) CDSDP_ITEM(4)
        }
#undef CDSDP_ITEM
    }
    batch_end();
}

template <typename T, int SMAX>
cudaError_t launch_ragged(int p, int limit, const int* off, const int* size, const void* W, void* X, double tolrel,
                          int max_sweeps, bool overlap, cudaStream_t st) {
    // entries per thread block: two thread blocks per SM where the batch
    // reaches that far (fewer leaves SMs idle, more leaves nothing to sort)
    const int run = std::max(1, std::min(32, (p + 2 * 152 - 1) / (2 * 152)));
    const size_t smem = kRaggedWarps * ragged_warp_bytes<T, SMAX>();
    cudaError_t e = cudaFuncSetAttribute(k_project_ragged<T, SMAX>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)smem);
    if (e != cudaSuccess) return e;
    return launch_beside(overlap, k_project_ragged<T, SMAX>, (p + run - 1) / run, 32 * kRaggedWarps, smem, st, p, run,
                         limit, off, size, (const T*)W, (T*)X, tolrel, max_sweeps);
}

// ---- orders 33..64 -------------------------------------------------------------

template <int S>
__device__ __noinline__ void project_block(double* shr, int s, const float* W, float* X,
                                           double tolrel, int max_sweeps) {
    using J = CTAJacobiReg<S>;
    extern __shared__ __align__(16) unsigned char smem[];
    J jac;
    jac.bind(smem);
    const int tid = threadIdx.x, npk = s * (s + 1) / 2;
    jac.clear();
    double nrm[1] = {0.0};
    for (int f = tid; f < npk; f += blockDim.x) {
        const int ab = packed_ab(f, s), a = ab >> 8, b = ab & 255;
        const float w = W[f];
        jac.put(a, b, w);
        nrm[0] += (a == b ? 1.0 : 2.0) * double(w) * double(w);
    }
    block_sum<1>(nrm, shr);
    if (tid == 0) shr[0] = nrm[0];
    __syncthreads();
    const float fro = float(sqrt(shr[0]));
    __syncthreads();
    jac.identity_basis();
    typename J::Plan plan;
    J::plan(plan);
    jac.run(float(tolrel) * fro, max_sweeps, fro > 0.0f ? 1.0f / fro : 0.0f, float(kThetaSolve * tolrel), plan);
    jac.project(plan);
    for (int f = tid; f < npk; f += blockDim.x) {
        const int ab = packed_ab(f, s);
        X[f] = jac.rebuild(ab >> 8, ab & 255, s);
    }
    __syncthreads();
}

constexpr int kRaggedCtaThreads = CTAJacobiReg<64>::NT;

__global__ void __launch_bounds__(kRaggedCtaThreads, 3) k_project_cta_ragged(int p, int limit,
                                                                             const int* __restrict__ off_arr,
                                                                             const int* __restrict__ size_arr,
                                                                             const float* W, float* X, double tolrel,
                                                                             int max_sweeps) {
    __shared__ double shr[32];
    batch_begin();
    for (int k = blockIdx.x; k < p; k += gridDim.x) {
        const int s = size_arr[k];
        if (s <= kMaxWarpOrder || s > limit) continue;  // block-uniform
        const float* w = W + off_arr[k];
        float* x = X + off_arr[k];
        switch ((s + 3) / 4) {
            case 9: project_block<36>(shr, s, w, x, tolrel, max_sweeps); break;
            case 10: project_block<40>(shr, s, w, x, tolrel, max_sweeps); break;
            case 11: project_block<44>(shr, s, w, x, tolrel, max_sweeps); break;
            case 12: project_block<48>(shr, s, w, x, tolrel, max_sweeps); break;
            case 13: project_block<52>(shr, s, w, x, tolrel, max_sweeps); break;
            case 14: project_block<56>(shr, s, w, x, tolrel, max_sweeps); break;
            case 15: project_block<60>(shr, s, w, x, tolrel, max_sweeps); break;
            case 16: project_block<64>(shr, s, w, x, tolrel, max_sweeps); break;
        }
    }
    batch_end();
}

}  // namespace cdsdp_dev

// Maximum-determinant positive definite completion (Section 7.1.1) of a
// partial matrix X given on the extended chordal pattern E*.
//
// The completion W is the unique positive definite matrix with W = X on E*
// and (W^-1)_ij = 0 off E* (Grone, Johnson, Sa and Wolkowicz 1984); on a
// chordal pattern it follows from a perfect elimination order v_1..v_n
// (Vandenberghe and Andersen, Chapter 10.2).  With N_k the neighbours of v_k
// eliminated after it (a clique),
//   t_k = X[N_k, N_k]^-1 X[N_k, v_k],   s_k = X[v_k, v_k] - X[v_k, N_k] t_k,
// all s_k > 0 exactly when every clique block of X is positive definite,
// log det W = sum_k log s_k, and, for k = n-1 down to 1, the free entries of
// column v_k are W[j, v_k] = W[j, N_k] t_k for every later j outside N_k.
//
// GPU design.
//   k_cmp_factor   one warp per vertex: gathers X[N, N] and X[N, v] from the
//                  pattern (binary search in the column-major lower pattern),
//                  Cholesky in shared memory, t_k and s_k.  Every vertex is
//                  independent, so this is one launch over all n vertices.
//   k_cmp_logdet   one thread block per component: sum of log s_k in a fixed
//                  order.
//   k_cmp_scatter  the given entries into the dense blocks.
//   k_cmp_rows     patterns with a full profile (below): every row of the
//                  completion is a chain of its own, so one launch runs all of
//                  them side by side.
//   k_cmp_step     other patterns: one launch per step of the recurrence (the
//                  launches are captured once into a CUDA graph and replayed);
//                  within a step each thread owns one later vertex j of one
//                  component (all components advance together, aligned at
//                  their last vertex), reads rows N_k of the block at column j
//                  (coalesced) and writes W[v_k, j] and W[j, v_k].
//
// Full profile: for every vertex u, all vertices eliminated between the first
// one that has u among its later neighbours and u itself have u among theirs
// (the Cholesky factor has no zeros inside its row envelope; bands and
// block-arrows in their own order are like that).  Then in
// W[j, v_k] = W[j, N_k] t_k an element u of N_k eliminated after j has the
// given entry (u, j), and one eliminated before j was computed by the same
// row j: row j needs nothing from other rows.  Without that property rows
// exchange computed entries, and the steps have to stay in order.
// The dense output holds one row-major n_c x n_c block per component
// (independent components complete independently; entries between them are
// zero), vertices of a block in ascending order.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <string>
#include <utility>
#include <vector>

#include "cdsdp_internal.h"

namespace cdsdp_impl {
namespace {

constexpr size_t kCmpAlign = 256;
constexpr int kStepThreads = 256;
constexpr int kRowWarps = 2, kRowsPerWarp = 8;  // k_cmp_rows: 8 rows a warp, 4 lanes a row
constexpr int kRowThreads = 32 * (kRowWarps + 1);  // and one warp that stages the recurrence coefficients
constexpr int kRowRing = 64;    // latest entries of a row kept in shared memory
constexpr int kRowFar = 8;      // prefetched older entries per lane
constexpr int kRowTerms = 1024; // coefficients per stage (at least one step)
constexpr size_t kMaxWarpSmem = 200 * 1024;  // largest shared block per warp of the factor kernel

inline size_t align_up(size_t x) { return (x + kCmpAlign - 1) / kCmpAlign * kCmpAlign; }

// Scratch layout (byte offsets, all 256-aligned).  The index section [0, idx_end)
// is copied from the host image; [idx_end, base_total) is written by the kernels.
// The tables of k_cmp_rows follow, from row_begin: they are built and copied
// only where it runs, for a dense result on a full profile, and a scratch that
// ends before them is served by k_cmp_step.
struct CmpLayout {
    size_t lt_ptr, lt_idx, colptr, prow, pcol, comp, loc, posl, peo_cat, peo_off, woff, idx_end;
    size_t T, schur, logdet, flag, base_total;
    size_t row_begin, lt_pos, lt_loc, first, rowblk, total;
    int smax = 0;
    int nrowblk = 0;  // blocks of k_cmp_rows
};

// Vertices of each component, ascending (local index) and in elimination order,
// and the offsets of the components' dense blocks.
struct CmpOrder {
    std::vector<int> cnt, loc, posl, peo_cat, peo_off;
    std::vector<long long> woff;
    int maxnc = 0;
};

// Offsets of the components' dense blocks, and the largest component.
void block_offsets(const HostProblem& hp, CmpOrder& o) {
    const int C = hp.ncomp;
    o.cnt.assign(C, 0);
    for (int v = 0; v < hp.n; ++v) ++o.cnt[hp.comp_of_vertex[v]];
    o.woff.assign(C + 1, 0);
    for (int c = 0; c < C; ++c) {
        o.woff[c + 1] = o.woff[c] + (long long)o.cnt[c] * o.cnt[c];
        o.maxnc = std::max(o.maxnc, o.cnt[c]);
    }
}

CmpLayout cmp_layout(const HostProblem& hp, const CmpOrder& ord) {
    CmpLayout L;
    const size_t n = hp.n, NE = hp.prow.size(), nl = hp.lt_idx.size(), C = hp.ncomp;
    size_t o = 0;
    auto take = [&](size_t bytes) { const size_t at = o; o = align_up(o + std::max<size_t>(bytes, 1)); return at; };
    L.lt_ptr = take((n + 1) * 4);
    L.lt_idx = take(nl * 4);
    L.colptr = take((n + 1) * 4);
    L.prow = take(NE * 4);
    L.pcol = take(NE * 4);
    L.comp = take(n * 4);
    L.loc = take(n * 4);
    L.posl = take(n * 4);
    L.peo_cat = take(n * 4);
    L.peo_off = take((C + 1) * 4);
    L.woff = take(C * 8);
    L.idx_end = o;
    L.T = take(nl * 8);
    L.schur = take(n * 8);
    L.logdet = take(C * 8);
    L.flag = take(16);
    L.base_total = L.row_begin = o;
    for (int nc : ord.cnt) L.nrowblk += (nc + kRowWarps * kRowsPerWarp - 1) / (kRowWarps * kRowsPerWarp);
    L.lt_pos = take(nl * 4);
    L.lt_loc = take(nl * 4);
    L.first = take(n * 4);
    L.rowblk = take((size_t)L.nrowblk * 8);
    L.total = o;
    for (int v = 0; v < hp.n; ++v) L.smax = std::max(L.smax, hp.lt_ptr[v + 1] - hp.lt_ptr[v]);
    return L;
}

// Host image of the index section.
void cmp_image(const HostProblem& hp, const CmpLayout& L, CmpOrder& ord, std::vector<unsigned char>& img) {
    const int n = hp.n, C = hp.ncomp;
    img.assign(L.idx_end, 0);
    auto put = [&](size_t off, const void* src, size_t bytes) { if (bytes) std::memcpy(img.data() + off, src, bytes); };
    put(L.lt_ptr, hp.lt_ptr.data(), (n + 1) * 4);
    put(L.lt_idx, hp.lt_idx.data(), hp.lt_idx.size() * 4);
    put(L.colptr, hp.colptr.data(), (n + 1) * 4);
    put(L.prow, hp.prow.data(), hp.prow.size() * 4);
    put(L.pcol, hp.pcol.data(), hp.pcol.size() * 4);
    put(L.comp, hp.comp_of_vertex.data(), n * 4);
    ord.loc.resize(n);
    ord.posl.resize(n);
    ord.peo_cat.resize(n);
    ord.peo_off.assign(C + 1, 0);
    for (int c = 0; c < C; ++c) ord.peo_off[c + 1] = ord.peo_off[c] + ord.cnt[c];
    std::vector<int> fill(C, 0);
    for (int v = 0; v < n; ++v) ord.loc[v] = fill[hp.comp_of_vertex[v]]++;
    std::fill(fill.begin(), fill.end(), 0);
    for (int k = 0; k < n; ++k) {
        const int v = hp.peo[k], c = hp.comp_of_vertex[v];
        ord.posl[v] = fill[c]++;
        ord.peo_cat[ord.peo_off[c] + ord.posl[v]] = v;
    }
    put(L.loc, ord.loc.data(), n * 4);
    put(L.posl, ord.posl.data(), n * 4);
    put(L.peo_cat, ord.peo_cat.data(), n * 4);
    put(L.peo_off, ord.peo_off.data(), (C + 1) * 4);
    put(L.woff, ord.woff.data(), C * 8);
}

// Whether the pattern has a full profile, and then the image of the tables of
// k_cmp_rows (scratch offsets row_begin .. total): elimination position and
// local index of every later neighbour; per position, the first position whose
// list holds it (itself when none does); the row blocks, longest chains first.
bool cmp_row_tables(const HostProblem& hp, const CmpLayout& L, const CmpOrder& ord, std::vector<unsigned char>& img) {
    const int n = hp.n, C = hp.ncomp;
    const std::vector<int>& peo_off = ord.peo_off;
    std::vector<int> first(n), seen(n, 0);
    for (int c = 0; c < C; ++c)
        for (int q = peo_off[c]; q < peo_off[c + 1]; ++q) first[q] = q - peo_off[c];
    for (int k = 0; k < n; ++k) {
        const int v = hp.peo[k], q0 = peo_off[hp.comp_of_vertex[v]], p = ord.posl[v];
        for (int e = hp.lt_ptr[v]; e < hp.lt_ptr[v + 1]; ++e) {
            const int qu = q0 + ord.posl[hp.lt_idx[e]];
            first[qu] = std::min(first[qu], p);
            ++seen[qu];
        }
    }
    for (int c = 0; c < C; ++c)
        for (int q = peo_off[c]; q < peo_off[c + 1]; ++q)
            if (seen[q] != (q - peo_off[c]) - first[q]) return false;
    img.assign(L.total - L.row_begin, 0);
    int* lpos = reinterpret_cast<int*>(img.data() + (L.lt_pos - L.row_begin));
    int* lloc = reinterpret_cast<int*>(img.data() + (L.lt_loc - L.row_begin));
    for (size_t e = 0; e < hp.lt_idx.size(); ++e) {
        lpos[e] = ord.posl[hp.lt_idx[e]];
        lloc[e] = ord.loc[hp.lt_idx[e]];
    }
    std::memcpy(img.data() + (L.first - L.row_begin), first.data(), (size_t)n * 4);
    std::vector<std::pair<int, int>> blk;  // (component, first row position)
    for (int c = 0; c < C; ++c)
        for (int r = 0; r < ord.cnt[c]; r += kRowWarps * kRowsPerWarp) blk.emplace_back(c, r);
    std::stable_sort(blk.begin(), blk.end(),
                     [](const std::pair<int, int>& a, const std::pair<int, int>& b) { return a.second > b.second; });
    int* flat = reinterpret_cast<int*>(img.data() + (L.rowblk - L.row_begin));
    for (const auto& b : blk) { *flat++ = b.first; *flat++ = b.second; }
    return true;
}

// Pattern value of entry (i, j): binary search of max(i, j) among the rows of
// column min(i, j).  Sets bit 2 of *flag when the entry is not in the pattern.
__device__ __forceinline__ double pattern_value(int i, int j, const int* __restrict__ colptr,
                                                const int* __restrict__ prow, const double* __restrict__ X,
                                                int* flag) {
    const int r = max(i, j), c = min(i, j);
    int lo = colptr[c], hi = colptr[c + 1] - 1;
    while (lo <= hi) {
        const int mid = (lo + hi) >> 1;
        const int pr = prow[mid];
        if (pr == r) return X[mid];
        if (pr < r) lo = mid + 1;
        else hi = mid - 1;
    }
    atomicOr(flag, 2);
    return 0.0;
}

// One warp per vertex v: t = X[N,N]^-1 X[N,v] and s = X[v,v] - X[v,N] t by a
// Cholesky factorisation X[N,N] = R R^T in shared memory (ld x ld lower block
// plus two vectors per warp).  A pivot or Schur complement that is not
// positive sets bit 1 of *flag (no completion); the pivot is then replaced by
// 1 so that the warp finishes with finite values.
__global__ void k_cmp_factor(int n, int ld, int wpb, const int* __restrict__ lt_ptr, const int* __restrict__ lt_idx,
                             const int* __restrict__ colptr, const int* __restrict__ prow,
                             const double* __restrict__ X, double* __restrict__ T, double* __restrict__ schur,
                             int* flag) {
    extern __shared__ double cmp_smem[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int v = blockIdx.x * wpb + warp;
    if (v >= n) return;  // warp-uniform
    double* M = cmp_smem + (size_t)warp * (ld * ld + 2 * ld);
    double* z = M + ld * ld;
    double* t = z + ld;
    const int beg = lt_ptr[v], s = lt_ptr[v + 1] - beg;
    const int* N = lt_idx + beg;
    for (int f = lane; f < s * s; f += 32) {
        const int a = f / s, b = f - a * s;
        if (b <= a) M[a * ld + b] = pattern_value(N[a], N[b], colptr, prow, X, flag);
    }
    for (int a = lane; a < s; a += 32) z[a] = pattern_value(N[a], v, colptr, prow, X, flag);
    __syncwarp();
    bool bad = false;
    // right-looking Cholesky, lower triangle
    for (int j = 0; j < s; ++j) {
        double d = M[j * ld + j];
        if (!(d > 0.0) || !isfinite(d)) { bad = true; d = 1.0; }
        const double rjj = sqrt(d);
        __syncwarp();
        if (lane == 0) M[j * ld + j] = rjj;
        for (int i = j + 1 + lane; i < s; i += 32) M[i * ld + j] /= rjj;
        __syncwarp();
        for (int i = j + 1 + lane; i < s; i += 32) {
            const double lij = M[i * ld + j];
            for (int k = j + 1; k <= i; ++k) M[i * ld + k] -= lij * M[k * ld + j];
        }
        __syncwarp();
    }
    // forward solve R w = r (in z), then s = x_vv - |w|^2
    for (int j = 0; j < s; ++j) {
        const double wj = z[j] / M[j * ld + j];
        __syncwarp();
        if (lane == 0) z[j] = wj;
        for (int i = j + 1 + lane; i < s; i += 32) z[i] -= M[i * ld + j] * wj;
        __syncwarp();
    }
    double q = 0.0;
    for (int a = lane; a < s; a += 32) q += z[a] * z[a];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) q += __shfl_xor_sync(0xffffffffu, q, o);
    // back solve R^T t = w
    for (int a = lane; a < s; a += 32) t[a] = z[a];
    __syncwarp();
    for (int j = s - 1; j >= 0; --j) {
        const double tj = t[j] / M[j * ld + j];
        __syncwarp();
        if (lane == 0) t[j] = tj;
        for (int i = lane; i < j; i += 32) t[i] -= M[j * ld + i] * tj;
        __syncwarp();
    }
    for (int a = lane; a < s; a += 32) T[beg + a] = t[a];
    if (lane == 0) {
        const double sv = X[colptr[v]] - q;  // the first row of column v is v itself
        if (!(sv > 0.0) || !isfinite(sv)) bad = true;
        schur[v] = sv;
        if (bad) atomicOr(flag, 1);
    }
}

// log det of each component's completion: sum of log s over its vertices, in
// elimination order, strided partials then a fixed tree.
__global__ void k_cmp_logdet(const int* __restrict__ peo_cat, const int* __restrict__ peo_off,
                             const double* __restrict__ schur, double* __restrict__ logdet) {
    __shared__ double part[256];
    const int c = blockIdx.x;
    double acc = 0.0;
    for (int q = peo_off[c] + threadIdx.x; q < peo_off[c + 1]; q += blockDim.x) acc += log(schur[peo_cat[q]]);
    part[threadIdx.x] = acc;
    __syncthreads();
    for (int w = blockDim.x / 2; w > 0; w >>= 1) {
        if (threadIdx.x < w) part[threadIdx.x] += part[threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x == 0) logdet[c] = part[0];
}

// Given entries into the dense blocks (both triangles).
__global__ void k_cmp_scatter(int NE, const int* __restrict__ prow, const int* __restrict__ pcol,
                              const int* __restrict__ comp, const int* __restrict__ loc,
                              const int* __restrict__ peo_off, const long long* __restrict__ woff,
                              const double* __restrict__ X, double* __restrict__ W) {
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < NE; e += gridDim.x * blockDim.x) {
        const int i = prow[e], j = pcol[e], c = comp[i];
        const size_t nc = peo_off[c + 1] - peo_off[c];
        double* Wc = W + woff[c];
        const size_t li = loc[i], lj = loc[j];
        Wc[li * nc + lj] = X[e];
        Wc[lj * nc + li] = X[e];
    }
}

// Step r of the recurrence: in every component with n_c > r, the vertex at
// elimination position k = n_c - 1 - r gets its free entries against every
// vertex eliminated after it.
__global__ void __launch_bounds__(kStepThreads) k_cmp_step(int n, int r, const int* __restrict__ lt_ptr,
                                                         const int* __restrict__ lt_idx, const int* __restrict__ comp,
                                                         const int* __restrict__ loc, const int* __restrict__ posl,
                                                         const int* __restrict__ peo_cat,
                                                         const int* __restrict__ peo_off,
                                                         const long long* __restrict__ woff,
                                                         const double* __restrict__ T, double* __restrict__ W) {
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= n) return;
    const int c = comp[j];
    const int nc = peo_off[c + 1] - peo_off[c];
    const int k = nc - 1 - r;
    if (k < 0 || posl[j] <= k) return;
    const int v = peo_cat[peo_off[c] + k];
    const int beg = lt_ptr[v], s = lt_ptr[v + 1] - beg;
    // j among the later neighbours of v: a given entry
    int lo = 0, hi = s - 1;
    while (lo <= hi) {
        const int mid = (lo + hi) >> 1;
        const int u = lt_idx[beg + mid];
        if (u == j) return;
        if (u < j) lo = mid + 1;
        else hi = mid - 1;
    }
    double* Wc = W + woff[c];
    const size_t lj = loc[j], ncz = nc;
    double acc = 0.0;
    for (int a = 0; a < s; ++a) acc += Wc[(size_t)loc[lt_idx[beg + a]] * ncz + lj] * T[beg + a];
    const size_t lv = loc[v];
    Wc[lv * ncz + lj] = acc;
    Wc[lj * ncz + lv] = acc;
}

// All rows of a full-profile completion (see the top of the file).  A block
// takes 16 consecutive elimination positions of one component, 8 rows a warp;
// the rows walk the positions k = (last row) - 1 .. 0 together, so that the
// coefficients t_k and the indices N_k are the same for all of them and one
// more warp stages them in shared memory, a stage ahead.  The 4 lanes of a row
// split the dot product W[j, N_k] t_k: elements of N_k at most 64 positions
// away come from a ring in shared memory, older ones (or, for rows past the
// element, given ones) from the dense block, loaded one step ahead; the loads
// of a step are 8 consecutive entries per element.
//
// Bound: the dependent chain of a row (n steps of a few float64 multiply-adds
// and two shuffles, 0.4 us a step), not bandwidth: 8 n^2 bytes are written
// once.  4 lanes a row and 16 rows a block put a chain on nearly every SM at
// n = 2000 (125 blocks).  Banded n = 2000, w = 10, whole call: 8.73 ms as
// 1999 dependent launches of k_cmp_step, 1.03 ms with this kernel (0.80 ms of
// it here).  A row past an element's position may read an entry of the dense
// block that nothing has written: by the profile property it is never used.
struct RowArgs {
    const int *lt_ptr, *lt_pos, *lt_loc, *loc, *peo_cat, *peo_off, *first, *rowblk;
    const long long* woff;
    const double* T;
    double* W;
    int smax, nstep;  // longest later-neighbour list; steps per stage
};

// A staged coefficient: t_k[a], and where its W[j, u] is: an offset into the
// ring, or (ring < 0) the local index `far` of u in the dense block.  Unused
// terms have t = 0 and the offset of the ring's row of zeros.
struct alignas(16) RowTerm {
    double t;
    int ring, far;
};

// U: terms per lane and step (4 U >= the longest list), 0: smax as given.
template <int U>
__global__ void __launch_bounds__(kRowThreads) k_cmp_rows(RowArgs g) {
    extern __shared__ __align__(16) unsigned char row_smem[];
    __shared__ double ring[kRowWarps][(kRowRing + 1) * kRowsPerWarp];  // [position & 63][row], then zeros
    __shared__ int step_loc[2][32], step_far[2][32];  // local index of v_k; some term of the step is far
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int nt = U > 0 ? 4 * U : (g.smax + 3) & ~3, cap = nt * g.nstep;  // terms of a step, of a stage
    RowTerm* st = reinterpret_cast<RowTerm*>(row_smem);                    // [2][cap]
    const int c = g.rowblk[2 * blockIdx.x], r0 = g.rowblk[2 * blockIdx.x + 1];
    const int q0 = g.peo_off[c], nc = g.peo_off[c + 1] - q0;
    const int kmax = min(r0 + kRowWarps * kRowsPerWarp, nc) - 2;  // highest position any row of the block needs
    const int nstage = (kmax + g.nstep) / g.nstep;
    double* Wc = g.W + g.woff[c];
    // rows of the computing warps
    const int sub = lane & 3, row = lane >> 2;
    const int pj = min(r0 + kRowsPerWarp * warp + row, nc - 1);
    const bool live = warp < kRowWarps && r0 + kRowsPerWarp * warp + row < nc;
    const size_t lj = g.loc[g.peo_cat[q0 + pj]], ncz = nc;
    const int fj = g.first[q0 + pj];
    int fmin = fj;  // below it every row of the warp computes
    for (int o = 4; o < 32; o <<= 1) fmin = min(fmin, __shfl_xor_sync(0xffffffffu, fmin, o));
    double* rg = ring[warp < kRowWarps ? warp : 0] + row;
    if (warp < kRowWarps) {  // ring: the entries at positions kmax + 1 .. kmax + 64 (given ones among them)
        for (int i = sub; i < kRowRing; i += 4) {
            const int p = kmax + 1 + i;
            if (p < nc) rg[(p & (kRowRing - 1)) * kRowsPerWarp] = Wc[(size_t)g.loc[g.peo_cat[q0 + p]] * ncz + lj];
        }
        if (sub == 0) rg[kRowRing * kRowsPerWarp] = 0.0;
    }
    auto stage = [&](int s) {  // the staging warp: coefficients of stage s into its half
        const int b = s & 1, k = kmax - s * g.nstep - lane;  // lane i: step i of the stage
        int beg = 0, sv = 0, any = 0;
        if (lane < g.nstep && k >= 0) {
            const int v = g.peo_cat[q0 + k];
            beg = g.lt_ptr[v];
            sv = g.lt_ptr[v + 1] - beg;
            step_loc[b][lane] = g.loc[v];
        }
        for (int f0 = 0; f0 < cap; f0 += 8 * 32) {  // eight coefficients a lane in flight
            double t[8];
            int p[8], l[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const int f = f0 + 32 * u + lane, i = f / nt, a = f - i * nt;
                const int bi = __shfl_sync(0xffffffffu, beg, i & 31), si = __shfl_sync(0xffffffffu, sv, i & 31);
                const bool ok = f < cap && a < si;
                t[u] = ok ? g.T[bi + a] : 0.0;
                p[u] = ok ? g.lt_pos[bi + a] : -1;
                l[u] = ok ? g.lt_loc[bi + a] : 0;
            }
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const int f = f0 + 32 * u + lane, i = f / nt, ki = kmax - s * g.nstep - i;
                const bool far = p[u] - ki > kRowRing;
                if (f < cap)
                    st[b * cap + f] = RowTerm{t[u], far ? -1 : (p[u] < 0 ? kRowRing : p[u] & (kRowRing - 1)) * kRowsPerWarp, l[u]};
                if (far) any |= 1u << (i & 31);
            }
        }
        any = __reduce_or_sync(0xffffffffu, any);
        step_far[b][lane] = (any >> lane) & 1;
    };
    if (warp == kRowWarps && nstage > 0) stage(0);
    __syncthreads();
    constexpr int NF = U > 0 ? U : kRowFar;
    for (int s = 0; s < nstage; ++s) {
        if (warp == kRowWarps) {
            if (s + 1 < nstage) stage(s + 1);
        } else {
            const int b = s & 1, k0 = kmax - s * g.nstep, ns = min(g.nstep, k0 + 1);
            const RowTerm* e0 = st + b * cap + sub;
            double far[NF];
            auto load_far = [&](int i) {  // the far entries of step i (older than 64 steps, or given)
#pragma unroll
                for (int u = 0; u < NF; ++u) {
                    if (U == 0 && 4 * u >= nt) break;
                    const RowTerm e = e0[i * nt + 4 * u];
                    far[u] = e.ring < 0 ? Wc[(size_t)e.far * ncz + lj] : 0.0;
                }
            };
            if (step_far[b][0]) load_far(0);
            for (int i = 0; i < ns; ++i) {
                const int k = k0 - i;
                const size_t lk = step_loc[b][i];
                const RowTerm* e = e0 + i * nt;
                double acc = 0.0;
                if (step_far[b][i]) {
#pragma unroll
                    for (int u = 0; u < NF; ++u) {
                        if (U == 0 && 4 * u >= nt) break;
                        acc += (e[4 * u].ring < 0 ? far[u] : rg[max(e[4 * u].ring, 0)]) * e[4 * u].t;
                    }
                } else {
#pragma unroll
                    for (int u = 0; u < NF; ++u) {
                        if (U == 0 && 4 * u >= nt) break;
                        acc += rg[e[4 * u].ring] * e[4 * u].t;
                    }
                }
                if (U == 0)
                    for (int u = kRowFar; 4 * u < nt; ++u) {
                        const RowTerm x = e[4 * u];
                        acc += (x.ring < 0 ? Wc[(size_t)x.far * ncz + lj] : rg[x.ring]) * x.t;
                    }
                acc += __shfl_xor_sync(0xffffffffu, acc, 1);
                acc += __shfl_xor_sync(0xffffffffu, acc, 2);
                bool given = false;  // (j, v_k) is in the pattern, or v_k is not eliminated before j
                if (k >= fmin) {
                    given = k >= fj;
                    if (given) acc = Wc[lk * ncz + lj];
                }
                if (sub == 0) rg[(k & (kRowRing - 1)) * kRowsPerWarp] = acc;
                if (!given && live) {
                    if (sub == 0) Wc[lk * ncz + lj] = acc;
                    if (sub == 1) Wc[lj * ncz + lk] = acc;
                }
                __syncwarp();
                if (i + 1 < ns && step_far[b][i + 1]) load_far(i + 1);
            }
        }
        __syncthreads();
    }
}

cudaError_t launch_rows(const RowArgs& a, int blocks, cudaStream_t st) {
    const int U = (a.smax + 3) / 4;
    const size_t smem = 2 * sizeof(RowTerm) * (size_t)(4 * U) * a.nstep;  // at most 32 KB
    switch (U <= kRowFar ? U : 0) {
        case 1: k_cmp_rows<1><<<blocks, kRowThreads, smem, st>>>(a); break;
        case 2: k_cmp_rows<2><<<blocks, kRowThreads, smem, st>>>(a); break;
        case 3: k_cmp_rows<3><<<blocks, kRowThreads, smem, st>>>(a); break;
        case 4: k_cmp_rows<4><<<blocks, kRowThreads, smem, st>>>(a); break;
        case 5: k_cmp_rows<5><<<blocks, kRowThreads, smem, st>>>(a); break;
        case 6: k_cmp_rows<6><<<blocks, kRowThreads, smem, st>>>(a); break;
        case 7: k_cmp_rows<7><<<blocks, kRowThreads, smem, st>>>(a); break;
        case 8: k_cmp_rows<8><<<blocks, kRowThreads, smem, st>>>(a); break;
        default: k_cmp_rows<0><<<blocks, kRowThreads, smem, st>>>(a);
    }
    return cudaGetLastError();
}

int cuda_fail(std::string* err, cudaError_t e, const char* what) {
    if (err) *err = std::string(what) + ": " + cudaGetErrorString(e);
    cudaGetLastError();
    return CDSDP_ERR_CUDA;
}

}  // namespace

void completion_release(CmpGraph& g) {
    if (g.exec) cudaGraphExecDestroy((cudaGraphExec_t)g.exec);
    g.exec = nullptr;
    g.scratch = nullptr;
    g.W = nullptr;
}

int completion_sizes(const HostProblem& hp, size_t* scratch_bytes, long long* w_elems, long long* w_offsets) {
    CmpOrder ord;
    block_offsets(hp, ord);
    if (scratch_bytes) *scratch_bytes = cmp_layout(hp, ord).total;
    if (w_elems) *w_elems = ord.woff[hp.ncomp];
    if (w_offsets) std::copy(ord.woff.begin(), ord.woff.end(), w_offsets);
    return CDSDP_SOLVED;
}

int completion_run(const HostProblem& hp, const double* d_X, void* d_scratch, size_t scratch_bytes, double* d_W,
                   double* logdet, void* stream, std::string* err, CmpGraph* cache) {
    if (!d_X || !d_scratch) return CDSDP_ERR_ARG;
    if (reinterpret_cast<uintptr_t>(d_scratch) % kCmpAlign) return CDSDP_ERR_ARG;
    CmpOrder ord;
    block_offsets(hp, ord);
    const CmpLayout L = cmp_layout(hp, ord);
    if (scratch_bytes < L.base_total) return CDSDP_ERR_NOMEM;
    const int ld = std::max(1, L.smax);
    const size_t per_warp = (size_t)(ld * ld + 2 * ld) * sizeof(double);
    if (per_warp > kMaxWarpSmem) return CDSDP_ERR_UNSUPPORTED;
    std::vector<unsigned char> img, row_img;
    cmp_image(hp, L, ord, img);
    const int maxnc = ord.maxnc;
    cudaStream_t st = (cudaStream_t)stream;
    unsigned char* g = (unsigned char*)d_scratch;
    const int n = hp.n, NE = (int)hp.prow.size(), C = hp.ncomp;
    cudaError_t e;
#define CMP_CK(call)                                        \
    do {                                                    \
        e = (call);                                         \
        if (e != cudaSuccess) return cuda_fail(err, e, #call); \
    } while (0)
    CMP_CK(cudaMemcpyAsync(g, img.data(), img.size(), cudaMemcpyHostToDevice, st));
    CMP_CK(cudaMemsetAsync(g + L.flag, 0, 16, st));
    const int* lt_ptr = (const int*)(g + L.lt_ptr);
    const int* lt_idx = (const int*)(g + L.lt_idx);
    const int* colptr = (const int*)(g + L.colptr);
    const int* prow = (const int*)(g + L.prow);
    const int* pcol = (const int*)(g + L.pcol);
    const int* comp = (const int*)(g + L.comp);
    const int* loc = (const int*)(g + L.loc);
    const int* posl = (const int*)(g + L.posl);
    const int* peo_cat = (const int*)(g + L.peo_cat);
    const int* peo_off = (const int*)(g + L.peo_off);
    const long long* dwoff = (const long long*)(g + L.woff);
    double* T = (double*)(g + L.T);
    double* schur = (double*)(g + L.schur);
    double* dlog = (double*)(g + L.logdet);
    int* flag = (int*)(g + L.flag);
    const int wpb = (int)std::max<size_t>(1, std::min<size_t>(8, (48 * 1024) / per_warp));
    const size_t smem = per_warp * wpb;
    if (smem > 48 * 1024) CMP_CK(cudaFuncSetAttribute(k_cmp_factor, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    k_cmp_factor<<<(n + wpb - 1) / wpb, 32 * wpb, smem, st>>>(n, ld, wpb, lt_ptr, lt_idx, colptr, prow, d_X, T,
                                                               schur, flag);
    CMP_CK(cudaGetLastError());
    // beside the factor kernel; a logdet alone and other patterns need no row tables
    const bool rows = d_W && scratch_bytes >= L.total && cmp_row_tables(hp, L, ord, row_img);
    int hflag = 0;
    CMP_CK(cudaMemcpyAsync(&hflag, flag, sizeof(int), cudaMemcpyDeviceToHost, st));
    CMP_CK(cudaStreamSynchronize(st));
    if (hflag & 2) {
        if (err) *err = "completion: pattern inconsistent with the elimination order";
        return CDSDP_ERR_ARG;
    }
    if (hflag & 1) return CDSDP_NOT_PD;
    if (rows) CMP_CK(cudaMemcpyAsync(g + L.row_begin, row_img.data(), row_img.size(), cudaMemcpyHostToDevice, st));
    k_cmp_logdet<<<C, 256, 0, st>>>(peo_cat, peo_off, schur, dlog);
    CMP_CK(cudaGetLastError());
    if (d_W) {
        const int gs = std::max(1, std::min(4096, (NE + 255) / 256));
        k_cmp_scatter<<<gs, 256, 0, st>>>(NE, prow, pcol, comp, loc, peo_off, dwoff, d_X, d_W);
        CMP_CK(cudaGetLastError());
        const int gn = (n + kStepThreads - 1) / kStepThreads;
        auto steps = [&](cudaStream_t s2) {
            for (int r = 1; r < maxnc; ++r)
                k_cmp_step<<<gn, kStepThreads, 0, s2>>>(n, r, lt_ptr, lt_idx, comp, loc, posl, peo_cat, peo_off,
                                                        dwoff, T, d_W);
            return cudaGetLastError();
        };
        if (rows) {  // full profile: rows are independent, one launch
            RowArgs ra;
            ra.lt_ptr = lt_ptr;
            ra.lt_pos = (const int*)(g + L.lt_pos);
            ra.lt_loc = (const int*)(g + L.lt_loc);
            ra.loc = loc;
            ra.peo_cat = peo_cat;
            ra.peo_off = peo_off;
            ra.first = (const int*)(g + L.first);
            ra.rowblk = (const int*)(g + L.rowblk);
            ra.woff = dwoff;
            ra.T = T;
            ra.W = d_W;
            ra.smax = std::max(1, L.smax);
            ra.nstep = std::max(1, std::min(32, kRowTerms / ((ra.smax + 3) / 4 * 4)));
            CMP_CK(launch_rows(ra, L.nrowblk, st));
        } else if (!cache || maxnc < 2) {
            CMP_CK(steps(st));
        } else {
            if (!cache->exec || cache->scratch != d_scratch || cache->W != d_W) {
                completion_release(*cache);
                cudaStream_t cs;
                CMP_CK(cudaStreamCreateWithFlags(&cs, cudaStreamNonBlocking));
                cudaGraph_t graph = nullptr;
                e = cudaStreamBeginCapture(cs, cudaStreamCaptureModeThreadLocal);
                if (e == cudaSuccess) {
                    const cudaError_t e2 = steps(cs);
                    e = cudaStreamEndCapture(cs, &graph);
                    if (e2 != cudaSuccess) e = e2;
                }
                cudaStreamDestroy(cs);
                cudaGraphExec_t exec = nullptr;
                if (e == cudaSuccess) e = cudaGraphInstantiate(&exec, graph, 0);
                if (graph) cudaGraphDestroy(graph);
                if (e != cudaSuccess) return cuda_fail(err, e, "completion graph");
                cache->exec = exec;
                cache->scratch = d_scratch;
                cache->W = d_W;
            }
            CMP_CK(cudaGraphLaunch((cudaGraphExec_t)cache->exec, st));
        }
    }
    if (logdet) {
        CMP_CK(cudaMemcpyAsync(logdet, dlog, C * sizeof(double), cudaMemcpyDeviceToHost, st));
        CMP_CK(cudaStreamSynchronize(st));
    }
#undef CMP_CK
    return CDSDP_SOLVED;
}

}  // namespace cdsdp_impl

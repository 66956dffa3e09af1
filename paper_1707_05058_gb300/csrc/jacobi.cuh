// Batched PSD projection P(W) = V max(Lambda, 0) V^T of clique blocks
// (Section 4.1.2, Eq. XkUpdate; Eq. zkUpdate; Eq. HsdeStep2), one warp per
// block of order s <= 32.
//
// Eigensolver: two-sided cyclic Jacobi (Jacobi 1846; 2x2 symmetric Schur step
// of Golub and Van Loan, Matrix Computations, Section 8.5) in the parallel
// ordering of Brent and Luk (1985).  The block is padded with zero rows to an
// even order S (padding rows never rotate: their entries stay exactly zero and
// their eigenvalues are 0).  Storage positions are paired as (2k, 2k+1),
// k < S/2; after every round the matrix is re-indexed by the round-robin
// permutation sigma (position 0 fixed, the other S-1 positions rotate along the
// circle 2, 4, ..., S-2, S-1, S-3, ..., 1), so over one sweep of S-1 rounds
// every pair of indices meets exactly once and the storage order returns to
// the identity.  Each lane owns fixed 2x2 pair-blocks (I, J), I >= J, of the
// lower triangle: per round it loads them from one shared-memory buffer,
// applies J_I^T B J_J and writes them to their permuted positions in the other
// buffer (one warp barrier per round).  Row `lane` of V stays in registers
// and its columns are re-indexed by the same sigma (static register moves).
// Every rotation is applied in Rutishauser's form (Handbook for Automatic
// Computation II, contribution II/1, 1971): with tau = s / (1 + c),
//   x' = c x - s y = x - s (y + tau x),   y' = s x + c y = y + s (x - tau y).
// For the small angles of the late sweeps c rounds to 1 while s = t does not,
// so the plain (c, s) products grow every rotated row and column by a factor
// 1 + t^2 (a bias, not noise); in float32 this bias, summed over a few hundred
// rotations per eigenvector, dominated the error of the projection.  The tau
// form carries 1 - c = s tau implicitly and has no such bias.
// A rotation is skipped when |a_pq| <= tol = 2 u ||W||_F (u the unit
// roundoff), and a sweep starts only while some off-diagonal entry exceeds tol
// (or until max_sweeps).  Eigenvalues clustered within rounding noise of each
// other (typical near zero at ADMM convergence) can keep off-diagonal entries
// at about S u ||W||_F forever; a block whose largest off-diagonal entry is
// below 4 S u ||W||_F and did not halve over the last sweep has reached that
// floor and stops.
// In a solve the sweeps end before that: what is rebuilt is P(W) to first order
// in the remaining off-diagonal part (project()), and a sweep is left out once
// an estimate of what that leaves out is at most a quarter of tol (run()).
// Warm start (ADMM iterates move little between iterations): each clique keeps
// its eigenvectors V from the previous iteration; the new block W is first
// rotated into that basis (A = V^T W V, two warp-level products) and the
// sweeps continue from V, which typically needs one sweep instead of five or
// six.  Every `restart` iterations the eigensolve starts from the identity, so
// rounding in the accumulated V cannot drift.
#pragma once

#include "reduce.cuh"
#include "proj_launch.h"

namespace cdsdp_dev {

// ---- round-robin ordering on S storage positions ---------------------------
template <int S>
struct RoundRobin {
    static constexpr int K = S / 2;
    static constexpr int R = S - 1;
    __host__ __device__ static constexpr int circ_index(int p) {  // p > 0
        return (p % 2 == 0) ? (p / 2 - 1) : (K - 1 + (K - 1 - (p - 1) / 2));
    }
    __host__ __device__ static constexpr int circ_pos(int c) {
        return c < K - 1 ? 2 * (c + 1) : 2 * (K - 1 - (c - (K - 1))) + 1;
    }
    __host__ __device__ static constexpr int sigma(int p) { return p == 0 ? 0 : circ_pos((circ_index(p) + 1) % R); }
    __host__ __device__ static constexpr int sigma_inv(int p) {
        return p == 0 ? 0 : circ_pos((circ_index(p) + R - 1) % R);
    }
};

// sigma in closed form: position 0 fixed, even positions one pair up, odd ones
// one pair down, turning round at both ends (the formulas of RoundRobin cost a
// modulo each; a launch evaluates four per owned pair-block).
template <int S>
__host__ __device__ constexpr int rr_sigma(int p) {
    return p == 0 ? 0 : (p == 1 ? (S == 2 ? 1 : 2) : ((p & 1) ? p - 2 : (p == S - 2 ? S - 1 : p + 2)));
}
template <int S>
constexpr bool rr_sigma_ok() {
    for (int p = 0; p < S; ++p)
        if (rr_sigma<S>(p) != RoundRobin<S>::sigma(p)) return false;
    return true;
}

// (a, b) of packed element f of an s x s block (s <= 128), a >= b, column-major.
// Column b starts where t - sqrt(t^2 - 8 f) = 2 b exactly (t = 2 s + 1) and the
// last entry of a column lies at least 4 / t below the next start, so an offset
// of 2e-3 covers the error of the approximate square root (2^-23 relative).
__device__ __forceinline__ int packed_ab(int f, int s) {
    const float t = float(2 * s + 1);
    float r;
    asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(fmaf(-8.0f, float(f), t * t)));
    const int b = int((t + 2e-3f - r) * 0.5f);
    const int a = b + f - ((b * (2 * s - b + 1)) >> 1);
    return (a << 8) | b;
}

// Rotation of a 2x2 symmetric block, half-angle form: (tau, s) with
// s = sin, tau = tan(theta/2) = s / (1 + c), zeros when |apq| <= tol.
//
// float: cos 2theta = |zeta| / r and sin 2theta = apq / r with
// zeta = (aqq - app)/2, r = sqrt(zeta^2 + apq^2); c^2 = (1 + cos 2theta)/2,
// s = sin 2theta / (2 c).  sc = 1 / ||W||_F brings the entries to order one, so
// that approximate reciprocal roots without denormal handling serve (a rotated
// entry exceeds 2 u ||W||_F, its square 1e-14).  1/(1 + c) comes from a
// quadratic fit on c in [1/sqrt 2, 1] (relative error 1.3e-4) and one Newton
// step (1.6e-8): two reciprocal square roots are the only special functions
// on the chain.  No branch: a lane without a rotation selects zeros.
// ta = tan(theta) apq is the change of the two diagonal entries.
__device__ __forceinline__ float rsqrt_ftz(float x) {
    float r;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
__device__ __forceinline__ float rcp_ftz(float x) {
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
__device__ __forceinline__ void rotation(float app, float aqq, float apq, float tol, float sc, float& tau, float& sn,
                                         float& ta) {
    const float zeta = (aqq - app) * (0.5f * sc), q = apq * sc;
    const float ri = rsqrt_ftz(zeta * zeta + q * q);
    const float c2 = 0.5f + 0.5f * fabsf(zeta) * ri;
    const float ci = rsqrt_ftz(c2);
    const float sx = copysignf(0.5f, zeta) * q * ri * ci;
    const float d = 1.0f + c2 * ci;
    float y = (0.1577689f * d - 0.8772993f) * d + 1.623585f;
    y += y * (1.0f - d * y);
    const bool on = fabsf(apq) > tol;
    sn = on ? sx : 0.0f;
    tau = on ? sx * y : 0.0f;
    ta = on ? sx * ci * apq : 0.0f;
}
// double: the float64 pipe does two operations a clock and SM, and its
// divisions and square roots take tens of them, so the angle is found in
// float32 (sc scales the entries to order one first) and only the pair
// (tau, s = 2 tau / (1 + tau^2)) is formed in double: the rotation is
// orthogonal to double precision, and an angle off by 1e-7 leaves 1e-7 of the
// off-diagonal entry behind, which the entry keeps (no entry is set to zero).
__device__ __forceinline__ void rotation(double app, double aqq, double apq, double tol, double sc, double& tau,
                                         double& sn, double& ta) {
    const float zeta = float((aqq - app) * (0.5 * sc)), q = float(apq * sc);
    const float ri = rsqrt_ftz(zeta * zeta + q * q);
    const float c2 = 0.5f + 0.5f * fabsf(zeta) * ri;
    const float ci = rsqrt_ftz(c2);
    float tf = copysignf(0.5f, zeta) * q * ri * ci * rcp_ftz(1.0f + c2 * ci);
    tf = fabs(apq) > tol ? tf : 0.0f;
    tau = double(tf);
    const double d = fma(tau, tau, 1.0);
    double y = double(rcp_ftz(fmaf(tf, tf, 1.0f)));
    y = fma(y, fma(-d, y, 1.0), y);
    y = fma(y, fma(-d, y, 1.0), y);
    sn = (tau + tau) * y;
    ta = 0.0;
}

// The same rotation through tan(theta) (Rutishauser's form of the 2x2 Schur
// step), for the smallest orders, where few rotations make each one's rounding
// show: 1,024 random blocks of order 2, 3 and 4 came out 0.81, 1.44 and 1.85
// u ||W||_F off with the half-angle form in float and 0.69, 1.38 and 1.78 through
// the tangent (order 5: 2.21 and 2.28); in double order 2 0.77 and 0.68, since an
// angle in float32 takes it two rotations, and no difference above.
// float: three special functions on the chain and no branch; the entries are of
// order one with sc, and 1/(1 + c) is found as in rotation().
__device__ __forceinline__ void rotation_small(float app, float aqq, float apq, float tol, float sc, float& tau,
                                               float& sn, float& ta) {
    const float zeta = (aqq - app) * (0.5f * sc), q = apq * sc;
    const float r2 = zeta * zeta + q * q;
    const float t = copysignf(1.0f, zeta) * q * rcp_ftz(fabsf(zeta) + r2 * rsqrt_ftz(r2));
    const float c = rsqrt_ftz(1.0f + t * t);
    const float d = 1.0f + c;
    float y = (0.1577689f * d - 0.8772993f) * d + 1.623585f;
    y += y * (1.0f - d * y);
    const bool on = fabsf(apq) > tol;
    const float s = t * c;
    sn = on ? s : 0.0f;
    tau = on ? s * y : 0.0f;
    ta = on ? t * apq : 0.0f;
}
// And, with sc = 1, for the unrolled passes: a derivative through the projections jumps
// where an eigenvalue changes sign, so gradients are only comparable between
// builds while the projections round alike, and these kept their arithmetic
// when the half-angle form above replaced it in the solves.
template <typename T>
__device__ __forceinline__ void rotation_tan(T app, T aqq, T apq, T tol, T sc, T& tau, T& sn, T& ta) {
    tau = T(0); sn = T(0); ta = T(0);
    if (fabs(apq) > tol) {
        const T zeta = T(0.5) * (aqq - app) * sc, q = apq * sc;
        const T r2 = zeta * zeta + q * q;
        const T r = r2 * rsqrt_t<T>(r2);
        const T tt = copysign(T(1), zeta) * div_t<T>(q, fabs(zeta) + r);
        const T c = rsqrt_t<T>(T(1) + tt * tt);
        sn = tt * c;
        tau = div_t<T>(sn, T(1) + c);
        ta = tt * apq;
    }
}

// Rows of N entries at 16-byte aligned addresses, as 16-byte accesses.
template <int N>
__device__ __forceinline__ void row_ld(const float* p, float (&v)[N]) {
#pragma unroll
    for (int j = 0; j + 4 <= N; j += 4) {
        const float4 q = *reinterpret_cast<const float4*>(p + j);
        v[j] = q.x; v[j + 1] = q.y; v[j + 2] = q.z; v[j + 3] = q.w;
    }
#pragma unroll
    for (int j = N & ~3; j < N; ++j) v[j] = p[j];
}
template <int N>
__device__ __forceinline__ void row_ld(const double* p, double (&v)[N]) {
#pragma unroll
    for (int j = 0; j + 2 <= N; j += 2) {
        const double2 q = *reinterpret_cast<const double2*>(p + j);
        v[j] = q.x; v[j + 1] = q.y;
    }
}
template <int N>
__device__ __forceinline__ void row_st(float* p, const float (&v)[N]) {
#pragma unroll
    for (int j = 0; j + 4 <= N; j += 4) *reinterpret_cast<float4*>(p + j) = make_float4(v[j], v[j + 1], v[j + 2], v[j + 3]);
#pragma unroll
    for (int j = N & ~3; j < N; ++j) p[j] = v[j];
}
template <int N>
__device__ __forceinline__ void row_st(double* p, const double (&v)[N]) {
#pragma unroll
    for (int j = 0; j + 2 <= N; j += 2) *reinterpret_cast<double2*>(p + j) = make_double2(v[j], v[j + 1]);
}
// sum_i a[i] p[i], two chains
template <typename T, int N>
__device__ __forceinline__ T row_dot(const T (&a)[N], const T* p) {
    T b[N];
    row_ld(p, b);
    T s0 = T(0), s1 = T(0);
#pragma unroll
    for (int i = 0; i < N; i += 2) {
        s0 += a[i] * b[i];
        s1 += a[i + 1] * b[i + 1];
    }
    return s0 + s1;
}

// The same sum in order, one chain.
template <typename T, int N>
__device__ __forceinline__ T row_dot_seq(const T (&a)[N], const T* p) {
    T b[N];
    row_ld(p, b);
    T s = T(0);
#pragma unroll
    for (int i = 0; i < N; ++i) s += a[i] * b[i];
    return s;
}

// (x, y) at an address aligned to both
template <typename T> struct PairOf;
template <> struct PairOf<float> { using P = float2; };
template <> struct PairOf<double> { using P = double2; };

// TAN: the arithmetic of the unrolled passes (rotation_tan, and projected
// blocks from the diagonal alone).
template <typename T, int S, int LW = 32, bool TAN = false>
struct BLJacobi {
    static_assert(LW == 32 || LW == 16 || LW == 8, "lanes per clique");
    static_assert(LW == 32 || S <= LW, "row `lane` of V needs a lane per row");
    static_assert(rr_sigma_ok<S>(), "closed form of sigma");
    using RR = RoundRobin<S>;
    // order 2: one rotation leaves an exact zero, so the diagonal alone is P(W)
    static constexpr bool DIAG = TAN || S == 2;
    static constexpr bool EXACT = TAN || S <= (sizeof(T) == 4 ? 4 : 2);  // through tan(theta)
    static constexpr int K = S / 2;
    static constexpr int R = S - 1;
    // row pitch: rows start on 16 bytes and eight consecutive rows read as
    // 16-byte vectors fall into different banks; one spare column at least
    static constexpr int LDA = sizeof(T) == 4 ? ((S + 4) / 8) * 8 + 4 : (((S / 2) & 1) == 0 ? S + 2 : S + 4);
    static_assert(LDA > S, "a spare column");
    static constexpr int BUF = S * LDA;
    static constexpr int NB = K * (K + 1) / 2;      // lower pair-blocks
    static constexpr int NS = (NB + LW - 1) / LW;   // blocks per lane
    static constexpr int NPK = S * (S + 1) / 2;
    static constexpr int MAXE = (NPK + LW - 1) / LW;  // packed elements per lane
    // per clique; an odd multiple of 64 bytes, so that the groups of a warp start in different banks
    static constexpr size_t bytes = (((2 * BUF + 4 * K) * sizeof(T) + 63) / 64 | 1) * 64;
    using P2 = typename PairOf<T>::P;

    T* X;    // current buffer
    T* Y;    // next buffer
    P2* rot;  // [2][K] (tau, s) of a round's rotations, double-buffered
    T v[S];  // row `lane` of V
    int src[NS], dst[NS][4];
    int bI[NS], bJ[NS];

    __device__ __forceinline__ void bind(unsigned char* base, int lane) {
        X = reinterpret_cast<T*>(base);
        Y = X + BUF;
        rot = reinterpret_cast<P2*>(Y + BUF);
#pragma unroll
        for (int t = 0; t < NS; ++t) {
            const int b = lane + LW * t;
            int I, J;
            if (b < K) {
                I = J = b;
            } else {  // o = I (I - 1) / 2 + J: (8 o + 1) is a square where a row starts
                const int o = b - K;
                float r;
                asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(float(8 * o + 1)));
                I = int((1.0f + r + 2e-3f) * 0.5f);
                J = o - I * (I - 1) / 2;
            }
            const bool ok = b < NB;
            if (!ok) I = J = 0;
            bI[t] = ok ? I : -1;
            bJ[t] = J;
            const int r0 = 2 * I, r1 = 2 * I + 1, c0 = 2 * J, c1 = 2 * J + 1;
            src[t] = r0 * LDA + c0;
            const int rr[4] = {r0, r1, r0, r1}, cc[4] = {c0, c0, c1, c1};
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const int si = rr_sigma<S>(rr[e]), sj = rr_sigma<S>(cc[e]);
                dst[t][e] = max(si, sj) * LDA + min(si, sj);
            }
        }
    }

    // entries (2I, 2J), (2I+1, 2J), (2I, 2J+1), (2I+1, 2J+1) of pair-block t;
    // the upper entry of a diagonal block is its lower one
    __device__ __forceinline__ void block_ld(int t, T (&b)[4]) const {
        const P2 u = *reinterpret_cast<const P2*>(X + src[t]), l = *reinterpret_cast<const P2*>(X + src[t] + LDA);
        b[0] = u.x;
        b[1] = l.x;
        b[2] = bI[t] == bJ[t] ? l.x : u.y;
        b[3] = l.y;
    }

    // Zero the working buffer (padding rows must read as exact zeros; a block of
    // full order fills every entry itself).
    __device__ __forceinline__ void clear(int lane, int s) {
        if (s < S)
            for (int i = lane; i < BUF; i += LW) X[i] = T(0);
        __syncwarp();
    }
    __device__ __forceinline__ void put(int a, int b, T w) {
        X[a * LDA + b] = w;
        X[b * LDA + a] = w;
    }

    // Largest |off-diagonal entry| of the lower triangle in X and, unless DIAG, with
    // sc = 1 / ||W||_F the sum over pairs sc a_ij^2 / (|a_ii| + |a_jj|) (see run();
    // same in all lanes of the group).
    __device__ __forceinline__ void off_diagonal(int lane, T sc, T& off, float& second) const {
        T m = T(0);
        float x2 = 0.0f;
#pragma unroll
        for (int t = 0; t < NS; ++t) {
            if (bI[t] < 0) continue;
            const T* p = X + src[t];
            const int r0 = 2 * bI[t] * (LDA + 1), c0 = 2 * bJ[t] * (LDA + 1);
            const float lr[2] = {float(fabs(X[r0]) * sc), float(fabs(X[r0 + LDA + 1]) * sc)};
            const float lc[2] = {float(fabs(X[c0]) * sc), float(fabs(X[c0 + LDA + 1]) * sc)};
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const int i = e & 1, j = e >> 1;
                const T x = fabs(p[i * LDA + j]);
                if (t == 0 && lane < K && e != 1) continue;  // of a diagonal block the lower entry only
                m = fmax(m, x);
                if constexpr (!DIAG) {
                    const float y = float(x * sc);
                    x2 += y * y * rcp_ftz(fmaxf(lr[i] + lc[j], 1.0e-30f));
                }
            }
        }
#pragma unroll
        for (int o = LW / 2; o > 0; o >>= 1) {  // within the group
            m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
            if constexpr (!DIAG) x2 += __shfl_xor_sync(0xffffffffu, x2, o);
        }
        off = m;
        second = x2;
    }

    // Warm start from the orthogonal V stored at Vc (column j of row r at
    // Vc[j s + r], so that a lane's row and the group's accesses are both in
    // order): v <- row `lane` of V (padded with the identity) and X <- V^T X V,
    // X holding the symmetric block (both triangles).  Every product entry is
    // the dot product of a register row with a row of shared memory that all
    // lanes read at once: T^T = (W V)^T row by row, then V^T T.
    __device__ __forceinline__ void rotate_into_stored(const T* __restrict__ Vc, int s, int lane) {
        const int row = lane < S ? lane : S - 1;
#pragma unroll
        for (int j = 0; j < S; ++j) v[j] = (lane < s && j < s) ? Vc[j * s + lane] : (j == lane ? T(1) : T(0));
        if (lane < S) {
#pragma unroll
            for (int j = 0; j < S; ++j) Y[j * LDA + lane] = v[j];  // Y = V^T
        }
        T x[S], vc[S];
        row_ld(X + row * LDA, x);
        __syncwarp();
        row_ld(Y + row * LDA, vc);  // column `lane` of V
        dots(x, Y, X, lane);        // X[j][r] = (W V)_{rj}
        __syncwarp();
        dots(vc, X, Y, lane);       // Y[j][i] = (V^T W V)_{ij}
        __syncwarp();
        T* t = X; X = Y; Y = t;
    }
    // out[j][lane] = sum_i a[i] in[j][i]
    __device__ __forceinline__ void dots(const T (&a)[S], const T* in, T* out, int lane) {
        constexpr int U = S % 4 == 0 ? 4 : 2;
#pragma unroll 1
        for (int j = 0; j < S; j += U) {
            T r[U];
#pragma unroll
            for (int u = 0; u < U; ++u) r[u] = TAN ? row_dot_seq(a, in + (j + u) * LDA) : row_dot(a, in + (j + u) * LDA);
            if (lane < S) {
#pragma unroll
                for (int u = 0; u < U; ++u) out[(j + u) * LDA + lane] = r[u];
            }
        }
    }

    __device__ __forceinline__ void store_basis(T* __restrict__ Vc, int s, int lane) const {
        if (lane < s) {
#pragma unroll
            for (int j = 0; j < S; ++j)
                if (j < s) Vc[j * s + lane] = v[j];
        }
    }

    // X <- V^T X V with the rows of V in v (X symmetric, both triangles; the
    // spare column of Y is left alone).
    __device__ void rotate_into_basis(int lane) {
        constexpr int NE1 = (S * S + LW - 1) / LW;
        if (lane < S) {
#pragma unroll
            for (int j = 0; j < S; ++j) Y[lane * LDA + j] = v[j];
        }
        __syncwarp();
        T acc[NE1];
#pragma unroll
        for (int e = 0; e < NE1; ++e) {  // (W V)_{rj}
            const int idx = lane + LW * e;
            T a = T(0);
            if (idx < S * S) {
                const int r = idx / S, j = idx - r * S;
                const T* xr = X + r * LDA;
#pragma unroll 4
                for (int i = 0; i < S; ++i) a += xr[i] * Y[i * LDA + j];
            }
            acc[e] = a;
        }
        __syncwarp();
#pragma unroll
        for (int e = 0; e < NE1; ++e) {
            const int idx = lane + LW * e;
            if (idx < S * S) {
                const int r = idx / S, j = idx - r * S;
                X[r * LDA + j] = acc[e];
            }
        }
        __syncwarp();
#pragma unroll
        for (int e = 0; e < NE1; ++e) {  // (V^T (W V))_{ij}
            const int idx = lane + LW * e;
            T a = T(0);
            if (idx < S * S) {
                const int i = idx / S, j = idx - i * S;
#pragma unroll 4
                for (int r = 0; r < S; ++r) a += Y[r * LDA + i] * X[r * LDA + j];
            }
            acc[e] = a;
        }
        __syncwarp();
#pragma unroll
        for (int e = 0; e < NE1; ++e) {
            const int idx = lane + LW * e;
            if (idx < S * S) {
                const int i = idx / S, j = idx - i * S;
                X[i * LDA + j] = acc[e];
            }
        }
        __syncwarp();
    }

    // X <- V X V^T (inverse of rotate_into_basis; X symmetric, both triangles).
    __device__ void rotate_out_of_basis(int lane) {
        constexpr int NE1 = (S * S + LW - 1) / LW;
        if (lane < S) {
#pragma unroll
            for (int j = 0; j < S; ++j) Y[lane * LDA + j] = v[j];
        }
        __syncwarp();
        T acc[NE1];
#pragma unroll
        for (int e = 0; e < NE1; ++e) {  // (X V^T)_{ib} = sum_j X_ij V_bj
            const int idx = lane + LW * e;
            T a = T(0);
            if (idx < S * S) {
                const int i = idx / S, b = idx - i * S;
#pragma unroll 4
                for (int j = 0; j < S; ++j) a += X[i * LDA + j] * Y[b * LDA + j];
            }
            acc[e] = a;
        }
        __syncwarp();
#pragma unroll
        for (int e = 0; e < NE1; ++e) {
            const int idx = lane + LW * e;
            if (idx < S * S) X[(idx / S) * LDA + idx % S] = acc[e];
        }
        __syncwarp();
#pragma unroll
        for (int e = 0; e < NE1; ++e) {  // (V (X V^T))_{ab} = sum_i V_ai (X V^T)_ib
            const int idx = lane + LW * e;
            T a = T(0);
            if (idx < S * S) {
                const int ar = idx / S, b = idx - ar * S;
#pragma unroll 4
                for (int i = 0; i < S; ++i) a += Y[ar * LDA + i] * X[i * LDA + b];
            }
            acc[e] = a;
        }
        __syncwarp();
#pragma unroll
        for (int e = 0; e < NE1; ++e) {
            const int idx = lane + LW * e;
            if (idx < S * S) X[(idx / S) * LDA + idx % S] = acc[e];
        }
        __syncwarp();
    }

    // V <- V J with the rotations of table B, columns re-indexed by sigma like A.
    template <int B>
    __device__ __forceinline__ void rotate_v(const T (&vin)[S], T (&vout)[S]) const {
#pragma unroll
        for (int k = 0; k < K; ++k) {
            const P2 r = rot[B * K + k];  // (tau, s)
            const T vp = vin[2 * k], vq = vin[2 * k + 1];
            vout[rr_sigma<S>(2 * k)] = vp - r.y * (vq + r.x * vp);
            vout[rr_sigma<S>(2 * k + 1)] = vq + r.y * (vp - r.x * vq);
        }
    }

    // One round: A (shared memory) from X into Y with the pair rotations, which
    // go into table B.  V follows a round behind: with V_STEP its row is taken
    // from vin into vout with the other table's rotations, work that fills the
    // wait for this round's rotation (the chain load, two reciprocal roots,
    // shuffle, store is what a round costs when few warps share an SM: 735
    // cycles at order 12 before, 540 now).
    template <int B, bool V_STEP>
    __device__ __forceinline__ void round(T tol, T sc, int lane, const T (&vin)[S], T (&vout)[S]) {
        T bv[NS][4];
#pragma unroll
        for (int t = 0; t < NS; ++t) block_ld(t, bv[t]);
        if (V_STEP) rotate_v<1 - B>(vin, vout);
        // rotation of pair `lane` (lanes < K own the diagonal blocks in slot 0)
        T tau, sn, ta;
        if constexpr (EXACT && !TAN && sizeof(T) == 4) rotation_small(bv[0][0], bv[0][3], bv[0][1], tol, sc, tau, sn, ta);
        else if constexpr (EXACT) rotation_tan(bv[0][0], bv[0][3], bv[0][1], tol, TAN ? T(1) : sc, tau, sn, ta);
        else rotation(bv[0][0], bv[0][3], bv[0][1], tol, sc, tau, sn, ta);
        if (lane < K) rot[B * K + lane] = P2{tau, sn};
        const bool schur = (EXACT || sizeof(T) == 4) && lane < K && sn != T(0);
#pragma unroll
        for (int t = 0; t < NS; ++t) {
            const int I = bI[t] >= 0 ? bI[t] : 0, J = bJ[t];
            const T uI = __shfl_sync(0xffffffffu, tau, I, LW), sI = __shfl_sync(0xffffffffu, sn, I, LW);
            const T uJ = __shfl_sync(0xffffffffu, tau, J, LW), sJ = __shfl_sync(0xffffffffu, sn, J, LW);
            // J_I^T B J_J, rows then columns, in the tau form
            const T r00 = bv[t][0] - sI * (bv[t][1] + uI * bv[t][0]);
            const T r10 = bv[t][1] + sI * (bv[t][0] - uI * bv[t][1]);
            const T r01 = bv[t][2] - sI * (bv[t][3] + uI * bv[t][2]);
            const T r11 = bv[t][3] + sI * (bv[t][2] - uI * bv[t][3]);
            T o00 = r00 - sJ * (r01 + uJ * r00);
            T o01 = r01 + sJ * (r00 - uJ * r01);
            T o10 = r10 - sJ * (r11 + uJ * r10);
            T o11 = r11 + sJ * (r10 - uJ * r11);
            if (t == 0) {  // diagonal block whose angle is exact to T: the 2x2 Schur result
                o00 = schur ? bv[t][0] - ta : o00;
                o11 = schur ? bv[t][3] + ta : o11;
                o10 = schur ? T(0) : o10;
                o01 = schur ? T(0) : o01;
            }
            if (bI[t] >= 0) {
                Y[dst[t][0]] = o00;
                Y[dst[t][2]] = o01;
                Y[dst[t][1]] = o10;
                Y[dst[t][3]] = o11;
            }
        }
        __syncwarp();
        T* tmp = X; X = Y; Y = tmp;
    }

    // fro = ||W||_F and sc = 1 / ||W||_F (0 for a zero block: nothing to rotate
    // there) from its square; sc only brings entries to order one.
    // float: a block whose squares leave the type's range takes a fixed scale, at
    // which its entries' squares are normal numbers, the lower end of the norm for
    // the threshold (0 below 1e-18, 3e18 above that), and no theta, so that it is
    // swept to single entries: read as a zero block, one of entries near 1e-24 came
    // back unprojected.
    // double: a float32 root serves for sc, without the hundreds of cycles of a
    // float64 root and division.  Blocks beyond 1e-145 and 1e145 are scaled by
    // their largest entry (X holds the block in both triangles) where WIDE is set:
    // the standalone kernels; in the solves its registers cost k_project_dual<double,
    // 16> 3% in spills.
    template <bool WIDE>
    __device__ __forceinline__ void norm(T nrm2, bool active, int lane, T& fro, T& sc, float& theta) const {
        if (TAN) {
            fro = sqrt(nrm2);
            sc = T(1);
            return;
        }
        if constexpr (sizeof(T) == 4) {
            fro = sqrt(nrm2);
            sc = 1.0f / fro;
            if (!(nrm2 >= 1.0e-36f && nrm2 <= 1.0e37f)) {
                fro = nrm2 < 1.0f ? 0.0f : 3.0e18f;
                sc = nrm2 < 1.0f ? 1.0e30f : 1.0e-30f;
                theta = -1.0f;
            }
            return;
        }
        if (nrm2 > T(1e-30) && nrm2 < T(1e30)) {
            sc = T(rsqrt_ftz(float(nrm2)));
            fro = nrm2 * sc;
        } else {
            fro = sqrt(nrm2);
            sc = nrm2 > T(0) ? T(1) / fro : T(0);
        }
        if (!WIDE) return;
        const bool out = active && !(nrm2 >= T(1e-290) && nrm2 <= T(1e290));
        if (!__any_sync(0xffffffffu, out)) return;
        T m = T(0), s = T(0);
#pragma unroll 1
        for (int i = lane; i < S * S; i += LW) m = fmax(m, fabs(X[(i / S) * LDA + i % S]));
        for (int o = LW / 2; o > 0; o >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
        // tiny entries are brought up by a constant first, so that 1 / m is finite
        const T up = m < T(1) ? T(1e250) : T(1);
        const T dn = T(1) / (m * up);
#pragma unroll 1
        for (int i = lane; i < S * S; i += LW) {
            const T x = X[(i / S) * LDA + i % S] * up * dn;
            s += x * x;
        }
        for (int o = LW / 2; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (!out || !(s > T(0)) || !(m <= T(1.7e308))) return;  // zero, NaN, infinite
        const T root = sqrt(s);
        fro = root * m;
        sc = fmin(dn / root * up, T(1.7e308));
    }

    // Diagonalise; returns the number of sweeps run.  Afterwards X holds the
    // (nearly) diagonal matrix and v the eigenvector row.  With v_preset the
    // sweeps start from the basis already in v (see rotate_into_stored);
    // otherwise from the identity.  A sweep runs only while some off-diagonal
    // entry exceeds tol = tolrel ||W||_F; nrm2 = ||W||_F^2 as summed.
    //
    // theta > 0 lets the sweeps end earlier, for callers that rebuild with
    // project(): that takes the remaining off-diagonal part to first order.  With
    // A = diag(l) + F the second-order term of P(A) is sum over k of F_ik F_kj
    // f[l_i, l_k, l_j], f = max(., 0), whose divided difference is at most
    // 1 / sqrt((|l_i| + |l_k|)(|l_k| + |l_j|)): with G_ij = |F_ij| / sqrt(|l_i| +
    // |l_j|) the term is at most |G|_F^2 = 2 sum over i < j of F_ij^2 / (|l_i| +
    // |l_j|).  That bounds this term only; of the whole error the sum was an
    // estimate from above in float64 replays (never below it on random blocks of
    // order 5..100 and on the blocks of banded, block-arrow and batched solves,
    // 1.02 to 5 times it in half of them).  The sweeps end once the sum is at most
    // theta ||W||_F.  In a solve whose clique blocks move little between
    // iterations this takes one sweep or none from the previous iteration's
    // eigenvectors, where reaching tol takes two or three.
    //
    // With LW < 32 the warp serves 32 / LW cliques, one per group of LW lanes;
    // the sweep loop runs while any group still sweeps, and a group that has
    // stopped (or is inactive) goes through the remaining rounds with every
    // rotation skipped (threshold +inf): its storage order returns to the
    // identity after each sweep and its matrix and V stay as they were, so each
    // clique's result is the one it gets alone.
    template <bool WIDE = true>
    __device__ int run(double tolrel, T nrm2, int max_sweeps, int lane, float theta = 0.0f, bool v_preset = false,
                       bool active = true) {
        T fro, sc;
        norm<WIDE>(nrm2, active, lane, fro, sc, theta);
        const T tol = T(tolrel) * fro;
        const T noise = tol * T(2 * S);  // 4 S u ||W||_F when tol = 2 u ||W||_F
        if (!v_preset) {
#pragma unroll
            for (int j = 0; j < S; ++j) v[j] = (j == lane) ? T(1) : T(0);
        }
        __syncwarp();
        int sw = 0;
        T w[S];
        T prev = T(3.0e38);
        bool go = active;
        while (true) {
            T off;
            float second;
            off_diagonal(lane, sc, off, second);
            if (go && (sw >= max_sweeps || off <= tol || (!DIAG && second <= theta) || (off <= noise && off > T(0.5) * prev)))
                go = false;  // converged, or stagnated at the rounding-noise level
            if (!__any_sync(0xffffffffu, go)) break;
            prev = off;
            if (go) ++sw;
            const T t_eff = go ? tol : T(INFINITY);
            // rounds in pairs, V (a round behind) ping-ponging between v and w (R = S - 1 is odd)
            round<0, false>(t_eff, sc, lane, v, w);
#pragma unroll 1
            for (int r = 1; r + 1 < R; r += 2) {
                round<1, true>(t_eff, sc, lane, v, w);
                round<0, true>(t_eff, sc, lane, w, v);
            }
            rotate_v<0>(v, w);
#pragma unroll
            for (int j = 0; j < S; ++j) v[j] = w[j];
            __syncwarp();  // the table is read before the next sweep writes it
        }
        return sw;
    }

    __device__ __forceinline__ void eigenvalues_to(T* lam_out, int s, int lane) const {
        // only valid before project()
        if (lane < s) lam_out[lane] = X[lane * LDA + lane];
    }

    // After run(): P(W) to first order in the off-diagonal part that is left,
    //   V (max(L, 0) + Gamma o F) V^T,  Gamma_ij = (f(l_i) - f(l_j)) / (l_i - l_j), f = max(., 0)
    // (Daleckii and Krein 1965): Gamma is 1 between positive diagonal entries,
    // 0 between others of one sign, and max(l_i, l_j) / (|l_i| + |l_j|) across.
    // Left in Y, entry (a, b) at Y[b LDA + a] (projected()).
    __device__ __forceinline__ void project(int lane) {
        if (DIAG) {  // V max(L, 0) V^T
            T w[S];
#pragma unroll
            for (int i = 0; i < S; ++i) {
                const T l = X[i * (LDA + 1)];
                w[i] = v[i] * (l > T(0) ? l : T(0));
            }
            __syncwarp();
            if (lane < S) row_st(X + lane * LDA, v);
            __syncwarp();
            dots(w, X, Y, lane);
            __syncwarp();
            return;
        }
#pragma unroll
        for (int t = 0; t < NS; ++t) {
            if (bI[t] < 0) continue;
            const int r0 = 2 * bI[t], c0 = 2 * bJ[t];
            T b[4];
            block_ld(t, b);
            const T lr[2] = {X[r0 * (LDA + 1)], X[(r0 + 1) * (LDA + 1)]};
            const T lc[2] = {X[c0 * (LDA + 1)], X[(c0 + 1) * (LDA + 1)]};
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const T li = lr[e & 1], lj = lc[e >> 1], hi = fmax(li, lj), lo = fmin(li, lj);
                T m = lo > T(0) ? b[e] : (hi > T(0) ? b[e] * gamma_across(hi, hi - lo) : T(0));
                if (t == 0 && lane < K && (e == 0 || e == 3)) m = li > T(0) ? li : T(0);
                const int i = r0 + (e & 1), j = c0 + (e >> 1);
                Y[i * LDA + j] = m;
                Y[j * LDA + i] = m;
            }
        }
        __syncwarp();
        dots(v, Y, X, lane);  // X[j][a] = (V M)_{aj}
        T w[S];
        const int row = lane < S ? lane : S - 1;
#pragma unroll
        for (int j = 0; j < S; ++j) w[j] = X[j * LDA + row];  // this lane's own entries
        __syncwarp();
        if (lane < S) row_st(X + lane * LDA, v);
        __syncwarp();
        dots(w, X, Y, lane);  // Y[b][a] = (V M V^T)_{ab}
        __syncwarp();
    }
    // hi / d for 0 < hi <= d
    __device__ __forceinline__ static float gamma_across(float hi, float d) {
        return d > 1.0e-37f ? hi * rcp_ftz(d) : 1.0f;
    }
    // F is at most about 1e-8 ||W||_F here, so 1e-14 of the quotient is enough
    __device__ __forceinline__ static double gamma_across(double hi, double d) {
        const float f = float(d);
        if (!(f > 1.0e-30f && f < 1.0e30f)) return hi / d;
        const double y = double(rcp_ftz(f));
        return hi * fma(y, fma(-d, y, 1.0), y);
    }
    __device__ __forceinline__ T projected(int a, int b) const { return Y[b * LDA + a]; }
};

// ---------------------------------------------------------------------------
// Algorithm 1, projection and multiplier step for every clique in `list`:
//   W = H_k x - lambda_k / rho,  x_k <- P(W),  lambda_k <- lambda_k + rho (x_k - H_k x)
// (Eqs. XkUpdate, LambdakUpdate).  x comes from k_xupd (pa.x_ready, the
// default) or is formed here on the clique's entries,
//   x_e = t_e - (A^T y)_e / D_e (Appendix A, Eq. KKTflops_s1),
// the first clique covering an entry storing it.  That clique also adds the
// entry's term of <c, x>.  Per-block sums of the stopping test (Eq.
// PrimalConsensusResidual and eps_lambda) go to the partial table:
//   |x_k - H_k x|^2, |x_k|^2, |H_k x|^2, |x_k - x_k_old|^2, |lambda_k|^2, <c, x>.
template <typename T, int S, bool UNROLLED>
__global__ void __launch_bounds__(32 * proj_max_warps(S, sizeof(T) == 4)) k_project_primal(Dev d, const int4* __restrict__ list, int nlist, ProjArgs pa,
                                                         FinishArgs fa) {
    constexpr int LW = proj_lanes(S), G = 32 / LW;  // lanes per clique, cliques per warp
    using J = BLJacobi<T, S, LW, UNROLLED>;
    extern __shared__ __align__(16) unsigned char smem[];
    const bool stop = stopped(d);
    const int lane = (threadIdx.x & 31) % LW, grp = (threadIdx.x & 31) / LW;  // lane within its group
    const int warp = threadIdx.x >> 5, wpb = blockDim.x >> 5;
    J jac;
    jac.bind(smem + (warp * G + grp) * J::bytes, lane);
    if (stop) return;
    T* xk = reinterpret_cast<T*>(d.ck0);
    T* lam = reinterpret_cast<T*>(d.ck1);
    T* vc = reinterpret_cast<T*>(d.vcache);
    const bool warm = pa.warm_start && (d.ctl[CTL_ITER] % pa.restart) != 0;
    double acc[6] = {0, 0, 0, 0, 0, 0};
    for (int li0 = (blockIdx.x * wpb + warp) * G; li0 < nlist; li0 += gridDim.x * wpb * G) {
        // group grp takes clique li0 + grp; a group past the list or on a
        // frozen clique is inactive: it touches no state and skips every rotation
        const int li = li0 + grp;
        const int4 rec = __ldg(list + (li < nlist ? li : li0));
        const int k = rec.x, off = rec.z, npk0 = li < nlist ? rec.y * (rec.y + 1) / 2 : 0;
        const bool active = li < nlist && !(d.comp_mode && d.comp_done[rec.w]);
        const double rho = d.rho[d.comp_mode ? rec.w : 0], ir = d.irho[d.comp_mode ? rec.w : 0];
        T nrm = T(0);
        T hx[J::MAXE];
        double cx = 0.0;
        T rho_t, irho;
        int s, npk;
        // The penalty and the clique's activity are on their way while the
        // entries load (a frozen clique's loads are dropped).
        auto settle = [&]() {
            s = active ? rec.y : 0;
            npk = s * (s + 1) / 2;
            rho_t = T(rho);
            irho = T(ir);
            jac.clear(lane, s);
        };
        if (pa.x_ready) {  // every load of this lane's entries issued before its use: indices, then values
            int ent[J::MAXE];
            T lm[J::MAXE];
            double xe[J::MAXE], ce[J::MAXE];
#pragma unroll
            for (int e = 0; e < J::MAXE; ++e) {
                const int f = lane + LW * e;
                const bool ok = f < npk0;
                ent[e] = ok ? __ldg(d.gmap + off + f) : -1;
                lm[e] = ok ? lam[off + f] : T(0);
                ce[e] = ok && __ldg(d.owner + off + f) != 0 ? 1.0 : 0.0;
            }
#pragma unroll
            for (int e = 0; e < J::MAXE; ++e) {
                xe[e] = ent[e] >= 0 ? d.x[ent[e]] : 0.0;
                if (ce[e] != 0.0) ce[e] = __ldg(d.c + ent[e]);
            }
            settle();
#pragma unroll
            for (int e = 0; e < J::MAXE; ++e) {
                const int f = lane + LW * e;
                hx[e] = T(xe[e]);
                if (f < npk) {
                    const int ab = packed_ab(f, s), a = ab >> 8, b = ab & 255;
                    cx += (a == b ? ce[e] : 2.0 * ce[e]) * xe[e];
                    const T w = hx[e] - lm[e] * irho;
                    jac.put(a, b, w);
                    nrm += (a == b ? T(1) : T(2)) * w * w;
                }
            }
        } else {
            settle();
#pragma unroll
            for (int e = 0; e < J::MAXE; ++e) {
                const int f = lane + LW * e;
                hx[e] = T(0);
                if (f < npk) {
                    const int ab = packed_ab(f, s), a = ab >> 8, b = ab & 255;
                    // read-only loads (__ldg): free to move past this kernel's stores
                    const int ent = __ldg(d.gmap + off + f);
                    const bool own = __ldg(d.owner + off + f) != 0;
                    double aty = 0.0;
                    const int q0 = __ldg(d.at_ptr + ent), q1 = __ldg(d.at_ptr + ent + 1);
#pragma unroll 8
                    for (int q = q0; q < q1; ++q) aty += __ldg(d.at_val + q) * __ldg(d.y + __ldg(d.at_col + q));
                    const double xe = __ldg(d.t + ent) - __ldg(d.dinv + ent) * aty;
                    if (own) {
                        d.x[ent] = xe;
                        cx += __ldg(d.wgt + ent) * __ldg(d.c + ent) * xe;
                    }
                    hx[e] = T(xe);
                    const T w = hx[e] - lam[off + f] * irho;
                    jac.put(a, b, w);
                    nrm += (a == b ? T(1) : T(2)) * w * w;
                }
            }
        }
        nrm = group_sum(nrm, LW);
        const double cxk = group_sum(cx, LW);
        __syncwarp();
        if (warm) jac.rotate_into_stored(vc + d.vv_off[k], s, lane);
        jac.template run<false>(pa.tolrel, nrm, pa.max_sweeps, lane, UNROLLED ? 0.0f : float(kThetaSolve * pa.tolrel), warm, active);
        if (pa.warm_start) jac.store_basis(vc + d.vv_off[k], s, lane);
        if (UNROLLED && d.estore) {  // the reverse pass takes the eigenvectors and eigenvalues from here
            const int slot = d.ctl[CTL_ITER];
            if (slot < d.estore_count) {
                T* rec = reinterpret_cast<T*>(d.estore) + 2 * ((size_t)slot * d.nd + off);
                jac.store_basis(rec, s, lane);
                jac.eigenvalues_to(rec + s * s, s, lane);
            }
        }
        T lm[J::MAXE], xo[J::MAXE];  // old state, on its way during the rebuild
#pragma unroll
        for (int e = 0; e < J::MAXE; ++e) {
            const int f = lane + LW * e;
            lm[e] = f < npk ? lam[off + f] : T(0);
            xo[e] = f < npk ? xk[off + f] : T(0);
        }
        jac.project(lane);
        // per-clique sums of the stopping test in the clique state's precision
        // (float32 values; the sums over cliques are float64)
        T p0 = 0, p1 = 0, p2 = 0, p3 = 0, p4 = 0;
#pragma unroll
        for (int e = 0; e < J::MAXE; ++e) {
            const int f = lane + LW * e;
            if (f < npk) {
                const int ab = packed_ab(f, s), a = ab >> 8, b = ab & 255;
                const T xn = jac.projected(a, b);
                const T ln = lm[e] + rho_t * (xn - hx[e]);
                xk[off + f] = xn;
                lam[off + f] = ln;
                const T w = (a == b) ? T(1) : T(2);
                const T dc = xn - hx[e], dx = xn - xo[e];
                p0 += w * dc * dc;
                p1 += w * xn * xn;
                p2 += w * hx[e] * hx[e];
                p3 += w * dx * dx;
                p4 += w * ln * ln;
            }
        }
        const double q[6] = {double(group_sum(p0, LW)), double(group_sum(p1, LW)), double(group_sum(p2, LW)),
                             double(group_sum(p3, LW)), double(group_sum(p4, LW)), cxk};
        if (d.comp_mode) {  // per-clique row, reduced per component
            if (lane == 0 && active)
#pragma unroll
                for (int c = 0; c < 6; ++c) d.part[(size_t)k * PART_COLS + c] = q[c];
        } else {
#pragma unroll
            for (int c = 0; c < 6; ++c) acc[c] += q[c];
        }
        __syncwarp();
    }
    if (d.comp_mode) return;
#pragma unroll
    for (int c = 0; c < 6; ++c)
        for (int o = LW; o < 32; o <<= 1) acc[c] += __shfl_xor_sync(0xffffffffu, acc[c], o);  // over the groups
    const int cols[6] = {0, 1, 2, 3, 4, 5};
    block_partial_row<6>(acc, d.part, pa.row_off + blockIdx.x, cols);
    if (fa.enabled && last_block_single_writer(d)) finish_primal_block(d, fa);
}

// Algorithm 2, z-step (Eq. zkUpdate): z_k <- P(v_k - lambda_k / rho);
// part[k][5] = |z_k - z_k_old|^2 (for eps_lambda).
template <typename T, int S>
__global__ void __launch_bounds__(32 * proj_max_warps(S, sizeof(T) == 4)) k_project_dual(Dev d, const int4* __restrict__ list, int nlist, ProjArgs pa) {
    constexpr int LW = proj_lanes(S), G = 32 / LW;  // lanes per clique, cliques per warp
    using J = BLJacobi<T, S, LW>;
    extern __shared__ __align__(16) unsigned char smem[];
    const bool stop = stopped(d);
    const int lane = (threadIdx.x & 31) % LW, grp = (threadIdx.x & 31) / LW;  // lane within its group
    const int warp = threadIdx.x >> 5, wpb = blockDim.x >> 5;
    J jac;
    jac.bind(smem + (warp * G + grp) * J::bytes, lane);
    if (stop) return;
    T* z = reinterpret_cast<T*>(d.ck0);
    const T* v = reinterpret_cast<const T*>(d.ck1);
    const T* lam = reinterpret_cast<const T*>(d.ck2);
    T* vc = reinterpret_cast<T*>(d.vcache);
    const bool warm = pa.warm_start && (d.ctl[CTL_ITER] % pa.restart) != 0;
    double acc[1] = {0};
    for (int li0 = (blockIdx.x * wpb + warp) * G; li0 < nlist; li0 += gridDim.x * wpb * G) {
        // group grp takes clique li0 + grp; a group past the list or on a
        // frozen clique is inactive: it touches no state and skips every rotation
        const int li = li0 + grp;
        const int4 rec = __ldg(list + (li < nlist ? li : li0));
        const int k = rec.x, off = rec.z, npk0 = li < nlist ? rec.y * (rec.y + 1) / 2 : 0;
        const bool active = li < nlist && !(d.comp_mode && d.comp_done[rec.w]);
        const double ir = d.irho[d.comp_mode ? rec.w : 0];
        T nrm = T(0);
        T zo[J::MAXE];
        T vv[J::MAXE], lm[J::MAXE];
#pragma unroll
        for (int e = 0; e < J::MAXE; ++e) {
            const int f = lane + LW * e;
            vv[e] = f < npk0 ? v[off + f] : T(0);
            lm[e] = f < npk0 ? lam[off + f] : T(0);
            zo[e] = f < npk0 ? z[off + f] : T(0);
        }
        const int s = active ? rec.y : 0, npk = s * (s + 1) / 2;
        const T irho = T(ir);
        jac.clear(lane, s);
        {
#pragma unroll
            for (int e = 0; e < J::MAXE; ++e) {
                const int f = lane + LW * e;
                if (f < npk) {
                    const int ab = packed_ab(f, s), a = ab >> 8, b = ab & 255;
                    const T w = vv[e] - lm[e] * irho;
                    jac.put(a, b, w);
                    nrm += (a == b ? T(1) : T(2)) * w * w;
                }
            }
        }
        nrm = group_sum(nrm, LW);
        __syncwarp();
        if (warm) jac.rotate_into_stored(vc + d.vv_off[k], s, lane);
        jac.template run<false>(pa.tolrel, nrm, pa.max_sweeps, lane, float(kThetaSolve * pa.tolrel), warm, active);
        if (pa.warm_start) jac.store_basis(vc + d.vv_off[k], s, lane);
        jac.project(lane);
        T p0 = 0;  // in the clique state's precision; float64 across cliques
#pragma unroll
        for (int e = 0; e < J::MAXE; ++e) {
            const int f = lane + LW * e;
            if (f < npk) {
                const int ab = packed_ab(f, s), a = ab >> 8, b = ab & 255;
                const T zn = jac.projected(a, b);
                const T dz = zn - zo[e];
                z[off + f] = zn;
                p0 += (a == b ? T(1) : T(2)) * dz * dz;
            }
        }
        const double q0 = double(group_sum(p0, LW));
        if (d.comp_mode) {
            if (lane == 0 && active) d.part[(size_t)k * PART_COLS + 5] = q0;
        } else {
            acc[0] += q0;
        }
        __syncwarp();
    }
    if (d.comp_mode) return;
    for (int o = LW; o < 32; o <<= 1) acc[0] += __shfl_xor_sync(0xffffffffu, acc[0], o);  // over the groups
    const int cols[1] = {5};
    block_partial_row<1>(acc, d.part, pa.row_off + blockIdx.x, cols);
}

// Algorithm 3, cone step on the s block (Eqs. HsdeStep2-3) with the pieces of
// the affine step that live on clique entries (Appendix B, Eqs.
// ThirBlkFlops_s2 and AppendixEqSigma2, then Eq. MatrixInverseResult with
// zeta_hat_s = H zeta_hat_x / 2, zeta_hat_t = -H zeta_hat_x / 2):
//   sigma_12 = (nu_12 - nu_22 + H sigma_11)/2,  sigma_22 = nu_22 - H sigma_11 + sigma_12
//   u_hat_s = sigma_12 - gamma zeta_hat_s,      u_hat_t = sigma_22 - gamma zeta_hat_t
//   u_s <- P(u_hat_s - v_z),  v_z <- v_z - u_hat_s + u_s,  u_t <- u_hat_t
// with nu_12 = u_s + v_z, nu_22 = u_t.  Partial sums for eps_c (Eq.
// HSDEconsensusResidual): |u_s - H u_x|^2, |u_s|^2, |H u_x|^2, |v_z - u_t|^2,
// |v_z|^2, |u_t|^2, where u_x = sigma_11 - gamma zeta_hat_x.
// Registers bound how many warps an SM holds, and with many cliques the time: two
// blocks an SM at orders up to 4 and in float at 20 and 24, and an epilogue of one entry at
// a time where it would take the registers of the sweeps (8,000 cliques: order 7
// 137 -> 124 us an iteration, order 20 524 -> 478, order 21 681 -> 571, order 24
// 719 -> 654).
template <typename T, int S>
__global__ void __launch_bounds__(32 * proj_max_warps(S, sizeof(T) == 4), S <= 4 || (sizeof(T) == 4 && (S == 20 || S == 24)) ? 2 : 1) k_project_hsde(Dev d, const int4* __restrict__ list, int nlist, ProjArgs pa) {
    constexpr int LW = proj_lanes(S), G = 32 / LW;  // lanes per clique, cliques per warp
    using J = BLJacobi<T, S, LW>;
    extern __shared__ __align__(16) unsigned char smem[];
    const bool stop = stopped(d);
    const int lane = (threadIdx.x & 31) % LW, grp = (threadIdx.x & 31) / LW;  // lane within its group
    const int warp = threadIdx.x >> 5, wpb = blockDim.x >> 5;
    J jac;
    jac.bind(smem + (warp * G + grp) * J::bytes, lane);
    if (stop) return;
    T* us = reinterpret_cast<T*>(d.ck0);
    T* vz = reinterpret_cast<T*>(d.ck1);
    T* ut = reinterpret_cast<T*>(d.ck2);
    T* vc = reinterpret_cast<T*>(d.vcache);
    const bool warm = pa.warm_start && (d.ctl[CTL_ITER] % pa.restart) != 0;
    double acc[6] = {0, 0, 0, 0, 0, 0};
    for (int li0 = (blockIdx.x * wpb + warp) * G; li0 < nlist; li0 += gridDim.x * wpb * G) {
        // group grp takes clique li0 + grp; a group past the list or on a
        // frozen clique is inactive: it touches no state and skips every rotation
        const int li = li0 + grp;
        const int4 rec = __ldg(list + (li < nlist ? li : li0));
        const int k = rec.x, off = rec.z;
        const bool active = li < nlist && !(d.comp_mode && d.comp_done[rec.w]);
        const double gamma = hs_gamma_c(d, rec.w);
        const int s = active ? rec.y : 0, npk = s * (s + 1) / 2;
        jac.clear(lane, s);
        T nrm = T(0);
        {
            int ent[J::MAXE];
            T cu[J::MAXE], cv[J::MAXE], ct[J::MAXE];
#pragma unroll
            for (int e = 0; e < J::MAXE; ++e) {
                const int f = lane + LW * e;
                const bool ok = f < npk;
                ent[e] = ok ? __ldg(d.gmap + off + f) : 0;
                cu[e] = ok ? us[off + f] : T(0);
                cv[e] = ok ? vz[off + f] : T(0);
                ct[e] = ok ? ut[off + f] : T(0);
            }
#pragma unroll
            for (int e = 0; e < J::MAXE; ++e) {
                const int f = lane + LW * e;
                const double hs = d.s11[ent[e]], zs = 0.5 * __ldg(d.zhx + ent[e]);
                if (f < npk) {
                    const int ab = packed_ab(f, s), a = ab >> 8, b = ab & 255;
                    const double u_s = cu[e], v_z = cv[e], u_t = ct[e];
                    const double s12 = 0.5 * (u_s + v_z - u_t + hs);
                    const double uh_s = s12 - gamma * zs;
                    const T w = T(uh_s - v_z);
                    jac.put(a, b, w);
                    nrm += (a == b ? T(1) : T(2)) * w * w;
                }
            }
        }
        nrm = group_sum(nrm, LW);
        __syncwarp();
        if (warm) jac.rotate_into_stored(vc + d.vv_off[k], s, lane);
        jac.template run<false>(pa.tolrel, nrm, pa.max_sweeps, lane, float(kThetaSolve * pa.tolrel), warm, active);
        if (pa.warm_start) jac.store_basis(vc + d.vv_off[k], s, lane);
        jac.project(lane);
        double p[6] = {0, 0, 0, 0, 0, 0};
constexpr int EU = (S <= 8 || S == 20 || S == 24) ? 1 : 4;
#pragma unroll EU
        for (int f = lane; f < npk; f += LW) {
            const int ab = packed_ab(f, s), a = ab >> 8, b = ab & 255;
            const int ent = __ldg(d.gmap + off + f);
            const double hs = d.s11[ent];
            const double zx = __ldg(d.zhx + ent), zs = 0.5 * zx;
            const double u_s = us[off + f], v_z = vz[off + f], u_t = ut[off + f];
            const double s12 = 0.5 * (u_s + v_z - u_t + hs);
            const double s22 = u_t - hs + s12;
            const T uhs = T(s12 - gamma * zs);
            const T utn = T(s22 + gamma * zs);
            const T hux = T(hs - gamma * zx);
            const T un = jac.projected(a, b);
            const T vn = T(v_z) - uhs + un;
            us[off + f] = un;
            vz[off + f] = vn;
            ut[off + f] = utn;
            const double w = (a == b) ? 1.0 : 2.0;
            const double d1 = double(un) - double(hux);
            const double d2 = double(vn) - double(utn);
            p[0] += w * d1 * d1;
            p[1] += w * double(un) * double(un);
            p[2] += w * double(hux) * double(hux);
            p[3] += w * d2 * d2;
            p[4] += w * double(vn) * double(vn);
            p[5] += w * double(utn) * double(utn);
        }
        double q[6];
#pragma unroll
        for (int c = 0; c < 6; ++c) q[c] = group_sum(p[c], LW);
        if (d.comp_mode) {  // per-clique row, reduced per component
            if (lane == 0 && active)
#pragma unroll
                for (int c = 0; c < 6; ++c) d.part[(size_t)k * PART_COLS + c] = q[c];
        } else {
#pragma unroll
            for (int c = 0; c < 6; ++c) acc[c] += q[c];
        }
        __syncwarp();
    }
    if (d.comp_mode) return;
#pragma unroll
    for (int c = 0; c < 6; ++c)
        for (int o = LW; o < 32; o <<= 1) acc[c] += __shfl_xor_sync(0xffffffffu, acc[c], o);  // over the groups
    const int cols[6] = {0, 1, 2, 3, 4, 5};
    block_partial_row<6>(acc, d.part, pa.row_off + blockIdx.x, cols);
}

// Standalone projection of packed blocks (the C ABI's cdsdp_psd_project).
template <typename T, int S>
__global__ void __launch_bounds__(128) k_project_standalone(int p, const int* __restrict__ off_arr,
                                                             const int* __restrict__ size_arr, const T* __restrict__ W,
                                                             T* X, T* eig, const int* __restrict__ voff, T* Vout,
                                                             const int* __restrict__ vvoff, double tolrel,
                                                             int max_sweeps) {
    using J = BLJacobi<T, S>;
    extern __shared__ __align__(16) unsigned char smem[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, wpb = blockDim.x >> 5;
    J jac;
    jac.bind(smem + warp * J::bytes, lane);
    for (int k = blockIdx.x * wpb + warp; k < p; k += gridDim.x * wpb) {
        const int s = size_arr[k];
        if (s > S || s < 1) continue;  // warp-uniform
        const int off = off_arr[k], npk = s * (s + 1) / 2;
        jac.clear(lane, s);
        T nrm = T(0);
        for (int f = lane; f < npk; f += 32) {
            const int ab = packed_ab(f, s), a = ab >> 8, b = ab & 255;
            const T w = W[off + f];
            jac.put(a, b, w);
            nrm += (a == b ? T(1) : T(2)) * w * w;
        }
        nrm = warp_sum(nrm);
        __syncwarp();
        // eigenvalues or vectors asked for: diagonalise to the threshold
        jac.run(tolrel, nrm, max_sweeps, lane, eig || Vout ? 0.0f : float(kThetaSolve * tolrel));
        if (eig) jac.eigenvalues_to(eig + voff[k], s, lane);
        if (Vout && lane < s) {
#pragma unroll
            for (int col = 0; col < S; ++col)
                if (col < s) Vout[vvoff[k] + col * s + lane] = jac.v[col];
        }
        __syncwarp();
        jac.project(lane);
        for (int f = lane; f < npk; f += 32) {
            const int ab = packed_ab(f, s), a = ab >> 8, b = ab & 255;
            X[off + f] = jac.projected(a, b);
        }
        __syncwarp();
    }
}

}  // namespace cdsdp_dev

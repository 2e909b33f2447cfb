// libsbp 3-D operator kernels: one curvilinear block of n1 x n2 x n3 nodes (the d = 3 form of
// Sec. 3.3, 4.3-4.7 and 5).  A leapfrog step is three kernel families:
//   k3_flux  -- the mixed fluxes q_ij = sum_{k != i} c_ijkl D_k u_l (9 fields) from u^n;
//   k3_lines -- the ends of every grid line of the three directions: closure rows of D_ii^FC and D_i q_i, and the
//               SATs of the two faces there (k3_face forms their fields along the face first), for the first rows
//               from each face, as partial sums;
//   k3_div   -- r_j = sum_i D_i q_ij + sum_i D_ii^FC(c_ijil) u_l with the interior rows of the other
//               directions on top of the partial sums, then the leapfrog store (MODE 0: increment form,
//               d = du + dt^2 w r, un = u + d; MODE 1: out = w r).
// Layout: every scalar field is [n3][n2][pitch] in the arithmetic type T, pitch = n1 rounded up
// to 128 bytes; field f of a group starts at f * fs (fs = n3 * n2 * pitch).
//   cm: 27 fields, M^{ik}_{jl} = c_ijkl for the pairs (i, k) = (1,2), (1,3), (2,3), field 9p + 3j + l
//       (the other ordering is its transpose: c_kjil = c_ilkj by major symmetry);
//   cd: 18 fields, c_ijil of direction i as a symmetric 3 x 3 (jl = 11 12 13 22 23 33), field 6i + s;
//   w : 1 / (rho J).
#pragma once
#include <utility>

#include "sbp_device.cuh"

namespace sbp3 {
using namespace sbp;

constexpr int BC_DISPLACEMENT = 0, BC_TRACTION = 1;

struct Grid3 {
    int n[3];               // nodes along x1, x2, x3
    long long s[3];         // element strides along x1, x2, x3 (1, pitch, n2 * pitch)
    long long fs;           // field stride (elements)
    double ih[3];           // 1 / h_i
};

__device__ __forceinline__ int sym3(int j, int l) {
    // index of (j, l) in 11 12 13 22 23 33
    const int a = j < l ? j : l, b = j < l ? l : j;
    return a == 0 ? b : (a == 1 ? 2 + b : 5);
}
// pair index of (i, k), i < k: (0,1) -> 0, (0,2) -> 1, (1,2) -> 2
__host__ __device__ __forceinline__ constexpr int pair3(int i, int k) { return i + k - 1; }

template <typename T> __device__ __forceinline__ T ldg(const T* p) { return __ldg(p); }

// c_ijkl at element offset o from the stored 45 fields
template <typename T>
__device__ __forceinline__ T cfull(const T* __restrict__ cm, const T* __restrict__ cd, long long fs, int i, int j,
                                   int k, int l, long long o) {
    if (i == k) return ldg(cd + (long long)(6 * i + sym3(j, l)) * fs + o);
    if (i < k) return ldg(cm + (long long)(9 * pair3(i, k) + 3 * j + l) * fs + o);
    return ldg(cm + (long long)(9 * pair3(k, i) + 3 * l + j) * fs + o);
}

// ------------------------------------------------------------------ narrow D_xx^FC for 3 components
// r_j += h^2 sum_l D_xx^FC(b_jl) u_l along one grid line; u(l, t) and b(s, t) read index t of
// the line, b symmetric with s = sym3(j, l).  Closure rows come from the coefficient table.  An
// interior row is sum_m E_m(i) (u_{i+m} - u_i) + E_m(i-m) (u_{i-m} - u_i) with the edge weights
// E_m(i) = sum_t e_{m,t} b_{i+t}; collecting the terms of each b_{i+k} (k = -Q..Q) gives
//   h^2 D_xx(b) u |_i = sum_k b_{i+k} L_k(u),  L_k(u) = sum_m e_{m,k} (u_{i+m} - u_i) + e_{m,k+m} (u_{i-m} - u_i),
// so every b value of the window is read once and the e's fold into compile-time constants.
template <int O, typename T> __device__ __forceinline__ T edge_wT(int m, int kk) {
    return Edge<O>::template e<T>(m, [&](int q) { return q == kk ? T(1) : T(0); });
}

// Closure rows of D_xx^FC, unrolled at compile time.  Row ROW of the table is a list of terms
// c_t b(k_t) u(j_t); grouping them by k gives r_j += sum_k sum_l b_jl(k) V_k(u_l) with
// V_k(u) = sum_{t: k_t = k} c_t u(j_t), so that every c_t, j_t, k_t is a constant and the window of u
// (NCLOSJ columns) and each column of b are read once for all the rows (k3_lines).
namespace tab {
#define SBP_TABLE static constexpr
#include "sbp_tables.inc"
#undef SBP_TABLE
}  // namespace tab

template <int O> struct CTab;
#define SBP3_CTAB(O)                                                                                   \
    template <> struct CTab<O> {                                                                       \
        static constexpr int NCLOS = SBP##O##_NCLOS, NJ = SBP##O##_NCLOSJ;                             \
        static constexpr const int* start = tab::sbp##O##_CLOS_START;                                  \
        static constexpr const int* cj = tab::sbp##O##_CLOS_J;                                         \
        static constexpr const int* ck = tab::sbp##O##_CLOS_K;                                         \
        static constexpr const double* cc = tab::sbp##O##_CLOS_C;                                      \
    };
SBP3_CTAB(2)
SBP3_CTAB(4)
SBP3_CTAB(6)
#undef SBP3_CTAB

template <int O> constexpr bool clos_has_k(int row, int k) {
    for (int t = CTab<O>::start[row]; t < CTab<O>::start[row + 1]; ++t)
        if (CTab<O>::ck[t] == k) return true;
    return false;
}

// rr[ROW - R0] += the terms of column K of the closure row ROW; bk: the column's six coefficients
template <int O, int ROW, int K, typename T, int W, int... I>
__device__ __forceinline__ void clos_term(const T (&uw)[3][W], const T bk[6], T rr[3], std::integer_sequence<int, I...>) {
    if constexpr (clos_has_k<O>(ROW, K)) {
        constexpr int T0 = CTab<O>::start[ROW];
        T V[3] = {T(0), T(0), T(0)};
        (
            [&] {
                if constexpr (CTab<O>::ck[T0 + I] == K) {
                    constexpr int j = CTab<O>::cj[T0 + I];
                    const T c = T(CTab<O>::cc[T0 + I]);
                    V[0] += c * uw[0][j];
                    V[1] += c * uw[1][j];
                    V[2] += c * uw[2][j];
                }
            }(),
            ...);
        rr[0] += bk[0] * V[0] + bk[1] * V[1] + bk[2] * V[2];
        rr[1] += bk[1] * V[0] + bk[3] * V[1] + bk[4] * V[2];
        rr[2] += bk[2] * V[0] + bk[4] * V[1] + bk[5] * V[2];
    }
}
template <int O, int K, int R0, typename T, int W, int NR, int... R>
__device__ __forceinline__ void clos_column(const T (&uw)[3][W], const T bk[6], T (&rr)[NR][3], std::integer_sequence<int, R...>) {
    (clos_term<O, R0 + R, K, T, W>(uw, bk, rr[R], std::make_integer_sequence<int, CTab<O>::start[R0 + R + 1] - CTab<O>::start[R0 + R]>()), ...);
}
// the closure rows R0 .. R0 + NR - 1 (those of them that are closure rows)
template <int O, int R0, typename T, int W, int NR, class FB, int... K>
__device__ __forceinline__ void clos_rows(const T (&uw)[3][W], FB b, T (&rr)[NR][3], std::integer_sequence<int, K...>) {
    constexpr int NC = CTab<O>::NCLOS - R0 < NR ? CTab<O>::NCLOS - R0 : NR;
    (
        [&] {
            T bk[6];
#pragma unroll
            for (int s6 = 0; s6 < 6; ++s6) bk[s6] = b(s6, K);
            clos_column<O, K, R0, T, W, NR>(uw, bk, rr, std::make_integer_sequence<int, (NC > 0 ? NC : 0)>());
        }(),
        ...);
}

template <int O, typename T, class FU, class FB>
__device__ __forceinline__ void dxx3_interior(int i, FU u, FB b, T r[3]) {
    constexpr int Q = Ord<O>::Q;
    T dp[3][Q], dm[3][Q];
#pragma unroll
    for (int l = 0; l < 3; ++l) {
        const T uc = u(l, i);
#pragma unroll
        for (int m = 1; m <= Q; ++m) {
            dp[l][m - 1] = u(l, i + m) - uc;
            dm[l][m - 1] = u(l, i - m) - uc;
        }
    }
#pragma unroll
    for (int k = -Q; k <= Q; ++k) {
        T L[3] = {T(0), T(0), T(0)};
#pragma unroll
        for (int m = 1; m <= Q; ++m) {
            const T cp = edge_wT<O, T>(m, k), cn = edge_wT<O, T>(m, k + m);
#pragma unroll
            for (int l = 0; l < 3; ++l) {
                if (cp != T(0)) L[l] += cp * dp[l][m - 1];
                if (cn != T(0)) L[l] += cn * dm[l][m - 1];
            }
        }
        const T b00 = b(0, i + k), b01 = b(1, i + k), b02 = b(2, i + k), b11 = b(3, i + k), b12 = b(4, i + k),
                b22 = b(5, i + k);
        r[0] += b00 * L[0] + b01 * L[1] + b02 * L[2];
        r[1] += b01 * L[0] + b11 * L[1] + b12 * L[2];
        r[2] += b02 * L[0] + b12 * L[1] + b22 * L[2];
    }
}

constexpr int BX = 32, BY = 8;

// element stride of direction D as a 32-bit int (a plane of the grid holds fewer than 2^31
// elements, checked at create): 1 along x1 (a compile-time constant), pitch or plane otherwise.
// Neighbour reads go through the node's own pointer plus (t - i) * stride, so interior stencil
// offsets fold into constants shared by every field.
template <int D> __device__ __forceinline__ int dstride(const Grid3& g) {
    if constexpr (D == 0) return 1;
    else return (int)g.s[D];
}

// D_D u_l (l = 0..2) at the node (index i along D), u at the node's pointer
template <typename T, int O, int D>
__device__ __forceinline__ void grad_dir(const Grid3& g, int i, const T* __restrict__ up, T gr[3]) {
    const int S = dstride<D>(g);
    const int N = g.n[D];
    const T ih = T(g.ih[D]);
#pragma unroll
    for (int l = 0; l < 3; ++l) {
        const T* p = up + l * g.fs;
        gr[l] = ih * dsum<O, T>(N, i, [&](int t) { return ldg(p + (t - i) * S); });
    }
}

template <typename T, int NV> __device__ __forceinline__ void vld(const T* p, T v[NV]) {
    if constexpr (NV == 2 && sizeof(T) == 4) {
        const float2 x = __ldg(reinterpret_cast<const float2*>(p));
        v[0] = x.x;
        v[1] = x.y;
    } else {
#pragma unroll
        for (int n = 0; n < NV; ++n) v[n] = __ldg(p + n);
    }
}
// Field access of the flux kernel: the field's base is the same for the whole grid and the node's
// offset, in bytes of type I, is 32 bits wide where the fields stay below 4 GB.  A neighbour then costs one 32-bit
// addition, shared by all the fields that are read there, where a pointer per field costs a 64-bit one for
// each of them.  160 x 151 x 144, FP32: k3_flux 140 -> 131 us (k3_div, whose offsets then take the registers that
// its rows need, 171 -> 189: it keeps pointers).
template <typename T, typename I> __device__ __forceinline__ const T* at(const T* base, I off) {
    return reinterpret_cast<const T*>(reinterpret_cast<const char*>(base) + off);
}
template <typename T, int NV, typename I> __device__ __forceinline__ void vldo(const T* base, I off, T v[NV]) {
    vld<T, NV>(at(base, off), v);
}
template <typename T, int NV> __device__ __forceinline__ void vst(T* p, const T v[NV]) {
    if constexpr (NV == 2 && sizeof(T) == 4) {
        *reinterpret_cast<float2*>(p) = make_float2(v[0], v[1]);
    } else {
#pragma unroll
        for (int n = 0; n < NV; ++n) p[n] = v[n];
    }
}

// D_D u_l of one node as a call of its own (the closure rows of the paired flux kernel)
template <typename T, int O, int D>
__device__ __noinline__ void grad_call(const Grid3& g, int i, const T* __restrict__ up, T* __restrict__ out) {
    T gr[3];
    grad_dir<T, O, D>(g, i, up, gr);
    out[0] = gr[0];
    out[1] = gr[1];
    out[2] = gr[2];
}

// ------------------------------------------------------------------ mixed fluxes
// Two x1-adjacent nodes per thread (FP32; one node in FP64).  A pair whose x1 rows are interior
// reads its x1 stencil as aligned vector windows; its x2 / x3 rows are vector loads at +-k
// strides (interior) or the general rows node by node (closure rows, the same for a whole warp).
// A pair near the x1 faces takes the general rows for everything.
template <typename T, int O, int NV, typename I>
__device__ __forceinline__ void flux_pair(const Grid3& g, int i1, int i2, int i3, const T* __restrict__ u, I ob,
                                          T gr[NV][3][3]) {
    using P = Ord<O>;
    constexpr int Q = P::Q;
    constexpr int QA = (Q + NV - 1) / NV * NV;
    constexpr int WN = NV + 2 * QA;
    const long long fs = g.fs;
    const T* up = at(u, ob);
    const bool x1int = i1 >= P::NB && i1 + NV - 1 <= g.n[0] - 1 - P::NB && i1 >= QA;
    if (x1int) {
        const T ih = T(g.ih[0]);
#pragma unroll
        for (int l = 0; l < 3; ++l) {
            T w[WN];
#pragma unroll
            for (int v = 0; v < WN / NV; ++v) vldo<T, NV>(u + l * fs, ob + I((v * NV - QA) * (int)sizeof(T)), w + v * NV);
#pragma unroll
            for (int n = 0; n < NV; ++n) {
                T acc = T(0);
#pragma unroll
                for (int k = 1; k <= Q; ++k) acc += P::template aT<T>(k - 1) * (w[QA + n + k] - w[QA + n - k]);
                gr[n][0][l] = ih * acc;
            }
        }
    } else {
#pragma unroll
        for (int n = 0; n < NV; ++n) grad_call<T, O, 0>(g, i1 + n, up + n, gr[n][0]);
    }
    auto strided = [&](auto dc, int i) {
        constexpr int D = decltype(dc)::value;
        const int N = g.n[D];
        if (i >= P::NB && i <= N - 1 - P::NB) {
            const I S = I(dstride<D>(g)) * I(sizeof(T));
            const T ih = T(g.ih[D]);
            T acc[3][NV];
#pragma unroll
            for (int l = 0; l < 3; ++l)
#pragma unroll
                for (int n = 0; n < NV; ++n) acc[l][n] = T(0);
#pragma unroll
            for (int k = 1; k <= Q; ++k) {
                const I op = ob + I(k) * S, om = ob - I(k) * S;
                const T ak = P::template aT<T>(k - 1);
#pragma unroll
                for (int l = 0; l < 3; ++l) {
                    T a[NV], b[NV];
                    vldo<T, NV>(u + l * fs, op, a);
                    vldo<T, NV>(u + l * fs, om, b);
#pragma unroll
                    for (int n = 0; n < NV; ++n) acc[l][n] += ak * (a[n] - b[n]);
                }
            }
#pragma unroll
            for (int l = 0; l < 3; ++l)
#pragma unroll
                for (int n = 0; n < NV; ++n) gr[n][D][l] = ih * acc[l][n];
        } else {
#pragma unroll
            for (int n = 0; n < NV; ++n) grad_call<T, O, D>(g, i, up + n, gr[n][D]);
        }
    };
    strided(std::integral_constant<int, 1>(), i2);
    strided(std::integral_constant<int, 2>(), i3);
}

template <typename T, int O, int NV, typename I>
__global__ void __launch_bounds__(BX * BY, 3) k3_flux(Grid3 g, const T* __restrict__ u, const T* __restrict__ cm,
                                                   T* __restrict__ q) {
    const int i1 = (blockIdx.x * BX + threadIdx.x) * NV, i2 = blockIdx.y * BY + threadIdx.y, i3 = blockIdx.z;
    if (i1 >= g.n[0] || i2 >= g.n[1]) return;
    const long long o = i1 + i2 * g.s[1] + i3 * g.s[2];
    const long long fs = g.fs;
    const T* up = u + o;
    const I ob = I(o) * I(sizeof(T));
    // the last pair of an odd row has one node: it runs alone through the general rows
    const bool full = i1 + NV - 1 < g.n[0];
    T gr[NV][3][3];                               // gr[n][k][l] = D_k u_l at node n
    if (full) {
        flux_pair<T, O, NV, I>(g, i1, i2, i3, u, ob, gr);
    } else {
#pragma unroll
        for (int n = 0; n < NV; ++n) {
            grad_call<T, O, 0>(g, i1, up, gr[n][0]);
            grad_call<T, O, 1>(g, i2, up, gr[n][1]);
            grad_call<T, O, 2>(g, i3, up, gr[n][2]);
        }
    }
    T qq[NV][3][3];
#pragma unroll
    for (int n = 0; n < NV; ++n)
#pragma unroll
        for (int i = 0; i < 3; ++i)
#pragma unroll
            for (int j = 0; j < 3; ++j) qq[n][i][j] = T(0);
#pragma unroll
    for (int p = 0; p < 3; ++p) {
        const int i = p == 2 ? 1 : 0, k = p == 0 ? 1 : 2;
#pragma unroll
        for (int j = 0; j < 3; ++j)
#pragma unroll
            for (int l = 0; l < 3; ++l) {
                T M[NV];
                if (full) {
                    vldo<T, NV>(cm + (9 * p + 3 * j + l) * fs, ob, M);
                } else {
                    M[0] = ldg(at(cm + (9 * p + 3 * j + l) * fs, ob));
#pragma unroll
                    for (int n = 1; n < NV; ++n) M[n] = T(0);
                }
#pragma unroll
                for (int n = 0; n < NV; ++n) {
                    qq[n][i][j] += M[n] * gr[n][k][l];       // c_ijkl D_k u_l
                    qq[n][k][l] += M[n] * gr[n][i][j];       // c_klij D_i u_j (major symmetry)
                }
            }
    }
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            T* qo = const_cast<T*>(at(static_cast<const T*>(q + (3 * i + j) * fs), ob));
            if (full) {
                T v[NV];
#pragma unroll
                for (int n = 0; n < NV; ++n) v[n] = qq[n][i][j];
                vst<T, NV>(qo, v);
            } else {
                *qo = qq[0][i][j];
            }
        }
}

// ------------------------------------------------------------------ divergence
// The rows that k3_lines takes: along x1 the columns outside [x1lo, x1hi) (x1lo a multiple of NV, so that
// k3_div reads its x1 windows as aligned vectors inside the row), along x2 and x3 the first and last
// line_rows<O>() planes.
template <int O> __host__ __device__ constexpr int line_rows() {
    return Ord<O>::NCLOS > Ord<O>::NCOL ? Ord<O>::NCLOS : Ord<O>::NCOL;
}
struct Box3 {
    int x1lo, x1hi;
    int rows;               // rows of the longer x1 end: max(x1lo, n1 - x1hi)
};

// x2 / x3 direction (stride S) for NV nodes: r[n][j] += ih D q_Dj + ih^2 D_xx(b) u, interior rows
template <typename T, int O, int NV>
__device__ __forceinline__ void div_int_strided(const T* __restrict__ qD, const T* __restrict__ cdD,
                                                const T* __restrict__ up, long long fs, int S, T ih, T r[NV][3]) {
    constexpr int Q = Ord<O>::Q;
#pragma unroll
    for (int j = 0; j < 3; ++j) {
        T acc[NV];
#pragma unroll
        for (int n = 0; n < NV; ++n) acc[n] = T(0);
        const T* p = qD + j * fs;
#pragma unroll
        for (int k = 1; k <= Q; ++k) {
            T a[NV], b[NV];
            vld<T, NV>(p + k * S, a);
            vld<T, NV>(p - k * S, b);
            const T ak = Ord<O>::template aT<T>(k - 1);
#pragma unroll
            for (int n = 0; n < NV; ++n) acc[n] += ak * (a[n] - b[n]);
        }
#pragma unroll
        for (int n = 0; n < NV; ++n) r[n][j] += ih * acc[n];
    }
    T dp[3][Q][NV], dm[3][Q][NV];
#pragma unroll
    for (int l = 0; l < 3; ++l) {
        T uc[NV];
        vld<T, NV>(up + l * fs, uc);
#pragma unroll
        for (int m = 1; m <= Q; ++m) {
            T a[NV], b[NV];
            vld<T, NV>(up + l * fs + m * S, a);
            vld<T, NV>(up + l * fs - m * S, b);
#pragma unroll
            for (int n = 0; n < NV; ++n) {
                dp[l][m - 1][n] = a[n] - uc[n];
                dm[l][m - 1][n] = b[n] - uc[n];
            }
        }
    }
    const T ih2 = ih * ih;
#pragma unroll
    for (int k = -Q; k <= Q; ++k) {
        T L[3][NV];
#pragma unroll
        for (int l = 0; l < 3; ++l)
#pragma unroll
            for (int n = 0; n < NV; ++n) L[l][n] = T(0);
#pragma unroll
        for (int m = 1; m <= Q; ++m) {
            const T cp = edge_wT<O, T>(m, k), cn = edge_wT<O, T>(m, k + m);
#pragma unroll
            for (int l = 0; l < 3; ++l)
#pragma unroll
                for (int n = 0; n < NV; ++n) {
                    if (cp != T(0)) L[l][n] += cp * dp[l][m - 1][n];
                    if (cn != T(0)) L[l][n] += cn * dm[l][m - 1][n];
                }
        }
        T bb[6][NV];
#pragma unroll
        for (int s6 = 0; s6 < 6; ++s6) vld<T, NV>(cdD + s6 * fs + k * S, bb[s6]);
#pragma unroll
        for (int n = 0; n < NV; ++n) {
            r[n][0] += ih2 * (bb[0][n] * L[0][n] + bb[1][n] * L[1][n] + bb[2][n] * L[2][n]);
            r[n][1] += ih2 * (bb[1][n] * L[0][n] + bb[3][n] * L[1][n] + bb[4][n] * L[2][n]);
            r[n][2] += ih2 * (bb[2][n] * L[0][n] + bb[4][n] * L[1][n] + bb[5][n] * L[2][n]);
        }
    }
}

// the same for FP32 node pairs, in packed FP32x2 arithmetic (one instruction for both nodes)
__device__ __forceinline__ float2 p2ffma(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 p2fmul(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 p2fsub(float2 a, float2 b) { return __ffma2_rn(b, make_float2(-1.f, -1.f), a); }
__device__ __forceinline__ float2 p2s(float a) { return make_float2(a, a); }

template <int O>
__device__ __forceinline__ void div_int_strided_f2(const float* __restrict__ qD, const float* __restrict__ cdD,
                                                   const float* __restrict__ up, long long fs, int S, float ih,
                                                   float r[2][3]) {
    constexpr int Q = Ord<O>::Q;
    auto ld2 = [](const float* p) { return __ldg(reinterpret_cast<const float2*>(p)); };
    float2 R[3];
#pragma unroll
    for (int j = 0; j < 3; ++j) {
        const float* p = qD + j * fs;
        float2 acc = make_float2(0.f, 0.f);
#pragma unroll
        for (int k = 1; k <= Q; ++k)
            acc = p2ffma(p2s(Ord<O>::template aT<float>(k - 1)), p2fsub(ld2(p + k * S), ld2(p - k * S)), acc);
        R[j] = p2fmul(p2s(ih), acc);
    }
    float2 dp[3][Q], dm[3][Q];
#pragma unroll
    for (int l = 0; l < 3; ++l) {
        const float *ul = up + l * fs, *pp = ul, *pm = ul;
        const float2 uc = ld2(ul);
#pragma unroll
        for (int m = 1; m <= Q; ++m) {
            pp += S;
            pm -= S;
            dp[l][m - 1] = p2fsub(ld2(pp), uc);
            dm[l][m - 1] = p2fsub(ld2(pm), uc);
        }
    }
    const float2 ih2 = p2s(ih * ih);
    const float* ck[6];
#pragma unroll
    for (int s6 = 0; s6 < 6; ++s6) ck[s6] = cdD + s6 * fs - Q * S;
#pragma unroll
    for (int k = -Q; k <= Q; ++k) {
        float2 L[3] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
#pragma unroll
        for (int m = 1; m <= Q; ++m) {
            const float cp = edge_wT<O, float>(m, k), cn = edge_wT<O, float>(m, k + m);
#pragma unroll
            for (int l = 0; l < 3; ++l) {
                if (cp != 0.f) L[l] = p2ffma(p2s(cp), dp[l][m - 1], L[l]);
                if (cn != 0.f) L[l] = p2ffma(p2s(cn), dm[l][m - 1], L[l]);
            }
        }
        float2 bb[6];
#pragma unroll
        for (int s6 = 0; s6 < 6; ++s6) {
            bb[s6] = ld2(ck[s6]);
            ck[s6] += S;
        }
        const float2 t0 = p2ffma(bb[2], L[2], p2ffma(bb[1], L[1], p2fmul(bb[0], L[0])));
        const float2 t1 = p2ffma(bb[4], L[2], p2ffma(bb[3], L[1], p2fmul(bb[1], L[0])));
        const float2 t2 = p2ffma(bb[5], L[2], p2ffma(bb[4], L[1], p2fmul(bb[2], L[0])));
        R[0] = p2ffma(ih2, t0, R[0]);
        R[1] = p2ffma(ih2, t1, R[1]);
        R[2] = p2ffma(ih2, t2, R[2]);
    }
#pragma unroll
    for (int j = 0; j < 3; ++j) {
        r[0][j] += R[j].x;
        r[1][j] += R[j].y;
    }
}

// x1 direction for NV consecutive nodes: windows of WN = NV + 2 QA values from i1 - QA (QA = Q
// rounded up to NV, so the window loads stay vector-aligned); node n sits at window index QA + n
template <typename T, int O, int NV>
__device__ __forceinline__ void div_int_x1(const T* __restrict__ q0, const T* __restrict__ cd0,
                                           const T* __restrict__ up, long long fs, T ih, T r[NV][3]) {
    constexpr int Q = Ord<O>::Q;
    constexpr int QA = (Q + NV - 1) / NV * NV;
    constexpr int WN = NV + 2 * QA;
    auto window = [&](const T* p, T w[WN]) {
#pragma unroll
        for (int v = 0; v < WN / NV; ++v) vld<T, NV>(p - QA + v * NV, w + v * NV);
    };
#pragma unroll
    for (int j = 0; j < 3; ++j) {
        T w[WN];
        window(q0 + j * fs, w);
#pragma unroll
        for (int n = 0; n < NV; ++n) {
            T acc = T(0);
#pragma unroll
            for (int k = 1; k <= Q; ++k) acc += Ord<O>::template aT<T>(k - 1) * (w[QA + n + k] - w[QA + n - k]);
            r[n][j] += ih * acc;
        }
    }
    // narrow rows one displacement component at a time (L_k of u_l for the NV nodes, then every
    // coefficient field b_jl that multiplies u_l), so only one component's L's are live
    const T ih2 = ih * ih;
#pragma unroll
    for (int l = 0; l < 3; ++l) {
        T L[2 * Q + 1][NV];
        {
            T w[WN];
            window(up + l * fs, w);
#pragma unroll
            for (int n = 0; n < NV; ++n) {
                const T uc = w[QA + n];
#pragma unroll
                for (int k = -Q; k <= Q; ++k) {
                    T acc = T(0);
#pragma unroll
                    for (int m = 1; m <= Q; ++m) {
                        const T cp = edge_wT<O, T>(m, k), cn = edge_wT<O, T>(m, k + m);
                        if (cp != T(0)) acc += cp * (w[QA + n + m] - uc);
                        if (cn != T(0)) acc += cn * (w[QA + n - m] - uc);
                    }
                    L[k + Q][n] = acc;
                }
            }
        }
        // fields b_jl with this l: (j, l) for j = 0..2, s6 = sym3 index
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            const int s6 = j <= l ? (j == 0 ? l : (j == 1 ? 2 + l : 5)) : (l == 0 ? j : (l == 1 ? 2 + j : 5));
            T w[WN];
            window(cd0 + s6 * fs, w);
#pragma unroll
            for (int n = 0; n < NV; ++n) {
                T acc = T(0);
#pragma unroll
                for (int k = -Q; k <= Q; ++k) acc += w[QA + n + k] * L[k + Q][n];
                r[n][j] += ih2 * acc;
            }
        }
    }
}

// ------------------------------------------------------------------ boundary SATs of the faces x_m = 0, 1
//   traction:     J SAT_J = -H^-1 P_f nu c_mJkL D_k u_L              (face node only)
//   displacement: J SAT_J = H^-1 [ sum_k D_k^T (nu c_mLkJ P_f u_L) - P_f (beta d / h1) c_mJmL u_L ]
// H^-1 P_f is 1 / (h_m hw_0) at a face node; D_m^T spreads the normal term over the first NCOL
// nodes of the normal line (H^-1 D_m^T at depth t: D_m[face][t] / (h_m hw_t)); the tangential
// D_k^T stays on the face, weighted by hw_k(a') / hw_k(a).  The normal term and the penalty act along
// the line and are formed by k3_lines itself.
// Along the face the term is (H_k^-1 D_k^T H_k b)(a) of the face field b_J = c_mLkJ u_L, which the SBP property
// turns into -(D_k b)(a), less b / H_k at the low end and plus it at the high end of the line.  k3_face forms the
// two fields of every displacement face once (fields 3 t + J of its buffer, t = 0, 1 the tangential directions in
// ascending order, each [B][A] with the lower one fastest), where each of the 12 taps of a node formed them again.
struct Faces3 {
    int kind[6];            // BC_DISPLACEMENT or BC_TRACTION per face
    double beta;
    long long at[6];        // element offset of the face's fields in the face buffer
};

template <typename T, int O, int M>
__device__ __forceinline__ void face_fields(const Grid3& g, int side, int t, const T* __restrict__ u,
                                            const T* __restrict__ cm, const T* __restrict__ cd, T* __restrict__ out) {
    constexpr int A = M == 0 ? 1 : 0, B = M == 2 ? 1 : 2;
    const int na = g.n[A], nb = g.n[B];
    if (t >= na * nb) return;
    const int ib = t / na, ia = t - ib * na;
    const long long o = ia * g.s[A] + ib * g.s[B] + (side ? (g.n[M] - 1) * g.s[M] : 0);
    T uf[3];
#pragma unroll
    for (int L = 0; L < 3; ++L) uf[L] = ldg(u + L * g.fs + o);
#pragma unroll
    for (int k = 0; k < 2; ++k)
#pragma unroll
        for (int J = 0; J < 3; ++J) {
            T v = T(0);
#pragma unroll
            for (int L = 0; L < 3; ++L) v += cfull(cm, cd, g.fs, M, L, k == 0 ? A : B, J, o) * uf[L];
            out[(long long)(3 * k + J) * na * nb + t] = v;
        }
}
// one launch for the six faces (blockIdx.y; traction faces have no fields)
template <typename T, int O>
__global__ void __launch_bounds__(128) k3_face(Grid3 g, Faces3 fc, const T* __restrict__ u, const T* __restrict__ cm,
                                               const T* __restrict__ cd, T* __restrict__ ff) {
    const int f = blockIdx.y, t = blockIdx.x * 128 + threadIdx.x;
    if (fc.kind[f] != BC_DISPLACEMENT) return;
    T* out = ff + fc.at[f];
    if (f < 2) face_fields<T, O, 0>(g, f, t, u, cm, cd, out);
    else if (f < 4) face_fields<T, O, 1>(g, f - 2, t, u, cm, cd, out);
    else face_fields<T, O, 2>(g, f - 4, t, u, cm, cd, out);
}

// one interior row of direction D at a node: r_j += D_D q_Dj + D_DD^FC(c_DjDl) u_l
template <typename T, int O, int D>
__device__ __noinline__ void int_row(const Grid3& g, const T* __restrict__ qo, const T* __restrict__ cp,
                                     const T* __restrict__ up, T r[3]) {
    const int S = dstride<D>(g);
    const long long fs = g.fs;
    const T ih = T(g.ih[D]);
    T rr[3] = {T(0), T(0), T(0)};
    dxx3_interior<O, T>(0, [&](int l, int t) { return ldg(up + l * fs + t * S); },
                        [&](int s, int t) { return ldg(cp + s * fs + t * S); }, rr);
#pragma unroll
    for (int j = 0; j < 3; ++j) {
        T d = T(0);
#pragma unroll
        for (int k = 1; k <= Ord<O>::Q; ++k)
            d += Ord<O>::template aT<T>(k - 1) * (ldg(qo + j * fs + k * S) - ldg(qo + j * fs - k * S));
        r[j] += ih * d + ih * ih * rr[j];
    }
}

// The ends of the grid lines of direction D: the partial sums
//   r_j = D_D q_Dj + D_DD^FC(c_DjDl) u_l + the SATs of the face there
// of the first rows from the face (line_rows<O>(); along x1 up to x1lo, or from x1hi), which k3_div completes.
// They go to the output field.  A node near several faces gets a sum from each direction: x3's goes there, x2's and x1's
// to planes of their own (LineParts), so that one launch takes all three.
// A closure row reads NCLOSJ columns of the line, the same ones for every row of the end: a
// thread reads the columns of u, q and the 6 coefficients once (order 6: 144 loads) for all its rows,
// where a thread per node read them for each row.  The lanes of a warp lie along x1 (D = 1, 2: coalesced)
// or x2 (D = 0), where a column is one word per line: the CTA copies its lines' ends to shared memory row by row
// and writes the sums back the same way.
// A line end is taken by three warps of a CTA, a third of the rows each (orders 4 and 6): the rows are straight-line code
// that a thread runs once (order 6: 2070 FP64 instructions; order 4: 780), and small blocks have few lines (40^3: 100 warps
// of line ends per direction for 152 SMs).  With a thread for all rows of an end, in a launch per direction one after the
// other, nothing hid the latencies of loads and instruction fetches: FP64 steps were slower than with a thread per node
// (a step of 40^3, order 6: 321 us with a thread per node, 436 with a thread per end, now 199; order 4: 184, 258, 147; the
// three launches of 64 x 61 x 57, order 4: 143 us, now 64).  FP32, 160 x 151 x 144, order 6: 91 us, now 78.
constexpr int kLines = 32;                                    // line ends of a CTA
template <int O> constexpr int kLineGroups = O == 2 ? 1 : 3;      // groups of rows
template <int O> constexpr int kLineThreads = kLines * kLineGroups<O>;
// rows formed here: along x1 one more than the closure for node pairs (the alignment of x1lo)
template <typename T, int O, int D> constexpr int kLineRows = line_rows<O>() + (D == 0 && sizeof(T) == 4 ? 1 : 0);
template <typename T, int O, int D> constexpr int line_window() {      // columns that the rows read
    constexpr int RX = kLineRows<T, O, D> + Ord<O>::Q, NJ = CTab<O>::NJ, NC = Ord<O>::NCOL;
    return NJ > RX ? (NJ > NC ? NJ : NC) : (RX > NC ? RX : NC);
}
template <typename T, int O> constexpr int line_smem() { return 12 * line_window<T, O, 0>() * (kLines + 1); }

// partial sums of x2 and x1 at nodes where another direction has one in the output field (planes over all the end rows;
// see Box3 for x1's rows)
template <typename T> struct LineParts {
    T *x2, *x1;
};
// whether index i of a direction is one of the rows that k3_lines takes there
template <int O> __device__ __forceinline__ bool line_row(int i, int n) { return i < line_rows<O>() || i >= n - line_rows<O>(); }
// element of the sum j at the node e-th row from the nearer face x2 (the rows of the high face after those of the low one)
template <int O> __device__ __forceinline__ long long part_x2(const Grid3& g, int e, int j, int i1, int i3) {
    return ((long long)(e * 3 + j) * g.n[2] + i3) * g.s[1] + i1;
}
// ... r-th row from the face x1 at `side`; line: i3 n2 + i2
__device__ __forceinline__ long long part_x1(const Grid3& g, const Box3& bx, int side, int j, long long line, int r) {
    return ((long long)(side * 3 + j) * g.n[1] * g.n[2] + line) * bx.rows + r;
}

// rows R0 .. of a line end, as many as rr holds or are left: u, q and the six coefficients through uat(l, c), qat(j, c),
// b(s6, c)
template <typename T, int O, int D, int R0, int NG, class FU, class FQ, class FB>
__device__ __forceinline__ void line_end_rows(const Grid3& g, const Faces3& fc, int side, int tl, int ia, int ib, FU uat, FQ qat,
                                              FB b, const T* __restrict__ ff, T (&rr)[NG][3]) {
    using P = Ord<O>;
    constexpr int LEFT = kLineRows<T, O, D> - R0, NR = NG < LEFT ? NG : LEFT;
    constexpr int NJ = CTab<O>::NJ, W = line_window<T, O, D>();
    constexpr int A = D == 0 ? 1 : 0, B = D == 2 ? 1 : 2;
    const int na = g.n[A], nb = g.n[B], N = g.n[D], lines = na * nb;
    const T ih = T(g.ih[D]), ih2 = ih * ih;
    T uw[3][W];
#pragma unroll
    for (int l = 0; l < 3; ++l)
#pragma unroll
        for (int c = 0; c < W; ++c) uw[l][c] = uat(l, c);
#pragma unroll
    for (int r = 0; r < NG; ++r) rr[r][0] = rr[r][1] = rr[r][2] = T(0);
    clos_rows<O, R0, T, W, NG>(uw, b, rr, std::make_integer_sequence<int, NJ>());
    // rows past the closure: order 2 has one that a SAT reaches; along x1 one more may be left here by the alignment of x1lo
#pragma unroll
    for (int r = 0; r < NR; ++r)
        if (R0 + r >= P::NCLOS) dxx3_interior<O, T>(R0 + r, [&](int l, int c) { return uw[l][c]; }, b, rr[r]);
#pragma unroll
    for (int r = 0; r < NR; ++r)
#pragma unroll
        for (int j = 0; j < 3; ++j) rr[r][j] *= ih2;
    // D_D q_Dj: rows of D from the face, mirrored with the opposite sign at the high end
    const T sg = side ? -ih : ih;
    T q0[3];
#pragma unroll
    for (int j = 0; j < 3; ++j) {
        T qw[W];
#pragma unroll
        for (int c = 0; c < W; ++c) qw[c] = qat(j, c);
        q0[j] = qw[0];
#pragma unroll
        for (int r = R0; r < R0 + NR; ++r) {
            T d = T(0);
            if (r < P::NB) {
#pragma unroll
                for (int c = 0; c < P::NCOL; ++c) d += P::template dqT<T>(r, c) * qw[c];
            } else {
#pragma unroll
                for (int k = 1; k <= P::Q; ++k) d += P::template aT<T>(k - 1) * (qw[r + k] - qw[r - k]);
            }
            rr[r - R0][j] += sg * d;
        }
    }
    if constexpr (R0 < P::NCOL) {
        // v_J -> c_DJDL v_L at the face node
        T b0[6];
#pragma unroll
        for (int s6 = 0; s6 < 6; ++s6) b0[s6] = b(s6, 0);
        auto cn = [&](const T v[3], T w[3]) {
            w[0] = b0[0] * v[0] + b0[1] * v[1] + b0[2] * v[2];
            w[1] = b0[1] * v[0] + b0[3] * v[1] + b0[4] * v[2];
            w[2] = b0[2] * v[0] + b0[4] * v[1] + b0[5] * v[2];
        };
        const T ihb = ih / hweightT<O, T>(N, 0);                       // H^-1 P_f at the face node
        const T nu = side ? T(1) : T(-1);
        T v[3], w[3];
        if (fc.kind[2 * D + side] == BC_TRACTION) {
            if constexpr (R0 == 0) {
                // c_DJkL D_k u_L = q_DJ + c_DJDL D_D u_L at the face
#pragma unroll
                for (int l = 0; l < 3; ++l) {
                    v[l] = T(0);
#pragma unroll
                    for (int c = 0; c < P::NCOL; ++c) v[l] += P::template dqT<T>(0, c) * uw[l][c];
                    v[l] *= sg;
                }
                cn(v, w);
#pragma unroll
                for (int j = 0; j < 3; ++j) rr[0][j] -= ihb * nu * (q0[j] + w[j]);
            }
        } else {
            // s_J = c_DJDL u_L at the face node: spread by H^-1 D_D^T nu over NCOL rows, and the penalty
            // -H^-1 P_f (beta d / h1) s_J at the face (h1 = h hw_0)
#pragma unroll
            for (int l = 0; l < 3; ++l) v[l] = uw[l][0];
            cn(v, w);
            const T pen = T(fc.beta * 3.0) * ihb * ihb;
#pragma unroll
            for (int r = R0; r < R0 + NR && r < P::NCOL; ++r) {
                T coef = -ih2 * P::template dqT<T>(0, r);
                if (r < P::NB) coef /= P::template hwT<T>(r);
                if (r == 0) coef -= pen;
#pragma unroll
                for (int j = 0; j < 3; ++j) rr[r - R0][j] += coef * w[j];
            }
            if constexpr (R0 == 0) {
                // tangential transposes of the face fields
                const T* F = ff + fc.at[2 * D + side];
                auto tang = [&](const T* Fk, int Nk, int a, int st, T ihk) {
#pragma unroll
                    for (int j = 0; j < 3; ++j) {
                        const T* p = Fk + (long long)j * lines + tl;
                        T d = -dsum<O, T>(Nk, a, [&](int x) { return p[(long long)(x - a) * st]; });
                        if (a == 0 || a == Nk - 1) d += (a == 0 ? -p[0] : p[0]) / P::template hwT<T>(0);
                        rr[0][j] += ihb * nu * ihk * d;
                    }
                };
                tang(F, na, ia, 1, T(g.ih[A]));
                tang(F + 3LL * lines, nb, ib, na, T(g.ih[B]));
            }
        }
    }
}

// the line ends `blk` kLines .. of direction D at `side`
template <typename T, int O, int D>
__device__ __forceinline__ void line_ends(const Grid3& g, const Box3& bx, const Faces3& fc, int blk, int side,
                                          const T* __restrict__ u, const T* __restrict__ q, const T* __restrict__ cd,
                                          const T* __restrict__ ff, T* __restrict__ un, const LineParts<T>& parts, T* sm) {
    constexpr int NL = kLines, G = kLineGroups<O>, NT = NL * G;
    constexpr int RX = kLineRows<T, O, D>, WS = line_window<T, O, D>();
    constexpr int A = D == 0 ? 1 : 0, B = D == 2 ? 1 : 2;
    const int na = g.n[A], nb = g.n[B], N = g.n[D], lines = na * nb;
    const int tx = threadIdx.x % NL, group = threadIdx.x / NL, t = blk * NL + tx;
    const long long fs = g.fs;
    const int S = dstride<D>(g), Ss = side ? -S : S;
    auto face_node = [&](int line) {
        const int b = line / na;
        return (line - b * na) * g.s[A] + b * g.s[B] + (side ? (long long)(N - 1) * g.s[D] : 0);
    };
    if constexpr (D == 0) {
        // column c of field f of line n at sm[(f * WS + c) * (NL + 1) + n]; fields u, q_1j, c_1j1l
        for (int idx = threadIdx.x; idx < NL * WS; idx += NT) {
            const int n = idx / WS, c = idx - n * WS, line = blk * NL + n;
            if (line >= lines || c >= N) continue;
            const long long oc = face_node(line) + c * Ss;
#pragma unroll
            for (int f = 0; f < 12; ++f) {
                const T* p = f < 3 ? u + f * fs : (f < 6 ? q + (f - 3) * fs : cd + (f - 6) * fs);
                sm[(f * WS + c) * (NL + 1) + n] = ldg(p + oc);
            }
        }
        __syncthreads();
    }
    const bool live = t < lines;
    const int tl = live ? t : lines - 1, ib = tl / na, ia = tl - ib * na;
    const long long o = face_node(tl);
    const T* cp = cd + 6 * D * fs + o;
    auto uat = [&](int l, int c) -> T {
        if constexpr (D == 0) return sm[(l * WS + c) * (NL + 1) + tx];
        else return ldg(u + l * fs + o + c * Ss);
    };
    auto qat = [&](int j, int c) -> T {
        if constexpr (D == 0) return sm[((3 + j) * WS + c) * (NL + 1) + tx];
        else return ldg(q + (3 * D + j) * fs + o + c * Ss);
    };
    auto b = [&](int s6, int c) -> T {
        if constexpr (D == 0) return sm[((6 + s6) * WS + c) * (NL + 1) + tx];
        else return ldg(cp + s6 * fs + c * Ss);
    };
    constexpr int R3 = (RX + G - 1) / G;                     // rows of a group (fewer in the last)
    T rr[R3][3];
    if (G == 1 || group == 0) line_end_rows<T, O, D, 0>(g, fc, side, tl, ia, ib, uat, qat, b, ff, rr);
    else if constexpr (G == 3) {
        if (group == 1) line_end_rows<T, O, D, R3>(g, fc, side, tl, ia, ib, uat, qat, b, ff, rr);
        else line_end_rows<T, O, D, 2 * R3>(g, fc, side, tl, ia, ib, uat, qat, b, ff, rr);
    }
    const int r0 = group * R3;
    if constexpr (D == 0) __syncthreads();                   // every thread has read the staged columns
#pragma unroll
    for (int r = 0; r < R3; ++r)
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            if (G * R3 > RX && r0 + r >= RX) continue;
            if constexpr (D == 0) sm[(j * RX + r0 + r) * (NL + 1) + tx] = rr[r][j];
            else if (live) {
                if (D == 1 && line_row<O>(ib, g.n[2])) parts.x2[part_x2<O>(g, side * line_rows<O>() + r0 + r, j, ia, ib)] = rr[r][j];
                else un[j * fs + o + (r0 + r) * Ss] = rr[r][j];
            }
        }
    if constexpr (D == 0) {
        const int rows1 = side ? N - bx.x1hi : bx.x1lo;     // at most RX; more only on the smallest order-2 blocks
        __syncthreads();
        const int nr = rows1 < RX ? rows1 : RX;
        for (int idx = threadIdx.x; idx < NL * nr; idx += NT) {
            const int n = idx / nr, r = idx - n * nr, line = blk * NL + n;
            if (line >= lines) continue;
            const int l3 = line / na, l2 = line - l3 * na;
            const bool own = line_row<O>(l2, g.n[1]) || line_row<O>(l3, g.n[2]);
            const long long ol = face_node(line) + r * Ss;
#pragma unroll
            for (int j = 0; j < 3; ++j) {
                const T v = sm[(j * RX + r) * (NL + 1) + n];
                if (own) parts.x1[part_x1(g, bx, side, j, line, r)] = v;
                else un[j * fs + ol] = v;
            }
        }
        if (live && group == 0) {
            const bool own = line_row<O>(ia, g.n[1]) || line_row<O>(ib, g.n[2]);
            for (int r = RX; r < rows1; ++r) {
                T v[3] = {T(0), T(0), T(0)};
                int_row<T, O, 0>(g, q + o + r * Ss, cp + r * Ss, u + o + r * Ss, v);
#pragma unroll
                for (int j = 0; j < 3; ++j) {
                    if (own) parts.x1[part_x1(g, bx, side, j, tl, r)] = v[j];
                    else un[j * fs + o + r * Ss] = v[j];
                }
            }
        }
    }
}

// CTAs of the three directions
struct LineGrid {
    int c2, c1;             // CTAs of x3's lines, then of x2's; the rest take x1's
};
template <typename T, int O>
__global__ void __launch_bounds__(kLineThreads<O>) k3_lines(Grid3 g, Box3 bx, Faces3 fc, LineGrid lg, const T* __restrict__ u,
                                                               const T* __restrict__ q, const T* __restrict__ cd,
                                                               const T* __restrict__ ff, T* __restrict__ un, LineParts<T> parts) {
    __shared__ T sm[line_smem<T, O>()];
    const int k = blockIdx.x, side = blockIdx.y;
    if (k < lg.c2) line_ends<T, O, 2>(g, bx, fc, k, side, u, q, cd, ff, un, parts, sm);
    else if (k < lg.c2 + lg.c1) line_ends<T, O, 1>(g, bx, fc, k - lg.c2, side, u, q, cd, ff, un, parts, sm);
    else line_ends<T, O, 0>(g, bx, fc, k - lg.c2 - lg.c1, side, u, q, cd, ff, un, parts, sm);
}

// interior rows of direction D = x2 or x3 for the NV nodes of a thread
template <typename T, int O, int NV, int D>
__device__ __forceinline__ void div_int_dir(const Grid3& g, const T* __restrict__ qo, const T* __restrict__ cdo,
                                            const T* __restrict__ up, T r[NV][3]) {
    const long long fs = g.fs;
    if constexpr (NV == 2 && sizeof(T) == 4)
        div_int_strided_f2<O>(qo + 3 * D * fs, cdo + 6 * D * fs, up, fs, dstride<D>(g), float(g.ih[D]), r);
    else
        div_int_strided<T, O, NV>(qo + 3 * D * fs, cdo + 6 * D * fs, up, fs, dstride<D>(g), T(g.ih[D]), r);
}

// launch shapes of k3_div (sbp3_set_tuning / sbp3_autotune): x2 rows per block and the
// minimum resident blocks per SM, which sets the register cap (65536 / (32 BY MINB))
struct DivShape {
    int by, minb;
};
constexpr DivShape kDivShapes[4] = {{4, 4}, {4, 6}, {8, 3}, {2, 10}};

// Every node: the interior rows of the directions whose end rows k3_lines has not taken, on top of its partial
// sums where it has, then the store.  NV consecutive x1 nodes per thread read as one vector
// (float2 for FP32); the last pair of an odd row covers one element of the row's padding, whose value no
// node reads.  160 x 151 x 144, FP32, order 6: 181 us, with the cap at 96 registers 183 (the
// kernel with closure rows and SATs behind calls: 328 us for the x1-interior columns).
template <typename T, int O, int MODE, int NV, int BY, int MINB>
__global__ void __launch_bounds__(32 * BY, MINB) k3_div(Grid3 g, Box3 bx, const T* __restrict__ u,
                                                        const T* __restrict__ q, const T* __restrict__ cd,
                                                        const T* __restrict__ w, T* __restrict__ du, T* un, LineParts<T> parts,
                                                        T dt2) {
    constexpr int NR = line_rows<O>();
    const int i1 = (blockIdx.x * 32 + threadIdx.x) * NV, i2 = blockIdx.y * BY + threadIdx.y, i3 = blockIdx.z;
    if (i1 >= g.n[0] || i2 >= g.n[1]) return;
    const long long o = i1 + i2 * g.s[1] + i3 * g.s[2];
    const long long fs = g.fs;
    const T* up = u + o;
    const bool in1 = i1 >= bx.x1lo && i1 < bx.x1hi, in2 = i2 >= NR && i2 < g.n[1] - NR, in3 = i3 >= NR && i3 < g.n[2] - NR;
    T r[NV][3];
#pragma unroll
    for (int n = 0; n < NV; ++n) r[n][0] = r[n][1] = r[n][2] = T(0);
    if (!(in1 && in2 && in3)) {
        auto add = [&](const T* p, int j) {
            T v[NV];
            if constexpr (NV == 2 && sizeof(T) == 4) {
                const float2 x = *reinterpret_cast<const float2*>(p);
                v[0] = x.x;
                v[1] = x.y;
            } else {
#pragma unroll
                for (int n = 0; n < NV; ++n) v[n] = p[n];
            }
#pragma unroll
            for (int n = 0; n < NV; ++n) r[n][j] += v[n];
        };
#pragma unroll
        for (int j = 0; j < 3; ++j) add(un + j * fs + o, j);
        if (!in2 && !in3) {
            const int e2 = i2 < NR ? i2 : NR + g.n[1] - 1 - i2;
#pragma unroll
            for (int j = 0; j < 3; ++j) add(parts.x2 + part_x2<O>(g, e2, j, i1, i3), j);
        }
        if (!in1 && !(in2 && in3)) {
            const int side = i1 >= bx.x1hi;
            const long long line = (long long)i3 * g.n[1] + i2;
#pragma unroll
            for (int j = 0; j < 3; ++j)
#pragma unroll
                for (int n = 0; n < NV; ++n)
                    if (i1 + n < g.n[0]) r[n][j] += parts.x1[part_x1(g, bx, side, j, line, side ? g.n[0] - 1 - i1 - n : i1 + n)];
        }
    }
    if (in1) div_int_x1<T, O, NV>(q + o, cd + o, up, fs, T(g.ih[0]), r);
    if (in2) div_int_dir<T, O, NV, 1>(g, q + o, cd + o, up, r);
    if (in3) div_int_dir<T, O, NV, 2>(g, q + o, cd + o, up, r);
    T wv[NV];
    vld<T, NV>(w + o, wv);
#pragma unroll
    for (int j = 0; j < 3; ++j) {
        const long long oj = j * fs + o;
        T out[NV];
        if constexpr (MODE == 0) {
            T d[NV], uc[NV];
            vld<T, NV>(du + oj, d);
            vld<T, NV>(up + j * fs, uc);
#pragma unroll
            for (int n = 0; n < NV; ++n) {
                d[n] += dt2 * wv[n] * r[n][j];
                out[n] = uc[n] + d[n];
            }
            vst<T, NV>(du + oj, d);
        } else {
#pragma unroll
            for (int n = 0; n < NV; ++n) out[n] = wv[n] * r[n][j];
        }
        vst<T, NV>(un + oj, out);
    }
}

// ------------------------------------------------------------------ setup: metric and material
// For the x3-planes k0 <= i3 < k0 + nk: G_iI = D_i X_I (FP64), J = det G, F = G^-1,
// c_ijkl = J F_Ii C_IjKl F_Kk for the 45 stored entries, w = 1 / (rho J).  rho and C45 are the
// compact host layout of those planes (C45 entry t = 9p - p(p-1)/2 + (q - p), p = 3I+J <= q = 3K+L).
__host__ __device__ __forceinline__ constexpr int tri45(int p, int q) {
    return p <= q ? 9 * p - p * (p - 1) / 2 + (q - p) : 9 * q - q * (q - 1) / 2 + (p - q);
}

template <typename T, int O>
__global__ void __launch_bounds__(128) k3_material(Grid3 g, const double* __restrict__ X, int k0, int nk,
                                                   const double* __restrict__ rho, const double* __restrict__ C45,
                                                   T* __restrict__ cm, T* __restrict__ cd, T* __restrict__ w,
                                                   int* __restrict__ err) {
    const int i1 = blockIdx.x * blockDim.x + threadIdx.x, i2 = blockIdx.y, kk = blockIdx.z;
    if (i1 >= g.n[0] || i2 >= g.n[1] || kk >= nk) return;
    const int i3 = k0 + kk;
    const int idx[3] = {i1, i2, i3};
    const long long o = i1 + i2 * g.s[1] + i3 * g.s[2];
    double G[3][3];
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        const long long si = g.s[i];
#pragma unroll
        for (int I = 0; I < 3; ++I) {
            const double* line = X + I * g.fs + o - idx[i] * si;
            G[i][I] = g.ih[i] * dsum<O, double>(g.n[i], idx[i], [&](int t) { return line[t * si]; });
        }
    }
    const double J = G[0][0] * (G[1][1] * G[2][2] - G[1][2] * G[2][1]) -
                     G[0][1] * (G[1][0] * G[2][2] - G[1][2] * G[2][0]) +
                     G[0][2] * (G[1][0] * G[2][1] - G[1][1] * G[2][0]);
    if (!(J > 0.0)) {
        atomicExch(err, 1);
        return;
    }
    // F_Ii = (G^-1)_Ii = cof(G)_iI / J
    double F[3][3];
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int I = 0; I < 3; ++I) {
            const int i1c = (i + 1) % 3, i2c = (i + 2) % 3, I1 = (I + 1) % 3, I2 = (I + 2) % 3;
            F[I][i] = (G[i1c][I1] * G[i2c][I2] - G[i1c][I2] * G[i2c][I1]) / J;
        }
    const long long np = (long long)g.n[0] * g.n[1];
    const long long hc = (long long)kk * np + (long long)i2 * g.n[0] + i1;     // compact index
    const long long cstr = (long long)nk * np;
    double Cn[45];
#pragma unroll
    for (int t = 0; t < 45; ++t) Cn[t] = C45[t * cstr + hc];
    auto cval = [&](int i, int j, int k, int l) {
        double s = 0.0;
#pragma unroll
        for (int I = 0; I < 3; ++I) {
            double sI = 0.0;
#pragma unroll
            for (int K = 0; K < 3; ++K) sI += Cn[tri45(3 * I + j, 3 * K + l)] * F[K][k];
            s += F[I][i] * sI;
        }
        return J * s;
    };
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j)
#pragma unroll
            for (int l = j; l < 3; ++l) cd[(long long)(6 * i + sym3(j, l)) * g.fs + o] = T(cval(i, j, i, l));
#pragma unroll
    for (int p = 0; p < 3; ++p) {
        const int i = p == 2 ? 1 : 0, k = p == 0 ? 1 : 2;
#pragma unroll
        for (int j = 0; j < 3; ++j)
#pragma unroll
            for (int l = 0; l < 3; ++l) cm[(long long)(9 * p + 3 * j + l) * g.fs + o] = T(cval(i, j, k, l));
    }
    w[o] = T(1.0 / (rho[hc] * J));
}

// ------------------------------------------------------------------ state conversion
// compact FP64 (3 components) <-> pitched T.  Load: u_cur, u_prev and the increment
// u_cur - u_prev formed in FP64.  Store: the two levels back to FP64.
template <typename T>
__global__ void k3_load_state(Grid3 g, const double* __restrict__ prev, const double* __restrict__ cur,
                              T* __restrict__ up, T* __restrict__ uc, T* __restrict__ du) {
    const int i1 = blockIdx.x * blockDim.x + threadIdx.x, i2 = blockIdx.y, i3 = blockIdx.z;
    if (i1 >= g.n[0]) return;
    const long long N = (long long)g.n[0] * g.n[1] * g.n[2];
    const long long hc = ((long long)i3 * g.n[1] + i2) * g.n[0] + i1;
    const long long o = i1 + i2 * g.s[1] + i3 * g.s[2];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const double a = prev[c * N + hc], b = cur[c * N + hc];
        up[c * g.fs + o] = T(a);
        uc[c * g.fs + o] = T(b);
        du[c * g.fs + o] = T(b - a);
    }
}

template <typename T>
__global__ void k3_store_field(Grid3 g, const T* __restrict__ f, double* __restrict__ out) {
    const int i1 = blockIdx.x * blockDim.x + threadIdx.x, i2 = blockIdx.y, i3 = blockIdx.z;
    if (i1 >= g.n[0]) return;
    const long long N = (long long)g.n[0] * g.n[1] * g.n[2];
    const long long hc = ((long long)i3 * g.n[1] + i2) * g.n[0] + i1;
    const long long o = i1 + i2 * g.s[1] + i3 * g.s[2];
#pragma unroll
    for (int c = 0; c < 3; ++c) out[c * N + hc] = double(f[c * g.fs + o]);
}

template <typename T>
__global__ void k3_load_field(Grid3 g, const double* __restrict__ in, T* __restrict__ f) {
    const int i1 = blockIdx.x * blockDim.x + threadIdx.x, i2 = blockIdx.y, i3 = blockIdx.z;
    if (i1 >= g.n[0]) return;
    const long long N = (long long)g.n[0] * g.n[1] * g.n[2];
    const long long hc = ((long long)i3 * g.n[1] + i2) * g.n[0] + i1;
    const long long o = i1 + i2 * g.s[1] + i3 * g.s[2];
#pragma unroll
    for (int c = 0; c < 3; ++c) f[c * g.fs + o] = T(in[c * N + hc]);
}

}  // namespace sbp3

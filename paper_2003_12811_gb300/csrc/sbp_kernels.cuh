// libsbp kernels: one leapfrog step of the SBP-SAT anisotropic elastic scheme (interior
// stencil, boundary strips with closures and SATs, face traces, interface/boundary SAT terms,
// point sources), the FP64 energy reduction, and the setup kernels (metric, material, CFL).
#pragma once
#include "sbp_device.cuh"

namespace sbp {

// ============================================================================ interior
// Tile of TX x TY output nodes, 256 threads (32 x 8), every thread computes TY/8 nodes.
// Nodes of the interior region are at least `strip` >= NCLOS, NCOL away from every face, so
// every row uses the interior stencils and no SAT reaches them.
//   r_j = sum_d [ D_dd^FC(c_djdl) u_l ] + D_1 (c_1j2l D_2 u_l) + D_2 (c_2j1l D_1 u_l)   (Sec. 4.6)
// with the narrow rows written through edge weights:
//   D_xx(b) u |_i = h^-2 sum_m E_m(i) (u_{i+m} - u_i) + E_m(i-m) (u_{i-m} - u_i).
constexpr int ITX = 32, ITY = 16, ITHREADS = 256;

template <typename T, int O> constexpr size_t interior_smem_elems() {
    constexpr int Q = Ord<O>::Q, SX = ITX + 2 * Q, SY = ITY + 2 * Q;
    return 2 * SY * SX + 3 * ITY * SX + 3 * SY * ITX + 4 * SY * SX + 2 * ITY * SX + 2 * SY * ITX +
           3 * Q * ITY * (ITX + Q) + 3 * Q * (ITY + Q) * ITX;
}

template <typename T, int O, int MODE>
__global__ void __launch_bounds__(ITHREADS) k_interior(BlockDev B, StepArgs a) {
    constexpr int Q = Ord<O>::Q;
    constexpr int TX = ITX, TY = ITY, SX = TX + 2 * Q, SY = TY + 2 * Q, EX = TX + Q, EY = TY + Q;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    T* su = reinterpret_cast<T*>(smem_raw);   // [2][SY][SX]
    T* snx = su + 2 * SY * SX;                 // [3][TY][SX]
    T* sny = snx + 3 * TY * SX;                // [3][SY][TX]
    T* smx = sny + 3 * SY * TX;                // [4][SY][SX]
    T* sg1 = smx + 4 * SY * SX;                // [2][TY][SX]
    T* sg2 = sg1 + 2 * TY * SX;                // [2][SY][TX]
    T* sex = sg2 + 2 * SY * TX;                // [3][Q][TY][EX]   E_m at i = ii - Q
    T* sey = sex + 3 * Q * TY * EX;            // [3][Q][EY][TX]   E_m at j = jj - Q

    const int S = B.strip;
    const int n1 = B.n1, n2 = B.n2, P = B.pitch;
    const int lim1 = n1 - S, lim2 = n2 - S;
    const int x0 = S + blockIdx.x * TX, y0 = S + blockIdx.y * TY;
    const int tid = threadIdx.y * 32 + threadIdx.x;
    const size_t plane = (size_t)n2 * P;
    const T* __restrict__ U = reinterpret_cast<const T*>(B.u[a.cur]);
    const T* __restrict__ C = reinterpret_cast<const T*>(B.c);

    auto load = [&](T* dst, const T* __restrict__ src, int rows, int cols, int gy0, int gx0) {
        for (int idx = tid; idx < rows * cols; idx += ITHREADS) {
            const int r = idx / cols, c = idx - r * cols;
            const int gy = gy0 + r, gx = gx0 + c;
            dst[idx] = (gy < n2 && gx < n1) ? __ldg(src + (size_t)gy * P + gx) : T(0);
        }
    };
    load(su, U, SY, SX, y0 - Q, x0 - Q);
    load(su + SY * SX, U + plane, SY, SX, y0 - Q, x0 - Q);
#pragma unroll
    for (int f = 0; f < 3; ++f) load(snx + f * TY * SX, C + f * plane, TY, SX, y0, x0 - Q);
#pragma unroll
    for (int f = 0; f < 3; ++f) load(sny + f * SY * TX, C + (3 + f) * plane, SY, TX, y0 - Q, x0);
#pragma unroll
    for (int f = 0; f < 4; ++f) load(smx + f * SY * SX, C + (6 + f) * plane, SY, SX, y0 - Q, x0 - Q);
    __syncthreads();

    const T ih1 = ih1T<T>(B), ih2 = ih2T<T>(B);
    // mixed fluxes g1_j = c_1j2l D_2 u_l on tile rows x (tile cols + x-halo)
    for (int idx = tid; idx < TY * SX; idx += ITHREADS) {
        const int r = idx / SX, c = idx - r * SX;
        const T* p0 = su + (r + Q) * SX + c;
        const T* p1 = p0 + SY * SX;
        T d0 = T(0), d1 = T(0);
#pragma unroll
        for (int k = 1; k <= Q; ++k) {
            const T ak = Ord<O>::template aT<T>(k - 1);
            d0 += ak * (p0[k * SX] - p0[-k * SX]);
            d1 += ak * (p1[k * SX] - p1[-k * SX]);
        }
        d0 *= ih2;
        d1 *= ih2;
        const int mi = (r + Q) * SX + c;
        const T m6 = smx[mi], m7 = smx[SY * SX + mi], m8 = smx[2 * SY * SX + mi], m9 = smx[3 * SY * SX + mi];
        sg1[r * SX + c] = m6 * d0 + m7 * d1;
        sg1[TY * SX + r * SX + c] = m8 * d0 + m9 * d1;
    }
    // mixed fluxes g2_j = c_2j1l D_1 u_l = c_1l2j D_1 u_l on (tile rows + y-halo) x tile cols
    for (int idx = tid; idx < SY * TX; idx += ITHREADS) {
        const int r = idx / TX, c = idx - r * TX;
        const T* p0 = su + r * SX + c + Q;
        const T* p1 = p0 + SY * SX;
        T d0 = T(0), d1 = T(0);
#pragma unroll
        for (int k = 1; k <= Q; ++k) {
            const T ak = Ord<O>::template aT<T>(k - 1);
            d0 += ak * (p0[k] - p0[-k]);
            d1 += ak * (p1[k] - p1[-k]);
        }
        d0 *= ih1;
        d1 *= ih1;
        const int mi = r * SX + c + Q;
        const T m6 = smx[mi], m7 = smx[SY * SX + mi], m8 = smx[2 * SY * SX + mi], m9 = smx[3 * SY * SX + mi];
        sg2[r * TX + c] = m6 * d0 + m8 * d1;
        sg2[SY * TX + r * TX + c] = m7 * d0 + m9 * d1;
    }
    // edge weights along x1 at i in [-Q, TX)
    for (int idx = tid; idx < 3 * TY * EX; idx += ITHREADS) {
        const int f = idx / (TY * EX);
        const int rem = idx - f * TY * EX;
        const int r = rem / EX, ii = rem - r * EX;
        const int i = ii - Q;
        const T* bl = snx + f * TY * SX + r * SX + (i + Q);
        auto Bf = [&](int k) { return bl[k]; };
#pragma unroll
        for (int m = 1; m <= Q; ++m)
            sex[((f * Q + (m - 1)) * TY + r) * EX + ii] = (i + Q + edge_lo<O>(m) >= 0) ? Edge<O>::template e<T>(m, Bf) : T(0);
    }
    // edge weights along x2 at j in [-Q, TY)
    for (int idx = tid; idx < 3 * EY * TX; idx += ITHREADS) {
        const int f = idx / (EY * TX);
        const int rem = idx - f * EY * TX;
        const int jj = rem / TX, c = rem - jj * TX;
        const int j = jj - Q;
        const T* bl = sny + f * SY * TX + (j + Q) * TX + c;
        auto Bf = [&](int k) { return bl[k * TX]; };
#pragma unroll
        for (int m = 1; m <= Q; ++m)
            sey[((f * Q + (m - 1)) * EY + jj) * TX + c] = (j + Q + edge_lo<O>(m) >= 0) ? Edge<O>::template e<T>(m, Bf) : T(0);
    }
    __syncthreads();

    const T* __restrict__ Wp = reinterpret_cast<const T*>(B.w);
#pragma unroll
    for (int rr = 0; rr < TY / 8; ++rr) {
        const int r = threadIdx.y + 8 * rr, c = threadIdx.x;
        const int gx = x0 + c, gy = y0 + r;
        if (gx >= lim1 || gy >= lim2) continue;
        const T* u0 = su + (r + Q) * SX + (c + Q);
        const T* u1 = u0 + SY * SX;
        const T uc0 = u0[0], uc1 = u1[0];
        T rx0 = T(0), rx1 = T(0), ry0 = T(0), ry1 = T(0);
#pragma unroll
        for (int m = 1; m <= Q; ++m) {
            const T* ex0 = sex + ((0 * Q + (m - 1)) * TY + r) * EX + (c + Q);
            const T* ex1 = ex0 + Q * TY * EX;
            const T* ex2 = ex1 + Q * TY * EX;
            const T dp0 = u0[m] - uc0, dp1 = u1[m] - uc1, dm0 = u0[-m] - uc0, dm1 = u1[-m] - uc1;
            rx0 += ex0[0] * dp0 + ex1[0] * dp1 + ex0[-m] * dm0 + ex1[-m] * dm1;
            rx1 += ex1[0] * dp0 + ex2[0] * dp1 + ex1[-m] * dm0 + ex2[-m] * dm1;
            const T* ey0 = sey + ((0 * Q + (m - 1)) * EY + (r + Q)) * TX + c;
            const T* ey1 = ey0 + Q * EY * TX;
            const T* ey2 = ey1 + Q * EY * TX;
            const T qp0 = u0[m * SX] - uc0, qp1 = u1[m * SX] - uc1, qm0 = u0[-m * SX] - uc0, qm1 = u1[-m * SX] - uc1;
            ry0 += ey0[0] * qp0 + ey1[0] * qp1 + ey0[-m * TX] * qm0 + ey1[-m * TX] * qm1;
            ry1 += ey1[0] * qp0 + ey2[0] * qp1 + ey1[-m * TX] * qm0 + ey2[-m * TX] * qm1;
        }
        T r0 = rx0 * ih1 * ih1 + ry0 * ih2 * ih2;
        T r1 = rx1 * ih1 * ih1 + ry1 * ih2 * ih2;
        const T* g10 = sg1 + r * SX + (c + Q);
        const T* g11 = g10 + TY * SX;
        const T* g20 = sg2 + (r + Q) * TX + c;
        const T* g21 = g20 + SY * TX;
        T m10 = T(0), m11 = T(0), m20 = T(0), m21 = T(0);
#pragma unroll
        for (int k = 1; k <= Q; ++k) {
            const T ak = Ord<O>::template aT<T>(k - 1);
            m10 += ak * (g10[k] - g10[-k]);
            m11 += ak * (g11[k] - g11[-k]);
            m20 += ak * (g20[k * TX] - g20[-k * TX]);
            m21 += ak * (g21[k * TX] - g21[-k * TX]);
        }
        r0 += m10 * ih1 + m20 * ih2;
        r1 += m11 * ih1 + m21 * ih2;
        const size_t gi = (size_t)gy * P + gx;
        if (a.with_data && B.jf) {
            const T* __restrict__ JF = reinterpret_cast<const T*>(B.jf);
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                if (k >= a.K) break;
                r0 += T(a.Tk[k]) * JF[(size_t)k * plane + gi];
                r1 += T(a.Tk[k]) * JF[(size_t)(a.K + k) * plane + gi];
            }
        }
        if (MODE == 0) {
            T* __restrict__ Un = reinterpret_cast<T*>(B.u[1 - a.cur]);
            const T wv = Wp[gi], dt2 = dt2T<T>(a);
            Un[gi] = T(2) * uc0 - Un[gi] + dt2 * wv * r0;
            Un[gi + plane] = T(2) * uc1 - Un[gi + plane] + dt2 * wv * r1;
        } else if (MODE == 2) {
            rk4_store<T>(B, a, gi, plane, Wp[gi], r0, r1);
        } else {
            T* __restrict__ R = reinterpret_cast<T*>(B.r);
            R[gi] = r0;
            R[gi + plane] = r1;
        }
    }
}

// ============================================================================ interior, FP64
// The FP64 units bound the double-precision interior: an SM retires two FP64 results per clock
// (152 SMs: 1.26 TFLOP/s against 6.8 TB/s, 0.19 operations per byte), so a warp's FP64 instruction
// holds its SM for 16 clocks and every one that is left out counts, while 232 B/node of traffic do not.
//  * The edge weights of the narrow rows depend on the material alone: k_edge_weights forms them once
//    and the step reads them (18 planes for order 6) instead of spending 100 of its 245 instructions per
//    node on them again.
//  * Only the displacement and the mixed fluxes, which neighbours share, sit in shared memory (34 KB for
//    32 x 16 nodes against the 177 KB that the kernel with its own weights needs, one CTA per SM).
//  * One launch covers every block (no tail per block), in tiles of a shape that launch_interior_f64
//    picks so that small grids still spread over all SMs.
// A step of 4 order-6 blocks of 401^2 (0.6 M interior nodes): 0.19 ms for the one launch, where the kernel
// with its own weights took 4 launches of 0.132 ms; at the FP64 units' rate the 157 instructions per node
// (counted by ncu: 227 operations) take 0.15 ms.
template <typename T, int O> __global__ void k_edge_weights(BlockDev B, T* __restrict__ E) {
    constexpr int Q = Ord<O>::Q;
    const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= (long long)B.n1 * B.n2) return;
    const int i2 = (int)(t / B.n1), i1 = (int)(t - (long long)i2 * B.n1);
    const size_t plane = (size_t)B.n2 * B.pitch, gi = (size_t)i2 * B.pitch + i1;
    const T* __restrict__ C = reinterpret_cast<const T*>(B.c);
#pragma unroll
    for (int d = 0; d < 2; ++d) {
        const int i = d == 0 ? i1 : i2, N = d == 0 ? B.n1 : B.n2;
        const long long st = d == 0 ? 1 : B.pitch;
        const T ih = d == 0 ? ih1T<T>(B) : ih2T<T>(B);
#pragma unroll
        for (int m = 1; m <= Q; ++m) {
            const bool in = i + edge_lo<O>(m) >= 0 && i + EdgeRange<O>::HI < N;   // the rows that use it are in range
#pragma unroll
            for (int f = 0; f < 3; ++f) {
                const T* b = C + (size_t)(3 * d + f) * plane + gi;
                const T e = in ? Edge<O>::template e<T>(m, [&](int k) { return b[k * st]; }) : T(0);
                E[(size_t)edge_plane<O>(d, f, m) * plane + gi] = e * ih * ih;
            }
        }
    }
}

constexpr int IE_MAX_BLOCKS = 32;
struct InteriorTiles {
    int nb, first;                     // blocks of this launch, the first one's index
    int start[IE_MAX_BLOCKS + 1];      // first tile of each
    int ncx[IE_MAX_BLOCKS];            // tiles across
};

// shared-memory elements of a tile: the displacement with its halo, g1 and g2
template <int O, int TX, int TY> constexpr int edge_tile_elems() {
    constexpr int SX = TX + 2 * Ord<O>::Q, SY = TY + 2 * Ord<O>::Q;
    return 2 * (SY * SX + TY * SX + SY * TX);
}
// tile `tile` (of ncx across) of block B by the NT threads of the CTA
template <typename T, int O, int MODE, int TX, int TY, int NT>
__device__ __forceinline__ void interior_edges_tile(const BlockDev& B, int tile, int ncx, const StepArgs& a, T* sm) {
    constexpr int Q = Ord<O>::Q;
    constexpr int SX = TX + 2 * Q, SY = TY + 2 * Q;
    T(*su)[SY][SX] = reinterpret_cast<T(*)[SY][SX]>(sm);
    T(*sg1)[TY][SX] = reinterpret_cast<T(*)[TY][SX]>(sm + 2 * SY * SX);
    T(*sg2)[SY][TX] = reinterpret_cast<T(*)[SY][TX]>(sm + 2 * (SY * SX + TY * SX));
    const int S = B.strip, n1 = B.n1, n2 = B.n2, P = B.pitch;
    const int x0 = S + (tile % ncx) * TX, y0 = S + (tile / ncx) * TY;
    const int lim1 = n1 - S, lim2 = n2 - S;
    const size_t plane = (size_t)n2 * P;
    const T* __restrict__ U = reinterpret_cast<const T*>(B.u[a.cur]);
    const T* __restrict__ M = reinterpret_cast<const T*>(B.c) + 6 * plane;
    const T* __restrict__ E = reinterpret_cast<const T*>(B.e);
    // nodes past the last interior row or column by more than Q are nobody's neighbours: zero
    const int xe = min(x0 - Q + SX, n1), ye = min(y0 - Q + SY, n2);
    for (int idx = threadIdx.x; idx < SY * SX; idx += NT) {
        const int r = idx / SX, c = idx - r * SX, gx = x0 - Q + c, gy = y0 - Q + r;
        const bool in = gx < xe && gy < ye;
        const size_t gi = (size_t)gy * P + gx;
        su[0][r][c] = in ? __ldg(U + gi) : T(0);
        su[1][r][c] = in ? __ldg(U + plane + gi) : T(0);
    }
    T a1[Q], a2[Q];
#pragma unroll
    for (int k = 0; k < Q; ++k) {
        a1[k] = T(B.ai1[k]);
        a2[k] = T(B.ai2[k]);
    }
    __syncthreads();
    // mixed fluxes g1_j = c_1j2l D_2 u_l on the tile's rows and its columns +- Q, g2_j = c_1l2j D_1 u_l
    // on its columns and its rows +- Q, one loop over both so that the CTA's warps share them evenly
    for (int idx = threadIdx.x; idx < TY * SX + SY * TX; idx += NT) {
        const bool first = idx < TY * SX;
        const int id = first ? idx : idx - TY * SX, w = first ? SX : TX;
        const int r = id / w, c = id - r * w;
        const int gx = first ? x0 - Q + c : x0 + c, gy = first ? y0 + r : y0 - Q + r;
        if (gx >= xe || gy >= ye) continue;
        const size_t gi = (size_t)gy * P + gx;
        const T m6 = __ldg(M + gi), m7 = __ldg(M + plane + gi), m8 = __ldg(M + 2 * plane + gi), m9 = __ldg(M + 3 * plane + gi);
        const T* p0 = first ? &su[0][r + Q][c] : &su[0][r][c + Q];
        const T* p1 = p0 + SY * SX;
        const int st = first ? SX : 1;
        T d0 = T(0), d1 = T(0);
#pragma unroll
        for (int k = 1; k <= Q; ++k) {
            const T ak = first ? a2[k - 1] : a1[k - 1];
            d0 += ak * (p0[k * st] - p0[-k * st]);
            d1 += ak * (p1[k * st] - p1[-k * st]);
        }
        if (first) {
            sg1[0][r][c] = m6 * d0 + m7 * d1;
            sg1[1][r][c] = m8 * d0 + m9 * d1;
        } else {
            sg2[0][r][c] = m6 * d0 + m8 * d1;
            sg2[1][r][c] = m7 * d0 + m9 * d1;
        }
    }
    __syncthreads();
#pragma unroll
    for (int n = 0; n < (TX * TY + NT - 1) / NT; ++n) {
        const int idx = threadIdx.x + n * NT, r = idx / TX, c = idx - r * TX;
        const int gx = x0 + c, gy = y0 + r;
        if (r >= TY || gx >= lim1 || gy >= lim2) continue;
        const size_t gi = (size_t)gy * P + gx;
        T r0 = T(0), r1 = T(0);
        dxx_edges<O, T>(
            0, [&](int k) { return su[0][r + Q][c + Q + k]; }, [&](int k) { return su[1][r + Q][c + Q + k]; },
            [&](int f, int m, int k) { return __ldg(E + (size_t)edge_plane<O>(0, f, m) * plane + gi + k); }, r0, r1);
        dxx_edges<O, T>(
            0, [&](int k) { return su[0][r + Q + k][c + Q]; }, [&](int k) { return su[1][r + Q + k][c + Q]; },
            [&](int f, int m, int k) { return __ldg(E + (size_t)edge_plane<O>(1, f, m) * plane + gi + (long long)k * P); },
            r0, r1);
#pragma unroll
        for (int k = 1; k <= Q; ++k) {
            r0 += a1[k - 1] * (sg1[0][r][c + Q + k] - sg1[0][r][c + Q - k]);
            r1 += a1[k - 1] * (sg1[1][r][c + Q + k] - sg1[1][r][c + Q - k]);
            r0 += a2[k - 1] * (sg2[0][r + Q + k][c] - sg2[0][r + Q - k][c]);
            r1 += a2[k - 1] * (sg2[1][r + Q + k][c] - sg2[1][r + Q - k][c]);
        }
        if (a.with_data && B.jf) {
            const T* __restrict__ JF = reinterpret_cast<const T*>(B.jf);
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                if (k >= a.K) break;
                r0 += T(a.Tk[k]) * JF[(size_t)k * plane + gi];
                r1 += T(a.Tk[k]) * JF[(size_t)(a.K + k) * plane + gi];
            }
        }
        if (MODE == 0) {
            leapfrog_store<T>(B, a, gi, plane, su[0][r + Q][c + Q], su[1][r + Q][c + Q],
                              reinterpret_cast<const T*>(B.w)[gi], r0, r1, false, T(0), T(0), T(0));
        } else if (MODE == 2) {
            rk4_store<T>(B, a, gi, plane, reinterpret_cast<const T*>(B.w)[gi], r0, r1);
        } else {
            T* __restrict__ R = reinterpret_cast<T*>(B.r);
            R[gi] = r0;
            R[gi + plane] = r1;
        }
    }
}

template <typename T, int O, int MODE, int TX, int TY>
__global__ void __launch_bounds__(TX * TY < 256 ? TX * TY : 256)
k_interior_edges(const BlockDev* __restrict__ blocks, const __grid_constant__ InteriorTiles tl, StepArgs a) {
    constexpr int NT = TX * TY < 256 ? TX * TY : 256;
    __shared__ T sm[edge_tile_elems<O, TX, TY>()];
    int b = 0;
    while (b + 1 < tl.nb && (int)blockIdx.x >= tl.start[b + 1]) ++b;
    interior_edges_tile<T, O, MODE, TX, TY, NT>(blocks[tl.first + b], blockIdx.x - tl.start[b], tl.ncx[b], a, sm);
}

// ============================================================================ faces
struct FaceRef {
    int block, face, start, nf;
};

__device__ __forceinline__ int find_face(const FaceRef* refs, int nrefs, int t) {
    int k = 0;
    while (k + 1 < nrefs && t >= refs[k + 1].start) ++k;
    return k;
}

// c planes at a face node: narrow of the normal direction m (c_mJmL) and the mixed c_mJtL
__device__ __forceinline__ int plane_nn(int m, int J, int L) { return 3 * m + J + L; }
__device__ __forceinline__ int plane_nt(int m, int J, int L) { return m == 0 ? 6 + 2 * J + L : 6 + 2 * L + J; }

// node (j1, j2) of face F at tangential index sp and depth d
__device__ __forceinline__ void face_at(const BlockDev& B, const FaceDev& F, int sp, int d, int& j1, int& j2) {
    if (F.m == 0) { j1 = F.side ? B.n1 - 1 - d : d; j2 = sp; }
    else { j2 = F.side ? B.n2 - 1 - d : d; j1 = sp; }
}

// J^ tau_J = nu_i c_iJkL D_k u_L at face node s (eq. n-C_conversion); u(L, j1, j2), c(pl, j1, j2)
template <typename T, int O, class UA, class CA>
__device__ __forceinline__ void face_traction(const BlockDev& B, const FaceDev& F, int s, UA u, CA c, T& t0, T& t1) {
    const int m = F.m, Nm = m == 0 ? B.n1 : B.n2, Nt = m == 0 ? B.n2 : B.n1;
    const T ihm = (m == 0 ? ih1T<T>(B) : ih2T<T>(B)), iht = (m == 0 ? ih2T<T>(B) : ih1T<T>(B));
    T dn[2], dt[2];
#pragma unroll
    for (int L = 0; L < 2; ++L) {
        dn[L] = dsum<O, T>(Nm, F.side ? Nm - 1 : 0, [&](int j) {
                    int j1, j2;
                    face_at(B, F, s, F.side ? Nm - 1 - j : j, j1, j2);
                    return u(L, j1, j2);
                }) * ihm;
        dt[L] = dsum<O, T>(Nt, s, [&](int j) {
                    int j1, j2;
                    face_at(B, F, j, 0, j1, j2);
                    return u(L, j1, j2);
                }) * iht;
    }
    int i1, i2;
    face_at(B, F, s, 0, i1, i2);
    const T nu = T(F.nu);
    t0 = nu * (c(plane_nn(m, 0, 0), i1, i2) * dn[0] + c(plane_nn(m, 0, 1), i1, i2) * dn[1] +
               c(plane_nt(m, 0, 0), i1, i2) * dt[0] + c(plane_nt(m, 0, 1), i1, i2) * dt[1]);
    t1 = nu * (c(plane_nn(m, 1, 0), i1, i2) * dn[0] + c(plane_nn(m, 1, 1), i1, i2) * dn[1] +
               c(plane_nt(m, 1, 0), i1, i2) * dt[0] + c(plane_nt(m, 1, 1), i1, i2) * dt[1]);
}

// SAT terms of face node s of face F of block B (Sec. 5.1 eq. sat_traction, Sec. 5.2 eq.
// dirichlet_ansatz with Z of Theorem 3, Sec. 6 eq. scheme_interface with V = Theta = 0), using
// J^ Z_JL = beta d / h1 * c_mJmL (boundary) and beta d / 4 (c^u_mJmL / h1^u + c^v / h1^v) (interface):
//   Fs_J: the term added at the face node itself,
//   As_J: the amplitude a_J = half nu c_mJmL w_L spread by D_m^T into the first NCOL nodes along
//         the normal (times F.fac[d]).
// u(L, j1, j2), c(pl, j1, j2) read this block's current level and coefficients; the interface
// neighbour is read from `blocks` (its current level in the same buffer parity a.cur).
template <typename T, int O, class UA, class CA>
__device__ void face_sat_node(const BlockDev* __restrict__ blocks, const BlockDev& B, const FaceDev& F, int s,
                              const StepArgs& a, double beta, UA u, CA c, T& Fs0, T& Fs1, T& As0, T& As1) {
    const int m = F.m, nf = F.nf;
    const T nu = T(F.nu);
    const T inv_h0 = T(F.inv_h0);
    int i1, i2;
    face_at(B, F, s, 0, i1, i2);
    const bool has_data = a.with_data && F.g;
    const T* __restrict__ g = reinterpret_cast<const T*>(F.g);
    if (F.kind == FACE_ROBIN) {
        T f0, f1;
        face_traction<T, O>(B, F, s, u, c, f0, f1);
        const T u0 = u(0, i1, i2), u1 = u(1, i1, i2);
        if (F.ju) {
            const T* ju = reinterpret_cast<const T*>(F.ju);
            const T a11 = ju[s], a12 = ju[nf + s], a22 = ju[2 * nf + s];
            f0 += a11 * u0 + a12 * u1;
            f1 += a12 * u0 + a22 * u1;
        }
        if (has_data) {
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                if (k >= a.K) break;
                f0 -= T(a.Tk[k]) * g[(size_t)k * nf + s];
                f1 -= T(a.Tk[k]) * g[(size_t)(a.K + k) * nf + s];
            }
        }
        Fs0 = -inv_h0 * f0;
        Fs1 = -inv_h0 * f1;
        As0 = As1 = T(0);
        return;
    }
    const bool intf = F.kind == FACE_INTF;
    // the neighbour across an interface: its block, face, current level and coefficients
    const BlockDev* V = intf ? &blocks[F.nbr_block] : nullptr;
    const FaceDev* FV = intf ? &V->f[F.nbr_face] : nullptr;
    const T* __restrict__ Uv = intf ? reinterpret_cast<const T*>(V->u[a.cur]) : nullptr;
    const T* __restrict__ Cv = intf ? reinterpret_cast<const T*>(V->c) : nullptr;
    const size_t pv = intf ? (size_t)V->n2 * V->pitch : 0;
    auto uv = [&](int L, int j1, int j2) { return Uv[(size_t)L * pv + (size_t)j2 * V->pitch + j1]; };
    auto cv = [&](int pl, int j1, int j2) { return Cv[(size_t)pl * pv + (size_t)j2 * V->pitch + j1]; };
    // traces of both sides (k_face_trace, same level): replace the neighbour's reads and both tractions
    const T* __restrict__ trU = intf ? reinterpret_cast<const T*>(F.tr) : nullptr;
    const T* __restrict__ trV = intf ? reinterpret_cast<const T*>(FV->tr) : nullptr;
    const bool traced = trU != nullptr && trV != nullptr;
    // jump w_L at face node sp (displacement: u - g(t); interface: u - v)
    auto jump = [&](int sp, T& w0, T& w1) {
        int j1, j2;
        face_at(B, F, sp, 0, j1, j2);
        w0 = u(0, j1, j2);
        w1 = u(1, j1, j2);
        if (intf) {
            const int svp = F.reversed ? nf - 1 - sp : sp;
            if (traced) {
                w0 -= trV[svp];
                w1 -= trV[nf + svp];
            } else {
                int v1, v2;
                face_at(*V, *FV, svp, 0, v1, v2);
                w0 -= uv(0, v1, v2);
                w1 -= uv(1, v1, v2);
            }
        } else if (has_data) {
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                if (k >= a.K) break;
                w0 -= T(a.Tk[k]) * g[(size_t)k * nf + sp];
                w1 -= T(a.Tk[k]) * g[(size_t)(a.K + k) * nf + sp];
            }
        }
    };
    const T half = intf ? T(0.5) : T(1);
    const double dd = 2.0;   // spatial dimension d
    T w0, w1;
    jump(s, w0, w1);
    const T c00 = c(plane_nn(m, 0, 0), i1, i2), c01 = c(plane_nn(m, 0, 1), i1, i2), c11 = c(plane_nn(m, 1, 1), i1, i2);
    T z00, z01, z11;
    if (!intf) {
        const T k = T(beta * dd * F.inv_h0);
        z00 = k * c00; z01 = k * c01; z11 = k * c11;
    } else if (traced) {
        const int sv = F.reversed ? nf - 1 - s : s;
        z00 = trU[4 * nf + s] + trV[4 * nf + sv];
        z01 = trU[5 * nf + s] + trV[5 * nf + sv];
        z11 = trU[6 * nf + s] + trV[6 * nf + sv];
    } else {
        const int sv = F.reversed ? nf - 1 - s : s;
        int v1, v2;
        face_at(*V, *FV, sv, 0, v1, v2);
        const int mv = FV->m;
        const T ku = T(beta * dd / 4.0 * F.inv_h0), kv = T(beta * dd / 4.0 * FV->inv_h0);
        const T zu00 = ku * c00, zu01 = ku * c01, zu11 = ku * c11;
        const T zv00 = kv * cv(plane_nn(mv, 0, 0), v1, v2), zv01 = kv * cv(plane_nn(mv, 0, 1), v1, v2),
                zv11 = kv * cv(plane_nn(mv, 1, 1), v1, v2);
        z00 = zu00 + zv00;
        z01 = zu01 + zv01;
        z11 = zu11 + zv11;
    }
    // normal-spread amplitude a_J = half nu c_mJmL w_L
    As0 = half * nu * (c00 * w0 + c01 * w1);
    As1 = half * nu * (c01 * w0 + c11 * w1);
    // tangential transpose term (1/H_t(s)) sum_s' D_t[s'][s] H_t(s') b_J(s'),  b_J = nu c_mLtJ w_L;
    // rows of D with a non-zero in column s: the interior band s-Q..s+Q plus, near an end, every
    // boundary row (boundary rows span columns 0..NCOL-1, which can reach past s+Q)
    const int Nt = nf;
    T tt0 = T(0), tt1 = T(0);
    auto tterm = [&](int sp, T wgt) {
        T v0, v1;
        jump(sp, v0, v1);
        int j1, j2;
        face_at(B, F, sp, 0, j1, j2);
        tt0 += wgt * nu * (c(plane_nt(m, 0, 0), j1, j2) * v0 + c(plane_nt(m, 1, 0), j1, j2) * v1);
        tt1 += wgt * nu * (c(plane_nt(m, 0, 1), j1, j2) * v0 + c(plane_nt(m, 1, 1), j1, j2) * v1);
    };
    if (s >= Ord<O>::NCOL && s < Nt - Ord<O>::NCOL) {
        // column s meets only interior rows s-Q..s+Q of D (weight 1): a fixed, unrolled sum whose
        // loads (the neighbour's traces across an interface) can all be in flight together
#pragma unroll
        for (int k = 1; k <= Ord<O>::Q; ++k) {
            const T ak = Ord<O>::template aT<T>(k - 1);
            tterm(s - k, ak);        // row s-k has +a_k in column s
            tterm(s + k, -ak);       // row s+k has -a_k in column s
        }
    } else {
        int lo = s - Ord<O>::Q, hi = s + Ord<O>::Q;
        if (s < Ord<O>::NCOL) { lo = 0; hi = max(hi, Ord<O>::NB - 1); }
        if (s >= Nt - Ord<O>::NCOL) { hi = Nt - 1; lo = min(lo, Nt - Ord<O>::NB); }
        if (lo < 0) lo = 0;
        if (hi > Nt - 1) hi = Nt - 1;
        for (int sp = lo; sp <= hi; ++sp) {
            const T dc = dcoefT<O, T>(Nt, sp, s);
            if (dc == T(0)) continue;
            tterm(sp, dc * hweightT<O, T>(Nt, sp));
        }
    }
    const T tfac = (m == 0 ? ih2T<T>(B) : ih1T<T>(B)) / hweightT<O, T>(Nt, s);
    T f0 = half * tt0 * tfac - (z00 * w0 + z01 * w1);
    T f1 = half * tt1 * tfac - (z01 * w0 + z11 * w1);
    if (intf) {
        T tu0, tu1, tv0, tv1;
        const int sv = F.reversed ? nf - 1 - s : s;
        if (traced) {
            tu0 = trU[2 * nf + s];
            tu1 = trU[3 * nf + s];
            tv0 = trV[2 * nf + sv];
            tv1 = trV[3 * nf + sv];
        } else {
            face_traction<T, O>(B, F, s, u, c, tu0, tu1);
            face_traction<T, O>(*V, *FV, sv, uv, cv, tv0, tv1);
        }
        f0 -= T(0.5) * (tu0 + tv0);
        f1 -= T(0.5) * (tu1 + tv1);
    }
    Fs0 = inv_h0 * f0;
    Fs1 = inv_h0 * f1;
}

// The same terms in SAT_PARTS independent parts, for as many threads; adds the part's share to Fs, As.  Part 0 has As
// and what needs the face node alone; the others the normal and the tangential share of a Robin face's traction, or
// the taps of the tangential transpose.  Interfaces have their traces here (the callers' steps form them first).  Apart from
// face_sat_node, whose callers sum the terms of a node in one go and have few registers left for them.
constexpr int SAT_PARTS = 4;
// face_traction's part of the normal derivative (NORMAL) or of the tangential one, added to t0, t1
template <typename T, int O, bool NORMAL, class UA, class CA>
__device__ __forceinline__ void face_traction_part(const BlockDev& B, const FaceDev& F, int s, UA u, CA c, T& t0, T& t1) {
    const int m = F.m, Nm = m == 0 ? B.n1 : B.n2, Nt = m == 0 ? B.n2 : B.n1;
    const T ih = ((m == 0) == NORMAL ? ih1T<T>(B) : ih2T<T>(B));
    T d[2];
#pragma unroll
    for (int L = 0; L < 2; ++L)
        d[L] = NORMAL ? dsum<O, T>(Nm, F.side ? Nm - 1 : 0, [&](int j) {
                            int j1, j2;
                            face_at(B, F, s, F.side ? Nm - 1 - j : j, j1, j2);
                            return u(L, j1, j2);
                        }) * ih
                      : dsum<O, T>(Nt, s, [&](int j) {
                            int j1, j2;
                            face_at(B, F, j, 0, j1, j2);
                            return u(L, j1, j2);
                        }) * ih;
    int i1, i2;
    face_at(B, F, s, 0, i1, i2);
    const T nu = T(F.nu);
    auto pl = [&](int J, int L) { return NORMAL ? plane_nn(m, J, L) : plane_nt(m, J, L); };
    t0 += nu * (c(pl(0, 0), i1, i2) * d[0] + c(pl(0, 1), i1, i2) * d[1]);
    t1 += nu * (c(pl(1, 0), i1, i2) * d[0] + c(pl(1, 1), i1, i2) * d[1]);
}
template <typename T, int O, class UA, class CA>
__device__ __forceinline__ void face_sat_part(int part, const BlockDev* __restrict__ blocks, const BlockDev& B, const FaceDev& F,
                                              int s, const StepArgs& a, double beta, UA u, CA c, T& Fs0, T& Fs1, T& As0,
                                              T& As1) {
    const int m = F.m, nf = F.nf;
    const T nu = T(F.nu);
    const T inv_h0 = T(F.inv_h0);
    int i1, i2;
    face_at(B, F, s, 0, i1, i2);
    const bool has_data = a.with_data && F.g;
    const T* __restrict__ g = reinterpret_cast<const T*>(F.g);
    if (F.kind == FACE_ROBIN) {
        T f0 = T(0), f1 = T(0);
        if (part == 1) face_traction_part<T, O, true>(B, F, s, u, c, f0, f1);
        else if (part == 2) face_traction_part<T, O, false>(B, F, s, u, c, f0, f1);
        else if (part == 0) {
            if (F.ju) {
                const T u0 = u(0, i1, i2), u1 = u(1, i1, i2);
                const T* ju = reinterpret_cast<const T*>(F.ju);
                const T a11 = ju[s], a12 = ju[nf + s], a22 = ju[2 * nf + s];
                f0 = a11 * u0 + a12 * u1;
                f1 = a12 * u0 + a22 * u1;
            }
            if (has_data) {
#pragma unroll
                for (int k = 0; k < 8; ++k) {
                    if (k >= a.K) break;
                    f0 -= T(a.Tk[k]) * g[(size_t)k * nf + s];
                    f1 -= T(a.Tk[k]) * g[(size_t)(a.K + k) * nf + s];
                }
            }
        }
        Fs0 -= inv_h0 * f0;
        Fs1 -= inv_h0 * f1;
        return;
    }
    const bool intf = F.kind == FACE_INTF;
    // traces of both sides of an interface (k_face_trace, same level): the neighbour's displacement, both tractions and
    // the penalty
    const T* __restrict__ trU = intf ? reinterpret_cast<const T*>(F.tr) : nullptr;
    const T* __restrict__ trV = intf ? reinterpret_cast<const T*>(blocks[F.nbr_block].f[F.nbr_face].tr) : nullptr;
    // jump w_L at face node sp (displacement: u - g(t); interface: u - v)
    auto jump = [&](int sp, T& w0, T& w1) {
        int j1, j2;
        face_at(B, F, sp, 0, j1, j2);
        w0 = u(0, j1, j2);
        w1 = u(1, j1, j2);
        if (intf) {
            const int svp = F.reversed ? nf - 1 - sp : sp;
            w0 -= trV[svp];
            w1 -= trV[nf + svp];
        } else if (has_data) {
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                if (k >= a.K) break;
                w0 -= T(a.Tk[k]) * g[(size_t)k * nf + sp];
                w1 -= T(a.Tk[k]) * g[(size_t)(a.K + k) * nf + sp];
            }
        }
    };
    const T half = intf ? T(0.5) : T(1);
    if (part == 0) {
        const double dd = 2.0;   // spatial dimension d
        T w0, w1;
        jump(s, w0, w1);
        const T c00 = c(plane_nn(m, 0, 0), i1, i2), c01 = c(plane_nn(m, 0, 1), i1, i2), c11 = c(plane_nn(m, 1, 1), i1, i2);
        T z00, z01, z11;
        if (!intf) {
            const T k = T(beta * dd * F.inv_h0);
            z00 = k * c00; z01 = k * c01; z11 = k * c11;
        } else {
            const int sv = F.reversed ? nf - 1 - s : s;
            z00 = trU[4 * nf + s] + trV[4 * nf + sv];
            z01 = trU[5 * nf + s] + trV[5 * nf + sv];
            z11 = trU[6 * nf + s] + trV[6 * nf + sv];
        }
        // normal-spread amplitude a_J = half nu c_mJmL w_L
        As0 += half * nu * (c00 * w0 + c01 * w1);
        As1 += half * nu * (c01 * w0 + c11 * w1);
        T f0 = -(z00 * w0 + z01 * w1), f1 = -(z01 * w0 + z11 * w1);
        if (intf) {
            const int sv = F.reversed ? nf - 1 - s : s;
            f0 -= T(0.5) * (trU[2 * nf + s] + trV[2 * nf + sv]);
            f1 -= T(0.5) * (trU[3 * nf + s] + trV[3 * nf + sv]);
        }
        Fs0 += inv_h0 * f0;
        Fs1 += inv_h0 * f1;
        return;
    }
    // tangential transpose term (1/H_t(s)) sum_s' D_t[s'][s] H_t(s') b_J(s'),  b_J = nu c_mLtJ w_L;
    // rows of D with a non-zero in column s: the interior band s-Q..s+Q plus, near an end, every
    // boundary row (boundary rows span columns 0..NCOL-1, which can reach past s+Q)
    const int Nt = nf;
    T tt0 = T(0), tt1 = T(0);
    auto tterm = [&](int sp, T wgt) {
        T v0, v1;
        jump(sp, v0, v1);
        int j1, j2;
        face_at(B, F, sp, 0, j1, j2);
        tt0 += wgt * nu * (c(plane_nt(m, 0, 0), j1, j2) * v0 + c(plane_nt(m, 1, 0), j1, j2) * v1);
        tt1 += wgt * nu * (c(plane_nt(m, 0, 1), j1, j2) * v0 + c(plane_nt(m, 1, 1), j1, j2) * v1);
    };
    constexpr int TP = SAT_PARTS - 1;
    T tfac = m == 0 ? ih2T<T>(B) : ih1T<T>(B);
    if (s >= Ord<O>::NCOL && s < Nt - Ord<O>::NCOL) {
        // column s meets only interior rows s-Q..s+Q of D (weight 1): s-k with a_k and s+k with -a_k, k = part
        static_assert(Ord<O>::Q <= TP, "a part per tap distance");
        if (part <= Ord<O>::Q) {
            const T ak = Ord<O>::template aT<T>(part - 1);
            tterm(s - part, ak);
            tterm(s + part, -ak);
        }
    } else {
        int lo = s - Ord<O>::Q, hi = s + Ord<O>::Q;
        if (s < Ord<O>::NCOL) { lo = 0; hi = max(hi, Ord<O>::NB - 1); }
        if (s >= Nt - Ord<O>::NCOL) { hi = Nt - 1; lo = min(lo, Nt - Ord<O>::NB); }
        if (lo < 0) lo = 0;
        if (hi > Nt - 1) hi = Nt - 1;
        for (int sp = lo + part - 1; sp <= hi; sp += TP) {
            const T dc = dcoefT<O, T>(Nt, sp, s);
            if (dc == T(0)) continue;
            tterm(sp, dc * hweightT<O, T>(Nt, sp));
        }
        tfac /= hweightT<O, T>(Nt, s);
    }
    Fs0 += inv_h0 * half * tfac * tt0;
    Fs1 += inv_h0 * half * tfac * tt1;
}

// SAT terms of every face node from global memory into F.sat (face term 2 x nf, spread amplitude
// 2 x nf); used with k_boundary (the strip tile kernel computes them itself)
template <typename T, int O>
__global__ void k_face_sat(const BlockDev* __restrict__ blocks, const FaceRef* __restrict__ refs, int nrefs,
                           int total, StepArgs a, double beta) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= total) return;
    const FaceRef fr = refs[find_face(refs, nrefs, t)];
    const int s = t - fr.start;
    const BlockDev& B = blocks[fr.block];
    const FaceDev& F = B.f[fr.face];
    const size_t plane = (size_t)B.n2 * B.pitch;
    const T* __restrict__ U = reinterpret_cast<const T*>(B.u[a.cur]);
    const T* __restrict__ C = reinterpret_cast<const T*>(B.c);
    T f0, f1, a0, a1;
    face_sat_node<T, O>(blocks, B, F, s, a, beta,
                        [&](int L, int j1, int j2) { return U[(size_t)L * plane + (size_t)j2 * B.pitch + j1]; },
                        [&](int pl, int j1, int j2) { return C[(size_t)pl * plane + (size_t)j2 * B.pitch + j1]; },
                        f0, f1, a0, a1);
    T* sat = reinterpret_cast<T*>(F.sat);
    const int nf = F.nf;
    sat[s] = f0;
    sat[nf + s] = f1;
    sat[2 * nf + s] = a0;
    sat[3 * nf + s] = a1;
}

// One side's trace at every node of up to TRACE_MAX interface faces: u_L, the traction
// J^ tau_J = nu c_mJkL D_k u_L (eq. n-C_conversion) and this side's share k c_mJmL of the
// interface penalty Z (Sec. 6, k = beta d / 4 / H_m[0]); the SAT terms of both sides then read
// the neighbour from these short arrays (face_sat_node).  The face geometry travels in the
// kernel parameters, so every load of a thread (NCOL nodes along the normal, the tangential
// stencil, 7 coefficient planes) is independent of the others.
constexpr int TRACE_MAX = 8;
struct TraceFace {
    const void* u;            // current level of the block (2 planes), type T
    const void* c;            // coefficient planes
    void* tr;                 // FaceDev::tr of this face (7 x nf)
    long long plane;          // plane stride (elements)
    int nf, start;            // face nodes, first thread index of this face
    int m, side, pitch, nm;   // normal direction, high side, row pitch, nodes along the normal
    double nu, ihm, iht, k;   // outward normal component, 1/h_m, 1/h_t, penalty share factor
};
struct TraceArgs {
    TraceFace f[TRACE_MAX];
    int nfaces, total;
};

template <typename T, int O>
__global__ void k_face_trace(const __grid_constant__ TraceArgs ta) {
    using P = Ord<O>;
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= ta.total) return;
    int fi = 0;
    while (fi + 1 < ta.nfaces && t >= ta.f[fi + 1].start) ++fi;
    const TraceFace& F = ta.f[fi];
    const int s = t - F.start, m = F.m, nf = F.nf;
    const T* __restrict__ U = reinterpret_cast<const T*>(F.u);
    const T* __restrict__ C = reinterpret_cast<const T*>(F.c);
    // face node offset, step into the block along the normal, step along the face
    long long o0, sn, st;
    if (m == 0) {
        o0 = (long long)s * F.pitch + (F.side ? F.nm - 1 : 0);
        sn = F.side ? -1 : 1;
        st = F.pitch;
    } else {
        o0 = (long long)(F.side ? F.nm - 1 : 0) * F.pitch + s;
        sn = F.side ? -(long long)F.pitch : (long long)F.pitch;
        st = 1;
    }
    // every operand first, so that all the loads are in flight together (8.1 us for 8002 nodes; 9.4 with the loads in the sums)
    T cn[4], ct[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        cn[k] = C[plane_nn(m, k >> 1, k & 1) * F.plane + o0];
        ct[k] = C[plane_nt(m, k >> 1, k & 1) * F.plane + o0];
    }
    T un[2][P::NCOL];
#pragma unroll
    for (int L = 0; L < 2; ++L)
#pragma unroll
        for (int j = 0; j < P::NCOL; ++j) un[L][j] = U[L * F.plane + o0 + j * sn];
    T dn[2], dt[2];
#pragma unroll
    for (int L = 0; L < 2; ++L) {
        const T* UL = U + L * F.plane;
        // boundary row of D along the normal (mirrored, with the opposite sign, on the high side)
        T acc = T(0);
#pragma unroll
        for (int j = 0; j < P::NCOL; ++j) acc += P::template dqT<T>(0, j) * un[L][j];
        dn[L] = (F.side ? -acc : acc) * T(F.ihm);
        dt[L] = dsum<O, T>(nf, s, [&](int j) { return UL[o0 + (long long)(j - s) * st]; }) * T(F.iht);
    }
    const T nu = T(F.nu);
    const T t0 = nu * (cn[0] * dn[0] + cn[1] * dn[1] + ct[0] * dt[0] + ct[1] * dt[1]);
    const T t1 = nu * (cn[2] * dn[0] + cn[3] * dn[1] + ct[2] * dt[0] + ct[3] * dt[1]);
    const T k = T(F.k);
    T* tr = reinterpret_cast<T*>(F.tr);
    tr[s] = un[0][0];
    tr[nf + s] = un[1][0];
    tr[2 * nf + s] = t0;
    tr[3 * nf + s] = t1;
    tr[4 * nf + s] = k * cn[0];
    tr[5 * nf + s] = k * cn[1];
    tr[6 * nf + s] = k * cn[3];
}

// Closure matrices of one direction of a block (dir 0: along x1, lines = rows i2; dir 1: along
// x2, lines = columns i1) from the coefficient planes (b0, b1, b2 = planes 0..2 or 3..5),
// accumulated in FP64 and stored in T (layout of dxx_closure_mat).
template <typename T, int O>
__global__ void k_closure_mats(BlockDev B, int dir, T* __restrict__ M) {
    using P = Ord<O>;
    constexpr int NC = P::NCLOS, NJ = P::NCLOSJ;
    const int N = dir == 0 ? B.n1 : B.n2, lines = dir == 0 ? B.n2 : B.n1;
    const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= 2LL * NC * NJ * lines) return;
    const int line = (int)(t % lines);
    long long q = t / lines;
    const int j = (int)(q % NJ);
    q /= NJ;
    const int r = (int)(q % NC), side = (int)(q / NC);
    const size_t plane = (size_t)B.n2 * B.pitch;
    const T* __restrict__ C = reinterpret_cast<const T*>(B.c);
    const int p0 = dir == 0 ? 0 : 3;
    double m0 = 0.0, m1 = 0.0, m2 = 0.0;
    for (int tt = P::cstart(r); tt < P::cstart(r + 1); ++tt) {
        if (P::cj(tt) != j) continue;
        const int k = side ? N - 1 - P::ck(tt) : P::ck(tt);
        const size_t gi = dir == 0 ? (size_t)line * B.pitch + k : (size_t)k * B.pitch + line;
        const double c = P::cc(tt);
        m0 += c * (double)C[(size_t)p0 * plane + gi];
        m1 += c * (double)C[(size_t)(p0 + 1) * plane + gi];
        m2 += c * (double)C[(size_t)(p0 + 2) * plane + gi];
    }
    T* Mo = M + ((long long)((side * NC + r) * NJ + j) * 3) * lines + line;
    Mo[0] = T(m0);
    Mo[lines] = T(m1);
    Mo[2LL * lines] = T(m2);
}

// ============================================================================ boundary strips
// Every node within `strip` of a face: generic rows (closures from the tables), mixed terms
// with the boundary rows of D, plus the SAT contributions prepared by k_face_sat:
//   at depth d < NCOL from face f:  D_m[face row][i_m] / H_m[i_m] * a_J(s)   (D_m^T spread)
//   on the face itself:             the face term of k_face_sat
// One strip node: narrow terms (closure triples or interior edge weights), mixed terms with the
// boundary rows of D, SAT contributions of k_face_sat, forcing, and the leapfrog update.
// u0(j1, j2), u1(j1, j2): displacement components; cc(plane, j1, j2): coefficient planes.
template <typename T, int O, int MODE, class FU0, class FU1, class FC>
__device__ __forceinline__ void strip_node(const BlockDev& B, const StepArgs& a, int i1, int i2, FU0 u0, FU1 u1, FC cc) {
    const int n1 = B.n1, n2 = B.n2, P = B.pitch;
    const size_t plane = (size_t)n2 * P;
    const T ih1 = ih1T<T>(B), ih2 = ih2T<T>(B);
    T rx0 = T(0), rx1 = T(0), ry0 = T(0), ry1 = T(0);
    dxx_vec<O, T>(n1, i1, [&](int j) { return u0(j, i2); }, [&](int j) { return u1(j, i2); },
                  [&](int k) { return cc(0, k, i2); }, [&](int k) { return cc(1, k, i2); },
                  [&](int k) { return cc(2, k, i2); }, rx0, rx1);
    dxx_vec<O, T>(n2, i2, [&](int j) { return u0(i1, j); }, [&](int j) { return u1(i1, j); },
                  [&](int k) { return cc(3, i1, k); }, [&](int k) { return cc(4, i1, k); },
                  [&](int k) { return cc(5, i1, k); }, ry0, ry1);
    T r0 = rx0 * ih1 * ih1 + ry0 * ih2 * ih2;
    T r1 = rx1 * ih1 * ih1 + ry1 * ih2 * ih2;
    {
        int lo, hi;
        drow_range<O>(n1, i1, lo, hi);
        T s0 = T(0), s1 = T(0);
        for (int aa = lo; aa <= hi; ++aa) {
            const T d = dcoefT<O, T>(n1, i1, aa);
            if (d == T(0)) continue;
            const T du0 = dsum<O, T>(n2, i2, [&](int bb) { return u0(aa, bb); }) * ih2;
            const T du1 = dsum<O, T>(n2, i2, [&](int bb) { return u1(aa, bb); }) * ih2;
            s0 += d * (cc(6, aa, i2) * du0 + cc(7, aa, i2) * du1);
            s1 += d * (cc(8, aa, i2) * du0 + cc(9, aa, i2) * du1);
        }
        r0 += s0 * ih1;
        r1 += s1 * ih1;
        drow_range<O>(n2, i2, lo, hi);
        s0 = T(0);
        s1 = T(0);
        for (int bb = lo; bb <= hi; ++bb) {
            const T d = dcoefT<O, T>(n2, i2, bb);
            if (d == T(0)) continue;
            const T du0 = dsum<O, T>(n1, i1, [&](int aa) { return u0(aa, bb); }) * ih1;
            const T du1 = dsum<O, T>(n1, i1, [&](int aa) { return u1(aa, bb); }) * ih1;
            s0 += d * (cc(6, i1, bb) * du0 + cc(8, i1, bb) * du1);
            s1 += d * (cc(7, i1, bb) * du0 + cc(9, i1, bb) * du1);
        }
        r0 += s0 * ih2;
        r1 += s1 * ih2;
    }
#pragma unroll
    for (int f = 0; f < 4; ++f) {
        const FaceDev& F = B.f[f];
        const int m = F.m;
        const int im = m == 0 ? i1 : i2, Nm = m == 0 ? n1 : n2;
        const int d = F.side ? Nm - 1 - im : im;
        if (d >= Ord<O>::NCOL) continue;
        const int s = m == 0 ? i2 : i1;
        const T* __restrict__ sat = reinterpret_cast<const T*>(F.sat);
        const int nf = F.nf;
        const T fac = facT<T>(F, d);
        r0 += fac * sat[2 * nf + s];
        r1 += fac * sat[3 * nf + s];
        if (d == 0) {
            r0 += sat[s];
            r1 += sat[nf + s];
        }
    }
    const size_t gi = (size_t)i2 * P + i1;
    if (a.with_data && B.jf) {
        const T* __restrict__ JF = reinterpret_cast<const T*>(B.jf);
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            if (k >= a.K) break;
            r0 += T(a.Tk[k]) * JF[(size_t)k * plane + gi];
            r1 += T(a.Tk[k]) * JF[(size_t)(a.K + k) * plane + gi];
        }
    }
    if (MODE == 0) {
        T* __restrict__ Un = reinterpret_cast<T*>(B.u[1 - a.cur]);
        const T wv = reinterpret_cast<const T*>(B.w)[gi], dt2 = dt2T<T>(a);
        Un[gi] = T(2) * u0(i1, i2) - Un[gi] + dt2 * wv * r0;
        Un[gi + plane] = T(2) * u1(i1, i2) - Un[gi + plane] + dt2 * wv * r1;
    } else {
        T* __restrict__ R = reinterpret_cast<T*>(B.r);
        R[gi] = r0;
        R[gi + plane] = r1;
    }
}

template <typename T, int O, int MODE>
__global__ void __launch_bounds__(256) k_boundary(BlockDev B, StepArgs a) {
    const int n1 = B.n1, n2 = B.n2, P = B.pitch, S = B.strip;
    const long long nstrip = (long long)n1 * n2 - (long long)(n1 - 2 * S) * (n2 - 2 * S);
    const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= nstrip) return;
    int i1, i2;
    {
        const long long top = (long long)S * n1;
        if (t < top) { i2 = (int)(t / n1); i1 = (int)(t - (long long)i2 * n1); }
        else if (t < 2 * top) { long long u = t - top; i2 = n2 - S + (int)(u / n1); i1 = (int)(u - (long long)(i2 - n2 + S) * n1); }
        else {
            long long u = t - 2 * top;
            const int row = (int)(u / (2 * S)), k = (int)(u - (long long)row * 2 * S);
            i2 = S + row;
            i1 = k < S ? k : n1 - 2 * S + k;
        }
    }
    const size_t plane = (size_t)n2 * P;
    const T* __restrict__ U0 = reinterpret_cast<const T*>(B.u[a.cur]);
    const T* __restrict__ U1 = U0 + plane;
    const T* __restrict__ C = reinterpret_cast<const T*>(B.c);
    strip_node<T, O, MODE>(
        B, a, i1, i2, [&](int j1, int j2) { return __ldg(U0 + (size_t)j2 * P + j1); },
        [&](int j1, int j2) { return __ldg(U1 + (size_t)j2 * P + j1); },
        [&](int pl, int j1, int j2) { return __ldg(C + pl * plane + (size_t)j2 * P + j1); });
}

// ============================================================================ point-source tables
struct SrcNode {
    int block, src;
    long long gi;             // node offset in the planes
    double wt0, wt1;          // dir_J * amplitude * w1 w2 / H
};
struct SrcParam {
    double alpha_p, t0;
};
// Ricker wavelet W(t) of a point source at the step's time (Sec. 7.4); graph mode reads the time of
// the captured step from the device array the host uploads
__device__ __forceinline__ double ricker_at(const SrcParam& p, const StepArgs& a) {
    const double tnow = a.tdev ? a.tdev[a.tstep] : a.t;
    const double x = 3.14159265358979323846 * p.alpha_p * (tnow - p.t0);
    return (1.0 - 2.0 * x * x) * exp(-x * x);
}

// ============================================================================ boundary strips, tiled
// The strips are cut into tiles of TL (32) nodes along the face x (strip width) nodes across it:
// bottom and top bands (tiles along x1), left and right bands (tiles along x2, between the
// bands).  The tile's region of the 2 displacement and 10 coefficient planes is staged in shared
// memory: for band tiles one elected thread issues two cp.async.bulk.tensor loads (a bounded
// mbarrier wait; on timeout the CTA sets bit 8 of the error flag, waits once more for its copies
// and returns); side tiles copy their narrow rows element-wise (cp.async) into rows of odd
// stride, since their warps walk columns.  Region extents:
//   across the face: the strip plus HN = Q nodes (the farthest reach past the strip of a closure
//     triple of D_xx^FC, of an interior edge weight and of the mixed terms);
//   along the face:  the tile plus HT nodes each side (the backward reach Q - LO of the edge
//     weights, rounded up to 4 so that the box starts on a 16-byte boundary).  Band tiles stage
//     the window of the 32 columns [xc, xc + 32), xc = min(x0, n1 - 32), so that the narrow last
//     tile still holds the whole closure of the block corner.
// The mixed fluxes g1_j = c_1j2l D_2 u_l (on the tile's rows) and g2_j = c_1l2j D_1 u_l (on its
// columns) are formed once per staged node, and the SAT terms of the tile's face nodes (every
// face whose first NCOL nodes the tile touches) are formed from the staged data (interfaces read
// the traces of k_face_trace), so every output node needs only the narrow rows, two <= NCOL-tap
// sums and shared-memory SAT terms.
//
// TL, the tile's length along the face: 32 in FP32 (a warp per row).  In FP64 the tile's arithmetic holds
// its SM (see k_interior_edges), so small grids are cut shorter, 16 or 8 nodes, until the tiles spread
// over all SMs (the host picks; the halo along the face repeats more of the fluxes the shorter the tile).
template <int O, int TL = 32, bool SPLIT = false> struct StripTile {
    static constexpr int Q = Ord<O>::Q;
    static constexpr int S = Ord<O>::NCLOS > Ord<O>::NCOL ? Ord<O>::NCLOS : Ord<O>::NCOL;
    static constexpr int HN = Q;
    static constexpr int HT = (Q - EdgeRange<O>::LO + 3) / 4 * 4;
    static constexpr int BWB = TL + 2 * HT + 4, BHB = S + HN;            // band box (tiles along x1)
    static constexpr int CWS = S + HN, BWS = CWS | 1, BHS = TL + 2 * HT; // side region: CWS columns, odd stride
    static constexpr int RMAX = BWB * BHB > BWS * BHS ? BWB * BHB : BWS * BHS;
    static constexpr int FLUXB = 2 * (S * BWB + BHB * TL), FLUXS = 2 * (TL * BWS + BHS * S);
    static constexpr int FLUX = FLUXB > FLUXS ? FLUXB : FLUXS;   // g1 on the tile rows, g2 on its columns
    static constexpr int FN = TL > S ? TL : S;          // face nodes of a tile: along it, or across it at a corner
    static constexpr int SN = 2 + 2 * (SPLIT ? SAT_PARTS : 1);   // per face node: As0, As1, and Fs0, Fs1 of each part
    static constexpr int SATS = 4 * FN * SN;
    static constexpr int THREADS = TL * S < 128 ? 128 : (TL * S + 31) / 32 * 32;
    // element offset of the coefficient box (128-byte aligned TMA destination), of the fluxes, and bytes
    template <typename T> static constexpr int coff() { return (int)((2 * RMAX * sizeof(T) + 127) / 128 * 128 / sizeof(T)); }
    template <typename T> static constexpr int foff() { return coff<T>() + 10 * RMAX; }
    template <typename T> static constexpr size_t bar_off() { return ((foff<T>() + FLUX + SATS) * sizeof(T) + 15) / 16 * 16; }
    template <typename T> static constexpr size_t bytes() { return bar_off<T>() + 16; }
};

// One launch covers the strips of every block: tiles[blockIdx.x] = (block, tile of that block,
// first and end index of the tile's point-source nodes in ssrc), ordered by the host so that the
// costliest tiles (interface bands, side bands) start first.  B.smaps holds the block's band-box
// tensor maps: u[0], u[1], c.  Point-source nodes inside the strips are added here (ssrc null:
// none, e.g. on the adjoint fields); the host launches k_sources only for interior source nodes.
// The body of one strip tile, by the NT threads of the calling CTA (NT a multiple of 32; with fewer
// than 32 S threads a warp takes several output rows).  Returns false when the bounded wait for
// the tile's staging copies ran out (the error word is set).  The staging mbarrier is
// invalidated before the return, so a persistent caller can reuse the shared memory for its next
// tile after a CTA barrier.
// SPLIT: a warp per part of the SAT terms.  One thread for all of a face node's terms is the tile's longest chain of
// dependent operations: the one-launch steps, which wait for it, gain (FP32 order 6: 101^2 20.6 -> 16.5 us, 601^2
// 24.8 -> 22.7; FP64 order 4: 101^2 31 -> 27), where many tiles fill the chip the repeated indexing costs (2 x
// 802 x 401: 43.4 -> 45.3 us).
template <typename T, int O, int MODE, int NT, int TL = 32, bool SPLIT = false>
__device__ __forceinline__ bool strip_tile_body(const BlockDev* __restrict__ blocks, const int4 tt, const StepArgs& a,
                                                double beta, int* err, const SrcNode* __restrict__ ssrc,
                                                const SrcParam* __restrict__ spar, unsigned char* strip_smem) {
    using ST = StripTile<O, TL, SPLIT>;
    constexpr int S = ST::S;
    T* sm = reinterpret_cast<T*>(strip_smem);
    uint64_t* bar = reinterpret_cast<uint64_t*>(strip_smem + ST::template bar_off<T>());
    const BlockDev& B = blocks[tt.x];
    const int n1 = B.n1, n2 = B.n2, P = B.pitch;
    const int nbx = (n1 + TL - 1) / TL, nby = (n2 - 2 * S + TL - 1) / TL;
    int t = tt.y, x0, y0, w, h, xs, ys, BW, BH, VW;   // VW: staged columns (BW: row stride)
    bool along_x;
    if (t < 2 * nbx) {
        along_x = true;
        const int band = t / nbx;
        x0 = (t - band * nbx) * TL;
        w = min(TL, n1 - x0);
        y0 = band ? n2 - S : 0;
        h = S;
        const int xc = min(x0, max(0, n1 - TL));
        xs = (xc & ~3) - ST::HT;
        ys = band ? n2 - S - ST::HN : 0;
        BW = VW = ST::BWB;
        BH = ST::BHB;
    } else {
        t -= 2 * nbx;
        along_x = false;
        const int side = t / nby;
        y0 = S + (t - side * nby) * TL;
        h = min(TL, n2 - S - y0);
        x0 = side ? n1 - S : 0;
        w = S;
        xs = side ? n1 - ST::CWS : 0;
        ys = y0 - ST::HT;
        BW = ST::BWS;
        VW = ST::CWS;
        BH = ST::BHS;
    }
    const int PS = BW * BH;                     // plane stride of the staged boxes
    const size_t plane = (size_t)n2 * P;
    // stage the tile's region (2 displacement planes at sm, 10 coefficient planes at sm + coff)
    if (along_x) {
        if (threadIdx.x == 0) {
            mbar_init(bar, 1);
            fence_barrier_init();
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            // the region may have been read and written by this CTA's threads for an earlier tile
            // (persistent callers): order those accesses before the bulk copies overwrite it
            fence_proxy_async();
            // (FP32 handles have a second set of maps for short tiles)
            const CUtensorMap* maps = reinterpret_cast<const CUtensorMap*>(B.smaps) + (sizeof(T) == 4 && TL != 32 ? 6 : 0);
            mbar_expect_tx(bar, (uint32_t)(12 * PS * sizeof(T)));
            tma_load_3d(sm, &maps[a.cur], xs, ys, 0, bar);
            tma_load_3d(sm + ST::template coff<T>(), &maps[2], xs, ys, 0, bar);
        }
        const bool staged = mbar_wait_bounded(bar, 0);
        if (__syncthreads_or(!staged)) {
            if (threadIdx.x == 0) {
                atomicOr(err, ERR_STRIP_WAIT);
                mbar_wait_bounded(bar, 0);
            }
            return false;
        }
        if (threadIdx.x == 0) mbar_inval(bar);   // every thread has seen the phase complete
    } else {
        const T* __restrict__ U = reinterpret_cast<const T*>(B.u[a.cur]);
        const T* __restrict__ C = reinterpret_cast<const T*>(B.c);
        const int r0 = max(0, ys), r1 = min(n2, ys + BH), nel = (r1 - r0) * ST::CWS;
        for (int pl = 0; pl < 12; ++pl) {
            const T* src = pl < 2 ? U + pl * plane : C + (pl - 2) * plane;
            T* dst = pl < 2 ? sm + pl * PS : sm + ST::template coff<T>() + (pl - 2) * PS;
            for (int e = threadIdx.x; e < nel; e += NT) {
                const int r = e / ST::CWS, c = e - r * ST::CWS;
                const unsigned sa = (unsigned)__cvta_generic_to_shared(dst + (r0 + r - ys) * BW + c);
                const T* gp = src + (size_t)(r0 + r) * P + xs + c;
                if (sizeof(T) == 8)
                    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(sa), "l"(gp) : "memory");
                else
                    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(sa), "l"(gp) : "memory");
            }
        }
        asm volatile("cp.async.commit_group;\ncp.async.wait_all;" ::: "memory");
        __syncthreads();
    }
    auto at = [&](int pl, int j1, int j2) -> T& {
        T* base = pl < 2 ? sm + pl * PS : sm + ST::template coff<T>() + (pl - 2) * PS;
        return base[(j2 - ys) * BW + (j1 - xs)];
    };
    // g1_J (J = 0, 1) at (j1, j2), j2 in the tile rows; g2_J at (j1, j2), j1 in the tile columns
    T* g1s = sm + ST::template foff<T>();
    T* g2s = g1s + 2 * h * BW;
    auto g1 = [&](int J, int j1, int j2) -> T& { return g1s[(J * h + (j2 - y0)) * BW + (j1 - xs)]; };
    auto g2 = [&](int J, int j1, int j2) -> T& { return g2s[(J * BH + (j2 - ys)) * w + (j1 - x0)]; };
    const T ih1 = ih1T<T>(B), ih2 = ih2T<T>(B);
    // SAT terms of the face nodes whose first NCOL nodes meet the tile: face f's tangential range
    // is the tile's y range (f = 0, 1) or x range (f = 2, 3)
    T* sats = sm + ST::template foff<T>() + ST::FLUX;
    auto face_meets = [&](int f) {
        if (f < 2) return f == 0 ? x0 < Ord<O>::NCOL : x0 + w > n1 - Ord<O>::NCOL;
        return f == 2 ? y0 < Ord<O>::NCOL : y0 + h > n2 - Ord<O>::NCOL;
    };
    // (split: two groups of warps where the CTA has eight, each with every other face)
    if constexpr (SPLIT) {
        const int wid = threadIdx.x >> 5, part = wid % SAT_PARTS, group = wid / SAT_PARTS;
        constexpr int GROUPS = NT / 32 / SAT_PARTS;
        static_assert(GROUPS >= 1, "a warp for every part");
        int nth = 0;
        for (int f = 0; f < 4; ++f) {
            if (!face_meets(f)) continue;
            if (nth++ % GROUPS != group) continue;
            for (int k = threadIdx.x & 31; k < (f < 2 ? h : w); k += 32) {
                T f0 = T(0), f1 = T(0), a0 = T(0), a1 = T(0);
                face_sat_part<T, O>(part, blocks, B, B.f[f], (f < 2 ? y0 : x0) + k, a, beta,
                                    [&](int L, int j1, int j2) { return at(L, j1, j2); },
                                    [&](int pl, int j1, int j2) { return at(2 + pl, j1, j2); }, f0, f1, a0, a1);
                T* q = sats + (f * ST::FN + k) * ST::SN;
                if (part == 0) {
                    q[0] = a0;
                    q[1] = a1;
                }
                q[2 + 2 * part] = f0;
                q[3 + 2 * part] = f1;
            }
        }
    }
    // g1 on the tile's rows (the staged columns inside the block), g2 on the tile's columns (the
    // staged rows inside the block)
    const int cx0 = max(0, xs), cx1 = min(n1, xs + VW), RWc = cx1 - cx0;
    const int cy0 = max(0, ys), cy1 = min(n2, ys + BH), RHc = cy1 - cy0;
    for (int idx = threadIdx.x; idx < h * RWc; idx += NT) {
        const int r = idx / RWc, c = idx - r * RWc;
        const int j1 = cx0 + c, j2 = y0 + r;
        const T d0 = dsum<O, T>(n2, j2, [&](int bb) { return at(0, j1, bb); }) * ih2;
        const T d1 = dsum<O, T>(n2, j2, [&](int bb) { return at(1, j1, bb); }) * ih2;
        g1(0, j1, j2) = at(8, j1, j2) * d0 + at(9, j1, j2) * d1;
        g1(1, j1, j2) = at(10, j1, j2) * d0 + at(11, j1, j2) * d1;
    }
    for (int idx = threadIdx.x; idx < RHc * w; idx += NT) {
        const int r = idx / w, c = idx - r * w;
        const int j1 = x0 + c, j2 = cy0 + r;
        const T d0 = dsum<O, T>(n1, j1, [&](int aa) { return at(0, aa, j2); }) * ih1;
        const T d1 = dsum<O, T>(n1, j1, [&](int aa) { return at(1, aa, j2); }) * ih1;
        g2(0, j1, j2) = at(8, j1, j2) * d0 + at(10, j1, j2) * d1;
        g2(1, j1, j2) = at(9, j1, j2) * d0 + at(11, j1, j2) * d1;
    }
    if constexpr (!SPLIT) {
        for (int idx = threadIdx.x; idx < 4 * ST::FN; idx += NT) {
            const int f = idx / ST::FN, k = idx % ST::FN;
            if (k >= (f < 2 ? h : w) || !face_meets(f)) continue;
            T f0, f1, a0, a1;
            face_sat_node<T, O>(blocks, B, B.f[f], (f < 2 ? y0 : x0) + k, a, beta,
                                [&](int L, int j1, int j2) { return at(L, j1, j2); },
                                [&](int pl, int j1, int j2) { return at(2 + pl, j1, j2); }, f0, f1, a0, a1);
            T* q = sats + (f * ST::FN + k) * ST::SN;
            q[0] = a0;
            q[1] = a1;
            q[2] = f0;
            q[3] = f1;
        }
    }
    __syncthreads();
    // output node of this thread: a warp per row of a band tile (lanes along the row), a warp per
    // column of a side tile (lanes along the column: one closure row per warp, and the odd row
    // stride of the side staging keeps the column accesses free of bank conflicts)
    auto out_node = [&](const int lane, const int wid) {
        const int i1 = along_x ? x0 + lane : x0 + wid;
        const int i2 = along_x ? y0 + wid : y0 + lane;
        if (i1 >= x0 + w || i2 >= y0 + h) return;
        // narrow rows: closure rows through the precomputed matrices, interior rows by edge weights (in
        // FP64 read from memory, where they are over h^2 already: into e0, e1)
        T rx0v = T(0), rx1v = T(0), ry0v = T(0), ry1v = T(0), e0 = T(0), e1 = T(0);
        const T* __restrict__ E = sizeof(T) == 8 ? reinterpret_cast<const T*>(B.e) : nullptr;
        const size_t gi = (size_t)i2 * P + i1;
        if (!dxx_closure_mat<O, T>(n1, i1, i2, n2, reinterpret_cast<const T*>(B.mx), [&](int j) { return at(0, j, i2); },
                                   [&](int j) { return at(1, j, i2); }, rx0v, rx1v)) {
            if (sizeof(T) == 8 && E)
                dxx_edges<O, T>(i1, [&](int j) { return at(0, j, i2); }, [&](int j) { return at(1, j, i2); },
                                [&](int f, int m, int k) { return __ldg(E + (size_t)edge_plane<O>(0, f, m) * plane + gi + (k - i1)); },
                                e0, e1);
            else dxx_interior<O, T>(i1, [&](int j) { return at(0, j, i2); }, [&](int j) { return at(1, j, i2); },
                               [&](int k) { return at(2, k, i2); }, [&](int k) { return at(3, k, i2); },
                               [&](int k) { return at(4, k, i2); }, rx0v, rx1v);
        }
        if (!dxx_closure_mat<O, T>(n2, i2, i1, n1, reinterpret_cast<const T*>(B.my), [&](int j) { return at(0, i1, j); },
                                   [&](int j) { return at(1, i1, j); }, ry0v, ry1v)) {
            if (sizeof(T) == 8 && E)
                dxx_edges<O, T>(i2, [&](int j) { return at(0, i1, j); }, [&](int j) { return at(1, i1, j); },
                                [&](int f, int m, int k) { return __ldg(E + (size_t)edge_plane<O>(1, f, m) * plane + gi + (long long)(k - i2) * P); },
                                e0, e1);
            else dxx_interior<O, T>(i2, [&](int j) { return at(0, i1, j); }, [&](int j) { return at(1, i1, j); },
                               [&](int k) { return at(5, i1, k); }, [&](int k) { return at(6, i1, k); },
                               [&](int k) { return at(7, i1, k); }, ry0v, ry1v);
        }
        T r0 = rx0v * ih1 * ih1 + ry0v * ih2 * ih2;
        T r1 = rx1v * ih1 * ih1 + ry1v * ih2 * ih2;
        if (sizeof(T) == 8) {
            r0 += e0;
            r1 += e1;
        }
        r0 += dsum<O, T>(n1, i1, [&](int aa) { return g1(0, aa, i2); }) * ih1 +
              dsum<O, T>(n2, i2, [&](int bb) { return g2(0, i1, bb); }) * ih2;
        r1 += dsum<O, T>(n1, i1, [&](int aa) { return g1(1, aa, i2); }) * ih1 +
              dsum<O, T>(n2, i2, [&](int bb) { return g2(1, i1, bb); }) * ih2;
    #pragma unroll
        for (int f = 0; f < 4; ++f) {
            const FaceDev& F = B.f[f];
            const int m = F.m;
            const int im = m == 0 ? i1 : i2, Nm = m == 0 ? n1 : n2;
            const int d = F.side ? Nm - 1 - im : im;
            if (d >= Ord<O>::NCOL) continue;
            const T* q = sats + (f * ST::FN + (m == 0 ? i2 - y0 : i1 - x0)) * ST::SN;
            const T fac = facT<T>(F, d);
            r0 += fac * q[0];
            r1 += fac * q[1];
            if (d == 0) {
#pragma unroll
                for (int p = 0; p < (SPLIT ? SAT_PARTS : 1); ++p) {
                    r0 += q[2 + 2 * p];
                    r1 += q[3 + 2 * p];
                }
            }
        }
        if (a.with_data && B.jf) {
            const T* __restrict__ JF = reinterpret_cast<const T*>(B.jf);
    #pragma unroll
            for (int k = 0; k < 8; ++k) {
                if (k >= a.K) break;
                r0 += T(a.Tk[k]) * JF[(size_t)k * plane + gi];
                r1 += T(a.Tk[k]) * JF[(size_t)(a.K + k) * plane + gi];
            }
        }
        // point-source nodes of this tile: J f_J = dir_J amp W(t) w1 w2 / H (Sec. 7.4, discrete delta)
        if (ssrc && a.with_data) {
            for (int k = tt.z; k < tt.w; ++k) {
                const SrcNode nd = ssrc[k];
                if (nd.gi != (long long)gi) continue;
                const double Wt = ricker_at(spar[nd.src], a);
                r0 += T(Wt * nd.wt0);
                r1 += T(Wt * nd.wt1);
            }
        }
        T dd00, dd01, dd11;
        const bool damped = MODE != 1 && robin_damping_at<T>(B, i1, i2, dd00, dd01, dd11);
        if (MODE == 0) {
            leapfrog_store<T>(B, a, gi, plane, at(0, i1, i2), at(1, i1, i2), reinterpret_cast<const T*>(B.w)[gi], r0, r1,
                              damped, dd00, dd01, dd11);
        } else if (MODE == 2) {
            if (damped) {
                T v0, v1;
                rk4_stage_velocity<T>(B, a.stage, rkhT<T>(a), gi, plane, v0, v1);
                r0 -= dd00 * v0 + dd01 * v1;
                r1 -= dd01 * v0 + dd11 * v1;
            }
            rk4_store<T>(B, a, gi, plane, reinterpret_cast<const T*>(B.w)[gi], r0, r1);
        } else {
            T* __restrict__ R = reinterpret_cast<T*>(B.r);
            R[gi] = r0;
            R[gi + plane] = r1;
        }
    };
    // one pass when the CTA has a thread per node (the strip kernel), else a loop
    if constexpr (NT == TL * S) out_node((int)(threadIdx.x % TL), (int)(threadIdx.x / TL));
    else
        for (int idx = threadIdx.x; idx < TL * S; idx += NT) out_node(idx % TL, idx / TL);
    return true;
}

template <typename T, int O, int MODE, int TL>
__global__ void __launch_bounds__(StripTile<O, TL>::THREADS, sizeof(T) == 4 ? 4 : (TL == 32 ? 2 : 4))
k_strip_tile(const BlockDev* __restrict__ blocks, const int4* __restrict__ tiles, StepArgs a, double beta, int* err,
             const SrcNode* __restrict__ ssrc, const SrcParam* __restrict__ spar) {
    extern __shared__ __align__(128) unsigned char strip_smem[];
    (void)strip_tile_body<T, O, MODE, StripTile<O, TL>::THREADS, TL>(blocks, tiles[blockIdx.x], a, beta, err, ssrc,
                                                                     spar, strip_smem);
}

// ============================================================================ point sources

// the share of source node nd in the step's output, after the node's own update
template <typename T, int MODE>
__device__ __forceinline__ void source_add(const BlockDev& B, const SrcNode& nd, const SrcParam* __restrict__ par, const StepArgs& a) {
    const double Wt = ricker_at(par[nd.src], a);
    const size_t plane = (size_t)B.n2 * B.pitch;
    if (MODE == 0) {
        // its share of dt^2 w r, into u^{n+1} and, in increment form, into d^{n+1}
        T* Un = reinterpret_cast<T*>(B.u[1 - a.cur]);
        T* DU = reinterpret_cast<T*>(B.du);
        const double fac = a.dt2 * (double)reinterpret_cast<const T*>(B.w)[nd.gi] * Wt;
        atomicAdd(Un + nd.gi, T(fac * nd.wt0));
        atomicAdd(Un + plane + nd.gi, T(fac * nd.wt1));
        if (DU) {
            atomicAdd(DU + nd.gi, T(fac * nd.wt0));
            atomicAdd(DU + plane + nd.gi, T(fac * nd.wt1));
        }
    } else if (MODE == 2) {
        // RK4, after the stage's kernels: the source's share of a_s, or of v_new = v + ... + h/6 a_4
        // (no stage input before the next stage depends on a_s: rk4_store)
        T* R = reinterpret_cast<T*>(B.rk) + (size_t)(a.stage < 4 ? 2 + 2 * a.stage : 2) * plane;
        const double fac = (double)reinterpret_cast<const T*>(B.w)[nd.gi] * Wt * (a.stage < 4 ? 1.0 : a.rkh / 6.0);
        atomicAdd(R + nd.gi, T(fac * nd.wt0));
        atomicAdd(R + plane + nd.gi, T(fac * nd.wt1));
    } else {
        T* R = reinterpret_cast<T*>(B.r);
        atomicAdd(R + nd.gi, T(Wt * nd.wt0));
        atomicAdd(R + plane + nd.gi, T(Wt * nd.wt1));
    }
}

template <typename T, int MODE>
__global__ void k_sources(const BlockDev* __restrict__ blocks, const SrcNode* __restrict__ nodes, int nnodes,
                          const SrcParam* __restrict__ par, StepArgs a) {
    const int tid = blockIdx.x * blockDim.x + threadIdx.x;
    if (tid >= nnodes || !a.with_data) return;
    const SrcNode nd = nodes[tid];
    source_add<T, MODE>(blocks[nd.block], nd, par, a);
}

// ============================================================================ wait probe
// Diagnostic for the kernels' timeout path: one thread waits, with the bounded wait the step
// kernels use, on an mbarrier that nothing ever arrives at (no copy is issued, so nothing is in
// flight); when its `polls` polls run out it sets ERR_SELFTEST_WAIT in the error word.
static __global__ void k_wait_probe(int polls, int* err) {
    __shared__ __align__(8) uint64_t bar;
    if (threadIdx.x == 0) {
        mbar_init(&bar, 1);
        fence_barrier_init();
    }
    __syncthreads();
    if (threadIdx.x == 0 && !mbar_wait_bounded(&bar, 0, polls)) atomicOr(err, ERR_SELFTEST_WAIT);
}

// ============================================================================ l2 distances
// sum over nodes of (u_J - ref_J) (J H) (u_J - ref_J) and ref_J (J H) ref_J (FP64 accumulation);
// ref is dense host layout (2 planes of n1*n2, x1 fastest)
template <typename T, int O>
__global__ void k_l2_diff(BlockDev B, const T* __restrict__ U, const double* __restrict__ ref, double* out) {
    const long long n = (long long)B.n1 * B.n2;
    double se = 0.0, sr = 0.0;
    for (long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x; t < n; t += (long long)gridDim.x * blockDim.x) {
        const int i2 = (int)(t / B.n1), i1 = (int)(t - (long long)i2 * B.n1);
        const size_t plane = (size_t)B.n2 * B.pitch, gi = (size_t)i2 * B.pitch + i1;
        const double wq = B.J[gi] * B.h1 * hweight<O>(B.n1, i1) * B.h2 * hweight<O>(B.n2, i2);
        const double r0 = ref[t], r1 = ref[n + t];
        const double e0 = (double)U[gi] - r0, e1 = (double)U[plane + gi] - r1;
        se += wq * (e0 * e0 + e1 * e1);
        sr += wq * (r0 * r0 + r1 * r1);
    }
    for (int o = 16; o > 0; o >>= 1) {
        se += __shfl_down_sync(0xffffffffu, se, o);
        sr += __shfl_down_sync(0xffffffffu, sr, o);
    }
    if ((threadIdx.x & 31) == 0) {
        atomicAdd(out, se);
        atomicAdd(out + 1, sr);
    }
}

// ============================================================================ layer dissipation
// Super-grid layer dissipation (Sec. 7.3; reading: J E = -H^-1 sum_i Dt_i^T diag(s) Dt_i per
// component, Dt_i the undivided second difference along x_i at the nodes 1 .. N-2 of a line, s >= 0
// the layer coefficient of the node at the difference's centre).  (H^-1 K v)(i1, i2) for a field
// v(j1, j2, component):
template <typename T, int O, class FV>
__device__ __forceinline__ void layer_kv(const BlockDev& B, int i1, int i2, FV v, T& k0, T& k1) {
    const T* __restrict__ S = reinterpret_cast<const T*>(B.sg);
    const int P = B.pitch;
    k0 = k1 = T(0);
#pragma unroll
    for (int dir = 0; dir < 2; ++dir) {
        const int N = dir == 0 ? B.n1 : B.n2, j = dir == 0 ? i1 : i2;
#pragma unroll
        for (int o = -1; o <= 1; ++o) {
            const int c = j + o;
            if (c < 1 || c > N - 2) continue;
            const int c1 = dir == 0 ? c : i1, c2 = dir == 0 ? i2 : c;
            const T sc = S[(size_t)c2 * P + c1];
            if (sc == T(0)) continue;
            const int e1 = dir == 0 ? 1 : 0, e2 = 1 - e1;
            const T coef = o == 0 ? T(-2) : T(1);
            const T d0 = v(c1 - e1, c2 - e2, 0) - T(2) * v(c1, c2, 0) + v(c1 + e1, c2 + e2, 0);
            const T d1 = v(c1 - e1, c2 - e2, 1) - T(2) * v(c1, c2, 1) + v(c1 + e1, c2 + e2, 1);
            k0 += coef * sc * d0;
            k1 += coef * sc * d1;
        }
    }
    const T ih = T(1.0 / (B.h1 * hweight<O>(B.n1, i1) * B.h2 * hweight<O>(B.n2, i2)));
    k0 *= ih;
    k1 *= ih;
}

// leapfrog, before the step: d = H^-1 K (u^n - u^{n-1}) / dt at the listed nodes (the backward
// velocity; u^{n-1} is overwritten by the step kernels)
template <typename T, int O>
__global__ void k_layer_pre(BlockDev B, const int2* __restrict__ nodes, int n, int cur, double idt, T* __restrict__ d) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n) return;
    const int2 nd = nodes[k];
    const size_t plane = (size_t)B.n2 * B.pitch;
    const T* __restrict__ U = reinterpret_cast<const T*>(B.u[cur]);
    const T* __restrict__ Up = reinterpret_cast<const T*>(B.u[1 - cur]);
    const T* __restrict__ DU = reinterpret_cast<const T*>(B.du);
    T k0, k1;
    layer_kv<T, O>(B, nd.x, nd.y, [&](int j1, int j2, int c) {
        const size_t g = (size_t)c * plane + (size_t)j2 * B.pitch + j1;
        return DU ? DU[g] : U[g] - Up[g];
    }, k0, k1);
    d[k] = k0 * T(idt);
    d[n + k] = k1 * T(idt);
}

// leapfrog, after the step: u^{n+1} -= dt^2 w d at the listed nodes (and d^{n+1} in increment form).  The layer term belongs to the
// right-hand side of the step, so at a face node with the dissipative Robin term (where the step
// solved (I + dt/2 w D) u^{n+1} = rhs) the correction is M^-1 (dt^2 w d), M = I + dt/2 w D.
template <typename T>
__global__ void k_layer_post(BlockDev B, const int2* __restrict__ nodes, int n, int cur, double dt, const T* __restrict__ d) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n) return;
    const int2 nd = nodes[k];
    const size_t plane = (size_t)B.n2 * B.pitch, gi = (size_t)nd.y * B.pitch + nd.x;
    T* __restrict__ Un = reinterpret_cast<T*>(B.u[1 - cur]);
    const T wv = reinterpret_cast<const T*>(B.w)[gi];
    const T fac = T(dt * dt) * wv;
    T c0 = fac * d[k], c1 = fac * d[n + k];
    T d00, d01, d11;
    if (robin_damping_at<T>(B, nd.x, nd.y, d00, d01, d11)) {
        const T al = T(0.5 * dt) * wv;
        const T m00 = T(1) + al * d00, m01 = al * d01, m11 = T(1) + al * d11;
        const T idet = T(1) / (m00 * m11 - m01 * m01);
        const T x0 = (m11 * c0 - m01 * c1) * idet, x1 = (m00 * c1 - m01 * c0) * idet;
        c0 = x0;
        c1 = x1;
    }
    Un[gi] -= c0;
    Un[plane + gi] -= c1;
    if (B.du) {
        T* __restrict__ DU = reinterpret_cast<T*>(B.du);
        DU[gi] -= c0;
        DU[plane + gi] -= c1;
    }
}

// RK4 stage, before the stage kernels: -H^-1 K V_s into the point-source planes of the operator
// output (rk4_store takes them into the operator sum)
template <typename T, int O>
__global__ void k_layer_rk(BlockDev B, const int2* __restrict__ nodes, int n, int stage, double h) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n) return;
    const int2 nd = nodes[k];
    const size_t plane = (size_t)B.n2 * B.pitch, gi = (size_t)nd.y * B.pitch + nd.x;
    T k0, k1;
    layer_kv<T, O>(B, nd.x, nd.y, [&](int j1, int j2, int c) {
        T v0, v1;
        rk4_stage_velocity<T>(B, stage, T(h), (size_t)j2 * B.pitch + j1, plane, v0, v1);
        return c == 0 ? v0 : v1;
    }, k0, k1);
    T* __restrict__ R = reinterpret_cast<T*>(B.r);
    R[gi] -= k0;
    R[plane + gi] -= k1;
}

// ============================================================================ energy
// E = 1/2 sum H/w |u1 - u0|^2 / dt^2 - 1/2 sum H u1 . r   (FP64 accumulation)
template <typename T, int O>
__global__ void k_energy(BlockDev B, int cur, double inv_dt2, double* out) {
    const long long n = (long long)B.n1 * B.n2;
    double acc = 0.0;
    const size_t plane = (size_t)B.n2 * B.pitch;
    const T* U1 = reinterpret_cast<const T*>(B.u[cur]);
    const T* U0 = reinterpret_cast<const T*>(B.u[1 - cur]);
    const T* R = reinterpret_cast<const T*>(B.r);
    const T* Wp = reinterpret_cast<const T*>(B.w);
    for (long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x; t < n; t += (long long)gridDim.x * blockDim.x) {
        const int i2 = (int)(t / B.n1), i1 = (int)(t - (long long)i2 * B.n1);
        const size_t gi = (size_t)i2 * B.pitch + i1;
        const double H = B.h1 * hweight<O>(B.n1, i1) * B.h2 * hweight<O>(B.n2, i2);
        const double d0 = (double)U1[gi] - (double)U0[gi], d1 = (double)U1[gi + plane] - (double)U0[gi + plane];
        const double mass = H / (double)Wp[gi];
        acc += 0.5 * mass * (d0 * d0 + d1 * d1) * inv_dt2 -
               0.5 * H * ((double)U1[gi] * (double)R[gi] + (double)U1[gi + plane] * (double)R[gi + plane]);
    }
    for (int off = 16; off > 0; off >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, off);
    __shared__ double red[32];
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x < 32) {
        acc = threadIdx.x < (blockDim.x >> 5) ? red[threadIdx.x] : 0.0;
        for (int off = 16; off > 0; off >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, off);
        if (threadIdx.x == 0) atomicAdd(out, acc);
    }
}

// ============================================================================ setup
// numerical metric (Sec. 3.3): G[2i+I] = D_i X_I, J = det; flags J <= 0
template <int O>
__global__ void k_metric(BlockDev B, int* flag) {
    const long long n = (long long)B.n1 * B.n2;
    const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= n) return;
    const int i2 = (int)(t / B.n1), i1 = (int)(t - (long long)i2 * B.n1);
    const size_t P = B.pitch, plane = (size_t)B.n2 * P, gi = (size_t)i2 * P + i1;
    const double* X0 = B.X;
    const double* X1 = B.X + plane;
    const double g00 = dsum<O, double>(B.n1, i1, [&](int j) { return X0[(size_t)i2 * P + j]; }) / B.h1;
    const double g01 = dsum<O, double>(B.n1, i1, [&](int j) { return X1[(size_t)i2 * P + j]; }) / B.h1;
    const double g10 = dsum<O, double>(B.n2, i2, [&](int j) { return X0[(size_t)j * P + i1]; }) / B.h2;
    const double g11 = dsum<O, double>(B.n2, i2, [&](int j) { return X1[(size_t)j * P + i1]; }) / B.h2;
    B.G[gi] = g00;
    B.G[plane + gi] = g01;
    B.G[2 * plane + gi] = g10;
    B.G[3 * plane + gi] = g11;
    const double J = g00 * g11 - g01 * g10;
    B.J[gi] = J;
    if (!(J > 0.0)) atomicOr(flag, 1);
}

// transformed stiffness c_ijkl = F_Ii J C_IjKl F_Kk and w = 1/(rho J) (eq. transf_density_stiffness)
template <typename T>
__global__ void k_material(BlockDev B, const double* __restrict__ rho, const double* __restrict__ Cp) {
    const long long n = (long long)B.n1 * B.n2;
    const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= n) return;
    const int i2 = (int)(t / B.n1), i1 = (int)(t - (long long)i2 * B.n1);
    const size_t P = B.pitch, plane = (size_t)B.n2 * P, gi = (size_t)i2 * P + i1;
    const double g00 = B.G[gi], g01 = B.G[plane + gi], g10 = B.G[2 * plane + gi], g11 = B.G[3 * plane + gi];
    const double J = B.J[gi];
    double F[2][2];   // F[I][i]
    F[0][0] = g11 / J;
    F[0][1] = -g01 / J;
    F[1][0] = -g10 / J;
    F[1][1] = g00 / J;
    // pair matrix M[p][q], p = 2I + J, upper triangle in 10 planes (host layout, n = n1*n2)
    double M[4][4];
    int idx = 0;
    for (int p = 0; p < 4; ++p)
        for (int q = p; q < 4; ++q) {
            M[p][q] = M[q][p] = Cp[(size_t)idx * n + t];
            ++idx;
        }
    auto cijkl = [&](int i, int j, int k, int l) {
        double s = 0.0;
        for (int I = 0; I < 2; ++I)
            for (int K = 0; K < 2; ++K) s = s + F[I][i] * M[2 * I + j][2 * K + l] * F[K][k];
        return J * s;
    };
    T* c = reinterpret_cast<T*>(const_cast<void*>(B.c));
    const int ijkl[10][4] = {{0, 0, 0, 0}, {0, 0, 0, 1}, {0, 1, 0, 1}, {1, 0, 1, 0}, {1, 0, 1, 1},
                             {1, 1, 1, 1}, {0, 0, 1, 0}, {0, 0, 1, 1}, {0, 1, 1, 0}, {0, 1, 1, 1}};
    for (int pl = 0; pl < 10; ++pl)
        c[pl * plane + gi] = T(cijkl(ijkl[pl][0], ijkl[pl][1], ijkl[pl][2], ijkl[pl][3]));
    reinterpret_cast<T*>(const_cast<void*>(B.w))[gi] = T(1.0 / (rho[t] * J));
}

// face scale factor J^ = |a_t|, a_t = dX/dx_t on the face (eq. surfj_app_2d)
static __global__ void k_face_jhat(BlockDev B, int face, double* jhat) {
    const FaceDev& F = B.f[face];
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= F.nf) return;
    int i1, i2;
    if (F.m == 0) { i1 = F.side ? B.n1 - 1 : 0; i2 = s; }
    else { i2 = F.side ? B.n2 - 1 : 0; i1 = s; }
    const size_t plane = (size_t)B.n2 * B.pitch, gi = (size_t)i2 * B.pitch + i1;
    const int tdir = 1 - F.m;
    const double a0 = B.G[(2 * tdir) * plane + gi], a1 = B.G[(2 * tdir + 1) * plane + gi];
    jhat[s] = sqrt(a0 * a0 + a1 * a1);
}

// out[k*n + s] = T(scale[s] * in[k*n + s])   (scale may be null)
template <typename T>
__global__ void k_scale_copy(T* out, const double* __restrict__ in, const double* __restrict__ scale, int n, int planes) {
    const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= (long long)n * planes) return;
    const int s = (int)(t % n);
    out[t] = T(scale ? scale[s] * in[t] : in[t]);
}

// pitched plane <-> dense double (optionally multiplied by the block's J)
// FP32 leapfrog increment from two dense FP64 levels: dst = (float)(cur - prev), rounded once
static __global__ void k_diff_to_pitched(float* dst, const double* __restrict__ cur, const double* __restrict__ prev, int n1,
                                  int n2, int pitch, int planes) {
    const long long n = (long long)n1 * n2;
    const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= n * planes) return;
    const int p = (int)(t / n);
    const long long node = t - (long long)p * n;
    const int i2 = (int)(node / n1), i1 = (int)(node - (long long)i2 * n1);
    dst[(size_t)p * n2 * pitch + (size_t)i2 * pitch + i1] = (float)(cur[t] - prev[t]);
}

// FP32 leapfrog increment from the two levels held in the state buffers (n elements each)
static __global__ void k_diff_levels(float* __restrict__ du, const float* __restrict__ cur, const float* __restrict__ prev,
                              long long n) {
    const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (t < n) du[t] = cur[t] - prev[t];
}

template <typename T>
__global__ void k_to_pitched(T* dst, const double* __restrict__ src, int n1, int n2, int pitch, int planes,
                             const double* __restrict__ Jmul) {
    const long long n = (long long)n1 * n2;
    const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= n * planes) return;
    const int p = (int)(t / n);
    const long long node = t - (long long)p * n;
    const int i2 = (int)(node / n1), i1 = (int)(node - (long long)i2 * n1);
    const size_t gi = (size_t)i2 * pitch + i1;
    double v = src[t];
    if (Jmul) v *= Jmul[gi];
    dst[(size_t)p * n2 * pitch + gi] = T(v);
}

template <typename T>
__global__ void k_from_pitched(double* dst, const T* __restrict__ src, int n1, int n2, int pitch, int planes) {
    const long long n = (long long)n1 * n2;
    const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= n * planes) return;
    const int p = (int)(t / n);
    const long long node = t - (long long)p * n;
    const int i2 = (int)(node / n1), i1 = (int)(node - (long long)i2 * n1);
    dst[t] = (double)src[(size_t)p * n2 * pitch + (size_t)i2 * pitch + i1];
}

// CFL (Sec. 7): per node min(h1,h2) / v_max with v_max^2 = max_theta lambda_max(Gamma(theta)) / (rho J),
// Gamma_jl = xi_i c_ijkl xi_k, xi = (cos theta, sin theta); lambda_max has period pi in theta.
// The maximisation is done in two precisions: 720 FP32 samples of [0, pi) locate the three best
// local maxima (cheap: GB300's FP64 rate is a small fraction of its FP32 rate), then each is
// refined in FP64 by Newton steps on d lambda/d theta = 0 with central differences (step 1e-4:
// the derivative error O(1e-8) leaves lambda exact to rounding), and the largest refined value wins.
template <typename R>
__device__ __forceinline__ R christoffel_lmax(const R* c, R x1, R x2) {
    const R g00 = x1 * x1 * c[0] + R(2) * x1 * x2 * c[6] + x2 * x2 * c[3];
    const R g01 = x1 * x1 * c[1] + x1 * x2 * (c[7] + c[8]) + x2 * x2 * c[4];
    const R g11 = x1 * x1 * c[2] + R(2) * x1 * x2 * c[9] + x2 * x2 * c[5];
    const R hm = R(0.5) * (g00 - g11);
    return R(0.5) * (g00 + g11) + sqrt(hm * hm + g01 * g01);
}

// CFL (Sec. 7, eq. christoffel; reading: the direction maximisation is a sampled sweep refined
// by Newton steps).  Pass 1 (every node): an FP32 sweep over NS directions gives the node's
// estimate r_f = min(h1, h2) / v_max; their minimum goes to *minf_bits.  Pass 2: only nodes with
// r_f within `margin` of that minimum (the FP32 sweep is accurate to ~1e-5, so the minimising
// node is always among them) refine their three best sampled maxima with FP64 Newton steps and
// take the exact minimum into *out_bits.
constexpr int CFL_NS = 720;

struct CflSweep {
    float best[3];
    int bk[3];
};

__device__ __forceinline__ CflSweep cfl_sweep(const float* cf) {
    CflSweep w{{-1.f, -1.f, -1.f}, {0, 0, 0}};
    float s, co;
    sincospif(-1.0f / CFL_NS, &s, &co);
    float prev = christoffel_lmax<float>(cf, co, s);
    sincospif(0.0f, &s, &co);
    float cur = christoffel_lmax<float>(cf, co, s);
    const float first = cur;
    for (int k = 0; k < CFL_NS; ++k) {
        float nxt;
        if (k + 1 < CFL_NS) {
            sincospif((float)(k + 1) / CFL_NS, &s, &co);
            nxt = christoffel_lmax<float>(cf, co, s);
        } else {
            nxt = first;
        }
        if (cur >= prev && cur >= nxt) {
            if (cur > w.best[0]) { w.best[2] = w.best[1]; w.bk[2] = w.bk[1]; w.best[1] = w.best[0]; w.bk[1] = w.bk[0]; w.best[0] = cur; w.bk[0] = k; }
            else if (cur > w.best[1]) { w.best[2] = w.best[1]; w.bk[2] = w.bk[1]; w.best[1] = cur; w.bk[1] = k; }
            else if (cur > w.best[2]) { w.best[2] = cur; w.bk[2] = k; }
        }
        prev = cur;
        cur = nxt;
    }
    return w;
}

template <typename T>
__device__ __forceinline__ void cfl_node(const BlockDev& B, long long t, double c[10], float cf[10], double& rhoJ) {
    const int i2 = (int)(t / B.n1), i1 = (int)(t - (long long)i2 * B.n1);
    const size_t plane = (size_t)B.n2 * B.pitch, gi = (size_t)i2 * B.pitch + i1;
    const T* C = reinterpret_cast<const T*>(B.c);
    for (int p = 0; p < 10; ++p) {
        c[p] = (double)C[p * plane + gi];
        cf[p] = (float)c[p];
    }
    rhoJ = 1.0 / (double)reinterpret_cast<const T*>(B.w)[gi];
}

template <typename T>
__global__ void k_cfl_sweep(BlockDev B, float* __restrict__ rf, unsigned* minf_bits) {
    const long long n = (long long)B.n1 * B.n2;
    const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= n) return;
    double c[10], rhoJ;
    float cf[10];
    cfl_node<T>(B, t, c, cf, rhoJ);
    const CflSweep w = cfl_sweep(cf);
    const float v = sqrtf(fmaxf(w.best[0], 0.f) / (float)rhoJ);
    const float r = (float)fmin(B.h1, B.h2) / v;
    rf[t] = r;
    atomicMin(minf_bits, __float_as_uint(r));    // positive floats order as their bit patterns
}

template <typename T>
__global__ void k_cfl_refine(BlockDev B, const float* __restrict__ rf, const unsigned* minf_bits, float margin,
                             unsigned long long* out_bits) {
    const long long n = (long long)B.n1 * B.n2;
    const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= n) return;
    if (!(rf[t] <= __uint_as_float(*minf_bits) * (1.f + margin))) return;
    double c[10], rhoJ;
    float cf[10];
    cfl_node<T>(B, t, c, cf, rhoJ);
    const CflSweep w = cfl_sweep(cf);
    const double PI = 3.14159265358979323846, dl = 1e-4;
    auto lam = [&](double th) { double sd, cd; sincos(th, &sd, &cd); return christoffel_lmax<double>(c, cd, sd); };
    double lmax = 0.0;
    for (int q = 0; q < 3; ++q) {
        if (w.best[q] < 0.f) continue;
        double th = w.bk[q] * PI / CFL_NS;
        double f0 = lam(th);
        lmax = fmax(lmax, f0);
        for (int it = 0; it < 3; ++it) {
            const double fp = lam(th + dl), fm = lam(th - dl);
            const double d1 = (fp - fm) / (2 * dl), d2 = (fp - 2 * f0 + fm) / (dl * dl);
            lmax = fmax(lmax, fmax(fp, fm));
            if (!(d2 < 0.0)) break;
            double step = -d1 / d2;
            step = fmax(-2 * PI / CFL_NS, fmin(2 * PI / CFL_NS, step));
            th += step;
            f0 = lam(th);
            lmax = fmax(lmax, f0);
        }
    }
    const double v = sqrt(lmax / rhoJ);
    const double r = fmin(B.h1, B.h2) / v;
    atomicMin(out_bits, (unsigned long long)__double_as_longlong(r));
}

}  // namespace sbp

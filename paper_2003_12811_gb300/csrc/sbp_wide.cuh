// Wide-stencil variant of the spatial operator (the comparison of Sec. 7.1): every term of
//   r_j = sum_{i,k} D_i (c_ijkl D_k u_l)
// is a first-derivative SBP operator applied twice, the narrow D_xx^FC(b) of the main scheme
// replaced by D b D -- the same SBP form H D b D = -D^T H b D + B b D without the remainder R(b),
// so the operator is fully compatible as well -- and the SATs are exactly those of the narrow
// scheme.  Two passes over each block:
//   k_wide_flux: the fluxes G_ij = sum_{k,l} c_ijkl D_k u_l at every node (boundary rows of D at the
//                faces), 4 planes G_10, G_11, G_20, G_21;
//   k_wide_div:  r_j = D_1 G_1j + D_2 G_2j + the SAT terms of k_face_sat + J f, and the step epilogue
//                (leapfrog update, operator output or RK4 stage).
// On all but small FP32 grids (wide_by_march) the two passes take only the frame of nodes near the faces (closure rows of
// D, SATs), and k_wide_march forms both in one pass over the interior.
#pragma once
#include "sbp_interior_march.cuh"
#include "sbp_kernels.cuh"

namespace sbp {

// nodes of an n1 x n2 block less than F from a face (every node where the two sides meet, or F is 0)
__host__ __device__ inline long long frame_nodes(int n1, int n2, int F) {
    if (F == 0 || n1 <= 2 * F || n2 <= 2 * F) return (long long)n1 * n2;
    return (long long)n1 * n2 - (long long)(n1 - 2 * F) * (n2 - 2 * F);
}
__device__ __forceinline__ void frame_node(int n1, int n2, int F, long long t, int& i1, int& i2) {
    if (F == 0 || n1 <= 2 * F || n2 <= 2 * F || t < (long long)F * n1) {
        i2 = (int)(t / n1);
        i1 = (int)(t - (long long)i2 * n1);
        return;
    }
    const long long top = (long long)F * n1;
    if (t < 2 * top) {
        const int r = (int)((t - top) / n1);
        i2 = n2 - F + r;
        i1 = (int)(t - top - (long long)r * n1);
        return;
    }
    const int u = (int)(t - 2 * top), row = u / (2 * F), k = u - row * 2 * F;
    i2 = F + row;
    i1 = k < F ? k : n1 - 2 * F + k;
}

// node t of the pass (FRAME: of the frame of width `frame`); false past the last
template <bool FRAME> __device__ __forceinline__ bool wide_node(const BlockDev& B, int frame, int& i1, int& i2) {
    const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if constexpr (FRAME) {
        if (t >= frame_nodes(B.n1, B.n2, frame)) return false;
        frame_node(B.n1, B.n2, frame, t, i1, i2);
    } else {
        if (t >= (long long)B.n1 * B.n2) return false;
        i2 = (int)(t / B.n1);
        i1 = (int)(t - (long long)i2 * B.n1);
    }
    return true;
}

template <typename T, int O, bool FRAME>
__global__ void k_wide_flux(BlockDev B, StepArgs a, T* __restrict__ G, int frame) {
    int i1, i2;
    if (!wide_node<FRAME>(B, frame, i1, i2)) return;
    const int P = B.pitch;
    const size_t plane = (size_t)B.n2 * P, gi = (size_t)i2 * P + i1;
    const T* __restrict__ U0 = reinterpret_cast<const T*>(B.u[a.cur]);
    const T* __restrict__ U1 = U0 + plane;
    const T* __restrict__ C = reinterpret_cast<const T*>(B.c);
    const T ih1 = ih1T<T>(B), ih2 = ih2T<T>(B);
    const T d10 = dsum<O, T>(B.n1, i1, [&](int aa) { return U0[(size_t)i2 * P + aa]; }) * ih1;
    const T d11 = dsum<O, T>(B.n1, i1, [&](int aa) { return U1[(size_t)i2 * P + aa]; }) * ih1;
    const T d20 = dsum<O, T>(B.n2, i2, [&](int bb) { return U0[(size_t)bb * P + i1]; }) * ih2;
    const T d21 = dsum<O, T>(B.n2, i2, [&](int bb) { return U1[(size_t)bb * P + i1]; }) * ih2;
    T c[10];
#pragma unroll
    for (int p = 0; p < 10; ++p) c[p] = C[p * plane + gi];
    // planes: 0 c0000 1 c0001 2 c0101 | 3 c1010 4 c1011 5 c1111 | 6 c0010 7 c0011 8 c0110 9 c0111,
    // with c_ijkl = c_klij for the entries not stored
    G[gi] = c[0] * d10 + c[1] * d11 + c[6] * d20 + c[7] * d21;                  // G_10
    G[plane + gi] = c[1] * d10 + c[2] * d11 + c[8] * d20 + c[9] * d21;          // G_11
    G[2 * plane + gi] = c[6] * d10 + c[8] * d11 + c[3] * d20 + c[4] * d21;      // G_20
    G[3 * plane + gi] = c[7] * d10 + c[9] * d11 + c[4] * d20 + c[5] * d21;      // G_21
}

template <typename T, int O, int MODE, bool FRAME>
__global__ void k_wide_div(BlockDev B, StepArgs a, const T* __restrict__ G, int frame) {
    const int n1 = B.n1, n2 = B.n2;
    int i1, i2;
    if (!wide_node<FRAME>(B, frame, i1, i2)) return;
    const int P = B.pitch;
    const size_t plane = (size_t)n2 * P, gi = (size_t)i2 * P + i1;
    const T ih1 = ih1T<T>(B), ih2 = ih2T<T>(B);
    T r0 = dsum<O, T>(n1, i1, [&](int aa) { return G[(size_t)i2 * P + aa]; }) * ih1 +
           dsum<O, T>(n2, i2, [&](int bb) { return G[2 * plane + (size_t)bb * P + i1]; }) * ih2;
    T r1 = dsum<O, T>(n1, i1, [&](int aa) { return G[plane + (size_t)i2 * P + aa]; }) * ih1 +
           dsum<O, T>(n2, i2, [&](int bb) { return G[3 * plane + (size_t)bb * P + i1]; }) * ih2;
    // SAT terms (k_face_sat): the face term at the face node, the D_m^T spread into the first
    // NCOL nodes along the normal
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
    if (a.with_data && B.jf) {
        const T* __restrict__ JF = reinterpret_cast<const T*>(B.jf);
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            if (k >= a.K) break;
            r0 += T(a.Tk[k]) * JF[(size_t)k * plane + gi];
            r1 += T(a.Tk[k]) * JF[(size_t)(a.K + k) * plane + gi];
        }
    }
    T dd00, dd01, dd11;
    const bool damped = MODE != 1 && robin_damping_at<T>(B, i1, i2, dd00, dd01, dd11);
    if (MODE == 0) {
        const T* __restrict__ U = reinterpret_cast<const T*>(B.u[a.cur]);
        leapfrog_store<T>(B, a, gi, plane, U[gi], U[gi + plane], reinterpret_cast<const T*>(B.w)[gi], r0, r1, damped,
                          dd00, dd01, dd11);
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
}

// ------------------------------------------------------------------ FP32 interior in one pass
// The two passes move 27 words per node through memory (the fluxes go out and come back) and read their
// neighbours from L1; one pass needs 19 (u, d, c, 1/(rho J) in, u, d out) and is bound by them.  Thread x
// marches down a column as in march_tile, with the same ring of TMA-filled rows: at row s it forms
// G(s) from the ring (D_1, c) and a register queue of its column (D_2), keeps G_2 in a queue of 2q + 1
// rows, exchanges G_1 through a shared row, and delays D_1 G_1(s) by q rows in registers until D_2 G_2 of that row is
// complete: row r = s - q goes out.  All 128 threads form fluxes, the inner WCOLS of them (a multiple of 4
// columns, for the TMA boxes) output nodes: no thread follows a second column.
// Bound by HBM and the row barrier: 2 x 2001 x 1001, order 6, 80 us for the interior (the two passes over every node
// took 157), 110 us a step with the frame's chain of kernels beside it (204).
// MODE: 3 leapfrog in increment form, 1 operator output, 2 RK4 stage.
constexpr int WCOLS = 120;
__host__ __device__ inline int wide_ncx(int n1, int strip) { return (n1 - strip - march_x0(strip) + WCOLS - 1) / WCOLS; }

template <int O, int MODE>
__device__ __forceinline__ bool wide_march_tile(const MarchMaps& maps, const BlockDev& B, const StepArgs& a, int rows_per_cta,
                                                int tile, int* err, unsigned char* smem) {
    using MC = MarchCfg<O>;
    constexpr int Q = MC::Q, W = MBOXW, L = 2 * Q + 1;
    // a node at least `strip` from every face sees interior rows of D in both applications
    static_assert((Ord<O>::NCLOS > Ord<O>::NCOL ? Ord<O>::NCLOS : Ord<O>::NCOL) >= Ord<O>::NB + Q, "strip covers the closures");
    constexpr int OFF = MXOFF / 2;                // thread 0 sits OFF columns before the tile's first
    static_assert(OFF >= Q && OFF + WCOLS + Q <= MTHREADS && OFF + MTHREADS + Q <= W, "every flux lies in the box");
    float* ring = reinterpret_cast<float*>(smem);
    float2* g1s = reinterpret_cast<float2*>(ring + MNCH * MC::CHUNK);     // [row parity][column]
    uint64_t* bars = reinterpret_cast<uint64_t*>(ring + MNCH * MC::CHUNK + MC::G1 + MC::HQ);
    const int S = B.strip, n1 = B.n1, n2 = B.n2, P = B.pitch;
    const int lim1 = n1 - S, lim2 = n2 - S, ncx = wide_ncx(n1, S);
    const int cx = tile % ncx, cy = tile / ncx;
    const int x0 = march_x0(S) + cx * WCOLS, ys = S + cy * rows_per_cta;
    if (ys >= lim2) return true;
    const int ye = min(lim2, ys + rows_per_cta), rb = ys - 2 * Q;
    const int tx = threadIdx.x, gx = x0 - OFF + tx, cc = tx + OFF;
    const bool out = tx >= OFF && tx < OFF + WCOLS && gx >= S && gx < lim1;
    const size_t plane = (size_t)n2 * P;
    constexpr uint32_t BYTES_U = 2 * MR * W * 4, BYTES_C = 10 * MR * W * 4;
    const int nchunks = (ye + 2 * Q - rb + MR - 1) / MR;
    if (tx == 0) {
        for (int k = 0; k < MNCH; ++k) mbar_init(&bars[k], 1);
        fence_barrier_init();
        fence_proxy_async();
    }
    __syncthreads();
    auto issue = [&](int ch) {
        float* dst = ring + (ch % MNCH) * MC::CHUNK;
        uint64_t* bar = &bars[ch % MNCH];
        mbar_expect_tx(bar, BYTES_U + BYTES_C);
        tma_load_3d(dst, &maps.u[a.cur], x0 - MXOFF, rb + ch * MR, 0, bar);
        tma_load_3d(dst + MC::UPAD, &maps.c, x0 - MXOFF, rb + ch * MR, 0, bar);
    };
    if (tx == 0)
        for (int ch = 0; ch < MNCH && ch < nchunks; ++ch) issue(ch);
    auto rowp = [&](int r) -> const float* {
        const unsigned rr = (unsigned)(r - rb);
        return ring + ((rr / MR) % MNCH) * MC::CHUNK + (rr % MR) * W;
    };
    auto poff = [](int p) { return p < 2 ? p * MR * W : MC::UPAD + (p - 2) * MR * W; };
    float ak1[Q], ak2[Q];                          // a_k / h_1, a_k / h_2
#pragma unroll
    for (int k = 0; k < Q; ++k) {
        ak1[k] = Ord<O>::template aT<float>(k) * B.ih1f;
        ak2[k] = Ord<O>::template aT<float>(k) * B.ih2f;
    }
    float2 qu[L], qg[L], dl[Q];                    // rows s-q .. s+q of u, s-2q .. s of G_2, s-1 .. s-q of D_1 G_1
#pragma unroll
    for (int k = 0; k < L; ++k) qu[k] = qg[k] = make_float2(0.f, 0.f);
#pragma unroll
    for (int k = 0; k < Q; ++k) dl[k] = make_float2(0.f, 0.f);
    bool ok = true;
    int waited = 0, next_issue = MNCH < nchunks ? MNCH : nchunks;
    auto push = [&](int r) {                       // row r of the column into the queue
        if (((unsigned)(r - rb) % MR) == 0) {
            const unsigned ch = (unsigned)(r - rb) / MR;
            ok = mbar_wait_bounded(&bars[ch % MNCH], (ch / MNCH) & 1) && ok;
            ++waited;
        }
#pragma unroll
        for (int k = 0; k < L - 1; ++k) qu[k] = qu[k + 1];
        const float* p = rowp(r) + cc;
        qu[L - 1] = make_float2(p[poff(0)], p[poff(1)]);
    };
    float w_c = 0.f, w_n = 0.f;                    // 1/(rho J) and d^n of the row going out, of the next
    float2 d_c = make_float2(0.f, 0.f), d_n = make_float2(0.f, 0.f);
    auto load_row = [&](int r, float& wv, float2& v) {
        if (MODE != 1 && out && r < ye) {
            const size_t gi = (size_t)r * P + gx;
            wv = __ldg(reinterpret_cast<const float*>(B.w) + gi);
            if (MODE == 3) {
                const float* D = reinterpret_cast<const float*>(B.du);
                v = make_float2(D[gi], D[gi + plane]);
            }
        }
    };
    load_row(ys, w_c, d_c);
    load_row(ys + 1, w_n, d_n);
    for (int r = rb; r < ys; ++r) push(r);
#pragma unroll 4
    for (int s = ys - Q; s < ye + Q; ++s) {
        push(s + Q);
        const int par = s & 1;
        {
            const float* p = rowp(s) + cc;
            float2 d1 = make_float2(0.f, 0.f), d2 = make_float2(0.f, 0.f);
#pragma unroll
            for (int k = 1; k <= Q; ++k) {
                d1 = ffma2(bc2(ak1[k - 1]), fsub2(make_float2(p[poff(0) + k], p[poff(1) + k]), make_float2(p[poff(0) - k], p[poff(1) - k])), d1);
                d2 = ffma2(bc2(ak2[k - 1]), fsub2(qu[Q + k], qu[Q - k]), d2);
            }
            float c[10];
#pragma unroll
            for (int k = 0; k < 10; ++k) c[k] = p[poff(2 + k)];
            // G_1 = (c0 d1x + c1 d1y + c6 d2x + c7 d2y, c1 d1x + c2 d1y + c8 d2x + c9 d2y), G_2 likewise with the
            // transposed mixed entries
            float2 g1 = fmul2(make_float2(c[0], c[1]), bc2(d1.x));
            g1 = ffma2(make_float2(c[1], c[2]), bc2(d1.y), g1);
            g1 = ffma2(make_float2(c[6], c[8]), bc2(d2.x), g1);
            g1 = ffma2(make_float2(c[7], c[9]), bc2(d2.y), g1);
            float2 g2 = fmul2(make_float2(c[6], c[7]), bc2(d1.x));
            g2 = ffma2(make_float2(c[8], c[9]), bc2(d1.y), g2);
            g2 = ffma2(make_float2(c[3], c[4]), bc2(d2.x), g2);
            g2 = ffma2(make_float2(c[4], c[5]), bc2(d2.y), g2);
            g1s[par * W + cc] = g1;
#pragma unroll
            for (int k = 0; k < L - 1; ++k) qg[k] = qg[k + 1];
            qg[L - 1] = g2;
        }
        if (__syncthreads_or(!ok)) {
            // a bounded wait ran out: record it, drain this CTA's issued copies (bounded), stop
            if (tx == 0) {
                atomicOr(err, ERR_MARCH_WAIT);
                for (int ch = waited; ch < next_issue; ++ch) mbar_wait_bounded(&bars[ch % MNCH], (ch / MNCH) & 1);
            }
            __syncthreads();
            return false;
        }
        if (tx == 0) {                             // every thread is past row s-1: refill the slots below row s
            const int below = (int)((unsigned)(s - rb) / MR);
            bool fenced = false;
            while (next_issue < nchunks && next_issue < below + MNCH) {
                if (!fenced) {
                    fence_proxy_async();
                    fenced = true;
                }
                issue(next_issue++);
            }
        }
        if (!out) continue;
        float2 m1 = make_float2(0.f, 0.f);
        const float2* g1r = g1s + par * W + cc;
#pragma unroll
        for (int k = 1; k <= Q; ++k) m1 = ffma2(bc2(ak1[k - 1]), fsub2(g1r[k], g1r[-k]), m1);
        float2 rr = dl[Q - 1];                     // D_1 G_1 of row s - q
#pragma unroll
        for (int k = Q - 1; k > 0; --k) dl[k] = dl[k - 1];
        dl[0] = m1;
        const int r = s - Q;
        if (r < ys) continue;
#pragma unroll
        for (int k = 1; k <= Q; ++k) rr = ffma2(bc2(ak2[k - 1]), fsub2(qg[Q + k], qg[Q - k]), rr);
        const size_t gi = (size_t)r * P + gx;
        if (a.with_data && B.jf) {
            const float* __restrict__ JF = reinterpret_cast<const float*>(B.jf);
#pragma unroll
            for (int kb = 0; kb < 8; ++kb) {
                if (kb >= a.K) break;
                rr = ffma2(bc2((float)a.Tk[kb]), make_float2(JF[(size_t)kb * plane + gi], JF[(size_t)(a.K + kb) * plane + gi]), rr);
            }
        }
        if constexpr (MODE == 3) {
            float* __restrict__ Un = reinterpret_cast<float*>(B.u[1 - a.cur]);
            float* __restrict__ DU = reinterpret_cast<float*>(B.du);
            const float2 d = ffma2(bc2(a.dt2f * w_c), rr, d_c), nu = fadd2(qu[0], d);
            Un[gi] = nu.x;
            Un[gi + plane] = nu.y;
            DU[gi] = d.x;
            DU[gi + plane] = d.y;
        } else if constexpr (MODE == 2) {
            rk4_store<float>(B, a, gi, plane, w_c, rr.x, rr.y);
        } else {
            float* __restrict__ R = reinterpret_cast<float*>(B.r);
            R[gi] = rr.x;
            R[gi + plane] = rr.y;
        }
        w_c = w_n;
        d_c = d_n;
        load_row(r + 2, w_n, d_n);
    }
    __syncthreads();
    if (tx == 0)
        for (int k = 0; k < MNCH; ++k) mbar_inval(&bars[k]);
    return true;
}

// (five CTAs' worth of registers for the four that shared memory holds: the frame's small kernels, which need none
// of it, fit beside them)
template <int O, int MODE>
__global__ void __launch_bounds__(MTHREADS, 5)
k_wide_march(const __grid_constant__ MarchMulti mm, StepArgs a, int* err) {
    extern __shared__ __align__(128) unsigned char march_smem[];
    const int k = blockIdx.x;
    int b = 0;
    while (b + 1 < mm.nb && k >= mm.start[b + 1]) ++b;
    (void)wide_march_tile<O, MODE>(mm.maps[b], mm.b[b], a, mm.rows[b], k - mm.start[b], err, march_smem);
}

}  // namespace sbp

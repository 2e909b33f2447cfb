// The kernels of one precision and order with the functions that launch them; instantiated by sbp_ops.cu.
#pragma once
#include "sbp_host.cuh"

namespace sbphost {

// interface traces of the level being read (k_face_trace), TRACE_MAX faces per launch, on stream tst
template <typename T, int O>
void launch_traces(sbp_handle* h, const StepArgs& a, cudaStream_t tst, bool adj) {
    TraceArgs ta{};
    auto flush = [&]() {
        if (ta.nfaces == 0) return;
        ProfScope ps(h, 2, tst, 1);
        k_face_trace<T, O><<<grid_for(ta.total, 128), 128, 0, tst>>>(ta);
        ta = TraceArgs{};
    };
    for (size_t b = 0; b < h->blocks.size(); ++b) {
        const HostBlock& hb = h->blocks[b];
        for (int f = 0; f < 4; ++f) {
            const HostFace& HF = hb.f[f];
            if (HF.kind != FACE_INTF) continue;
            TraceFace& F = ta.f[ta.nfaces++];
            F.u = adj ? hb.psi[a.cur] : hb.u[a.cur];
            F.c = hb.c;
            F.tr = HF.tr;
            F.plane = (long long)hb.n2 * hb.pitch;
            F.nf = HF.nf;
            F.start = ta.total;
            F.m = f / 2;
            F.side = f % 2;
            F.pitch = hb.pitch;
            F.nm = F.m == 0 ? hb.n1 : hb.n2;
            F.nu = (f % 2 == 0) ? -1.0 : 1.0;
            const double hm = F.m == 0 ? hb.h1 : hb.h2, ht = F.m == 0 ? hb.h2 : hb.h1;
            F.ihm = 1.0 / hm;
            F.iht = 1.0 / ht;
            F.k = h->beta * 2.0 / 4.0 * (1.0 / (hm * host_hweight(h->order, F.nm, 0)));
            ta.total += HF.nf;
            if (ta.nfaces == TRACE_MAX) flush();
        }
    }
    flush();
}

// the wide-stencil operator (sbp_wide.cuh): traces, the SAT terms of every face node, the flux and
// divergence passes of every block (by wide_by_march only of its frame near the faces, beside one marching kernel over
// the interior, which they share nothing with), then the point sources (every source node: the wide path has
// no strip kernel)
template <typename T, int O>
int launch_wide(sbp_handle* h, const StepArgs& a, int mode, cudaStream_t st) {
    constexpr bool f32 = std::is_same<T, float>::value;
    const bool march = f32 && wide_by_march(h);
    const int S = std::max(order_nclos(h->order), order_ncol(h->order));
    // the frame's chain of small kernels on the high-priority stream, queued before the interior
    const bool par = march && h->hi && !h->prof;
    cudaStream_t fst = par ? h->hi : st;
    if (par) {
        cudaEventRecord(h->ev_fork, st);
        cudaStreamWaitEvent(h->hi, h->ev_fork, 0);
    }
    if (h->ntrefs > 0) launch_traces<T, O>(h, a, fst, false);
    if (h->nface_nodes > 0) {
        ProfScope ps(h, 1, fst, 1);
        k_face_sat<T, O><<<grid_for(h->nface_nodes, 64), 64, 0, fst>>>(h->d_blocks, h->d_refs, h->nrefs, h->nface_nodes, a, h->beta);
    }
    if constexpr (f32) {
        MarchMulti mm{};
        int tiles = 0;
        auto flush = [&]() {
            if (mm.nb == 0) return;
            mm.start[mm.nb] = tiles;
            ProfScope ps(h, 0, st, 1);
            constexpr size_t msm = MarchCfg<O>::BYTES;
            if (mode == 0) k_wide_march<O, 3><<<tiles, MTHREADS, msm, st>>>(mm, a, h->d_err);
            else if (mode == 2) k_wide_march<O, 2><<<tiles, MTHREADS, msm, st>>>(mm, a, h->d_err);
            else k_wide_march<O, 1><<<tiles, MTHREADS, msm, st>>>(mm, a, h->d_err);
            mm = MarchMulti{};
            tiles = 0;
        };
        for (auto& hb : h->blocks) {
            if (!march) break;
            const int ncx = wide_ncx(hb.n1, S), n2i = hb.n2 - 2 * S, rows = march_rows(h, ncx, n2i), k = mm.nb++;
            mm.maps[k] = hb.mmaps;
            mm.b[k] = make_view(h, hb);
            mm.start[k] = tiles;
            mm.rows[k] = rows;
            tiles += ncx * ((n2i + rows - 1) / rows);
            if (mm.nb == MARCH_MAX_BLOCKS) flush();
        }
        flush();
    }
    auto passes = [&](auto fc) {
        constexpr bool F = decltype(fc)::value;
        for (auto& hb : h->blocks) {
            const BlockDev b = make_view(h, hb);
            const int ff = F ? S + Ord<O>::Q : 0, fd = F ? S : 0;
            const long long nf = frame_nodes(hb.n1, hb.n2, ff), nd = frame_nodes(hb.n1, hb.n2, fd);
            ProfScope ps(h, F ? 1 : 0, fst, 2);
            k_wide_flux<T, O, F><<<grid_for(nf), 256, 0, fst>>>(b, a, (T*)hb.gw, ff);
            if (mode == 0) k_wide_div<T, O, 0, F><<<grid_for(nd), 256, 0, fst>>>(b, a, (const T*)hb.gw, fd);
            else if (mode == 2) k_wide_div<T, O, 2, F><<<grid_for(nd), 256, 0, fst>>>(b, a, (const T*)hb.gw, fd);
            else k_wide_div<T, O, 1, F><<<grid_for(nd), 256, 0, fst>>>(b, a, (const T*)hb.gw, fd);
        }
    };
    if constexpr (f32) {
        if (march) passes(std::true_type());
        else passes(std::false_type());
    } else {
        passes(std::false_type());
    }
    if (par) {
        cudaEventRecord(h->ev_join_hi, h->hi);
        cudaStreamWaitEvent(st, h->ev_join_hi, 0);
    }
    if (!h->src_nodes.empty()) {
        ProfScope ps(h, 3, st, 1);
        const int ns = (int)h->src_nodes.size();
        if (mode == 2) k_sources<T, 2><<<grid_for(ns), 256, 0, st>>>(h->d_blocks, h->d_src_nodes, ns, h->d_src_params, a);
        else if (mode == 0) k_sources<T, 0><<<grid_for(ns), 256, 0, st>>>(h->d_blocks, h->d_src_nodes, ns, h->d_src_params, a);
        else k_sources<T, 1><<<grid_for(ns), 256, 0, st>>>(h->d_blocks, h->d_src_nodes, ns, h->d_src_params, a);
    }
    return check_cuda(h, "wide operator launch");
}

template <int O>
void launch_interior_f64(sbp_handle* h, const BlockDev* tab, const StepArgs& a, int mode, cudaStream_t st) {
    const int best = pick_edge_shape(h);
    for (int first = 0; first < h->nblocks; first += IE_MAX_BLOCKS) {
        InteriorTiles tl;
        const int tiles = edge_tiles(h, first, best, tl);
        ProfScope ps(h, 0, st, 1);
        auto run = [&](auto kc) {
            constexpr int TX = kEdgeShapes[decltype(kc)::value][0], TY = kEdgeShapes[decltype(kc)::value][1], NT = TX * TY < 256 ? TX * TY : 256;
            if (mode == 0) k_interior_edges<double, O, 0, TX, TY><<<tiles, NT, 0, st>>>(tab, tl, a);
            else if (mode == 2) k_interior_edges<double, O, 2, TX, TY><<<tiles, NT, 0, st>>>(tab, tl, a);
            else k_interior_edges<double, O, 1, TX, TY><<<tiles, NT, 0, st>>>(tab, tl, a);
        };
        if (best == 0) run(std::integral_constant<int, 0>());
        else if (best == 1) run(std::integral_constant<int, 1>());
        else if (best == 2) run(std::integral_constant<int, 2>());
        else run(std::integral_constant<int, 3>());
    }
}

template <typename T, int O>
int launch_step(sbp_handle* h, const StepArgs& a, int mode, cudaStream_t st, bool adj) {
    if (h->ntrefs > 0) launch_traces<T, O>(h, a, st, adj);
    StepStrips ss{};
    const bool sh = h->shorts.d_tiles != nullptr;
    ss.blocks = adj ? h->d_blocks_adj : h->d_blocks;
    ss.tiles = sh ? h->shorts.d_tiles : h->d_tiles;
    ss.n = sh ? (int)h->shorts.tiles.size() : h->ntiles;
    ss.ssrc = adj ? nullptr : (sh ? h->shorts.d_src : h->d_src_strip);
    ss.spar = h->d_src_params;
    ss.beta = h->beta;
    const bool inside = !adj && h->n_src_int > 0 && h->n_src_int <= STEP_MAX_SOURCES;
    ss.isrc = inside ? h->d_src_int : nullptr;
    ss.nisrc = inside ? h->n_src_int : 0;
    {
        ProfScope ps(h, 0, st, 1);
        if constexpr (std::is_same<T, float>::value) {
            MarchMulti mm{};
            int tiles = 0;
            const int S = std::max(order_nclos(h->order), order_ncol(h->order));
            std::vector<int2> grids;
            for (auto& hb : h->blocks) grids.push_back(make_int2(march_ncx(hb.n1, S), hb.n2 - 2 * S));
            const int even = h->rows_per_cta > 0 ? h->rows_per_cta : item_rows(4 * h->num_sms, grids, ss.n, false);
            for (auto& hb : h->blocks) {
                const int ncx = march_ncx(hb.n1, S), n2i = hb.n2 - 2 * S, most = std::min(n2i, even), bands = (n2i + most - 1) / most;
                const int rows = h->rows_per_cta > 0 ? most : (n2i + bands - 1) / bands;
                const int k = mm.nb++;
                mm.maps[k] = adj ? hb.pmaps : hb.mmaps;
                mm.b[k] = adj ? make_view_adj(h, hb) : make_view(h, hb);
                mm.start[k] = tiles;
                mm.rows[k] = rows;
                tiles += ncx * ((n2i + rows - 1) / rows);
            }
            mm.start[mm.nb] = tiles;
            constexpr size_t sm = step_smem_f32<O>();
            const int grid = ss.n + tiles;
            if (adj && sh) k_step_f32<O, 0, SHORT_TILE><<<grid, MTHREADS, sm, st>>>(mm, ss, a, h->d_err);
            else if (adj) k_step_f32<O, 0, 32><<<grid, MTHREADS, sm, st>>>(mm, ss, a, h->d_err);
            else if (sh) k_step_f32<O, 3, SHORT_TILE><<<grid, MTHREADS, sm, st>>>(mm, ss, a, h->d_err);
            else k_step_f32<O, 3, 32><<<grid, MTHREADS, sm, st>>>(mm, ss, a, h->d_err);
        } else {
            const int best = step_edge_shape(h);
            InteriorTiles tl;
            const int grid = ss.n + edge_tiles(h, 0, best, tl);
            auto run = [&](auto kc) {
                constexpr int TX = kEdgeShapes[decltype(kc)::value][0], TY = kEdgeShapes[decltype(kc)::value][1];
                constexpr size_t sm = step_smem_f64<O, TX, TY>();
                constexpr int NT = step_threads_f64<TX, TY>();
                if (mode == 0) k_step_f64<O, 0, TX, TY><<<grid, NT, sm, st>>>(tl, ss, a, h->d_err);
                else k_step_f64<O, 2, TX, TY><<<grid, NT, sm, st>>>(tl, ss, a, h->d_err);
            };
            if (best == 0) run(std::integral_constant<int, 0>());
            else if (best == 1) run(std::integral_constant<int, 1>());
            else if (best == 2) run(std::integral_constant<int, 2>());
            else run(std::integral_constant<int, 3>());
        }
    }
    if (!adj && h->n_src_int > 0 && !inside) {
        ProfScope ps(h, 3, st, 1);
        const int ns = h->n_src_int;
        if (mode == 2) k_sources<T, 2><<<grid_for(ns), 256, 0, st>>>(h->d_blocks, h->d_src_int, ns, h->d_src_params, a);
        else k_sources<T, 0><<<grid_for(ns), 256, 0, st>>>(h->d_blocks, h->d_src_int, ns, h->d_src_params, a);
    }
    return check_cuda(h, "step launch");
}

// one operator application (mode 1) or leapfrog step (mode 0) on the state fields, or, with adj,
// on the adjoint fields (the same kernels; the sources are skipped)
template <typename T, int O>
int launch_operator(sbp_handle* h, const StepArgs& a, int mode, cudaStream_t st, bool adj) {
    if (one_launch(h, mode)) return launch_step<T, O>(h, a, mode, st, adj);
    const BlockDev* tab = adj ? h->d_blocks_adj : h->d_blocks;
    constexpr size_t smem = interior_smem_elems<T, O>() * sizeof(T);
    // interior kernels on st; strip kernels on the auxiliary stream when overlapping (profiling
    // runs serialise so that every family's events time that family alone)
    const bool ovl = h->overlap && h->aux && !h->prof;
    // the interface traces run on the auxiliary stream beside the interior kernel (in its tail
    // or its free slots); the strips that read them follow on that stream or wait for it
    const bool tr_async = h->aux && !h->prof && h->ntrefs > 0;
    cudaStream_t sst = ovl ? h->aux : st;
    cudaStream_t ist = ovl ? h->hi : st;
    cudaStream_t tst = (ovl || tr_async) ? h->aux : st;
    if (ovl || tr_async) {
        cudaEventRecord(h->ev_fork, st);
        cudaStreamWaitEvent(h->aux, h->ev_fork, 0);
        if (ovl) cudaStreamWaitEvent(h->hi, h->ev_fork, 0);
    }
    if constexpr (std::is_same<T, float>::value) {
        // column-marching kernel: the interior tiles of up to MARCH_MAX_BLOCKS blocks per launch,
        // rows per tile chosen for one wave of ~4 CTAs per SM per block
        MarchMulti mmul{};
        int tiles = 0;
        auto flush = [&]() {
            if (mmul.nb == 0) return;
            mmul.start[mmul.nb] = tiles;
            ProfScope ps(h, 0, ist, 1);
            constexpr size_t msm = MarchCfg<O>::BYTES;
            if (mode == 0 && !adj) k_interior_march_multi<O, 3><<<tiles, MTHREADS, msm, ist>>>(mmul, a, h->d_err);
            else if (mode == 0) k_interior_march_multi<O, 0><<<tiles, MTHREADS, msm, ist>>>(mmul, a, h->d_err);
            else if (mode == 2 && a.stage == 1) k_interior_march_multi<O, 4><<<tiles, MTHREADS, msm, ist>>>(mmul, a, h->d_err);
            else if (mode == 2 && a.stage == 2) k_interior_march_multi<O, 5><<<tiles, MTHREADS, msm, ist>>>(mmul, a, h->d_err);
            else if (mode == 2 && a.stage == 3) k_interior_march_multi<O, 6><<<tiles, MTHREADS, msm, ist>>>(mmul, a, h->d_err);
            else if (mode == 2) k_interior_march_multi<O, 7><<<tiles, MTHREADS, msm, ist>>>(mmul, a, h->d_err);
            else k_interior_march_multi<O, 1><<<tiles, MTHREADS, msm, ist>>>(mmul, a, h->d_err);
            mmul = MarchMulti{};
            tiles = 0;
        };
        for (auto& hb : h->blocks) {
            const int S2 = std::max(order_nclos(h->order), order_ncol(h->order));
            const int ncx = march_ncx(hb.n1, S2);
            const int n2i = hb.n2 - 2 * S2;
            const int rows = march_rows(h, ncx, n2i), ncy = (n2i + rows - 1) / rows;
            const int k = mmul.nb++;
            mmul.maps[k] = adj ? hb.pmaps : hb.mmaps;
            mmul.b[k] = adj ? make_view_adj(h, hb) : make_view(h, hb);
            mmul.start[k] = tiles;
            mmul.rows[k] = rows;
            tiles += ncx * ncy;
            if (mmul.nb == MARCH_MAX_BLOCKS) flush();
        }
        flush();
    } else if (h->blocks[0].e) {
        launch_interior_f64<O>(h, tab, a, mode, ist);
    } else for (auto& hb : h->blocks) {   // no room for the edge weights: the kernel that forms them
        BlockDev b = adj ? make_view_adj(h, hb) : make_view(h, hb);
        const int S = b.strip;
        const int ni1 = hb.n1 - 2 * S, ni2 = hb.n2 - 2 * S;
        dim3 grid((ni1 + ITX - 1) / ITX, (ni2 + ITY - 1) / ITY);
        {
            ProfScope ps(h, 0, ist, 1);
            {
                if (mode == 0) k_interior<T, O, 0><<<grid, dim3(32, 8), smem, ist>>>(b, a);
                else if (mode == 2) k_interior<T, O, 2><<<grid, dim3(32, 8), smem, ist>>>(b, a);
                else k_interior<T, O, 1><<<grid, dim3(32, 8), smem, ist>>>(b, a);
            }
        }
    }
    if (h->ntrefs > 0) launch_traces<T, O>(h, a, tst, adj);
    if (tr_async && !ovl) {    // the strips wait for the traces formed beside the interior
        cudaEventRecord(h->ev_join, h->aux);
        cudaStreamWaitEvent(st, h->ev_join, 0);
    }
    {
        ProfScope ps(h, 1, sst, 1);
        const SrcNode* ss = adj ? nullptr : h->d_src_strip;
        auto run = [&](auto lc) {
            constexpr int TL = decltype(lc)::value;
            using ST = StripTile<O, TL>;
            constexpr size_t ssm = ST::template bytes<T>();
            if (mode == 0)
                k_strip_tile<T, O, 0, TL><<<h->ntiles, ST::THREADS, ssm, sst>>>(tab, h->d_tiles, a, h->beta, h->d_err, ss, h->d_src_params);
            else if (mode == 2)
                k_strip_tile<T, O, 2, TL><<<h->ntiles, ST::THREADS, ssm, sst>>>(tab, h->d_tiles, a, h->beta, h->d_err, ss, h->d_src_params);
            else
                k_strip_tile<T, O, 1, TL><<<h->ntiles, ST::THREADS, ssm, sst>>>(tab, h->d_tiles, a, h->beta, h->d_err, ss, h->d_src_params);
        };
        if constexpr (std::is_same<T, double>::value) {
            if (h->strip_len == 8) run(std::integral_constant<int, 8>());
            else if (h->strip_len == 16) run(std::integral_constant<int, 16>());
            else run(std::integral_constant<int, 32>());
        } else {
            run(std::integral_constant<int, 32>());
        }
    }
    if (ovl) {
        cudaEventRecord(h->ev_join, h->aux);
        cudaEventRecord(h->ev_join_hi, h->hi);
        cudaStreamWaitEvent(st, h->ev_join, 0);
        cudaStreamWaitEvent(st, h->ev_join_hi, 0);
    }
    if (!adj && h->n_src_int > 0) {   // source nodes off the strips (the strip kernel adds the others)
        ProfScope ps(h, 3, st, 1);
        const int ns = h->n_src_int;
        if (mode == 2) k_sources<T, 2><<<grid_for(ns), 256, 0, st>>>(h->d_blocks, h->d_src_int, ns, h->d_src_params, a);
        else if (mode == 0) k_sources<T, 0><<<grid_for(ns), 256, 0, st>>>(h->d_blocks, h->d_src_int, ns, h->d_src_params, a);
        else k_sources<T, 1><<<grid_for(ns), 256, 0, st>>>(h->d_blocks, h->d_src_int, ns, h->d_src_params, a);
    }
    return check_cuda(h, "operator launch");
}

// layer dissipation around the step kernels (leapfrog: the backward-velocity term is formed before
// the step overwrites u^{n-1} and added after it; RK4: added into the stage's operator sum before)
template <typename T, int O>
void layer_launch(sbp_handle* h, const StepArgs& a, int mode, cudaStream_t st, bool post) {
    if (mode == 0 && !(a.dt > 0)) return;   // tuning steps advance nothing (dt = 0)
    for (auto& hb : h->blocks) {
        if (hb.nln == 0) continue;
        const BlockDev b = make_view(h, hb);
        const unsigned g = grid_for(hb.nln);
        if (mode == 2) {
            if (!post) k_layer_rk<T, O><<<g, 256, 0, st>>>(b, hb.d_lnodes, hb.nln, a.stage, a.rkh);
        } else if (!post) {
            k_layer_pre<T, O><<<g, 256, 0, st>>>(b, hb.d_lnodes, hb.nln, a.cur, 1.0 / a.dt, (T*)hb.lscr);
        } else {
            k_layer_post<T><<<g, 256, 0, st>>>(b, hb.d_lnodes, hb.nln, a.cur, a.dt, (const T*)hb.lscr);
        }
    }
}

template <typename T, int O>
void launch_noalloc(sbp_handle* h, const BlockDev* views, int nviews, BlockDev* d_views, FaceRef* d_refs,
                    const StepArgs& a, cudaStream_t st) {
    const int total = h->nface_nodes;
    if (total > 0) k_face_sat<T, O><<<grid_for(total), 256, 0, st>>>(d_views, d_refs, h->nrefs, total, a, h->beta);
    constexpr size_t smem = interior_smem_elems<T, O>() * sizeof(T);
    bool edges = false;
    if constexpr (std::is_same<T, double>::value) {
        edges = views[0].e != nullptr;
        if (edges) launch_interior_f64<O>(h, d_views, a, 1, st);
    }
    for (int b = 0; b < nviews; ++b) {
        const BlockDev& v = views[b];
        const int S = v.strip;
        const int ni1 = v.n1 - 2 * S, ni2 = v.n2 - 2 * S;
        dim3 grid((ni1 + ITX - 1) / ITX, (ni2 + ITY - 1) / ITY);
        if (!edges) k_interior<T, O, 1><<<grid, dim3(32, 8), smem, st>>>(v, a);
        const long long nstrip = (long long)v.n1 * v.n2 - (long long)ni1 * ni2;
        k_boundary<T, O, 1><<<grid_for(nstrip), 256, 0, st>>>(v, a);
    }
    if (!h->src_nodes.empty()) {
        const int ns = (int)h->src_nodes.size();
        k_sources<T, 1><<<grid_for(ns), 256, 0, st>>>(d_views, h->d_src_nodes, ns, h->d_src_params, a);
    }
}

// gradient contributions of the nl levels of one segment
template <typename T, int O>
void launch_grad(sbp_handle* h, const GradDev* d_grad, const std::vector<GradDev>& grads, int nl, double dt2,
                 cudaStream_t st) {
    const int total = h->nface_nodes, nfc = std::min(GRAD_MAX_CHUNKS, nl);
    if (total > 0) {
        ProfScope ps(h, 6, st, 1);
        k_grad_face<T, O><<<dim3(grid_for(total, 64), nfc), 64, 0, st>>>(h->d_blocks_adj, d_grad, h->d_refs, h->nrefs, total, nl, nfc, h->beta);
    }
    constexpr int GS = GradCfg<O>::GS;
    for (size_t b = 0; b < h->blocks.size(); ++b) {
        const HostBlock& hb = h->blocks[b];
        const BlockDev v = make_view_adj(h, hb);
        {
            ProfScope ps(h, 4, st, 1);
            dim3 gi((hb.n1 - 2 * GS + 31) / 32, (hb.n2 - 2 * GS + 7) / 8);
            k_grad_interior<T, O><<<gi, dim3(32, 8), 0, st>>>(v, grads[b], nl, dt2);
        }
        {
            ProfScope ps(h, 5, st, 3);
            const long long nstrip = grad_strip_nodes(hb, GS);
            const int nchunk = grad_strip_chunks(h, nstrip, nl);
            k_grad_lines<T, O><<<dim3(grid_for(2LL * (hb.n1 + hb.n2), 64), nchunk), 64, 0, st>>>(v, grads[b], nl, nchunk, nstrip);
            k_grad_strip<T, O><<<dim3(grid_for(nstrip), nchunk), 256, 0, st>>>(v, grads[b], nl, nchunk, nstrip);
            k_grad_strip_sum<T, O><<<grid_for(nstrip), 256, 0, st>>>(v, grads[b], nchunk, nfc, nstrip, dt2);
        }
    }
}

template <typename T, int O> void set_smem_attr() {
    constexpr size_t smem = interior_smem_elems<T, O>() * sizeof(T);
    auto strip = [](auto lc) {
        constexpr int TL = decltype(lc)::value;
        constexpr int ssm = (int)StripTile<O, TL>::template bytes<T>();
        cudaFuncSetAttribute(k_strip_tile<T, O, 0, TL>, cudaFuncAttributeMaxDynamicSharedMemorySize, ssm);
        cudaFuncSetAttribute(k_strip_tile<T, O, 1, TL>, cudaFuncAttributeMaxDynamicSharedMemorySize, ssm);
        cudaFuncSetAttribute(k_strip_tile<T, O, 2, TL>, cudaFuncAttributeMaxDynamicSharedMemorySize, ssm);
    };
    strip(std::integral_constant<int, 32>());
    if constexpr (std::is_same<T, float>::value) {
        constexpr int sm = (int)step_smem_f32<O>();
        cudaFuncSetAttribute(k_step_f32<O, 0, SHORT_TILE>, cudaFuncAttributeMaxDynamicSharedMemorySize, sm);
        cudaFuncSetAttribute(k_step_f32<O, 3, SHORT_TILE>, cudaFuncAttributeMaxDynamicSharedMemorySize, sm);
        cudaFuncSetAttribute(k_step_f32<O, 0, 32>, cudaFuncAttributeMaxDynamicSharedMemorySize, sm);
        cudaFuncSetAttribute(k_step_f32<O, 3, 32>, cudaFuncAttributeMaxDynamicSharedMemorySize, sm);
    } else {
        auto step = [](auto kc) {
            constexpr int TX = kEdgeShapes[decltype(kc)::value][0], TY = kEdgeShapes[decltype(kc)::value][1];
            constexpr int sm = (int)step_smem_f64<O, TX, TY>();
            cudaFuncSetAttribute(k_step_f64<O, 0, TX, TY>, cudaFuncAttributeMaxDynamicSharedMemorySize, sm);
            cudaFuncSetAttribute(k_step_f64<O, 2, TX, TY>, cudaFuncAttributeMaxDynamicSharedMemorySize, sm);
        };
        step(std::integral_constant<int, 0>());
        step(std::integral_constant<int, 1>());
        step(std::integral_constant<int, 2>());
        step(std::integral_constant<int, 3>());
    }
    if constexpr (std::is_same<T, double>::value) {
        strip(std::integral_constant<int, 16>());
        strip(std::integral_constant<int, 8>());
    }
    cudaFuncSetAttribute(k_interior<T, O, 0>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    cudaFuncSetAttribute(k_interior<T, O, 1>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    cudaFuncSetAttribute(k_interior<T, O, 2>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (std::is_same<T, float>::value) {
        cudaFuncSetAttribute(k_wide_march<O, 1>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)MarchCfg<O>::BYTES);
        cudaFuncSetAttribute(k_wide_march<O, 2>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)MarchCfg<O>::BYTES);
        cudaFuncSetAttribute(k_wide_march<O, 3>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)MarchCfg<O>::BYTES);
        cudaFuncSetAttribute(k_interior_march_multi<O, 0>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)MarchCfg<O>::BYTES);
        cudaFuncSetAttribute(k_interior_march_multi<O, 3>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)MarchCfg<O>::BYTES);
        cudaFuncSetAttribute(k_interior_march_multi<O, 1>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)MarchCfg<O>::BYTES);
        cudaFuncSetAttribute(k_interior_march_multi<O, 4>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)MarchCfg<O>::BYTES);
        cudaFuncSetAttribute(k_interior_march_multi<O, 5>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)MarchCfg<O>::BYTES);
        cudaFuncSetAttribute(k_interior_march_multi<O, 6>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)MarchCfg<O>::BYTES);
        cudaFuncSetAttribute(k_interior_march_multi<O, 7>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)MarchCfg<O>::BYTES);
    }
}

template <int O> int batch_ctas_per_sm() {
    cudaFuncSetAttribute(k_batch_step<O>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)batch_smem_bytes<O>());
    int per_sm = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_batch_step<O>, MTHREADS, batch_smem_bytes<O>());
    return per_sm;
}
template <int O> void batch_step_launch(int ctas, BatchHead* head, int* err, cudaStream_t st) {
    k_batch_step<O><<<ctas, MTHREADS, batch_smem_bytes<O>(), st>>>(head, err);
}

}  // namespace sbphost

// Host side shared by the translation units of libsbp: the handle, its block and face records, the device views, and
// the rules that pick launches.  sbp_api.cu holds the entry points; the kernels of each precision and order, with the
// functions that launch them (sbp_launch.cuh), are compiled by a translation unit of their own (sbp_ops.cu).
#pragma once
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <mutex>
#include <string>
#include <type_traits>
#include <vector>

#include <cuda.h>
#include <cudaTypedefs.h>


#include "../../include/sbp.h"
#include "sbp_interior_march.cuh"
#include "sbp_kernels.cuh"
#include "sbp_adjoint.cuh"
#include "sbp_batch.cuh"
#include "sbp_wide.cuh"
#include "sbp_step.cuh"

using namespace sbp;

namespace sbphost {
#define SBP_TABLE static const
#include "sbp_tables.inc"
#undef SBP_TABLE

struct HostFace {
    int kind = -1, nbr_block = -1, nbr_face = -1, reversed = 0;
    int nf = 0;
    double* jhat = nullptr;
    void* ju = nullptr;
    void* g = nullptr;
    void* sat = nullptr;      // wide stencil: SAT terms of the face nodes (k_face_sat); else unused (sbp_apply_noalloc
                              // points its views at its own scratch)
    void* tr = nullptr;       // interface faces: trace of this side (k_face_trace), 7 x nf
    void* jv = nullptr;       // Robin faces with damping: J^ V (3 x nf, type T)
};

struct HostBlock {
    int n1 = 0, n2 = 0, pitch = 0;
    double h1 = 0, h2 = 0;
    void* u[2] = {nullptr, nullptr};
    void* du = nullptr;       // FP32: the leapfrog increment u^n - u^{n-1} (2 planes)
    void* c = nullptr;
    void* w = nullptr;
    void* jf = nullptr;
    void* r = nullptr;
    double* X = nullptr;
    double* G = nullptr;
    double* J = nullptr;
    bool material = false;
    HostFace f[4];
    MarchMaps mmaps;          // FP32 column-marching interior kernel tensor maps
    void* psi[2] = {nullptr, nullptr};   // adjoint fields (sbp_misfit_gradient), allocated on first use
    MarchMaps pmaps;          // marching-kernel maps over the adjoint fields
    CUtensorMap* d_smaps = nullptr;   // strip-tile band-box maps on the device: [0..2] state u0, u1, c; [3..5] adjoint;
                                      // [6..11] the same for short tiles
    void* rk = nullptr;       // RK4 state (u, v, a_1, a_2, a_3; sbp_set_state_rk4), allocated on first use
    void* gw = nullptr;       // wide stencil: the fluxes G_1j, G_2j (4 planes, type T)
    void* sg = nullptr;       // layer dissipation coefficient s (1 plane, type T)
    int2* d_lnodes = nullptr; // nodes the layer dissipation reaches, (i1, i2)
    int nln = 0;
    void* lscr = nullptr;     // leapfrog: the dissipation of the listed nodes between the pre and post kernels
    void* mx = nullptr;       // closure matrices of D_xx^FC along x1 / x2 (k_closure_mats, type T)
    void* my = nullptr;
    void* e = nullptr;        // FP64 narrow stencil: interior edge weights (6 Q planes, k_edge_weights), optional (take_edges)
};

inline int order_nb(int o) { return o == 2 ? SBP2_NB : (o == 4 ? SBP4_NB : SBP6_NB); }
inline int order_ncol(int o) { return o == 2 ? SBP2_NCOL : (o == 4 ? SBP4_NCOL : SBP6_NCOL); }
inline int order_nclos(int o) { return o == 2 ? SBP2_NCLOS : (o == 4 ? SBP4_NCLOS : SBP6_NCLOS); }
inline int order_nclosj(int o) { return o == 2 ? SBP2_NCLOSJ : (o == 4 ? SBP4_NCLOSJ : SBP6_NCLOSJ); }
// elements of the closure matrices of one direction with `lines` lines (layout of dxx_closure_mat)
inline size_t closure_elems(int o, int lines) { return 2 * (size_t)order_nclos(o) * order_nclosj(o) * 3 * lines; }
inline int order_q(int o) { return o / 2; }
inline int order_min_n(int o) { return o == 2 ? 5 : (o == 4 ? 18 : 27); }
inline double order_hw(int o, int i) {
    return o == 2 ? sbphost::sbp2_HW[i] : (o == 4 ? sbphost::sbp4_HW[i] : sbphost::sbp6_HW[i]);
}
inline double order_dq0(int o, int c) {
    return o == 2 ? sbphost::sbp2_DQ[0][c] : (o == 4 ? sbphost::sbp4_DQ[0][c] : sbphost::sbp6_DQ[0][c]);
}
inline double host_hweight(int o, int N, int i) {
    const int nb = order_nb(o);
    if (i < nb) return order_hw(o, i);
    if (i >= N - nb) return order_hw(o, N - 1 - i);
    return 1.0;
}

}  // namespace sbphost

struct sbp_handle;
namespace sbphost {
bool reclaim_edges(sbp_handle* h);
cudaError_t device_malloc(void** p, size_t bytes);
}

struct sbp_handle {
    int order = 0, precision = 0, nblocks = 0;
    int stencil = SBP_STENCIL_NARROW;
    bool layers = false;          // some block has layer dissipation (sbp_set_layer_dissipation)
    bool damping = false;         // some face has Robin damping or some block layers
    double beta = 1.0;
    size_t esize = 8;
    std::vector<sbphost::HostBlock> blocks;
    BlockDev* d_blocks = nullptr;
    FaceRef* d_refs = nullptr;
    int nrefs = 0, nface_nodes = 0;
    int ntrefs = 0;               // interface faces (their traces: k_face_trace)
    int cur = 0;
    double t = 0.0;
    int nbasis = 0;
    int basis_kind[8] = {0};
    double basis_omega[8] = {0};
    std::vector<SrcNode> src_nodes;
    std::vector<SrcParam> src_params;
    SrcNode* d_src_nodes = nullptr;     // every source node (sbp_apply_noalloc)
    SrcNode* d_src_int = nullptr;       // source nodes off the boundary strips (k_sources)
    int n_src_int = 0;
    SrcNode* d_src_strip = nullptr;     // source nodes on the strips, grouped by strip tile (k_strip_tile)
    SrcParam* d_src_params = nullptr;
    bool src_dirty = false;
    double* d_scalar = nullptr;
    int* d_flag = nullptr;
    int* d_err = nullptr;       // kernel error flags (bounded waits that ran out)
    int num_sms = 0;
    int device = 0;             // CUDA device current at sbp_grid_create (holds every buffer)
    std::string err;
    std::vector<void*> allocs;
    // held by every call on the handle: another handle's call that finds no memory takes the edge weights from a handle
    // that is not in use (reclaim_edges)
    std::recursive_mutex use;
    bool edges_wanted = true;     // sbp_edge_weights
    size_t edge_bytes = 0;        // bytes of HostBlock::e over the blocks
    bool captured = false;        // a caller has captured steps that read them: they stay for good
    // kernel timing (benchmarks): the families of sbp_profile in include/sbp.h
    bool prof = false;
    double prof_ms[SBP_PROF_FAMILIES] = {0};
    long long launches[SBP_PROF_FAMILIES] = {0};
    std::vector<cudaEvent_t> ev_pool;
    struct Pending { int fam; cudaEvent_t a, b; };
    std::vector<Pending> pending;
    // CUDA-graph step loop (sbp_step_graph): graph of `graph_steps` steps of size `graph_dt`
    cudaGraphExec_t graph_exec = nullptr;
    int graph_steps = 0;
    double graph_dt = 0.0;
    double* d_time = nullptr;     // device copies of the step times of a graph launch
    int d_time_cap = 0;
    // marching-kernel rows per CTA chosen by sbp_autotune (0 = default heuristic)
    int rows_per_cta = 0;
    // optionally (sbp_autotune, sbp_set_tuning) the boundary strips run on a second stream
    // concurrently with the interior kernel (they write disjoint nodes); both are forked from and
    // joined back into the launch stream every step, the interior on a high-priority stream so
    // that its CTAs are placed first
    bool overlap = false;
    cudaStream_t hi = nullptr;
    cudaEvent_t ev_join_hi = nullptr;
    // strip tiles of every block, costliest first (one k_strip_tile launch per step)
    int4* d_tiles = nullptr;            // (block, tile, first, end source node of the tile) in launch order
    int ntiles = 0;
    int strip_len = 32;                 // nodes of a strip tile along the face (pick_strip_len)
    std::vector<int4> tiles_host;
    std::vector<std::vector<int>> tile_pos;   // [block][tile of the block] -> position in the launch order
    // FP32 grids whose strips make few tiles: a second set, SHORT_TILE nodes long, for the one-launch step (the
    // batch kernel and the others keep to 32)
    struct StripSet {
        int4* d_tiles = nullptr;
        SrcNode* d_src = nullptr;
        std::vector<int4> tiles;
        std::vector<std::vector<int>> pos;
    } shorts;
    cudaStream_t aux = nullptr;
    cudaEvent_t ev_fork = nullptr, ev_join = nullptr;
    // adjoint: block views whose state buffers are the adjoint fields; receivers
    BlockDev* d_blocks_adj = nullptr;
    std::vector<RecDev> recs;
    RecDev* d_recs = nullptr;

    cudaEvent_t get_event() {
        if (!ev_pool.empty()) {
            cudaEvent_t e = ev_pool.back();
            ev_pool.pop_back();
            return e;
        }
        cudaEvent_t e;
        cudaEventCreate(&e);
        return e;
    }

    int fail(int code, const std::string& msg) {
        err = msg;
        return code;
    }
    // one grow-only device staging buffer for host uploads and downloads: setup and transfer calls
    // use it instead of allocating and freeing temporaries (a free synchronises the whole device,
    // which would stall work other streams run meanwhile, e.g. a batch of served shots)
    void* stage = nullptr;
    size_t stage_bytes = 0;
    void* staging(size_t bytes) {
        if (bytes <= stage_bytes) return stage;
        if (stage) dfree(stage);
        stage = dalloc(bytes + bytes / 4);
        stage_bytes = stage ? bytes + bytes / 4 : 0;
        return stage;
    }
    void* dalloc(size_t bytes, bool clear = true) {
        void* p = nullptr;
        while (cudaMalloc(&p, bytes) != cudaSuccess) {
            cudaGetLastError();   // reported as SBP_E_OOM by the caller; the next launch check starts clean
            if (!sbphost::reclaim_edges(this)) return nullptr;
        }
        if (clear) cudaMemset(p, 0, bytes);
        allocs.push_back(p);
        return p;
    }
    void dfree(void* p) {
        if (!p) return;
        allocs.erase(std::remove(allocs.begin(), allocs.end(), p), allocs.end());
        cudaFree(p);
    }
};

namespace sbphost {

// records CUDA events around one kernel family when profiling is on; counts launches always
struct ProfScope {
    sbp_handle* h;
    int fam;
    cudaStream_t st;
    cudaEvent_t a = nullptr, b = nullptr;
    ProfScope(sbp_handle* h_, int fam_, cudaStream_t st_, int nlaunch) : h(h_), fam(fam_), st(st_) {
        h->launches[fam] += nlaunch;
        if (h->prof) {
            a = h->get_event();
            b = h->get_event();
            cudaEventRecord(a, st);
        }
    }
    ~ProfScope() {
        if (h->prof) {
            cudaEventRecord(b, st);
            h->pending.push_back({fam, a, b});
        }
    }
};

inline int check_cuda(sbp_handle* h, const char* where) {
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return h->fail(SBP_E_CUDA, std::string(where) + ": " + cudaGetErrorString(e));
    return SBP_OK;
}

inline BlockDev make_view(const sbp_handle* h, const HostBlock& hb) {
    BlockDev b{};
    b.n1 = hb.n1;
    b.n2 = hb.n2;
    b.pitch = hb.pitch;
    b.strip = std::max(order_nclos(h->order), order_ncol(h->order));
    b.h1 = hb.h1;
    b.h2 = hb.h2;
    b.ih1 = 1.0 / hb.h1;
    b.ih2 = 1.0 / hb.h2;
    b.ih1f = (float)b.ih1;
    b.ih2f = (float)b.ih2;
    b.u[0] = hb.u[0];
    b.u[1] = hb.u[1];
    b.du = hb.du;
    b.c = hb.c;
    b.w = hb.w;
    b.jf = hb.jf;
    b.r = hb.r;
    b.X = hb.X;
    b.G = hb.G;
    b.J = hb.J;
    for (int f = 0; f < 4; ++f) {
        const HostFace& F = hb.f[f];
        FaceDev& D = b.f[f];
        D.kind = F.kind;
        D.m = f / 2;
        D.side = f % 2;
        D.nf = F.nf;
        D.nbr_block = F.nbr_block;
        D.nbr_face = F.nbr_face;
        D.reversed = F.reversed;
        D.nu = (f % 2 == 0) ? -1.0 : 1.0;
        const int Nm = (f / 2 == 0) ? hb.n1 : hb.n2;
        const double hm = (f / 2 == 0) ? hb.h1 : hb.h2;
        D.hm0 = hm * host_hweight(h->order, Nm, 0);
        D.inv_h0 = 1.0 / D.hm0;
        // D_m[face row][i_m] / (h_m^2 hw(i_m)) at depth d: the boundary row of D (mirrored with the
        // opposite sign at the high end) over the norm weight
        for (int d = 0; d < 12; ++d) {
            const double dq0 = d < order_ncol(h->order) ? order_dq0(h->order, d) : 0.0;
            D.fac[d] = ((f % 2) ? -dq0 : dq0) / (hm * hm * host_hweight(h->order, Nm, (f % 2) ? Nm - 1 - d : d));
            D.facf[d] = (float)D.fac[d];
        }
        D.jhat = F.jhat;
        D.ju = F.ju;
        D.g = F.g;
        D.sat = F.sat;
        D.tr = F.tr;
        D.jv = F.jv;
        if (F.jv) b.damped = 1;
    }
    b.smaps = hb.d_smaps;
    b.rk = hb.rk;
    b.sg = hb.sg;
    b.mx = hb.mx;
    b.my = hb.my;
    b.e = hb.e;
    for (int k = 0; k < order_q(h->order); ++k) {
        const double ak = h->order == 2 ? sbphost::sbp2_A[k] : (h->order == 4 ? sbphost::sbp4_A[k] : sbphost::sbp6_A[k]);
        b.ai1[k] = ak * b.ih1;
        b.ai2[k] = ak * b.ih2;
    }
    return b;
}

// the same view with the adjoint fields as its state buffers
inline BlockDev make_view_adj(const sbp_handle* h, const HostBlock& hb) {
    BlockDev b = make_view(h, hb);
    b.u[0] = hb.psi[0];
    b.u[1] = hb.psi[1];
    b.du = nullptr;             // the adjoint fields step from their two levels
    b.smaps = hb.d_smaps ? hb.d_smaps + 3 : nullptr;
    return b;
}

inline unsigned grid_for(long long n, int bs = 256) { return (unsigned)((n + bs - 1) / bs); }

// length of the short strip tiles of FP32 grids (sbp_handle::shorts)
constexpr int SHORT_TILE = 8;

// rows per CTA of a marching kernel on a block with ncx tiles across: one wave of about 4 CTAs per SM, at least
// 16 rows (a tile streams 2q rows or more beyond its own), or the height that was tuned
inline int march_rows(const sbp_handle* h, int ncx, int n2i) {
    if (h->rows_per_cta > 0) return std::min(h->rows_per_cta, n2i);
    const int ncy = std::max(1, (4 * h->num_sms + ncx / 2) / ncx);
    return std::max((n2i + ncy - 1) / ncy, std::min(16, n2i));
}

// the FP64 interior of every block by k_interior_edges, up to IE_MAX_BLOCKS blocks a launch.  The tile
// shape is the one whose busiest SM executes the fewest FP64 instructions (the kernel is bound by
// them): 32 x 16 nodes repeat the fewest fluxes on their halos and win once there are several tiles per
// SM, 16 x 4 nodes leave no SM idle on a 101^2 grid (138 tiles against 18).   Order 4, 101^2: 13 us
// against 38 us for 32 x 16 tiles with their own weights.
constexpr int kEdgeShapes[4][2] = {{32, 16}, {32, 8}, {32, 4}, {16, 4}};
inline int pick_edge_shape(const sbp_handle* h) {
    const int Q = order_q(h->order), S = std::max(order_nclos(h->order), order_ncol(h->order));
    const int node = 8 * Q * 4 + 12, flux = 6 * Q + 4;
    int best = 0;
    long long least = -1;
    for (int k = 0; k < 4; ++k) {
        const int tx = kEdgeShapes[k][0], ty = kEdgeShapes[k][1];
        long long tiles = 0;
        for (auto& hb : h->blocks)
            tiles += (long long)((hb.n1 - 2 * S + tx - 1) / tx) * ((hb.n2 - 2 * S + ty - 1) / ty);
        const long long cost = (tiles + h->num_sms - 1) / h->num_sms *
                               (tx * ty * node + flux * ((tx + 2 * Q) * ty + tx * (ty + 2 * Q)));
        if (least < 0 || cost < least) {
            least = cost;
            best = k;
        }
    }
    return best;
}
// the interior tiles of blocks [first, first + IE_MAX_BLOCKS) in shape k; returns their number
inline int edge_tiles(const sbp_handle* h, int first, int k, InteriorTiles& tl) {
    const int S = std::max(order_nclos(h->order), order_ncol(h->order)), tx = kEdgeShapes[k][0], ty = kEdgeShapes[k][1];
    tl = InteriorTiles{};
    tl.first = first;
    int tiles = 0;
    for (int b = first; b < std::min(h->nblocks, first + IE_MAX_BLOCKS); ++b) {
        const HostBlock& hb = h->blocks[b];
        tl.ncx[tl.nb] = (hb.n1 - 2 * S + tx - 1) / tx;
        tl.start[tl.nb++] = tiles;
        tiles += tl.ncx[tl.nb - 1] * ((hb.n2 - 2 * S + ty - 1) / ty);
    }
    tl.start[tl.nb] = tiles;
    return tiles;
}

// Rows of the interior items (128 columns of a marching kernel, bands of equal height per grid) that share `slots`
// CTAs with `strips` strip tiles.  An item costs its rows and about ITEM_ROWS more (the rows it marches before
// its first output, its start), a strip tile about STRIP_ROWS; the height minimises the larger of the mean load
// and the rounds of the longest item.  grids: (tiles across, interior rows).
inline int item_rows(int slots, const std::vector<int2>& grids, long long strips, bool queued) {
    constexpr double ITEM_ROWS = 14, STRIP_ROWS = 10;
    double least = 1e300;
    int best = 64;
    for (int rows = 8; rows <= 256; rows += rows < 32 ? 1 : 4) {
        long long items = 0;
        double work = strips * STRIP_ROWS, longest = 0;
        for (const int2& s : grids) {
            const int bands = (s.y + rows - 1) / rows, high = (s.y + bands - 1) / bands;
            items += (long long)s.x * bands;
            work += (double)s.x * (s.y + bands * ITEM_ROWS);
            longest = std::max(longest, high + ITEM_ROWS);
        }
        // (strip tiles first, one per slot, or queued behind the items)
        const double cost = std::max(work / slots, (double)((items + (queued ? 0 : strips) + slots - 1) / slots) * longest);
        if (cost < least) {
            least = cost;
            best = rows;
        }
    }
    return best;
}

// Whether a step runs as one launch (sbp_step.cuh): the blocks fit the launch's tables.  A property of the handle, whatever
// its tuning and whether its kernels are being timed, so that neither changes the rounding of a result (the one-launch
// kernels sum a face node's SAT terms by parts) and sbp_profile times the launches that steps make.  FP32: leapfrog steps of the state or the adjoint fields, up to as many strip tiles as SMs
// (1200^2; larger grids fill the chip with either kernel, see the figures there) and without interfaces, whose
// traces now form beside the interior (2 x 402 x 201: 38 us a step, 41 with the traces first).  FP64: leapfrog steps and RK4 stages
// with strip tiles of 8 nodes, or 16 without interfaces (4 blocks of 401^2: 264 us in one launch, 258 in two), not on
// the largest grids, where FP64 arithmetic alone counts.  (Where it is one launch there is nothing for the overlap of
// sbp_set_tuning to run side by side.)
inline bool one_launch(const sbp_handle* h, int mode) {
    if (h->nblocks > MARCH_MAX_BLOCKS || h->stencil != SBP_STENCIL_NARROW) return false;
    if (h->precision == SBP_FP32) return mode == 0 && h->ntrefs == 0 && (h->shorts.d_tiles || h->ntiles <= h->num_sms);
    return mode != 1 && h->blocks[0].e && (h->strip_len == 8 || (h->strip_len == 16 && h->ntrefs == 0));
}

// the interior shape that goes with the strip tiles of an FP64 step in one launch
inline int step_edge_shape(const sbp_handle* h) { return h->strip_len == 16 ? 0 : std::max(1, pick_edge_shape(h)); }

// strip nodes of the gradient (bands of width gs along every face)
inline long long grad_strip_nodes(const HostBlock& hb, int gs) {
    return (long long)hb.n1 * hb.n2 - (long long)(hb.n1 - 2 * gs) * (hb.n2 - 2 * gs);
}
inline int order_gs(int o) { return o == 2 ? SBP2_GS : (o == 4 ? SBP4_GS : SBP6_GS); }
// level chunks of the strip gradient: about 4 waves of 256-thread CTAs over the SMs, at most
// one chunk per level and at most GRAD_MAX_CHUNKS
constexpr int GRAD_MAX_CHUNKS = 16;
inline int grad_strip_chunks(const sbp_handle* h, long long nstrip, int nl) {
    const long long want = 4LL * h->num_sms * 2048;
    long long c = (want + nstrip - 1) / std::max(1LL, nstrip);
    c = std::min<long long>(c, GRAD_MAX_CHUNKS);
    c = std::min<long long>(c, nl);
    return (int)std::max(1LL, c);
}

// Whether an FP32 wide-stencil operator marches over the interior (k_wide_march beside the frame's kernels) or takes
// two passes over every node.  The march reads each node once, but costs a launch and a fork and join of streams, which the
// host pays where the kernels are short.  The line lies where the two are equal, in nodes of all blocks (a block's own two
// launches move it up): order 6 about 300 k on one block, 450 k on four (us a step, two passes / march: 601 x 477 38.2 /
// 42.4, 801 x 627 43.1 / 41.4; 4 x 301^2 87 / 98, 4 x 401^2 103 / 99; 2 x 201 x 177 59 / 62, 2 x 601 x 477 68 / 65); orders 2
// and 4, whose marches save less, 350 k and 950 k (order 4: 601 x 477 33.7 / 33.9, 801 x 627 38.6 / 34.3; order 2: 2 x
// 401 x 327 43.4 / 50.8, 2 x 801 x 627 65 / 52; 4 x 401^2 77 / 84, 4 x 601^2 124 / 118).
inline bool wide_by_march(const sbp_handle* h) {
    long long nodes = 0;
    for (auto& hb : h->blocks) nodes += (long long)hb.n1 * hb.n2;
    const long long nb = h->nblocks;
    return nodes >= (h->order == 6 ? 250000 + 50000 * nb : 150000 + 200000 * nb);
}

// ------------------------------------------------------------------ per precision and order (sbp_launch.cuh)
template <typename T, int O> int launch_operator(sbp_handle* h, const StepArgs& a, int mode, cudaStream_t st, bool adj);
template <typename T, int O> int launch_wide(sbp_handle* h, const StepArgs& a, int mode, cudaStream_t st);
template <typename T, int O> void layer_launch(sbp_handle* h, const StepArgs& a, int mode, cudaStream_t st, bool post);
template <typename T, int O> void set_smem_attr();
template <typename T, int O>
void launch_noalloc(sbp_handle* h, const BlockDev* views, int nviews, BlockDev* d_views, FaceRef* d_refs, const StepArgs& a,
                    cudaStream_t st);
template <typename T, int O>
void launch_grad(sbp_handle* h, const GradDev* d_grad, const std::vector<GradDev>& grads, int nl, double dt2, cudaStream_t st);
// the persistent batch kernel (FP32): CTAs that are resident on an SM, one step of the batch
template <int O> int batch_ctas_per_sm();
template <int O> void batch_step_launch(int ctas, BatchHead* head, int* err, cudaStream_t st);

}  // namespace sbphost

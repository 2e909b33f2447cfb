// A whole step in one launch (after the interface traces, where there are interfaces: read by the strip tiles
// themselves, the neighbour's tractions made a tile's 17 us 38): the first CTAs take the boundary-strip tiles, the others the interior tiles.
// All of them read level n and write level n + 1 at disjoint nodes, so they run side by side: a small or
// middling grid leaves most of the chip idle in either kernel and waits for each one's latency and launch in
// turn.  An interior tile then adds the off-strip source nodes that lie in it (as k_sources does after the step kernels; the same
// arithmetic), which saves that launch as well.
// A step of one block, FP32, order 6, with a source inside, against separate launches: 201^2 36.6 -> 14.7 us, 601^2
// 37.7 -> 20.6, 1001^2 46.1 -> 28.7, but 1401^2 66.6 -> 72.7 (the strips by 128 threads then cost more than the
// launches do); FP64, order 6: 201^2 45 -> 32 us, 601^2 158 -> 135; order 4: 101^2 41 -> 23.
#pragma once
#include "sbp_interior_march.cuh"
#include "sbp_kernels.cuh"

namespace sbp {

struct StepStrips {
    const BlockDev* blocks;
    const int4* tiles;            // strip tiles in launch order
    int n;                        // their number: CTAs 0 .. n-1
    int nisrc;                    // off-strip source nodes
    const SrcNode* ssrc;          // strip source nodes (by tile) or null
    const SrcNode* isrc;
    const SrcParam* spar;
    double beta;
};
// with more off-strip source nodes than this, k_sources takes them (every tile looks through the list)
constexpr int STEP_MAX_SOURCES = 512;

// the off-strip source nodes of block b in [lo1, hi1) x [lo2, hi2), once the tile's nodes are stored
template <typename T, int MODE>
__device__ __forceinline__ void tile_sources(const StepStrips& s, int b, int lo1, int hi1, int lo2, int hi2, const StepArgs& a) {
    if (s.nisrc == 0 || !a.with_data) return;
    __syncthreads();
    const BlockDev& B = s.blocks[b];
    for (int k = threadIdx.x; k < s.nisrc; k += blockDim.x) {
        const SrcNode nd = s.isrc[k];
        if (nd.block != b) continue;
        const int i2 = (int)(nd.gi / B.pitch), i1 = (int)(nd.gi - (long long)i2 * B.pitch);
        if (i1 >= lo1 && i1 < hi1 && i2 >= lo2 && i2 < hi2) source_add<T, MODE>(B, nd, s.spar, a);
    }
}

template <int O> constexpr size_t step_smem_f32() {
    return MarchCfg<O>::BYTES > StripTile<O, 32, (O > 2)>::template bytes<float>() ? MarchCfg<O>::BYTES
                                                                                  : StripTile<O, 32, (O > 2)>::template bytes<float>();
}

// FP32 leapfrog step; MODE 3: increment form, 0: the adjoint fields' two levels
template <int O, int MODE, int TL>
__global__ void __launch_bounds__(MTHREADS, 4)
k_step_f32(const __grid_constant__ MarchMulti mm, const __grid_constant__ StepStrips ss, StepArgs a, int* err) {
    extern __shared__ __align__(128) unsigned char step_smem[];
    const int k = (int)blockIdx.x - ss.n;
    if (k < 0) {
        (void)strip_tile_body<float, O, 0, MTHREADS, TL, (O > 2)>(ss.blocks, ss.tiles[blockIdx.x], a, ss.beta, err, ss.ssrc, ss.spar, step_smem);
        return;
    }
    int b = 0;
    while (b + 1 < mm.nb && k >= mm.start[b + 1]) ++b;
    const int tile = k - mm.start[b];
    (void)march_tile<O, MODE>(mm.maps[b], mm.b[b], a, mm.rows[b], tile, err, step_smem);
    const int S = mm.b[b].strip, ncx = march_ncx(mm.b[b].n1, S), x0 = march_x0(S) + (tile % ncx) * MTHREADS;
    const int y0 = S + (tile / ncx) * mm.rows[b];
    tile_sources<float, 0>(ss, b, x0, x0 + MTHREADS, y0, y0 + mm.rows[b], a);
}

// FP64 leapfrog step (MODE 0) or RK4 stage (MODE 2): strip tiles of 16 nodes beside interior tiles of 32 x 16,
// of 8 nodes beside the smaller ones
template <int TX, int TY> constexpr int step_len_f64() { return TX * TY == 512 ? 16 : 8; }
template <int TX, int TY> constexpr int step_threads_f64() { return TX * TY == 512 ? 256 : 128; }
template <int O, int TX, int TY> constexpr size_t step_smem_f64() {
    constexpr size_t strip = StripTile<O, step_len_f64<TX, TY>(), (O > 2)>::template bytes<double>();
    return edge_tile_elems<O, TX, TY>() * sizeof(double) > strip ? edge_tile_elems<O, TX, TY>() * sizeof(double) : strip;
}
template <int O, int MODE, int TX, int TY>
__global__ void __launch_bounds__(step_threads_f64<TX, TY>(), 512 / step_threads_f64<TX, TY>())
k_step_f64(const __grid_constant__ InteriorTiles tl, const __grid_constant__ StepStrips ss, StepArgs a, int* err) {
    constexpr int NT = step_threads_f64<TX, TY>();
    extern __shared__ __align__(128) unsigned char step_smem[];
    const int k = (int)blockIdx.x - ss.n;
    if (k < 0) {
        (void)strip_tile_body<double, O, MODE, NT, step_len_f64<TX, TY>(), (O > 2)>(ss.blocks, ss.tiles[blockIdx.x], a, ss.beta, err,
                                                                           ss.ssrc, ss.spar, step_smem);
        return;
    }
    int b = 0;
    while (b + 1 < tl.nb && k >= tl.start[b + 1]) ++b;
    const int tile = k - tl.start[b], ncx = tl.ncx[b];
    const BlockDev& B = ss.blocks[b];
    interior_edges_tile<double, O, MODE, TX, TY, NT>(B, tile, ncx, a, reinterpret_cast<double*>(step_smem));
    const int x0 = B.strip + (tile % ncx) * TX, y0 = B.strip + (tile / ncx) * TY;
    tile_sources<double, MODE>(ss, b, x0, x0 + TX, y0, y0 + TY, a);
}

}  // namespace sbp

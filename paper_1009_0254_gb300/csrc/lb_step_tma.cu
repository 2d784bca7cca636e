// lb_step_tma.cu -- the fused fluctuating D2Q9 step of FP32 lattices, TMA-staged and persistent (FP16
// lattices: lb_step_half.cu).
//
// Same arithmetic as lb_step.cu (collide_node), two nodes at a time (collide_pair of lb_pair.cuh),
// and different data movement:
//   * a persistent grid (resident CTAs only) walks the lattice in TX x TY tiles (the shape
//     chosen per noise mode, tma_default_tile) in row-major tile order, so the
//     tiles in flight form a band whose halo rows are still in L2 when the neighbouring tile
//     reads them;
//   * for each tile one thread issues nine 3D TMA loads (cp.async.bulk.tensor), one per
//     population plane, of the box [x0 - 4, x0 + TX + 4) x [y0 - 1 - cy_i, y0 + TY + 1 - cy_i)
//     into shared memory; the y offset of plane i absorbs its streaming shift, so node
//     (lx, ly) of the tile reads f_i at box[ly + 1][lx + 4 - cx_i].  The x start is rounded
//     down to a 16-byte boundary (four floats) as TMA requires;
//   * every thread pulls its pairs' nine deviations from shared memory into registers and
//     writes their density to a tile-plus-ring array (the ring from the halo); after one
//     barrier the next tile is loaded into the same stage while every pair collides.  Nodes
//     beyond a ragged edge of the lattice take part in the density pass (their values are
//     never used);
//   * the post-collision planes go to a tile in shared memory, which leaves with one TMA store
//     (a box of nine planes, clipped to the lattice) behind the next tile's density pass; the
//     periodic ghost copies of a tile near an edge are stored by its threads.
//
// One load in flight per CTA, not two: with the tile after next requested early the 4096^2 step
// had 190 KB of requests outstanding per SM, and DRAM then answers more slowly (no noise 250 us
// against 191 on the same tiles; a plain copy of nine planes shows the same, 183 us with 55 KB
// in flight per SM and 233 us with 147 KB).
//
// Step at 4096^2, before and after this form (scalar nodes, two stages, stores by thread):
// without noise 262 -> 186 us, uncorrelated 212 -> 191 (6.32 TB/s of the 72 bytes a node), k-space
// correlated (the step kernel alone) 235 -> 221, real space 333 -> 263, local density 219 -> 194.  What
// bounds it now: DRAM; the real-space noise the SM (FMA-heavy pipe 60 % busy, half of it the wide
// multiplies of Philox, and the barriers between the passes).
//
// Waits on the mbarriers are bounded by the global timer; a CTA that gives up sets the
// error word, gives its loads in flight a bounded chance to land, and returns.
#include <cuda.h>

#include "lb_limits.cuh"
#include "lb_pair.cuh"

namespace lbf {

// What one launch reads, by value: the lattice's coefficients as lb_pair.cuh takes them, the
// time and the Philox round keys.
struct TmaArgs : PairCoef, PairStencil {
    PairLocal loc;     // POLY and MODE 4
    Grid g;
    float* dst;
    const float2* xi49;
    int ntx, nty;      // tiles along x and y
    int* err;          // device error word (1 = a TMA wait timed out)
    uint32_t t_lo, t_hi;
    RoundKeys rk;
};

// POLY: the double-well equation of state (the bulk pressure's quartic in drho)
template <int TX, int TY, int NT, int MODE, bool POLY = false>
__global__ void __launch_bounds__(NT, (pair_min_blocks<TX, TY, NT, MODE == 3>()))
    step_tma_kernel(const __grid_constant__ CUtensorMap lmap, const __grid_constant__ CUtensorMap smap,
                    const TmaArgs a) {
    using TT = TmaTile<TX, TY>;
    using M = PairMap<TX, TY, NT>;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    float* S = reinterpret_cast<float*>(smem_raw);
    float* out = reinterpret_cast<float*>(smem_raw + TT::OUT);
    float* R = reinterpret_cast<float*>(smem_raw + TT::RHO);
    const uint32_t bar = smem_u32(smem_raw + TT::BAR);
    unsigned char* xch = smem_raw + TT::SMEM_BYTES;     // MODE 3: StencilTile
    const Grid g = a.g;
    const int tid = threadIdx.x;
    const int ntiles = a.ntx * a.nty;

    if (tid == 0) {
        mbar_init(bar, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&lmap)) : "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&smap)) : "memory");
    }
    __syncthreads();
    grid_wait();
    grid_next();

    // the nine boxes of the tile in column col, row row of the tiling
    auto load = [&](int col, int row) {
        const int x0 = col * TX, y0 = row * TY;
        mbar_expect_tx(bar, TT::TX_BYTES);
#pragma unroll
        for (int i = 0; i < Q; ++i)
            tma_load_3d(smem_u32(S + i * TT::PS), &lmap, x0 - TT::XO + g.gx, y0 - 1 - kCYt[i] + GY, i, bar);
    };

    // a tile's column and row, advanced by the grid stride without a division per tile
    const int first = blockIdx.x;
    const int stx = (int)gridDim.x % a.ntx, sty = (int)gridDim.x / a.ntx;
    int tcol = first % a.ntx, trow = first / a.ntx;
    if (tid == 0 && first < ntiles) load(tcol, trow);
    int px0 = 0, py0 = 0;                  // the tile whose results are in `out`
    uint32_t k = 0;
    for (int tile = first; tile < ntiles; tile += gridDim.x, ++k) {
        // bounded wait for this tile's nine boxes; the decision to give up is collective (the
        // barrier also orders the previous tile's reads of R and writes of `out` before this
        // tile's writes and the store)
        const bool ok = mbar_wait_bounded(bar, k & 1u);
        if (__syncthreads_or(!ok)) {
            if (tid == 0) {
                atomicExch(a.err, 1);
                // give the loads still in flight into this CTA's shared memory a bounded
                // chance to land before the CTA exits
                mbar_wait_bounded(bar, k & 1u);
                tma_store_wait();
            }
            return;
        }
        if (tid == 0 && k > 0 && !tile_direct<TX>(g, px0)) {
            tma_store_3d(&smap, smem_u32(out), px0, py0, 0);
            tma_store_commit();
        }
        const int x0 = tcol * TX, y0 = trow * TY;
        px0 = x0;
        py0 = y0;
        tcol += stx;                       // now the next tile's
        trow += sty;
        if (tcol >= a.ntx) {
            tcol -= a.ntx;
            ++trow;
        }

        // each thread pulls its pairs of nodes once, keeps them in registers across the barrier
        // and writes their density to the tile; the ring is formed separately
        F2 fr[M::RPT][Q];
        tile_pull<TX, TY, NT, MODE == 3>(S, R, fr);
        F2 z4[M::RPT], z9[M::RPT];
        if constexpr (MODE == 3) stencil_tile<TX, TY, NT>(a, xch, x0, y0, g.nx, g.ny, z4, z9);
        if (tid == 0) tma_store_wait_read();
        __syncthreads();
        // the collision pass reads no population from the stage: load the next tile now
        if (tid == 0 && tile + (int)gridDim.x < ntiles) {
            fence_async_smem();
            load(tcol, trow);
        }
        tile_collide<MODE, POLY, TX, TY, NT>(a, &a.loc, fr, R, g, x0, y0, out, a.dst, a.xi49, z4, z9, xch);
        fence_async_smem();
    }
    __syncthreads();
    if (tid == 0 && k > 0) {
        if (!tile_direct<TX>(g, px0)) {
            tma_store_3d(&smap, smem_u32(out), px0, py0, 0);
            tma_store_commit();
        }
        tma_store_wait();              // of earlier tiles too, if the last one left by its threads
    }
}

// --- host side ----------------------------------------------------------------------

EncodeTiledFn tensor_map_encoder() {
    static const EncodeTiledFn fn = [] {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        const bool ok = cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
                            cudaSuccess && q == cudaDriverEntryPointSuccess;
        return ok ? (EncodeTiledFn)p : (EncodeTiledFn) nullptr;
    }();
    return fn;
}

// Tile shapes (TX x TY nodes, NT threads): 0 = 32x16/256, 1 = 32x32/256, 2 = 64x8/256,
// 3 = 64x16/512, 4 = 32x16/128.
static const int kTiles[5][3] = {{32, 16, 256}, {32, 32, 256}, {64, 8, 256}, {64, 16, 512}, {32, 16, 128}};

int tma_tile_count() { return 5; }

// The fastest shape per noise mode (0 off, 1 uncorrelated, 2 correlated, 3 correlated built in real
// space, 4 local density) and storage, measured at 4096^2 (FP32, us a step, shapes 0 to 4):
//   off 191 208 186 205 190, uncorrelated 194 213 191 209 193, correlated (kernel alone) 232 257
//   221 225 229, real space 294 281 304 402 263, local 195 218 194 211 198.
// Four CTAs per SM hide each other's barriers: one pair a thread where the registers allow 32 warps
// (shape 2), two pairs and 16 warps where the contributions of the real-space noise need them
// (shape 4: their exchange stays within a thread for half the rows).  2048^2 and 3000^2 agree; below
// 512^2 a step is bound by its launch and the shape does not matter.  FP16 (lb_step_half.cu): the shapes
// its recorded states were computed with, the fastest of that kernel.
int tma_default_tile(int noise_mode, int fp16, const Grid& g) {
    static const int best[2][5] = {{2, 2, 2, 4, 2}, {4, 1, 3, 0, 1}};
    const int m = noise_mode < 0 ? 0 : (noise_mode > 4 ? 4 : noise_mode);
    // real space, up to four CTAs a SM of 256 threads: one row of pairs a thread instead of two shortens the
    // step, which is a tile's latency there (33 x 47 9.7 us against 11.7, 128^2 8.7 and 10.0, 512^2 12.6 and
    // 13.6; 700^2 16.3 and 16.4, 1000 x 600 19.9 and 18.9)
    if (!fp16 && m == 3 && (long long)((g.nx + 31) / 32) * ((g.ny + 15) / 16) <= 4LL * device_sms()) return 0;
    return best[fp16 ? 1 : 0][m];
}

// Tensor maps over one population buffer.  For loads: dims (pitch, ny + 2 GY, 9), a plane's box of
// the tile with its halo.  For stores (FP32): dims (nx, ny, 9) from node (0, 0), so that a ragged tile
// is clipped to the lattice, the nine planes of the tile in one box.
bool make_pop_tensor_maps(const void* buf, const Grid& g, int tile, int fp16, void* load_map, void* store_map) {
    EncodeTiledFn fn = tensor_map_encoder();
    if (!fn || tile < 0 || tile >= tma_tile_count()) return false;
    const cuuint64_t es = fp16 ? 2 : 4;
    const int xo = fp16 ? Elem<__half>::XO : Elem<float>::XO;
    const CUtensorMapDataType dt = fp16 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT16 : CU_TENSOR_MAP_DATA_TYPE_FLOAT32;
    cuuint64_t strides[2] = {(cuuint64_t)g.pitch * es, (cuuint64_t)g.plane * es};
    cuuint32_t estr[3] = {1, 1, 1};
    cuuint64_t ldims[3] = {(cuuint64_t)g.pitch, (cuuint64_t)(g.ny + 2 * GY), (cuuint64_t)Q};
    cuuint32_t lbox[3] = {(cuuint32_t)(kTiles[tile][0] + 2 * xo), (cuuint32_t)kTiles[tile][1] + 2, 1};
    if (fn(reinterpret_cast<CUtensorMap*>(load_map), dt, 3, (void*)buf, ldims, strides, lbox, estr,
           CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
           CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
        return false;
    if (fp16) return true;
    cuuint64_t sdims[3] = {(cuuint64_t)g.nx, (cuuint64_t)g.ny, (cuuint64_t)Q};
    cuuint32_t sbox[3] = {(cuuint32_t)kTiles[tile][0], (cuuint32_t)kTiles[tile][1], (cuuint32_t)Q};
    return fn(reinterpret_cast<CUtensorMap*>(store_map), dt, 3, (char*)buf + g.at(0, 0) * es, sdims, strides, sbox, estr,
              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_NONE,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

size_t tensor_map_bytes() { return sizeof(CUtensorMap); }

template <int TX, int TY, int NT, int MODE, bool POLY = false>
static cudaError_t launch_cfg(const void* const map[2], TmaArgs ta, cudaStream_t s) {
    using TT = TmaTile<TX, TY>;
    auto kern = step_tma_kernel<TX, TY, NT, MODE, POLY>;
    constexpr int smem = TT::SMEM_BYTES + (MODE == 3 ? StencilTile<TX, TY, NT>::BYTES : 0);
    static GridCache cache;
    int grid_max = 0;
    cudaError_t e = resident_grid(kern, NT, smem, cache, &grid_max);
    if (e != cudaSuccess) return e;
    ta.ntx = (ta.g.nx + TX - 1) / TX;
    ta.nty = (ta.g.ny + TY - 1) / TY;
    const int ntiles = ta.ntx * ta.nty;
    const int grid = ntiles < grid_max ? ntiles : grid_max;
    return launch_chained(kern, grid, NT, smem, s, *static_cast<const CUtensorMap*>(map[0]),
                          *static_cast<const CUtensorMap*>(map[1]), ta);
}

template <int MODE>
static cudaError_t launch_mode(const void* const map[2], const TmaArgs& ta, int tile, cudaStream_t s) {
    switch (tile) {
        case 1: return launch_cfg<32, 32, 256, MODE>(map, ta, s);
        case 2: return launch_cfg<64, 8, 256, MODE>(map, ta, s);
        case 3: return launch_cfg<64, 16, 512, MODE>(map, ta, s);
        case 4: return launch_cfg<32, 16, 128, MODE>(map, ta, s);
        default: return launch_cfg<32, 16, 256, MODE>(map, ta, s);
    }
}

// the double-well equation of state, FP32 storage: the default tile of each noise mode
// (tma_default_tile; the caller encodes the tensor maps for it)
static cudaError_t launch_poly(const void* const map[2], const TmaArgs& ta, int noise_mode, int tile, cudaStream_t s) {
    switch (noise_mode) {
        case 0: return launch_cfg<64, 8, 256, 0, true>(map, ta, s);
        case 1: return launch_cfg<64, 8, 256, 1, true>(map, ta, s);
        case 3: return tile == 0 ? launch_cfg<32, 16, 256, 3, true>(map, ta, s) : launch_cfg<32, 16, 128, 3, true>(map, ta, s);
        case 4: return launch_cfg<64, 8, 256, 4, true>(map, ta, s);
        default: return launch_cfg<64, 8, 256, 2, true>(map, ta, s);
    }
}

cudaError_t launch_step_tma(const StepArgs& a, const StepArgsD& d, const void* src_map, const void* dst_map, int* err, int noise_mode, int tile,
                            cudaStream_t s, bool poly) {
    TmaArgs ta;
    // the coefficients from FP64, rounded once
    const double L[4] = {d.L44, d.L49, d.L94, d.L99}, s3[3] = {d.s5, d.s6, d.s7};
    pair_coef(d.rho0, d.cs2m, d.kappa, d.lb, d.ls, d.lq, d.le, L, s3, &ta);
    pair_stencil(d.sL, &ta);
    pair_local(d.e2, d.e3, d.e4, d.cq, d.lu, &ta.loc);
    ta.g = a.g;
    ta.dst = static_cast<float*>(a.dst);
    ta.xi49 = a.xi49;
    ta.ntx = ta.nty = 0;
    ta.err = err;
    ta.t_lo = a.t_lo;
    ta.t_hi = a.t_hi;
    ta.rk = a.rk;
    const void* const map[2] = {src_map, dst_map};
    if (poly) return launch_poly(map, ta, noise_mode, tile, s);
    switch (noise_mode) {
        case 0: return launch_mode<0>(map, ta, tile, s);
        case 1: return launch_mode<1>(map, ta, tile, s);
        case 3: return launch_mode<3>(map, ta, tile, s);
        case 4: return launch_mode<4>(map, ta, tile, s);
        default: return launch_mode<2>(map, ta, tile, s);
    }
}

}  // namespace lbf

// lb_step_half.cu -- the fused fluctuating D2Q9 step of FP16 lattices, TMA-staged and persistent: one node
// a lane, collide_node in the stored form g_i = df_i / w_i, two tiles in flight per CTA.
//
// Why not the pairs of lb_step_tma.cu.  Every stored value is an FP32 sum rounded to FP16, and a sum that
// is fused or ordered otherwise rounds the values next to a boundary of FP16 the other way: after some tens
// of steps two such runs differ by 2^-11 of a value everywhere, and their structure factors by 1e-4 to 1e-3
// a bin, where this library's FP32 outputs repeat to 2e-5.  So what an FP16 lattice computes is tied to
// this kernel, its tile shapes and its order of operations (golden/fp16_states.txt of the tests has it bit
// for bit).  On pairs with one tile in flight and TMA stores 2048^2 took 53 us a step instead of 69 and
// 4096^2 182 instead of 222, with other roundings; the pairs' data movement around collide_node took 207 and
// had other roundings too, as the compiler fuses the same source otherwise in another kernel.
//
// What bounds it: issue (368 instructions a node at 71 % issue, FP32 arithmetic on half the bytes).  4096^2, us a step: no
// noise 162, uncorrelated 222, k-space correlated 228 (the step kernel), real space 339, local density 233.
#include <cuda.h>

#include "lb_collide.cuh"
#include "lb_tma.cuh"

namespace lbf {

// Shared memory of one CTA: two stages (nine boxes each), the density tile with its one-node ring, the
// mbarriers and, with MODE 3, the 2 x 2-box noise contributions.
template <int TX, int TY>
struct HalfTile {
    static constexpr int XO = Elem<__half>::XO;                         // 16 bytes of elements
    static constexpr int BW = TX + 2 * XO;                              // box width (elements)
    static constexpr int BH = TY + 2;                                   // box height
    static constexpr int PLANE_BYTES = BW * BH * 2;
    static constexpr int PS = ((PLANE_BYTES + 127) / 128) * 128 / 2;    // plane stride (elements)
    static constexpr int STAGE = Q * PS;                                // elements per stage
    static constexpr int STAGE_BYTES = STAGE * 2;
    static constexpr int RW = TX + 2, RH = TY + 2;                      // density tile + ring
    static constexpr int SMEM_BYTES = 2 * STAGE_BYTES + RW * RH * 4 + 2 * 8;
    static constexpr uint32_t TX_BYTES = Q * PLANE_BYTES;
    // real-space correlated noise: h00, h10, h01, h11 (float2 each) of the tile's nodes and of
    // the column left of it and the row below it, (TX + 1) x (TY + 1) nodes, after the mbarriers
    static constexpr int HW = TX + 1;
    static constexpr int HN = (TX + 1) * (TY + 1);
    static constexpr int H_BYTES = 4 * HN * 8;
    static constexpr int H_OFFSET = SMEM_BYTES;
    static_assert(H_OFFSET % 16 == 0, "H must be 16-byte aligned");
};

// The nine pulled values of the node whose unshifted box index is b: plane i is read at
// b - cx_i (its y shift is already in the box origin).
template <int PS>
__device__ __forceinline__ void load9_g(const __half* S, int b, float f[Q]) {
    f[0] = Elem<__half>::load_g(S[b]);
    f[1] = Elem<__half>::load_g(S[PS + b - 1]);
    f[2] = Elem<__half>::load_g(S[2 * PS + b]);
    f[3] = Elem<__half>::load_g(S[3 * PS + b + 1]);
    f[4] = Elem<__half>::load_g(S[4 * PS + b]);
    f[5] = Elem<__half>::load_g(S[5 * PS + b - 1]);
    f[6] = Elem<__half>::load_g(S[6 * PS + b + 1]);
    f[7] = Elem<__half>::load_g(S[7 * PS + b + 1]);
    f[8] = Elem<__half>::load_g(S[8 * PS + b - 1]);
}

// Real-space correlated noise of a tile (LB_NOISE_FULL_RS): the contributions h_d(q) of a
// node q of the tile, or of the column left of it / row below it (local coordinates -1),
// go to H[d][(ly + 1) * HW + lx + 1]; the (xi_4, xi_9) of a tile node are then
// h00(r) + h10(r - e_x) + h01(r - e_y) + h11(r - e_x - e_y).
template <int HW>
__device__ __forceinline__ void stencil_store(const StepArgs& a, float2* H, int HN, int lx, int ly, uint32_t node) {
    float h[8];
    stencil_h(a, node, h);
    const int q = (ly + 1) * HW + lx + 1;
    H[q] = make_float2(h[0], h[1]);
    H[HN + q] = make_float2(h[2], h[3]);
    H[2 * HN + q] = make_float2(h[4], h[5]);
    H[3 * HN + q] = make_float2(h[6], h[7]);
}

// the halo nodes of the tile at (x0, y0): j in [0, TY] -> column x0 - 1, rows y0 - 1 ..
// y0 + TY - 1; j in (TY, TX + TY] -> row y0 - 1, columns x0 .. x0 + TX - 1 (periodic; nodes
// past a ragged edge are skipped, no tile node reads them).  They go to the last threads of
// the block, which form no density-ring node, so the work before the tile's barrier evens out.
template <int TX, int TY, int HW>
__device__ __forceinline__ void stencil_halo(const StepArgs& a, float2* H, int HN, int x0, int y0, int nx, int ny,
                                             int tid, int nthreads) {
    for (int j = nthreads - 1 - tid; j < TX + TY + 1; j += nthreads) {
        int lx, ly;
        if (j <= TY) { lx = -1; ly = j - 1; }
        else { lx = j - (TY + 1); ly = -1; }
        int gx = x0 + lx, gy = y0 + ly;
        if (gx < 0) gx += nx;
        if (gy < 0) gy += ny;
        if (gx < nx && gy < ny) stencil_store<HW>(a, H, HN, lx, ly, (uint32_t)gy * (uint32_t)nx + (uint32_t)gx);
    }
}

template <int HW>
__device__ __forceinline__ float2 stencil_xi(const float2* H, int HN, int lx, int ly) {
    const int q = (ly + 1) * HW + lx + 1;
    const float2 a = H[q], b = H[HN + q - 1], c = H[2 * HN + q - HW], d = H[3 * HN + q - HW - 1];
    return make_float2((a.x + b.x) + (c.x + d.x), (a.y + b.y) + (c.y + d.y));
}

struct HalfArgs {
    StepArgs a;
    int ntx, nty;      // tiles along x and y
    int* err;          // device error word (1 = a TMA wait timed out)
};

template <int TX, int TY, int NT, int MODE>
__global__ void __launch_bounds__(NT) step_half_kernel(const __grid_constant__ CUtensorMap tmap, const HalfArgs ta) {
    using TT = HalfTile<TX, TY>;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    __half* smem = reinterpret_cast<__half*>(smem_raw);
    float* R = reinterpret_cast<float*>(smem_raw + 2 * TT::STAGE_BYTES);
    uint64_t* mbar = reinterpret_cast<uint64_t*>(R + TT::RW * TT::RH);
    const StepArgs& a = ta.a;
    const Grid g = a.g;
    const int tid = threadIdx.x;
    const int ntiles = ta.ntx * ta.nty;
    // MODE 3: the noise contributions, kept apart from the stages (filling them into the consumed
    // stage and refilling it after the collision measured slower: two more barriers)
    float2* H = reinterpret_cast<float2*>(smem_raw + TT::H_OFFSET);

    if (tid == 0) {
        mbar_init(smem_u32(&mbar[0]), 1);
        mbar_init(smem_u32(&mbar[1]), 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&tmap)) : "memory");
    }
    __syncthreads();
    grid_wait();
    grid_next();

    // the nine boxes of the tile in column col, row row of the tiling into stage s
    auto issue = [&](int col, int row, int s) {
        const int x0 = col * TX, y0 = row * TY;
        const uint32_t bar = smem_u32(&mbar[s]);
        mbar_expect_tx(bar, TT::TX_BYTES);
        __half* st = smem + s * TT::STAGE;
#pragma unroll
        for (int i = 0; i < Q; ++i)
            tma_load_3d(smem_u32(st + i * TT::PS), &tmap, x0 - TT::XO + g.gx, y0 - 1 - kCYt[i] + GY, i, bar);
    };

    // a tile's column and row, advanced by the grid stride without a division per tile
    const int first = blockIdx.x;
    const int stx = (int)gridDim.x % ta.ntx, sty = (int)gridDim.x / ta.ntx;
    auto advance = [&](int& col, int& row) {
        col += stx;
        row += sty;
        if (col >= ta.ntx) {
            col -= ta.ntx;
            ++row;
        }
    };
    int tcol = first % ta.ntx, trow = first / ta.ntx;
    if (tid == 0) {
        if (first < ntiles) issue(tcol, trow, 0);
        int c1 = tcol, r1 = trow;
        advance(c1, r1);
        if (first + (int)gridDim.x < ntiles) issue(c1, r1, 1);
    }
    int k = 0;
    for (int tile = first; tile < ntiles; tile += gridDim.x, ++k) {
        const int s = k & 1;
        const uint32_t parity = (uint32_t)((k >> 1) & 1);
        // bounded wait for this tile's nine boxes; the decision to give up is collective
        // (this barrier also orders the previous tile's reads of R before this tile's writes)
        const bool ok = mbar_wait_bounded(smem_u32(&mbar[s]), parity);
        if (__syncthreads_or(!ok)) {
            if (tid == 0) {
                atomicExch(ta.err, 1);
                // give the loads still in flight into this CTA's shared memory a bounded
                // chance to land before the CTA exits
                mbar_wait_bounded(smem_u32(&mbar[s]), parity);
                if (tile + (int)gridDim.x < ntiles)
                    mbar_wait_bounded(smem_u32(&mbar[s ^ 1]), (uint32_t)(((k + 1) >> 1) & 1));
            }
            return;
        }
        const __half* S = smem + s * TT::STAGE;
        const int x0 = tcol * TX, y0 = trow * TY;
        advance(tcol, trow);        // now the next tile's

        static_assert((TX * TY) % NT == 0, "tile must be a multiple of the block");
        constexpr int NN = TX * TY / NT;
        // each thread pulls its nodes' nine values once, keeps them in registers across
        // the barrier and writes their density to the tile; the ring is formed separately
        float fr[NN][Q];
#pragma unroll
        for (int it = 0; it < NN; ++it) {
            const int q = tid + it * NT;
            const int ly = q / TX, lx = q - ly * TX;
            load9_g<TT::PS>(S, (ly + 1) * TT::BW + lx + TT::XO, fr[it]);
            R[(ly + 1) * TT::RW + lx + 1] = drho_of_g(fr[it]);
        }
        // real-space correlated noise: every node's contributions, then the halo's
        if (MODE == 3) {
#pragma unroll 1
            for (int it = 0; it < NN; ++it) {
                const int q = tid + it * NT;
                const int ly = q / TX, lx = q - ly * TX;
                const int x = x0 + lx, y = y0 + ly;
                if (x < g.nx && y < g.ny)
                    stencil_store<TT::HW>(a, H, TT::HN, lx, ly, (uint32_t)y * (uint32_t)g.nx + (uint32_t)x);
            }
            stencil_halo<TX, TY, TT::HW>(a, H, TT::HN, x0, y0, g.nx, g.ny, tid, NT);
        }
        // the ring: rows 0 and TY + 1 (TX + 2 each), then columns 0 and TX + 1, on the last
        // threads (the first issues the refill); with MODE 3 on the first (the last form the
        // noise contributions of the halo)
        constexpr int NB = 2 * (TX + 2) + 2 * TY;
        for (int j = MODE == 3 ? tid : NT - 1 - tid; j < NB; j += NT) {
            int rx, ry;
            if (j < TX + 2) { rx = j; ry = 0; }
            else if (j < 2 * (TX + 2)) { rx = j - (TX + 2); ry = TY + 1; }
            else { const int u = j - 2 * (TX + 2); ry = 1 + (u >> 1); rx = (u & 1) ? TX + 1 : 0; }
            float h[Q];
            load9_g<TT::PS>(S, ry * TT::BW + rx + TT::XO - 1, h);
            R[ry * TT::RW + rx] = drho_of_g(h);
        }
        __syncthreads();
        // the collision pass reads no population from stage s: refill it now with the tile
        // two steps ahead
        if (tid == 0 && tile + 2 * (int)gridDim.x < ntiles) {
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            int c2 = tcol, r2 = trow;
            advance(c2, r2);
            issue(c2, r2, s);
        }

        // collide every node of the tile; the nodes of one thread are independent, so
        // their random-number and collision chains interleave
#pragma unroll
        for (int it = 0; it < NN; ++it) {
            const int q = tid + it * NT;
            const int ly = q / TX, lx = q - ly * TX;
            const int x = x0 + lx, y = y0 + ly;
            if (x >= g.nx || y >= g.ny) continue;
            const float* f = fr[it];
            const int rc = (ly + 1) * TT::RW + lx + 1;
            Nbr r;
            r.C = R[rc];
            r.E = R[rc + 1]; r.W = R[rc - 1];
            r.N = R[rc + TT::RW]; r.S = R[rc - TT::RW];
            r.NE = R[rc + TT::RW + 1]; r.NW = R[rc + TT::RW - 1];
            r.SE = R[rc - TT::RW + 1]; r.SW = R[rc - TT::RW - 1];
            const uint32_t node = (uint32_t)y * (uint32_t)g.nx + (uint32_t)x;
            float2 z = make_float2(0.f, 0.f);
            if (MODE == 2) z = a.xi49[(long long)y * g.nx + x];
            if (MODE == 3) z = stencil_xi<TT::HW>(H, TT::HN, lx, ly);
            float o[Q];
            collide_node<MODE, false, true>(a, f, r, node, z, o);
            store9<__half, float, true>(static_cast<__half*>(a.dst), g.plane, g, x, y, o);
        }
    }
}

// --- host side ----------------------------------------------------------------------

template <int TX, int TY, int NT, int MODE>
static cudaError_t launch_cfg(const void* map, HalfArgs ta, cudaStream_t s) {
    using TT = HalfTile<TX, TY>;
    auto kern = step_half_kernel<TX, TY, NT, MODE>;
    constexpr int smem = TT::SMEM_BYTES + (MODE == 3 ? TT::H_BYTES : 0);
    static GridCache cache;
    int grid_max = 0;
    cudaError_t e = resident_grid(kern, NT, smem, cache, &grid_max);
    if (e != cudaSuccess) return e;
    ta.ntx = (ta.a.g.nx + TX - 1) / TX;
    ta.nty = (ta.a.g.ny + TY - 1) / TY;
    const int ntiles = ta.ntx * ta.nty;
    const int grid = ntiles < grid_max ? ntiles : grid_max;
    return launch_chained(kern, grid, NT, smem, s, *static_cast<const CUtensorMap*>(map), ta);
}

// the tile shapes of lb_step_tma.cu
template <int MODE>
static cudaError_t launch_mode(const void* map, const HalfArgs& ta, int tile, cudaStream_t s) {
    switch (tile) {
        case 1: return launch_cfg<32, 32, 256, MODE>(map, ta, s);
        case 2: return launch_cfg<64, 8, 256, MODE>(map, ta, s);
        case 3: return launch_cfg<64, 16, 512, MODE>(map, ta, s);
        case 4: return launch_cfg<32, 16, 128, MODE>(map, ta, s);
        default: return launch_cfg<32, 16, 256, MODE>(map, ta, s);
    }
}

cudaError_t launch_step_half(const StepArgs& a, const void* src_map, int* err, int noise_mode, int tile, cudaStream_t s) {
    HalfArgs ta;
    ta.a = a;
    ta.ntx = ta.nty = 0;
    ta.err = err;
    switch (noise_mode) {
        case 0: return launch_mode<0>(src_map, ta, tile, s);
        case 1: return launch_mode<1>(src_map, ta, tile, s);
        case 3: return launch_mode<3>(src_map, ta, tile, s);
        case 4: return launch_mode<4>(src_map, ta, tile, s);
        default: return launch_mode<2>(src_map, ta, tile, s);
    }
}

}  // namespace lbf

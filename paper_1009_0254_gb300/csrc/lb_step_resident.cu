// lb_step_resident.cu -- many steps of a small FP32 D2Q9 lattice in one launch, its populations resident in
// the shared memory of a cluster of CTAs.
//
// A step of a lattice of up to 128^2 nodes is all latency: launched one by one it takes 3.8 us (launch,
// TMA load from L2, density, collision, store, with at most 32 CTAs at work), of which the arithmetic is
// half a microsecond.  Here 16 CTAs of one cluster each keep a band of rows, with two rows of each
// neighbour's, for the whole launch: a step is a density pass, a barrier of the CTA, the collision
// (collide_pair, one pair of nodes a thread), stores into the other buffer and, for the two outermost
// rows, into the neighbours' (distributed shared memory), and a barrier of the cluster.  Global memory is
// read once and written once per launch.  Arithmetic and order are those of the TMA-staged kernel, so the
// trajectory does not depend on which of the two runs a step.  Uncorrelated noise, us a step in calls of
// 1,000 steps, by launches and here: 32^2 3.64, 1.01; 64^2 3.84, 1.33; 64 x 100 3.73, 1.57; 128^2 3.69,
// 2.68.  What bounds it: two barriers a step and the collision of one to eight rows by one CTA (128^2: 16
// of the 152 SMs).  A launch with its load and store costs 5.5 us.
#include <cooperative_groups.h>

#include <atomic>

#include "lb_limits.cuh"
#include "lb_pair.cuh"

namespace lbf {

constexpr int RES_CTAS = 16;          // CTAs of the cluster
constexpr int RES_MAX_NX = 128;       // one pair a thread: at most 8 rows of 64 pairs and two ring rows

// coefficients, key and the time of the step, as collide_pair takes them
struct ResCoef : PairCoef {
    RoundKeys rk;
    uint32_t t_lo, t_hi;
};

struct ResArgs {
    ResCoef c;
    PairLocal loc;
    Grid g;
    const float* src;
    float* dst;
    long long t;
    int steps;
    int pw, ps;        // elements per stored row (nx + 8) and per plane
    int nown;          // threads that may own a pair; the ring's follow
};

// bytes of the two population buffers; the density tile follows
__host__ __device__ inline int res_buf_bytes(const ResArgs& a) { return 2 * Q * a.ps * (int)sizeof(float); }

template <int MODE, bool POLY>
__global__ void __launch_bounds__(RES_MAX_NX / 2 * 10) step_resident_kernel(const __grid_constant__ ResArgs a) {
    namespace cg = cooperative_groups;
    extern __shared__ __align__(16) unsigned char res_smem[];
    cg::cluster_group cluster = cg::this_cluster();
    const int rank = (int)cluster.block_rank();
    const Grid g = a.g;
    const int nx = g.nx, ny = g.ny, hx = nx >> 1, pw = a.pw, ps = a.ps;
    const int y0 = rank * ny / RES_CTAS, rows = (rank + 1) * ny / RES_CTAS - y0;
    const int below = (rank + RES_CTAS - 1) % RES_CTAS, above = (rank + 1) % RES_CTAS;
    const int rows_below = (below + 1) * ny / RES_CTAS - below * ny / RES_CTAS;
    float* buf = reinterpret_cast<float*>(res_smem);           // [2][Q][rows + 4][pw], node (x, r) at (r + 2) pw + x + 4
    float* R = reinterpret_cast<float*>(res_smem + res_buf_bytes(a));   // node (x, r) at (r + 1)(nx + 4) + x + 2
    const int tid = threadIdx.x, rw = nx + 4;

    // the band and its halo from the stored planes (columns -2 .. nx + 1, rows -2 .. rows + 1)
    {
        const float* src = a.src;
        const int w = hx + 2, n = w * (rows + 4);
        for (int e = tid; e < n; e += blockDim.x) {
            const int r = e / w, x = 2 * (e - r * w) - 2;
            const long long o = g.at(x, y0 + r - 2);
#pragma unroll
            for (int i = 0; i < Q; ++i) {
                float* d = buf + i * ps + r * pw + x + 4;
                d[0] = src[i * g.plane + o];
                d[1] = src[i * g.plane + o + 1];
            }
        }
    }
    // this thread's pair: one of the band's, or of the ring rows -1 and `rows`
    int r, p;
    bool own = false, ring = false;
    if (tid < a.nown) {
        r = tid / hx;
        p = tid - r * hx;
        own = r < rows;
    } else {
        const int q = tid - a.nown;
        ring = q < nx;
        r = q < hx ? -1 : rows;
        p = q < hx ? q : q - hx;
    }
    const int x = 2 * p, y = y0 + r;
    const int at = (r + 2) * pw + x + 4;
    float* pr = R + (r + 1) * rw + x + 2;
    const uint32_t node = (uint32_t)y * (uint32_t)nx + (uint32_t)x;
    // offsets of the pair in the halo rows of the neighbours that hold a copy of it (rows >= 2)
    const bool to_below = own && r < 2, to_above = own && r >= rows - 2;
    float* const nb_below = cluster.map_shared_rank(buf, below);
    float* const nb_above = cluster.map_shared_rank(buf, above);
    const int at_below = (rows_below + r + 2) * pw + x + 4, at_above = (r - rows + 2) * pw + x + 4;
    const int wrap = x < 2 ? nx : (x >= nx - 2 ? -nx : 0);
    cluster.sync();        // every CTA runs and has loaded its band

    ResCoef c = a.c;
    for (int k = 0; k < a.steps; ++k) {
        const float* S = buf + (k & 1) * Q * ps;
        const int to = ((k & 1) ^ 1) * Q * ps;
        F2 f[Q];
        if (own || ring) {
            constexpr int cx[Q] = {0, 1, 0, -1, 0, 1, -1, -1, 1}, cy[Q] = {0, 0, 1, 0, -1, 1, 1, -1, -1};
#pragma unroll
            for (int i = 0; i < Q; ++i) {
                const float* s = S + i * ps + at - cy[i] * pw - cx[i];
                f[i] = make_float2(s[0], s[1]);
            }
            const F2 rho = drho_pair(f);
            *reinterpret_cast<F2*>(pr) = rho;
            if (x == 0) pr[nx] = rho.x;                    // column nx
            if (x == nx - 2) pr[1 - nx] = rho.y;           // column -1
        }
        __syncthreads();
        if (own) {
            const unsigned long long t = (unsigned long long)(a.t + k);
            c.t_lo = (uint32_t)t;
            c.t_hi = (uint32_t)(t >> 32);
            const RhoRow m = rho_row(pr - rw), d = rho_row(pr), n = rho_row(pr + rw);
            const F2 lap6 = fma2(d.C, bc(-20.0f), fma2(add2(d.s, add2(n.C, m.C)), bc(4.0f), add2(n.s, m.s)));
            const F2 gx12 = fma2(d.d, bc(4.0f), add2(n.d, m.d));
            const F2 gy12 = fma2(sub2(n.C, m.C), bc(4.0f), sub2(n.s, m.s));
            F2 o[Q];
            collide_pair<MODE, POLY>(c, &a.loc, f, d.C, lap6, gx12, gy12, node, bc(0.f), bc(0.f), o);
            if (k + 1 < a.steps) {
#pragma unroll
                for (int i = 0; i < Q; ++i) {
                    float* q = buf + to + i * ps + at;
                    put_pair(q, o[i]);
                    if (wrap) put_pair(q + wrap, o[i]);
                }
                if (to_below) {
#pragma unroll
                    for (int i = 0; i < Q; ++i) {
                        float* q = nb_below + to + i * ps + at_below;
                        put_pair(q, o[i]);
                        if (wrap) put_pair(q + wrap, o[i]);
                    }
                }
                if (to_above) {
#pragma unroll
                    for (int i = 0; i < Q; ++i) {
                        float* q = nb_above + to + i * ps + at_above;
                        put_pair(q, o[i]);
                        if (wrap) put_pair(q + wrap, o[i]);
                    }
                }
            } else {
                store_pair(a.dst, g.plane, g, x, y, o);
                ghost_pair(a.dst, g.plane, g, x, y, o);
            }
        }
        // every CTA's stores into this one's next buffer are done and visible, and this one's reads of
        // the last buffer are over; no CTA leaves while another may still write to it
        cluster.sync();
    }
}

// --- host side ------------------------------------------------------------------------------------

// Which lattices: even nx (pairs) of 32 to 128 columns, at least two rows a CTA (a halo row comes from
// the nearest neighbour) and at most eight.
bool resident_fits(const Grid& g) {
    return g.nx % 2 == 0 && g.nx >= 32 && g.nx <= RES_MAX_NX && g.ny >= 2 * RES_CTAS && g.ny <= 8 * RES_CTAS;
}

template <int MODE, bool POLY>
static cudaError_t launch_res(const ResArgs& a, int threads, size_t smem, cudaStream_t s) {
    constexpr auto kern = step_resident_kernel<MODE, POLY>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e == cudaSuccess) e = all_shared_memory<kern>();
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t c = {};
    c.gridDim = dim3(RES_CTAS);
    c.blockDim = dim3(threads);
    c.dynamicSmemBytes = smem;
    c.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = RES_CTAS;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    c.attrs = at;
    c.numAttrs = 1;
    return cudaLaunchKernelEx(&c, kern, a);
}

// Whether this device can hold such a cluster at its largest (a launch that it cannot hold is refused);
// asked once per device.
bool resident_available() {
    static std::atomic<int> known[MAX_DEVICES];
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= MAX_DEVICES) return false;
    int k = known[dev].load(std::memory_order_acquire);
    if (k == 0) {
        constexpr auto kern = step_resident_kernel<1, false>;
        const int smem = 2 * Q * (RES_MAX_NX + 8) * 12 * 4 + 10 * (RES_MAX_NX + 4) * 4;
        cudaLaunchConfig_t c = {};
        c.gridDim = dim3(RES_CTAS);
        c.blockDim = dim3(RES_MAX_NX / 2 * 10);
        c.dynamicSmemBytes = smem;
        cudaLaunchAttribute at[1];
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = RES_CTAS;
        at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
        c.attrs = at;
        c.numAttrs = 1;
        int n = 0;
        const bool ok = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess &&
                        all_shared_memory<kern>() == cudaSuccess &&
                        cudaOccupancyMaxActiveClusters(&n, kern, &c) == cudaSuccess && n > 0;
        if (!ok) cudaGetLastError();
        k = ok ? 1 : 2;
        known[dev].store(k, std::memory_order_release);
    }
    return k == 1;
}

// nsteps steps from src (time t) into dst; noise modes 0, 1 and 4
cudaError_t launch_step_resident(const StepArgs& a, const StepArgsD& d, long long t, int nsteps, int noise_mode, bool poly,
                                 cudaStream_t s) {
    ResArgs r;
    const double L[4] = {d.L44, d.L49, d.L94, d.L99}, s3[3] = {d.s5, d.s6, d.s7};
    pair_coef(d.rho0, d.cs2m, d.kappa, d.lb, d.ls, d.lq, d.le, L, s3, &r.c);
    pair_local(d.e2, d.e3, d.e4, d.cq, d.lu, &r.loc);
    r.c.rk = a.rk;
    r.c.t_lo = r.c.t_hi = 0;
    r.g = a.g;
    r.src = static_cast<const float*>(a.src);
    r.dst = static_cast<float*>(a.dst);
    r.t = t;
    r.steps = nsteps;
    const int rows = (a.g.ny + RES_CTAS - 1) / RES_CTAS;
    r.pw = a.g.nx + 8;
    r.ps = r.pw * (rows + 4);
    r.nown = rows * a.g.nx / 2;
    const int threads = (r.nown + a.g.nx + 31) / 32 * 32;
    const size_t smem = res_buf_bytes(r) + (size_t)(rows + 2) * (a.g.nx + 4) * sizeof(float);
    switch (noise_mode) {
        case 0: return poly ? launch_res<0, true>(r, threads, smem, s) : launch_res<0, false>(r, threads, smem, s);
        case 1: return poly ? launch_res<1, true>(r, threads, smem, s) : launch_res<1, false>(r, threads, smem, s);
        default: return poly ? launch_res<4, true>(r, threads, smem, s) : launch_res<4, false>(r, threads, smem, s);
    }
}

}  // namespace lbf

// lb_ens.cuh -- device pieces shared by the engines that step many independent lattices
// in one launch (batched ensembles, the request server): the per-lattice record and its copy
// in shared memory that the collision of a staged tile reads.
#pragma once

#include "lb_internal.cuh"
#include "lb_pair.cuh"
#include "lb_tma.cuh"

#include <type_traits>

namespace lbf {

// Per-replica record (device).
struct RepRec : PairCoef, PairStencil {
    float a44, b44, a49, b49, a99, b99;   // Xi(k) of the (4,9) block = a + b s(k) (correlated noise)
    int mode;                 // 0 no noise, 1 uncorrelated, 2 correlated (k-space), 3 correlated (real space)
    uint32_t k0, k1;          // Philox key = the replica's seed
    long long toff;           // time = K + toff
};

// What the collision of one tile of one replica reads, in shared memory (the engines step the
// linearised equation of state).
struct __align__(16) TileArgs : PairCoef {
    RoundKeys4 rk;            // the lattice's Philox round keys
    uint32_t t_lo, t_hi;
    int mode;                 // RepRec::mode
};

// The same with the real-space correlated-noise factors: the record of the engines' step
// kernel variant that steps such lattices (the lean variant keeps the smaller record).
struct TileArgsRS : TileArgs, PairStencil {};

template <bool RS>
using TileArgsOf = typename std::conditional<RS, TileArgsRS, TileArgs>::type;

// Copies a lattice's record, for its time t, to the tile's shared copy a: one word a thread on the
// first warps, so that it costs one load latency between the tile's barriers (by a single thread,
// forty loads and the ten key additions sat on the tile's critical path).
template <bool RS>
__device__ __forceinline__ void load_tile_args(const RepRec* rp, long long t, TileArgsOf<RS>* a) {
    constexpr int NC = sizeof(PairCoef) / 4, NS = sizeof(PairStencil) / 4;
    static_assert(NC + 11 <= 32 && NS <= 32, "one word a lane");
    const int tid = threadIdx.x;
    if (tid < NC) {
        reinterpret_cast<float*>(static_cast<PairCoef*>(a))[tid] =
            __ldg(reinterpret_cast<const float*>(static_cast<const PairCoef*>(rp)) + tid);
    } else if (tid < NC + 10) {
        const uint32_t r = (uint32_t)(tid - NC);
        uint32_t* k = reinterpret_cast<uint32_t*>(&a->rk) + 2 * r;
        k[0] = __ldg(&rp->k0) + r * 0x9E3779B9u;
        k[1] = __ldg(&rp->k1) + r * 0xBB67AE85u;
    } else if (tid == NC + 10) {
        a->t_lo = (uint32_t)((unsigned long long)t & 0xffffffffu);
        a->t_hi = (uint32_t)((unsigned long long)t >> 32);
        a->mode = __ldg(&rp->mode);
    }
    if constexpr (RS) {
        if (tid >= 32 && tid < 32 + NS)
            reinterpret_cast<float*>(static_cast<PairStencil*>(a))[tid - 32] =
                __ldg(reinterpret_cast<const float*>(static_cast<const PairStencil*>(rp)) + tid - 32);
    }
}

// host: fills the parameter fields of a record (defined in lb_batch.cu)
void fill_rep_record(double rho0, double cs2, double kT, double kappa, double tau_s, double tau_b,
                     double tau_ghost, int noise_mode, RepRec* rec);

}  // namespace lbf

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

// Copies a lattice's record to the tile's shared copy a, for its time K + toff: one word a thread on the first
// warps, every load issued before any is used, so that the copy costs one load latency between the tile's
// barriers: with a branch for each kind of word, each waiting for its own load, and the time formed by all
// threads, eight replicas of 32^2 to 256^2 took 10.2 us a step (uncorrelated noise, graph replay) and 512 of
// them 174; this way 10.0 and 169.
template <bool RS>
__device__ __forceinline__ void load_tile_args(const RepRec* rp, long long K, TileArgsOf<RS>* a) {
    constexpr int NC = sizeof(PairCoef) / 4, NS = sizeof(PairStencil) / 4, NT = NC + 20, NM = NT + 2;
    static_assert(NM + 1 + NS <= 64, "the words must fit the first two warps");
    const int tid = threadIdx.x;
    if (tid > NM + (RS ? NS : 0)) return;
    // the coefficients, the round keys (k0, k1) + r (W0, W1), the time, the mode and the noise factors
    const uint32_t* src = reinterpret_cast<const uint32_t*>(static_cast<const PairCoef*>(rp)) + tid;
    uint32_t* dst = reinterpret_cast<uint32_t*>(static_cast<PairCoef*>(a)) + tid;
    uint32_t add = 0;
    if (tid >= NC) {
        const uint32_t k = (uint32_t)(tid - NC);
        src = (k & 1u) ? &rp->k1 : &rp->k0;
        dst = reinterpret_cast<uint32_t*>(&a->rk) + k;
        add = (k >> 1) * ((k & 1u) ? 0xBB67AE85u : 0x9E3779B9u);
    }
    if (tid >= NT) dst = tid == NT ? &a->t_lo : &a->t_hi;
    if (tid == NM) {
        src = reinterpret_cast<const uint32_t*>(&rp->mode);
        dst = reinterpret_cast<uint32_t*>(&a->mode);
    }
    if (tid >= NM) add = 0;
    if constexpr (RS) {
        if (tid > NM) {
            src = reinterpret_cast<const uint32_t*>(static_cast<const PairStencil*>(rp)) + (tid - NM - 1);
            dst = reinterpret_cast<uint32_t*>(static_cast<PairStencil*>(a)) + (tid - NM - 1);
        }
    }
    const long long toff = __ldg(&rp->toff);
    uint32_t v = __ldg(src) + add;
    const unsigned long long t = (unsigned long long)(K + toff);
    if (tid == NT) v = (uint32_t)t;
    if (tid == NT + 1) v = (uint32_t)(t >> 32);
    *dst = v;
}

// host: fills the parameter fields of a record (defined in lb_batch.cu)
void fill_rep_record(double rho0, double cs2, double kT, double kappa, double tau_s, double tau_b,
                     double tau_ghost, int noise_mode, RepRec* rec);

}  // namespace lbf

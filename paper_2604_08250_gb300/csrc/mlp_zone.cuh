// mlp_zone.cuh -- the interaction zone of an MLP trial, the shared-memory
// layouts of the network kernels and their evaluators, shared by the sweeps
// that evaluate every row (sweep_mlp.cu) and by the tabulated ones
// (mlp_table.cu).
#pragma once

#include <type_traits>

#include "mlp_common.cuh"
#include "mlp_tc.cuh"
#include "mlpnet_tc.cuh"
#include "sweep_common.cuh"

namespace smc {

constexpr int kOmega = 40;       // sites of a trial's interaction zone
constexpr int kMlpChunk = 64;    // most trials of a mini-step evaluated together (40 rows each)
constexpr int kTraceTB = 3;      // trials per trace step (120 rows: one tile)
constexpr int kTcMaxCtasPerSm = 512 / (2 * kTcCols);  // for the 2-warpgroup kernels
constexpr int kTinfo = 16;       // ints of per-trial information

// Omega of a trial for each (trial sublattice, partner direction): rel = 0
// for a site of the trial sublattice, 1 for the partner's; (dxo, dy, dz) its
// cell offset from the trial site's cell.  Entry 0 is a, entry 1 is b.
struct OmegaEntry {
    signed char rel, dy, dz, dxo;
    signed char ma, mb;  // shell (1-3) in which the site sees a / b, 0 if none
    signed char pad[2];
};
struct MlpGeo {
    OmegaEntry om[2][8][kOmega];
};

// Shared memory of the MLP kernels: weights, the warpgroups' tiles, then
// kernel-specific parts from END on.
template <int NWG>
struct MlpSmem {
    static constexpr uint32_t W1 = 0;
    static constexpr uint32_t W2 = W1 + kTcW1;
    static constexpr uint32_t X = W2 + kTcW2;        // [NWG] tiles
    static constexpr uint32_t H = X + NWG * kTcX;    // [NWG] tiles
    static constexpr uint32_t B1 = H + NWG * kTcH;
    static constexpr uint32_t B2 = B1 + 256;
    static constexpr uint32_t W3 = B2 + 256;
    static constexpr uint32_t B3 = W3 + 256;
    static constexpr uint32_t MBAR = B3 + 16;        // [NWG][2]
    static constexpr uint32_t TSLOT = MBAR + 16 * NWG;
    static constexpr uint32_t CTL = TSLOT + 4;       // CTA-wide flag
    static constexpr uint32_t RED = (CTL + 4 + 15) / 16 * 16;  // 4 doubles / long longs for reductions
    static constexpr uint32_t TINFO = RED + 64;      // int [kMlpChunk][kTinfo]
    static constexpr uint32_t ACT = TINFO + kMlpChunk * kTinfo * 4;  // int [kMlpChunk]: trials with A != B
    static constexpr uint32_t D = ACT + kMlpChunk * 4;  // pair table (kDEntries floats)
    static constexpr uint32_t GEO = D + kDEntries * 4;
    static constexpr uint32_t END = (uint32_t)((GEO + sizeof(MlpGeo) + 127) / 128 * 128);
    static_assert(X % 128 == 0 && H % 128 == 0 && W2 % 128 == 0, "tile alignment");
    static_assert(MBAR % 8 == 0 && RED % 8 == 0, "alignment");
};
constexpr int kSweepWG = 4;  // warpgroups of the sweep kernel (64-wide network)
constexpr int kEvalWG = 2;   // warpgroups of the trace kernel
// Warpgroups of the kernels that stream rows through the network (site
// energies; the MLP's table): one CTA per SM with all 512 tensor-memory columns.
// With two warpgroups per CTA the driver kept one CTA per SM (the occupancy
// query gives 1, eight warps), and the special-function pipe idled half the
// time: 50.6 ms for the 9.46e8 rows of the five-species table (MLP), 72 ms
// (MLPNet).
constexpr int kStreamWG = 4;

// Shared memory of the MLPNet kernels (96-wide, three ReLU layers): the same
// kernel-specific parts as MlpSmem from CTL on, without the pair table.
template <int NWG>
struct NetSmem {
    static constexpr uint32_t W0 = 0;
    static constexpr uint32_t W1 = W0 + kNetW0;
    static constexpr uint32_t W2 = W1 + kNetW12;
    static constexpr uint32_t X = W2 + kNetW12;      // [NWG] tiles
    static constexpr uint32_t XSIZE = NWG <= 4 ? kNetX : kNetXc;
    static constexpr uint32_t H = X + NWG * XSIZE;   // [NWG] tiles
    static constexpr uint32_t W3 = H + NWG * kNetHt;
    static constexpr uint32_t B3 = W3 + kNetHid * 4;
    static constexpr uint32_t MBAR = B3 + 16;        // [NWG][2]
    static constexpr uint32_t TSLOT = MBAR + 16 * NWG;
    static constexpr uint32_t CTL = TSLOT + 4;
    static constexpr uint32_t RED = (CTL + 4 + 15) / 16 * 16;
    static constexpr uint32_t TINFO = RED + 64;      // (the table kernel's shared memory ends here)
    static constexpr uint32_t ACT = TINFO + kMlpChunk * kTinfo * 4;
    static constexpr uint32_t GEO = ACT + kMlpChunk * 4;
    static constexpr uint32_t END = (uint32_t)((GEO + sizeof(MlpGeo) + 127) / 128 * 128);
    static_assert(X % 128 == 0 && XSIZE % 128 == 0 && H % 128 == 0 && W1 % 128 == 0 && W2 % 128 == 0, "tile alignment");
    static_assert(MBAR % 8 == 0 && RED % 8 == 0, "alignment");
};

// The two site-energy networks the MLP kernels run: evaluator, layouts and
// warpgroups of the sweep.
struct NetSilu64 {  // MLP of mlp_tc.cuh: 20 -> 64 -> 64 -> 1, SiLU
    using Eval = TcEval;
    using Block = MlpBlock;
    template <int NWG>
    using Smem = MlpSmem<NWG>;
    static constexpr int kSweepNWG = kSweepWG;
    static constexpr int kFillNWG = kStreamWG;
    template <int NWG>
    static __device__ TcLayout layout(uint32_t wg)
    {
        using M = MlpSmem<NWG>;
        return TcLayout{M::X + wg * kTcX, M::H + wg * kTcH, M::W1, M::W2, M::B1, M::B2, M::W3, M::B3,
                        M::MBAR + 16 * wg, M::TSLOT};
    }
};
struct NetRelu96 {  // MLPNet of mlpnet_tc.cuh: 20 -> 96 -> 96 -> 96 -> 1, ReLU
    using Eval = NetEval;
    using Block = NetBlock;
    template <int NWG>
    using Smem = NetSmem<NWG>;
    static constexpr int kSweepNWG = 2;  // the 28 KB hidden tiles of four would not fit
    static constexpr int kFillNWG = 5;   // all tensor memory: 96 columns each
    template <int NWG>
    static __device__ NetLayout layout(uint32_t wg)
    {
        using M = NetSmem<NWG>;
        return NetLayout{M::X + wg * M::XSIZE, M::H + wg * kNetHt, M::W0, M::W1, M::W2, M::W3, M::B3, M::MBAR + 16 * wg,
                         M::TSLOT, NWG <= 4 ? 512u : 384u};
    }
};

// Site-energy models of the tensor-core sweep.
constexpr int kModeMlp = 0, kModeMlpPair = 1;

// The evaluator of this thread's warpgroup.
template <class Net, int NWG>
__device__ __forceinline__ typename Net::Eval mlp_evaluator(long long timeout_ns, int *status, int *abort_flag)
{
    const uint32_t wg = threadIdx.x >> 7;
    typename Net::Eval E;
    E.L = Net::template layout<NWG>(wg);
    E.timeout_ns = timeout_ns;
    E.status = status;
    E.abort_flag = abort_flag;
    E.tmem = 0;
    E.phase1 = E.phase2 = 0;
    E.bar = 1 + wg;
    return E;
}

// Pair part of dE (pair + MLP models) from the packed post-swap neighbour
// histograms of a (species B now) and b (species A now), 3 shells each; the
// swapped partner is removed from shell 1.  Dt: D[m][A][B][q].
__device__ __forceinline__ float pair_part(const float *Dt, int nshells, int S, const int *ha, const int *hb, int A,
                                           int B)
{
    float dp = 0.f;
    for (int m = 0; m < nshells; ++m) {
        const float *D = Dt + ((m * kMaxSpecies + A) * kMaxSpecies + B) * kMaxSpecies;
        for (int q = 0; q < S; ++q) {
            float ca = (float)(((uint32_t)ha[m] >> (4 * q)) & 15u);
            float cb = (float)(((uint32_t)hb[m] >> (4 * q)) & 15u);
            if (m == 0) {
                ca -= (q == A) ? 1.f : 0.f;
                cb -= (q == B) ? 1.f : 0.f;
            }
            dp = fmaf(ca - cb, D[q], dp);
        }
    }
    return dp;
}

// Copies the model (weights, pair table, geometry) and sets up the evaluators.
template <class Net, int NWG>
__device__ void mlp_cta_setup(typename Net::Eval &E, const void *W, const float *Dsrc, const MlpGeo *geo)
{
    using M = typename Net::template Smem<NWG>;
    tc_load_weights((const typename Net::Block *)W, E.L);
    const int tid = threadIdx.x, n = blockDim.x;
    if constexpr (std::is_same<Net, NetSilu64>::value) {
        if (Dsrc)
            for (int i = tid; i < kDEntries; i += n) ((float *)(g_smem + M::D))[i] = Dsrc[i];
    }
    if (geo)
        for (int i = tid; i < (int)(sizeof(MlpGeo) / 4); i += n) ((int *)(g_smem + M::GEO))[i] = ((const int *)geo)[i];
    tc_setup(E, NWG);
}

// Host pieces of sweep_mlp.cu: the zone table (false on a geometry
// inconsistency), the network's weight block copied to dst (device), and the
// pair table D of a pair + MLP model.
bool build_mlp_geo(MlpGeo &G);
smc_status mlp_copy_weights(const smc_model *m, void *dst, cudaStream_t stream);
// Sweeps with f tabulated over all feature vectors (mlp_table.cu), where that
// is the faster route.  *taken: kMlpEvaluate, the caller runs the evaluating
// sweep (also when the table finds no room); kMlpTabulate, the call is done;
// kMlpEither, the device decides by the lattice: the tabulated sweep runs if
// **route is not 0, and the caller enqueues the evaluating one to run if it is.
// D: pair table (host).  eval_passes: columns that a CTA of the evaluating
// sweep takes in turn.  The workspace grows to `least` bytes at least: those of
// the evaluating sweep, which shares it.
enum MlpTaken { kMlpEvaluate, kMlpTabulate, kMlpEither };
smc_status launch_mlp_table_sweep(const smc_lattice *lat, const smc_model *m, int8_t *occ, uint64_t seed,
                                  uint32_t replica, uint64_t sweep0, int nsweeps, const double *kT, double *e_acc,
                                  int64_t *n_acc, const float *D, size_t least, int eval_passes, MlpTaken *taken,
                                  const int **route, cudaStream_t stream);
constexpr size_t kWeightBytes = sizeof(MlpBlock) > sizeof(NetBlock) ? sizeof(MlpBlock) : sizeof(NetBlock);

}  // namespace smc

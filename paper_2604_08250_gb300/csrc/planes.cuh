// planes.cuh -- neighbour counts from species bit planes (planes.cu).
#pragma once

#include "smc_common.cuh"

namespace smc {

enum PlaneLattice { kPlanesBcc = 0, kPlanesFcc = 1 };

// The bit planes of an occupancy: uint4 (planes 0-2) per 32 cells of a row,
// rows in (sublattice, z, y) order.
struct Planes {
    const uint4 *words;
    int nx, ny, nz, num_sms;
    PlaneLattice lat;
};

// Sites from which on the planes pay for their own launch: below, the
// byte-wise kernels of the callers finish in the time of one launch more.
constexpr long long kPlanesMinSites = 1 << 16;

// Builds the planes on the stream.  False, with *st = SMC_OK, when their
// buffer cannot be had (captured stream, no memory): the caller has a kernel
// without planes.
bool planes_build(PlaneLattice lat, int nx, int ny, int nz, const int8_t *occ, int num_sms, Planes &P, smc_status *st,
                  cudaStream_t stream);
// counts[m][p][q] += ordered pair counts of shells 1..nsh, species < S.
smc_status planes_pairs(const Planes &P, int nsh, int S, unsigned long long *counts, cudaStream_t stream);
// Own-species counts of every site into cache (1 byte per site for 1-2
// shells, 2 for 3: bit fields at 0, 4, 7; rows of a multiple of four cells,
// 4-byte aligned) and their squares' sums per shell and species into
// quad[m][8] (+=); either may be NULL.
smc_status planes_own(const Planes &P, int nsh, void *cache, unsigned long long *quad, cudaStream_t stream);

// nx % 32 == 0, occ 16-byte aligned (observables.cu).
void launch_planes_aligned(const int8_t *occ, long long nwords, uint4 *planes, int num_sms, cudaStream_t stream);
void *planes_buffer(int which, size_t bytes, smc_status *st, cudaStream_t stream);

}  // namespace smc

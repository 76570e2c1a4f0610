// row_group.cuh -- one launch per group of four mini-steps for the one-thread-
// per-trial sweeps (FCC pair models, qSRO models on both lattices).
//
// The four mini-steps dx = 0..3 of one (sublattice, dz, dy) are consecutive,
// and the trials of one row of link cells (a column: fixed link-cell y, z)
// read and write within 3 half units of the trial row along y and z, so with
// columns 8 half units apart no two columns of a group touch the same row.
// A block takes C columns: it copies the rows they touch into shared memory
// (with four cells of periodic x-halo on each side, so that a neighbour is one
// byte at a fixed offset from the trial site whatever the box face), runs
// dx = 0..3 with a block barrier in between, and writes the changed rows
// back.  Against one launch per mini-step with neighbours read from L2 this
// saves three of four launches and reads each row once for four mini-steps.
// Rows start a multiple of 128 bytes apart in the pair kernel, so that the rows
// that different lanes pick by their partner direction share no bank beyond
// the cell offset (256^3 FCC cells, two shells, us per group: 35.1, with 64
// 34.8, with 32 36.2; three shells 65.5, 65.5, 67.6), and a multiple of 64 in
// the qSRO kernels, which keep twice the bytes per column (90 us, 101 with 32,
// 104 with 128, which leaves room for fewer columns).
#pragma once

#include <algorithm>

#include "sweep_common.cuh"

namespace smc {

constexpr int kRgRows = 49;     // most rows of a column: half-unit offsets -3..3 along y and z
constexpr int kRgBody = 16;     // cells before cell 0 in a row
constexpr int kRgThreads = 256;
constexpr int kRgRowBytes = 52 * 4;  // row numbers of a column in shared memory

// Rows of a column, relative to the trial row: sublattice, cell offsets along
// y and z; the first nwr of them hold the sites that a swap changes.
struct RowSet {
    int n, nwr;
    signed char sub[kRgRows], dy[kRgRows], dz[kRgRows];
};

// Rows (A, B) of 8 words in shared memory, kRgDA A + kRgDB B words from the
// start of their shell.  The lanes of a warp read words of unrelated rows; these
// strides spread the S^3 words in use over the 32 banks: 2.8 accesses for a
// warp's 32 random words of five species, 4.0 with rows of 8 words one after the
// other, where a bank belongs to one species (eight species: 3.3 either way).
// Legs of two sweeps, two shells, five species: 256^3 FCC cells 5.14 -> 4.77 ms,
// 128^3 1.64 -> 1.38 ms; three shells, 160 x 128 x 128 2.98 -> 2.71 ms; eight
// species unchanged.
constexpr int kRgDA = 83, kRgDB = 9, kRgDShell = 652;
static_assert(7 * kRgDA + 7 * kRgDB + 8 <= kRgDShell && kRgDShell % 4 == 0, "room for a shell's rows");
__host__ __device__ constexpr int rg_d_at(int i)  // word i of the tables [shell][A][B][8]
{
    return (i >> 9) * kRgDShell + ((i >> 6) & 7) * kRgDA + ((i >> 3) & 7) * kRgDB + (i & 7);
}

// What staging needs to know about the box and the launch.
struct RowGroup {
    int nx, ny, nz, NLx, NLy, ncol;
    int C, tpc;               // columns per block, threads per column (a multiple of 32)
    int pitch, pitchq;        // bytes between occupancy rows and between count rows (qSRO)
    int unit, unitq;          // bytes per copy of an occupancy row (16, 4 or 1, by alignment) and of a count row
    uint32_t inv, invq;       // ceil(2^32 / copies per row)
    int dy, dz, sub, dx0, dx1;
    RowSet rows;
};


// Row numbers ((sublattice, z, y) order) of a column's rows, by its team, into
// rown; a barrier follows.
__device__ __forceinline__ void rg_rows(const RowGroup &G, int *rown, int y0, int z0, int tt)
{
    for (int r = tt; r < G.rows.n; r += G.tpc) {
        const int y = wrapc(y0 + G.rows.dy[r], G.ny), z = wrapc(z0 + G.rows.dz[r], G.nz);
        rown[r] = (G.rows.sub[r] * G.nz + z) * G.ny + y;
    }
}

template <int N>
__device__ __forceinline__ void rg_copy_async(uint32_t dst, const void *src)
{
    if (N == 16)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
    else
        asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(dst), "l"(src) : "memory");
}

// Starts the copies of a column's rows (ES-byte cells at src) to shared memory
// offset base, by the tpc threads of its team (thread tt).  unit: 16, 4 or 1.
template <int ES>
__device__ __forceinline__ void rg_stage(const RowGroup &G, const unsigned char *src, uint32_t base, int pitch,
                                         int unit, uint32_t inv, const int *rown, int tt)
{
    const uint32_t s0 = (uint32_t)__cvta_generic_to_shared(g_smem) + base;
    const int rowb = G.nx * ES;
    if (unit == 1) {
        for (int j = tt; j < G.rows.n * rowb; j += G.tpc) {
            const int r = j / rowb, q = j - r * rowb;
            const unsigned char v = src[(size_t)rown[r] * rowb + q];
            unsigned char *row = g_smem + base + r * pitch + kRgBody * ES;
            row[q] = v;
            if (q < 4 * ES) row[rowb + q] = v;
            if (q >= rowb - 4 * ES) row[q - rowb] = v;
        }
        return;
    }
    const int per = rowb / unit, n = G.rows.n * per;
    for (int j = tt; j < n; j += G.tpc) {
        const int r = (int)__umulhi((uint32_t)j, inv), q = j - r * per;
        const unsigned char *p = src + (size_t)rown[r] * rowb + q * unit;
        const uint32_t d = s0 + r * pitch + kRgBody * ES + q * unit;
        if (unit == 16)
            rg_copy_async<16>(d, p);
        else
            rg_copy_async<4>(d, p);
    }
    for (int j = tt; j < G.rows.n * 2 * ES; j += G.tpc) {  // halo words: ES on each side
        const int r = j / (2 * ES), h = j % (2 * ES);
        const unsigned char *p = src + (size_t)rown[r] * rowb + (h < ES ? 4 * h : rowb - 4 * ES + 4 * (h - ES));
        rg_copy_async<4>(s0 + r * pitch + kRgBody * ES + (h < ES ? rowb + 4 * h : 4 * (h - ES) - 4 * ES), p);
    }
}

// Writes the first nrow rows of a column back.
template <int ES>
__device__ __forceinline__ void rg_store(const RowGroup &G, unsigned char *dst, uint32_t base, int pitch, int unit,
                                         uint32_t inv, int nrow, const int *rown, int tt)
{
    const int rowb = G.nx * ES, per = rowb / unit;
    for (int j = tt; j < nrow * per; j += G.tpc) {
        const int r = unit == 1 ? j / per : (int)__umulhi((uint32_t)j, inv), q = j - r * per;
        unsigned char *p = dst + (size_t)rown[r] * rowb + q * unit;
        const unsigned char *s = g_smem + base + r * pitch + kRgBody * ES + q * unit;
        if (unit == 16)
            *(uint4 *)p = *(const uint4 *)s;
        else if (unit == 4)
            *(uint32_t *)p = *(const uint32_t *)s;
        else
            *p = *s;
    }
}

__device__ __forceinline__ void rg_wait()
{
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
}

// Copies the periodic x-halos of the first nrow rows of a column from their
// bodies (ES-byte cells), after the block's stores and a barrier.
template <int ES>
__device__ __forceinline__ void rg_halos(const RowGroup &G, uint32_t base, int pitch, int nrow, int tt)
{
    for (int j = tt; j < nrow * 2 * ES; j += G.tpc) {
        const int r = j / (2 * ES), h = j % (2 * ES), rowb = G.nx * ES;
        uint32_t *row = (uint32_t *)(g_smem + base + r * pitch + kRgBody * ES);
        if (h < ES)
            row[rowb / 4 + h] = row[h];  // right halo: the first four cells
        else
            row[h - 2 * ES] = row[rowb / 4 + h - 2 * ES];  // left halo: the last four
    }
}

__device__ __forceinline__ int rg_wrap(int x, int nx)
{
    x = x < 0 ? x + nx : x;
    return x >= nx ? x - nx : x;
}

// Stores v at the cell at byte offset `at` (cell x of its row, possibly a halo
// cell) and at the cell's other copy when it has one.
template <class V>
__device__ __forceinline__ void rg_put(uint32_t at, int x, int nx, V v)
{
    *(V *)(g_smem + at) = v;
    int o = 0;
    if (x < 4) o = nx;               // -4..-1 (halo): body copy; 0..3: right halo
    else if (x >= nx - 4) o = -nx;   // nx-4..nx-1: left halo; nx..nx+3 (halo): body copy
    if (o) *(V *)(g_smem + at + o * (int)sizeof(V)) = v;
}

// Copies of 16 bytes need rows of more than one of them (rg_stage divides by
// their number with a 32-bit reciprocal).
inline void rg_unit(int row_bytes, uintptr_t base, int &unit, uint32_t &inv)
{
    unit = (row_bytes % 16 == 0 && row_bytes > 16 && base % 16 == 0) ? 16 : (base % 4 == 0 ? 4 : 1);
    const uint32_t per = (uint32_t)(row_bytes / unit);
    inv = (uint32_t)((0x100000000ull + per - 1) / per);
}

// Fills the launch geometry: columns per block from the shared memory a
// column takes (per_col bytes beside `fixed`), the block's threads and an even
// share of the SMs.  esq: bytes per cell of the count rows (0: none).  False
// if a column does not fit.
inline bool rg_plan(const smc_lattice *lat, const void *occ, int num_sms, size_t smem_max, size_t fixed, int max_rows,
                    int esq, RowGroup &G)
{
    G.nx = lat->nx;
    G.ny = lat->ny;
    G.nz = lat->nz;
    G.NLx = lat->nx / 4;
    G.NLy = lat->ny / 4;
    G.ncol = G.NLy * (lat->nz / 4);
    const int align = esq ? 64 : 128;
    G.pitch = (kRgBody + lat->nx + 4 + align - 1) / align * align;
    G.pitchq = esq * G.pitch;  // a count row has the layout of a species row, scaled by the cell size
    const size_t per_col = (size_t)max_rows * (size_t)(G.pitch + G.pitchq) + kRgRowBytes;  // rows of every launch are at most max_rows
    if (G.NLx > kRgThreads || fixed + per_col > smem_max) return false;
    G.tpc = (G.NLx + 31) / 32 * 32;
    // Columns per block: the most columns resident on an SM (228 KB of shared
    // memory, 1 KB of it per block), no more than an even share of the SMs.
    const size_t sm_bytes = 228 * 1024;
    const int even = (G.ncol + num_sms - 1) / num_sms, cmax = std::max(1, std::min(kRgThreads / G.tpc, even));
    size_t best = 0;
    G.C = 1;
    for (int c = 1; c <= cmax && fixed + c * per_col <= smem_max; ++c) {
        const size_t resident = std::min<size_t>(c * (sm_bytes / (fixed + c * per_col + 1024)), even);
        if (resident >= best) {  // of equals the largest: a block loads the model's tables once
            best = resident;
            G.C = c;
        }
    }
    rg_unit(lat->nx, (uintptr_t)occ, G.unit, G.inv);
    rg_unit(lat->nx * (esq ? esq : 1), 0, G.unitq, G.invq);
    return true;
}

}  // namespace smc

// sweep_cta.cu -- the pair-model sweep of a small box by one CTA, the whole
// lattice in its shared memory for the length of a call.
//
// A mini-step of a small box has few trials (8 on 8^3 cells, one when no axis
// is cut into four-cell link cells), and the sweep is a chain of n_A of them:
// what counts is the latency of one.  The kernels that spread columns over CTAs
// pay a hand-over between CTAs per group (5.7 us per group of four mini-steps
// at 8^3), or between the warps of a CTA and global memory.  Here one CTA per
// replica runs all mini-steps:
//   - species sit in a box extended by two halo cells on each side, every cell
//     at all its periodic positions, so that a neighbour is one byte at a fixed
//     offset; an accepted swap writes the (at most eight) positions of a and b;
//   - LPT lanes share a trial: each sums the table entries Q_m[A, B](q) of its
//     share of the neighbours of a and (negative) of b, in int32 modulo 2^32,
//     which is the dE_fix of pair_fixed.cuh in any order (the pair a-b, which
//     both sums contain, is taken out by a term of (A, B));
//   - other warps of the CTA compute the Philox words and positions of the
//     trials ahead, into a ring in shared memory.
// Mini-steps are separated by a warp barrier when the trials fill one warp, by a
// named barrier of the compute warps otherwise.
#include <algorithm>
#include <cstring>
#include <vector>

#include "pair_fixed.cuh"

namespace smc {

namespace {

constexpr int kCtaRing = 1024;      // ring entries per half
constexpr int kCtaRngWarps = 4;

// Shared-memory layout of one replica.
struct CtaLayout {
    int EX, EY, EZ;       // extended box
    int ntr, lpt, cthr;   // trials per mini-step, lanes per trial, compute threads (a multiple of 32)
    int E, units, nunit;  // mini-steps per unit (4 or 1), units per ring half, units per sweep
    uint32_t q, off, ring, occ, bytes;
};

__host__ __device__ inline CtaLayout cta_layout(int nx, int ny, int nz, int nsh)
{
    CtaLayout L;
    const int Lx = lc_edge(nx), Ly = lc_edge(ny), Lz = lc_edge(nz);
    L.EX = nx + 4;
    L.EY = ny + 4;
    L.EZ = nz + 4;
    L.ntr = (nx / Lx) * (ny / Ly) * (nz / Lz);
    L.lpt = L.ntr <= 1 ? 32 : (L.ntr <= 2 ? 16 : (L.ntr <= 4 ? 8 : 4));
    L.cthr = (L.ntr * L.lpt + 31) / 32 * 32;
    L.E = Lx == 4 && nx % 4 == 0 ? 4 : 1;  // the four sites of a link cell's row share a Philox block
    L.units = kCtaRing / (L.ntr * L.E) > 0 ? kCtaRing / (L.ntr * L.E) : 1;
    L.nunit = 2 * Lx * Ly * Lz / L.E;
    L.q = 0;
    L.off = L.q + (uint32_t)nsh * 64 * 8 * 4;
    L.ring = L.off + 2 * 32 * 4;
    L.occ = L.ring + 2 * kCtaRing * 16;
    L.bytes = L.occ + (uint32_t)(2 * L.EX * L.EY * L.EZ);
    return L;
}

// Vector t of shells 1-3 (8, 6, 12 of them) from a site of sublattice sub, as
// cell offsets; shell 1 changes the sublattice.
__device__ __forceinline__ int3 cta_vector(int sub, int t)
{
    if (t < 8) {
        const int o = sub == 0 ? -1 : 0;
        return make_int3(o + ((t >> 2) & 1), o + ((t >> 1) & 1), o + (t & 1));
    }
    if (t < 14) {
        const int a = (t - 8) >> 1, s = (t & 1) ? 1 : -1;
        return make_int3(a == 0 ? s : 0, a == 1 ? s : 0, a == 2 ? s : 0);
    }
    const int a = (t - 14) >> 2, s = ((t >> 1) & 1) ? 1 : -1, u = (t & 1) ? 1 : -1;  // a: the axis without offset
    return make_int3(a == 0 ? 0 : s, a == 1 ? 0 : (a == 0 ? s : u), a == 2 ? 0 : u);
}

// Whether the warps that draw the words also bound the accepted dE (one
// compare in the mini-step's chain instead of a table load or an exponential).
// Integer models always (8^3, 100 sweeps: 37 us per sweep against 49);
// floating-point ones when a warp holds one trial (11^3: 435 against 514 us),
// not when the undecided range's branch divides a warp (8^3: 41 against 38).
__host__ __device__ constexpr bool cta_bounded(bool is_int, int lpt) { return is_int || lpt == 32; }

// Width of the undecided range above cta_accept's bound, in dE_fix.
__device__ __forceinline__ int32_t cta_band(float cx)
{
    const float w = 2.5e-4f / -cx;  // twice the margin of cta_accept, and the rounding of both bounds
    return w < 2147480000.f ? __float2int_ru(w) + 512 : 0x7FFFFFFF;
}

template <bool IS_INT, int NSH, int LPT>
__device__ void cta_compute(const SweepParams &P, const CtaLayout &L, const RepDesc &RD, int tid, long long &accE,
                            long long &accN, int rep)
{
    constexpr int NV = NSH >= 3 ? 26 : 14;
    constexpr int kTerms = (2 * NV + LPT - 1) / LPT;
    const int lane = tid % LPT, trial = tid / LPT;
    const bool on = trial < L.ntr;
    const int32_t *Q = (const int32_t *)(g_smem + L.q);
    unsigned char *occ = g_smem + L.occ;
    const int plane = L.EX * L.EY * L.EZ, strY = L.EX, strZ = L.EX * L.EY;
    const int nx = RD.nx, ny = RD.ny, nz = RD.nz;
    const bool one_warp = L.cthr == 32;
    // this lane's neighbours: their offsets from a (or, second half, from b) for
    // a trial on either sublattice, their shell's table and sign
    int o0[kTerms], o1[kTerms], qm[kTerms], sg[kTerms];
    __syncthreads();  // the offset table is written
#pragma unroll
    for (int i = 0; i < kTerms; ++i) {
        const int *off = (const int *)(g_smem + L.off);  // [2][32]
        const int j = i * LPT + lane, v = j < NV ? j : j - NV;
        const bool any = j < 2 * NV;
        o0[i] = any ? off[(j < NV ? 0 : 32) + v] : 0;
        o1[i] = any ? off[(j < NV ? 32 : 0) + v] : 0;
        qm[i] = any ? (v < 8 ? 0 : (v < 14 ? 512 : 1024)) : 0;
        sg[i] = any ? (j < NV ? 1 : -1) : 0;
    }
    int half = 0;
    for (int t = 0; t < P.nsweeps; ++t) {
        float cx = 0.f;
        int32_t band = 0;  // floating-point models: dE in (lo, lo + band] needs the exact test
        if constexpr (!IS_INT) {
            cx = P.temp.beta[P.beta_stride ? rep * P.beta_stride + t : rep];
            if (cta_bounded(IS_INT, LPT)) band = cta_band(cx);
        }
        for (int u0 = 0; u0 < L.nunit; u0 += L.units) {
            __syncthreads();  // this half of the ring is written
            const uint4 *ring = (const uint4 *)(g_smem + L.ring) + half * kCtaRing;
            half ^= 1;
            const int steps = min(L.units, L.nunit - u0) * L.E;
            int accS = 0;  // accepted trials of this unit: those of a launch may exceed 32 bits
            uint4 e = on ? ring[trial] : make_uint4(0, 0, 0, 0);
            for (int k = 0; k < steps; ++k) {
                // entry: word, offset of a, its extended coordinates (10 bits each) and sublattice, accepted dE
                const uint32_t word = e.x;
                const int pa = (int)e.y, co = (int)e.z, lo = (int)e.w;
                if (on && k + 1 < steps) e = ring[(k + 1) * L.ntr + trial];
                const int sub = (int)((uint32_t)co >> 30), dir = (int)(word >> kRBits);
                const int s_off = sub - 1, kx = (dir >> 2) + s_off, ky = ((dir >> 1) & 1) + s_off, kz = (dir & 1) + s_off;
                const int pb = pa + (sub ? -plane : plane) + kz * strZ + ky * strY + kx;
                int q[kTerms];
                int A = 0, B = 0;
                if (on) {
                    A = occ[pa];
                    B = occ[pb];
#pragma unroll
                    for (int i = 0; i < kTerms; ++i)
                        q[i] = occ[(i * LPT + lane < NV ? pa : pb) + (sub ? o1[i] : o0[i])];
                }
                // where a's and b's other periodic positions lie (0: none along that axis)
                const int xa = co & 1023, ya = (co >> 10) & 1023, za = (co >> 20) & 1023;
                auto copy = [](int e, int n, int str) { return e < 4 ? n * str : (e >= n ? -n * str : 0); };
                const int ax = copy(xa, nx, 1), ay = copy(ya, ny, strY), az = copy(za, nz, strZ);
                const int bx = copy(xa + kx, nx, 1), by = copy(ya + ky, ny, strY), bz = copy(za + kz, nz, strZ);
                constexpr int kPut = LPT >= 8 ? 1 : 8 / LPT;
                int wa[kPut], wb[kPut];
#pragma unroll
                for (int i = 0; i < kPut; ++i) {
                    const int h = (i * LPT + lane) & 7;
                    wa[i] = pa + (h & 1 ? ax : 0) + (h & 2 ? ay : 0) + (h & 4 ? az : 0);
                    wb[i] = pb + (h & 1 ? bx : 0) + (h & 2 ? by : 0) + (h & 4 ? bz : 0);
                }
                const int32_t *row = Q + (A * 8 + B) * 8;  // (all zero where A = B)
                int32_t s = 0;
                if (on) {
#pragma unroll
                    for (int i = 0; i < kTerms; i += 2) s += sg[i] * row[qm[i] + q[i]];
                    int32_t s2 = lane == 0 ? row[A] - row[B] : 0;  // the pair a-b itself
#pragma unroll
                    for (int i = 1; i < kTerms; i += 2) s2 += sg[i] * row[qm[i] + q[i]];
                    s += s2;
                }
                if constexpr (LPT == 32) {
                    s = __reduce_add_sync(0xffffffffu, s);
                } else {
#pragma unroll
                    for (int o = LPT / 2; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
                }
                bool acc;
                if constexpr (cta_bounded(IS_INT, LPT)) {
                    acc = s <= lo;
                    if constexpr (!IS_INT) {
                        if (!acc && (int64_t)s <= (int64_t)lo + band)
                            acc = accept_fixed<false>(s, word & kRMask, cx, nullptr, make_int2(0, 0));
                    }
                } else {
                    acc = accept_fixed<false>(s, word & kRMask, cx, nullptr, make_int2(0, 0));
                }
                acc = acc && on;
                if (acc) {
#pragma unroll
                    for (int i = 0; i < kPut; ++i) {
                        occ[wa[i]] = (unsigned char)B;
                        occ[wb[i]] = (unsigned char)A;
                    }
                    if (lane == 0) {
                        accE += s;
                        ++accS;
                    }
                }
                if (one_warp)
                    __syncwarp();
                else
                    asm volatile("bar.sync 1, %0;" ::"r"(L.cthr) : "memory");
            }
            accN += accS;
        }
    }
}

// Largest dE accepted with random number r.  Integer models: the last entry of
// the (non-increasing) acceptance table above r, exactly.  Floating-point
// models: the test 2r + 1 < ceil(2^(dE cx + 30)) is certain to hold up to here;
// cta_band() further up it is certain to fail.  In between (the errors of
// log2, ex2.approx and FP32 are below 1e-5 in the exponent; 1e-4 is allowed
// for) the compute warps evaluate it.
constexpr float kCtaMargin = 1e-4f;

template <bool IS_INT>
__device__ __forceinline__ int32_t cta_accept(uint32_t r, float cx, const uint32_t *tab, int2 ti)
{
    if constexpr (IS_INT) {
        int lo = 0, hi = ti.y;  // entries below lo are > r, those from hi on are not
        while (lo < hi) {
            const int mid = (lo + hi) >> 1;
            if (__ldg(tab + ti.x + mid) > r)
                lo = mid + 1;
            else
                hi = mid;
        }
        return lo > 0 ? lo - 1 : 0;  // dE <= 0 is always accepted
    } else {
        const float t = (log2f((float)(2u * r + 1u)) - kAcceptBias + kCtaMargin) / cx;  // cx <= 0: t >= -margin / |cx|
        return t >= 2147483000.f || !(t == t) ? 0x7FFFFFFF : max(0, __float2int_rd(t));
    }
}

// The words and positions of one unit's trials: ring[(unit * E + mini-step) * ntr + trial].
template <bool IS_INT>
__device__ void cta_rng(const SweepParams &P, const CtaLayout &L, const RepDesc &RD, int tid, int nthr, int rep)
{
    const int Lx = lc_edge(RD.nx), Ly = lc_edge(RD.ny), Lz = lc_edge(RD.nz);
    const int NLx = RD.nx / Lx, NLy = RD.ny / Ly;
    int half = 0;
    for (int t = 0; t < P.nsweeps; ++t) {
        const uint64_t sweep = P.sweep0 + (uint64_t)t;
        const int idx = P.beta_stride ? rep * P.beta_stride + t : rep;
        float cxp = 0.f;
        int2 ti = make_int2(0, 0);
        if constexpr (IS_INT)
            ti = P.temp.tabinfo[idx];
        else
            cxp = P.temp.beta[idx];
        for (int u0 = 0; u0 < L.nunit; u0 += L.units) {
            uint4 *ring = (uint4 *)(g_smem + L.ring) + half * kCtaRing;
            half ^= 1;
            const int n = min(L.units, L.nunit - u0) * L.ntr;
            for (int j = tid; j < n; j += nthr) {
                const int u = j / L.ntr, c = j - u * L.ntr, k = (u0 + u) * L.E;
                const int dx = k % Lx, dy = (k / Lx) % Ly, dz = (k / (Lx * Ly)) % Lz, sub = k / (Lx * Ly * Lz);
                const int cx = c % NLx, cy = (c / NLx) % NLy, cz = c / (NLx * NLy);
                const int x = cx * Lx + dx, y = cy * Ly + dy, z = cz * Lz + dz;
                const uint32_t site = (uint32_t)(((sub * RD.nz + z) * RD.ny + y) * RD.nx + x);
                const U4 w = philox10(U4{site >> 2, RD.rep, (uint32_t)sweep, (uint32_t)(sweep >> 32)}, (uint32_t)P.seed,
                                      (uint32_t)(P.seed >> 32));
                const uint32_t o = (uint32_t)(((sub * L.EZ + z + 2) * L.EY + y + 2) * L.EX + x + 2);
                const uint32_t co = (uint32_t)(x + 2) | (uint32_t)(y + 2) << 10 | (uint32_t)(z + 2) << 20 | (uint32_t)sub << 30;
                for (int d = 0; d < L.E; ++d) {
                    const uint32_t word = pick_word(w, (site + (uint32_t)d) & 3u);
                    const uint32_t lo =
                        cta_bounded(IS_INT, L.lpt) ? (uint32_t)cta_accept<IS_INT>(word & kRMask, cxp, P.tab, ti) : 0u;
                    ring[(u * L.E + d) * L.ntr + c] = make_uint4(word, o + d, co + d, lo);
                }
            }
            __syncthreads();  // handed over; the compute warps are done with the other half
        }
    }
}

// The bounds are those of the largest block.  Without them ptxas aims at fewer
// registers than the chain of a mini-step wants (64 instead of 90): 8^3 cells,
// us per sweep, integer / FP32: 36.4 / 42.4, with them 29.3 / 32.4; 11^3, one
// trial per mini-step: 393 / 450 and 388 / 438; 12^3 three shells of eight species:
// 60 / 55 and 52 / 54.
template <bool IS_INT, int NSH>
__global__ void __launch_bounds__(4 * kCtaMaxTrials + 32 * kCtaRngWarps, 1) k_sweep_cta(const __grid_constant__ SweepParams P, int check)
{
    const int rep = blockIdx.x, tid = threadIdx.x, nthr = blockDim.x;
    const RepDesc &RD = P.rep[rep];
    const CtaLayout L = cta_layout(RD.nx, RD.ny, RD.nz, NSH);
    const int nx = RD.nx, ny = RD.ny, nz = RD.nz, N = 2 * nx * ny * nz;
    unsigned char *occ = g_smem + L.occ;
    __shared__ unsigned long long s_e, s_n;
    // Q_m[A, B](q) from the byte planes of the table rows
    int32_t *Q = (int32_t *)(g_smem + L.q);
    const int sw = (P.qrow - 4) / (NSH * 4) >= 2 ? 2 : 1;
    for (int i = tid; i < NSH * 512; i += nthr) {
        const int m = i >> 9, row = (i >> 3) & 63, q = i & 7;
        uint32_t v = 0;
        if (q < 4 * sw)
            for (int k = 0; k < 4; ++k)
                v |= ((P.qtab[row * P.qrow + (m * sw + (q >> 2)) * 4 + k] >> (8 * (q & 3))) & 0xFFu) << (8 * k);
        Q[i] = (int32_t)v;
    }
    for (int i = tid; i < 64; i += nthr) {
        const int sub = i >> 5, t = i & 31;
        int o = 0;
        if (t < 26) {
            const int3 v = cta_vector(sub, t);
            o = (v.z * L.EY + v.y) * L.EX + v.x + (t < 8 ? (sub ? -1 : 1) * L.EX * L.EY * L.EZ : 0);
        }
        ((int *)(g_smem + L.off))[i] = o;
    }
    if (tid == 0) s_e = s_n = 0;
    bool bad = false;
    for (int i = tid; i < 2 * L.EX * L.EY * L.EZ; i += nthr) {
        const int ex = i % L.EX, ey = (i / L.EX) % L.EY, ez = (i / (L.EX * L.EY)) % L.EZ, sub = i / (L.EX * L.EY * L.EZ);
        const int x = wrapc(ex - 2, nx), y = wrapc(ey - 2, ny), z = wrapc(ez - 2, nz);
        const int v = RD.occ[((sub * nz + z) * ny + y) * nx + x];
        bad |= v < 0 || v >= P.S;
        occ[i] = (unsigned char)(v & 7);
    }
    if (bad && check) atomicCAS(P.status, 0, (int)SMC_ERR_ARG);
    long long accE = 0, accN = 0;
    if (tid >= L.cthr) {
        // (threads of a larger replica's block that this one does not need draw words as well)
        __syncthreads();  // the compute warps read the offset table
        cta_rng<IS_INT>(P, L, RD, tid - L.cthr, nthr - L.cthr, rep);
    } else {
        switch (L.lpt) {
        case 32: cta_compute<IS_INT, NSH, 32>(P, L, RD, tid, accE, accN, rep); break;
        case 16: cta_compute<IS_INT, NSH, 16>(P, L, RD, tid, accE, accN, rep); break;
        case 8: cta_compute<IS_INT, NSH, 8>(P, L, RD, tid, accE, accN, rep); break;
        default: cta_compute<IS_INT, NSH, 4>(P, L, RD, tid, accE, accN, rep); break;
        }
        if (accE) atomicAdd(&s_e, (unsigned long long)accE);
        if (accN) atomicAdd(&s_n, (unsigned long long)accN);
    }
    __syncthreads();
    for (int i = tid; i < N; i += nthr) {
        const int x = i % nx, y = (i / nx) % ny, z = (i / (nx * ny)) % nz, sub = i / (nx * ny * nz);
        RD.occ[i] = (int8_t)occ[((sub * L.EZ + z + 2) * L.EY + y + 2) * L.EX + x + 2];
    }
    if (tid == 0) {
        if (RD.e_acc) *RD.e_acc += (double)(long long)s_e * P.escale;
        if (RD.n_acc) *RD.n_acc += (long long)s_n;
    }
}

}  // namespace

// One CTA per replica is taken for boxes of at least 4 cells per axis whose
// lattice and ring fit, with up to `most` trials per mini-step.
bool cta_takes(int R, const smc_lattice *lats, int nsh, int most, size_t smem_max)
{
    for (int r = 0; r < R; ++r) {
        const smc_lattice &l = lats[r];
        if (l.nx < 4 || l.ny < 4 || l.nz < 4 || l.nx > 1000 || l.ny > 1000 || l.nz > 1000) return false;
        if ((long long)(l.nx + 4) * (l.ny + 4) * (l.nz + 4) * 2 > (long long)smem_max) return false;
        const CtaLayout L = cta_layout(l.nx, l.ny, l.nz, nsh);
        if (L.ntr > most || L.ntr * L.E > kCtaRing || L.bytes + 16 > smem_max) return false;
    }
    return true;
}

smc_status launch_pair_sweep_cta(int R, const smc_lattice *lats, const smc_model *m, const PairTable &pt,
                                 int8_t *const *occ, uint64_t seed, uint32_t replica0, uint64_t sweep0, int nsweeps,
                                 const double *kT, int most, bool check, double *e_acc, int64_t *n_acc,
                                 cudaStream_t stream)
{
    smc_status st;
    Workspace *ws = workspace(&st);
    if (!ws) return st;
    if (!cta_takes(R, lats, pt.nsh, std::min(most, kCtaMaxTrials), ws->smem_optin)) return SMC_ERR_UNSUPPORTED;
    const bool is_int = m->kind == SMC_PAIR_I32;
    static SweepParams P;
    memset(&P, 0, sizeof P);
    P.R = R;
    P.S = lats[0].nspecies;
    P.nshells = m->nshells;
    P.seed = seed;
    P.status = ws->status;
    P.qrow = pt.rw;
    P.escale = pt.scale;
    memcpy(P.qtab, pt.rows.data(), pt.rows.size() * 4);
    size_t smem = 0;
    int cthr = 0;
    for (int r = 0; r < R; ++r) {
        RepDesc &d = P.rep[r];
        d.occ = occ[r];
        d.e_acc = e_acc ? e_acc + r : nullptr;
        d.n_acc = n_acc ? (long long *)n_acc + r : nullptr;
        d.nx = lats[r].nx;
        d.ny = lats[r].ny;
        d.nz = lats[r].nz;
        d.rep = replica0 + (uint32_t)r;
        const CtaLayout L = cta_layout(d.nx, d.ny, d.nz, pt.nsh);
        smem = std::max<size_t>(smem, L.bytes);
        cthr = std::max(cthr, L.cthr);
    }
    bool constant = true;
    for (int r = 0; r < R && constant; ++r)
        for (int t = 1; t < nsweeps; ++t)
            if (kT[(size_t)r * nsweeps + t] != kT[(size_t)r * nsweeps]) constant = false;
    const int cap = is_int ? kMaxBeta / 2 : kMaxBeta;
    const int chunk = constant ? nsweeps : std::max(1, cap / R);
    std::vector<uint32_t> tabs;  // integer acceptance tables, one per distinct kT
    std::vector<std::pair<double, int2>> tindex;
    auto table_of = [&](double kt) -> int2 {
        for (auto &p : tindex)
            if (p.first == kt) return p.second;
        std::vector<uint32_t> t = int_table(m->unit_ev, kt);
        const int2 ti = make_int2((int)tabs.size(), (int)t.size());
        tabs.insert(tabs.end(), t.begin(), t.end());
        tindex.push_back({kt, ti});
        return ti;
    };
    cudaError_t e;
    if (is_int) {
        for (int r = 0; r < R; ++r)
            for (int t = 0; t < nsweeps; ++t) table_of(kT[(size_t)r * nsweeps + t]);
        unsigned char *scr = (unsigned char *)workspace_scratch(ws, tabs.size() * 4 + 16, &st);
        if (!scr) return st;
        e = cudaMemcpyAsync(scr, tabs.data(), tabs.size() * 4, cudaMemcpyHostToDevice, stream);
        if (e != cudaSuccess) return cuda_fail(e, "cudaMemcpyAsync(acceptance tables)");
        P.tab = (const uint32_t *)scr;
    }
    auto kern = is_int ? (pt.nsh >= 3 ? k_sweep_cta<true, 3> : k_sweep_cta<true, 2>)
                       : (pt.nsh >= 3 ? k_sweep_cta<false, 3> : k_sweep_cta<false, 2>);
    e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return cuda_fail(e, "cudaFuncSetAttribute(k_sweep_cta)");
    for (int t0 = 0; t0 < nsweeps; t0 += chunk) {
        const int nc = std::min(chunk, nsweeps - t0);
        P.sweep0 = sweep0 + (uint64_t)t0;
        P.nsweeps = nc;
        P.beta_stride = constant ? 0 : nc;
        for (int r = 0; r < R; ++r)
            for (int t = 0; t < (constant ? 1 : nc); ++t) {
                const double kt = kT[(size_t)r * nsweeps + t0 + t];
                const int idx = constant ? r : r * nc + t;
                if (is_int)
                    P.temp.tabinfo[idx] = table_of(kt);
                else
                    P.temp.beta[idx] = accept_cx(pt.scale, kt);
            }
        kern<<<R, cthr + 32 * kCtaRngWarps, smem, stream>>>(P, check ? 1 : 0);
        e = cudaGetLastError();
        if (e != cudaSuccess) return cuda_fail(e, "k_sweep_cta");
    }
    return SMC_OK;
}

}  // namespace smc

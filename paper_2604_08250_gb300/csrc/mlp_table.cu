// mlp_table.cu -- swap-MC sweeps with the MLP and MLPNet site energies read
// from a table of f over every feature vector.
//
// The features of a site (its species and the species counts of its three
// shells) take S n1 n2 n3 values, n_m = C(z_m + S - 1, S - 1) ways to fill
// the z_m = 8, 6, 12 neighbours: 9.46e8 for five species, 2.5e7 for four,
// 3.4e5 for three.  A sweep evaluates f for 40 sites per trial of unlike
// species, 1.07e9 of them on an equiatomic 256^3 lattice, so from about one
// such sweep per call on it is cheaper to evaluate every vector once
// (k_table_fill, on the tensor cores, 4 B per vector) and to look f up: f is
// a fixed function of the features with the same bits wherever it is
// evaluated (mlp_tc.cuh), so the looked-up sweep takes the same decisions as
// the evaluating one.  Measured (GB300, 256^3, five species): the table 35 ms
// (MLP) or 36 ms (MLPNet), then 22 ms per sweep, against 60 ms (MLP) and 90 ms
// (MLPNet) per sweep of the evaluating kernel.  Which of the two a call takes
// depends on the box and on its share of unlike bonds (table_gain).
//
// Feature vectors are numbered shell by shell: r_m is the rank of the shell's
// composition among the n_m, most probable (largest multinomial coefficient)
// first, which keeps the part of the table that a random alloy visits
// together.  A site's word packs (species, r_1, r_2, r_3) into 31 bits, so
// the state of the sweep is 8 bytes per site (word, f), against the 20 of the
// evaluating sweep (packed counts and f).  A swap moves one A neighbour to B
// in the shell where a zone site sees a, and one B to A where it sees b; a
// move goes through the composition without the removed neighbour (two 16-bit
// loads, 43 KB of shared memory for five species; one load from tables of all
// ordered pairs would take 101 KB, see k_table_sweep).
//
// k_table_sweep runs the four mini-steps of a group (one launch per group of
// the 32): columns of one group share no zone site, so no block waits for
// another.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <map>
#include <mutex>
#include <vector>

#include "mlp_zone.cuh"

namespace smc {

namespace {

__host__ __device__ constexpr int shell_z(int m) { return m == 0 ? 8 : (m == 1 ? 6 : 12); }
// fields of a site word: r_3 in bits 0-10, r_2 in 11-18, r_1 in 19-27, species in 28-30
__host__ __device__ constexpr int word_sh(int m) { return m == 0 ? 19 : (m == 1 ? 11 : 0); }
__host__ __device__ constexpr uint32_t word_mask(int m) { return m == 0 ? 511u : (m == 1 ? 255u : 2047u); }
constexpr int kWordSp = 28;

// Numbers of a species count S: ranks, their compositions and the moves.
struct TableDims {
    int S;
    int n[3];              // compositions per shell
    int nd[3];             // compositions of z_m - 1 neighbours
    uint32_t rem[3];       // offset of shell m's removals (16-bit units): [species][rank] -> rank among nd
    uint32_t add[3];       // offset of shell m's additions: [species][rank among nd] -> rank
    uint32_t mv_total;     // 16-bit units, padded to 8
    uint32_t rk[3];        // offset of shell m's rank map (16-bit units), by sum_q c_q (z+1)^q, q < S-1
    uint32_t rk_total;     // 16-bit units, padded to 8
    uint32_t un[3];        // offset of shell m's packed counts (32-bit units)
    uint32_t un_total;     // padded to 4
    long long entries;     // S n1 n2 n3
};

struct TableHost {
    TableDims d;
    std::vector<uint16_t> moves, ranks;
    std::vector<uint32_t> unrank;
    std::vector<uint32_t> rows;  // per composition (at 4 (un[m] + rank)): its BF16 counts as words of a feature row
};

void enumerate(int left, int q, int S, std::vector<int> &c, std::vector<std::vector<int>> &out)
{
    if (q == S - 1) {
        c[q] = left;
        out.push_back(c);
        return;
    }
    for (int k = left; k >= 0; --k) {
        c[q] = k;
        enumerate(left - k, q + 1, S, c, out);
    }
}

void build_table_host(int S, TableHost &T)
{
    TableDims &d = T.d;
    memset(&d, 0, sizeof d);
    d.S = S;
    d.entries = S;
    uint32_t mv = 0, rk = 0, un = 0;
    std::vector<std::vector<int>> comp[3], part[3];
    for (int m = 0; m < 3; ++m) {
        const int z = shell_z(m);
        std::vector<int> c((size_t)S, 0);
        enumerate(z, 0, S, c, comp[m]);
        auto weight = [](const std::vector<int> &v) {  // -log of the multinomial coefficient, up to a constant
            double w = 0.0;
            for (int x : v)
                for (int k = 2; k <= x; ++k) w += std::log((double)k);
            return w;
        };
        std::stable_sort(comp[m].begin(), comp[m].end(),
                         [&](const std::vector<int> &a, const std::vector<int> &b) { return weight(a) < weight(b) - 1e-9; });
        d.n[m] = (int)comp[m].size();
        d.entries *= d.n[m];
        enumerate(z - 1, 0, S, c, part[m]);
        d.nd[m] = (int)part[m].size();
        d.rem[m] = mv;
        mv += (uint32_t)(S * d.n[m]);
        d.add[m] = mv;
        mv += (uint32_t)(S * d.nd[m]);
        d.rk[m] = rk;
        d.un[m] = un;
        uint32_t span = 1;
        for (int q = 0; q < S - 1; ++q) span *= (uint32_t)(z + 1);
        rk += span;
        un += (uint32_t)d.n[m];
    }
    d.mv_total = (mv + 7) / 8 * 8;
    d.rk_total = (rk + 7) / 8 * 8;
    d.un_total = (un + 3) / 4 * 4;
    T.moves.assign(std::max<size_t>(d.mv_total, 8), 0);
    T.ranks.assign(d.rk_total, 0);
    T.unrank.assign(d.un_total, 0);
    T.rows.assign(4 * (size_t)d.un_total, 0);
    for (int m = 0; m < 3; ++m) {
        const int z = shell_z(m);
        auto radix = [&](const std::vector<int> &c) {
            uint32_t v = 0, p = 1;
            for (int q = 0; q < S - 1; ++q) {
                v += (uint32_t)c[(size_t)q] * p;
                p *= (uint32_t)(z + 1);
            }
            return v;
        };
        for (int r = 0; r < d.n[m]; ++r) {
            const std::vector<int> &c = comp[m][(size_t)r];
            T.ranks[d.rk[m] + radix(c)] = (uint16_t)r;
            uint32_t h = 0;
            for (int q = 0; q < S; ++q) h += (uint32_t)c[(size_t)q] << (4 * q);
            T.unrank[d.un[m] + (uint32_t)r] = h;
            for (int q = 0; q < S; ++q) {  // column 5 (m + 1) + q of the row, relative to the word of the shell's first
                const float f = (float)c[(size_t)q];
                uint32_t b;
                memcpy(&b, &f, 4);
                const int col = (5 * (m + 1) & 1) + q;
                T.rows[4 * (size_t)(d.un[m] + (uint32_t)r) + (size_t)(col / 2)] |= (b >> 16) << (16 * (col & 1));
            }
        }
        std::map<std::vector<int>, int> rank;
        for (int r = 0; r < d.n[m]; ++r) rank[comp[m][(size_t)r]] = r;
        for (int r = 0; r < d.nd[m]; ++r)
            for (int A = 0; A < S; ++A) {
                std::vector<int> c = part[m][(size_t)r];
                ++c[(size_t)A];
                const int to = rank[c];
                T.moves[d.add[m] + (uint32_t)(A * d.nd[m] + r)] = (uint16_t)to;
                // the removal that undoes it; one of an absent species (never made) stays 0
                T.moves[d.rem[m] + (uint32_t)(A * d.n[m] + to)] = (uint16_t)r;
            }
    }
}

// The tables of S species, built once per process.
const TableHost &table_host(int S)
{
    static TableHost T[6];
    static std::once_flag once[6];
    std::call_once(once[S], [S] { build_table_host(S, T[S]); });
    return T[S];
}

struct TableParams {
    TableDims d;
    int nx, ny, nz, NLx, NLy, NLz, ncol;
    int K, team_threads;     // teams per block (a column each) and their threads
    int nshells;             // of the pair part (0: none)
    int8_t *occ;
    uint2 *state;            // per site (word, bits of f)
    const float *table;      // f by feature vector
    const uint16_t *moves, *ranks;
    const uint32_t *unrank;
    const uint32_t *geo;     // [2][8][kOmega]
    const float *D;          // pair table (kDEntries)
    double *part_e;          // per link cell
    long long *part_n;
    uint64_t seed, sweep;
    uint32_t replica;
    float beta;
    int g;                   // group
    const int *route;        // 0 there: the call evaluates its rows, nothing to do here (NULL: tabulated for certain)
    int *status;
    long long timeout_ns;
};

// Table index of a site word.  Plain rank order spreads the probable vectors
// over the whole of the five-species table, 3.8 GB: a random alloy finds half
// of its look-ups in 256 of the 1900 2 MB pages.  There (SPLIT) every shell's
// ranks are cut into probable and other ones, and the eight combinations lie
// one after the other, the most probable first: 50 % of the look-ups in 98
// pages, and a group of mini-steps at 256^3 takes 0.70 ms instead of 0.80
// (cuts at 64, 48, 400 and 96, 96, 768: 0.71 and 0.72).  A finer cut by digits
// with a table of places took 0.76, one by bit fields 0.80 (its power-of-two
// strides crowd the cache sets).
constexpr uint32_t kCut1 = 96, kCut2 = 64, kCut3 = 512;
constexpr uint32_t kRest1 = 495 - kCut1, kRest2 = 210 - kCut2, kRest3 = 1820 - kCut3;

template <bool SPLIT>
__device__ __forceinline__ uint32_t word_index(const TableDims &D, uint32_t w)
{
    const uint32_t s = w >> kWordSp, r1 = (w >> word_sh(0)) & word_mask(0), r2 = (w >> word_sh(1)) & word_mask(1),
                   r3 = w & word_mask(2);
    if (!SPLIT) return ((s * (uint32_t)D.n[0] + r1) * (uint32_t)D.n[1] + r2) * (uint32_t)D.n[2] + r3;
    constexpr uint32_t a1 = kCut1, a2 = kCut2, a3 = kCut3, b1 = kRest1, b2 = kRest2, b3 = kRest3;
    // starts of the combinations (shell 1, 2, 3 beyond its cut)
    constexpr uint32_t z001 = 5 * a1 * a2 * a3, z010 = z001 + 5 * a1 * a2 * b3, z100 = z010 + 5 * a1 * b2 * a3,
                       z011 = z100 + 5 * b1 * a2 * a3, z101 = z011 + 5 * a1 * b2 * b3, z110 = z101 + 5 * b1 * a2 * b3,
                       z111 = z110 + 5 * b1 * b2 * a3;
    static_assert((unsigned long long)z111 + 5ull * b1 * b2 * b3 == 5ull * 495 * 210 * 1820, "the blocks fill the table");
    const bool c1 = r1 >= a1, c2 = r2 >= a2, c3 = r3 >= a3;
    const uint32_t d1 = c1 ? b1 : a1, d2 = c2 ? b2 : a2, d3 = c3 ? b3 : a3;
    const uint32_t q1 = c1 ? r1 - a1 : r1, q2 = c2 ? r2 - a2 : r2, q3 = c3 ? r3 - a3 : r3;
    const uint32_t z = c1 ? (c2 ? (c3 ? z111 : z110) : (c3 ? z101 : z100)) : (c2 ? (c3 ? z011 : z010) : (c3 ? z001 : 0u));
    return z + ((s * d1 + q1) * d2 + q2) * d3 + q3;
}

// ---------------------------------------------------------------------------
// f of every feature vector.  Tile t holds vectors 128 t .. 128 t + 127.
//
// Bound by the chain of a tile (products, barriers, epilogues) and the ALU
// under it, so that what a row costs besides its network counts: ranks advance
// by the stride of the grid with carries (no divisions), and a row is put
// together from the words of its three compositions (three 16-byte loads)
// instead of from counts.  945 M vectors: MLP 37.9 -> 35.3 ms (its tanh alone
// would take 26), MLPNet 42.4 -> 38.5 ms, and 35.7 ms with five warpgroups on
// all tensor memory instead of four.
// ---------------------------------------------------------------------------
template <class Net>
__global__ void __launch_bounds__(128 * Net::kFillNWG) k_table_fill(const void *W, const TableDims D,
                                                              const uint4 *__restrict__ rows, float *table,
                                                              const int *route, long long timeout_ns, int *status,
                                                              int *abort_flag)
{
    if (route && *route == 0) return;
    constexpr int NWG = Net::kFillNWG;
    constexpr uint32_t xg = NWG <= 4 ? 512 : 384;  // bytes of 8 rows of the X tile
    typename Net::Eval E = mlp_evaluator<Net, NWG>(timeout_ns, status, abort_flag);
    mlp_cta_setup<Net, NWG>(E, W, nullptr, nullptr);
    const int r = threadIdx.x & 127, wg = threadIdx.x >> 7;
    const uint32_t nv = (uint32_t)D.entries, ntile = (nv + kTcRows - 1) / kTcRows;
    const uint32_t step = (uint32_t)NWG * gridDim.x;
    uint32_t tl = (uint32_t)NWG * blockIdx.x + wg;
    // species and ranks of vector 128 tl + r, and of the stride
    uint32_t t = tl * kTcRows + r;
    const uint32_t n1 = (uint32_t)D.n[0], n2 = (uint32_t)D.n[1], n3 = (uint32_t)D.n[2];
    uint32_t r3 = t % n3, r2 = (t /= n3) % n2, r1 = (t /= n2) % n1, q = t / n1;
    t = step * kTcRows;
    const uint32_t d3 = t % n3, d2 = (t /= n3) % n2, d1 = (t /= n2) % n1, dq = t / n1;
    unsigned char *const row = g_smem + E.L.x + (r >> 3) * xg + (r & 7) * 16;  // chunks of 8 columns 128 bytes apart
    for (int kc = 0; kc < (NWG <= 4 || r >= 120 ? 4 : 3); ++kc) *(uint4 *)(row + 128 * kc) = make_uint4(0u, 0u, 0u, 0u);
    wg_sync(E.bar);
    // writes the row of vector 128 tl + r and advances; its place in the table (~0: past the last)
    auto build = [&](uint32_t tl) {
        uint32_t at = ~0u;
        if (q < (uint32_t)D.S) {
            const uint4 a = __ldg(rows + D.un[0] + r1), b = __ldg(rows + D.un[1] + r2), c = __ldg(rows + D.un[2] + r3);
            const uint32_t one = 0x3F80u << (16 * (q & 1));  // columns 0-4: the species
            *(uint4 *)row =
                make_uint4(q < 2 ? one : 0u, (q >> 1) == 1 ? one : 0u, (q == 4 ? one : 0u) | a.x, a.y);
            *(uint4 *)(row + 128) = make_uint4(a.z, b.x, b.y, b.z | c.x);
            *(uint4 *)(row + 256) = make_uint4(c.y, c.z, 0x3F803F80u, 0x00003F80u);
            at = D.S == 5 ? word_index<true>(D, q << kWordSp | r1 << word_sh(0) | r2 << word_sh(1) | r3) : tl * kTcRows + r;
        }
        fence_async_smem();
        r3 += d3;
        uint32_t carry = r3 >= n3;
        r3 -= carry ? n3 : 0u;
        r2 += d2 + carry;
        carry = r2 >= n2;
        r2 -= carry ? n2 : 0u;
        r1 += d1 + carry;
        carry = r1 >= n1;
        r1 -= carry ? n1 : 0u;
        q += dq + carry;
        return at;
    };
    uint32_t at = ~0u;
    if (tl < ntile) {
        at = build(tl);
        tc_issue1(E);
    }
    while (tl < ntile) {
        tc_stage2(E);
        const uint32_t next = tl + step;
        uint32_t at_next = ~0u;
        if (next < ntile) {
            at_next = build(next);
            tc_issue1(E);
        }
        const float f = tc_finish(E);
        if (at != ~0u) table[at] = f;
        at = at_next;
        tl = next;
    }
    tc_teardown(E, NWG);
}

// Position of cell x in a row of states: cells of one residue x mod 4 are
// contiguous, so that neighbouring link cells are neighbouring words (the
// threads of a warp read 8-byte states without bank conflicts).
__device__ __forceinline__ int state_pos(int x, int NLx) { return (x & 3) * NLx + (x >> 2); }

// The state of every site from the occupancy.
__global__ void __launch_bounds__(256) k_table_state(const __grid_constant__ TableParams P)
{
    if (P.route && *P.route == 0) return;
    const long long N = 2LL * P.nx * P.ny * P.nz;
    const int S = P.d.S;
    auto spec = [&](int sb, int xx, int yy, int zz) { return occ_at(P.occ, P.nx, P.ny, P.nz, sb, xx, yy, zz); };
    for (long long s = blockIdx.x * (long long)blockDim.x + threadIdx.x; s < N; s += (long long)gridDim.x * blockDim.x) {
        uint32_t t = (uint32_t)s;
        const int x = (int)(t % (uint32_t)P.nx);
        t /= (uint32_t)P.nx;
        const int y = (int)(t % (uint32_t)P.ny);
        t /= (uint32_t)P.ny;
        const int z = (int)(t % (uint32_t)P.nz);
        const int sub = (int)(t / (uint32_t)P.nz);
        uint32_t h[3];
        site_hist(spec, sub, x, y, z, h[0], h[1], h[2]);
        // species outside [0, S) make no composition: their index is clamped into the table
        uint32_t w = min((uint32_t)(P.occ[s] & 7), (uint32_t)S - 1u) << kWordSp;
#pragma unroll
        for (int m = 0; m < 3; ++m) {
            uint32_t v = 0, p = 1;
            for (int q = 0; q < S - 1; ++q) {
                v += min((h[m] >> (4 * q)) & 15u, (uint32_t)shell_z(m)) * p;
                p *= (uint32_t)(shell_z(m) + 1);
            }
            w |= (uint32_t)__ldg(P.ranks + P.d.rk[m] + v) << word_sh(m);
        }
        P.state[s - x + state_pos(x, P.NLx)] = make_uint2(w, __float_as_uint(__ldg(P.table + (S == 5 ? word_index<true>(P.d, w) : word_index<false>(P.d, w)))));
    }
}

// ---------------------------------------------------------------------------
// One group of mini-steps.  A team of warps takes a column at a time: the 25
// rows of site states that its trials touch (9 of the trial sublattice, 16 of
// the other) are copied to shared memory, the four mini-steps run there, and
// the rows are written back.  Four lanes share a trial, ten zone sites each.
// What bounds it are the look-ups, 40 per trial of unlike species: with five
// species three in four miss L2 and cost a 128-byte DRAM read each (a
// microbenchmark of such loads runs 39 G/s), and the loads that an SM can have
// in flight need room in L1.  So shared memory is kept small: with move tables
// of ordered pairs (204 KB used, 28 KB of L1) a group took 1.03 ms, with the
// factored ones 0.80 ms, and with the vectors of probable compositions in
// blocks of their own (word_index) 0.70 ms, 48 G/s (256^3); a thread per
// trial, eight lanes per trial and whole-block barriers were within 5 % of each
// other, and so were lanes with ten consecutive zone entries each.
// ---------------------------------------------------------------------------
constexpr int kTabTrials = 128;               // most trials of a block's mini-step
constexpr int kLanes = 4;                     // lanes of a trial
constexpr int kTabThreads = kLanes * kTabTrials;
constexpr int kTabRows = 25;
constexpr int kMoveBases = 64;
constexpr int kPer = kOmega / kLanes;         // zone sites per lane

// Shared memory of a team: row numbers (28 ints), Philox words, rows.
__host__ __device__ constexpr size_t table_team_bytes(int nx) { return 28 * 4 + (size_t)nx * 4 + (size_t)kTabRows * nx * 8; }

// Row r of a column (cells y0, z0 of sublattice sub): 0-8 the trial
// sublattice, dy, dz in -1..1; 9-24 the other, dy, dz in o..o+3 with o = -2
// for sublattice 0, -1 for 1.  Returned as (sublattice, y, z) row number.
__device__ __forceinline__ int table_row(int r, int sub, int y0, int z0, int ny, int nz)
{
    const bool own = r < 9;
    const int q = own ? r : r - 9, o = own ? -1 : (sub == 0 ? -2 : -1), per = own ? 3 : 4;
    const int y = wrapc(y0 + o + q / per, ny), z = wrapc(z0 + o + q % per, nz);
    return ((own ? sub : 1 - sub) * nz + z) * ny + y;
}

// Site word after one neighbour in shell m (0: none) changes from A to B;
// rem[m], add[m]: shell m's removals of A and additions of B.
__device__ __forceinline__ uint32_t table_move(uint32_t w, uint32_t m, const uint16_t *mv, const uint32_t *rem,
                                               const uint32_t *add)
{
    const uint32_t sh = m == 1 ? word_sh(0) : (m == 2 ? word_sh(1) : word_sh(2));
    const uint32_t mask = m == 1 ? word_mask(0) : (m == 2 ? word_mask(1) : word_mask(2));
    const uint32_t r = (w >> sh) & mask;
    return m ? w + (((uint32_t)mv[add[m] + mv[rem[m] + r]] - r) << sh) : w;
}

// Waits until the shared counter at a reaches need; false after timeout_ns.
__device__ __forceinline__ bool table_wait(uint32_t a, uint32_t need, long long timeout_ns)
{
    uint64_t t0 = 0;
    for (;;) {
        uint32_t v;
        asm volatile("ld.acquire.cta.shared::cta.u32 %0, [%1];" : "=r"(v) : "r"(a) : "memory");
        if (v >= need) return true;
        if (t0 == 0) t0 = global_ns();
        if ((long long)(global_ns() - t0) > timeout_ns) return false;
        __nanosleep(32);
    }
}

// Barrier of one team (id 1 + team): n threads, a multiple of 32.
__device__ __forceinline__ void team_sync(int team, int n)
{
    asm volatile("bar.sync %0, %1;" ::"r"(team + 1), "r"(n) : "memory");
}

template <bool HAS_PAIR, bool SPLIT>
__global__ void __launch_bounds__(kTabThreads, 1) k_table_sweep(const __grid_constant__ TableParams P)
{
    if (P.route && *P.route == 0) return;
    // shared memory: moves | zone table | the moves' offsets | progress | (pair) D | per team: row numbers,
    // Philox words, rows
    uint16_t *mv = (uint16_t *)g_smem;
    uint32_t *geo = (uint32_t *)(g_smem + P.d.mv_total * 2);
    uint32_t *base = geo + kOmega * 8;
    uint32_t *prog = base + kMoveBases;  // mini-steps done by each warp
    float *Dt = (float *)(prog + kTabThreads / 32);
    const int tid = threadIdx.x, nthr = blockDim.x;
    const int nx = P.nx, ny = P.ny, nz = P.nz, NLx = P.NLx;
    const int tthr = P.team_threads, team = tid / tthr, tt = tid - team * tthr;  // thread of the team
    int *rown = (int *)((unsigned char *)(Dt + (HAS_PAIR ? kDEntries : 0)) + (size_t)team * table_team_bytes(nx));
    uint4 *words = (uint4 *)(rown + 28);
    uint2 *rows = (uint2 *)(words + NLx);
    const int dy = P.g & 3, dz = (P.g >> 2) & 3, sub = P.g >> 4;
    for (uint32_t i = tid; i < P.d.mv_total / 8; i += nthr) ((uint4 *)mv)[i] = __ldg((const uint4 *)P.moves + i);
    for (int i = tid; i < kOmega * 8; i += nthr) geo[i] = __ldg(P.geo + sub * kOmega * 8 + i);
    if (tid < 32) {  // removals of species p, shell m at base[4 p + m], additions at base[32 + 4 p + m]
        const int m = (tid & 3) - 1, p = tid >> 2;
        const bool ok = m >= 0 && p < P.d.S;
        base[tid] = ok ? P.d.rem[m] + (uint32_t)(p * P.d.n[m]) : 0u;
        base[32 + tid] = ok ? P.d.add[m] + (uint32_t)(p * P.d.nd[m]) : 0u;
    }
    if (HAS_PAIR)
        for (int i = tid; i < kDEntries; i += nthr) Dt[i] = __ldg(P.D + i);
    if ((tid & 31) == 0) prog[tid >> 5] = 0;
    __syncthreads();
    constexpr int kPerWarp = 32 / kLanes;  // trials of a warp
    const int i = tt / kLanes, sl = tt % kLanes;
    const int quads = nx / 2;  // 16-byte pieces of a row
    // Between mini-steps a trial depends on its neighbouring link cells only:
    // a warp waits for the warps left and right of it (periodic) when the
    // link cells fill whole warps, else the team waits for all of its own.
    const bool pairwise = NLx % kPerWarp == 0;
    const int w0 = team * tthr / 32, wpc = tthr / 32, wt = tt >> 5;
    const uint32_t prog0 = (uint32_t)__cvta_generic_to_shared(prog);
    const uint32_t mine = prog0 + 4 * (w0 + wt), look = prog0 + 4 * (w0 + (wt + ((tt & 1) ? 1 : wpc - 1)) % wpc);
    uint32_t step = 0;
    const bool active = i < NLx;
    uint2 *st0 = rows;
    for (int col = blockIdx.x + gridDim.x * team; col < P.ncol; col += gridDim.x * P.K) {
        const int y0 = 4 * (col % P.NLy) + dy, z0 = 4 * (col / P.NLy) + dz;
        if (tt < kTabRows) rown[tt] = table_row(tt, sub, y0, z0, ny, nz);
        team_sync(team, tthr);
        for (int j = tt; j < kTabRows * quads; j += tthr) {
            const int r = j / quads, q = j - r * quads;
            const uint32_t dst = (uint32_t)__cvta_generic_to_shared((uint4 *)rows + j);
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst),
                         "l"((const uint4 *)(P.state + (size_t)rown[r] * nx) + q)
                         : "memory");
        }
        for (int j = tt; j < NLx; j += tthr) {
            const int site = ((sub * nz + z0) * ny + y0) * nx;
            const U4 w = philox10(U4{((uint32_t)site >> 2) + (uint32_t)j, P.replica, (uint32_t)P.sweep,
                                     (uint32_t)(P.sweep >> 32)},
                                  (uint32_t)P.seed, (uint32_t)(P.seed >> 32));
            words[j] = make_uint4(w.x, w.y, w.z, w.w);
        }
        asm volatile("cp.async.wait_all;" ::: "memory");
        team_sync(team, tthr);
        double accE = 0.0;
        int accN = 0;
        for (int dx = 0; dx < 4; ++dx) {
            // The lanes of a warp stay together (full-mask shuffles); lanes of a
            // trial that changes nothing, or of none, look nothing up.
            const uint32_t word = ((const uint32_t *)(words + (active ? i : 0)))[dx];
            const int dir = (int)(word >> kRBits);
            const uint32_t *gd = geo + dir * kOmega;
            // zone site of entry word gw: row offset gw & 0x7FFF, cell 4 i + dx + dxo
            auto pos = [&](uint32_t gw) {
                const int u = dx + (int)((gw >> 15) & 7u) - 3;
                int l = i + (u >> 2);
                l = l < 0 ? l + NLx : (l >= NLx ? l - NLx : l);
                return (gw & 0x7FFFu) + (uint32_t)((u & 3) * NLx + l);
            };
            uint32_t A = 0, B = 0;
            if (active) {
                A = st0[pos(gd[0])].x >> kWordSp;
                B = st0[pos(gd[1])].x >> kWordSp;
                if (A == B) ++accN;  // dE = 0: accepted, nothing changes
            }
            const bool live = A != B;
            if (__any_sync(0xffffffffu, live)) {
                uint32_t at[kPer], nw[kPer];
                float nf[kPer], df[kPer];
#pragma unroll
                for (int k = 0; k < kPer; ++k) {
                    at[k] = nw[k] = 0;
                    nf[k] = 0.f;
                }
                if (live) {
                    const uint32_t *ra = base + 4 * A, *rb = base + 4 * B;
#pragma unroll
                    for (int k = 0; k < kPer; ++k) {
                        const uint32_t gw = gd[kLanes * k + sl];
                        at[k] = pos(gw);
                        uint32_t w = st0[at[k]].x;
                        w = table_move(w, (gw >> 18) & 3u, mv, ra, rb + 32);  // the shell that sees a: A -> B
                        w = table_move(w, gw >> 20, mv, rb, ra + 32);         // the shell that sees b: B -> A
                        if (k == 0 && sl < 2)  // a, b themselves
                            w = (w & ((1u << kWordSp) - 1u)) | (sl == 0 ? B : A) << kWordSp;
                        nw[k] = w;
                        nf[k] = __ldg(P.table + word_index<SPLIT>(P.d, w));
                    }
                }
#pragma unroll
                for (int k = 0; k < kPer; ++k) df[k] = live ? nf[k] - __uint_as_float(st0[at[k]].y) : 0.f;
                // dE in zone order, every lane of the trial
                float dE = 0.f;
#pragma unroll
                for (int e = 0; e < kOmega; ++e) dE += __shfl_sync(0xffffffffu, df[e / kLanes], e % kLanes, kLanes);
                const uint32_t wa = HAS_PAIR ? __shfl_sync(0xffffffffu, nw[0], 0, kLanes) : 0u,
                               wb = HAS_PAIR ? __shfl_sync(0xffffffffu, nw[0], 1, kLanes) : 0u;
                if (live) {
                    if (HAS_PAIR) {
                        int ha[3], hb[3];
#pragma unroll
                        for (int m = 0; m < 3; ++m) {
                            ha[m] = (int)__ldg(P.unrank + P.d.un[m] + ((wa >> word_sh(m)) & word_mask(m)));
                            hb[m] = (int)__ldg(P.unrank + P.d.un[m] + ((wb >> word_sh(m)) & word_mask(m)));
                        }
                        dE += pair_part(Dt, P.nshells, P.d.S, ha, hb, (int)A, (int)B);
                    }
                    if (metropolis<false>(dE, word & kRMask, P.beta, nullptr, make_int2(0, 0))) {
#pragma unroll
                        for (int k = 0; k < kPer; ++k) st0[at[k]] = make_uint2(nw[k], __float_as_uint(nf[k]));
                        if (sl < 2) {
                            const int o = sl == 0 ? 0 : (sub == 0 ? -1 : 0), kk = sl == 0 ? 0 : dir;
                            const int y = wrapc(y0 + o + ((kk >> 1) & 1), ny), z = wrapc(z0 + o + (kk & 1), nz),
                                      xs = wrapc(4 * i + dx + o + (kk >> 2), nx), ss = sl == 0 ? sub : 1 - sub;
                            P.occ[((ss * nz + z) * ny + y) * nx + xs] = (int8_t)(sl == 0 ? B : A);
                        }
                        accE += (double)dE;
                        ++accN;
                    }
                }
            }
            if (pairwise && dx < 3) {
                ++step;
                __syncwarp();
                if ((tid & 31) == 0)
                    asm volatile("st.release.cta.shared::cta.u32 [%0], %1;" ::"r"(mine), "r"(step) : "memory");
                if ((tid & 31) < 2 && !table_wait(look, step, P.timeout_ns))
                    atomicCAS(P.status, 0, (int)SMC_ERR_TIMEOUT);
                __syncwarp();
            } else {
                team_sync(team, tthr);
            }
        }
        for (int j = tt; j < kTabRows * quads; j += tthr) {
            const int r = j / quads, q = j - r * quads;
            ((uint4 *)(P.state + (size_t)rown[r] * nx))[q] = ((const uint4 *)rows)[j];
        }
        if (active && sl == 0) {
            const int lc = col * NLx + i;
            P.part_e[lc] += accE;
            P.part_n[lc] += accN;
        }
        team_sync(team, tthr);
    }
}

// Shared memory besides the teams'.
size_t table_sweep_fixed(const TableDims &d, bool pair)
{
    return (size_t)d.mv_total * 2 + (size_t)kOmega * 8 * 4 + kMoveBases * 4 + kTabThreads / 32 * 4 +
           (pair ? (size_t)kDEntries * 4 : 0);
}

template <class Net>
smc_status fill_launch(Workspace *ws, const void *W, const TableDims &d, const uint4 *rows, float *table,
                       const int *route, int *abort_flag, cudaStream_t stream)
{
    constexpr int NWG = Net::kFillNWG;
    const size_t smem = (Net::template Smem<NWG>::TINFO + 127) / 128 * 128;
    auto kern = k_table_fill<Net>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return cuda_fail(e, "cudaFuncSetAttribute(k_table_fill)");
    const long long tiles = (d.entries + kTcRows - 1) / kTcRows;
    const int grid = (int)std::max(1LL, std::min<long long>(ws->num_sms, (tiles + NWG - 1) / NWG));
    kern<<<grid, 128 * NWG, smem, stream>>>(W, d, rows, table, route, debug_timeout_ns(), ws->status, abort_flag);
    e = cudaGetLastError();
    return e == cudaSuccess ? SMC_OK : cuda_fail(e, "k_table_fill");
}

// The zone table of the sweep: offset of the row (table_row) in a column's
// rows in bits 0-14, dx + 3 in 15-17, the shells that see a and b in 18-19 and
// 20-21; [sub][dir][entry].
bool pack_zone(int nx, std::vector<uint32_t> &out)
{
    static MlpGeo G;
    if (!build_mlp_geo(G)) return false;
    out.assign(2 * kOmega * 8, 0);
    for (int s = 0; s < 2; ++s)
        for (int d = 0; d < 8; ++d)
            for (int e = 0; e < kOmega; ++e) {
                const OmegaEntry &o = G.om[s][d][e];
                const int base = o.rel ? (s == 0 ? -2 : -1) : -1, per = o.rel ? 4 : 3;
                const int qy = o.dy - base, qz = o.dz - base;
                if (qy < 0 || qy >= per || qz < 0 || qz >= per || o.dxo < -3 || o.dxo > 3) return false;
                if (o.mb && o.mb == o.ma) return false;
                out[(size_t)((s * 8 + d) * kOmega + e)] =
                    (uint32_t)(((o.rel ? 9 : 0) + qy * per + qz) * nx | (o.dxo + 3) << 15 | o.ma << 18 | o.mb << 20);
            }
    return true;
}

// ---------------------------------------------------------------------------
// The choice between evaluating and tabulating.  Both times follow the share
// f of unlike first-shell bonds, since only trials of unlike species evaluate or
// look up: a column of n trials has f n of them per mini-step, and none with
// probability (1 - f)^n.  In us, fitted to 23 boxes of 8^3 to 256^3 cells (cubes,
// single columns and plates), two, four and five species, f = 0.02 to 0.8, to
// 12 % (root mean square):
//   evaluating  per mini-step of a column
//               1.65 + 1.55 (1 - (1 - f)^n) + 0.28 f n (MLPNet: 0.46 f n) + 0.0085 n,
//               columns one after the other on an SM;
//   tabulated   per group of a block's K columns (c0..c3)
//               c0 + c1 (1 - (1 - f)^n) + (c2 f + c3) K n,
//               and per call 37 ps per vector (the table) and 60 us (launches, copies).
// Over these boxes and calls of 1 to 5000 sweeps the slower route is taken, by
// more than 5 %, for 1 in 100; with the rows of an alloy in equal parts over the
// number of vectors alone it was 1 in 6.  Per call, evaluating / tabulated (ms):
//   256^3, 2 sweeps: Dirichlet fractions 122 / 84, 1 % of one solute 26 / 49
//   128^3, 12 sweeps: Dirichlet 102 / 78, two of five species 82 / 54, 1 % 26 / 49
//   32^3, 600 sweeps: equal fractions 389 / 566, 1 % 198 / 380; MLPNet 541 / 565
//   16^3, 10 sweeps of three species 5.1 / 5.4; 64^3 15.9 / 6.0
// f moves during a call (order sets in, or phases separate); the share at its
// start decides.
// ---------------------------------------------------------------------------
struct TableGain {  // of tabulating (us): g0 + g1 (1 - (1 - f)^n) + g2 f
    double g0, g1, g2, n;
    __host__ __device__ double at(double f) const { return g0 + g1 * (1.0 - pow(1.0 - f, n)) + g2 * f; }
};

TableGain table_gain(int S, bool net, int nsweeps, int NLx, int eval_passes, int table_passes, int K, double entries)
{
    static const double c[3][4] = {{10.6, 5.6, 0.05, 0.015}, {12.2, 5.5, 0.09, 0.0}, {14.7, 6.8, 0.26, 0.0}};
    const double *t = c[S <= 3 ? 0 : S - 3];
    const double ev = 128.0 * nsweeps * eval_passes, look = 32.0 * nsweeps * table_passes, kn = (double)K * NLx;
    return TableGain{ev * (1.65 + 0.0085 * NLx) - look * (t[0] + t[3] * kn) - 37e-6 * entries - 60.0,
                     ev * 1.55 - look * t[1], ev * (net ? 0.46 : 0.28) * NLx - look * t[2] * kn, (double)NLx};
}

// Unlike first-shell bonds, each once: sublattice 0's sites with their eight
// neighbours, four cells of a row (a word) at a time (512^3: 0.19 ms, 0.71 by bytes).
template <bool ALIGNED>
__device__ __forceinline__ uint32_t four_species(const int8_t *p)
{
    if (ALIGNED) return *(const uint32_t *)p & 0x07070707u;
    return (uint32_t)(p[0] & 7) | (uint32_t)(p[1] & 7) << 8 | (uint32_t)(p[2] & 7) << 16 | (uint32_t)(p[3] & 7) << 24;
}

template <bool ALIGNED>
__global__ void __launch_bounds__(256) k_unlike_bonds(const int8_t *__restrict__ occ, int nx, int ny, int nz,
                                                      unsigned long long *count)
{
    const uint32_t nw = (uint32_t)nx / 4, words = nw * ny * nz;  // rows are multiples of four cells; < 2^28
    const int8_t *other = occ + 4 * (size_t)words;
    uint32_t n = 0;
    for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < words; i += gridDim.x * blockDim.x) {
        const int w = (int)(i % nw), t = (int)(i / nw), y = t % ny, z = t / ny;
        const uint32_t a = four_species<ALIGNED>(occ + 4 * (size_t)i);
        const int left = w ? 4 * w - 1 : nx - 1;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int8_t *row = other + (size_t)(wrapc(z - (k >> 1), nz) * ny + wrapc(y - (k & 1), ny)) * nx;
            const uint32_t b = four_species<ALIGNED>(row + 4 * w), c = b << 8 | (uint32_t)(row[left] & 7);  // x, x - 1
            n += __popc(__vcmpne4(a, b)) + __popc(__vcmpne4(a, c));
        }
    }
    n = __reduce_add_sync(0xffffffffu, n / 8);  // eight bits per unlike pair
    if ((threadIdx.x & 31) == 0 && n) atomicAdd(count, (unsigned long long)n);
}

// The choice (1: tabulated), and for the host to see (echo, pinned) with the
// call's number: 2 call + choice.
__global__ void k_table_route(TableGain gain, double bonds, const unsigned long long *unlike, uint32_t call, int *route,
                              volatile uint32_t *echo)
{
    const int r = gain.at((double)*unlike / bonds) > 0.0 ? 1 : 0;
    *route = r;
    if (echo) *echo = 2u * call + (uint32_t)r;
}

// The host never waits for the choice: it looks before it enqueues each sweep,
// and what was enqueued before the word came ends at once where it is not
// needed.  (A look is a load: an event query would break a capture that another
// thread has under way.)
struct RouteEcho {
    uint32_t *word = nullptr;  // pinned
    uint32_t call = 0;         // 31 bits
};
RouteEcho *route_echo()
{
    static RouteEcho echo[64];
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev >= 64) return nullptr;
    RouteEcho &r = echo[dev];
    if (!r.word) {
        if (cudaHostAlloc((void **)&r.word, sizeof(uint32_t), cudaHostAllocDefault) != cudaSuccess) {
            cudaGetLastError();
            r.word = nullptr;
            return nullptr;
        }
        *r.word = 0;
    }
    r.call = (r.call + 1) & 0x7FFFFFFFu;
    return &r;
}

}  // namespace

smc_status launch_mlp_table_sweep(const smc_lattice *lat, const smc_model *m, int8_t *occ, uint64_t seed,
                                  uint32_t replica, uint64_t sweep0, int nsweeps, const double *kT, double *e_acc,
                                  int64_t *n_acc, const float *D, size_t least, int eval_passes, MlpTaken *taken,
                                  const int **route, cudaStream_t stream)
{
    *taken = kMlpEvaluate;
    *route = nullptr;
    const int fixed_route = debug_mlp_table();  // 0: chosen here; 1: evaluating; 2: tabulated where it fits
    if (lat->nspecies < 2 || fixed_route == 1) return SMC_OK;
    smc_status st;
    Workspace *ws = workspace(&st);
    if (!ws) return st;
    const TableHost &T = table_host(lat->nspecies);
    const bool pair = m->kind == SMC_PAIR_F32_MLP_BF16, net = m->kind == SMC_MLPNET_BF16;
    TableParams P;
    memset(&P, 0, sizeof P);
    P.d = T.d;
    P.nx = lat->nx;
    P.ny = lat->ny;
    P.nz = lat->nz;
    P.NLx = lat->nx / 4;
    P.NLy = lat->ny / 4;
    P.NLz = lat->nz / 4;
    P.ncol = P.NLy * P.NLz;
    // teams per block: what fits beside the tables, at most a block's threads, 15 barriers and an even share of the SMs
    const size_t fixed = table_sweep_fixed(T.d, pair), per = table_team_bytes(P.nx);
    P.team_threads = (kLanes * P.NLx + 31) / 32 * 32;
    if (fixed + per > ws->smem_optin || P.team_threads > kTabThreads) return SMC_OK;
    P.K = (int)std::min<size_t>((ws->smem_optin - fixed) / per,
                                std::min({kTabThreads / P.team_threads, 15, (P.ncol + ws->num_sms - 1) / ws->num_sms}));
    const size_t smem = fixed + per * (size_t)P.K;
    const int blocks = std::min(P.ncol, ws->num_sms), per_pass = blocks * P.K;
    const TableGain gain = table_gain(lat->nspecies, net, nsweeps, P.NLx, eval_passes,
                                      (P.ncol + per_pass - 1) / per_pass, P.K, (double)T.d.entries);
    // worth a look at the lattice if it would be for a random alloy in equal parts
    if (fixed_route == 0 && !(gain.at(1.0 - 1.0 / lat->nspecies) > 0.0)) return SMC_OK;
    const bool certain = fixed_route == 2 || (gain.g0 > 0.0 && gain.g1 >= 0.0 && gain.g2 >= 0.0);  // for any lattice
    P.nshells = pair ? m->nshells : 0;
    std::vector<uint32_t> zone;
    if (!pack_zone(P.nx, zone)) {
        set_error("internal error: MLP interaction-zone geometry");
        return SMC_ERR_STATE;
    }
    // workspace: [part_e | part_n | abort | weights | moves | ranks | packed counts | feature words | zone | D | state];
    // the table (4 bytes per vector, whatever the lattice) has a buffer of its own
    const size_t nc = (size_t)P.NLx * P.ncol, N = 2ull * lat->nx * lat->ny * lat->nz;
    auto up = [](size_t v) { return (v + 255) / 256 * 256; };
    const size_t o_pn = nc * 8, o_abort = o_pn + nc * 8, o_w = up(o_abort + 16), o_mv = up(o_w + kWeightBytes),
                 o_rk = up(o_mv + T.moves.size() * 2), o_un = up(o_rk + T.ranks.size() * 2),
                 o_rows = up(o_un + T.unrank.size() * 4), o_zone = up(o_rows + T.rows.size() * 4), o_D = up(o_zone + zone.size() * 4),
                 o_red = up(o_D + kDEntries * 4), o_state = up(o_red + lc_reduce_bytes()),
                 need = std::max(o_state + N * 8, least);
    unsigned char *scr = (unsigned char *)workspace_scratch(ws, need, &st);
    if (!scr) return out_of_memory() ? SMC_OK : st;  // no room beside the table: the evaluating sweep may have it
    void *table = nullptr;
    const size_t table_bytes = up((size_t)T.d.entries * 4);  // then the count and the route word
    const cudaError_t room = table_buffer(table_bytes + 16, &table);
    if (room == cudaErrorMemoryAllocation) return SMC_OK;
    if (room != cudaSuccess) return cuda_fail(room, "cudaMalloc(MLP table)");
    *taken = certain ? kMlpTabulate : kMlpEither;
    P.part_e = (double *)scr;
    P.part_n = (long long *)(scr + o_pn);
    P.occ = occ;
    P.state = (uint2 *)(scr + o_state);
    P.table = (const float *)table;
    P.moves = (const uint16_t *)(scr + o_mv);
    P.ranks = (const uint16_t *)(scr + o_rk);
    P.unrank = (const uint32_t *)(scr + o_un);
    P.geo = (const uint32_t *)(scr + o_zone);
    P.D = (const float *)(scr + o_D);
    P.seed = seed;
    P.replica = replica;
    P.status = ws->status;
    P.timeout_ns = debug_timeout_ns();
    cudaError_t e = cudaSuccess;
    RouteEcho *echo = nullptr;
    if (!certain) {
        unsigned long long *unlike = (unsigned long long *)((unsigned char *)table + table_bytes);
        int *word = (int *)(unlike + 1);
        e = cudaMemsetAsync(unlike, 0, 16, stream);
        if (e != cudaSuccess) return cuda_fail(e, "cudaMemsetAsync(unlike bonds)");
        const int cb = (int)std::max<size_t>(1, std::min<size_t>((N / 8 + 255) / 256, (size_t)ws->num_sms * 8));
        if ((uintptr_t)occ % 4 == 0)
            k_unlike_bonds<true><<<cb, 256, 0, stream>>>(occ, P.nx, P.ny, P.nz, unlike);
        else
            k_unlike_bonds<false><<<cb, 256, 0, stream>>>(occ, P.nx, P.ny, P.nz, unlike);
        echo = route_echo();
        k_table_route<<<1, 1, 0, stream>>>(gain, 4.0 * (double)N, unlike, echo ? echo->call : 0u, word,
                                           echo ? echo->word : nullptr);
        e = cudaGetLastError();
        if (e != cudaSuccess) return cuda_fail(e, "k_table_route");
        P.route = *route = word;
    }
    // looks whether the route is known by now; false: the rest of the tabulated sweep is not needed
    auto go_on = [&]() {
        if (*taken != kMlpEither || !echo) return true;
        const uint32_t w = *(volatile uint32_t *)echo->word;
        if (w >> 1 == echo->call) *taken = w & 1u ? kMlpTabulate : kMlpEvaluate;
        return *taken != kMlpEvaluate;
    };
    st = mlp_copy_weights(m, scr + o_w, stream);
    if (st != SMC_OK) return st;
    e = cudaMemsetAsync(scr, 0, o_abort + 16, stream);
    // (in pieces: a copy of more than 64 KB of pageable memory waits for the work ahead of it on the stream)
    auto put = [&](size_t off, const void *src, size_t bytes) {
        for (size_t o = 0; o < bytes && e == cudaSuccess; o += 32768)
            e = cudaMemcpyAsync(scr + off + o, (const char *)src + o, std::min<size_t>(32768, bytes - o),
                                cudaMemcpyHostToDevice, stream);
    };
    put(o_mv, T.moves.data(), T.moves.size() * 2);
    put(o_rk, T.ranks.data(), T.ranks.size() * 2);
    put(o_un, T.unrank.data(), T.unrank.size() * 4);
    put(o_rows, T.rows.data(), T.rows.size() * 4);
    put(o_zone, zone.data(), zone.size() * 4);
    if (pair) put(o_D, D, kDEntries * 4);
    if (e != cudaSuccess) return cuda_fail(e, "cudaMemcpyAsync(MLP table sweep)");
    st = net ? fill_launch<NetRelu96>(ws, scr + o_w, T.d, (const uint4 *)(scr + o_rows), (float *)table, P.route, (int *)(scr + o_abort), stream)
             : fill_launch<NetSilu64>(ws, scr + o_w, T.d, (const uint4 *)(scr + o_rows), (float *)table, P.route, (int *)(scr + o_abort), stream);
    if (st != SMC_OK) return st;
    const int sb = (int)std::max<size_t>(1, std::min<size_t>((N + 255) / 256, (size_t)ws->num_sms * 64));
    k_table_state<<<sb, 256, 0, stream>>>(P);
    e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_fail(e, "k_table_state");
    auto kern = T.d.S == 5 ? (pair ? k_table_sweep<true, true> : k_table_sweep<false, true>)
                           : (pair ? k_table_sweep<true, false> : k_table_sweep<false, false>);
    e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return cuda_fail(e, "cudaFuncSetAttribute(k_table_sweep)");
    const int threads = P.team_threads * P.K;
    for (int t = 0; t < nsweeps; ++t) {
        if (!go_on()) return SMC_OK;
        P.sweep = sweep0 + (uint64_t)t;
        P.beta = (float)(1.0 / kT[t]);
        for (int g = 0; g < 32; ++g) {
            P.g = g;
            kern<<<blocks, threads, smem, stream>>>(P);
        }
        e = cudaGetLastError();
        if (e != cudaSuccess) return cuda_fail(e, "k_table_sweep");
    }
    if (!go_on()) return SMC_OK;
    if (e_acc || n_acc)  // (sums of zeros where the sweep was not needed)
        return launch_lc_reduce(P.part_e, P.part_n, (long long)nc, scr + o_red, e_acc, (long long *)n_acc, stream);
    return SMC_OK;
}

}  // namespace smc

// planes.cu -- neighbour counts from species bit planes, for both lattices and
// rows of any length: ordered pair counts n_m^{pq}, the own-species counts of
// every site (the qSRO sweeps' cache) and the sums Q_m^p of their squares.
//
// A word of a row holds 32 consecutive cells; plane k bit i is bit k of the
// species of cell i.  The cells past the end of a row's last word repeat the
// row from its start, so that the word of the cells x + 1 is a funnel shift
// everywhere.  Against byte-wise kernels that visit every neighbour of every
// site this takes a few instructions per neighbour and 32 sites:
//   pairs      popc((M_p & N_q) | (M_q & N_p)) per unordered species pair and
//              visited vector (half of each shell, as in observables.cu)
//   own counts bit-sliced counters of the words that agree in all planes
//   squares    sum over sites of species p of c^2 = sum_{i,j} 2^(i+j)
//              popc(b_i & b_j & M_p) over the counters' bits
// 2 shells, 5 species: pair counts of 256^3 FCC cells 2.40 -> 0.125 ms with the
// planes' own pass; own-count cache of 128^3 FCC cells 0.25 -> 0.023 ms, of
// 256^3 BCC cells 0.80 -> 0.060, squares there 0.93 -> 0.067.
#include <algorithm>
#include <cstring>

#include "planes.cuh"

namespace smc {

namespace {

// Vector t of a shell list from a site of sublattice s: target sublattice and
// cell offsets (+ 2) packed as nsub | dx << 4 | dy << 8 | dz << 12; the visited
// half of each shell (first non-zero component of the vector positive) first.
struct VecSet {
    uint32_t v[4][42];
};
__constant__ VecSet c_vec[2];  // by PlaneLattice

__host__ __device__ constexpr int shell_size(int lat, int m)
{
    return lat == 0 ? (m == 0 ? 8 : (m == 1 ? 6 : 12)) : (m == 0 ? 12 : (m == 1 ? 6 : 24));
}
__host__ __device__ constexpr int shell_first(int lat, int m)
{
    return m == 0 ? 0 : (m == 1 ? shell_size(lat, 0) : shell_size(lat, 0) + shell_size(lat, 1));
}

// Bits of the count of shell m (at most 8, 6, 12 / 12, 6, 24 neighbours) and
// its position in the cache entry.
__host__ __device__ constexpr int count_bits(int lat, int m) { return m == 1 ? 3 : (lat == 1 && m == 2 ? 5 : 4); }
__host__ __device__ constexpr int count_pos(int m) { return m == 0 ? 0 : (m == 1 ? 4 : 7); }

__global__ void __launch_bounds__(256) k_planes_rows(const int8_t *__restrict__ occ, int nx, int nw, long long nwords,
                                                     uint4 *__restrict__ planes)
{
    const int lane = threadIdx.x & 31;
    const long long nwarps = (long long)gridDim.x * (blockDim.x >> 5);
    for (long long t = (long long)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); t < nwords; t += nwarps) {
        const long long row = t / nw;
        const int w = (int)(t - row * nw), x = 32 * w + lane;
        const int v = __ldg(occ + row * nx + (x < nx ? x : x % nx));
        const uint32_t a = __ballot_sync(0xffffffffu, v & 1), b = __ballot_sync(0xffffffffu, v & 2),
                       c = __ballot_sync(0xffffffffu, v & 4);
        if (lane == 0) planes[t] = make_uint4(a, b, c, 0u);
    }
}

// A word's place, and the words of its neighbours.
struct PlaneView {
    const uint4 *planes;
    int nw, ny, nz, last;  // last: cells of a row's last word (1-32)
    int sub, y, z, w;
    __device__ __forceinline__ uint4 at(uint32_t row, int ww) const { return __ldg(planes + (size_t)row * nw + ww); }
    __device__ __forceinline__ uint4 neighbour(uint32_t v) const
    {
        const int dx = (int)((v >> 4) & 15u) - 2, dy = (int)((v >> 8) & 15u) - 2, dz = (int)((v >> 12) & 15u) - 2;
        const uint32_t row = ((v & 3u) * (uint32_t)nz + (uint32_t)wrapc(z + dz, nz)) * (uint32_t)ny + (uint32_t)wrapc(y + dy, ny);
        const uint4 c = at(row, w);
        if (dx == 0) return c;
        if (dx > 0) {  // cells x + 1
            const uint4 n = at(row, w + 1 < nw ? w + 1 : 0);
            // (the last word of a ragged row continues with the row's start by itself)
            const bool own = w + 1 == nw && last < 32;
            const uint32_t k = 1u;
            return own ? make_uint4(c.x >> k, c.y >> k, c.z >> k, 0u)
                       : make_uint4(__funnelshift_r(c.x, n.x, k), __funnelshift_r(c.y, n.y, k), __funnelshift_r(c.z, n.z, k), 0u);
        }
        uint4 p = at(row, w > 0 ? w - 1 : nw - 1);  // cells x - 1
        if (w == 0 && last < 32) {
            const int s = 32 - last;
            p = make_uint4(p.x << s, p.y << s, p.z << s, 0u);
        }
        return make_uint4(__funnelshift_l(p.x, c.x, 1), __funnelshift_l(p.y, c.y, 1), __funnelshift_l(p.z, c.z, 1), 0u);
    }
    __device__ __forceinline__ uint32_t valid() const { return w + 1 == nw && last < 32 ? (1u << last) - 1u : 0xffffffffu; }
};

__device__ __forceinline__ PlaneView plane_view(const uint4 *planes, int nx, int ny, int nz, long long t)
{
    PlaneView V;
    V.planes = planes;
    V.nw = (nx + 31) / 32;
    V.ny = ny;
    V.nz = nz;
    V.last = nx - 32 * (V.nw - 1);
    const uint32_t row = (uint32_t)(t / V.nw);
    V.w = (int)(t - (long long)row * V.nw);
    const uint32_t q = row / (uint32_t)ny;
    V.y = (int)(row - q * (uint32_t)ny);
    V.sub = (int)(q / (uint32_t)nz);
    V.z = (int)(q - (uint32_t)V.sub * (uint32_t)nz);
    return V;
}

template <int S>
__device__ __forceinline__ void masks(const uint4 &w, uint32_t (&M)[S])
{
#pragma unroll
    for (int p = 0; p < S; ++p) M[p] = ((p & 1) ? w.x : ~w.x) & ((p & 2) ? w.y : ~w.y) & ((p & 4) ? w.z : ~w.z);
}

// Ordered pair counts of shells M0 .. M1-1.
template <int LAT, int M0, int M1, int S>
__global__ void __launch_bounds__(256) k_plane_pairs(const uint4 *__restrict__ planes, int nx, int ny, int nz,
                                                     unsigned long long *counts)
{
    constexpr int NP = S * (S + 1) / 2, NM = M1 - M0;
    __shared__ unsigned long long bins[NM * NP];
    for (int i = threadIdx.x; i < NM * NP; i += blockDim.x) bins[i] = 0;
    __syncthreads();
    uint32_t acc[NM][NP];  // p < q: n^{pq}; p = q: n^{pp} / 2
#pragma unroll
    for (int m = 0; m < NM; ++m)
#pragma unroll
        for (int k = 0; k < NP; ++k) acc[m][k] = 0u;
    const long long total = (long long)(LAT == 0 ? 2 : 4) * ny * nz * ((nx + 31) / 32);
    for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < total;
         t += (long long)gridDim.x * blockDim.x) {
        const PlaneView V = plane_view(planes, nx, ny, nz, t);
        const uint32_t ok = V.valid();
        uint32_t A[S];
        masks<S>(__ldg(planes + t), A);
#pragma unroll
        for (int p = 0; p < S; ++p) A[p] &= ok;
#pragma unroll
        for (int m = M0; m < M1; ++m)
            for (int i = 0; i < shell_size(LAT, m) / 2; ++i) {
                uint32_t B[S];
                masks<S>(V.neighbour(c_vec[LAT].v[V.sub][shell_first(LAT, m) + i]), B);
                int k = 0;
#pragma unroll
                for (int p = 0; p < S; ++p) {
                    acc[m - M0][k++] += __popc(A[p] & B[p]);
#pragma unroll
                    for (int q = p + 1; q < S; ++q) acc[m - M0][k++] += __popc((A[p] & B[q]) | (A[q] & B[p]));
                }
            }
    }
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int m = 0; m < NM; ++m)
#pragma unroll
        for (int k = 0; k < NP; ++k) {
            const unsigned v = __reduce_add_sync(0xffffffffu, acc[m][k]);
            if (lane == 0 && v) atomicAdd(&bins[m * NP + k], (unsigned long long)v);
        }
    __syncthreads();
    for (int i = threadIdx.x; i < NM * S * S; i += blockDim.x) {
        const int m = i / (S * S), p = (i / S) % S, q = i % S;
        const int a = p < q ? p : q, b = p < q ? q : p;
        const unsigned long long v = bins[m * NP + a * S - a * (a - 1) / 2 + (b - a)];
        if (v) atomicAdd(counts + M0 * S * S + i, p == q ? 2 * v : v);
    }
}

// Own-species counts of every site: the cache entries (ES bytes per site: bit
// fields of the shells), and with QUAD the sums of squares per shell and
// species ([shell][8], added).
template <int LAT, int NSH, bool QUAD>
__global__ void __launch_bounds__(256) k_plane_own(const uint4 *__restrict__ planes, int nx, int ny, int nz, void *cache,
                                                   unsigned long long *quad)
{
    constexpr int ES = NSH == 3 ? 2 : 1;
    __shared__ unsigned long long bins[QUAD ? NSH * 8 : 1];
    uint32_t sq[QUAD ? NSH : 1][8];
    if (QUAD) {
        for (int i = threadIdx.x; i < NSH * 8; i += blockDim.x) bins[i] = 0;
        __syncthreads();
#pragma unroll
        for (int m = 0; m < NSH; ++m)
#pragma unroll
            for (int p = 0; p < 8; ++p) sq[m][p] = 0u;
    }
    const long long total = (long long)(LAT == 0 ? 2 : 4) * ny * nz * ((nx + 31) / 32);
    // whole warps take each turn (the reduction below follows the loop)
    for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < total;
         t += (long long)gridDim.x * blockDim.x) {
        const PlaneView V = plane_view(planes, nx, ny, nz, t);
        const uint4 a = __ldg(planes + t);
        uint32_t bits[12];  // the cache entry's bits, each for 32 sites
#pragma unroll
        for (int k = 0; k < 12; ++k) bits[k] = 0u;
#pragma unroll
        for (int m = 0; m < NSH; ++m) {
            uint32_t c[5] = {0u, 0u, 0u, 0u, 0u};
            constexpr int kBits = 5;
#pragma unroll 6
            for (int i = 0; i < shell_size(LAT, m); ++i) {
                const uint4 b = V.neighbour(c_vec[LAT].v[V.sub][shell_first(LAT, m) + i]);
                uint32_t e = ~((a.x ^ b.x) | (a.y ^ b.y) | (a.z ^ b.z));
#pragma unroll
                for (int k = 0; k < kBits; ++k) {
                    if (k >= count_bits(LAT, m)) break;
                    const uint32_t carry = c[k] & e;
                    c[k] ^= e;
                    e = carry;
                }
            }
#pragma unroll
            for (int k = 0; k < kBits; ++k)
                if (k < count_bits(LAT, m)) bits[count_pos(m) + k] = c[k];
            if (QUAD) {
                uint32_t M[8];
                masks<8>(a, M);
                const uint32_t ok = V.valid();
#pragma unroll
                for (int p = 0; p < 8; ++p) {
                    const uint32_t mp = M[p] & ok;
                    if (mp == 0u) continue;
                    uint32_t s = 0;
#pragma unroll
                    for (int i = 0; i < kBits; ++i)
#pragma unroll
                        for (int j = i; j < kBits; ++j)
                            if (j < count_bits(LAT, m)) s += (uint32_t)__popc(c[i] & c[j] & mp) << (i + j + (j > i));
                    sq[m][p] += s;
                }
            }
        }
        if (cache) {
            const uint32_t row = (uint32_t)(t / V.nw);
            unsigned char *dst = (unsigned char *)cache + ((size_t)row * nx + 32 * V.w) * ES;
            const int n = V.w + 1 == V.nw ? V.last : 32;  // rows are multiples of four cells
            if (ES == 1) {
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    uint32_t o = 0;
#pragma unroll
                    for (int k = 0; k < 7; ++k) o |= ((((bits[k] >> (4 * j)) & 15u) * 0x00204081u) & 0x01010101u) << k;
                    if (4 * j < n) *(uint32_t *)(dst + 4 * j) = o;
                }
            } else {
#pragma unroll
                for (int j = 0; j < 16; ++j) {
                    uint32_t o = 0;
#pragma unroll
                    for (int k = 0; k < 12; ++k) o |= ((((bits[k] >> (2 * j)) & 3u) * 0x8001u) & 0x00010001u) << k;
                    if (2 * j < n) *(uint32_t *)(dst + 4 * j) = o;
                }
            }
        }
    }
    if (QUAD) {
        const int lane = threadIdx.x & 31;
        __syncwarp();
#pragma unroll
        for (int m = 0; m < NSH; ++m)
#pragma unroll
            for (int p = 0; p < 8; ++p) {
                const unsigned v = __reduce_add_sync(0xffffffffu, sq[m][p]);
                if (lane == 0 && v) atomicAdd(&bins[m * 8 + p], (unsigned long long)v);
            }
        __syncthreads();
        for (int i = threadIdx.x; i < NSH * 8; i += blockDim.x)
            if (bins[i]) atomicAdd(quad + i, bins[i]);
    }
}

bool g_vec_ready[64];

// The vector tables of both lattices, in half units from a site of sublattice
// s: BCC (+-1)^3, (+-2, 0, 0), (+-2, +-2, 0); FCC of squared length 2, 4, 6
// with an even component sum.
smc_status vec_tables()
{
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return cuda_fail(e, "cudaGetDevice");
    if (dev < 64 && g_vec_ready[dev]) return SMC_OK;
    static const int fcc[4][3] = {{0, 0, 0}, {1, 1, 0}, {1, 0, 1}, {0, 1, 1}};
    VecSet h[2];
    memset(h, 0, sizeof h);
    for (int lat = 0; lat < 2; ++lat)
        for (int s = 0; s < (lat == 0 ? 2 : 4); ++s)
            for (int m = 0; m < 3; ++m) {
                int n = shell_first(lat, m);
                for (int half = 0; half < 2; ++half)
                    for (int x = -2; x <= 2; ++x)
                        for (int y = -2; y <= 2; ++y)
                            for (int z = -2; z <= 2; ++z) {
                                const int d2 = x * x + y * y + z * z;
                                const bool in = lat == 0 ? (((x & 1) == (y & 1) && (y & 1) == (z & 1)) &&
                                                            d2 == (m == 0 ? 3 : (m == 1 ? 4 : 8)))
                                                         : (d2 == 2 * (m + 1) && ((x + y + z) & 1) == 0);
                                const bool first = x > 0 || (x == 0 && (y > 0 || (y == 0 && z > 0)));
                                if (!in || first != (half == 0)) continue;
                                int q[3] = {x, y, z}, ns = 0;
                                if (lat == 0) {
                                    for (int &v : q) v += s;
                                    ns = q[0] & 1;
                                } else {
                                    for (int k = 0; k < 3; ++k) q[k] += fcc[s][k];
                                    while (fcc[ns][0] != (q[0] & 1) || fcc[ns][1] != (q[1] & 1) || fcc[ns][2] != (q[2] & 1)) ++ns;
                                }
                                h[lat].v[s][n++] = (uint32_t)(ns | (floor_half(q[0]) + 2) << 4 | (floor_half(q[1]) + 2) << 8 |
                                                              (floor_half(q[2]) + 2) << 12);
                            }
                if (n != shell_first(lat, m) + shell_size(lat, m)) {
                    set_error("internal error: shell vectors");
                    return SMC_ERR_STATE;
                }
            }
    e = cudaMemcpyToSymbol(c_vec, h, sizeof h);
    if (e != cudaSuccess) return cuda_fail(e, "cudaMemcpyToSymbol(shell vectors)");
    if (dev < 64) g_vec_ready[dev] = true;
    return SMC_OK;
}

template <int LAT, int M0, int M1>
bool pairs_launch(const Planes &P, int blocks, int S, unsigned long long *counts, cudaStream_t stream)
{
#define SMC_PP(s)                                                                                                   \
    case s: k_plane_pairs<LAT, M0, M1, s><<<blocks, 256, 0, stream>>>(P.words, P.nx, P.ny, P.nz, counts); return true;
    switch (S) {
        SMC_PP(1) SMC_PP(2) SMC_PP(3) SMC_PP(4) SMC_PP(5) SMC_PP(6) SMC_PP(7) SMC_PP(8)
    }
#undef SMC_PP
    return false;
}

template <int LAT, int NSH>
void own_launch(const Planes &P, int blocks, void *cache, unsigned long long *quad, cudaStream_t stream)
{
    if (quad)
        k_plane_own<LAT, NSH, true><<<blocks, 256, 0, stream>>>(P.words, P.nx, P.ny, P.nz, cache, quad);
    else
        k_plane_own<LAT, NSH, false><<<blocks, 256, 0, stream>>>(P.words, P.nx, P.ny, P.nz, cache, quad);
}

}  // namespace

// The planes' buffer: one per device, grown when needed, kept apart from the
// workspace's scratch (which the callers already use for the counts).  NULL, with nothing
// changed, without memory or when a captured stream would have to grow it
// (*st = SMC_OK), and on any other error (*st).
// Graphs may hold the buffer of the pair counts of aligned rows (0), so other
// calls, never captured, grow one of their own (1).
void *planes_buffer(int which, size_t bytes, smc_status *st, cudaStream_t stream)
{
    Workspace *ws = workspace(st);
    if (!ws) return nullptr;
    auto &p = ws->planes[which];
    if (bytes > p.cap) {
        if (stream_capturing(stream)) return nullptr;
        void *buf = nullptr;
        cudaError_t e = cudaDeviceSynchronize();
        if (e == cudaSuccess) e = device_alloc(&buf, bytes);
        if (e == cudaErrorMemoryAllocation) return nullptr;
        if (e != cudaSuccess) {
            *st = cuda_fail(e, "cudaMalloc(planes)");
            return nullptr;
        }
        release(p.buf, p.held);
        p.buf = buf;
        p.cap = bytes;
        p.held = false;
    }
    if (call_captured()) p.held = true;
    return p.buf;
}

bool planes_build(PlaneLattice lat, int nx, int ny, int nz, const int8_t *occ, int num_sms, Planes &P, smc_status *st,
                  cudaStream_t stream)
{
    *st = SMC_OK;
    if (stream_capturing(stream)) return false;
    *st = vec_tables();
    if (*st != SMC_OK) return false;
    P.nx = nx;
    P.ny = ny;
    P.nz = nz;
    P.lat = lat;
    P.num_sms = num_sms;
    const long long rows = (long long)(lat == kPlanesBcc ? 2 : 4) * ny * nz;
    const int nw = (nx + 31) / 32;
    uint4 *words = (uint4 *)planes_buffer(1, (size_t)(rows * nw) * sizeof(uint4), st, stream);
    if (!words) return false;
    P.words = words;
    if (nx % 32 == 0 && (uintptr_t)occ % 16 == 0) {
        launch_planes_aligned(occ, rows * nw, words, num_sms, stream);
    } else {
        const int blocks = (int)std::max(1LL, std::min<long long>((rows * nw + 7) / 8, (long long)num_sms * 32));
        k_planes_rows<<<blocks, 256, 0, stream>>>(occ, nx, nw, rows * nw, words);
    }
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) {
        *st = cuda_fail(e, "k_planes");
        return false;
    }
    return true;
}

smc_status planes_pairs(const Planes &P, int nsh, int S, unsigned long long *counts, cudaStream_t stream)
{
    const long long words = (long long)(P.lat == kPlanesBcc ? 2 : 4) * P.ny * P.nz * ((P.nx + 31) / 32);
    const int blocks = (int)std::max(1LL, std::min<long long>((words + 255) / 256, (long long)P.num_sms * 4));
    bool ok = true;
    // (three shells of eight species would take 108 counters per thread: the third shell goes alone)
    if (P.lat == kPlanesBcc) {
        if (nsh == 1) ok = pairs_launch<0, 0, 1>(P, blocks, S, counts, stream);
        if (nsh >= 2) ok = pairs_launch<0, 0, 2>(P, blocks, S, counts, stream);
        if (nsh == 3) ok = ok && pairs_launch<0, 2, 3>(P, blocks, S, counts, stream);
    } else {
        if (nsh == 1) ok = pairs_launch<1, 0, 1>(P, blocks, S, counts, stream);
        if (nsh >= 2) ok = pairs_launch<1, 0, 2>(P, blocks, S, counts, stream);
        if (nsh == 3) ok = ok && pairs_launch<1, 2, 3>(P, blocks, S, counts, stream);
    }
    if (!ok) {
        set_error("internal error: pair counts of %d species", S);
        return SMC_ERR_STATE;
    }
    const cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? SMC_OK : cuda_fail(e, "k_plane_pairs");
}

smc_status planes_own(const Planes &P, int nsh, void *cache, unsigned long long *quad, cudaStream_t stream)
{
    const long long words = (long long)(P.lat == kPlanesBcc ? 2 : 4) * P.ny * P.nz * ((P.nx + 31) / 32);
    const int blocks = (int)std::max(1LL, std::min<long long>((words + 255) / 256, (long long)P.num_sms * 8));
    if (P.lat == kPlanesBcc) {
        if (nsh == 1) own_launch<0, 1>(P, blocks, cache, quad, stream);
        if (nsh == 2) own_launch<0, 2>(P, blocks, cache, quad, stream);
        if (nsh == 3) own_launch<0, 3>(P, blocks, cache, quad, stream);
    } else {
        if (nsh == 1) own_launch<1, 1>(P, blocks, cache, quad, stream);
        if (nsh == 2) own_launch<1, 2>(P, blocks, cache, quad, stream);
        if (nsh == 3) own_launch<1, 3>(P, blocks, cache, quad, stream);
    }
    const cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? SMC_OK : cuda_fail(e, "k_plane_own");
}

}  // namespace smc

// init.cu -- composition-conserving random initial configuration.
//
// Definition: sites ordered by the compound key K(s) = (k64(s), s), with
// k64(s) = (hi(s) << 32) | lo(s), hi/lo the Philox words of site s at the two
// reserved sweep indices; the sites at sorted positions [C_{p}, C_{p+1}) get
// species p (C = cumulative counts).
//
// No sort is needed: species(s) = #{t : K(s) >= T_t}, where T_t is the
// element of rank C_t.  The leading word hi is enough for nearly every site,
// so each of three passes over the sites computes one Philox block per four
// sites: a histogram of the leading 11 bits of hi, which gives the bin of every
// T_t; the collection of the sites in those bins (N / 2048 each) with their
// whole keys; and, after T_t is selected from its list, the assignment, which
// computes lo only where hi equals that of a T_t.  (A radix select over the 12
// bytes of K, recomputing both words in each of 12 passes, took 558 us for
// 4.2e6 sites and 8 species against 60 us.)
#include <algorithm>
#include <cstring>

#include "smc_common.cuh"

namespace smc {

constexpr int kMaxTargets = kMaxSpecies - 1;

constexpr int kInitBits = 11, kInitBins = 1 << kInitBits;

struct Threshold {
    unsigned long long k64;
    unsigned s;
    unsigned rank;   // rank still to skip inside the bin
    int bin;         // leading bits of hi
    int list;        // candidate list (targets of one bin share it)
    int active;      // 0: beyond the last site
    unsigned count;  // entries of list `t` (as a list, not as a target)
};
struct InitState {
    Threshold t[kMaxTargets];
    unsigned hist[kInitBins];
};

__device__ __forceinline__ U4 site_hi(uint64_t seed, uint32_t rep, uint32_t q)
{
    return philox10(U4{q, rep, 0xFFFFFFFEu, 0xFFFFFFFFu}, (uint32_t)seed, (uint32_t)(seed >> 32));
}
__device__ __forceinline__ U4 site_lo(uint64_t seed, uint32_t rep, uint32_t q)
{
    return philox10(U4{q, rep, 0xFFFFFFFFu, 0xFFFFFFFFu}, (uint32_t)seed, (uint32_t)(seed >> 32));
}

__global__ void __launch_bounds__(512) k_init_hist(uint64_t seed, uint32_t rep, long long N, InitState *st)
{
    __shared__ unsigned h[kInitBins];
    for (int i = threadIdx.x; i < kInitBins; i += blockDim.x) h[i] = 0;
    __syncthreads();
    const long long nq = (N + 3) / 4;
    for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < nq; q += (long long)gridDim.x * blockDim.x) {
        const U4 hi = site_hi(seed, rep, (uint32_t)q);
#pragma unroll
        for (int i = 0; i < 4; ++i)
            if (4 * q + i < N) atomicAdd(&h[pick_word(hi, i) >> (32 - kInitBits)], 1u);
    }
    __syncthreads();
    for (int i = threadIdx.x; i < kInitBins; i += blockDim.x)
        if (h[i]) atomicAdd(st->hist + i, h[i]);
}

// The bin and the rank inside it of every target (one block of kInitBins / 2 threads).
__global__ void __launch_bounds__(kInitBins / 2) k_init_bins(int ntarget, InitState *st)
{
    __shared__ unsigned sum[kInitBins / 2];
    const int i = threadIdx.x;
    const unsigned a = st->hist[2 * i], b = st->hist[2 * i + 1];
    sum[i] = a + b;
    __syncthreads();
    for (int o = 1; o < kInitBins / 2; o <<= 1) {
        const unsigned v = i >= o ? sum[i - o] : 0u;
        __syncthreads();
        sum[i] += v;
        __syncthreads();
    }
    const unsigned before = sum[i] - a - b;
    for (int t = 0; t < ntarget; ++t) {
        Threshold &T = st->t[t];
        if (!T.active) continue;
        const unsigned r = T.rank;
        __syncthreads();
        if (r >= before && r < before + a) {
            T.bin = 2 * i;
            T.rank = r - before;
        } else if (r >= before + a && r < before + a + b) {
            T.bin = 2 * i + 1;
            T.rank = r - before - a;
        }
        __syncthreads();
    }
    if (i == 0)
        for (int t = 0; t < ntarget; ++t) {
            Threshold &T = st->t[t];
            T.list = t;
            T.count = 0;
            for (int u = t - 1; u >= 0; --u)
                if (T.active && st->t[u].active && st->t[u].bin == T.bin) T.list = u;
        }
}

struct Candidate {
    unsigned hi, lo, s;
};

// Appends every site of a target's bin to the bin's list.
__global__ void __launch_bounds__(256) k_init_collect(uint64_t seed, uint32_t rep, long long N, int ntarget,
                                                      InitState *st, Candidate *lists, unsigned cap)
{
    __shared__ int bin[kMaxTargets];
    if (threadIdx.x < ntarget) {
        const Threshold &T = st->t[threadIdx.x];
        bin[threadIdx.x] = T.active && T.list == (int)threadIdx.x ? T.bin : -1;
    }
    __syncthreads();
    const long long nq = (N + 3) / 4;
    for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < nq; q += (long long)gridDim.x * blockDim.x) {
        const U4 hi = site_hi(seed, rep, (uint32_t)q);
        for (int t = 0; t < ntarget; ++t) {
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const uint32_t h = pick_word(hi, i);
                if ((int)(h >> (32 - kInitBits)) != bin[t] || 4 * q + i >= N) continue;
                const U4 lo = site_lo(seed, rep, (uint32_t)q);
                const unsigned k = atomicAdd(&st->t[t].count, 1u);
                if (k < cap) lists[(size_t)t * cap + k] = Candidate{h, pick_word(lo, i), (unsigned)(4 * q + i)};
            }
        }
    }
}

// Target blockIdx.x: the element of its rank among its list, by bytes of the
// 96-bit key from the top until one element is left.
__global__ void __launch_bounds__(1024) k_init_select(InitState *st, const Candidate *lists, unsigned cap, int *status)
{
    __shared__ unsigned h[256];
    __shared__ unsigned s_byte, s_rank, s_left;
    Threshold &T = st->t[blockIdx.x];
    if (!T.active) return;
    const unsigned n = st->t[T.list].count;
    const Candidate *L = lists + (size_t)T.list * cap;
    if (n > cap || n <= T.rank) {  // (a bin of uniform keys never holds 1.25 times its share and 4096 more)
        if (threadIdx.x == 0) atomicCAS(status, 0, (int)SMC_ERR_STATE);
        return;
    }
    unsigned rank = T.rank, pre[3] = {0u, 0u, 0u};
    int d = 0;
    for (; d < 12; ++d) {
        const int w = d >> 2, sh = 24 - 8 * (d & 3);
        auto match = [&](const Candidate &c) {  // leading d bytes equal
            const unsigned v[3] = {c.hi, c.lo, c.s};
            for (int k = 0; k < w; ++k)
                if (v[k] != pre[k]) return false;
            return sh == 24 || (v[w] >> (sh + 8)) == (pre[w] >> (sh + 8));
        };
        auto byte = [&](const Candidate &c) { return ((w == 0 ? c.hi : (w == 1 ? c.lo : c.s)) >> sh) & 255u; };
        for (int i = threadIdx.x; i < 256; i += blockDim.x) h[i] = 0;
        __syncthreads();
        for (unsigned i = threadIdx.x; i < n; i += blockDim.x)
            if (match(L[i])) atomicAdd(&h[byte(L[i])], 1u);
        __syncthreads();
        if (threadIdx.x < 32) {  // lane l: bytes 8 l .. 8 l + 7
            const int l = threadIdx.x;
            unsigned c[8], sum = 0;
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                c[k] = h[8 * l + k];
                sum += c[k];
            }
            unsigned incl = sum;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const unsigned v = __shfl_up_sync(0xffffffffu, incl, o);
                if (l >= o) incl += v;
            }
            unsigned acc = incl - sum;
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                if (rank >= acc && rank < acc + c[k]) {
                    s_byte = (unsigned)(8 * l + k);
                    s_rank = rank - acc;
                    s_left = c[k];
                }
                acc += c[k];
            }
        }
        __syncthreads();
        pre[w] |= s_byte << sh;
        rank = s_rank;
        const unsigned left = s_left;
        __syncthreads();
        if (left == 1) break;
    }
    // the one element with these leading bytes
    if (d > 11) d = 11;
    const int w = d >> 2, sh = 24 - 8 * (d & 3);
    for (unsigned i = threadIdx.x; i < n; i += blockDim.x) {
        const unsigned v[3] = {L[i].hi, L[i].lo, L[i].s};
        bool ok = (v[w] >> sh) == (pre[w] >> sh);
        for (int k = 0; k < w; ++k) ok = ok && v[k] == pre[k];
        if (ok) {
            T.k64 = ((unsigned long long)v[0] << 32) | v[1];
            T.s = v[2];
        }
    }
}

__global__ void __launch_bounds__(256) k_init_assign(uint64_t seed, uint32_t rep, long long N, int ntarget,
                                                     const InitState *st, int8_t *occ)
{
    __shared__ Threshold T[kMaxTargets];
    if (threadIdx.x < ntarget) T[threadIdx.x] = st->t[threadIdx.x];
    __syncthreads();
    const long long nq = (N + 3) / 4;
    for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < nq; q += (long long)gridDim.x * blockDim.x) {
        const U4 hi = site_hi(seed, rep, (uint32_t)q);
        uint32_t out = 0;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const uint32_t h = pick_word(hi, i);
            uint32_t sp = 0;
            for (int t = 0; t < ntarget; ++t) {
                const uint32_t th = (uint32_t)(T[t].k64 >> 32);
                if (!T[t].active) continue;
                if (h > th) {
                    ++sp;
                } else if (h == th) {
                    const uint32_t l = pick_word(site_lo(seed, rep, (uint32_t)q), i), tl = (uint32_t)T[t].k64;
                    if (l > tl || (l == tl && (unsigned)(4 * q + i) >= T[t].s)) ++sp;
                }
            }
            out |= sp << (8 * i);
        }
        if (4 * q + 3 < N && (reinterpret_cast<uintptr_t>(occ) & 3) == 0)
            *(uint32_t *)(occ + 4 * q) = out;
        else
            for (int i = 0; i < 4 && 4 * q + i < N; ++i) occ[4 * q + i] = (int8_t)(out >> (8 * i));
    }
}

smc_status launch_init(const smc_lattice *lat, const int64_t *counts, uint64_t seed, uint32_t replica, int8_t *occ,
                       cudaStream_t stream)
{
    smc_status stt;
    Workspace *ws = workspace(&stt);
    if (!ws) return stt;
    const long long N = 2LL * lat->nx * lat->ny * lat->nz;
    const int ntarget = lat->nspecies - 1;
    static InitState h0;
    memset(&h0, 0, sizeof h0);
    long long cum = 0;
    for (int t = 0; t < ntarget; ++t) {
        cum += counts[t];
        h0.t[t].rank = (unsigned)cum;
        h0.t[t].active = cum < N ? 1 : 0;
    }
    // candidate lists: in the workspace's first megabyte for small boxes, in
    // the occupancy (written last) for others, 0.052 N + 0.4 MB bytes
    const unsigned cap = (unsigned)std::min<long long>(N, N / kInitBins + N / kInitBins / 4 + 4096);
    const size_t off_lists = (sizeof(InitState) + 15) / 16 * 16, lists_bytes = (size_t)ntarget * cap * sizeof(Candidate);
    const bool in_occ = off_lists + lists_bytes > (1u << 20) - 512;
    unsigned char *scr = (unsigned char *)workspace_scratch(ws, off_lists + (in_occ ? 0 : lists_bytes), &stt);
    if (!scr) return stt;
    InitState *st = (InitState *)scr;
    Candidate *lists = in_occ ? (Candidate *)(((uintptr_t)occ + 15) / 16 * 16) : (Candidate *)(scr + off_lists);
    cudaError_t e = cudaMemcpyAsync(st, &h0, sizeof h0, cudaMemcpyHostToDevice, stream);
    if (e != cudaSuccess) return cuda_fail(e, "cudaMemcpyAsync(init state)");
    const long long nq = (N + 3) / 4;
    const int blocks = (int)std::max<long long>(1, std::min<long long>((nq + 255) / 256, ws->num_sms * 8LL));
    if (ntarget > 0) {
        const int hb = (int)std::max<long long>(1, std::min<long long>((nq + 511) / 512, ws->num_sms * 2LL));
        k_init_hist<<<hb, 512, 0, stream>>>(seed, replica, N, st);
        k_init_bins<<<1, kInitBins / 2, 0, stream>>>(ntarget, st);
        k_init_collect<<<blocks, 256, 0, stream>>>(seed, replica, N, ntarget, st, lists, cap);
        k_init_select<<<ntarget, 1024, 0, stream>>>(st, lists, cap, ws->status);
    }
    k_init_assign<<<blocks, 256, 0, stream>>>(seed, replica, N, ntarget, st, occ);
    e = cudaGetLastError();
    return e == cudaSuccess ? SMC_OK : cuda_fail(e, "init kernels");
}

}  // namespace smc

// mlp_grad.cu -- dE/dtheta of the MLP energy E = sum_i f(x_i) with respect to
// every MLP parameter (W1, b1, W2, b2, W3, b3), by back-propagation at every
// site, on the tcgen05 tensor cores.
//
// For one site, with z1 = W1 x + b1, h1 = silu(z1), z2 = W2 h1 + b2,
// h2 = silu(z2), f = W3 h2 + b3:
//   d2 = W3 .* silu'(z2),  d1 = (W2^T d2) .* silu'(z1),
//   dE/dW3 = sum_i h2,  dE/db3 = N,  dE/dW2 = sum_i d2 h1^T,  dE/db2 = sum_i d2,
//   dE/dW1 = sum_i d1 x^T,  dE/db1 = sum_i d1.
// A warpgroup takes 128 sites per tile, thread t owning site t (TMEM lane t):
//   layer 1  D = [x | 1] [W1 | b1]^T / 2 = z1/2                    (2 MMAs)
//   epilogue h1 = silu(z1) -> columns 0-63 of the HX tile (BF16), 2 silu'(z1) kept in registers
//   layer 2  D = [h1 | 1] [W2 | b2]^T / 2 = z2/2                   (5 MMAs)
//   epilogue h2, d2 -> the two slots of the Z tile (BF16)
//   back     D = d2 W2 / 2, the W2 tile read along its other axis  (4 MMAs)
//            GH[64 x 8] += h2^T [x16..x19 1 1 1 0]                 (8 MMAs, K = 16 sites): column 4 is dW3
//   epilogue d1 = D .* 2 silu'(z1) -> the slot of h2
//   G[128 x 96] += [d1 | d2]^T [h1 | x | 1]                        (8 MMAs): rows d2: dW2 (columns 0-63), db2 (84);
//                                                                  rows d1: dW1 (columns 64-83), db1 (84)
// The tiles are site-major (each site's values contiguous), which makes them,
// read with MN-major descriptors (leading byte offset = stride between 8-site
// groups, stride byte offset = 128 B between 8-value groups), the operands of
// the contractions over sites, accumulated in TMEM across tiles.  Every
// kFlushEvery tiles a warpgroup adds its accumulators into the CTA's FP64
// copy, the warpgroups in turn (their order is fixed); a second kernel adds
// the CTA copies in CTA order, so the result is bit-reproducible for a device.
//
// Bound by the chain of a tile (four products, each with a barrier before and
// a wait after it, and the epilogues between them): one warpgroup leaves its
// schedulers idle two cycles of three.  So three warpgroups run at their own
// pace; what each needs was cut to a third of an SM: 56 KB of tiles (HX
// shared by both contractions, d1 over h2) and 168 TMEM columns.  The
// activations and derivatives are computed two at a time (fma.rn.f32x2), and
// the neighbours of the next tile are read while the second layer runs.
// Random 5-species boxes, whole gradient: 512^3 49.3 -> 24.5 ms (from two
// warpgroups with tiles of their own for either contraction, scalar epilogues
// and the FP64 additions behind a CTA barrier, bank conflicts in them), 128^3
// 0.83 -> 0.45 ms, 32^3 72 -> 63 us.  Straight-line code matters: unrolling
// the flush further, or integer conversions in it, cost 6 % in fetches.
#include "mlp_common.cuh"
#include "mlp_tc.cuh"
#include "sweep_common.cuh"

namespace smc {

constexpr int kGradWG = 3;
constexpr int kGradThreads = 128 * kGradWG;
constexpr int kMlpParams = 64 * 20 + 64 + 64 * 64 + 64 + 64 + 1;
constexpr int kFlushEvery = 8;
constexpr int kOffW1 = 0, kOffB1 = kOffW1 + 64 * 20, kOffW2 = kOffB1 + 64, kOffB2 = kOffW2 + 64 * 64,
              kOffW3 = kOffB2 + 64, kOffB3 = kOffW3 + 64;
// FP64 copy: [column][row of 64], lanes side by side: W2 and b2 (65 columns), W1 and b1 (21), W3 (1)
constexpr int kAccW1 = 65 * 64, kAccW3 = kAccW1 + 21 * 64, kAccN = kAccW3 + 64;
static_assert(kAccN == kMlpParams - 1 && kAccN % 32 == 0, "all parameters but b3");
constexpr uint32_t kHXGroup = 8 * 96 * 2;  // HX tile: h1 | x | 1, 96 BF16 a site; bytes of 8 sites
constexpr uint32_t kZGroup = 8 * 128 * 2;  // Z tile: two slots of 64 BF16 a site
// TMEM columns: per warpgroup 64 for the layers (D), 96 (G) and 8 (GH); 504 of the SM's 512
constexpr uint32_t kColD = 0, kColG = 64 * kGradWG, kColGH = kColG + 96 * kGradWG;
static_assert(kColGH + 8 * kGradWG <= 512, "tensor memory");

struct GradSmem {
    static constexpr uint32_t W1 = 0;
    static constexpr uint32_t W2 = W1 + kTcW1;
    static constexpr uint32_t W3 = W2 + kTcW2;
    static constexpr uint32_t B3 = W3 + 256;
    static constexpr uint32_t WG = (B3 + 16 + 127) / 128 * 128;  // per-warpgroup tiles from here
    static constexpr uint32_t HX = 0, Z = HX + 16 * kHXGroup, WGSIZE = Z + 16 * kZGroup;  // offsets within a warpgroup
    static constexpr uint32_t MBAR = WG + kGradWG * WGSIZE;  // [kGradWG][4]
    static constexpr uint32_t TSLOT = MBAR + 32 * kGradWG;
    static constexpr uint32_t TURN = TSLOT + 8;  // flushes done by the CTA's warpgroups
    static constexpr uint32_t ACC = (TURN + 8 + 15) / 16 * 16;  // FP64 [kAccN]
    static constexpr uint32_t END = ACC + kAccN * 8;
};
static_assert(GradSmem::WG % 128 == 0 && GradSmem::WGSIZE % 128 == 0, "tile alignment");
static_assert(GradSmem::END <= 227 * 1024, "shared memory");

// Byte offset of chunk kc (8 BF16) of site row r in the HX tile and in the Z tile.
__host__ __device__ constexpr uint32_t hx_off(uint32_t r, uint32_t kc) { return (r >> 3) * kHXGroup + kc * 128 + (r & 7) * 16; }
__host__ __device__ constexpr uint32_t z_off(uint32_t r, uint32_t kc) { return (r >> 3) * kZGroup + kc * 128 + (r & 7) * 16; }

// Pairs of FP32 values, rounded as the scalar operations round.
__device__ __forceinline__ uint64_t pair2(float a, float b)
{
    uint64_t v;
    asm("mov.b64 %0, {%1, %2};" : "=l"(v) : "f"(a), "f"(b));
    return v;
}
__device__ __forceinline__ void unpair2(uint64_t v, float &a, float &b) { asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v)); }
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c)
{
    uint64_t d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ uint64_t mul2(uint64_t a, uint64_t b)
{
    uint64_t d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b)
{
    uint64_t d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ uint32_t pack2(uint64_t v)
{
    float a, b;
    unpair2(v, a, b);
    return pack_bf16(a, b);
}

// Of a pair h: silu(2h) = h + h t and 2 silu'(2h) = (1 + t)(1 + h (1 - t)), t = tanh(h).
__device__ __forceinline__ void silu_pair2(uint32_t ha, uint32_t hb, uint64_t &s, uint64_t &ds)
{
    float ta, tb;
    asm("tanh.approx.f32 %0, %1;" : "=f"(ta) : "f"(__uint_as_float(ha)));
    asm("tanh.approx.f32 %0, %1;" : "=f"(tb) : "f"(__uint_as_float(hb)));
    const uint64_t one = pair2(1.f, 1.f), neg = pair2(-1.f, -1.f);
    const uint64_t h = pair2(__uint_as_float(ha), __uint_as_float(hb)), t = pair2(ta, tb);
    s = fma2(h, t, h);
    ds = mul2(add2(t, one), fma2(h, fma2(t, neg, one), one));
}

// One column of TMEM, this warp's 32 lanes.
__device__ __forceinline__ uint32_t tc_ld1(uint32_t taddr)
{
    uint32_t v;
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x1.b32 {%0}, [%1];" : "=r"(v) : "r"(taddr) : "memory");
    asm volatile("tcgen05.wait::ld.sync.aligned;" : "+r"(v) : : "memory");
    return v;
}

__device__ __forceinline__ void grad_wait(uint32_t mbar, uint32_t &phase, long long timeout_ns, int *status,
                                          int *abort_flag)
{
    if (!mbar_wait(mbar, phase, timeout_ns)) {
        atomicCAS(status, 0, (int)SMC_ERR_TIMEOUT);
        atomicExch(abort_flag, 1);
    }
    phase ^= 1;
    tc_fence_after();
}

__global__ void __launch_bounds__(kGradThreads, 1) k_mlp_grad(const MlpBlock *W, const int8_t *__restrict__ occ,
                                                              int nx, int ny, int nz, double *part,
                                                              long long timeout_ns, int *status, int *abort_flag)
{
    const int tid = threadIdx.x, r = tid & 127, wg = tid >> 7, wq = r >> 5;
    const uint32_t s0 = (uint32_t)__cvta_generic_to_shared(g_smem);
    const uint32_t base = GradSmem::WG + wg * GradSmem::WGSIZE;
    const uint32_t HX = base + GradSmem::HX, Z = base + GradSmem::Z, mbar = s0 + GradSmem::MBAR + 32 * wg;
    // weights: W1, W2 halved with the biases folded in; b2 moves to where the tile has x16..x19 1 1 1 0
    {
        TcLayout L{HX, HX, GradSmem::W1, GradSmem::W2, 0, 0, GradSmem::W3, GradSmem::B3, 0, 0};
        tc_load_weights(W, L);
    }
    __syncthreads();
    for (int i = tid; i < 64; i += kGradThreads) {
        uint4 *b = (uint4 *)(g_smem + GradSmem::W2 + tc_off80(i, 8));
        *b = make_uint4(0u, 0u, b->x, b->y);
        ((float *)(g_smem + GradSmem::W3))[i] *= 0.5f;  // d2 = (W3 / 2) .* 2 silu'
    }
    double *acc64 = (double *)(g_smem + GradSmem::ACC);
    for (int i = tid; i < kAccN; i += kGradThreads) acc64[i] = 0.0;
    volatile uint32_t *turn = (volatile uint32_t *)(g_smem + GradSmem::TURN);
    if (tid == 0) *turn = 0;
    if (r == 0)
        for (int b = 0; b < 4; ++b) mbar_init(mbar + 8 * b, 1);
    if (tid < 32) tc_alloc(s0 + GradSmem::TSLOT, 512);
    fence_async_smem();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *(const uint32_t *)(g_smem + GradSmem::TSLOT);
    const uint32_t D = tmem + kColD + 64 * wg, G = tmem + kColG + 96 * wg, GH = tmem + kColGH + 8 * wg;
    const uint32_t bar = 1 + wg;
    const uint32_t lane_base = (uint32_t)(32 * wq) << 16;
    uint32_t ph[4] = {0, 0, 0, 0};
    // slots of d2 and of h2, then d1: the other way round in the second warpgroup, so that its d2 sums (three
    // quarters of the FP64 additions) fall on the other two schedulers
    const uint32_t sd = wg == 1 ? 0 : 1, sh = 1 - sd;
    const float4 *w3 = (const float4 *)(g_smem + GradSmem::W3);
    auto spec = [&](int sb, int xx, int yy, int zz) {
        return occ[(unsigned)((sb * nz + wrapc(zz, nz)) * ny + wrapc(yy, ny)) * (unsigned)nx + (unsigned)wrapc(xx, nx)] & 7;
    };
    constexpr uint32_t kIdBack = tc_idesc(128, 64, false, true), kIdG = tc_idesc(128, 96, true, true),
                       kIdGH = tc_idesc(64, 8, true, true);
    const long long N = 2LL * nx * ny * nz;  // < 2^31
    const long long ntile = (N + kTcRows - 1) / kTcRows;
    const long long rounds = (ntile + (long long)kGradWG * gridDim.x - 1) / ((long long)kGradWG * gridDim.x);
    uint32_t g_acc = 0;    // 0: the next weight-gradient products start the accumulators afresh
    bool g_busy = false;   // the last tile's products still read HX and Z

    // species and neighbour histograms of this thread's site of tile tl (q0 < 0: no site)
    int q0 = -1;
    uint32_t n1 = 0, n2 = 0, n3 = 0;
    auto site = [&](long long tl) {
        const long long s = tl * kTcRows + r;
        q0 = -1;
        n1 = n2 = n3 = 0;
        if (s < N) {
            unsigned t = (unsigned)s;
            const int x = (int)(t % (unsigned)nx);
            t /= (unsigned)nx;
            const int y = (int)(t % (unsigned)ny);
            t /= (unsigned)ny;
            const int z = (int)(t % (unsigned)nz);
            q0 = occ[s] & 7;
            site_hist(spec, (int)(t / (unsigned)nz), x, y, z, n1, n2, n3);
        }
    };

    // adds the TMEM accumulators of this warpgroup into the FP64 copy
    auto flush = [&]() {
        const int k = r & 63;
        uint32_t v[32];
        if ((uint32_t)(r >> 6) == sd) {
#pragma unroll 1
            for (int c = 0; c < 64; c += 32) {
                tc_ld32(G + lane_base + c, v);
                tc_wait_ld(v);
#pragma unroll
                for (int j = 0; j < 32; ++j) acc64[(c + j) * 64 + k] += (double)__uint_as_float(v[j]);
            }
            acc64[64 * 64 + k] += (double)__uint_as_float(tc_ld1(G + lane_base + 84));
        } else {
            tc_ld32(G + lane_base + 64, v);
            tc_wait_ld(v);
#pragma unroll
            for (int j = 0; j < 21; ++j) acc64[kAccW1 + j * 64 + k] += (double)__uint_as_float(v[j]);
        }
        // 64-row accumulator: rows 16 w .. 16 w + 15 in the first 16 lanes of warp w
        const uint32_t h = tc_ld1(GH + lane_base + 4);
        if ((r & 31) < 16) acc64[kAccW3 + 16 * wq + (r & 31)] += (double)__uint_as_float(h);
    };

    long long tl = (long long)blockIdx.x * kGradWG + wg;
    if (tl < ntile) site(tl);
    for (long long rd = 0; rd < rounds; ++rd, tl += (long long)gridDim.x * kGradWG) {
        if (tl < ntile) {
            const bool valid = q0 >= 0;
            if (g_busy) grad_wait(mbar + 24, ph[3], timeout_ns, status, abort_flag);  // HX, Z free again
            // ---- features of this row's site ----
            {
                uint32_t w[16];
                tc_feature_words(q0, n1, n2, n3, w);
#pragma unroll
                for (int kc = 0; kc < 4; ++kc)
                    *(uint4 *)(g_smem + HX + hx_off(r, 8 + kc)) = make_uint4(w[4 * kc], w[4 * kc + 1], w[4 * kc + 2], w[4 * kc + 3]);
            }
            fence_async_smem();
            tc_fence_before();
            wg_sync(bar);
            if (r == 0) {
                tc_fence_after();
#pragma unroll
                for (int k = 0; k < 2; ++k)
                    tc_mma(D, tc_desc(s0 + HX + 1024 + k * 256, 128, kHXGroup),
                           tc_desc(s0 + GradSmem::W1 + k * 256, 128, 512), k > 0);
                tc_commit(mbar);
            }
            grad_wait(mbar, ph[0], timeout_ns, status, abort_flag);
            // ---- layer-1 epilogue: h1 -> HX, 2 silu'(z1) kept ----
            uint64_t ds1[32];
#pragma unroll
            for (int half = 0; half < 2; ++half) {
                uint32_t v[32];
                tc_ld32(D + lane_base + 32 * half, v);
                tc_wait_ld(v);
#pragma unroll
                for (int kc = 0; kc < 4; ++kc) {
                    uint32_t w[4];
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        uint64_t h;
                        silu_pair2(v[8 * kc + 2 * u], v[8 * kc + 2 * u + 1], h, ds1[16 * half + 4 * kc + u]);
                        w[u] = pack2(h);
                    }
                    *(uint4 *)(g_smem + HX + hx_off(r, 4 * half + kc)) = make_uint4(w[0], w[1], w[2], w[3]);
                }
            }
            fence_async_smem();
            tc_fence_before();
            wg_sync(bar);
            if (r == 0) {
                tc_fence_after();
#pragma unroll
                for (int k = 0; k < 5; ++k)  // the last: columns 80-95 (x16..x19 1 1 1 0 ..) against the bias parts
                    tc_mma(D, tc_desc(s0 + HX + (k < 4 ? k * 256 : 1280), 128, kHXGroup),
                           tc_desc(s0 + GradSmem::W2 + k * 256, 128, 1280), k > 0);
                tc_commit(mbar + 8);
            }
            {  // the next tile's neighbours, meanwhile
                const long long next = tl + (long long)gridDim.x * kGradWG;
                if (next < ntile) site(next);
            }
            grad_wait(mbar + 8, ph[1], timeout_ns, status, abort_flag);
            // ---- layer-2 epilogue: h2 and d2 = W3 .* silu'(z2) -> Z ----
#pragma unroll
            for (int half = 0; half < 2; ++half) {
                uint32_t v[32];
                tc_ld32(D + lane_base + 32 * half, v);
                tc_wait_ld(v);
#pragma unroll
                for (int kc = 0; kc < 4; ++kc) {
                    uint32_t wh[4], wd[4];
                    const float4 wa = w3[8 * half + 2 * kc], wb = w3[8 * half + 2 * kc + 1];
                    const uint64_t wv[4] = {pair2(wa.x, wa.y), pair2(wa.z, wa.w), pair2(wb.x, wb.y), pair2(wb.z, wb.w)};
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        uint64_t h, d;
                        silu_pair2(v[8 * kc + 2 * u], v[8 * kc + 2 * u + 1], h, d);
                        wh[u] = pack2(h);
                        wd[u] = pack2(mul2(wv[u], d));
                    }
                    *(uint4 *)(g_smem + Z + z_off(r, 8 * sh + 4 * half + kc)) = make_uint4(wh[0], wh[1], wh[2], wh[3]);
                    *(uint4 *)(g_smem + Z + z_off(r, 8 * sd + 4 * half + kc)) = make_uint4(wd[0], wd[1], wd[2], wd[3]);
                }
            }
            if (!valid)  // rows past the last site
#pragma unroll 1
                for (int kc = 0; kc < 16; ++kc) *(uint4 *)(g_smem + Z + z_off(r, kc)) = make_uint4(0u, 0u, 0u, 0u);
            fence_async_smem();
            tc_fence_before();
            wg_sync(bar);
            if (r == 0) {
                tc_fence_after();
                // back-propagation through W2 / 2 (its tile as a K x N operand: K = its rows)
#pragma unroll
                for (int k = 0; k < 4; ++k)
                    tc_mma_i(D, tc_desc(s0 + Z + 1024 * sd + k * 256, 128, kZGroup),
                             tc_desc(s0 + GradSmem::W2 + k * 2 * 1280, 1280, 128), kIdBack, k > 0);
                // GH += h2^T [x16..x19 1 1 1 0], contraction over the 128 sites
#pragma unroll
                for (int k = 0; k < 8; ++k)
                    tc_mma_i(GH, tc_desc(s0 + Z + 1024 * sh + k * 2 * kZGroup, kZGroup, 128),
                             tc_desc(s0 + HX + 1280 + k * 2 * kHXGroup, kHXGroup, 128), kIdGH, (k > 0) | g_acc);
                tc_commit(mbar + 16);
            }
            grad_wait(mbar + 16, ph[2], timeout_ns, status, abort_flag);
            // ---- back epilogue: d1 = D .* 2 silu'(z1) over h2 ----
#pragma unroll
            for (int half = 0; half < 2; ++half) {
                uint32_t v[32];
                tc_ld32(D + lane_base + 32 * half, v);
                tc_wait_ld(v);
#pragma unroll
                for (int kc = 0; kc < 4; ++kc) {
                    uint32_t w[4];
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        const uint64_t d = pair2(__uint_as_float(v[8 * kc + 2 * u]), __uint_as_float(v[8 * kc + 2 * u + 1]));
                        w[u] = pack2(mul2(d, ds1[16 * half + 4 * kc + u]));
                    }
                    *(uint4 *)(g_smem + Z + z_off(r, 8 * sh + 4 * half + kc)) = make_uint4(w[0], w[1], w[2], w[3]);
                }
            }
            if (!valid)
#pragma unroll 1
                for (int kc = 0; kc < 8; ++kc) *(uint4 *)(g_smem + Z + z_off(r, 8 * sh + kc)) = make_uint4(0u, 0u, 0u, 0u);
            fence_async_smem();
            tc_fence_before();
            wg_sync(bar);
            if (r == 0) {
                tc_fence_after();
                // G += [slot 0 | slot 1]^T [h1 | x | 1]
#pragma unroll
                for (int k = 0; k < 8; ++k)
                    tc_mma_i(G, tc_desc(s0 + Z + k * 2 * kZGroup, kZGroup, 128),
                             tc_desc(s0 + HX + k * 2 * kHXGroup, kHXGroup, 128), kIdG, (k > 0) | g_acc);
                tc_commit(mbar + 24);
            }
            g_busy = true;
            g_acc = 1;
        }
        // ---- every kFlushEvery rounds (and after the last): FP64 accumulation, the warpgroups in turn ----
        if ((rd + 1) % kFlushEvery == 0 || rd + 1 == rounds) {
            if (g_busy) grad_wait(mbar + 24, ph[3], timeout_ns, status, abort_flag);
            g_busy = false;
            const uint32_t mine = (uint32_t)(rd / kFlushEvery) * kGradWG + wg;
            if (r == 0 && *turn != mine) {
                const uint64_t t0 = global_ns();
                while (*turn != mine)
                    if ((long long)(global_ns() - t0) > timeout_ns) {
                        atomicCAS(status, 0, (int)SMC_ERR_TIMEOUT);
                        atomicExch(abort_flag, 1);
                        break;
                    }
            }
            __threadfence_block();
            wg_sync(bar);
            if (g_acc) flush();
            g_acc = 0;
            __threadfence_block();
            tc_fence_before();
            wg_sync(bar);
            tc_fence_after();
            if (r == 0) *turn = mine + 1;
        }
    }
    __syncthreads();
    double *dst = part + (size_t)blockIdx.x * kAccN;
    for (int i = tid; i < kAccN; i += kGradThreads) dst[i] = acc64[i];
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (tid < 32) tc_dealloc(tmem, 512);
}

// grad = sum over CTAs of part[cta]: eight warps of a block add an eighth of the CTAs each, in CTA order, then their
// sums are added in order; db3 is the number of sites.  (The additions of one thread wait for each other, and a
// scheduler's FP64 unit takes 64 cycles for a warp: one thread for all 152 CTAs took 16 us.)
__global__ void __launch_bounds__(256) k_mlp_grad_finish(const double *part, int nparts, double nsites, float *grad)
{
    __shared__ double sum[8][32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, i = blockIdx.x * 32 + lane;  // kAccN is a multiple of 32
    const int each = (nparts + 7) / 8, b1 = min(nparts, (w + 1) * each);
    double s = 0.0;
#pragma unroll 8
    for (int b = w * each; b < b1; ++b) s += part[(size_t)b * kAccN + i];
    sum[w][lane] = s;
    __syncthreads();
    if (w > 0) return;
    for (int k = 1; k < 8; ++k) s += sum[k][lane];
    if (i == 0) grad[kOffB3] = (float)nsites;
    const int row = i & 63;
    int at;
    if (i < kAccW1)
        at = i < 64 * 64 ? kOffW2 + row * 64 + (i >> 6) : kOffB2 + row;
    else if (i < kAccW3)
        at = i < kAccW1 + 20 * 64 ? kOffW1 + row * 20 + ((i - kAccW1) >> 6) : kOffB1 + row;
    else
        at = kOffW3 + row;
    grad[at] = (float)s;
}

smc_status launch_mlp_grad(const smc_lattice *lat, const smc_model *m, const int8_t *occ, float *grad,
                           cudaStream_t stream)
{
    smc_status st;
    Workspace *ws = workspace(&st);
    if (!ws) return st;
    const size_t smem = GradSmem::END;
    cudaError_t e = cudaFuncSetAttribute(k_mlp_grad, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return cuda_fail(e, "cudaFuncSetAttribute(k_mlp_grad)");
    int per_sm = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_mlp_grad, kGradThreads, smem);
    if (e != cudaSuccess) return cuda_fail(e, "cudaOccupancyMaxActiveBlocksPerMultiprocessor");
    if (per_sm != 1) {  // each CTA holds all 512 tensor-memory columns of its SM
        set_error("MLP gradient kernel occupancy %d (expected 1 CTA per SM)", per_sm);
        return SMC_ERR_STATE;
    }
    const long long N = 2LL * lat->nx * lat->ny * lat->nz;
    const long long ntile = (N + kTcRows - 1) / kTcRows;
    const int grid = (int)std::max(1LL, std::min<long long>((long long)ws->num_sms, (ntile + kGradWG - 1) / kGradWG));
    // scratch: [pair counts | abort word | MlpBlock | CTA partials]
    const size_t off_abort = (sizeof(unsigned long long) * kMaxShells * 64 + 15) / 16 * 16;
    const size_t off_w = off_abort + 16;
    const size_t off_part = (off_w + sizeof(MlpBlock) + 15) / 16 * 16;
    unsigned char *scr =
        (unsigned char *)workspace_scratch(ws, off_part + sizeof(double) * kAccN * (size_t)grid, &st);
    if (!scr) return st;
    int npair = 0;
    if (m->kind == SMC_PAIR_F32_MLP_BF16) {
        npair = m->nshells * lat->nspecies * (lat->nspecies + 1) / 2;
        unsigned long long *cnt = (unsigned long long *)scr;
        st = launch_pair_counts(lat, m->nshells, occ, cnt, stream);
        if (st != SMC_OK) return st;
        st = launch_pair_grad_finish(lat, m, cnt, grad, stream);
        if (st != SMC_OK) return st;
    }
    static MlpBlock W;
    make_mlp_block(m, W);
    e = cudaMemcpyAsync(scr + off_w, &W, sizeof W, cudaMemcpyHostToDevice, stream);
    if (e != cudaSuccess) return cuda_fail(e, "cudaMemcpyAsync(MLP weights)");
    e = cudaMemsetAsync(scr + off_abort, 0, 16, stream);
    if (e != cudaSuccess) return cuda_fail(e, "cudaMemsetAsync(abort word)");
    double *part = (double *)(scr + off_part);
    k_mlp_grad<<<grid, kGradThreads, smem, stream>>>((const MlpBlock *)(scr + off_w), occ, lat->nx, lat->ny, lat->nz,
                                                     part, debug_timeout_ns(), ws->status, (int *)(scr + off_abort));
    e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_fail(e, "k_mlp_grad");
    k_mlp_grad_finish<<<kAccN / 32, 256, 0, stream>>>(part, grid, (double)N, grad + npair);
    e = cudaGetLastError();
    return e == cudaSuccess ? SMC_OK : cuda_fail(e, "k_mlp_grad_finish");
}

}  // namespace smc

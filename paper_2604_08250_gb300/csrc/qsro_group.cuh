// qsro_group.cuh -- qSRO trials (Eq. quadratic_local_SRO), one launch per group
// of four mini-steps (row_group.cuh), for the BCC and FCC lattices.
//
// A column's rows of species and of own-species counts are copied to shared
// memory; a zone site is one byte of each at a fixed offset from the trial
// site (table per partner direction), and an accepted swap updates both
// there.  The sums run in the order of the one-mini-step kernels
// (qsro_bcc.cu, fcc.cu), so both give the same bits.
#pragma once

#include <type_traits>

#include "row_group.cuh"

namespace smc {

// Tables of a launch (32-bit words): Dz[m][A][B][q] at m * 512 + (A * 8 + B) * 8
// + q, Wz[m][p] at kQgW + m * 8 + p, then per sublattice, for each partner
// direction d (kQgDirs of them): the zone's offsets [e][d] from a (cells times
// 16, plus dx + 8), and b's at [kQgZone][d].
constexpr int kQgW = kMaxShells * 512, kQgOff = kQgW + kMaxShells * 8, kQgDirs = 16, kQgZone = 58,
              kQgSub = (kQgZone + 1) * kQgDirs;
__host__ __device__ constexpr int qg_words(int nsub) { return kQgOff + nsub * kQgSub; }
inline uint32_t qg_pack(int slot, int pitch, int dx) { return (uint32_t)(((slot * pitch + dx) << 4) | (dx + 8)); }

struct QsroGroup {
    RowGroup G;
    uint64_t seed, sweep;
    uint32_t replica;
    float beta;
    const uint32_t *tables;
    int8_t *occ;
    void *qcache;
    double *part_e;
    long long *part_n;
    float *dE_out;
    uint8_t *acc_out;
};

// Bytes of shared memory beside the rows.
inline size_t qg_fixed(int nsh, int nz) { return (size_t)(nsh * (kRgDShell + 8) + (nz + 1) * kQgDirs) * 4; }

// Lat: zone(nsh) sites, code(nsh, e) = (shell to a) * 4 + (shell to b), count
// fields qoff(m), qmask(m), and draw(P, a, word set) -> (r, dir).
template <class Lat, int NSH>
__global__ void __launch_bounds__(kRgThreads) k_qsro_group(const __grid_constant__ QsroGroup P)
{
    using QT = typename std::conditional<NSH == 3, uint16_t, uint8_t>::type;
    constexpr int NZ = Lat::zone(NSH), ES = (int)sizeof(QT);
    const RowGroup &G = P.G;
    // shared memory: Dz (rows laid out by rg_d_at: 256^3 BCC cells 2.14 -> 2.07 ms per sweep, boxes that do not
    // fill the SMs within 0.2 %) | Wz | offsets [NZ + 1][16] | row numbers per column | per column: species rows, count rows
    const float *sT = (const float *)g_smem;
    const float *sW = sT + NSH * kRgDShell;
    int *sZ = (int *)(g_smem + (size_t)(NSH * (kRgDShell + 8)) * 4);
    constexpr uint32_t rows0 = (uint32_t)(NSH * (kRgDShell + 8) + (NZ + 1) * kQgDirs) * 4;
    const int tid = threadIdx.x, c = tid / G.tpc, tt = tid - c * G.tpc, col = blockIdx.x * G.C + c;
    const bool on = col < G.ncol;
    const int y0 = 4 * (col % G.NLy) + G.dy, z0 = 4 * (col / G.NLy) + G.dz;
    int *rown = (int *)(g_smem + rows0 + c * kRgRowBytes);
    const uint32_t base = rows0 + G.C * kRgRowBytes + (uint32_t)(c * G.rows.n * (G.pitch + G.pitchq)),
                   baseq = base + G.rows.n * G.pitch;
    if (on) rg_rows(G, rown, y0, z0, tt);
    __syncthreads();
    if (on) {
        rg_stage<1>(G, (const unsigned char *)P.occ, base, G.pitch, G.unit, G.inv, rown, tt);
        rg_stage<ES>(G, (const unsigned char *)P.qcache, baseq, G.pitchq, G.unitq, G.invq, rown, tt);
    }
    for (int i = tid; i < NSH * 520; i += blockDim.x) {
        const int w = i - NSH * 512;  // from W on
        ((uint32_t *)g_smem)[w < 0 ? rg_d_at(i) : NSH * kRgDShell + w] = __ldg(P.tables + (w < 0 ? i : kQgW + w));
    }
    for (int i = tid; i < (NZ + 1) * kQgDirs; i += blockDim.x) {
        const int e = i / kQgDirs, src = e < NZ ? i : kQgZone * kQgDirs + i % kQgDirs;
        sZ[i] = (int)__ldg(P.tables + kQgOff + G.sub * kQgSub + src);
    }
    const bool active = on && tt < G.NLx;
    const int lc = col * G.NLx + tt;
    double accE = 0.0;
    long long accN = 0;
    const typename Lat::Words words = Lat::words(P, ((G.sub * G.nz + z0) * G.ny + y0) * G.nx + 4 * tt);
    rg_wait();
    unsigned char *occ = g_smem + base + kRgBody;
    QT *Qc = (QT *)(g_smem + baseq) + kRgBody;
    for (int dx = G.dx0; dx < G.dx1; ++dx) {
        if (active) {
            const int x = 4 * tt + dx;
            uint32_t r;
            int dir;
            Lat::draw(P, words, ((G.sub * G.nz + z0) * G.ny + y0) * G.nx + x, dx, r, dir);
            const int *zone = sZ + dir;
            const int bw = zone[NZ * kQgDirs], ob = bw >> 4;
            const int A = occ[x] & 7, B = occ[x + ob] & 7;
            // packed per-shell counts (byte m-1): species B around a (b among them), A around b (a among them);
            // those of A around a and B around b are a's and b's own counts
            uint32_t cBa = 1u, cAb = 1u;
            const int ca = Qc[x], cb = Qc[x + ob];
            uint32_t zq[NZ];  // species | count cache << 4 of every zone site, for the update of an accepted swap
            float dE = 0.f;
            if (A != B) {
                const float *row = sT + A * kRgDA + B * kRgDB;
                float wA[NSH], wB[NSH];  // W_m^A / z_m^2, W_m^B / z_m^2
#pragma unroll
                for (int m = 0; m < NSH; ++m) {
                    wA[m] = sW[m * 8 + A];
                    wB[m] = sW[m * 8 + B];
                }
                float lin = 0.f, wz = 0.f;
#pragma unroll
                for (int e = 0; e < NZ; ++e) {
                    const int code = Lat::code(NSH, e), ma = code >> 2, mb = code & 3;
                    const int o = x + (zone[e * kQgDirs] >> 4);
                    const int sj = occ[o] & 7;
                    const bool isA = sj == A, isB = sj == B;
                    if (ma) {
                        lin += row[(ma - 1) * kRgDShell + sj];
                        cBa += isB ? 1u << (8 * (ma - 1)) : 0u;
                    }
                    if (mb) {
                        lin -= row[(mb - 1) * kRgDShell + sj];
                        cAb += isA ? 1u << (8 * (mb - 1)) : 0u;
                    }
                    zq[e] = (uint32_t)sj;
                    if (ma != mb) {
                        const int q = Qc[o];
                        zq[e] |= (uint32_t)q << 4;
                        // a leaves j's shell ma as A and arrives as B (2n + 1 more or 2n - 1 less); b the reverse
                        // in shell mb.  The products are rounded before they are added.
                        float t = 0.f;
                        if (ma) {
                            const int n = (q >> Lat::qoff(ma - 1)) & Lat::qmask(ma - 1);
                            t += __fmul_rn(isA ? wA[ma - 1] : (isB ? wB[ma - 1] : 0.f), (float)(isA ? 1 - 2 * n : 2 * n + 1));
                        }
                        if (mb) {
                            const int n = (q >> Lat::qoff(mb - 1)) & Lat::qmask(mb - 1);
                            t += __fmul_rn(isA ? wA[mb - 1] : (isB ? wB[mb - 1] : 0.f), (float)(isB ? 1 - 2 * n : 2 * n + 1));
                        }
                        wz += t;
                    }
                }
                float wa = 0.f, wbb = 0.f;
#pragma unroll
                for (int m = 0; m < NSH; ++m) {
                    const int nAa = (ca >> Lat::qoff(m)) & Lat::qmask(m), nBa = ((cBa >> (8 * m)) & 255) - (m == 0 ? 1 : 0);
                    const int nAb = ((cAb >> (8 * m)) & 255) - (m == 0 ? 1 : 0), nBb = (cb >> Lat::qoff(m)) & Lat::qmask(m);
                    wa += wB[m] * (float)(nBa * nBa) - wA[m] * (float)(nAa * nAa);
                    wbb += wA[m] * (float)(nAb * nAb) - wB[m] * (float)(nBb * nBb);
                }
                dE = 2.f * lin + wa + wbb + wz;
            }
            const bool acc = metropolis<false>(dE, r, P.beta, nullptr, make_int2(0, 0));
            if (acc) {
                if (A != B) {
                    const int wrapb = rg_wrap(x + (bw & 15) - 8, G.nx) - (x + (bw & 15) - 8);
                    occ[x] = (unsigned char)B;
                    occ[x + ob + wrapb] = (unsigned char)A;
                    int qa = 0, qb = 0;  // a now B: its B neighbours other than b; b now A likewise
#pragma unroll
                    for (int m = 0; m < NSH; ++m) {
                        qa += (int)(((cBa >> (8 * m)) & 255u) - (m == 0 ? 1u : 0u)) << Lat::qoff(m);
                        qb += (int)(((cAb >> (8 * m)) & 255u) - (m == 0 ? 1u : 0u)) << Lat::qoff(m);
                    }
                    Qc[x] = (QT)qa;
                    Qc[x + ob + wrapb] = (QT)qb;
#pragma unroll
                    for (int e = 0; e < NZ; ++e) {
                        const int code = Lat::code(NSH, e), ma = code >> 2, mb = code & 3;
                        if (ma == mb) continue;
                        const int sj = (int)(zq[e] & 15u), q = (int)(zq[e] >> 4);
                        // A sites lose a (shell ma) and gain b (shell mb); B sites the reverse
                        const int d = (ma ? 1 << Lat::qoff(ma - 1) : 0) - (mb ? 1 << Lat::qoff(mb - 1) : 0);
                        const int zw = zone[e * kQgDirs], j = x + (zw & 15) - 8;
                        if (sj == A || sj == B)
                            Qc[x + (zw >> 4) + rg_wrap(j, G.nx) - j] = (QT)(sj == A ? q - d : q + d);
                    }
                }
                accE += (double)dE;
                ++accN;
            }
            if (P.dE_out) P.dE_out[lc] = dE;
            if (P.acc_out) P.acc_out[lc] = acc ? 1 : 0;
        }
        __syncthreads();
        if (dx + 1 < G.dx1) {
            if (on) {
                rg_halos<1>(G, base, G.pitch, G.rows.nwr, tt);
                rg_halos<ES>(G, baseq, G.pitchq, G.rows.n, tt);
            }
            __syncthreads();
        }
    }
    if (on) {
        rg_store<1>(G, (unsigned char *)P.occ, base, G.pitch, G.unit, G.inv, G.rows.nwr, rown, tt);
        rg_store<ES>(G, (unsigned char *)P.qcache, baseq, G.pitchq, G.unitq, G.invq, G.rows.n, rown, tt);
    }
    if (active && accN) {
        P.part_e[lc] += accE;
        P.part_n[lc] += accN;
    }
}

// All groups (trace_k < 0) or the one mini-step trace_k of nsweeps sweeps;
// dz and dy are the next slower digits of k after dx, then the sublattice.
template <class Kernel>
smc_status qg_launch(Kernel kern, QsroGroup &gp, const RowSet *rows, size_t smem, uint64_t sweep0, int nsweeps,
                     const double *kT, int groups, int trace_k, cudaStream_t stream)
{
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return cuda_fail(e, "cudaFuncSetAttribute(k_qsro_group)");
    const int blocks = (gp.G.ncol + gp.G.C - 1) / gp.G.C;
    const int g0 = trace_k >= 0 ? trace_k >> 2 : 0, g1 = trace_k >= 0 ? g0 + 1 : groups;
    gp.G.dx0 = trace_k >= 0 ? trace_k & 3 : 0;
    gp.G.dx1 = trace_k >= 0 ? gp.G.dx0 + 1 : 4;
    for (int t = 0; t < nsweeps; ++t) {
        gp.sweep = sweep0 + (uint64_t)t;
        gp.beta = (float)(1.0 / kT[t]);
        for (int g = g0; g < g1; ++g) {
            gp.G.dy = g & 3;
            gp.G.dz = (g >> 2) & 3;
            gp.G.sub = g >> 4;
            gp.G.rows = rows[gp.G.sub];
            kern<<<blocks, gp.G.C * gp.G.tpc, smem, stream>>>(gp);
        }
        e = cudaGetLastError();
        if (e != cudaSuccess) return cuda_fail(e, "k_qsro_group");
    }
    return SMC_OK;
}

}  // namespace smc

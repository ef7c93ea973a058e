// Batched realisations: K copies of Eq. 1 that differ only in the on-site field (K disorder
// phases, Sec. 3 "many layers of disorder"), evolved together.  Vectors are interleaved
// [state][K] complex, so one rank computation and one neighbour lookup serve K contiguous
// amplitudes (a 512-byte row at K = 64 complex64).  Each realisation keeps its own Lanczos
// recurrence (alpha_k, beta_k, reorthogonalisation coefficients) in FP64; all share the
// time grid, so the step size is the smallest step every realisation accepts.
//
//   k_apply_b      y = H x for all K (warp per state, lanes over k)
//   k_hv_b         u = H v_j for all K (pass A, part 1)
//   k_alpha_b      alpha_j per realisation (one-read form, from 32,768 elements on)
//   k_ortho_b      update and the dots of the new vector in one read (one-read form)
//   k_dots_b       all dots <v_i, u> and ||u||^2 per realisation (two-pass form: pass A, part 2)
//   k_lincomb_b    update (two-pass form) / correction / combine / load with per-realisation
//                  coefficients, and the dots of the new vector with the earlier ones (pass C1)
//   k_reduce_b     per-realisation sum of the per-CTA partials (deterministic) and the
//                  scalar epilogue of each pass
#include <cuda_runtime.h>

#include <algorithm>
#include <type_traits>

#include "kry_device.cuh"

namespace kry {

struct SmemHeadB {
    uint32_t koff[20];
    uint32_t bsz[20];
};

// Row r of H x for every realisation: the rank arithmetic is the same for all k, the
// lanes of the warp run over k = lane + 32 q (k0 = lane), or one realisation k0 per lane.
template <class V, int KQ>
__device__ __forceinline__ void hv_row_b(const DevBasis &b, const DevHam &hm, const V *__restrict__ x,
                                         int K, uint32_t hi, uint32_t off, int klo,
                                         const uint32_t *koff_s, const uint16_t *rl, V out[KQ], int k0)
{
    using R = typename VT<V>::R;
    const int lane = k0;
    const int Llo = b.Llo, L = b.L;
    const uint32_t pos = koff_s[klo] + off;
    const uint32_t lo = __ldg(b.lolist + pos);
    const uint32_t s = (hi << Llo) | lo;
    const uint32_t base = __ldg(b.blk + hi);
    const uint32_t lomask = (1u << Llo) - 1u;
    const uint32_t obc = (L >= 2) ? ((1u << (L - 1)) - 1u) : 0u;
    const uint32_t anti = (s ^ (s >> 1)) & obc;
    const uint32_t wrap = hm.pbc ? ((s ^ (s >> (L - 1))) & 1u) : 0u;
    const int nanti = __popc(anti) + (int)wrap;
    const R dz = (R)hm.cz * (R)(hm.nbonds - 2 * nanti);
    typename Arith<V>::HvSum acc[KQ];
#pragma unroll
    for (int q = 0; q < KQ; ++q) acc[q] = typename Arith<V>::HvSum{};
    // Neighbour rows in chunks of 4 bond positions (bit 31 = ring bond): the ranks are the
    // same for all lanes; every lane issues its loads of the whole chunk before summing.
    const uint32_t hops = anti | (wrap << 31);
#pragma unroll
    for (int c0 = 0; c0 < 32; c0 += 4) {
        if (!((hops >> c0) & 0xFu)) continue;
        V v[4][KQ];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int p = c0 + u;
#pragma unroll
            for (int q = 0; q < KQ; ++q) v[u][q] = VT<V>::zero();
            if ((hops >> p) & 1u) {
                uint32_t t2;
                if (p == 31) {
                    const uint32_t s2 = s ^ ((1u << (L - 1)) | 1u);
                    t2 = __ldg(b.blk + (s2 >> Llo)) + rl[s2 & lomask];
                } else if (p < Llo - 1) {
                    t2 = base + rl[lo ^ (3u << p)];
                } else if (p == Llo - 1) {
                    const uint32_t s2 = s ^ (3u << p);
                    t2 = __ldg(b.blk + (s2 >> Llo)) + rl[s2 & lomask];
                } else {
                    t2 = __ldg(b.blk + (hi ^ (3u << (p - Llo)))) + off;
                }
                const V *xr = x + (size_t)t2 * K;
#pragma unroll
                for (int q = 0; q < KQ; ++q) {
                    const int k = lane + 32 * q;
                    if (k < K) v[u][q] = ldg(xr + k);
                }
            }
        }
#pragma unroll
        for (int u = 0; u < 4; ++u)
#pragma unroll
            for (int q = 0; q < KQ; ++q) hv_add(acc[q], v[u][q]);
    }
    const V *xr = x + (size_t)(base + off) * K;
#pragma unroll
    for (int q = 0; q < KQ; ++q) {
        const int k = lane + 32 * q;
        if (k < K) {
            const R d = dz + VT<V>::ehlo(hm, pos * K + k) + VT<V>::ehhi(hm, hi * K + k);
            out[q] = hv_finish(d, ldg(xr + k), (R)hm.halfJ, acc[q]);
        } else {
            out[q] = VT<V>::zero();
        }
    }
}

// ---------------------------------------------------------------- y = H x (batched)

template <class V, int KQ>
__global__ void __launch_bounds__(NTHR) k_apply_b(DevBasis b, DevHam hm, int K, const V *__restrict__ x,
                                                  V *__restrict__ y, int rl_smem)
{
    extern __shared__ __align__(16) unsigned char smem[];
    SmemHeadB *hd = (SmemHeadB *)smem;
    uint16_t *rl_s = (uint16_t *)(smem + sizeof(SmemHeadB));
    stage_tables(b, hd->koff, hd->bsz, rl_s, rl_smem);
    __syncthreads();
    const uint16_t *rl = rl_smem ? rl_s : b.ranklo;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t ntiles = (b.D + TROWS - 1) / TROWS;
    for (uint32_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
        const uint32_t r0 = tile * TROWS;
        for (int rr = warp; rr < TROWS; rr += NTHR / 32) {
            if (r0 + rr >= b.D) break;
            uint32_t hi, off;
            int klo;
            tile_unrank(b, hd->bsz, r0, rr, hi, off, klo);
            V u[KQ];
            hv_row_b<V, KQ>(b, hm, x, K, hi, off, klo, hd->koff, rl, u, lane);
#pragma unroll
            for (int q = 0; q < KQ; ++q) {
                const int k = lane + 32 * q;
                if (k < K) y[(size_t)(r0 + rr) * K + k] = u[q];
            }
        }
    }
}

// ---------------------------------------------------------------- pass A (batched)

// Part 1: U[:, k] = sigma_j[k] H_k W_j[:, k] for every realisation (warp per state, lanes over
// k), at full occupancy: nothing but the gathers.  FLAT (K <= 16): a thread per element instead, its
// realisation fixed, because a warp per state would leave half its lanes and more idle.
template <class V, int KQ, bool FLAT>
__global__ void __launch_bounds__(NTHR) k_hv_b(EvArgsB<V> a, int jj)
{
    using R = typename VT<V>::R;
    KryCtlB *ctl = a.ctl;
    if (ctl->hd.done || jj >= ctl->hd.m_run) return;
    extern __shared__ __align__(16) unsigned char smem[];
    SmemHeadB *hd = (SmemHeadB *)smem;
    uint16_t *rl_s = (uint16_t *)(smem + sizeof(SmemHeadB));
    stage_tables(a.b, hd->koff, hd->bsz, rl_s, a.rl_smem);
    __syncthreads();
    const uint16_t *rl = a.rl_smem ? rl_s : a.b.ranklo;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, K = a.K;
    const V *x = a.W + (size_t)jj * a.ldW;
    const uint32_t D = a.b.D;
    if constexpr (FLAT) {
        const uint32_t per = NTHR / K * K;   // elements of a CTA's unit: whole states
        const int k = threadIdx.x % K;
        const R sg = (R)ctl->sigma[jj][k];
        const uint32_t rows = per / K, ntiles = (D + rows - 1) / rows;
        for (uint32_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
            const uint32_t r = tile * rows + threadIdx.x / K;
            if (threadIdx.x >= per || r >= D) break;
            uint32_t hi, off;
            int klo;
            tile_unrank(a.b, hd->bsz, r & ~(uint32_t)(TILE - 1), r & (uint32_t)(TILE - 1), hi, off, klo);
            V u[1];
            hv_row_b<V, 1>(a.b, a.h, x, K, hi, off, klo, hd->koff, rl, u, k);
            a.U[(size_t)r * K + k] = scale(u[0], sg);
        }
    } else {
        R sg[KQ];
#pragma unroll
        for (int q = 0; q < KQ; ++q) {
            const int k = lane + 32 * q;
            sg[q] = (k < K) ? (R)ctl->sigma[jj][k] : (R)0;
        }
        const uint32_t ntiles = (D + TROWS - 1) / TROWS;
        for (uint32_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
            const uint32_t r0 = tile * TROWS;
            for (int rr = warp; rr < TROWS; rr += NTHR / 32) {
                if (r0 + rr >= D) break;
                uint32_t hi, off;
                int klo;
                tile_unrank(a.b, hd->bsz, r0, rr, hi, off, klo);
                V u[KQ];
                hv_row_b<V, KQ>(a.b, a.h, x, K, hi, off, klo, hd->koff, rl, u, lane);
#pragma unroll
                for (int q = 0; q < KQ; ++q) {
                    const int k = lane + 32 * q;
                    if (k < K) a.U[(size_t)(r0 + rr) * K + k] = scale(u[q], sg[q]);
                }
            }
        }
    }
}

// Part 1 in chunks of KCH realisations: the work items are (chunk, tile) pairs in chunk-major
// order and a warp holds 32 / KCH states, KCH lanes each.  The CTAs sweep all tiles of one
// chunk before the next, so the gathered part of W_j (D x KCH amplitudes, e.g. 90 MB for
// L = 22 and KCH = 16 in complex64) stays in L2 while its rows are gathered about eleven
// times each; without chunks the whole [D][K] block (361 MB at K = 64) exceeds L2 and
// gathered rows come from HBM several times.  The rank arithmetic is repeated per chunk.
// Same hop order per amplitude as k_hv_b: the same bits.
template <class V, int KCH>
__global__ void __launch_bounds__(NTHR) k_hv_bc(EvArgsB<V> a, int jj)
{
    using R = typename VT<V>::R;
    KryCtlB *ctl = a.ctl;
    if (ctl->hd.done || jj >= ctl->hd.m_run) return;
    extern __shared__ __align__(16) unsigned char smem[];
    SmemHeadB *hd = (SmemHeadB *)smem;
    uint16_t *rl_s = (uint16_t *)(smem + sizeof(SmemHeadB));
    stage_tables(a.b, hd->koff, hd->bsz, rl_s, a.rl_smem);
    __syncthreads();
    const uint16_t *rl = a.rl_smem ? rl_s : a.b.ranklo;
    constexpr int SPW = 32 / KCH;   // states per warp
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, K = a.K;
    const int sub = lane / KCH, kk = lane % KCH;
    const V *x = a.W + (size_t)jj * a.ldW;
    const uint32_t D = a.b.D, ntiles = (D + TROWS - 1) / TROWS;
    const uint32_t nch = (uint32_t)((K + KCH - 1) / KCH);
    for (uint32_t item = blockIdx.x; item < nch * ntiles; item += gridDim.x) {
        const uint32_t ch = item / ntiles, tile = item - ch * ntiles;
        const int k = (int)ch * KCH + kk;
        const R sg = (k < K) ? (R)ctl->sigma[jj][k] : (R)0;
        const uint32_t r0 = tile * TROWS;
        for (int rr = warp * SPW + sub; rr < TROWS; rr += (NTHR / 32) * SPW) {
            if (r0 + rr >= D) break;
            uint32_t hi, off;
            int klo;
            tile_unrank(a.b, hd->bsz, r0, rr, hi, off, klo);
            V u[1];
            hv_row_b<V, 1>(a.b, a.h, x, K, hi, off, klo, hd->koff, rl, u, k);
            if (k < K) a.U[(size_t)(r0 + rr) * K + k] = scale(u[0], sg);
        }
    }
}

// Part 2: the dots Re <W_i[:, k], U[:, k]>, i <= j, and ||U[:, k]||^2 of every realisation.
// Thread (k, g) takes column k and the vectors i = g, g + NG, ...; the rows of U of a tile
// are loaded once and serve all of them.
template <class V, int KQ>
__global__ void __launch_bounds__(NTHR, 2) k_dots_b(EvArgsB<V> a, int jj)
{
    KryCtlB *ctl = a.ctl;
    if (ctl->hd.done || jj >= ctl->hd.m_run) return;
    // vectors i = g + NG q < MMAX (j <= MMAX - 1)
    constexpr int Kp = 32 * KQ, NG = NTHR / Kp, QD = (MMAX + NG - 1) / NG;
    // rows in registers at a time (16-byte elements with the 16 accumulators of K > 64: four)
    constexpr int RH = sizeof(V) == 16 && KQ == 4 ? TROWS / 4 : TROWS / 2;
    const int tid = threadIdx.x, K = a.K;
    const int k = tid % Kp, g = tid / Kp;
    const uint32_t D = a.b.D, ntiles = (D + TROWS - 1) / TROWS;
    RealAcc<V> acc[QD], nrm;
    if (k < K) {
        for (uint32_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
            const uint32_t r0 = tile * TROWS;
            // rows past D are skipped by one test per RH rows, not per element
            // (a select of FP64 values occupies the FP64 pipe)
#pragma unroll
            for (int h = 0; h < TROWS / RH; ++h) {
                const uint32_t rh = r0 + h * RH;
                const int nr = rh >= D ? 0 : (int)min((uint32_t)RH, D - rh);
                V uu[RH];
#pragma unroll
                for (int rr = 0; rr < RH; ++rr) uu[rr] = VT<V>::zero();
                if (nr == RH) {
#pragma unroll
                    for (int rr = 0; rr < RH; ++rr) uu[rr] = ldg(a.U + (size_t)(rh + rr) * K + k);
                } else {
#pragma unroll
                    for (int rr = 0; rr < RH; ++rr)
                        if (rr < nr) uu[rr] = ldg(a.U + (size_t)(rh + rr) * K + k);
                }
                typename RealAcc<V>::Pre up[RH];
#pragma unroll
                for (int rr = 0; rr < RH; ++rr) up[rr] = RealAcc<V>::pre(uu[rr]);
                if (g == 0) {
#pragma unroll
                    for (int rr = 0; rr < RH; ++rr) nrm.add(uu[rr], up[rr]);
                }
                // rows rh .. rh + RH of vector iv, column k (zero past D)
                auto load = [&](int iv, V *dst) {
                    const V *wi = a.W + (size_t)iv * a.ldW + (size_t)rh * K + k;
                    if (nr == RH) {
#pragma unroll
                        for (int rr = 0; rr < RH; ++rr) dst[rr] = ldg(wi + (size_t)rr * K);
                    } else {
#pragma unroll
                        for (int rr = 0; rr < RH; ++rr) dst[rr] = (rr < nr) ? ldg(wi + (size_t)rr * K) : VT<V>::zero();
                    }
                };
                // (loading the next vector's rows before this one's products
                // needs more registers than the eight accumulators of K = 64 leave, and spills)
#pragma unroll
                for (int q = 0; q < QD; ++q) {
                    const int iv = g + NG * q;
                    if (iv <= jj) {
                        V vv[RH];
                        load(iv, vv);
#pragma unroll
                        for (int rr = 0; rr < RH; ++rr) acc[q].add(vv[rr], up[rr]);
                    }
                }
            }
            // fold the float-float compensations back once per tile
#pragma unroll
            for (int q = 0; q < QD; ++q)
                if (g + NG * q <= jj) acc[q].renorm();
            nrm.renorm();
        }
    }
    double2 *pc = a.part + (size_t)blockIdx.x * PSB * Kp;
#pragma unroll
    for (int q = 0; q < QD; ++q) {
        const int iv = g + NG * q;
        if (iv <= jj) pc[(size_t)iv * Kp + k] = make_double2(to_double(acc[q].sum()), 0.0);
    }
    if (g == 0) pc[(size_t)SLOT_NRM * Kp + k] = make_double2(to_double(nrm.sum()), 0.0);
}


// ---------------------------------------------------------------- linear combinations (batched)

// MODE 0: w = U - sum_i c_i W_i (pure update); 1: the correction of pass C2; 2: combine;
// 3: load psi0; 4: the dots <W_i, W_{j+1}> of pass C1 (no update), for realisations that
// flagged them.
template <class V, int MODE, int KQ>
__global__ void __launch_bounds__(NTHR, 1) k_lincomb_b(EvArgsB<V> a, int jj)
{
    KryCtlB *ctl = a.ctl;
    if (ctl->hd.done) return;
    if ((MODE <= 1 || MODE == 4) && jj >= ctl->hd.m_run) return;
    if (MODE == 1 && !ctl->hd.corr_any) return;
    if (MODE == 4 && !ctl->hd.dots_any) return;
    constexpr int Kp = 32 * KQ, NG = NTHR / Kp, QD = (MMAX + NG) / NG;
    const int nvec = (MODE == 2) ? ctl->hd.m_run : ((MODE == 3 || MODE == 4) ? 0 : jj + 1);
    extern __shared__ __align__(16) unsigned char smem[];
    // modes 0 and 1 subtract real multiples (RealAcc), the combine takes complex ones
    constexpr bool RE = MODE <= 1;
    using Lin = typename std::conditional<RE, RealLin<V>, CplxLin<V>>::type;
    using Coef = typename Lin::RCoef;
    static_assert(sizeof(Coef) <= sizeof(V), "coefficient slots have the element size");
    Coef *coef = (Coef *)smem;                    // [MMAX+1][Kp]
    V *wtile = (V *)smem + (MMAX + 1) * Kp;       // [TROWS][Kp]
    double2 *nred = (double2 *)(wtile + TROWS * Kp);   // [NG][Kp] (norm), then [NG][Kp] (G)
    const int tid = threadIdx.x, K = a.K;
    for (int e = tid; e < nvec * Kp; e += NTHR) {
        const int i = e / Kp, k = e % Kp;
        if constexpr (RE) coef[i * Kp + k] = Lin::coef(k >= K ? 0.0 : MODE == 0 ? ctl->coefA[i][k] : ctl->coefC[i][k]);
        else coef[i * Kp + k] = Lin::coef(k < K ? ctl->coefY[i][k] : make_double2(0.0, 0.0));
    }
    __syncthreads();
    V *out = (MODE == 2 || MODE == 3) ? a.W : a.W + (size_t)(jj + 1) * a.ldW;
    const V *src = (MODE == 0) ? a.U : (MODE == 1 || MODE == 4) ? out : (MODE == 3) ? a.G : nullptr;
    const uint32_t D = a.b.D, ntiles = (D + TROWS - 1) / TROWS;
    const int k = tid % Kp, g = tid / Kp;
    RealAcc<V> acc[QD], nrm;
    DotAcc<V> gacc;
    for (uint32_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
        const uint32_t r0 = tile * TROWS;
        for (int rr = g; rr < TROWS; rr += NG) {
            V w = VT<V>::zero();
            if (r0 + rr < D && k < K) {
                const size_t idx = (size_t)(r0 + rr) * K + k;
                if (src) w = src[idx];
                if (MODE != 4) {
                    Lin wl(w);
                    if (MODE == 2) {
#pragma unroll 8
                        for (int i = 0; i < nvec; ++i) wl.fms(coef[i * Kp + k], a.W[(size_t)i * a.ldW + idx]);
                    } else {
#pragma unroll 8
                        for (int i = 0; i < nvec; ++i) wl.fms(coef[i * Kp + k], ldg(a.W + (size_t)i * a.ldW + idx));
                    }
                    w = (MODE == 3) ? w : wl.out();
                    out[idx] = w;
                    nrm.add(w, RealAcc<V>::pre(w));
                    if (a.G && MODE != 3) gacc.add(ldg(a.G + idx), w);
                }
            }
            if (MODE == 4) wtile[rr * Kp + k] = w;
        }
        nrm.renorm();
        gacc.renorm();
        if (MODE == 4) {
            __syncthreads();
            if (k < K) {
#pragma unroll
                for (int q = 0; q < QD; ++q) {
                    const int iv = g + NG * q;
                    if (iv <= jj) {
                        const V *wi = a.W + (size_t)iv * a.ldW + (size_t)r0 * K + k;
                        V vv[TROWS];
#pragma unroll
                        for (int rr = 0; rr < TROWS; ++rr)
                            vv[rr] = (r0 + rr < D) ? ldg(wi + (size_t)rr * K) : VT<V>::zero();
#pragma unroll
                        for (int rr = 0; rr < TROWS; ++rr) acc[q].add(vv[rr], RealAcc<V>::pre(wtile[rr * Kp + k]));
                        acc[q].renorm();
                    }
                }
            }
            __syncthreads();
        }
    }
    double2 *pc = a.part + (size_t)blockIdx.x * PSB * Kp;
    if (MODE == 4) {
#pragma unroll
        for (int q = 0; q < QD; ++q) {
            const int iv = g + NG * q;
            if (iv <= jj) pc[(size_t)iv * Kp + k] = make_double2(to_double(acc[q].sum()), 0.0);
        }
        return;
    }
    nred[g * Kp + k] = make_double2(to_double(nrm.sum()), 0.0);
    nred[(NG + g) * Kp + k] = gacc.value();
    __syncthreads();
    for (int kk = tid; kk < Kp; kk += NTHR) {
        double2 s = make_double2(0.0, 0.0), t = make_double2(0.0, 0.0);
        for (int gg = 0; gg < NG; ++gg) {
            s.x += nred[gg * Kp + kk].x;
            t.x += nred[(NG + gg) * Kp + kk].x;
            t.y += nred[(NG + gg) * Kp + kk].y;
        }
        pc[(size_t)SLOT_NRM * Kp + kk] = s;
        pc[(size_t)SLOT_G * Kp + kk] = t;
    }
}

// ---------------------------------------------------------------- the one-read pass (batched)

// Threads of a group: the elements of whole states that fit 64 threads, or 128 where that leaves fewer idle.
static __host__ __device__ int ortho_group(int K) { return K > 64 || (K > 32 && K < 64) ? 128 : 64; }
// Threads of a CTA: an even number of groups
// (the 64-bit indices and the coefficients per lane need more registers than k_ortho's)
template <class V, int T> constexpr int ORTHO_B_NTHR = T == 64 && !std::is_same<V, ffc>::value ? 384 : 256;

constexpr int ALPHA_NTHR = 512;

// Re <W_j[:, k], U[:, k]> of every realisation, on k_ortho_b's split of the elements: the CTAs' shares go to
// part[CTA][Kp] (doubles).  A pass of its own, because the H.v's forms split the states in different ways
// and alpha_j's bits must not depend on them; two of the step's j + 5 vector reads.  In the first Krylov step
// also c_0 = Re <W_0[:, k], U[:, k]> (see alpha_epilogue), to part[gridDim + CTA][Kp].
template <class V, int T>
__global__ void __launch_bounds__(ALPHA_NTHR) k_alpha_b(EvArgsB<V> a, int jj)
{
    KryCtlB *ctl = a.ctl;
    if (ctl->hd.done || jj >= ctl->hd.m_run) return;
    constexpr int NGRP = ALPHA_NTHR / T, NU = 4;
    using Sum = typename RealAcc<V>::Sum;
    __shared__ Sum sums[ALPHA_NTHR];
    const int K = a.K, tid = threadIdx.x, g = tid / T, t = tid % T;
    const uint32_t unit = T / K * K;
    const size_t n = (size_t)a.b.D * K;
    const uint32_t nu = (uint32_t)((n + unit - 1) / unit), du = gridDim.x * NGRP;
    const bool first = jj > 0 && ctl->hd.n_steps == 0;
    auto dots = [&](const V *x, double *out) {
        RealAcc<V> al;
        for (uint32_t u0 = blockIdx.x * NGRP + g; u0 < nu; u0 += NU * du) {
            V xv[NU], uv[NU];
#pragma unroll
            for (int q = 0; q < NU; ++q) {
                const size_t r = (size_t)(u0 + q * du) * unit + t;
                const bool in = t < (int)unit && u0 + q * du < nu && r < n;
                xv[q] = ldg_if(in, x + r);
                uv[q] = ldg_if(in, a.U + r);
            }
#pragma unroll
            for (int q = 0; q < NU; ++q) al.add(xv[q], RealAcc<V>::pre(uv[q]));
            al.renorm();
        }
        __syncthreads();
        sums[tid] = al.sum();
        __syncthreads();
        if (tid < a.Kp) {
            Sum tot{};
            if (tid < K)
                for (int gg = 0; gg < NGRP; ++gg)
                    for (uint32_t r = tid; r < unit; r += K) tot = add2(tot, sums[gg * T + r]);
            out[(size_t)blockIdx.x * a.Kp + tid] = to_double(tot);
        }
    };
    double *part = (double *)a.part;
    dots(a.W + (size_t)jj * a.ldW, part);
    if (!first) return;
    part += (size_t)gridDim.x * a.Kp;
    if (a.G) dots(a.W, part);
    else if (tid < a.Kp)   // basis states: one element
        part[(size_t)blockIdx.x * a.Kp + tid] =
            blockIdx.x == 0 && tid < K ? real_part(a.U + (size_t)ctl->r0k[tid] * K + tid) : 0.0;
}

// k_ortho for K realisations: thread t of a group takes the element of state t / K and realisation t % K of
// its unit of T / K states, so that its accumulators belong to one realisation; the coefficients are kept
// per realisation in shared memory.  At the end the sums of a realisation's threads go to part[CTA][slot].
// The two-pass form pads K to 32, 64 or 128 lanes and reads the vectors twice.
template <class V, int T>
__global__ void __launch_bounds__(ORTHO_B_NTHR<V, T>, 1) k_ortho_b(EvArgsB<V> a, int jj)
{
    KryCtlB *ctl = a.ctl;
    if (ctl->hd.done || jj >= ctl->hd.m_run) return;
    constexpr int QV = ORTHO_QV, NT = ORTHO_B_NTHR<V, T>, NGRP = NT / T;
    using RCoef = typename RealLin<V>::RCoef;
    using Sum = typename RealAcc<V>::Sum;
    extern __shared__ __align__(16) unsigned char smem[];
    const int K = a.K, tid = threadIdx.x, g = tid / T, t = tid % T;
    const uint32_t unit = T / K * K;
    const int k = t % K;   // (threads past the unit sum zeros)
    RCoef *coef = (RCoef *)smem;                              // [MMAX + 1][K]
    float *mcoef = (float *)(coef + (MMAX + 1) * K);          // [MMAX + 1][K]
    const size_t off = ((sizeof(RCoef) + sizeof(float)) * (MMAX + 1) * K + 15) & ~(size_t)15;
    V *xch = (V *)(smem + off);                               // [2][NGRP][T][XU]
    Sum *sums = (Sum *)(smem + off);                          // afterwards [QV + 3][NT]
    bool mine = true;
    for (int e = tid; e < (jj + 1) * K; e += NT) {
        const double c = ctl->coefA[e / K][e % K];
        coef[e] = RealLin<V>::coef(c);
        mcoef[e] = -(float)c;
    }
    if (MinorSum<V>::use && tid < K) mine = ctl->minor[tid] != 0;
    const bool minor = __syncthreads_and(mine) && MinorSum<V>::use;
    const int nv = jj + 1;
    const int nvg = nv <= QV ? 1 : 2, nrp = NGRP / nvg;
    const int rp = g / nvg, vg = (g + rp) % nvg;
    const int i0 = (nv * vg) / nvg, nq = (nv * (vg + 1)) / nvg - i0, pad = ortho_pad(nq);
    const size_t n = (size_t)a.b.D * K;
    const uint32_t nu = (uint32_t)((n + unit - 1) / unit), du = gridDim.x * nrp;
    RealAcc<V> acc[QV], nrm;
    DotAcc<V> gacc;
    V *out = a.W + (size_t)(jj + 1) * a.ldW;
#define KRY_ORTHO(NQ, NU, KIND)                                                                                      \
    ortho_rows<V, NQ, NU, KIND, T, NGRP, 2>(a.W, a.ldW, a.U, a.G, out, n, unit, t, i0, nq, minor, rp, blockIdx.x * nrp + rp, \
                                      du, nu, jj & 1, coef + k, mcoef + k, K, xch, acc, nrm, gacc)
#define KRY_ORTHO_N(NQ, NU) \
    case NQ: KRY_ORTHO(NQ, NU, ORTHO_ONLY); break;
#define KRY_ORTHO_3(NQ)                                           \
    case NQ:                                                      \
        if (nvg == 1) KRY_ORTHO(NQ, 1, ORTHO_ONLY);               \
        else if (vg == 0) KRY_ORTHO(NQ, 1, ORTHO_FIRST);          \
        else KRY_ORTHO(NQ, 1, ORTHO_LAST);                        \
        break;
    if (rp < nrp) {
        switch (nq + pad) {
            KRY_ORTHO_N(1, 8)
            KRY_ORTHO_N(2, 4)
            KRY_ORTHO_N(3, 4)
            KRY_ORTHO_N(4, 4)
            KRY_ORTHO_N(6, 2)
            KRY_ORTHO_3(8)
            KRY_ORTHO_3(10)
            KRY_ORTHO_3(12)
            KRY_ORTHO_3(14)
            KRY_ORTHO_3(15)
            KRY_ORTHO_3(16)
        default: break;
        }
    }
#undef KRY_ORTHO_3
#undef KRY_ORTHO_N
#undef KRY_ORTHO
    __syncthreads();   // (the exchange buffers become the sums)
#pragma unroll
    for (int q = 0; q < QV; ++q) {
        acc[q].renorm();
        sums[q * NT + tid] = acc[q].sum();
    }
    nrm.renorm();
    sums[QV * NT + tid] = nrm.sum();
    if (a.G) {
        gacc.renorm();
        const double2 gv = gacc.value();
        sums[(QV + 1) * NT + tid] = from_double<Sum>(gv.x);
        sums[(QV + 2) * NT + tid] = from_double<Sum>(gv.y);
    }
    __syncthreads();
    double2 *pc = a.part + (size_t)blockIdx.x * PSB * a.Kp;
    const int nslot = nv + 1 + (a.G ? 2 : 0);
    for (int e = tid; e < nslot * K; e += NT) {
        const int i = e / K, kk = e % K;
        int s = 0, q;   // the share and slot that hold sum i
        if (i < nv) {
            s = nvg == 1 || i < nv / 2 ? 0 : 1;
            const int f = s ? nv / 2 : 0, ns = nvg == 1 ? nv : s ? nv - nv / 2 : nv / 2;
            q = i - f + ortho_pad(ns);
        } else {
            q = QV + (i - nv);
        }
        Sum tot{};
        for (int p = 0; p < nrp; ++p) {
            const int gg = p * nvg + (nvg == 1 ? 0 : (s + p) & 1);   // the group of share s in part p
            for (uint32_t r = kk; r < unit; r += K) tot = add2(tot, sums[q * NT + gg * T + r]);
        }
        const double v = to_double(tot);
        if (i < nv) pc[(size_t)i * a.Kp + kk] = make_double2(v, 0.0);
        else if (i == nv) pc[(size_t)SLOT_NRM * a.Kp + kk] = make_double2(v, 0.0);
        else if (i == nv + 1) pc[(size_t)SLOT_G * a.Kp + kk].x = v;
        else pc[(size_t)SLOT_G * a.Kp + kk].y = v;
    }
}

// ---------------------------------------------------------------- per-realisation reductions

// mode: 0 pass A, 1 pass B, 3 pass C1 (dots of w), 2 pass C2 (correction), 4 combine,
// 5 load of a general psi0; one-read form: 6 alpha_j, c_0 and the update's coefficients (partials of
// k_alpha_b), 7 the dots and the norm of the update (see k_ortho).  One CTA per realisation.  A warp takes a whole slot (lanes over the
// CTAs' partials) and lane i of warp 0 the scalars of vector i: GB300 issues
// one FP64 warp instruction per about 77 cycles and SM sub-partition whatever its active lanes, so
// block-wide trees slot by slot and loops over the vectors in one thread cost tens of us at j = 30.
__global__ void __launch_bounds__(256) k_reduce_b(KryCtlB *ctl, const double2 *__restrict__ part,
                                                  int grid, int Kp, int mode, int jj, int general, float *Cb,
                                                  float *db)
{
    KryHdrB &H = ctl->hd;
    if (H.done) return;
    if ((mode <= 3 || mode >= 6) && jj >= H.m_run) return;
    const int k = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (mode == 2 && !H.corr_any) return;   // pass C2 did not run
    if (mode == 3 && !H.dots_any) return;   // pass C1 did not run
    __shared__ double2 fin[PSB];
    __shared__ float Cs[MMAX * MMAX], ds[MMAX + 1];
    // one-read form: lane i's coefficient c_i, after pass C2 with its correction (1 / sigma_i is the norm that
    // made v_i)
    double ci = 0.0;
    if (Cb && (mode == 7 || mode == 2) && tid <= jj)
        ci = (ctl->coefA[tid][k] + (mode == 2 ? ctl->coefC[tid][k] : 0.0)) * (tid ? ctl->beta[tid - 1][k] : ctl->beta0[k]);
    const int nd = (mode == 0 || mode == 3 || mode == 7) ? jj + 1 : 0;
    const int ns = mode == 6 ? 0 : nd + (mode != 3 ? 1 : 0) + (general && mode != 0 && mode != 3 ? 1 : 0);
    if (mode == 6) {
        for (int e = tid; e < MMAX * MMAX; e += 256) Cs[e] = Cb[(size_t)k * MMAX * MMAX + e];
        if (tid <= MMAX) ds[tid] = tid < jj ? db[(size_t)k * MMAX + tid] : 0.f;
        if (warp == 0 || (warp == 1 && jj > 0 && H.n_steps == 0)) {   // alpha_j; c_0
            const double *pa = (const double *)part + (size_t)warp * grid * Kp;
            double s = 0.0;
            for (int c0 = 0; c0 < grid; c0 += 256) {
                double x[8];
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const int c = c0 + 32 * i + lane;
                    x[i] = c < grid ? __ldg(pa + (size_t)c * Kp + k) : 0.0;
                }
                s += warp_sum_int<8>(x);
            }
            if (lane == 0) fin[warp].x = s;
        }
    }
    for (int q = warp; q < ns; q += 8) {
        const int slot = q < nd ? q : q == nd ? SLOT_NRM : SLOT_G;
        double2 s = make_double2(0.0, 0.0);
        const bool cplx = slot == SLOT_G;   // the others are real
        for (int c0 = 0; c0 < grid; c0 += 256) {
            double x[8], y[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const int c = c0 + 32 * i + lane;
                double2 v = make_double2(0.0, 0.0);
                if (c < grid) v = __ldg(part + ((size_t)c * PSB + slot) * Kp + k);
                x[i] = v.x;
                y[i] = v.y;
            }
            s.x += warp_sum_int<8>(x);
            if (cplx) s.y += warp_sum_int<8>(y);
        }
        if (lane == 0) fin[slot] = s;
    }
    __syncthreads();
    if (tid >= 32) return;
    const double nw2 = (mode == 3) ? ctl->wnorm2[k] : fin[SLOT_NRM].x;
    const double2 gdot = (mode == 3) ? ctl->wg[k]
                                     : ((general && mode != 0) ? fin[SLOT_G] : make_double2(0.0, 0.0));
    // lane i: Re <v_i, y> = c, c sigma_i (modes 0 and 3)
    double c = 0.0, cs = 0.0;
    if (lane < nd) {
        const double s = ctl->sigma[lane][k];
        c = fin[lane].x * s;
        cs = c * s;
    }
    if (mode == 6) {
        if (k == 0 && lane == 0) {
            H.n_hv += 1;
            H.vec_passes += 2;
            H.vp_kind[KIND_HV] += 2;
            H.corr_any = 0;
            H.dots_any = 0;
        }
        const bool run = jj < ctl->m_eff[k], inv = lane <= jj;
        const double s = inv ? ctl->sigma[lane][k] : 0.0, alpha = fin[0].x * ctl->sigma[jj][k];
        double cc = 0.0;
        if (lane < jj) {
            float f = 0.f;
            for (int i = 0; i <= lane; ++i) f = fmaf(Cs[i * MMAX + lane], ds[i], f);
            const double b = ctl->beta[lane][k];
            const bool sub = lane == jj - 1;   // d_j = 1
            cc = fma(b, (double)(sub ? f : f + ds[lane + 1]), sub ? b : 0.0);
        } else if (lane == jj) {
            cc = alpha;
        }
        if (lane == 0 && jj > 0 && H.n_steps == 0) cc = fin[1].x * s;
        if (!run) cc = 0.0;   // (invariant subspace already reached: the next vectors stay zero)
        const double q2 = cc * cc, c2 = warp_sum_int<1>(&q2);
        const bool small = lane + 1 < jj;
        const double cm = small ? q2 : 0.0, m2 = warp_sum_int<1>(&cm), big = small ? 0.0 : q2, b2 = warp_sum_int<1>(&big);
        // rounding level (MinorSum; its bound for complex128, the smaller one, for both types)
        const bool minor = __all_sync(0xffffffffu, !small || !run || (s >= 0x1p-40 && s <= 0x1p40)) &&
                           m2 <= MinorSum<double2>::eta * MinorSum<double2>::eta * b2;
        if (inv) ctl->coefA[lane][k] = cc * s;
        if (lane != 0) return;
        ctl->c2[k] = c2;
        ctl->minor[k] = minor ? 1 : 0;
        if (run) ctl->alpha[jj][k] = alpha;
        return;
    }
    auto finalize = [&](double w2, double2 gd) {
        const double bt = sqrt(w2);
        ctl->beta[jj][k] = bt;
        if (!(bt > H.eta_bd * sqrt(ctl->normu2[k]))) {
            ctl->m_eff[k] = jj + 1;
            atomicAdd(&H.n_bd, 1ull);
            ctl->sigma[jj + 1][k] = 0.0;
        } else {
            const double s = 1.0 / bt;
            ctl->sigma[jj + 1][k] = s;
            ctl->g[jj + 1][k] = make_double2(gd.x * s, gd.y * s);
        }
    };
    if (mode == 0) {
        if (k == 0 && lane == 0) {
            H.n_hv += 1;
            H.vec_passes += jj + 4;
            H.vp_kind[KIND_PASSA] += jj + 2;   // u and v_0 .. v_j
            H.vp_kind[KIND_HV] += 2;                  // the H.v: v_j read, u written
            H.corr_any = 0;
            H.dots_any = 0;
        }
        // (invariant subspace already reached: this realisation's next vectors stay zero)
        const bool run = jj < ctl->m_eff[k];
        if (lane <= jj) ctl->coefA[lane][k] = run ? cs : 0.0;
        if (run && lane == jj) ctl->alpha[jj][k] = c;
        if (run && lane == 0) ctl->normu2[k] = nw2;
    } else if (mode == 1) {
        if (k == 0 && lane == 0) {
            H.vec_passes += jj + 3 + (general ? 1 : 0);
            H.vp_kind[KIND_PASSB] += jj + 3 + (general ? 1 : 0);
        }
        if (lane <= jj) ctl->coefC[lane][k] = 0.0;
        if (lane != 0) return;
        ctl->corr[k] = 0;
        ctl->dots[k] = 0;
        if (jj >= ctl->m_eff[k]) return;
        // One classical Gram-Schmidt pass is enough unless the projection cancelled most of
        // u (||w|| < eta ||u||, the Daniel-Gragg-Kaufman-Stewart test); then this
        // realisation takes the dots of w with every previous vector (pass C1).
        if (H.verify || nw2 < H.eta_cancel * H.eta_cancel * ctl->normu2[k]) {
            ctl->dots[k] = 1;
            ctl->wnorm2[k] = nw2;
            ctl->wg[k] = gdot;
            H.dots_any = 1;
        } else {
            finalize(nw2, gdot);
        }
    } else if (mode == 7) {
        if (k == 0 && lane == 0) {
            H.vec_passes += jj + 3 + (general ? 1 : 0);
            H.vp_kind[KIND_PASSB] += jj + 3 + (general ? 1 : 0);
        }
        const double cc = c * c, nd2 = warp_sum_int<1>(&cc);
        const bool run = jj < ctl->m_eff[k];
        const double normu2 = ctl->c2[k] + nw2;   // ||u||^2 = ||c||^2 + ||w||^2
        const bool dead = !(nw2 > H.eta_bd * H.eta_bd * normu2);
        const bool sub = run && nw2 > 0.0 && nd2 > H.eta_corr * H.eta_corr * nw2;   // (as in k_ortho)
        if (lane <= jj) {
            const double rb = rsqrt(nw2);
            const bool off = sub || dead || !run;   // (after a subtraction mode 2 sets C)
            ctl->coefC[lane][k] = sub ? cs : 0.0;
            Cb[((size_t)k * MMAX + lane) * MMAX + jj] = off ? 0.f : (float)(ci * rb);
            db[(size_t)k * MMAX + lane] = off ? 0.f : (float)(c * rb);
        }
        if (sub && lane == jj) ctl->alpha[jj][k] += c;
        if (lane != 0) return;
        ctl->corr[k] = sub ? 1 : 0;
        if (!run) return;
        ctl->normu2[k] = normu2;
        if ((H.verify || sub) && nw2 > 0.0) ctl->orth[k] = fmax(ctl->orth[k], sqrt(nd2 / nw2));
        if (sub) H.corr_any = 1;
        else finalize(nw2, gdot);
    } else if (mode == 3) {
        if (k == 0 && lane == 0) {
            H.vec_passes += jj + 2;
            H.vp_kind[KIND_PASSC] += jj + 2;
        }
        if (!ctl->dots[k] || jj >= ctl->m_eff[k]) return;
        const double cc = c * c, nd2 = warp_sum_int<1>(&cc);
        const bool sub = nw2 > 0.0 && sqrt(nd2) > H.eta_corr * sqrt(nw2);
        if (sub && lane <= jj) ctl->coefC[lane][k] = cs;
        if (sub && lane == jj) ctl->alpha[jj][k] += c;
        if (lane != 0) return;
        if (nw2 > 0.0) ctl->orth[k] = fmax(ctl->orth[k], sqrt(nd2 / nw2));
        if (sub) {
            ctl->corr[k] = 1;
            H.corr_any = 1;
        } else {
            finalize(nw2, gdot);
        }
    } else if (mode == 2) {
        if (Cb && lane <= jj && jj < ctl->m_eff[k] && ctl->corr[k])
            Cb[((size_t)k * MMAX + lane) * MMAX + jj] = (float)(ci * rsqrt(nw2));
        if (lane != 0) return;
        if (k == 0) {
            H.vec_passes += jj + 3 + (general ? 1 : 0);
            H.vp_kind[KIND_PASSC] += jj + 3 + (general ? 1 : 0);
        }
        if (jj < ctl->m_eff[k] && ctl->corr[k]) {
            atomicAdd(&H.n_corr, 1ull);
            finalize(nw2, gdot);
        }
    } else if (lane == 0) {   // 4 combine, 5 load of psi0
        const double b0 = sqrt(nw2);
        if (!(b0 > 0.0)) {
            H.err = KRY_EINVAL;
            H.done = 1;
            return;
        }
        ctl->beta0[k] = b0;
        ctl->sigma[0][k] = 1.0 / b0;
        ctl->g[0][k] = (mode == 5) ? make_double2(b0, 0.0) : make_double2(gdot.x / b0, gdot.y / b0);
        ctl->m_eff[k] = H.m;
        ctl->corr[k] = 0;
    }
}

// Shared bookkeeping after the combine (one thread): advance time, count the step.
__global__ void k_step_done_b(KryCtlB *ctl, int general)
{
    KryHdrB &H = ctl->hd;
    if (H.done) return;
    double e = 0.0;
    for (int k = 0; k < H.K; ++k) e = fmax(e, ctl->err_k[k]);
    H.err_sum += e;
    H.n_steps += 1;
    H.vec_passes += H.m_run + 1 + (general ? 1 : 0);
    H.vp_kind[KIND_COMBINE] += H.m_run + 1 + (general ? 1 : 0);
    H.t_now = H.t_next;
    H.next_out = H.next_out_new;
    H.m_run = H.m;
    H.corr_any = 0;
    if (H.finishing) H.done = 1;
}

// m_run refresh after pass C ran (all per-realisation epilogues of pass C are complete).
__global__ void k_mrun_b(KryCtlB *ctl)
{
    KryHdrB &H = ctl->hd;
    if (H.done) return;
    int mr = 0;
    for (int k = 0; k < H.K; ++k) mr = max(mr, ctl->m_eff[k]);
    H.m_run = mr;
}

// psi0_k = e_{r0_k}: each realisation starts from its own basis state
template <class V>
__global__ void k_set_basis_state_b(V *W0, int K, const KryCtlB *ctl)
{
    const int k = threadIdx.x;
    if (k < K) W0[(size_t)ctl->r0k[k] * K + k] = VT<V>::from(make_double2(1.0, 0.0));
}

// ---------------------------------------------------------------- launchers

static int sm_count_b()
{
    static int n = 0;
    if (!n) {
        int dev = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
        if (n <= 0) n = 1;
    }
    return n;
}

static size_t hv_b_smem(const DevBasis &b, int rl_smem)
{
    return sizeof(SmemHeadB) + (rl_smem ? (sizeof(uint16_t) << b.Llo) : 0);
}

static size_t lincomb_b_smem(int Kp, size_t es)
{
    return es * (MMAX + 1) * Kp + es * TROWS * Kp + sizeof(double2) * 2 * NTHR;
}

template <class K_>
static int set_smem(K_ kernel, size_t smem)
{
    if (smem > 48 * 1024) KRY_CU(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    return KRY_OK;
}

#define KRY_KQ_SWITCH(Kp, ...)                                \
    switch (Kp) {                                             \
    case 32: { constexpr int KQ = 1; __VA_ARGS__; } break;    \
    case 64: { constexpr int KQ = 2; __VA_ARGS__; } break;    \
    default: { constexpr int KQ = 4; __VA_ARGS__; } break;    \
    }

// CTAs of the batched dots (returned) and of the updates (*gridB): whole SMs times the
// resident CTAs of each.
template <class V>
int batched_grid(const DevBasis &b, int Kp, int rl_smem, int *gridB)
{
    const size_t es = sizeof(V);
    int o1 = 1, o2 = 1;
    KRY_KQ_SWITCH(Kp, {
        if (int rc = set_smem(k_hv_b<V, KQ, false>, hv_b_smem(b, rl_smem))) return -rc;
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&o1, k_dots_b<V, KQ>, NTHR, 0);
        const size_t sL = lincomb_b_smem(Kp, es);
        if (int rc = set_smem(k_lincomb_b<V, 0, KQ>, sL)) return -rc;
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&o2, k_lincomb_b<V, 0, KQ>, NTHR, sL);
    });
    const uint32_t ntiles = (b.D + TROWS - 1) / TROWS;
    auto fit = [&](int occ) {
        return (int)std::max<uint32_t>(1u, std::min<uint32_t>(ntiles, (uint32_t)(sm_count_b() * std::max(1, occ))));
    };
    *gridB = fit(o2);
    return fit(o1);
}

// The H.v at full occupancy, its own grid
template <class V>
static int launch_hv_b(const EvArgsB<V> &a, int jj, cudaStream_t s)
{
    const size_t sH = hv_b_smem(a.b, a.rl_smem);
    auto go = [&](auto kernel, uint32_t items) {
        int oh = 0;
        if (int rc = set_smem(kernel, sH)) return rc;
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&oh, kernel, NTHR, sH);
        const int grid = (int)std::max<uint32_t>(1u, std::min<uint32_t>(items, (uint32_t)(sm_count_b() * std::max(1, oh))));
        kernel<<<grid, NTHR, sH, s>>>(a, jj);
        KRY_CU(cudaGetLastError());
        return (int)KRY_OK;
    };
    if (a.K <= 16) {
        const uint32_t rows = (uint32_t)(NTHR / a.K);
        return go(k_hv_b<V, 1, true>, (a.b.D + rows - 1) / rows);
    }
    KRY_KQ_SWITCH(a.Kp, { return go(k_hv_b<V, KQ, false>, (a.b.D + TROWS - 1) / TROWS); });
    return KRY_OK;
}

// alpha_j's partial sums; returns the CTAs (the reduction's grid), or minus a status
template <class V>
int launch_alpha_b(const EvArgsB<V> &a, int jj, cudaStream_t s)
{
    const size_t units = ((size_t)a.b.D * a.K + ALPHA_NTHR - 1) / ALPHA_NTHR;
    const int grid = (int)std::max<size_t>(1, std::min<size_t>((units + 3) / 4, (size_t)sm_count_b() * 2));
    if (ortho_group(a.K) == 64) k_alpha_b<V, 64><<<grid, ALPHA_NTHR, 0, s>>>(a, jj);
    else k_alpha_b<V, 128><<<grid, ALPHA_NTHR, 0, s>>>(a, jj);
    const cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? grid : -cuda_fail(e, "k_alpha_b");
}

template <class V>
int launch_ortho_b(const EvArgsB<V> &a, int jj, int grid, cudaStream_t s)
{
    auto go = [&](auto kernel, int nt) {
        const size_t off = ((sizeof(typename RealLin<V>::RCoef) + sizeof(float)) * (MMAX + 1) * a.K + 15) & ~(size_t)15;
        const size_t sm = off + std::max(sizeof(V) * 2 * nt * ORTHO_XU, sizeof(typename RealAcc<V>::Sum) * (ORTHO_QV + 3) * nt);
        if (int rc = set_smem(kernel, sm)) return rc;
        kernel<<<grid, nt, sm, s>>>(a, jj);
        KRY_CU(cudaGetLastError());
        return (int)KRY_OK;
    };
    return ortho_group(a.K) == 64 ? go(k_ortho_b<V, 64>, ORTHO_B_NTHR<V, 64>) : go(k_ortho_b<V, 128>, ORTHO_B_NTHR<V, 128>);
}

// pass A: the H.v at full occupancy (its own grid), then the dots on the common grid
// (their partials feed k_reduce_b); part 1 launches the H.v alone, part 2 the dots alone
template <class V>
int launch_passA_b(const EvArgsB<V> &a, int jj, int grid, cudaStream_t s, int part)
{
    if (part == 2) {
        KRY_KQ_SWITCH(a.Kp, { k_dots_b<V, KQ><<<grid, NTHR, 0, s>>>(a, jj); });
        KRY_CU(cudaGetLastError());
        return KRY_OK;
    }
    if (a.b.list) {
        if (int rc = launch_list_hv_b<V>(a, jj, s)) return rc;
        if (part == 1) return KRY_OK;
        KRY_KQ_SWITCH(a.Kp, { k_dots_b<V, KQ><<<grid, NTHR, 0, s>>>(a, jj); });
        KRY_CU(cudaGetLastError());
        return KRY_OK;
    }
    const size_t sH = hv_b_smem(a.b, a.rl_smem);
    const uint32_t ntiles = (a.b.D + TROWS - 1) / TROWS;
    auto hv_grid = [&](auto kernel, uint32_t items) {
        int oh = 0;
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&oh, kernel, NTHR, sH);
        return (int)std::max<uint32_t>(1u, std::min<uint32_t>(items, (uint32_t)(sm_count_b() * std::max(1, oh))));
    };
    if (a.kch == 8 || a.kch == 16) {   // chunks of realisations (launch shape part 4)
        const uint32_t items = ntiles * (uint32_t)((a.K + a.kch - 1) / a.kch);
        if (a.kch == 8) {
            if (int rc = set_smem(k_hv_bc<V, 8>, sH)) return rc;
            k_hv_bc<V, 8><<<hv_grid(k_hv_bc<V, 8>, items), NTHR, sH, s>>>(a, jj);
        } else {
            if (int rc = set_smem(k_hv_bc<V, 16>, sH)) return rc;
            k_hv_bc<V, 16><<<hv_grid(k_hv_bc<V, 16>, items), NTHR, sH, s>>>(a, jj);
        }
        KRY_CU(cudaGetLastError());
    } else {
        if (int rc = launch_hv_b<V>(a, jj, s)) return rc;
    }
    if (part == 1) return KRY_OK;
    KRY_KQ_SWITCH(a.Kp, { k_dots_b<V, KQ><<<grid, NTHR, 0, s>>>(a, jj); });
    KRY_CU(cudaGetLastError());
    return KRY_OK;
}

template <class V>
int launch_lincomb_b(const EvArgsB<V> &a, int mode, int jj, int grid, cudaStream_t s)
{
    const size_t sL = lincomb_b_smem(a.Kp, sizeof(V));
    KRY_KQ_SWITCH(a.Kp, {
        switch (mode) {
        case 0: if (int rc = set_smem(k_lincomb_b<V, 0, KQ>, sL)) return rc; k_lincomb_b<V, 0, KQ><<<grid, NTHR, sL, s>>>(a, jj); break;
        case 1: if (int rc = set_smem(k_lincomb_b<V, 1, KQ>, sL)) return rc; k_lincomb_b<V, 1, KQ><<<grid, NTHR, sL, s>>>(a, jj); break;
        case 2: if (int rc = set_smem(k_lincomb_b<V, 2, KQ>, sL)) return rc; k_lincomb_b<V, 2, KQ><<<grid, NTHR, sL, s>>>(a, jj); break;
        case 4: if (int rc = set_smem(k_lincomb_b<V, 4, KQ>, sL)) return rc; k_lincomb_b<V, 4, KQ><<<grid, NTHR, sL, s>>>(a, jj); break;
        default: if (int rc = set_smem(k_lincomb_b<V, 3, KQ>, sL)) return rc; k_lincomb_b<V, 3, KQ><<<grid, NTHR, sL, s>>>(a, jj); break;
        }
    });
    KRY_CU(cudaGetLastError());
    return KRY_OK;
}

// mode 0, 1 follow passes A, B; 3 and 2 passes C1 and C2; 4 the combine (then the shared
// step bookkeeping); 5 the load of a general psi0.
int launch_reduce_b(KryCtlB *ctl, const double2 *part, int grid, int K, int Kp, int mode, int jj,
                    int general, cudaStream_t s, float *C, float *d)
{
    k_reduce_b<<<K, 256, 0, s>>>(ctl, part, grid, Kp, mode, jj, general, C, d);
    KRY_CU(cudaGetLastError());
    if (mode == 2) {
        k_mrun_b<<<1, 1, 0, s>>>(ctl);
        KRY_CU(cudaGetLastError());
    }
    if (mode == 4) {
        k_step_done_b<<<1, 1, 0, s>>>(ctl, general);
        KRY_CU(cudaGetLastError());
    }
    return KRY_OK;
}

int launch_apply_b(const DevBasis &b, const DevHam &h, int c64, int K, const void *x, void *y,
                   int rl_smem, cudaStream_t s)
{
    if (b.list) return launch_list_apply(b, h, c64, K, x, y, s);
    int Kp = 32;
    while (Kp < K) Kp *= 2;
    const size_t smem = sizeof(SmemHeadB) + (rl_smem ? (sizeof(uint16_t) << b.Llo) : 0);
    const uint32_t ntiles = (b.D + TROWS - 1) / TROWS;
    const int grid = (int)std::min<uint32_t>(ntiles, (uint32_t)sm_count_b() * 8u);
    KRY_KQ_SWITCH(Kp, {
        if (c64) {
            if (int rc = set_smem(k_apply_b<float2, KQ>, smem)) return rc;
            k_apply_b<float2, KQ><<<grid, NTHR, smem, s>>>(b, h, K, (const float2 *)x, (float2 *)y, rl_smem);
        } else {
            if (int rc = set_smem(k_apply_b<double2, KQ>, smem)) return rc;
            k_apply_b<double2, KQ><<<grid, NTHR, smem, s>>>(b, h, K, (const double2 *)x, (double2 *)y, rl_smem);
        }
    });
    KRY_CU(cudaGetLastError());
    return KRY_OK;
}

int launch_set_basis_state_b(void *W0, int c64, int K, const KryCtlB *ctl, cudaStream_t s, int ff)
{
    if (c64) k_set_basis_state_b<float2><<<1, KBMAX, 0, s>>>((float2 *)W0, K, ctl);
    else if (ff) k_set_basis_state_b<ffc><<<1, KBMAX, 0, s>>>((ffc *)W0, K, ctl);
    else k_set_basis_state_b<double2><<<1, KBMAX, 0, s>>>((double2 *)W0, K, ctl);
    KRY_CU(cudaGetLastError());
    return KRY_OK;
}

template int launch_alpha_b<ffc>(const EvArgsB<ffc> &, int, cudaStream_t);
template int launch_ortho_b<ffc>(const EvArgsB<ffc> &, int, int, cudaStream_t);
template int batched_grid<ffc>(const DevBasis &, int, int, int *);
template int launch_passA_b<ffc>(const EvArgsB<ffc> &, int, int, cudaStream_t, int);
template int launch_lincomb_b<ffc>(const EvArgsB<ffc> &, int, int, int, cudaStream_t);
template int launch_alpha_b<double2>(const EvArgsB<double2> &, int, cudaStream_t);
template int launch_ortho_b<double2>(const EvArgsB<double2> &, int, int, cudaStream_t);
template int batched_grid<double2>(const DevBasis &, int, int, int *);
template int launch_alpha_b<float2>(const EvArgsB<float2> &, int, cudaStream_t);
template int launch_ortho_b<float2>(const EvArgsB<float2> &, int, int, cudaStream_t);
template int batched_grid<float2>(const DevBasis &, int, int, int *);
template int launch_passA_b<double2>(const EvArgsB<double2> &, int, int, cudaStream_t, int);
template int launch_passA_b<float2>(const EvArgsB<float2> &, int, int, cudaStream_t, int);
template int launch_lincomb_b<double2>(const EvArgsB<double2> &, int, int, int, cudaStream_t);
template int launch_lincomb_b<float2>(const EvArgsB<float2> &, int, int, int, cudaStream_t);

}  // namespace kry

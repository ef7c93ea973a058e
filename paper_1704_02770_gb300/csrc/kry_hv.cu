// Vector kernels of the Krylov step (Sec. 2, "Krylov subspace methods"):
//   k_apply     y = H x (matrix-free, Eq. 1)
//   k_hv        u = sigma_j H v_j (pass A, part 1); in the one-read form also alpha_j = Re <v_j, u>
//   k_dots      Re <v_i, y> for the Krylov vectors, a tall-skinny GEMV with plain loads (two-pass
//               form: pass A part 2 with y = u, alpha_j and ||u||^2 included; pass C1 with y = w)
//   k_ortho     the one-read form: the update w, written as W_{j+1}, ||w||^2 and the dots of w with
//               every Krylov vector, which give the next update's coefficients
//   k_lincomb   w = src - sum_i c_i W_i (MODE 0: Lanczos update, pass B of the two-pass form; 1: the
//               second Gram-Schmidt subtraction, pass C2; 2: combine psi = beta V y; 3: load the
//               initial vector)
//   k_vecout    psi at output times inside the step (adjoint)
// Every reduction ends in the last CTA to finish (ticket counter), which sums the per-CTA
// partials as integers of one exponent: results are bitwise reproducible for a fixed grid.
#include <cuda_runtime.h>

#include <algorithm>
#include <type_traits>

#include "kry_device.cuh"

namespace kry {

constexpr int DOTS_NTHR = 512;   // threads of a CTA of the dots
// Loads of hops issued together in the forms of the H.v: inside the lower bits (bit 0 of the form) and
// inside the upper bits (bit 1); eight of 16 bytes would spill
template <class V, int BIT> constexpr int HV_RND =
    sizeof(V) == 8 ? (BIT == 0 ? 4 : 8) : (BIT == 0) == std::is_same<V, double2>::value ? 2 : 4;

// ---------------------------------------------------------------- y = H x

// Bond energies (J Delta / 4)(nbonds - 2 n) for n antiparallel bonds.
template <class R>
__device__ __forceinline__ void stage_dz(const DevBasis &b, const DevHam &hm, R *dz)
{
    if (threadIdx.x <= (unsigned)b.L) dz[threadIdx.x] = (R)(hm.cz * (double)(hm.nbonds - 2 * (int)threadIdx.x));
}

template <class V>
__global__ void __launch_bounds__(HV_NTHR, sizeof(V) == 8 ? 4 : 3) k_apply(DevBasis b, DevHam hm, HvPlan pl,
                                                                          const V *__restrict__ x, V *__restrict__ y)
{
    using R = typename VT<V>::R;
    __shared__ R dz[64];
    __shared__ __align__(16) HvWarp w[HV_NTHR / 32];
    stage_dz(b, hm, dz);
    __syncthreads();
    hv_items<V, 4, 4, false>(b, hm, pl, x, y, w[threadIdx.x >> 5], dz, (R)1, (R)hm.halfJ,
                                               (RealAcc<V> *)nullptr);
}

// ---------------------------------------------------------------- reductions

// Sum per-thread values over the CTA (warp shuffles, then warps in order) into red[slot].
__device__ __forceinline__ void cta_sum_into(double2 v, double2 *red, int slot, double2 *wtmp)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    v = make_double2(warp_sum_int<1>(&v.x), warp_sum_int<1>(&v.y));
    if (lane == 0) wtmp[warp] = v;
    __syncthreads();
    if (threadIdx.x == 0) {
        double2 s = make_double2(0.0, 0.0);
        for (int w = 0; w < (int)blockDim.x / 32; ++w) { s.x += wtmp[w].x; s.y += wtmp[w].y; }
        red[slot] = s;
    }
    __syncthreads();
}

// The same for per-thread dot accumulators (float-float warp sums for complex64): complex ones
// (warp_value) and real ones.
template <class Acc>
__device__ __forceinline__ double2 acc_warp_value(const Acc &acc) { return acc.warp_value(); }
template <class V>
__device__ __forceinline__ double2 acc_warp_value(const RealAcc<V> &acc)
{
    typename RealAcc<V>::Sum v[1] = {acc.sum()};
    return make_double2(to_double(warp_totals<1>(v)), 0.0);
}
template <class Acc>
__device__ __forceinline__ void cta_sum_into(const Acc &acc, double2 *red, int slot, double2 *wtmp)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const double2 v = acc_warp_value(acc);
    if (lane == 0) wtmp[warp] = v;
    __syncthreads();
    if (threadIdx.x == 0) {
        double2 s = make_double2(0.0, 0.0);
        for (int w = 0; w < (int)blockDim.x / 32; ++w) { s.x += wtmp[w].x; s.y += wtmp[w].y; }
        red[slot] = s;
    }
    __syncthreads();
}

// ---------------------------------------------------------------- pass A

// u = sigma_j H W_j, written to U (pass A, part 1): the gathers of hv_items at full occupancy.  Without
// ALPHA (two-pass form) nothing else: alpha_j, ||u||^2 and the dots with the earlier vectors are taken
// by the streaming pass that follows (k_dots, mode 0).  With ALPHA (one-read form, k_ortho) the pass
// also takes alpha_j and sets up the update's coefficients (L = 24 c64: 40 us without, 50 with), and with A0 (a
// general psi0) in the first Krylov step c_0 (alpha_epilogue).
// FORM: how many loads are issued together inside the lower and the upper bits (HV_RND); every form
// gives the same bits, the launch shape picks the fastest (kry_autotune).
template <class V, int FORM, bool ALPHA, bool A0>
__global__ void __launch_bounds__(HV_NTHR, sizeof(V) == 8 ? 4 : 3) k_hv(EvArgs<V> a, HvPlan pl, int jj)
{
    using R = typename VT<V>::R;
    __shared__ R dz[64];
    __shared__ __align__(16) HvWarp w[HV_NTHR / 32];
    stage_dz(a.b, a.h, dz);   // (does not depend on the kernels before this one)
    __syncthreads();
    pdl_begin();
    KryCtl *ctl = a.ctl;
    if (ctl->done || jj >= ctl->m_eff) return;
    const double s = ctl->sigma[jj];
    RealAcc<V> al;
    hv_items<V, HV_RND<V, (FORM & 1)>, HV_RND<V, (FORM >> 1)>, ALPHA>(
        a.b, a.h, pl, a.W + (size_t)jj * a.ldW, a.U, w[threadIdx.x >> 5], dz, (R)s, (R)(s * a.h.halfJ), &al);
    if constexpr (ALPHA) {
        const bool first = jj > 0 && ctl->n_steps == 0;
        RealAcc<V> a0;
        if (A0 && first) hv_items_dot<V>(a.b, pl, a.W, a.U, &a0);
        alpha_epilogue<V, A0>(al, a0, first, a.U, a.part, ctl, jj);
    }
}

// The row loop of k_dots for one group of 64 threads: NQ vectors from Wg, NU units of rows at a time
// (all their loads issued before the products), and with NORM also ||y||^2.  NQ is a template
// parameter because a predicated-off multiply-add takes the FP64 pipe like any other: with a loop
// over eight vectors and a test in it, the dots with 1 to 8 vectors all took 91 us at L = 24.
template <class V, int NQ, int NU, bool NORM>
__device__ __forceinline__ void dots_rows(const V *y, const V *Wg, size_t ldW, uint32_t u0, uint32_t du,
                                          uint32_t nu, uint32_t D, RealAcc<V> *acc, RealAcc<V> &nrm)
{
    constexpr int RPC = 16 / sizeof(V);
    // units between two foldings of the float-float compensations (8 rows of complex64, 4 else)
    constexpr uint32_t FOLD = 4;
    const uint32_t col = threadIdx.x & 63;
    uint32_t it = 0;
    for (uint32_t u = u0; u < nu; u += NU * du) {
        V x[NU][NQ][RPC], yy[NU][RPC];
#pragma unroll
        for (int n = 0; n < NU; ++n) {
            const uint32_t r = ((u + n * du) * 64 + col) * RPC;
            // zero past D; the second row of a complex64 pair may be the first past D, where the
            // vectors are padded (ldW is a multiple of 64) and the value is dropped
#pragma unroll
            for (int e = 0; e < RPC; ++e) {
                yy[n][e] = VT<V>::zero();
#pragma unroll
                for (int q = 0; q < NQ; ++q) x[n][q][e] = VT<V>::zero();
            }
            if (r < D) {
                ldg_chunk(y + r, yy[n]);
#pragma unroll
                for (int q = 0; q < NQ; ++q) ldg_chunk(Wg + q * ldW + r, x[n][q]);
            }
            if (RPC == 2 && r + 1 == D) {
                yy[n][RPC - 1] = VT<V>::zero();
#pragma unroll
                for (int q = 0; q < NQ; ++q) x[n][q][RPC - 1] = VT<V>::zero();
            }
        }
#pragma unroll
        for (int n = 0; n < NU; ++n) {
            if (NU == 1 || u + n * du < nu) {
#pragma unroll
                for (int e = 0; e < RPC; ++e) {
                    const typename RealAcc<V>::Pre p = RealAcc<V>::pre(yy[n][e]);
                    if (NORM) nrm.add(yy[n][e], p);
#pragma unroll
                    for (int q = 0; q < NQ; ++q) acc[q].add(x[n][q][e], p);
                }
                if (++it % FOLD == 0) {
#pragma unroll
                    for (int q = 0; q < NQ; ++q) acc[q].renorm();
                    nrm.renorm();
                }
            }
        }
    }
}

// Dots Re <W_i, y>, i <= j, of a right-hand vector y with the Krylov vectors: a tall-skinny
// GEMV with plain loads, bound by HBM (complex64, float-float) or the FP64 pipe (complex128).
// 64 threads (two warps) read 16 bytes each of consecutive rows -- one row, or two of complex64 --
// of up to QV = 8 vectors, all loads issued before the products are accumulated (one real
// accumulator per vector and thread); with few vectors they take two or four units of rows at a time
// (MU = 0: always one, a launch-shape choice of kry_autotune; the bits are the same).  The 64-thread
// groups of a CTA split the vectors into NVG = 1, 2 or 4 nearly equal shares of at most eight, and
// the groups left over take other rows, so every warp has the same work at every j.  One CTA of 512
// threads per SM keeps up to 64 KB of loads in flight per SM (45 bytes per ns and SM at the HBM rate
// and about 0.8 us of latency need 36 KB) and leaves 152 partial sums per slot to add at the end.
//   MODE 0 (pass A): y = U = sigma_j H W_j; fills coefA[0..j], alpha_j and ||u||^2.
//   MODE 1 (pass C1, when pass B flagged it): y = W_{j+1}; measures the loss of
//          orthogonality and sets up the subtraction of pass C2 when it exceeds eta_corr.
template <class V, int MODE, int MU>
__global__ void __launch_bounds__(DOTS_NTHR, 1) k_dots(EvArgs<V> a, int jj)
{
    pdl_begin();
    KryCtl *ctl = a.ctl;
    if (ctl->done || jj >= ctl->m_eff) return;
    if (MODE == 1 && !ctl->corr) return;
    constexpr int RPC = 16 / sizeof(V);                 // rows of a thread's 16 bytes
    constexpr int QV = 8;                               // vectors of a group, at most
    __shared__ double2 red[PSTRIDE];
    __shared__ double wred[DOTS_NTHR / 32][QV + 1];
    __shared__ int flag;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, ngrp = blockDim.x >> 6, g = tid >> 6;
    if (tid < PSTRIDE) red[tid] = make_double2(0.0, 0.0);
    const V *y = (MODE == 0) ? a.U : a.W + (size_t)(jj + 1) * a.ldW;
    const int nv = jj + 1;   // vectors W_0 .. W_j
    const int nvg = nv <= QV ? 1 : nv <= 2 * QV ? 2 : 4, nrp = ngrp / nvg;   // shares of the vectors, of the rows
    const int rp = g / nvg, vg = (g + rp) % nvg;   // (rotated: the shares differ by one vector)
    const int i0 = (nv * vg) / nvg, nq = (nv * (vg + 1)) / nvg - i0;   // this group's vectors i0 .. i0 + nq - 1
    const uint32_t D = a.b.D, nu = (D + 64 * RPC - 1) / (64 * RPC);   // units of 64 threads' rows
    RealAcc<V> acc[QV], nrm;
    const V *Wg = a.W + (size_t)i0 * a.ldW;
    const uint32_t u0 = blockIdx.x * nrp + rp, du = gridDim.x * nrp;
#define KRY_DOTS_ROWS(NQ, NU)                                                                          \
    case NQ:                                                                                           \
        if (MODE == 0 && vg == 0) dots_rows<V, NQ, MU ? NU : 1, MODE == 0>(y, Wg, a.ldW, u0, du, nu, D, acc, nrm); \
        else dots_rows<V, NQ, MU ? NU : 1, false>(y, Wg, a.ldW, u0, du, nu, D, acc, nrm);              \
        break;
    switch (nq) {
        KRY_DOTS_ROWS(1, 4)
        KRY_DOTS_ROWS(2, 4)
        KRY_DOTS_ROWS(3, 2)
        KRY_DOTS_ROWS(4, 2)
        KRY_DOTS_ROWS(5, 2)
        KRY_DOTS_ROWS(6, 2)
        KRY_DOTS_ROWS(7, 1)
        KRY_DOTS_ROWS(8, 1)
    default: break;
    }
#undef KRY_DOTS_ROWS
    // per warp: the totals of its vectors (accumulators that were not used are zero); then the
    // warps of a vector's groups, in order
    {
        typename RealAcc<V>::Sum v[QV];
#pragma unroll
        for (int q = 0; q < QV; ++q) {
            acc[q].renorm();
            v[q] = acc[q].sum();
        }
        const double t = to_double(warp_totals<QV>(v));
        if (lane % (32 / QV) == 0) wred[warp][lane / (32 / QV)] = t;
    }
    if (MODE == 0) {
        nrm.renorm();
        typename RealAcc<V>::Sum v[1] = {nrm.sum()};
        const double t = to_double(warp_totals<1>(v));
        if (lane == 0) wred[warp][QV] = t;
    }
    __syncthreads();
    if (tid < nv || (MODE == 0 && tid == SLOT_NRM)) {
        const bool isn = tid == SLOT_NRM;
        int s = 0;   // the share that holds vector tid
        while (!isn && tid >= (nv * (s + 1)) / nvg) ++s;
        const int q = isn ? QV : tid - (nv * s) / nvg;
        double t = 0.0;
        for (int p = 0; p < nrp; ++p) {
            const int w = 2 * (p * nvg + (s + (nvg - 1) * p) % nvg);   // the group of share s in row part p
            t += wred[w][q] + wred[w + 1][q];
        }
        red[tid] = make_double2(t, 0.0);
    }
    __syncthreads();
    double2 *fin = red;
    if (!finish_partials(red, a.part, ctl, fin, &flag, nullptr, nv, MODE == 0, false)) return;
    // Scalar epilogue, one lane of warp 0 per vector.  GB300 issues one FP64 warp instruction per
    // about 77 cycles and SM sub-partition whatever its active lanes, so a loop over the vectors
    // in one thread cost 4 us at j = 30.
    if (tid >= 32) return;
    const bool in = tid <= jj;
    const double s = in ? ctl->sigma[tid] : 0.0;
    const double c = fin[tid].x * s;   // Re <v_i, y>
    const double cc = c * c, c2 = warp_sum_int<1>(&cc);
    if (MODE == 0) {
        if (in) ctl->coefA[tid] = c * s;
        if (tid == jj) ctl->alpha[jj] = c;
        bool minor = false;
        if (MinorSum<V>::use) {
            // rounding level: sum_{i<j-1} c_i^2 <= (eta ||u||)^2, with scales inside the FP32 range
            const bool small = tid + 1 < jj;
            const double cm = small ? c * c : 0.0, m2 = warp_sum_int<1>(&cm);
            minor = __all_sync(0xffffffffu, !small || (s >= 0x1p-40 && s <= 0x1p40)) &&
                    m2 <= MinorSum<V>::eta * MinorSum<V>::eta * fin[SLOT_NRM].x;
        }
        if (tid != 0) return;
        ctl->minor = minor ? 1 : 0;
        ctl->c2 = c2;
        ctl->normu2 = fin[SLOT_NRM].x;
        ctl->n_hv += 1;
        ctl->vec_passes += jj + 4;
        ctl->vp_kind[KIND_PASSA] += jj + 2;   // u and v_0 .. v_j
        ctl->vp_kind[KIND_HV] += 2;          // the H.v: v_j read, u written
        ctl->counter = 0;
        return;
    }
    const double nw2 = ctl->wnorm2;
    const bool sub = nw2 > 0.0 && sqrt(c2) > ctl->eta_corr * sqrt(nw2);
    if (sub && in) ctl->coefC[tid] = c * s;
    if (sub && tid == jj) ctl->alpha[jj] += c;
    if (tid != 0) return;
    if (nw2 > 0.0) ctl->max_orth = fmax(ctl->max_orth, sqrt(c2 / nw2));
    ctl->n_c1 += 1;
    ctl->vec_passes += jj + 2;
    ctl->vp_kind[KIND_PASSC] += jj + 2;
    ctl->corr = 0;
    ctl->corr2 = sub ? 1 : 0;
    if (!sub) finalize_beta(ctl, jj, nw2, ctl->wg);
    ctl->counter = 0;
}

// ---------------------------------------------------------------- the one-read pass

// Pass B and pass A's dots in one read of the Krylov vectors: w = u - sum_i c_i W_i, written as W_{j+1},
// ||w||^2 and the dots Re <W_i, w>, i <= j.  Every vector is orthogonalised against all the earlier ones,
// with coefficients c_i = Re <v_i, u>, u = (H - s) v_j, that need no pass of their own: H is symmetric, so
// c_i = Re <(H - s) v_i, v_j>, and the update that made v_{i+1} says what (H - s) v_i is,
//     (H - s) v_i = sum_{k<=i} C_ki v_k + beta_i v_{i+1}   (C_ki its coefficients c_k),
// up to the rounding of that update.  With the dots d_k = Re <v_k, v_j> that this kernel measured when it
// made v_j (d_j = 1), c_i = beta_i (sum_{k<=i} (C_ki / beta_i) d_k + d_{i+1}): beta_{j-1} for i = j - 1, rounding level
// below, and c_j = alpha_j comes from the H.v pass (as c_0 does in the first Krylov step, see alpha_epilogue).
// What the recurrence leaves out is the rounding of the stored u along v_i, which stays in the new vector, and
// the next dots see it: of the order of the rounding of w itself, except where v_i is a few elements and P
// reads it, which is v_0.  The Krylov vectors, whose
// reads bound the step, are read once per Lanczos index instead of twice.
// 64 threads take one row each of up to 16 vectors at a time; from 17 vectors on two such groups share a
// row.  (Eight vectors per group, with teams of up to four, took
// 98.7 us where this takes 90.4, L = 24 c64, and 107.5 against 93.2, L = 23 c128e.)  Sixteen vectors' rows and
// accumulators do not fit the 128 registers of 512 threads: complex64 spills 368 bytes per thread (708 loaded
// back), complex128 108 (348); c128e has 168 and no spills.
// Odd indices run backwards, so that the rows a pass ends with are still in L2 for the next.  When the
// dots exceed eta_corr, pass C2 (k_lincomb, mode 1) takes them off.
template <class V, int COND>
__global__ void __launch_bounds__(ORTHO_NTHR<V>, 1) k_ortho(EvArgs<V> a, int jj)
{
    pdl_begin();
    KryCtl *ctl = a.ctl;
    if (ctl->done || jj >= ctl->m_eff) return;
    constexpr int QV = ORTHO_QV, NW = ORTHO_NTHR<V> / 32, NGRP = ORTHO_NTHR<V> / 64;
    __shared__ double2 red[PSTRIDE];
    __shared__ double wred[NW][QV + 3];
    __shared__ typename RealLin<V>::RCoef coef[MMAX + 1];
    __shared__ float mcoef[MMAX + 1];
    __shared__ __align__(16) V xch[2 * ORTHO_NTHR<V> * ORTHO_XU];
    __shared__ int flag;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, g = tid >> 6;
    if (tid < PSTRIDE) red[tid] = make_double2(0.0, 0.0);
    if (tid <= jj) {
        const double c = ctl->coefA[tid];
        coef[tid] = RealLin<V>::coef(c);
        mcoef[tid] = -(float)c;
    }
    __syncthreads();
    const bool minor = MinorSum<V>::use && ctl->minor;
    const int nv = jj + 1;
    const int nvg = nv <= QV ? 1 : 2, nrp = NGRP / nvg;
    const int rp = g / nvg, vg = (g + rp) % nvg;   // (rotated: the shares differ by one vector)
    const int i0 = (nv * vg) / nvg, nq = (nv * (vg + 1)) / nvg - i0;
    const uint32_t D = a.b.D, nu = (D + 63) / 64, du = gridDim.x * nrp;
    RealAcc<V> acc[QV], nrm;
    DotAcc<V> gacc;
    V *out = a.W + (size_t)(jj + 1) * a.ldW;
    const int pad = ortho_pad(nq);
#define KRY_ORTHO(NQ, NU, KIND) \
    ortho_rows<V, NQ, NU, KIND, 64, NGRP, 1>(a.W, a.ldW, a.U, a.G, out, a.b.D, 64u, tid & 63, i0, nq, minor, rp, \
                                       blockIdx.x * nrp + rp, du, nu, jj & 1, coef, mcoef, 1, xch, acc, nrm, gacc)
#define KRY_ORTHO_N(NQ, NU) \
    case NQ: KRY_ORTHO(NQ, NU, ORTHO_ONLY); break;
#define KRY_ORTHO_3(NQ, NU)                                       \
    case NQ:                                                      \
        if (nvg == 1) KRY_ORTHO(NQ, NU, ORTHO_ONLY);              \
        else if (vg == 0) KRY_ORTHO(NQ, NU, ORTHO_FIRST);         \
        else KRY_ORTHO(NQ, NU, ORTHO_LAST);                       \
        break;
    switch (nq + pad) {
        KRY_ORTHO_N(1, 8)
        KRY_ORTHO_N(2, 4)
        KRY_ORTHO_N(3, 4)
        KRY_ORTHO_N(4, 4)
        KRY_ORTHO_N(6, 2)
        case 8:
            if (nvg == 1) KRY_ORTHO(8, 2, ORTHO_ONLY);
            else if (vg == 0) KRY_ORTHO(8, 1, ORTHO_FIRST);
            else KRY_ORTHO(8, 1, ORTHO_LAST);
            break;
        KRY_ORTHO_3(10, 1)
        KRY_ORTHO_3(12, 1)
        KRY_ORTHO_3(14, 1)
        KRY_ORTHO_3(15, 1)
        KRY_ORTHO_3(16, 1)
    default: break;
    }
#undef KRY_ORTHO_3
#undef KRY_ORTHO_N
#undef KRY_ORTHO
    {
        typename RealAcc<V>::Sum v[QV];
#pragma unroll
        for (int q = 0; q < QV; ++q) {
            acc[q].renorm();
            v[q] = acc[q].sum();
        }
        const double t = to_double(warp_totals<QV>(v));
        if (lane % (32 / QV) == 0) wred[warp][lane / (32 / QV)] = t;
        nrm.renorm();
        typename RealAcc<V>::Sum n1[1] = {nrm.sum()};
        const double tn = to_double(warp_totals<1>(n1));
        if (lane == 0) wred[warp][QV] = tn;
        if (a.G) {
            gacc.renorm();
            const double2 tg = gacc.warp_value();
            if (lane == 0) { wred[warp][QV + 1] = tg.x; wred[warp][QV + 2] = tg.y; }
        }
    }
    // c_i (1 / sigma_i is the norm that made v_i) in warp 1; loaded here, its latency passes beside the reduction
    const double ci = warp == 1 && lane <= jj ? ctl->coefA[lane] * (lane ? ctl->beta[lane - 1] : ctl->beta0) : 0.0;
    __syncthreads();
    if (tid < nv) {
        const int s = nvg == 1 || tid < nv / 2 ? 0 : 1;   // the share that holds vector tid
        const int f = nvg == 1 ? 0 : s ? nv / 2 : 0, n = nvg == 1 ? nv : s ? nv - nv / 2 : nv / 2;
        const int q = tid - f + ortho_pad(n);
        double t = 0.0;
        for (int p = 0; p < nrp; ++p) {
            const int w = 2 * (p * nvg + (nvg == 1 ? 0 : (s + p) & 1));   // the group of share s in row part p
            t += wred[w][q] + wred[w + 1][q];
        }
        red[tid] = make_double2(t, 0.0);
    } else if (tid >= 64 && tid < 67) {   // ||w||^2 and the two parts of <psi0, w>, from the groups of share 0
        double t = 0.0;
        if (tid == 64 || a.G)
            for (int w = 0; w < NW; ++w)
                if (((w >> 1) + (w >> 1) / nvg) % nvg == 0) t += wred[w][QV + tid - 64];
        if (tid == 64) red[SLOT_NRM] = make_double2(t, 0.0);
        else if (tid == 65) red[SLOT_G].x = t;
        else red[SLOT_G].y = t;
    }
    __syncthreads();
    double2 *fin = red;
    if (!finish_partials(red, a.part, ctl, fin, &flag, nullptr, nv, true, a.G != nullptr)) return;
    // Scalar epilogue, lane i for vector i: warp 1 keeps C and d of the new vector while warp 0 ends the index (the
    // FP64 square roots of both in one warp, and the sums of alpha_epilogue, took 1 us longer: P at L = 24 c64 76.6 -> 76.1 ms).
    if (tid >= 64) return;
    const bool inv = lane <= jj;
    const double s = inv ? ctl->sigma[lane] : 0.0, dd = fin[lane].x * s;   // Re <v_i, w>
    const double d2 = dd * dd, nd2 = warp_sum_int<1>(&d2), nw2 = fin[SLOT_NRM].x;
    const double normu2 = ctl->c2 + nw2;   // ||u||^2 = ||c||^2 + ||w||^2 for orthonormal v_i
    const bool dead = !(nw2 > ctl->eta_bd * ctl->eta_bd * normu2);   // an invariant subspace
    // (where the space ends too: w is rounding then, its dots refine alpha_j and its length the error estimate)
    const bool sub = nw2 > 0.0 && nd2 > ctl->eta_corr * ctl->eta_corr * nw2;
    if (warp == 1) {
        const double rb = rsqrt(nw2);
        if (inv && !sub && !dead) ctl->C[lane][jj] = (float)(ci * rb);   // (after a subtraction pass C2 sets C)
        // d of the new vector; after pass C2 it is at rounding level and taken as zero
        if (inv) ctl->d[lane] = sub || dead ? 0.f : (float)(dd * rb);
        return;
    }
    if (inv && sub) ctl->coefC[lane] = dd * s;
    if (sub && tid == jj) ctl->alpha[jj] += dd;
    if (tid != 0) return;
    ctl->normu2 = normu2;
    ctl->vec_passes += jj + 3 + (a.G ? 1 : 0);
    ctl->vp_kind[KIND_PASSB] += jj + 3 + (a.G ? 1 : 0);
    if (ctl->verify || sub) {
        ctl->n_c1 += 1;
        if (nw2 > 0.0) ctl->max_orth = fmax(ctl->max_orth, sqrt(nd2 / nw2));
    }
    ctl->corr2 = sub ? 1 : 0;
    if (!sub) finalize_beta(ctl, jj, nw2, fin[SLOT_G]);
    if (COND && a.use_cond) cudaGraphSetConditional(a.cond, sub ? 1u : 0u);
    ctl->counter = 0;
}

// ---------------------------------------------------------------- linear combinations

// w = src - sum_i c_i W_i, the terms taken in index order; w is then dotted with psi0.
// Plain loads, RR rows per thread (r, r + TILE, ...) and eight vectors unrolled (8 RR loads
// in flight per thread), four CTAs per SM (two with RR = 4): a pure stream, which this form
// keeps near the HBM rate.  RR is a launch-shape choice (kry_autotune); it changes which
// rows a thread sums into its partial norms, so results agree to rounding.
template <class V, int MODE, int RR, int COND = 0>
__global__ void __launch_bounds__(NTHR, RR == 4 ? 2 : 4) k_lincomb(EvArgs<V> a, int jj)
{
    pdl_begin();
    KryCtl *ctl = a.ctl;
    if (ctl->done) return;
    if (MODE <= 1 && jj >= ctl->m_eff) return;
    if (MODE == 1 && !ctl->corr2) return;
    const int nvec = (MODE == 2) ? ctl->m_eff : ((MODE == 3) ? 0 : jj + 1);
    // modes 0 and 1 subtract real multiples (RealAcc), the combine takes complex ones
    constexpr bool RE = MODE <= 1;
    using Lin = typename std::conditional<RE, RealLin<V>, CplxLin<V>>::type;
    __shared__ typename Lin::RCoef coef[MMAX + 1];
    __shared__ double2 red[PSTRIDE];
    __shared__ double2 wtmp[NTHR / 32];
    __shared__ float mcoef[MMAX + 1];
    __shared__ int flag;
    const int tid = threadIdx.x;
    const uint32_t nt = blockDim.x;
    // pass B: the first nminor terms are summed in FP32 (MinorSum)
    const int nminor = MODE == 0 && MinorSum<V>::use && ctl->minor ? max(jj - 1, 0) : 0;
    if (tid < PSTRIDE) red[tid] = make_double2(0.0, 0.0);
    if (tid < nvec) {
        if (MODE == 0) mcoef[tid] = -(float)ctl->coefA[tid];
        if constexpr (RE) coef[tid] = Lin::coef(MODE == 0 ? ctl->coefA[tid] : ctl->coefC[tid]);
        else coef[tid] = Lin::coef(ctl->coefY[tid]);
    }
    __syncthreads();
    V *out = (MODE >= 2) ? a.W : a.W + (size_t)(jj + 1) * a.ldW;
    const V *src = (MODE == 0) ? a.U : (MODE == 1) ? out : (MODE == 3) ? a.G : nullptr;
    const uint32_t D = a.b.D;
    RealAcc<V> nrm;
    DotAcc<V> gacc;
    const uint32_t ntr = (D + RR * nt - 1) / (RR * nt);
    for (uint32_t tile = blockIdx.x; tile < ntr; tile += gridDim.x) {
        const uint32_t r = tile * RR * nt + tid;
        if (r >= D) continue;
        uint32_t q[RR];
        bool in[RR];
#pragma unroll
        for (int k = 0; k < RR; ++k) {
            in[k] = r + k * nt < D;
            q[k] = in[k] ? r + k * nt : r;   // past D a row repeats the first, unstored
        }
        Lin w[RR];
#pragma unroll
        for (int k = 0; k < RR; ++k) w[k] = Lin(src ? src[q[k]] : VT<V>::zero());
        if (MODE == 2) {   // reads W_0 while overwriting it: plain loads
#pragma unroll 8
            for (int i = 0; i < nvec; ++i) {
                const V *wi = a.W + (size_t)i * a.ldW;
                V x[RR];
#pragma unroll
                for (int k = 0; k < RR; ++k) x[k] = wi[q[k]];
#pragma unroll
                for (int k = 0; k < RR; ++k) w[k].fms(coef[i], x[k]);
            }
        } else {
            if constexpr (MODE == 0 && MinorSum<V>::use) {
                if (nminor > 0) {
                    float2 f[RR];
#pragma unroll
                    for (int k = 0; k < RR; ++k) f[k] = make_float2(0.f, 0.f);
#pragma unroll 8
                    for (int i = 0; i < nminor; ++i) {
                        const V *wi = a.W + (size_t)i * a.ldW;
                        V x[RR];
#pragma unroll
                        for (int k = 0; k < RR; ++k) x[k] = ldg(wi + q[k]);
#pragma unroll
                        for (int k = 0; k < RR; ++k)
                            f[k] = __ffma2_rn(make_float2(mcoef[i], mcoef[i]), MinorSum<V>::lead(x[k]), f[k]);
                    }
#pragma unroll
                    for (int k = 0; k < RR; ++k) MinorSum<V>::add(w[k], f[k]);
                }
            }
#pragma unroll 8
            for (int i = nminor; i < nvec; ++i) {
                const V *wi = a.W + (size_t)i * a.ldW;
                V x[RR];
#pragma unroll
                for (int k = 0; k < RR; ++k) x[k] = ldg(wi + q[k]);
#pragma unroll
                for (int k = 0; k < RR; ++k) w[k].fms(coef[i], x[k]);
            }
        }
#pragma unroll
        for (int k = 0; k < RR; ++k) {
            if (!in[k]) continue;
            const V wv = (MODE == 3) ? src[q[k]] : w[k].out();   // (the load is a plain copy)
            out[q[k]] = wv;
            nrm.add(wv, RealAcc<V>::pre(wv));
            if (a.G && MODE != 3) gacc.add(ldg(a.G + q[k]), wv);
        }
        nrm.renorm();
        gacc.renorm();
    }
    cta_sum_into(nrm, red, SLOT_NRM, wtmp);
    if (a.G) cta_sum_into(gacc, red, SLOT_G, wtmp);
    double2 *fin = red;
    if (!finish_partials(red, a.part, ctl, fin, &flag, nullptr, 0, true, a.G != nullptr)) return;
    const double nw2 = fin[SLOT_NRM].x;
    if (MODE == 1 && a.one_read && tid <= jj)
        ctl->C[tid][jj] =
            (float)((ctl->coefA[tid] + ctl->coefC[tid]) * (tid ? ctl->beta[tid - 1] : ctl->beta0) * rsqrt(nw2));
    if (tid != 0) return;
    const double2 gdot = fin[SLOT_G];
    if (MODE == 0) {
        ctl->vec_passes += jj + 3 + (a.G ? 1 : 0);
        ctl->vp_kind[KIND_PASSB] += jj + 3 + (a.G ? 1 : 0);
        // One classical Gram-Schmidt pass is enough unless the projection cancelled most of
        // u (||w|| < eta ||u||, the Daniel-Gragg-Kaufman-Stewart test), or the lengths show a
        // loss of orthogonality: with c = V^H u and G = V^H V = I + E, ||w||^2 = ||u||^2 -
        // ||c||^2 + c^H E c, so |||w||^2 - (||u||^2 - ||c||^2)| / (||c|| ||w||) estimates
        // ||E c|| / ||w|| = ||V^H w|| / ||w|| (Pythagoras test).  Either way the dots of w
        // with every previous vector are taken (pass C1) and subtracted if needed (C2).
        // With orth_check set the dots are taken after every update.
        const double c2 = ctl->c2;
        // (floor: the noise of the lengths of vectors in storage precision; the square root is
        // taken only above it)
        const double pyth = fabs(nw2 - (ctl->normu2 - c2)), floor = 0.1 * ctl->eta_bd * ctl->normu2;
        const bool lost = pyth > floor && pyth > ctl->eta_corr * sqrt(c2 * nw2) + floor;
        if (ctl->verify || nw2 < ctl->eta_cancel * ctl->eta_cancel * ctl->normu2 || lost) {
            ctl->corr = 1;
            ctl->wnorm2 = nw2;
            ctl->wg = gdot;
        } else {
            ctl->corr = 0;
            finalize_beta(ctl, jj, nw2, gdot);
        }
        // (COND = 0 leaves the device graph call out of the kernel: profilers skip kernels
        // that make it, and the plain step graph does not need it)
        if (COND && a.use_cond) cudaGraphSetConditional(a.cond, ctl->corr ? 1u : 0u);
    } else if (MODE == 1) {
        ctl->n_corr += 1;
        ctl->vec_passes += jj + 3 + (a.G ? 1 : 0);
        ctl->vp_kind[KIND_PASSC] += jj + 3 + (a.G ? 1 : 0);
        ctl->corr2 = 0;
        finalize_beta(ctl, jj, nw2, gdot);
    } else {
        const double b0 = sqrt(nw2);
        if (!(b0 > 0.0)) {
            ctl->err = KRY_EINVAL;
            ctl->done = 1;
        } else {
            ctl->beta0 = b0;
            ctl->sigma[0] = 1.0 / b0;
            ctl->g[0] = (MODE == 3) ? make_double2(b0, 0.0)
                                    : make_double2(gdot.x / b0, gdot.y / b0);
        }
        ctl->vec_passes += nvec + 1 + ((a.G && MODE == 2) ? 1 : 0);
        if (MODE == 2) ctl->vp_kind[KIND_COMBINE] += nvec + 1 + (a.G ? 1 : 0);
        ctl->m_eff = ctl->m;
        ctl->corr = 0;
        ctl->corr2 = 0;
        if (MODE == 2 && ctl->finishing) ctl->done = 1;
    }
    ctl->counter = 0;
}

template <class V>
__global__ void k_set_basis_state(V *W0, uint32_t r0)
{
    V one = VT<V>::zero();
    one.x = 1;
    W0[r0] = one;
}

__global__ void k_set_basis_state_ff(ffc *W0, uint32_t r0) { W0[r0] = ffc{1.f, 0.f, 0.f, 0.f}; }

// ---------------------------------------------------------------- dense vector output

constexpr int VECOUT_NTHR = 128;

// psi(t_o) = sum_j Yout[o][j] W_j for every output time o inside the current step (the
// small exponential fills Yout and [out_begin, out_end)); runs before the combine
// overwrites W_0.  Bound by the multiply-adds (FP64: 4 per element, vector and output): eight outputs
// share a vector's load (one output at a time re-read all vectors, 819 us for 20 outputs at L = 18).
template <class V>
__global__ void __launch_bounds__(VECOUT_NTHR) k_vecout(VecOutArgs<V> a)
{
    pdl_begin();
    KryCtl *ctl = a.ctl;
    if (ctl->done) return;
    const int ob = ctl->out_begin, oe = ctl->out_end, me = ctl->m_eff;
    if (ob >= oe) return;
    constexpr int NO = 8;
    __shared__ V cf[MMAX][NO];
    for (int o0 = ob; o0 < oe; o0 += NO) {
        const int no = min(NO, oe - o0);
        __syncthreads();
        for (int e = threadIdx.x; e < me * NO; e += VECOUT_NTHR) {
            const int j = e / NO, q = e % NO;
            cf[j][q] = q < no ? VT<V>::from(a.Yout[(size_t)(o0 + q) * MMAX + j]) : VT<V>::zero();
        }
        __syncthreads();
        for (size_t r = (size_t)blockIdx.x * VECOUT_NTHR + threadIdx.x; r < a.D; r += (size_t)gridDim.x * VECOUT_NTHR) {
            V w[NO];
#pragma unroll
            for (int q = 0; q < NO; ++q) w[q] = VT<V>::zero();
            V next = a.W[r];
#pragma unroll 2
            for (int j = 0; j < me; ++j) {
                const V v = next;
                if (j + 1 < me) next = a.W[(size_t)(j + 1) * a.ldW + r];
#pragma unroll
                for (int q = 0; q < NO; ++q) {
                    if (q < 4 || no > 4) {   // (a full or a half block: a predicated-off FP64 multiply-add costs as much)
                        const V c = cf[j][q];
                        w[q].x = fma(c.x, v.x, fma(-c.y, v.y, w[q].x));
                        w[q].y = fma(c.x, v.y, fma(c.y, v.x, w[q].y));
                    }
                }
            }
#pragma unroll
            for (int q = 0; q < NO; ++q)
                if (q < no) a.out[(size_t)(o0 + q) * a.ldOut + r] = w[q];
        }
    }
}

// Copy psi (= W_0 after the combine) into checkpoint slot n_steps/every - 1 after every
// `every`-th Krylov step, and record its time.
template <class V>
__global__ void __launch_bounds__(NTHR) k_ckpt(const V *__restrict__ W0, V *__restrict__ ck, size_t ldC,
                                               KryCtl *ctl, uint32_t D)
{
    pdl_begin();
    if (ctl->done || ctl->ckpt_every <= 0) return;
    const long long ns = ctl->n_steps;
    if (ns % ctl->ckpt_every != 0) return;
    const long long slot = ns / ctl->ckpt_every - 1;
    if (slot < 0 || slot >= ctl->ckpt_cap) return;
    V *dst = ck + (size_t)slot * ldC;
    for (size_t r = (size_t)blockIdx.x * NTHR + threadIdx.x; r < D; r += (size_t)gridDim.x * NTHR) dst[r] = W0[r];
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        ctl->ckpt_t[slot] = ctl->t_now;
        ctl->n_ckpt = (int)slot + 1;
    }
}

// ---------------------------------------------------------------- gradient integrand

__global__ void __launch_bounds__(NTHR) k_grad_acc(DevBasis b, DevHam hm, double J, const double2 *__restrict__ psi,
                                                   const double2 *__restrict__ lam, size_t ld,
                                                   const double *__restrict__ w, int nq, double2 *part,
                                                   double2 *acc_out, unsigned *counter, int site0)
{
    __shared__ uint32_t koff_s[20], bsz_s[20];
    __shared__ double2 red[PSTRIDE];
    __shared__ double2 wtmp[NTHR / 32];
    __shared__ int flag;
    const int tid = threadIdx.x, L = b.L;
    if (!b.list) stage_tables(b, koff_s, bsz_s, nullptr, 0);
    if (tid < PSTRIDE) red[tid] = make_double2(0.0, 0.0);
    __syncthreads();
    double2 acc[MMAX + 1];
#pragma unroll
    for (int i = 0; i <= MMAX; ++i) acc[i] = make_double2(0.0, 0.0);
    const uint32_t D = b.D, ntiles = (D + TILE - 1) / TILE;
    const uint64_t obc = (L >= 2) ? ((1ull << (L - 1)) - 1ull) : 0ull;
    const double czz = 0.25 * J;
    for (uint32_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
        const uint32_t r = tile * TILE + tid;
        if (r >= D) continue;
        uint64_t s;
        if (b.list) {
            s = __ldg(b.states + r);
        } else {
            uint32_t hi, off;
            int klo;
            tile_unrank(b, bsz_s, tile * TILE, tid, hi, off, klo);
            s = ((uint64_t)hi << b.Llo) | __ldg(b.lolist + koff_s[klo] + off);
        }
        double2 S = make_double2(0.0, 0.0);
        for (int q = 0; q < nq; ++q) {
            const double2 l = __ldg(lam + (size_t)(nq - 1 - q) * ld + r), p = __ldg(psi + (size_t)q * ld + r);
            const double wq = __ldg(w + q);
            S.x += wq * (l.x * p.x + l.y * p.y);
            S.y += wq * (l.x * p.y - l.y * p.x);
        }
#pragma unroll
        for (int i = 0; i < MMAX; ++i) {
            if (site0 + i < L) {
                const double z = ((s >> (site0 + i)) & 1ull) ? 0.5 : -0.5;
                acc[i].x += z * S.x;
                acc[i].y += z * S.y;
            }
        }
        if (site0 == 0) {
            const int nanti = __popcll((long long)((s ^ (s >> 1)) & obc)) +
                              (hm.pbc ? (int)((s ^ (s >> (L - 1))) & 1ull) : 0);
            const double zz = czz * (double)(hm.nbonds - 2 * nanti);
            acc[MMAX].x += zz * S.x;
            acc[MMAX].y += zz * S.y;
        }
    }
#pragma unroll
    for (int i = 0; i <= MMAX; ++i) {
        if (site0 + i < L || i == MMAX) cta_sum_into(acc[i], red, i, wtmp);
    }
    double2 *fin = red;
    if (!finish_partials(red, part, nullptr, fin, &flag, counter)) return;
    if (tid < MMAX && site0 + tid < L) {
        acc_out[site0 + tid].x += fin[tid].x;
        acc_out[site0 + tid].y += fin[tid].y;
    } else if (tid == MMAX && site0 == 0) {
        acc_out[L].x += fin[MMAX].x;
        acc_out[L].y += fin[MMAX].y;
    }
    if (tid == 0) *counter = 0;
}

// ---------------------------------------------------------------- launchers

static int sm_count()
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

// Threads of a CTA of the updates: 64 in sectors whose rows, at two per thread, would not give every SM
// two CTAs of 256 (D < 155,648 on 152 SMs), so that more SMs share them.
static int lincomb_threads(uint32_t D) { return D < (uint32_t)sm_count() * 4u * NTHR ? 64 : NTHR; }

// Blocks per item of the H.v: more share the lower part's ranks, fewer give more items.  One below four
// items of 32 rows per warp slot, two below 16, four below 200 and eight from there on.  kry_apply with one, two,
// four and eight, in us (complex64; complex128), by items of 32 rows per slot:
//   0.3 (L = 18)   9.3 9.3 9.3 12.2; 8.9 10.0 16.4 24.6     17 (L = 24)   53.8 41.5 37.3 37.3; 171 160 158 158
//   4.5 (L = 22)   18.5 14.4 15.9 16.4; 50.0 47.2 52.8 54.8 67 (L = 26)   200 154 141 130; 694 641 623 618
//   8.7 (L = 23)   28.8 22.6 22.6 24.6; 88 82 80 81         258 (L = 28)  975 724 655 616; 3450 3215 3121 3050
static HvPlan hv_plan(const DevBasis &b)
{
    HvPlan p{};
    const uint64_t warps = (uint64_t)b.D / 32u, full = (uint64_t)sm_count() * 32u;
    p.nh = warps >= 200u * full ? 8 : warps >= 16u * full ? 4 : warps >= 4u * full ? 2 : 1;
    auto binom = [](int n, int k) {
        if (k < 0 || k > n) return (uint32_t)0;
        uint64_t r = 1;
        for (int i = 1; i <= k; ++i) r = r * (uint64_t)(n - k + i) / (uint64_t)i;
        return (uint32_t)r;
    };
    uint32_t kofs[18] = {0};   // group offsets of lolist
    for (int k = 0; k <= b.Llo; ++k) kofs[k + 1] = kofs[k] + binom(b.Llo, k);
    for (int c = 0; c <= b.Lhi; ++c) {
        const uint32_t nhi = binom(b.Lhi, c);
        const int kl = b.N - c;
        p.hoff[c + 1] = p.hoff[c] + nhi;
        p.first[c + 1] = p.first[c];
        if (kl < 0 || kl > b.Llo) continue;
        p.nlo[c] = kofs[kl + 1] - kofs[kl];
        p.koff[c] = kofs[kl];
        p.first[c + 1] += ((p.nlo[c] + 31u) / 32u) * ((nhi + p.nh - 1) / p.nh);
    }
    return p;
}

int launch_apply(const DevBasis &b, const DevHam &h, int c64, const void *x, void *y, cudaStream_t s)
{
    if (b.list) return launch_list_apply(b, h, c64, 1, x, y, s);
    const HvPlan pl = hv_plan(b);
    const uint32_t ctas = (pl.first[b.Lhi + 1] + HV_NTHR / 32 - 1) / (HV_NTHR / 32);
    const int grid = (int)std::min<uint32_t>(ctas, (uint32_t)sm_count() * (c64 ? 4u : 3u));
    if (c64) k_apply<float2><<<grid, HV_NTHR, 0, s>>>(b, h, pl, (const float2 *)x, (float2 *)y);
    else k_apply<double2><<<grid, HV_NTHR, 0, s>>>(b, h, pl, (const double2 *)x, (double2 *)y);
    KRY_CU(cudaGetLastError());
    return KRY_OK;
}

// CTAs of the vector kernels, whole SMs times their resident CTAs: the streaming dots
// (returned; also pass C1), the H.v of pass A (*gridH) and the updates, combine and
// outputs (*gridB).
template <class V>
int vector_grid(const DevBasis &b, int *gridH, int *gridB)
{
    const uint32_t es = sizeof(V);
    int occB = 0, occH = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occH, k_hv<V, 0, true, false>, HV_NTHR, 0);   // (the same for every form)
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occB, k_lincomb<V, 0, 2>, NTHR, 0);
    const uint32_t ntiles = (b.D + TILE - 1) / TILE;
    auto fit = [&](int occ, uint32_t most) {
        return (int)std::max<uint32_t>(1u, std::min<uint32_t>(most, (uint32_t)(sm_count() * std::max(1, occ))));
    };
    if (b.list) {
        *gridH = fit(occH, ntiles);
        if (int rc = list_hv_grid<V>(b, gridH)) return -rc;
    } else {
        *gridH = fit(occH, (hv_plan(b).first[b.Lhi + 1] + HV_NTHR / 32 - 1) / (HV_NTHR / 32));
    }
    // (the updates of small sectors: CTAs of 64 threads, two rows each)
    *gridB = lincomb_threads(b.D) == NTHR ? fit(occB, ntiles) : (int)std::max<uint32_t>(1u, std::min<uint32_t>((b.D + 127) / 128, (uint32_t)sm_count() * 4u));
    // the dots: one CTA per SM, fewer when there are not two units of 64 threads' rows for each
    const uint32_t nu = (b.D + 64 * (16 / es) - 1) / (64 * (16 / es));
    return (int)std::max<uint32_t>(1u, std::min<uint32_t>((nu + 1) / 2, (uint32_t)sm_count()));
}

template <class V>
int launch_hv(const EvArgs<V> &a, int jj, int grid, cudaStream_t s, int pdl)
{
    if (a.b.list) return launch_list_hv<V>(a, jj, grid, s, pdl);
    const HvPlan pl = hv_plan(a.b);
    auto go = [&](auto k0, auto k1, auto k2, auto k3) {
        return launch_ex(pdl, a.hv_form == 0 ? k0 : a.hv_form == 1 ? k1 : a.hv_form == 2 ? k2 : k3, grid, HV_NTHR, 0, s, a, pl, jj);
    };
    if (a.one_read && a.G) KRY_CU(go(k_hv<V, 0, true, true>, k_hv<V, 1, true, true>, k_hv<V, 2, true, true>, k_hv<V, 3, true, true>));
    else if (a.one_read) KRY_CU(go(k_hv<V, 0, true, false>, k_hv<V, 1, true, false>, k_hv<V, 2, true, false>, k_hv<V, 3, true, false>));
    else KRY_CU(go(k_hv<V, 0, false, false>, k_hv<V, 1, false, false>, k_hv<V, 2, false, false>, k_hv<V, 3, false, false>));
    KRY_CU(cudaGetLastError());
    return KRY_OK;
}

template <class V, int MODE, int COND>
static cudaError_t launch_lincomb_rr(const EvArgs<V> &a, int jj, int grid, cudaStream_t s, int pdl)
{
    const int nt = lincomb_threads(a.b.D);
    switch (a.upd_rows) {
    case 1: return launch_ex(pdl, k_lincomb<V, MODE, 1, COND>, grid, nt, 0, s, a, jj);
    case 4: return launch_ex(pdl, k_lincomb<V, MODE, 4, COND>, grid, nt, 0, s, a, jj);
    default: return launch_ex(pdl, k_lincomb<V, MODE, 2, COND>, grid, nt, 0, s, a, jj);
    }
}

template <class V>
int launch_lincomb(const EvArgs<V> &a, int mode, int jj, int grid, cudaStream_t s, int pdl)
{
    switch (mode) {
    case 0:
        if (a.use_cond) KRY_CU((launch_lincomb_rr<V, 0, 1>(a, jj, grid, s, pdl)));
        else KRY_CU((launch_lincomb_rr<V, 0, 0>(a, jj, grid, s, pdl)));
        break;
    case 1: KRY_CU((launch_lincomb_rr<V, 1, 0>(a, jj, grid, s, pdl))); break;
    case 2: KRY_CU(launch_ex(pdl, k_lincomb<V, 2, 2>, grid, lincomb_threads(a.b.D), 0, s, a, jj)); break;
    default: KRY_CU(launch_ex(pdl, k_lincomb<V, 3, 2>, grid, lincomb_threads(a.b.D), 0, s, a, jj)); break;
    }
    KRY_CU(cudaGetLastError());
    return KRY_OK;
}

int launch_set_basis_state(void *W0, int c64, uint32_t r0, cudaStream_t s, int ff)
{
    if (c64) k_set_basis_state<float2><<<1, 1, 0, s>>>((float2 *)W0, r0);
    else if (ff) k_set_basis_state_ff<<<1, 1, 0, s>>>((ffc *)W0, r0);
    else k_set_basis_state<double2><<<1, 1, 0, s>>>((double2 *)W0, r0);
    KRY_CU(cudaGetLastError());
    return KRY_OK;
}

// complex128 <-> float-float vectors (dtype KRY_C128E): in at the initial vector, out at psi(t)
__global__ void __launch_bounds__(NTHR) k_c128_to_ffc(const double2 *__restrict__ src, ffc *__restrict__ dst, size_t n)
{
    for (size_t r = (size_t)blockIdx.x * NTHR + threadIdx.x; r < n; r += (size_t)gridDim.x * NTHR)
        dst[r] = VT<ffc>::from(__ldg(src + r));
}
__global__ void __launch_bounds__(NTHR) k_ffc_to_c128(const ffc *__restrict__ src, double2 *__restrict__ dst, size_t n)
{
    for (size_t r = (size_t)blockIdx.x * NTHR + threadIdx.x; r < n; r += (size_t)gridDim.x * NTHR) {
        const ffc v = ldg(src + r);
        dst[r] = make_double2(ff2d(v.xh, v.xl), ff2d(v.yh, v.yl));
    }
}
static unsigned convert_grid(size_t n)
{
    return (unsigned)std::max<size_t>(1, std::min<size_t>((n + NTHR - 1) / NTHR, (size_t)sm_count() * 8));
}
int launch_c128_to_ffc(const void *src, void *dst, size_t n, cudaStream_t s)
{
    if (n == 0) return KRY_OK;
    k_c128_to_ffc<<<convert_grid(n), NTHR, 0, s>>>((const double2 *)src, (ffc *)dst, n);
    KRY_CU(cudaGetLastError());
    return KRY_OK;
}
int launch_ffc_to_c128(const void *src, void *dst, size_t n, cudaStream_t s)
{
    if (n == 0) return KRY_OK;
    k_ffc_to_c128<<<convert_grid(n), NTHR, 0, s>>>((const ffc *)src, (double2 *)dst, n);
    KRY_CU(cudaGetLastError());
    return KRY_OK;
}

template <class V>
int launch_vecout(const VecOutArgs<V> &a, cudaStream_t s)
{
    const int g = (int)std::max<uint32_t>(1u, std::min<uint32_t>((a.D + VECOUT_NTHR - 1) / VECOUT_NTHR, (uint32_t)sm_count() * 4u));
    KRY_CU(launch_pdl(k_vecout<V>, g, VECOUT_NTHR, 0, s, a));
    KRY_CU(cudaGetLastError());
    return KRY_OK;
}

template <class V>
int launch_ckpt(const V *W0, V *ckpt, size_t ldC, KryCtl *ctl, uint32_t D, int grid, cudaStream_t s)
{
    KRY_CU(launch_pdl(k_ckpt<V>, grid, NTHR, 0, s, W0, ckpt, ldC, ctl, D));
    KRY_CU(cudaGetLastError());
    return KRY_OK;
}

int launch_grad_acc(const DevBasis &b, const DevHam &h, double J, const double2 *psi, const double2 *lam,
                    size_t ld, const double *w, int nq, double2 *part, double2 *acc, unsigned *counter,
                    int grid, cudaStream_t s)
{
    for (int site0 = 0; site0 < b.L; site0 += MMAX) {   // 32 sites per launch (L > 32: two)
        k_grad_acc<<<grid, NTHR, 0, s>>>(b, h, J, psi, lam, ld, w, nq, part, acc, counter, site0);
        KRY_CU(cudaGetLastError());
    }
    return KRY_OK;
}

template int launch_vecout<double2>(const VecOutArgs<double2> &, cudaStream_t);
template int launch_vecout<float2>(const VecOutArgs<float2> &, cudaStream_t);
template int launch_ckpt<double2>(const double2 *, double2 *, size_t, KryCtl *, uint32_t, int, cudaStream_t);
template int launch_ckpt<float2>(const float2 *, float2 *, size_t, KryCtl *, uint32_t, int, cudaStream_t);
template <class V>
int launch_dots(const EvArgs<V> &a, int mode, int jj, int grid, cudaStream_t s, int pdl)
{
    const int mu = a.dots_form == 0;
    if (mode == 0) KRY_CU(launch_ex(pdl, mu ? k_dots<V, 0, 1> : k_dots<V, 0, 0>, grid, DOTS_NTHR, 0, s, a, jj));
    else KRY_CU(launch_ex(pdl, mu ? k_dots<V, 1, 1> : k_dots<V, 1, 0>, grid, DOTS_NTHR, 0, s, a, jj));
    KRY_CU(cudaGetLastError());
    return KRY_OK;
}

template <class V>
int launch_ortho(const EvArgs<V> &a, int jj, int grid, cudaStream_t s, int pdl)
{
    KRY_CU(launch_ex(pdl, a.use_cond ? k_ortho<V, 1> : k_ortho<V, 0>, grid, ORTHO_NTHR<V>, 0, s, a, jj));
    KRY_CU(cudaGetLastError());
    return KRY_OK;
}

template int launch_ortho<double2>(const EvArgs<double2> &, int, int, cudaStream_t, int);
template int launch_ortho<float2>(const EvArgs<float2> &, int, int, cudaStream_t, int);
template int launch_ortho<ffc>(const EvArgs<ffc> &, int, int, cudaStream_t, int);
template int launch_dots<double2>(const EvArgs<double2> &, int, int, int, cudaStream_t, int);
template int launch_dots<float2>(const EvArgs<float2> &, int, int, int, cudaStream_t, int);
template int launch_dots<ffc>(const EvArgs<ffc> &, int, int, int, cudaStream_t, int);
template int vector_grid<double2>(const DevBasis &, int *, int *);
template int vector_grid<float2>(const DevBasis &, int *, int *);
template int vector_grid<ffc>(const DevBasis &, int *, int *);
template int launch_hv<double2>(const EvArgs<double2> &, int, int, cudaStream_t, int);
template int launch_hv<float2>(const EvArgs<float2> &, int, int, cudaStream_t, int);
template int launch_hv<ffc>(const EvArgs<ffc> &, int, int, cudaStream_t, int);
template int launch_lincomb<double2>(const EvArgs<double2> &, int, int, int, cudaStream_t, int);
template int launch_lincomb<float2>(const EvArgs<float2> &, int, int, int, cudaStream_t, int);
template int launch_lincomb<ffc>(const EvArgs<ffc> &, int, int, int, cudaStream_t, int);

}  // namespace kry

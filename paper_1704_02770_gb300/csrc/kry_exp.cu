// Small exponential, error estimate and step control of one Krylov step (Sec. 2:
// psi(t + tau) ~ beta V_m exp(-i tau T_m) e_1 with time stepping and error estimation),
// run by one CTA in FP64 without a host round trip.
//
// T (m_eff x m_eff, symmetric tridiagonal from Lanczos) is shifted and scaled into
// [-1, 1]: T~ = (T - c)/r with c, r the centre and half-width of its Gershgorin interval.
// Then (Jacobi-Anger expansion)
//     exp(-i tau T) e_1 = exp(-i tau c) sum_k w_k J_k(tau r) T_k(T~) e_1,
//     w_0 = 1, w_k = 2 (-i)^k,
// with Bessel functions J_k from Miller's backward recurrence normalised by
// J_0 + 2 sum J_2k = 1.  The leading term of the Krylov error (Saad 1992; the estimate
// of Sidje's Expokit that the paper relies on) is
//     err(tau) = beta h |e_m^T tau phi_1(-i tau (T - c)) e_1|
//              = (beta h / r) |sum_k w_k I_k(tau r) [T_k(T~) e_1]_m|,
// where I_k(x) = int_0^x J_k = 2 sum_n J_{k+2n+1}(x) (Abramowitz & Stegun 11.1.2) and h is
// the coupling of v_m to the next Krylov vector.  A ladder of 32 candidate steps (one per
// lane) is scanned and the largest tau with err(tau) <= 0.05 tol tau / t_end is taken;
// the Krylov basis is reused, so a rejected candidate costs no H.v.  Every output time in
// [t, t + tau] is read from the same expansion (dense output):
//     <psi0|psi(t + tau')> = beta exp(-i tau' c) sum_k w_k J_k(tau' r) sum_j g_j [T_k(T~) e_1]_j,
// g_j = <psi0|v_j>.
#include <cuda_runtime.h>

#include "kry_device.cuh"

namespace kry {

constexpr double STEP_SAFETY = 0.1;   // fraction of the local error budget a step may use
constexpr double LADDER = 0.85;       // ratio of consecutive candidate steps

struct ExpSmem {
    double al[MMAX], be[MMAX];
    double2 g[MMAX];
    double tch[(KMAX + 1) * 32];      // T_k(T~) e_1, component j at [k * 32 + j]
    double jb[32 * (KMAX + 2)];       // per-lane Bessel sequences
    double2 gk[KMAX + 1];             // sum_j g_j [T_k(T~) e_1]_j
};

__device__ __forceinline__ int cheb_degree(double x)
{
    const int K = (int)ceil(x + 8.0 * cbrt(x) + 24.0);
    return K < KMAX ? K : KMAX;
}

__device__ __forceinline__ double2 cmul(double2 a, double2 b)
{
    return make_double2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}

__device__ double2 gershgorin(const ExpSmem &sm, int me)
{
    const int j = threadIdx.x & 31;
    const double a = (j < me) ? sm.al[j] : 0.0;
    const double bl = (j >= 1 && j < me) ? fabs(sm.be[j - 1]) : 0.0;
    const double br = (j + 1 < me) ? fabs(sm.be[j]) : 0.0;
    double lo = (j < me) ? a - bl - br : 1e300, hi = (j < me) ? a + bl + br : -1e300;
    for (int o = 16; o > 0; o >>= 1) {
        lo = fmin(lo, __shfl_xor_sync(0xffffffffu, lo, o));
        hi = fmax(hi, __shfl_xor_sync(0xffffffffu, hi, o));
    }
    const double r = 0.5 * (hi - lo);
    const double rmin = 1e-12 * fmax(1.0, fmax(fabs(lo), fabs(hi)));
    return make_double2(0.5 * (lo + hi), r > rmin ? r : rmin);
}

// Gershgorin centre c and half-width r of T (lanes own rows), then the Chebyshev vectors
// T_k(T~) e_1 for k = 0..K into sm.tch.  Returns (c, r) in every lane.
__device__ double2 chebyshev_basis(ExpSmem &sm, int me, int K)
{
    const int j = threadIdx.x & 31;
    const double a = (j < me) ? sm.al[j] : 0.0;
    const double bl = (j >= 1 && j < me) ? fabs(sm.be[j - 1]) : 0.0;
    const double br = (j + 1 < me) ? fabs(sm.be[j]) : 0.0;
    double lo = (j < me) ? a - bl - br : 1e300, hi = (j < me) ? a + bl + br : -1e300;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        lo = fmin(lo, __shfl_xor_sync(0xffffffffu, lo, o));
        hi = fmax(hi, __shfl_xor_sync(0xffffffffu, hi, o));
    }
    const double c = 0.5 * (lo + hi);
    double r = 0.5 * (hi - lo);
    const double rmin = 1e-12 * fmax(1.0, fmax(fabs(lo), fabs(hi)));
    if (!(r > rmin)) r = rmin;
    const double ir = 1.0 / r;
    const double dj = (j < me) ? (a - c) * ir : 0.0;
    const double ol = (j >= 1 && j < me) ? sm.be[j - 1] * ir : 0.0;
    const double orr = (j + 1 < me) ? sm.be[j] * ir : 0.0;
    double v0 = (j == 0) ? 1.0 : 0.0;
    sm.tch[j] = v0;
    double up = __shfl_up_sync(0xffffffffu, v0, 1), dn = __shfl_down_sync(0xffffffffu, v0, 1);
    double v1 = dj * v0 + ol * up + orr * dn;
    if (K >= 1) sm.tch[32 + j] = v1;
    for (int k = 2; k <= K; ++k) {
        up = __shfl_up_sync(0xffffffffu, v1, 1);
        dn = __shfl_down_sync(0xffffffffu, v1, 1);
        const double v2 = 2.0 * (dj * v1 + ol * up + orr * dn) - v0;
        sm.tch[k * 32 + j] = v2;
        v0 = v1;
        v1 = v2;
    }
    __syncwarp();
    return make_double2(c, r);
}

// ---- sums over the Bessel functions straight from the backward recurrence
constexpr int NKD = KMAX + 64;   // table of the doubles k: the recurrence starts at most at KMAX + 41

// Miller's recurrence for J_K(x) .. J_0(x), unnormalised, handed to f from k = K down; the caller's
// sums are scaled along by f.scale when the values are.  Returns 1 / (J_0 + 2 sum J_2k), the factor
// that normalises them.  Integer tests of the exponent and a table of the doubles k spare the FP64
// pipe (77 issue cycles per instruction of a warp): two and a half instructions per index.  ANY: arguments
// above the table too, which a Krylov step does not have (x <= XMAX) and kry_tridiag_expv takes.
template <bool ANY = false, class F>
__device__ __forceinline__ double bessel_down(double x, int K, const double *kd, F &f)
{
    if (x < 1e-6) {
        if (K >= 3) f.add(3, x * x * x / 48.0);
        if (K >= 2) f.add(2, x * x / 8.0);
        if (K >= 1) f.add(1, 0.5 * x - x * x * x / 16.0);
        f.add(0, 1.0 - 0.25 * x * x);
        return 1.0;
    }
    const int xi = ANY ? (int)fmin(x, 1048576.0) : (int)x;   // (the expansion holds to about x = 100)
    int ns = (K > xi ? K : xi) + 40;
    ns += ns & 1;
    const double inv = 2.0 / x;
    double jp1 = 0.0, jk = 1e-280, sum = 0.0, j0 = 0.0;
    if constexpr (ANY) {
        for (; ns >= NKD; --ns) {
            const double jm1 = (double)ns * inv * jk - jp1;
            jp1 = jk;
            jk = jm1;
            if (ns & 1) sum += jm1;
            if (fabs(jk) > 1e250) {
                jk *= 1e-250;
                jp1 *= 1e-250;
                sum *= 1e-250;
            }
        }
    }
    for (int k = ns; k >= 1; --k) {
        const double jm1 = kd[k] * inv * jk - jp1;
        jp1 = jk;
        jk = jm1;
        const int idx = k - 1;
        if (idx <= K) f.add(idx, jm1);
        if (idx >= 2 && !(idx & 1)) sum += jm1;
        if (idx == 0) j0 = jm1;
        if (((unsigned)__double2hiint(jk) & 0x7fffffffu) > 0x73e00000u) {   // above 1e250, about
            const double sc = 1e-250;
            jk *= sc;
            jp1 *= sc;
            sum *= sc;
            j0 *= sc;
            f.scale(idx, sc);
        }
    }
    return 1.0 / (j0 + 2.0 * sum);
}
struct BesselStore {   // J_k itself, for the combine's and the vector outputs' coefficients
    double *out;
    int K;
    __device__ __forceinline__ void add(int k, double j) { out[k] = j; }
    __device__ __forceinline__ void scale(int k, double s)
    {
        for (int t = k; t <= K; ++t) out[t] *= s;
    }
};
// sum_k 2 J_k S_k with S_k = sum of w_l [T_l e_1]_m over l < k of the other parity: the error estimate's
// sum_l w_l I_l [T_l e_1]_m, I_l = 2 (J_{l+1} + J_{l+3} + ...), with the order of summation exchanged, so
// that the inner sums are the same for every candidate step
struct BesselErr {
    const double *S;
    double odd = 0.0, even = 0.0;
    __device__ __forceinline__ void add(int k, double j)
    {
        if (k & 1) odd = fma(j, S[k], odd);
        else even = fma(j, S[k], even);
    }
    __device__ __forceinline__ void scale(int, double s) { odd *= s; even *= s; }
    // the sum's magnitude (scaled by the normalisation n before it is squared: unnormalised the parts
    // reach 1e+-280)
    __device__ __forceinline__ double value(double n) const { return sqrt(odd * n * (odd * n) + even * n * (even * n)); }
};
struct BesselErrStore : BesselErr {
    BesselStore st;
    __device__ __forceinline__ void add(int k, double j) { BesselErr::add(k, j); st.add(k, j); }
    __device__ __forceinline__ void scale(int k, double s) { BesselErr::scale(k, s); st.scale(k, s); }
};
struct BesselRead {   // sum_k J_k w_k G_k
    const double2 *g;
    double re = 0.0, im = 0.0;
    __device__ __forceinline__ void add(int k, double j)
    {
        const double2 v = g[k];
        re = fma(j, v.x, re);
        im = fma(j, v.y, im);
    }
    __device__ __forceinline__ void scale(int, double s) { re *= s; im *= s; }
};

constexpr int EXPW = 4;   // warps of the small exponential, one per SM sub-partition (each has its own FP64 pipe)
struct ExpSmem4 : ExpSmem {
    double S[KMAX + 2];        // sums of BesselErr
    double kd[NKD];            // the doubles 0, 1, 2, ...
    double2 yp[EXPW][32];      // partial sums of y
    double cr[2], inv[32];     // T's centre and half-width; normalisation of the candidates' sequences
    double tau, err;
    int pick, next;
    double integ[40][2];       // int P over [t_now, output o] and over the step, by halves of the nodes
};

// <psi0|psi(t_now + tp)> and P there
__device__ __forceinline__ double read_P(const ExpSmem4 &sm, double tp, double r, int K, double beta0)
{
    BesselRead f{sm.gk};
    // (the sums are scaled before they are squared: unnormalised they reach 1e+-280; the phase
    // exp(-i tp c) drops out)
    const double n = bessel_down(tp * r, K, sm.kd, f) * beta0, re = f.re * n, im = f.im * n;
    return re * re + im * im;
}

// Chebyshev vectors of the step's T and the sums S of BesselErr (one warp).
__device__ __forceinline__ void exp_basis(ExpSmem4 &sm, int me, int K, double shift)
{
    const int lane = threadIdx.x & 31;
    const double2 cr = chebyshev_basis(sm, me, K);
    if (lane == 0) { sm.cr[0] = cr.x + shift; sm.cr[1] = cr.y; }
    // w_0 = 1, w_k = 2 (-i)^k: S_k is real for odd k, imaginary for even k; lane 0 sums the even l,
    // lane 1 the odd l
    if (lane < 2) {
        double acc = 0.0;
        for (int l = lane; l <= K; l += 2) {
            const double t = sm.tch[l * 32 + me - 1] * (l == 0 ? 1.0 : 2.0);
            const int q = l & 3;   // (-i)^l = 1, -i, -1, i
            acc += (q == 0 || q == 3) ? t : -t;
            sm.S[l + 1] = 2.0 * acc;
        }
        if (lane == 0) sm.S[0] = 0.0;
    }
    __syncwarp();
}

// w_k G_k = w_k sum_j g_j [T_k e_1]_j for k = first, first + step, ...
__device__ __forceinline__ void exp_gk(ExpSmem4 &sm, int me, int K, int first, int step)
{
    for (int k = first; k <= K; k += step) {
        double re = 0.0, im = 0.0;
        for (int j = 0; j < me; ++j) {
            const double t = sm.tch[k * 32 + j];
            re = fma(sm.g[j].x, t, re);
            im = fma(sm.g[j].y, t, im);
        }
        const double w = k == 0 ? 1.0 : 2.0;
        re *= w;
        im *= w;
        sm.gk[k] = (k & 3) == 0 ? make_double2(re, im) : (k & 3) == 1 ? make_double2(im, -re)
                   : (k & 3) == 2 ? make_double2(-re, -im) : make_double2(-im, re);
    }
}

// sum_k w_k J_k T_kj over k = warp, warp + 4, ... for component j = lane ((-i)^k is the same for all of a
// warp's k), and the phase and sum of the four parts: y_j of the combine
__device__ __forceinline__ void exp_parts(ExpSmem4 &sm, const double *J, int me, int K)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    double t = 0.0;
    for (int k = warp; k <= K; k += 4) t = fma(J[k], sm.tch[k * 32 + lane], t);
    t *= 2.0;
    if (warp == 0) t -= J[0] * sm.tch[lane];
    sm.yp[warp][lane] = lane >= me ? make_double2(0.0, 0.0)
                        : warp == 0 ? make_double2(t, 0.0) : warp == 1 ? make_double2(0.0, -t)
                        : warp == 2 ? make_double2(-t, 0.0) : make_double2(0.0, t);
}
__device__ __forceinline__ double2 exp_y(const ExpSmem4 &sm, double phase)
{
    const int lane = threadIdx.x & 31;
    const double2 a = sm.yp[0][lane], b = sm.yp[1][lane], d = sm.yp[2][lane], e = sm.yp[3][lane];
    double sn, cs;
    sincos(phase, &sn, &cs);
    return cmul(make_double2(cs, -sn), make_double2(a.x + d.x, b.y + e.y));
}

// First output past the step [t_now, t_now + tau] (times are sorted; one warp).
__device__ __forceinline__ int exp_next(const double *times, int next0, int n_times, double t_now, double tau, bool last)
{
    int nx = next0;
    for (;;) {
        const int o = nx + (threadIdx.x & 31);
        const bool in = o < n_times && (last || times[o] - t_now <= tau * (1.0 + 1e-12));
        const unsigned mk = __ballot_sync(0xffffffffu, in);
        const int cnt = __popc(mk & ~(mk + 1u));
        nx += cnt;
        if (cnt < 32) return nx;
    }
}

// Temporal autocorrelation (Sec. 4): put(o, int P over [t_now, times[o]]) for the step's outputs and, unless
// it is the last step, put(next, int P over the whole step), by NGL-point Gauss-Legendre on the step's
// expansion (the frequencies of P are bounded by twice the half-width r, and tau r <= 50, so 64 nodes
// integrate it to rounding); (integral, half of the nodes) pairs are shared by the warps.
template <class F>
__device__ __forceinline__ void exp_integrals(ExpSmem4 &sm, const double *times, const double *glx, const double *glw,
                                              int next0, int next, bool last, double t_now, double tau, double r, int K,
                                              double beta0, F put)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int ob = next0; ob <= next; ob += 39) {
        const int nb = min(39, next + 1 - ob);   // integrals ob .. ob + nb - 1
        __syncthreads();
        for (int q = warp; q < 2 * nb; q += EXPW) {
            const int o = ob + (q >> 1), nd = 32 * (q & 1) + lane;
            if (o == next && last) continue;
            const double s = o == next ? tau : fmax(times[o] - t_now, 0.0);
            double acc = glw[nd] * read_P(sm, 0.5 * s * (1.0 + glx[nd]), r, K, beta0);
#pragma unroll
            for (int z = 16; z > 0; z >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, z);
            if (lane == 0) sm.integ[q >> 1][q & 1] = 0.5 * s * acc;
        }
        __syncthreads();
        for (int q = threadIdx.x; q < nb; q += 32 * EXPW)
            if (ob + q != next || !last) put(ob + q, sm.integ[q][0] + sm.integ[q][1]);
    }
}

// One CTA of four warps.  While warp 0 scans the candidate steps' Bessel sequences, warp 1 builds the
// Chebyshev vectors; the sums over the expansion, the outputs and the quadrature nodes are shared by all.
// (One warp doing this in turn took 130 us a step, 410 us with C(t): a quarter of a small sector's step.)
__global__ void __launch_bounds__(32 * EXPW) k_smallexp(ExpArgs ea)
{
    pdl_begin();
    KryCtl *ctl = ea.ctl;
    if (ctl->done) return;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    ExpSmem4 &sm = *(ExpSmem4 *)smem_raw;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int me = ctl->m_eff;
    if (warp == 0 && lane < me) {
        sm.al[lane] = ctl->alpha[lane];
        sm.be[lane] = ctl->beta[lane];
        double2 g;
        if (ctl->r0 >= 0) {
            const size_t idx = (size_t)lane * ea.ldW + (size_t)ctl->r0;
            double2 w;
            if (ea.c64) { float2 f = ((const float2 *)ea.W)[idx]; w = make_double2(f.x, f.y); }
            else if (ea.ff) { float4 f = ((const float4 *)ea.W)[idx]; w = make_double2((double)f.x + (double)f.z, (double)f.y + (double)f.w); }
            else w = ((const double2 *)ea.W)[idx];
            // <psi0|v_j> with psi0 = e_{r0}: the (real-valued psi0) conjugate is trivial
            const double s = ctl->sigma[lane];
            g = make_double2(w.x * s, w.y * s);
        } else {
            g = ctl->g[lane];
        }
        sm.g[lane] = g;
    }
    for (int k = threadIdx.x; k < NKD; k += 32 * EXPW) sm.kd[k] = (double)k;
    __syncthreads();
    const double beta0 = ctl->beta0, h = sm.be[me - 1];
    const double t_now = ctl->t_now, t_end = ctl->t_end, tol = ctl->tol;
    const double remaining = t_end - t_now;
    const double2 gc = gershgorin(sm, me);   // (every warp)
    const double tau_hi = fmin(remaining, XMAX / gc.y);
    const int K = cheb_degree(tau_hi * gc.y);
    // ---- Chebyshev vectors and the sums S; T holds H - s I: the phase centre gets s back
    if (warp == 1) exp_basis(sm, me, K, ctl->shift);
    __syncthreads();
    const double c = sm.cr[0], r = sm.cr[1];
    // ---- G_k w_k = w_k sum_j g_j [T_k e_1]_j (warps 1 to 3) and the step-size ladder (warp 0)
    if (warp > 0) {
        exp_gk(sm, me, K, threadIdx.x - 32, 32 * (EXPW - 1));
    } else {
        double tau_top = tau_hi, tau = 0.0, err = 0.0;
        int pick = -1;
        for (int round = 0; round < 4 && pick < 0; ++round) {
            const double tq = tau_top * pow(LADDER, (double)lane);
            BesselErrStore f;
            f.S = sm.S;
            f.st = BesselStore{sm.jb + lane * (KMAX + 2), K};
            if (tq * r < 1e-6)
                for (int k = 4; k <= K; ++k) f.st.out[k] = 0.0;
            const double nrm = bessel_down(tq * r, K, sm.kd, f);
            sm.inv[lane] = nrm;
            const double eq = h != 0.0 ? beta0 * fabs(h) / r * f.value(nrm) : 0.0;
            // a step's error budget must stay above the FP64 rounding unit of psi, otherwise
            // the tolerance is unreachable (KRY_ETOL) rather than met by ever smaller steps
            const double budget = STEP_SAFETY * 0.5 * tol * tq / t_end;
            const bool ok = tq > 0.0 && budget >= 2.3e-16 * beta0 && eq <= budget;
            const unsigned mask = __ballot_sync(0xffffffffu, ok || (remaining <= 0.0));
            if (mask) {
                pick = __ffs(mask) - 1;
                tau = __shfl_sync(0xffffffffu, tq, pick);
                err = __shfl_sync(0xffffffffu, eq, pick);
            } else {
                tau_top *= pow(LADDER, 32.0);
            }
        }
        if (lane == 0) { sm.pick = pick; sm.tau = tau; sm.err = err; }
    }
    __syncthreads();
    const int pick = sm.pick;
    const double tau = sm.tau;
    if (pick < 0) {
        if (threadIdx.x == 0) { ctl->err = KRY_ETOL; ctl->done = 1; }
        return;
    }
    const bool last = (tau >= remaining);
    // ---- y(tau) -> combine coefficients, and the outputs inside the step
    exp_parts(sm, sm.jb + pick * (KMAX + 2), me, K);
    const int next0 = ctl->next_out;
    if (warp == 0) {
        const int nx = exp_next(ea.times, next0, ctl->n_times, t_now, tau, last);
        if (lane == 0) sm.next = nx;
    }
    __syncthreads();
    const int next = sm.next;
    if (warp == 0 && lane < me) {
        const double2 y = exp_y(sm, tau * c);
        const double f = -beta0 * ctl->sigma[lane] * sm.inv[pick];
        ctl->coefY[lane] = make_double2(f * y.x, f * y.y);
    }
    // ---- dense output of P: one output per lane, 32 at a time, the warps in turn (warp 0 last)
    for (int o = next0 + 32 * ((warp + EXPW - 1) % EXPW) + lane; o - lane < next; o += 32 * EXPW)
        if (o < next) ea.P[o] = read_P(sm, fmax(ea.times[o] - t_now, 0.0), r, K, beta0);
    if (ea.Yout) {
        // whole-vector dense output: psi(t_o) = sum_j Yout[o][j] W_j with
        // Yout[o][j] = beta sigma_j [exp(-i tau' T) e_1]_j; 32 outputs' Bessel sequences at a time
        for (int ob = next0; ob < next; ob += 32) {
            __syncthreads();
            if (warp == 0) {
                const int o = ob + lane;
                const double tp = fmax(ea.times[o < next ? o : next - 1] - t_now, 0.0);
                BesselStore f{sm.jb + lane * (KMAX + 2), K};
                if (tp * r < 1e-6)
                    for (int k = 4; k <= K; ++k) f.out[k] = 0.0;
                sm.inv[lane] = bessel_down(tp * r, K, sm.kd, f);
            }
            __syncthreads();
            for (int o = ob + warp; o < min(next, ob + 32); o += EXPW) {
                if (lane >= me) continue;
                // sum_k w_k J_k T_kj, the degrees by k mod 4 (phases 1, -i, -1, i): one multiply-add each
                const double *J = sm.jb + (o - ob) * (KMAX + 2);
                double part[4] = {0.0, 0.0, 0.0, 0.0};
                for (int k0 = 0; k0 <= K; k0 += 4) {
#pragma unroll
                    for (int q = 0; q < 4; ++q)
                        if (k0 + q <= K) part[q] = fma(J[k0 + q], sm.tch[(k0 + q) * 32 + lane], part[q]);
                }
                const double2 s = make_double2(2.0 * (part[0] - part[2]) - J[0] * sm.tch[lane], 2.0 * (part[3] - part[1]));
                double sn, cs;
                sincos(fmax(ea.times[o] - t_now, 0.0) * c, &sn, &cs);
                const double2 y = cmul(make_double2(cs, -sn), s);
                const double f = beta0 * ctl->sigma[lane] * sm.inv[o - ob];
                ea.Yout[(size_t)o * MMAX + lane] = make_double2(f * y.x, f * y.y);
            }
        }
    }
    if (ea.C) {
        const double pint = ctl->pint;
        exp_integrals(sm, ea.times, ea.glx, ea.glw, next0, next, last, t_now, tau, r, K, beta0, [&](int o, double I) {
            if (o == next) ctl->pint = pint + I;
            else ea.C[o] = ea.times[o] > 0.0 ? (pint + I) / ea.times[o] : 1.0;
        });
    }
    if (threadIdx.x == 0) {
        ctl->out_begin = next0;
        ctl->out_end = next;
        ctl->next_out = next;
        ctl->t_now = last ? t_end : t_now + tau;
        ctl->tau_prev = tau;
        ctl->n_steps += 1;
        ctl->err_sum += sm.err;
        if (next >= ctl->n_times) ctl->finishing = 1;
    }
}

// y = exp(-i tau T) e_1 and err(tau) for given T, h (beta = 1): the step's own functions on one CTA of four warps.
__global__ void __launch_bounds__(32 * EXPW) k_expv(const double *alpha, const double *beta, int me, double h,
                                                    double tau, double *y, double *err)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    ExpSmem4 &sm = *(ExpSmem4 *)smem_raw;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (warp == 0 && lane < me) {
        sm.al[lane] = alpha[lane];
        sm.be[lane] = (lane + 1 < me) ? beta[lane] : h;
    }
    for (int k = threadIdx.x; k < NKD; k += 32 * EXPW) sm.kd[k] = (double)k;
    __syncthreads();
    const double x = tau * gershgorin(sm, me).y;   // (every warp)
    const int K = cheb_degree(x);
    if (warp == 1) exp_basis(sm, me, K, 0.0);
    __syncthreads();
    if (threadIdx.x == 0) {
        BesselErrStore f;
        f.S = sm.S;
        f.st = BesselStore{sm.jb, K};
        if (x < 1e-6)
            for (int k = 4; k <= K; ++k) f.st.out[k] = 0.0;
        sm.inv[0] = bessel_down<true>(x, K, sm.kd, f);
        *err = fabs(h) / sm.cr[1] * f.value(sm.inv[0]);
    }
    __syncthreads();
    exp_parts(sm, sm.jb, me, K);
    __syncthreads();
    if (warp == 0 && lane < me) {
        const double2 v = exp_y(sm, tau * sm.cr[0]);
        y[2 * lane] = v.x * sm.inv[0];
        y[2 * lane + 1] = v.y * sm.inv[0];
    }
}

// ---------------------------------------------------------------- batched realisations
// Every realisation k has its own T_k, coupling h_k and norm beta_k.  k_exp_scan_b finds,
// per realisation, the largest ladder step that meets the error budget; k_exp_apply_b takes
// the smallest of those (the leading error term grows with the step, so every realisation
// stays within its budget), builds exp(-i tau T_k) e_1 for the combine and reads P_k at
// every output time inside the step.

__device__ void load_tridiag_b(ExpSmem &sm, const KryCtlB *ctl, int k, int me, const ExpArgsB &ea)
{
    const int lane = threadIdx.x;
    if (lane < me) {
        sm.al[lane] = ctl->alpha[lane][k];
        sm.be[lane] = ctl->beta[lane][k];
        double2 g;
        if (ctl->hd.r0 >= 0) {
            const size_t idx = (size_t)lane * ea.ldW + (size_t)ctl->r0k[k] * ea.K + k;
            double2 w;
            if (ea.c64) { float2 f = ((const float2 *)ea.W)[idx]; w = make_double2(f.x, f.y); }
            else if (ea.ff) { float4 f = ((const float4 *)ea.W)[idx]; w = make_double2((double)f.x + (double)f.z, (double)f.y + (double)f.w); }
            else w = ((const double2 *)ea.W)[idx];
            const double s = ctl->sigma[lane][k];
            g = make_double2(w.x * s, w.y * s);
        } else {
            g = ctl->g[lane][k];
        }
        sm.g[lane] = g;
    }
    __syncwarp();
}

// Largest ladder step of realisation blockIdx.x that meets its error budget (one warp).
__global__ void __launch_bounds__(32) k_exp_scan_b(ExpArgsB ea)
{
    KryCtlB *ctl = ea.ctl;
    const KryHdrB &H = ctl->hd;
    if (H.done) return;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    ExpSmem4 &sm = *(ExpSmem4 *)smem_raw;
    const int k = blockIdx.x, lane = threadIdx.x;
    const int me = ctl->m_eff[k];
    load_tridiag_b(sm, ctl, k, me, ea);
    for (int q = lane; q < NKD; q += 32) sm.kd[q] = (double)q;
    __syncwarp();
    const double beta0 = ctl->beta0[k], h = sm.be[me - 1];
    const double remaining = H.t_end - H.t_now;
    const double2 cr = gershgorin(sm, me);
    const double tau_hi = fmin(remaining, XMAX / cr.y);
    const int Kc = cheb_degree(tau_hi * cr.y);
    exp_basis(sm, me, Kc, 0.0);
    const double r = sm.cr[1];
    double tau_top = tau_hi, tau = 0.0;
    int pick = -1;
    for (int round = 0; round < 4 && pick < 0; ++round) {
        const double tq = tau_top * pow(LADDER, (double)lane);
        BesselErr f{sm.S};
        const double nrm = bessel_down(tq * r, Kc, sm.kd, f);
        const double eq = h != 0.0 ? beta0 * fabs(h) / r * f.value(nrm) : 0.0;
        const double budget = STEP_SAFETY * 0.5 * H.tol * tq / H.t_end;
        const bool ok = tq > 0.0 && budget >= 2.3e-16 * beta0 && eq <= budget;
        const unsigned mask = __ballot_sync(0xffffffffu, ok || (remaining <= 0.0));
        if (mask) {
            pick = __ffs(mask) - 1;
            tau = __shfl_sync(0xffffffffu, tq, pick);
        } else {
            tau_top *= pow(LADDER, 32.0);
        }
    }
    if (lane == 0) {
        ctl->tau_ok[k] = (pick < 0) ? -1.0 : tau;
        if (pick < 0) ctl->hd.err = KRY_ETOL;
    }
}

// The common step of realisation blockIdx.x: combine coefficients, P (and C) at the outputs inside it.  Four
// warps, as in k_smallexp.
__global__ void __launch_bounds__(32 * EXPW) k_exp_apply_b(ExpArgsB ea)
{
    KryCtlB *ctl = ea.ctl;
    KryHdrB &H = ctl->hd;
    if (H.done) return;
    const int k = blockIdx.x, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (H.err) {
        if (k == 0 && threadIdx.x == 0) H.done = 1;
        return;
    }
    extern __shared__ __align__(16) unsigned char smem_raw[];
    ExpSmem4 &sm = *(ExpSmem4 *)smem_raw;
    double tau = 1e300;
    for (int kk = lane; kk < ea.K; kk += 32) tau = fmin(tau, ctl->tau_ok[kk]);
    for (int o = 16; o > 0; o >>= 1) tau = fmin(tau, __shfl_xor_sync(0xffffffffu, tau, o));
    const int me = ctl->m_eff[k];
    if (warp == 0) load_tridiag_b(sm, ctl, k, me, ea);
    for (int q = threadIdx.x; q < NKD; q += 32 * EXPW) sm.kd[q] = (double)q;
    __syncthreads();
    const double beta0 = ctl->beta0[k], h = sm.be[me - 1];
    const double t_now = H.t_now, t_end = H.t_end, remaining = t_end - t_now;
    const bool last = (tau >= remaining);
    const double2 cr = gershgorin(sm, me);   // (every warp)
    const int Kc = cheb_degree(tau * cr.y);
    if (warp == 1) {
        exp_basis(sm, me, Kc, ctl->shift[k]);   // T holds H_k - s_k I
    } else if (threadIdx.x == 0) {   // (one lane: the sequence is rescaled in place)
        BesselStore f{sm.jb, Kc};
        if (tau * cr.y < 1e-6)
            for (int q = 4; q <= Kc; ++q) f.out[q] = 0.0;
        sm.inv[0] = bessel_down(tau * cr.y, Kc, sm.kd, f);
    }
    __syncthreads();
    const double c = sm.cr[0], r = sm.cr[1];
    exp_gk(sm, me, Kc, threadIdx.x, 32 * EXPW);
    exp_parts(sm, sm.jb, me, Kc);
    const int next0 = H.next_out;
    if (warp == 0) {
        const int nx = exp_next(ea.times, next0, H.n_times, t_now, tau, last);
        if (lane == 0) sm.next = nx;
    } else if (warp == 1) {   // the error estimate of this step
        double odd = 0.0, even = 0.0;
        for (int q = lane; q <= Kc; q += 32) {
            const double t = sm.jb[q] * sm.inv[0] * sm.S[q];
            if (q & 1) odd += t;
            else even += t;
        }
        for (int o = 16; o > 0; o >>= 1) {
            odd += __shfl_xor_sync(0xffffffffu, odd, o);
            even += __shfl_xor_sync(0xffffffffu, even, o);
        }
        if (lane == 0)
            ctl->err_k[k] = h != 0.0 ? beta0 * fabs(h) / r * sqrt(odd * odd + even * even) : 0.0;
    }
    __syncthreads();
    const int next = sm.next;
    if (warp == 0) {
        double2 y = make_double2(0.0, 0.0);
        if (lane < me) {
            y = exp_y(sm, tau * c);
            const double f = -beta0 * ctl->sigma[lane][k] * sm.inv[0];
            y = make_double2(f * y.x, f * y.y);
        }
        ctl->coefY[lane][k] = y;
    }
    for (int o = next0 + 32 * ((warp + EXPW - 1) % EXPW) + lane; o - lane < next; o += 32 * EXPW)
        if (o < next) ea.P[(size_t)o * ea.K + k] = read_P(sm, fmax(ea.times[o] - t_now, 0.0), r, Kc, beta0);
    if (ea.C) {
        const double pint = ctl->pint[k];
        exp_integrals(sm, ea.times, ea.glx, ea.glw, next0, next, last, t_now, tau, r, Kc, beta0, [&](int o, double I) {
            if (o == next) ctl->pint[k] = pint + I;
            else ea.C[(size_t)o * ea.K + k] = ea.times[o] > 0.0 ? (pint + I) / ea.times[o] : 1.0;
        });
    }
    if (k == 0 && threadIdx.x == 0) {
        H.next_out_new = next;
        H.t_next = last ? t_end : t_now + tau;
        H.finishing = (next >= H.n_times) ? 1 : 0;
    }
}

int launch_exp_b(const ExpArgsB &a, cudaStream_t s)
{
    KRY_CU(cudaFuncSetAttribute(k_exp_scan_b, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(ExpSmem4)));
    KRY_CU(cudaFuncSetAttribute(k_exp_apply_b, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(ExpSmem4)));
    k_exp_scan_b<<<a.K, 32, sizeof(ExpSmem4), s>>>(a);
    KRY_CU(cudaGetLastError());
    k_exp_apply_b<<<a.K, 32 * EXPW, sizeof(ExpSmem4), s>>>(a);
    KRY_CU(cudaGetLastError());
    return KRY_OK;
}

int launch_smallexp(const ExpArgs &a, cudaStream_t s, int pdl)
{
    KRY_CU(cudaFuncSetAttribute(k_smallexp, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)sizeof(ExpSmem4)));
    KRY_CU(launch_ex(pdl, k_smallexp, 1, 32 * EXPW, sizeof(ExpSmem4), s, a));
    KRY_CU(cudaGetLastError());
    return KRY_OK;
}

}  // namespace kry

using namespace kry;

extern "C" int kry_tridiag_expv(const double *alpha, const double *beta, int m, double h, double tau,
                                double *y_out, double *err_out, void *stream)
{
    if (!alpha || (m > 1 && !beta) || !y_out || !err_out || m < 1 || m > MMAX || !(tau >= 0.0) ||
        !(tau * 1.0 < 1e300)) {
        set_error("kry_tridiag_expv: bad arguments");
        return KRY_EINVAL;
    }
    cudaStream_t s = (cudaStream_t)stream;
    double *d = nullptr;
    KRY_CU(cudaMalloc(&d, sizeof(double) * (4 * MMAX + 2)));
    double *da = d, *db = d + MMAX, *dy = d + 2 * MMAX, *de = d + 4 * MMAX;
    cudaError_t e = cudaMemcpyAsync(da, alpha, sizeof(double) * m, cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess && m > 1)
        e = cudaMemcpyAsync(db, beta, sizeof(double) * (m - 1), cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_expv, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(ExpSmem4));
    if (e == cudaSuccess) {
        k_expv<<<1, 32 * EXPW, sizeof(ExpSmem4), s>>>(da, db, m, h, tau, dy, de);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaMemcpyAsync(y_out, dy, sizeof(double) * 2 * m, cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaMemcpyAsync(err_out, de, sizeof(double), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    cudaFree(d);
    if (e != cudaSuccess) return cuda_fail(e, "kry_tridiag_expv");
    return KRY_OK;
}

// ---------------------------------------------------------------- allocation-free variant
//
// kry_tridiag_expv_noalloc runs the same kernel as kry_tridiag_expv, but its device-side
// copies of alpha, beta and the results live in the fixed array below instead of memory
// from cudaMalloc.  It serves callers that hand all device memory to their own pool with a
// hard cap, and callers that cannot accept the device-wide synchronisation that cudaFree
// performs while their other streams are busy.
//
// The array holds alpha[32], beta[32], y[64] and err (about 1 KB).  Every GPU that loads
// this library keeps it for the life of the process.  Host code cannot pass the array's
// name to a kernel (in host code it is a stand-in, not a device address), so the call looks
// up the real address with cudaGetSymbolAddress while the caller's device is current, once
// per device and CUDA context: the address is kept together with the id of the context it
// was looked up in, and looked up again when the current context differs (after a
// cudaDeviceReset the module is loaded anew and the array may move).  When the driver
// cannot report a context id the address is looked up on every call.

#include <mutex>

static __device__ __align__(256) double g_expv_scratch[4 * kry::MMAX + 8];

namespace {
constexpr int kMaxDevices = 64;
std::mutex g_expv_mu;
struct ScratchAddr {
    unsigned long long ctx_id;   // 0 = not looked up
    double *ptr;
};
ScratchAddr g_expv_addr[kMaxDevices] = {};

// Id of the calling thread's current CUDA context (unique over the process's lifetime), or 0
// if there is none or the driver cannot say.  The two driver calls are fetched through the
// runtime, so the library does not link the driver library itself.
unsigned long long current_context_id()
{
    typedef int (*get_current_t)(void **);
    typedef int (*get_id_t)(void *, unsigned long long *);
    static get_current_t get_current = nullptr;
    static get_id_t get_id = nullptr;
    static std::once_flag once;
    std::call_once(once, [] {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q = cudaDriverEntryPointSymbolNotFound;
        if (cudaGetDriverEntryPointByVersion("cuCtxGetCurrent", &p, 12000, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            get_current = (get_current_t)p;
        p = nullptr;
        q = cudaDriverEntryPointSymbolNotFound;
        if (cudaGetDriverEntryPointByVersion("cuCtxGetId", &p, 12000, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            get_id = (get_id_t)p;
        cudaGetLastError();
    });
    if (!get_current || !get_id) return 0;
    void *ctx = nullptr;
    if (get_current(&ctx) != 0 || !ctx) return 0;
    unsigned long long id = 0;
    if (get_id(ctx, &id) != 0) return 0;
    return id;
}

int expv_scratch(double **out)
{
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return cuda_fail(e, "cudaGetDevice");
    if (dev < 0 || dev >= kMaxDevices) {
        set_error("kry_tridiag_expv_noalloc: device ordinal %d is above %d", dev, kMaxDevices - 1);
        return KRY_EINVAL;
    }
    const unsigned long long id = current_context_id();
    std::lock_guard<std::mutex> lock(g_expv_mu);
    ScratchAddr &a = g_expv_addr[dev];
    if (id == 0 || a.ctx_id != id || !a.ptr) {
        void *p = nullptr;
        e = cudaGetSymbolAddress(&p, g_expv_scratch);
        if (e != cudaSuccess) return cuda_fail(e, "cudaGetSymbolAddress(g_expv_scratch)");
        a.ptr = (double *)p;
        a.ctx_id = current_context_id();   // the lookup made the runtime's context current
    }
    *out = a.ptr;
    return KRY_OK;
}
}  // namespace

extern "C" int kry_tridiag_expv_noalloc(const double *alpha, const double *beta, int m, double h,
                                        double tau, double *y_out, double *err_out, void *stream)
{
    if (m > MMAX) {
        set_error("kry_tridiag_expv_noalloc: m = %d exceeds the maximum %d that its fixed "
                  "device scratch holds", m, MMAX);
        return KRY_EINVAL;
    }
    if (!alpha || (m > 1 && !beta) || !y_out || !err_out || m < 1 || !(tau >= 0.0) ||
        !(tau < 1e300)) {
        set_error("kry_tridiag_expv_noalloc: bad arguments");
        return KRY_EINVAL;
    }
    double *d = nullptr;
    if (int rc = expv_scratch(&d)) return rc;
    cudaStream_t s = (cudaStream_t)stream;
    double *da = d, *db = d + MMAX, *dy = d + 2 * MMAX, *de = d + 4 * MMAX;
    // Every element the kernel reads is copied in below and every element read back is
    // written by the kernel, so nothing left over from an earlier call is used.
    cudaError_t e = cudaMemcpyAsync(da, alpha, sizeof(double) * m, cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess && m > 1)
        e = cudaMemcpyAsync(db, beta, sizeof(double) * (m - 1), cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_expv, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)sizeof(ExpSmem4));
    if (e == cudaSuccess) {
        k_expv<<<1, 32 * EXPW, sizeof(ExpSmem4), s>>>(da, db, m, h, tau, dy, de);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaMemcpyAsync(y_out, dy, sizeof(double) * 2 * m, cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaMemcpyAsync(err_out, de, sizeof(double), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) return cuda_fail(e, "kry_tridiag_expv_noalloc");
    return KRY_OK;
}

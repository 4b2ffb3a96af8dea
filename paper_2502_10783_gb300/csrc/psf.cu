// psf.cu -- batched differentiable PSF model and Levenberg-Marquardt fit
// (paper-silent reading of the photometry of Sec. 2.2.5; elliptical Moffat or
// Gaussian, 7 parameters x0, y0, F, sky, sx, sy, theta, point-sampled at the
// pixel centres of an S x S stamp).
//
// The fit (k_psf_fit) runs one stamp per lane: each lane keeps its LM state,
// J'WJ (28 terms), J'W r (7) and chi^2 in registers and evaluates its stamp from
// a column of the warp's shared-memory tile.  The damped 7 x 7 normal equations
// are solved in FP64 (LDL', no square roots), one system per lane, so one FP64
// instruction of the warp serves 32 stamps.  The forward model and its adjoint
// (k_psf_fwd, k_psf_adj) evaluate the same point-sampled model.
#include <math.h>

#include <algorithm>

#include "jobs.cuh"

namespace ipp {

constexpr float F_PI = 3.14159265358979f;

// The FP64 pipe of this part is narrow (1/64 of the FP32 rate), so the solve
// spends it on the arithmetic of the factorisation alone: the widening of the
// FP32 normal equations, the pivot tests and the reciprocal seeds are integer
// operations on the IEEE-754 bit patterns.

// Exact float -> double (sign, exponent rebiased by 1023 - 127, mantissa
// shifted up by 52 - 23 bits); zeros, infinities and NaNs map to their double
// counterparts, subnormals take the conversion instruction.
__device__ __forceinline__ double widen(float f) {
    const uint32_t u = __float_as_uint(f);
    const uint32_t e = (u >> 23) & 0xffu, m = u & 0x7fffffu, sg = u & 0x80000000u;
    if (e == 0u && m != 0u) return (double)f;
    const uint32_t e64 = e == 0u ? 0u : (e == 0xffu ? 0x7ffu : e + 896u);
    return __hiloint2double((int)(sg | (e64 << 20) | (m >> 3)), (int)(m << 29));
}

// double -> float rounded to nearest (ties away from zero) for |v| in the
// normal single range, 0 below it and infinity above it.
__device__ __forceinline__ float narrow(double v) {
    const uint32_t hi = (uint32_t)__double2hiint(v), lo = (uint32_t)__double2loint(v);
    const int e = (int)((hi >> 20) & 0x7ffu) - 896;
    const uint32_t sg = hi & 0x80000000u;
    if (e <= 0) return __uint_as_float(sg);
    if (e >= 255) return __uint_as_float(sg | 0x7f800000u);
    // exponent and the top 23 mantissa bits, plus the first discarded bit
    // (a carry out of the mantissa moves into the exponent, as it should)
    const uint32_t body = ((uint32_t)e << 23) | ((hi & 0xfffffu) << 3) | (lo >> 29);
    return __uint_as_float(sg | (body + ((lo >> 28) & 1u)));
}

// 1/d for a pivot d by Newton's iteration x <- x + x (1 - d x) from a
// single-precision seed; each step doubles the correct bits (about 22 -> 44 ->
// beyond double precision).  Pivots outside 2^-100 .. 2^100 divide.
__device__ __forceinline__ double recip_pivot(double d) {
    const int e = (__double2hiint(d) >> 20) & 0x7ff;
    if (e > 923 && e < 1123) {
        double x = widen(__fdividef(1.0f, narrow(d)));
        x = fma(x, fma(-d, x, 1.0), x);
        return fma(x, fma(-d, x, 1.0), x);
    }
    return 1.0 / d;
}

// d > 0, finite and normal: sign clear, exponent field in 1 .. 2046
__device__ __forceinline__ bool pivot_ok(double d) {
    const uint32_t hi = (uint32_t)__double2hiint(d);
    return hi - 0x00100000u < 0x7fe00000u;
}

__device__ __forceinline__ int tri(int i, int j) { return i * (i - 1) / 2 + j; }  // strictly lower, j < i

// Solve (H + lambda D) x = g, D = diag(H) floored at 1e-9 max(diag), in FP64 by
// an LDL' factorisation (no square roots).  H packed upper-triangular row-major
// (28 entries).  Row-oriented: row i of L is formed from the earlier rows with
// W(q) = L(i,q) D(q) held as a temporary, so each product L(i,q) D(q) L(j,q)
// costs one fused multiply-add.  Returns false if a pivot is not positive.
__device__ __forceinline__ bool solve7(const float Hf[28], const float gf[7], double lam, double x[7]) {
    double L[21], iD[7];
    float dmaxf = 0.f;
#pragma unroll
    for (int a = 0; a < 7; a++) dmaxf = fmaxf(dmaxf, Hf[a * 7 - a * (a - 1) / 2]);
    const double floor_d = 1e-9 * widen(dmaxf);
    bool ok = true;
#pragma unroll
    for (int i = 0; i < 7; i++) {
        double W[7];
#pragma unroll
        for (int j = 0; j < i; j++) {
            // H(j, i) from the upper row-major packing
            double t = widen(Hf[j * 7 - j * (j - 1) / 2 + (i - j)]);
#pragma unroll
            for (int q = 0; q < j; q++) t = fma(-W[q], L[tri(j, q)], t);
            W[j] = t;
            L[tri(i, j)] = t * iD[j];
        }
        const double h = widen(Hf[i * 7 - i * (i - 1) / 2]);
        double d = fma(lam, fmax(h, floor_d), h);
#pragma unroll
        for (int q = 0; q < i; q++) d = fma(-W[q], L[tri(i, q)], d);
        ok = ok && pivot_ok(d);
        iD[i] = recip_pivot(d);
    }
    if (!ok) return false;
    double z[7];
#pragma unroll
    for (int i = 0; i < 7; i++) {
        double t = widen(gf[i]);
#pragma unroll
        for (int q = 0; q < i; q++) t = fma(-L[tri(i, q)], z[q], t);
        z[i] = t;
    }
#pragma unroll
    for (int i = 6; i >= 0; i--) {
        double t = z[i] * iD[i];
#pragma unroll
        for (int q = i + 1; q < 7; q++) t = fma(-L[tri(q, i)], x[q], t);
        x[i] = t;
    }
    return true;
}

// ---------------------------------------------------------------------------
// LM fit, G lanes per stamp.  A warp (one block) owns a contiguous chunk of
// stamps and fits 32/G of them at a time, one per slot; the G lanes of a slot
// hold identical copies of its LM state and all slots step through the same
// round:
//   (1) idle slots take the next stamps of the chunk, in slot order; the warp
//       stages each new stamp in shared memory (pixel k of slot s at
//       k fit_pitch(G) + s) and computes its default starting point together;
//   (2) slots with a fit in progress solve their damped normal equations (FP64); one
//       whose step promises little takes its convergence test, a second solve -- at
//       G = 1 it is put on hold until that can be made for several slots at once;
//   (3) every slot with a point to try evaluates chi^2, J'WJ and J'Wr there,
//       each lane of the slot over every G-th stamp row, and the slot's lanes
//       add their sums with shuffles;
//   (4) each slot accepts, rejects or stops.
// The Jacobian is evaluated at every trial point, not only after an accepted
// step: a rejected trial wastes its normal equations, but no slot of the warp
// waits for another slot's extra evaluation.  Per-lane accumulation over the
// pixels is sequential; chi^2 is summed per stamp row first, so its rounding
// stays near that of a 2 x S-term sum.
//
// G = 1 for large batches: one FP64 instruction serves 32 solves, and G = 2
// (12 warps an SM instead of 7) measured slower on 200,000 stamps because it
// repeats every solve on both lanes of a slot, the FP64 pipe of this part
// running at 1/64 of the FP32 rate.  Batches too small to give every lane a
// stamp take G = 2 or 4 (fit_lanes_per_stamp), where the shorter rounds win.
//
// Bound by the latency of one lane's model evaluation with the two warps a scheduler
// that the stamps' tiles leave room for, so at G = 1 a tile has no padding column
// (15 x 15 stamps: 28.1 KB, eight warps an SM; 29 KB and seven before): a row, one
// pixel of 32 stamps, is read without conflicts, and only the staging stores, one
// stamp's column, meet in one bank (the registers, 248 and more a thread, hold eight
// warps as well).  200,000 stamps of 15 x 15: 15.3 -> 12.7 ms with the forms of eval_lane
// and border_pair below.
constexpr int FL_MAX_WARPS = 8;

// G = 1: slots on hold for which the undamped system is solved (fewer when nothing else is
// left to do in the warp, or no stamp waits for a slot).  A solve costs the warp the same
// FP64 time for one lane as for 32, and with 32 fits a warp one of them converges in
// almost every round: solved at once, the second solve doubled the FP64 work; waiting
// costs a slot a round or two, which only a waiting stamp can make good: 50,000 stamps of
// 11 x 11, Gaussian, 2510 us solved at once, 2600 held to the end, 2450 so.
constexpr int HOLD_MIN = 4;

// Base-2 logarithm of the hardware without the steps for subnormal arguments: 1 + q >= 1
// has none.  (The exponential and the quotient keep theirs: a profile far out is part of a
// fit whose star lies off its stamp.)
__device__ __forceinline__ float lg2_fast(float x) {
    float y;
    asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// chi^2, J'WJ and J'Wr of one stamp at pp.  The model of k_psf_fwd with the
// per-trial constants (reciprocal widths, normalisation, trig) taken out of the
// pixel loop and its derivatives regrouped around T = 2 dP/dq, a = u/sx^2 and
// b = v/sy^2:
//   dm/dx0 = T (b s - a c),  dm/dy0 = -T (a s + b c),  dm/dF = P/F,  dm/dsky = 1,
//   dm/dsx = -(P + T a u)/sx,  dm/dsy = -(P + T b v)/sy,
//   dm/dtheta = T u v (sy^2 - sx^2)/(sx^2 sy^2).
// Moffat (1+q)^-beta is exp2(-beta log2(1+q)) with the fast base-2 logarithm
// (absolute error ~2^-22 on the exponent, a few ulp in P).
template <int MODEL, bool WEIGHTED, int G, int PITCH>
__device__ __forceinline__ float eval_lane(const float* __restrict__ col, const float* __restrict__ wts, int S,
                                           float beta, const float pp[7], float Ht[28], float gt[7], float* sm2) {
    const int h = (threadIdx.x & 31) % G;
#pragma unroll
    for (int a = 0; a < 28; a++) Ht[a] = 0.f;
#pragma unroll
    for (int a = 0; a < 7; a++) gt[a] = 0.f;
    float sn, cs;
    sincosf(pp[6], &sn, &cs);
    const float x0 = pp[0], F = pp[2], sky = pp[3];
    const float isx = 1.0f / pp[4], isy = 1.0f / pp[5];
    const float isx2 = isx * isx, isy2 = isy * isy;
    const float kth = (pp[5] - pp[4]) * (pp[5] + pp[4]) * isx2 * isy2;
    const float A0 = (MODEL == IPP_PSF_GAUSS ? 0.5f / F_PI : (beta - 1.0f) / F_PI) * isx * isy;
    const float tq = MODEL == IPP_PSF_GAUSS ? -1.0f : -2.0f * beta;  // T = tq P / (1+q) (Moffat), -P (Gauss)
    float chi = 0.f, star2 = 0.f;  // chi^2 and sum w P^2 (the star part of the model, squared)
    for (int i = h; i < S; i += G) {
        const float dy = (float)i - pp[1];
        const float sdy = sn * dy, cdy = cs * dy;
        const float* row = col + i * S * PITCH;
        float rowc = 0.f, rows = 0.f;
        float jf = 0.f;
#pragma unroll 5
        for (int j = 0; j < S; j++, jf += 1.0f) {
            const float dx = jf - x0;
            const float u = fmaf(cs, dx, sdy), v = fmaf(-sn, dx, cdy);
            const float a = u * isx2, b = v * isy2;
            const float q = fmaf(u, a, v * b);
            float A1, P, T;
            if (MODEL == IPP_PSF_GAUSS) {
                A1 = A0 * exp2f(-0.72134752f * q);  // exp(-q/2)
                P = F * A1;
                T = -P;
            } else {
                const float base = 1.0f + q;
                A1 = A0 * exp2f(-beta * lg2_fast(base));
                P = F * A1;
                T = __fdividef(tq * P, base);
            }
            const float wk = WEIGHTED ? __ldg(wts + i * S + j) : 1.0f;
            const float r = row[j * PITCH] - (P + sky);
            rowc = fmaf(wk * r, r, rowc);
            rows = fmaf(wk * P, P, rows);
            float e[7];
            e[0] = T * fmaf(b, sn, -a * cs);
            e[1] = -T * fmaf(a, sn, b * cs);
            e[2] = A1;
            e[3] = 1.0f;
            e[4] = -isx * fmaf(T * a, u, P);
            e[5] = -isy * fmaf(T * b, v, P);
            e[6] = T * u * v * kth;
            int t = 0;
#pragma unroll
            for (int c = 0; c < 7; c++) {
                const float wa = wk * e[c];
                gt[c] = fmaf(wa, r, gt[c]);
#pragma unroll
                for (int d = c; d < 7; d++) {
                    if (WEIGHTED || c != 3 || d != 3) Ht[t] = fmaf(wa, e[d], Ht[t]);
                    t++;
                }
            }
        }
        chi += rowc;
        star2 += rows;
    }
    if (!WEIGHTED) Ht[18] = (float)((S - h + G - 1) / G * S);   // (sky, sky): the lane's pixels
    if (G > 1) {  // all lanes of the slot are here (their states are identical)
        const unsigned pm = ((1u << G) - 1u) << ((threadIdx.x & 31) & ~(G - 1));
#pragma unroll
        for (int o = 1; o < G; o <<= 1) {
#pragma unroll
            for (int a = 0; a < 28; a++) Ht[a] += __shfl_xor_sync(pm, Ht[a], o);
#pragma unroll
            for (int a = 0; a < 7; a++) gt[a] += __shfl_xor_sync(pm, gt[a], o);
            chi += __shfl_xor_sync(pm, chi, o);
            star2 += __shfl_xor_sync(pm, star2, o);
        }
    }
    *sm2 = star2;
    return chi;
}

// Pixel index of border pixel b (0 <= b < 4S-4) of an S x S stamp: the top
// row, the bottom row, then rows 1..S-2 alternating left and right edge.
__device__ __forceinline__ int border_k(int b, int S) {
    if (b < S) return b;
    if (b < 2 * S) return (S - 1) * S + (b - S);
    const int c = b - 2 * S;
    return (1 + (c >> 1)) * S + ((c & 1) ? S - 1 : 0);
}

// Order statistics k0 <= k1 of the border's keys, the same values in every lane.
// Each lane holds at most 4 of the nb keys (S <= 32) and counts, for each, the keys
// below and at most equal to it as every key passes by in a shuffle: the loads,
// compares and shuffles are independent, where a bisection of the key range is 32
// dependent rounds (0.6 against 2 K cycles of a warp for 15 x 15 stamps, with its
// other lanes' fits waiting).
template <int NK>
__device__ __forceinline__ void border_pair(const uint32_t* key, int nb, int k0, int k1, uint32_t& ka, uint32_t& kb) {
    const int lane = threadIdx.x & 31;
    int lt[NK], le[NK];
#pragma unroll
    for (int s = 0; s < NK; s++) lt[s] = le[s] = 0;
#pragma unroll
    for (int t = 0; t < NK; t++) {
        const int m = min(32, nb - 32 * t);
#pragma unroll 4
        for (int l = 0; l < m; l++) {
            const uint32_t v = __shfl_sync(0xffffffffu, key[t], l);
#pragma unroll
            for (int s = 0; s < NK; s++) {
                lt[s] += v < key[s];
                le[s] += v <= key[s];
            }
        }
    }
    ka = kb = 0u;
#pragma unroll
    for (int s = 0; s < NK; s++) {
        const bool mine = lane + 32 * s < nb;
        const unsigned a = __ballot_sync(0xffffffffu, mine && lt[s] <= k0 && k0 < le[s]);
        const unsigned b = __ballot_sync(0xffffffffu, mine && lt[s] <= k1 && k1 < le[s]);
        if (a) ka = __shfl_sync(0xffffffffu, key[s], __ffs(a) - 1);
        if (b) kb = __shfl_sync(0xffffffffu, key[s], __ffs(b) - 1);
    }
}

// Default start of the stamp at src: centre, border-median sky, sum above sky,
// widths 1.6 / 1.4, theta 0.  All lanes of the warp take part and all return the
// same values.
__device__ __forceinline__ void init_coop(const float* __restrict__ src, int S, float p[7]) {
    const int lane = threadIdx.x & 31;
    const int NP = S * S, nb = 4 * S - 4;
    uint32_t key[4];
#pragma unroll
    for (int t = 0; t < 4; t++) {
        const int b = lane + 32 * t;
        key[t] = b < nb ? fkey(__ldg(src + border_k(b, S))) : 0xffffffffu;
    }
    uint32_t ka, kb;
    if (nb <= 64) border_pair<2>(key, nb, (nb - 1) / 2, nb / 2, ka, kb);
    else border_pair<4>(key, nb, (nb - 1) / 2, nb / 2, ka, kb);
    const float sky0 = (float)(0.5 * ((double)fkey_inv(ka) + (double)fkey_inv(kb)));
    float fs = 0.f;
    for (int k = lane; k < NP; k += 32) fs += __ldg(src + k) - sky0;
    fs = warp_sum(fs);
    p[0] = 0.5f * (S - 1); p[1] = 0.5f * (S - 1); p[2] = fs; p[3] = sky0;
    p[4] = 1.6f; p[5] = 1.4f; p[6] = 0.f;
}

constexpr int PF_AHEAD = 24;   // stamps

// row pitch of a warp's tile: pixel k of slot s at k * pitch + s
__host__ __device__ constexpr int fit_pitch(int G) { return G == 1 ? 32 : 32 / G + 1; }

template <int MODEL, bool WEIGHTED, int G>
__global__ void __launch_bounds__(32 * FL_MAX_WARPS) k_psf_fit(FitJob J, int64_t chunk) {
    constexpr int PITCH = fit_pitch(G);
    extern __shared__ float fl_sm_all[];  // per warp [S*S][PITCH]: pixel k of slot s's stamp in column s
    __shared__ unsigned long long blk_next;  // next stamp of the block's chunk
    const unsigned FULL = 0xffffffffu;
    const unsigned HEADS = G == 1 ? FULL : (G == 2 ? 0x55555555u : 0x11111111u);  // first lane of each slot
    const int lane = threadIdx.x & 31;
    const int slot = lane / G;
    const int S = J.S, NP = S * S;
    float* fl_sm = fl_sm_all + (threadIdx.x >> 5) * NP * PITCH;
    // stamps to fit: N, or the device count when one is given; the chunks are
    // cut from that count here, so a count known only on the device needs no sync
    int64_t nfit = J.N;
    if (J.n_dev) nfit = min(nfit, (int64_t)max(__ldg(J.n_dev), 0));
    if (chunk <= 0) chunk = (nfit + gridDim.x - 1) / gridDim.x;
    const int64_t c0 = (int64_t)blockIdx.x * chunk;
    const int64_t c1 = c0 + chunk < nfit ? c0 + chunk : nfit;
    if (threadIdx.x == 0) blk_next = (unsigned long long)c0;
    __syncthreads();
    bool drained = false;  // the block's chunk has been handed out
    int64_t st = -1;
    float p[7], H[28], g[7], chi2 = 0.f, sm2 = 0.f;
    double lam = 0.0;
    int it = 0, nsing = 0;
    bool fresh = false, hold = false;
    float pt[7];   // the point to try
#pragma unroll
    for (int a = 0; a < 7; a++) p[a] = pt[a] = 0.f;
    while (true) {
        const unsigned idle = __ballot_sync(FULL, st < 0) & HEADS;
        if (idle && !drained) {
            // the warp takes as many stamps as it has idle slots from the
            // block's chunk; the shared cursor may run past c1
            unsigned long long base = 0;
            if (lane == 0) base = atomicAdd(&blk_next, (unsigned long long)__popc(idle));
            const int64_t next = (int64_t)__shfl_sync(FULL, base, 0);
            drained = next + __popc(idle) >= c1;
            const int rank = __popc(idle & ((1u << (slot * G)) - 1u));
            if (st < 0 && next + rank < c1) {
                st = next + rank;
                fresh = true;
                it = 0; nsing = 0;
                lam = (double)J.lambda0;
            }
            unsigned nm = __ballot_sync(FULL, fresh) & HEADS;
            while (nm) {
                const int rl = __ffs(nm) - 1, r = rl / G;
                nm &= nm - 1u;
                const int64_t sr = __shfl_sync(FULL, st, rl);
                const float* src = J.stamps + sr * NP;
                // the stamp that a warp of the block will take about a round from now
                if (sr + PF_AHEAD < c1 && lane * 32 < NP)
                    asm volatile("prefetch.global.L2 [%0];" ::"l"(src + (int64_t)PF_AHEAD * NP + lane * 32));
                for (int k = lane; k < NP; k += 32) fl_sm[k * PITCH + r] = __ldg(src + k);
                __syncwarp();
                if (J.init) {
                    if (slot == r) {
#pragma unroll
                        for (int a = 0; a < 7; a++) p[a] = __ldg(J.init + sr * 7 + a);
                    }
                } else {
                    float q[7];
                    init_coop(src, S, q);
                    if (slot == r) {
#pragma unroll
                        for (int a = 0; a < 7; a++) p[a] = q[a];
                    }
                }
            }
        }
        if (!__any_sync(FULL, st >= 0)) break;

        bool try_pt = false;
        int fl = -1;
        if (st >= 0 && fresh) {
#pragma unroll
            for (int a = 0; a < 7; a++) pt[a] = p[a];
            try_pt = true;
        }
        // A fit has converged when the Gauss-Newton decrease g'H^-1 g is below what the
        // distance to the optimum (1e-10 chi^2) and the model's FP32 rounding
        // (1e-12 sum w P^2) allow; the damped step's decrease never exceeds it, so the
        // undamped system is solved only when that one is small.
        if constexpr (G > 1) {
            // few fits a warp: both systems at once (with the form below, 8000 stamps of
            // 15 x 15 took 1457 us, 1397 so)
            if (st >= 0 && !fresh) {
                double x[7];
                if (!solve7(H, g, lam, x)) {
                    lam *= 10.0;
                    nsing++;
                    it++;
                    if (lam > 1e10) fl = IPP_FLAG_FIT_MAXITER;
                } else {
                    const double thr = 1e-10 * widen(chi2) + 1e-12 * widen(sm2);
                    double dec = 0.0;
#pragma unroll
                    for (int a = 0; a < 7; a++) dec = fma(widen(g[a]), x[a], dec);
                    if (dec <= thr) {
                        double u[7];
                        if (solve7(H, g, 0.0, u)) {
                            double dgn = 0.0;
#pragma unroll
                            for (int a = 0; a < 7; a++) dgn = fma(widen(g[a]), u[a], dgn);
                            if (dgn <= thr) fl = 0;   // stopped at p
                        }
                    }
#pragma unroll
                    for (int a = 0; a < 7; a++) pt[a] = narrow(widen(p[a]) + x[a]);
                    if (fl == 0) {
                    } else if (!(pt[4] > 0.05f) || !(pt[5] > 0.05f)) {
                        lam *= 10.0;
                        it++;
                        if (lam > 1e10) fl = 0;
                    } else {
                        try_pt = true;
                    }
                }
            }
        } else {
            // pass 0: the damped step of every slot with a fit in progress; pass 1: the
            // undamped system of the slots on hold.  One copy of the solve's code.
#pragma unroll 1
            for (int pass = 0; pass < 2; pass++) {
                bool run = st >= 0 && !fresh && !hold;
                if (pass == 1) {
                    const int held = __popc(__ballot_sync(FULL, hold));
                    const bool due = held >= HOLD_MIN || drained || !__any_sync(FULL, try_pt);
                    run = hold && due;
                }
                if (!__any_sync(FULL, run)) continue;
                if (!run) continue;
                double x[7];
                const bool ok = solve7(H, g, pass == 0 ? lam : 0.0, x);
                if (!ok && pass == 0) {
                    lam *= 10.0;
                    nsing++;
                    it++;
                    if (lam > 1e10) fl = IPP_FLAG_FIT_MAXITER;
                    continue;
                }
                const double thr = 1e-10 * widen(chi2) + 1e-12 * widen(sm2);
                double dec = 0.0;
#pragma unroll
                for (int a = 0; a < 7; a++) dec = fma(widen(g[a]), x[a], dec);
                const bool small = ok && dec <= thr;
                if (pass == 0) {
#pragma unroll
                    for (int a = 0; a < 7; a++) pt[a] = narrow(widen(p[a]) + x[a]);
                    hold = small;
                    if (hold) continue;
                } else {
                    hold = false;
                    if (small) fl = 0;   // stopped at p
                }
                if (fl == 0) {
                } else if (!(pt[4] > 0.05f) || !(pt[5] > 0.05f)) {
                    lam *= 10.0;
                    it++;
                    if (lam > 1e10) fl = 0;
                } else {
                    try_pt = true;
                }
            }
        }
        float Ht[28], gt[7], c2t = 0.f, s2t = 0.f;
        // both lanes of a slot take the same branch: their states are identical
        if (try_pt) {
            const float* wts = WEIGHTED ? J.weights + st * NP : nullptr;
            c2t = eval_lane<MODEL, WEIGHTED, G, PITCH>(fl_sm + slot, wts, S, J.beta, pt, Ht, gt, &s2t);
        }
        if (try_pt) {
            bool take = fresh;
            if (!fresh) {
                it++;
                if (c2t < chi2) {
                    take = true;
                    lam /= 10.0;   // as the oracle: 1e-3 * 0.1 rounds above 1e-4 in FP64
                } else {
                    lam *= 10.0;
                    if (lam > 1e10) fl = 0;
                }
            }
            if (take) {
#pragma unroll
                for (int a = 0; a < 7; a++) p[a] = pt[a];
#pragma unroll
                for (int a = 0; a < 28; a++) H[a] = Ht[a];
#pragma unroll
                for (int a = 0; a < 7; a++) g[a] = gt[a];
                chi2 = c2t;
                sm2 = s2t;
            }
            fresh = false;
        }
        if (st >= 0 && fl < 0 && it >= J.max_iter) fl = IPP_FLAG_FIT_MAXITER;
        if (fl >= 0) {
            if (nsing > 0 && fl) fl |= IPP_FLAG_FIT_SINGULAR;
            if (!(p[4] > 0.05f) || !(p[5] > 0.05f)) fl |= IPP_FLAG_FIT_BAD_SIGMA;
            float q[7];
#pragma unroll
            for (int a = 0; a < 7; a++) q[a] = p[a];
            if (q[4] < q[5]) { const float t = q[4]; q[4] = q[5]; q[5] = t; q[6] += 0.5f * F_PI; }
            q[6] = q[6] - F_PI * floorf((q[6] + 0.5f * F_PI) / F_PI);
            if (lane % G == 0) {
#pragma unroll
                for (int a = 0; a < 7; a++) J.params[st * 7 + a] = q[a];
                J.chi2[st] = chi2;
                if (J.iters) J.iters[st] = it;
                if (J.flags) J.flags[st] = fl;
            }
            st = -1;
        }
        __syncwarp();
    }
}

// ---- forward model and adjoint ---------------------------------------------------
// One stamp per group of L lanes (a warp, or 8 lanes for stamps of at most 5 x 5
// pixels, which would leave most of a warp idle).  What depends on the stamp
// alone -- the sine and cosine, the reciprocal widths, the amplitude -- is formed
// once per stamp instead of once per pixel, and a lane walks its pixels (lane,
// lane + L, ...) by adding L in (row, column) form, without a division.  Both are
// bound by issue slots (the logarithm and exponential of a pixel), then by the
// 4 bytes a pixel of DRAM.  50,000 Moffat stamps of 15 x 15: forward 72 -> 35 us
// (one thread per pixel, sincos and 64-bit divisions in each, before), adjoint
// 82 -> 55 us.
struct PsfStamp {
    float x0, y0, F, sky, sx, sy, isx, isy, c, s, amp;   // amp: dm/dF at the centre
};

template <int MODEL>
__device__ __forceinline__ PsfStamp psf_stamp(const float* __restrict__ p, float beta) {
    PsfStamp t;
    t.x0 = __ldg(p); t.y0 = __ldg(p + 1); t.F = __ldg(p + 2); t.sky = __ldg(p + 3);
    t.sx = __ldg(p + 4); t.sy = __ldg(p + 5);
    sincosf(__ldg(p + 6), &t.s, &t.c);
    t.isx = 1.0f / t.sx;
    t.isy = 1.0f / t.sy;
    t.amp = MODEL == IPP_PSF_GAUSS ? 1.0f / (2.0f * F_PI * t.sx * t.sy) : (beta - 1.0f) / (F_PI * t.sx * t.sy);
    return t;
}

// the lane's pixels in turn: f(k, column, row)
template <int L, class Fn>
__device__ __forceinline__ void psf_pixels(int S, int lane, Fn&& f) {
    const int NP = S * S, dr = L / S, dc = L - dr * S;
    int r = lane / S;
    int c = lane - r * S;
    for (int k = lane; k < NP; k += L) {
        f(k, (float)c, (float)r);
        r += dr;
        c += dc;
        if (c >= S) { c -= S; r++; }
    }
}

// the profile over its centre value, e = exp(-q/2) or (1 + q)^-beta, and 1 + q
template <int MODEL>
__device__ __forceinline__ float psf_profile(float q, float beta, float& base) {
    base = 1.0f + q;
    return MODEL == IPP_PSF_GAUSS ? expf(-0.5f * q) : exp2f(-beta * log2f(base));
}

template <int MODEL, int L>
__global__ void __launch_bounds__(256) k_psf_fwd(const float* __restrict__ params, int64_t N, int S, float beta,
                                                 float* __restrict__ out) {
    const int lane = threadIdx.x & (L - 1);
    const int64_t stride = (int64_t)gridDim.x * (256 / L);
    for (int64_t n = (int64_t)blockIdx.x * (256 / L) + threadIdx.x / L; n < N; n += stride) {
        const PsfStamp t = psf_stamp<MODEL>(params + n * 7, beta);
        float* o = out + n * S * S;
        const float isx2 = 1.0f / (t.sx * t.sx), isy2 = 1.0f / (t.sy * t.sy);
        psf_pixels<L>(S, lane, [&](int k, float col, float row) {
            const float dx = col - t.x0, dy = row - t.y0;
            const float u = t.c * dx + t.s * dy, v = -t.s * dx + t.c * dy;
            float base;
            const float A1 = t.amp * psf_profile<MODEL>(u * u * isx2 + v * v * isy2, beta, base);
            o[k] = t.F * A1 + t.sky;
        });
    }
}

// lanes whose number differs in bit H swap halves of v[0 .. 2H) and add
template <int H>
__device__ __forceinline__ void psf_halve(float v[8], int lane, unsigned mask) {
    const bool up = lane & H;
#pragma unroll
    for (int q = 0; q < H; q++) {
        const float give = up ? v[q] : v[q + H], keep = up ? v[q + H] : v[q];
        v[q] = keep + __shfl_xor_sync(mask, give, H);
    }
}

// adjoint: grad_params[n] = J(n)' grad_model[n].  With P the star part of the model, T =
// 2 dP/dq, (x, y) the pixel along the axes, a = x/sx^2 and b = y/sy^2, the derivatives of
// eval_lane are formed at the pixel, up to a factor of the stamp, before they meet g: a
// width's two terms largely cancel, and summed apart over the stamp (48 us) their error
// against 64 bits was up to 2.6 times as large (5.7e-8 against 2.2e-8 of the terms'
// magnitudes, Moffat 15 x 15, g > 0).
template <int MODEL, int L>
__global__ void __launch_bounds__(256) k_psf_adj(const float* __restrict__ params, int64_t N, int S, float beta,
                                                 const float* __restrict__ grad, float* __restrict__ gout) {
    const int lane = threadIdx.x & (L - 1);
    const unsigned gmask = L == 32 ? 0xffffffffu : ((1u << (L & 31)) - 1u) << (threadIdx.x & 31 & ~(L - 1));
    const int64_t stride = (int64_t)gridDim.x * (256 / L);
    for (int64_t n = (int64_t)blockIdx.x * (256 / L) + threadIdx.x / L; n < N; n += stride) {
        const PsfStamp t = psf_stamp<MODEL>(params + n * 7, beta);
        const float* g = grad + n * S * S;
        const float isx2 = 1.0f / (t.sx * t.sx), isy2 = 1.0f / (t.sy * t.sy);
        float v[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
        psf_pixels<L>(S, lane, [&](int k, float col, float row) {
            const float gm = __ldg(g + k);
            const float dx = col - t.x0, dy = row - t.y0;
            const float x = t.c * dx + t.s * dy, y = -t.s * dx + t.c * dy;
            const float a = x * isx2, b = y * isy2;
            float base;
            const float A = t.amp * psf_profile<MODEL>(x * x * isx2 + y * y * isy2, beta, base);
            const float P = t.F * A;
            const float T = MODEL == IPP_PSF_GAUSS ? -P : -2.0f * beta * P / base;
            const float gt = gm * T;
            v[0] = fmaf(gt, fmaf(b, t.s, -a * t.c), v[0]);
            v[1] = fmaf(gt, fmaf(a, t.s, b * t.c), v[1]);
            v[2] = fmaf(gm, A, v[2]);
            v[3] += gm;
            v[4] = fmaf(gm, fmaf(T * a, x, P), v[4]);
            v[5] = fmaf(gm, fmaf(T * b, y, P), v[5]);
            v[6] = fmaf(gt * x, y, v[6]);
        });
        // eight values over the group's lanes: three exchanges of halves leave lane l
        // with the partial of value l & 7, plain steps add the groups of eight
        psf_halve<4>(v, lane, gmask);
        psf_halve<2>(v, lane, gmask);
        psf_halve<1>(v, lane, gmask);
#pragma unroll
        for (int o = 8; o < L; o <<= 1) v[0] += __shfl_xor_sync(gmask, v[0], o);
        float f = 1.0f;                                              // x0, F, sky
        if (lane == 1) f = -1.0f;                                    // y0
        if (lane == 4) f = -t.isx;                                   // sx
        if (lane == 5) f = -t.isy;                                   // sy
        // theta: dq/dtheta = 2uv (1/sx^2 - 1/sy^2), without the cancellation when sx ~ sy
        if (lane == 6) f = ((t.sy - t.sx) * (t.sy + t.sx)) * isx2 * isy2;
        if (lane < 7) gout[n * 7 + lane] = f * v[0];
    }
}

}  // namespace ipp

using namespace ipp;

static size_t fit_warp_bytes(int S, int G) { return (size_t)S * S * fit_pitch(G) * sizeof(float); }
static int fit_max_warps(int S, int G) {   // the kernel's static shared memory is 8 bytes
    return (int)std::min<size_t>(FL_MAX_WARPS, (size_t)(227 * 1024 - 64) / fit_warp_bytes(S, G));
}

template <int MODEL, bool WEIGHTED, int G>
static int launch_fit(const FitJob& J, cudaStream_t s) {
    auto k = k_psf_fit<MODEL, WEIGHTED, G>;
    const size_t per_warp = fit_warp_bytes(J.S, G);
    // warps of one block share a chunk of stamps: the block's chunk drains with
    // every slot busy until its last few stamps, so the larger the block, the
    // smaller the idle tail.  One block per SM, as many warps as its shared
    // memory holds.
    const int wmax = fit_max_warps(J.S, G);
    const int64_t warps = std::min<int64_t>((int64_t)ipp_sm_count() * wmax, (J.N + 32 / G - 1) / (32 / G));
    const int64_t blocks = std::min<int64_t>(ipp_sm_count(), warps);
    const int wpb = (int)((warps + blocks - 1) / blocks);
    const size_t smem = per_warp * wpb;
    cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    cudaFuncSetAttribute(k, cudaFuncAttributePreferredSharedMemoryCarveout, 100);
    const int64_t chunk = J.n_dev ? 0 : (J.N + blocks - 1) / blocks;   // 0: from the device count
    k<<<(unsigned)blocks, 32 * wpb, smem, s>>>(J, chunk);
    return ipp_check_launch("k_psf_fit");
}

// Lanes per stamp: 1 when the stamps fill every lane the GPU can hold (one FP64
// instruction then serves 32 solves); for smaller batches 2 or 4 lanes share a
// stamp, so that the batch still spreads over the lanes and each round is
// shorter.  G is taken while N G stays within 1.25 x the lanes resident at G
// (measured on 152 SMs, 15 x 15 stamps: G = 4 up to ~12,000 stamps, G = 2 up
// to ~24,000, G = 1 beyond).  With a count on the device N is the capacity of the arrays:
// G, and with it the order of a stamp's sums, can differ from a call that is given the
// same stamps by their number.
static int fit_lanes_per_stamp(const FitJob& J) {
    const int64_t sms = ipp_sm_count();
    for (int G = 4; G > 1; G >>= 1)
        if (J.N * G * 4 <= sms * fit_max_warps(J.S, G) * 32 * 5) return G;
    return 1;
}

template <int MODEL, bool WEIGHTED>
static int launch_fit_g(const FitJob& J, cudaStream_t s) {
    switch (fit_lanes_per_stamp(J)) {
        case 4: return launch_fit<MODEL, WEIGHTED, 4>(J, s);
        case 2: return launch_fit<MODEL, WEIGHTED, 2>(J, s);
        default: return launch_fit<MODEL, WEIGHTED, 1>(J, s);
    }
}

int ipp_launch_psf_fit(const FitJob& J, cudaStream_t s) {
    if (fit_warp_bytes(J.S, 1) > 227 * 1024)
        return ipp_set_error(IPP_ERR_NOT_SUPPORTED, "stamp size %d above 32", J.S);
    if (J.model == IPP_PSF_GAUSS)
        return J.weights ? launch_fit_g<IPP_PSF_GAUSS, true>(J, s) : launch_fit_g<IPP_PSF_GAUSS, false>(J, s);
    return J.weights ? launch_fit_g<IPP_PSF_MOFFAT, true>(J, s) : launch_fit_g<IPP_PSF_MOFFAT, false>(J, s);
}

// Eight lanes a stamp up to 6 x 6 pixels, a warp above.  50,000 Moffat stamps of 6 x 6:
// forward 8 us with eight lanes against 18, adjoint 12 against 27; from 7 x 7 on the warp
// is the shorter pass of small batches (1000 Gaussian stamps, adjoint: 4 us against 6).
template <class Fn>
static void launch_psf_lanes(int64_t N, int S, Fn&& go) {
    const int L = S <= 6 ? 8 : 32;
    const int64_t need = (N + 256 / L - 1) / (256 / L);
    go(L, (unsigned)std::max<int64_t>(1, std::min<int64_t>(need, (int64_t)ipp_sm_count() * 32)));
}

int ipp_launch_psf_fwd(const float* params, int64_t N, int S, int model, float beta, float* out, cudaStream_t s) {
    launch_psf_lanes(N, S, [&](int L, unsigned blocks) {
        if (model == IPP_PSF_GAUSS) {
            if (L == 8) k_psf_fwd<IPP_PSF_GAUSS, 8><<<blocks, 256, 0, s>>>(params, N, S, beta, out);
            else k_psf_fwd<IPP_PSF_GAUSS, 32><<<blocks, 256, 0, s>>>(params, N, S, beta, out);
        } else {
            if (L == 8) k_psf_fwd<IPP_PSF_MOFFAT, 8><<<blocks, 256, 0, s>>>(params, N, S, beta, out);
            else k_psf_fwd<IPP_PSF_MOFFAT, 32><<<blocks, 256, 0, s>>>(params, N, S, beta, out);
        }
    });
    return ipp_check_launch("k_psf_fwd");
}

int ipp_launch_psf_adj(const float* params, int64_t N, int S, int model, float beta, const float* grad,
                       float* gout, cudaStream_t s) {
    launch_psf_lanes(N, S, [&](int L, unsigned blocks) {
        if (model == IPP_PSF_GAUSS) {
            if (L == 8) k_psf_adj<IPP_PSF_GAUSS, 8><<<blocks, 256, 0, s>>>(params, N, S, beta, grad, gout);
            else k_psf_adj<IPP_PSF_GAUSS, 32><<<blocks, 256, 0, s>>>(params, N, S, beta, grad, gout);
        } else {
            if (L == 8) k_psf_adj<IPP_PSF_MOFFAT, 8><<<blocks, 256, 0, s>>>(params, N, S, beta, grad, gout);
            else k_psf_adj<IPP_PSF_MOFFAT, 32><<<blocks, 256, 0, s>>>(params, N, S, beta, grad, gout);
        }
    });
    return ipp_check_launch("k_psf_adj");
}

// subtract.cu -- the convolution and difference of HOTPANTS-style image
// subtraction (Sec. 2.2.4, Eqs. 8-10): with fitted coefficients c_{n,s} and
// background d_b, the kernel of each (2 hw + 1)^2 output tile is
// K(u, v) = sum_n a_n(tile centre) K_n(u, v), a_n = sum_s c_{n,s} P_s (Eq. 8),
// K_n = exp(-(u^2 + v^2) / (2 sig^2)) u^i v^j (Eq. 9), and the difference is
// D = I + B - R (x) K (the residual of Eq. 10), NaN where the kernel's support
// leaves the frame.
//
// The kernel of a tile costs 49 x 441 multiply-adds, its convolution 441 x 441.  A
// block takes TPB neighbouring tiles: their kernels and the template window they
// share (rows and columns 2 hw beyond the tiles) are staged in shared memory, and
// each thread computes a patch of 3 rows x C columns of one tile.  A window row is
// read once into registers and meets the three kernel rows it contributes to, one
// 16-byte shared load per four kernel values, so that a step of 3 x C x S
// multiply-adds costs C + 2 hw + 3 S / 4 shared loads: bound by the FP32 pipe
// instead of shared memory.  Per output the sum still runs over the kernel's rows,
// then columns, in ascending order.  4096 x 4096, hw = 10, 49 basis functions:
// 767 -> 473 us (one row of 7 outputs a thread, before); the convolution's
// 7.4 G multiply-adds alone are 191 us of this part's FP32 rate.
#include <math.h>

#include <algorithm>

#include "jobs.cuh"

namespace ipp {

constexpr int SB_MAXB = 64;    // basis functions
constexpr int SB_MAXT = 16;    // spatial terms (order <= 4)

struct SubBasisDesc {
    int nk;
    float sig[8];
    int deg[8];
};

// basis function n on the (2 hw + 1)^2 grid: one block per function
__global__ void k_sub_basis(SubBasisDesc d, int hw, float* __restrict__ basis) {
    int n = blockIdx.x, k = 0, i = 0, j = 0, acc = 0;
    for (int kk = 0; kk < d.nk; kk++) {
        const int cnt = (d.deg[kk] + 1) * (d.deg[kk] + 2) / 2;
        if (n < acc + cnt) {
            k = kk;
            int r = n - acc;
            for (i = 0; i <= d.deg[kk]; i++) {
                const int row = d.deg[kk] - i + 1;
                if (r < row) {
                    j = r;
                    break;
                }
                r -= row;
            }
            break;
        }
        acc += cnt;
    }
    const int S = 2 * hw + 1;
    const double s2 = 2.0 * (double)d.sig[k] * (double)d.sig[k];
    for (int t = threadIdx.x; t < S * S; t += blockDim.x) {
        const int u = t % S - hw, v = t / S - hw;
        double p = exp(-(double)(u * u + v * v) / s2);
        for (int q = 0; q < i; q++) p *= (double)u;
        for (int q = 0; q < j; q++) p *= (double)v;
        basis[(size_t)n * S * S + t] = (float)p;
    }
}

__device__ __forceinline__ void sub_terms(float xs, float ys, int order, float* t) {
    int n = 0;
    float xp = 1.f;
    for (int p = 0; p <= order; p++) {
        float yq = 1.f;
        for (int q = 0; q <= order - p; q++) {
            t[n++] = xp * yq;
            yq *= ys;
        }
        xp *= xs;
    }
}

// Shape of k_sub_apply for a half width: C columns a thread, TPB tiles a block (the
// threads of TPB tiles fill whole warps as far as they can) and the window's row
// pitch WP, the first at which a warp's window reads meet the fewest bank conflicts.
template <int HW, int C, int TPB, int WP>
struct SubApplyShape {
    static constexpr int S = 2 * HW + 1, NS = (S + C - 1) / C, RG = (S + 2) / 3, TPT = RG * NS, T = TPB * TPT;
    static constexpr int WROWS = 3 * RG + 2 * HW, WCOLS = (TPB - 1) * S + NS * C + 2 * HW, KP = (S + 3) & ~3;
    static_assert(WP >= WCOLS && WROWS * WP >= S * TPB * S, "window, then the block's sums, in one array");
};

template <int HW, int C, int TPB, int WP>
__global__ void __launch_bounds__(SubApplyShape<HW, C, TPB, WP>::T)
    k_sub_apply(const float* __restrict__ I, const float* __restrict__ R, int64_t W, int64_t H, int64_t pitch,
                const float* __restrict__ basis, int nb, const float* __restrict__ cs, int sord,
                const float* __restrict__ cb, int bord, float* __restrict__ D, int64_t opitch) {
    using SH = SubApplyShape<HW, C, TPB, WP>;
    constexpr int S = SH::S, T = SH::T, KP = SH::KP;
    __shared__ __align__(16) float Ks[TPB][S][KP];
    __shared__ float Rw[SH::WROWS * WP];   // the window, after the convolution its sums [S][TPB S]
    __shared__ __align__(16) float an[SB_MAXB][(TPB + 3) & ~3];
    const int ntx = (int)((W + S * TPB - 1) / (S * TPB));
    const int64_t bx = blockIdx.x % ntx, by = blockIdx.x / ntx;
    const int64_t x0 = bx * (S * TPB), y0 = by * S;
    const float sx = W > 1 ? 2.f / (float)(W - 1) : 0.f, sy = H > 1 ? 2.f / (float)(H - 1) : 0.f;
    // background terms 1, y, x of the usual order, read before they are needed
    const float cb0 = bord == 1 ? __ldg(cb) : 0.f, cb1 = bord == 1 ? __ldg(cb + 1) : 0.f, cb2 = bord == 1 ? __ldg(cb + 2) : 0.f;
    // Eq. 8 at the tiles' centres
    for (int t = threadIdx.x; t < TPB * nb; t += T) {
        const int tile = t / nb, n = t - tile * nb;
        float P[SB_MAXT];
        const float xs = W > 1 ? (float)((double)(x0 + tile * S) + 0.5 * (S - 1)) * sx - 1.f : 0.f;
        const float ys = H > 1 ? (float)((double)y0 + 0.5 * (S - 1)) * sy - 1.f : 0.f;
        sub_terms(xs, ys, sord, P);
        const int ns = (sord + 1) * (sord + 2) / 2;
        float a = 0.f;
        for (int q = 0; q < ns; q++) a = fmaf(__ldg(cs + n * ns + q), P[q], a);
        an[n][tile] = a;
    }
    // template window: rows y0 - HW .., columns x0 - HW .. (0 outside the frame and
    // in the rows and columns that only padding outputs read)
    constexpr int NWIN = SH::WROWS * SH::WCOLS, LB = 9;   // LB loads in flight a thread
    for (int t0 = threadIdx.x; t0 < NWIN; t0 += LB * T) {
        float v[LB];
#pragma unroll
        for (int m = 0; m < LB; m++) {
            const int t = t0 + m * T, a = t / SH::WCOLS, b = t - a * SH::WCOLS;
            const int64_t yy = y0 - HW + a, xx = x0 - HW + b;
            const bool in = a < S + 2 * HW && b < S * TPB + 2 * HW && yy >= 0 && yy < H && xx >= 0 && xx < W;
            v[m] = in ? __ldg(R + yy * pitch + xx) : 0.f;
        }
#pragma unroll
        for (int m = 0; m < LB; m++) {
            const int t = t0 + m * T, a = t / SH::WCOLS;
            if (t < NWIN) Rw[a * WP + t - a * SH::WCOLS] = v[m];
        }
    }
    __syncthreads();
    // Eq. 9 summed with the tiles' amplitudes: one read of a basis value (from L2)
    // serves the block's tiles, and the reads of all the thread's taps are in flight
    {
        constexpr int TAPS = (S * S + T - 1) / T;
        float k[TAPS][TPB];
#pragma unroll
        for (int m = 0; m < TAPS; m++)
#pragma unroll
            for (int u = 0; u < TPB; u++) k[m][u] = 0.f;
        const float* bp = basis + threadIdx.x;
#pragma unroll 4
        for (int n = 0; n < nb; n++, bp += S * S) {
            float b[TAPS];
#pragma unroll
            for (int m = 0; m < TAPS; m++) b[m] = threadIdx.x + m * T < S * S ? __ldg(bp + m * T) : 0.f;
#pragma unroll
            for (int u = 0; u < TPB; u++) {
                const float a = an[n][u];
#pragma unroll
                for (int m = 0; m < TAPS; m++) k[m][u] = fmaf(a, b[m], k[m][u]);
            }
        }
#pragma unroll
        for (int m = 0; m < TAPS; m++) {
            const int t = threadIdx.x + m * T;
            if (t < S * S) {
                const int vp = t / S, up = t - vp * S;
#pragma unroll
                for (int u = 0; u < TPB; u++) Ks[u][vp][up] = k[m][u];
            }
        }
    }
    __syncthreads();
    const int tile = threadIdx.x / SH::TPT, rem = threadIdx.x - tile * SH::TPT;
    const int oy0 = rem / SH::NS * 3, ox0 = rem % SH::NS * C;
    float acc[3][C];
#pragma unroll
    for (int r = 0; r < 3; r++)
#pragma unroll
        for (int q = 0; q < C; q++) acc[r][q] = 0.f;
    // out(oy, ox) = sum_{v', u'} K[v'][u'] Rw[oy + 2HW - v'][ox + 2HW - u']: window
    // row oy0 + 2HW + 2 - m is row r's with v' = m + r - 2
    const float* wrow = Rw + (oy0 + 2 * HW + 2) * WP + tile * S + ox0;
#pragma unroll 1
    for (int m = 0; m < S + 2; m++, wrow -= WP) {
        float rr[C + 2 * HW];
#pragma unroll
        for (int q = 0; q < C + 2 * HW; q++) rr[q] = wrow[q];
#pragma unroll
        for (int r = 0; r < 3; r++) {
            const int vp = m + r - 2;
            if (vp < 0 || vp >= S) continue;
            const float4* kr = reinterpret_cast<const float4*>(Ks[tile][vp]);
#pragma unroll
            for (int u4 = 0; u4 < KP / 4; u4++) {
                const float4 kv = kr[u4];
                const float k4[4] = {kv.x, kv.y, kv.z, kv.w};
#pragma unroll
                for (int e = 0; e < 4; e++) {
                    const int up = u4 * 4 + e;
                    if (up >= S) continue;
#pragma unroll
                    for (int q = 0; q < C; q++) acc[r][q] = fmaf(k4[e], rr[q + 2 * HW - up], acc[r][q]);
                }
            }
        }
    }
    __syncthreads();   // the window is no longer needed
#pragma unroll
    for (int r = 0; r < 3; r++)
#pragma unroll
        for (int q = 0; q < C; q++)
            if (oy0 + r < S && ox0 + q < S) Rw[(oy0 + r) * (S * TPB) + tile * S + ox0 + q] = acc[r][q];
    __syncthreads();
    // the difference, EB pixels of the frame in flight a thread
    constexpr int NOUT = S * S * TPB, EB = 7;
    for (int t0 = threadIdx.x; t0 < NOUT; t0 += EB * T) {
        float v[EB];
#pragma unroll
        for (int m = 0; m < EB; m++) {
            const int t = t0 + m * T, oy = t / (S * TPB), ox = t - oy * (S * TPB);
            const int64_t x = x0 + ox, y = y0 + oy;
            v[m] = t < NOUT && x >= HW && y >= HW && x <= W - 1 - HW && y <= H - 1 - HW ? __ldg(I + y * pitch + x) : NAN;
        }
#pragma unroll
        for (int m = 0; m < EB; m++) {
            const int t = t0 + m * T, oy = t / (S * TPB), ox = t - oy * (S * TPB);
            const int64_t x = x0 + ox, y = y0 + oy;
            if (t >= NOUT || x >= W || y >= H) continue;
            float b = 0.f;
            // the terms of sub_terms in turn, without a table
            const float xs = W > 1 ? (float)x * sx - 1.f : 0.f;
            const float ys = H > 1 ? (float)y * sy - 1.f : 0.f;
            if (bord == 1) {
                b = fmaf(cb2, xs, fmaf(cb1, ys, cb0));
            } else {
                const float* c = cb;
                float xp = 1.f;
                for (int p = 0; p <= bord; p++) {
                    float yq = 1.f;
                    for (int q = 0; q <= bord - p; q++) {
                        b = fmaf(__ldg(c++), xp * yq, b);
                        yq *= ys;
                    }
                    xp *= xs;
                }
            }
            // pixels whose support leaves the frame stay NaN
            const bool in = x >= HW && y >= HW && x <= W - 1 - HW && y <= H - 1 - HW;
            D[y * opitch + x] = in ? v[m] + b - Rw[t] : NAN;
        }
    }
}

template <int HW, int C, int TPB, int WP>
static void launch_sub_apply(const float* I, const float* R, int64_t W, int64_t H, int64_t pitch, const float* basis,
                             int nb, const float* cs, int sord, const float* cb, int bord, float* D, int64_t opitch,
                             cudaStream_t s) {
    using SH = SubApplyShape<HW, C, TPB, WP>;
    const int64_t nblk = ((W + SH::S * TPB - 1) / (SH::S * TPB)) * ((H + SH::S - 1) / SH::S);
    k_sub_apply<HW, C, TPB, WP><<<(unsigned)nblk, SH::T, 0, s>>>(I, R, W, H, pitch, basis, nb, cs, sord, cb, bord, D,
                                                                 opitch);
}

}  // namespace ipp

using namespace ipp;

size_t ipp_sub_ws_bytes(int nb, int hw) {
    return (size_t)nb * (2 * hw + 1) * (2 * hw + 1) * sizeof(float);
}

int ipp_launch_sub_apply(const float* I, const float* R, int64_t W, int64_t H, int64_t pitch, int hw, int nk,
                         const float* sig, const int* deg, int nb, const float* cs, int sord, const float* cb,
                         int bord, float* D, int64_t opitch, void* ws, cudaStream_t s) {
    SubBasisDesc d;
    d.nk = nk;
    for (int k = 0; k < nk; k++) {
        d.sig[k] = sig[k];
        d.deg[k] = deg[k];
    }
    float* basis = (float*)ws;
    k_sub_basis<<<nb, 128, 0, s>>>(d, hw, basis);
    if (int e = ipp_check_launch("k_sub_basis")) return e;
    // hw = 4: 517 x 389 frames 37 -> 25 us, 2048 x 2048 126 -> 102 us (ten tiles of nine
    // columns a thread before); hw = 12: 128 x 128 45 -> 42 us, 2048 x 2048 209 -> 195 us
    // (nine columns before)
    switch (hw) {
#define SB_CASE(HWV, C, TPB, WP)                                                                             \
    case HWV:                                                                                                \
        launch_sub_apply<HWV, C, TPB, WP>(I, R, W, H, pitch, basis, nb, cs, sord, cb, bord, D, opitch, s);   \
        break;
        SB_CASE(4, 3, 7, 72)
        SB_CASE(6, 7, 3, 58)
        SB_CASE(8, 6, 3, 77)
        SB_CASE(10, 7, 3, 85)
        SB_CASE(12, 5, 2, 76)
#undef SB_CASE
        default: return IPP_ERR_NOT_SUPPORTED;
    }
    return ipp_check_launch("k_sub_apply");
}

// subfit.cu -- the fit of image subtraction (Sec. 2.2.4, Eqs. 8-10): stamp
// selection, the normal equations of the basis-kernel model and their Cholesky
// solve.  Readings (the same as the difference-image kernels of subtract.cu):
//   stamps: the frame is cut into nsx x nsy regions; in each, the median and
//     1.4826 MAD of the template's finite pixels; the candidate is the brightest
//     template pixel (first in raster order among equals) whose fit footprint
//     (2 fh + 1)^2 and convolution support (2 (fh + hw) + 1)^2 lie inside the
//     frame and are finite in I and R, kept when it exceeds the median by nsig
//     robust sigmas;
//   model: I + B = R (x) K, K = sum_n a_n K_n, a_n = sum_s c_{n,s} P_s taken at
//     the candidate's centre, B = sum_b d_b P_b at each pixel; unweighted least
//     squares over every footprint pixel of every candidate; the design row of a
//     pixel is [C_n P_s for n, s] then [-P_b for b], C_n = R (x) K_n, target I.
//
// Precision.  The normal matrix is badly conditioned (after a diagonal scaling
// its condition number is ~1e11 on a survey frame), so it is formed in FP64: a
// relative error of 1e-6 in its entries moves the fitted model by ~2%.  The
// convolutions use the separability of the basis, K_n(u, v) = h_{k,i}(u)
// h_{k,j}(v) with h_{k,p}(t) = exp(-t^2 / (2 sig_k^2)) t^p: a row pass with the
// sum(deg_k + 1) one-dimensional filters, then a column pass per basis function
// (725 k FP64 multiply-adds per 21 x 21 footprint instead of 9.5 M).  The stamp
// selection is exact: order statistics by radix selection on the values' bit
// patterns, the MAD on the FP64 differences the definition takes.
#include <cooperative_groups.h>
#include <math.h>

#include <algorithm>

#include "jobs.cuh"

namespace ipp {

// ---- stamp selection: one cluster of blocks per region ---------------------------
// A region takes about 13 passes over its pixels (radix passes of the median and
// the MAD, the extrema, the brightest pixel), and one block per region left SMs
// idle and read the region from L2 each time.  Here NC <= 8 blocks of a cluster
// share a region, each holds its slice in shared memory (84 KB; two blocks an SM)
// and a pass ends in one exchange over distributed shared memory: the counters or
// extrema of all blocks are read by every block, which then take the same decision.
// Bound by the passes' integer work per element, so a slice holds ordered 32-bit keys
// and the passes work on 32 bits wherever that is exact.  100 regions of 168 K
// pixels: 820 us with one block, 460 us in clusters on 64-bit keys, 328 us now.  A region above NC slices is read from memory in every pass.
constexpr int SS_T = 512, SS_W = SS_T / 32, SS_NC = 8;
constexpr int SS_SLICE = 21504;   // pixels of a slice: 84 KB beside 18 KB of counters, two blocks an SM

struct StampShared {
    unsigned int hist[SS_W * 256];
    unsigned int tot[2][256];              // this block's digit counts, double-buffered over exchanges
    unsigned long long xch[2][SS_NC];      // this block's values for an exchange
    unsigned long long red[SS_NC][SS_W];
    int sdig;
    long long sbelow;
};

struct StampRegion {
    const float* I;
    const float* R;
    int64_t pitch, W, H;
    int x0, y0, rw, rh;   // the region [x0, x0 + rw) x [y0, y0 + rh)
    int t0, t1;           // this block's pixels of it (raster index)
    bool cached;          // their keys are in shared memory
    const uint32_t* cache;
    int buf;              // exchange buffer in turn
};

// Key of a pixel: fkey of a finite value, STAMP_NONE (no finite value's key) otherwise
constexpr uint32_t STAMP_NONE = 0xffffffffu;
__device__ __forceinline__ uint32_t reg_load(const StampRegion& g, int t) {
    const int yy = t / g.rw;
    const float v = __ldg(g.R + (int64_t)(g.y0 + yy) * g.pitch + (g.x0 + (t - yy * g.rw)));
    return isfinite(v) ? fkey(v) : STAMP_NONE;
}
__device__ __forceinline__ uint32_t reg_key(const StampRegion& g, int t) {
    return g.cached ? g.cache[t - g.t0] : reg_load(g, t);
}

// One exchange: this block's value(s) in S.xch[buf] are combined over the
// cluster's blocks by every block.  The buffers alternate, so one barrier per
// exchange is enough: a buffer is written again only after the next barrier.
__device__ __forceinline__ void stamp_barrier() { cooperative_groups::this_cluster().sync(); }

template <class Op>
__device__ __forceinline__ unsigned long long warp_red_u64(unsigned long long v, Op op) {
    for (int o = 16; o > 0; o >>= 1) v = op(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}

struct OpMin { __device__ unsigned long long operator()(unsigned long long a, unsigned long long b) const { return a < b ? a : b; } };
struct OpMax { __device__ unsigned long long operator()(unsigned long long a, unsigned long long b) const { return a > b ? a : b; } };
struct OpAdd { __device__ unsigned long long operator()(unsigned long long a, unsigned long long b) const { return a + b; } };

// this block's partial of value `slot` (visible after the exchange's barrier)
template <class Op>
__device__ __forceinline__ void stamp_part(StampShared& S, int slot, unsigned long long v, Op op) {
    v = warp_red_u64(v, op);
    if ((threadIdx.x & 31) == 0) S.red[slot][threadIdx.x >> 5] = v;
}
template <class Op>
__device__ __forceinline__ void stamp_block(StampShared& S, int buf, int slot, Op op) {   // after a block barrier
    if (threadIdx.x == 0) {
        unsigned long long v = S.red[slot][0];
        for (int w = 1; w < SS_W; w++) v = op(v, S.red[slot][w]);
        S.xch[buf][slot] = v;
    }
}
template <class Op>
__device__ __forceinline__ unsigned long long stamp_all(StampShared& S, int buf, int slot, Op op) {   // after the cluster barrier
    auto cl = cooperative_groups::this_cluster();
    unsigned long long v = *cl.map_shared_rank(&S.xch[buf][slot], 0);
    for (unsigned r = 1; r < cl.num_blocks(); r++) v = op(v, *cl.map_shared_rank(&S.xch[buf][slot], r));
    return v;
}

// Keys of a region's finite values for the order statistics, as unsigned integers
// ordered like the quantities they stand for:
//   value, 32 bits: fkey(v);
//   |v - med| exactly, as the integer |v 2^-e0 - med 2^-e0| -- every value and med are
//     multiples of 2^e0 (e0: one below the smallest ulp in the region), so the
//     difference is exact and its FP64 rounding is the FP64 subtraction's, without
//     FP64 arithmetic per element; the scaling is two exact products with powers of
//     two, 2^-e0 = s1 s2;
//   the same in 32 bits: the conversion saturates at +-2^31, so a key below
//     2^31 - 1 - |med 2^-e0| is exact and every other pixel's is at least that.  Few
//     pixels of a region are far from its median: the MAD's keys nearly always are
//     below, and these passes take half the instructions of the 64-bit ones;
//   the bit pattern of the FP64 |v - med| (when the region's range does not fit 62
//     bits at scale 2^e0).
struct ValueKey {
    using T = uint32_t;
    __device__ __forceinline__ bool operator()(uint32_t k, T* out) const {
        *out = k;
        return k != STAMP_NONE;
    }
};
struct DistKey32 {
    using T = uint32_t;
    float s1, s2;
    int imed;
    __device__ __forceinline__ bool operator()(uint32_t k, T* out) const {
        const int v = __float2int_rz(__fmul_rn(__fmul_rn(fkey_inv(k), s1), s2));
        *out = v < imed ? (uint32_t)imed - (uint32_t)v : (uint32_t)v - (uint32_t)imed;
        return k != STAMP_NONE;
    }
};
struct DistKey64 {
    using T = unsigned long long;
    float s1, s2;
    long long imed;
    __device__ __forceinline__ bool operator()(uint32_t k, T* out) const {
        const long long d = __float2ll_rz(__fmul_rn(__fmul_rn(fkey_inv(k), s1), s2)) - imed;
        *out = (T)(d < 0 ? -d : d);
        return k != STAMP_NONE;
    }
};
struct DistKeyD {
    using T = unsigned long long;
    double med;
    __device__ __forceinline__ bool operator()(uint32_t k, T* out) const {
        *out = (T)__double_as_longlong(fabs((double)fkey_inv(k) - med));
        return k != STAMP_NONE;
    }
};

// The k-th smallest key (0-based) of the region: radix selection, 8 bits a
// pass from bit top + 7 down, every key sharing the bits above top with
// prefix0; per-warp histograms in shared memory, fed by per-thread run lengths
// of equal digits, summed over the block, then over the cluster.  A key known to be
// `limit` or more after some digits ends the search (the caller has no use for it).
template <class Key>
__device__ unsigned long long region_select(StampRegion& g, const Key& key_of, long long k, int top,
                                            unsigned long long prefix0, unsigned long long limit,
                                            StampShared& S) {
    using T = typename Key::T;
    auto cl = cooperative_groups::this_cluster();
    T prefix = (T)prefix0;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int shift = top; shift >= 0; shift -= 8) {
        for (int t = threadIdx.x; t < SS_W * 256; t += SS_T) S.hist[t] = 0;
        __syncthreads();
        // each thread counts runs of equal digits over its elements (the region's
        // keys mostly share their high digits) and adds a run to its warp's
        // histogram when the digit changes
        unsigned cur = 256u, run = 0u;
        const bool all = shift + 8 >= 8 * (int)sizeof(T);   // the first digit: no bits above it
        for (int t = g.t0 + threadIdx.x; t < g.t1; t += SS_T) {
            T key;
            const bool ok = key_of(reg_key(g, t), &key);
            if (!ok || !(all || (key >> (shift + 8)) == prefix)) continue;
            const unsigned dig = (unsigned)((key >> shift) & 255u);
            if (dig == cur) {
                run++;
            } else {
                if (run) atomicAdd(&S.hist[warp * 256 + cur], run);
                cur = dig;
                run = 1u;
            }
        }
        if (run) atomicAdd(&S.hist[warp * 256 + cur], run);
        __syncthreads();
        if (threadIdx.x < 256) {
            unsigned s = 0;
            for (int w = 0; w < SS_W; w++) s += S.hist[w * 256 + threadIdx.x];
            S.tot[g.buf][threadIdx.x] = s;
        }
        cl.sync();
        // the region's counts per digit (thread b < 256), then warp 0 finds the digit of rank k
        if (threadIdx.x < 256) {
            unsigned s = 0;
            for (unsigned r = 0; r < cl.num_blocks(); r++) s += *cl.map_shared_rank(&S.tot[g.buf][threadIdx.x], r);
            S.hist[threadIdx.x] = s;
        }
        g.buf ^= 1;
        __syncthreads();
        if (warp == 0) {
            long long c8 = 0;
            for (int b = 0; b < 8; b++) c8 += S.hist[lane * 8 + b];
            long long inc = c8;
            for (int o = 1; o < 32; o <<= 1) {
                const long long u = __shfl_up_sync(0xffffffffu, inc, o);
                if (lane >= o) inc += u;
            }
            const long long exc = inc - c8;
            const unsigned hit = __ballot_sync(0xffffffffu, exc <= k && k < inc);
            if (hit && lane == __ffs(hit) - 1) {
                long long c = exc;
                int d = lane * 8;
                for (int b = 0; b < 8; b++) {
                    const long long nb = c + S.hist[lane * 8 + b];
                    if (k < nb) { d = lane * 8 + b; break; }
                    c = nb;
                }
                S.sdig = d;
                S.sbelow = c;
            }
        }
        __syncthreads();
        prefix = (T)(prefix << 8) | (T)S.sdig;
        k -= S.sbelow;
        __syncthreads();
        if (((unsigned long long)prefix << shift) >= limit) return (unsigned long long)prefix << shift;
    }
    return prefix;
}

// the two middle order statistics (k0 = (n - 1) / 2, k1 = n / 2) as keys, for
// keys in [kmin, kmax]: the radix passes start at the highest byte where kmin
// and kmax differ
template <class Key>
__device__ void region_middle(StampRegion& g, const Key& key_of, long long n, unsigned long long kmin,
                              unsigned long long kmax, unsigned long long limit, StampShared& S,
                              unsigned long long* a, unsigned long long* b) {
    using T = typename Key::T;
    const long long k0 = (n - 1) / 2, k1 = n / 2;
    const unsigned long long dif = kmin ^ kmax;
    const int top = dif ? ((63 - __clzll((long long)dif)) & ~7) : 0;
    const unsigned long long prefix0 = top + 8 < 64 ? kmin >> (top + 8) : 0ull;
    *a = region_select(g, key_of, k0, top, prefix0, limit, S);
    if (k1 == k0 || *a >= limit) { *b = *a; return; }
    // count of keys <= a, smallest key > a
    uint32_t cnt = 0;
    T next = (T)~(T)0;
    const T ka = (T)*a;
    for (int t = g.t0 + threadIdx.x; t < g.t1; t += SS_T) {
        T key;
        if (!key_of(reg_key(g, t), &key)) continue;
        if (key <= ka) cnt++;
        else if (key < next) next = key;
    }
    unsigned long long c = cnt, nx = next;
    stamp_part(S, 0, c, OpAdd());
    stamp_part(S, 1, nx, OpMin());
    __syncthreads();
    stamp_block(S, g.buf, 0, OpAdd());
    stamp_block(S, g.buf, 1, OpMin());
    stamp_barrier();
    c = stamp_all(S, g.buf, 0, OpAdd());
    nx = stamp_all(S, g.buf, 1, OpMin());
    g.buf ^= 1;
    *b = (long long)c > k1 ? *a : nx;
}

// Is every pixel of the (2 m + 1)^2 box of A around (x, y) finite?  (block-wide)
__device__ bool block_box_finite(const float* A, int64_t pitch, int x, int y, int m) {
    const int s = 2 * m + 1;
    bool bad = false;
    for (int t = threadIdx.x; t < s * s; t += SS_T) {
        const int dy = t / s, dx = t - dy * s;
        if (!isfinite(__ldg(A + (int64_t)(y - m + dy) * pitch + (x - m + dx)))) bad = true;
    }
    return !__syncthreads_or(bad);
}

// One cluster per region: the candidate's pixel or -1.  Every block of the
// cluster follows the same control flow on the same exchanged values.
__global__ void __launch_bounds__(SS_T, 2) k_sub_stamps(const float* I, const float* R, int64_t W, int64_t H,
                                                        int64_t pitch, int nsx, int nsy, int hw, int fh, double nsig,
                                                        int slice, int2* reg_out) {
    extern __shared__ uint32_t stamp_cache[];   // [slice]
    __shared__ StampShared S;
    auto cl = cooperative_groups::this_cluster();
    const int nc = (int)cl.num_blocks(), rank = (int)cl.block_rank();
    const int reg = (int)blockIdx.x / nc;
    const int sx = reg % nsx, sy = reg / nsx;
    StampRegion g;
    g.I = I; g.R = R; g.pitch = pitch; g.W = W; g.H = H;
    g.x0 = (int)(sx * W / nsx);
    g.y0 = (int)(sy * H / nsy);
    g.rw = (int)((sx + 1) * W / nsx) - g.x0;
    g.rh = (int)((sy + 1) * H / nsy) - g.y0;
    const int64_t npix = (int64_t)g.rw * g.rh;
    g.t0 = (int)(npix * rank / nc);
    g.t1 = (int)(npix * (rank + 1) / nc);
    g.cached = false;
    g.cache = stamp_cache;
    g.buf = 0;
    const bool fits = g.t1 - g.t0 <= slice;   // per block: no decision of the cluster depends on it
    // the finite values: count, key range, smallest ulp exponent, largest |v|
    uint32_t c = 0, kmin = ~0u, kmax = 0, emin = ~0u, amax = 0;
    for (int t = g.t0 + threadIdx.x; t < g.t1; t += SS_T) {
        const uint32_t k = reg_load(g, t);
        if (fits) stamp_cache[t - g.t0] = k;
        if (k == STAMP_NONE) continue;
        c++;
        kmin = min(kmin, k);
        kmax = max(kmax, k);
        const uint32_t bits = __float_as_uint(fkey_inv(k)) & 0x7fffffffu;
        emin = min(emin, max(bits >> 23, 1u));      // ulp 2^(be - 150), denormals as be = 1
        amax = max(amax, bits);
    }
    g.cached = fits;   // a thread reads back its own elements only
    stamp_part(S, 0, c, OpAdd());
    stamp_part(S, 1, kmin, OpMin());
    stamp_part(S, 2, kmax, OpMax());
    stamp_part(S, 3, emin, OpMin());
    stamp_part(S, 4, amax, OpMax());
    __syncthreads();
    stamp_block(S, 0, 0, OpAdd());
    stamp_block(S, 0, 1, OpMin());
    stamp_block(S, 0, 2, OpMax());
    stamp_block(S, 0, 3, OpMin());
    stamp_block(S, 0, 4, OpMax());
    stamp_barrier();
    const long long n = (long long)stamp_all(S, 0, 0, OpAdd());
    const unsigned long long gmin = stamp_all(S, 0, 1, OpMin()), gmax = stamp_all(S, 0, 2, OpMax());
    emin = (uint32_t)stamp_all(S, 0, 3, OpMin());
    amax = (uint32_t)stamp_all(S, 0, 4, OpMax());
    g.buf = 1;
    if (n == 0) {
        if (rank == 0 && threadIdx.x == 0) reg_out[reg] = make_int2(-1, -1);
        stamp_barrier();   // no block leaves while another reads its exchange buffer
        return;
    }
    // median (Eq. 1's even-count mean of the middle pair)
    unsigned long long ka, kb;
    region_middle(g, ValueKey{}, n, gmin, gmax, ~0ull, S, &ka, &kb);
    const double va = (double)fkey_inv((uint32_t)ka), vb = (double)fkey_inv((uint32_t)kb);
    const double med = (n & 1) ? vb : __dmul_rn(0.5, __dadd_rn(va, vb));
    // MAD: exact integer differences at scale 2^e0 when they fit 62 bits
    const int e0 = (int)emin - 150 - 1;
    const double span = ldexp((double)__uint_as_float(amax) + fabs(med), -e0);
    double da, db;
    if (span < 4.6e18) {
        // -150 <= e0 <= 103: two powers of two within the normal range, of one sign
        const int h1 = -e0 / 2, h2 = -e0 - h1;
        const float s1 = __uint_as_float((uint32_t)(h1 + 127) << 23), s2 = __uint_as_float((uint32_t)(h2 + 127) << 23);
        const long long imed = __double2ll_rz(ldexp(med, -e0));
        const unsigned long long top = (unsigned long long)span + 1ull;
        // the same in every block: n, med, the extrema and the selected keys are the region's
        const long long exact32 = 2147483647ll - (imed < 0 ? -imed : imed);
        bool done = false;
        if (exact32 > 0) {
            region_middle(g, DistKey32{s1, s2, (int)imed}, n, 0ull, top < 0xffffffffull ? top : 0xffffffffull,
                          (unsigned long long)exact32, S, &ka, &kb);
            done = (long long)kb < exact32;
        }
        if (!done) region_middle(g, DistKey64{s1, s2, imed}, n, 0ull, top, ~0ull, S, &ka, &kb);
        da = ldexp((double)ka, e0);
        db = ldexp((double)kb, e0);
    } else {
        region_middle(g, DistKeyD{med}, n, 0ull, ~0ull, ~0ull, S, &ka, &kb);
        da = __longlong_as_double((long long)ka);
        db = __longlong_as_double((long long)kb);
    }
    const double mad = (n & 1) ? db : __dmul_rn(0.5, __dadd_rn(da, db));
    const double sgm = __dmul_rn(1.4826, mad);
    const double thr = __dadd_rn(med, __dmul_rn(nsig, sgm));
    // the brightest eligible pixel: arg-max rounds over the keys below the last
    // rejected one (fkey(v) << 32 | ~raster index: ties to the first pixel)
    const int m = fh + hw;
    unsigned long long bound = ~0ull;
    int bx = -1, by = -1;
    float best = 0.f;
    for (;;) {
        unsigned long long mk = 0;
        for (int t = g.t0 + threadIdx.x; t < g.t1; t += SS_T) {
            const uint32_t fk = reg_key(g, t);
            if (fk == STAMP_NONE || fk < (uint32_t)(mk >> 32) || fk > (uint32_t)(bound >> 32)) continue;
            const int yy = t / g.rw, y = g.y0 + yy, x = g.x0 + (t - yy * g.rw);
            if (x < m || y < m || x > W - 1 - m || y > H - 1 - m) continue;
            const unsigned long long key =
                ((unsigned long long)fk << 32) | (unsigned long long)(~(uint32_t)((int64_t)y * W + x));
            if (key < bound && key > mk) mk = key;
        }
        stamp_part(S, 0, mk, OpMax());
        __syncthreads();
        stamp_block(S, g.buf, 0, OpMax());
        stamp_barrier();
        mk = stamp_all(S, g.buf, 0, OpMax());
        g.buf ^= 1;
        if (mk == 0) break;                              // no eligible pixel left
        const uint32_t idx = ~(uint32_t)(mk & 0xffffffffu);
        const int x = (int)(idx % (uint32_t)W), y = (int)(idx / (uint32_t)W);
        if (block_box_finite(R, pitch, x, y, m) && block_box_finite(I, pitch, x, y, fh)) {
            bx = x; by = y;
            best = fkey_inv((uint32_t)(mk >> 32));
            break;
        }
        bound = mk;
    }
    if (rank == 0 && threadIdx.x == 0)
        reg_out[reg] = (bx >= 0 && (double)best > thr) ? make_int2(bx, by) : make_int2(-1, -1);
    stamp_barrier();   // no block leaves while another reads its exchange buffer
}

// Candidates in region order (row-major over the regions) and their count.
__global__ void __launch_bounds__(1024) k_sub_compact(const int2* reg, int nreg, int32_t* cx, int32_t* cy,
                                                      int32_t* n_dev) {
    dep_begin();
    __shared__ int red[32];
    __shared__ int carry;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (threadIdx.x == 0) carry = 0;
    __syncthreads();
    for (int base = 0; base < nreg; base += 1024) {
        const int r = base + threadIdx.x;
        const int2 v = r < nreg ? reg[r] : make_int2(-1, -1);
        const int f = v.x >= 0 ? 1 : 0;
        int inc = f;
        for (int o = 1; o < 32; o <<= 1) {
            const int t = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc += t;
        }
        if (lane == 31) red[warp] = inc;
        __syncthreads();
        int before = carry;
        for (int w = 0; w < warp; w++) before += red[w];
        if (f) { cx[before + inc - 1] = v.x; cy[before + inc - 1] = v.y; }
        __syncthreads();
        if (threadIdx.x == 1023) carry = before + inc;
        __syncthreads();
    }
    if (threadIdx.x == 0) *n_dev = carry;
}

// ---- normal equations ---------------------------------------------------------
struct SubFitJob {
    const float* I;
    const float* R;
    int64_t pitch, W, H;
    const int32_t* cx;
    const int32_t* cy;
    const int32_t* n_dev;
    int max_c;
    int hw, fh, nk, nf;          // nf = sum (deg_k + 1) one-dimensional filters
    double sig[8];
    int fo[9];                   // first filter of Gaussian k
    int sord, bord, nb, ns, ng, np;
    int deg[8];
    double* C;                   // [max_c][nb][nfp]
    double* G;                   // [max_c][nb][nb] (m <= n)
    double* X;                   // [max_c][nb][ng]
    double* Y;                   // [max_c][nb]
    double* BB;                  // [max_c][ng][ng]
    double* BI;                  // [max_c][ng]
    double* Ps;                  // [max_c][ns]
    double* AtA;                 // [np][np]
    double* Atb;                 // [np]
};

// Spatial terms x^p y^q (p outer, q inner, p + q <= order) of the normalised
// coordinates xs = 2x / (W - 1) - 1, ys = 2y / (H - 1) - 1 (0 for one column / row).
__device__ void sub_terms_dev(double x, double y, int64_t W, int64_t H, int order, double* t) {
    const double xs = W > 1 ? __dsub_rn(__ddiv_rn(2.0 * x, (double)(W - 1)), 1.0) : 0.0;
    const double ys = H > 1 ? __dsub_rn(__ddiv_rn(2.0 * y, (double)(H - 1)), 1.0) : 0.0;
    int n = 0;
    double xp = 1.0;
    for (int p = 0; p <= order; p++) {
        double yq = 1.0;
        for (int q = 0; q <= order - p; q++) {
            t[n++] = __dmul_rn(xp, yq);
            yq = __dmul_rn(yq, ys);
        }
        xp = __dmul_rn(xp, xs);
    }
}

// The footprint's C_n = R (x) K_n, separably.  FP64-bound (2 lanes a clock an SM:
// one candidate's 725 K multiply-adds are 190 us of one SM), so a candidate is cut
// into `parts` blocks that share nothing: block part takes the row filters
// [f0, f1) -- a cut of about equal work -- and the basis functions built on them.
// 100 candidates on 152 SMs: 200 -> 173 us with three parts each.
__global__ void __launch_bounds__(256) k_sub_conv(SubFitJob J, int parts) {
    dep_begin();
    extern __shared__ double sm[];
    const int c = blockIdx.x / parts, part = blockIdx.x - c * parts;
    if (c >= min(*J.n_dev, J.max_c)) return;
    const int S = 2 * J.hw + 1, m = J.hw + J.fh, WS = 2 * m + 1, FW = 2 * J.fh + 1, nfp = FW * FW;
    double* h = sm;                    // [nf][S] one-dimensional filters
    double* Rw = h + J.nf * S;         // [WS][WS] the template around the candidate
    double* T = Rw + WS * WS;          // [nf][WS][FW] row-filtered template
    int2* bf = reinterpret_cast<int2*>(T + (size_t)J.nf * WS * FW);   // [nb] row and column filter of basis n
    // row filters [f0, f1) and basis functions [n0, n1) of this part.  A filter's work:
    // its rows (WS per footprint column) and, for each basis function on it, the
    // footprint's columns (FW); it goes to the part that holds the middle of its share.
    int f0 = -1, f1 = -1, n0 = 0, n1 = 0;
    {
        int total = 0, done = 0, n = 0;
        for (int k = 0; k < J.nk; k++)
            for (int i = 0; i <= J.deg[k]; i++) total += WS + FW * (J.deg[k] - i + 1);
        for (int k = 0; k < J.nk; k++)
            for (int i = 0; i <= J.deg[k]; i++) {
                const int nj = J.deg[k] - i + 1, w = WS + FW * nj;
                if ((2 * done + w) * parts / (2 * total) == part) {
                    if (f0 < 0) { f0 = J.fo[k] + i; n0 = n; }
                    f1 = J.fo[k] + i + 1;
                    n1 = n + nj;
                }
                done += w;
                if (threadIdx.x == 0)
                    for (int j = 0; j < nj; j++) bf[n + j] = make_int2(J.fo[k] + i, J.fo[k] + j);
                n += nj;
            }
    }
    if (f0 < 0) return;
    for (int t = threadIdx.x; t < J.nf * S; t += 256) {
        const int f = t / S, u = t - f * S - J.hw;
        int k = 0;
        while (k + 1 < J.nk && f >= J.fo[k + 1]) k++;
        const int p = f - J.fo[k];
        double v = exp(-(double)(u * u) / (2.0 * J.sig[k] * J.sig[k]));
        for (int q = 0; q < p; q++) v *= (double)u;
        h[t] = v;
    }
    const int x0 = J.cx[c] - m, y0 = J.cy[c] - m;
    // a candidate whose support leaves the frame contributes nothing
    const bool inb = x0 >= 0 && y0 >= 0 && x0 + WS <= J.W && y0 + WS <= J.H;
    for (int t = threadIdx.x; t < WS * WS; t += 256) {
        const int r = t / WS, q = t - r * WS;
        Rw[t] = inb ? (double)dep_ld(J.R + (int64_t)(y0 + r) * J.pitch + (x0 + q)) : 0.0;
    }
    __syncthreads();
    // rows: T[f][r][q] = sum_u h_f(u) R(x - u, row r), x = footprint column q
    for (int t = f0 * WS * FW + threadIdx.x; t < f1 * WS * FW; t += 256) {
        const int f = t / (WS * FW), rq = t - f * WS * FW, r = rq / FW, q = rq - r * FW;
        const double* hf = h + f * S;
        const double* rr = Rw + r * WS + q + 2 * J.hw;   // R at column offset u = -hw .. hw: rr[-(u + hw)]
        double s = 0.0;
        for (int u = 0; u < S; u++) s = fma(hf[u], rr[-u], s);
        T[t] = s;
    }
    __syncthreads();
    // columns: C_n(p) = sum_v h_{k,j}(v) T_{k,i}(x, y - v)
    double* C = J.C + (size_t)c * J.nb * nfp;
    for (int t = n0 * nfp + threadIdx.x; t < n1 * nfp; t += 256) {
        const int n = t / nfp, p = t - n * nfp, pr = p / FW, pq = p - pr * FW;
        const int fi = bf[n].x, fj = bf[n].y;
        const double* hv = h + fj * S;
        const double* tc = T + (size_t)fi * WS * FW + (pr + 2 * J.hw) * FW + pq;
        double s = 0.0;
        for (int v = 0; v < S; v++) s = fma(hv[v], tc[-v * FW], s);
        C[t] = s;
    }
}

// A candidate's Gram matrix of the C_n, the cross terms with the background terms
// and the target, and the candidate's spatial terms.  FP64-bound as k_sub_conv, and
// cut into `parts` blocks in the same way: each takes an equal run of
// the sums.  100 candidates: 180 -> 138 us.
__global__ void __launch_bounds__(256) k_sub_gram(SubFitJob J, int parts) {
    dep_begin();
    extern __shared__ double sm[];
    const int c = blockIdx.x / parts, part = blockIdx.x - c * parts;
    if (c >= min(*J.n_dev, J.max_c)) return;
    const int FW = 2 * J.fh + 1, nfp = FW * FW, nb = J.nb, ng = J.ng;
    double* Cs = sm;                   // [nb][nfp]
    double* Is = Cs + nb * nfp;        // [nfp]
    double* Pb = Is + nfp;             // [ng][nfp]
    const double* C = J.C + (size_t)c * nb * nfp;
    for (int t = threadIdx.x; t < nb * nfp; t += 256) Cs[t] = C[t];
    const int cx = J.cx[c], cy = J.cy[c], m = J.hw + J.fh;
    const bool inb = cx >= m && cy >= m && cx + m < J.W && cy + m < J.H;   // else every part is 0
    for (int p = threadIdx.x; p < nfp; p += 256) {
        const int pr = p / FW, pq = p - pr * FW;
        const int x = cx - J.fh + pq, y = cy - J.fh + pr;
        Is[p] = inb ? (double)dep_ld(J.I + (int64_t)y * J.pitch + x) : 0.0;
        if (ng) {
            double tb[64];
            sub_terms_dev((double)x, (double)y, J.W, J.H, J.bord, tb);
            for (int b = 0; b < ng; b++) Pb[b * nfp + p] = inb ? tb[b] : 0.0;
        }
    }
    if (part == 0 && threadIdx.x == 0) {
        double ts[64];
        sub_terms_dev((double)cx, (double)cy, J.W, J.H, J.sord, ts);
        for (int s = 0; s < J.ns; s++) J.Ps[(size_t)c * J.ns + s] = ts[s];
    }
    __syncthreads();
    const int ntri = nb * (nb + 1) / 2;
    const int ntask = ntri + nb * ng + nb + ng * ng + ng;
    const int share = (ntask + parts - 1) / parts, tend = min(ntask, (part + 1) * share);
    for (int t = part * share + threadIdx.x; t < tend; t += 256) {
        const double *a, *b;
        double* out;
        if (t < ntri) {                                   // G[n][m], m <= n
            int n = (int)((sqrt(8.0 * t + 1.0) - 1.0) * 0.5);
            while (n * (n + 1) / 2 > t) n--;
            while ((n + 1) * (n + 2) / 2 <= t) n++;
            const int mm = t - n * (n + 1) / 2;
            a = Cs + n * nfp; b = Cs + mm * nfp;
            out = J.G + ((size_t)c * nb + n) * nb + mm;
        } else if (t < ntri + nb * ng) {                  // X[n][b] = sum C_n P_b
            const int u = t - ntri, n = u / ng, g = u - n * ng;
            a = Cs + n * nfp; b = Pb + g * nfp;
            out = J.X + ((size_t)c * nb + n) * ng + g;
        } else if (t < ntri + nb * ng + nb) {             // Y[n] = sum C_n I
            const int n = t - ntri - nb * ng;
            a = Cs + n * nfp; b = Is;
            out = J.Y + (size_t)c * nb + n;
        } else if (t < ntri + nb * ng + nb + ng * ng) {   // BB[g][h] = sum P_g P_h
            const int u = t - ntri - nb * ng - nb, g = u / ng, hh = u - g * ng;
            a = Pb + g * nfp; b = Pb + hh * nfp;
            out = J.BB + ((size_t)c * ng + g) * ng + hh;
        } else {                                          // BI[g] = sum P_g I
            const int g = t - ntri - nb * ng - nb - ng * ng;
            a = Pb + g * nfp; b = Is;
            out = J.BI + (size_t)c * ng + g;
        }
        double s = 0.0;
        for (int p = 0; p < nfp; p++) s = fma(a[p], b[p], s);
        *out = s;
    }
}

// AtA and Atb from the candidates' parts, summed in candidate order: one thread
// per entry of the lower triangle (both halves written).  Bound by latency: a
// candidate's parts lie apart, so eight candidates' loads are issued before their
// sums are formed.  100 candidates, 297 unknowns: 50 -> 40 us.
template <class Load, class Term>
__device__ __forceinline__ double sum_candidates(int nc, Load&& load, Term&& term) {
    constexpr int B = 8;
    double s = 0.0;
    for (int c0 = 0; c0 < nc; c0 += B) {
        double v[B][3];
#pragma unroll
        for (int q = 0; q < B; q++) load(min(c0 + q, nc - 1), v[q]);
#pragma unroll
        for (int q = 0; q < B; q++)
            if (c0 + q < nc) term(s, v[q]);
    }
    return s;
}

__global__ void __launch_bounds__(256) k_sub_assemble(SubFitJob J) {
    dep_begin();
    const int nc = min(*J.n_dev, J.max_c);
    const int np = J.np, nk = J.nb * J.ns, ns = J.ns, nb = J.nb, ng = J.ng;
    const int ntri = np * (np + 1) / 2;
    for (int t = blockIdx.x * 256 + threadIdx.x; t < ntri + np; t += gridDim.x * 256) {
        if (t >= ntri) {                                   // Atb
            const int a = t - ntri;
            double s = 0.0;
            if (a < nk) {
                const int n = a / ns, sa = a - n * ns;
                for (int c = 0; c < nc; c++) s += J.Ps[(size_t)c * ns + sa] * J.Y[(size_t)c * nb + n];
            } else {
                const int g = a - nk;
                for (int c = 0; c < nc; c++) s -= J.BI[(size_t)c * ng + g];
            }
            J.Atb[a] = s;
            continue;
        }
        int a = (int)((sqrt(8.0 * t + 1.0) - 1.0) * 0.5);
        while (a * (a + 1) / 2 > t) a--;
        while ((a + 1) * (a + 2) / 2 <= t) a++;
        const int b = t - a * (a + 1) / 2;                 // b <= a
        double s;
        if (a < nk) {                                      // both kernel unknowns
            const int n = a / ns, sa = a - n * ns, mm = b / ns, sb = b - mm * ns;
            const int hi = max(n, mm), lo = min(n, mm);
            s = sum_candidates(
                nc,
                [&](int c, double* v) {
                    v[0] = J.Ps[(size_t)c * ns + sa];
                    v[1] = J.Ps[(size_t)c * ns + sb];
                    v[2] = J.G[((size_t)c * nb + hi) * nb + lo];
                },
                [](double& t, const double* v) { t += v[0] * v[1] * v[2]; });
        } else if (b < nk) {                               // background row a, kernel column b
            const int g = a - nk, mm = b / ns, sb = b - mm * ns;
            s = sum_candidates(
                nc,
                [&](int c, double* v) {
                    v[0] = J.Ps[(size_t)c * ns + sb];
                    v[1] = J.X[((size_t)c * nb + mm) * ng + g];
                },
                [](double& t, const double* v) { t -= v[0] * v[1]; });
        } else {                                           // both background
            const int g = a - nk, hh = b - nk;
            s = sum_candidates(
                nc, [&](int c, double* v) { v[0] = J.BB[((size_t)c * ng + g) * ng + hh]; },
                [](double& t, const double* v) { t += v[0]; });
        }
        J.AtA[(size_t)a * np + b] = s;
        J.AtA[(size_t)b * np + a] = s;
    }
}

// Cholesky solve of AtA x = Atb in place, blocked and right-looking: for each
// panel of CB columns, the diagonal block is factored in shared memory
// (k_chol_diag), the rows below it are solved against it (k_chol_trsm, a warp
// per row), and the trailing lower triangle takes the panel's rank-CB update
// (k_chol_syrk, a tile per block).  Then the two triangular solves,
// CB rows at a time (k_chol_solve).  FP64 throughout.  A pivot that is not
// positive sets *status = 1; the later kernels then leave everything as is.
constexpr int CB = 32;

__global__ void k_chol_init(int32_t* status) {
    dep_begin();
    *status = 0;
}

// The diagonal block.  Bound by the chain square root -> reciprocal -> scaled
// column -> next pivot, so warp 0 runs that chain alone, one column ahead: it
// brings column j + 1 up to date and factors it while the other warps apply column
// j to the columns from j + 2 on; one barrier a column.  An entry still takes its
// updates in ascending column order.  32 columns: 44 -> 28 us.
constexpr int CD_T = 256, CD_W = CD_T / 32;

__global__ void __launch_bounds__(CD_T) k_chol_diag(double* A, int n, int k0, int32_t* status) {
    dep_begin();
    __shared__ double D[CB][CB + 1];
    if (__ldcg(status)) return;
    const int b = min(CB, n - k0), lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int t = threadIdx.x; t < CB * CB; t += CD_T) {
        const int i = t >> 5, j = t & 31;
        D[i][j] = i < b && j <= i ? A[(size_t)(k0 + i) * n + k0 + j] : 0.0;
    }
    __syncthreads();
    // column c, already up to date in lane i's v = D[i][c]: scaled by its pivot;
    // returns whether the pivot is not positive
    auto factor = [&](int c, double v) {
        const double d = __shfl_sync(0xffffffffu, v, c);
        const bool ok = d > 0.0;
        const double r = ok ? sqrt(d) : 1.0;
        const double rinv = 1.0 / r;
        if (lane == c) D[lane][c] = r;
        else if (lane > c) D[lane][c] = v * rinv;
        return !ok;
    };
    bool bad = warp == 0 && factor(0, D[lane][0]);
    bool fail = __syncthreads_or(bad);
    for (int j = 0; j + 1 < b && !fail; j++) {
        const double lj = lane > j ? D[lane][j] : 0.0;
        if (warp == 0) {
            const int c = j + 1;
            double v = D[lane][c];
            if (lane >= c) v -= lj * D[c][j];
            bad = factor(c, v);
        } else {
            for (int c = j + 1 + warp; c < b; c += CD_W - 1) {
                const double m = D[c][j];
                if (lane >= c) D[lane][c] -= lj * m;
            }
        }
        fail = __syncthreads_or(bad);
    }
    if (fail) {
        if (threadIdx.x == 0) *status = 1;
        return;
    }
    for (int t = threadIdx.x; t < CB * CB; t += CD_T) {
        const int i = t >> 5, j = t & 31;
        if (i < b && j <= i) A[(size_t)(k0 + i) * n + k0 + j] = D[i][j];
    }
}

// a / b from y = RN(1 / b), correctly rounded (Markstein, IBM J. Res. Dev. 34,
// 1990): the residual of a quotient within one ulp, formed exactly by an FMA, times
// y corrects it to the rounded one.  The first product may be two ulps off, so the
// correction is applied twice.  Outside the range in which no step can overflow or
// lose bits the division itself.
__device__ __forceinline__ double div_by_recip(double a, double b, double y) {
    // exponents of a within 2^-600 .. 2^600 and of b within 2^-250 .. 2^250 (tested on the
    // bits: FP64 compares share the pipe)
    const uint32_t ea = ((uint32_t)__double2hiint(a) >> 20) & 0x7ffu, eb = ((uint32_t)__double2hiint(b) >> 20) & 0x7ffu;
    if (ea - 423u < 1200u && eb - 773u < 500u) {
        double q = a * y;
        q = fma(fma(-q, b, a), y, q);
        return fma(fma(-q, b, a), y, q);
    }
    return a / b;
}

// rows i >= k0 + CB: L21[i] = A21[i] L11^-T, one warp per row (lane j holds column
// j).  A step is a quotient, a broadcast and a multiply-add; the quotients come from
// the diagonal's reciprocals, taken once per block.  FP64 instructions of one SM
// share a pipe of 2 lanes a clock, so two warps a block spread the rows over as many
// SMs as there are.  265 rows: 23 -> 18 us (eight warps a block, a division a step).
constexpr int CT_T = 64;

__global__ void __launch_bounds__(CT_T) k_chol_trsm(double* A, int n, int k0, const int32_t* status) {
    dep_begin();
    __shared__ double L[CB][CB + 1];
    if (__ldcg(status)) return;
    const int b = min(CB, n - k0);
    for (int t = threadIdx.x; t < CB * CB; t += CT_T) {
        const int i = t >> 5, j = t & 31;
        L[i][j] = i < b && j <= i ? A[(size_t)(k0 + i) * n + k0 + j] : (i == j ? 1.0 : 0.0);
    }
    __syncthreads();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const double dl = L[lane][lane], yl = 1.0 / dl;
    for (int i = k0 + b + blockIdx.x * (CT_T / 32) + warp; i < n; i += gridDim.x * (CT_T / 32)) {
        double a = lane < b ? A[(size_t)i * n + k0 + lane] : 0.0;
        double x = 0.0;
        for (int j = 0; j < b; j++) {
            const double xj = __shfl_sync(0xffffffffu, lane == j ? div_by_recip(a, dl, yl) : 0.0, j);
            if (lane == j) x = xj;
            if (lane > j) a -= xj * L[lane][j];
        }
        if (lane < b) A[(size_t)i * n + k0 + lane] = x;
    }
}

// trailing update of the lower triangle from row / column k0 + CB on: tile
// (ti, tc), ti >= tc, of CS x CS, A[i][c] -= sum_m L[i][k0 + m] L[c][k0 + m].  Tiles
// of 16 give every SM one at the first panels of ~300 unknowns (FP64-bound: 14 ->
// 6 us with 32 x 32, which left two thirds of the SMs idle).
constexpr int CS = 16;

__global__ void __launch_bounds__(CS * CS) k_chol_syrk(double* A, int n, int k0, const int32_t* status) {
    dep_begin();
    __shared__ double Li[CS][CB + 1], Lc[CS][CB + 1];
    if (__ldcg(status)) return;
    const int r0 = k0 + CB;
    const int t = blockIdx.x;
    int ti = (int)((sqrtf(8.0f * t + 1.0f) - 1.0f) * 0.5f);
    while (ti * (ti + 1) / 2 > t) ti--;
    while ((ti + 1) * (ti + 2) / 2 <= t) ti++;
    const int tc = t - ti * (ti + 1) / 2;
    const int i0 = r0 + ti * CS, c0 = r0 + tc * CS;
    for (int q = threadIdx.x; q < CS * CB; q += CS * CS) {
        const int r = q / CB, m = q - r * CB;
        Li[r][m] = i0 + r < n ? A[(size_t)(i0 + r) * n + k0 + m] : 0.0;
        Lc[r][m] = c0 + r < n ? A[(size_t)(c0 + r) * n + k0 + m] : 0.0;
    }
    __syncthreads();
    const int r = threadIdx.x / CS, c = threadIdx.x % CS;
    const int i = i0 + r, cc = c0 + c;
    if (i >= n || cc >= n || cc > i) return;
    double acc = 0.0;
#pragma unroll
    for (int m = 0; m < CB; m++) acc = fma(Li[r][m], Lc[c][m], acc);
    A[(size_t)i * n + cc] -= acc;
}

// L y = b, then L' x = y, CB rows at a time: the block's warps first take the
// dot products with the part already solved (a warp per row), then warp 0
// solves the CB x CB triangle.  The solution goes to b (and x64 / x32).
// the CB x CB diagonal block of L at r0 (bsz rows) in shared memory, and the
// reciprocals of its diagonal, for the sequential part of a solve step
__device__ __forceinline__ void chol_stage_block(const double* A, int n, int r0, int bsz, double (*Ld)[CB + 1],
                                                 double* rd) {
    for (int t = threadIdx.x; t < bsz * bsz; t += 1024) {
        const int i = t / bsz, j = t - i * bsz;
        Ld[i][j] = A[(size_t)(r0 + i) * n + r0 + j];
    }
    if (threadIdx.x < bsz) rd[threadIdx.x] = 1.0 / A[(size_t)(r0 + threadIdx.x) * n + r0 + threadIdx.x];
}

__global__ void __launch_bounds__(1024) k_chol_solve(const double* A, double* b, int n, double* x64, float* x32,
                                                     const int32_t* status) {
    dep_begin();
    __shared__ double part[CB], rd[CB];
    __shared__ double Ld[CB][CB + 1];
    if (__ldcg(status)) return;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int r0 = 0; r0 < n; r0 += CB) {                 // forward
        const int bsz = min(CB, n - r0);
        chol_stage_block(A, n, r0, bsz, Ld, rd);
        if (warp < bsz) {
            const int i = r0 + warp;
            double s = 0.0;
            for (int k = lane; k < r0; k += 32) s = fma(A[(size_t)i * n + k], b[k], s);
            for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
            if (lane == 0) part[warp] = b[i] - s;
        }
        __syncthreads();
        if (warp == 0) {
            double y = lane < bsz ? part[lane] : 0.0, x = 0.0;
            for (int j = 0; j < bsz; j++) {
                const double xj = __shfl_sync(0xffffffffu, y * rd[j], j);
                if (lane == j) x = xj;
                if (lane > j && lane < bsz) y -= Ld[lane][j] * xj;
            }
            if (lane < bsz) b[r0 + lane] = x;
        }
        __syncthreads();
    }
    const int nblk = (n + CB - 1) / CB;
    for (int blk = nblk - 1; blk >= 0; blk--) {          // backward with L'
        const int r0 = blk * CB, bsz = min(CB, n - r0);
        chol_stage_block(A, n, r0, bsz, Ld, rd);
        if (warp < bsz) {
            const int i = r0 + warp;
            double s = 0.0;
            for (int k = r0 + bsz + lane; k < n; k += 32) s = fma(A[(size_t)k * n + i], b[k], s);
            for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
            if (lane == 0) part[warp] = b[i] - s;
        }
        __syncthreads();
        if (warp == 0) {
            double y = lane < bsz ? part[lane] : 0.0, x = 0.0;
            for (int j = bsz - 1; j >= 0; j--) {
                const double xj = __shfl_sync(0xffffffffu, y * rd[j], j);
                if (lane == j) x = xj;
                if (lane < j) y -= Ld[j][lane] * xj;
            }
            if (lane < bsz) b[r0 + lane] = x;
        }
        __syncthreads();
    }
    for (int i = threadIdx.x; i < n; i += 1024) {
        if (x64) x64[i] = b[i];
        if (x32) x32[i] = (float)b[i];
    }
}

}  // namespace ipp

using namespace ipp;

namespace {
size_t a256s(size_t x) { return (x + 255) & ~(size_t)255; }

struct SubDims {
    int nb, ns, ng, np, nf, nfp, WS, S;
    size_t conv_smem, gram_smem;
};

SubDims sub_dims(int hw, int fh, int nk, const int32_t* deg, int sord, int bord) {
    SubDims d{};
    for (int k = 0; k < nk; k++) { d.nb += (deg[k] + 1) * (deg[k] + 2) / 2; d.nf += deg[k] + 1; }
    d.ns = (sord + 1) * (sord + 2) / 2;
    d.ng = bord >= 0 ? (bord + 1) * (bord + 2) / 2 : 0;
    d.np = d.nb * d.ns + d.ng;
    d.S = 2 * hw + 1;
    d.WS = 2 * (hw + fh) + 1;
    const int FW = 2 * fh + 1;
    d.nfp = FW * FW;
    d.conv_smem = sizeof(double) * ((size_t)d.nf * d.S + (size_t)d.WS * d.WS + (size_t)d.nf * d.WS * FW) +
                  sizeof(int2) * (size_t)d.nb;
    d.gram_smem = sizeof(double) * ((size_t)d.nb * d.nfp + d.nfp + (size_t)d.ng * d.nfp);
    return d;
}

// Blocks a candidate of the FP64-bound kernels, one block an SM: the cut whose
// waves take the least time (100 candidates: one part
// fills 100 SMs once, three fill 152 twice with a third of the work each).
int sub_parts(int max_c) {
    const int64_t sms = ipp_sm_count();
    int best = 1;
    double cost = 1e30;
    for (int p = 1; p <= 6; p++) {
        const double t = (double)cdiv((int64_t)max_c * p, sms) / p;
        if (t < cost * 0.95) { cost = t; best = p; }
    }
    return best;
}

// workspace: region results, then the per-candidate parts, the normal
// equations and the candidate list of ipp_sub_fit
size_t sub_carve(const SubDims& d, int max_c, int nreg, void* base, SubFitJob* J, int2** reg, int32_t** cxy) {
    const size_t mc = (size_t)std::max(max_c, 1);
    const size_t sz[] = {(size_t)std::max(nreg, 1) * sizeof(int2), mc * d.nb * d.nfp * 8, mc * d.nb * d.nb * 8,
                         mc * d.nb * std::max(d.ng, 1) * 8, mc * d.nb * 8, mc * std::max(d.ng * d.ng, 1) * 8,
                         mc * std::max(d.ng, 1) * 8, mc * d.ns * 8, (size_t)d.np * d.np * 8, (size_t)d.np * 8,
                         (2 * mc + 1) * sizeof(int32_t)};
    constexpr int NA = sizeof(sz) / sizeof(sz[0]);
    size_t off[NA], o = 0;
    for (int k = 0; k < NA; k++) { off[k] = o; o += a256s(sz[k]); }
    if (base) {
        unsigned char* b = static_cast<unsigned char*>(base);
        if (reg) *reg = reinterpret_cast<int2*>(b + off[0]);
        if (J) {
            J->C = reinterpret_cast<double*>(b + off[1]);
            J->G = reinterpret_cast<double*>(b + off[2]);
            J->X = reinterpret_cast<double*>(b + off[3]);
            J->Y = reinterpret_cast<double*>(b + off[4]);
            J->BB = reinterpret_cast<double*>(b + off[5]);
            J->BI = reinterpret_cast<double*>(b + off[6]);
            J->Ps = reinterpret_cast<double*>(b + off[7]);
            J->AtA = reinterpret_cast<double*>(b + off[8]);
            J->Atb = reinterpret_cast<double*>(b + off[9]);
        }
        if (cxy) *cxy = reinterpret_cast<int32_t*>(b + off[10]);
    }
    return o;
}
}  // namespace

size_t ipp_subfit_ws_bytes(int max_c, int nreg, int hw, int fh, int nk, const int32_t* deg, int sord, int bord) {
    return sub_carve(sub_dims(hw, fh, nk, deg, sord, bord), max_c, nreg, nullptr, nullptr, nullptr, nullptr);
}

size_t ipp_subfit_smem(int hw, int fh, int nk, const int32_t* deg, int sord, int bord) {
    const SubDims d = sub_dims(hw, fh, nk, deg, sord, bord);
    return std::max(d.conv_smem, d.gram_smem);
}

int ipp_launch_sub_stamps(const float* I, const float* R, int64_t W, int64_t H, int64_t pitch, int nsx, int nsy,
                          int hw, int fh, double nsig, int32_t* cx, int32_t* cy, int32_t* n_dev, void* ws,
                          cudaStream_t s) {
    int2* reg = static_cast<int2*>(ws);   // the first array of the workspace
    // Blocks a region: as few as hold the largest region in their slices, then more
    // while the grid stays within one wave of two blocks an SM and a slice keeps
    // at least 8 pixels a thread (below that a pass is mostly its exchange).
    const int64_t nreg = (int64_t)nsx * nsy, npix = ((W + nsx - 1) / nsx) * ((H + nsy - 1) / nsy);
    int nc = 1;
    while (nc < SS_NC && (npix > (int64_t)nc * SS_SLICE ||
                          (nreg * nc * 2 <= 2 * ipp_sm_count() && npix >= (int64_t)nc * 2 * 8 * SS_T)))
        nc *= 2;
    const int slice = (int)std::min<int64_t>(SS_SLICE, npix / nc + 1);
    auto fn = k_sub_stamps;
    if (cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, SS_SLICE * (int)sizeof(float)) !=
        cudaSuccess)
        return ipp_check_launch("k_sub_stamps shared memory");
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)(nreg * nc));
    cfg.blockDim = dim3(SS_T);
    cfg.dynamicSmemBytes = (size_t)slice * sizeof(float);
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)nc;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    if (cudaLaunchKernelEx(&cfg, fn, I, R, W, H, pitch, nsx, nsy, hw, fh, nsig, slice, reg) != cudaSuccess)
        return ipp_check_launch("k_sub_stamps");
    if (int e = ipp_check_launch("k_sub_stamps")) return e;
    ipp_launch_dep(k_sub_compact, dim3(1), 1024, 0, s, reg, nsx * nsy, cx, cy, n_dev);
    return ipp_check_launch("k_sub_compact");
}

int ipp_launch_sub_normal(const float* I, const float* R, int64_t W, int64_t H, int64_t pitch, const int32_t* cx,
                          const int32_t* cy, const int32_t* n_dev, int max_c, int nreg, int hw, int fh, int nk,
                          const double* sig, const int32_t* deg, int sord, int bord, double* AtA, double* Atb,
                          void* ws, cudaStream_t s) {
    const SubDims d = sub_dims(hw, fh, nk, deg, sord, bord);
    SubFitJob J{};
    sub_carve(d, max_c, nreg, ws, &J, nullptr, nullptr);
    J.I = I; J.R = R; J.pitch = pitch; J.W = W; J.H = H;
    J.cx = cx; J.cy = cy; J.n_dev = n_dev; J.max_c = max_c;
    J.hw = hw; J.fh = fh; J.nk = nk; J.nf = d.nf;
    J.fo[0] = 0;
    for (int k = 0; k < nk; k++) { J.sig[k] = sig[k]; J.deg[k] = deg[k]; J.fo[k + 1] = J.fo[k] + deg[k] + 1; }
    J.sord = sord; J.bord = bord; J.nb = d.nb; J.ns = d.ns; J.ng = d.ng; J.np = d.np;
    if (AtA) J.AtA = AtA;
    if (Atb) J.Atb = Atb;
    if (max_c < 1) return IPP_OK;
    cudaFuncSetAttribute(k_sub_conv, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)d.conv_smem);
    cudaFuncSetAttribute(k_sub_gram, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)d.gram_smem);
    const int parts = sub_parts(max_c);
    ipp_launch_dep(k_sub_conv, dim3((unsigned)(max_c * parts)), 256, d.conv_smem, s, J, parts);
    if (int e = ipp_check_launch("k_sub_conv")) return e;
    ipp_launch_dep(k_sub_gram, dim3((unsigned)(max_c * parts)), 256, d.gram_smem, s, J, parts);
    if (int e = ipp_check_launch("k_sub_gram")) return e;
    const int nt = d.np * (d.np + 1) / 2 + d.np;
    ipp_launch_dep(k_sub_assemble, dim3((unsigned)((nt + 255) / 256)), 256, 0, s, J);
    return ipp_check_launch("k_sub_assemble");
}

int ipp_launch_sub_solve(double* AtA, double* Atb, int np, double* coef64, float* coef, int32_t* status,
                         cudaStream_t s) {
    ipp_launch_dep(k_chol_init, dim3(1), 1, 0, s, status);
    if (int e = ipp_check_launch("k_chol_init")) return e;
    for (int k0 = 0; k0 < np; k0 += CB) {
        ipp_launch_dep(k_chol_diag, dim3(1), CD_T, 0, s, AtA, np, k0, status);
        if (int e = ipp_check_launch("k_chol_diag")) return e;
        const int rest = np - k0 - CB;
        if (rest <= 0) break;
        ipp_launch_dep(k_chol_trsm, dim3((unsigned)((rest + CT_T / 32 - 1) / (CT_T / 32))), CT_T, 0, s, AtA, np, k0, status);
        if (int e = ipp_check_launch("k_chol_trsm")) return e;
        const int nt = (rest + CS - 1) / CS;
        ipp_launch_dep(k_chol_syrk, dim3((unsigned)(nt * (nt + 1) / 2)), CS * CS, 0, s, AtA, np, k0, status);
        if (int e = ipp_check_launch("k_chol_syrk")) return e;
    }
    ipp_launch_dep(k_chol_solve, dim3(1), 1024, 0, s, AtA, Atb, np, coef64, coef, status);
    return ipp_check_launch("k_chol_solve");
}

int ipp_launch_sub_fit(const float* I, const float* R, int64_t W, int64_t H, int64_t pitch, int nsx, int nsy,
                       double nsig, int hw, int fh, int nk, const double* sig, const int32_t* deg, int sord, int bord,
                       double* coef64, float* coef, int32_t* cx_out, int32_t* cy_out, int32_t* n_out,
                       int32_t* status, void* ws, cudaStream_t s) {
    const SubDims d = sub_dims(hw, fh, nk, deg, sord, bord);
    const int nreg = nsx * nsy;
    SubFitJob J{};
    int32_t* cxy = nullptr;
    sub_carve(d, nreg, nreg, ws, &J, nullptr, &cxy);
    int32_t* cx = cx_out ? cx_out : cxy;
    int32_t* cy = cy_out ? cy_out : cxy + nreg;
    int32_t* nd = n_out ? n_out : cxy + 2 * nreg;
    if (int e = ipp_launch_sub_stamps(I, R, W, H, pitch, nsx, nsy, hw, fh, nsig, cx, cy, nd, ws, s)) return e;
    if (int e = ipp_launch_sub_normal(I, R, W, H, pitch, cx, cy, nd, nreg, nreg, hw, fh, nk, sig, deg, sord, bord,
                                      nullptr, nullptr, ws, s))
        return e;
    return ipp_launch_sub_solve(J.AtA, J.Atb, d.np, coef64, coef, status, s);
}

// Preconditioner of the correlated-noise gap filling: block-Jacobi over the
// gaps of the Schur operator S = E^T C^T diag(gamma) C E.  Within a gap of
// L consecutive flagged samples S is (away from the detscan ends) the
// symmetric Toeplitz matrix T_ij = h(|i-j|) with
//   h(d) = (1/n) sum_{k>=1} gamma_k cos(pi k d / n),
//   gamma_k = sigma0^2 r/(1+r),  r = (f_k/f_knee)^-alpha,  f_k = k f_samp/(2n).
// The kernel is evaluated per detector at a reference length H (cz_href, a
// power of two at least the longest detscan; the preconditioner only has to
// be symmetric positive definite, and a kernel shared by all detscans of a
// detector is close enough), at every lag d < H at once: h(d) is the real
// part of the length-2H DFT of the even sequence a_k = gamma_k (k < H),
// a_{2H-k} = gamma_k, a_H = 0, divided by 2H.  The transform of a real even
// sequence is real, so one complex FP32 FFT serves two detectors (one in the
// real, one in the imaginary part), each brought to a peak between 1 and 2 by
// a power of two first: the rounding of the transform goes by the larger of
// the two, and a detector far below its partner, or beside one whose noise
// parameters are not finite, keeps its own kernel.  A scan then stores, for the coarse
// correction, the prefix sums H(x) = sum_{d<x} h(d) and G(x) = sum_{d<x} d h(d)
// (FP32 double-words); the gap blocks take the first TOEP_LMAX lags.
// A second kernel finds, for every order L, the first column
// x = T_L^{-1} e_1 (Durbin's solutions, Golub & Van Loan, Section 4.7) by the
// Schur recursion.  The CG then applies T_L^{-1} by the Gohberg-Semencul
// formula T^{-1} = (L(x) L(x)^T - L(w) L(w)^T) / x_0, w = (0, x_{L-1}, ..,
// x_1), L(v) the lower-triangular Toeplitz matrix with first column v.
#include "common.cuh"
#include "fft_reg.cuh"
#include "internal.cuh"

namespace tg {

constexpr int CZ_T = 256;       // threads per CTA of the FFT passes and the scans
constexpr int CZ_C = 32;        // columns (consecutive j) of an FFT tile
constexpr int CZ_PER = 8;       // lags per thread of the scans
constexpr int CZ_CHUNK = CZ_T * CZ_PER;

// FP32 double-word (head + tail, |tail| <= ulp(head)/2): about 2^-45 relative
// per operation, at the FP32 rate (FP64 issues at 1/64 of it on this part).
struct DW { float h, l; };
__device__ __forceinline__ DW dw_renorm(float s, float r) {
    DW o;
    o.h = __fadd_rn(s, r);
    o.l = __fsub_rn(r, __fsub_rn(o.h, s));
    return o;
}
// x + (p + e), e small against p
__device__ __forceinline__ DW dw_add2(DW x, float p, float e) {
    const float s = __fadd_rn(x.h, p);
    const float bb = __fsub_rn(s, x.h);
    float r = __fadd_rn(__fsub_rn(x.h, __fsub_rn(s, bb)), __fsub_rn(p, bb));
    r = __fadd_rn(r, __fadd_rn(x.l, e));
    return dw_renorm(s, r);
}
__device__ __forceinline__ DW dw_add(DW x, DW y) { return dw_add2(x, y.h, y.l); }
// x + a b
__device__ __forceinline__ DW dw_fma(DW x, DW a, DW b) {
    const float p = __fmul_rn(a.h, b.h);
    float e = __fmaf_rn(a.h, b.h, -p);
    e = __fmaf_rn(a.h, b.l, e);
    e = __fmaf_rn(a.l, b.h, e);
    return dw_add2(x, p, e);
}
// a / b
__device__ __forceinline__ DW dw_div(DW a, DW b) {
    const float inv = __frcp_rn(b.h);
    const float q = __fmul_rn(a.h, inv);
    const float p = __fmul_rn(q, b.h);
    float r = __fsub_rn(a.h, p);
    r = __fsub_rn(r, __fmaf_rn(q, b.h, -p));
    r = __fadd_rn(r, __fmaf_rn(-q, b.l, a.l));
    return dw_renorm(q, __fmul_rn(r, inv));
}

// A detector's sequence: gamma_k / sigma0^2 = r / (1 + r) at mode k of the
// length-2H sequence (f_k = k f_samp / (2H); a_0 = a_H = 0), in units of the
// power of two `unit` at or below its largest value (the first or the last:
// it is monotone in k).
struct CzDet { float unit, fscale, mal; };
__device__ __forceinline__ float cz_ratio(const CzDet &c, int kk) {
    const float r = exp2f(c.mal * log2f(static_cast<float>(kk) * c.fscale));
    return 1.0f / (1.0f + 1.0f / r);          // r / (1 + r), also for r = 0 or inf
}
__device__ __forceinline__ CzDet cz_det(const double *__restrict__ psd, int det, int href, double fsamp, float &peak) {
    CzDet c{1.0f, static_cast<float>(fsamp / (2.0 * href * psd[3 * det + 1])), static_cast<float>(-psd[3 * det + 2])};
    const float lo = cz_ratio(c, 1), hi = cz_ratio(c, href - 1);
    peak = lo + hi >= 0.f ? fmaxf(lo, hi) : lo + hi;                   // NaN where one of them is
    c.unit = __uint_as_float(max(__float_as_uint(peak >= 0.f ? peak : 0.f) & 0x7f800000u, 0x00800000u));
    return c;
}
// in units; a value that is not a number would spread to the partner: zero
// (the detector's kernel is marked by cz_scale)
__device__ __forceinline__ float cz_gamma(const CzDet &c, int k, int href) {
    const int kk = k <= href ? k : 2 * href - k;
    if (kk == 0 || kk >= href) return 0.f;
    const float g = cz_ratio(c, kk) * __uint_as_float(0x7f000000u - __float_as_uint(c.unit));
    return g >= 0.f ? g : 0.f;
}
// what the transform's output is multiplied by: NaN for parameters that give
// no kernel (the tables then end at order 0 and the detector goes without)
__device__ __forceinline__ float cz_scale(const CzDet &c, float peak, double sig0) {
    const float s2 = static_cast<float>(sig0 * sig0);
    return peak >= 0.f && s2 < __int_as_float(0x7f800000) ? s2 * c.unit : __int_as_float(0x7fffffff);
}

// One radix-R Stockham pass (R = 8 A, forward DFT) over the length-M sequence
// of every detector pair, Ns points of each sub-transform done (powers of
// two).  Point j < M/R reads x[j + r M/R], twiddles by exp(-2 pi i r k /
// (Ns R)), k = j mod Ns, and writes output r' to (j - k) R + k + r' Ns.
// A CTA takes CZ_C consecutive j: the R-point DFTs are A-point DFTs of the
// rows r = 8 n1 + n2 in registers, a table twiddle, one exchange through
// shared memory, and 8-point DFTs over n2.  FIRST evaluates gamma in place
// of a load (and writes through shared memory, since its outputs of one j
// are consecutive), and leaves the detectors' scales; LAST keeps the lags
// d < H only, real part to the first detector's kernel, imaginary part to the
// second's, each times its scale.
// Every radix-R pass reads and writes the sequence once, so R up to 128
// takes three passes where radix 4 took ten; per point one sincospif in
// eight instead of three in four.  Bound: L2 bandwidth and the gamma
// evaluations.  Fill, FFT and tables of 12 detectors, H = 262144: 1022 us by
// radix-4 passes per detector and FP64 scans, 151 us so; of 2 detectors,
// H = 32768: 166 us, 37 us.
template <int A, bool FIRST, bool LAST>
__global__ void __launch_bounds__(CZ_T)
k_cz_fft(const float2 *__restrict__ src, float2 *__restrict__ dst, const double *__restrict__ psd, int ndet, int href,
         double fsamp, int Ns, float *__restrict__ scale, float *__restrict__ hout)
{
    constexpr int R = 8 * A;
    constexpr int IT = (A * CZ_C + CZ_T - 1) / CZ_T;
    __shared__ float2 t[R * (CZ_C + 1)];
    __shared__ float2 wt[R];                   // W_R^{n2 k1} at n2 A + k1
    __shared__ CzDet s_det[2];
    const int pair = blockIdx.y, M = 2 * href, MR = M / R;
    const int j0 = blockIdx.x * CZ_C;
    if (threadIdx.x < R) {
        const int n2 = threadIdx.x / A, k1 = threadIdx.x % A;
        float sn, cs;
        sincospif(-2.0f * static_cast<float>(n2 * k1) / static_cast<float>(R), &sn, &cs);
        wt[threadIdx.x] = make_float2(cs, sn);
    }
    if (FIRST && threadIdx.x < 2) {
        const int det = min(2 * pair + static_cast<int>(threadIdx.x), ndet - 1);
        float peak;
        const CzDet c = cz_det(psd, det, href, fsamp, peak);
        s_det[threadIdx.x] = c;
        if (blockIdx.x == 0) scale[det] = cz_scale(c, peak, psd[3 * det]);
    }
    __syncthreads();
    {
        const int c = threadIdx.x & (CZ_C - 1), n2 = threadIdx.x / CZ_C;
        const int j = j0 + c;
        float2 v[A];
        if (FIRST) {
            const CzDet d0 = s_det[0], d1 = s_det[1];
            const bool two = 2 * pair + 1 < ndet;
#pragma unroll
            for (int n1 = 0; n1 < A; ++n1) {
                const int k = j + (8 * n1 + n2) * MR;
                v[n1] = make_float2(cz_gamma(d0, k, href), two ? cz_gamma(d1, k, href) : 0.f);
            }
        } else {
            const float2 *x = src + static_cast<int64_t>(pair) * M;
#pragma unroll
            for (int n1 = 0; n1 < A; ++n1) v[n1] = x[j + (8 * n1 + n2) * MR];
            // W^{r k}, r = 8 n1 + n2: the factors of n2 and of each bit of n1
            const int k = j & (Ns - 1);
            const float inv = -2.0f / (static_cast<float>(Ns) * static_cast<float>(R));     // a power of two
            float2 w[A];
            {
                float sn, cs;
                sincospif(static_cast<float>(n2 * k) * inv, &sn, &cs);
                w[0] = make_float2(cs, sn);
            }
#pragma unroll
            for (int b = 1; b < A; b <<= 1) {
                float sn, cs;
                sincospif(static_cast<float>(8 * b * k) * inv, &sn, &cs);
#pragma unroll
                for (int n1 = 0; n1 < b; ++n1) w[n1 + b] = vmul(w[n1], make_float2(cs, sn));
            }
#pragma unroll
            for (int n1 = 0; n1 < A; ++n1) v[n1] = vmul(v[n1], w[n1]);
        }
        RDft<A, false, float2>::run(v);
#pragma unroll
        for (int k1 = 0; k1 < A; ++k1) t[(n2 * A + k1) * CZ_C + c] = vmul(v[k1], wt[n2 * A + k1]);
    }
    __syncthreads();
    float2 u[IT][8];
#pragma unroll
    for (int i = 0; i < IT; ++i) {
        const int w = threadIdx.x + i * CZ_T, c = w & (CZ_C - 1), k1 = w / CZ_C;
        if (k1 >= A) continue;
#pragma unroll
        for (int n2 = 0; n2 < 8; ++n2) u[i][n2] = t[(n2 * A + k1) * CZ_C + c];
        RDft<8, false, float2>::run(u[i]);
    }
    if (FIRST) __syncthreads();                // t is reused for the outputs
    const float sc0 = LAST ? scale[2 * pair] : 0.f, sc1 = LAST ? scale[min(2 * pair + 1, ndet - 1)] : 0.f;
    float2 *y = dst + static_cast<int64_t>(pair) * M;
#pragma unroll
    for (int i = 0; i < IT; ++i) {
        const int w = threadIdx.x + i * CZ_T, c = w & (CZ_C - 1), k1 = w / CZ_C;
        if (k1 >= A) continue;
        const int j = j0 + c, k = j & (Ns - 1);
#pragma unroll
        for (int k2 = 0; k2 < 8; ++k2) {
            const int r = k1 + A * k2;
            if (FIRST) {
                t[c * (R + 1) + r] = u[i][k2];
            } else if (LAST) {
                const int d = j + r * Ns;      // Ns = M/R: j < Ns
                if (d < href) {
                    const float inv = 1.0f / static_cast<float>(M);              // a power of two
                    hout[static_cast<int64_t>(2 * pair) * href + d] = u[i][k2].x * inv * sc0;
                    if (2 * pair + 1 < ndet) hout[static_cast<int64_t>(2 * pair + 1) * href + d] = u[i][k2].y * inv * sc1;
                }
            } else {
                y[(j - k) * R + k + r * Ns] = u[i][k2];
            }
        }
    }
    if (FIRST) {
        __syncthreads();
        for (int e = threadIdx.x; e < R * CZ_C; e += CZ_T) y[j0 * R + e] = t[(e / R) * (R + 1) + (e & (R - 1))];
    }
}

// tab[x] = (H(x), G(x)) for x <= H as double-words.  The lags of a detector
// are cut into chunks of CZ_CHUNK, one CTA each: k_cz_sums adds up every
// chunk, k_cz_tables scans within its chunk from the sum of the chunks
// before it.  Fixed order of the sums throughout.
struct HG { DW h, g; };
__device__ __forceinline__ HG hg_zero() { return HG{{0.f, 0.f}, {0.f, 0.f}}; }
__device__ __forceinline__ HG hg_add(const HG &a, const HG &b) { return HG{dw_add(a.h, b.h), dw_add(a.g, b.g)}; }
__device__ __forceinline__ void hg_lag(HG &a, float h, int d) {
    const float fd = static_cast<float>(d);                 // d < 2^24: exact
    const float p = __fmul_rn(fd, h);
    a.h = dw_add2(a.h, h, 0.f);
    a.g = dw_add2(a.g, p, __fmaf_rn(fd, h, -p));
}
__device__ __forceinline__ HG hg_shfl_up(const HG &a, int o) {
    return HG{{__shfl_up_sync(0xffffffffu, a.h.h, o), __shfl_up_sync(0xffffffffu, a.h.l, o)},
              {__shfl_up_sync(0xffffffffu, a.g.h, o), __shfl_up_sync(0xffffffffu, a.g.l, o)}};
}
// Exclusive scan of one value per thread over the CTA (the total in *tot)
__device__ __forceinline__ HG hg_exscan(const HG &own, HG *s_w, HG *tot) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    HG inc = own;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const HG up = hg_shfl_up(inc, o);
        if (lane >= o) inc = hg_add(up, inc);
    }
    HG ex = hg_shfl_up(inc, 1);
    if (lane == 0) ex = hg_zero();
    if (lane == 31) s_w[warp] = inc;
    __syncthreads();
    HG base = hg_zero(), all = hg_zero();
    for (int w = 0; w < CZ_T / 32; ++w) {
        if (w == warp) base = all;
        all = hg_add(all, s_w[w]);
    }
    *tot = all;
    __syncthreads();
    return hg_add(base, ex);
}

__global__ void __launch_bounds__(CZ_T)
k_cz_sums(const float *__restrict__ hk, int href, float4 *__restrict__ csum)
{
    __shared__ HG s_w[CZ_T / 32];
    const int det = blockIdx.y, d0 = blockIdx.x * CZ_CHUNK + threadIdx.x * CZ_PER;
    const float *h = hk + static_cast<int64_t>(det) * href;
    HG s = hg_zero(), tot;
    if (d0 < href) {
#pragma unroll
        for (int i = 0; i < CZ_PER; ++i) hg_lag(s, h[d0 + i], d0 + i);
    }
    hg_exscan(s, s_w, &tot);
    if (threadIdx.x == 0) csum[det * gridDim.x + blockIdx.x] = make_float4(tot.h.h, tot.h.l, tot.g.h, tot.g.l);
}

__global__ void __launch_bounds__(CZ_T)
k_cz_tables(const float *__restrict__ hk, int href, const float4 *__restrict__ csum, float4 *__restrict__ tab)
{
    __shared__ HG s_w[CZ_T / 32];
    const int det = blockIdx.y, ch = blockIdx.x, nch = gridDim.x;
    const int d0 = ch * CZ_CHUNK + threadIdx.x * CZ_PER;
    const float *h = hk + static_cast<int64_t>(det) * href;
    float4 *t = tab + static_cast<int64_t>(det) * (href + 1);
    // the chunks before this one
    HG b = hg_zero(), base, tot;
    for (int c = threadIdx.x; c < ch; c += CZ_T) {
        const float4 v = csum[det * nch + c];
        b = hg_add(b, HG{{v.x, v.y}, {v.z, v.w}});
    }
    hg_exscan(b, s_w, &base);
    float x[CZ_PER];
    HG s = hg_zero();
    if (d0 < href) {
#pragma unroll
        for (int i = 0; i < CZ_PER; ++i) { x[i] = h[d0 + i]; hg_lag(s, x[i], d0 + i); }
    }
    HG run = hg_add(base, hg_exscan(s, s_w, &tot));
    if (d0 >= href) return;
#pragma unroll
    for (int i = 0; i < CZ_PER; ++i) {
        t[d0 + i] = make_float4(run.h.h, run.h.l, run.g.h, run.g.l);
        hg_lag(run, x[i], d0 + i);
    }
    if (d0 + CZ_PER == href) t[href] = make_float4(run.h.h, run.h.l, run.g.h, run.g.l);
}

// One CTA per detector.  xtab[det] holds, at offset L(L-1)/2, the L values
// of T_L^{-1} e_1 for L = 1..TOEP_LMAX; lvalid[det] is the largest order the
// recursion reached with a positive pivot.
//
// The 511 orders are one serial chain, so the time is the length of an
// order.  The Durbin recursion needs two dot products per order (in FP64, a
// CTA reduction of about 5 us); the Schur recursion (Kailath, "A theorem of
// I. Schur and its impact on modern signal processing", 1986) carries the
// sequences those dot products evaluate instead: with a^(k) = (1, y^(k)),
//   P_k[m] = sum_i a_i r(k + 1 + m - i),  Q_k[m] = sum_i a_{k-i} r(k + m - i),
// the reflection coefficient is alpha = -P_k[0] / Q_k[0], the pivot
// 1 + r . y^(k) is Q_k[0], and
//   P_{k+1}[m] = P_k[m+1] + alpha Q_k[m+1],  Q_{k+1}[m] = Q_k[m] + alpha P_k[m],
//   y^(k+1) = (y^(k) + alpha reversed y^(k), alpha):
// element-wise, one barrier per order.  A thread of the first half of the CTA
// owns four consecutive (P, Q) elements (an order needs one neighbour's value
// through shared memory), one of the second half two pairs (i, k - 1 - i) of
// y; both updates are two multiply-adds with one alpha, the lanes of packed
// double-words (about 2^-45 relative: the input lags carry the 2^-24 of an
// FP32 transform; FP64 issues at 1/64 of the FP32 rate on this part and one
// dependent FP64 division costs more than a whole order does here).  The
// first thread forms the next order's alpha while the others still update.
// Measured, 1 to 12 detectors: 2540 us with the dot products, 223 us with
// scalar double-words and a thread per element and per y, 176 us packed,
// 162 us with four elements a thread (an order is bound by its
// chain of dependent operations and the barrier).
constexpr int DTE = 4, DTY = 2;                    // elements, y pairs per thread
constexpr int DTH = TOEP_LMAX / DTE;               // threads of each half
constexpr int DT = 2 * DTH;
static_assert(DTH * DTY * 2 == TOEP_LMAX, "the second half covers every pair of y");

// double-words in the two lanes: x + a b with a one double-word for both
struct DW2 { PF h, l; };
__device__ __forceinline__ DW2 dw2_fma(DW2 x, DW a, DW2 b) {
    const PF ah = pdup<PF>(a.h), al = pdup<PF>(a.l);
    const PF p = pmul(ah, b.h);
    PF e = pfma(ah, b.h, pneg(p));
    e = pfma(ah, b.l, e);
    e = pfma(al, b.h, e);
    const PF s = padd(x.h, p);
    const PF bb = psub(s, x.h);
    PF r = padd(psub(x.h, psub(s, bb)), psub(p, bb));
    r = padd(r, padd(x.l, e));
    DW2 o;
    o.h = padd(s, r);
    o.l = psub(r, psub(o.h, s));
    return o;
}

// (alpha of the next order, 1 / (its pivot h(0)), the pivot) from P[0], Q[0].
// The reciprocal approximation gets one Newton step; alpha a correction.
__device__ __forceinline__ float4 schur_pivot(DW P, DW Q, float it0) {
    float inv;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(inv) : "f"(Q.h));
    inv = __fmaf_rn(__fmaf_rn(-Q.h, inv, 1.0f), inv, inv);
    const float q = __fmul_rn(-P.h, inv);
    // the remainder -P - q Q
    float r = __fmaf_rn(-q, Q.h, -P.h);
    r = __fadd_rn(r, __fmaf_rn(-q, Q.l, -P.l));
    const DW al = dw_renorm(q, __fmul_rn(r, inv));
    return make_float4(al.h, al.l, it0 * inv, Q.h);
}

__global__ void __launch_bounds__(DT)
k_toep_durbin(const float *__restrict__ hk, int href, float *__restrict__ xtab, int32_t *__restrict__ lvalid)
{
    const int det = blockIdx.x;
    const bool pq = threadIdx.x < DTH;
    const int g = pq ? threadIdx.x : threadIdx.x - DTH;
    __shared__ float4 s_pq[2][DTH + 1];                 // first (P, Q) of each thread: heads, tails; by parity
    __shared__ DW s_y[2][TOEP_LMAX];
    __shared__ float4 s_pv[2];                          // the order's pivot values (schur_pivot)
    const float *h = hk + static_cast<int64_t>(det) * href;
    float *xt = xtab + static_cast<int64_t>(det) * (TOEP_LMAX * (TOEP_LMAX + 1) / 2);
    const float t0 = h[0];
    if (!(t0 > 0.0f)) { if (threadIdx.x == 0) lvalid[det] = 0; return; }
    const float it0 = 1.0f / t0;
    DW2 V[DTE];                                         // lanes P, Q
    if (pq) {
        // order 0: P[m] = r(1 + m), Q[m] = r(m), r = h / h(0)
        const DW d0{t0, 0.f};
#pragma unroll
        for (int i = 0; i < DTE; ++i) {
            const int e = DTE * g + i;
            const DW P = dw_div(DW{e + 1 < TOEP_LMAX ? h[e + 1] : 0.f, 0.f}, d0), Q = dw_div(DW{h[e], 0.f}, d0);
            V[i] = DW2{{P.h, Q.h}, {P.l, Q.l}};
        }
        s_pq[0][g] = make_float4(V[0].h.a, V[0].h.b, V[0].l.a, V[0].l.b);
        if (g == 0) {
            s_pq[0][DTH] = s_pq[1][DTH] = make_float4(0.f, 0.f, 0.f, 0.f);
            s_pv[0] = schur_pivot(DW{V[0].h.a, V[0].l.a}, DW{V[0].h.b, V[0].l.b}, it0);
            xt[0] = it0;
        }
    }
    __syncthreads();
    int valid = 1;
    float *xk = xt;                                     // the row of order k (length k)
    for (int k = 0; k < TOEP_LMAX; ++k) {
        const int cur = k & 1;
        const float4 pv = s_pv[cur];
        if (!(pv.w > 0.0f) || pv.w > 3.0e38f) break;    // pivot not positive, or not finite
        xk += k;                                        // the row of order k + 1
        if (k > 0) valid = k + 1;
        const bool last = k + 1 >= TOEP_LMAX;
        const DW alpha{pv.x, pv.y};
        if (pq) {
            if (last) break;
            if (DTE * g < TOEP_LMAX - k) {
                const float4 n4 = s_pq[cur][g + 1];
                const DW2 nx{{n4.x, n4.y}, {n4.z, n4.w}};
#pragma unroll
                for (int i = 0; i < DTE; ++i) {
                    // (P[e+1], Q[e]) + alpha (Q[e+1], P[e])
                    const DW2 up = i + 1 < DTE ? V[i + 1] : nx;
                    V[i] = dw2_fma(DW2{{up.h.a, V[i].h.b}, {up.l.a, V[i].l.b}}, alpha,
                                   DW2{{up.h.b, V[i].h.a}, {up.l.b, V[i].l.a}});
                    if (i == 0) {
                        s_pq[cur ^ 1][g] = make_float4(V[0].h.a, V[0].h.b, V[0].l.a, V[0].l.b);
                        if (g == 0) s_pv[cur ^ 1] = schur_pivot(DW{V[0].h.a, V[0].l.a}, DW{V[0].h.b, V[0].l.b}, it0);
                    }
                }
            }
        } else {
            // order k + 1: x = (1, y^(k)) / (pivot h(0)); then y^(k+1)
#pragma unroll
            for (int i = 0; i < DTY; ++i) {
                const int t = g + i * DTH, j = k - 1 - t;       // an element and its partner
                if (t > j) break;
                const DW a = s_y[cur][t], b = s_y[cur][j];
                const DW2 n = dw2_fma(DW2{{a.h, b.h}, {a.l, b.l}}, alpha, DW2{{b.h, a.h}, {b.l, a.l}});
                s_y[cur ^ 1][t] = DW{n.h.a, n.l.a};
                if (j != t) s_y[cur ^ 1][j] = DW{n.h.b, n.l.b};
                xk[t + 1] = (a.h + a.l) * pv.z;
                if (j != t) xk[j + 1] = (b.h + b.l) * pv.z;
            }
            if (g == 0) {
                if (k > 0) xk[0] = pv.z;
                s_y[cur ^ 1][k] = alpha;
            }
        }
        if (last) break;
        __syncthreads();
    }
    if (threadIdx.x == 0) lvalid[det] = valid;
}

template <bool FIRST, bool LAST>
static void cz_fft_pass(const Plan &p, int lgR, const float2 *src, float2 *dst, const double *psd, int Ns, float *h,
                        cudaStream_t st)
{
    const int M = 2 * p.cz_href;
    const dim3 grid(M >> (lgR + 5), (p.ndet + 1) / 2);
    static_assert(CZ_C == 32, "grid");
    KTIME(TOD_KT_TOEP_KERNEL);
    switch (lgR) {
    case 5:
        k_cz_fft<4, FIRST, LAST><<<grid, CZ_T, 0, st>>>(src, dst, psd, p.ndet, p.cz_href, p.fsamp, Ns, p.czscale, h);
        break;
    case 6:
        k_cz_fft<8, FIRST, LAST><<<grid, CZ_T, 0, st>>>(src, dst, psd, p.ndet, p.cz_href, p.fsamp, Ns, p.czscale, h);
        break;
    default:
        k_cz_fft<16, FIRST, LAST><<<grid, CZ_T, 0, st>>>(src, dst, psd, p.ndet, p.cz_href, p.fsamp, Ns, p.czscale, h);
        break;
    }
}

cudaError_t launch_toeplitz_prep(const Plan &p, const double *psd, cudaStream_t st)
{
    // passes of radix 32, 64 or 128, as equal as log2(M) allows (M >= 2048:
    // two passes at least; every factor has at least five bits)
    const int M = 2 * p.cz_href;
    int lg = 0;
    while ((1 << lg) < M) ++lg;
    const int np = (lg + 6) / 7;
    const int64_t half = static_cast<int64_t>((p.ndet + 1) / 2) * M;
    float2 *buf[2] = {p.czfft, p.czfft + half};
    int cur = 0, Ns = 1;
    for (int i = 0; i < np; ++i) {
        const int lgR = (lg + np - 1 - i) / np;
        // the last pass leaves the kernels (FP32) where its output would go
        float *h = reinterpret_cast<float *>(buf[cur ^ 1]);
        if (i == 0) cz_fft_pass<true, false>(p, lgR, nullptr, buf[cur ^ 1], psd, Ns, nullptr, st);
        else if (i + 1 < np) cz_fft_pass<false, false>(p, lgR, buf[cur], buf[cur ^ 1], psd, Ns, nullptr, st);
        else cz_fft_pass<false, true>(p, lgR, buf[cur], nullptr, psd, Ns, h, st);
        cur ^= 1;
        Ns <<= lgR;
    }
    const float *h = reinterpret_cast<const float *>(buf[cur]);
    float4 *csum = reinterpret_cast<float4 *>(buf[cur ^ 1]);        // the last pass's input is free
    const int nch = (p.cz_href + CZ_CHUNK - 1) / CZ_CHUNK;
    {
        KTIME(TOD_KT_TOEP_KERNEL);
        k_cz_sums<<<dim3(nch, p.ndet), CZ_T, 0, st>>>(h, p.cz_href, csum);
    }
    {
        KTIME(TOD_KT_TOEP_KERNEL);
        k_cz_tables<<<dim3(nch, p.ndet), CZ_T, 0, st>>>(h, p.cz_href, csum, p.cztab);
    }
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    {
        KTIME(TOD_KT_TOEP_DURBIN);
        k_toep_durbin<<<p.ndet, DT, 0, st>>>(h, p.cz_href, p.xtab, p.lvalid);
    }
    return cudaGetLastError();
}

// The tables are first read by the coarse correction, after the draw's flag
// index, right-hand side and x0: beside those, on the plan's own stream, most
// of the preparation's chain (0.2 to 0.3 ms) is hidden.  Every later kernel of
// the caller's stream waits for it (the draw waits for prep_done), so nothing
// on the side stream outlives the call's work there, and psd may be freed in
// stream order as before.  After an error there is no draw to wait: the
// caller's stream is joined here (a capture keeps no loose branch; by the host
// if even the event fails), and the first error returned.
cudaError_t fork_toeplitz_prep(const Plan &p, const double *psd, cudaStream_t st)
{
    cudaError_t e = cudaEventRecord(p.prep_fork, st);
    if (e != cudaSuccess) return e;
    if ((e = cudaStreamWaitEvent(p.prep_stream, p.prep_fork, 0)) != cudaSuccess) return e;
    e = launch_toeplitz_prep(p, psd, p.prep_stream);
    const cudaError_t e2 = cudaEventRecord(p.prep_done, p.prep_stream);
    if (e == cudaSuccess) e = e2;
    if (e != cudaSuccess && (e2 != cudaSuccess || cudaStreamWaitEvent(st, p.prep_done, 0) != cudaSuccess))
        cudaStreamSynchronize(p.prep_stream);
    return e;
}

}  // namespace tg

// A3 batched DCT-II (the mirrored FFT of Sect. 4.2) as passes through
// memory, and on it A4 (gain draw), A5 (correlated-noise draw with CG gap
// filling; Eq. `gibbsstart`, Sect. 5) and A8 (TOD chi^2 and gradients).
//
// A length-n real DCT-II is an m = n/2 complex FFT of the even/odd-packed,
// reversed-odd sequence z_j = (v_{2j}, v_{2j+1}), v_i = x_{2i} (i < m),
// x_{2n-1-2i} (i >= m) (Makhoul 1980), plus a real split.  The FFT is
// four-step, m = m1 x m2, with j = j1 m2 + j2 and k = k1 + m1 k2:
//   column pass: for a tile of column pairs {c, m2-1-c}: FFTs of length m1
//     along j1, times W_m^{c k1}, written to the intermediate Y;
//     z_j and z_{m-1-j} together are the four samples x_{4j..4j+3}, so the
//     tile reads and writes whole runs of samples;
//   row pass: for a tile of row pairs {k1, m1-k1}: FFTs of length m2 along
//     k2, the real split (Z_k with Z_{m-k}) into packed orthonormal
//     coefficients (X_k, X_{n-k}) (slot 0: (X_0, X_m)), a per-mode filter,
//     the inverse split and inverse FFTs, written back to Y;
//   inverse column pass: times W_m^{-c k1}, inverse FFTs, samples out.
// The two members of a pair are the two lanes of every value the passes
// compute with (fft_reg.cuh): one packed FP32 instruction, one 16-byte
// shared-memory access and one twiddle for both.  Every tile is independent:
// a CTA holds one tile in shared memory, passes are separate grid-wide
// phases, and the intermediate goes through L2/HBM.
#include <cooperative_groups.h>
#include <type_traits>
#include "fft_reg.cuh"

namespace cgrp = cooperative_groups;

namespace tg {

// ---------------------------------------------------------------------------
// per-item context
// ---------------------------------------------------------------------------
struct TxCtx {
    TxLen L;
    float s2, inv_s2, inv_s, fscale, alpha, g;   // detector noise, detscan gain
    int q, blk, det;
    int mode;                                    // CgState mode of the detscan (n_corr)
    int64_t o;                                   // first sample of the detscan
    int64_t yb;                                  // first complex value of its Y block
    int64_t koff;                                // first flagged rank (n_corr)
    int2 fw[3];                                  // ItemFeed: items by turn, and their length indices
    int fl[3];
};

__device__ __forceinline__ void cp_async_bytes4(void *dst, const void *src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n"
                 ::"r"(static_cast<uint32_t>(__cvta_generic_to_shared(dst))), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_bytes8(void *dst, const void *src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n"
                 ::"r"(static_cast<uint32_t>(__cvta_generic_to_shared(dst))), "l"(src) : "memory");
}

// A CTA's share of a list of n items, i0, i0 + stride, ..: the items (detscan,
// tile) and the detscans' length indices, fetched by thread 0 two tiles and
// one tile ahead of their use into a ring in shared memory (two dependent
// loads, about a microsecond, in front of every tile otherwise; in registers
// the row passes spilled more).  n_corr draw of 6 x 18 detscans at 44 GHz, this
// and the single round of loads in tx_begin: 2335 -> 2196 us; chi^2 of 52M
// samples, with the spectrum's logarithm once per detscan: 2336 -> 2240 us.
struct ItemFeed {
    const int2 *__restrict__ items;
    const int32_t *__restrict__ q_tx;
    int last, k;
    __device__ __forceinline__ ItemFeed(TxCtx &X, const int2 *items_, const int32_t *q_tx_, int i0, int n)
        : items(items_), q_tx(q_tx_), last(n - 1), k(0) {
        if (threadIdx.x == 0 && i0 <= last) {
            X.fw[0] = items[i0];
            if (i0 + static_cast<int>(gridDim.x) <= last) X.fw[1] = items[i0 + static_cast<int>(gridDim.x)];
            X.fl[0] = q_tx[X.fw[0].x];
        }
    }
    // by thread 0 alone, ahead of the barrier that the others read the turn's
    // slot behind: waits for it, and fetches for the turns to come (none is
    // left in flight after the last)
    __device__ __forceinline__ void fetch(TxCtx &X, int it) const {
        asm volatile("cp.async.wait_all;\n" ::: "memory");
        const int k1 = k == 2 ? 0 : k + 1, k2 = k1 == 2 ? 0 : k1 + 1;
        const int st = static_cast<int>(gridDim.x);
        if (it + st <= last) cp_async_bytes4(&X.fl[k1], q_tx + X.fw[k1].x);
        if (it + 2 * st <= last) cp_async_bytes8(&X.fw[k2], items + it + 2 * st);
    }
    __device__ __forceinline__ void next() { k = k == 2 ? 0 : k + 1; }
};

// The item (q, blk) set up: the length plan li copied into shared memory
// (skipped when the previous item had the same length) and the detscan's
// scalars, from qsc those of the call, from cgs its CG mode and first rank.
// All threads call it; it ends with a barrier.  A tile takes 5 to 20 us, and
// its FFT waits for all of this: the loads go out together, ahead of the first
// barrier.
struct TxItem { int64_t o, koff; float4 a0, a1; int mode; };
__device__ __forceinline__ TxItem tx_load(const int64_t *__restrict__ off, int q, const float4 *__restrict__ qsc,
                                          const CgState *cgs)
{
    TxItem t;
    t.a0 = t.a1 = make_float4(0.f, 0.f, 0.f, 0.f);
    t.mode = 0;
    t.koff = 0;
    t.o = off[q];
    if (qsc) { t.a0 = qsc[2 * q]; t.a1 = qsc[2 * q + 1]; }
    if (cgs) { t.mode = cgs[q].mode; t.koff = cgs[q].koff; }
    return t;
}
__device__ __forceinline__ void tx_set(TxCtx &X, const TxLen *__restrict__ txl, const TxItem &t, int q, int blk, int li,
                                       int64_t obase, int ndet, int &cur)
{
    if (li != cur) {
        const int4 *src = reinterpret_cast<const int4 *>(txl + li);
        int4 *dst = reinterpret_cast<int4 *>(&X.L);
        for (int i = threadIdx.x; i < static_cast<int>(sizeof(TxLen) / 16); i += blockDim.x) dst[i] = src[i];
    }
    if (threadIdx.x == 0) {
        X.q = q;
        X.blk = blk;
        X.det = q % ndet;
        X.o = t.o;
        X.yb = (t.o - obase) >> 1;
        X.s2 = t.a0.x; X.inv_s2 = t.a0.y; X.inv_s = t.a0.z; X.fscale = t.a0.w;
        X.alpha = t.a1.x;
        X.g = t.a1.y;
        X.mode = t.mode;
        X.koff = t.koff;
    }
    cur = li;
    __syncthreads();
}
__device__ __forceinline__ void tx_begin(TxCtx &X, const TxLen *__restrict__ txl, int li,
                                         const int64_t *__restrict__ off, int q, int blk, int64_t obase, int ndet,
                                         int &cur, const float4 *__restrict__ qsc = nullptr,
                                         const CgState *cgs = nullptr)
{
    TxItem t{};
    if (threadIdx.x == 0) t = tx_load(off, q, qsc, cgs);
    __syncthreads();                 // earlier readers of X are done
    tx_set(X, txl, t, q, blk, li, obase, ndet, cur);
}
// the feed's next item
__device__ __forceinline__ void tx_begin(TxCtx &X, ItemFeed &feed, int it, const TxLen *__restrict__ txl,
                                         const int64_t *__restrict__ off, int64_t obase, int ndet, int &cur,
                                         const float4 *__restrict__ qsc = nullptr, const CgState *cgs = nullptr)
{
    TxItem t{};
    if (threadIdx.x == 0) {
        feed.fetch(X, it);
        t = tx_load(off, X.fw[feed.k].x, qsc, cgs);
    }
    __syncthreads();                 // earlier readers of X are done, the turn's slot is there
    const int2 w = X.fw[feed.k];
    tx_set(X, txl, t, w.x, w.y, X.fl[feed.k], obase, ndet, cur);
    feed.next();
}

// The FP32 scalars of every detscan of a call, from the FP64 noise
// parameters (and gains): (sigma0^2, 1/sigma0^2, 1/sigma0, fsamp/(2 n f_knee)),
// (alpha, g, 0, 0).  Computed once per call instead of in every tile.
__device__ __forceinline__ void det_scalars_q(const double *psd, const double *gain, const int64_t *off, int ndet,
                                              double fsamp, int q, float4 *qsc)
{
    const int det = q % ndet;
    const double sig0 = psd[3 * det], fk = psd[3 * det + 1], al = psd[3 * det + 2];
    const double n = static_cast<double>(off[q + 1] - off[q]);
    qsc[2 * q] = make_float4(static_cast<float>(sig0 * sig0), static_cast<float>(1.0 / (sig0 * sig0)),
                             static_cast<float>(1.0 / sig0), static_cast<float>(fsamp / (2.0 * n * fk)));
    qsc[2 * q + 1] = make_float4(static_cast<float>(al), gain ? static_cast<float>(gain[q]) : 1.0f, 0.f, 0.f);
}
__global__ void k_det_scalars(const double *__restrict__ psd, const double *__restrict__ gain,
                              const int64_t *__restrict__ off, int ndet, double fsamp, int q0, int q1,
                              float4 *__restrict__ qsc)
{
    const int q = q0 + blockIdx.x * blockDim.x + threadIdx.x;
    if (q < q1) det_scalars_q(psd, gain, off, ndet, fsamp, q, qsc);
}

// The SFU's approximate base-2 logarithm and exponential and reciprocal
// (PTX lg2/ex2/rcp.approx: absolute error about 2^-22 in the logarithm,
// relative about 2^-22 in the others).  Used for the per-mode noise weights,
// where their error (below 1e-6 relative in a weight) is far inside the
// transforms' FP32 budget.
__device__ __forceinline__ float sfu_lg2(float x) {
    float y;
    asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float sfu_ex2(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float sfu_rcp(float x) {
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// (f_k / f_knee)^alpha at DCT mode k >= 1, FP32 (fscale = fsamp / (2 n f_knee))
__device__ __forceinline__ float tx_fpow(int k, float fscale, float alpha) {
    return sfu_ex2(alpha * sfu_lg2(static_cast<float>(k) * fscale));
}

// twiddle block of a length: W_m1^i and W_m2^i (both lanes of a pair), then
// plain complex values: hq W_4n^{k1}, W_4n^{m1 k2}, hq W_4n^{5 k1},
// W_4n^{5 m1 k2} (hq = 1/(2 sqrt(m)): the real split's scale, the same both
// ways), W_m^{64 i}, W_m^i (i < 64)
template <class V> struct PairOf;
template <> struct PairOf<CF2> { typedef float2 Z; };
template <> struct PairOf<CD2> { typedef double2 Z; };
__device__ __forceinline__ float2 zmul(float2 a, float2 b) {
    return make_float2(fmaf(-a.y, b.y, a.x * b.x), fmaf(a.x, b.y, a.y * b.x));
}
__device__ __forceinline__ double2 zmul(double2 a, double2 b) {
    return make_double2(fma(-a.y, b.y, a.x * b.x), fma(a.x, b.y, a.y * b.x));
}
template <class V, class Z> __device__ __forceinline__ V vtwo(Z a, Z b) {
    return vmake<V>(pset(a.x, b.x), pset(a.y, b.y));
}
template <class V> struct TwB {
    typedef typename PairOf<V>::Z Z;
    const V *tw1, *tw2;
    const Z *sa1, *sb1, *sa5, *sb5, *t4hi, *t4lo;
    __device__ __forceinline__ TwB(const Z *base, const TxLen &L) {
        tw1 = reinterpret_cast<const V *>(base);
        tw2 = tw1 + L.m1;
        sa1 = reinterpret_cast<const Z *>(tw2 + L.m2);
        sb1 = sa1 + L.m1;
        sa5 = sb1 + L.m2;
        sb5 = sa5 + L.m1;
        t4hi = sb5 + L.m2;
        t4lo = t4hi + L.m / 64 + 1;
    }
    __device__ __forceinline__ Z w4(int r) const { return zmul(vld(t4hi + (r >> 6)), vld(t4lo + (r & 63))); }
};

// flagged-sample mask (bit u: sample t + u) of samples t..t+cnt-1, cnt <= 4
__device__ __forceinline__ uint32_t flag_bits(const uint32_t *__restrict__ fl, int64_t t, int cnt) {
    const int64_t w = t >> 5;
    const int b = static_cast<int>(t & 31);
    uint32_t v = __ldg(fl + w) >> b;
    if (b + cnt > 32) v |= __ldg(fl + w + 1) << (32 - b);
    return v & ((1u << cnt) - 1u);
}

// The four samples of unit j (x_{4j..4j+3}; two at the centre j = m-1-j):
// z_j = (x0, x2), z_{m-1-j} = (x3, x1).
__device__ __forceinline__ float4 ld4(const float *__restrict__ x, int64_t t, bool centre) {
    const float2 a = __ldg(reinterpret_cast<const float2 *>(x + t));
    if (centre) return make_float4(a.x, a.y, 0.f, 0.f);
    const float2 b = __ldg(reinterpret_cast<const float2 *>(x + t + 2));
    return make_float4(a.x, a.y, b.x, b.y);
}

// Asynchronous global -> shared copies (cp.async, Ampere and later): every
// copy of a tile is in flight at once; cp_wait ends them (a barrier must
// follow before other threads read the tile).
__device__ __forceinline__ void cp_async(PF *dst, const float2 *src) {
    const uint32_t d = static_cast<uint32_t>(__cvta_generic_to_shared(dst));
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(d), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async(PD *dst, const double2 *src) {
    const uint32_t d = static_cast<uint32_t>(__cvta_generic_to_shared(dst));
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(d), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_wait() { asm volatile("cp.async.wait_all;\n" ::: "memory"); }

// ---------------------------------------------------------------------------
// The intermediate Y of a detscan (m complex values): row pairs {p, m1 - p}
// (p = 0: rows 0 and m1/2), two planes of m2 values each: the pair's real
// parts (re_a, re_b), then its imaginary parts.  With m1 odd row 0 has no
// partner: it is stored last, as plain complex values.
// ---------------------------------------------------------------------------
__device__ __forceinline__ int y_plane(int m1, int p) { return (m1 & 1) ? 2 * (p - 1) : 2 * p; }

// ---------------------------------------------------------------------------
// column tiles: column pairs {c, m2-1-c}, c in [p0, p0 + np); the pair's two
// columns are the two lanes; element (j1, i) at j1 TP + i.  TP is a power of
// two dividing TX_T: thread t keeps pair t mod TP and takes rows r0 = t / TP,
// r0 + rstep, .. (at most TX_ROWS of the m1/2 rows, since TP m1 <= TX_TILE/2).
// Unit j = j1 m2 + c holds z_j and its mirror z_{m-1-j}, which lies in the
// other lane at row m1-1-j1: the two units of row j1 fill both lanes of the
// elements j1 and m1-1-j1.
// ---------------------------------------------------------------------------
constexpr int TX_ROWS = 4;
// CTAs per SM of the column passes and the chi^2 passes: at three (80
// registers) the four rows of loads that a thread keeps in flight spill; two
// at 128 registers are faster (82M samples: k_gain_cols 359 -> 343 us,
// k_nc_gather_final 476 -> 418; chi^2 rows of 52M 1093 -> 840 us, there with a
// grid that is resident at once).  The scatter, which holds no samples, keeps
// three (the draw of 72 x 225k samples without its preparation 2009 us; 2102
// with two).
constexpr int TX_CTAS_COL = 2;
struct ColThread {
    int m, m1, m2, TP, np, i, c, c2, r0, rstep, m1h;
    __device__ __forceinline__ ColThread(const TxLen &L, int blk) {
        m = L.m; m1 = L.m1; m2 = L.m2; TP = L.TP;
        const int p0 = blk * TP;
        np = min(TP, L.P2 - p0);
        i = threadIdx.x & (TP - 1);
        r0 = threadIdx.x >> L.lgW;
        rstep = TX_T >> L.lgW;
        c = i < np ? p0 + i : -1;          // -1: no column
        c2 = m2 - 1 - c;
        m1h = (m1 + 1) >> 1;
    }
    __device__ __forceinline__ int row(int r) const { return r0 + r * rstep; }
    __device__ __forceinline__ bool mid(int j1) const { return 2 * j1 == m1 - 1; }
    __device__ __forceinline__ bool centre(int j1) const { return mid(j1) && c == c2; }
    __device__ __forceinline__ bool second(int j1) const { return !mid(j1) && c != c2; }   // unit (j1, c2) too
};

// The flag bits of a thread's units, loaded ahead of the transform (all
// loads in flight together): nibble 2r + u is unit u (column c, c2) of the
// thread's r-th row.  Zero without flags (fl null) or without a column.
__device__ __forceinline__ uint32_t unit_flags(const ColThread &C, const uint32_t *__restrict__ fl, int64_t o)
{
    uint32_t nib = 0;
    if (!fl || C.c < 0) return nib;
#pragma unroll
    for (int r = 0; r < TX_ROWS; ++r) {
        const int j1 = C.row(r);
        if (j1 >= C.m1h) continue;
        const int64_t t = o + 4 * static_cast<int64_t>(j1 * C.m2);
        nib |= flag_bits(fl, t + 4 * C.c, C.centre(j1) ? 2 : 4) << (8 * r);
        if (C.second(j1)) nib |= flag_bits(fl, t + 4 * C.c2, 4) << (8 * r + 4);
    }
    return nib;
}

// The second half of a forward column pass, the tile in b0: the column FFTs,
// the four-step twiddle W_m^{c k1}, and the tile out to Y.
template <class V>
__device__ __forceinline__ void col_forward_out(const TxCtx &X, const ColThread &C, V *b0, V *b1,
                                                typename PairOf<V>::Z *__restrict__ Y,
                                                const typename PairOf<V>::Z *__restrict__ twb)
{
    typedef typename PairOf<V>::Z Z;
    const int m1 = C.m1, m2 = C.m2, TP = C.TP;
    __syncthreads();
    const TwB<V> T(twb, X.L);
    V *R = sp_transform<false, TX_T, true>(b0, b1, m1, X.L.s1, X.L.nr1, X.L.lgW, 0, T.tw1);
    if (C.c < 0) return;
    Z *Yq = Y + X.yb;
    // W_m^{c p} from the table at the thread's first row, then by steps of
    // W_m^{c rstep} (at most three products); row m1 - p takes W_m2^c conj(W_m^{c p})
    const V wc = vtwo<V>(Z{vld(T.tw2 + C.c).x.a, vld(T.tw2 + C.c).y.a}, Z{vld(T.tw2 + C.c2).x.a, vld(T.tw2 + C.c2).y.a});
    V w = C.r0 < m1 ? vtwo<V>(T.w4(C.c * C.r0), T.w4(C.c2 * C.r0)) : vzero<V>();
    const V wstep = C.rstep < m1 ? vtwo<V>(T.w4(C.c * C.rstep), T.w4(C.c2 * C.rstep)) : vzero<V>();
#pragma unroll
    for (int r = 0; r < TX_ROWS; ++r) {
        const int p = C.row(r);
        if (p >= C.m1h) break;
        const V za = vmul(sld(R + p * TP + C.i), w);
        if (p == 0 && (m1 & 1)) {
            Z *y = Yq + static_cast<int64_t>(m1 - 1) * m2;
            y[C.c] = Z{za.x.a, za.y.a};
            if (C.c2 != C.c) y[C.c2] = Z{za.x.b, za.y.b};
        } else {
            const int pr = p ? m1 - p : m1 >> 1;
            const V wr = p ? vmul<true>(wc, w) : vtwo<V>(T.w4(C.c * pr), T.w4(C.c2 * pr));
            const V zb = vmul(sld(R + pr * TP + C.i), wr);
            Z *y = Yq + static_cast<int64_t>(y_plane(m1, p)) * m2;
            y[C.c] = Z{za.x.a, zb.x.a};
            y[m2 + C.c] = Z{za.y.a, zb.y.a};
            if (C.c2 != C.c) {
                y[C.c2] = Z{za.x.b, zb.x.b};
                y[m2 + C.c2] = Z{za.y.b, zb.y.b};
            }
        }
        w = vmul(w, wstep);
    }
}

// Forward column pass.  D = ld(j, centre, fb) issues a unit's loads (UNR rows
// per thread at a time; fb: the unit's flag bits, from fl at sample o + 4j,
// read ahead), val(D, j, centre, fb, wa, wb, v) gives its samples
// v[0..3] (two at the centre).  With NORM, pre(tile) first fills the tile
// and wa, wb are the tile's values at z_j and z_{m-1-j}.
template <bool NORM, int UNR, class V, class Pre, class Ld, class Val>
__device__ __forceinline__ void col_forward(const TxCtx &X, V *b0, V *b1, typename PairOf<V>::Z *__restrict__ Y,
                                            const typename PairOf<V>::Z *__restrict__ twb,
                                            const uint32_t *__restrict__ fl, Pre pre, Ld ld, Val val)
{
    typedef typename PairOf<V>::Z Z;
    typedef typename VecT<V>::S S;
    const ColThread C(X.L, X.blk);
    const int m1 = C.m1, m2 = C.m2, TP = C.TP;
    if (C.c < 0)
        for (int j1 = C.r0; j1 < m1; j1 += C.rstep) sst(b0 + j1 * TP + C.i, vzero<V>());
    pre(b0);
    const uint32_t fnib = unit_flags(C, fl, X.o);
    if (NORM) __syncthreads();
    if (C.c >= 0) {
#pragma unroll
        for (int r1 = 0; r1 < TX_ROWS; r1 += UNR) {
            decltype(ld(0, false, 0u)) D[UNR][2];
#pragma unroll
            for (int u = 0; u < UNR; ++u) {
                const int j1 = C.row(r1 + u);
                if (j1 >= C.m1h) continue;
                const uint32_t fb = fnib >> (8 * (r1 + u));
                D[u][0] = ld(j1 * m2 + C.c, C.centre(j1), fb & 15u);
                if (C.second(j1)) D[u][1] = ld(j1 * m2 + C.c2, false, (fb >> 4) & 15u);
            }
#pragma unroll
            for (int u = 0; u < UNR; ++u) {
                const int j1 = C.row(r1 + u);
                if (j1 >= C.m1h) continue;
                const uint32_t fb = fnib >> (8 * (r1 + u));
                V *ea = b0 + j1 * TP + C.i, *eb = b0 + (m1 - 1 - j1) * TP + C.i;
                V na = vzero<V>(), nb = na;
                if (NORM) { na = sld(ea); nb = sld(eb); }
                S va[4], vb[4];
                val(D[u][0], j1 * m2 + C.c, C.centre(j1), fb & 15u, Z{na.x.a, na.y.a}, Z{nb.x.b, nb.y.b}, va);
                if (C.mid(j1)) {
                    sst(ea, C.c == C.c2 ? vmake<V>(pset(va[0], va[0]), pset(va[1], va[1]))
                                        : vmake<V>(pset(va[0], va[3]), pset(va[2], va[1])));
                    continue;
                }
                if (C.c == C.c2) {
#pragma unroll
                    for (int s = 0; s < 4; ++s) vb[s] = va[s];
                } else {
                    val(D[u][1], j1 * m2 + C.c2, false, (fb >> 4) & 15u, Z{na.x.b, na.y.b}, Z{nb.x.a, nb.y.a}, vb);
                }
                sst(ea, vmake<V>(pset(va[0], vb[0]), pset(va[2], vb[2])));
                sst(eb, vmake<V>(pset(vb[3], va[3]), pset(vb[1], va[1])));
            }
        }
    }
    col_forward_out(X, C, b0, b1, Y, twb);
}

// Inverse column pass: the tile's Y values (every load of a thread in
// flight), the conjugate twiddle, inverse FFT of the columns; then for every
// unit out(D, j, centre, v, fb) with v its samples, D = ld(j, centre, fb) issued
// ahead of the transform (the flag bits are read while the tile loads).  Where
// again() then asks for it, the thread's units are gone through once more, as
// redo(D, j, centre, v, fb).
struct NoRedo {
    __device__ __forceinline__ bool again() const { return false; }
};
template <class V, class Ld, class Out, class Redo = NoRedo>
__device__ __forceinline__ void col_inverse(const TxCtx &X, V *b0, V *b1,
                                            const typename PairOf<V>::Z *__restrict__ Y,
                                            const typename PairOf<V>::Z *__restrict__ twb,
                                            const uint32_t *__restrict__ fl, Ld ld, Out out, Redo redo = Redo())
{
    typedef typename PairOf<V>::Z Z;
    typedef typename VecT<V>::S S;
    const ColThread C(X.L, X.blk);
    const int m1 = C.m1, m2 = C.m2, TP = C.TP;
    const TwB<V> T(twb, X.L);
    uint32_t fnib = 0;
    if (C.c < 0) {
        for (int k1 = C.r0; k1 < m1; k1 += C.rstep) sst(b0 + k1 * TP + C.i, vzero<V>());
    } else {
        const Z *Yq = Y + X.yb;
        Z A[TX_ROWS][4];
#pragma unroll
        for (int r = 0; r < TX_ROWS; ++r) {
            const int p = C.row(r);
            if (p >= C.m1h) break;
            if (p == 0 && (m1 & 1)) {
                const Z *y = Yq + static_cast<int64_t>(m1 - 1) * m2;
                A[r][0] = __ldcg(&y[C.c]);
                A[r][1] = __ldcg(&y[C.c2]);
            } else {
                const Z *y = Yq + static_cast<int64_t>(y_plane(m1, p)) * m2;
                A[r][0] = __ldcg(&y[C.c]);
                A[r][1] = __ldcg(&y[C.c2]);
                A[r][2] = __ldcg(&y[m2 + C.c]);
                A[r][3] = __ldcg(&y[m2 + C.c2]);
            }
        }
        fnib = unit_flags(C, fl, X.o);
        const V wc = vtwo<V>(Z{vld(T.tw2 + C.c).x.a, vld(T.tw2 + C.c).y.a},
                             Z{vld(T.tw2 + C.c2).x.a, vld(T.tw2 + C.c2).y.a});
        V w = C.r0 < m1 ? vtwo<V>(T.w4(C.c * C.r0), T.w4(C.c2 * C.r0)) : vzero<V>();
        const V wstep = C.rstep < m1 ? vtwo<V>(T.w4(C.c * C.rstep), T.w4(C.c2 * C.rstep)) : vzero<V>();
#pragma unroll
        for (int r = 0; r < TX_ROWS; ++r) {
            const int p = C.row(r);
            if (p >= C.m1h) break;
            if (p == 0 && (m1 & 1)) {
                sst(b0 + C.i, vmul<true>(vtwo<V>(A[r][0], A[r][1]), w));
            } else {
                const int pr = p ? m1 - p : m1 >> 1;
                const V wr = p ? vmul<true>(wc, w) : vtwo<V>(T.w4(C.c * pr), T.w4(C.c2 * pr));
                const V za = vmake<V>(pset(A[r][0].x, A[r][1].x), pset(A[r][2].x, A[r][3].x));
                const V zb = vmake<V>(pset(A[r][0].y, A[r][1].y), pset(A[r][2].y, A[r][3].y));
                sst(b0 + p * TP + C.i, vmul<true>(za, w));
                sst(b0 + pr * TP + C.i, vmul<true>(zb, wr));
            }
            w = vmul(w, wstep);
        }
    }
    // the units' loads, in flight through the transform
    decltype(ld(0, false, 0u)) D[TX_ROWS][2];
    if (C.c >= 0) {
#pragma unroll
        for (int r = 0; r < TX_ROWS; ++r) {
            const int j1 = C.row(r);
            if (j1 >= C.m1h) continue;
            const uint32_t fb = fnib >> (8 * r);
            D[r][0] = ld(j1 * m2 + C.c, C.centre(j1), fb & 15u);
            if (C.second(j1)) D[r][1] = ld(j1 * m2 + C.c2, false, (fb >> 4) & 15u);
        }
    }
    __syncthreads();
    V *R = sp_transform<true, TX_T, true>(b0, b1, m1, X.L.s1, X.L.nr1, X.L.lgW, 0, T.tw1);
    if (C.c < 0) return;
    // the units of the thread's r-th row
    const auto units = [&](int r, const auto &Da, const auto &Db, auto &fn) {
        const int j1 = C.row(r);
        const uint32_t fb = fnib >> (8 * r);
        const V ea = sld(R + j1 * TP + C.i), eb = sld(R + (m1 - 1 - j1) * TP + C.i);
        if (C.centre(j1)) {
            const S v[4] = {ea.x.a, ea.y.a, S(0), S(0)};
            fn(Da, j1 * m2 + C.c, true, v, fb & 15u);
        } else {
            const S v[4] = {ea.x.a, eb.y.b, ea.y.a, eb.x.b};
            fn(Da, j1 * m2 + C.c, false, v, fb & 15u);
        }
        if (C.second(j1)) {
            const S v[4] = {ea.x.b, eb.y.a, ea.y.b, eb.x.a};
            fn(Db, j1 * m2 + C.c2, false, v, (fb >> 4) & 15u);
        }
    };
#pragma unroll
    for (int r = 0; r < TX_ROWS; ++r)
        if (C.row(r) < C.m1h) units(r, D[r][0], D[r][1], out);
    if constexpr (!std::is_same<Redo, NoRedo>::value) {
        if (!redo.again()) return;
#pragma unroll 1
        for (int r = 0; C.row(r) < C.m1h; ++r) {
            const int j1 = C.row(r);
            const uint32_t fb = fnib >> (8 * r);
            const auto Da = ld(j1 * m2 + C.c, C.centre(j1), fb & 15u);
            const auto Db = C.second(j1) ? ld(j1 * m2 + C.c2, false, (fb >> 4) & 15u) : Da;
            units(r, Da, Db, redo);
        }
    }
}

// ---------------------------------------------------------------------------
// row tiles: row pairs p in [r0, r0 + nr); the pair's rows are the two lanes
// (lane a: row p; lane b: row m1 - p, or m1/2 for p = 0, absent when m1 is
// odd); element (p, k2) at (p - r0) m2p + k2.
//
// Row pass.  The tile's rows in from Y, forward row FFTs, then pre(nubuf)
// (NORM: a second tile-sized buffer filled with a value per mode; a barrier
// follows), the real split, Y' = f(k0, k1, mask, Y, nu) for the packed slots
// of modes k0, k1 (lanes; Y = (X_k, X_{n-k}), or (X_0, X_m) for k = 0; mask
// bit l: lane l holds a mode not met before, for sums; nu the second buffer's
// values), the inverse split, inverse row FFTs, and the rows back to Y.
//
// Split: with e1 = W_4n^k, e5 = W_4n^{5k} and Za = Z_k, Zb = Z_{m-k},
//   P = e1 (Za + conj Zb), Q = e5 (-i)(Za - conj Zb),
//   Y_k = hq conj(P + Q), Y_{m-k} = hq e^{i pi/4} (P - Q)
// (the twiddles of m - k are those of k rotated by e^{-i pi/4}); the inverse
// runs it backwards with the same factors.  Mode m - k of row p lies in
// row m1 - p at m2 - 1 - k2, the other lane of that element, so one thread
// takes elements k2 and m2 - 1 - k2 together: lane a the pair based in row p,
// lane b the pair based in row m1 - p.  Rows 0 and m1/2 pair with themselves
// (p = 0).  The conjugates of P and Q are carried, so no sign is flipped.
//
// stop(), asked of every thread after the modes: where one says so the pass
// ends there, Y as it was, and returns false.
// ---------------------------------------------------------------------------
struct NeverStop {};
// A CTA's threads as groups of whole warps, a power of two of threads at least
// n wide: a loop over the n elements of each of several rows takes the rows by
// groups, so that short rows keep the CTA at work (one row after the other left
// seven of eight warps idle in the split at m2 = 64: FP64 chi^2 of 16 x 4096
// samples 955 us, 432 so; the gain of 800 x 2000 89 us, 74 so).  A warp has one
// row: groups of fewer threads than a warp cost the long rows registers (gain of
// 72 x 225k samples 325 us, 308 so, 311 with one row after the other).
struct RowGroups {
    int first, step, row, nrow;
    __device__ __forceinline__ explicit RowGroups(int n) {
        const int lg = min(8, max(5, 32 - __clz(n - 1)));
        first = threadIdx.x & ((1 << lg) - 1);
        step = 1 << lg;
        row = __shfl_sync(0xffffffffu, static_cast<int>(threadIdx.x >> lg), 0);      // uniform, and known to be
        nrow = __shfl_sync(0xffffffffu, TX_T >> lg, 0);
    }
};
static_assert(TX_T == 256, "a group is at most the CTA");

template <bool NORM, class V, class Pre, class F, class Stop = NeverStop>
__device__ __forceinline__ bool row_pass(const TxCtx &X, V *b0, V *b1, typename PairOf<V>::Z *__restrict__ Y,
                                         const typename PairOf<V>::Z *__restrict__ twb, Pre pre, F f,
                                         Stop stop = Stop())
{
    typedef typename PairOf<V>::Z Z;
    typedef typename VecT<V>::S S;
    typedef typename VecT<V>::C C;
    const int m = X.L.m, m1 = X.L.m1, m2 = X.L.m2, m2p = X.L.m2p, TR = X.L.TR;
    const int p0 = X.blk * TR, nr = min(TR, X.L.P1 - p0);
    const bool odd = m1 & 1;
    const RowGroups W(m2), H((m2 + 1) >> 1);
    Z *Yq = Y + X.yb;
    for (int pl = W.row; pl < TR; pl += W.nrow) {
        const int p = p0 + pl;
        V *dst = b0 + pl * m2p;
        if (pl >= nr) {
            for (int k2 = W.first; k2 < m2; k2 += W.step) sst(dst + k2, vzero<V>());
        } else if (odd && p == 0) {
            const Z *y = Yq + static_cast<int64_t>(m1 - 1) * m2;
            for (int k2 = W.first; k2 < m2; k2 += W.step) {
                const Z z = y[k2];
                sst(dst + k2, vmake<V>(pset(z.x, S(0)), pset(z.y, S(0))));
            }
        } else {
            const Z *y = Yq + static_cast<int64_t>(y_plane(m1, p)) * m2;
            for (int k2 = W.first; k2 < m2; k2 += W.step) {
                cp_async(&dst[k2].x, y + k2);
                cp_async(&dst[k2].y, y + m2 + k2);
            }
        }
    }
    cp_wait();
    __syncthreads();
    const TwB<V> T(twb, X.L);
    V *R = sp_transform<false, TX_T, false>(b0, b1, m2, X.L.s2, X.L.nr2, X.L.lgS, m2p, T.tw2);
    V *Fr = R == b0 ? b1 : b0;
    if (NORM) {
        pre(Fr);
        __syncthreads();
    }
    const C h = pdup<C>(static_cast<S>(0.70710678118654752440));
    for (int pl = H.row; pl < nr; pl += H.nrow) {
        const int p = p0 + pl;
        const int ra = p, rb = p ? m1 - p : (odd ? 0 : m1 >> 1);
        V *t = R + pl * m2p, *nt = Fr + pl * m2p;
        const V A1 = vtwo<V>(vld(T.sa1 + ra), vld(T.sa1 + rb)), A5 = vtwo<V>(vld(T.sa5 + ra), vld(T.sa5 + rb));
        const int cnt = p ? (m2 + 1) >> 1 : (m2 >> 1) + 1;
        for (int k2 = H.first; k2 < cnt; k2 += H.step) {
            const int q = m2 - 1 - k2;                       // partner element (p = 0: lane b)
            const int q0 = k2 ? m2 - k2 : 0;                 // p = 0: lane a's partner
            int mb = 3, mp = 3;
            V Za = sld(t + k2), Zb, nua = vzero<V>(), nub = nua;
            if (p) {
                Zb = vswap(sld(t + q));
                if (NORM) { nua = sld(nt + k2); nub = vswap(sld(nt + q)); }
                if (q == k2) mb = mp = 1;
            } else {
                const int qb = max(q, 0);
                Zb = vmake<V>(pset(t[q0].x.a, t[qb].x.b), pset(t[q0].y.a, t[qb].y.b));
                if (NORM) {
                    nua = sld(nt + k2);
                    nub = vmake<V>(pset(nt[q0].x.a, nt[qb].x.b), pset(nt[q0].y.a, nt[qb].y.b));
                }
                mb = 1 | ((!odd && k2 <= q) ? 2 : 0);
                mp = ((k2 && q0 != k2) ? 1 : 0) | ((!odd && k2 < q) ? 2 : 0);
            }
            const Z s1 = vld(T.sb1 + k2), s5 = vld(T.sb5 + k2);
            const V e1 = vmul(A1, vtwo<V>(s1, s1)), e5 = vmul(A5, vtwo<V>(s5, s5));
            const V cP = vmul<true>(vmake<V>(padd(Za.x, Zb.x), psub(Zb.y, Za.y)), e1);
            const V cQ = vmul<true>(vmake<V>(padd(Za.y, Zb.y), psub(Za.x, Zb.x)), e5);
            V Ya = vadd(cP, cQ);
            const V cm = vsub(cP, cQ);
            V Yb = vmake<V>(pmul(h, padd(cm.x, cm.y)), pmul(h, psub(cm.x, cm.y)));
            const int k0 = ra + m1 * k2, k1 = rb + m1 * k2;
            if (k0 == 0) {
                const S s0f = static_cast<S>(X.L.s0_fwd);
                Ya.x.a = (Za.x.a + Za.y.a) * s0f;
                Ya.y.a = (Za.x.a - Za.y.a) * s0f;
            }
            Ya = f(k0, k1, mb, Ya, nua);
            Yb = f(m - k0, m - k1, mp, Yb, nub);
            const V cn = vmake<V>(pmul(h, padd(Yb.x, Yb.y)), pmul(h, psub(Yb.x, Yb.y)));
            const V cs = vmul(vadd(Ya, cn), e1), cd = vmul(vsub(Ya, cn), e5);
            Za = vmake<V>(padd(cs.x, cd.y), psub(cd.x, cs.y));
            Zb = vmake<V>(psub(cs.x, cd.y), padd(cd.x, cs.y));
            if (p) {
                sst(t + k2, Za);
                if (q != k2) sst(t + q, vswap(Zb));
            } else {
                if (k2 == 0) {
                    const S s0i = static_cast<S>(X.L.s0_inv), v0 = Ya.x.a * s0i, vm = Ya.y.a * s0i;
                    Za.x.a = static_cast<S>(0.5) * (v0 + vm);
                    Za.y.a = static_cast<S>(0.5) * (v0 - vm);
                }
                t[k2].x.a = Za.x.a;
                t[k2].y.a = Za.y.a;
                if (mp & 1) { t[q0].x.a = Zb.x.a; t[q0].y.a = Zb.y.a; }
                if (mb & 2) { t[k2].x.b = Za.x.b; t[k2].y.b = Za.y.b; }
                if (mp & 2) { t[q].x.b = Zb.x.b; t[q].y.b = Zb.y.b; }
            }
        }
    }
    if constexpr (std::is_same<Stop, NeverStop>::value) __syncthreads();
    else if (__syncthreads_or(stop())) return false;
    const V *Ri = sp_transform<true, TX_T, false>(R, Fr, m2, X.L.s2, X.L.nr2, X.L.lgS, m2p, T.tw2);
    for (int pl = W.row; pl < nr; pl += W.nrow) {
        const int p = p0 + pl;
        const V *src = Ri + pl * m2p;
        if (odd && p == 0) {
            Z *y = Yq + static_cast<int64_t>(m1 - 1) * m2;
            for (int k2 = W.first; k2 < m2; k2 += W.step) y[k2] = Z{src[k2].x.a, src[k2].y.a};
        } else {
            Z *y = Yq + static_cast<int64_t>(y_plane(m1, p)) * m2;
            for (int k2 = W.first; k2 < m2; k2 += W.step) {
                const V v = sld(src + k2);
                y[k2] = Z{v.x.a, v.x.b};
                y[m2 + k2] = Z{v.y.a, v.y.b};
            }
        }
    }
    return true;
}

// ---------------------------------------------------------------------------
// CTA reductions: FP32 double-word partials, warps merged by shuffles, the
// warp results added in FP64 in a fixed order by thread 0.
// ---------------------------------------------------------------------------
__device__ __forceinline__ Acc2 acc_merge_tx(const Acc2 &a, const Acc2 &b) {
    Acc2 r = a;
    acc_add(r, b.s);
    r.c = __fadd_rn(r.c, b.c);
    return r;
}
__device__ __forceinline__ Acc2 warp_acc(Acc2 x) {
#pragma unroll
    for (int o = 16; o; o >>= 1) {
        Acc2 y;
        y.s = __shfl_xor_sync(0xffffffffu, x.s, o);
        y.c = __shfl_xor_sync(0xffffffffu, x.c, o);
        x = acc_merge_tx(x, y);
    }
    return x;
}
// NV values per thread summed over the CTA; the totals land in out[0..NV)
// (shared) for every thread after the call.  s_red holds NV * TX_T/32.
template <int NV>
__device__ __forceinline__ void block_sums(const Acc2 (&a)[NV], double *s_red, double *out) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
#pragma unroll
    for (int v = 0; v < NV; ++v) {
        const Acc2 w = warp_acc(a[v]);
        if (lane == 0) s_red[v * (TX_T / 32) + warp] = acc_value(w);
    }
    __syncthreads();
    if (threadIdx.x < NV) {
        double t = 0.0;
        for (int w = 0; w < TX_T / 32; ++w) t += s_red[threadIdx.x * (TX_T / 32) + w];
        out[threadIdx.x] = t;
    }
    __syncthreads();
}
template <int NV>
__device__ __forceinline__ void block_sums_d(const double (&a)[NV], double *s_red, double *out) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
#pragma unroll
    for (int v = 0; v < NV; ++v) {
        double x = a[v];
#pragma unroll
        for (int o = 16; o; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
        if (lane == 0) s_red[v * (TX_T / 32) + warp] = x;
    }
    __syncthreads();
    if (threadIdx.x < NV) {
        double t = 0.0;
        for (int w = 0; w < TX_T / 32; ++w) t += s_red[threadIdx.x * (TX_T / 32) + w];
        out[threadIdx.x] = t;
    }
    __syncthreads();
}

// ===========================================================================
// A4: gain.  a = sum_{k>=1} shat_k^2 / P_k (row pass), u = C^T(shat / P) and
// b = sum_t M_t d_t u_t (inverse column pass): b = sum_k shat_k dhat_k / P_k.
// ===========================================================================
struct GainTx {
    const float *d, *s;
    const uint32_t *flags;
    const double *psd;
    const int64_t *off;
    const TxLen *txl;
    const int32_t *q_tx;
    const float2 *tw;
    const int2 *items;
    int item0, nitems;
    int ndet;
    double fsamp;
    int64_t obase;
    float2 *Y;
    double *part;                 // [item][4]
    const float4 *qsc;            // per-detscan FP32 scalars of the call
};

// A pair of FP32 double-word accumulators (one per lane)
struct PAcc { PF s, c; };
__device__ __forceinline__ PAcc pacc_zero() { return PAcc{{0.f, 0.f}, {0.f, 0.f}}; }
__device__ __forceinline__ void pacc_add(PAcc &a, PF v) {
    const PF s = padd(a.s, v);
    const PF bb = psub(s, a.s);
    const PF e = padd(psub(a.s, psub(s, bb)), psub(v, bb));
    a.s = s;
    a.c = padd(a.c, e);
}
__device__ __forceinline__ void pacc_add_prod(PAcc &a, PF x, PF y) {
    const PF p = pmul(x, y);
    const PF e = pfma(x, y, pneg(p));
    pacc_add(a, p);
    a.c = padd(a.c, e);
}
__device__ __forceinline__ Acc2 pacc_total(const PAcc &a) { return acc_merge_tx(Acc2{a.s.a, a.c.a}, Acc2{a.s.b, a.c.b}); }
// the lanes of v that mask names (the others zero)
__device__ __forceinline__ PF pmask(PF v, int mask) { return PF{(mask & 1) ? v.a : 0.f, (mask & 2) ? v.b : 0.f}; }
__device__ __forceinline__ PD pmask(PD v, int mask) { return PD{(mask & 1) ? v.a : 0.0, (mask & 2) ? v.b : 0.0}; }

__global__ void __launch_bounds__(TX_T, TX_CTAS_COL) k_gain_cols(GainTx a)
{
    extern __shared__ __align__(16) CF2 tx_smem[];
    __shared__ TxCtx X;
    CF2 *b0 = tx_smem, *b1 = tx_smem + TX_PAIRS;
    int cur = -1;
    ItemFeed feed(X, a.items + a.item0, a.q_tx, blockIdx.x, a.nitems);
    for (int it = blockIdx.x; it < a.nitems; it += gridDim.x) {
        tx_begin(X, feed, it, a.txl, a.off, a.obase, a.ndet, cur);
        const float *sq = a.s + X.o;
        col_forward<false, 4>(X, b0, b1, a.Y, a.tw + X.L.twb, a.flags, [](CF2 *) {},
                    [&](int j, bool ctr, uint32_t) { return ld4(sq, 4 * static_cast<int64_t>(j), ctr); },
                    [&](const float4 &x, int, bool, uint32_t fb, float2, float2, float (&v)[4]) {
                        v[0] = (fb & 1) ? 0.f : x.x;
                        v[1] = (fb & 2) ? 0.f : x.y;
                        v[2] = (fb & 4) ? 0.f : x.z;
                        v[3] = (fb & 8) ? 0.f : x.w;
                    });
    }
}

__global__ void __launch_bounds__(TX_T, 3) k_gain_rows(GainTx a)
{
    extern __shared__ __align__(16) CF2 tx_smem[];
    __shared__ TxCtx X;
    __shared__ double s_red[TX_T / 32], s_out[1];
    CF2 *b0 = tx_smem, *b1 = tx_smem + TX_PAIRS;
    int cur = -1;
    ItemFeed feed(X, a.items + a.item0, a.q_tx, blockIdx.x, a.nitems);
    for (int it = blockIdx.x; it < a.nitems; it += gridDim.x) {
        tx_begin(X, feed, it, a.txl, a.off, a.obase, a.ndet, cur, a.qsc);
        const float fscale = X.fscale, alpha = X.alpha, s2 = X.s2;
        const int n = X.L.n, m = X.L.m;
        PAcc sum = pacc_zero();
        const auto weight = [&](int k) { return sfu_rcp(s2 * (1.0f + tx_fpow(k, fscale, alpha))); };
        row_pass<false>(X, b0, b1, a.Y, a.tw + X.L.twb, [](CF2 *) {}, [&](int k0, int k1, int mask, CF2 S, CF2) {
            const PF wa = pset(k0 ? weight(k0) : 0.f, k1 ? weight(k1) : 0.f);
            const PF wb = pset(weight(k0 ? n - k0 : m), weight(k1 ? n - k1 : m));
            const CF2 W{pmul(S.x, wa), pmul(S.y, wb)};
            if (mask != 3) { S.x = pmask(S.x, mask); S.y = pmask(S.y, mask); }
            pacc_add_prod(sum, S.x, W.x);
            pacc_add_prod(sum, S.y, W.y);
            return W;
        });
        const Acc2 sa[1] = {pacc_total(sum)};
        block_sums<1>(sa, s_red, s_out);
        if (threadIdx.x == 0) a.part[4 * static_cast<int64_t>(a.item0 + it)] = s_out[0];
    }
}

__global__ void __launch_bounds__(TX_T, TX_CTAS_COL) k_gain_colsinv(GainTx a)
{
    extern __shared__ __align__(16) CF2 tx_smem[];
    __shared__ TxCtx X;
    __shared__ double s_red[TX_T / 32], s_out[1];
    CF2 *b0 = tx_smem, *b1 = tx_smem + TX_PAIRS;
    int cur = -1;
    ItemFeed feed(X, a.items + a.item0, a.q_tx, blockIdx.x, a.nitems);
    for (int it = blockIdx.x; it < a.nitems; it += gridDim.x) {
        tx_begin(X, feed, it, a.txl, a.off, a.obase, a.ndet, cur);
        const float *dq = a.d + X.o;
        PAcc sum = pacc_zero();
        col_inverse(X, b0, b1, a.Y, a.tw + X.L.twb, a.flags, [&](int j, bool ctr, uint32_t) {
            return ld4(dq, 4 * static_cast<int64_t>(j), ctr);
        }, [&](const float4 &dv, int, bool, const float (&v)[4], uint32_t fb) {
            // at the centre the last two samples are zero
            pacc_add_prod(sum, pset((fb & 1) ? 0.f : dv.x, (fb & 2) ? 0.f : dv.y), pset(v[0], v[1]));
            pacc_add_prod(sum, pset((fb & 4) ? 0.f : dv.z, (fb & 8) ? 0.f : dv.w), pset(v[2], v[3]));
        });
        const Acc2 sb[1] = {pacc_total(sum)};
        block_sums<1>(sb, s_red, s_out);
        if (threadIdx.x == 0) a.part[4 * static_cast<int64_t>(a.item0 + it) + 1] = s_out[0];
    }
}

// The sum over items [i0, i1) of value k of their partials, one warp (lanes
// stride, then a tree: a fixed order); every lane gets it.  A thread adding
// the items one after the other waits out an FP64 add (about 40 ns here)
// for each.
__device__ __forceinline__ double item_sum(const double *__restrict__ part, int i0, int i1, int k)
{
    double t = 0.0;
    for (int i = i0 + static_cast<int>(threadIdx.x & 31); i < i1; i += 32) t += part[4 * static_cast<int64_t>(i) + k];
#pragma unroll
    for (int o = 16; o; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    return t;
}

// Per detscan (one warp): a and b summed over its row and column items, then
// the draw g ~ N(b/a, 1/a); a <= 0 (no usable sample) or a non-finite sum
// gives g = 0 and TOD_ERR_ARG.
__global__ void __launch_bounds__(256) k_gain_fin(const double *__restrict__ rpart, const double *__restrict__ cpart,
                                                  const int32_t *__restrict__ row_off,
                                                  const int32_t *__restrict__ col_off, int q0, int q1, tod_rng rng,
                                                  int mode, double *g_out, double *mu_out, double *sig_out,
                                                  int32_t *status)
{
    const int q = q0 + static_cast<int>((blockIdx.x * blockDim.x + threadIdx.x) >> 5);
    if (q >= q1) return;
    const double A = item_sum(rpart, row_off[q], row_off[q + 1], 0);
    const double B = item_sum(cpart, col_off[q], col_off[q + 1], 1);
    if (threadIdx.x & 31) return;
    if (!(A > 0.0) || !isfinite(A) || !isfinite(B)) {
        set_status(status, q, TOD_ERR_ARG);
        g_out[q] = 0.0;
        if (mu_out) mu_out[q] = 0.0;
        if (sig_out) sig_out[q] = 0.0;
        return;
    }
    const double mu = B / A, sg = 1.0 / sqrt(A);
    double z = 0.0;
    if (mode == TOD_MODE_DRAW) {
        const uint64_t it = rng.gibbs_iter_dev ? *rng.gibbs_iter_dev : rng.gibbs_iter;
        const u64x4 wv = philox4x64(0, static_cast<uint64_t>(q), 0, it, rng.seed, rng.band);
        const double u1 = (static_cast<double>(wv.x[0] >> 11) + 0.5) * 1.1102230246251565e-16;
        const double u2 = (static_cast<double>(wv.x[1] >> 11) + 0.5) * 1.1102230246251565e-16;
        z = sqrt(-2.0 * log(u1)) * cospi(2.0 * u2);
    }
    g_out[q] = mu + z * sg;
    if (mu_out) mu_out[q] = mu;
    if (sig_out) sig_out[q] = sg;
}

// ===========================================================================
// A8: chi^2 with n_corr marginalised and its gradients, FP32 or FP64
// transforms.  rhat = C(M(d - g s)); L = 1/2 sum_{k>=1} [rhat^2/P + ln P];
// dL/dtheta = 1/2 sum_k (1/P - rhat^2/P^2) dP/dtheta (row pass);
// v = M C^T(rhat / P), dL/dg = -<M s, v> (inverse column pass).
// ===========================================================================
// the samples of unit j of s in the pass's precision (float or double s)
template <class S>
__device__ __forceinline__ void ld4s(const void *x, int64_t t, bool centre, S (&v)[4]) {
    if constexpr (sizeof(S) == sizeof(float)) {
        const float4 a = ld4(static_cast<const float *>(x), t, centre);
        v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w;
    } else {
        const double *p = static_cast<const double *>(x) + t;     // t even: 16-byte aligned
        const double2 a = __ldg(reinterpret_cast<const double2 *>(p));
        v[0] = a.x; v[1] = a.y; v[2] = 0.0; v[3] = 0.0;
        if (!centre) {
            const double2 b = __ldg(reinterpret_cast<const double2 *>(p + 2));
            v[2] = b.x; v[3] = b.y;
        }
    }
}

template <class V> struct Chi2Tx {
    typedef typename PairOf<V>::Z Z;
    const float *d;
    const void *s;                // float or double [N] as V
    const double *gain;
    const uint32_t *flags;
    const double *psd;
    const int64_t *off;
    const TxLen *txl;
    const int32_t *q_tx;
    const Z *tw;
    const int2 *items;
    int item0, nitems;
    int ndet;
    double fsamp;
    int64_t obase;
    Z *Y;
    double *part;                 // [item][4]
    double2 *par;                 // [nq][2] (sigma0, ln(fsamp/(2 n f_knee))), (alpha, f_knee): the row pass's
    void *v_out;                  // float or double [N] (global sample index), or null
    bool v_al;                    // v_out aligned to two values
};

// Sums over a CTA's modes or samples, one per lane: FP32 double-words (2^-44
// relative; FP64 adds issue at 1/64 of the FP32 rate) or FP64.  A double-word
// sum reaches 3.4e38, and an infinite term leaves NaN in its tail: what is
// not finite the caller adds up again in FP64.
template <class C> struct LaneSum;
template <> struct LaneSum<PF> {
    PAcc a = pacc_zero();
    __device__ __forceinline__ void add(PF v) { pacc_add(a, v); }
    __device__ __forceinline__ void add_prod(PF x, PF y) { pacc_add_prod(a, x, y); }
    __device__ __forceinline__ double total() const { return acc_value(pacc_total(a)); }
};
struct WideSum {                          // FP32 terms added in FP64
    double a = 0.0;
    __device__ __forceinline__ void add(PF v) { a += static_cast<double>(v.a) + static_cast<double>(v.b); }
    __device__ __forceinline__ double total() const { return a; }
};
template <> struct LaneSum<PD> {
    double a = 0.0;
    __device__ __forceinline__ void add(PD v) { a += v.a + v.b; }
    __device__ __forceinline__ void add_prod(PD x, PD y) { a += x.a * y.a + x.b * y.b; }
    __device__ __forceinline__ double total() const { return a; }
};

template <class V>
__global__ void __launch_bounds__(TX_T, sizeof(V) == sizeof(CF2) ? TX_CTAS_COL : 1) k_chi2_cols(Chi2Tx<V> a)
{
    typedef typename VecT<V>::S S;
    typedef typename PairOf<V>::Z Z;
    extern __shared__ __align__(16) CD2 tx_smem64[];
    __shared__ TxCtx X;
    V *b0 = reinterpret_cast<V *>(tx_smem64), *b1 = b0 + TX_PAIRS;
    int cur = -1;
    ItemFeed feed(X, a.items + a.item0, a.q_tx, blockIdx.x, a.nitems);
    for (int it = blockIdx.x; it < a.nitems; it += gridDim.x) {
        tx_begin(X, feed, it, a.txl, a.off, a.obase, a.ndet, cur);
        const double gq = a.gain[X.q];
        const S g = static_cast<S>(gq);
        const float *dq = a.d + X.o;
        const int64_t o = X.o;
        struct U4 { float4 dv; S sx[4]; };
        col_forward<false, 2>(X, b0, b1, a.Y, a.tw + X.L.twb, a.flags, [](V *) {},
                    [&](int j, bool ctr, uint32_t) {
                        const int64_t t = 4 * static_cast<int64_t>(j);
                        U4 D;
                        D.dv = ld4(dq, t, ctr);
                        ld4s<S>(a.s, o + t, ctr, D.sx);
                        return D;
                    },
                    [&](const U4 &D, int, bool, uint32_t fb, Z, Z, S (&v)[4]) {
                        v[0] = (fb & 1) ? S(0) : static_cast<S>(D.dv.x) - g * D.sx[0];
                        v[1] = (fb & 2) ? S(0) : static_cast<S>(D.dv.y) - g * D.sx[1];
                        v[2] = (fb & 4) ? S(0) : static_cast<S>(D.dv.z) - g * D.sx[2];
                        v[3] = (fb & 8) ? S(0) : static_cast<S>(D.dv.w) - g * D.sx[3];
                    });
        if (X.blk == 0 && threadIdx.x == 0) {      // once per detscan: a chain of FP64 operations, 40 ns each
            const double *ps = a.psd + 3 * X.det;
            a.par[2 * X.q] = make_double2(ps[0], log(a.fsamp / (2.0 * X.L.n * ps[1])));
            a.par[2 * X.q + 1] = make_double2(ps[2], ps[1]);
        }
    }
}

// The weights and gradient factors of the modes in the pass's precision, the
// sums as LaneSum.
template <class V>
__global__ void __launch_bounds__(TX_T, sizeof(V) == sizeof(CF2) ? TX_CTAS_COL : 1) k_chi2_rows(Chi2Tx<V> a)
{
    typedef typename VecT<V>::S S;
    typedef typename VecT<V>::C C;
    extern __shared__ __align__(16) CD2 tx_smem64[];
    __shared__ TxCtx X;
    constexpr bool kF64 = sizeof(S) == sizeof(double);
    __shared__ double s_red[4 * (TX_T / 32)], s_out[4];
    V *b0 = reinterpret_cast<V *>(tx_smem64), *b1 = b0 + TX_PAIRS;
    int cur = -1;
    ItemFeed feed(X, a.items + a.item0, a.q_tx, blockIdx.x, a.nitems);
    for (int it = blockIdx.x; it < a.nitems; it += gridDim.x) {
        tx_begin(X, feed, it, a.txl, a.off, a.obase, a.ndet, cur);
        const double2 *par = a.par + 2 * X.q;                        // written by k_chi2_cols
        const double2 pa = __ldg(par), pb = __ldg(par + 1);
        const S sig0 = static_cast<S>(pa.x), lfs = static_cast<S>(pa.y), al = static_cast<S>(pb.x);
        const S fk = static_cast<S>(pb.y);
        const S s2 = sig0 * sig0;
        const S d1 = S(2) / sig0, d2 = -s2 * al / fk;
        const int n = X.L.n, m = X.L.m;
        // the modes k0, k1 of coefficients r: r / P, their terms added; in
        // FP64 all but ln P (P in the mask's lanes, 1 elsewhere, left in Pm).  The
        // sums: 2 L, dL/dsigma0, dL/dfknee, dL/dalpha
        const auto mode_terms = [&](auto &sum, int k0, int k1, int mask, C r, C &Pm) -> C {
            // ln(f/fk) = ln k + ln(fsamp/(2 n fk)); P = s2 (1 + e^{alpha ln(f/fk)})
            const C lr = pset(log(static_cast<S>(max(k0, 1))) + lfs, log(static_cast<S>(max(k1, 1))) + lfs);
            const C pw = pset(exp(al * lr.a), exp(al * lr.b));
            const C P = pmul(pdup<C>(s2), padd(pw, pdup<C>(S(1))));
            const C iP = pset(S(1) / P.a, S(1) / P.b);
            const C rP = pmul(r, iP), r2P = pmul(r, rP);
            const C hh = pmul(pdup<C>(S(0.5)), psub(iP, pmul(r2P, iP)));     // 1/2 (1/P - r^2/P^2)
            const C sp = pmul(pdup<C>(s2), pmul(pw, lr));
            C t0 = r2P, tl, t1 = pmul(hh, pmul(P, pdup<C>(d1)));
            C t2 = pmul(hh, pmul(pw, pdup<C>(d2))), t3 = pmul(hh, sp);
            if constexpr (kF64) Pm = mask == 3 ? P : pset((mask & 1) ? P.a : S(1), (mask & 2) ? P.b : S(1));
            else tl = pset(log(P.a), log(P.b));
            if (mask != 3) {
                t0 = pmask(t0, mask); t1 = pmask(t1, mask);
                t2 = pmask(t2, mask); t3 = pmask(t3, mask);
                if constexpr (!kF64) tl = pmask(tl, mask);
            }
            sum[0].add(t0);
            if constexpr (!kF64) sum[0].add(tl);
            sum[1].add(t1);
            sum[2].add(t2);
            sum[3].add(t3);
            return rP;
        };
        const auto modes = [&](auto &sum, int k0, int k1, int mask, V Rv) {
            const int on = (k0 ? 1 : 0) | (k1 ? 2 : 0);         // the offset mode does not enter
            C P0, P1;
            const C x = mode_terms(sum, k0, k1, mask & on, Rv.x, P0);
            const C y = mode_terms(sum, k0 ? n - k0 : m, k1 ? n - k1 : m, mask, Rv.y, P1);
            if constexpr (kF64) {
                // one logarithm for the four modes (an FP64 one takes about 30
                // operations, at 1/64 of the FP32 rate: 25 scans of 4 x 65536,
                // rows 2168 -> 1815 us) of the product, which leaves the range
                // only past 1e72 a mode: then one each (also where half the
                // product is below 2^-963, which the other half may hide)
                const S pa = P0.a * P0.b, pb = P1.a * P1.b, pr = pa * pb;
                if (min(__double2hiint(pa), __double2hiint(pb)) > 0x03c00000 && pr > S(1e-290) && pr < S(1e290)) {
                    sum[0].add(pset(log(pr), S(0)));
                } else {
                    sum[0].add(pset(log(P0.a), log(P0.b)));
                    sum[0].add(pset(log(P1.a), log(P1.b)));
                }
            }
            return vmake<V>(on == 3 ? x : pmask(x, on), y);
        };
        double acc[4];
        const auto totals = [&](auto &sum) {
#pragma unroll
            for (int k = 0; k < 4; ++k) acc[k] = (k == 0 ? 0.5 : 1.0) * sum[k].total();
        };
        const auto none = [](V *) {};
        LaneSum<C> sum[4];
        const auto pass = [&](int k0, int k1, int mask, V Rv, V) { return modes(sum, k0, k1, mask, Rv); };
        if constexpr (kF64) {
            row_pass<false>(X, b0, b1, a.Y, a.tw + X.L.twb, none, pass);
            totals(sum);
        } else {
            // a sum past FP32's range, or an infinite term: the tile once more,
            // its terms added in FP64
            const auto stop = [&] {
                totals(sum);
                return !(isfinite(acc[0]) && isfinite(acc[1]) && isfinite(acc[2]) && isfinite(acc[3]));
            };
            if (!row_pass<false>(X, b0, b1, a.Y, a.tw + X.L.twb, none, pass, stop)) {
                WideSum wide[4];
                row_pass<false>(X, b0, b1, a.Y, a.tw + X.L.twb, none,
                                [&](int k0, int k1, int mask, V Rv, V) { return modes(wide, k0, k1, mask, Rv); });
                totals(wide);
            }
        }
        block_sums_d<4>(acc, s_red, s_out);
        if (threadIdx.x < 4) a.part[4 * static_cast<int64_t>(a.item0 + it) + threadIdx.x] = s_out[threadIdx.x];
    }
}

template <class V>
__global__ void __launch_bounds__(TX_T, sizeof(V) == sizeof(CF2) ? TX_CTAS_COL : 1) k_chi2_colsinv(Chi2Tx<V> a)
{
    typedef typename VecT<V>::S S;
    typedef typename VecT<V>::C C;
    extern __shared__ __align__(16) CD2 tx_smem64[];
    __shared__ TxCtx X;
    __shared__ double s_red[TX_T / 32], s_out[1];
    V *b0 = reinterpret_cast<V *>(tx_smem64), *b1 = b0 + TX_PAIRS;
    int cur = -1;
    ItemFeed feed(X, a.items + a.item0, a.q_tx, blockIdx.x, a.nitems);
    for (int it = blockIdx.x; it < a.nitems; it += gridDim.x) {
        tx_begin(X, feed, it, a.txl, a.off, a.obase, a.ndet, cur);
        const int64_t o = X.o;
        LaneSum<C> sum;
        struct U4 { S sx[4]; };
        const auto load = [&](int j, bool ctr, uint32_t) {
            U4 D;
            ld4s<S>(a.s, o + 4 * static_cast<int64_t>(j), ctr, D.sx);
            return D;
        };
        const auto unit = [&](const U4 &D, int j, bool ctr, const S (&u)[4], uint32_t fb) {
            const S v[4] = {(fb & 1) ? S(0) : u[0], (fb & 2) ? S(0) : u[1], (fb & 4) ? S(0) : u[2],
                            (fb & 8) ? S(0) : u[3]};
            // at the centre the last two samples are zero
            sum.add_prod(pset(D.sx[0], D.sx[1]), pset(v[0], v[1]));
            sum.add_prod(pset(D.sx[2], D.sx[3]), pset(v[2], v[3]));
            if (a.v_out) {
                typedef typename PairOf<V>::Z Z;
                Z *vo = reinterpret_cast<Z *>(static_cast<S *>(a.v_out) + o + 4 * static_cast<int64_t>(j));
                if (a.v_al) {
                    vo[0] = Z{v[0], v[1]};
                    if (!ctr) vo[1] = Z{v[2], v[3]};
                } else {
                    S *vs = reinterpret_cast<S *>(vo);
                    for (int s = 0; s < (ctr ? 2 : 4); ++s) vs[s] = v[s];
                }
            }
        };
        double total;
        if constexpr (sizeof(S) == sizeof(float)) {
            // a sum past FP32's range, or with a product past it: formed again in FP64
            struct Again {
                LaneSum<C> *sum;
                double *t;
                __device__ __forceinline__ bool again() const {
                    *t = sum->total();
                    if (isfinite(*t)) return false;
                    *t = 0.0;
                    return true;
                }
                __device__ __forceinline__ void operator()(const U4 &D, int, bool, const S (&u)[4], uint32_t fb) const {
                    for (int s = 0; s < 4; ++s) *t += static_cast<double>(D.sx[s]) * ((fb >> s & 1) ? 0.0 : u[s]);
                }
            };
            total = 0.0;                              // threads without a column add nothing
            col_inverse(X, b0, b1, a.Y, a.tw + X.L.twb, a.flags, load, unit, Again{&sum, &total});
        } else {
            col_inverse(X, b0, b1, a.Y, a.tw + X.L.twb, a.flags, load, unit);
            total = sum.total();
        }
        const double acc[1] = {-total};
        block_sums_d<1>(acc, s_red, s_out);
        if (threadIdx.x == 0) a.part[4 * static_cast<int64_t>(a.item0 + it) + 1] = s_out[0];
    }
}

// Per detscan (one warp): chi^2 and its PSD-parameter terms from the row
// items, the gain derivative from the column items.
__global__ void __launch_bounds__(256) k_chi2_fin(const double *__restrict__ rpart, const double *__restrict__ cpart,
                                                  const int32_t *__restrict__ row_off,
                                                  const int32_t *__restrict__ col_off, int q0, int q1,
                                                  double *chi2_q, double *dgain, double *dpsd_q)
{
    const int q = q0 + static_cast<int>((blockIdx.x * blockDim.x + threadIdx.x) >> 5);
    if (q >= q1) return;
    double s[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) s[k] = item_sum(rpart, row_off[q], row_off[q + 1], k);
    const double g = item_sum(cpart, col_off[q], col_off[q + 1], 1);
    if (threadIdx.x & 31) return;
    chi2_q[q] = s[0];
    dgain[q] = g;
    for (int k = 0; k < 3; ++k) dpsd_q[3 * static_cast<int64_t>(q) + k] = s[k + 1];
}

// Band totals, one CTA each in a fixed order (strided lanes, then a tree):
// chi^2 (CTA 0) and the PSD gradient of every detector (CTA 1 + det).  One
// thread adding 800 detscans, and 200 for each of 12 derivatives, took 225 us.
__global__ void __launch_bounds__(256) k_chi2_total(const double *__restrict__ chi2_q,
                                                    const double *__restrict__ dpsd_q, int nq, int ndet,
                                                    double *total, double *dpsd_det)
{
    __shared__ double s_red[3 * (TX_T / 32)], s_out[3];
    double t[3] = {0.0, 0.0, 0.0};
    if (blockIdx.x == 0) {
        for (int q = threadIdx.x; q < nq; q += TX_T) t[0] += chi2_q[q];
    } else {
        for (int q = static_cast<int>(blockIdx.x) - 1 + ndet * static_cast<int>(threadIdx.x); q < nq; q += ndet * TX_T)
#pragma unroll
            for (int k = 0; k < 3; ++k) t[k] += dpsd_q[3 * static_cast<int64_t>(q) + k];
    }
    block_sums_d<3>(t, s_red, s_out);
    if (blockIdx.x == 0) { if (threadIdx.x == 0) total[0] = s_out[0]; }
    else if (threadIdx.x < 3) dpsd_det[3 * (blockIdx.x - 1) + threadIdx.x] = s_out[threadIdx.x];
}

// ===========================================================================
// A5: correlated noise.  x0 = B^{-1} b with B = C^T diag(phi + 1/sigma0^2) C
// is the draw of a gap-free detscan; flagged detscans then solve the Schur
// complement S y = E^T x0, S = sigma0^2 I - E^T B^{-1} E
// = E^T C^T diag(gamma) C E (E: flagged samples), by CG preconditioned with
// the exact inverse of each gap's Toeplitz block, and x = x0 + B^{-1} E y
// (Woodbury): x = A^{-1} b, A = B - E E^T / sigma0^2.  A detscan with every
// sample flagged has A = C^T diag(phi) C: x is its exact spectral solution
// (the offset mode, unconstrained, set to zero).
//
// One launch per pass, and one cooperative launch (grid barriers between its
// passes) for the CG iterations past the launched ones.
// ===========================================================================
struct NcorrTx {
    const float *d, *s;
    const double *gain;
    const uint32_t *flags;
    const double *psd;
    const int64_t *off;
    const TxLen *txl;
    const int32_t *q_tx;
    const float2 *tw;
    const int2 *colitems, *rowitems;
    const int32_t *col_off, *row_off;
    int q0, q1;                   // detscan range of this launch
    int ndet;
    double fsamp;
    tod_rng rng;
    int mode;
    float tol;
    int maxit;
    float *x_out;
    int32_t *iters;
    int32_t *status;
    float *spec_out;
    const float *xtab;            // Toeplitz inverses' first columns per detector (null: no preconditioner)
    const int32_t *lvalid;
    // coarse correction (null czsz: none)
    const float4 *cztab;          // [ndet][href + 1] prefix sums of the gap kernel
    int href;
    int32_t *gbpos;               // [nq][TX_GBMAX] first sample of each block
    float *czsz;                  // [czcap][TX_CZJ] S Z rows by flagged rank
    int64_t czcap;
    float *czl;                   // [nq][2 TX_CBMAX][TX_CZB + 1] factor of E
    // scratch
    float2 *Y;                    // launch-range intermediate
    int64_t *wpre;                // [range words + 1]
    int64_t *chunk;               // [gridDim + 1]
    CgState *cgs;                 // [nq]
    int2 *gblk;                   // [nq][TX_GBMAX]
    int32_t *gnb;                 // [nq]
    float *cgv;                   // [5][cgcap]
    int64_t cgcap;
    int32_t *count;               // [3] active detscans (alternating), arrivals at the list
    float4 *qsc;                  // [nq][2] per-detscan FP32 scalars, written in the index phase
    // the detscans a CG pass works on, in order, with the running counts of
    // their column and row items: list[0] = n, then q[nq], col[nq + 1], row[nq + 1]
    int32_t *list;
};
__device__ __forceinline__ int32_t *nl_q(const NcorrTx &a) { return a.list + 1; }
__device__ __forceinline__ int32_t *nl_col(const NcorrTx &a) { return a.list + 1 + (a.q1 - a.q0); }
__device__ __forceinline__ int32_t *nl_row(const NcorrTx &a) { return a.list + 2 + 2 * (a.q1 - a.q0); }

struct CgVec { float *y, *r, *p, *q, *z; };
__device__ __forceinline__ CgVec cg_vecs(const NcorrTx &a) {
    CgVec v;
    v.y = a.cgv; v.r = v.y + a.cgcap; v.p = v.r + a.cgcap; v.q = v.p + a.cgcap; v.z = v.q + a.cgcap;
    return v;
}

// flagged samples of the launch range before sample t (global index)
__device__ __forceinline__ int64_t flag_rank(const uint32_t *__restrict__ fl, const int64_t *__restrict__ wpre,
                                             int64_t w_lo, int64_t obase, int64_t t) {
    const int64_t w = t >> 5;
    uint32_t bits = __ldg(fl + w) & ((1u << (t & 31)) - 1u);
    if (w == w_lo) bits &= ~((1u << (obase & 31)) - 1u);
    return wpre[w - w_lo] + __popc(bits);
}

// Shared memory of the n_corr kernel besides the tiles.
struct NcShared {
    TxCtx X;
    double red[4 * (TX_T / 32)];
    double out[4];
    int3 scan[TX_T / 32 + 1];
    int gbeg[TX_GBMAX], gend[TX_GBMAX];
    int next, grab[TX_T / 64];         // gap blocks handed out to the warp pairs
    int64_t i64[2];
    double d64[4];
    int flag;
};

// Exclusive scan of one int3 per thread over the CTA; total gets the sum.
__device__ int3 cta_exscan3(int3 v, int3 *s_w, int3 &total)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int3 inc = v;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const int x = __shfl_up_sync(0xffffffffu, inc.x, d);
        const int y = __shfl_up_sync(0xffffffffu, inc.y, d);
        const int z = __shfl_up_sync(0xffffffffu, inc.z, d);
        if (lane >= d) { inc.x += x; inc.y += y; inc.z += z; }
    }
    if (lane == 31) s_w[warp] = inc;
    __syncthreads();
    if (warp == 0) {
        constexpr int NW = TX_T / 32;
        const int3 w = lane < NW ? s_w[lane] : make_int3(0, 0, 0);
        int3 wi = w;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const int x = __shfl_up_sync(0xffffffffu, wi.x, d);
            const int y = __shfl_up_sync(0xffffffffu, wi.y, d);
            const int z = __shfl_up_sync(0xffffffffu, wi.z, d);
            if (lane >= d) { wi.x += x; wi.y += y; wi.z += z; }
        }
        __syncwarp();
        if (lane < NW) s_w[lane] = make_int3(wi.x - w.x, wi.y - w.y, wi.z - w.z);
        if (lane == NW - 1) s_w[NW] = wi;
    }
    __syncthreads();
    const int3 b = s_w[warp];
    total = s_w[TX_T / 32];
    __syncthreads();
    return make_int3(b.x + inc.x - v.x, b.y + inc.y - v.y, b.z + inc.z - v.z);
}

// Flagged-sample prefix over the range's flag words, in chunks of words per
// CTA: count (chunk totals), then write (the per-word prefix from the totals
// of the chunks before).
struct FlagChunk {
    int64_t w_lo, nw, c0, c1, t0, per, obase, oend;
};
__device__ __forceinline__ FlagChunk flag_chunk(const NcorrTx &a) {
    FlagChunk f;
    f.obase = a.off[a.q0];
    f.oend = a.off[a.q1];
    f.w_lo = f.obase >> 5;
    f.nw = ((f.oend + 31) >> 5) - f.w_lo;
    const int64_t cw = (f.nw + gridDim.x - 1) / gridDim.x;
    f.c0 = min(f.nw, static_cast<int64_t>(blockIdx.x) * cw);
    f.c1 = min(f.nw, f.c0 + cw);
    f.per = (f.c1 - f.c0 + TX_T - 1) / TX_T;
    f.t0 = f.c0 + threadIdx.x * f.per;
    return f;
}
// word w_lo + i restricted to the range
__device__ __forceinline__ uint32_t flag_word(const NcorrTx &a, const FlagChunk &f, int64_t i) {
    const int64_t w = f.w_lo + i;
    uint32_t b = __ldg(a.flags + w);
    const int64_t base = w << 5;
    if (base < f.obase) b &= ~0u << static_cast<int>(f.obase - base);
    if (base + 32 > f.oend) b &= (f.oend - base >= 32) ? ~0u : ((1u << static_cast<int>(f.oend - base)) - 1u);
    return b;
}
__device__ void nc_flag_count(const NcorrTx &a, NcShared &S)
{
    const FlagChunk f = flag_chunk(a);
    int mine = 0;
    for (int64_t i = f.t0; i < min(f.c1, f.t0 + f.per); ++i) mine += __popc(flag_word(a, f, i));
    int3 tot3;
    cta_exscan3(make_int3(mine, 0, 0), S.scan, tot3);
    if (threadIdx.x == 0) a.chunk[blockIdx.x] = tot3.x;
}
__device__ void nc_flag_write(const NcorrTx &a, NcShared &S)
{
    const FlagChunk f = flag_chunk(a);
    // the chunks before this one: at most a grid's worth of counts, summed by
    // the CTA (a serial scan of them by one thread took 20-50 us)
    long long before = 0;
    for (int c = threadIdx.x; c < static_cast<int>(blockIdx.x); c += TX_T) before += __ldg(a.chunk + c);
#pragma unroll
    for (int o = 16; o; o >>= 1) before += __shfl_xor_sync(0xffffffffu, before, o);
    __shared__ long long s_before[TX_T / 32];
    if ((threadIdx.x & 31) == 0) s_before[threadIdx.x >> 5] = before;
    int mine = 0;
    for (int64_t i = f.t0; i < min(f.c1, f.t0 + f.per); ++i) mine += __popc(flag_word(a, f, i));
    int3 tot3;
    const int3 ex = cta_exscan3(make_int3(mine, 0, 0), S.scan, tot3);       // barriers: s_before is complete
    int64_t run = ex.x;
#pragma unroll
    for (int w = 0; w < TX_T / 32; ++w) run += s_before[w];
    if (blockIdx.x == gridDim.x - 1 && threadIdx.x == 0) a.wpre[f.nw] = run + tot3.x;
    for (int64_t i = f.t0; i < min(f.c1, f.t0 + f.per); ++i) {
        a.wpre[i] = run;
        run += __popc(flag_word(a, f, i));
    }
}

// Phase 2 (per detscan): flagged count and rank offset, CG mode, and the
// gap blocks of the preconditioner (gaps split into blocks of at most lmax).
__device__ void nc_detscan_index(const NcorrTx &a, NcShared &S, int q)
{
    const int64_t obase = a.off[a.q0];
    const int64_t w_lo = obase >> 5;
    const int64_t o = a.off[q], n = a.off[q + 1] - o;
    const int det = q % a.ndet;
    if (threadIdx.x == 0) {
        const int64_t k0 = flag_rank(a.flags, a.wpre, w_lo, obase, o);
        const int64_t k1 = (a.off[q + 1] == a.off[a.q1] && ((a.off[q + 1] & 31) == 0))
                               ? a.wpre[((a.off[q + 1]) >> 5) - w_lo]
                               : flag_rank(a.flags, a.wpre, w_lo, obase, a.off[q + 1]);
        S.i64[0] = k0;
        S.i64[1] = k1 - k0;
    }
    __syncthreads();
    const int64_t koff = S.i64[0];
    const int K = static_cast<int>(S.i64[1]);
    // gaps: runs of flagged samples
    const int64_t wb0 = o >> 5, wb1 = (o + n - 1) >> 5;
    const int nw = static_cast<int>(wb1 - wb0 + 1);
    const int per = (nw + TX_T - 1) / TX_T;
    auto wbits = [&](int wi) -> uint32_t {
        if (wi < 0 || wi >= nw) return 0u;
        uint32_t bits = __ldg(a.flags + wb0 + wi);
        const int64_t base = ((wb0 + wi) << 5) - o;
        if (base < 0) bits &= ~0u << static_cast<int>(-base);
        if (base + 32 > n) bits &= (n - base >= 32) ? ~0u : ((1u << static_cast<int>(n - base)) - 1u);
        return bits;
    };
    int3 mine = make_int3(0, 0, 0);
    for (int i = 0; i < per; ++i) {
        const int wi = threadIdx.x * per + i;
        if (wi >= nw) break;
        const uint32_t bits = wbits(wi), prev = wbits(wi - 1) >> 31, next = wbits(wi + 1) & 1u;
        mine.y += __popc(bits & ~((bits << 1) | prev));
        mine.z += __popc(bits & ~((bits >> 1) | (next << 31)));
    }
    int3 tot3;
    const int3 ex = cta_exscan3(mine, S.scan, tot3);
    const int ngap = tot3.y;
    if (ngap <= TX_GBMAX) {
        int gpos = ex.y, epos = ex.z;
        for (int i = 0; i < per; ++i) {
            const int wi = threadIdx.x * per + i;
            if (wi >= nw) break;
            const uint32_t bits = wbits(wi), prev = wbits(wi - 1) >> 31, next = wbits(wi + 1) & 1u;
            uint32_t st = bits & ~((bits << 1) | prev), en = bits & ~((bits >> 1) | (next << 31));
            const int base = static_cast<int>(((wb0 + wi) << 5) - o);
            while (st) { S.gbeg[gpos++] = base + __ffs(st) - 1; st &= st - 1; }
            while (en) { S.gend[epos++] = base + __ffs(en); en &= en - 1; }
        }
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        det_scalars_q(a.psd, a.gain, a.off, a.ndet, a.fsamp, q, a.qsc);
        CgState cs;
        cs.rz = 0.0; cs.stop = 0.0; cs.koff = koff; cs.K = K; cs.it = 0; cs.ncz = 0;
        if (K == 0) cs.mode = CG_NONE;
        else if (K == n) cs.mode = CG_ALLFLAG;
        else if (koff + K > a.cgcap) cs.mode = CG_OVER;
        else cs.mode = CG_ACTIVE;
        a.cgs[q] = cs;
        // preconditioner blocks (rank within the detscan, length)
        int nb = 0;
        // (blocks of TOEP_LMAX: the tables may not be there yet, see nc_resplit)
        const int lmax = a.xtab ? TOEP_LMAX : 0;
        if (cs.mode == CG_ACTIVE && ngap <= TX_GBMAX && lmax >= 1) {
            int rank = 0;
            for (int g = 0; g < ngap && nb >= 0; ++g)
                for (int b0 = S.gbeg[g]; b0 < S.gend[g]; b0 += lmax) {
                    const int len = min(lmax, S.gend[g] - b0);
                    if (nb >= TX_GBMAX) { nb = -1; break; }
                    a.gblk[static_cast<int64_t>(q) * TX_GBMAX + nb] = make_int2(rank, len);
                    a.gbpos[static_cast<int64_t>(q) * TX_GBMAX + nb] = b0;
                    ++nb;
                    rank += len;
                }
        } else {
            nb = -1;
        }
        a.gnb[q] = nb;
    }
}

// Phase 3, column pass of the right-hand side: M (r/sigma0^2 + w1/sigma0),
// r = d - g s; w1 of z_j is normal pair j of the NC_W1 stream (pair j mod 4
// of Philox block j/4).
__device__ void nc_rhs_cols(const NcorrTx &a, const TxCtx &X, CF2 *b0, CF2 *b1, uint64_t gi)
{
    const bool draw = a.mode == TOD_MODE_DRAW;
    const float *dq = a.d + X.o, *sq = a.s + X.o;
    const float g = X.g, inv_s2 = X.inv_s2, inv_s = X.inv_s;
    const uint64_t q = static_cast<uint64_t>(X.q);
    struct U8 { float4 dv, sv; };
    col_forward<true, 2>(X, b0, b1, a.Y, a.tw + X.L.twb, a.flags,
                [&](CF2 *U) {
                    // the tile's normals: one Philox block per thread and
                    // round, its four pairs to the elements whose index j
                    // falls in it.  Lane a of row j1 holds columns p0 ..
                    // p0 + np - 1, lane b their mirrors: np consecutive j each.
                    const ColThread C(X.L, X.blk);
                    const int TP = C.TP, np = C.np, m1 = C.m1, m2 = C.m2, p0 = X.blk * TP;
                    if (!draw) {
                        for (int e = threadIdx.x; e < m1 * TP; e += TX_T) sst(U + e, vzero<CF2>());
                        return;
                    }
                    // a side's j range of a row touches at most (np + 6) / 4
                    // blocks; 2^lb >= that, so that no division is needed
                    int lb = 0;
                    while ((4 << lb) < np + 3) ++lb;
                    const int total = m1 << (lb + 1);
                    for (int w = threadIdx.x; w < total; w += TX_T) {
                        const int j1 = w >> (lb + 1), side = (w >> lb) & 1, bi = w & ((1 << lb) - 1);
                        const int ja = j1 * m2 + (side ? m2 - p0 - np : p0), jb = ja + np;
                        const int bk = (ja >> 2) + bi;
                        if (4 * bk >= jb) continue;
                        const u64x4 rw = philox4x64(static_cast<uint64_t>(bk), q, 1, gi, a.rng.seed, a.rng.band);
                        float *row = reinterpret_cast<float *>(U + j1 * TP);
#pragma unroll
                        for (int u = 0; u < 4; ++u) {
                            const int j = 4 * bk + u;
                            if (j < ja || j >= jb) continue;
                            const int i = side ? jb - 1 - j : j - ja;
                            const float2 z = philox_normal_pair(rw, u);
                            row[4 * i + side] = z.x;
                            row[4 * i + 2 + side] = z.y;
                        }
                    }
                },
                [&](int j, bool ctr, uint32_t) {
                    const int64_t t = 4 * static_cast<int64_t>(j);
                    return U8{ld4(dq, t, ctr), ld4(sq, t, ctr)};
                },
                [&](const U8 &D, int, bool ctr, uint32_t fb, float2 wa, float2 wb, float (&v)[4]) {
                    const float4 dv = D.dv, sv = D.sv;
                    // samples 4j, 4j+2 -> z_j; 4j+3, 4j+1 -> z_{m-1-j}; at the centre 4j, 4j+1 -> z_j
                    v[0] = (fb & 1) ? 0.f : fmaf(dv.x - g * sv.x, inv_s2, wa.x * inv_s);
                    v[1] = (fb & 2) ? 0.f : fmaf(dv.y - g * sv.y, inv_s2, (ctr ? wa.y : wb.y) * inv_s);
                    v[2] = (fb & 4) ? 0.f : fmaf(dv.z - g * sv.z, inv_s2, wa.y * inv_s);
                    v[3] = (fb & 8) ? 0.f : fmaf(dv.w - g * sv.w, inv_s2, wb.x * inv_s);
                });
}

// Filter weights of a mode: beta = 1/(phi + 1/sigma0^2) = sigma0^2/(1 + r),
// gamma = sigma0^2 r/(1 + r) with r = sigma0^2 phi = (f/f_knee)^-alpha (r = 0
// at mode 0).  With every sample flagged beta is 1/phi = sigma0^2 / r (0 at
// mode 0).
__device__ __forceinline__ float nc_r(int k, const TxCtx &X) {
    return k == 0 ? 0.f : tx_fpow(k, X.fscale, -X.alpha);
}
__device__ __forceinline__ float nc_beta(int k, float s2, const TxCtx &X) { return s2 * sfu_rcp(1.0f + nc_r(k, X)); }
__device__ __forceinline__ float nc_gamma(int k, float s2, const TxCtx &X) {
    const float r = nc_r(k, X);
    return s2 * r * sfu_rcp(1.0f + r);
}

// Phase 3, row pass of the right-hand side: + sqrt(phi) w2 (mode pair k of
// the NC_W2 stream), times beta; the spectrum beta (C b + prior term) is
// written when asked for.
__device__ void nc_rhs_rows(const NcorrTx &a, const TxCtx &X, CF2 *b0, CF2 *b1, uint64_t gi)
{
    const bool draw = a.mode == TOD_MODE_DRAW;
    const bool allf = X.mode == CG_ALLFLAG;
    const uint64_t q = static_cast<uint64_t>(X.q);
    const float s2 = X.s2, inv_s2 = X.inv_s2;
    const int n = X.L.n, m = X.L.m;
    float *spec = a.spec_out ? a.spec_out + X.o : nullptr;
    row_pass<true>(X, b0, b1, a.Y, a.tw + X.L.twb,
        [&](CF2 *Fr) {
            const int m1 = X.L.m1, m2 = X.L.m2, m2p = X.L.m2p, TR = X.L.TR;
            const int p0 = X.blk * TR, npl = min(TR, X.L.P1 - p0);
            if (!draw) {
                for (int e = threadIdx.x; e < TR * m2p; e += TX_T) sst(Fr + e, vzero<CF2>());
                return;
            }
            // for a fixed k2 lane a holds k = p0 + pl + m1 k2 and lane b
            // k = m1 - p0 - pl + m1 k2 (row m1/2, or none, for pair 0): runs
            // of consecutive modes, one Philox block for up to four of them
            const int lo = p0 ? p0 : 1;                        // first pair whose lane b runs with the others
            const float zero = 0.f;
            for (int w = threadIdx.x; w < 2 * m2; w += TX_T) {
                const int side = w >= m2, k2 = w - (side ? m2 : 0);
                const int ka = (side ? m1 - p0 - (npl - 1) : p0) + m1 * k2;
                const int kb = ka + (side ? p0 + npl - lo : npl);       // modes [ka, kb)
                float *e0 = reinterpret_cast<float *>(Fr + k2) + side;
                for (int bk = ka >> 2; 4 * bk < kb; ++bk) {
                    const u64x4 rw = philox4x64(static_cast<uint64_t>(bk), q, 2, gi, a.rng.seed, a.rng.band);
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        const int k = 4 * bk + u;
                        if (k < ka || k >= kb) continue;
                        const int pl = side ? npl - 1 - (k - ka) : k - ka;
                        const float2 z = philox_normal_pair(rw, u);
                        e0[4 * pl * m2p] = z.x;
                        e0[4 * pl * m2p + 2] = z.y;
                    }
                }
                if (side && p0 == 0) {
                    float2 z = make_float2(zero, zero);
                    if (!(m1 & 1)) {
                        const int k = (m1 >> 1) + m1 * k2;
                        z = stream_normal_pair(a.rng.seed, a.rng.band, q, 2, gi, 2 * static_cast<int64_t>(k));
                    }
                    e0[0] = z.x;
                    e0[2] = z.y;
                }
            }
        },
        [&](int k0, int k1, int mask, CF2 Y, CF2 nu) {
            const int l0 = k0 ? n - k0 : m, l1 = k1 ? n - k1 : m;
            const float r0 = nc_r(k0, X), r1 = nc_r(k1, X), u0 = nc_r(l0, X), u1 = nc_r(l1, X);
            PF bx, by;
            if (allf) {
                bx = pset(k0 ? s2 * sfu_rcp(r0) : 0.f, k1 ? s2 * sfu_rcp(r1) : 0.f);
                by = pset(s2 * sfu_rcp(u0), s2 * sfu_rcp(u1));
            } else {
                bx = pset(s2 * sfu_rcp(1.0f + r0), s2 * sfu_rcp(1.0f + r1));
                by = pset(s2 * sfu_rcp(1.0f + u0), s2 * sfu_rcp(1.0f + u1));
            }
            const PF px = pset(sqrtf(r0 * inv_s2), sqrtf(r1 * inv_s2)), py = pset(sqrtf(u0 * inv_s2), sqrtf(u1 * inv_s2));
            const CF2 xs{pmul(pfma(px, nu.x, Y.x), bx), pmul(pfma(py, nu.y, Y.y), by)};
            if (spec) {
                if (mask & 1) { spec[k0] = xs.x.a; spec[l0] = xs.y.a; }
                if (mask & 2) { spec[k1] = xs.x.b; spec[l1] = xs.y.b; }
            }
            return xs;
        });
}

// Phase 3, inverse column pass: x0 out; its flagged samples are the CG
// right-hand side E^T x0.
__device__ void nc_x0_cols(const NcorrTx &a, const TxCtx &X, CF2 *b0, CF2 *b1)
{
    const bool cg = X.mode == CG_ACTIVE;
    float *xq = a.x_out + X.o;
    const int64_t o = X.o, obase = a.off[a.q0], w_lo = obase >> 5;
    float *r = a.cgv + a.cgcap;
    col_inverse(X, b0, b1, a.Y, a.tw + X.L.twb, cg ? a.flags : nullptr, [&](int, bool, uint32_t) { return 0; },
                [&](int, int j, bool ctr, const float (&v)[4], uint32_t fb) {
        const int64_t t = 4 * static_cast<int64_t>(j);
        reinterpret_cast<float2 *>(xq + t)[0] = make_float2(v[0], v[1]);
        if (!ctr) reinterpret_cast<float2 *>(xq + t + 2)[0] = make_float2(v[2], v[3]);
        while (fb) {                  // cg only: no flags are read otherwise
            const int u = __ffs(fb) - 1;
            fb &= fb - 1;
            r[flag_rank(a.flags, a.wpre, w_lo, obase, o + t + u)] = u == 0 ? v[0] : u == 1 ? v[1] : u == 2 ? v[2] : v[3];
        }
    });
}

// CG column pass: z = E vec (the flagged samples' entries of vec, zero
// elsewhere), forward columns.  The thread zeroes its tile elements and places
// the entries of its flagged units, about one sample in fifty: no value is held
// for the others (four rows of values, and the lookup of their ranks written out
// eight times, spilled 412 bytes at 80 registers: the draw of 72 x 225k samples
// without its preparation 2107 -> 2009 us).
// Sample s of unit (j1, c): z_j = (x_0, x_2) in lane a of row j1, its mirror
// z_{m-1-j} = (x_3, x_1) in lane b of row m1-1-j1; of unit (j1, c2) the lanes
// change places; a column that is its own mirror fills both.
__device__ void nc_scatter_cols(const NcorrTx &a, const TxCtx &X, CF2 *b0, CF2 *b1, const float *vec)
{
    const int64_t o = X.o, obase = a.off[a.q0], w_lo = obase >> 5;
    const ColThread C(X.L, X.blk);
    const int m1 = C.m1, TP = C.TP;
    uint32_t fnib = unit_flags(C, a.flags, o);
    for (int j1 = C.r0; j1 < (C.c < 0 ? m1 : C.m1h); j1 += C.rstep) {
        sst(b0 + j1 * TP + C.i, vzero<CF2>());
        if (C.c >= 0) sst(b0 + (m1 - 1 - j1) * TP + C.i, vzero<CF2>());
    }
#pragma unroll 1
    for (int k = 0; fnib; ++k, fnib >>= 4) {
        const uint32_t fb = fnib & 15u;
        if (!fb) continue;
        const int j1 = C.row(k >> 1), side = k & 1;
        const int64_t t = o + 4 * static_cast<int64_t>(j1 * C.m2 + (side ? C.c2 : C.c));
        const float *v = vec + flag_rank(a.flags, a.wpre, w_lo, obase, t);
        float *ea = reinterpret_cast<float *>(b0 + j1 * TP + C.i);
        float *eb = reinterpret_cast<float *>(b0 + (m1 - 1 - j1) * TP + C.i);
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            if (!(fb >> u & 1u)) continue;
            const float val = v[__popc(fb & ((1u << u) - 1u))];
            float *e = ((u & 1) ? eb : ea) + ((u == 1 || u == 2) ? 2 : 0);     // x_1, x_2: imaginary parts
            if (C.c == C.c2) e[0] = e[1] = val;
            else e[side ^ (u & 1)] = val;
        }
    }
    col_forward_out(X, C, b0, b1, a.Y, a.tw + X.L.twb);
}

// CG row pass: times gamma (apply S), or times beta (the final B^{-1} E y,
// whose spectrum is added to the one written at the right-hand side).
template <bool BETA>
__device__ void nc_filter_rows(const NcorrTx &a, const TxCtx &X, CF2 *b0, CF2 *b1)
{
    const float s2 = X.s2;
    const int n = X.L.n, m = X.L.m;
    float *spec = (BETA && a.spec_out) ? a.spec_out + X.o : nullptr;
    const auto weight = [&](int k) { return BETA ? nc_beta(k, s2, X) : nc_gamma(k, s2, X); };
    row_pass<false>(X, b0, b1, a.Y, a.tw + X.L.twb, [](CF2 *) {}, [&](int k0, int k1, int mask, CF2 Y, CF2) {
        const int l0 = k0 ? n - k0 : m, l1 = k1 ? n - k1 : m;
        const CF2 r{pmul(Y.x, pset(weight(k0), weight(k1))), pmul(Y.y, pset(weight(l0), weight(l1)))};
        if (spec) {
            if (mask & 1) { spec[k0] += r.x.a; spec[l0] += r.y.a; }
            if (mask & 2) { spec[k1] += r.x.b; spec[l1] += r.y.b; }
        }
        return r;
    });
}

// CG inverse column pass: q = E^T (...) (gather), or x += (...) (final).
template <bool ADD>
__device__ void nc_gather_cols(const NcorrTx &a, const TxCtx &X, CF2 *b0, CF2 *b1, float *qv)
{
    const int64_t o = X.o, obase = a.off[a.q0], w_lo = obase >> 5;
    float *xq = a.x_out + X.o;
    col_inverse(X, b0, b1, a.Y, a.tw + X.L.twb, ADD ? nullptr : a.flags, [&](int j, bool ctr, uint32_t) {
        // ADD: the unit's x0 (written earlier in this launch: coherent loads,
        // not the read-only path); the gather needs only the flag bits
        float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
        if (ADD) {
            const int64_t t = 4 * static_cast<int64_t>(j);
            const float2 a01 = reinterpret_cast<const float2 *>(xq + t)[0];
            const float2 a23 = ctr ? make_float2(0.f, 0.f) : reinterpret_cast<const float2 *>(xq + t + 2)[0];
            x = make_float4(a01.x, a01.y, a23.x, a23.y);
        }
        return x;
    }, [&](const float4 &x0, int j, bool ctr, const float (&v)[4], uint32_t fb) {
        const int64_t t = 4 * static_cast<int64_t>(j);
        if (ADD) {
            float2 *p = reinterpret_cast<float2 *>(xq + t);
            p[0] = make_float2(x0.x + v[0], x0.y + v[1]);
            if (!ctr) p[1] = make_float2(x0.z + v[2], x0.w + v[3]);
            return;
        }
        while (fb) {
            const int u = __ffs(fb) - 1;
            fb &= fb - 1;
            qv[flag_rank(a.flags, a.wpre, w_lo, obase, o + t + u)] = u == 0 ? v[0] : u == 1 ? v[1] : u == 2 ? v[2] : v[3];
        }
    });
}

// z = M^{-1} r over the detscan's gap blocks: T_L^{-1} = (L(x) L(x)^T -
// L(w) L(w)^T) / x_0 (Gohberg-Semencul; x = T_L^{-1} e_1 from the Toeplitz
// tables, w = (0, x_{L-1}, .., x_1)).  Returns r.z (CTA total, every thread)
// with RZ.  z may be r (a block reads its r before it writes its z).
//
// A block is taken by a group of two warps, the next free one by each group
// (the blocks are independent and of very different lengths); a warp forms
// 128 outputs at a time, four per lane:
//   u[i] = sum_k (x, w)[k] r[i + k],  z[i] = (1/x_0) sum_s x[s] u1[i-s] - w[s] u2[i-s],
// with x, w and u1, u2 the lanes of packed FMAs.  A step of four k takes 16
// packed FMAs, two broadcast loads of (x, w) and one (u: two) 16-byte load of
// the sliding window, so the FMA pipe is the bound; with the whole CTA on one
// round of blocks after the other, every operand loaded per output, it was
// shared memory, and the barriers between the rounds (cg_init of 240
// detscans of 30 GHz: 151 -> 110 us; of 360 of 70 GHz 268 -> 214, of which
// these products are 119).
// gb: GB_FLOATS of shared memory.
constexpr int GB_GROUPS = TX_T / 64;
constexpr int GB_TILE = 128;                             // outputs of a warp tile
constexpr int GB_PAD = GB_TILE + 8;                      // zeros beyond r, and before u
constexpr int GB_XW = 2 * TOEP_LMAX, GB_U = 2 * (GB_PAD + TOEP_LMAX), GB_R = TOEP_LMAX + GB_PAD;
constexpr int GB_GROUP_FLOATS = GB_XW + GB_U + GB_R;
constexpr int GB_FLOATS = GB_GROUPS * GB_GROUP_FLOATS;
static_assert(GB_XW % 4 == 0 && GB_U % 4 == 0 && GB_R % 4 == 0 && GB_PAD % 4 == 0, "16-byte accesses");

__device__ __forceinline__ void group_sync(int group) {
    asm volatile("bar.sync %0, 64;" ::"r"(group + 1) : "memory");
}
template <bool RZ>
__device__ double nc_precond_m1(const NcorrTx &a, NcShared &S, int q, const float *r, float *z, float *gb)
{
    const int nb = a.gnb[q];
    const CgState &cs = a.cgs[q];
    const int K = cs.K;
    Acc2 rz[1] = {{0.f, 0.f}};
    if (nb < 0) {             // no preconditioner: z = r
        for (int i = threadIdx.x; i < K; i += TX_T) {
            const float v = r[i];
            z[i] = v;
            acc_add_prod(rz[0], v, v);
        }
        if (!RZ) return 0.0;
        block_sums<1>(rz, S.red, S.out);
        return S.out[0];
    }
    const float *xt_det = a.xtab + static_cast<int64_t>(q % a.ndet) * (TOEP_LMAX * (TOEP_LMAX + 1) / 2);
    const int2 *gbl = a.gblk + static_cast<int64_t>(q) * TX_GBMAX;
    const int group = threadIdx.x >> 6, gt = threadIdx.x & 63, wg = gt >> 5, lane = threadIdx.x & 31;
    float *g0 = gb + group * GB_GROUP_FLOATS;
    PF *xw = reinterpret_cast<PF *>(g0), *u0 = reinterpret_cast<PF *>(g0 + GB_XW), *u = u0 + GB_PAD;
    float *rb = g0 + GB_XW + GB_U;
    for (int i = gt; i < GB_PAD; i += 64) u0[i] = PF{0.f, 0.f};
    if (threadIdx.x == 0) S.next = GB_GROUPS;
    __syncthreads();
    for (int b = group; b < nb;) {
        const int2 bl = gbl[b];
        const int L = bl.y, L4 = (L + 3) & ~3;
        const float *xt = xt_det + L * (L - 1) / 2;
        if (gt == 0) S.grab[group] = atomicAdd(&S.next, 1);
        for (int i = gt; i < L; i += 64) {
            const float xv = xt[i];
            xw[i].a = xv;
            xw[i ? L - i : 0].b = i ? xv : 0.f;
            rb[i] = r[bl.x + i];
        }
        for (int i = L + gt; i < L4 + GB_PAD; i += 64) {
            if (i < L4) xw[i] = PF{0.f, 0.f};
            rb[i] = 0.f;                                  // L4 + GB_PAD <= GB_R
        }
        group_sync(group);
        const float inv = 1.0f / xw[0].a;
        const int nt = (L + GB_TILE - 1) / GB_TILE;
        // tiles to warps, balancing the triangular sums (u: long first tiles; z: long last ones)
        for (int t = 0; t < nt; ++t) {
            if (((t == 1 || t == 2) ? 1 : 0) != wg) continue;
            const int i0 = t * GB_TILE + 4 * lane;
            PF acc[4] = {{0.f, 0.f}, {0.f, 0.f}, {0.f, 0.f}, {0.f, 0.f}};
            float4 rc = *reinterpret_cast<const float4 *>(rb + i0);
#pragma unroll 2
            for (int k = 0; k < L - t * GB_TILE; k += 4) {
                const float4 rn = *reinterpret_cast<const float4 *>(rb + i0 + k + 4);
                const float4 p = *reinterpret_cast<const float4 *>(xw + k), q4 = *reinterpret_cast<const float4 *>(xw + k + 2);
                const PF w4[4] = {{p.x, p.y}, {p.z, p.w}, {q4.x, q4.y}, {q4.z, q4.w}};
                const float rw[7] = {rc.x, rc.y, rc.z, rc.w, rn.x, rn.y, rn.z};
#pragma unroll
                for (int kk = 0; kk < 4; ++kk)
#pragma unroll
                    for (int j = 0; j < 4; ++j) acc[j] = pfma(w4[kk], pdup<PF>(rw[kk + j]), acc[j]);
                rc = rn;
            }
#pragma unroll
            for (int j = 0; j < 4; ++j) u[i0 + j] = acc[j];
        }
        group_sync(group);
        for (int t = 0; t < nt; ++t) {
            if ((nt == 3 ? (t == 2 ? 1 : 0) : (t == 1 || t == 2) ? 1 : 0) != wg) continue;
            const int i0 = t * GB_TILE + 4 * lane;
            PF acc[4] = {{0.f, 0.f}, {0.f, 0.f}, {0.f, 0.f}, {0.f, 0.f}};
            float4 ua = *reinterpret_cast<const float4 *>(u + i0), ub = *reinterpret_cast<const float4 *>(u + i0 + 2);
            const int smax = min((t + 1) * GB_TILE, L4);
#pragma unroll 2
            for (int s = 0; s < smax; s += 4) {
                const float4 va = *reinterpret_cast<const float4 *>(u + i0 - s - 4);
                const float4 vb = *reinterpret_cast<const float4 *>(u + i0 - s - 2);
                const float4 p = *reinterpret_cast<const float4 *>(xw + s), q4 = *reinterpret_cast<const float4 *>(xw + s + 2);
                const PF w4[4] = {{p.x, p.y}, {p.z, p.w}, {q4.x, q4.y}, {q4.z, q4.w}};
                // u[i0 - s - 3 .. i0 - s + 3]
                const PF uw[7] = {{va.z, va.w}, {vb.x, vb.y}, {vb.z, vb.w}, {ua.x, ua.y}, {ua.z, ua.w},
                                  {ub.x, ub.y}, {ub.z, ub.w}};
#pragma unroll
                for (int ss = 0; ss < 4; ++ss)
#pragma unroll
                    for (int j = 0; j < 4; ++j) acc[j] = pfma(w4[ss], uw[3 + j - ss], acc[j]);
                ua = va;
                ub = vb;
            }
#pragma unroll
            for (int j = 0; j < 4; ++j)
                if (i0 + j < L) z[bl.x + i0 + j] = (acc[j].a - acc[j].b) * inv;
        }
        b = S.grab[group];
        group_sync(group);
    }
    __syncthreads();
    if (!RZ) return 0.0;
#pragma unroll 4
    for (int i = threadIdx.x; i < K; i += TX_T) acc_add_prod(rz[0], r[i], z[i]);
    block_sums<1>(rz, S.red, S.out);
    return S.out[0];
}

// ---------------------------------------------------------------------------
// Coarse correction (two-level preconditioner, balancing form):
//   M r = P^T M1 P r + Z E^{-1} Z^T r,  P = I - S Z E^{-1} Z^T,  E = Z^T S Z,
// with M1 the gap-block inverses above and Z two vectors per gap block: its
// indicator and its centred ramp (z(l) = (l - c) / c, c = (L - 1) / 2, over
// the block's L samples; zero for L = 1).  M is symmetric positive definite
// for any S Z and E^{-1} used consistently, so the CG converges to the same
// solution; the correction takes out the smooth modes spread over several
// gaps, which the block inverses leave to the iterations.  S Z is taken from
// the Toeplitz kernel alone, (S Z)_{i,(b,s)} = sum_{j in b} h(|p_i - p_j|)
// z_{b,s}(j), and only for the TX_CZW blocks either side of the row's own
// block (farther terms dropped), so E is banded (half-bandwidth TX_CZB in
// scalar rows) and one banded Cholesky factor per detscan applies E^{-1}.
// The sums over a block come from prefix sums of h:
//   sum_{delta=lo..hi} h(|delta|)       from H(x) = sum_{d<x} h(d),
//   sum_{delta=lo..hi} delta h(|delta|) from G(x) = sum_{d<x} d h(d),
// held as FP32 pairs and differenced in pair arithmetic (the differences of
// far blocks cancel most of the prefix values).
// ---------------------------------------------------------------------------
constexpr int CZ_LROW = TX_CZB + 1;                   // factor row: 1 / L_ii, then L_{i,i-k}, k = 1..TX_CZB
constexpr int CZ_FLOATS = 2 * TX_CBMAX * CZ_LROW + 3 * 2 * TX_CBMAX + TX_CBMAX * TX_CZJ + CZ_LROW * TX_CZB;

__device__ __forceinline__ float cz_ramp(int l, int L) {
    if (L < 2) return 0.f;
    const float c = 0.5f * static_cast<float>(L - 1);
    return (static_cast<float>(l) - c) * (1.0f / c);
}

// FP32 pair (hi + lo) arithmetic: Knuth's two-sum and an FMA two-product.
struct F2 { float h, l; };
__device__ __forceinline__ F2 f2_add(F2 x, F2 y) {
    const float s = x.h + y.h;
    const float bp = s - x.h;
    float e = (x.h - (s - bp)) + (y.h - bp);
    e += x.l + y.l;
    const float h = s + e;
    return {h, e - (h - s)};
}
__device__ __forceinline__ F2 f2_mulf(F2 x, float f) {
    const float p = __fmul_rn(x.h, f);        // not contracted into the sum below
    float e = fmaf(x.h, f, -p);
    e = fmaf(x.l, f, e);
    const float h = p + e;
    return {h, e - (h - p)};
}

// (S Z) entries of the row at sample p for a block of L samples from s:
// the indicator's sum over delta = p - j, and the ramp's.  Each table
// entry holds (H, G) at one x, loaded once.
__device__ __forceinline__ float2 cz_entry(const float4 *__restrict__ t, int p, int s, int L) {
    const int lo = p - (s + L - 1), hi = p - s;
    F2 I, Mo;
    if (lo >= 0) {
        const float4 A = __ldg(t + hi + 1), B = __ldg(t + lo);
        I = f2_add(F2{A.x, A.y}, F2{-B.x, -B.y});
        Mo = f2_add(F2{A.z, A.w}, F2{-B.z, -B.w});
    } else if (hi < 0) {
        const float4 A = __ldg(t + 1 - lo), B = __ldg(t - hi);
        I = f2_add(F2{A.x, A.y}, F2{-B.x, -B.y});
        Mo = f2_add(F2{B.z, B.w}, F2{-A.z, -A.w});
    } else {
        const float4 A = __ldg(t + hi + 1), B = __ldg(t + 1 - lo), C = __ldg(t + 1);
        I = f2_add(f2_add(F2{A.x, A.y}, F2{B.x, B.y}), F2{-C.x, -C.y});
        Mo = f2_add(F2{A.z, A.w}, F2{-B.z, -B.w});
    }
    float ramp = 0.f;
    if (L > 1) {
        // sum_j (j - c_b) h = (p - c_b) I - Mo, c_b = s + (L - 1)/2
        const float pc = 0.5f * static_cast<float>(2 * (p - s) - (L - 1));
        const F2 v = f2_add(f2_mulf(I, pc), F2{-Mo.h, -Mo.l});
        ramp = (v.h + v.l) * (1.0f / (0.5f * static_cast<float>(L - 1)));
    }
    return make_float2(I.h + I.l, ramp);
}

// Cuts detscan q's gaps anew when the tables stop short of TOEP_LMAX (a pivot
// of the recursion was not positive): blocks of at most lvalid samples, or no
// preconditioner when there are too many of them or no table at all.
__device__ void nc_resplit(const NcorrTx &a, int q)
{
    if (!a.xtab) return;
    const int lmax = a.lvalid[q % a.ndet], nb = a.gnb[q];
    if (lmax >= TOEP_LMAX || nb < 0) return;
    __shared__ int3 s_old[TX_GBMAX];              // rank, length, first sample
    int2 *gbl = a.gblk + static_cast<int64_t>(q) * TX_GBMAX;
    int32_t *pos = a.gbpos + static_cast<int64_t>(q) * TX_GBMAX;
    for (int b = threadIdx.x; b < nb; b += TX_T) s_old[b] = make_int3(gbl[b].x, gbl[b].y, pos[b]);
    __syncthreads();
    if (threadIdx.x == 0) {
        int n = lmax >= 1 ? 0 : -1;
        for (int b = 0; b < nb && n >= 0;) {
            // a gap: blocks that follow one another without a sample between
            int e = b + 1, len = s_old[b].y;
            while (e < nb && s_old[e].z == s_old[b].z + len) len += s_old[e++].y;
            for (int i = 0; i < len; i += lmax) {
                if (n >= TX_GBMAX) { n = -1; break; }
                gbl[n] = make_int2(s_old[b].x + i, min(lmax, len - i));
                pos[n] = s_old[b].z + i;
                ++n;
            }
            b = e;
        }
        a.gnb[q] = n;
    }
    __syncthreads();
}

// Builds the coarse correction of detscan q (after the index phase): S Z
// rows, E, its banded Cholesky factor.  On success cgs[q].ncz = blocks.
__device__ void nc_coarse_setup(const NcorrTx &a, int q)
{
    __shared__ int s_rank[TX_CBMAX], s_len[TX_CBMAX], s_pos[TX_CBMAX];
    __shared__ float s_E[TX_CBMAX][4 * (2 * TX_CZW + 1)];
    __shared__ float s_L[2 * TX_CBMAX][CZ_LROW];
    __shared__ int s_ok;
    const CgState cs = a.cgs[q];
    const int nb = a.gnb[q];
    if (cs.mode != CG_ACTIVE || nb < 1 || nb > TX_CBMAX || !a.czsz || cs.koff + cs.K > a.czcap) return;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int det = q % a.ndet;
    const float4 *tab = a.cztab + static_cast<int64_t>(det) * (a.href + 1);
    for (int b = threadIdx.x; b < nb; b += TX_T) {
        const int2 bl = a.gblk[static_cast<int64_t>(q) * TX_GBMAX + b];
        s_rank[b] = bl.x;
        s_len[b] = bl.y;
        s_pos[b] = a.gbpos[static_cast<int64_t>(q) * TX_GBMAX + b];
    }
    __syncthreads();
    float *sz = a.czsz + cs.koff * TX_CZJ;
    // S Z rows, one warp per block, with the block's rows of E: for the
    // neighbour j and the row/column vector kinds (s', s), sum over the
    // block's samples of z_{s'} (S Z)_s
    for (int b = warp; b < nb; b += TX_T / 32) {
        const int L = s_len[b];
        float e[4 * (2 * TX_CZW + 1)];
#pragma unroll
        for (int k = 0; k < 4 * (2 * TX_CZW + 1); ++k) e[k] = 0.f;
        for (int l = lane; l < L; l += 32) {
            const int i = s_rank[b] + l, p = s_pos[b] + l;
            const float zr = cz_ramp(l, L);
            float2 *row = reinterpret_cast<float2 *>(sz + static_cast<int64_t>(i) * TX_CZJ);
#pragma unroll
            for (int j = 0; j < 2 * TX_CZW + 1; ++j) {
                const int c = b - TX_CZW + j;
                float2 v = make_float2(0.f, 0.f);
                if (c >= 0 && c < nb) v = cz_entry(tab, p, s_pos[c], s_len[c]);
                row[j] = v;
                e[4 * j + 0] += v.x;
                e[4 * j + 1] += v.y;
                e[4 * j + 2] = fmaf(zr, v.x, e[4 * j + 2]);
                e[4 * j + 3] = fmaf(zr, v.y, e[4 * j + 3]);
            }
        }
#pragma unroll
        for (int k = 0; k < 4 * (2 * TX_CZW + 1); ++k) {
            float v = e[k];
            for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
            if (lane == 0) s_E[b][k] = v;
        }
    }
    __syncthreads();
    // E's lower band, s_L[x][k] = E(x, x - k), x = 2b + s', y = 2c + s: from
    // block b's rows s_E[b][4 (c - b + W) + 2 s' + s], averaged with block
    // c's; a ramp of a one-sample block is zero (its row of E set to the
    // identity's)
    const int nc = 2 * nb;
    for (int i = threadIdx.x; i < nc * CZ_LROW; i += TX_T) {
        const int x = i / CZ_LROW, k = i % CZ_LROW, y = x - k;
        float v = 0.f;
        if (y >= 0) {
            const int b = x >> 1, sp = x & 1, c = y >> 1, sc = y & 1;
            if ((sp && s_len[b] < 2) || (sc && s_len[c] < 2)) v = x == y ? 1.f : 0.f;
            else if (b - c <= TX_CZW)
                v = 0.5f * (s_E[b][4 * (c - b + TX_CZW) + 2 * sp + sc] + s_E[c][4 * (b - c + TX_CZW) + 2 * sc + sp]);
        }
        s_L[x][k] = v;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        // banded Cholesky in place (FP32: E is a small, well-conditioned
        // Gram matrix of smooth vectors); s_L[x][0] becomes 1 / L_xx
        int ok = 1;
        for (int x = 0; x < nc && ok; ++x) {
            const float exx = s_L[x][0];
            float dsum = exx;
            for (int k = TX_CZB; k >= 1; --k) {
                const int y = x - k;
                float v = 0.f;
                if (y >= 0) {
                    v = s_L[x][k];
                    // sum over m < y of L(x, m) L(y, m), both within the band
                    for (int m = max(0, x - TX_CZB); m < y; ++m) v = fmaf(-s_L[x][x - m], s_L[y][y - m], v);
                    v *= s_L[y][0];
                }
                s_L[x][k] = v;
                dsum = fmaf(-v, v, dsum);
            }
            if (!(dsum > 1e-5f * fabsf(exx))) ok = 0;
            else s_L[x][0] = rsqrtf(dsum);
        }
        s_ok = ok;
        if (ok) a.cgs[q].ncz = nb;
    }
    __syncthreads();
    if (s_ok) {
        float *Lq = a.czl + static_cast<int64_t>(q) * (2 * TX_CBMAX * CZ_LROW);
        for (int i = threadIdx.x; i < nc * CZ_LROW; i += TX_T) Lq[i] = s_L[i / CZ_LROW][i % CZ_LROW];
    }
    __syncthreads();
}

// t = E^{-1} u with the banded factor staged in shared memory (rows of
// CZ_LROW; rows nc .. nc + TX_CZB - 1 zero).  One thread.
__device__ __forceinline__ void cz_solve(const float *L, int nc, const float *u, float *t)
{
    float w[TX_CZB];
#pragma unroll
    for (int k = 0; k < TX_CZB; ++k) w[k] = 0.f;
    for (int x = 0; x < nc; ++x) {
        const float *l = L + x * CZ_LROW;
        float v = u[x];
#pragma unroll
        for (int k = 1; k <= TX_CZB; ++k) v = fmaf(-l[k], w[k - 1], v);
        v *= l[0];
#pragma unroll
        for (int k = TX_CZB - 1; k > 0; --k) w[k] = w[k - 1];
        w[0] = v;
        t[x] = v;
    }
#pragma unroll
    for (int k = 0; k < TX_CZB; ++k) w[k] = 0.f;
    for (int x = nc - 1; x >= 0; --x) {
        float v = t[x];
#pragma unroll
        for (int k = 1; k <= TX_CZB; ++k) v = fmaf(-L[(x + k) * CZ_LROW + k], w[k - 1], v);
        v *= L[x * CZ_LROW];
#pragma unroll
        for (int k = TX_CZB - 1; k > 0; --k) w[k] = w[k - 1];
        w[0] = v;
        t[x] = v;
    }
}

// z = M r (two-level when the detscan has a coarse correction, else the
// block inverses alone).  Returns r.z (CTA total, every thread).  gb: the
// block inverses' GB_FLOATS, then CZ_FLOATS for the coarse vectors.
__device__ double nc_precond(const NcorrTx &a, NcShared &S, int q, const float *r, float *z, float *gb)
{
    const CgState cs = a.cgs[q];
    const int nb = cs.ncz;
    if (nb <= 0) return nc_precond_m1<true>(a, S, q, r, z, gb);
    const int nc = 2 * nb;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    float *cL = gb + GB_FLOATS;                      // [(nc + TX_CZB) rows][CZ_LROW]
    float *ct = cL + (2 * TX_CBMAX + TX_CZB) * CZ_LROW;  // t = E^{-1} Z^T r
    float *cu = ct + 2 * TX_CBMAX;                      // Z^T r, then (S Z)^T z1
    float *cs2 = cu + 2 * TX_CBMAX;                     // t - E^{-1} (S Z)^T z1
    float *cP = cs2 + 2 * TX_CBMAX;                     // [nb][TX_CZJ] per-block partial sums
    const int2 *gbl = a.gblk + static_cast<int64_t>(q) * TX_GBMAX;
    const float *Lq = a.czl + static_cast<int64_t>(q) * (2 * TX_CBMAX * CZ_LROW);
    const float *sz = a.czsz + cs.koff * TX_CZJ;
    for (int i = threadIdx.x; i < (nc + TX_CZB) * CZ_LROW; i += TX_T) cL[i] = i < nc * CZ_LROW ? Lq[i] : 0.f;
    // Z^T r: one warp per block
    for (int b = warp; b < nb; b += TX_T / 32) {
        const int2 bl = gbl[b];
        float s0 = 0.f, s1 = 0.f;
#pragma unroll 4
        for (int l = lane; l < bl.y; l += 32) {
            const float v = r[bl.x + l];
            s0 += v;
            s1 = fmaf(cz_ramp(l, bl.y), v, s1);
        }
        for (int o = 16; o; o >>= 1) {
            s0 += __shfl_xor_sync(0xffffffffu, s0, o);
            s1 += __shfl_xor_sync(0xffffffffu, s1, o);
        }
        if (lane == 0) { cu[2 * b] = s0; cu[2 * b + 1] = s1; }
    }
    __syncthreads();
    if (threadIdx.x == 0) cz_solve(cL, nc, cu, ct);
    __syncthreads();
    // w = r - (S Z) t, into z
    for (int b = warp; b < nb; b += TX_T / 32) {
        const int2 bl = gbl[b];
#pragma unroll 4
        for (int l = lane; l < bl.y; l += 32) {
            const int i = bl.x + l;
            const float2 *row = reinterpret_cast<const float2 *>(sz + static_cast<int64_t>(i) * TX_CZJ);
            float v = r[i];
#pragma unroll
            for (int j = 0; j < 2 * TX_CZW + 1; ++j) {
                const int c = b - TX_CZW + j;
                if (c >= 0 && c < nb) {
                    const float2 e = row[j];
                    v = fmaf(-e.x, ct[2 * c], v);
                    v = fmaf(-e.y, ct[2 * c + 1], v);
                }
            }
            z[i] = v;
        }
    }
    __syncthreads();
    // z1 = M1 w, in place
    nc_precond_m1<false>(a, S, q, z, z, gb);
    __syncthreads();
    // (S Z)^T z1: per block the sums over its rows of each stored column
    for (int b = warp; b < nb; b += TX_T / 32) {
        const int2 bl = gbl[b];
        float e[TX_CZJ];
#pragma unroll
        for (int k = 0; k < TX_CZJ; ++k) e[k] = 0.f;
#pragma unroll 4
        for (int l = lane; l < bl.y; l += 32) {
            const int i = bl.x + l;
            const float2 *row = reinterpret_cast<const float2 *>(sz + static_cast<int64_t>(i) * TX_CZJ);
            const float zi = z[i];
#pragma unroll
            for (int j = 0; j < 2 * TX_CZW + 1; ++j) {
                const float2 v = row[j];
                e[2 * j] = fmaf(v.x, zi, e[2 * j]);
                e[2 * j + 1] = fmaf(v.y, zi, e[2 * j + 1]);
            }
        }
#pragma unroll
        for (int k = 0; k < TX_CZJ; ++k) {
            float v = e[k];
            for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
            if (lane == 0) cP[b * TX_CZJ + k] = v;
        }
    }
    __syncthreads();
    for (int x = threadIdx.x; x < nc; x += TX_T) {
        const int c = x >> 1, sc = x & 1;
        float v = 0.f;
        for (int bp = max(0, c - TX_CZW); bp <= min(nb - 1, c + TX_CZW); ++bp)
            v += cP[bp * TX_CZJ + 2 * (c - bp + TX_CZW) + sc];
        cu[x] = v;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        cz_solve(cL, nc, cu, cs2);
        for (int x = 0; x < nc; ++x) cs2[x] = ct[x] - cs2[x];
    }
    __syncthreads();
    // z = z1 + Z (t - E^{-1} (S Z)^T z1);  r.z
    Acc2 rz[1] = {{0.f, 0.f}};
    for (int b = warp; b < nb; b += TX_T / 32) {
        const int2 bl = gbl[b];
        const float c0 = cs2[2 * b], c1 = cs2[2 * b + 1];
#pragma unroll 4
        for (int l = lane; l < bl.y; l += 32) {
            const int i = bl.x + l;
            const float zi = z[i] + fmaf(c1, cz_ramp(l, bl.y), c0);
            z[i] = zi;
            acc_add_prod(rz[0], r[i], zi);
        }
    }
    block_sums<1>(rz, S.red, S.out);
    return S.out[0];
}

// CG start of detscan q: r = E^T x0 (already gathered), y = 0, z = M^{-1} r,
// p = z, (r.r, r.z); nothing to do when r = 0.
__device__ void nc_cg_init(const NcorrTx &a, NcShared &S, int q, float *gb)
{
    CgState cs = a.cgs[q];
    if (cs.mode != CG_ACTIVE) return;
    const CgVec V = cg_vecs(a);
    const int64_t k0 = cs.koff;
    const int K = cs.K;
    Acc2 rr[1] = {{0.f, 0.f}};
#pragma unroll 4
    for (int i = threadIdx.x; i < K; i += TX_T) {
        const float v = V.r[k0 + i];
        V.y[k0 + i] = 0.f;
        acc_add_prod(rr[0], v, v);
    }
    block_sums<1>(rr, S.red, S.out);
    const double rr0 = S.out[0];
    const double rz = nc_precond(a, S, q, V.r + k0, V.z + k0, gb);
#pragma unroll 4
    for (int i = threadIdx.x; i < K; i += TX_T) V.p[k0 + i] = V.z[k0 + i];
    if (threadIdx.x == 0) {
        cs.rz = rz;
        cs.stop = static_cast<double>(a.tol) * a.tol * rr0;
        cs.it = 0;
        if (rr0 == 0.0) cs.mode = CG_DONE;
        a.cgs[q] = cs;
        if (cs.mode == CG_ACTIVE) atomicAdd(a.count, 1);
    }
}

// One CG iteration of detscan q after q = S p is gathered.
__device__ void nc_cg_update(const NcorrTx &a, NcShared &S, int q, float *gb, int32_t *count_next)
{
    CgState cs = a.cgs[q];
    if (cs.mode != CG_ACTIVE) return;
    const CgVec V = cg_vecs(a);
    const int64_t k0 = cs.koff;
    const int K = cs.K;
    Acc2 pq[1] = {{0.f, 0.f}};
#pragma unroll 4
    for (int i = threadIdx.x; i < K; i += TX_T) acc_add_prod(pq[0], V.p[k0 + i], V.q[k0 + i]);
    block_sums<1>(pq, S.red, S.out);
    const float alp = static_cast<float>(cs.rz / S.out[0]);
    Acc2 rr[1] = {{0.f, 0.f}};
#pragma unroll 4
    for (int i = threadIdx.x; i < K; i += TX_T) {
        V.y[k0 + i] = fmaf(alp, V.p[k0 + i], V.y[k0 + i]);
        const float rn = fmaf(-alp, V.q[k0 + i], V.r[k0 + i]);
        V.r[k0 + i] = rn;
        acc_add_prod(rr[0], rn, rn);
    }
    block_sums<1>(rr, S.red, S.out);
    const double rrn = S.out[0];
    ++cs.it;
    bool cont = true;
    if (rrn <= cs.stop) { cs.mode = CG_DONE; cont = false; }
    else if (cs.it >= a.maxit || !(rrn == rrn)) {
        cs.mode = CG_DONE;
        cont = false;
        if (threadIdx.x == 0) set_status(a.status, q, TOD_ERR_NOT_CONVERGED);
    }
    if (cont) {
        const double rzn = nc_precond(a, S, q, V.r + k0, V.z + k0, gb);
        const float beta = static_cast<float>(rzn / cs.rz);
#pragma unroll 4
    for (int i = threadIdx.x; i < K; i += TX_T) V.p[k0 + i] = fmaf(beta, V.p[k0 + i], V.z[k0 + i]);
        cs.rz = rzn;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        a.cgs[q] = cs;
        if (cs.mode == CG_ACTIVE) atomicAdd(count_next, 1);
    }
}

// ---------------------------------------------------------------------------
// The n_corr kernels.  Each pass is its own launch over the tiles of the
// launch range, or of the detscans a CG pass concerns (a list rebuilt after
// every CG update); the CG runs a fixed number of iterations as launches of
// their own (each returns at once when no detscan is iterating), and a
// cooperative tail kernel finishes any detscan still iterating (grid
// barriers between its passes; it returns at once when none is).
// ---------------------------------------------------------------------------
// Every work item of the launch range, grid-stride: neighbouring tiles run at
// the same time on neighbouring CTAs, so the runs of 64 to 256 bytes that a
// column tile reads and writes of every row come as whole rows while their
// DRAM pages are open (a contiguous share per CTA, one tile after the other:
// k_gain_cols on 82M samples 422 us, k_gain_colsinv 622; so 358, 509).
template <class Fn>
__device__ __forceinline__ void nc_items(const NcorrTx &a, TxCtx &X, bool rows, int &cur, Fn fn)
{
    const int2 *items = rows ? a.rowitems : a.colitems;
    const int j0 = rows ? a.row_off[a.q0] : a.col_off[a.q0];
    const int j1 = rows ? a.row_off[a.q1] : a.col_off[a.q1];
    const int64_t obase = a.off[a.q0];
    ItemFeed feed(X, items, a.q_tx, j0 + blockIdx.x, j1);
    for (int it = j0 + blockIdx.x; it < j1; it += gridDim.x) {
        tx_begin(X, feed, it, a.txl, a.off, obase, a.ndet, cur, a.qsc, a.cgs);
        fn();
    }
}

// The list of the launch range's detscans in CG mode `want` (ascending),
// with exclusive running counts of their column and row items.  One CTA
// builds it (modes read past L1: other CTAs of the launch have written them).
__device__ void nc_build_list(const NcorrTx &a, int want)
{
    __shared__ int s_w[32][3];
    __shared__ int s_base[3], s_tot[3];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    if (threadIdx.x == 0) { s_base[0] = 0; s_base[1] = 0; s_base[2] = 0; }
    __syncthreads();
    int32_t *lq = nl_q(a), *lc = nl_col(a), *lr = nl_row(a);
    for (int c0 = a.q0; c0 < a.q1; c0 += blockDim.x) {
        const int q = c0 + threadIdx.x;
        const bool in = q < a.q1 && __ldcg(&a.cgs[q].mode) == want;
        int v[3] = {in ? 1 : 0, in ? a.col_off[q + 1] - a.col_off[q] : 0, in ? a.row_off[q + 1] - a.row_off[q] : 0};
        int x[3];
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            int t = v[k];
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int u = __shfl_up_sync(0xffffffffu, t, o);
                if (lane >= o) t += u;
            }
            x[k] = t - v[k];                       // exclusive within the warp
            if (lane == 31) s_w[warp][k] = t;
        }
        __syncthreads();
        if (threadIdx.x < 3) {                     // warp totals -> exclusive warp offsets
            int acc = 0;
            for (int w = 0; w < nw; ++w) { const int t = s_w[w][threadIdx.x]; s_w[w][threadIdx.x] = acc; acc += t; }
            s_tot[threadIdx.x] = acc;
        }
        __syncthreads();
        if (in) {
            const int i = s_base[0] + s_w[warp][0] + x[0];
            lq[i] = q;
            lc[i] = s_base[1] + s_w[warp][1] + x[1];
            lr[i] = s_base[2] + s_w[warp][2] + x[2];
        }
        __syncthreads();
        if (threadIdx.x < 3) s_base[threadIdx.x] += s_tot[threadIdx.x];
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        a.list[0] = s_base[0];
        lc[s_base[0]] = s_base[1];
        lr[s_base[0]] = s_base[2];
    }
}
// Called by every CTA at the end of a launch that set the detscans' modes: the
// last one to arrive builds the list of those still iterating (a launch of
// its own for the list cost 3 us an iteration; count[2] counts arrivals).
__device__ void nc_list_by_last(const NcorrTx &a)
{
    __shared__ int s_last;
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        s_last = atomicAdd(a.count + 2, 1) == static_cast<int>(gridDim.x) - 1;
        __threadfence();
    }
    __syncthreads();
    if (!s_last) return;
    if (threadIdx.x == 0) a.count[2] = 0;
    nc_build_list(a, CG_ACTIVE);
}

// The listed detscans' column (or row) items, grid-stride.
template <class Fn>
__device__ __forceinline__ void nc_list_items(const NcorrTx &a, TxCtx &X, bool rows, int &cur, Fn fn)
{
    const int n = *reinterpret_cast<volatile const int32_t *>(a.list);
    if (n <= 0) return;
    const int32_t *lq = nl_q(a), *lo = rows ? nl_row(a) : nl_col(a);
    const int i0 = blockIdx.x, i1 = lo[n];
    const int64_t obase = a.off[a.q0];
    int pos = 0;                                  // last detscan whose items start at or before the current one
    for (int ii = i0; ii < i1; ii += gridDim.x) {
        // the detscan of item ii: the warp's lanes probe every 16th of the next 512,
        // then those between.  One step after the other walks a grid's worth of
        // detscans when they have one item each, in dependent loads (draw of 800 x
        // 2000 samples 883 us, by bisection 550, 530 so), and bisection takes more
        // of them than the walk when they have many (3600 x 144k: 40.60 ms, by
        // bisection 41.41, 39.67 so).
        const int lane = threadIdx.x & 31;
        for (int c = 32; c == 32; pos += 16 * c) {
            const int p = pos + 16 * (lane + 1);
            c = __popc(__ballot_sync(0xffffffffu, p < n && lo[min(p, n)] <= ii));
        }
        const int p = pos + lane + 1;
        pos += __popc(__ballot_sync(0xffffffffu, lane < 16 && p < n && lo[min(p, n)] <= ii));
        const int q = lq[pos];
        tx_begin(X, a.txl, a.q_tx[q], a.off, q, ii - lo[pos], obase, a.ndet, cur, a.qsc, a.cgs);
        fn();
    }
}


__global__ void __launch_bounds__(TX_T) k_nc_flag_count(NcorrTx a)
{
    __shared__ NcShared S;
    nc_flag_count(a, S);
}
__global__ void __launch_bounds__(TX_T) k_nc_flag_write(NcorrTx a)
{
    __shared__ NcShared S;
    nc_flag_write(a, S);
}
__global__ void __launch_bounds__(TX_T) k_nc_index(NcorrTx a)
{
    __shared__ NcShared S;
    if (blockIdx.x == 0 && threadIdx.x == 0) { a.count[0] = 0; a.count[1] = 0; a.count[2] = 0; }
    for (int q = a.q0 + blockIdx.x; q < a.q1; q += gridDim.x) {
        nc_detscan_index(a, S, q);
        __syncthreads();
    }
}
__global__ void __launch_bounds__(TX_T) k_nc_coarse(NcorrTx a)
{
    for (int q = a.q0 + blockIdx.x; q < a.q1; q += gridDim.x) {
        nc_resplit(a, q);
        nc_coarse_setup(a, q);
    }
}
__global__ void __launch_bounds__(TX_T, TX_CTAS_COL) k_nc_rhs_cols(NcorrTx a)
{
    extern __shared__ __align__(16) CF2 tx_smem[];
    __shared__ TxCtx X;
    const uint64_t gi = a.rng.gibbs_iter_dev ? *a.rng.gibbs_iter_dev : a.rng.gibbs_iter;
    int cur = -1;
    nc_items(a, X, false, cur, [&] { nc_rhs_cols(a, X, tx_smem, tx_smem + TX_PAIRS, gi); });
}
__global__ void __launch_bounds__(TX_T, 3) k_nc_rhs_rows(NcorrTx a)
{
    extern __shared__ __align__(16) CF2 tx_smem[];
    __shared__ TxCtx X;
    const uint64_t gi = a.rng.gibbs_iter_dev ? *a.rng.gibbs_iter_dev : a.rng.gibbs_iter;
    int cur = -1;
    nc_items(a, X, true, cur, [&] { nc_rhs_rows(a, X, tx_smem, tx_smem + TX_PAIRS, gi); });
}
__global__ void __launch_bounds__(TX_T, TX_CTAS_COL) k_nc_x0_cols(NcorrTx a)
{
    extern __shared__ __align__(16) CF2 tx_smem[];
    __shared__ TxCtx X;
    int cur = -1;
    nc_items(a, X, false, cur, [&] { nc_x0_cols(a, X, tx_smem, tx_smem + TX_PAIRS); });
}
__global__ void __launch_bounds__(TX_T, 3) k_nc_cg_init(NcorrTx a)
{
    extern __shared__ __align__(16) CF2 tx_smem[];
    __shared__ NcShared S;
    for (int q = a.q0 + blockIdx.x; q < a.q1; q += gridDim.x) {
        __syncthreads();
        nc_cg_init(a, S, q, reinterpret_cast<float *>(tx_smem));
    }
    nc_list_by_last(a);
}
// One CG iteration (parity par: count[par] active detscans going in, the
// update counts into count[par ^ 1]), or with FINAL the correction B^{-1} E y.
template <bool FINAL>
__global__ void __launch_bounds__(TX_T, 3) k_nc_scatter(NcorrTx a, int par)
{
    extern __shared__ __align__(16) CF2 tx_smem[];
    __shared__ TxCtx X;
    if (!FINAL) {
        if (blockIdx.x == 0 && threadIdx.x == 0) a.count[par ^ 1] = 0;
        if (*reinterpret_cast<volatile const int32_t *>(a.count + par) == 0) return;
    }
    const CgVec V = cg_vecs(a);
    int cur = -1;
    nc_list_items(a, X, false, cur, [&] { nc_scatter_cols(a, X, tx_smem, tx_smem + TX_PAIRS, FINAL ? V.y : V.p); });
}
template <bool FINAL>
__global__ void __launch_bounds__(TX_T, 3) k_nc_filter(NcorrTx a, int par)
{
    extern __shared__ __align__(16) CF2 tx_smem[];
    __shared__ TxCtx X;
    if (!FINAL && *reinterpret_cast<volatile const int32_t *>(a.count + par) == 0) return;
    int cur = -1;
    nc_list_items(a, X, true, cur, [&] { nc_filter_rows<FINAL>(a, X, tx_smem, tx_smem + TX_PAIRS); });
}
template <bool FINAL>
__global__ void __launch_bounds__(TX_T, TX_CTAS_COL) k_nc_gather(NcorrTx a, int par)
{
    extern __shared__ __align__(16) CF2 tx_smem[];
    __shared__ TxCtx X;
    if (!FINAL && *reinterpret_cast<volatile const int32_t *>(a.count + par) == 0) return;
    const CgVec V = cg_vecs(a);
    int cur = -1;
    nc_list_items(a, X, false, cur,
                  [&] { nc_gather_cols<FINAL>(a, X, tx_smem, tx_smem + TX_PAIRS, FINAL ? nullptr : V.q); });
}
// the listed (iterating) detscans' CG update
__device__ __forceinline__ void nc_update_listed(const NcorrTx &a, NcShared &S, float *gb, int32_t *count_next)
{
    const int n = *reinterpret_cast<volatile const int32_t *>(a.list);
    for (int i = blockIdx.x; i < n; i += gridDim.x) {
        __syncthreads();
        nc_cg_update(a, S, nl_q(a)[i], gb, count_next);
    }
}
__global__ void __launch_bounds__(TX_T, 3) k_nc_update(NcorrTx a, int par)
{
    extern __shared__ __align__(16) CF2 tx_smem[];
    __shared__ NcShared S;
    if (*reinterpret_cast<volatile const int32_t *>(a.count + par) == 0) return;
    nc_update_listed(a, S, reinterpret_cast<float *>(tx_smem), a.count + (par ^ 1));
    nc_list_by_last(a);
}
// The iterations left after the launched ones, in one cooperative launch, two
// CTAs per SM (at three, the bodies of all passes in one kernel spill 330 bytes:
// with PREC_NONE, most of whose iterations run here, the draw of 40 x 115k
// samples takes 3990 us, 3829 so; 72 x 225k 5312, 5226): the passes over the listed detscans with grid
// barriers between them, the list rebuilt by CTA 0 after each update.  Then
// the list of the detscans that ran the CG (for the correction), the
// iteration counts, and the status of detscans left at x0 for want of CG room.
__global__ void __launch_bounds__(TX_T, 2) k_nc_tail(NcorrTx a, int par)
{
    extern __shared__ __align__(16) CF2 tx_smem[];
    __shared__ NcShared S;
    cgrp::grid_group grid = cgrp::this_grid();
    const CgVec V = cg_vecs(a);
    int cur = -1;
    while (*reinterpret_cast<volatile const int32_t *>(a.count + par) != 0) {
        if (blockIdx.x == 0 && threadIdx.x == 0) a.count[par ^ 1] = 0;
        nc_list_items(a, S.X, false, cur, [&] { nc_scatter_cols(a, S.X, tx_smem, tx_smem + TX_PAIRS, V.p); });
        grid.sync();
        nc_list_items(a, S.X, true, cur, [&] { nc_filter_rows<false>(a, S.X, tx_smem, tx_smem + TX_PAIRS); });
        grid.sync();
        nc_list_items(a, S.X, false, cur, [&] { nc_gather_cols<false>(a, S.X, tx_smem, tx_smem + TX_PAIRS, V.q); });
        grid.sync();
        nc_update_listed(a, S, reinterpret_cast<float *>(tx_smem), a.count + (par ^ 1));
        grid.sync();
        par ^= 1;
        if (*reinterpret_cast<volatile const int32_t *>(a.count + par) == 0) break;
        if (blockIdx.x == 0) nc_build_list(a, CG_ACTIVE);
        grid.sync();
    }
    if (blockIdx.x == 0) nc_build_list(a, CG_DONE);
    for (int q = a.q0 + blockIdx.x * TX_T + threadIdx.x; q < a.q1; q += gridDim.x * TX_T) {
        if (a.iters) a.iters[q] = __ldcg(&a.cgs[q].it);
        if (__ldcg(&a.cgs[q].mode) == CG_OVER) set_status(a.status, q, TOD_ERR_NOT_CONVERGED);
    }
}

// ===========================================================================
// launchers
// ===========================================================================
static size_t tx_smem_bytes(bool fp64) { return (fp64 ? sizeof(CD2) : sizeof(CF2)) * 2 * TX_PAIRS; }
constexpr size_t kGbBytes = (GB_FLOATS + CZ_FLOATS) * sizeof(float);   // preconditioner staging
static_assert(kGbBytes <= sizeof(CF2) * 2 * TX_PAIRS, "the preconditioner staging fits the tile buffers");
// CG iterations as separate launches.  The two-level preconditioner takes 2.1
// on average and 4 to 5 at most on the 30 to 70 GHz bands; the rest runs in
// the cooperative tail, whose grid barriers cost what a launch does.  Launches
// past the last iteration return at once but cost 2 us each (four an
// iteration), and the tail costs as much as they do: three launched
// iterations leave it the few stragglers.  With eight the two-level draw of
// 16 x 4096 samples takes 465 us instead of 383, of 72 x 225k 2228 instead of
// 2175; without a preconditioner (12 and 21 iterations on average and at most)
// that of 72 x 225k 5102 instead of 5226, of 40 x 115k 3811 instead of 3829.
constexpr int NC_LAUNCHED_ITERS = 3;

template <class K>
static cudaError_t smem_attr(K k, size_t bytes) {
    return cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(bytes));
}

cudaError_t setup_tx_kernels(Plan &p)
{
    cudaError_t e;
    const size_t s32 = tx_smem_bytes(false), s64 = tx_smem_bytes(true);
    const size_t sgb = std::max(s32, kGbBytes);
    if ((e = smem_attr(k_gain_cols, s32)) || (e = smem_attr(k_gain_rows, s32)) || (e = smem_attr(k_gain_colsinv, s32)))
        return e;
    if ((e = smem_attr(k_chi2_cols<CF2>, s32)) || (e = smem_attr(k_chi2_rows<CF2>, s32)) ||
        (e = smem_attr(k_chi2_colsinv<CF2>, s32)))
        return e;
    if ((e = smem_attr(k_chi2_cols<CD2>, s64)) || (e = smem_attr(k_chi2_rows<CD2>, s64)) ||
        (e = smem_attr(k_chi2_colsinv<CD2>, s64)))
        return e;
    if ((e = smem_attr(k_nc_rhs_cols, s32)) || (e = smem_attr(k_nc_rhs_rows, s32)) ||
        (e = smem_attr(k_nc_x0_cols, s32)) || (e = smem_attr(k_nc_cg_init, sgb)) ||
        (e = smem_attr(k_nc_scatter<false>, s32)) || (e = smem_attr(k_nc_scatter<true>, s32)) ||
        (e = smem_attr(k_nc_filter<false>, s32)) || (e = smem_attr(k_nc_filter<true>, s32)) ||
        (e = smem_attr(k_nc_gather<false>, s32)) || (e = smem_attr(k_nc_gather<true>, s32)) ||
        (e = smem_attr(k_nc_update, sgb)) || (e = smem_attr(k_nc_tail, sgb)))
        return e;
    int dev = 0, nsm = 0, per = 0;
    if ((e = cudaGetDevice(&dev))) return e;
    if ((e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev))) return e;
    if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_nc_tail, TX_T, sgb))) return e;
    p.coop_grid = std::max(1, per) * nsm;
    if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_gain_rows, TX_T, s32))) return e;
    p.pass_grid = std::max(1, per) * nsm;
    p.sm_count = nsm;
    return cudaSuccess;
}

// persistent grids: the row passes', and that of kernels with `ctas` per SM
static int grid_for(const Plan &p, int nitems) { return std::max(1, std::min(nitems, p.pass_grid)); }
static int grid_ctas(const Plan &p, int nitems, int ctas) { return std::max(1, std::min(nitems, p.sm_count * ctas)); }

cudaError_t launch_tx_gain(const Plan &p, const float *d, const float *s, const uint32_t *flags, const double *psd,
                           tod_rng rng, int mode, double *g, double *mu, double *sig, cudaStream_t st, int q0, int q1)
{
    if (q1 <= q0) return cudaSuccess;
    GainTx a = {};
    a.d = d; a.s = s; a.flags = flags; a.psd = psd; a.off = p.off; a.txl = p.txl; a.q_tx = p.q_tx; a.tw = p.txtw;
    a.ndet = p.ndet; a.fsamp = p.fsamp; a.obase = p.h_off[q0]; a.Y = p.ybuf; a.part = p.part; a.qsc = p.qsc;
    const int c0 = p.h_col_off[q0], c1 = p.h_col_off[q1], r0 = p.h_row_off[q0], r1 = p.h_row_off[q1];
    const size_t sm = tx_smem_bytes(false);
    {
        KTIME(TOD_KT_DET_SCALARS);
        k_det_scalars<<<(q1 - q0 + 127) / 128, 128, 0, st>>>(psd, nullptr, p.off, p.ndet, p.fsamp, q0, q1, p.qsc);
    }
    // column items' partials at part[4 c], row items' at part[4 (ncol + r)]
    double *cpart = p.part;
    double *rpart = p.part + 4 * static_cast<int64_t>(p.h_col_off[p.nq]);
    a.items = p.colitems; a.item0 = c0; a.nitems = c1 - c0; a.part = cpart;
    {
        KTIME(TOD_KT_GAIN_COLS);
        k_gain_cols<<<grid_ctas(p, a.nitems, TX_CTAS_COL), TX_T, sm, st>>>(a);
    }
    a.items = p.rowitems; a.item0 = r0; a.nitems = r1 - r0; a.part = rpart;
    {
        KTIME(TOD_KT_GAIN_ROWS);
        k_gain_rows<<<grid_for(p, a.nitems), TX_T, sm, st>>>(a);
    }
    a.items = p.colitems; a.item0 = c0; a.nitems = c1 - c0; a.part = cpart;
    {
        KTIME(TOD_KT_GAIN_COLSINV);
        k_gain_colsinv<<<grid_ctas(p, a.nitems, TX_CTAS_COL), TX_T, sm, st>>>(a);
    }
    {
        KTIME(TOD_KT_GAIN_FIN);
        k_gain_fin<<<(q1 - q0 + 7) / 8, 256, 0, st>>>(rpart, cpart, p.row_off, p.col_off, q0, q1, rng, mode, g, mu, sig,
                                                      p.status);
    }
    return cudaGetLastError();
}

template <class V>
static cudaError_t chi2_range(const Plan &p, const float *d, const void *s, const double *gain,
                              const uint32_t *flags, const double *psd, double *chi2_q, double *dgain, double *dpsd_q,
                              void *v_out, cudaStream_t st, int q0, int q1)
{
    Chi2Tx<V> a = {};
    a.d = d; a.s = s; a.gain = gain; a.flags = flags; a.psd = psd; a.off = p.off; a.txl = p.txl; a.q_tx = p.q_tx;
    typedef typename PairOf<V>::Z Z;
    constexpr bool f32 = sizeof(Z) == sizeof(float2);
    a.tw = reinterpret_cast<const Z *>(f32 ? static_cast<const void *>(p.txtw) : static_cast<const void *>(p.txtw64));
    a.ndet = p.ndet; a.fsamp = p.fsamp; a.obase = p.h_off[q0];
    a.par = reinterpret_cast<double2 *>(p.qsc);
    a.Y = reinterpret_cast<Z *>(p.ybuf);
    a.v_out = v_out;
    a.v_al = (reinterpret_cast<uintptr_t>(v_out) & (sizeof(Z) - 1)) == 0;
    const size_t sm = tx_smem_bytes(!f32);
    const int c0 = p.h_col_off[q0], c1 = p.h_col_off[q1], r0 = p.h_row_off[q0], r1 = p.h_row_off[q1];
    double *cpart = p.part;
    double *rpart = p.part + 4 * static_cast<int64_t>(p.h_col_off[p.nq]);
    a.items = p.colitems; a.item0 = c0; a.nitems = c1 - c0; a.part = cpart;
    {
        KTIME(TOD_KT_CHI2_COLS);
        k_chi2_cols<V><<<grid_ctas(p, a.nitems, f32 ? TX_CTAS_COL : 3), TX_T, sm, st>>>(a);
    }
    a.items = p.rowitems; a.item0 = r0; a.nitems = r1 - r0; a.part = rpart;
    {
        KTIME(TOD_KT_CHI2_ROWS);
        k_chi2_rows<V><<<grid_ctas(p, a.nitems, f32 ? TX_CTAS_COL : 3), TX_T, sm, st>>>(a);
    }
    a.items = p.colitems; a.item0 = c0; a.nitems = c1 - c0; a.part = cpart;
    {
        KTIME(TOD_KT_CHI2_COLSINV);
        k_chi2_colsinv<V><<<grid_ctas(p, a.nitems, f32 ? TX_CTAS_COL : 3), TX_T, sm, st>>>(a);
    }
    {
        KTIME(TOD_KT_CHI2_FIN);
        k_chi2_fin<<<(q1 - q0 + 7) / 8, 256, 0, st>>>(rpart, cpart, p.row_off, p.col_off, q0, q1, chi2_q, dgain, dpsd_q);
    }
    return cudaGetLastError();
}

cudaError_t launch_tx_chi2(const Plan &p, bool fp64, const float *d, const void *s, const double *gain,
                           const uint32_t *flags, const double *psd, double *chi2_q, double *dgain, double *dpsd_q,
                           double *total, double *dpsd_det, void *v_out, cudaStream_t st)
{
    cudaError_t e = cudaSuccess;
    if (!fp64) {
        e = chi2_range<CF2>(p, d, s, gain, flags, psd, chi2_q, dgain, dpsd_q, v_out, st, 0, p.nq);
    } else {
        // the intermediate holds ybuf_floats / 4 double2: waves of detscans of
        // at most ybuf_floats / 2 samples (a whole detscan always fits)
        int q = 0;
        while (q < p.nq && e == cudaSuccess) {
            int q1 = q + 1;
            while (q1 < p.nq && p.h_off[q1 + 1] - p.h_off[q] <= p.ybuf_floats / 2) ++q1;
            e = chi2_range<CD2>(p, d, s, gain, flags, psd, chi2_q, dgain, dpsd_q, v_out, st, q, q1);
            q = q1;
        }
    }
    if (e != cudaSuccess) return e;
    {
        KTIME(TOD_KT_CHI2_FIN);
        k_chi2_total<<<1 + p.ndet, TX_T, 0, st>>>(chi2_q, dpsd_q, p.nq, p.ndet, total, dpsd_det);
    }
    return cudaGetLastError();
}

cudaError_t launch_tx_ncorr(const Plan &p, const float *d, const float *s, const double *gain,
                            const uint32_t *flags, const double *psd, tod_rng rng, int mode, float tol, int maxit,
                            float *x, int32_t *iters, cudaStream_t st, int q0, int q1, const TxNcorrScratch &sc,
                            int grid, cudaEvent_t prepared)
{
    if (q1 <= q0) return cudaSuccess;
    NcorrTx a = {};
    a.d = d; a.s = s; a.gain = gain; a.flags = flags; a.psd = psd; a.off = p.off; a.txl = p.txl; a.q_tx = p.q_tx;
    a.tw = p.txtw; a.colitems = p.colitems; a.rowitems = p.rowitems; a.col_off = p.col_off; a.row_off = p.row_off;
    a.q0 = q0; a.q1 = q1; a.ndet = p.ndet; a.fsamp = p.fsamp; a.rng = rng; a.mode = mode; a.tol = tol;
    a.maxit = maxit; a.x_out = x; a.iters = iters; a.status = p.status; a.spec_out = p.spec_out;
    a.xtab = p.use_prec ? p.xtab : nullptr; a.lvalid = p.lvalid;
    a.cztab = p.cztab; a.href = p.cz_href; a.gbpos = p.gbpos; a.czsz = (p.use_prec && p.use_coarse) ? p.czsz : nullptr;
    a.czcap = p.czcap; a.czl = p.czl;
    a.Y = sc.Y; a.wpre = sc.wpre; a.chunk = p.chunk; a.cgs = p.cgs; a.gblk = p.gblk; a.gnb = p.gnb;
    a.cgv = sc.cgv; a.cgcap = sc.cgcap; a.count = p.cg_count; a.qsc = p.qsc; a.list = p.nclist;
    const size_t s32 = tx_smem_bytes(false), sgb = std::max(s32, kGbBytes);
    const int nq = q1 - q0;
    const int ncol = p.h_col_off[q1] - p.h_col_off[q0], nrow = p.h_row_off[q1] - p.h_row_off[q0];
    const int gc = std::min(grid_for(p, ncol), grid), gr = std::min(grid_for(p, nrow), grid);
    const int gc2 = std::min(gc, grid_ctas(p, ncol, TX_CTAS_COL));
    const int gq = std::min(nq, std::max(1, grid));
    // flag index (count and write use the same grid)
    const int gf = std::max(1, std::min(p.pass_grid, grid));
    {
        KTIME(TOD_KT_NC_FLAG_COUNT);
        k_nc_flag_count<<<gf, TX_T, 0, st>>>(a);
    }
    {
        KTIME(TOD_KT_NC_FLAG_WRITE);
        k_nc_flag_write<<<gf, TX_T, 0, st>>>(a);
    }
    {
        KTIME(TOD_KT_NC_INDEX);
        k_nc_index<<<gq, TX_T, 0, st>>>(a);
    }
    // x0 = B^{-1} b
    {
        KTIME(TOD_KT_NC_RHS_COLS);
        k_nc_rhs_cols<<<gc2, TX_T, s32, st>>>(a);
    }
    {
        KTIME(TOD_KT_NC_RHS_ROWS);
        k_nc_rhs_rows<<<gr, TX_T, s32, st>>>(a);
    }
    {
        KTIME(TOD_KT_NC_X0_COLS);
        k_nc_x0_cols<<<gc2, TX_T, s32, st>>>(a);
    }
    // CG on the Schur complement
    if (prepared) {
        const cudaError_t ew = cudaStreamWaitEvent(st, prepared, 0);
        if (ew != cudaSuccess) return ew;
    }
    {
        KTIME(TOD_KT_NC_COARSE);
        k_nc_coarse<<<gq, TX_T, 0, st>>>(a);
    }
    {
        KTIME(TOD_KT_NC_CG_INIT);
        k_nc_cg_init<<<gq, TX_T, sgb, st>>>(a);
    }
    int par = 0;
    for (int it = 0; it < NC_LAUNCHED_ITERS; ++it, par ^= 1) {
        {
            KTIME(TOD_KT_NC_SCATTER);
            k_nc_scatter<false><<<gc, TX_T, s32, st>>>(a, par);
        }
        {
            KTIME(TOD_KT_NC_FILTER);
            k_nc_filter<false><<<gr, TX_T, s32, st>>>(a, par);
        }
        {
            KTIME(TOD_KT_NC_GATHER);
            k_nc_gather<false><<<gc2, TX_T, s32, st>>>(a, par);
        }
        {
            KTIME(TOD_KT_NC_UPDATE);
            k_nc_update<<<gq, TX_T, sgb, st>>>(a, par);
        }
    }
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    int tail_par = par;
    void *args[] = {&a, &tail_par};
    {
        KTIME(TOD_KT_NC_TAIL);
        e = cudaLaunchCooperativeKernel(reinterpret_cast<const void *>(k_nc_tail),
                                        dim3(std::max(1, std::min(grid, p.coop_grid))), dim3(TX_T), args, sgb, st);
    }
    if (e != cudaSuccess) return e;
    // x = x0 + B^{-1} E y for every detscan that ran the CG
    {
        KTIME(TOD_KT_NC_SCATTER_FINAL);
        k_nc_scatter<true><<<gc, TX_T, s32, st>>>(a, 0);
    }
    {
        KTIME(TOD_KT_NC_FILTER_FINAL);
        k_nc_filter<true><<<gr, TX_T, s32, st>>>(a, 0);
    }
    {
        KTIME(TOD_KT_NC_GATHER_FINAL);
        k_nc_gather<true><<<gc2, TX_T, s32, st>>>(a, 0);
    }
    return cudaGetLastError();
}

}  // namespace tg

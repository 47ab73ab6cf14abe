// Packed complex arithmetic, register DFTs and one Stockham pass over a tile
// of vectors in shared memory.
//
// The transform passes work on pairs of complex values: two lanes a, b that
// go through the same butterflies (two columns of a column tile, two rows of
// a row tile), stored as (re_a, re_b, im_a, im_b).  In FP32 an operation on
// both lanes is one packed instruction (add/mul/fma.f32x2, sm_100 and
// later): the FP32 pipe does the same number of operations a cycle either
// way, but half the issue slots go to them, and shared-memory accesses,
// twiddle loads and index arithmetic are per pair too (the passes are bound
// by instruction issue).  In FP64 the pair is two scalars.  Every routine is
// written once: V is a complex type with components of type C (float2 with
// float, Cx2<PF> with PF, Cx2<PD> with PD).
#pragma once
#include <cstdint>
#include <cuda_runtime.h>
#include "internal.cuh"

namespace tg {

// ---------------------------------------------------------------------------
// component types: a scalar or a pair of lanes
// ---------------------------------------------------------------------------
struct alignas(8) PF { float a, b; };
struct alignas(16) PD { double a, b; };
template <class P> struct alignas(2 * sizeof(P)) Cx2 { P x, y; };
typedef Cx2<PF> CF2;
typedef Cx2<PD> CD2;

template <class C> struct ScalarOf { typedef C S; };
template <> struct ScalarOf<PF> { typedef float S; };
template <> struct ScalarOf<PD> { typedef double S; };
template <class V> struct VecT { typedef decltype(V::x) C; typedef typename ScalarOf<C>::S S; };

__device__ __forceinline__ float2 pf2(PF p) { return make_float2(p.a, p.b); }
__device__ __forceinline__ PF f2p(float2 v) { return PF{v.x, v.y}; }
__device__ __forceinline__ PF pset(float a, float b) { return PF{a, b}; }
__device__ __forceinline__ PD pset(double a, double b) { return PD{a, b}; }
template <class C> __device__ __forceinline__ C pdup(typename ScalarOf<C>::S s);
template <> __device__ __forceinline__ float pdup<float>(float s) { return s; }
template <> __device__ __forceinline__ PF pdup<PF>(float s) { return PF{s, s}; }
template <> __device__ __forceinline__ PD pdup<PD>(double s) { return PD{s, s}; }

__device__ __forceinline__ float padd(float a, float b) { return a + b; }
__device__ __forceinline__ float psub(float a, float b) { return a - b; }
__device__ __forceinline__ float pmul(float a, float b) { return a * b; }
__device__ __forceinline__ float pfma(float a, float b, float c) { return fmaf(a, b, c); }
__device__ __forceinline__ float pneg(float a) { return -a; }
__device__ __forceinline__ PF padd(PF a, PF b) { return f2p(__fadd2_rn(pf2(a), pf2(b))); }
__device__ __forceinline__ PF pmul(PF a, PF b) { return f2p(__fmul2_rn(pf2(a), pf2(b))); }
__device__ __forceinline__ PF pfma(PF a, PF b, PF c) { return f2p(__ffma2_rn(pf2(a), pf2(b), pf2(c))); }
// a sign, a swap of the lanes or one scalar in both lanes is a modifier of the
// packed instruction that takes it as an operand: none costs an instruction
__device__ __forceinline__ PF pneg(PF a) { return PF{-a.a, -a.b}; }
__device__ __forceinline__ PF psub(PF a, PF b) { return padd(a, pneg(b)); }
__device__ __forceinline__ PD padd(PD a, PD b) { return PD{a.a + b.a, a.b + b.b}; }
__device__ __forceinline__ PD psub(PD a, PD b) { return PD{a.a - b.a, a.b - b.b}; }
__device__ __forceinline__ PD pmul(PD a, PD b) { return PD{a.a * b.a, a.b * b.b}; }
__device__ __forceinline__ PD pfma(PD a, PD b, PD c) { return PD{fma(a.a, b.a, c.a), fma(a.b, b.b, c.b)}; }
__device__ __forceinline__ PD pneg(PD a) { return PD{-a.a, -a.b}; }
__device__ __forceinline__ PF pswap(PF a) { return PF{a.b, a.a}; }
__device__ __forceinline__ PD pswap(PD a) { return PD{a.b, a.a}; }

// ---------------------------------------------------------------------------
// complex arithmetic
// ---------------------------------------------------------------------------
template <class V> __device__ __forceinline__ V vmake(typename VecT<V>::C a, typename VecT<V>::C b) {
    V v;
    v.x = a;
    v.y = b;
    return v;
}
template <class V> __device__ __forceinline__ V vadd(V a, V b) { return vmake<V>(padd(a.x, b.x), padd(a.y, b.y)); }
template <class V> __device__ __forceinline__ V vsub(V a, V b) { return vmake<V>(psub(a.x, b.x), psub(a.y, b.y)); }
// a b (INV: a conj(b)), each part one product and one fused product-sum
template <bool INV = false, class V> __device__ __forceinline__ V vmul(V a, V b) {
    const auto ny = pneg(b.y);
    const auto wp = INV ? b.y : ny, wm = INV ? ny : b.y;
    return vmake<V>(pfma(a.y, wp, pmul(a.x, b.x)), pfma(a.x, wm, pmul(a.y, b.x)));
}
// a +- i b
template <bool PLUS, class V> __device__ __forceinline__ V vaddi(V a, V b) {
    return PLUS ? vmake<V>(psub(a.x, b.y), padd(a.y, b.x)) : vmake<V>(padd(a.x, b.y), psub(a.y, b.x));
}
// lanes swapped
template <class V> __device__ __forceinline__ V vswap(V v) { return vmake<V>(pswap(v.x), pswap(v.y)); }
template <class V> __device__ __forceinline__ V vzero() {
    typedef typename VecT<V>::C C;
    return vmake<V>(pdup<C>(0), pdup<C>(0));
}
__device__ __forceinline__ float2 vld(const float2 *p) { return __ldg(p); }
__device__ __forceinline__ double2 vld(const double2 *p) { return __ldg(p); }
__device__ __forceinline__ CF2 vld(const CF2 *p) {
    const float4 v = __ldg(reinterpret_cast<const float4 *>(p));
    return CF2{{v.x, v.y}, {v.z, v.w}};
}
__device__ __forceinline__ CD2 vld(const CD2 *p) {
    const double2 x = __ldg(reinterpret_cast<const double2 *>(p)), y = __ldg(reinterpret_cast<const double2 *>(p) + 1);
    return CD2{{x.x, x.y}, {y.x, y.y}};
}
// shared-memory accesses of a pair as 16-byte words
__device__ __forceinline__ CF2 sld(const CF2 *p) {
    const float4 v = *reinterpret_cast<const float4 *>(p);
    return CF2{{v.x, v.y}, {v.z, v.w}};
}
__device__ __forceinline__ void sst(CF2 *p, const CF2 &v) {
    *reinterpret_cast<float4 *>(p) = make_float4(v.x.a, v.x.b, v.y.a, v.y.b);
}
__device__ __forceinline__ CD2 sld(const CD2 *p) { return *p; }
__device__ __forceinline__ void sst(CD2 *p, const CD2 &v) { *p = v; }

// ---------------------------------------------------------------------------
// Twiddle constants of the composite register DFTs: cos and sin of 2 pi j/R
// from Taylor series after a quarter-turn reduction (|x| < pi/2, 14 terms:
// below 1e-17), evaluated by the compiler.
// ---------------------------------------------------------------------------
constexpr double kTwoPiR = 6.283185307179586476925286766559;
__host__ __device__ constexpr double rq_sin(double x) {
    double term = x, sum = x;
    for (int i = 1; i < 14; ++i) { term *= -x * x / ((2.0 * i) * (2.0 * i + 1.0)); sum += term; }
    return sum;
}
__host__ __device__ constexpr double rq_cos(double x) {
    double term = 1.0, sum = 1.0;
    for (int i = 1; i < 14; ++i) { term *= -x * x / ((2.0 * i - 1.0) * (2.0 * i)); sum += term; }
    return sum;
}
__host__ __device__ constexpr double turn_cos(int j, int R) {
    const int jj = ((j % R) + R) % R;
    const int q = (4 * jj) / R, rem = 4 * jj - q * R;
    const double x = 0.25 * kTwoPiR * rem / R;
    return q == 0 ? rq_cos(x) : q == 1 ? -rq_sin(x) : q == 2 ? -rq_cos(x) : rq_sin(x);
}
__host__ __device__ constexpr double turn_sin(int j, int R) {
    const int jj = ((j % R) + R) % R;
    const int q = (4 * jj) / R, rem = 4 * jj - q * R;
    const double x = 0.25 * kTwoPiR * rem / R;
    return q == 0 ? rq_sin(x) : q == 1 ? rq_cos(x) : q == 2 ? -rq_sin(x) : -rq_cos(x);
}
// a k + c and a k for a constant k
template <class C> __device__ __forceinline__ C pfmak(C a, typename ScalarOf<C>::S k, C c) { return pfma(a, pdup<C>(k), c); }
template <class C> __device__ __forceinline__ C pmulk(C a, typename ScalarOf<C>::S k) { return pmul(a, pdup<C>(k)); }
// v * W_R^J with W = exp(-+2 pi i/R); exact at the quarter turns
template <int R, int J, bool INV, class V>
__device__ __forceinline__ V rtwiddle(V v) {
    typedef typename VecT<V>::S S;
    constexpr int j = J % R;
    if constexpr (j == 0) return v;
    else if constexpr (2 * j == R) return vmake<V>(pneg(v.x), pneg(v.y));
    else if constexpr (4 * j == R) return INV ? vmake<V>(pneg(v.y), v.x) : vmake<V>(v.y, pneg(v.x));
    else if constexpr (4 * j == 3 * R) return INV ? vmake<V>(v.y, pneg(v.x)) : vmake<V>(pneg(v.y), v.x);
    else {
        constexpr S c = static_cast<S>(turn_cos(j, R));
        constexpr S sn = static_cast<S>(INV ? turn_sin(j, R) : -turn_sin(j, R));
        return vmake<V>(pfmak(v.y, -sn, pmulk(v.x, c)), pfmak(v.x, sn, pmulk(v.y, c)));
    }
}

// ---------------------------------------------------------------------------
// Register DFTs of radix 2, 3, 4, 5 (textbook butterflies) and composite
// radices by Cooley-Tukey in registers.  Sign -1 forward, +1 inverse; no
// normalisation.
// ---------------------------------------------------------------------------
template <int R, bool INV, class V> struct RDft;

template <bool INV, class V> struct RDft<2, INV, V> {
    static __device__ __forceinline__ void run(V *v) {
        const V a = v[0], b = v[1];
        v[0] = vadd(a, b);
        v[1] = vsub(a, b);
    }
};
template <bool INV, class V> struct RDft<3, INV, V> {
    static __device__ __forceinline__ void run(V *v) {
        typedef typename VecT<V>::S S;
        const S s3 = static_cast<S>(0.86602540378443864676);
        const V a = v[0], t1 = vadd(v[1], v[2]), dd = vsub(v[1], v[2]);
        const V t2 = vmake<V>(pfmak(t1.x, static_cast<S>(-0.5), a.x), pfmak(t1.y, static_cast<S>(-0.5), a.y));
        const S sp = INV ? s3 : -s3;
        v[0] = vadd(a, t1);
        v[1] = vmake<V>(pfmak(dd.y, -sp, t2.x), pfmak(dd.x, sp, t2.y));      // t2 + i sp dd
        v[2] = vmake<V>(pfmak(dd.y, sp, t2.x), pfmak(dd.x, -sp, t2.y));
    }
};
template <bool INV, class V> struct RDft<4, INV, V> {
    static __device__ __forceinline__ void run(V *v) {
        const V s0 = vadd(v[0], v[2]), d0 = vsub(v[0], v[2]);
        const V s1 = vadd(v[1], v[3]), d1 = vsub(v[1], v[3]);
        v[0] = vadd(s0, s1);
        v[2] = vsub(s0, s1);
        v[1] = vaddi<INV>(d0, d1);
        v[3] = vaddi<!INV>(d0, d1);
    }
};
template <bool INV, class V> struct RDft<5, INV, V> {
    static __device__ __forceinline__ void run(V *v) {
        typedef typename VecT<V>::S S;
        const S c1 = static_cast<S>(0.30901699437494742410), c2 = static_cast<S>(-0.80901699437494742410);
        const S s1 = static_cast<S>(0.95105651629515357212), s2 = static_cast<S>(0.58778525229247312917);
        const V a = v[0];
        const V be = vadd(v[1], v[4]), bm = vsub(v[1], v[4]);
        const V cd = vadd(v[2], v[3]), cm = vsub(v[2], v[3]);
        const V r1 = vmake<V>(pfmak(cd.x, c2, pfmak(be.x, c1, a.x)), pfmak(cd.y, c2, pfmak(be.y, c1, a.y)));
        const V r2 = vmake<V>(pfmak(cd.x, c1, pfmak(be.x, c2, a.x)), pfmak(cd.y, c1, pfmak(be.y, c2, a.y)));
        const V q1 = vmake<V>(pfmak(cm.x, s2, pmulk(bm.x, s1)), pfmak(cm.y, s2, pmulk(bm.y, s1)));
        const V q2 = vmake<V>(pfmak(cm.x, -s1, pmulk(bm.x, s2)), pfmak(cm.y, -s1, pmulk(bm.y, s2)));
        v[0] = vadd(a, vadd(be, cd));
        v[1] = vaddi<INV>(r1, q1);
        v[4] = vaddi<!INV>(r1, q1);
        v[2] = vaddi<INV>(r2, q2);
        v[3] = vaddi<!INV>(r2, q2);
    }
};

__host__ __device__ constexpr int rdft_first(int R) {
    return (R % 4 == 0) ? 4 : (R % 3 == 0) ? 3 : (R % 5 == 0) ? 5 : 2;
}
// R = A B: X[k1 + A k2] = sum_n2 W_B^{n2 k2} W_R^{n2 k1} sum_n1 x[B n1 + n2] W_A^{n1 k1}
template <int A, int B, bool INV, class V> struct RDftAB {
    template <int N2, int K1>
    static __device__ __forceinline__ void tw(V *u) {
        if constexpr (K1 < A) {
            u[K1] = rtwiddle<A * B, N2 * K1, INV>(u[K1]);
            tw<N2, K1 + 1>(u);
        }
    }
    template <int N2>
    static __device__ __forceinline__ void inner(const V *v, V (&t)[B][A]) {
        if constexpr (N2 < B) {
            V u[A];
#pragma unroll
            for (int n1 = 0; n1 < A; ++n1) u[n1] = v[B * n1 + N2];
            RDft<A, INV, V>::run(u);
            tw<N2, 0>(u);
#pragma unroll
            for (int k1 = 0; k1 < A; ++k1) t[N2][k1] = u[k1];
            inner<N2 + 1>(v, t);
        }
    }
    static __device__ __forceinline__ void run(V *v) {
        V t[B][A];
        inner<0>(v, t);
#pragma unroll
        for (int k1 = 0; k1 < A; ++k1) {
            V w[B];
#pragma unroll
            for (int n2 = 0; n2 < B; ++n2) w[n2] = t[n2][k1];
            RDft<B, INV, V>::run(w);
#pragma unroll
            for (int k2 = 0; k2 < B; ++k2) v[k1 + A * k2] = w[k2];
        }
    }
};
template <int R, bool INV, class V> struct RDft {
    static_assert(R % rdft_first(R) == 0 && R / rdft_first(R) > 1, "composite radix");
    static __device__ __forceinline__ void run(V *v) { RDftAB<rdft_first(R), R / rdft_first(R), INV, V>::run(v); }
};

// ---------------------------------------------------------------------------
// One out-of-place Stockham pass (radix R after Ns points are done) over
// the 2^lgv vectors of length L of a tile in shared memory: element e of
// vector c at c + e 2^lgv (COL: a tile of columns) or c * stride + e (rows).
// Thread t keeps vector t mod 2^lgv (2^lgv divides NT) and takes the
// butterflies j = t >> lgv, j + (NT >> lgv), ..; pass twiddles
// W_L^{r k L/(Ns R)} (k = j mod Ns) from tw (W_L^i in both lanes, i < L,
// global).  The caller synchronises.  Radices 10, 9, 8, 6, 5, 4, 3, 2 (a
// radix-16 butterfly of pairs needs 64 registers for its values alone).
// ---------------------------------------------------------------------------
template <int R, bool INV, int NT, bool COL, class V>
__device__ __forceinline__ void sp_pass(const V *__restrict__ src, V *__restrict__ dst, int L, const DctStage &st,
                                        int lgv, int stride, const V *__restrict__ tw)
{
    const int LR = L / R;
    const int Ns = st.Ns;
    const int tstep = fdiv(LR, st.fNs);                                             // L / (Ns R)
    const int vec = threadIdx.x & ((1 << lgv) - 1);
    const int es = COL ? (1 << lgv) : 1;
    const int base = COL ? vec : vec * stride;
    const V *s0 = src + base;
    V *d0 = dst + base;
    const int ls = LR * es, ns = Ns * es;
    for (int j = threadIdx.x >> lgv; j < LR; j += NT >> lgv) {
        const V *p = s0 + j * es;
        V v[R];
#pragma unroll
        for (int r = 0; r < R; ++r) v[r] = sld(p + r * ls);
        const int jq = fdiv(j, st.fNs);
        const int k = j - jq * Ns;
        if (Ns > 1) {
            const int ts = k * tstep;
#pragma unroll
            for (int r = 1; r < R; ++r) v[r] = vmul<INV>(v[r], vld(tw + r * ts));
        }
        RDft<R, INV, V>::run(v);
        V *q = d0 + (jq * Ns * R + k) * es;
#pragma unroll
        for (int r = 0; r < R; ++r) sst(q + r * ns, v[r]);
    }
}

// All passes of a sub-transform, ping-ponging between the two tile buffers
// (a barrier after each); returns the buffer holding the result.
template <bool INV, int NT, bool COL, class V>
__device__ V *sp_transform(V *a, V *b, int L, const DctStage *stages, int nr, int lgv, int stride,
                           const V *__restrict__ tw)
{
    for (int s = 0; s < nr; ++s) {
        const DctStage st = stages[s];
        switch (st.R) {
        case 10: sp_pass<10, INV, NT, COL>(a, b, L, st, lgv, stride, tw); break;
        case 9: sp_pass<9, INV, NT, COL>(a, b, L, st, lgv, stride, tw); break;
        case 8: sp_pass<8, INV, NT, COL>(a, b, L, st, lgv, stride, tw); break;
        case 6: sp_pass<6, INV, NT, COL>(a, b, L, st, lgv, stride, tw); break;
        case 5: sp_pass<5, INV, NT, COL>(a, b, L, st, lgv, stride, tw); break;
        case 4: sp_pass<4, INV, NT, COL>(a, b, L, st, lgv, stride, tw); break;
        case 3: sp_pass<3, INV, NT, COL>(a, b, L, st, lgv, stride, tw); break;
        default: sp_pass<2, INV, NT, COL>(a, b, L, st, lgv, stride, tw); break;
        }
        __syncthreads();
        V *t = a; a = b; b = t;
    }
    return a;
}

}  // namespace tg

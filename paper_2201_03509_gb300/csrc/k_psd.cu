// A10 noise PSD step: random-walk Metropolis on (ln f_knee, alpha) of every
// detector, from the DCT spectra of the n_corr draws (the paper lists the
// noise PSD step among the TOD steps of Sect. 5 and defers its sampler to
// the noise companion paper; the reading taken is the Gaussian density of
// n_corr under its 1/f prior, sigma0 fixed, flat prior on a box).
//
// With L = ln f_knee, a = alpha, N the detector's modes k >= 1 and
// f_{q,k} = k fsamp / (2 n_q) = k e^{c_q}:
//   ln L(L, a) = -1/2 [ e^{a L} / sigma0^2 S(a) + N ln sigma0^2
//                       + a (sum ln f - N L) ],
//   S(a) = sum_q e^{-a c_q} sum_{k>=1} xhat_{q,k}^2 k^{-a}.
// One evaluation is one pass over the spectra (k_psd_sums, one CTA per
// element tile of a detscan, partial sums per tile) and a fixed-order
// reduction per detector (k_psd_step), which also takes the Metropolis
// decision, draws the next proposal and forms its detscan factors
// e^{-a c_q}.  Deterministic.  An FP64 transcendental takes microseconds on
// this part (a chain of dependent operations at 1/64 of the FP32 rate), so
// the sums' CTAs take none and the
// step's run on different warps at once.  27M samples: an evaluation 61 ->
// 50 us, a step 17.7 -> 14.4 us.
#include <algorithm>
#include "common.cuh"
#include "fft_reg.cuh"
#include "internal.cuh"

namespace tg {

namespace {

constexpr int PSD_T = 256;
// state per detector: ln f_knee, alpha, ln L, proposal (ln f_knee, alpha,
// in box), accepted count
constexpr int PS_LNFK = 0, PS_AL = 1, PS_LOGL = 2, PS_PLNFK = 3, PS_PAL = 4, PS_PVALID = 5, PS_ACC = 6;

__device__ __forceinline__ bool psd_in_box(double lnfk, double al) {
    return lnfk >= TOD_PSD_LNFK_MIN && lnfk <= TOD_PSD_LNFK_MAX && al >= TOD_PSD_ALPHA_MIN &&
           al <= TOD_PSD_ALPHA_MAX;
}

// The numbers of Metropolis step `step` of detector det: 53-bit uniforms
// from words 0 and 1 (Box-Muller pair of the proposal), word 2 (acceptance).
__device__ void psd_numbers(const tod_rng &rng, uint64_t it, int det, int step, double &z1, double &z2,
                            double &ua)
{
    const u64x4 w = philox4x64(static_cast<uint64_t>(step), static_cast<uint64_t>(det), TOD_PURPOSE_PSD, it,
                               rng.seed, rng.band);
    const double u1 = (static_cast<double>(w.x[0] >> 11) + 0.5) * 1.1102230246251565e-16;
    const double u2 = (static_cast<double>(w.x[1] >> 11) + 0.5) * 1.1102230246251565e-16;
    ua = (static_cast<double>(w.x[2] >> 11) + 0.5) * 1.1102230246251565e-16;
    const double r = sqrt(-2.0 * log(u1));
    z1 = r * cospi(2.0 * u2);
    z2 = r * sinpi(2.0 * u2);
}

// The factors e^{-alpha c_q} of a detector's detscans (the CTA's threads).
__device__ __forceinline__ void psd_factors(double al, int det, int ndet, int nq, const double *__restrict__ lnfs,
                                            double *__restrict__ wq)
{
    for (int q = det + ndet * static_cast<int>(threadIdx.x); q < nq; q += ndet * PSD_T) wq[q] = exp(-al * lnfs[q]);
}

__global__ void __launch_bounds__(PSD_T) k_psd_begin(const double *__restrict__ psd_in, double *state, int ndet,
                                                     int nq, const double *__restrict__ lnfs, double *wq,
                                                     double *psd_out, int32_t *acc_out)
{
    const int det = blockIdx.x;
    const double fk = psd_in[3 * det + 1], al = psd_in[3 * det + 2];
    psd_factors(al, det, ndet, nq, lnfs, wq);
    if (threadIdx.x != 0) return;
    double *st = state + 8 * det;
    st[PS_LNFK] = log(fk);
    st[PS_AL] = al;
    st[PS_LOGL] = 0.0;
    st[PS_PLNFK] = st[PS_LNFK];        // the first evaluation is at the current state
    st[PS_PAL] = al;
    st[PS_PVALID] = 1.0;
    st[PS_ACC] = 0.0;
    psd_out[3 * det] = psd_in[3 * det];
    psd_out[3 * det + 1] = fk;
    psd_out[3 * det + 2] = al;
    if (acc_out) acc_out[det] = 0;
}

// partial S(alpha') of `per` (at most PSD_TILES) consecutive element tiles (each
// one detscan's samples t0..t1).  The tiles' parameters take a chain of three
// dependent loads, longer than a tile's work: fetched once for all of them by
// the first lanes.
// Several tiles a CTA only once the grid keeps PSD_CTAS CTAs on every SM: below,
// a tile's work is not shared with anything and the tiles of a CTA just wait for
// one another.
constexpr int PSD_TILES = 4, PSD_CTAS = 4;
__global__ void __launch_bounds__(PSD_T) k_psd_sums(const float *__restrict__ spec, const int64_t *__restrict__ off,
                                                    const int32_t *__restrict__ tile_q,
                                                    const int64_t *__restrict__ tile_t0, int ntile, int per,
                                                    const double *__restrict__ wq, const float2 *__restrict__ lnk,
                                                    const double *__restrict__ state, int ndet,
                                                    double *__restrict__ part)
{
    struct Tile { const float *x; int k0, k1; float na, na_lo; double w; };
    __shared__ Tile s_tile[PSD_TILES];
    __shared__ double s_w[PSD_TILES][PSD_T / 32];
    const int first = blockIdx.x * per, nt = min(per, ntile - first);
    if (threadIdx.x < nt) {
        const int q = tile_q[first + threadIdx.x];
        const int64_t t0 = tile_t0[first + threadIdx.x];
        const double *st = state + 8 * (q % ndet);
        const int64_t o = off[q], n = off[q + 1] - o;
        const double al = st[PS_PAL];
        Tile t;
        t.x = spec + o;
        t.k0 = static_cast<int>(t0 - o);
        t.k1 = static_cast<int>(min(static_cast<int64_t>(t.k0) + ELEM_TILE, n));
        t.na = static_cast<float>(-al);
        t.na_lo = static_cast<float>(-al - static_cast<double>(t.na));
        t.w = wq[q];
        if (st[PS_PVALID] == 0.0) t.k1 = t.k0;         // proposal outside the box: rejected anyway
        s_tile[threadIdx.x] = t;
    }
    __syncthreads();
    for (int j = 0; j < nt; ++j) {
        const Tile T = s_tile[j];
        // eight modes per thread and round, every load in flight; the
        // double-word sums of two modes are the lanes of packed operations
        constexpr int U = 8;
        const PF nh = pdup<PF>(T.na), nl = pdup<PF>(T.na_lo);
        PF as[U / 2], ac[U / 2];
#pragma unroll
        for (int u = 0; u < U / 2; ++u) as[u] = ac[u] = PF{0.f, 0.f};
        for (int kb = T.k0 + static_cast<int>(threadIdx.x); kb < T.k1; kb += U * PSD_T) {
            float x[U];
            float2 l[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int k = kb + u * PSD_T;
                x[u] = 0.f;                            // the offset mode (k = 0) does not enter
                l[u] = make_float2(0.f, 0.f);
                if (k < T.k1 && k > 0) { x[u] = __ldg(T.x + k); l[u] = __ldg(lnk + k); }    // ln k = l.x + l.y
            }
#pragma unroll
            for (int u = 0; u < U; u += 2) {
                // -alpha ln k as a double-float (p + e), then k^-alpha = e^p (1 + e)
                const PF lx{l[u].x, l[u + 1].x}, ly{l[u].y, l[u + 1].y}, xx{x[u], x[u + 1]};
                const PF p = pmul(nh, lx);
                const PF e = padd(pfma(nh, lx, pneg(p)), pfma(nh, ly, pmul(nl, lx)));
                const PF w = pmul(PF{expf(p.a), expf(p.b)}, padd(pdup<PF>(1.0f), e));
                // the exact product x^2 w added as a double-word
                const PF x2 = pmul(xx, xx);
                const PF v = pmul(x2, w), ve = pfma(x2, w, pneg(v));
                const PF s = padd(as[u / 2], v);
                const PF bb = psub(s, as[u / 2]);
                const PF er = padd(psub(as[u / 2], psub(s, bb)), psub(v, bb));
                as[u / 2] = s;
                ac[u / 2] = padd(ac[u / 2], padd(er, ve));
            }
        }
        Acc2 acc = Acc2{as[0].a, ac[0].a};
        const auto merge = [&](float s, float c) {
            acc_add(acc, s);
            acc.c = __fadd_rn(acc.c, c);
        };
        merge(as[0].b, ac[0].b);
#pragma unroll
        for (int u = 1; u < U / 2; ++u) {
            merge(as[u].a, ac[u].a);
            merge(as[u].b, ac[u].b);
        }
        // fixed-order reduction: warp trees, then the warps in order (FP64)
#pragma unroll
        for (int ofs = 16; ofs; ofs >>= 1)
            merge(__shfl_xor_sync(0xffffffffu, acc.s, ofs), __shfl_xor_sync(0xffffffffu, acc.c, ofs));
        if ((threadIdx.x & 31) == 0) s_w[j][threadIdx.x >> 5] = acc_value(acc);
    }
    __syncthreads();
    if (threadIdx.x < nt) {
        double sum = 0.0;
        for (int w = 0; w < PSD_T / 32; ++w) sum += s_w[threadIdx.x][w];
        part[first + threadIdx.x] = s_tile[threadIdx.x].w * sum;
    }
}

// One CTA per detector: S from the tiles' partials in a fixed order, ln L of
// the proposal, the Metropolis decision (step >= 0) or the first evaluation
// (step < 0), then the proposal of the next step and the outputs.
__global__ void __launch_bounds__(PSD_T) k_psd_step(int step, int nsteps, const double *__restrict__ part,
                                                    const int32_t *__restrict__ tile_q, int ntile, int ndet,
                                                    double *state, const double *__restrict__ psd_in,
                                                    const double *__restrict__ nmodes,
                                                    const double *__restrict__ sumlnf, int nq,
                                                    const double *__restrict__ lnfs, double *wq, tod_rng rng,
                                                    double step_lnfk, double step_al, double *psd_out,
                                                    int32_t *acc_out, double *loglike_out)
{
    // the tiles' sum on the first half of the CTA; on the other warps, one
    // lane each, what the decision and the proposal need besides it
    constexpr int SUM_T = PSD_T / 2;
    __shared__ double s_r[SUM_T];
    __shared__ double s_v[5], s_next[2];     // ln u, z1, z2, e^{a L} / sigma0^2, ln sigma0^2; ln f_knee, next alpha
    const int det = blockIdx.x;
    double *st = state + 8 * det;
    const double s0 = psd_in[3 * det];
    const double L = st[PS_PLNFK], a = st[PS_PAL];
    const int warp = threadIdx.x >> 5;
    if (threadIdx.x < SUM_T) {
        double sum = 0.0;
        for (int i = threadIdx.x; i < ntile; i += SUM_T)
            if (tile_q[i] % ndet == det) sum += part[i];
        s_r[threadIdx.x] = sum;
    } else if ((threadIdx.x & 31) == 0) {
        const uint64_t it = rng.gibbs_iter_dev ? *rng.gibbs_iter_dev : rng.gibbs_iter;
        double z1, z2, ua;
        if (warp == SUM_T / 32 && step >= 0) {
            psd_numbers(rng, it, det, step, z1, z2, ua);
            s_v[0] = log(ua);
        } else if (warp == SUM_T / 32 + 1 && step + 1 < nsteps) {
            psd_numbers(rng, it, det, step + 1, z1, z2, ua);
            s_v[1] = z1;
            s_v[2] = z2;
        } else if (warp == SUM_T / 32 + 2) {
            s_v[3] = exp(a * L) / (s0 * s0);
        } else if (warp == SUM_T / 32 + 3) {
            s_v[4] = log(s0 * s0);
        }
    }
    __syncthreads();
    for (int h = SUM_T / 2; h; h >>= 1) {
        if (threadIdx.x < h) s_r[threadIdx.x] += s_r[threadIdx.x + h];
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        const double N = nmodes[det];
        const double ll = -0.5 * (s_v[3] * s_r[0] + N * s_v[4] + a * (sumlnf[det] - N * L));
        double lnfk = st[PS_LNFK], al = st[PS_AL], logl = st[PS_LOGL], acc = st[PS_ACC];
        if (step < 0) {
            logl = ll;
        } else if (st[PS_PVALID] != 0.0 && s_v[0] < ll - logl) {
            lnfk = L;
            al = a;
            logl = ll;
            acc += 1.0;
        }
        st[PS_LNFK] = lnfk;
        st[PS_AL] = al;
        st[PS_LOGL] = logl;
        st[PS_ACC] = acc;
        s_next[0] = lnfk;
        if (step + 1 < nsteps) {
            const double lp = lnfk + step_lnfk * s_v[1], ap = al + step_al * s_v[2];
            st[PS_PLNFK] = lp;
            st[PS_PAL] = ap;
            st[PS_PVALID] = psd_in_box(lp, ap) ? 1.0 : 0.0;
            s_next[1] = ap;
        }
        psd_out[3 * det] = s0;
        psd_out[3 * det + 2] = al;
        if (acc_out) acc_out[det] = static_cast<int32_t>(acc);
        if (loglike_out) loglike_out[det] = logl;
    }
    __syncthreads();
    if (step + 1 < nsteps) psd_factors(s_next[1], det, ndet, nq, lnfs, wq);
    if (threadIdx.x == PSD_T - 1 && step + 1 >= nsteps) psd_out[3 * det + 1] = exp(s_next[0]);
}

}  // namespace

cudaError_t launch_noise_psd(const Plan &p, const float *spec, const double *psd_in, tod_rng rng, int nsteps,
                             double step_lnfk, double step_al, double *psd_out, int32_t *acc_out,
                             double *loglike_out, cudaStream_t st)
{
    const int per = std::max(1, std::min(PSD_TILES, p.ntile / (PSD_CTAS * std::max(1, p.sm_count))));
    {
        KTIME(TOD_KT_PSD_STEP);
        k_psd_begin<<<p.ndet, PSD_T, 0, st>>>(psd_in, p.psd_state, p.ndet, p.nq, p.lnfs, p.psd_w, psd_out, acc_out);
    }
    cudaError_t e = cudaGetLastError();
    for (int s = -1; s < nsteps && e == cudaSuccess; ++s) {
        if (p.ntile > 0)
            {
                KTIME(TOD_KT_PSD_SUMS);
                k_psd_sums<<<(p.ntile + per - 1) / per, PSD_T, 0, st>>>(spec, p.off, p.tile_q, p.tile_t0, p.ntile, per,
                                                                        p.psd_w, p.lnk, p.psd_state, p.ndet,
                                                                        p.psd_part);
            }
        {
            KTIME(TOD_KT_PSD_STEP);
            k_psd_step<<<p.ndet, PSD_T, 0, st>>>(s, nsteps, p.psd_part, p.tile_q, p.ntile, p.ndet, p.psd_state,
                                                 psd_in, p.psd_nmodes, p.psd_sumlnf, p.nq, p.lnfs, p.psd_w, rng, step_lnfk, step_al,
                                                 psd_out, acc_out, loglike_out);
        }
        e = cudaGetLastError();
    }
    return e;
}

}  // namespace tg

// A6 binning into per-pixel normal equations and A7 per-pixel 3x3 solve
// (paper Sect. 5 table rows "TOD binning" and "Map solution (Ax=b for each
// pixel)"; Sect. 2.4: coadded on the fly, synchronised once).
//
// Binning is a deterministic two-level segmented reduction.  The plan holds,
// for every detscan, its pixel-sorted order (stable in time), the runs of
// equal pixel ("pairs" of detscan and pixel) ranked over the band by (pixel,
// detscan), and tiles of consecutive whole runs of one detscan (at most
// BIN_TILE samples, or one longer run alone).
//   k_bin:    one CTA per tile gathers the tile's data, residual and
//             psi/flag words in sorted order into shared memory (the
//             detscan's samples stay in L2 while its tiles run), then four
//             lanes sum each run.  Products of FP32 values are formed
//             exactly and summed as FP32 double-words (FP64 accuracy at FP32
//             issue rate), the residual d - x taken exactly as a
//             double-word; each run's sums are scaled by the detscan's
//             g^2/sigma0^2, g/sigma0^2 in FP64 and written at the run's rank.
//             A run longer than a tile is summed by the whole CTA with a
//             fixed-order tree.
//   k_reduce: one lane per pixel and value adds the pixel's contiguous runs
//             in FP64, in ascending detscan order.
#include <algorithm>
#include "common.cuh"
#include "fft_reg.cuh"
#include "internal.cuh"

namespace tg {

constexpr int BIN_T = 256;

struct BinArgs {
    const uint16_t *psi;
    const float *d, *x;
    const double *gain;
    const uint32_t *flags;
    const double *psd;
    const int64_t *off;
    const uint32_t *ld_t;         // load order -> time index within the detscan
    const uint16_t *ld_pos;       // load order -> run-major position within the tile
    const int64_t *pair_start;
    const int32_t *pair_len, *pair_slot;
    const int32_t *tile_q, *tile_r0;
    const float2 *trig;
    int ndet;
    double *rec;
    // adjoint of the projection: no mask (flags null), weights 0 and g, and,
    // when y64 is set, the FP64 input y = hi + lo read as d = hi, x = -lo
    bool adjoint;
    const double *y64;
};

// the per-run sums: 1 (as hits), c, s, cc, cs, ss, r, cr, sr with r = d - x
// (taken exactly as a double-word: its head and tail), as the lanes of packed
// double-words: (c, s), (cc, ss), (cs, r), (cr, sr)
constexpr int NSUM = 4;
struct PSum { PF s, c; };
struct RunSums {
    PSum a[NSUM];
    int hits;
};
__device__ __forceinline__ void sums_zero(RunSums &r) {
#pragma unroll
    for (int i = 0; i < NSUM; ++i) r.a[i] = PSum{{0.f, 0.f}, {0.f, 0.f}};
    r.hits = 0;
}
__device__ __forceinline__ void psum_add(PSum &a, PF v) {
    const PF s = padd(a.s, v);
    const PF bb = psub(s, a.s);
    const PF e = padd(psub(a.s, psub(s, bb)), psub(v, bb));
    a.s = s;
    a.c = padd(a.c, e);
}
// add the exact products x y and the small values t
__device__ __forceinline__ void psum_add_prod(PSum &a, PF x, PF y, PF t) {
    const PF p = pmul(x, y);
    const PF e = pfma(x, y, pneg(p));
    psum_add(a, p);
    a.c = padd(a.c, padd(e, t));
}
__device__ __forceinline__ void psum_merge(PSum &a, const PSum &b) {
    psum_add(a, b.s);
    a.c = padd(a.c, b.c);
}
__device__ __forceinline__ void sums_add(RunSums &r, float2 cs, float dv, float xv) {
    ++r.hits;
    const PF v{cs.x, cs.y}, zero{0.f, 0.f};
    // r = d - x exactly: head rh (rounded difference) and tail rl (two-sum)
    const float rh = __fsub_rn(dv, xv);
    const float bb = __fsub_rn(rh, dv);
    const float rl = __fadd_rn(__fsub_rn(dv, __fsub_rn(rh, bb)), __fsub_rn(-xv, bb));
    psum_add(r.a[0], v);
    psum_add_prod(r.a[1], v, v, zero);
    // the tail of r, and its products with c and s (below 2^-24 of the
    // heads'), go to the compensation words
    psum_add_prod(r.a[2], PF{cs.x, rh}, PF{cs.y, 1.0f}, PF{0.f, rl});
    psum_add_prod(r.a[3], v, PF{rh, rh}, pmul(v, PF{rl, rl}));
}
__device__ __forceinline__ PF shfl_xor(PF v, int m) {
    return PF{__shfl_xor_sync(0xffffffffu, v.a, m), __shfl_xor_sync(0xffffffffu, v.b, m)};
}
// the sums of lanes l and l ^ m, the lower lane's first, in both
__device__ __forceinline__ void sums_merge_xor(RunSums &r, int m) {
    const bool up = (threadIdx.x & m) != 0;
#pragma unroll
    for (int k = 0; k < NSUM; ++k) {
        PSum p = r.a[k], o{shfl_xor(p.s, m), shfl_xor(p.c, m)};
        if (up) {
            psum_merge(o, p);
            r.a[k] = o;
        } else {
            psum_merge(p, o);
            r.a[k] = p;
        }
    }
    r.hits += __shfl_xor_sync(0xffffffffu, r.hits, m);
}
// the ten outputs as double-words (hits exact below 2^24, else in two words)
__device__ __forceinline__ void sums_out(const RunSums &r, Acc2 *o) {
    const float h = static_cast<float>(r.hits);
    const float hl = static_cast<float>(r.hits - static_cast<int>(h));
    o[0] = o[9] = Acc2{h, hl};
    o[1] = Acc2{r.a[0].s.a, r.a[0].c.a};
    o[2] = Acc2{r.a[0].s.b, r.a[0].c.b};
    o[3] = Acc2{r.a[1].s.a, r.a[1].c.a};
    o[4] = Acc2{r.a[2].s.a, r.a[2].c.a};
    o[5] = Acc2{r.a[1].s.b, r.a[1].c.b};
    o[6] = Acc2{r.a[2].s.b, r.a[2].c.b};
    o[7] = Acc2{r.a[3].s.a, r.a[3].c.a};
    o[8] = Acc2{r.a[3].s.b, r.a[3].c.b};
}
// float to double, exactly, by integer instructions (the conversion itself
// issues with the FP64 ones): normal numbers and zeros, the rest converted
__device__ __forceinline__ double widen(float x) {
    const uint32_t u = __float_as_uint(x), m = u & 0x7FFFFFFFu;
    if (m - 0x00800000u >= 0x7F000000u && m != 0u) return static_cast<double>(x);
    const uint32_t hi = (u & 0x80000000u) | (m ? (m >> 3) + (896u << 20) : 0u);
    return __hiloint2double(static_cast<int>(hi), static_cast<int>(m << 29));
}

__device__ __forceinline__ uint16_t psi_flag(const BinArgs &a, int64_t tg) {
    const uint32_t fb = a.flags ? (__ldg(a.flags + (tg >> 5)) >> (tg & 31)) & 1u : 0u;
    return static_cast<uint16_t>((__ldg(a.psi + tg) & 0x0FFF) | (fb << 15));
}

// data and residual of sample tg (the adjoint's input: y, or the head and
// negated tail of the FP64 y, whose difference is y to FP64 accuracy)
__device__ __forceinline__ void load_dx(const BinArgs &a, int64_t tg, float &dv, float &xv) {
    if (a.y64) {
        const double y = __ldg(a.y64 + tg);
        const float hi = static_cast<float>(y);
        dv = hi;
        xv = -static_cast<float>(y - static_cast<double>(hi));
    } else {
        dv = __ldg(a.d + tg);
        xv = a.x ? __ldg(a.x + tg) : 0.f;
    }
}

// copies into shared memory past the registers; zeros where !take
__device__ __forceinline__ void cp_async4(float *dst, const float *src, bool take) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;"
                 :: "r"(static_cast<uint32_t>(__cvta_generic_to_shared(dst))), "l"(src), "r"(take ? 4 : 0) : "memory");
}
__device__ __forceinline__ void cp_async8(float2 *dst, const float2 *src, bool take) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;"
                 :: "r"(static_cast<uint32_t>(__cvta_generic_to_shared(dst))), "l"(src), "r"(take ? 8 : 0) : "memory");
}

// Bound by the gather: its loads and the sectors they touch take three
// quarters of the time (324 of 401 us with the sums left out).  A branch per
// sample put the psi -> cos, sin chains of a thread's eight samples one behind
// the other; here each kind of load is issued for all eight first, and data,
// residual and cos, sin go past the registers, which also keeps five CTAs on
// an SM (four: 441 against 409 us; six, by spilling: 449).  FP64 issues at 1/64
// of the FP32 rate, so the weights' divisions run on one thread of the last
// warp beside the sums, and the outputs of 64 runs are scaled by all threads,
// every lane of an FP64 instruction at work; the sums are packed FP32
// double-words.  Four lanes per run: eight are even at 33 runs a tile (409
// against 401 us) and slower at 40 (963 against 876).
// 45M samples of 44 GHz: 596 -> 401 us; 102M of 70 GHz: 1324 -> 876 us.
constexpr int BIN_LANES = 4;                         // lanes per run
constexpr int BIN_CTAS = 5;                          // CTAs per SM
constexpr int BIN_BATCH = 64;                        // runs whose outputs are staged together

__global__ void __launch_bounds__(BIN_T, BIN_CTAS) k_bin(BinArgs a)
{
    __shared__ float s_d[BIN_TILE], s_x[BIN_TILE];
    __shared__ float2 s_cs[BIN_TILE];
    __shared__ Acc2 s_out[BIN_BATCH][10];            // the outputs of a batch's runs
    __shared__ double s_w[2];
    __shared__ RunSums s_red[BIN_T / 32];
    const int tile = blockIdx.x;
    const int q = a.tile_q[tile];
    const int r0 = a.tile_r0[tile], nr = a.tile_r0[tile + 1] - r0;
    const int64_t o = a.off[q];
    const int64_t s0 = a.pair_start[r0];
    const int cnt = static_cast<int>(a.pair_start[r0 + nr - 1] + a.pair_len[r0 + nr - 1] - s0);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const bool whole = cnt > BIN_TILE;               // one run longer than a tile

    if (!whole) {
        // gather in the tile's load order (the k-th sample of each run, k = 0,
        // 1, ..: a warp's 32 samples are close in time, so they share sectors),
        // each value into its run-major slot: the positions first, then every
        // psi, flag, data and residual load of the thread in flight together
        // (data and residual straight into shared memory), then cos 2psi and
        // sin 2psi, both zero for a flagged sample
        constexpr int PER = BIN_TILE / BIN_T;
        int idx[PER], pos[PER];
#pragma unroll
        for (int u = 0; u < PER; ++u) {
            const int i = threadIdx.x + u * BIN_T;
            idx[u] = i < cnt ? static_cast<int>(__ldg(a.ld_t + s0 + i)) : -1;
            pos[u] = i < cnt ? __ldg(a.ld_pos + s0 + i) : 0;
        }
        uint32_t fw[PER];
        uint16_t pf[PER];
#pragma unroll
        for (int u = 0; u < PER; ++u) {
            const int64_t tg = o + idx[u];
            pf[u] = idx[u] >= 0 ? __ldg(a.psi + tg) : 0;
            fw[u] = a.flags && idx[u] >= 0 ? __ldg(a.flags + (tg >> 5)) >> (tg & 31) : 0u;
        }
        if (a.y64) {
#pragma unroll
            for (int u = 0; u < PER; ++u)
                if (idx[u] >= 0) load_dx(a, o + idx[u], s_d[pos[u]], s_x[pos[u]]);
        } else {
#pragma unroll
            for (int u = 0; u < PER; ++u)
                if (idx[u] >= 0) {
                    cp_async4(s_d + pos[u], a.d + o + idx[u], true);
                    cp_async4(s_x + pos[u], a.x ? a.x + o + idx[u] : a.d, a.x != nullptr);
                }
        }
#pragma unroll
        for (int u = 0; u < PER; ++u)
            if (idx[u] >= 0) cp_async8(s_cs + pos[u], a.trig + (pf[u] & 0x0FFF), !(fw[u] & 1u));
        asm volatile("cp.async.wait_all;" ::: "memory");
        __syncthreads();
    }
    // the detscan's weights g^2/sigma0^2 and g/sigma0^2
    if (threadIdx.x == BIN_T - 1) {
        const double gq = a.gain[q];
        if (a.adjoint) {
            s_w[0] = 0.0;
            s_w[1] = gq;
        } else {
            const double sig0 = a.psd[3 * (q % a.ndet)];
            s_w[0] = gq * gq / (sig0 * sig0);
            s_w[1] = gq / (sig0 * sig0);
        }
    }
    for (int rb = 0; rb < nr; rb += BIN_BATCH) {
        const int nb = min(BIN_BATCH, nr - rb);
        if (whole) {
            // strided partial sums, then a fixed-order tree
            RunSums rs;
            sums_zero(rs);
            for (int i = threadIdx.x; i < cnt; i += BIN_T) {
                const int64_t tg = o + __ldg(a.ld_t + s0 + i);     // a single run: run order
                const uint16_t pf = psi_flag(a, tg);
                if (pf >> 15) continue;
                float dv, xv;
                load_dx(a, tg, dv, xv);
                sums_add(rs, __ldg(a.trig + (pf & 0x0FFF)), dv, xv);
            }
#pragma unroll 1
            for (int m = 1; m < 32; m <<= 1) sums_merge_xor(rs, m);
            if (lane == 0) s_red[warp] = rs;
            __syncthreads();
            if (threadIdx.x == 0) {
                for (int w = 1; w < BIN_T / 32; ++w) {
#pragma unroll
                    for (int k = 0; k < NSUM; ++k) psum_merge(rs.a[k], s_red[w].a[k]);
                    rs.hits += s_red[w].hits;
                }
                sums_out(rs, s_out[0]);
            }
        } else {
            // lane j of a run's quad takes its samples j, j + 4, ...; their
            // sums are merged in a fixed order (deterministic)
            const int sub = lane / BIN_LANES, ql = lane % BIN_LANES;
            for (int g = warp * (32 / BIN_LANES); g < nb; g += BIN_T / BIN_LANES) {
                const int r = g + sub;
                RunSums rs;
                sums_zero(rs);
                if (r < nb) {
                    const int st = static_cast<int>(a.pair_start[r0 + rb + r] - s0);
                    const int end = st + a.pair_len[r0 + rb + r];
                    for (int i = st + ql; i < end; i += BIN_LANES) {
                        const float2 cs = s_cs[i];
                        if (cs.x == 0.0f && cs.y == 0.0f) continue;
                        sums_add(rs, cs, s_d[i], s_x[i]);
                    }
                }
                __syncwarp();
#pragma unroll
                for (int m = 1; m < BIN_LANES; m <<= 1) sums_merge_xor(rs, m);
                if (r < nb && ql == 0) sums_out(rs, s_out[r]);
            }
        }
        __syncthreads();
        const double wA = s_w[0], wb = s_w[1];
        for (int e = threadIdx.x; e < nb * 10; e += BIN_T) {
            const int r = e / 10, i = e - 10 * r;
            const Acc2 v = s_out[r][i];
            const double w = i == 9 ? 1.0 : (i <= 5 ? wA : wb);
            a.rec[static_cast<int64_t>(a.pair_slot[r0 + rb + r]) * 10 + i] = w * (widen(v.s) + widen(v.c));
        }
        if (rb + BIN_BATCH < nr) __syncthreads();    // the next batch overwrites s_out
    }
}

// Per pixel, its runs added in ascending detscan order as a double-double
// (Knuth two-sum: hi + lo carries the sum to about 2^-104 of its size), then
// rounded once.  The rounded total is the sum of the runs correctly rounded
// but for sums within ~2^-104 of a rounding tie, whatever the grouping: the
// normal equations of a band split into scan ranges and combined with
// tod_combine_partials equal those of the whole band.
struct DD { double hi, lo; };
__device__ __forceinline__ void dd_add(DD &a, double x) {
    const double s = a.hi + x;
    const double bb = s - a.hi;
    const double e = (a.hi - (s - bb)) + (x - bb);
    a.hi = s;
    a.lo += e;
}
__device__ __forceinline__ void dd_add_dd(DD &a, const DD &b) {
    dd_add(a, b.hi);
    a.lo += b.lo;
}

// A CTA takes RED_T pixels at a time: it lists those with runs, zeroes the
// others, and gives the listed ones NV lanes each, lane v the record's value
// V0 + v (V0 = 0, NV = 10: all of them, three pixels a warp; V0 = 6, NV = 3: the
// adjoint's three, ten pixels a warp).  FP64 adds bound it (this part issues
// a warp's FP64 instruction over 71 cycles, whatever its active lanes; the
// hits are summed by the same instructions, exactly): with a thread per pixel
// a warp ran as long as its longest of 32 pixels, read its records 80 bytes
// apart and added zeros for the empty ones.  45M samples at Nside 512: 597 ->
// 183 us; 102M at Nside 1024, 5 % of the pixels hit: 1068 ->
// 544 us; the adjoint of 52M samples at Nside 256: 1259 -> 215 us.
constexpr int RED_T = 256;
template <int V0, int NV>
__global__ void __launch_bounds__(RED_T)
k_reduce(const double *__restrict__ rec, const int64_t *__restrict__ pix_slot_off, int npix,
         double *__restrict__ A, double *__restrict__ b, int32_t *__restrict__ hits, double *__restrict__ part)
{
    constexpr int PW = 32 / NV;          // pixels per warp and round
    __shared__ int64_t s_off[RED_T + 1];
    __shared__ uint16_t s_list[RED_T];
    __shared__ int s_cnt[RED_T / 32];
    const int lane = threadIdx.x & 31, wi = threadIdx.x >> 5;
    const int pl = lane / NV, v = lane - pl * NV;
    for (int64_t p0 = static_cast<int64_t>(blockIdx.x) * RED_T; p0 < npix; p0 += static_cast<int64_t>(gridDim.x) * RED_T) {
        const int np = static_cast<int>(min(static_cast<int64_t>(RED_T), npix - p0));
        for (int i = threadIdx.x; i <= np; i += RED_T) s_off[i] = pix_slot_off[p0 + i];
        __syncthreads();
        const int i = threadIdx.x;
        const bool has = i < np && s_off[i + 1] > s_off[i];
        const uint32_t full = __ballot_sync(0xffffffffu, has);
        if (lane == 0) s_cnt[wi] = __popc(full);
        __syncthreads();
        int before = 0, nf = 0;
#pragma unroll
        for (int w = 0; w < RED_T / 32; ++w) {
            if (w == wi) before = nf;
            nf += s_cnt[w];
        }
        if (has) s_list[before + __popc(full & ((1u << lane) - 1u))] = static_cast<uint16_t>(i);
        // pixels without runs, 32 of them by each warp
        const int64_t pw = p0 + 32 * wi;
        const int nw = min(32, np - 32 * wi);
        if (part) {
            for (int k = lane; k < nw * 20; k += 32)
                if (!(full >> (k / 20) & 1u)) part[pw * 20 + k] = 0.0;
        } else {
            if (A)
                for (int k = lane; k < nw * 6; k += 32)
                    if (!(full >> (k / 6) & 1u)) A[pw * 6 + k] = 0.0;
            for (int k = lane; k < nw * 3; k += 32)
                if (!(full >> (k / 3) & 1u)) b[pw * 3 + k] = 0.0;
            if (hits && i < np && !has) hits[p0 + i] = 0;
        }
        __syncthreads();
        if (pl < PW) {
            for (int slot = wi * PW + pl; slot < nf; slot += PW * (RED_T / 32)) {
                const int ip = s_list[slot];
                const int64_t p = p0 + ip, k0 = s_off[ip];
                const int c = static_cast<int>(s_off[ip + 1] - k0);
                const double *r = rec + k0 * 10 + V0 + v;
                DD s{0.0, 0.0};
#pragma unroll 2
                for (int k = 0; k < c; ++k, r += 10) dd_add(s, *r);
                if (part) {          // the unrounded pairs (hi, lo) of the ten sums
                    double *o = part + (p * 10 + V0 + v) * 2;
                    o[0] = s.hi;
                    o[1] = s.lo;
                } else if (V0 + v < 6) {
                    if (A) A[p * 6 + V0 + v] = s.hi + s.lo;
                } else if (V0 + v < 9) {
                    b[p * 3 + V0 + v - 6] = s.hi + s.lo;
                } else if (hits) {
                    hits[p] = static_cast<int32_t>(s.hi);
                }
            }
        }
        __syncthreads();
    }
}

// at most a few waves of resident CTAs
static unsigned reduce_grid(const Plan &p)
{
    const int64_t ctas = (static_cast<int64_t>(p.npix) + RED_T - 1) / RED_T;
    return static_cast<unsigned>(std::max<int64_t>(1, std::min<int64_t>(ctas, static_cast<int64_t>(p.sm_count) * 8 * 8)));
}

// Shards' pairs of pixels [0, np) added in rank order as double-doubles,
// rounded once: parts [nparts][np][20] -> A [np][6], b [np][3], hits [np].
__global__ void __launch_bounds__(256)
k_combine(const double *__restrict__ parts, int nparts, int64_t np, double *__restrict__ A, double *__restrict__ b,
          int32_t *__restrict__ hits)
{
    const int64_t p = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
    if (p >= np) return;
    DD s[10];
#pragma unroll
    for (int i = 0; i < 10; ++i) s[i] = DD{0.0, 0.0};
    for (int r = 0; r < nparts; ++r) {
        const double *o = parts + (static_cast<int64_t>(r) * np + p) * 20;
#pragma unroll
        for (int i = 0; i < 10; ++i) dd_add_dd(s[i], DD{o[2 * i], o[2 * i + 1]});
    }
#pragma unroll
    for (int i = 0; i < 6; ++i) A[p * 6 + i] = s[i].hi + s[i].lo;
#pragma unroll
    for (int i = 0; i < 3; ++i) b[p * 3 + i] = s[6 + i].hi + s[6 + i].lo;
    hits[p] = static_cast<int32_t>(s[9].hi + s[9].lo);
}

// ---------------------------------------------------------------------------
// A7: FP64 3x3 Cholesky per pixel, validity by hits and Hadamard ratio.
// ---------------------------------------------------------------------------
// Pixels [0, npix) of A, b, hits (a whole map, or one range of it: the
// outputs are indexed like the inputs).  FP64 bounds the pixels that hold
// data: one reciprocal square root per pivot serves the divisions of its row
// and of the two triangular solves (five divisions and three square roots
// before); a pixel without data (A_TT = 0, as bits) takes none: its determinant
// ratio is zero.  Nside 1024 with 5 % of the pixels hit: 1032 -> 193 us.
__global__ void __launch_bounds__(256)
k_solve(const double *__restrict__ A, const double *__restrict__ b, const int32_t *__restrict__ hits,
        int npix, double rcond_min, double *__restrict__ map, float4 *__restrict__ map32,
        double *__restrict__ rcond, uint8_t *__restrict__ valid)
{
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= npix) return;
    const double *a = A + static_cast<int64_t>(p) * 6;
    const double a00 = a[0];
    double x0 = 0.0, x1 = 0.0, x2 = 0.0, had = 0.0;
    bool ok = false;
    if (__double_as_longlong(a00) != 0) {
        const double a01 = a[1], a02 = a[2], a11 = a[3], a12 = a[4], a22 = a[5];
        const double det = a00 * (a11 * a22 - a12 * a12) - a01 * (a01 * a22 - a12 * a02)
                         + a02 * (a01 * a12 - a11 * a02);
        const double dp = a00 * a11 * a22;
        had = dp > 0.0 ? det / dp : 0.0;
        ok = hits[p] >= 3 && had >= rcond_min && a00 > 0.0 && a11 > 0.0 && a22 > 0.0;
        if (ok) {
            const double i0 = rsqrt(a00);                       // 1 / l00
            const double l10 = a01 * i0, l20 = a02 * i0;
            const double i1 = rsqrt(a11 - l10 * l10);           // 1 / l11
            const double l21 = (a12 - l20 * l10) * i1;
            const double i2 = rsqrt(a22 - l20 * l20 - l21 * l21);
            const double *bb = b + static_cast<int64_t>(p) * 3;
            const double y0 = bb[0] * i0;
            const double y1 = (bb[1] - l10 * y0) * i1;
            const double y2 = (bb[2] - l20 * y0 - l21 * y1) * i2;
            x2 = y2 * i2;
            x1 = (y1 - l21 * x2) * i1;
            x0 = (y0 - l10 * x1 - l20 * x2) * i0;
        }
    }
    map[p] = x0;
    map[npix + p] = x1;
    map[2 * static_cast<int64_t>(npix) + p] = x2;
    if (map32) map32[p] = make_float4(static_cast<float>(x0), static_cast<float>(x1), static_cast<float>(x2), 0.f);
    if (rcond) rcond[p] = had;
    if (valid) valid[p] = ok ? 1 : 0;
}

cudaError_t setup_bin_kernel(Plan &)
{
    return cudaSuccess;
}

cudaError_t launch_bin(const Plan &p, const uint16_t *psi, const float *d, const float *ncorr,
                       const double *gain, const uint32_t *flags, const double *psd, double *A,
                       double *b, int32_t *hits, double *part, cudaStream_t st)
{
    if (p.nq == 0) return cudaSuccess;
    BinArgs a;
    a.psi = psi; a.d = d; a.x = ncorr; a.gain = gain; a.flags = flags; a.psd = psd; a.off = p.off;
    a.ld_t = p.ld_t; a.ld_pos = p.ld_pos; a.pair_start = p.pair_start; a.pair_len = p.pair_len; a.pair_slot = p.pair_slot;
    a.tile_q = p.bin_tile_q; a.tile_r0 = p.bin_tile_r0; a.trig = p.trig; a.ndet = p.ndet; a.rec = p.rec;
    a.adjoint = false; a.y64 = nullptr;
    if (p.nbin_tiles > 0) {
        KTIME(TOD_KT_BIN);
        k_bin<<<p.nbin_tiles, BIN_T, 0, st>>>(a);
    }
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    {
        KTIME(TOD_KT_REDUCE);
        k_reduce<0, 10><<<reduce_grid(p), RED_T, 0, st>>>(p.rec, p.pix_slot_off, p.npix, A, b, hits, part);
    }
    return cudaGetLastError();
}

cudaError_t launch_combine(const double *parts, int nparts, int64_t np, double *A, double *b, int32_t *hits,
                           cudaStream_t st)
{
    if (np <= 0) return cudaSuccess;
    k_combine<<<static_cast<unsigned>((np + 255) / 256), 256, 0, st>>>(parts, nparts, np, A, b, hits);
    return cudaGetLastError();
}

cudaError_t launch_project_adjoint(const Plan &p, const uint16_t *psi, const void *y, bool fp64, const double *gain,
                                   double *out, cudaStream_t st)
{
    if (p.nq == 0) return cudaSuccess;
    BinArgs a;
    a.psi = psi; a.d = fp64 ? nullptr : static_cast<const float *>(y); a.x = nullptr; a.gain = gain;
    a.flags = nullptr; a.psd = nullptr; a.off = p.off;
    a.ld_t = p.ld_t; a.ld_pos = p.ld_pos; a.pair_start = p.pair_start; a.pair_len = p.pair_len; a.pair_slot = p.pair_slot;
    a.tile_q = p.bin_tile_q; a.tile_r0 = p.bin_tile_r0; a.trig = p.trig; a.ndet = p.ndet; a.rec = p.rec;
    a.adjoint = true; a.y64 = fp64 ? static_cast<const double *>(y) : nullptr;
    if (p.nbin_tiles > 0) {
        KTIME(TOD_KT_BIN);
        k_bin<<<p.nbin_tiles, BIN_T, 0, st>>>(a);
    }
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    {
        KTIME(TOD_KT_REDUCE);
        k_reduce<6, 3><<<reduce_grid(p), RED_T, 0, st>>>(p.rec, p.pix_slot_off, p.npix, nullptr, out, nullptr,
                                                           nullptr);
    }
    return cudaGetLastError();
}

cudaError_t launch_solve(const Plan &p, const double *A, const double *b, const int32_t *hits,
                         double rcond_min, double *map, float4 *map32, double *rcond,
                         uint8_t *valid, cudaStream_t st)
{
    KTIME(TOD_KT_SOLVE);
    return launch_solve_n(p.npix, A, b, hits, rcond_min, map, map32, rcond, valid, st);
}

cudaError_t launch_solve_n(int64_t npix, const double *A, const double *b, const int32_t *hits, double rcond_min,
                           double *map, float4 *map32, double *rcond, uint8_t *valid, cudaStream_t st)
{
    if (npix <= 0) return cudaSuccess;
    const int nb = static_cast<int>((npix + 255) / 256);
    k_solve<<<nb, 256, 0, st>>>(A, b, hits, static_cast<int>(npix), rcond_min, map, map32, rcond, valid);
    return cudaGetLastError();
}

}  // namespace tg

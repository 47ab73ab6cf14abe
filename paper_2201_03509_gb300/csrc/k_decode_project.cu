// A1 Huffman decode (paper Sect. 4.1) and A2 projection (Eq. `todmodel`).
//
// Decode: every checkpoint block (TOD_CKPT_BLOCK symbols of one detscan) is
// decoded by one thread, starting from the block's bit offset and the value
// preceding it, so a band's ~10^6 blocks decode in parallel.  One CTA takes
// up to DEC_T consecutive blocks of one scan and stages that scan's code
// (a 2^DEC_LUTB-entry first-level table, per-length limits for the long
// codes) in shared memory; the rare long codes read their symbol through
// the cache.  Values are undone from their differences on the fly, staged
// DEC_ROUND at a time per thread in shared memory, and written by their own
// warp in pairs (no CTA barrier after the table is staged).
//
// A block is one long dependency chain, and what it waits for decides the
// speed.  Threads run out of bits at different symbols, so a load of the next
// word where it is needed stalls the warp at nearly every symbol for a trip
// to L2.  Each thread's words come through a ring of four 16-byte chunks in
// shared memory instead, filled by asynchronous copies two groups of symbols
// ahead (a group of DEC_GROUP symbols takes less than one chunk, 24 bits each
// at most, so one copy per group keeps the ring full); and a symbol takes no
// branch but those to a refill and to the long codes, whose symbols are staged
// in shared memory too when a scan has at most DEC_CANON of them (30 % of the
// 70 GHz pixel symbols are longer than the table).  27M samples of pointing:
// 474 -> 268 us; of TOD 305 -> 151, of flags 149 -> 73 us; 65k samples 111 -> 63 us
// a stream; 102M samples of 70 GHz pointing 1972 -> 784 us.  A symbol's chain of
// dependent operations is the bound.  (Asking L2 for a block's lines at its
// start cost 15 %, a ring of eight chunks gained nothing.)
//
// The same decoder serves the TOD and quality-flag streams (Sect. 4.1:
// the ADC integers and flag words are differenced and coded like the
// pointing; Listing `tod`: tod and flag held as compressed bytes).  What a
// decoded value becomes is the kernel's KIND: the value itself (pointing),
// the FP32 TOD d = fl32(scale_q * count) (the FP64 product, rounded once),
// or the flag bit (word & select) != 0, collected per DEC_ROUND samples and
// ORed into the sample bitmask with at most two atomics.
#include <type_traits>

#include "common.cuh"
#include "internal.cuh"

namespace tg {

constexpr int DEC_GROUP = 4;                  // symbols between two refills of the ring
constexpr int DEC_CANON = 8192;               // most symbols of a code staged in shared memory
constexpr int DEC_RING = 16;                  // words of a thread's ring (four chunks)
constexpr int DEC_RSTRIDE = DEC_RING + 4;     // its stride, 16-byte aligned
static_assert(DEC_ROUND % DEC_GROUP == 0 && DEC_GROUP * TOD_HUFF_MAXLEN < 128, "a group takes less than a chunk");
static_assert(DEC_ROUND == 16 && TOD_CKPT_BLOCK % DEC_ROUND == 0, "flags are packed 16 at a time");
static_assert((1 << DEC_LUTB) % (4 * DEC_T) == 0, "the table is staged 16 bytes a thread");

// fl32 of the FP64 product c * scale (scale = s1 + s2 + ..., FP32 parts) in
// FP32: the product as head + tail to about 2^-46, rounded; where that lies
// too near a rounding boundary to be sure (or out of the easy range), the
// FP64 product itself (FP64 issues at 1/64 of the FP32 rate here).  A count of
// zero is zero whatever the scale, which is positive and finite but may lie
// past FP32's range.
__device__ __forceinline__ float tod_value(int32_t c, float s1, float s2, double scale) {
    const float fc = static_cast<float>(c);
    const float ph = __fmul_rn(fc, s1);
    const float l = __fadd_rn(__fmaf_rn(fc, s1, -ph), __fmul_rn(fc, s2));
    const float r = __fadd_rn(ph, l);
    const float e = fabsf(__fsub_rn(l, __fsub_rn(r, ph)));       // distance to the rounded value
    const uint32_t rb = __float_as_uint(r);
    const float half = __uint_as_float(rb & 0x7f800000u) * 5.9604644775390625e-08f;    // half an ulp of r
    const bool sure = c == 0 || (e < 0.9999f * half && (rb & 0x7fffffu) != 0u && abs(c) < (1 << 24) &&
                                 fabsf(r) > 1e-25f && fabsf(r) < 1e25f);
    return !sure ? __double2float_rn(static_cast<double>(c) * scale) : c == 0 ? 0.0f : r;
}

template <typename OutT, int KIND>
__global__ void __launch_bounds__(DEC_T)
k_decode(const uint32_t *__restrict__ words, int64_t nchunks, const int64_t *__restrict__ word_off,
         const int64_t *__restrict__ nbits, const int64_t *__restrict__ blk_off,
         const uint32_t *__restrict__ ckpt_bit, const int32_t *__restrict__ ckpt_val,
         const int32_t *__restrict__ blk_q, const int32_t *__restrict__ lut,
         const unsigned long long *__restrict__ lim_g, const int32_t *__restrict__ base_g,
         const int32_t *__restrict__ canon_off, const int32_t *__restrict__ canon_vals,
         const int32_t *__restrict__ cta_scan, const int64_t *__restrict__ cta_blk0,
         const int32_t *__restrict__ cta_nblk, const int64_t *__restrict__ off,
         const double *__restrict__ scale, uint32_t select, bool staged, OutT *__restrict__ out, bool pairs,
         int32_t *status)
{
    struct alignas(2 * sizeof(OutT)) Pair { OutT a, b; };
    constexpr int TS = DEC_ROUND / 2 + 1;                  // pairs per thread of the tile, odd
    extern __shared__ __align__(16) int32_t s_lut[];       // [1 << DEC_LUTB], then the rings
    uint32_t *s_ring = reinterpret_cast<uint32_t *>(s_lut + (1 << DEC_LUTB));
    __shared__ unsigned long long s_lim[26];
    __shared__ int32_t s_base[26];
    __shared__ Pair s_tile[KIND == DEC_FLAG ? 1 : DEC_T * TS];
    __shared__ int64_t s_out0[DEC_T];
    __shared__ int32_t s_cnt[DEC_T];

    const int tid = threadIdx.x, lane = tid & 31, w32 = tid & ~31;
    const int scan = cta_scan[blockIdx.x];
    const int64_t b0 = cta_blk0[blockIdx.x];
    const int nb = cta_nblk[blockIdx.x];

    {
        const int4 *src = reinterpret_cast<const int4 *>(lut + (static_cast<int64_t>(scan) << DEC_LUTB));
        int4 *dst = reinterpret_cast<int4 *>(s_lut);
#pragma unroll
        for (int i = 0; i < (1 << DEC_LUTB) / (4 * DEC_T); ++i) dst[tid + i * DEC_T] = src[tid + i * DEC_T];
    }
    if (tid < 26) { s_lim[tid] = lim_g[scan * 26 + tid]; s_base[tid] = base_g[scan * 26 + tid]; }
    // symbols of long codes (longer than DEC_LUTB bits)
    const int c0 = canon_off[scan], nc = canon_off[scan + 1] - c0;
    int32_t *s_canon = reinterpret_cast<int32_t *>(s_ring + DEC_T * DEC_RSTRIDE);
    if (staged)
        for (int i = tid; i < nc; i += DEC_T) s_canon[i] = __ldg(canon_vals + c0 + i);
    const int32_t *canon = staged ? s_canon : canon_vals + c0;

    // this thread's block
    int q = 0, cnt = 0;
    int64_t end = 0, out0 = 0;
    int32_t x = 0;
    double sc = 0.0;                    // DEC_TOD: the detscan's ADC quantum
    float s1 = 0.f, s2 = 0.f;
    uint32_t hi = 0, lo = 0;            // the next bits, left-aligned
    int have = 64;                      // valid bits in hi:lo
    int64_t chunk0 = 0;                 // first chunk of the ring's numbering
    int wi = 0, fetched = 0;            // next word, next chunk to copy, relative to chunk0
    bool ok = true;
    uint32_t *ring = s_ring + tid * DEC_RSTRIDE;
    const auto fetch = [&]() {          // the next chunk, once its place is free
        if (fetched < (wi >> 2) + DEC_RING / 4 && chunk0 + fetched < nchunks) {
            const uint32_t d = static_cast<uint32_t>(__cvta_generic_to_shared(ring + 4 * (fetched & (DEC_RING / 4 - 1))));
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(d), "l"(words + 4 * (chunk0 + fetched)) : "memory");
            ++fetched;
        }
        asm volatile("cp.async.commit_group;\n" ::: "memory");
    };
    if (tid < nb) {
        const int64_t b = b0 + tid;
        q = blk_q[b];
        const int64_t j = b - blk_off[q];
        const int64_t n = off[q + 1] - off[q];
        cnt = static_cast<int>((n - j * TOD_CKPT_BLOCK < TOD_CKPT_BLOCK ? n - j * TOD_CKPT_BLOCK : TOD_CKPT_BLOCK));
        out0 = off[q] + j * TOD_CKPT_BLOCK;
        const int64_t w0 = word_off[q] * 32;
        const int64_t pos = w0 + ckpt_bit[b];
        end = w0 + nbits[q];
        x = ckpt_val[b];
        if constexpr (KIND == DEC_TOD) {
            sc = scale[q];
            s1 = static_cast<float>(sc);
            s2 = static_cast<float>(sc - static_cast<double>(s1));
        }
        chunk0 = pos >> 7;
        wi = static_cast<int>((pos >> 5) & 3);
#pragma unroll
        for (int i = 0; i < DEC_RING / 4; ++i) fetch();
        asm volatile("cp.async.wait_all;\n" ::: "memory");
        const int sh = static_cast<int>(pos & 31);
        const uint32_t a = ring[wi], c = ring[wi + 1];
        hi = __funnelshift_l(c, a, sh);
        lo = c << sh;
        have = 64 - sh;
        wi += 2;
    }
    s_cnt[tid] = cnt;
    s_out0[tid] = out0;
    uint32_t nw = ring[wi & (DEC_RING - 1)];               // the word after hi:lo
    __syncthreads();
    // the limits of the first lengths past the table
    constexpr int NL = 4;
    unsigned long long lim[NL];
#pragma unroll
    for (int l = 0; l < NL; ++l) lim[l] = s_lim[DEC_LUTB + 1 + l];

    for (int round = 0; round < TOD_CKPT_BLOCK / DEC_ROUND; ++round) {
        uint32_t bits = 0;
#pragma unroll
        for (int g = 0; g < DEC_ROUND / DEC_GROUP; ++g) {
            if (cnt > 0) fetch();
            else asm volatile("cp.async.commit_group;\n" ::: "memory");
            // every chunk but the last two copies' has arrived: the current
            // chunk and the next, more than a group can take
            asm volatile("cp.async.wait_group 2;\n" ::: "memory");
            OutT val[DEC_GROUP];
#pragma unroll
            for (int i = 0; i < DEC_GROUP; ++i) {
                const int idx = round * DEC_ROUND + g * DEC_GROUP + i;
                const int32_t e = s_lut[hi >> (32 - DEC_LUTB)];
                int len = e & 31;
                int32_t v = e >> 5;
                if (len == 0 || v == DEC_WIDE) {
                    // a code longer than the table (its length found from the
                    // canonical limits above DEC_LUTB), or a value too wide for
                    // the packed entry (length known)
                    int L = len;
                    if (len == 0) {
                        L = DEC_LUTB + 1;
#pragma unroll
                        for (int l = 0; l < NL; ++l) L += hi >= lim[l];
                        if (L == DEC_LUTB + 1 + NL)
                            while (L <= TOD_HUFF_MAXLEN && static_cast<unsigned long long>(hi) >= s_lim[L]) ++L;
                    }
                    const int ci = L > TOD_HUFF_MAXLEN ? -1 : s_base[L] + static_cast<int>(hi >> (32 - L));
                    if (ci < 0 || ci >= nc) {
                        if (idx < cnt) ok = false;
                        v = 0;
                        len = L > TOD_HUFF_MAXLEN ? 1 : L;
                    } else {
                        v = canon[ci];
                        len = L;
                    }
                }
                if (idx >= cnt) { len = 0; v = 0; }         // past a short block: nothing more is taken
                x += v;
                hi = __funnelshift_l(lo, hi, len);
                lo <<= len;
                have -= len;
                // 8 <= have: codes have at most 24 bits
                const bool need = have < 32;
                hi |= need ? nw >> (have & 31) : 0u;
                lo = need ? nw << (32 - have & 31) : lo;
                have += need ? 32 : 0;
                if (need) { ++wi; nw = ring[wi & (DEC_RING - 1)]; }
                if constexpr (KIND == DEC_TOD) val[i] = tod_value(x, s1, s2, sc);
                else if constexpr (KIND == DEC_FLAG) {
                    if (idx < cnt && (static_cast<uint32_t>(x) & select) != 0u) bits |= 1u << (g * DEC_GROUP + i);
                } else val[i] = static_cast<OutT>(x);
            }
            if constexpr (KIND != DEC_FLAG) {
#pragma unroll
                for (int i = 0; i < DEC_GROUP; i += 2)
                    s_tile[tid * TS + (g * DEC_GROUP + i) / 2] = Pair{val[i], val[i + 1]};
            }
        }
        if constexpr (KIND == DEC_FLAG) {
            // DEC_ROUND consecutive samples' flags into the bitmask (bit
            // t & 31 of word t >> 5; the words start zeroed)
            if (bits) {
                const int64_t g0 = out0 + round * DEC_ROUND;
                const unsigned long long v = static_cast<unsigned long long>(bits) << (g0 & 31);
                atomicOr(out + (g0 >> 5), static_cast<uint32_t>(v));
                if (v >> 32) atomicOr(out + (g0 >> 5) + 1, static_cast<uint32_t>(v >> 32));
            }
        } else {
            // the warp's values: eight lanes a block, two values each
            __syncwarp();
#pragma unroll
            for (int k = 0; k < DEC_ROUND / 2; ++k) {
                const int bl = w32 + 4 * k + (lane >> 3), pi = lane & 7;
                const int idx = round * DEC_ROUND + 2 * pi;
                const Pair v = s_tile[bl * TS + pi];
                OutT *o = out + s_out0[bl] + idx;
                const int left = s_cnt[bl] - idx;
                if (pairs && left >= 2) *reinterpret_cast<Pair *>(o) = v;
                else {
                    if (left >= 1) o[0] = v.a;
                    if (left >= 2) o[1] = v.b;
                }
            }
            __syncwarp();
        }
    }
    // the bits taken: the next word's place less what is still in hi:lo
    if (cnt > 0 && (!ok || (chunk0 * 4 + wi) * 32 - have > end)) set_status(status, q, TOD_ERR_CORRUPT_STREAM);
}

// shared memory of a launch: the table, the rings, and the symbols when staged
static size_t dec_smem(int canon) {
    return sizeof(int32_t) * ((1 << DEC_LUTB) + DEC_T * DEC_RSTRIDE + (canon <= DEC_CANON ? (canon + 3 & ~3) : 0));
}

cudaError_t setup_decode_kernel()
{
    const int smem = static_cast<int>(dec_smem(DEC_CANON));
    cudaError_t e = cudaFuncSetAttribute(k_decode<int32_t, DEC_VALUE>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_decode<uint16_t, DEC_VALUE>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_decode<float, DEC_TOD>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_decode<uint32_t, DEC_FLAG>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    return e;
}

namespace {

template <int KIND> constexpr int32_t kind_id() {
    return KIND == DEC_TOD ? TOD_KT_DECODE_TOD : KIND == DEC_FLAG ? TOD_KT_DECODE_FLAGS : TOD_KT_DECODE;
}

template <typename OutT, int KIND>
cudaError_t decode_into(const Plan &p, const HuffDev &h, const double *scale, uint32_t select, OutT *out,
                        cudaStream_t st)
{
    if (h.ncta == 0) return cudaSuccess;
    // pairs of values: every detscan starts at an even sample
    const bool pairs = (reinterpret_cast<uintptr_t>(out) & (2 * sizeof(OutT) - 1)) == 0;
    {
        KTIME(kind_id<KIND>());
        k_decode<OutT, KIND><<<h.ncta, DEC_T, dec_smem(h.max_canon), st>>>(
            h.words, h.nchunks, h.word_off, h.nbits, h.blk_off, h.ckpt_bit, h.ckpt_val, h.blk_q, h.lut, h.lim, h.base,
            h.canon_off, h.canon_vals, h.cta_scan, h.cta_blk0, h.cta_nblk, p.off, scale, select,
            h.max_canon <= DEC_CANON, out, pairs, p.status);
    }
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_decode(const Plan &p, const HuffDev &h, int32_t *pix_out, uint16_t *psi_out,
                          cudaStream_t st)
{
    if (pix_out) return decode_into<int32_t, DEC_VALUE>(p, h, nullptr, 0u, pix_out, st);
    return decode_into<uint16_t, DEC_VALUE>(p, h, nullptr, 0u, psi_out, st);
}

cudaError_t launch_decode_tod(const Plan &p, float *d_out, cudaStream_t st)
{
    return decode_into<float, DEC_TOD>(p, p.htod, p.tod_scale, 0u, d_out, st);
}

cudaError_t launch_decode_flags(const Plan &p, uint32_t *flags_out, cudaStream_t st)
{
    cudaError_t e = cudaMemsetAsync(flags_out, 0, sizeof(uint32_t) * ((p.N + 31) / 32), st);
    if (e != cudaSuccess) return e;
    return decode_into<uint32_t, DEC_FLAG>(p, p.hflag, nullptr, p.flag_select, flags_out, st);
}

// ---------------------------------------------------------------------------
// A2 projection: one 16-byte map gather per sample, psi angle from the FP32
// table (L1-resident), gain per detscan.  Tiles of ELEM_TILE samples never
// cross a detscan.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256)
k_project(const float4 *__restrict__ map, const int32_t *__restrict__ pix,
          const uint16_t *__restrict__ psi, const double *__restrict__ gain,
          const float2 *__restrict__ trig, const int32_t *__restrict__ tile_q,
          const int64_t *__restrict__ tile_t0, const int64_t *__restrict__ off,
          int32_t npix, float *__restrict__ s_out, int32_t *status)
{
    const int q = tile_q[blockIdx.x];
    const int64_t t0 = tile_t0[blockIdx.x];
    const int64_t t1 = (t0 + ELEM_TILE < off[q + 1]) ? t0 + ELEM_TILE : off[q + 1];
    const float g = gain ? static_cast<float>(gain[q]) : 1.0f;
    for (int64_t t = t0 + threadIdx.x; t < t1; t += blockDim.x) {
        const int32_t pp = pix[t];
        const uint32_t b = psi[t];
        if (static_cast<uint32_t>(pp) >= static_cast<uint32_t>(npix) || b >= TOD_N_PSI) {
            set_status(status, q, TOD_ERR_ARG);      // out-of-range pointing: no gather
            s_out[t] = 0.0f;
            continue;
        }
        const float4 m = __ldg(map + pp);
        const float2 cs = __ldg(trig + b);
        s_out[t] = g * fmaf(m.z, cs.y, fmaf(m.y, cs.x, m.x));
    }
}

// The same in FP64: map double[3][npix] (rows T, Q, U), the FP32 table
// values read as FP64, s in FP64.
__global__ void __launch_bounds__(256)
k_project64(const double *__restrict__ map, const int32_t *__restrict__ pix,
            const uint16_t *__restrict__ psi, const double *__restrict__ gain,
            const float2 *__restrict__ trig, const int32_t *__restrict__ tile_q,
            const int64_t *__restrict__ tile_t0, const int64_t *__restrict__ off,
            int32_t npix, double *__restrict__ s_out, int32_t *status)
{
    const int q = tile_q[blockIdx.x];
    const int64_t t0 = tile_t0[blockIdx.x];
    const int64_t t1 = (t0 + ELEM_TILE < off[q + 1]) ? t0 + ELEM_TILE : off[q + 1];
    const double g = gain ? gain[q] : 1.0;
    for (int64_t t = t0 + threadIdx.x; t < t1; t += blockDim.x) {
        const int32_t pp = pix[t];
        const uint32_t b = psi[t];
        if (static_cast<uint32_t>(pp) >= static_cast<uint32_t>(npix) || b >= TOD_N_PSI) {
            set_status(status, q, TOD_ERR_ARG);
            s_out[t] = 0.0;
            continue;
        }
        const float2 cs = __ldg(trig + b);
        const double T = __ldg(map + pp), Q = __ldg(map + npix + pp), U = __ldg(map + 2 * static_cast<int64_t>(npix) + pp);
        s_out[t] = g * (T + Q * static_cast<double>(cs.x) + U * static_cast<double>(cs.y));
    }
}

cudaError_t launch_project64(const Plan &p, const double *map, const int32_t *pix, const uint16_t *psi,
                             const double *gain, double *s_out, cudaStream_t st)
{
    if (p.ntile == 0) return cudaSuccess;
    {
        KTIME(TOD_KT_PROJECT64);
        k_project64<<<p.ntile, 256, 0, st>>>(map, pix, psi, gain, p.trig, p.tile_q, p.tile_t0, p.off, p.npix,
                                             s_out, p.status);
    }
    return cudaGetLastError();
}

// One sample of the projection (out-of-range pointing: status, zero).
__device__ __forceinline__ float project_one(const float4 *__restrict__ map, const float2 *__restrict__ trig,
                                             int32_t pp, uint32_t b, int32_t npix, float g, int32_t *status, int q)
{
    if (static_cast<uint32_t>(pp) >= static_cast<uint32_t>(npix) || b >= TOD_N_PSI) {
        set_status(status, q, TOD_ERR_ARG);
        return 0.0f;
    }
    const float4 m = __ldg(map + pp);
    const float2 cs = __ldg(trig + b);
    return g * fmaf(m.z, cs.y, fmaf(m.y, cs.x, m.x));
}

// The same, four samples per thread: 16-byte pixel loads, 8-byte angle
// loads and 16-byte stores on the tile's aligned body (global sample index a
// multiple of 4; the caller checks the base pointers), its up to three head
// and tail samples one per thread.  Bound by the gathers' latency: the four
// of a thread go out together, out-of-range pointing taking the last entries
// and a zero afterwards (with a branch per sample each gather waited for the
// one before: 102M samples at Nside 1024, whose map is larger than L2, 474 ->
// 447 us; 27M at Nside 512 118.5 -> 117.3 us).  A map that stays in L1 leaves
// the instructions and the warps in flight as the bound: the index clamped by a
// minimum, the test of the range after the loads, and registers for eight CTAs
// per SM (18M samples at Nside 16: 59.1 us with a branch per sample, 60.1 with
// the index selected by the test at 38 registers, 58.7 so).
__global__ void __launch_bounds__(256, 8)
k_project4(const float4 *__restrict__ map, const int32_t *__restrict__ pix,
           const uint16_t *__restrict__ psi, const double *__restrict__ gain,
           const float2 *__restrict__ trig, const int32_t *__restrict__ tile_q,
           const int64_t *__restrict__ tile_t0, const int64_t *__restrict__ off,
           int32_t npix, float *__restrict__ s_out, int32_t *status)
{
    const int q = tile_q[blockIdx.x];
    const int64_t t0 = tile_t0[blockIdx.x];
    const int64_t t1 = (t0 + ELEM_TILE < off[q + 1]) ? t0 + ELEM_TILE : off[q + 1];
    const float g = gain ? static_cast<float>(gain[q]) : 1.0f;
    const int64_t a0 = min(t1, (t0 + 3) & ~static_cast<int64_t>(3));
    const int64_t a1 = max(a0, t1 & ~static_cast<int64_t>(3));
    if (threadIdx.x < a0 - t0) {
        const int64_t t = t0 + threadIdx.x;
        s_out[t] = project_one(map, trig, pix[t], psi[t], npix, g, status, q);
    }
    if (threadIdx.x < t1 - a1) {
        const int64_t t = a1 + threadIdx.x;
        s_out[t] = project_one(map, trig, pix[t], psi[t], npix, g, status, q);
    }
    for (int64_t t = a0 + 4 * static_cast<int64_t>(threadIdx.x); t < a1; t += 4 * blockDim.x) {
        const int4 p4 = *reinterpret_cast<const int4 *>(pix + t);
        const uint2 b4 = *reinterpret_cast<const uint2 *>(psi + t);
        const int32_t pp[4] = {p4.x, p4.y, p4.z, p4.w};
        const uint32_t bb[4] = {b4.x & 0xFFFFu, b4.x >> 16, b4.y & 0xFFFFu, b4.y >> 16};
        float4 m[4];
        float2 cs[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            m[u] = __ldg(map + min(static_cast<uint32_t>(pp[u]), static_cast<uint32_t>(npix) - 1u));
            cs[u] = __ldg(trig + min(bb[u], static_cast<uint32_t>(TOD_N_PSI) - 1u));
        }
        float v[4];
        bool in = true;
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            v[u] = g * fmaf(m[u].z, cs[u].y, fmaf(m[u].y, cs[u].x, m[u].x));
            in = in && static_cast<uint32_t>(pp[u]) < static_cast<uint32_t>(npix) && bb[u] < TOD_N_PSI;
        }
        if (!in) {
            set_status(status, q, TOD_ERR_ARG);
#pragma unroll
            for (int u = 0; u < 4; ++u)
                if (!(static_cast<uint32_t>(pp[u]) < static_cast<uint32_t>(npix) && bb[u] < TOD_N_PSI)) v[u] = 0.0f;
        }
        const float4 o = make_float4(v[0], v[1], v[2], v[3]);
        *reinterpret_cast<float4 *>(s_out + t) = o;
    }
}

cudaError_t launch_project(const Plan &p, const float4 *map, const int32_t *pix, const uint16_t *psi,
                           const double *gain, float *s_out, cudaStream_t st)
{
    if (p.ntile == 0) return cudaSuccess;
    const bool vec = (reinterpret_cast<uintptr_t>(pix) & 15u) == 0 && (reinterpret_cast<uintptr_t>(psi) & 7u) == 0 &&
                     (reinterpret_cast<uintptr_t>(s_out) & 15u) == 0;
    {
        KTIME(TOD_KT_PROJECT);
        if (vec)
            k_project4<<<p.ntile, 256, 0, st>>>(map, pix, psi, gain, p.trig, p.tile_q, p.tile_t0, p.off, p.npix,
                                                s_out, p.status);
        else
            k_project<<<p.ntile, 256, 0, st>>>(map, pix, psi, gain, p.trig, p.tile_q, p.tile_t0, p.off, p.npix,
                                               s_out, p.status);
    }
    return cudaGetLastError();
}

}  // namespace tg

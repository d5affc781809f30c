// Front end of the receiver: 12-bit unpack, Kramers-Kronig field reconstruction
// by overlap-save FFT Hilbert transform with carrier / gain reduction, and the
// matched filters (KK with downshift and 4 -> 2 decimation; PAM with DC removal).
//
// Paper: Sec. 2 -- 12-bit samples in 2^22-sample buffers; the KK front end takes
// the square root and logarithm inside the overlap-save step, recovers the phase
// with an FD Hilbert transform (FFT, IFFT), mixes it with the square-root term and
// downshifts (Fig. 1d: one thread per sample, amplitude and phase in, complex out);
// the signal is then filtered and reduced to 2 samples/symbol.
//
// Hilbert FFT layout.  One complex FFT of length N = 16 * N2 transforms two real
// overlap-save blocks at once (z = u_a + j u_b; the Hilbert multiplier -j sgn(k)
// is complex-linear, so phi_a + j phi_b = IFFT(h * FFT(z))).  N is split four-step
// style into a radix-16 pass over the stride-N2 index (K1a, registers only), an
// N2-point FFT per row with the multiplier and the inverse in shared memory (K1b),
// and the inverse radix-16 pass fused with sqrt/exp/field assembly (K1c).
#include <string.h>

#include <numeric>

#include <cooperative_groups.h>

#include "rx_async.cuh"
#include "rx_common.cuh"
#include "rx_internal.cuh"

namespace rxk {

// ================================================================== unpack
// Two 12-bit samples per three bytes.  Eight samples (12 bytes, three aligned
// 32-bit words) per thread; the output is [history | this buffer] as uint16 codes.
__device__ __forceinline__ void decode_pair(uint32_t b0, uint32_t b1, uint32_t b2, int order,
                                            uint32_t &s0, uint32_t &s1)
{
    if (order == 0) {
        s0 = b0 | ((b1 & 0xFu) << 8);
        s1 = (b1 >> 4) | (b2 << 4);
    } else {
        s0 = (b0 << 4) | (b1 >> 4);
        s1 = ((b1 & 0xFu) << 8) | b2;
    }
}

// With `sums` (PAM) also the buffer's integer sums; the CTA that takes the last ticket turns
// them into the call's mean and 1 / deviation (slot) and clears them: the division and the
// square root in FP64 (a few thousand cycles on this part) run once per call instead of at
// the start of every CTA of the filter.
constexpr int kUnpackThreads = 256, kUnpackPer = 2;   // threads per CTA, groups of 8 samples per thread
__global__ void __launch_bounds__(kUnpackThreads)
    k_unpack(const uint8_t *in, uint16_t *codes, const uint16_t *codes_prev,
             long long nb, int nhist, long long prev_off, int first_call, int order, DevState *sums, int slot,
             LatRecord *lat, int lat_slot)
{
    pdl_wait();
    if (lat && blockIdx.x == 0 && threadIdx.x == 0) lat_start(lat, lat_slot);
    const long long ngroups = nb / 8, g0 = (long long)blockIdx.x * (kUnpackPer * kUnpackThreads) + threadIdx.x;
    const uint32_t *in32 = reinterpret_cast<const uint32_t *>(in);
    uint32_t w[kUnpackPer][3];
#pragma unroll
    for (int k = 0; k < kUnpackPer; k++) {   // every load issues first
        const long long g = g0 + k * kUnpackThreads;
        if (g < ngroups)
#pragma unroll
            for (int i = 0; i < 3; i++) w[k][i] = in32[3 * g + i];
    }
    unsigned lsum = 0;                // 8 samples of 12 bits per group
    unsigned long long wsq = 0;       // lane 0: the warp's squares (256 samples: below 2^32 per group)
#pragma unroll
    for (int k = 0; k < kUnpackPer; k++) {
        const long long g = g0 + k * kUnpackThreads;
        unsigned lsq = 0;
        if (g < ngroups) {
            uint32_t by[12];
#pragma unroll
            for (int i = 0; i < 12; i++) by[i] = (w[k][i >> 2] >> (8 * (i & 3))) & 0xFFu;
            uint32_t s[8];
#pragma unroll
            for (int p = 0; p < 4; p++)
                decode_pair(by[3 * p], by[3 * p + 1], by[3 * p + 2], order, s[2 * p], s[2 * p + 1]);
            *reinterpret_cast<uint4 *>(codes + nhist + 8 * g) =
                make_uint4(s[0] | (s[1] << 16), s[2] | (s[3] << 16), s[4] | (s[5] << 16), s[6] | (s[7] << 16));
#pragma unroll
            for (int i = 0; i < 8; i++) { lsum += s[i]; lsq += s[i] * s[i]; }
        } else if (g < ngroups + nhist) {
            const long long j = g - ngroups;   // history sample j
            uint16_t v;
            if (first_call) {            // before the stream: first sample replicated
                uint32_t a, b;
                decode_pair(in[0], in[1], in[2], order, a, b);
                v = (uint16_t)a;
            } else {
                v = codes_prev[prev_off + j];
            }
            codes[j] = v;
        }
        if (sums) wsq += __reduce_add_sync(0xffffffffu, lsq);
    }
    if (!sums) return;
    // one atomic per CTA and sum (integer: exact and order free)
    __shared__ unsigned long long r[2][kUnpackThreads / 32];
    const unsigned wsum = __reduce_add_sync(0xffffffffu, lsum);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (lane == 0) { r[0][wid] = wsum; r[1][wid] = wsq; }
    __syncthreads();
    if (wid != 0) return;
    unsigned long long *S[2] = {reinterpret_cast<unsigned long long *>(&sums->pam_s1),
                                reinterpret_cast<unsigned long long *>(&sums->pam_s2)};
    unsigned last = 0;
    if (lane == 0) {
#pragma unroll
        for (int q = 0; q < 2; q++) {
            unsigned long long a = 0;
#pragma unroll
            for (int i = 0; i < kUnpackThreads / 32; i++) a += r[q][i];
            if (a) atomicAdd(S[q], a);
        }
        last = take_ticket(&sums->pam_ticket) == gridDim.x - 1;
    }
    if (!__shfl_sync(0xffffffffu, last, 0)) return;
    __syncwarp();   // what lane 0's ticket acquired, for the other lanes
    // lane 0 divides the sum, lane 1 the sum of squares
    double q = 0.0;
    if (lane < 2) q = (double)(long long)atomicExch(lane ? S[1] : S[0], 0ull) / (double)nb;
    const double mu = __shfl_sync(0xffffffffu, q, 0), m2 = __shfl_sync(0xffffffffu, q, 1);
    if (lane == 0) {
        const double var = m2 - mu * mu;
        const double inv = (var > 0.0) ? 1.0 / sqrt(var) : 1.0;
        sums->pam_nd[slot][0] = mu;
        sums->pam_nd[slot][1] = inv;
        sums->pam_nf[slot][0] = (float)mu;
        sums->pam_nf[slot][1] = (float)inv;
        sums->pam_ticket = 0u;
    }
}

cudaError_t launch_unpack(const uint8_t *in, uint16_t *codes, const uint16_t *codes_prev,
                          long long nb, int nhist, long long prev_off, int first_call,
                          int pack_order, DevState *sums, int slot, cudaStream_t st, LatRecord *lat,
                          int lat_slot, bool pdl)
{
    long long items = nb / 8 + nhist;
    const int per = kUnpackPer * kUnpackThreads;
    unsigned grid = (unsigned)((items + per - 1) / per);
    return launch_k(k_unpack, grid, kUnpackThreads, 0, st, pdl, in, codes, codes_prev, nb, nhist, prev_off, first_call,
                    pack_order, sums, slot, lat, lat_slot);
}

// ============================================================= KK Hilbert
// window start of overlap-save block j (the last block ends at the newest sample)
__device__ __forceinline__ long long ols_ws(const KkGeom &g, int j)
{
    return (j < g.J - 1) ? g.e_prev - g.V / 2 + (long long)j * g.hop : g.avail - g.N;
}
// kept positions [t_lo, t_hi) of block j inside its window
__device__ __forceinline__ void ols_kept(const KkGeom &g, int j, int &t_lo, int &t_hi)
{
    if (j < g.J - 1) {
        t_lo = g.V / 2;
        t_hi = g.V / 2 + g.hop;
    } else {
        int cnt = (int)(g.e_k - (g.e_prev + (long long)(g.J - 1) * g.hop));
        t_hi = g.N - g.V / 2;
        t_lo = t_hi - cnt;
    }
}

// u = ln(I)/2 - ln(2048)/2 (the constant is annihilated by the Hilbert transform
// and only keeps the FP32 FFT well scaled) and sqrt(I), I = code (0.5 for code 0):
// the codes are 12-bit, so both are exact lookup tables computed in double.
static int tw_split(int M)
{
    int m = 0;
    while ((1 << m) < M) m++;
    return (m + 1) / 2;
}
int kk_tw_entries(int M) { return (1 << tw_split(M)) + M / (1 << tw_split(M)); }

static void factored_twiddles(int M, float2 *out)
{
    const double pi = 3.14159265358979323846;
    int s = tw_split(M), lo = 1 << s, hi = M / lo;
    for (int a = 0; a < lo; a++) {
        double t = -2.0 * pi * (double)a / (double)M;
        out[a] = make_float2((float)cos(t), (float)sin(t));
    }
    for (int a = 0; a < hi; a++) {
        double t = -2.0 * pi * (double)a * (double)lo / (double)M;
        out[lo + a] = make_float2((float)cos(t), (float)sin(t));
    }
}

void kk_host_tables(int N, float *lnt, float2 *twN, float2 *twN2)
{
    for (int c = 0; c < kLutCodes; c++) {
        double I = c ? (double)c : 0.5;
        lnt[c] = (float)(0.5 * log(I / 2048.0));
    }
    factored_twiddles(N, twN);
    factored_twiddles(N / 16, twN2);
}

// factored twiddle table staged in shared memory
struct TwSmem {
    const float2 *lo, *hi;
    int s, mask;
    __device__ __forceinline__ float2 operator()(int a) const { return cmul(hi[a >> s], lo[a & mask]); }
};
// x[r] times W^(a r), r = 1..15 (conjugated twiddles when CONJ), W the table's root.
// Four twiddles come from the table (exponents a, 4a, 8a, 12a); the others are the
// powers w^2 = w w, w^3 = w^2 w of the first and the products W^(4qa) w^b, a few
// roundings more than a table value each.  The caller keeps 15 a below the table's
// length.
template <bool CONJ>
__device__ __forceinline__ void twiddle16(float2 (&x)[16], const TwSmem &tw, int a)
{
    const float2 w1 = tw(a), w2 = cmul(w1, w1), w3 = cmul(w2, w1);
    const float2 wb[4] = {make_float2(1.f, 0.f), w1, w2, w3};
#pragma unroll
    for (int q = 0; q < 4; q++) {
        const float2 wq = q ? tw(4 * q * a) : make_float2(1.f, 0.f);
#pragma unroll
        for (int b = (q ? 0 : 1); b < 4; b++) {
            const float2 w = q ? (b ? cmul(wq, wb[b]) : wq) : wb[b];
            x[4 * q + b] = CONJ ? cmulc(x[4 * q + b], w) : cmul(x[4 * q + b], w);
        }
    }
}
// Stages the factored table asynchronously: the caller waits (cp_async_wait_all) before the
// barrier in front of its first use, so the copies are in flight beside the input's loads
// (also asynchronous, stage_rows) instead of a round trip before them.  2^22 samples: K1a
// 10.7 us against 13.0, K1c 16.4 against 17.6 (ncu); a batch 60.8 us per buffer against 63.1.
__device__ __forceinline__ TwSmem stage_tw(const float2 *__restrict__ gtab, int M, float2 *sm)
{
    int m = 31 - __clz(M);
    int s = (m + 1) / 2, lo = 1 << s, n = lo + (M >> s);
    for (int i = threadIdx.x; i < n; i += blockDim.x) cp_async8(sm + i, gtab + i, true);
    cp_async_commit();
    TwSmem t;
    t.lo = sm;
    t.hi = sm + lo;
    t.s = s;
    t.mask = lo - 1;
    return t;
}

// Packed 12-bit input of the KK front end, read directly (the unpack is fused):
// stream sample n lives at byte 1.5 (n - cbase) of the virtual buffer
// [history (the nhist samples before this buffer) | this buffer].  A CTA covers
// 256 columns of a block pair; its 32 rows (2 blocks x 16 radix-16 rows) are 256
// consecutive samples each, whose 384 bytes start on a 48-byte boundary and are
// staged into shared memory with 16-byte loads.
struct KkPacked {
    const uint8_t *hist;   // packed history (nhist samples)
    const uint8_t *in;     // this buffer
    uint8_t *hist_next;    // history of the next call, or null
    long long hist_bytes;  // nhist * 3 / 2
    long long in_bytes;    // buf_len * 3 / 2
    int order, first_call;
    LatRecord *lat;        // latency record whose slot the call's first kernel stamps, or null
    int lat_slot;
};
constexpr int kRawWords = 100;   // 384 bytes of a row + spare word, 16-byte multiple

// 16 bytes of the packed stream of one code repeated, from byte vb (the pairs start at the
// multiples of three)
__device__ __forceinline__ uint4 code_bytes(uint32_t c, int order, unsigned vb)
{
    // the pair's three bytes, least significant first
    const uint32_t pat = order == 0 ? c | (c << 12) : (c >> 4) | ((((c & 0xFu) << 4) | (c >> 8)) << 8) | ((c & 0xFFu) << 16);
    const unsigned long long rep = (unsigned long long)pat * 0x1000001ull;   // six bytes
    const unsigned s = vb % 3;
    const uint32_t w0 = (uint32_t)(rep >> (8 * s)), w1 = (uint32_t)(rep >> (8 * ((s + 1) % 3))),
                   w2 = (uint32_t)(rep >> (8 * ((s + 2) % 3)));
    return make_uint4(w0, w1, w2, w0);
}

// Whether a block of the pair starts before the stream, whose samples read as the stream's
// first code (uniform in a CTA).
__device__ __forceinline__ bool before_stream(const KkGeom &g, int pair, bool hb)
{
    return ols_ws(g, 2 * pair) < 0 || (hb && ols_ws(g, 2 * pair + 1) < 0);
}

// The rows of a CTA's columns (kCtaK1 threads) by asynchronous copies, which the caller waits
// for.  Samples before the stream are staged as c_first.  Byte offsets fit 32 bits: a buffer
// is at most 2^30 samples.
template <int N2T>
__device__ __forceinline__ void stage_rows(const KkGeom &g, const KkPacked &pk, int pair, int c0,
                                           uint32_t (*raw)[kRawWords], bool hb, uint32_t c_first)
{
    static_assert((32 * 24) % kCtaK1 == 0, "whole iterations");
    // virtual-buffer byte of the first sample of this CTA's row 0, per block (>= 0 for every
    // window of the call), and of stream sample 0 (a multiple of 16: buffers and histories
    // are multiples of 32 samples)
    const unsigned v0 = (unsigned)((ols_ws(g, 2 * pair) + c0 - g.cbase) * 3 / 2);
    const unsigned v1 = hb ? (unsigned)((ols_ws(g, 2 * pair + 1) + c0 - g.cbase) * 3 / 2) : 0u;
    const unsigned vs = g.cbase < 0 ? (unsigned)(-g.cbase * 3 / 2) : 0u;
    const unsigned hbytes = (unsigned)pk.hist_bytes;
    const uint8_t *in0 = pk.in - hbytes;
#pragma unroll
    for (int k = 0; k < 32 * 24 / kCtaK1; k++) {
        const int i = threadIdx.x + k * kCtaK1;
        const int row = i / 24, ch = i - 24 * row;
        if (row >= 16 && !hb) continue;
        const unsigned vb = (row < 16 ? v0 : v1) + (unsigned)(row & 15) * (N2T * 3 / 2) + 16 * ch;
        uint32_t *dst = &raw[row][4 * ch];
        if (vb < vs) *reinterpret_cast<uint4 *>(dst) = code_bytes(c_first, pk.order, vb);
        else cp_async16(dst, (vb < hbytes ? pk.hist : in0) + vb);
    }
    cp_async_commit();
}

// 12-bit code of column t of a staged row.  The row is a stream of 12-bit fields,
// two per three bytes.  In pack order 0 sample t fills bits [12 t, 12 t + 12) of the
// little-endian stream: one funnel shift of the two words that hold them and a mask.
// In pack order 1 the code's high nibble comes first: the two bytes that hold it are
// swapped, then a shift takes the high 12 bits (even t) or the low 12 bits (odd t).
// The word index and the shifts depend on t only, so a thread computes them once.
struct ColPos {
    int w;         // first of the two words
    unsigned fs;   // funnel shift
    unsigned ps;   // pack order 1: shift after the byte swap
};
template <int ORD>
__device__ __forceinline__ ColPos col_pos(int t)
{
    const int b = (3 * t) >> 1;   // first byte of the sample
    ColPos c;
    c.w = b >> 2;
    c.fs = 8 * (b & 3) + (ORD == 0 ? 4 * (t & 1) : 0);
    c.ps = ORD == 0 ? 0u : 4u * (1 - (t & 1));
    return c;
}
template <int ORD>
__device__ __forceinline__ uint32_t col_code(const uint32_t *rw, const ColPos &c)
{
    uint32_t v = __funnelshift_r(rw[c.w], rw[c.w + 1], c.fs);
    if (ORD == 1) v = __byte_perm(v, 0u, 0x4401) >> c.ps;   // (byte 0 << 8) | byte 1
    return v & 0xFFFu;
}

// (dst may be null on a stream's first call)
__device__ __forceinline__ uint32_t first_code(const KkPacked &pk, const DevState *dst)
{
    if (!pk.first_call) return (uint32_t)dst->first_code;
    uint32_t a, b;
    decode_pair(pk.in[0], pk.in[1], pk.in[2], pk.order, a, b);
    return a;
}

// the ln table into shared memory, asynchronously like stage_tw: a gather over 32 random codes
// costs a few bank conflicts there instead of one L1 wavefront per distinct cache line
__device__ __forceinline__ void stage_ln(const float *__restrict__ lnt, float *s_ln)
{
    for (int i = threadIdx.x; i < kLutCodes / 4; i += blockDim.x) cp_async16(s_ln + 4 * i, lnt + 4 * i);
    cp_async_commit();
}

// u = ln(I)/2 of both blocks of a pair at this column's 16 window positions
template <int ORD>
__device__ __forceinline__ void load_columns(bool hb, const uint32_t (*raw)[kRawWords], const ColPos &cp, const float *s_ln,
                                             float2 (&x)[16])
{
#pragma unroll
    for (int q = 0; q < 16; q++) {
        const float ua = s_ln[col_code<ORD>(raw[q], cp)];
        const float ub = hb ? s_ln[col_code<ORD>(raw[16 + q], cp)] : 0.f;
        x[q] = make_float2(ua, ub);
    }
}

// packed history of the next call, samples [avail - nhist, avail) = virtual bytes
// [in_bytes, in_bytes + hist_bytes), copied by CTAs 0 .. ncta - 1 (this one is cta)
__device__ __forceinline__ void copy_hist(const KkPacked &pk, int cta, int ncta)
{
    const long long nch = pk.hist_bytes / 16;
    const long long step = (long long)ncta * blockDim.x;
    for (long long c = (long long)cta * blockDim.x + threadIdx.x; c < nch; c += 2 * step) {
        uint4 v[2];
#pragma unroll
        for (int k = 0; k < 2; k++) {   // every load issues before the first one is stored
            const long long vb = pk.in_bytes + 16 * (c + k * step);
            const uint8_t *src = vb < pk.hist_bytes ? pk.hist + vb : pk.in + (vb - pk.hist_bytes);
            if (c + k * step < nch) v[k] = *reinterpret_cast<const uint4 *>(src);
        }
#pragma unroll
        for (int k = 0; k < 2; k++)
            if (c + k * step < nch) reinterpret_cast<uint4 *>(pk.hist_next)[c + k * step] = v[k];
    }
}

// K1a: unpack, u = ln(I)/2 by table, radix-16 pass over the stride-N2 index of two
// packed blocks, twiddle.  CTAs with blockIdx.y == npairs copy the next history.
// ORD: the pack order of the 12-bit input; N2T: the row length N / 16 (256 or 4096), so
// that the stride-N2 accesses take compile-time offsets.
template <int ORD, int N2T>
__global__ void __launch_bounds__(kCtaK1) k_kk_fwd(KkGeom g, KkPacked pk, float2 *fftws,
                                                  const KkTables tb, DevState *dst)
{
    __shared__ float2 s_tw[512];
    __shared__ __align__(16) uint32_t raw[32][kRawWords];
    __shared__ __align__(16) float s_ln[kLutCodes];
    int pair = blockIdx.y;
    const TwSmem tw = stage_tw(tb.twN, g.N, s_tw);
    stage_ln(tb.lnt, s_ln);
    pdl_wait();
    if (pk.lat && blockIdx.x == 0 && pair == 0 && threadIdx.x == 0) lat_start(pk.lat, pk.lat_slot);
    if (pair == g.npairs) {
        copy_hist(pk, blockIdx.x, gridDim.x);
        cp_async_wait_all();
        return;
    }
    const int c0 = blockIdx.x * blockDim.x;
    const bool hb = 2 * pair + 1 < g.J;
    const uint32_t c_first = before_stream(g, pair, hb) || pk.first_call ? first_code(pk, dst) : 0u;
    stage_rows<N2T>(g, pk, pair, c0, raw, hb, c_first);
    if (pk.first_call && dst && blockIdx.x == 0 && pair == 0 && threadIdx.x == 0) dst->first_code = (int)c_first;
    cp_async_wait_all();
    __syncthreads();
    const int t = threadIdx.x, n1 = c0 + t;
    const ColPos cp = col_pos<ORD>(t);
    float2 x[16];
    load_columns<ORD>(hb, raw, cp, s_ln, x);
    dft16<false>(x);
    twiddle16<false>(x, tw, n1);
    float2 *out = fftws + (size_t)pair * g.N + n1;
#pragma unroll
    for (int k2 = 0; k2 < 16; k2++) out[k2 * N2T] = x[k2];
}

// digit reversal of a P-digit base-16 index
template <int P>
__device__ __forceinline__ int drev16(int pos)
{
    int r = 0;
#pragma unroll
    for (int i = 0; i < P; i++) { r = (r << 4) | (pos & 15); pos >>= 4; }
    return r;
}

// Hilbert multiplier of bin k of an N-point spectrum: -j (0<k<N/2), +j (k>N/2), 0 at 0 and N/2
__device__ __forceinline__ float2 hilbert_mul(float2 v, int k, int N)
{
    if (k == 0 || 2 * k == N) return make_float2(0.f, 0.f);
    return (2 * k < N) ? make_float2(v.y, -v.x) : make_float2(-v.y, v.x);
}

// K1b: per row k2 of a block pair of 2^16-point blocks, 4096-point FFT (radix-16
// decimation in frequency, digit-reversed output), Hilbert multiplier on the bins
// k = k2 + 16 k1, inverse FFT (radix-16 decimation in time back to natural order).  In
// place, one row per CTA.
constexpr int kRowN2 = 4096, kRowPad = kRowN2 + kRowN2 / 16;   // row and padded row
__global__ void __launch_bounds__(256, 3) k_kk_rows(KkGeom g, float2 *fftws,
                                                   const float2 *__restrict__ twN2g)
{
    constexpr int P = 3, N2 = kRowN2, TPR = N2 / 16;
    extern __shared__ float2 s[];                 // the padded row
    __shared__ float2 s_tw[128];
    const TwSmem tw2 = stage_tw(twN2g, N2, s_tw);
    pdl_wait();
    const int t = threadIdx.x, row = blockIdx.x, k2 = row & 15;
    float2 *d = fftws + (size_t)row * N2;
    float2 x[16];
    // forward pass 0 (sub-transform size N2) straight from global memory
#pragma unroll
    for (int r = 0; r < 16; r++) x[r] = d[t + r * TPR];
    cp_async_wait_all();
    __syncthreads();   // staged twiddles
    dft16<false>(x);
    twiddle16<false>(x, tw2, t);
    // a pass's 16 elements base + r stride sit at pad16(base) + r (stride + stride / 16)
    // when stride is a multiple of 16, or base is one and stride is 1: one pointer per
    // pass and compile-time offsets
    float2 *const s0 = s + pad16(t);
    constexpr int STR0 = TPR + TPR / 16;
#pragma unroll
    for (int r = 0; r < 16; r++) s0[r * STR0] = x[r];
    __syncthreads();
    // remaining forward passes; the last one is fused with the multiplier and the
    // first inverse pass
#pragma unroll
    for (int p = 1; p < P; p++) {
        const int M = N2 >> (4 * p), sub = M / 16, str = sub + sub / 16;
        int o = (t / sub) * M, j = t % sub;
        float2 *const sb = s + pad16(o + j);
#pragma unroll
        for (int r = 0; r < 16; r++) x[r] = sb[r * str];
        dft16<false>(x);
        if (p < P - 1) {
            twiddle16<false>(x, tw2, j * (N2 / M));
#pragma unroll
            for (int r = 0; r < 16; r++) sb[r * str] = x[r];
            __syncthreads();
        } else {
            // M = 16: positions o + r hold X[k2 + 16 * drev(o + r)]
#pragma unroll
            for (int r = 0; r < 16; r++) x[r] = hilbert_mul(x[r], k2 + 16 * drev16<P>(o + r), g.N);
            dft16<true>(x);
#pragma unroll
            for (int r = 0; r < 16; r++) sb[r] = x[r];   // sub = 1, j = 0
            __syncthreads();
        }
    }
    // inverse passes P-2 .. 1
#pragma unroll
    for (int p = P - 2; p >= 1; p--) {
        const int M = N2 >> (4 * p), sub = M / 16, str = sub + sub / 16;
        int o = (t / sub) * M, j = t % sub;
        float2 *const sb = s + pad16(o + j);
#pragma unroll
        for (int r = 0; r < 16; r++) x[r] = sb[r * str];
        twiddle16<true>(x, tw2, j * (N2 / M));
        dft16<true>(x);
#pragma unroll
        for (int r = 0; r < 16; r++) sb[r * str] = x[r];
        __syncthreads();
    }
    // inverse pass 0 to global memory
#pragma unroll
    for (int r = 0; r < 16; r++) x[r] = s0[r * STR0];
    twiddle16<true>(x, tw2, t);
    dft16<true>(x);
#pragma unroll
    for (int r = 0; r < 16; r++) d[t + r * TPR] = x[r];
}

// Carrier and intensity sums of a call, from which its carrier and gain follow.
// Each warp's FP32 sums of E become exact integers in units of 2^-24 (a warp's sum
// is below 2^17 in magnitude and a call holds at most 2^30 samples of |E| <= 64, so
// every total fits a signed 64-bit integer).  One 64-bit atomic per CTA and quantity
// adds them to the slot's totals.  Integer addition does not depend on order, so the
// totals, and the carrier, are the same whatever order the CTAs run in.  The CTA that
// takes the last ticket forms, in FP64, the carrier c = sum E / n, the mean intensity
// sum 2I / 2n and the gain 1 / sqrt(sps (mean I - |c|^2)), then clears the totals and
// the ticket for the slot's next call.
constexpr double kCarrierUnit = 16777216.0;   // 2^24
__device__ __forceinline__ void carrier_sums(const KkGeom &g, DevState *dst, float sre, float sim, int si2,
                                             int ncta)
{
    if (!dst) return;   // field only
    __shared__ long long s_q[3][32];
    sre = warp_sum_f(sre);
    sim = warp_sum_f(sim);
    si2 = (int)__reduce_add_sync(0xffffffffu, (unsigned)si2);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    // the power-of-two scaling is exact in FP32 (a warp's sum is far from overflow), so this
    // rounds once, to the nearest integer
    if (lane < 2) s_q[lane][wid] = __float2ll_rn((lane ? sim : sre) * (float)kCarrierUnit);
    if (lane == 2) s_q[2][wid] = si2;
    __syncthreads();
    if (wid != 0) return;
    // lane q < 3 carries total q from here on
    unsigned long long *S = dst->csum[g.slot];
    if (lane < 3) {
        long long a = 0;
        for (int i = 0; i < (int)(blockDim.x >> 5); i++) a += s_q[lane][i];
        atomicAdd(S + lane, (unsigned long long)a);
        __threadfence();   // three threads' adds before lane 0's ticket
    }
    __syncwarp();
    unsigned last = 0;
    if (lane == 0) last = take_ticket(&dst->ticket[g.slot]) == (unsigned)(ncta - 1);
    if (!__shfl_sync(0xffffffffu, last, 0)) return;
    __syncwarp();   // what lane 0's ticket acquired, for the other lanes
    const double cnt = (double)(g.e_k - g.e_prev);
    double m = 0.0;
    if (lane < 3) {
        const double t = (double)(long long)atomicExch(S + lane, 0ull);
        m = lane < 2 ? t * (1.0 / kCarrierUnit) / cnt : t / (2.0 * cnt);   // the scaling is exact
    }
    const double cr = __shfl_sync(0xffffffffu, m, 0), ci = __shfl_sync(0xffffffffu, m, 1),
                 ibar = __shfl_sync(0xffffffffu, m, 2);
    if (lane == 0) {
        const double P = ibar - (cr * cr + ci * ci);
        dst->cg[g.slot][0] = cr;
        dst->cg[g.slot][1] = ci;
        dst->cg[g.slot][2] = (P > 0.0) ? 1.0 / sqrt((double)g.sps * P) : 1.0;
        dst->ticket[g.slot] = 0u;
    }
}

// field history for the matched filter: E[n], n in [e_prev - kEHist, e_prev) (E_prev null:
// the caller keeps none), the samples first, first + step, .. by one thread, NB loads at a time
template <int NB>
__device__ __forceinline__ void carry_field(const KkGeom &g, float2 *E, const float2 *E_prev, int first, int step)
{
    if (!E_prev) return;
    for (int i0 = first; i0 < kEHist; i0 += NB * step) {
        float2 v[NB];
#pragma unroll
        for (int k = 0; k < NB; k++) {   // every load issues before the first one is stored
            const int i = i0 + k * step;
            const long long n = g.e_prev - kEHist + i;
            v[k] = i < kEHist && n >= 0 ? E_prev[n - g.ebase_prev] : make_float2(0.f, 0.f);
        }
#pragma unroll
        for (int k = 0; k < NB; k++)
            if (i0 + k * step < kEHist) E[i0 + k * step] = v[k];
    }
}

// E = sqrt(I) exp(j phi) (Fig. 1d) of the kept outputs of a column of a block pair: x[q]
// holds N times the phase of both blocks at window position n1 + N2T q; the codes come from
// the staged rows.  Adds to the carrier sums and to the sum of the intensities (halves and
// integers below 2^24: exact in FP32).
template <int ORD, int N2T>
__device__ __forceinline__ void emit_field(const KkGeom &g, int pair, int n1, const float2 (&x)[16],
                                           const uint32_t (*raw)[kRawWords], const ColPos &cp, float2 *E,
                                           float &sre, float &sim, float &sint)
{
    const float invN = 1.0f / (float)g.N;
#pragma unroll
    for (int half = 0; half < 2; half++) {
        int j = 2 * pair + half;
        if (j >= g.J) break;
        int tlo, thi;
        ols_kept(g, j, tlo, thi);
        float2 *Eb = E + (ols_ws(g, j) - g.ebase) + n1;
        // rows q whose position n1 + N2T q lies in [tlo, thi), as a bit mask
        const int qlo = max((tlo - n1 + N2T - 1) / N2T, 0), qhi = min((thi - n1 + N2T - 1) / N2T, 16);
        const unsigned keep = qhi > qlo ? ((1u << qhi) - 1u) & ~((1u << qlo) - 1u) : 0u;
#pragma unroll
        for (int q = 0; q < 16; q++) {
            if (!(keep & (1u << q))) continue;
            const uint32_t code = col_code<ORD>(raw[16 * half + q], cp);
            float phi = (half ? x[q].y : x[q].x) * invN;
            float sn, cs;
            __sincosf(phi, &sn, &cs);   // |phi| < pi: absolute error <= 2^-21.41
            // the hardware square-root approximation (sqrt.approx.f32) in place of the
            // correctly rounded sequence; the field is held to the FP64 reference
            // within 1e-5 relative RMS
            const float in = fmaxf((float)code, 0.5f);
            const float A = sqrt_approx(in);
            float2 e = make_float2(A * cs, A * sn);
            Eb[N2T * q] = e;
            sre += e.x;
            sim += e.y;
            sint += in;
        }
    }
}

// K1c: inverse radix-16 pass, then the field of every kept output, written at its stream
// position, and the per-call carrier / intensity sums (exact integer totals,
// carrier_sums).  ORD: the pack order; N2T: the row length N / 16.
template <int ORD, int N2T>
__global__ void __launch_bounds__(kCtaK1) k_kk_inv(KkGeom g, KkPacked pk, const float2 *fftws,
                                                  const KkTables tb, float2 *E,
                                                  const float2 *E_prev, DevState *dst)
{
    __shared__ float2 s_tw[512];
    __shared__ __align__(16) uint32_t raw[32][kRawWords];
    const TwSmem tw = stage_tw(tb.twN, g.N, s_tw);
    pdl_wait();
    int pair = blockIdx.y;
    const int c0 = blockIdx.x * blockDim.x;
    const bool hb = 2 * pair + 1 < g.J;
    stage_rows<N2T>(g, pk, pair, c0, raw, hb, before_stream(g, pair, hb) ? first_code(pk, dst) : 0u);
    float sre = 0.f, sim = 0.f, sint = 0.f;
    if (blockIdx.y == 0) carry_field<1>(g, E, E_prev, c0 + threadIdx.x, gridDim.x * blockDim.x);
    const int t = threadIdx.x, n1 = c0 + t;
    const ColPos cp = col_pos<ORD>(t);
    float2 x[16];
    const float2 *in = fftws + (size_t)pair * g.N + n1;
#pragma unroll
    for (int k2 = 0; k2 < 16; k2++) x[k2] = in[k2 * N2T];
    cp_async_wait_all();
    __syncthreads();   // staged twiddles and rows
    twiddle16<true>(x, tw, n1);
    dft16<true>(x);
    emit_field<ORD, N2T>(g, pair, n1, x, raw, cp, E, sre, sim, sint);
    carrier_sums(g, dst, sre, sim, (int)(2.f * sint), gridDim.x * gridDim.y);
}

// ============================================== KK front end, 4096-point blocks
// A pair of 4096-point blocks (32 KB of complex spectrum) fits one CTA, so the whole
// Hilbert transform of the pair runs in one kernel: thread t takes column t of the 16 x 256
// four-step layout (codes, u = ln(I)/2, radix-16 DFT, twiddle), then a sixteenth of row
// t / 16 (256-point FFT in two radix-16 passes, multiplier, inverse; a row belongs to half a
// warp), then column t again (inverse DFT, field, carrier sums).  The arithmetic is that of
// the three-kernel form of the 2^16-point blocks, pass by pass.  CTAs from npairs on copy
// the next call's history.
// Bound by latency: a chain of six passes at three CTAs per SM.  41,984 samples with V = 512
// (six CTAs): 7.0 us per call of rx_kk_field_noalloc; 28.7 us as three kernels (column DFT, rows,
// column DFT and field, the spectrum through global memory twice), a clear and a copy.
constexpr int kBkN2 = 256, kBkRow = kBkN2 + kBkN2 / 16;   // row length and padded row
struct BkSmem {
    static constexpr int FFT = 0;                                    // float2 [16][kBkRow]; before it the ln table
    static constexpr int RAW = FFT + 16 * kBkRow * 8;                // staged packed rows
    static constexpr int TW = RAW + 32 * kRawWords * 4;              // factored W_4096 (128), W_256 (32)
    static constexpr int TOTAL = TW + (128 + 32) * 8;
};
static_assert(kLutCodes * 4 <= BkSmem::RAW, "the ln table fits the spectrum's place");

template <int ORD>
__global__ void __launch_bounds__(kCtaK1, 3) k_kk_block(KkGeom g, KkPacked pk, const KkTables tb,
                                                       float2 *E, const float2 *E_prev,
                                                       DevState *dst)
{
    extern __shared__ __align__(16) unsigned char bksm[];
    float2 *fft = reinterpret_cast<float2 *>(bksm + BkSmem::FFT);
    float *s_ln = reinterpret_cast<float *>(bksm + BkSmem::FFT);
    uint32_t(*raw)[kRawWords] = reinterpret_cast<uint32_t(*)[kRawWords]>(bksm + BkSmem::RAW);
    float2 *s_tw = reinterpret_cast<float2 *>(bksm + BkSmem::TW);
    const int pair = blockIdx.x, t = threadIdx.x;
    const TwSmem tw = stage_tw(tb.twN, 16 * kBkN2, s_tw);
    const TwSmem tw2 = stage_tw(tb.twN2, kBkN2, s_tw + 128);
    stage_ln(tb.lnt, s_ln);
    pdl_wait();
    if (pk.lat && pair == 0 && t == 0) lat_start(pk.lat, pk.lat_slot);
    if (pair >= g.npairs) {
        copy_hist(pk, pair - g.npairs, gridDim.x - g.npairs);
        cp_async_wait_all();
        return;
    }
    const bool hb = 2 * pair + 1 < g.J;
    const uint32_t c_first = before_stream(g, pair, hb) || pk.first_call ? first_code(pk, dst) : 0u;
    stage_rows<kBkN2>(g, pk, pair, 0, raw, hb, c_first);
    if (pk.first_call && dst && pair == 0 && t == 0) dst->first_code = (int)c_first;
    if (pair == 0) carry_field<kEHist / kCtaK1>(g, E, E_prev, t, kCtaK1);
    cp_async_wait_all();
    __syncthreads();
    const ColPos cp = col_pos<ORD>(t);
    float2 x[16];
    load_columns<ORD>(hb, raw, cp, s_ln, x);
    __syncthreads();   // the ln table has been read: the spectrum takes its place
    dft16<false>(x);
    twiddle16<false>(x, tw, t);
    float2 *const col = fft + pad16(t);
#pragma unroll
    for (int k2 = 0; k2 < 16; k2++) col[k2 * kBkRow] = x[k2];
    __syncthreads();
    {
        const int k2 = t >> 4, tt = t & 15;
        float2 *const r0 = fft + k2 * kBkRow + tt;             // positions tt + 16 r: pad16 = tt + 17 r
        float2 *const r1 = fft + k2 * kBkRow + pad16(16 * tt);   // positions 16 tt + r
#pragma unroll
        for (int r = 0; r < 16; r++) x[r] = r0[17 * r];
        dft16<false>(x);
        twiddle16<false>(x, tw2, tt);
#pragma unroll
        for (int r = 0; r < 16; r++) r0[17 * r] = x[r];
        __syncwarp();
#pragma unroll
        for (int r = 0; r < 16; r++) x[r] = r1[r];
        dft16<false>(x);
#pragma unroll
        for (int r = 0; r < 16; r++) x[r] = hilbert_mul(x[r], k2 + 16 * drev16<2>(16 * tt + r), 16 * kBkN2);
        dft16<true>(x);
#pragma unroll
        for (int r = 0; r < 16; r++) r1[r] = x[r];
        __syncwarp();
#pragma unroll
        for (int r = 0; r < 16; r++) x[r] = r0[17 * r];
        twiddle16<true>(x, tw2, tt);
        dft16<true>(x);
#pragma unroll
        for (int r = 0; r < 16; r++) r0[17 * r] = x[r];
    }
    __syncthreads();
#pragma unroll
    for (int k2 = 0; k2 < 16; k2++) x[k2] = col[k2 * kBkRow];
    twiddle16<true>(x, tw, t);
    dft16<true>(x);
    float sre = 0.f, sim = 0.f, sint = 0.f;
    emit_field<ORD, kBkN2>(g, pair, t, x, raw, cp, E, sre, sim, sint);
    carrier_sums(g, dst, sre, sim, (int)(2.f * sint), g.npairs);
}

// ====================================================== KK front end, fused
// One thread-block cluster of kClC CTAs per block pair computes the whole
// Hilbert transform of the pair in distributed shared memory (the 2^16-point
// case, N2 = 4096): CTA c owns rows k2 = 2c, 2c+1 of the 16 x 4096 four-step
// layout, padded as in K1b.
//   A  columns:  CTA c takes columns n1 in [512 c, 512 c + 512): 12-bit codes
//      straight from the packed input, u = ln(I)/2, radix-16 DFT over the
//      stride-N2 index, twiddle, each result stored into the shared memory of
//      the CTA that owns its row;
//   B  rows:     forward 4096-point FFT, Hilbert multiplier, inverse FFT of the
//      CTA's two rows in its own shared memory (the passes of K1b);
//   C  columns:  the 16 values of each of its columns gathered back from the
//      owners, inverse radix-16 DFT, E = sqrt(I) exp(j phi) for the kept
//      outputs and the carrier sums (the reduction of K1c).
// Cluster barriers separate the phases, so the 512 KB of a pair never leave the
// chip; global traffic is the packed input and the field.
constexpr int kClC = 8;
constexpr int kClThreads = 256;
constexpr int kClN2 = 4096;
constexpr int kClRow = kClN2 + kClN2 / 16;   // padded row
constexpr int kClCols = kClN2 / kClC;        // columns per CTA
constexpr size_t kClSmem = (size_t)(2 * kClRow + 512 + 128) * sizeof(float2);

// 12-bit codes of 32 consecutive stream samples (one per lane) starting at
// virtual-buffer offset t0 (a multiple of 32, so its 48 bytes start on 16 bytes
// and lie wholly in the history or in this buffer): lanes 0..11 load one word
// each, every lane takes its two bytes from the owners by shuffle.
__device__ __forceinline__ uint32_t warp_codes(const KkPacked &pk, long long t0, int lane)
{
    long long vb = (3 * t0) >> 1;
    const uint32_t *src = reinterpret_cast<const uint32_t *>(vb < pk.hist_bytes ? pk.hist + vb
                                                                                : pk.in + (vb - pk.hist_bytes));
    uint32_t w = lane < 12 ? src[lane] : 0u;
    int b = (3 * lane) >> 1;
    uint32_t w0 = __shfl_sync(0xffffffffu, w, b >> 2);
    uint32_t w1 = __shfl_sync(0xffffffffu, w, min((b >> 2) + 1, 31));
    uint32_t v = __funnelshift_r(w0, w1, 8 * (b & 3));
    uint32_t lo = v & 0xFFu, hi = (v >> 8) & 0xFFu;
    if (pk.order == 0) return (lane & 1) ? ((lo >> 4) | (hi << 4)) : (lo | ((hi & 0xFu) << 8));
    return (lane & 1) ? (((lo & 0xFu) << 8) | hi) : ((lo << 4) | (hi >> 4));
}

__global__ void __cluster_dims__(kClC, 1, 1) __launch_bounds__(kClThreads, 3)
    k_kk_cluster(KkGeom g, KkPacked pk, const KkTables tb, float2 *E,
                 const float2 *E_prev, DevState *dst)
{
    namespace cg = cooperative_groups;
    cg::cluster_group cl = cg::this_cluster();
    extern __shared__ float2 smc[];
    float2 *rows = smc;                         // [2][kClRow]
    const TwSmem tw = stage_tw(tb.twN, g.N, smc + 2 * kClRow);
    const TwSmem tw2 = stage_tw(tb.twN2, kClN2, smc + 2 * kClRow + 512);
    pdl_wait();
    const int c = (int)cl.block_rank();
    const int pair = blockIdx.x / kClC;
    const int t = threadIdx.x;
    if (pk.lat && blockIdx.x == 0 && t == 0) lat_start(pk.lat, pk.lat_slot);
    const bool hb = 2 * pair + 1 < g.J;
    const uint32_t c_first = first_code(pk, dst);
    if (pk.first_call && blockIdx.x == 0 && t == 0) dst->first_code = (int)c_first;
    // history of the next call (packed bytes [in_bytes, in_bytes + hist_bytes) of
    // the virtual buffer), spread over the grid
    if (pk.hist_next) copy_hist(pk, blockIdx.x, gridDim.x);
    if (blockIdx.x == 0) carry_field<kEHist / kClThreads>(g, E, E_prev, t, kClThreads);
    cp_async_wait_all();
    __syncthreads();   // staged twiddles

    // ---- A: forward column DFTs, scattered to the row owners
    const long long wsa = ols_ws(g, 2 * pair), wsb = hb ? ols_ws(g, 2 * pair + 1) : 0;
    cl.sync();         // every CTA of the cluster is running before remote stores
#pragma unroll 1
    for (int h = 0; h < kClCols / kClThreads; h++) {
        const int n1 = c * kClCols + h * kClThreads + t;
        float2 x[16];
        const int lane = t & 31;
        const int n1w = n1 - lane;                  // first column of the warp
#pragma unroll
        for (int q = 0; q < 16; q++) {
            long long na = wsa + n1w + (long long)kClN2 * q;   // warp-uniform, a multiple of 32
            uint32_t ca = na < 0 ? c_first : warp_codes(pk, na - g.cbase, lane);
            float ub = 0.f;
            if (hb) {
                long long nb2 = wsb + n1w + (long long)kClN2 * q;
                ub = __ldg(tb.lnt + (nb2 < 0 ? c_first : warp_codes(pk, nb2 - g.cbase, lane)));
            }
            x[q] = make_float2(__ldg(tb.lnt + ca), ub);
        }
        dft16<false>(x);
#pragma unroll
        for (int k2 = 0; k2 < 16; k2++) {
            float2 *dstp = cl.map_shared_rank(rows + (k2 & 1) * kClRow, k2 >> 1);
            dstp[pad16(n1)] = k2 ? cmul(x[k2], tw(n1 * k2)) : x[0];
        }
    }
    cl.sync();

    // ---- B: the CTA's two rows, FFT / Hilbert / inverse FFT (passes of K1b, P = 3)
#pragma unroll 1
    for (int lr = 0; lr < 2; lr++) {
        const int k2 = 2 * c + lr;
        float2 *s = rows + lr * kClRow;
        float2 x[16];
#pragma unroll
        for (int r = 0; r < 16; r++) x[r] = s[pad16(t + r * 256)];
        dft16<false>(x);
#pragma unroll
        for (int r = 1; r < 16; r++) x[r] = cmul(x[r], tw2(t * r));
#pragma unroll
        for (int r = 0; r < 16; r++) s[pad16(t + r * 256)] = x[r];
        __syncthreads();
        {   // pass 1 (M = 256)
            int o = (t / 16) * 256, j = t % 16;
#pragma unroll
            for (int r = 0; r < 16; r++) x[r] = s[pad16(o + j + r * 16)];
            dft16<false>(x);
#pragma unroll
            for (int r = 1; r < 16; r++) x[r] = cmul(x[r], tw2(j * r * 16));
#pragma unroll
            for (int r = 0; r < 16; r++) s[pad16(o + j + r * 16)] = x[r];
        }
        __syncthreads();
        {   // pass 2 (M = 16), Hilbert multiplier on X[k2 + 16 drev(o + r)], first inverse pass
            int o = t * 16;
#pragma unroll
            for (int r = 0; r < 16; r++) x[r] = s[pad16(o + r)];
            dft16<false>(x);
#pragma unroll
            for (int r = 0; r < 16; r++) x[r] = hilbert_mul(x[r], k2 + 16 * drev16<3>(o + r), g.N);
            dft16<true>(x);
#pragma unroll
            for (int r = 0; r < 16; r++) s[pad16(o + r)] = x[r];
        }
        __syncthreads();
        {   // inverse pass 1
            int o = (t / 16) * 256, j = t % 16;
#pragma unroll
            for (int r = 0; r < 16; r++) {
                x[r] = s[pad16(o + j + r * 16)];
                if (r) x[r] = cmulc(x[r], tw2(j * r * 16));
            }
            dft16<true>(x);
#pragma unroll
            for (int r = 0; r < 16; r++) s[pad16(o + j + r * 16)] = x[r];
        }
        __syncthreads();
        // inverse pass 0, in place
#pragma unroll
        for (int r = 0; r < 16; r++) {
            x[r] = s[pad16(t + r * 256)];
            if (r) x[r] = cmulc(x[r], tw2(t * r));
        }
        dft16<true>(x);
#pragma unroll
        for (int r = 0; r < 16; r++) s[pad16(t + r * 256)] = x[r];
    }
    cl.sync();

    // ---- C: inverse column DFTs from the row owners, field and carrier sums
    float sre = 0.f, sim = 0.f;
    int si2 = 0;
    const float invN = 1.0f / (float)g.N;
#pragma unroll 1
    for (int h = 0; h < kClCols / kClThreads; h++) {
        const int n1 = c * kClCols + h * kClThreads + t;
        float2 x[16];
#pragma unroll
        for (int k2 = 0; k2 < 16; k2++) {
            const float2 *srcp = cl.map_shared_rank(rows + (k2 & 1) * kClRow, k2 >> 1);
            x[k2] = srcp[pad16(n1)];
        }
#pragma unroll
        for (int k2 = 1; k2 < 16; k2++) x[k2] = cmulc(x[k2], tw(n1 * k2));
        dft16<true>(x);
#pragma unroll
        for (int half = 0; half < 2; half++) {
            int j = 2 * pair + half;
            if (j >= g.J) break;
            long long ws = half ? wsb : wsa;
            int tlo, thi;
            ols_kept(g, j, tlo, thi);
            const int lane = t & 31;
#pragma unroll
            for (int q = 0; q < 16; q++) {
                int tt = n1 + kClN2 * q;
                int tw0 = tt - lane;                    // warp-uniform
                if (tw0 + 31 < tlo || tw0 >= thi) continue;
                long long n = ws + tt;
                long long nw = ws + tw0;
                uint32_t code = nw < 0 ? c_first : warp_codes(pk, nw - g.cbase, lane);
                if (tt < tlo || tt >= thi) continue;
                float phi = (half ? x[q].y : x[q].x) * invN;
                float sn, cs;
                __sincosf(phi, &sn, &cs);   // |phi| < pi: absolute error <= 2^-21.41
                float A = sqrt_approx(code ? (float)code : 0.5f);
                float2 e = make_float2(A * cs, A * sn);
                E[n - g.ebase] = e;
                sre += e.x;
                sim += e.y;
                si2 += code ? 2 * (int)code : 1;
            }
        }
    }
    cl.sync();   // no CTA leaves while its rows may still be read

    carrier_sums(g, dst, sre, sim, si2, gridDim.x);
}

__global__ void k_kk_hist(KkPacked pk)
{
    pdl_wait();
    if (pk.lat && blockIdx.x == 0 && threadIdx.x == 0) lat_start(pk.lat, pk.lat_slot);
    copy_hist(pk, blockIdx.x, gridDim.x);
}

cudaError_t launch_kk_hist(const KkInput &inp, cudaStream_t st, const KkSync &sync)
{
    if (sync.wait_fwd) cudaStreamWaitEvent(st, sync.wait_fwd, 0);
    KkPacked pk;
    pk.hist = inp.hist;
    pk.in = inp.in;
    pk.hist_next = inp.hist_next;
    pk.hist_bytes = inp.hist_bytes;
    pk.in_bytes = inp.in_bytes;
    pk.order = inp.order;
    pk.first_call = inp.first_call;
    pk.lat = inp.lat;
    pk.lat_slot = inp.lat_slot;
    const cudaError_t e = launch_k(k_kk_hist, 32, 256, 0, st, sync.pdl_first, pk);
    if (sync.rec_fwd) cudaEventRecord(sync.rec_fwd, st);
    return e;
}

cudaError_t prepare_kk_front()
{
    cudaError_t e = cudaFuncSetAttribute(k_kk_cluster, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kClSmem);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_kk_block<0>, cudaFuncAttributeMaxDynamicSharedMemorySize, BkSmem::TOTAL);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_kk_block<1>, cudaFuncAttributeMaxDynamicSharedMemorySize, BkSmem::TOTAL);
    return e;
}

cudaError_t launch_kk_front(const KkGeom &g, const KkInput &inp, float2 *fftws, const KkTables &tb,
                            float2 *E, const float2 *E_prev, DevState *dst, cudaStream_t st, void *prof,
                            const KkSync &sync)
{
    KkPacked pk;
    pk.hist = inp.hist;
    pk.in = inp.in;
    pk.hist_next = inp.hist_next;
    pk.hist_bytes = inp.hist_bytes;
    pk.in_bytes = inp.in_bytes;
    pk.order = inp.order;
    pk.first_call = inp.first_call;
    pk.lat = inp.lat;
    pk.lat_slot = inp.lat_slot;
    cudaError_t e = cudaSuccess;
    if (sync.wait_fwd) cudaStreamWaitEvent(st, sync.wait_fwd, 0);
    if ((g.N2 == kClN2 && g.fused) || g.N2 == kBkN2) {
        // one kernel: the cluster form of 2^16-point blocks or the one-CTA form of
        // 4096-point blocks (profiled as the K1a stage)
        if (sync.wait_inv) cudaStreamWaitEvent(st, sync.wait_inv, 0);
        prof_stage(prof, 1, st);
        if (g.N2 == kClN2)
            e = launch_k(k_kk_cluster, g.npairs * kClC, kClThreads, kClSmem, st, sync.pdl_first, g, pk, tb, E, E_prev, dst);
        else
            e = launch_k(pk.order ? k_kk_block<1> : k_kk_block<0>, g.npairs + (inp.hist_next ? 1 : 0), kCtaK1,
                         BkSmem::TOTAL, st, sync.pdl_first, g, pk, tb, E, E_prev, dst);
        if (sync.rec_fwd) cudaEventRecord(sync.rec_fwd, st);
        prof_stage(prof, -2, st);
        prof_stage(prof, -3, st);
        prof_stage(prof, -4, st);
        return e;
    }
    if (g.N2 != kRowN2) return cudaErrorInvalidValue;   // N is 65536 or 4096
    dim3 grid(kRowN2 / kCtaK1, g.npairs);
    dim3 grid_a(kRowN2 / kCtaK1, g.npairs + (inp.hist_next ? 1 : 0));
    prof_stage(prof, 1, st);
    e = launch_k(pk.order ? k_kk_fwd<1, kRowN2> : k_kk_fwd<0, kRowN2>, grid_a, kCtaK1, 0, st, sync.pdl_first, g, pk, fftws, tb,
                 dst);
    if (sync.rec_fwd) cudaEventRecord(sync.rec_fwd, st);
    prof_stage(prof, -2, st);
    if (e == cudaSuccess)
        e = launch_k(k_kk_rows, g.npairs * 16, 256, kRowPad * sizeof(float2), st, sync.pdl, g, fftws, tb.twN2);
    if (sync.wait_inv) cudaStreamWaitEvent(st, sync.wait_inv, 0);
    prof_stage(prof, -3, st);
    if (e == cudaSuccess)
        e = launch_k(pk.order ? k_kk_inv<1, kRowN2> : k_kk_inv<0, kRowN2>, grid, kCtaK1, 0, st, sync.pdl, g, pk, fftws, tb,
                     E, E_prev, dst);
    prof_stage(prof, -4, st);
    return e;
}

// ============================================================ KK matched filter
// y[m] = g * sum_i h_i * (E[2m - i] - c) * exp(-j 2 pi ds (2m - i)),  x[n < 0] = 0.
// 256 outputs per CTA from a shared-memory tile of the carrier-removed,
// downshifted field.  CTA 0 also carries the equaliser history [ybase, f_prev).
constexpr int kMfOut = 256;

__global__ void __launch_bounds__(kMfOut) k_kk_mf(const float2 *E, long long ebase, long long e_k,
                                                 long long f_prev, long long f_k, const float *__restrict__ rrc,
                                                 int hmf, const float2 *__restrict__ ds_tab, int ds_num,
                                                 int ds_den, const double *cg,
                                                 float2 *Y, long long ybase,
                                                 const float2 *Y_prev, long long ybase_prev)
{
    extern __shared__ float2 xs[];
    pdl_wait();
    long long m0 = f_prev + (long long)blockIdx.x * kMfOut;
    int L = 2 * kMfOut + 2 * hmf;
    float2 c = make_float2((float)cg[0], (float)cg[1]);
    float gn = (float)cg[2];
    long long n0 = 2 * m0 - hmf;
    for (int i = threadIdx.x; i < L; i += blockDim.x) {
        long long n = n0 + i;
        float2 v = make_float2(0.f, 0.f);
        if (n >= 0 && n < e_k) {
            int p = (int)(((n % ds_den) * ds_num) % ds_den);
            v = cmul(csub(E[n - ebase], c), __ldg(ds_tab + p));
        }
        xs[i] = v;
    }
    if (blockIdx.x == 0) {
        for (long long m = ybase + threadIdx.x; m < f_prev; m += blockDim.x)
            Y[m - ybase] = (m < 0) ? make_float2(0.f, 0.f) : Y_prev[m - ybase_prev];
    }
    __syncthreads();
    long long m = m0 + threadIdx.x;
    if (m >= f_k) return;
    const float2 *xc = xs + 2 * threadIdx.x + hmf;
    float ar = 0.f, ai = 0.f;
    for (int i = -hmf; i <= hmf; i++) {
        float h = __ldg(rrc + i + hmf);
        float2 v = xc[-i];
        ar = fmaf(h, v.x, ar);
        ai = fmaf(h, v.y, ai);
    }
    Y[m - ybase] = make_float2(gn * ar, gn * ai);
}

// Register-tiled form for a compile-time half length HMF (even).  With the tile
// starting at n0 = 2 m0 - HMF, the pairs P[p] = (x[n0 + 2p], x[n0 + 2p + 1])
// turn the decimating filter into two plain FIRs over the pair index:
//   y[m0 + j] = g * sum_{u=0..HMF} (ge[u] P[j+u].first + go[u] P[j+u].second)
// with ge[u] = h[HMF - 2u], go[u] = h[HMF - 2u - 1].  Each thread computes 8
// consecutive outputs from a sliding window of 8 pairs held in registers (one
// 16-byte shared load per tap); the pair layout keeps one spare slot per 8 pairs,
// which makes the stride-8-pair loads of a warp free of bank conflicts.  The real
// and imaginary parts of an output accumulate as one packed FP32 pair (one
// fma.rn.f32x2 per tap and output, the same roundings as two scalar FMAs in the
// same order); the taps are kernel parameters, read from the constant bank as (g, g).
// A thread stages the pairs t, t + STRIDE, ..: where STRIDE is a multiple of the downshift's
// period in pairs (FIXED), they all turn by the same two phases, looked up once; otherwise
// the phases are looked up pair by pair.  STRIDE 120 serves every period that divides it
// (the default 11/80 cycles per sample: 40) and covers a tile in as many steps as 128.
// Bound by the shared-memory pipe and the packed FMAs (two issue cycles each: 7 us of the
// FMA pipe for 2^21 outputs) in 1.2 waves of CTAs.  2^22-sample buffer: 17.4 us on warm caches and
// 7.6 M warp instructions; 19.5 us and 10.1 M with taps in shared memory, phases per
// sample and 64-bit phase and range arithmetic.  Persistent CTAs that load the next tile
// into registers during the FIR took 16.5 us alone on warm caches against 17.4 but 1 to 3 us
// more in the receiver, where their 95 to 116 registers leave no room for other kernels.
// A thread's loads go out in two halves (40 registers): all at once they take 50, and six
// pipelined 2^20-sample buffers behind the cluster front end 500 us against 430, since the
// cluster of the next buffer then finds no room beside the filter.
template <int HMF>
struct MfTaps {
    f2x ge[HMF + 1];   // (ge, ge)
    f2x go[HMF];       // (go, go)
};
// (ph0 + n step) mod den with ph0, step < den: the 64-bit remainder only where the product
// needs it
__device__ __forceinline__ unsigned phase_at(unsigned ph0, unsigned step, unsigned long long n, unsigned den)
{
    const unsigned long long v = ph0 + n * step;
    return (v >> 32) ? (unsigned)(v % den) : (unsigned)v % den;
}

constexpr int kMfThreads = 128, kMfR = 8, kMfTileOut = kMfThreads * kMfR;
__host__ __device__ __forceinline__ int pad8(int p) { return p + (p >> 3); }

template <int HMF, int STRIDE, bool FIXED>
__global__ void __launch_bounds__(kMfThreads)
    k_kk_mf_t(const float2 *E, long long ebase, long long e_k, long long f_prev, long long f_k,
              const __grid_constant__ MfTaps<HMF> taps, const float2 *__restrict__ ds_tab, int ds_num, int ds_den,
              unsigned ph0, const double *cg, float2 *Y, long long ybase,
              const float2 *Y_prev, long long ybase_prev)
{
    constexpr int NPAIR = kMfTileOut + HMF + kMfR, NIT = (NPAIR + STRIDE - 1) / STRIDE;
    static_assert(STRIDE <= kMfThreads && STRIDE % 8 == 0, "one padded slot per 8 pairs");
    extern __shared__ float4 pr[];     // padded pair tile
    const long long m0 = f_prev + (long long)blockIdx.x * kMfTileOut;
    const long long n0 = 2 * m0 - HMF;
    // integer phase index of the downshift: ph0 + 2 ds_num pp (mod ds_den) at pair pp from the
    // call's first one on
    const unsigned den = (unsigned)ds_den, two = 2u * (unsigned)ds_num % den, odd = (unsigned)ds_num % den;
    unsigned idx = phase_at(ph0, two, (unsigned long long)blockIdx.x * kMfTileOut + threadIdx.x, den);
    const unsigned step = FIXED ? 0u : phase_at(0u, two, STRIDE, den);
    auto phases = [&](unsigned i) {    // e^{-2 pi j i / den} and the next sample's
        unsigned j = i + odd;
        j = j >= den ? j - den : j;
        const float2 a = __ldg(ds_tab + i), b = __ldg(ds_tab + j);
        return make_float4(a.x, a.y, b.x, b.y);
    };
    float4 w = phases(idx);
    // tile samples [lo, hi) lie inside the stream and the field; inner tiles load 16-byte
    // pairs where the field's origin allows it
    const int lo = n0 < 0 ? (int)-n0 : 0, hi = (int)min(e_k - n0, (long long)(2 * NPAIR));
    const float2 *Et = E + (n0 - ebase);
    const bool inner = lo == 0 && hi == 2 * NPAIR && ((uintptr_t)Et & 15) == 0;
    const bool act = STRIDE == kMfThreads || threadIdx.x < STRIDE;
    float4 *const ps = pr + pad8(threadIdx.x);
    pdl_wait();
    const float2 c = make_float2((float)cg[0], (float)cg[1]);
    const float gn = (float)cg[2];
    if (inner) {
        constexpr int HALF = (NIT + 1) / 2;
#pragma unroll
        for (int k0 = 0; k0 < NIT; k0 += HALF) {
            float4 v[HALF];   // the loads of half the pairs issue before the first one is used
#pragma unroll
            for (int k = k0; k < k0 + HALF && k < NIT; k++)
                if (act && threadIdx.x + k * STRIDE < NPAIR)
                    v[k - k0] = reinterpret_cast<const float4 *>(Et)[threadIdx.x + k * STRIDE];
#pragma unroll
            for (int k = k0; k < k0 + HALF && k < NIT; k++) {
                if (!FIXED && k) {
                    idx += step;
                    idx = idx >= den ? idx - den : idx;
                    w = phases(idx);
                }
                const float4 x = v[k - k0];
                const float2 a = cmul(csub(make_float2(x.x, x.y), c), make_float2(w.x, w.y));
                const float2 b = cmul(csub(make_float2(x.z, x.w), c), make_float2(w.z, w.w));
                if (act && threadIdx.x + k * STRIDE < NPAIR) ps[k * pad8(STRIDE)] = make_float4(a.x, a.y, b.x, b.y);
            }
        }
    } else if (act) {
#pragma unroll 1
        for (int k = 0; k < NIT; k++) {
            const int pp = threadIdx.x + k * STRIDE, n = 2 * pp;
            if (pp >= NPAIR) break;
            float2 a = make_float2(0.f, 0.f), b = a;
            if (n >= lo && n < hi) a = cmul(csub(Et[n], c), make_float2(w.x, w.y));
            if (n + 1 >= lo && n + 1 < hi) b = cmul(csub(Et[n + 1], c), make_float2(w.z, w.w));
            ps[k * pad8(STRIDE)] = make_float4(a.x, a.y, b.x, b.y);
            if (!FIXED) {
                idx += step;
                idx = idx >= den ? idx - den : idx;
                w = phases(idx);
            }
        }
    }
    if (blockIdx.x == 0) {
        for (long long m = ybase + threadIdx.x; m < f_prev; m += blockDim.x)
            Y[m - ybase] = (m < 0) ? make_float2(0.f, 0.f) : Y_prev[m - ybase_prev];
    }
    __syncthreads();
    const ulonglong2 *prp = reinterpret_cast<const ulonglong2 *>(pr);
    const int j0 = kMfR * threadIdx.x;
    ulonglong2 win[kMfR];
#pragma unroll
    for (int r = 0; r < kMfR; r++) win[r] = prp[pad8(j0 + r)];
    f2x acc[kMfR];
#pragma unroll
    for (int r = 0; r < kMfR; r++) acc[r] = 0ull;   // (+0, +0)
#pragma unroll
    for (int u = 0; u <= HMF; u++) {
#pragma unroll
        for (int r = 0; r < kMfR; r++) acc[r] = f2_fma(taps.ge[u], win[r].x, acc[r]);
        if (u < HMF) {
#pragma unroll
            for (int r = 0; r < kMfR; r++) acc[r] = f2_fma(taps.go[u], win[r].y, acc[r]);
#pragma unroll
            for (int r = 0; r < kMfR - 1; r++) win[r] = win[r + 1];
            win[kMfR - 1] = prp[pad8(j0 + u + kMfR)];
        }
    }
    const f2x g2 = f2_pack(gn, gn);
    float2 out[kMfR];
#pragma unroll
    for (int r = 0; r < kMfR; r++) out[r] = f2_unpack(f2_mul(g2, acc[r]));
    long long mb = m0 + j0;
    if (mb + kMfR <= f_k) {
        float4 *o = reinterpret_cast<float4 *>(Y + (mb - ybase));
        bool al = (((uintptr_t)o) & 15) == 0;
        if (al) {
#pragma unroll
            for (int r = 0; r < kMfR; r += 2)
                o[r / 2] = make_float4(out[r].x, out[r].y, out[r + 1].x, out[r + 1].y);
        } else {
#pragma unroll
            for (int r = 0; r < kMfR; r++) Y[mb + r - ybase] = out[r];
        }
    } else {
#pragma unroll
        for (int r = 0; r < kMfR; r++)
            if (mb + r < f_k) Y[mb + r - ybase] = out[r];
    }
}

cudaError_t launch_kk_mf(const float2 *E, long long ebase, long long e_k, long long f_prev,
                         long long f_k, const float *rrc, int hmf, const float2 *ds_tab,
                         int ds_num, int ds_den, const double *cg, float2 *Y, long long ybase,
                         const float2 *Y_prev, long long ybase_prev, cudaStream_t st,
                         const float *rrc_host, bool pdl)
{
    long long n = f_k - f_prev;
    if (hmf == 32 && rrc_host) {
        MfTaps<32> t;
        auto twice = [](float h) {
            uint32_t b;
            memcpy(&b, &h, 4);
            return (f2x)b << 32 | b;
        };
        for (int u = 0; u <= 32; u++) t.ge[u] = twice(rrc_host[32 + (32 - 2 * u)]);
        for (int u = 0; u < 32; u++) t.go[u] = twice(rrc_host[32 + (32 - 2 * u - 1)]);
        unsigned grid = (unsigned)((n + kMfTileOut - 1) / kMfTileOut);
        size_t smem = (size_t)pad8(kMfTileOut + 32 + kMfR) * sizeof(float4) + 16;
        const long long n0 = 2 * f_prev - hmf, r0 = (n0 % ds_den + ds_den) % ds_den;
        const unsigned ph0 = (unsigned)(r0 * ds_num % ds_den);   // downshift phase of the call's first input
        const long long period = ds_den / std::gcd(2LL * ds_num % ds_den, (long long)ds_den);   // in pairs
        return launch_k(120 % period == 0 ? k_kk_mf_t<32, 120, true> : k_kk_mf_t<32, kMfThreads, false>, grid, kMfThreads,
                        smem, st, pdl, E, ebase, e_k, f_prev, f_k, t, ds_tab, ds_num, ds_den, ph0, cg, Y, ybase, Y_prev,
                        ybase_prev);
    }
    unsigned grid = (unsigned)((n + kMfOut - 1) / kMfOut);
    size_t smem = (size_t)(2 * kMfOut + 2 * hmf) * sizeof(float2);
    return launch_k(k_kk_mf, grid, kMfOut, smem, st, pdl, E, ebase, e_k, f_prev, f_k, rrc, hmf, ds_tab, ds_num, ds_den, cg, Y,
                    ybase, Y_prev, ybase_prev);
}

// ================================================ resampler to the transmitter's grid
// The ADC runs on its own clock (Sec. 2: the DSP recovers the clock phase).  Nominal
// sample m of the transmitter's grid lies at ADC position psi_m / 2^32 with the exact
// integer accumulator psi_m = psi_{m0} + (m - m0) step; its field is the 16-tap
// Hann-windowed sinc interpolation sum_{j=-7..8} c_j(mu) E[i + j] of the
// reconstructed field at i = floor(psi / 2^32) and the fraction mu rounded down to
// 10 bits (a 1024 x 16 table).  The host splits psi_{m0} (m0 = this call's first
// output) into its integer part i0 and fraction f0, so every offset inside a call
// fits in 64 bits.  One CTA per kRsOut outputs stages their ADC window in shared
// memory first.
constexpr int kRsThreads = 256, kRsPer = 4, kRsOut = kRsThreads * kRsPer, kRsWin = kRsOut + kRsOut / 64 + 24;

__global__ void __launch_bounds__(kRsThreads) k_kk_resample(const float2 *__restrict__ E, long long ebase,
                                                       long long r_prev, long long r_k, long long i0,
                                                       unsigned f0, long long step, const float *__restrict__ tab,
                                                       float2 *__restrict__ R, long long rbase,
                                                       const float2 *__restrict__ R_prev, long long rbase_prev)
{
    __shared__ float2 xs[kRsWin];
    const long long m0 = r_prev + (long long)blockIdx.x * kRsOut;
    // the CTA's first output in integer part and fraction; with step = 2^32 + delta
    // (|delta| < 2^32 / 64) thread t sits at i_b + t + floor((f_b + t delta) / 2^32)
    const long long accb = (long long)f0 + (m0 - r_prev) * step;
    const long long i_b = i0 + (accb >> 32);
    const long long f_b = accb & 0xFFFFFFFFLL;
    const int delta = (int)(step - (1LL << 32));
    const int nout = (int)min((long long)kRsOut, r_k - m0);
    const long long a0 = i_b - 7;
    const int len = (nout - 1) + (int)((f_b + (long long)(nout - 1) * delta) >> 32) + 16;
    for (int t = threadIdx.x; t < len && t < kRsWin; t += blockDim.x) {
        const long long n = a0 + t;
        xs[t] = n < 0 ? make_float2(0.f, 0.f) : E[n - ebase];
    }
    if (blockIdx.x == 0)   // the filter's history on the nominal grid
        for (long long m = rbase + threadIdx.x; m < r_prev; m += blockDim.x)
            R[m - rbase] = (m < 0) ? make_float2(0.f, 0.f) : R_prev[m - rbase_prev];
    __syncthreads();
#pragma unroll
    for (int k = 0; k < kRsPer; k++) {   // outputs t, t + 256, ...: coalesced stores
        const int t = threadIdx.x + kRsThreads * k;
        if (t >= nout) return;
        const long long v = f_b + (long long)t * delta;   // |v| < 2^39
        const int li = t + (int)(v >> 32);                  // local index of E[i - 7]
        const float4 *c4 = reinterpret_cast<const float4 *>(tab + ((unsigned)(v & 0xFFFFFFFFLL) >> 22) * 16);
        float cj[16];
#pragma unroll
        for (int q = 0; q < 4; q++) {   // the 64-byte row in four 16-byte loads
            const float4 w = __ldg(c4 + q);
            cj[4 * q] = w.x;
            cj[4 * q + 1] = w.y;
            cj[4 * q + 2] = w.z;
            cj[4 * q + 3] = w.w;
        }
        float re = 0.f, im = 0.f;
#pragma unroll
        for (int j = 0; j < 16; j++) {
            const float2 x = xs[li + j];
            re = fmaf(cj[j], x.x, re);
            im = fmaf(cj[j], x.y, im);
        }
        R[m0 + t - rbase] = make_float2(re, im);
    }
}

cudaError_t launch_kk_resample(const float2 *E, long long ebase, long long r_prev, long long r_k, long long i0,
                               unsigned f0, long long step, const float *tab, float2 *R, long long rbase,
                               const float2 *R_prev, long long rbase_prev, cudaStream_t st)
{
    // the window of kRsOut outputs spans at most kRsOut step / 2^32 + 17 ADC samples
    if (step < (1LL << 32) - (1LL << 32) / 64 || step > (1LL << 32) + (1LL << 32) / 64) return cudaErrorInvalidValue;
    const long long n = r_k - r_prev;
    if (n <= 0) return cudaSuccess;
    k_kk_resample<<<(unsigned)((n + kRsOut - 1) / kRsOut), kRsThreads, 0, st>>>(E, ebase, r_prev, r_k, i0, f0, step, tab,
                                                                           R, rbase, R_prev, rbase_prev);
    return cudaGetLastError();
}

// ============================================ frequency-domain reduction (KK)
// The paper's form of the filter before the equaliser (Sec. 2, KK chain): a
// static filter applied in the frequency domain on overlap-save blocks of N =
// fd_n samples with hop N/2, and an N/2-point inverse transform of the kept bins
// -N/4 <= k < N/4 as the downsampler to 2 samples/symbol.  One CTA per block b:
//   - the N inputs from stream index N/2 b - N/4 (carrier removed, downshifted by
//     the exact integer phase; zero before the stream start) are staged in
//     shared memory;
//   - a radix-4 Stockham FFT (natural order in and out, two ping-pong buffers,
//     a last radix-2 pass when log2 N is odd) transforms them;
//   - the kept bins times the filter response (pre-scaled by 1/N) form the
//     N/2-point spectrum, which the inverse Stockham FFT brings back;
//   - the central half, N/4 outputs, leaves at 2 samples/symbol times the gain.
constexpr int kFdThreads = 128;

// Stockham passes of an n-point transform (n = N or N/2) on shared buffers a, b;
// tw is the N-point table e^{-2 pi i t / N}; returns the buffer with the result
template <bool INV>
__device__ float2 *stockham(float2 *a, float2 *b, int n, int N, const float2 *__restrict__ tw)
{
    int ns = 1;
    for (; ns * 4 <= n; ns *= 4) {
        const int q4 = n >> 2, ts = N / (4 * ns);
        for (int j = threadIdx.x; j < q4; j += blockDim.x) {
            const int k = j & (ns - 1);
            float2 v0 = a[j], v1 = a[j + q4], v2 = a[j + 2 * q4], v3 = a[j + 3 * q4];
            if (ns > 1) {
                float2 w1 = __ldg(tw + k * ts), w2 = __ldg(tw + 2 * k * ts), w3 = __ldg(tw + 3 * k * ts);
                if (INV) {
                    w1 = cconj(w1);
                    w2 = cconj(w2);
                    w3 = cconj(w3);
                }
                v1 = cmul(v1, w1);
                v2 = cmul(v2, w2);
                v3 = cmul(v3, w3);
            }
            dft4<INV>(v0, v1, v2, v3);
            const int o = ((j - k) << 2) + k;
            b[o] = v0;
            b[o + ns] = v1;
            b[o + 2 * ns] = v2;
            b[o + 3 * ns] = v3;
        }
        __syncthreads();
        float2 *t = a;
        a = b;
        b = t;
    }
    if (ns < n) {   // one radix-2 pass
        const int h2 = n >> 1, ts = N / (2 * ns);
        for (int j = threadIdx.x; j < h2; j += blockDim.x) {
            const int k = j & (ns - 1);
            float2 w = __ldg(tw + k * ts);
            if (INV) w = cconj(w);
            const float2 v0 = a[j], v1 = cmul(a[j + h2], w);
            const int o = ((j - k) << 1) + k;
            b[o] = cadd(v0, v1);
            b[o + ns] = csub(v0, v1);
        }
        __syncthreads();
        a = b;
    }
    return a;
}

__global__ void __launch_bounds__(kFdThreads) k_kk_fdmf(const float2 *E, long long ebase,
                                                       long long b_first, int N, const float2 *__restrict__ H,
                                                       const float2 *__restrict__ tw,
                                                       const float2 *__restrict__ ds_tab, int ds_num, int ds_den,
                                                       const double *cg, float2 *Y,
                                                       long long ybase, long long f_prev,
                                                       const float2 *Y_prev, long long ybase_prev,
                                                       float2 *clk, int wbin)
{
    extern __shared__ float2 fbuf[];   // [2][N]
    float2 *a = fbuf, *b = fbuf + N;
    pdl_wait();
    const long long blk = b_first + blockIdx.x;
    const long long n0 = (N / 2) * blk - N / 4;   // stream index of the block's first input
    const float2 c = make_float2((float)cg[0], (float)cg[1]);
    const float gn = (float)cg[2];
    // integer phase index of the downshift: p(n) = n ds_num mod ds_den, advanced by the thread stride
    long long r0 = (n0 + threadIdx.x) % ds_den;
    if (r0 < 0) r0 += ds_den;
    int p = (int)((r0 * ds_num) % ds_den);
    const int step = (int)(((long long)kFdThreads * ds_num) % ds_den);
    for (int t = threadIdx.x; t < N; t += kFdThreads) {
        const long long n = n0 + t;
        a[t] = n < 0 ? make_float2(0.f, 0.f) : cmul(csub(E[n - ebase], c), __ldg(ds_tab + p));
        p += step;
        p = p >= ds_den ? p - ds_den : p;
    }
    if (blockIdx.x == 0)
        for (long long m = ybase + threadIdx.x; m < f_prev; m += kFdThreads)
            Y[m - ybase] = (m < 0) ? make_float2(0.f, 0.f) : Y_prev[m - ybase_prev];
    __syncthreads();
    float2 *X = stockham<false>(a, b, N, N, tw);
    float2 *Z = X == a ? b : a;
    const int half = N >> 1, q = N >> 2;
    for (int kp = threadIdx.x; kp < half; kp += kFdThreads) Z[kp] = cmul(X[kp < q ? kp : kp + half], __ldg(H + kp));
    __syncthreads();
    if (clk && threadIdx.x < 32) {   // band-edge clock correlation: Y_k conj(Y_{k - N/4}), |k - N/8| <= w
        float2 acc = make_float2(0.f, 0.f);
        for (int k = N / 8 - wbin + (int)threadIdx.x; k <= N / 8 + wbin; k += 32) {
            const float2 a = Z[k], b = Z[k + q];   // kept positions k and (k - N/4) mod N - N/2
            acc = cadd(acc, cmulc(a, b));
        }
#pragma unroll
        for (int o = 16; o; o >>= 1)
            acc = make_float2(acc.x + __shfl_xor_sync(0xffffffffu, acc.x, o), acc.y + __shfl_xor_sync(0xffffffffu, acc.y, o));
        if (threadIdx.x == 0) clk[blockIdx.x] = acc;
    }
    float2 *z = stockham<true>(Z, X, half, N, tw);
    const long long s0 = (long long)(N / 4) * blk - ybase;   // 2-sps index of the block's first output
    for (int m = threadIdx.x; m < q; m += kFdThreads) Y[s0 + m] = cscale(z[m + N / 8], gn);
}

// W32^k = e^{-2 pi i k / 32} for k = 0..15 (cos and sin of pi k / 16)
__device__ __forceinline__ float2 w32(int k)
{
    switch (k) {
    case 0: return make_float2(1.f, 0.f);
    case 1: return make_float2(0.98078528040323043f, -0.19509032201612825f);
    case 2: return make_float2(0.92387953251128674f, -0.38268343236508978f);
    case 3: return make_float2(0.83146961230254524f, -0.55557023301960218f);
    case 4: return make_float2(0.70710678118654752f, -0.70710678118654752f);
    case 5: return make_float2(0.55557023301960218f, -0.83146961230254524f);
    case 6: return make_float2(0.38268343236508978f, -0.92387953251128674f);
    case 7: return make_float2(0.19509032201612825f, -0.98078528040323043f);
    case 8: return make_float2(0.f, -1.f);
    case 9: return make_float2(-0.19509032201612825f, -0.98078528040323043f);
    case 10: return make_float2(-0.38268343236508978f, -0.92387953251128674f);
    case 11: return make_float2(-0.55557023301960218f, -0.83146961230254524f);
    case 12: return make_float2(-0.70710678118654752f, -0.70710678118654752f);
    case 13: return make_float2(-0.83146961230254524f, -0.55557023301960218f);
    case 14: return make_float2(-0.92387953251128674f, -0.38268343236508978f);
    default: return make_float2(-0.98078528040323043f, -0.19509032201612825f);   // k = 15
    }
}

// 32-point DFT in registers, natural order in and out, unscaled: two 16-point
// DFTs over the even and odd samples and one radix-2 combination
template <bool INV>
__device__ __forceinline__ void dft32(float2 (&x)[32])
{
    float2 e[16], o[16];
#pragma unroll
    for (int i = 0; i < 16; i++) {
        e[i] = x[2 * i];
        o[i] = x[2 * i + 1];
    }
    dft16<INV>(e);
    dft16<INV>(o);
#pragma unroll
    for (int k = 0; k < 16; k++) {
        float2 w = w32(k);
        if (INV) w.y = -w.y;
        const float2 t = cmul(o[k], w);
        x[k] = cadd(e[k], t);
        x[k + 16] = csub(e[k], t);
    }
}

// The 1024-point form, one warp per block, as a 32 x 32 four-step transform with
// n = lane + 32 q and k = k2 + 32 k1:
//   forward: 32-point DFTs over q in registers, twiddle W1024^(lane k2), a padded
//     shared-memory transpose, 32-point DFTs over the former lane index: lane k2
//     then holds the bins k2 + 32 k1;
//   the kept bins (k1 < 8 or k1 >= 24) times the response give the 512-point
//     spectrum at k' = lane + 32 j (j = k1, or k1 - 16);
//   inverse with m = m_a + 16 m_b: 16-point inverse DFTs over j in registers,
//     twiddle e^{+2 pi i lane m_a / 512}, a transpose, then per m_a the inverse
//     32-point DFT over the lanes split between a lane pair (even / odd lanes,
//     16 points each, halves exchanged by shuffles), evaluated only at the kept
//     outputs m_b = 8 .. 23 (m = 128 .. 383).
constexpr int kFdWarps = 4, kFdPitch = 33;

__global__ void __launch_bounds__(32 * kFdWarps, 4)
    k_kk_fd1024(const float2 *E, long long ebase, long long b_first, long long nblk,
                const float2 *__restrict__ H, const float2 *__restrict__ tw, const float2 *__restrict__ ds_tab,
                int ds_num, int ds_den, const double *cg, float2 *Y, long long ybase,
                long long f_prev, const float2 *Y_prev, long long ybase_prev,
                float2 *clk, int wbin)
{
    __shared__ float2 s_tw[1024];
    __shared__ float2 s_t[kFdWarps][32 * kFdPitch];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    for (int i = threadIdx.x; i < 1024; i += blockDim.x) s_tw[i] = tw[i];
    pdl_wait();
    if (blockIdx.x == 0)
        for (long long m = ybase + threadIdx.x; m < f_prev; m += blockDim.x)
            Y[m - ybase] = (m < 0) ? make_float2(0.f, 0.f) : Y_prev[m - ybase_prev];
    __syncthreads();
    const long long bi = (long long)blockIdx.x * kFdWarps + w;
    if (bi >= nblk) return;
    const long long blk = b_first + bi, n0 = 512 * blk - 256;
    const float2 c = make_float2((float)cg[0], (float)cg[1]);
    const float gn = (float)cg[2];
    long long r0 = (n0 + lane) % ds_den;
    if (r0 < 0) r0 += ds_den;
    int p = (int)((r0 * ds_num) % ds_den);
    const int step = (int)((32LL * ds_num) % ds_den);
    float2 x[32];
#pragma unroll
    for (int q = 0; q < 32; q++) {
        const long long n = n0 + lane + 32 * q;
        x[q] = n < 0 ? make_float2(0.f, 0.f) : cmul(csub(E[n - ebase], c), __ldg(ds_tab + p));
        p += step;
        p = p >= ds_den ? p - ds_den : p;
    }
    dft32<false>(x);
#pragma unroll
    for (int k2 = 1; k2 < 32; k2++) x[k2] = cmul(x[k2], s_tw[lane * k2]);
    float2 *T = s_t[w];
#pragma unroll
    for (int k2 = 0; k2 < 32; k2++) T[lane * kFdPitch + k2] = x[k2];
    __syncwarp();
#pragma unroll
    for (int n1 = 0; n1 < 32; n1++) x[n1] = T[n1 * kFdPitch + lane];
    __syncwarp();
    dft32<false>(x);
    float2 z[16];
#pragma unroll
    for (int j = 0; j < 16; j++) z[j] = cmul(x[j < 8 ? j : j + 16], __ldg(H + lane + 32 * j));
    if (clk) {   // band-edge clock correlation: bins k = lane + 32 k1 (k1 = 3, 4) with k - 256 (k1 + 24 -> j + 8)
        float2 acc = make_float2(0.f, 0.f);
#pragma unroll
        for (int k1 = 3; k1 <= 4; k1++) {
            const int k = lane + 32 * k1;
            if (k >= 128 - wbin && k <= 128 + wbin) acc = cadd(acc, cmulc(z[k1], z[k1 + 8]));
        }
#pragma unroll
        for (int o = 16; o; o >>= 1)
            acc = make_float2(acc.x + __shfl_xor_sync(0xffffffffu, acc.x, o), acc.y + __shfl_xor_sync(0xffffffffu, acc.y, o));
        if (lane == 0) clk[bi] = acc;
    }
    dft16<true>(z);
#pragma unroll
    for (int ma = 1; ma < 16; ma++) z[ma] = cmulc(z[ma], s_tw[2 * lane * ma]);
#pragma unroll
    for (int ma = 0; ma < 16; ma++) T[lane * 17 + ma] = z[ma];
    __syncwarp();
    const int ma = lane >> 1, h = lane & 1;
#pragma unroll
    for (int i = 0; i < 16; i++) z[i] = T[(2 * i + h) * 17 + ma];
    dft16<true>(z);   // h = 0: even-lane half E[r]; h = 1: odd-lane half O[r]
    const long long s0 = 256 * blk - ybase;
#pragma unroll
    for (int i = 0; i < 8; i++) {
        // lane h = 0 emits m_b = 8 + i (r = 8 + i), lane h = 1 emits m_b = 16 + i (r = i)
        const float2 send = h ? z[8 + i] : z[i];
        const float2 other = make_float2(__shfl_xor_sync(0xffffffffu, send.x, 1),
                                         __shfl_xor_sync(0xffffffffu, send.y, 1));
        const float2 Ev = h ? other : z[8 + i], Ov = h ? z[i] : other;
        float2 wv = h ? w32(i) : w32(8 + i);   // e^{+2 pi i m_b / 32} = conj(W32^r), negated for m_b >= 16
        wv.y = -wv.y;
        if (h) wv = make_float2(-wv.x, -wv.y);
        Y[s0 + ma + 16 * (8 * h + i)] = cscale(cadd(Ev, cmul(wv, Ov)), gn);
    }
}

cudaError_t launch_kk_fdmf(const float2 *E, long long ebase, long long f_prev, long long f_k, int N,
                           const float2 *H, const float2 *tw, const float2 *ds_tab, int ds_num, int ds_den,
                           const double *cg, float2 *Y, long long ybase, const float2 *Y_prev,
                           long long ybase_prev, cudaStream_t st, float2 *clk, int wbin, bool pdl)
{
    const int per = N / 4;   // outputs per block
    if (N < 16 || (N & (N - 1)) || f_prev % per || f_k % per || wbin < 0 || wbin >= N / 8 || (N == 1024 && wbin > 31))
        return cudaErrorInvalidValue;
    const long long nblk = (f_k - f_prev) / per;
    if (nblk <= 0) return cudaSuccess;
    if (N == 1024) {
        return launch_k(k_kk_fd1024, (unsigned)((nblk + kFdWarps - 1) / kFdWarps), 32 * kFdWarps, 0, st, pdl, E, ebase,
                        f_prev / per, nblk, H, tw, ds_tab, ds_num, ds_den, cg, Y, ybase, f_prev, Y_prev, ybase_prev, clk,
                        wbin);
    }
    return launch_k(k_kk_fdmf, (unsigned)nblk, kFdThreads, 2 * N * sizeof(float2), st, pdl, E, ebase, f_prev / per, N, H, tw,
                    ds_tab, ds_num, ds_den, cg, Y, ybase, f_prev, Y_prev, ybase_prev, clk, wbin);
}

// =========================================================== PAM matched filter
// x[n] = (code[n] - mu) / sd with the buffer's exact integer moments, x[n < 0] = 0;
// y[m] = sum_i h_i x[m - i] at 2 samples/symbol.

// first CTA of a filter: the equaliser's history [ybase, f_prev), and the debug view of the
// call's mean and deviation
__device__ __forceinline__ void pam_carry(DevState *dst, int slot, float *Y, long long ybase, long long f_prev,
                                          const float *Y_prev, long long ybase_prev)
{
    for (long long m = ybase + threadIdx.x; m < f_prev; m += blockDim.x)
        Y[m - ybase] = (m < 0) ? 0.f : Y_prev[m - ybase_prev];
    if (threadIdx.x == 0) {
        dst->pam_mu = dst->pam_nd[slot][0];
        dst->pam_inv_sd = dst->pam_nd[slot][1];
    }
}

__global__ void __launch_bounds__(kMfOut) k_pam_mf(const uint16_t *codes, long long cbase,
                                                  long long n_end, long long f_prev, long long f_k,
                                                  const float *__restrict__ rrc, int hmf, DevState *dst,
                                                  int slot, float *Y, long long ybase,
                                                  const float *Y_prev, long long ybase_prev)
{
    extern __shared__ float xf[];
    pdl_wait_late();
    const float s_mu = dst->pam_nf[slot][0], s_inv = dst->pam_nf[slot][1];
    long long m0 = f_prev + (long long)blockIdx.x * kMfOut;
    int L = kMfOut + 2 * hmf;
    long long n0 = m0 - hmf;
    for (int i = threadIdx.x; i < L; i += blockDim.x) {
        long long n = n0 + i;
        float v = 0.f;
        if (n >= 0 && n < n_end) v = ((float)codes[n - cbase] - s_mu) * s_inv;
        xf[i] = v;
    }
    if (blockIdx.x == 0) pam_carry(dst, slot, Y, ybase, f_prev, Y_prev, ybase_prev);
    __syncthreads();
    long long m = m0 + threadIdx.x;
    if (m >= f_k) return;
    const float *xc = xf + threadIdx.x + hmf;
    float a = 0.f;
    for (int i = -hmf; i <= hmf; i++) a = fmaf(__ldg(rrc + i + hmf), xc[-i], a);
    Y[m - ybase] = a;
    pdl_release();
}

// ========================================== PAM resampler path (ADC off the transmitter's clock)
// The normalised code x[n] = (code - mu) / sd of the call (complex, imaginary part 0)
// for stream samples [cbase, n_end), the input of the resampler (which treats
// samples before the stream as zero); the call's mean and deviation come from the
// exact integer sums.
__global__ void k_pam_norm(const uint16_t *__restrict__ codes, long long cbase, long long n_end, DevState *dst, int slot,
                           float2 *__restrict__ X)
{
    const float mu = dst->pam_nf[slot][0], inv = dst->pam_nf[slot][1];
    const long long n = cbase + (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (n < n_end) X[n - cbase] = make_float2(((float)codes[n - cbase] - mu) * inv, 0.f);
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        dst->pam_mu = (double)mu;
        dst->pam_inv_sd = (double)inv;
    }
}

// the PAM matched filter (2 samples/symbol, no decimation) on the resampled series
// (real parts of R, stream index m at R[m - rbase]; zero before the stream)
__global__ void __launch_bounds__(kMfOut) k_pam_mf_r(const float2 *__restrict__ R, long long rbase, long long f_prev,
                                                    long long f_k, const float *__restrict__ rrc, int hmf,
                                                    float *__restrict__ Y, long long ybase,
                                                    const float *__restrict__ Y_prev, long long ybase_prev)
{
    extern __shared__ float xf[];
    long long m0 = f_prev + (long long)blockIdx.x * kMfOut;
    int L = kMfOut + 2 * hmf;
    long long n0 = m0 - hmf;
    for (int i = threadIdx.x; i < L; i += blockDim.x) {
        long long n = n0 + i;
        xf[i] = n < 0 ? 0.f : R[n - rbase].x;
    }
    if (blockIdx.x == 0)
        for (long long m = ybase + threadIdx.x; m < f_prev; m += blockDim.x)
            Y[m - ybase] = (m < 0) ? 0.f : Y_prev[m - ybase_prev];
    __syncthreads();
    long long m = m0 + threadIdx.x;
    if (m >= f_k) return;
    const float *xc = xf + threadIdx.x + hmf;
    float a = 0.f;
    for (int i = -hmf; i <= hmf; i++) a = fmaf(__ldg(rrc + i + hmf), xc[-i], a);
    Y[m - ybase] = a;
}

cudaError_t launch_pam_norm(const uint16_t *codes, long long cbase, long long n_end, DevState *dst, int slot, float2 *X,
                            cudaStream_t st)
{
    const long long n = n_end - cbase;
    k_pam_norm<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(codes, cbase, n_end, dst, slot, X);
    return cudaGetLastError();
}

cudaError_t launch_pam_mf_r(const float2 *R, long long rbase, long long f_prev, long long f_k, const float *rrc, int hmf,
                            float *Y, long long ybase, const float *Y_prev, long long ybase_prev, cudaStream_t st)
{
    long long n = f_k - f_prev;
    unsigned grid = (unsigned)((n + kMfOut - 1) / kMfOut);
    size_t smem = (size_t)(kMfOut + 2 * hmf) * sizeof(float);
    k_pam_mf_r<<<grid, kMfOut, smem, st>>>(R, rbase, f_prev, f_k, rrc, hmf, Y, ybase, Y_prev, ybase_prev);
    return cudaGetLastError();
}

// ===================================================== PAM frequency-domain filter
// The paper's PAM form (Sec. 2): a static filter applied on 1024-point
// overlap-save blocks (hop 512) at the input rate.  One warp per block: the
// normalised codes x[n] = (code - mu) / sd of the N inputs from 512 b - 256 go
// through the same 32 x 32 four-step forward transform as the KK form (lane k2
// holds the bins k2 + 32 k1), every bin is multiplied by the response (times
// 1/N), and the 1024-point inverse runs as a second four-step with m = m_a + 32
// m_b: 32-point inverse DFTs over k1 in registers, twiddle e^{+2 pi i lane m_a /
// 1024}, a transpose, 32-point inverse DFTs over the former lane index; lane m_a
// keeps m_b = 8 .. 23 (m = 256 .. 767), whose real part is y.
__global__ void __launch_bounds__(32 * kFdWarps, 4)
    k_pam_fd1024(const uint16_t *codes, long long cbase, long long n_end,
                 long long b_first, long long nblk, const float2 *__restrict__ H, const float2 *__restrict__ tw,
                 DevState *dst, int slot, float *Y, long long ybase, long long f_prev,
                 const float *Y_prev, long long ybase_prev, float2 *clk, int wbin)
{
    __shared__ float2 s_tw[1024];
    __shared__ float2 s_t[kFdWarps][32 * kFdPitch];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    for (int i = threadIdx.x; i < 1024; i += blockDim.x) s_tw[i] = tw[i];
    pdl_wait_late();
    __syncthreads();
    if (blockIdx.x == 0) pam_carry(dst, slot, Y, ybase, f_prev, Y_prev, ybase_prev);
    const long long bi = (long long)blockIdx.x * kFdWarps + w;
    if (bi >= nblk) return;
    const long long blk = b_first + bi, n0 = 512 * blk - 256;
    const float mu = dst->pam_nf[slot][0], inv = dst->pam_nf[slot][1];
    float2 x[32];
#pragma unroll
    for (int q = 0; q < 32; q++) {
        const long long n = n0 + lane + 32 * q;
        x[q] = make_float2(n >= 0 && n < n_end ? ((float)codes[n - cbase] - mu) * inv : 0.f, 0.f);
    }
    dft32<false>(x);
#pragma unroll
    for (int k2 = 1; k2 < 32; k2++) x[k2] = cmul(x[k2], s_tw[lane * k2]);
    float2 *T = s_t[w];
#pragma unroll
    for (int k2 = 0; k2 < 32; k2++) T[lane * kFdPitch + k2] = x[k2];
    __syncwarp();
#pragma unroll
    for (int n1 = 0; n1 < 32; n1++) x[n1] = T[n1 * kFdPitch + lane];
    __syncwarp();
    dft32<false>(x);   // x[k1] = X[lane + 32 k1]
#pragma unroll
    for (int k1 = 0; k1 < 32; k1++) x[k1] = cmul(x[k1], __ldg(H + lane + 32 * k1));
    if (clk) {   // band-edge clock correlation at 2 samples/symbol: bins k = lane + 32 k1 (k1 = 7, 8)
                 // around N/4 with k - N/2 (k1 + 16)
        float2 acc = make_float2(0.f, 0.f);
#pragma unroll
        for (int k1 = 7; k1 <= 8; k1++) {
            const int k = lane + 32 * k1;
            if (k >= 256 - wbin && k <= 256 + wbin) acc = cadd(acc, cmulc(x[k1], x[k1 + 16]));
        }
#pragma unroll
        for (int o = 16; o; o >>= 1)
            acc = make_float2(acc.x + __shfl_xor_sync(0xffffffffu, acc.x, o), acc.y + __shfl_xor_sync(0xffffffffu, acc.y, o));
        if (lane == 0) clk[bi] = acc;
    }
    dft32<true>(x);    // over k1 -> m_a
#pragma unroll
    for (int ma = 1; ma < 32; ma++) x[ma] = cmulc(x[ma], s_tw[lane * ma]);
#pragma unroll
    for (int ma = 0; ma < 32; ma++) T[lane * kFdPitch + ma] = x[ma];
    __syncwarp();
#pragma unroll
    for (int l = 0; l < 32; l++) x[l] = T[l * kFdPitch + lane];
    dft32<true>(x);    // lane m_a: x[m_b] = z[m_a + 32 m_b]
    const long long s0 = 512 * blk - ybase;
#pragma unroll
    for (int mb = 8; mb < 24; mb++) Y[s0 + lane + 32 * (mb - 8)] = x[mb].x;
    pdl_release();
}

cudaError_t launch_pam_fd1024(const uint16_t *codes, long long cbase, long long n_end,
                              long long f_prev, long long f_k, const float2 *H, const float2 *tw, DevState *dst,
                              int slot, float *Y, long long ybase, const float *Y_prev, long long ybase_prev,
                              cudaStream_t st, float2 *clk, int wbin, bool pdl)
{
    if (f_prev % 512 || f_k % 512 || wbin < 0 || wbin > 31) return cudaErrorInvalidValue;
    const long long nblk = (f_k - f_prev) / 512;
    if (nblk <= 0) return cudaSuccess;
    return launch_k(k_pam_fd1024, (unsigned)((nblk + kFdWarps - 1) / kFdWarps), 32 * kFdWarps, 0, st, pdl, codes, cbase,
                    n_end, f_prev / 512, nblk, H, tw, dst, slot, Y, ybase, f_prev, Y_prev, ybase_prev, clk, wbin);
}

// Register-tiled PAM matched filter for a compile-time half length HMF (a multiple of 4):
// each thread computes kPmR consecutive outputs from a window of kPmR + 2 HMF inputs held in
// registers, read from shared memory in 16-byte pieces; four spare floats per 32 keep the
// stride-8 reads (and the staging stores) free of most bank conflicts.  The codes are loaded
// eight at a time, the taps are kernel parameters (constant operands of the FMAs).  Per
// output the products are accumulated in the same order as k_pam_mf (tap index ascending),
// so the outputs are the same bit for bit.  Bound by latency (one tile per CTA, 264 FMAs a
// thread).  2^20 samples: 6.3 us; 12.7 us with a 4-byte conflicting load per tap, 2-byte
// code loads and the FP64 mean and deviation formed in every CTA.
constexpr int kPmThreads = 128, kPmR = 8, kPmTile = kPmThreads * kPmR;
__host__ __device__ __forceinline__ constexpr int pad32(int i) { return i + ((i >> 5) << 2); }
template <int HMF>
struct PmTaps {
    float h[2 * HMF + 1];
};

template <int HMF>
__global__ void __launch_bounds__(kPmThreads)
    k_pam_mf_t(const uint16_t *codes, long long cbase, long long n_end, long long f_prev, long long f_k,
               const __grid_constant__ PmTaps<HMF> taps, DevState *dst, int slot, float *Y, long long ybase,
               const float *Y_prev, long long ybase_prev)
{
    constexpr int L = kPmTile + 2 * HMF, NW = kPmR + 2 * HMF;
    static_assert(HMF % 4 == 0 && L % 8 == 0 && kPmR == 8, "16-byte pieces");
    __shared__ __align__(16) float xf[pad32(L) + 4];
    pdl_wait_late();
    const float mu = dst->pam_nf[slot][0], inv = dst->pam_nf[slot][1];
    const long long m0 = f_prev + (long long)blockIdx.x * kPmTile, n0 = m0 - HMF;
    const uint16_t *ct = codes + (n0 - cbase);
    if (n0 >= 0 && n0 + L <= n_end && ((uintptr_t)ct & 15) == 0) {
#pragma unroll
        for (int k = 0; k < (L / 8 + kPmThreads - 1) / kPmThreads; k++) {
            const int c = threadIdx.x + k * kPmThreads;
            if (c >= L / 8) break;
            const uint4 v = reinterpret_cast<const uint4 *>(ct)[c];
            const uint32_t w[4] = {v.x, v.y, v.z, v.w};
            float x[8];
#pragma unroll
            for (int i = 0; i < 4; i++) {
                x[2 * i] = ((float)(w[i] & 0xFFFFu) - mu) * inv;
                x[2 * i + 1] = ((float)(w[i] >> 16) - mu) * inv;
            }
            float4 *d = reinterpret_cast<float4 *>(xf + pad32(8 * c));
            d[0] = make_float4(x[0], x[1], x[2], x[3]);
            d[1] = make_float4(x[4], x[5], x[6], x[7]);
        }
    } else {
        for (int i = threadIdx.x; i < L; i += kPmThreads) {
            const long long n = n0 + i;
            xf[pad32(i)] = (n >= 0 && n < n_end) ? ((float)ct[i] - mu) * inv : 0.f;
        }
    }
    if (blockIdx.x == 0) pam_carry(dst, slot, Y, ybase, f_prev, Y_prev, ybase_prev);
    __syncthreads();
    // output j = j0 + r: y = sum_{i=-HMF}^{HMF} h[i + HMF] xf[j + HMF - i], i ascending
    const int j0 = kPmR * threadIdx.x;
    float x[NW];
#pragma unroll
    for (int q = 0; q < NW / 4; q++) {
        const float4 v = *reinterpret_cast<const float4 *>(xf + pad32(j0 + 4 * q));
        x[4 * q] = v.x;
        x[4 * q + 1] = v.y;
        x[4 * q + 2] = v.z;
        x[4 * q + 3] = v.w;
    }
    float acc[kPmR];
#pragma unroll
    for (int r = 0; r < kPmR; r++) acc[r] = 0.f;
#pragma unroll
    for (int i = 0; i <= 2 * HMF; i++)
#pragma unroll
        for (int r = 0; r < kPmR; r++) acc[r] = fmaf(taps.h[i], x[2 * HMF - i + r], acc[r]);
    const long long mb = m0 + j0;
    float *Yo = Y + (mb - ybase);
    if (mb + kPmR <= f_k && ((uintptr_t)Yo & 15) == 0) {
        reinterpret_cast<float4 *>(Yo)[0] = make_float4(acc[0], acc[1], acc[2], acc[3]);
        reinterpret_cast<float4 *>(Yo)[1] = make_float4(acc[4], acc[5], acc[6], acc[7]);
    } else {
#pragma unroll
        for (int r = 0; r < kPmR; r++)
            if (mb + r < f_k) Yo[r] = acc[r];
    }
    pdl_release();
}

cudaError_t launch_pam_mf(const uint16_t *codes, long long cbase, long long n_end, long long f_prev,
                          long long f_k, const float *rrc, const float *rrc_host, int hmf, DevState *dst, int slot,
                          float *Y, long long ybase, const float *Y_prev, long long ybase_prev,
                          cudaStream_t st, bool pdl)
{
    long long n = f_k - f_prev;
    if (hmf == 16) {   // the default span (16 symbols at 2 samples/symbol)
        PmTaps<16> t;
        memcpy(t.h, rrc_host, sizeof t.h);
        unsigned grid = (unsigned)((n + kPmTile - 1) / kPmTile);
        return launch_k(k_pam_mf_t<16>, grid, kPmThreads, 0, st, pdl, codes, cbase, n_end, f_prev, f_k, t, dst, slot, Y, ybase,
                        Y_prev, ybase_prev);
    }
    unsigned grid = (unsigned)((n + kMfOut - 1) / kMfOut);
    size_t smem = (size_t)(kMfOut + 2 * hmf) * sizeof(float);
    return launch_k(k_pam_mf, grid, kMfOut, smem, st, pdl, codes, cbase, n_end, f_prev, f_k, rrc, hmf, dst, slot, Y, ybase,
                    Y_prev, ybase_prev);
}

// bin and clear every latency slot still holding a record (rx_stats)
__global__ void k_lat_flush(LatRecord *r)
{
    const int i = threadIdx.x;
    if (i < kLatSlots) {
        const unsigned long long t0 = r->slot[i].t0, t1 = r->slot[i].t1;
        r->slot[i].t0 = 0ull;
        r->slot[i].t1 = 0ull;
        lat_bin(r, t0, t1);
    }
}

cudaError_t launch_lat_flush(LatRecord *r, cudaStream_t st)
{
    k_lat_flush<<<1, kLatSlots, 0, st>>>(r);
    return cudaGetLastError();
}

}  // namespace rxk

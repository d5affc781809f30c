// Block-Toeplitz FIR on the fifth-generation tensor cores (tcgen05).
//
// The equaliser's filter z_k = sum_i conj(w_i) y[2k + TH - i] with taps that are
// fixed for a whole call (the frozen form) is one dense contraction: rows of 16
// consecutive symbols, each row a K = 2 (30 + NT) real slice (padded to 128) of
// the 2-sps sequence as stored (complex interleaved; consecutive rows overlap,
// a Hankel matrix), times a K x 32 real Toeplitz matrix of the taps (complex
// split to real: re / im output of each symbol).  Tiles of 128 rows (2048
// symbols) run through M = 128, N = 32 tcgen05.mma in BF16, FP16 or FP8-E4M3
// with FP32 accumulation in tensor memory.  Persistent CTAs, per tile:
//   - the threads load the tile's 4.1 k complex FP32 inputs into registers, coalesced and
//     once, convert them and store them into the K-major no-swizzle operand layout (core
//     matrices of 8 rows x 16 bytes); FP8 first takes a power-of-two scale per block of
//     rows_per_scale rows from the block's largest input;
//   - one thread issues the MMAs and commits them to an mbarrier, while the next tile's
//     loads are in flight;
//   - each warp reads its 32 accumulator lanes (tcgen05.ld 32x32b), rescales and stores
//     them.
// The taps' Toeplitz operand is built once per CTA.  Every wait is bounded: on
// time-out the kernel records RX_ETIMEOUT, waits (bounded) for its own MMAs, frees its
// tensor memory and returns.
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_fp8.h>

#include "rx_async.cuh"
#include "rx_internal.cuh"

namespace rxk {
namespace {

constexpr int kRowSyms = 16;                       // symbols per GEMM row
constexpr int kTileRows = 128;                     // M of one MMA
constexpr int kN = 2 * kRowSyms;                   // real outputs per row
constexpr uint32_t kTmemCols = 32;

template <int PREC> struct Fmt;
template <> struct Fmt<RX_FIR_BF16> {
    static constexpr uint32_t code = 1;   // kind::f16, BF16
};
template <> struct Fmt<RX_FIR_FP16> {
    static constexpr uint32_t code = 0;   // kind::f16, F16
};
// 8 consecutive K elements -> one 16-byte core-matrix row
template <int PREC>
__device__ __forceinline__ uint4 pack16(const float *v);
template <>
__device__ __forceinline__ uint4 pack16<RX_FIR_BF16>(const float *v)
{
    uint32_t w[4];
#pragma unroll
    for (int i = 0; i < 4; i++) {
        __nv_bfloat162 h = __floats2bfloat162_rn(v[2 * i], v[2 * i + 1]);
        w[i] = *reinterpret_cast<uint32_t *>(&h);
    }
    return make_uint4(w[0], w[1], w[2], w[3]);
}
template <>
__device__ __forceinline__ uint4 pack16<RX_FIR_FP16>(const float *v)
{
    uint32_t w[4];
#pragma unroll
    for (int i = 0; i < 4; i++) {
        __half2 h = __floats2half2_rn(v[2 * i], v[2 * i + 1]);
        w[i] = *reinterpret_cast<uint32_t *>(&h);
    }
    return make_uint4(w[0], w[1], w[2], w[3]);
}
// power-of-two scale that brings the largest magnitude m to at most 448 (E4M3 max)
__device__ __forceinline__ int fp8_exp(float m)
{
    if (!(m > 0.f)) return 0;
    int e;
    frexpf(448.f / m, &e);   // 448/m = f 2^e, f in [0.5, 1)
    return min(max(e - 1, -60), 60);
}

// FP8 form.  Output row r (symbols k = k_lo + 16 (r0 + r) + j, j < 16) reads the samples
// 32 r .. 32 r + 30 + NT - 1 of the tile, counted from stream sample 2 (k_lo + 16 r0) - TH:
// K elements 0..63 are block row r (32 samples), 64..127 the start of block row r + 1, zero
// from sample 30 + NT on.  A scale belongs to rows_per_scale consecutive rows and follows
// from the largest input any of them reads (the first samples of the next block's first row
// included), so the two halves of a row are stored apart: a sample is converted with its own
// block's scale into the first half of row r and with row r - 1's scale into the second half
// of that row; the two conversions differ at the first row of a block only.  Lanes hold
// consecutive samples of a block row: loads are coalesced, a row's maximum is one warp
// reduction of the magnitudes' bit patterns, and planes 16 bytes apart modulo 128 take the
// 2-byte stores without conflicts.  Every input is read once, into registers; the next
// tile's loads are in flight while this tile's MMAs and stores run.
// 777 x 1024 symbols, scale block 1024: 8.1 us a call; 28.7 us when each row gathered its 122
// K elements from a staged copy twice (once for the maxima) through a rotated read order.
// Three CTAs per SM: the tile's chain (maxima, scales, conversion, MMA, store) is latency
// bound.
constexpr int kT8Planes = 8;                         // 128 K elements, 16 per 16-byte core row
constexpr int kT8Plane = kTileRows * 16 + 16;        // plane pitch
constexpr int kT8BPlane = kN * 16;
constexpr int kT8OffB = kT8Planes * kT8Plane;
constexpr int kT8OffW = kT8OffB + kT8Planes * kT8BPlane;      // the taps (32 complex)
constexpr int kT8OffMax = kT8OffW + 32 * 8;                   // row maxima [129], halo maxima [129] (bit patterns)
constexpr int kT8OffExp = kT8OffMax + 2 * (kTileRows + 1) * 4;   // scale exponents [<= 128]
constexpr int kT8OffBar = (kT8OffExp + kTileRows * 4 + 7) & ~7;
constexpr int kT8Smem = kT8OffBar + 16;
constexpr int kT8Threads = 256, kT8Warps = kT8Threads / 32, kT8PerSm = 3;
constexpr int kT8Iter = (kTileRows + 1 + kT8Warps - 1) / kT8Warps;   // block rows per warp
static_assert(kT8Plane % 16 == 0 && kT8OffB % 16 == 0 && kT8OffW % 8 == 0, "16-byte aligned operands");
static_assert(kT8Smem <= 48 * 1024, "no shared-memory attribute needed");

// two scaled values as E4M3 (round to nearest even, saturating)
__device__ __forceinline__ uint16_t fp8_pair(float2 v, float s)
{
    return __nv_cvt_float2_to_fp8x2(make_float2(v.x * s, v.y * s), __NV_SATFINITE, __NV_E4M3);
}

__global__ void __launch_bounds__(kT8Threads, kT8PerSm)
    k_fir_tc8(const float2 *Y, long long ybase, long long k_lo, int nrows,
              const float2 *taps, int ntaps, int rows_per_scale, float2 *z, int *err)
{
    extern __shared__ __align__(1024) unsigned char sm[];
    unsigned char *sA = sm, *sB = sm + kT8OffB;
    float2 *s_w = reinterpret_cast<float2 *>(sm + kT8OffW);
    unsigned *s_max = reinterpret_cast<unsigned *>(sm + kT8OffMax), *s_halo = s_max + kTileRows + 1;
    int *s_exp = reinterpret_cast<int *>(sm + kT8OffExp);
    uint64_t *bar = reinterpret_cast<uint64_t *>(sm + kT8OffBar);
    uint32_t *tslot = reinterpret_cast<uint32_t *>(bar + 1);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, quarter = warp & 3, half = warp >> 2;
    const int th = (ntaps - 1) / 2, ns = 2 * kRowSyms - 2 + ntaps;   // complex inputs per row
    const int nhalo = ns - 32;                                       // of them in the next block row (may be <= 0)
    const int ntiles = (nrows + kTileRows - 1) / kTileRows, rshift = 31 - __clz(rows_per_scale);
    float2 v[kT8Iter];
    // lane = sample of block row warp + 8 i; zero outside what the rows read (with one tap, ns
    // is 31: no row reads sample 31, which then has no say in the scales either)
    auto load_tile = [&](int t) {
        const int r0 = t * kTileRows, n = lane < ns ? 32 * (min(kTileRows, nrows - r0) - 1) + ns : 0;
        const float2 *Yb = Y + (2 * (k_lo + (long long)r0 * kRowSyms) - th - ybase);
#pragma unroll
        for (int i = 0; i < kT8Iter; i++) {
            const int j = tid + i * kT8Threads;
            v[i] = j < n ? Yb[j] : make_float2(0.f, 0.f);
        }
    };
    int t = blockIdx.x;
    if (tid == 0) mbar_init(bar, 1);
    if (warp == 0) tmem_alloc(tslot, kTmemCols);
    pdl_wait();
    if (tid < 32) s_w[tid] = tid < ntaps ? taps[tid] : make_float2(0.f, 0.f);
    if (t < ntiles) load_tile(t);
    __syncthreads();   // the taps in shared memory
    // B: Toeplitz matrix of the taps, rows n = 2 j + c (c: re / im output of symbol j), K
    // index 2 s + d (d: re / im of input s); tap i = 2 j + 2 TH - s
    const float2 wl = s_w[lane];
    const int eB = fp8_exp(__uint_as_float(
        __reduce_max_sync(0xffffffffu, __float_as_uint(fmaxf(fmaxf(0.f, fabsf(wl.x)), fabsf(wl.y))))));
    const float sBv = ldexpf(1.f, eB);
    {
        const int n = tid % kN, pl = tid / kN, j = n >> 1, c = n & 1;
        uint16_t h[8];
#pragma unroll
        for (int q = 0; q < 8; q++) {
            const int s = 8 * pl + q, i = 2 * j + 2 * th - s;
            float2 a = make_float2(0.f, 0.f);
            if (s < ns && i >= 0 && i < ntaps) {
                const float2 w = s_w[i];
                // conj(w) y: re = a yr + b yi, im = a yi - b yr
                a = c == 0 ? w : make_float2(-w.y, w.x);
            }
            h[q] = fp8_pair(a, sBv);
        }
        *reinterpret_cast<uint4 *>(sB + pl * kT8BPlane + n * 16) =
            make_uint4(h[0] | (uint32_t)h[1] << 16, h[2] | (uint32_t)h[3] << 16, h[4] | (uint32_t)h[5] << 16,
                       h[6] | (uint32_t)h[7] << 16);
    }
    static_assert(kN * kT8Planes == kT8Threads, "one core row of B per thread");
    const uint32_t idesc = umma_idesc(0, kTileRows, kN);   // kind::f8f6f4, E4M3
    bool ok = true;
    for (int it = 0; t < ntiles; t += gridDim.x, it++) {
        const int r0 = t * kTileRows, rows = min(kTileRows, nrows - r0);
        // largest magnitude of each block row and, where it starts a scale block, of the
        // part of it that the last row of the block before reads
#pragma unroll
        for (int i = 0; i < kT8Iter; i++) {
            const int q = warp + kT8Warps * i;
            if (q > kTileRows) break;
            const unsigned m = __float_as_uint(fmaxf(fmaxf(0.f, fabsf(v[i].x)), fabsf(v[i].y)));
            const unsigned mr = __reduce_max_sync(0xffffffffu, m);
            if (lane == 0) s_max[q] = mr;
            if ((q & (rows_per_scale - 1)) == 0) {
                const unsigned mh = __reduce_max_sync(0xffffffffu, lane < nhalo ? m : 0u);
                if (lane == 0) s_halo[q] = mh;
            }
        }
        __syncthreads();
        for (int b = warp; b < (kTileRows >> rshift); b += kT8Warps) {
            unsigned m = lane == 0 ? s_halo[(b + 1) << rshift] : 0u;
            for (int r = lane; r < rows_per_scale; r += 32) m = max(m, s_max[(b << rshift) + r]);
            m = __reduce_max_sync(0xffffffffu, m);
            if (lane == 0) s_exp[b] = fp8_exp(__uint_as_float(m));
        }
        __syncthreads();
#pragma unroll
        for (int i = 0; i < kT8Iter; i++) {
            const int q = warp + kT8Warps * i;
            if (q > kTileRows) break;
            unsigned char *dst = sA + (lane >> 3) * kT8Plane + (lane & 7) * 2;
            const int e0 = q < kTileRows ? s_exp[q >> rshift] : 0;
            const uint16_t h = fp8_pair(v[i], ldexpf(1.f, e0));
            if (q < kTileRows) *reinterpret_cast<uint16_t *>(dst + q * 16) = h;
            if (q > 0) {
                uint16_t h1 = h;
                if ((q & (rows_per_scale - 1)) == 0) h1 = fp8_pair(v[i], ldexpf(1.f, s_exp[(q - 1) >> rshift]));
                *reinterpret_cast<uint16_t *>(dst + (kT8Planes / 2) * kT8Plane + (q - 1) * 16) = lane < nhalo ? h1 : 0;
            }
        }
        fence_async_smem();
        tc_fence_before();
        __syncthreads();
        tc_fence_after();
        const uint32_t tmem = *tslot;
        if (t + (int)gridDim.x < ntiles) load_tile(t + gridDim.x);
        if (tid == 0) {
            const uint32_t a0 = smem_u32(sA), b0 = smem_u32(sB);
#pragma unroll
            for (int q = 0; q < kT8Planes / 2; q++)
                umma_f8(tmem, umma_sdesc(a0 + q * 2 * kT8Plane, kT8Plane, 128),
                        umma_sdesc(b0 + q * 2 * kT8BPlane, kT8BPlane, 128), idesc, q > 0);
            umma_commit(bar);
        }
        bool done = mbar_wait(bar, (unsigned)(it & 1));
        if (!done) {
            atomicExch(err, (int)RX_ETIMEOUT);
            mbar_wait(bar, (unsigned)(it & 1));
        }
        ok = __syncthreads_and(done) != 0;
        tc_fence_after();
        if (!ok) break;
        // warp (quarter, half): accumulator lanes (rows) 32 quarter .. + 31, columns
        // 16 half .. + 15 = symbols 8 half .. + 7 of the row, unscaled exactly
        uint32_t acc[16];
        tmem_ld16(tmem + ((uint32_t)(32 * quarter) << 16) + 16 * half, acc);
        const int r = 32 * quarter + lane;
        if (r < rows) {
            const float inv = ldexpf(1.f, -(eB + s_exp[r >> rshift]));
            float4 *zr = reinterpret_cast<float4 *>(z + ((long long)(r0 + r) * kRowSyms + 8 * half));
#pragma unroll
            for (int q = 0; q < 4; q++)
                zr[q] = make_float4(__uint_as_float(acc[4 * q]) * inv, __uint_as_float(acc[4 * q + 1]) * inv,
                                    __uint_as_float(acc[4 * q + 2]) * inv, __uint_as_float(acc[4 * q + 3]) * inv);
        }
        tc_fence_before();
        __syncthreads();   // A, the scales and the accumulator are free again
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) tmem_dealloc(*tslot, kTmemCols);
}

// ---------------------------------------------------------------------------
// 16-bit forms (BF16, FP16): each input sample is converted once.  Block row q of
// a tile holds the 32 complex samples that start at stream sample
// 2 (k_lo + 16 (r0 + q)) - 16, i.e. 64 K elements in 8 core-matrix columns whose
// rows lie 16 bytes apart across 8-row groups (SBO = 128).  Output row r (symbols
// k = k_lo + 16 (r0 + r) + j, j < 16) needs samples 2k - TH .. 2k + TH with TH <= 15,
// all inside block rows r and r + 1: the tile is X[r] B0 + X[r + 1] B1, two sets
// of four K = 16 MMAs over the same planes, the second with its descriptors
// shifted by one row (16 bytes).  Persistent CTAs, two per SM: the next tile's
// samples are loaded into registers while this tile's MMAs and stores run (a
// launch of one CTA per tile spent its first 4 us bringing 512 CTAs up).
constexpr int kT2Rows = kTileRows + 8;            // block rows a plane holds (129 used)
constexpr int kT2Plane = kT2Rows * 16 + 16;       // plane pitch: + 16 bytes skews the planes by 4 banks
constexpr int kT2Planes = 2 * kRowSyms * 2 / 8;   // 64 K elements of a block row, 8 per core row
constexpr int kT2BPlane = kN * 16;                // one K core-matrix column of B (32 rows)
constexpr int kT2OffB = kT2Planes * kT2Plane;
constexpr int kT2OffW = kT2OffB + 2 * kT2Planes * kT2BPlane;   // the taps (32 complex)
constexpr int kT2OffBar = kT2OffW + 32 * 8;
constexpr int kT2Smem = kT2OffBar + 16;
constexpr int kT2Threads = 256, kT2PerSm = 2;
constexpr int kT2Samples = (kTileRows + 1) * 2 * kRowSyms;   // complex samples a tile converts
constexpr int kT2Iter = (kT2Samples + kT2Threads - 1) / kT2Threads;
static_assert(kT2Plane % 16 == 0 && kT2OffB % 16 == 0 && kT2OffBar % 8 == 0, "16-byte aligned operands");
static_assert((kT2Plane / 4) % 32 == 4, "planes four banks apart: a warp's 32 samples store conflict-free");

template <int PREC>
__device__ __forceinline__ uint32_t pack2(float a, float b)
{
    if (PREC == RX_FIR_BF16) {
        __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
        return *reinterpret_cast<uint32_t *>(&h);
    } else {
        __half2 h = __floats2half2_rn(a, b);
        return *reinterpret_cast<uint32_t *>(&h);
    }
}

template <int PREC>
__global__ void __launch_bounds__(kT2Threads, kT2PerSm)
    k_fir_tc2(const float2 *Y, long long ybase, long long k_lo, int nrows,
              const float2 *taps, int ntaps, float2 *z, int *err)
{
    extern __shared__ __align__(1024) unsigned char sm[];
    unsigned char *sA = sm, *sB = sm + kT2OffB;
    uint64_t *bar = reinterpret_cast<uint64_t *>(sm + kT2OffBar);
    uint32_t *tslot = reinterpret_cast<uint32_t *>(bar + 1);
    float2 *s_w = reinterpret_cast<float2 *>(sm + kT2OffW);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, quarter = warp & 3, half = warp >> 2;
    const int th = (ntaps - 1) / 2;
    const int ntiles = (nrows + kTileRows - 1) / kTileRows;
    // a tile's samples into registers: sample j of tile t is stream sample
    // 2 (k_lo + 16 r0) - 16 + j; zero outside the samples its symbols use, so that
    // nothing outside the caller's range is read
    float2 v[kT2Iter];
    auto load_tile = [&](int t) {
        const int r0 = t * kTileRows, rows = min(kTileRows, nrows - r0);
        const long long n0 = 2 * (k_lo + (long long)r0 * kRowSyms) - 16;
        const int jlo = 16 - th, jhi = 2 * (rows * kRowSyms - 1) + th + 16;
        const float2 *Yb = Y + (n0 - ybase);
#pragma unroll
        for (int i = 0; i < kT2Iter; i++) {
            const int j = tid + i * kT2Threads;
            v[i] = (j >= jlo && j <= jhi && j < kT2Samples) ? Yb[j] : make_float2(0.f, 0.f);
        }
    };
    int t = blockIdx.x;
    if (tid == 0) mbar_init(bar, 1);
    if (warp == 0) tmem_alloc(tslot, kTmemCols);
    pdl_wait();
    if (tid < 32) s_w[tid] = tid < ntaps ? taps[tid] : make_float2(0.f, 0.f);
    if (t < ntiles) load_tile(t);
    __syncthreads();   // the taps in shared memory
    // B: rows n = 2 j + c (c: re / im output of symbol j), K index k = 64 h + 2 s + d
    // (block row r + h, sample s, d: re / im); sample 32 h + s of the pair is stream
    // sample 2 k_row - 16 + 32 h + s, so tap i = 2 j + TH + 16 - (32 h + s)
    for (int u = tid; u < kN * 2 * kT2Planes; u += kT2Threads) {
        const int n = u % kN, pl = u / kN;
        const int j = n >> 1, c = n & 1;
        float vb[16];
#pragma unroll
        for (int q = 0; q < 8; q++) {
            const int k = 8 * pl + q, hb = k >> 6, sp = (k & 63) >> 1, d = k & 1;
            const int i = 2 * j + th + 16 - (32 * hb + sp);
            float val = 0.f;
            if (i >= 0 && i < ntaps) {
                const float2 w = s_w[i];
                // conj(w) y: re = a yr + b yi, im = a yi - b yr
                val = c == 0 ? (d == 0 ? w.x : w.y) : (d == 0 ? -w.y : w.x);
            }
            vb[q] = val;
        }
        *reinterpret_cast<uint4 *>(sB + pl * kT2BPlane + n * 16) = pack16<PREC>(vb);
    }
    const uint32_t idesc = umma_idesc(Fmt<PREC>::code, kTileRows, kN);
    bool ok = true;
    for (int it = 0; t < ntiles; t += gridDim.x, it++) {
        const int r0 = t * kTileRows, rows = min(kTileRows, nrows - r0);
        // A: sample j of the tile -> block row j / 32, K elements 2 (j % 32) and + 1
#pragma unroll
        for (int i = 0; i < kT2Iter; i++) {
            const int j = tid + i * kT2Threads;
            if (j < kT2Samples) {
                const int q = j >> 5, s = j & 31;
                *reinterpret_cast<uint32_t *>(sA + (s >> 2) * kT2Plane + q * 16 + (s & 3) * 4) =
                    pack2<PREC>(v[i].x, v[i].y);
            }
        }
        fence_async_smem();
        tc_fence_before();
        __syncthreads();
        tc_fence_after();
        const uint32_t tmem = *tslot;
        // the next tile's loads are in flight while this tile's MMAs and stores run
        if (t + (int)gridDim.x < ntiles) load_tile(t + gridDim.x);
        if (tid == 0) {
            const uint32_t a0 = smem_u32(sA), b0 = smem_u32(sB);
#pragma unroll
            for (int q = 0; q < kT2Planes; q++) {
                const uint32_t shift = q < kT2Planes / 2 ? 0u : 16u;   // block row r, then r + 1
                const uint64_t ad = umma_sdesc(a0 + shift + (q % (kT2Planes / 2)) * 2 * kT2Plane, kT2Plane, 128);
                const uint64_t bd = umma_sdesc(b0 + q * 2 * kT2BPlane, kT2BPlane, 128);
                umma_f16(tmem, ad, bd, idesc, q > 0);
            }
            umma_commit(bar);
        }
        bool done = mbar_wait(bar, (unsigned)(it & 1));
        if (!done) {
            atomicExch(err, (int)RX_ETIMEOUT);
            mbar_wait(bar, (unsigned)(it & 1));
        }
        ok = __syncthreads_and(done) != 0;
        tc_fence_after();
        if (!ok) break;
        // warp (quarter, half): accumulator lanes (rows) 32 quarter .. + 31, columns
        // 16 half .. + 15 = symbols 8 half .. + 7 of the row, stored as four 16-byte pieces
        uint32_t acc[16];
        tmem_ld16(tmem + ((uint32_t)(32 * quarter) << 16) + 16 * half, acc);
        const int r = 32 * quarter + lane;
        if (r < rows) {
            float4 *zr = reinterpret_cast<float4 *>(z + ((long long)(r0 + r) * kRowSyms + 8 * half));
#pragma unroll
            for (int q = 0; q < 4; q++)
                zr[q] = make_float4(__uint_as_float(acc[4 * q]), __uint_as_float(acc[4 * q + 1]),
                                    __uint_as_float(acc[4 * q + 2]), __uint_as_float(acc[4 * q + 3]));
        }
        tc_fence_before();
        __syncthreads();   // A and the accumulator are free again
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) tmem_dealloc(*tslot, kTmemCols);
}

}  // namespace

cudaError_t prepare_fir_tc(int prec)
{
    // every form's shared memory is under the default limit
    return prec == RX_FIR_BF16 || prec == RX_FIR_FP16 || prec == RX_FIR_FP8 ? cudaSuccess : cudaErrorInvalidValue;
}

cudaError_t launch_fir_tc(int prec, const float2 *Y, long long ybase, long long k_lo, long long nsym,
                          const float2 *taps, int ntaps, int scale_block, float2 *z, int *err, int nsm,
                          cudaStream_t st, bool pdl)
{
    if (nsym <= 0) return cudaSuccess;
    if (nsym % kRowSyms || ntaps < 1 || ntaps > 31 || !(ntaps & 1) || scale_block % kRowSyms ||
        (kTileRows * kRowSyms) % scale_block)
        return cudaErrorInvalidValue;
    int nrows = (int)(nsym / kRowSyms);
    int rps = scale_block / kRowSyms;
    int ntiles = (nrows + kTileRows - 1) / kTileRows;
    if (prec == RX_FIR_BF16 || prec == RX_FIR_FP16) {
        const unsigned g2 = (unsigned)min(ntiles, kT2PerSm * nsm);   // persistent CTAs
        return launch_k(prec == RX_FIR_BF16 ? k_fir_tc2<RX_FIR_BF16> : k_fir_tc2<RX_FIR_FP16>, g2, kT2Threads, kT2Smem, st,
                        pdl, Y, ybase, k_lo, nrows, taps, ntaps, z, err);
    }
    if (prec != RX_FIR_FP8) return cudaErrorInvalidValue;
    const unsigned g8 = (unsigned)min(ntiles, kT8PerSm * nsm);   // persistent CTAs
    return launch_k(k_fir_tc8, g8, kT8Threads, kT8Smem, st, pdl, Y, ybase, k_lo, nrows, taps, ntaps, rps, z, err);
}

}  // namespace rxk

// Learned equaliser: a 1-D CNN over the 2-sps matched-filter output, trained on
// the GPU by its own forward and backward kernels (BF16 operands on the tensor
// cores for the forward convolutions, FP32 accumulation, FP32 master weights and
// Adam).
//
// Network (the configured workload's learned equaliser): input y as two channels
// (real, imaginary); three valid convolutions of 32 channels, kernel 9, each
// followed by GELU (exact erf form); at every symbol position an MLP
// 32 -> 64 (GELU) -> 2 gives the soft symbol in unit-power units.  A segment of
// S = 64 symbols starting at symbol k0 reads y[2 k0 - 12, 2 k0 + 140).
// Parameter vector: W1[32][9][2] b1[32] W2[32][9][32] b2[32] W3[32][9][32] b3[32]
//                   M1[64][32] c1[64] M2[2][64] c2[2].
// Activations are channel-last, so the im2col row of output position p of a 32-channel
// layer is 9 consecutive rows of 32 channels: the convolution is a plain GEMM of the rows
// from p on against W[o][k], k = 9 x 32, computed with mma.sync m16n8k16 (BF16 in, FP32
// accumulate); the receiver's inference kernel (tcgen05) is further below.
#include <math.h>
#include <stdlib.h>
#include <string.h>

#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include "rx_async.cuh"
#include "rx_common.cuh"
#include "rx_internal.cuh"

namespace rxk {

constexpr int CC = 32, CK = 9, CH = 64, CS = 64;          // channels, kernel, hidden, symbols per segment
constexpr int L0 = 2 * CS + 24, L1 = L0 - 8, L2 = L1 - 8;
constexpr int KW = CK * CC;                               // 288
constexpr int OW1 = 0, OB1 = OW1 + CC * CK * 2, OW2 = OB1 + CC, OB2 = OW2 + CC * KW, OW3 = OB2 + CC,
              OB3 = OW3 + CC * KW, OM1 = OB3 + CC, OC1 = OM1 + CH * CC, OM2 = OC1 + CH, OC2 = OM2 + 2 * CH,
              NPRM = OC2 + 2;

__device__ __forceinline__ float gelu_f(float u) { return 0.5f * u * (1.0f + erff(u * 0.70710678118654752f)); }
__device__ __forceinline__ float gelu_df(float u)
{
    return 0.5f * (1.0f + erff(u * 0.70710678118654752f)) + u * 0.3989422804014327f * __expf(-0.5f * u * u);
}

__device__ __forceinline__ void mma_bf16(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1)
{
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
                 "{%0,%1,%2,%3};"
                 : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
                 : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// ------------------------------------------------- shared-memory operand tiles
// Activations are rows of 32 channels (64 bytes, four 16-byte chunks), read by
// ldmatrix.  Eight consecutive rows at a 64-byte pitch would fall on two groups of four
// banks; the chunk index is therefore exclusive-ored with bits 1-2 of the row, which
// spreads the eight rows of every 8 x 8 matrix over all 32 banks, for any row offset
// (a tap moves the rows) and for plain and transposed loads.  Weight rows (288 values,
// 36 chunks) have the same pitch modulo 128 bytes and take the same rule.
__device__ __forceinline__ uint32_t row_off(int row, int chunk) { return row * 64 + ((chunk ^ ((row >> 1) & 3)) << 4); }
__device__ __forceinline__ uint32_t w_off(int o, int chunk) { return o * (KW * 2) + ((chunk ^ ((o >> 1) & 3)) << 4); }
// rows of 64 values (128 bytes, eight chunks)
__device__ __forceinline__ uint32_t row128_off(int row, int chunk) { return row * 128 + ((chunk ^ (row & 7)) << 4); }

__device__ __forceinline__ void ldsm4(uint32_t (&r)[4], uint32_t addr)
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(addr)
                 : "memory");
}
__device__ __forceinline__ void ldsm4_t(uint32_t (&r)[4], uint32_t addr)
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(addr)
                 : "memory");
}
__device__ __forceinline__ uint32_t bf2(float a, float b)
{
    __nv_bfloat162 h = __halves2bfloat162(__float2bfloat16(a), __float2bfloat16(b));
    return *reinterpret_cast<uint32_t *>(&h);
}

// BF16 weights of a 32-channel layer, global [32][288] -> shared rows with swizzled chunks
template <int NTH>
__device__ __forceinline__ void stage_w(unsigned char *dst, const __nv_bfloat16 *src, int tid)
{
    for (int i = tid; i < CC * (KW / 8); i += NTH) {
        const int o = i / (KW / 8), ch = i - o * (KW / 8);
        cp_async16(dst + w_off(o, ch), src + o * KW + 8 * ch);
    }
}

// Layer 1 (2 -> 32, K = 18) in FP32, a channel pair per lane (2 cp, 2 cp + 1) as one
// packed FP32 pair, RPH consecutive rows per half-warp.  xs holds every input value
// twice, (re, re, im, im), so that one 16-byte load feeds both channels.  Products are
// accumulated from the bias on in tap order, re before im.
struct L1Weights {
    f2x b, w[18];
};
// shared copy of the weights and biases as channel pairs: [k][pair], row 18 the biases
constexpr int kW1Floats = 19 * CC;
template <int NTH>
__device__ __forceinline__ void stage_l1(float *w1, const float *prm, int tid)
{
    for (int i = tid; i < kW1Floats; i += NTH) {
        const int k = i / CC, o = i % CC;
        w1[i] = k < 18 ? prm[OW1 + o * 18 + k] : prm[OB1 + o];
    }
}
__device__ __forceinline__ void load_l1(L1Weights &W, const float *w1, int cp)
{
    const f2x *p = reinterpret_cast<const f2x *>(w1) + cp;
#pragma unroll
    for (int k = 0; k < 18; k++) W.w[k] = p[k * (CC / 2)];
    W.b = p[18 * (CC / 2)];
}
template <int RPH, typename Emit>
__device__ __forceinline__ void layer1_rows(const L1Weights &W, const float4 *xs, int p0, Emit emit)
{
    ulonglong2 x[RPH + 8];
#pragma unroll
    for (int i = 0; i < RPH + 8; i++) x[i] = reinterpret_cast<const ulonglong2 *>(xs)[p0 + i];
#pragma unroll
    for (int i = 0; i < RPH; i++) {
        f2x a = W.b;
#pragma unroll
        for (int t = 0; t < CK; t++) {
            a = f2_fma(W.w[2 * t], x[i + t].x, a);
            a = f2_fma(W.w[2 * t + 1], x[i + t].y, a);
        }
        emit(p0 + i, f2_unpack(a));
    }
}

// One 16-row tile of a 32-channel, 9-tap convolution: acc[n] += A B over K = 288 in steps
// of 16 (tap ks / 2, channels 16 (ks % 2) ..), 2 NP blocks of 8 output channels from n0.
// a_addr(tap, chunk) is this lane's row address (row lane % 16 of the tile).
template <int NP, typename Addr>
__device__ __forceinline__ void conv_tile(float (&acc)[2 * NP][4], uint32_t w, int n0, int lane, Addr a_addr)
{
    uint32_t wa[2][NP];
#pragma unroll
    for (int p = 0; p < NP; p++) {
        const int n = n0 + 16 * p + (lane & 7) + ((lane >> 4) << 3);
        wa[0][p] = w + w_off(n, (lane >> 3) & 1);
        wa[1][p] = w + w_off(n, 2 + ((lane >> 3) & 1));
    }
#pragma unroll
    for (int n = 0; n < 2 * NP; n++)
#pragma unroll
        for (int i = 0; i < 4; i++) acc[n][i] = 0.f;
#pragma unroll
    for (int ks = 0; ks < KW / 16; ks++) {
        uint32_t a[4], b[NP][4];
        ldsm4(a, a_addr(ks >> 1, 2 * (ks & 1) + (lane >> 4)));
#pragma unroll
        for (int p = 0; p < NP; p++) ldsm4(b[p], wa[ks & 1][p] + 64 * (ks >> 1));
#pragma unroll
        for (int p = 0; p < NP; p++) {
            mma_bf16(acc[2 * p], a, b[p][0], b[p][1]);
            mma_bf16(acc[2 * p + 1], a, b[p][2], b[p][3]);
        }
    }
}

// ------------------------------------------------------------------- inference
// rx_cnn_forward: persistent CTAs of nine warps, three per SM, each looping over
// segments with the weights staged once.  Nine warps because layer 2 has nine row tiles
// of 16 (144 computed positions) and layer 1 144 rows: every warp does one tile with all
// 32 channels.  Layer 3 runs at the symbol (even) positions only, the ones the MLP reads:
// layer 2 stores even and odd positions in two row sets, tap t reads set t & 1.
// The MLP's first layer takes its FP32 weights as three BF16 terms (8 + 8 + 8 bits, the
// sum exact), so its products with the BF16 activations are those of the FP32 weights,
// accumulated in FP32 on the tensor cores.
// Bound: FP32 issue of the erf GELU (472 warp-wide evaluations a segment).  4096 segments:
// 126 us; 457 us with one 128-thread CTA per segment that staged all weights for it, layer
// 3 at every position, 4-byte operand loads and the MLP on the CUDA cores.
constexpr int kFwThreads = 288, kFwPerSm = 3;
constexpr int kH1Rows = L1 + 8;              // rows L1 .. are zero (read by the last tile's taps)
constexpr int kH2Half = L2 / 2;              // rows of each of layer 2's even / odd sets
struct FwdSmem {
    static constexpr int W2 = 0;
    static constexpr int W3 = W2 + CC * KW * 2;
    static constexpr int M1 = W3 + CC * KW * 2;            // bf16 [3 terms][64][32]
    static constexpr int H1 = M1 + 3 * CH * CC * 2;        // bf16 [kH1Rows][32]; then h3 [64][32]
    static constexpr int H2 = H1 + kH1Rows * CC * 2;       // bf16 [2][kH2Half][32]
    static constexpr int XD = H2;                          // float4 [L0]: the input, every value twice (layer 1 only)
    static constexpr int X = H2 + 2 * kH2Half * CC * 2;    // float2 [2][L0]: this and the next segment's input
    static constexpr int W1 = X + 2 * L0 * 8;              // float [19][32]
    static constexpr int B = W1 + kW1Floats * 4;           // float b2, b3 [64], c1 [64], M2 [128], c2 [2] (+ 2)
    static constexpr int OUT = B + (64 + CH + 2 * CH + 4) * 4;   // float [2 halves][64][2]
    static constexpr int TOTAL = OUT + 2 * CS * 2 * 4;
};
static_assert(kFwPerSm * (FwdSmem::TOTAL + 1024) <= 228 * 1024, "three CTAs per SM");
static_assert(FwdSmem::H1 % 16 == 0 && FwdSmem::X % 16 == 0 && FwdSmem::XD % 16 == 0, "16-byte rows");
static_assert(L0 * 16 <= 2 * kH2Half * CC * 2, "the doubled input fits the layer-2 rows");

__global__ void __launch_bounds__(kFwThreads, kFwPerSm)
    k_cnn_fwd(const float *prm, const __nv_bfloat16 *prm_bf, const float2 *y,
              const long long *seg_start, int nseg, float *out)
{
    extern __shared__ __align__(16) unsigned char sm[];
    float2 *x2 = reinterpret_cast<float2 *>(sm + FwdSmem::X);
    float4 *xd = reinterpret_cast<float4 *>(sm + FwdSmem::XD);
    float *b2 = reinterpret_cast<float *>(sm + FwdSmem::B), *b3 = b2 + CC, *c1 = b3 + CC, *m2 = c1 + CH;
    float *os = reinterpret_cast<float *>(sm + FwdSmem::OUT);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, g = lane >> 2, tq = lane & 3;
    const uint32_t sW2 = smem_u32(sm + FwdSmem::W2), sW3 = smem_u32(sm + FwdSmem::W3), sM1 = smem_u32(sm + FwdSmem::M1);
    const uint32_t sH1 = smem_u32(sm + FwdSmem::H1), sH2 = smem_u32(sm + FwdSmem::H2);
    auto prefetch = [&](int s, int buf) {
        const float2 *src = y + seg_start[s];
        for (int i = tid; i < L0; i += kFwThreads) cp_async8(x2 + buf * L0 + i, src + i, true);
        cp_async_commit();
    };
    int s = blockIdx.x;
    pdl_wait();
    if (s < nseg) prefetch(s, 0);
    stage_w<kFwThreads>(sm + FwdSmem::W2, prm_bf + OW2, tid);
    stage_w<kFwThreads>(sm + FwdSmem::W3, prm_bf + OW3, tid);
    cp_async_commit();
    for (int i = tid; i < CH * CC; i += kFwThreads) {   // w = t0 + t1 + t2, every remainder exact in FP32
        const int m = i >> 5, c = i & 31;
        float w = prm[OM1 + i];
#pragma unroll
        for (int t = 0; t < 3; t++) {
            const __nv_bfloat16 h = __float2bfloat16(w);
            w -= __bfloat162float(h);
            *reinterpret_cast<__nv_bfloat16 *>(sm + FwdSmem::M1 + t * CH * CC * 2 + row_off(m, c >> 3) + 2 * (c & 7)) = h;
        }
    }
    if (tid < CC) {
        b2[tid] = prm[OB2 + tid];
        b3[tid] = prm[OB3 + tid];
        reinterpret_cast<uint4 *>(sm + FwdSmem::H1 + L1 * 64)[tid] = make_uint4(0, 0, 0, 0);   // 8 rows of 64 bytes
    }
    for (int i = tid; i < CH; i += kFwThreads) c1[i] = prm[OC1 + i];
    for (int i = tid; i < 2 * CH + 2; i += kFwThreads) m2[i] = prm[OM2 + i];
    float *w1 = reinterpret_cast<float *>(sm + FwdSmem::W1);
    stage_l1<kFwThreads>(w1, prm, tid);
    for (int buf = 0; s < nseg; s += gridDim.x, buf ^= 1) {
        cp_async_wait_all();
        __syncthreads();   // this segment's input (and, the first time, the weights)
        if (s + (int)gridDim.x < nseg) prefetch(s + gridDim.x, buf ^ 1);
        for (int i = tid; i < L0; i += kFwThreads) {
            const float2 v = x2[buf * L0 + i];
            xd[i] = make_float4(v.x, v.x, v.y, v.y);
        }
        __syncthreads();
        L1Weights W1;
        load_l1(W1, w1, lane & 15);
        layer1_rows<8>(W1, xd, 16 * warp + 8 * (lane >> 4), [&](int p, float2 u) {
            const int cp = lane & 15;
            *reinterpret_cast<uint32_t *>(sm + FwdSmem::H1 + row_off(p, cp >> 2) + 4 * (cp & 3)) =
                bf2(gelu_f(u.x), gelu_f(u.y));
        });
        __syncthreads();
        {   // layer 2: rows 16 warp ..
            float acc[4][4];
            conv_tile<2>(acc, sW2, 0, lane, [&](int t, int ch) { return sH1 + row_off(16 * warp + (lane & 15) + t, ch); });
#pragma unroll
            for (int n = 0; n < 4; n++) {
                const float2 b = *reinterpret_cast<const float2 *>(b2 + 8 * n + 2 * tq);
#pragma unroll
                for (int h = 0; h < 2; h++) {
                    const int r = 16 * warp + g + 8 * h;
                    if (r < L2)
                        *reinterpret_cast<uint32_t *>(sm + FwdSmem::H2 + (r & 1) * kH2Half * 64 + row_off(r >> 1, n) + 4 * tq) =
                            bf2(gelu_f(acc[n][2 * h] + b.x), gelu_f(acc[n][2 * h + 1] + b.y));
                }
            }
        }
        __syncthreads();
        if (warp < 8) {   // layer 3 at the symbols 16 tile ..: channels 16 half ..
            const int tile = warp >> 1, half = warp & 1;
            float acc[2][4];
            conv_tile<1>(acc, sW3, 16 * half, lane, [&](int t, int ch) {
                return sH2 + (t & 1) * kH2Half * 64 + row_off(16 * tile + (lane & 15) + (t >> 1), ch);
            });
#pragma unroll
            for (int n = 0; n < 2; n++) {
                const float2 b = *reinterpret_cast<const float2 *>(b3 + 16 * half + 8 * n + 2 * tq);
#pragma unroll
                for (int h = 0; h < 2; h++)
                    *reinterpret_cast<uint32_t *>(sm + FwdSmem::H1 + row_off(16 * tile + g + 8 * h, 2 * half + n) + 4 * tq) =
                        bf2(gelu_f(acc[n][2 * h] + b.x), gelu_f(acc[n][2 * h + 1] + b.y));
            }
        }
        __syncthreads();
        if (warp < 8) {   // MLP: symbols 16 tile .., hidden units 32 half ..
            const int tile = warp >> 1, half = warp & 1;
            float acc[4][4];
#pragma unroll
            for (int n = 0; n < 4; n++)
#pragma unroll
                for (int i = 0; i < 4; i++) acc[n][i] = 0.f;
            uint32_t a[2][4];
#pragma unroll
            for (int ks = 0; ks < 2; ks++) ldsm4(a[ks], sH1 + row_off(16 * tile + (lane & 15), 2 * ks + (lane >> 4)));
#pragma unroll
            for (int t = 2; t >= 0; t--)   // smallest terms first
#pragma unroll
                for (int ks = 0; ks < 2; ks++)
#pragma unroll
                    for (int p = 0; p < 2; p++) {
                        uint32_t b[4];
                        ldsm4(b, sM1 + t * CH * CC * 2 +
                                     row_off(32 * half + 16 * p + (lane & 7) + ((lane >> 4) << 3), 2 * ks + ((lane >> 3) & 1)));
                        mma_bf16(acc[2 * p], a[ks], b[0], b[1]);
                        mma_bf16(acc[2 * p + 1], a[ks], b[2], b[3]);
                    }
            float o[2][2] = {{0.f, 0.f}, {0.f, 0.f}};   // [row g, g + 8][output]
#pragma unroll
            for (int n = 0; n < 4; n++)
#pragma unroll
                for (int i = 0; i < 2; i++) {
                    const int m = 32 * half + 8 * n + 2 * tq + i;
                    const float c = c1[m], ma = m2[m], mb = m2[CH + m];
#pragma unroll
                    for (int h = 0; h < 2; h++) {
                        const float z = gelu_f(acc[n][2 * h + i] + c);
                        o[h][0] = fmaf(ma, z, o[h][0]);
                        o[h][1] = fmaf(mb, z, o[h][1]);
                    }
                }
#pragma unroll
            for (int h = 0; h < 2; h++)
#pragma unroll
                for (int q = 0; q < 2; q++) {
                    o[h][q] += __shfl_xor_sync(0xffffffffu, o[h][q], 1);
                    o[h][q] += __shfl_xor_sync(0xffffffffu, o[h][q], 2);
                }
            if (tq == 0)
#pragma unroll
                for (int h = 0; h < 2; h++)
                    *reinterpret_cast<float2 *>(os + 2 * (CS * half + 16 * tile + g + 8 * h)) = make_float2(o[h][0], o[h][1]);
        }
        __syncthreads();
        if (tid < 2 * CS) out[(size_t)s * 2 * CS + tid] = os[tid] + os[2 * CS + tid] + m2[2 * CH + (tid & 1)];
    }
    cp_async_wait_all();
}

// --------------------------------------------------------------------- training
// Forward and backward pass of one segment per CTA, everything between them in shared
// memory: 18 warps, since layer 2 has 9 row tiles x 2 channel halves, its input gradient
// the same, and a weight gradient 2 x 9 (output-channel half, tap) units.  The GELU
// derivative is taken with the GELU (they share the erf) and kept in FP32 in place of the
// pre-activation.  The transposed operands of the backward products (du and the layer
// inputs with the positions along K, the weights with the output channels along K) are
// read with transposing ldmatrix from the forward's own tiles, so nothing is rearranged.
// A step of 64 segments (this kernel, the reduction and Adam, each launched as the
// dependent of the one before): 26 us; 146 us with a forward
// and a backward kernel that passed activations through global memory and rearranged their
// operands in shared memory.  Bound: the chain of eleven phases, each a few hundred cycles
// of one CTA per SM.
// BF16 operands, FP32 accumulation over the positions in order (mma.sync m16n8k16: the
// contractions of a segment are 32 wide, below a tcgen05 tile); GELU derivatives, dM2,
// biases and the 2-channel layer 1 in FP32.
constexpr int kTrThreads = 576, kTrWarps = kTrThreads / 32;
constexpr int kZP = CH + 1;                                  // padded row of the hidden units
struct TrainSmem {
    static constexpr int W2 = 0;
    static constexpr int W3 = W2 + CC * KW * 2;
    static constexpr int M1B = W3 + CC * KW * 2;             // bf16 [64][32]
    static constexpr int M1 = M1B + CH * CC * 2;             // float [64][32]
    static constexpr int H1 = M1 + CH * CC * 4;              // bf16 [kH1Rows][32]
    static constexpr int H2 = H1 + kH1Rows * CC * 2;         // bf16 [L2][32]
    static constexpr int H3 = H2 + L2 * CC * 2;              // bf16 [64][32] (symbols)
    static constexpr int DVB = H3 + CS * CC * 2;             // bf16 [64 symbols][64 units] dv
    static constexpr int DU3 = DVB + CS * CH * 2;            // bf16 [160][32]: du3 from row 8 on
    static constexpr int DU2 = DU3 + 160 * CC * 2;           // bf16 [160][32]: du2 from row 8 on
    static constexpr int D1 = DU2 + 160 * CC * 2;            // float [L1][32]: gelu'(u1), then du1
    static constexpr int D2 = D1 + L1 * CC * 4;              // float [L2][32]: gelu'(u2)
    static constexpr int D3 = D2 + L2 * CC * 4;              // float [64][32]: gelu'(u3)
    static constexpr int Z = D3 + CS * CC * 4;               // float [64][kZP] hidden units
    static constexpr int DZ = Z + CS * kZP * 4;              // float [64][kZP] gelu'(v), then dv
    static constexpr int XD = DZ + CS * kZP * 4;             // float4 [L0]
    static constexpr int W1 = XD + L0 * 16;                  // float [19][32]
    static constexpr int B = W1 + kW1Floats * 4;             // float b2, b3 [64], c1 [64], M2 [128] c2 [2] (+ 2)
    static constexpr int DO = B + (64 + CH + 2 * CH + 4) * 4;   // float [64][2] gradient at the outputs
    static constexpr int RED = DO + CS * 2 * 4;              // float [18][32] bias partials, [4] loss
    static constexpr int TOTAL = RED + (kTrWarps * CC + 4) * 4;
    static constexpr int P1 = D2;                            // float [18][576] layer-1 partials (D2, D3, Z are free)
};
static_assert(TrainSmem::TOTAL <= 227 * 1024, "one training CTA per SM");
static_assert(TrainSmem::P1 + kTrWarps * CC * 18 * 4 <= TrainSmem::DZ, "layer-1 partials fit");
static_assert(TrainSmem::M1 % 16 == 0 && TrainSmem::H1 % 16 == 0 && TrainSmem::DU3 % 16 == 0 && TrainSmem::XD % 16 == 0,
              "16-byte rows");

__global__ void __launch_bounds__(kTrThreads, 1)
    k_cnn_train(const float *prm, const __nv_bfloat16 *prm_bf, const float2 *y,
                const long long *seg_start, const float *tgt, float norm,
                float *gpart, float *lpart)
{
    extern __shared__ __align__(16) unsigned char sm[];
    float4 *xd = reinterpret_cast<float4 *>(sm + TrainSmem::XD);
    float *b2 = reinterpret_cast<float *>(sm + TrainSmem::B), *b3 = b2 + CC, *c1 = b3 + CC, *m2 = c1 + CH;
    float *m1 = reinterpret_cast<float *>(sm + TrainSmem::M1);
    float *d1 = reinterpret_cast<float *>(sm + TrainSmem::D1), *d2 = reinterpret_cast<float *>(sm + TrainSmem::D2);
    float *d3 = reinterpret_cast<float *>(sm + TrainSmem::D3);
    float *zs = reinterpret_cast<float *>(sm + TrainSmem::Z), *dz = reinterpret_cast<float *>(sm + TrainSmem::DZ);
    float *dout = reinterpret_cast<float *>(sm + TrainSmem::DO), *red = reinterpret_cast<float *>(sm + TrainSmem::RED);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, g = lane >> 2, tq = lane & 3;
    const uint32_t sW2 = smem_u32(sm + TrainSmem::W2), sW3 = smem_u32(sm + TrainSmem::W3);
    const uint32_t sH1 = smem_u32(sm + TrainSmem::H1), sH2 = smem_u32(sm + TrainSmem::H2), sH3 = smem_u32(sm + TrainSmem::H3);
    const uint32_t sDV = smem_u32(sm + TrainSmem::DVB), sM1B = smem_u32(sm + TrainSmem::M1B);
    const int s = blockIdx.x;
    float *G = gpart + (size_t)s * NPRM;

    // ---- stage: the input and what layer 1 needs first, the weights behind it
    pdl_wait();
    stage_w<kTrThreads>(sm + TrainSmem::W2, prm_bf + OW2, tid);
    stage_w<kTrThreads>(sm + TrainSmem::W3, prm_bf + OW3, tid);
    for (int i = tid; i < CH * 4; i += kTrThreads)
        cp_async16(sm + TrainSmem::M1B + row_off(i >> 2, i & 3), prm_bf + OM1 + 8 * i);
    for (int i = tid; i < CH * CC / 4; i += kTrThreads) cp_async16(m1 + 4 * i, prm + OM1 + 4 * i);
    cp_async_commit();
    {
        const float2 *src = y + seg_start[s];
        for (int i = tid; i < L0; i += kTrThreads) {
            const float2 v = src[i];
            xd[i] = make_float4(v.x, v.x, v.y, v.y);
        }
    }
    if (tid < CC) {
        b2[tid] = prm[OB2 + tid];
        b3[tid] = prm[OB3 + tid];
        reinterpret_cast<uint4 *>(sm + TrainSmem::H1 + L1 * 64)[tid] = make_uint4(0, 0, 0, 0);
    }
    for (int i = tid; i < CH; i += kTrThreads) c1[i] = prm[OC1 + i];
    for (int i = tid; i < 2 * CH + 2; i += kTrThreads) m2[i] = prm[OM2 + i];
    // du3 is zero at the odd positions and both du in the rows around them
    for (int i = tid; i < 160 * 4; i += kTrThreads) {
        reinterpret_cast<uint4 *>(sm + TrainSmem::DU3)[i] = make_uint4(0, 0, 0, 0);
        if (i < 8 * 4 || i >= (8 + L2) * 4) reinterpret_cast<uint4 *>(sm + TrainSmem::DU2)[i] = make_uint4(0, 0, 0, 0);
    }
    float *w1 = reinterpret_cast<float *>(sm + TrainSmem::W1);
    stage_l1<kTrThreads>(w1, prm, tid);
    __syncthreads();
    // ---- layer 1
    L1Weights W1;
    load_l1(W1, w1, lane & 15);
    layer1_rows<4>(W1, xd, 8 * warp + 4 * (lane >> 4), [&](int p, float2 u) {
        const int cp = lane & 15;
        *reinterpret_cast<uint32_t *>(sm + TrainSmem::H1 + row_off(p, cp >> 2) + 4 * (cp & 3)) =
            bf2(gelu_f(u.x), gelu_f(u.y));
        *reinterpret_cast<float2 *>(d1 + p * CC + 2 * cp) = make_float2(gelu_df(u.x), gelu_df(u.y));
    });
    cp_async_wait_all();
    __syncthreads();
    const int tile9 = warp % 9, half2 = warp / 9;   // a row tile and a half of the channels
    {   // ---- layer 2
        float acc[2][4];
        conv_tile<1>(acc, sW2, 16 * half2, lane, [&](int t, int ch) { return sH1 + row_off(16 * tile9 + (lane & 15) + t, ch); });
#pragma unroll
        for (int n = 0; n < 2; n++) {
            const int o = 16 * half2 + 8 * n + 2 * tq;
            const float2 b = *reinterpret_cast<const float2 *>(b2 + o);
#pragma unroll
            for (int h = 0; h < 2; h++) {
                const int r = 16 * tile9 + g + 8 * h;
                if (r < L2) {
                    const float u0 = acc[n][2 * h] + b.x, u1 = acc[n][2 * h + 1] + b.y;
                    *reinterpret_cast<uint32_t *>(sm + TrainSmem::H2 + row_off(r, 2 * half2 + n) + 4 * tq) =
                        bf2(gelu_f(u0), gelu_f(u1));
                    *reinterpret_cast<float2 *>(d2 + r * CC + o) = make_float2(gelu_df(u0), gelu_df(u1));
                }
            }
        }
    }
    __syncthreads();
    if (warp < 8) {   // ---- layer 3 at the symbol (even) positions
        const int tile = warp >> 1, half = warp & 1;
        float acc[2][4];
        conv_tile<1>(acc, sW3, 16 * half, lane,
                     [&](int t, int ch) { return sH2 + row_off(2 * (16 * tile + (lane & 15)) + t, ch); });
#pragma unroll
        for (int n = 0; n < 2; n++) {
            const int o = 16 * half + 8 * n + 2 * tq;
            const float2 b = *reinterpret_cast<const float2 *>(b3 + o);
#pragma unroll
            for (int h = 0; h < 2; h++) {
                const int r = 16 * tile + g + 8 * h;
                const float u0 = acc[n][2 * h] + b.x, u1 = acc[n][2 * h + 1] + b.y;
                *reinterpret_cast<uint32_t *>(sm + TrainSmem::H3 + row_off(r, 2 * half + n) + 4 * tq) =
                    bf2(gelu_f(u0), gelu_f(u1));
                *reinterpret_cast<float2 *>(d3 + r * CC + o) = make_float2(gelu_df(u0), gelu_df(u1));
            }
        }
    }
    __syncthreads();
    if (warp < 16) {   // ---- MLP hidden layer in FP32: 8 units per warp, a symbol per lane
        const int j = 32 * (warp & 1) + lane, m0 = 8 * (warp >> 1);
        float hv[CC];
#pragma unroll
        for (int q = 0; q < 4; q++) {
            const uint4 v = *reinterpret_cast<const uint4 *>(sm + TrainSmem::H3 + row_off(j, q));
            const uint32_t u[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
            for (int i = 0; i < 4; i++) {
                hv[8 * q + 2 * i] = __uint_as_float(u[i] << 16);
                hv[8 * q + 2 * i + 1] = __uint_as_float(u[i] & 0xFFFF0000u);
            }
        }
#pragma unroll 2
        for (int mm = 0; mm < 8; mm++) {
            const int m = m0 + mm;
            float a = c1[m];
            const float4 *w4 = reinterpret_cast<const float4 *>(m1 + m * CC);
#pragma unroll
            for (int q = 0; q < 8; q++) {
                const float4 w = w4[q];
                a = fmaf(w.x, hv[4 * q], a);
                a = fmaf(w.y, hv[4 * q + 1], a);
                a = fmaf(w.z, hv[4 * q + 2], a);
                a = fmaf(w.w, hv[4 * q + 3], a);
            }
            zs[j * kZP + m] = gelu_f(a);
            dz[j * kZP + m] = gelu_df(a);
        }
    }
    __syncthreads();
    if (tid < 2 * CS) {   // ---- outputs, loss, gradient at the outputs: two threads per symbol, 32 units each
        const int j = tid >> 1, half = tid & 1;
        float o0 = 0.f, o1 = 0.f;
#pragma unroll 8
        for (int mm = 0; mm < CH / 2; mm++) {
            const int m = half * (CH / 2) + mm;
            const float z = zs[j * kZP + m];
            o0 = fmaf(m2[m], z, o0);
            o1 = fmaf(m2[CH + m], z, o1);
        }
        o0 += __shfl_xor_sync(0xffffffffu, o0, 1);
        o1 += __shfl_xor_sync(0xffffffffu, o1, 1);
        const float o = (half ? o1 : o0) + m2[2 * CH + half];
        const float e = o - tgt[(size_t)s * 2 * CS + tid];
        dout[tid] = 2.f * e * norm;
        const float l = warp_sum_f(e * e);
        if (lane == 0) red[kTrWarps * CC + warp] = l;
    }
    __syncthreads();
    if (tid == 0) {
        const float *l = red + kTrWarps * CC;
        lpart[s] = (l[0] + l[1]) + (l[2] + l[3]);
    }
    for (int i = tid; i < CS * CH / 2; i += kTrThreads) {   // ---- dv = (dout . M2) gelu'(v)
        const int j = i >> 5, m = 2 * (i & 31);
        const float g0 = dout[2 * j], g1 = dout[2 * j + 1];
        float d[2];
#pragma unroll
        for (int q = 0; q < 2; q++) {
            const float dzv = g0 * m2[m + q] + g1 * m2[CH + m + q];
            d[q] = dzv * dz[j * kZP + m + q];
            dz[j * kZP + m + q] = d[q];
        }
        *reinterpret_cast<uint32_t *>(sm + TrainSmem::DVB + row128_off(j, m >> 3) + 2 * (m & 7)) = bf2(d[0], d[1]);
    }
    __syncthreads();
    // ---- tasks 0..6: dM2, dc2, dc1 in FP32 (one sum over the symbols per lane);
    // 7..22: du3[j][c] = gelu'(u3) sum_m dv[j][m] M1[m][c] (16 symbols x 8 channels);
    // 23..38: dM1[m][c] = sum_j dv[j][m] h3[j][c] (16 units x 8 channels)
    for (int task = warp; task < 39; task += kTrWarps) {
        if (task < 7) {
            const int i = 32 * task + lane;   // dM2 [2][64], dc2 [2] (contiguous in G), then dc1 from 160 on
            float a = 0.f;
            if (i < 2 * CH) {
                const int oc = i >> 6, m = i & 63;
#pragma unroll 8
                for (int j = 0; j < CS; j++) a = fmaf(dout[2 * j + oc], zs[j * kZP + m], a);
                G[OM2 + i] = a;
            } else if (i < 2 * CH + 2) {
                for (int j = 0; j < CS; j++) a += dout[2 * j + i - 2 * CH];
                G[OM2 + i] = a;
            } else if (i >= 160) {
#pragma unroll 8
                for (int j = 0; j < CS; j++) a += dz[j * kZP + i - 160];
                G[OC1 + i - 160] = a;
            }
            continue;
        }
        const bool in = task < 23;
        const int mt = (in ? task - 7 : task - 23) >> 2, nt = (in ? task - 7 : task - 23) & 3;
        float acc[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int ks = 0; ks < 4; ks++) {
            uint32_t a[4], b[4];
            if (in) {   // A: dv rows (symbols); B: M1 with the units along K
                ldsm4(a, sDV + row128_off(16 * mt + (lane & 15), 2 * ks + (lane >> 4)));
                ldsm4_t(b, sM1B + row_off(16 * ks + (lane & 15), nt));
            } else {    // A: dv with the symbols along K; B: h3 with the symbols along K
                ldsm4_t(a, sDV + row128_off(16 * ks + (lane & 7) + ((lane >> 4) << 3), 2 * mt + ((lane >> 3) & 1)));
                ldsm4_t(b, sH3 + row_off(16 * ks + (lane & 15), nt));
            }
            mma_bf16(acc, a, b[0], b[1]);
        }
        if (in) {
            float cs[2] = {0.f, 0.f};
#pragma unroll
            for (int h = 0; h < 2; h++) {
                const int j = 16 * mt + g + 8 * h, c = 8 * nt + 2 * tq;
                const float2 f = *reinterpret_cast<const float2 *>(d3 + j * CC + c);
                const float v0 = acc[2 * h] * f.x, v1 = acc[2 * h + 1] * f.y;
                *reinterpret_cast<uint32_t *>(sm + TrainSmem::DU3 + row_off(8 + 2 * j, nt) + 4 * tq) = bf2(v0, v1);
                cs[0] += v0;
                cs[1] += v1;
            }
#pragma unroll
            for (int q = 0; q < 2; q++)
#pragma unroll
                for (int o = 4; o < 32; o <<= 1) cs[q] += __shfl_xor_sync(0xffffffffu, cs[q], o);
            if (g == 0) *reinterpret_cast<float2 *>(red + mt * CC + 8 * nt + 2 * tq) = make_float2(cs[0], cs[1]);
        } else {
#pragma unroll
            for (int h = 0; h < 2; h++)
                *reinterpret_cast<float2 *>(G + OM1 + (16 * mt + g + 8 * h) * CC + 8 * nt + 2 * tq) =
                    make_float2(acc[2 * h], acc[2 * h + 1]);
        }
    }
    __syncthreads();
    // ---- convolution layers 3 and 2: per warp one unit of the weight gradient
    // dW[o][t][c] = sum_p du[p][o] h_in[p + t][c] (16 output channels, one tap, 32 input
    // channels) and one of the input gradient dh_in[q][c] = sum_{t, o} W[o][t][c] du[q - t][o]
    // (16 positions, 16 channels; row q of the padded du from row q on, tap 8 - t at row
    // q + 8 - t), which times gelu' is the du of the layer below
#pragma unroll
    for (int l = 3; l >= 2; l--) {
        const uint32_t sDU = smem_u32(sm + (l == 3 ? TrainSmem::DU3 : TrainSmem::DU2));
        const uint32_t sHin = l == 3 ? sH2 : sH1, sW = l == 3 ? sW3 : sW2;
        const int OW = l == 3 ? OW3 : OW2, OB = l == 3 ? OB3 : OB2;
        const int nred = l == 3 ? 4 : 9;   // bias partials left by the step before
        if (warp == kTrWarps - 1) {
            float a = 0.f;
            for (int w = 0; w < nred; w++) a += red[w * CC + lane];
            G[OB + lane] = a;
        }
        {
            const int t = tile9;
            float acc[4][4];
#pragma unroll
            for (int n = 0; n < 4; n++)
#pragma unroll
                for (int i = 0; i < 4; i++) acc[n][i] = 0.f;
            // positions 16 ks ..; layer 3's du is zero from position 128 on
#pragma unroll
            for (int ks = 0; ks < (l == 3 ? 8 : 9); ks++) {
                uint32_t a[4], b[2][4];
                ldsm4_t(a, sDU + row_off(8 + 16 * ks + (lane & 7) + ((lane >> 4) << 3), 2 * half2 + ((lane >> 3) & 1)));
#pragma unroll
                for (int p = 0; p < 2; p++) ldsm4_t(b[p], sHin + row_off(16 * ks + (lane & 15) + t, 2 * p + (lane >> 4)));
#pragma unroll
                for (int p = 0; p < 2; p++) {
                    mma_bf16(acc[2 * p], a, b[p][0], b[p][1]);
                    mma_bf16(acc[2 * p + 1], a, b[p][2], b[p][3]);
                }
            }
#pragma unroll
            for (int n = 0; n < 4; n++)
#pragma unroll
                for (int h = 0; h < 2; h++)
                    *reinterpret_cast<float2 *>(G + OW + (16 * half2 + g + 8 * h) * KW + t * CC + 8 * n + 2 * tq) =
                        make_float2(acc[n][2 * h], acc[n][2 * h + 1]);
        }
        float acc[2][4];
#pragma unroll
        for (int n = 0; n < 2; n++)
#pragma unroll
            for (int i = 0; i < 4; i++) acc[n][i] = 0.f;
#pragma unroll
        for (int ks = 0; ks < KW / 16; ks++) {
            uint32_t a[4], b[4];
            ldsm4(a, sDU + row_off(16 * tile9 + (lane & 15) + (ks >> 1), 2 * (ks & 1) + (lane >> 4)));
            ldsm4_t(b, sW + w_off(16 * (ks & 1) + (lane & 15), 4 * (CK - 1 - (ks >> 1)) + 2 * half2 + (lane >> 4)));
            mma_bf16(acc[0], a, b[0], b[1]);
            mma_bf16(acc[1], a, b[2], b[3]);
        }
        __syncthreads();   // the partials in red are read
        const int Lin = l == 3 ? L2 : L1;
        float cs[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int n = 0; n < 2; n++)
#pragma unroll
            for (int h = 0; h < 2; h++) {
                const int q = 16 * tile9 + g + 8 * h, c = 16 * half2 + 8 * n + 2 * tq;
                if (q >= Lin) continue;
                float2 *f = reinterpret_cast<float2 *>((l == 3 ? d2 : d1) + q * CC + c);
                const float v0 = acc[n][2 * h] * f->x, v1 = acc[n][2 * h + 1] * f->y;
                if (l == 3)
                    *reinterpret_cast<uint32_t *>(sm + TrainSmem::DU2 + row_off(8 + q, 2 * half2 + n) + 4 * tq) = bf2(v0, v1);
                else
                    *f = make_float2(v0, v1);
                cs[2 * n] += v0;
                cs[2 * n + 1] += v1;
            }
#pragma unroll
        for (int q = 0; q < 4; q++)
#pragma unroll
            for (int o = 4; o < 32; o <<= 1) cs[q] += __shfl_xor_sync(0xffffffffu, cs[q], o);
        if (g == 0)
#pragma unroll
            for (int n = 0; n < 2; n++)
                *reinterpret_cast<float2 *>(red + tile9 * CC + 16 * half2 + 8 * n + 2 * tq) =
                    make_float2(cs[2 * n], cs[2 * n + 1]);
        __syncthreads();
    }
    // ---- layer 1 in FP32: dW1[o][t][c] = sum_p du1[p][o] x[p + t][c], eight positions per
    // warp with an output channel per lane, then the 18 partials of each weight
    {
        float a[18], du[8];
#pragma unroll
        for (int i = 0; i < 8; i++) du[i] = d1[(8 * warp + i) * CC + lane];
#pragma unroll
        for (int k = 0; k < 18; k++) a[k] = 0.f;
#pragma unroll
        for (int i = 0; i < 16; i++) {
            const float4 x = xd[8 * warp + i];
#pragma unroll
            for (int q = 0; q < 8; q++) {
                const int t = i - q;
                if (t < 0 || t >= CK) continue;
                a[2 * t] = fmaf(du[q], x.x, a[2 * t]);
                a[2 * t + 1] = fmaf(du[q], x.z, a[2 * t + 1]);
            }
        }
        float *part = reinterpret_cast<float *>(sm + TrainSmem::P1);
#pragma unroll
        for (int k = 0; k < 18; k++) part[warp * (18 * CC) + k * CC + lane] = a[k];
        __syncthreads();
        float v = 0.f;
#pragma unroll
        for (int w = 0; w < kTrWarps; w++) v += part[w * (18 * CC) + tid];
        G[OW1 + (tid & 31) * 18 + (tid >> 5)] = v;
        if (warp == 0) {
            float b = 0.f;
            for (int w = 0; w < 9; w++) b += red[w * CC + lane];
            G[OB1 + lane] = b;
        }
    }
}

// grad[i] = sum_s gpart[s][i] in segment order, copied to the caller's buffer (or null);
// the last CTA sums the segments' loss parts
constexpr int kRedThreads = 128;
__global__ void __launch_bounds__(kRedThreads)
    k_cnn_reduce(const float *gpart, const float *lpart, int nseg, float norm,
                 float *grad, float *grad_out, float *loss, float *loss_out)
{
    pdl_wait();
    if (blockIdx.x == gridDim.x - 1) {
        __shared__ float part[kRedThreads / 32];
        float a = 0.f;
        for (int s = threadIdx.x; s < nseg; s += kRedThreads) a += lpart[s];
        a = warp_sum_f(a);
        if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = a;
        __syncthreads();
        if (threadIdx.x == 0) {
            const float v = ((part[0] + part[1]) + (part[2] + part[3])) * norm;
            *loss = v;
            if (loss_out) *loss_out = v;
        }
        return;
    }
    const int i = blockIdx.x * kRedThreads + threadIdx.x;
    if (i >= NPRM) return;
    float a = 0.f;
#pragma unroll 16
    for (int s = 0; s < nseg; s++) a += gpart[(size_t)s * NPRM + i];
    grad[i] = a;
    if (grad_out) grad_out[i] = a;
}

// Adam on the FP32 master weights; refreshes the BF16 copy
__global__ void k_cnn_adam(float *prm, __nv_bfloat16 *prm_bf,
                           float *m, float *v, const float *grad, float lr,
                           float b1t, float b2t)
{
    pdl_wait();
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= NPRM) return;
    const float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
    float g = grad[i];
    float mi = b1 * m[i] + (1.f - b1) * g, vi = b2 * v[i] + (1.f - b2) * g * g;
    m[i] = mi;
    v[i] = vi;
    float mh = mi / (1.f - b1t), vh = vi / (1.f - b2t);
    float w = prm[i] - lr * mh / (sqrtf(vh) + eps);
    prm[i] = w;
    prm_bf[i] = __float2bfloat16(w);
}

__global__ void k_cnn_tobf(const float *__restrict__ prm, __nv_bfloat16 *__restrict__ prm_bf)
{
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < NPRM) prm_bf[i] = __float2bfloat16(prm[i]);
}

// ====================================================================
// Receiver inference on the fifth-generation tensor cores (tcgen05).
//
// Tiles of kTS = 128 symbols (two 64-symbol windows).  One persistent CTA per SM
// runs kRxGroups independent groups of 8 warps, each with its own tile loop,
// activation planes, mbarrier, 128 tensor-memory columns and named barrier, and all
// reading the weights staged once per CTA: while one group waits on its MMAs or its
// tensor-memory loads, the others issue, so kRxGroups tiles are in flight per SM.  In
// a group two warps share each tensor-memory lane quarter, each taking half of the
// accumulator columns.  Activations live
// in shared memory as "planes" of 8 channels, each position one 16-byte row: with
// this layout the im2col operand of a 32-channel, 9-tap convolution at K-step ks
// (tap ks/2, channel groups 2 (ks % 2) and +1) is the plane pair read from
// position p + ks/2 onwards, i.e. a K-major no-swizzle matrix descriptor whose
// start address moves by whole 16-byte rows; no im2col copy is made.
//   layer 1 (2 -> 32, K = 18 padded to 32): one FP16 plane whose row p holds the
//      8 reals of positions p .. p+3; a descriptor whose two K core matrices sit
//      4 rows apart (leading offset 64 bytes) reads rows p, p+4 (K 0..15) and,
//      8 rows on, p+8, p+12 (K 16..31): the whole im2col row of position p;
//   layer 2 (32 -> 32): 18 tcgen05.mma (M = 128, N = 32, K = 16) per 128
//      positions; its epilogue stores the even and the odd positions in two
//      separate plane sets;
//   layer 3 (32 -> 32) only at the symbol (even) positions 2j: tap 2e reads the
//      even set from row j + e, tap 2e + 1 the odd set from row j + e, so one
//      M = 128 tile covers the tile's 128 symbols;
//   MLP 32 -> 64 (M = 128, N = 64) on the symbols, bias + GELU into FP16
//      planes, then 64 -> 2 as one more MMA (N = 16, two live columns);
//   decisions by the lanes that hold the outputs, window records as the FIR receiver.
// Row tiles of layers 1 and 2 are committed one by one, so that a tile's epilogue runs
// while the next one's MMAs do, and a group passes six barriers per tile.  Bound by the
// latency of each tile's chain of MMA commits, tensor-memory loads and barriers with four
// tiles in flight per SM (tensor pipe 21 % active): 192 us per 2^20 symbols; 196 us with one
// commit per layer, eleven barriers and the decisions on two of eight warps.
// Inference precision: BF16 operands by default, FP16 as the alternative
// (activations and weights, converted from the FP32 master weights), FP32
// accumulation in tensor memory; bias and GELU in the same packed type, GELU by its
// tanh form 0.5 u (1 + tanh(sqrt(2/pi) (u + 0.044715 u^3))) with the hardware tanh
// (tanh.approx.bf16x2 / .f16x2): its distance to the erf form (< 2.2e-4 absolute)
// stays below the resolution the activations are stored with (2^-8 / 2^-11).
constexpr int kTS = 128;
constexpr int kP0 = 2 * kTS + 24, kP1 = kP0 - 8, kP2 = kP1 - 8;   // 280 272 264 input / layer-1 / layer-2 positions
constexpr int kMT1 = (kP1 + 127) / 128, kMT2 = (kP2 + 127) / 128;  // 3, 3 row tiles
constexpr int kRX = 128 * kMT1 + 12;         // rows of the layer-1 input plane (396)
constexpr int kR1 = 128 * kMT2 + 8;          // rows of the h1 planes (rows >= kP1 stay zero); h3 reuses rows < 128
constexpr int kRE = kP2 / 2 + 4;             // rows of each even / odd h2 plane (136; rows < 132 written)
constexpr int kWinT = kTS / 64;              // windows per tile
constexpr int kRxGroups = 4;                 // tile groups per CTA (tiles in flight per SM)
constexpr int kRxGroupThreads = 256;         // 8 warps: two per tensor-memory lane quarter
constexpr int kRxThreads = kRxGroups * kRxGroupThreads;
constexpr uint32_t kRxTmemGroup = 128;       // accumulator columns of one group
constexpr uint32_t kRxTmem = 512;            // the CTA's allocation (a power of two)
constexpr uint32_t kColOut = 96;             // accumulator columns of the 64 -> 2 projection
static_assert(kRxGroups * kRxTmemGroup <= kRxTmem && kRxTmem <= 512, "tensor memory of one SM");
// Shared memory: the weights (read by every group), then one block per group.
struct RxSmem {
    static constexpr int W2 = 0;                          // fp16 planes [36][32 rows][16 B]
    static constexpr int W3 = W2 + 36 * 512;
    static constexpr int M1 = W3 + 36 * 512;              // fp16 planes [4][64 rows][16 B]
    static constexpr int M2 = M1 + 4 * 1024;              // fp16 planes [8][16 rows][16 B] (rows 0, 1 live)
    static constexpr int B1 = M2 + 8 * 256;               // fp16 planes [4][32 rows][16 B]
    static constexpr int BH = B1 + 4 * 512;               // half2 biases: layers 1..3 [3][16], MLP [32]
    static constexpr int C2 = BH + 80 * 4;                // float [2]: output bias
    static constexpr int GRP = (C2 + 16 + 1023) & ~1023;  // first group block
    // one group's block, offsets from its start
    static constexpr int H1 = 0;                          // fp16 planes [4][kR1][16 B] (h1, then h3)
    static constexpr int HX = H1 + 4 * kR1 * 16;          // the layer-1 input plane [kRX][16 B], then the
                                                          // even/odd h2 planes [2][4][kRE][16 B], then the
                                                          // hidden planes [8][128][16 B]
    static constexpr int HXB = 2 * 4 * kRE * 16;
    static constexpr int XS = HX + HXB;                   // float2 [kP0]: the next tile's input (async copy)
    static constexpr int BAR = XS + kP0 * 8;              // mbarriers, one per row tile of layers 1 and 2, one of the exit
    static constexpr int REC = BAR + 32;                  // uint32 [2 tiles][kWinT][4]: window records being summed
    static constexpr int GROUP = (REC + 2 * kWinT * 16 + 127) & ~127;
    static constexpr int SLOT = GRP + kRxGroups * GROUP;  // tensor-memory base address
    static constexpr int TOTAL = SLOT + 16;
};
static_assert(kRX * 16 <= RxSmem::HXB && 8 * 128 * 16 <= RxSmem::HXB, "aliases of the HX region fit");
static_assert(RxSmem::TOTAL <= 227 * 1024, "one receiver CNN CTA per SM");
static_assert(kMT1 <= 3 && kMT2 <= 3 && kWinT == 2, "one mbarrier per row tile, two windows per tile");
static_assert(2 * (kRE - 4) == kP2, "even / odd h2 rows cover the layer-2 positions");

// barrier of one group's 256 threads (named barrier id, 1 + group); the second form
// also returns whether pred held in every thread of the group
__device__ __forceinline__ void group_sync(int id)
{
    asm volatile("bar.sync %0, %1;" ::"r"(id), "n"(kRxGroupThreads) : "memory");
}
__device__ __forceinline__ bool group_and(int id, bool pred)
{
    uint32_t r;
    asm volatile("{\n .reg .pred q, o;\n setp.ne.u32 q, %1, 0;\n bar.red.and.pred o, %2, %3, q;\n"
                 " selp.u32 %0, 1, 0, o;\n}"
                 : "=r"(r)
                 : "r"((uint32_t)pred), "r"(id), "n"(kRxGroupThreads)
                 : "memory");
    return r != 0;
}

__device__ __forceinline__ uint32_t h2_bits(__half2 h) { return *reinterpret_cast<uint32_t *>(&h); }
__device__ __forceinline__ __half2 bits_h2(uint32_t u) { return *reinterpret_cast<__half2 *>(&u); }

__device__ __forceinline__ uint32_t b2_bits(__nv_bfloat162 h) { return *reinterpret_cast<uint32_t *>(&h); }
__device__ __forceinline__ __nv_bfloat162 bits_b2(uint32_t u) { return *reinterpret_cast<__nv_bfloat162 *>(&u); }

// two FP32 values as one packed 16-bit pair (round to nearest even): FP16 or BF16
template <bool BF>
__device__ __forceinline__ uint32_t pack2(float a, float b)
{
    if constexpr (BF) return b2_bits(__floats2bfloat162_rn(a, b));
    else return h2_bits(__floats2half2_rn(a, b));
}

// bias + GELU of two FP32 accumulators in packed FP16 (tanh form, hardware tanh),
// returned doubled: u = acc + b; t = tanh(u (c0 + c1 u^2)); 2 GELU(u) = u (1 + t) =
// u + u t.  The layers that read these activations take their weights halved, so the
// products they accumulate are those of GELU(u) and the true weights: a factor of two
// commutes with rounding, so the result is that of the undoubled form (BF16; FP16
// where no value is subnormal) at one operation less per pair.
__device__ __forceinline__ uint32_t gelu_h2(uint32_t a, uint32_t b, uint32_t bias)
{
    const __half2 c0 = __float2half2_rn(0.7978845608028654f), c1 = __float2half2_rn(0.7978845608028654f * 0.044715f);
    const __half2 u = __hadd2(__floats2half2_rn(__uint_as_float(a), __uint_as_float(b)), bits_h2(bias));
    const __half2 arg = __hmul2(u, __hfma2(__hmul2(u, u), c1, c0));
    uint32_t th;
    asm("tanh.approx.f16x2 %0, %1;" : "=r"(th) : "r"(h2_bits(arg)));
    return h2_bits(__hfma2(u, bits_h2(th), u));
}
// the same in packed BF16
__device__ __forceinline__ uint32_t gelu_b2(uint32_t a, uint32_t b, uint32_t bias)
{
    const __nv_bfloat162 c0 = __float2bfloat162_rn(0.7978845608028654f),
                         c1 = __float2bfloat162_rn(0.7978845608028654f * 0.044715f);
    const __nv_bfloat162 u = __hadd2(__floats2bfloat162_rn(__uint_as_float(a), __uint_as_float(b)), bits_b2(bias));
    const __nv_bfloat162 arg = __hmul2(u, __hfma2(__hmul2(u, u), c1, c0));
    uint32_t th;
    asm("tanh.approx.bf16x2 %0, %1;" : "=r"(th) : "r"(b2_bits(arg)));
    return b2_bits(__hfma2(u, bits_b2(th), u));
}
template <bool BF>
__device__ __forceinline__ uint32_t gelu2(uint32_t a, uint32_t b, uint32_t bias)
{
    if constexpr (BF) return gelu_b2(a, b, bias);
    else return gelu_h2(a, b, bias);
}

template <bool BF>
__global__ void __launch_bounds__(kRxThreads, 1)
    k_cnn_rx_tc(const float *prm, const float2 *y,
                long long seg_base, long long y_end, int nwin, uint8_t *dec, uint8_t *winb,
                uint4 *winrec, const uint32_t *__restrict__ prbs_bits, long long k_first, float scale,
                int mq, float2 *soft, int *err)
{
    extern __shared__ __align__(16) unsigned char sm[];   // no-swizzle operands: 16-byte rows
    unsigned char *sW2 = sm + RxSmem::W2, *sW3 = sm + RxSmem::W3, *sM1 = sm + RxSmem::M1, *sM2 = sm + RxSmem::M2;
    unsigned char *sB1 = sm + RxSmem::B1;
    uint32_t *bh = reinterpret_cast<uint32_t *>(sm + RxSmem::BH);   // half2 bias pairs
    float *c2 = reinterpret_cast<float *>(sm + RxSmem::C2);
    uint32_t *tslot = reinterpret_cast<uint32_t *>(sm + RxSmem::SLOT);
    const int tid = threadIdx.x, grp = tid / kRxGroupThreads, gtid = tid % kRxGroupThreads;
    const int lane = tid & 31, warp = tid >> 5, gwarp = gtid >> 5, quarter = gwarp & 3, ch = gwarp >> 2;
    const int gbar = 1 + grp;   // the group's named barrier
    unsigned char *gb = sm + RxSmem::GRP + grp * RxSmem::GROUP;
    unsigned char *sH1 = gb + RxSmem::H1, *sHX = gb + RxSmem::HX;
    uint32_t *rec = reinterpret_cast<uint32_t *>(gb + RxSmem::REC);
    float2 *xs = reinterpret_cast<float2 *>(gb + RxSmem::XS);
    uint64_t *bar = reinterpret_cast<uint64_t *>(gb + RxSmem::BAR);
    constexpr int PL1 = kR1 * 16, PLE = kRE * 16, EO = 4 * PLE;

    if (gtid < 4) mbar_init(bar + gtid, 1);
    if (gtid < 2 * kWinT * 4) rec[gtid] = 0;
    __syncwarp();
    if (warp == 0) tmem_alloc(tslot, kRxTmem);
    pdl_wait();
    // weights: B operands as K-major planes (chunk (row n, K column kk) at kk * rows * 16 + n * 16)
    // 8 FP32 weights of a layer that reads GELU outputs -> 16 bytes of FP16 / BF16,
    // halved (the epilogues store 2 GELU(u))
    auto h8 = [&](const float *src) {
        uint32_t w[4];
#pragma unroll
        for (int i = 0; i < 4; i++) w[i] = pack2<BF>(0.5f * src[2 * i], 0.5f * src[2 * i + 1]);
        return make_uint4(w[0], w[1], w[2], w[3]);
    };
    for (int u = tid; u < 36 * 32; u += kRxThreads) {
        int n = u & 31, kk = u >> 5;
        *reinterpret_cast<uint4 *>(sW2 + kk * 512 + n * 16) = h8(prm + OW2 + n * KW + 8 * kk);
        *reinterpret_cast<uint4 *>(sW3 + kk * 512 + n * 16) = h8(prm + OW3 + n * KW + 8 * kk);
    }
    for (int u = tid; u < 4 * CH; u += kRxThreads) {
        int n = u & 63, kk = u >> 6;
        *reinterpret_cast<uint4 *>(sM1 + kk * 1024 + n * 16) = h8(prm + OM1 + n * CC + 8 * kk);
    }
    for (int u = tid; u < 8 * 16; u += kRxThreads) {   // output projection: rows 0, 1 = the two outputs
        int n = u & 15, kk = u >> 4;
        *reinterpret_cast<uint4 *>(sM2 + kk * 256 + n * 16) =
            n < 2 ? h8(prm + OM2 + n * CH + 8 * kk) : make_uint4(0, 0, 0, 0);
    }
    for (int u = tid; u < 4 * 32; u += kRxThreads) {   // layer-1 weights, FP16, K padded to 32
        int n = u & 31, kk = u >> 5;
        uint32_t w[4];
#pragma unroll
        for (int i = 0; i < 4; i++) {
            int k0 = 8 * kk + 2 * i;
            float a = k0 < 18 ? prm[OW1 + n * 18 + k0] : 0.f, b = k0 + 1 < 18 ? prm[OW1 + n * 18 + k0 + 1] : 0.f;
            w[i] = pack2<BF>(a, b);
        }
        *reinterpret_cast<uint4 *>(sB1 + kk * 512 + n * 16) = make_uint4(w[0], w[1], w[2], w[3]);
    }
    for (int i = tid; i < 3 * 16; i += kRxThreads) {
        const int off = (i < 16 ? OB1 : i < 32 ? OB2 : OB3) + 2 * (i & 15);
        bh[i] = pack2<BF>(prm[off], prm[off + 1]);
    }
    for (int i = tid; i < 32; i += kRxThreads) bh[48 + i] = pack2<BF>(prm[OC1 + 2 * i], prm[OC1 + 2 * i + 1]);
    if (tid < 2) c2[tid] = prm[OC2 + tid];
    const int ntiles = (nwin + kWinT - 1) / kWinT;
    const int t0 = (int)blockIdx.x * kRxGroups + grp, tstep = (int)gridDim.x * kRxGroups;
    // a tile's input, copied asynchronously into the group's buffer (zero past the stream end)
    auto prefetch = [&](int t) {
        for (int i = gtid; i < kP0; i += kRxGroupThreads) {
            const long long g = seg_base + 2LL * kTS * t + i;
            cp_async8(xs + i, g < y_end ? y + g : y, g < y_end);
        }
        cp_async_commit();
    };
    if (t0 < ntiles) prefetch(t0);
    // rows past the computed positions are read by the last row tiles: zero once
    for (int i = gtid; i < 4 * kR1; i += kRxGroupThreads)
        *reinterpret_cast<uint4 *>(sH1 + (i / kR1) * PL1 + (i % kR1) * 16) = make_uint4(0, 0, 0, 0);
    fence_async_smem();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tslot + (uint32_t)grp * kRxTmemGroup;   // the group's columns
    constexpr uint32_t kFmt = BF ? 1u : 0u;   // kind::f16 operand format: F16 or BF16
    const uint32_t id16 = umma_idesc(kFmt, 128, 16), id32 = umma_idesc(kFmt, 128, 32), id64 = umma_idesc(kFmt, 128, 64);
    const uint32_t aB1 = smem_u32(sB1), aH1 = smem_u32(sH1), aHX = smem_u32(sHX), aW2 = smem_u32(sW2),
                   aW3 = smem_u32(sW3), aM1 = smem_u32(sM1), aM2 = smem_u32(sM2);
    const uint32_t tq = tmem + ((uint32_t)(32 * quarter) << 16);   // this warp's lane quarter
    // matrix descriptors at the operand bases; an operand offset of o bytes adds o >> 4
    // to the start-address field, so the issue loops add compile-time constants
    const uint64_t dX = umma_sdesc(aHX, 64, 128), dB1 = umma_sdesc(aB1, 512, 128);
    const uint64_t dH1 = umma_sdesc(aH1, PL1, 128), dW2 = umma_sdesc(aW2, 512, 128), dW3 = umma_sdesc(aW3, 512, 128);
    const uint64_t dEO = umma_sdesc(aHX, PLE, 128), dM1 = umma_sdesc(aM1, 1024, 128);
    const uint64_t dHid = umma_sdesc(aHX, 2048, 128), dM2 = umma_sdesc(aM2, 256, 128);
    unsigned phase = 0;   // bit b: phase of mbarrier b
    bool ok = true;

    // wait for the MMAs committed to mbarrier b.  A wait that ran out is flagged and ends the
    // group's loop at its next tile; until then a thread that gave up waits for nothing more,
    // and the issuing one issues nothing more (the others' waits for it run out as well)
    auto wait_mma = [&](int b) {
        if (ok && !mbar_wait(bar + b, (phase >> b) & 1u)) {
            atomicExch(err, (int)RX_ETIMEOUT);
            ok = false;
        }
        phase ^= 1u << b;
        __syncwarp();   // the tensor-memory loads that follow are warp-wide
        tc_fence_after();
    };
    // conv epilogue of row tile m: rows of this warp's lane quarter, channel groups 2 ch and
    // 2 ch + 1 (8 channels each); row -> address of its 16-byte row of channel group cq in
    // the destination
    auto conv_epi = [&](int m, int valid, const uint32_t *bias, auto dst_row) {
        if (128 * m + 32 * quarter >= valid) return;   // warp-uniform
        uint32_t r[16];
        tmem_ld16(tq + 32 * m + 16 * ch, r);
        const int row = 128 * m + 32 * quarter + lane;
        if (row >= valid) return;
#pragma unroll
        for (int c = 0; c < 2; c++) {
            const int cq = 2 * ch + c;
            const uint4 b = *reinterpret_cast<const uint4 *>(bias + 4 * cq);
            const uint32_t *q = r + 8 * c;
            *reinterpret_cast<uint4 *>(dst_row(row, cq)) =
                make_uint4(gelu2<BF>(q[0], q[1], b.x), gelu2<BF>(q[2], q[3], b.y), gelu2<BF>(q[4], q[5], b.z),
                           gelu2<BF>(q[6], q[7], b.w));
        }
    };
    // records of tile t (buffer tp), complete once the group has passed a barrier after it
    auto put_records = [&](int t, int tp) {
        if (gtid < kWinT && kWinT * t + gtid < nwin) {
            uint4 *rc = reinterpret_cast<uint4 *>(rec + 4 * (kWinT * tp + gtid));
            const uint4 v = *rc;
            const int s = kWinT * t + gtid;
            winb[s] = 0;
            winrec[s] = make_uint4(v.x, v.y, v.z, v.w << 8);
            *rc = make_uint4(0, 0, 0, 0);
        }
    };

    const int NB = mq == 2 ? 1 : 2, BPS = 2 * NB;
    int tlast = -1, tp = 0;   // the tile whose records are being summed, and its buffer
    // PRBS position of the tile's first bit, and how far it moves per tile of this group
    int pos_t = (int)((long long)BPS * (k_first + (long long)kTS * t0) % 32767);
    const int pos_step = (int)((long long)BPS * kTS * tstep % 32767);
    for (int t = t0; t < ntiles; t += tstep) {
        // layer-1 input plane: row p = positions p .. p+3 (8 reals) in FP16, zero past kP0
        cp_async_wait_all();
        if (!group_and(gbar, ok)) break;   // the tile's input is in xs
        if (tlast >= 0) put_records(tlast, tp);
        tlast = t;
        tp ^= 1;
        for (int p = gtid; p < kRX; p += kRxGroupThreads) {
            uint32_t w[4];
#pragma unroll
            for (int i = 0; i < 4; i++) {
                const float2 v = p + i < kP0 ? xs[p + i] : make_float2(0.f, 0.f);
                w[i] = pack2<BF>(v.x, v.y);
            }
            *reinterpret_cast<uint4 *>(sHX + p * 16) = make_uint4(w[0], w[1], w[2], w[3]);
        }
        fence_async_smem();
        group_sync(gbar);
        if (t + tstep < ntiles) prefetch(t + tstep);   // lands while this tile computes
        if (gtid == 0 && ok) {
            tc_fence_after();
#pragma unroll
            for (int m = 0; m < kMT1; m++) {
#pragma unroll
                for (int ks = 0; ks < 2; ks++)
                    umma_f16(tmem + 32 * m, dX + (((128 * m + 8 * ks) * 16) >> 4), dB1 + ((2 * ks * 512) >> 4), id32,
                             ks > 0);
                umma_commit(bar + m);
            }
        }
        // the reference bits of this lane's symbol, long before the decisions
        const int js = 32 * quarter + lane;                       // symbol of the tile
        const long long ksym = (long long)kTS * t + js;           // payload symbol
        int ref = 0;
        if (ch == 0 && ksym < 64LL * nwin) {
            int pos = pos_t + BPS * js;
            pos = pos >= 32767 ? pos - 32767 : pos;
            const uint32_t w0 = __ldg(prbs_bits + (pos >> 5)), w1w = __ldg(prbs_bits + (pos >> 5) + 1);
            ref = (int)(__funnelshift_l(w1w, w0, pos & 31) >> (32 - BPS));
        }
        pos_t += pos_step;
        pos_t = pos_t >= 32767 ? pos_t - 32767 : pos_t;
        __syncwarp();
#pragma unroll
        for (int m = 0; m < kMT1; m++) {
            wait_mma(m);
            conv_epi(m, kP1, bh, [&](int row, int cq) { return sH1 + cq * PL1 + row * 16; });
        }
        __syncwarp();
        fence_async_smem();
        tc_fence_before();
        group_sync(gbar);
        // layer 2 (reads h1; the input plane is free): the epilogue of a row tile runs while
        // the MMAs of the next one do
        if (gtid == 0 && ok) {
            tc_fence_after();
#pragma unroll
            for (int m = 0; m < kMT2; m++) {
#pragma unroll
                for (int ks = 0; ks < 18; ks++)
                    umma_f16(tmem + 32 * m, dH1 + (((128 * m + ks / 2) * 16 + 2 * (ks & 1) * PL1) >> 4),
                             dW2 + ((2 * ks * 512) >> 4), id32, ks > 0);
                umma_commit(bar + m);
            }
        }
        __syncwarp();
#pragma unroll
        for (int m = 0; m < kMT2; m++) {
            wait_mma(m);
            conv_epi(m, kP2, bh + 16, [&](int row, int cq) { return sHX + (row & 1) * EO + cq * PLE + (row >> 1) * 16; });
        }
        __syncwarp();
        fence_async_smem();
        tc_fence_before();
        group_sync(gbar);
        // layer 3 at the symbol positions: tap d reads set d & 1 from row j + d / 2
        if (gtid == 0 && ok) {
            tc_fence_after();
#pragma unroll
            for (int ks = 0; ks < 18; ks++) {
                const int d = ks >> 1;
                umma_f16(tmem, dEO + (((d & 1) * EO + (d >> 1) * 16 + 2 * (ks & 1) * PLE) >> 4),
                         dW3 + ((2 * ks * 512) >> 4), id32, ks > 0);
            }
            umma_commit(bar);
        }
        __syncwarp();
        wait_mma(0);
        conv_epi(0, kTS, bh + 32, [&](int row, int cq) { return sH1 + cq * PL1 + row * 16; });   // h3, row = symbol
        __syncwarp();
        fence_async_smem();
        tc_fence_before();
        group_sync(gbar);
        // MLP 32 -> 64 on the symbols (M = 128, N = 64, K = 32)
        if (gtid == 0 && ok) {
            tc_fence_after();
#pragma unroll
            for (int ks = 0; ks < 2; ks++)
                umma_f16(tmem, dH1 + ((2 * ks * PL1) >> 4), dM1 + ((2 * ks * 1024) >> 4), id64, ks > 0);
            umma_commit(bar);
        }
        __syncwarp();
        wait_mma(0);
#pragma unroll
        for (int c = 0; c < 2; c++) {
            // hidden units 16 hq .. + 15 of symbol row -> planes 2 hq, 2 hq + 1 (the h2 planes are free)
            const int hq = 2 * ch + c;
            uint32_t r[16];
            tmem_ld16(tq + 16 * hq, r);
            const int row = 32 * quarter + lane;
            const uint4 b0 = *reinterpret_cast<const uint4 *>(bh + 48 + 8 * hq);
            const uint4 b1 = *reinterpret_cast<const uint4 *>(bh + 48 + 8 * hq + 4);
            *reinterpret_cast<uint4 *>(sHX + (2 * hq) * 2048 + row * 16) =
                make_uint4(gelu2<BF>(r[0], r[1], b0.x), gelu2<BF>(r[2], r[3], b0.y), gelu2<BF>(r[4], r[5], b0.z),
                           gelu2<BF>(r[6], r[7], b0.w));
            *reinterpret_cast<uint4 *>(sHX + (2 * hq + 1) * 2048 + row * 16) =
                make_uint4(gelu2<BF>(r[8], r[9], b1.x), gelu2<BF>(r[10], r[11], b1.y), gelu2<BF>(r[12], r[13], b1.z),
                           gelu2<BF>(r[14], r[15], b1.w));
        }
        fence_async_smem();
        tc_fence_before();
        group_sync(gbar);
        // 64 -> 2 (M = 128, N = 16 with rows 2..15 of B zero, K = 64)
        if (gtid == 0 && ok) {
            tc_fence_after();
#pragma unroll
            for (int ks = 0; ks < 4; ks++)
                umma_f16(tmem + kColOut, dHid + ((2 * ks * 2048) >> 4), dM2 + ((2 * ks * 256) >> 4), id16, ks > 0);
            umma_commit(bar);
        }
        __syncwarp();
        wait_mma(0);
        // decisions and window records: the lanes that hold the outputs decide their symbol,
        // two warps per window; the other warps go on to the next tile's input
        if (ch == 0 && __all_sync(0xffffffffu, ok)) {
            uint32_t r[8];
            tmem_ld8(tq + kColOut, r);
            const float o0 = __uint_as_float(r[0]) + c2[0], o1 = __uint_as_float(r[1]) + c2[1];
            unsigned eA = 0, eB = 0, se = 0, nr = 0;
            if (ksym < 64LL * nwin) {
                if (soft) soft[ksym] = make_float2(o0, o1);
                const float vr = scale * o0, vi = scale * o1;
                int LI = 0, LQ = 0;
                bool near = false;
                for (int jj = 0; jj < mq - 1; jj++) {
                    float th = (float)(2 * jj - (mq - 2));
                    LI += vr >= th;
                    LQ += vi >= th;
                    near |= fabsf(vr - th) < 1e-4f || fabsf(vi - th) < 1e-4f;
                }
                dec[ksym] = (uint8_t)(LI | (LQ << 3) | (near ? 64 : 0));
                // bit errors under the four rotations (qam_window's codes)
                const int cm = mq == 2 ? 1 : 2, gI = LI ^ (LI >> 1), gQ = LQ ^ (LQ >> 1);
                const int X = ((gI << NB) | gQ) ^ ref, Xs = ((gQ << NB) | gI) ^ ref;
                const unsigned n0 = __popc(X), n1 = __popc(Xs ^ cm), n2 = __popc(X ^ ((cm << NB) | cm)),
                               n3 = __popc(Xs ^ (cm << NB));
                eA = n0 + (n1 << 16);
                eB = n2 + (n3 << 16);
                se = (unsigned)(n0 > 0) | ((unsigned)(n1 > 0) << 8) | ((unsigned)(n2 > 0) << 16) |
                     ((unsigned)(n3 > 0) << 24);
                nr = near;
            }
            eA = __reduce_add_sync(0xffffffffu, eA);
            eB = __reduce_add_sync(0xffffffffu, eB);
            se = __reduce_add_sync(0xffffffffu, se);
            nr = __reduce_add_sync(0xffffffffu, nr);
            uint32_t *rw = rec + 4 * (kWinT * tp + (quarter >> 1));
            if (lane < 4) atomicAdd(rw + lane, lane == 0 ? eA : lane == 1 ? eB : lane == 2 ? se : nr);
        }
        tc_fence_before();
    }
    cp_async_wait_all();   // a prefetch may still be in flight after an early exit
    if (group_and(gbar, ok)) {
        if (tlast >= 0) put_records(tlast, tp);
    } else if (gtid == 0) {   // MMAs may still be in flight: wait (bounded) for all this thread issued
        umma_commit(bar + 3);
        mbar_wait(bar + 3, 0);
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) tmem_dealloc(*tslot, kRxTmem);
}

cudaError_t prepare_cnn_rx()
{
    cudaError_t e = cudaFuncSetAttribute(k_cnn_rx_tc<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, RxSmem::TOTAL);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_cnn_rx_tc<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, RxSmem::TOTAL);
    return e;
}

cudaError_t launch_cnn_decide(const float *prm, const float2 *y, long long seg_base, long long y_end,
                              int nwin, uint8_t *dec, uint8_t *winb, uint4 *winrec, const uint32_t *prbs_bits,
                              long long k_first, float scale, int mq, float2 *soft, int *err, int nsm, cudaStream_t st,
                              int bf16, bool pdl)
{
    if (nwin <= 0) return cudaSuccess;
    int ntiles = (nwin + kWinT - 1) / kWinT, nctas = (ntiles + kRxGroups - 1) / kRxGroups;
    unsigned grid = (unsigned)(nctas < nsm ? nctas : nsm);   // one persistent CTA per SM
    return launch_k(bf16 ? k_cnn_rx_tc<true> : k_cnn_rx_tc<false>, grid, kRxThreads, RxSmem::TOTAL, st, pdl, prm, y, seg_base,
                    y_end, nwin, dec, winb, winrec, prbs_bits, k_first, scale, mq, soft, err);
}

}  // namespace rxk

using namespace rxk;

struct rx_cnn {
    int max_seg, nsm;
    float *prm, *grad, *m, *v, *gpart, *lpart, *loss;   // gpart, lpart: gradient and loss of each segment
    __nv_bfloat16 *prm_bf;
    long long step;
};

extern "C" {

int rx_cnn_nparams(void) { return NPRM; }

void rx_cnn_destroy(rx_cnn *c)
{
    if (!c) return;
    void *p[] = {c->prm, c->grad, c->m, c->v, c->gpart, c->lpart, c->loss, c->prm_bf};
    for (void *q : p)
        if (q) cudaFree(q);
    free(c);
}

rx_status rx_cnn_create(int max_seg, rx_cnn **out)
{
    if (!out || max_seg <= 0) return RX_EINVAL;
    *out = nullptr;
    rx_cnn *c = (rx_cnn *)calloc(1, sizeof(rx_cnn));
    if (!c) return RX_ENOMEM;
    c->max_seg = max_seg;
    size_t S = (size_t)max_seg;
    struct {
        void **p;
        size_t b;
    } al[] = {{(void **)&c->prm, NPRM * 4},
              {(void **)&c->grad, NPRM * 4},
              {(void **)&c->m, NPRM * 4},
              {(void **)&c->v, NPRM * 4},
              {(void **)&c->gpart, S * NPRM * 4},
              {(void **)&c->lpart, S * 4},
              {(void **)&c->loss, 16},
              {(void **)&c->prm_bf, NPRM * 2 + 64}};
    for (auto &a : al) {
        if (cudaMalloc(a.p, a.b) != cudaSuccess || cudaMemset(*a.p, 0, a.b) != cudaSuccess) {
            cudaGetLastError();
            rx_cnn_destroy(c);
            return RX_ENOMEM;
        }
    }
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&c->nsm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
        cudaFuncSetAttribute(k_cnn_fwd, cudaFuncAttributeMaxDynamicSharedMemorySize, FwdSmem::TOTAL) != cudaSuccess ||
        cudaFuncSetAttribute(k_cnn_train, cudaFuncAttributeMaxDynamicSharedMemorySize, TrainSmem::TOTAL) != cudaSuccess) {
        cudaGetLastError();
        rx_cnn_destroy(c);
        return RX_ECUDA;
    }
    *out = c;
    return RX_OK;
}

rx_status rx_cnn_set_params(rx_cnn *c, const float *host, int n)
{
    if (!c || !host || n != NPRM) return RX_EINVAL;
    if (cudaMemcpy(c->prm, host, NPRM * 4, cudaMemcpyHostToDevice) != cudaSuccess) return RX_ECUDA;
    cudaMemset(c->m, 0, NPRM * 4);
    cudaMemset(c->v, 0, NPRM * 4);
    c->step = 0;
    k_cnn_tobf<<<(NPRM + 255) / 256, 256>>>(c->prm, c->prm_bf);
    if (cudaDeviceSynchronize() != cudaSuccess) return RX_ECUDA;
    return RX_OK;
}

rx_status rx_cnn_get_params(rx_cnn *c, float *host, int n)
{
    if (!c || !host || n != NPRM) return RX_EINVAL;
    if (cudaMemcpy(host, c->prm, NPRM * 4, cudaMemcpyDeviceToHost) != cudaSuccess) return RX_ECUDA;
    return RX_OK;
}

rx_status rx_cnn_forward(rx_cnn *c, const float *y, const int64_t *seg_start, int nseg, float *out, void *stream)
{
    if (!c || !y || !seg_start || !out || nseg <= 0) return RX_EINVAL;
    const int grid = nseg < kFwPerSm * c->nsm ? nseg : kFwPerSm * c->nsm;   // persistent CTAs
    return launch_k(k_cnn_fwd, grid, kFwThreads, FwdSmem::TOTAL, (cudaStream_t)stream, true, c->prm, c->prm_bf, (const float2 *)y,
                    (const long long *)seg_start, nseg, out) == cudaSuccess
               ? RX_OK
               : RX_ECUDA;
}

rx_status rx_cnn_grad(rx_cnn *c, const float *y, const int64_t *seg_start, const float *tgt, int nseg, float *grad_out,
                      float *loss_out, void *stream)
{
    if (!c || !y || !seg_start || !tgt || nseg <= 0 || nseg > c->max_seg) return RX_EINVAL;
    cudaStream_t st = (cudaStream_t)stream;
    float norm = 1.f / ((float)nseg * CS);
    cudaError_t e = launch_k(k_cnn_train, nseg, kTrThreads, TrainSmem::TOTAL, st, true, c->prm, c->prm_bf, (const float2 *)y,
                             (const long long *)seg_start, tgt, norm, c->gpart, c->lpart);
    // the caller's buffers are written by the reduction itself where they are aligned
    float *go = ((uintptr_t)grad_out & 3) ? nullptr : grad_out, *lo = ((uintptr_t)loss_out & 3) ? nullptr : loss_out;
    if (e == cudaSuccess)
        e = launch_k(k_cnn_reduce, (NPRM + kRedThreads - 1) / kRedThreads + 1, kRedThreads, 0, st, true, c->gpart, c->lpart,
                     nseg, norm, c->grad, go, c->loss, lo);
    if (e == cudaSuccess && grad_out && !go)
        e = cudaMemcpyAsync(grad_out, c->grad, NPRM * 4, cudaMemcpyDeviceToDevice, st);
    if (e == cudaSuccess && loss_out && !lo) e = cudaMemcpyAsync(loss_out, c->loss, 4, cudaMemcpyDeviceToDevice, st);
    return e == cudaSuccess ? RX_OK : RX_ECUDA;
}

rx_status rx_cnn_adam_step(rx_cnn *c, float lr, void *stream)
{
    if (!c || !(lr > 0)) return RX_EINVAL;
    c->step++;
    float b1t = powf(0.9f, (float)c->step), b2t = powf(0.999f, (float)c->step);
    return launch_k(k_cnn_adam, (NPRM + 255) / 256, 256, 0, (cudaStream_t)stream, true, c->prm, c->prm_bf, c->m, c->v, c->grad,
                    lr, b1t, b2t) == cudaSuccess
               ? RX_OK
               : RX_ECUDA;
}

// device pointers of the parameters (for the receiver's CNN path)
const float *rx_cnn_dev_params(const rx_cnn *c) { return c ? c->prm : nullptr; }

}  // extern "C"

// Learned warm start for the pressure solve: a small 3-level encoder/decoder
// CNN (16/32 channels) on BF16 activations and weights with FP32 accumulation,
// trained on the GPU by these kernels (forward, backward-data,
// backward-weight, loss, Adam).  The network maps (b / s, (1/rho) / max) to
// p / s, s the rms of the mean-free right-hand side; the multigrid solve then
// continues from s * (y - mean y) to the requested residual.
//
// Convolutions are implicit GEMMs on the tensor cores (mma.sync m16n8k16,
// BF16 in, FP32 accumulate): an 8 x 16 output tile (M = 128 pixels) per CTA,
// the input tile with its 1-pixel halo and all weights staged in shared
// memory with padded strides (conflict-free fragment loads), K = 9 taps x
// input channels.  Activations are NHWC with channel counts padded to 16.
// The weight gradient is split over pixel chunks and reduced in a fixed
// order, so training is deterministic.
#include <cuda_bf16.h>
#include <math.h>

#include <algorithm>
#include <vector>

#include "ib_internal.cuh"

namespace ibk {
namespace {

using bf16 = __nv_bfloat16;
constexpr int CH = 8, CW = 16;  // conv output tile: 8 rows x 16 columns

__device__ __forceinline__ void mma_bf16(float *d, const uint32_t *a, const uint32_t *b)
{
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 "
        "{%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};\n"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}

// keep each bf16 half of v where the matching half of the mask is > 0
__device__ __forceinline__ uint32_t relu_mask(uint32_t v, uint32_t m)
{
    uint32_t r = 0;
    if ((m & 0x8000u) == 0 && (m & 0x7fffu) != 0) r |= v & 0xffffu;
    if ((m & 0x80000000u) == 0 && (m & 0x7fff0000u) != 0) r |= v & 0xffff0000u;
    return r;
}

// 16-byte asynchronous copy (both addresses 16-byte aligned); src-size 0 writes zeros.
__device__ __forceinline__ void cp_async16(uint32_t sa, const void *gsrc, bool valid)
{
    const int sz = valid ? 16 : 0;
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(sa), "l"(gsrc), "r"(sz));
}
__device__ __forceinline__ void cp_async4(uint32_t sa, const void *gsrc, bool valid)
{
    const int sz = valid ? 4 : 0;
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;\n" ::"r"(sa), "l"(gsrc), "r"(sz));
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;\n" ::"n"(N)); }

// Address of channels [8q, 8q + 8) of the convolution input at pixel
// (bz, gy, gx) (inside the image).  With CUP > 0 the input is the channel
// concatenation up2(xu) ++ x: channels below CUP come from the half-resolution
// tensor xu (nearest upsampling, CUP channels), the rest from x (CIN - CUP
// channels); the concatenated tensor is never stored.
template <int CIN, int CUP>
__device__ __forceinline__ const bf16 *in_chunk(const bf16 *x, const bf16 *xu, int bz, int H, int W,
                                                int gy, int gx, int q)
{
    if (CUP > 0 && q < CUP / 8)
        return xu + (((long)bz * (H / 2) + gy / 2) * (W / 2) + gx / 2) * CUP + 8 * q;
    return x + (((long)bz * H + gy) * W + gx) * (CIN - CUP) + 8 * q - CUP;
}

// Four 8 x 8 BF16 matrices from (lane l gives row l & 7 of matrix l >> 3) or
// to shared memory; ldsm4t transposes them.
__device__ __forceinline__ void ldsm4(uint32_t *r, uint32_t addr)
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];\n"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
}
__device__ __forceinline__ void ldsm4t(uint32_t *r, uint32_t addr)
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];\n"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
}
__device__ __forceinline__ void stsm4(uint32_t addr, const uint32_t *r)
{
    asm volatile("stmatrix.sync.aligned.m8n8.x4.shared.b16 [%0], {%1,%2,%3,%4};\n"
                 ::"r"(addr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]) : "memory");
}

// 8 channels (16 bytes) as floats and back.
__device__ __forceinline__ void unpack8(uint4 v, float *f)
{
    const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int q = 0; q < 4; q++) {
        f[2 * q] = __uint_as_float(w[q] << 16);
        f[2 * q + 1] = __uint_as_float(w[q] & 0xffff0000u);
    }
}
__device__ __forceinline__ uint4 pack8(const float *f)
{
    uint32_t w[4];
#pragma unroll
    for (int q = 0; q < 4; q++) {
        const __nv_bfloat162 h = __floats2bfloat162_rn(f[2 * q], f[2 * q + 1]);
        w[q] = *(const uint32_t *)&h;
    }
    return make_uint4(w[0], w[1], w[2], w[3]);
}
__device__ __forceinline__ uint4 relu_mask8(uint4 v, uint4 m)
{
    return make_uint4(relu_mask(v.x, m.x), relu_mask(v.y, m.y), relu_mask(v.z, m.z), relu_mask(v.w, m.w));
}
// scale * sum of four 8-channel groups, in order, as BF16
__device__ __forceinline__ uint4 sum4(uint4 v0, uint4 v1, uint4 v2, uint4 v3, float scale)
{
    float a[8], f[8];
    unpack8(v0, a);
    unpack8(v1, f);
#pragma unroll
    for (int q = 0; q < 8; q++) a[q] += f[q];
    unpack8(v2, f);
#pragma unroll
    for (int q = 0; q < 8; q++) a[q] += f[q];
    unpack8(v3, f);
#pragma unroll
    for (int q = 0; q < 8; q++) a[q] = (a[q] + f[q]) * scale;
    return pack8(a);
}

// A tile's image, row and column among tw x th tiles an image, advanced by a
// fixed number of tiles without a division per step.
struct TilePos {
    int b, r, c;
    __device__ TilePos(int tl, int tw, int th) { b = tl / (tw * th); const int m = tl - b * tw * th; r = m / tw; c = m - r * tw; }
    __device__ void advance(const TilePos &d, int tw, int th)
    {
        c += d.c; r += d.r; b += d.b;
        if (c >= tw) { c -= tw; r++; }
        if (r >= th) { r -= th; b++; }
    }
};

// What a convolution's epilogue makes of its output tile (plain: y, masked
// where ymask is given).
enum ConvEpi {
    kEpiPlain = 0,
    kEpiPool = 1,   // y, and its 2 x 2 mean into y2 (half resolution)
    kEpiSplit = 2   // gradient of up2(a) ++ b, a of 32 channels: the 2 x 2 sum of
                    // those channels, masked, into y2 (half resolution), the rest into y
};

template <int CIN, int COUT>
struct ConvCfg {
    static constexpr int XS = CIN + 8, WS = 9 * CIN + 8, TP = (CH + 2) * (CW + 2);
    static constexpr int ES = COUT + 8;                      // pitch of an output pixel (values)
    static constexpr bool REGW = CIN * COUT <= 512;          // weight fragments kept in registers
    static constexpr int ST = CIN <= 16 ? 4 : 3;             // stages of the input ring
    static constexpr size_t smem = ((size_t)ST * TP * XS + (size_t)COUT * WS + (size_t)4 * 32 * ES) * 2;
};

// y = act(conv3x3(x) + bias), NHWC, zero padding, with the epilogues above.
// w: [COUT][9][CIN] (tap = 3 dy + dx multiplies x[i + dy - 1, j + dx - 1]).
// Persistent: each CTA stages all weights once, then walks output tiles of
// 8 x 16 pixels; the next tiles' inputs are copied into a ring by cp.async
// while the current one is on the tensor cores.
// CUP > 0: the input is up2(xu) ++ x (see in_chunk).  CST: channels stored of
// x, CIN or 2 (the other channels are zero and neither stored nor copied).
// ymask (NULL: none; the backward-data passes): the ReLU mask of the gradient
// written, so that its readers take it as it is.  y may be NULL with y32,
// which receives channel 0 in FP32.
// Each warp takes two rows of 16 pixels.  The layers are skinny (K = 16 to 64
// a tap, N = 16 to 64) and their bytes few, so the cost is instructions and
// latency: one fragment load (ldmatrix) for four 4-byte reads, the weights'
// fragments in registers where they fit, copies three tiles ahead, addresses
// of a thread's chunks formed once, output tiles through shared memory in
// 16-byte rows with the pooling of the forward pass and the up-sampling fold
// and split of the backward pass done on them there.  With 4-byte fragment
// reads, two buffers and separate pooling and folding launches the layers
// took (us) 25.5 (16 -> 16, 8 x 256^2), 44.9 (48 -> 16), 33.1 (64 -> 32, half
// resolution), 12.6 (32 -> 32, half and quarter) in all; now
// 13, 41, 26 and 10.
template <int CIN, int COUT, int CUP, int CST, int EPI>
__global__ void __launch_bounds__(128)
k_conv_fwd(int B, int H, int W, const bf16 *__restrict__ x, const bf16 *__restrict__ xu,
           const bf16 *__restrict__ ymask,
           const bf16 *__restrict__ w, const float *__restrict__ bias, int relu,
           bf16 *__restrict__ y, bf16 *__restrict__ y2, float *__restrict__ y32)
{
    using C = ConvCfg<CIN, COUT>;
    constexpr int XS = C::XS, WS = C::WS, NT = COUT / 8, TP = C::TP, ES = C::ES, ST = C::ST, KC = CIN / 16;
    static_assert(CIN % 16 == 0 && CUP % 8 == 0 && (CST == CIN - CUP || CST == 2), "channel layout");
    static_assert(EPI != kEpiSplit || COUT > 32, "split outputs");
    extern __shared__ __align__(16) unsigned char conv_sm[];
    bf16 *xs0 = (bf16 *)conv_sm, *ws = xs0 + ST * TP * XS, *es0 = ws + COUT * WS;
    const int tw = (W + CW - 1) / CW, th = (H + CH - 1) / CH, ntiles = B * tw * th;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane >> 2, t4 = lane & 3;
    for (int k = tid; k < COUT * (9 * CIN / 8); k += 128) {
        const int co = k / (9 * CIN / 8), q = k - co * (9 * CIN / 8);
        *(uint4 *)(ws + co * WS + 8 * q) = *(const uint4 *)(w + (long)co * 9 * CIN + 8 * q);
    }
    if (CST == 2)  // the channels that no copy writes
        for (int k = tid; k < ST * TP * XS / 8; k += 128) *(uint4 *)(xs0 + 8 * k) = make_uint4(0u, 0u, 0u, 0u);
    // this thread's chunks of a tile: window row and column, offset from the
    // tile's corner in x (or xu; a tile's corner is even, so the up-sampled
    // part's offset is the same for every tile)
    constexpr int NCH = CST == 2 ? TP : TP * (CIN / 8), PER = (NCH + 127) / 128;
    int go[PER], rc[PER], so[PER];
    unsigned up = 0;
#pragma unroll
    for (int i = 0; i < PER; i++) {
        const int k = tid + 128 * i, pix = CST == 2 ? k : k / (CIN / 8), q = CST == 2 ? 0 : k - pix * (CIN / 8);
        const int r = pix / (CW + 2), c = pix - r * (CW + 2);
        rc[i] = k < NCH ? r | c << 8 : -1;
        so[i] = (pix * XS + 8 * q) * 2;
        if (CST == 2) go[i] = (r * W + c) * 2;
        else if (CUP > 0 && q < CUP / 8) {
            go[i] = (((r - 1) >> 1) * (W / 2) + ((c - 1) >> 1)) * CUP + 8 * q;
            up |= 1u << i;
        } else go[i] = (r * W + c) * CST + 8 * q - CUP;
    }
    const TilePos stride(gridDim.x, tw, th);
    TilePos pi(blockIdx.x, tw, th);  // the next tile to copy
    int ti = blockIdx.x;
    const uint32_t xsa = (uint32_t)__cvta_generic_to_shared(xs0);
    __syncthreads();
    auto issue = [&](int st) {
        if (ti < ntiles) {
            const int ty0 = pi.r * CH, tx0 = pi.c * CW;
            const bf16 *xt = x + (((long)pi.b * H + ty0 - 1) * W + tx0 - 1) * CST;
            const bf16 *ut = CUP > 0 ? xu + (((long)pi.b * (H / 2) + ty0 / 2) * (W / 2) + tx0 / 2) * CUP : nullptr;
            const uint32_t sb = xsa + st * (TP * XS * 2);
#pragma unroll
            for (int i = 0; i < PER; i++) {
                if (PER * 128 > NCH && i == PER - 1 && rc[i] < 0) break;
                const bool in = (unsigned)(ty0 - 1 + (rc[i] & 255)) < (unsigned)H && (unsigned)(tx0 - 1 + (rc[i] >> 8)) < (unsigned)W;
                const bf16 *src = (CUP > 0 && (up >> i & 1u) ? ut : xt) + go[i];
                if (CST == 2) cp_async4(sb + so[i], in ? src : x, in);
                else cp_async16(sb + so[i], in ? src : x, in);
            }
        }
        ti += gridDim.x;
        pi.advance(stride, tw, th);
        cp_async_commit();  // an empty group past the last tile keeps the count
    };
    pdl_enter();  // the weights above are older than the kernel before this one
    for (int k = 0; k < ST - 1; k++) issue(k);
    float bv[2 * NT];  // this lane's biases
#pragma unroll
    for (int nt = 0; nt < NT; nt++) {
        bv[2 * nt] = bias ? bias[nt * 8 + 2 * t4] : 0.0f;
        bv[2 * nt + 1] = bias ? bias[nt * 8 + 2 * t4 + 1] : 0.0f;
    }
    // weight fragments: rows n (co) of 8 k values, two n blocks a load
    const uint32_t wa = (uint32_t)__cvta_generic_to_shared(ws) +
                        (((lane & 7) + (lane >> 4) * 8) * WS + ((lane >> 3) & 1) * 8) * 2;
    uint32_t wr[C::REGW ? 9 * KC * (NT / 2) : 1][4];
    if constexpr (C::REGW) {
#pragma unroll
        for (int t = 0; t < 9 * KC; t++)
#pragma unroll
            for (int n2 = 0; n2 < NT / 2; n2++) ldsm4(wr[t * (NT / 2) + n2], wa + (n2 * 16 * WS + t * 16) * 2);
    }
    const uint32_t xa0 = (uint32_t)__cvta_generic_to_shared(xs0) +
                         ((2 * warp * (CW + 2) + (lane & 7) + ((lane >> 3) & 1) * 8) * XS + (lane >> 4) * 8) * 2;
    bf16 *es = es0 + warp * 32 * ES;
    const uint32_t ea = (uint32_t)__cvta_generic_to_shared(es) +
                        (((lane & 7) + ((lane >> 3) & 1) * 8) * ES + (lane >> 4) * 8) * 2;
    int st = 0;
    TilePos po(blockIdx.x, tw, th);
    for (int tl = blockIdx.x; tl < ntiles; tl += gridDim.x, po.advance(stride, tw, th)) {
        cp_async_wait<ST - 2>();
        __syncthreads();  // this tile's copies are visible; the slot of the one before is free
        issue((st + ST - 1) % ST);
        const uint32_t xa = xa0 + st * (TP * XS * 2);
        st = (st + 1) % ST;
        float acc[2][NT][4];
#pragma unroll
        for (int a = 0; a < 2; a++)
#pragma unroll
            for (int b = 0; b < NT; b++)
#pragma unroll
                for (int q = 0; q < 4; q++) acc[a][b][q] = 0.0f;
        auto step = [&](int tap, int kc, uint32_t xo) {
            uint32_t af[2][4];
#pragma unroll
            for (int mt = 0; mt < 2; mt++) ldsm4(af[mt], xo + (mt * (CW + 2) * XS + kc * 16) * 2);
#pragma unroll
            for (int n2 = 0; n2 < NT / 2; n2++) {
                uint32_t bq[4];
                const uint32_t *bf = bq;
                if constexpr (C::REGW) bf = wr[(tap * KC + kc) * (NT / 2) + n2];
                else ldsm4(bq, wa + (n2 * 16 * WS + tap * CIN + kc * 16) * 2);
#pragma unroll
                for (int mt = 0; mt < 2; mt++) {
                    mma_bf16(acc[mt][2 * n2], af[mt], bf);
                    mma_bf16(acc[mt][2 * n2 + 1], af[mt], bf + 2);
                }
            }
        };
        if constexpr (C::REGW) {
#pragma unroll
            for (int tap = 0; tap < 9; tap++)
#pragma unroll
                for (int kc = 0; kc < KC; kc++)
                    step(tap, kc, xa + ((tap / 3) * (CW + 2) + tap % 3) * (XS * 2));
        } else {
#pragma unroll 1
            for (int tap = 0; tap < 9; tap++) {
                const uint32_t xo = xa + ((tap / 3) * (CW + 2) + tap - 3 * (tap / 3)) * (XS * 2);
#pragma unroll
                for (int kc = 0; kc < KC; kc++) step(tap, kc, xo);
            }
        }
        // epilogue: bias, ReLU, BF16, and through shared memory
        const int oy0 = po.r * CH + 2 * warp, tx0 = po.c * CW;
        const long o0 = ((long)po.b * H + oy0) * W + tx0;                        // first pixel of the warp's rows
        const long h0 = ((long)po.b * (H / 2) + oy0 / 2) * (W / 2) + tx0 / 2;    // the same at half resolution
        __syncwarp();  // the last tile's rows of this warp have been read
#pragma unroll
        for (int nt = 0; nt < NT; nt += 2) {
            const float b0 = bv[2 * nt], b1 = bv[2 * nt + 1], b2 = bv[2 * nt + 2], b3 = bv[2 * nt + 3];
#pragma unroll
            for (int mt = 0; mt < 2; mt++) {
                float v[8] = {acc[mt][nt][0] + b0, acc[mt][nt][1] + b1, acc[mt][nt][2] + b0, acc[mt][nt][3] + b1,
                              acc[mt][nt + 1][0] + b2, acc[mt][nt + 1][1] + b3, acc[mt][nt + 1][2] + b2, acc[mt][nt + 1][3] + b3};
                if (relu)
#pragma unroll
                    for (int q = 0; q < 8; q++) v[q] = fmaxf(v[q], 0.0f);
                if (y32 && nt == 0 && t4 == 0 && oy0 + mt < H) {
                    float *o = y32 + o0 + mt * W + g;
                    if (tx0 + g < W) o[0] = v[0];
                    if (tx0 + g + 8 < W) o[8] = v[2];
                }
                const uint4 pk = pack8(v);
                const uint32_t rg[4] = {pk.x, pk.y, pk.z, pk.w};
                if (y) stsm4(ea + (mt * 16 * ES + nt * 8) * 2, rg);
            }
        }
        if (!y) continue;
        __syncwarp();
        // rows oy0, oy0 + 1: 16 pixels of COUT channels each in es
        constexpr int C8 = COUT / 8;
        if constexpr (EPI == kEpiSplit) {
            constexpr int S8 = C8 - 4;  // chunks of the rest
            {
                const int px = lane >> 2, c = lane & 3, ox = tx0 / 2 + px;
                if (oy0 < H && 2 * ox < W) {
                    const bf16 *e = es + 2 * px * ES + 8 * c;
                    const long o = (h0 + px) * 32 + 8 * c;
                    const uint4 v = sum4(*(const uint4 *)e, *(const uint4 *)(e + ES), *(const uint4 *)(e + 16 * ES),
                                         *(const uint4 *)(e + 17 * ES), 1.0f);
                    *(uint4 *)(y2 + o) = relu_mask8(v, *(const uint4 *)(ymask + o));
                }
            }
#pragma unroll
            for (int k = lane; k < 32 * S8; k += 32) {
                const int px = k / S8, c = k % S8, oy = oy0 + (px >> 4), ox = tx0 + (px & 15);
                if (oy < H && ox < W)
                    *(uint4 *)(y + o0 * (8 * S8) + ((px >> 4) * W + (px & 15)) * (8 * S8) + 8 * c) =
                        *(const uint4 *)(es + px * ES + 32 + 8 * c);
            }
        } else {
#pragma unroll
            for (int k = lane; k < 32 * C8; k += 32) {
                const int px = k / C8, c = k % C8, oy = oy0 + (px >> 4), ox = tx0 + (px & 15);
                if (oy < H && ox < W) {
                    const long o = o0 * COUT + ((px >> 4) * W + (px & 15)) * COUT + 8 * c;
                    uint4 v = *(const uint4 *)(es + px * ES + 8 * c);
                    if (ymask) v = relu_mask8(v, *(const uint4 *)(ymask + o));
                    *(uint4 *)(y + o) = v;
                }
            }
            if constexpr (EPI == kEpiPool) {
                const int px = lane / C8, c = lane % C8, ox = tx0 / 2 + px;
                if (lane < 8 * C8 && oy0 < H && 2 * ox < W) {
                    const bf16 *e = es + 2 * px * ES + 8 * c;
                    *(uint4 *)(y2 + (h0 + px) * COUT + 8 * c) =
                        sum4(*(const uint4 *)e, *(const uint4 *)(e + ES), *(const uint4 *)(e + 16 * ES),
                             *(const uint4 *)(e + 17 * ES), 0.25f);
                }
            }
        }
    }
    cp_async_wait<0>();
}

// ---- fifth-generation tensor cores (tcgen05) --------------------------
// Shared-memory matrix descriptor of a K-major operand without swizzling:
// core matrices of 8 rows x 16 bytes stored as 128 contiguous bytes; lbo =
// byte distance between core matrices adjacent along K, sbo = along M (or
// N); start, lbo, sbo are multiples of 16 (encoded >> 4); bits 46-47 carry
// the descriptor version (1).
__device__ __forceinline__ uint64_t umma_desc(uint32_t saddr, uint32_t lbo, uint32_t sbo)
{
    return (uint64_t)((saddr >> 4) & 0x3FFFu) | ((uint64_t)((lbo >> 4) & 0x3FFFu) << 16) |
           ((uint64_t)((sbo >> 4) & 0x3FFFu) << 32) | (1ull << 46);
}

// Instruction descriptor of kind::f16 with BF16 A and B, FP32 D, both
// operands K-major, no negation or sparsity: D format bits 4-5 (1 = F32), A
// and B format bits 7-9 and 10-12 (1 = BF16), N >> 3 in bits 17-22, M >> 4
// in bits 24-28.
__host__ __device__ constexpr uint32_t umma_idesc_bf16(int M, int N)
{
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

__device__ __forceinline__ unsigned long long cnn_gtimer()
{
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;\n" : "=l"(t));
    return t;
}

// Wait for the phase of a shared-memory barrier with the given parity: true
// once it has completed, false when limit_ns of global time (or 2^26 polls)
// pass first.
__device__ __forceinline__ bool cnn_mbar_wait(unsigned long long *bar, unsigned parity,
                                              unsigned long long limit_ns)
{
    const unsigned a = (unsigned)__cvta_generic_to_shared(bar);
    const unsigned long long t0 = cnn_gtimer();
    for (int it = 0; it < (1 << 26); it++) {
        unsigned done;
        asm volatile("{\n .reg .pred P;\n mbarrier.try_wait.parity.shared::cta.b64 P, [%1], %2;\n"
                     " selp.u32 %0, 1, 0, P;\n}\n" : "=r"(done) : "r"(a), "r"(parity) : "memory");
        if (done) return true;
        if (cnn_gtimer() - t0 > limit_ns) return false;
    }
    return false;
}

// Set by a tensor-core convolution whose completion wait ran out (checked by
// the synchronising network calls).
__device__ int g_cnn_fault = 0;

template <int N>
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t *r);
template <>
__device__ __forceinline__ void tmem_ld32<16>(uint32_t taddr, uint32_t *r)
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,"
                 "%12,%13,%14,%15}, [%16];\n"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]),
                   "=r"(r[6]), "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]),
                   "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
                 : "r"(taddr));
}
template <>
__device__ __forceinline__ void tmem_ld32<32>(uint32_t taddr, uint32_t *r)
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,"
                 "%12,%13,%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,"
                 "%31}, [%32];\n"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]),
                   "=r"(r[6]), "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]),
                   "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]),
                   "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
                   "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]),
                   "=r"(r[30]), "=r"(r[31])
                 : "r"(taddr));
}

constexpr int kTcPix = 128;              // output pixels of a row segment
constexpr int kTcNP = kTcPix + 2;        // input pixels of a staged row (with halo)

template <int CIN, int COUT>
constexpr size_t conv_tc_smem()
{
    return (size_t)(CIN / 8) * 4 * kTcNP * 16 + (size_t)9 * (CIN / 8) * COUT * 16 + 16;
}

// y = act(conv3x3(x) + bias) on the fifth-generation tensor cores.  A work
// unit is a strip of 128 output pixels (a row segment) over rpu rows;
// each output row is an implicit GEMM D[128 x COUT] = sum over the 9 taps
// and 16-channel chunks of A_tap[128 x 16] B_tap[16 x COUT]
// (tcgen05.mma kind::f16, M = 128, N = COUT, K = 16: BF16 operands from
// shared memory, FP32 accumulators in tensor memory), issued by one thread
// and committed to a shared barrier (bounded wait).  Persistent: a CTA
// allocates its accumulator columns and stages all weights once
// ([tap][8-channel plane][cout][8]), then walks units.  Input rows live in a
// ring of four slots, plane by plane (8 channels a plane, 130 pixels at
// 16-byte steps, zero outside the image; channels below CUP from the
// half-resolution xu, nearest up-sampling, as k_conv_fwd): a unit stages
// its first three rows, then one new row per output row while the tensor
// cores work on the previous one, and a tap's A is the
// slot of row r - 1 + dy shifted by dx pixels, so its core matrices (8
// consecutive pixels x 8 channels) are 128 contiguous bytes, 128 bytes apart
// along M and one plane apart along K.  Each warp reads its 32 accumulator
// lanes (one pixel a thread) and writes bias + ReLU as BF16 NHWC (and the
// FP32 channel 0 when y32 is given).  W must be a multiple of 128.  The
// accumulation order (taps, then 16-channel chunks) is k_conv_fwd's.
template <int CIN, int COUT, int CUP>
__global__ void __launch_bounds__(128)
k_conv_tc(int B, int H, int W, int rpu, const bf16 *__restrict__ x, const bf16 *__restrict__ xu,
          const bf16 *__restrict__ w, const float *__restrict__ bias, int relu,
          bf16 *__restrict__ y, float *__restrict__ y32)
{
    static_assert(CIN % 16 == 0 && (COUT == 16 || COUT == 32) && CUP % 8 == 0, "shapes");
    constexpr int KP = CIN / 8;                  // 8-channel planes
    constexpr uint32_t SL = kTcNP * 16;          // bytes of a row slot in a plane
    constexpr uint32_t PL = 4 * SL;              // bytes of an input plane (4 slots)
    constexpr uint32_t WPL = COUT * 16;          // bytes of a weight plane
    extern __shared__ __align__(1024) unsigned char tc_sm[];
    unsigned char *xs = tc_sm;
    unsigned char *wsm = tc_sm + KP * PL;
    unsigned long long *mbar = (unsigned long long *)(wsm + 9 * KP * WPL);
    uint32_t *tslot = (uint32_t *)(mbar + 1);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int segs = W / kTcPix, bands = (H + rpu - 1) / rpu;
    const int units = B * segs * bands;
    if (warp == 0) {
        // 32 accumulator columns (COUT <= 32), the minimum allocation
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n"
                     ::"r"((unsigned)__cvta_generic_to_shared(tslot)), "r"(32u));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::);
    }
    if (tid == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n"
                     ::"r"((unsigned)__cvta_generic_to_shared(mbar)));
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::);
    }
    // weights: [tap][plane][cout][8] from [cout][tap][CIN], 16-byte chunks
    for (int k = tid; k < 9 * KP * COUT; k += 128) {
        const int co = k % COUT, rest = k / COUT, k8 = rest % KP, tap = rest / KP;
        const uint4 v = *(const uint4 *)(w + ((long)co * 9 + tap) * CIN + 8 * k8);
        *(uint4 *)(wsm + ((tap * KP + k8) * COUT + co) * 16) = v;
    }
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    const uint32_t taddr = *tslot;
    const uint32_t xb = (unsigned)__cvta_generic_to_shared(xs);
    const uint32_t wb = (unsigned)__cvta_generic_to_shared(wsm);
    constexpr uint32_t idesc = umma_idesc_bf16(kTcPix, COUT);
    unsigned phase = 0;
    bool fail = false, stuck = false;
    // input row gy of the strip at x0 into ring slot gy & 3
    auto stage = [&](int bz, int gy, int x0) {
        const int slot = gy & 3;
        for (int k = tid; k < kTcNP * KP; k += 128) {
            const int px = k % kTcNP, k8 = k / kTcNP, gx = x0 - 1 + px;
            uint4 v = make_uint4(0u, 0u, 0u, 0u);
            if (gy >= 0 && gy < H && gx >= 0 && gx < W)
                v = *(const uint4 *)in_chunk<CIN, CUP>(x, xu, bz, H, W, gy, gx, k8);
            *(uint4 *)(xs + k8 * PL + slot * SL + px * 16) = v;
        }
    };
    for (int u = blockIdx.x; u < units && !fail; u += gridDim.x) {
        const int seg = u % segs, band = (u / segs) % bands, bz = u / (segs * bands);
        const int x0 = seg * kTcPix, r0 = band * rpu, r1 = min(r0 + rpu, H);
        stage(bz, r0 - 1, x0);
        stage(bz, r0, x0);
        stage(bz, r0 + 1, x0);
        for (int row = r0; row < r1; row++) {
            // the operands, written by the generic proxy, are read by the
            // tensor cores through the async proxy
            asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
            asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
            __syncthreads();
            asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
            if (tid == 0) {
#pragma unroll 1
                for (int tap = 0; tap < 9; tap++) {
                    const int dy = tap / 3, dx = tap - 3 * (tap / 3);
                    const uint32_t a0 = xb + ((row - 1 + dy) & 3) * SL + dx * 16;
#pragma unroll
                    for (int kc = 0; kc < CIN / 16; kc++) {
                        const uint64_t ad = umma_desc(a0 + 2 * kc * PL, PL, 128);
                        const uint64_t bd = umma_desc(wb + (tap * KP + 2 * kc) * WPL, WPL, 128);
                        const unsigned acc = (tap > 0 || kc > 0) ? 1u : 0u;
                        asm volatile("{\n .reg .pred p;\n setp.ne.u32 p, %4, 0;\n"
                                     " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n"
                                     ::"r"(taddr), "l"(ad), "l"(bd), "r"(idesc), "r"(acc));
                    }
                }
                asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n"
                             ::"r"((unsigned)__cvta_generic_to_shared(mbar)) : "memory");
            }
            // the next row's input while the tensor cores work: its slot
            // held row - 2, which no MMA of this row reads
            if (row + 1 < r1) stage(bz, row + 2, x0);
            const bool done = cnn_mbar_wait(mbar, phase, 50000000ull);
            if (__syncthreads_or(!done)) {
                // the MMAs did not complete in 50 ms: report and stop; wait
                // up to 0.5 s more for them before the accumulators are
                // released
                if (tid == 0) atomicExch(&g_cnn_fault, 1);
                stuck = !__syncthreads_and(cnn_mbar_wait(mbar, phase, 500000000ull));
                fail = true;
                break;
            }
            phase ^= 1;
            asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
            uint32_t acc[COUT];
            tmem_ld32<COUT>(taddr + ((uint32_t)(32 * warp) << 16), acc);
            asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
            const long off = (((long)bz * H + row) * W + x0 + 32 * warp + lane) * COUT;
            uint32_t packed[COUT / 2];
#pragma unroll
            for (int c = 0; c < COUT; c += 2) {
                float v0 = __uint_as_float(acc[c]) + bias[c], v1 = __uint_as_float(acc[c + 1]) + bias[c + 1];
                if (relu) { v0 = fmaxf(v0, 0.0f); v1 = fmaxf(v1, 0.0f); }
                if (c == 0 && y32) y32[off / COUT] = v0;
                __nv_bfloat162 b2 = __floats2bfloat162_rn(v0, v1);
                packed[c / 2] = *(uint32_t *)&b2;
            }
#pragma unroll
            for (int q = 0; q < COUT / 8; q++)
                *(uint4 *)(y + off + 8 * q) = make_uint4(packed[4 * q], packed[4 * q + 1],
                                                         packed[4 * q + 2], packed[4 * q + 3]);
            // the accumulators are read before the next row's MMAs overwrite
            // them, and the ring slot of row - 1 before it is restaged
            asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
            __syncthreads();
            asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    // MMAs that never completed leave their columns allocated rather than
    // released under them
    if (warp == 0 && !stuck)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(taddr), "r"(32u));
}

// Work split of k_conv_dw: one CTA for a 16 x 16 block of channels (outputs x
// inputs) and a chunk of tiles; with a single such block (16 -> 16) one CTA
// for each row of taps.  Three warps take the products (three taps each, or
// one), the fourth the bias.
template <int CIN, int COUT>
struct DwSplit {
    static constexpr int NP = CIN / 16, G = (COUT / 16) * NP, DY = G == 1 ? 3 : 1;
    static constexpr int TAPS = DY == 3 ? 1 : 3, T = 128, ST = 4;  // taps a warp, threads, stages
    static constexpr int XS = 24, XR = DY == 3 ? CH : CH + 2;      // pitch (values) of a pixel, rows staged
    static constexpr int XP = XR * (CW + 2), GP = CH * CW;
    static constexpr size_t smem = (size_t)ST * (XP + GP) * XS * 2;
    static constexpr long n = (long)COUT * 9 * CIN + COUT;         // values of a chunk's partial
};

// Partial weight and bias gradients over a chunk of output tiles:
// dW[co][tap][ci] += sum_p g[p][co] x[p + tap][ci], g the (masked) output
// gradient.  Per tap a GEMM with M = COUT, N = CIN, K = pixels, on the tensor
// cores (mma.sync m16n8k16: the products are skinny, 16 channels wide, and
// both operands are stored pixel-major, so the transposing fragment load
// takes them as they lie).  A chunk's tiles (the input tile with its halo and
// the gradient tile, 16 channels of each) are staged once for the CTA's taps
// by cp.async into a ring of four, so that three tiles' copies cover the L2's
// latency.  Each product's pixels are summed in one chain over the chunk, and
// the chunks (64) in order, so the result does not depend on the split.
// What bounds it is that chain and the fragment loads (four a 16-pixel step
// for six products).  One CTA per tap with element-wise fragment reads took
// 325 us (16 -> 16), 528 us (48 -> 16) and 260 us (64 -> 32, half resolution)
// at 8 x 256^2; this takes 45, 71 and 39 us.
template <int CIN, int COUT, int CUP, int CSX, int CSG>
__global__ void __launch_bounds__(128)
k_conv_dw(int B, int H, int W, int tiles_per_chunk, const bf16 *__restrict__ x,
          const bf16 *__restrict__ xu, const bf16 *__restrict__ gy, float *__restrict__ part)
{
    using D = DwSplit<CIN, COUT>;
    constexpr int XS = D::XS, T = D::T, ST = D::ST, XP = D::XP, GP = D::GP, TAPS = D::TAPS;
    extern __shared__ __align__(16) unsigned char conv_sm[];
    bf16 *xs0 = (bf16 *)conv_sm, *gs0 = xs0 + ST * XP * XS;
    // CSX, CSG = 2: only two channels of x or gy are stored, the rest are zero
    // (written here once; no copy touches them)
    if (CSX == 2 || CSG == 2) {
        for (int k = threadIdx.x; k < ST * (XP + GP) * XS / 8; k += T)
            *(uint4 *)(xs0 + 8 * k) = make_uint4(0u, 0u, 0u, 0u);
        __syncthreads();
    }
    const int tw = (W + CW - 1) / CW, th = (H + CH - 1) / CH, ntiles = B * tw * th;
    const int chunk = blockIdx.y, t0 = chunk * tiles_per_chunk, t1 = min(ntiles, t0 + tiles_per_chunk);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t4 = lane & 3;
    const int grp = blockIdx.x / D::DY, dy0 = D::DY == 3 ? blockIdx.x % 3 : 0;
    const int mt = grp / D::NP, np = grp % D::NP;
    const bool bias = np == 0 && (D::DY == 1 || dy0 == 0);
    // this thread's chunks of a tile: pixel (tid / 2 + 64 i), half (tid & 1)
    // of the 16 channels, or pixel tid + 128 i of two stored channels; their
    // offsets from the tile's corner, formed once
    constexpr int XN = CSX == 2 ? 1 : 2, GN = CSG == 2 ? 1 : 2;   // chunks a pixel
    constexpr int XI = (XP * XN + T - 1) / T, GI = (GP * GN) / T;
    const bool up = CUP > 0 && np < CUP / 16;                     // the CTA's channels come from xu
    int xo[XI], xrc[XI], go[GI];
#pragma unroll
    for (int i = 0; i < XI; i++) {
        const int pix = (threadIdx.x + T * i) / XN, q = (threadIdx.x + T * i) % XN;
        const int r = pix / (CW + 2), c = pix - r * (CW + 2);
        xrc[i] = pix < XP ? r | c << 8 : -1;
        if (CSX == 2) xo[i] = (r * W + c) * 2;
        else if (up) xo[i] = (((r - 1) >> 1) * (W / 2) + ((c - 1) >> 1)) * CUP + 16 * np + 8 * q;
        else xo[i] = (r * W + c) * (CIN - CUP) + 16 * np + 8 * q - CUP;
    }
#pragma unroll
    for (int i = 0; i < GI; i++) {
        const int pix = (threadIdx.x + T * i) / GN, q = (threadIdx.x + T * i) % GN;
        go[i] = ((pix / CW) * W + pix % CW) * CSG + (CSG == 2 ? 0 : 16 * mt + 8 * q);
    }
    const uint32_t xsa = (uint32_t)__cvta_generic_to_shared(xs0), gsa = (uint32_t)__cvta_generic_to_shared(gs0);
    TilePos pi(t0, tw, th);
    const TilePos one(1, tw, th);
    int ti = t0;
    auto issue = [&](int st) {
        if (ti < t1) {
            const int ty0 = pi.r * CH, tx0 = pi.c * CW, ys = ty0 + dy0 - 1;
            const bf16 *xt = up ? xu + (((long)pi.b * (H / 2) + ty0 / 2) * (W / 2) + tx0 / 2) * CUP
                                : x + (((long)pi.b * H + ys) * W + tx0 - 1) * (CSX == 2 ? 2 : CIN - CUP);
            const bf16 *gt = gy + (((long)pi.b * H + ty0) * W + tx0) * CSG;
            const uint32_t xd = xsa + st * (XP * XS * 2) + (threadIdx.x / XN * XS + threadIdx.x % XN * 8) * 2;
            const uint32_t gd = gsa + st * (GP * XS * 2) + (threadIdx.x / GN * XS + threadIdx.x % GN * 8) * 2;
#pragma unroll
            for (int i = 0; i < XI; i++) {
                if (XI * T > XP * XN && i == XI - 1 && xrc[i] < 0) break;
                const bool in = (unsigned)(ys + (xrc[i] & 255)) < (unsigned)H && (unsigned)(tx0 - 1 + (xrc[i] >> 8)) < (unsigned)W;
                if (CSX == 2) cp_async4(xd + i * (T / XN) * XS * 2, in ? xt + xo[i] : x, in);
                else cp_async16(xd + i * (T / XN) * XS * 2, in ? xt + xo[i] : x, in);
            }
#pragma unroll
            for (int i = 0; i < GI; i++) {
                const int pix = (threadIdx.x + T * i) / GN;
                const bool in = ty0 + pix / CW < H && tx0 + pix % CW < W;  // beyond the image: no gradient
                if (CSG == 2) cp_async4(gd + i * (T / GN) * XS * 2, in ? gt + go[i] : gy, in);
                else cp_async16(gd + i * (T / GN) * XS * 2, in ? gt + go[i] : gy, in);
            }
        }
        ti++;
        pi.advance(one, tw, th);
        cp_async_commit();  // an empty group past the chunk's end keeps the count
    };
    float acc[TAPS][2][4], accb[4] = {0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll
    for (int t = 0; t < TAPS; t++)
#pragma unroll
        for (int q = 0; q < 8; q++) acc[t][q >> 2][q & 3] = 0.0f;
    // the warp's first tap: row (warp) and column 0, or row dy0 and column (warp)
    const int tap0 = D::DY == 3 ? 3 * dy0 + warp : 3 * warp;
    const int shift = D::DY == 3 ? warp : warp * (CW + 2);
    const uint32_t xa0 = (uint32_t)__cvta_generic_to_shared(xs0) +
                         ((shift + (lane & 7) + ((lane >> 3) & 1) * 8) * XS + (lane >> 4) * 8) * 2;
    const uint32_t ga0 = (uint32_t)__cvta_generic_to_shared(gs0) +
                         (((lane & 7) + (lane >> 4) * 8) * XS + ((lane >> 3) & 1) * 8) * 2;
    for (int k = 0; k < ST - 1; k++) issue(k);
    int st = 0;
    for (int tl = t0; tl < t1; tl++) {
        cp_async_wait<ST - 2>();
        __syncthreads();  // this tile's copies are visible; the slot of the one before is free
        issue((st + ST - 1) % ST);
        if (warp < 3) {
            const uint32_t xa = xa0 + st * (XP * XS * 2), ga = ga0 + st * (GP * XS * 2);
#pragma unroll 4
            for (int r = 0; r < CH; r++) {  // K step = the 16 pixels of output row r
                uint32_t af[4], bf[TAPS][4];
                ldsm4t(af, ga + r * (CW * XS * 2));
#pragma unroll
                for (int t = 0; t < TAPS; t++) ldsm4t(bf[t], xa + (r * (CW + 2) + t) * (XS * 2));
#pragma unroll
                for (int t = 0; t < TAPS; t++) {
                    mma_bf16(acc[t][0], af, bf[t]);
                    mma_bf16(acc[t][1], af, bf[t] + 2);
                }
            }
        } else if (bias) {
            // the gradient's column sums: its product with a matrix of ones
            const uint32_t ga = ga0 + st * (GP * XS * 2), ones[2] = {0x3f803f80u, 0x3f803f80u};
#pragma unroll 4
            for (int r = 0; r < CH; r++) {
                uint32_t af[4];
                ldsm4t(af, ga + r * (CW * XS * 2));
                mma_bf16(accb, af, ones);
            }
        }
        st = (st + 1) % ST;
    }
    // C fragment: rows co (g, g + 8), columns ci (2 t4, 2 t4 + 1)
    float *pw = part + (long)chunk * D::n;
    const int co0 = mt * 16 + g;
    if (warp < 3) {
#pragma unroll
        for (int t = 0; t < TAPS; t++)
#pragma unroll
            for (int b = 0; b < 2; b++) {
                float *o = pw + (long)co0 * 9 * CIN + (tap0 + t) * CIN + np * 16 + b * 8 + 2 * t4;
                *(float2 *)o = make_float2(acc[t][b][0], acc[t][b][1]);
                *(float2 *)(o + 8L * 9 * CIN) = make_float2(acc[t][b][2], acc[t][b][3]);
            }
    } else if (bias && t4 == 0) {
        pw[(long)COUT * 9 * CIN + co0] = accb[0];
        pw[(long)COUT * 9 * CIN + co0 + 8] = accb[2];
    }
}

// Gradients of every parameter from the chunk partials of all layers, in one
// launch: each thread sums the chunks of one value in order and scatters it
// from the padded layout [COP][9][CIP], [COP] into the master one.
constexpr int kLayers = 9, kDwChunks = 64;
struct ReduceArgs {
    const float *part[kLayers];
    float *gw[kLayers], *gb[kLayers];
    int nchunks[kLayers], ci[kLayers], co[kLayers], cip[kLayers], cop[kLayers];
    int first[kLayers + 1];  // first CTA of each layer
};
__global__ void __launch_bounds__(128) k_reduce_grads(const __grid_constant__ ReduceArgs a)
{
    int l = 0;
    while ((int)blockIdx.x >= a.first[l + 1]) l++;
    const int nw = a.cop[l] * 9 * a.cip[l], n = nw + a.cop[l];
    const int e = ((int)blockIdx.x - a.first[l]) * 128 + threadIdx.x;
    if (e >= n) return;
    float s = 0.0f;
    const float *p = a.part[l] + e;
#pragma unroll 16
    for (int c = 0; c < a.nchunks[l]; c++) s += p[(long)c * n];
    if (e < nw) {
        const int co = e / (9 * a.cip[l]), r = e - co * 9 * a.cip[l], tap = r / a.cip[l], i = r - tap * a.cip[l];
        if (co < a.co[l] && i < a.ci[l]) a.gw[l][((long)co * 9 + tap) * a.ci[l] + i] = s;
    } else if (e - nw < a.co[l]) {
        a.gb[l][e - nw] = s;
    }
}

// --- layout helpers (bf16 NHWC), 8 channels (16 bytes) a thread ------------
// 2 x 2 mean after a tcgen05 convolution (the warp-level kernel pools in its
// epilogue).  n8: 8-channel groups of the output (H2 x W2, C channels)
__global__ void __launch_bounds__(256)
k_pool2(int n8, int H2, int W2, int C, const bf16 *__restrict__ x, bf16 *__restrict__ y)
{
    const int k = blockIdx.x * 256 + threadIdx.x;
    if (k >= n8) return;
    const int c8 = C / 8, c = (k % c8) * 8;
    int p = k / c8;
    const int j = p % W2;
    p /= W2;
    const int i = p % H2, b = p / H2, W = 2 * W2;
    const bf16 *a = x + (((long)b * (2 * H2) + 2 * i) * W + 2 * j) * C + c;
    *(uint4 *)(y + 8L * k) = sum4(*(const uint4 *)a, *(const uint4 *)(a + C), *(const uint4 *)(a + (long)W * C),
                                  *(const uint4 *)(a + (long)W * C + C), 0.25f);
}

// gskip = [mask > 0] * (gs + pool2_bwd(gp)), C channels (gp at half
// resolution); may be in place (gskip = gs).  One channel a thread took 38 us
// at 8 x 256^2 (instructions), 8 take 8 us.
__global__ void __launch_bounds__(256)
k_skip_grad(int n8, int H, int W, int C, const bf16 *gs, const bf16 *__restrict__ gp,
            const bf16 *__restrict__ mask, bf16 *gskip)
{
    const int k = blockIdx.x * 256 + threadIdx.x;
    if (k >= n8) return;
    const int c8 = C / 8, c = (k % c8) * 8;
    int p = k / c8;
    const int j = p % W;
    p /= W;
    const int i = p % H, b = p / H;
    float v[8], f[8];
    unpack8(*(const uint4 *)(gs + 8L * k), v);
    unpack8(*(const uint4 *)(gp + (((long)b * (H / 2) + i / 2) * (W / 2) + j / 2) * C + c), f);
#pragma unroll
    for (int q = 0; q < 8; q++) v[q] += 0.25f * f[q];
    *(uint4 *)(gskip + 8L * k) = relu_mask8(pack8(v), *(const uint4 *)(mask + 8L * k));
}

// --- features, loss, output ----------------------------------------------
// Per-sample statistics of the network input, in two launches: partial sums
// over kRedBlocks CTAs per sample, then a fixed-order fold.  One pass gives
// sum (b - b0) and sum (b - b0)^2 with b0 the sample's first value (a shift
// that keeps the variance free of cancellation), and min rho (max(1/rho) is
// 1/min(rho) exactly, IEEE division being monotone).
// stats[kStat * smp + ...]: 0 mean b, 1 s = rms(b - mean) (1 if zero),
// 2 1/s, 3 min rho, 4 1/(s pscale), 5 mean of the network output.
constexpr int kRedBlocks = 256, kStat = 8;

__device__ __forceinline__ void block_fold3(double (*sh)[256], double &a, double &b, double &c, bool cmin)
{
    sh[0][threadIdx.x] = a; sh[1][threadIdx.x] = b; sh[2][threadIdx.x] = c;
    __syncthreads();
    for (int o = 128; o; o >>= 1) {
        if (threadIdx.x < o) {
            sh[0][threadIdx.x] += sh[0][threadIdx.x + o];
            sh[1][threadIdx.x] += sh[1][threadIdx.x + o];
            sh[2][threadIdx.x] = cmin ? fmin(sh[2][threadIdx.x], sh[2][threadIdx.x + o])
                                      : sh[2][threadIdx.x] + sh[2][threadIdx.x + o];
        }
        __syncthreads();
    }
    a = sh[0][0]; b = sh[1][0]; c = sh[2][0];
}

__global__ void __launch_bounds__(256)
k_stats_part(int N2, const double *__restrict__ b, const double *__restrict__ rho,
             double *__restrict__ part)
{
    __shared__ double sh[3][256];
    pdl_enter();
    const int smp = blockIdx.y;
    const double *bb = b + (long)smp * N2, *rr = rho + (long)smp * N2;
    const double b0 = bb[0];
    double sd = 0.0, sq = 0.0, mn = INFINITY;
    for (int k = blockIdx.x * 256 + threadIdx.x; k < N2; k += 256 * kRedBlocks) {
        const double d = bb[k] - b0;
        sd += d; sq += d * d; mn = fmin(mn, rr[k]);
    }
    block_fold3(sh, sd, sq, mn, true);
    if (threadIdx.x == 0) {
        double *o = part + ((long)smp * kRedBlocks + blockIdx.x) * 3;
        o[0] = sd; o[1] = sq; o[2] = mn;
    }
}

__global__ void __launch_bounds__(256)
k_stats_final(int N2, const double *__restrict__ b, const double *__restrict__ part, double pscale,
              double *__restrict__ stats)
{
    __shared__ double sh[3][256];
    pdl_enter();
    const int smp = blockIdx.x;
    double sd = 0.0, sq = 0.0, mn = INFINITY;
    if (threadIdx.x < kRedBlocks) {
        const double *o = part + ((long)smp * kRedBlocks + threadIdx.x) * 3;
        sd = o[0]; sq = o[1]; mn = o[2];
    }
    block_fold3(sh, sd, sq, mn, true);
    if (threadIdx.x == 0) {
        const double md = sd / N2, var = fmax(sq / N2 - md * md, 0.0), r = sqrt(var);
        const double sc = r > 0.0 ? r : 1.0;
        double *st = stats + kStat * smp;
        st[0] = b[(long)smp * N2] + md;
        st[1] = sc;
        st[2] = 1.0 / sc;
        st[3] = mn;
        st[4] = 1.0 / (sc * pscale);
    }
}

// Mean of the network output per sample (partials, then the fold into stats[5]).
__global__ void __launch_bounds__(256)
k_ysum_part(int N2, const float *__restrict__ y32, double *__restrict__ part)
{
    __shared__ double sh[3][256];
    pdl_enter();
    const int smp = blockIdx.y;
    const float *yy = y32 + (long)smp * N2;
    double s = 0.0, z0 = 0.0, z1 = 0.0;
    for (int k = blockIdx.x * 256 + threadIdx.x; k < N2; k += 256 * kRedBlocks) s += (double)yy[k];
    block_fold3(sh, s, z0, z1, false);
    if (threadIdx.x == 0) part[(long)smp * kRedBlocks + blockIdx.x] = s;
}

__global__ void __launch_bounds__(256)
k_ymean_final(int N2, const double *__restrict__ part, double *__restrict__ stats)
{
    __shared__ double sh[3][256];
    pdl_enter();
    double s = threadIdx.x < kRedBlocks ? part[(long)blockIdx.x * kRedBlocks + threadIdx.x] : 0.0;
    double z0 = 0.0, z1 = 0.0;
    block_fold3(sh, s, z0, z1, false);
    if (threadIdx.x == 0) stats[kStat * blockIdx.x + 5] = s / N2;
}

// x[..., 0] = (b - mean)/s, x[..., 1] = (1/rho)/max(1/rho) = min(rho)/rho
// (BF16, rounded from FP32; the first layer's other 14 input channels are
// zero and not stored); and (training)
// t = p / (s pscale), pscale = h^2 c.
__global__ void k_features(long n, int N2, const double *__restrict__ b, const double *__restrict__ rho,
                           const double *__restrict__ p, const double *__restrict__ stats,
                           bf16 *__restrict__ x, float *__restrict__ t)
{
    pdl_enter();
    long k = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n) return;
    const double *st = stats + kStat * (k / N2);
    const float f0 = (float)((b[k] - st[0]) * st[2]);
    const float f1 = (float)st[3] / (float)rho[k];
    __nv_bfloat162 v = __floats2bfloat162_rn(f0, f1);
    *(__nv_bfloat162 *)(x + k * 2) = v;
    if (t) t[k] = (float)(p[k] * st[4]);
}

// Mean-removed squared error per sample: loss partial and the gradient
// 2 d / (B n) minus its mean, written as BF16 channel 0 of two.  Three launches over kLossBlk CTAs a sample, each folding the
// partial sums of the one before in a fixed order: the means; the loss and
// the gradient's mean; the gradient.  (One CTA a sample: 288 us at 8 x 256^2
// on 8 of the SMs; this takes 8 us.)
constexpr int kLossBlk = 32;
__device__ __forceinline__ float2 block_sum2(float2 v)
{
    __shared__ float2 sh[8];
#pragma unroll
    for (int o = 16; o; o >>= 1) {
        v.x += __shfl_xor_sync(0xffffffffu, v.x, o);
        v.y += __shfl_xor_sync(0xffffffffu, v.y, o);
    }
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
    __syncthreads();
    v = sh[0];
#pragma unroll
    for (int w = 1; w < 8; w++) { v.x += sh[w].x; v.y += sh[w].y; }
    return v;
}
__device__ __forceinline__ float2 fold_parts(const float2 *part)
{
    float2 v = part[threadIdx.x & 31];  // kLossBlk = 32 partials, every warp the same tree
#pragma unroll
    for (int o = 16; o; o >>= 1) {
        v.x += __shfl_xor_sync(0xffffffffu, v.x, o);
        v.y += __shfl_xor_sync(0xffffffffu, v.y, o);
    }
    return v;
}
__global__ void __launch_bounds__(256)
k_loss_means(int N2, const float *__restrict__ y32, const float *__restrict__ t, float2 *__restrict__ part)
{
    const long base = (long)blockIdx.y * N2;
    float2 s = make_float2(0.0f, 0.0f);
    for (int k = blockIdx.x * 256 + threadIdx.x; k < N2; k += 256 * kLossBlk) {
        s.x += y32[base + k];
        s.y += t[base + k];
    }
    s = block_sum2(s);
    if (threadIdx.x == 0) part[blockIdx.y * kLossBlk + blockIdx.x] = s;
}
__global__ void __launch_bounds__(256)
k_loss_sums(int N2, float sc, const float *__restrict__ y32, const float *__restrict__ t,
            const float2 *__restrict__ means, float2 *__restrict__ part)
{
    const float2 m = fold_parts(means + blockIdx.y * kLossBlk);
    const float my = m.x / N2, mt = m.y / N2;
    const long base = (long)blockIdx.y * N2;
    float2 s = make_float2(0.0f, 0.0f);
    for (int k = blockIdx.x * 256 + threadIdx.x; k < N2; k += 256 * kLossBlk) {
        const float d = (y32[base + k] - my) - (t[base + k] - mt);
        s.x += d * d;
        s.y += sc * d;
    }
    s = block_sum2(s);
    if (threadIdx.x == 0) part[blockIdx.y * kLossBlk + blockIdx.x] = s;
}
__global__ void __launch_bounds__(256)
k_loss_grad(int N2, int Bn, float sc, const float *__restrict__ y32, const float *__restrict__ t,
            const float2 *__restrict__ means, const float2 *__restrict__ sums, bf16 *__restrict__ gy,
            float *__restrict__ lsum)
{
    const float2 m = fold_parts(means + blockIdx.y * kLossBlk), s = fold_parts(sums + blockIdx.y * kLossBlk);
    const float my = m.x / N2, mt = m.y / N2, gmean = s.y / N2;
    const long base = (long)blockIdx.y * N2;
    for (int k = blockIdx.x * 256 + threadIdx.x; k < N2; k += 256 * kLossBlk) {
        const float d = (y32[base + k] - my) - (t[base + k] - mt);
        const __nv_bfloat162 v = __floats2bfloat162_rn(sc * d - gmean, 0.0f);
        *(__nv_bfloat162 *)(gy + (base + k) * 2) = v;
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) lsum[blockIdx.y] = s.x / ((float)Bn * (float)N2);
}

// p0 = s pscale (y - mean y), FP64 out.
__global__ void k_output(long n, int N2, const float *__restrict__ y32, const double *__restrict__ stats,
                         double pscale, double *__restrict__ p0)
{
    pdl_enter();
    const long k = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n) return;
    const double *st = stats + kStat * (k / N2);
    p0[k] = st[1] * pscale * ((double)y32[k] - st[5]);
}

// 2x2 mean of B samples of (2 Nc) x (2 Nc) into Nc x Nc.
__global__ void k_restrict2(long nc, int Nc, const double *__restrict__ in, double *__restrict__ out)
{
    const long k = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= nc) return;
    const long N2c = (long)Nc * Nc, smp = k / N2c;
    const int r = (int)(k - smp * N2c), J = r / Nc, I = r - J * Nc, N = 2 * Nc;
    const double *a = in + smp * 4 * N2c + (long)(2 * J) * N + 2 * I;
    out[k] = 0.25 * (a[0] + a[1] + a[N] + a[N + 1]);
}

// Cell-centred bilinear interpolation (9, 3, 3, 1)/16 of Nc x Nc samples to
// (2 Nc) x (2 Nc), zero-gradient at the walls.
__global__ void k_prolong2(long nf, int Nc, const double *__restrict__ ec, double *__restrict__ ef)
{
    const long k = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= nf) return;
    const int N = 2 * Nc;
    const long N2 = (long)N * N, smp = k / N2;
    const int r = (int)(k - smp * N2), j = r / N, i = r - j * N;
    const int I = i >> 1, J = j >> 1;
    const int I2 = min(max(I + ((i & 1) ? 1 : -1), 0), Nc - 1);
    const int J2 = min(max(J + ((j & 1) ? 1 : -1), 0), Nc - 1);
    const double *c = ec + smp * (long)Nc * Nc;
    ef[k] = (9.0 * c[J * Nc + I] + 3.0 * c[J * Nc + I2] + 3.0 * c[J2 * Nc + I] + c[J2 * Nc + I2]) *
            0.0625;
}

// Adam with bias correction on FP32 master weights.
__global__ void k_adam(long n, float *__restrict__ w, float *__restrict__ m, float *__restrict__ v,
                       const float *__restrict__ g, float lr, float b1, float b2, float eps,
                       float c1, float c2)
{
    long k = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n) return;
    const float gk = g[k];
    const float mk = b1 * m[k] + (1.0f - b1) * gk, vk = b2 * v[k] + (1.0f - b2) * gk * gk;
    m[k] = mk;
    v[k] = vk;
    w[k] -= lr * (mk / c1) / (sqrtf(vk / c2) + eps);
}

// Master [co][3][3][ci] FP32 -> forward BF16 [COP][9][CIP] (zero padded) and
// backward-data BF16 [CIP][9][COP] with the taps flipped.
__global__ void k_pack(int ci, int co, int cip, int cop, const float *__restrict__ w,
                       bf16 *__restrict__ wf, bf16 *__restrict__ wb)
{
    int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= cop * 9 * cip) return;
    const int o = k / (9 * cip), r = k - o * 9 * cip, tap = r / cip, i = r - tap * cip;
    const float v = (o < co && i < ci) ? w[((long)o * 9 + tap) * ci + i] : 0.0f;
    wf[k] = __float2bfloat16_rn(v);
    if (wb) wb[((long)i * 9 + (8 - tap)) * cop + o] = __float2bfloat16_rn(v);
}

}  // namespace

// rms of (a - mean a) of each sample (one CTA per sample, fixed order: the
// mean first, then the squared deviations).
__global__ void __launch_bounds__(256) k_sample_rms(int N2, const double *__restrict__ a,
                                                    double *__restrict__ out)
{
    __shared__ double sh[256];
    const double *x = a + (long)blockIdx.x * N2;
    double t = 0.0;
    for (int k = threadIdx.x; k < N2; k += 256) t += x[k];
    sh[threadIdx.x] = t;
    __syncthreads();
    for (int o = 128; o; o >>= 1) {
        if (threadIdx.x < o) sh[threadIdx.x] += sh[threadIdx.x + o];
        __syncthreads();
    }
    const double m = sh[0] / N2;
    __syncthreads();
    double q = 0.0;
    for (int k = threadIdx.x; k < N2; k += 256) {
        const double d = x[k] - m;
        q += d * d;
    }
    sh[threadIdx.x] = q;
    __syncthreads();
    for (int o = 128; o; o >>= 1) {
        if (threadIdx.x < o) sh[threadIdx.x] += sh[threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0) out[blockIdx.x] = sqrt(sh[0] / N2);
}

// Mini-batch gather: sample idx[i] of each set into slot i.
__global__ void k_gather3(long n, int N2, const int *__restrict__ idx, const double *__restrict__ a,
                          const double *__restrict__ b, const double *__restrict__ c,
                          double *__restrict__ ga, double *__restrict__ gb, double *__restrict__ gc)
{
    const long k = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n) return;
    const long src = (long)idx[k / N2] * N2 + k % N2;
    ga[k] = a[src];
    gb[k] = b[src];
    gc[k] = c[src];
}

// The batch loss (sum of the per-sample partials, in order) into out.
__global__ void k_loss_record(int B, const float *__restrict__ lsum, float *__restrict__ out)
{
    if (threadIdx.x != 0) return;
    float t = 0.0f;
    for (int b = 0; b < B; b++) t += lsum[b];
    *out = t;
}

// ======================================================================= host
struct CnnLayer {
    int ci, co, cip, cop;     // real and padded channel counts
    bool relu;
    size_t woff, boff;        // offsets in the flat FP32 parameter vector
    size_t part_off = 0;      // chunk partials of the gradients ([COP][9][CIP], [COP] a chunk)
    bf16 *wf = nullptr, *wb = nullptr;
};

struct Cnn {
    int c1 = 16, c2 = 32;
    std::vector<CnnLayer> L;
    size_t nparam = 0;
    float *w = nullptr, *m = nullptr, *v = nullptr, *g = nullptr;  // flat FP32
    void *wmem = nullptr;
    int step = 0;
    int tc = 1;               // forward convolutions on tcgen05: 0 none, 1 where faster, 2 all that fit
    double out_scale = 1.0;   // c in the pressure scale s h^2 c
    // activation workspace, sized for B x N x N
    int capB = 0, capN = 0;
    void *amem = nullptr;
    bf16 *x = nullptr, *a1 = nullptr, *s1 = nullptr, *p1 = nullptr, *a2 = nullptr, *s2 = nullptr,
         *p2 = nullptr, *a3 = nullptr, *t3 = nullptr, *t4 = nullptr,
         *a5 = nullptr, *y = nullptr, *gbig = nullptr, *gbig2 = nullptr,
         *gmid = nullptr, *gmid2 = nullptr, *gsmall = nullptr, *gsmall2 = nullptr, *gcat = nullptr,
         *gup = nullptr;
    float *y32 = nullptr, *t = nullptr, *lsum = nullptr, *part = nullptr;
    double *stats = nullptr, *rpart = nullptr;
    // the weight gradients' streams (see cnn_backward), one event per layer's
    // output gradient and one per weight gradient
    static constexpr int kSide = 3;
    cudaStream_t side[kSide] = {};
    cudaEvent_t ev_gy[9] = {}, ev_dw[9] = {};
    // coarse-grid inference: restricted inputs and prolongated outputs
    double *cbuf = nullptr;
    size_t cbuf_cap = 0;
};

namespace {

int g_sms = 0;

int sm_count()
{
    if (!g_sms) {
        int dev = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&g_sms, cudaDevAttrMultiProcessorCount, dev);
        if (g_sms <= 0) g_sms = 152;
    }
    return g_sms;
}

// tc: 0, 1 the warp-level kernel; 2 tcgen05 wherever the width is a multiple
// of 128 (forward layers; bound by operand staging and latency, where the
// warp-level kernel's ring of 8 x 16 tiles stages less per output: 16 -> 32
// channels at 8 x 128^2 take 18.7 us there, 10.4 us here).
// ymask: mask of the output (backward-data passes), NULL for none.
template <int CIN, int COUT, int CUP = 0, int CST = CIN - CUP, int EPI = kEpiPlain>
void conv_launch(int B, int H, int W, const bf16 *x, const bf16 *xu, const bf16 *ymask, const bf16 *w,
                 const float *bias, int relu, bf16 *y, bf16 *y2, float *y32, cudaStream_t s, int tc = 0,
                 bool pdl = false)
{
    if constexpr ((COUT == 16 || COUT == 32) && CST == CIN - CUP && EPI != kEpiSplit) {
        if (tc == 2 && y && W % kTcPix == 0) {
            constexpr size_t smt = conv_tc_smem<CIN, COUT>();
            raise_smem_limit((const void *)k_conv_tc<CIN, COUT, CUP>, (int)smt);
            // rows per unit: as many as keep every SM busy, up to 8 (a unit
            // stages rpu + 2 input rows for rpu output rows); CTAs per SM by
            // shared memory (at most 8: 256 of the 512 tensor-memory columns)
            const int per_sm = std::max(1, std::min(8, (int)((227 * 1024) / smt)));
            const long rows = (long)B * H * (W / kTcPix);
            const int rpu = (int)std::max(1L, std::min(std::min((long)H, 8L), rows / sm_count()));
            const long units = (long)B * (W / kTcPix) * ((H + rpu - 1) / rpu);
            const int grid = (int)std::min(units, (long)sm_count() * per_sm);
            note_launch();
            k_conv_tc<CIN, COUT, CUP><<<grid, 128, smt, s>>>(B, H, W, rpu, x, xu, w, bias, relu, y, y32);
            if (EPI == kEpiPool) {
                const int n8 = B * (H / 2) * (W / 2) * (COUT / 8);
                note_launch();
                k_pool2<<<cdiv(n8, 256), 256, 0, s>>>(n8, H / 2, W / 2, COUT, y, y2);
            }
            return;
        }
    }
    constexpr size_t sm = ConvCfg<CIN, COUT>::smem;
    raise_smem_limit((const void *)k_conv_fwd<CIN, COUT, CUP, CST, EPI>, (int)sm);
    const int ntiles = B * (int)cdiv(W, CW) * (int)cdiv(H, CH);
    const int per_sm = std::max(1, std::min(5, (int)((227 * 1024) / (sm + 1024))));
    const int grid = std::min(ntiles, sm_count() * per_sm);
    note_launch();
    if (pdl)
        launch_pdl(k_conv_fwd<CIN, COUT, CUP, CST, EPI>, grid, 128, sm, s, B, H, W, x, xu, ymask, w, bias, relu, y, y2, y32);
    else
        k_conv_fwd<CIN, COUT, CUP, CST, EPI><<<grid, 128, sm, s>>>(B, H, W, x, xu, ymask, w, bias, relu, y, y2, y32);
}

// Partial gradients of layer k (input x, or up2(xu) ++ x; gy its masked
// output gradient); records the chunk count for k_reduce_grads.
template <int CIN, int COUT, int CUP = 0, int CSX = CIN - CUP, int CSG = COUT>
void conv_dw(Cnn &n, ReduceArgs &ra, int k, int B, int H, int W, const bf16 *x, const bf16 *gy,
             cudaStream_t s, const bf16 *xu = nullptr)
{
    using D = DwSplit<CIN, COUT>;
    const int ntiles = B * (int)cdiv(W, CW) * (int)cdiv(H, CH);
    const int nchunks = std::min(ntiles, kDwChunks), tpc = (int)cdiv(ntiles, nchunks);
    raise_smem_limit((const void *)k_conv_dw<CIN, COUT, CUP, CSX, CSG>, (int)D::smem);
    ra.part[k] = n.part + n.L[k].part_off;
    ra.nchunks[k] = nchunks;
    note_launch();
    k_conv_dw<CIN, COUT, CUP, CSX, CSG><<<dim3(D::G * D::DY, nchunks), D::T, D::smem, s>>>(B, H, W, tpc, x, xu, gy, n.part + n.L[k].part_off);
}

size_t al(size_t b) { return (b + 255) & ~(size_t)255; }

}  // namespace

Cnn *cnn_new(int c1, int c2, unsigned long long seed, cudaStream_t s, cudaError_t *err)
{
    (void)s;
    Cnn *n = new Cnn();
    n->c1 = c1;
    n->c2 = c2;
    auto pad = [](int c) { return (c + 15) / 16 * 16; };
    const int spec[9][3] = {{2, c1, 1}, {c1, c1, 1}, {c1, c2, 1}, {c2, c2, 1}, {c2, c2, 1},
                            {c2, c2, 1}, {2 * c2, c2, 1}, {c2 + c1, c1, 1}, {c1, 1, 0}};
    size_t off = 0;
    for (auto &sp : spec) {
        CnnLayer l;
        l.ci = sp[0]; l.co = sp[1]; l.relu = sp[2] != 0;
        l.cip = pad(l.ci); l.cop = pad(l.co);
        l.woff = off; off += (size_t)l.co * 9 * l.ci;
        l.boff = off; off += (size_t)l.co;
        n->L.push_back(l);
    }
    n->nparam = off;
    size_t bytes = al(off * 4) * 4;
    for (auto &l : n->L) bytes += 2 * al((size_t)l.cop * 9 * l.cip * 2);
    *err = cudaMalloc(&n->wmem, bytes);
    if (*err != cudaSuccess) { n->wmem = nullptr; cnn_free(n); return nullptr; }
    char *q = (char *)n->wmem;
    auto take = [&](size_t b) { char *r = q; q += al(b); return (void *)r; };
    n->w = (float *)take(off * 4); n->m = (float *)take(off * 4);
    n->v = (float *)take(off * 4); n->g = (float *)take(off * 4);
    for (auto &l : n->L) {
        l.wf = (bf16 *)take((size_t)l.cop * 9 * l.cip * 2);
        l.wb = (bf16 *)take((size_t)l.cop * 9 * l.cip * 2);
    }
    // He-normal initial weights (Box-Muller on a splitmix64 stream), zero biases
    std::vector<float> h(off, 0.0f);
    unsigned long long st = seed ^ 0x9E3779B97F4A7C15ULL;
    auto next = [&]() {
        st += 0x9E3779B97F4A7C15ULL;
        unsigned long long z = st;
        z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ULL;
        z = (z ^ (z >> 27)) * 0x94D049BB133111EBULL;
        return (double)((z ^ (z >> 31)) >> 11) * (1.0 / 9007199254740992.0);
    };
    for (auto &l : n->L) {
        const double sd = sqrt(2.0 / (9.0 * l.ci));
        for (size_t k = 0; k < (size_t)l.co * 9 * l.ci; k++) {
            double u1 = next(), u2 = next();
            if (u1 < 1e-300) u1 = 1e-300;
            h[l.woff + k] = (float)(sd * sqrt(-2.0 * log(u1)) * cos(6.283185307179586 * u2));
        }
    }
    *err = cudaMemcpy(n->w, h.data(), off * 4, cudaMemcpyHostToDevice);
    if (*err == cudaSuccess) *err = cudaMemset(n->m, 0, off * 4 * 3);
    for (auto &q : n->side)
        if (*err == cudaSuccess) *err = cudaStreamCreateWithFlags(&q, cudaStreamNonBlocking);
    for (int k = 0; k < kLayers; k++) {
        if (*err == cudaSuccess) *err = cudaEventCreateWithFlags(&n->ev_gy[k], cudaEventDisableTiming);
        if (*err == cudaSuccess) *err = cudaEventCreateWithFlags(&n->ev_dw[k], cudaEventDisableTiming);
    }
    if (*err != cudaSuccess) { cnn_free(n); return nullptr; }
    return n;
}

void cnn_free(Cnn *n)
{
    if (!n) return;
    if (n->wmem) cudaFree(n->wmem);
    if (n->amem) cudaFree(n->amem);
    if (n->cbuf) cudaFree(n->cbuf);
    for (auto &q : n->side)
        if (q) cudaStreamDestroy(q);
    for (int k = 0; k < kLayers; k++) {
        if (n->ev_gy[k]) cudaEventDestroy(n->ev_gy[k]);
        if (n->ev_dw[k]) cudaEventDestroy(n->ev_dw[k]);
    }
    delete n;
}

cudaError_t cnn_pack(Cnn &n, cudaStream_t s)
{
    for (auto &l : n.L) {
        int tot = l.cop * 9 * l.cip;
        note_launch();
        k_pack<<<cdiv(tot, 256), 256, 0, s>>>(l.ci, l.co, l.cip, l.cop, n.w + l.woff, l.wf, l.wb);
    }
    return cudaGetLastError();
}

cudaError_t cnn_workspace(Cnn &n, int B, int N)
{
    if (B <= n.capB && N <= n.capN && n.amem) return cudaSuccess;
    if (n.amem) cudaFree(n.amem);
    n.amem = nullptr;
    const size_t P = (size_t)B * N * N, P2 = P / 4, P4 = P / 16;
    const int c1 = n.c1, c2 = n.c2;
    size_t bytes = al(P * 2 * 2) +                        // x
                   al(P * c1 * 2) * 2 +                    // a1, s1
                   al(P2 * c1 * 2) + al(P2 * c2 * 2) * 2 + // p1, a2, s2
                   al(P4 * c2 * 2) * 3 +                   // p2, a3, t3
                   al(P2 * c2 * 2) +                       // t4
                   al(P * c1 * 2) + al(P * 16 * 2) +       // a5, y
                   al(P * c1 * 2) * 2 + al(P2 * c2 * 2) * 2 + al(P4 * c2 * 2) * 2 +  // grads
                   al(P * c1 * 2) + al(P2 * c2 * 2) +      // gcat, gup (skip parts)
                   al(P * 4) + al(P * 4) + al(B * 4) + al(B * kStat * 8) +
                   al(B * kRedBlocks * 3 * 8);
    // chunk partials of the weight gradients, layer after layer
    size_t part = 0;
    for (auto &l : n.L) {
        l.part_off = part;
        part += (size_t)kDwChunks * ((size_t)l.cop * 9 * l.cip + l.cop);
    }
    bytes += al(part * 4);
    cudaError_t e = cudaMalloc(&n.amem, bytes);
    if (e != cudaSuccess) { n.amem = nullptr; return e; }
    char *q = (char *)n.amem;
    auto take = [&](size_t b) { char *r = q; q += al(b); return (void *)r; };
    n.x = (bf16 *)take(P * 2 * 2);
    n.a1 = (bf16 *)take(P * c1 * 2); n.s1 = (bf16 *)take(P * c1 * 2);
    n.p1 = (bf16 *)take(P2 * c1 * 2); n.a2 = (bf16 *)take(P2 * c2 * 2); n.s2 = (bf16 *)take(P2 * c2 * 2);
    n.p2 = (bf16 *)take(P4 * c2 * 2); n.a3 = (bf16 *)take(P4 * c2 * 2); n.t3 = (bf16 *)take(P4 * c2 * 2);
    n.t4 = (bf16 *)take(P2 * c2 * 2);
    n.a5 = (bf16 *)take(P * c1 * 2);
    n.y = (bf16 *)take(P * 16 * 2);
    n.gbig = (bf16 *)take(P * c1 * 2); n.gbig2 = (bf16 *)take(P * c1 * 2);
    n.gmid = (bf16 *)take(P2 * c2 * 2); n.gmid2 = (bf16 *)take(P2 * c2 * 2);
    n.gsmall = (bf16 *)take(P4 * c2 * 2); n.gsmall2 = (bf16 *)take(P4 * c2 * 2);
    n.gcat = (bf16 *)take(P * c1 * 2); n.gup = (bf16 *)take(P2 * c2 * 2);
    n.y32 = (float *)take(P * 4); n.t = (float *)take(P * 4); n.lsum = (float *)take(B * 4);
    n.stats = (double *)take(B * kStat * 8);
    n.rpart = (double *)take(B * kRedBlocks * 3 * 8);
    n.part = (float *)take(part * 4);
    n.capB = B;
    n.capN = N;
    return cudaSuccess;
}

// Forward pass on B samples of N x N (N a multiple of 4).  Fills the
// activation workspace; y32 holds the FP32 output (one channel).  Programmatic
// launches: a layer's weights are staged while the layer before drains
// (inference at 512^2: 130 us by plain launches, 117 so; gradients at 8 x 256^2
// 615 and 576).  Not in the backward pass, whose
// waiting CTAs would hold the slots of the weight gradients beside them.
void cnn_forward(Cnn &n, int B, int N, double h, const double *rhs, const double *rho,
                 const double *p, cudaStream_t s)
{
    const int N2 = N * N, H2 = N / 2, H4 = N / 4;
    const long P = (long)B * N2;
    note_launch();
    launch_pdl(k_stats_part, dim3(kRedBlocks, B), 256, 0, s, N2, rhs, rho, n.rpart);
    note_launch();
    launch_pdl(k_stats_final, B, 256, 0, s, N2, rhs, n.rpart, h * h * n.out_scale, n.stats);
    note_launch();
    launch_pdl(k_features, cdiv(P, 256), 256, 0, s, P, N2, rhs, rho, p, n.stats, n.x, p ? n.t : nullptr);
    auto &L = n.L;
    auto bias = [&](int k) { return n.w + L[k].boff; };
    const int tc = n.tc;
    conv_launch<16, 16, 0, 2>(B, N, N, n.x, nullptr, nullptr, L[0].wf, bias(0), 1, n.a1, nullptr, nullptr, s, tc, true);
    conv_launch<16, 16, 0, 16, kEpiPool>(B, N, N, n.a1, nullptr, nullptr, L[1].wf, bias(1), 1, n.s1, n.p1, nullptr, s, tc, true);
    conv_launch<16, 32>(B, H2, H2, n.p1, nullptr, nullptr, L[2].wf, bias(2), 1, n.a2, nullptr, nullptr, s, tc, true);
    conv_launch<32, 32, 0, 32, kEpiPool>(B, H2, H2, n.a2, nullptr, nullptr, L[3].wf, bias(3), 1, n.s2, n.p2, nullptr, s, tc, true);
    conv_launch<32, 32>(B, H4, H4, n.p2, nullptr, nullptr, L[4].wf, bias(4), 1, n.a3, nullptr, nullptr, s, tc, true);
    conv_launch<32, 32>(B, H4, H4, n.a3, nullptr, nullptr, L[5].wf, bias(5), 1, n.t3, nullptr, nullptr, s, tc, true);
    conv_launch<64, 32, 32>(B, H2, H2, n.s2, n.t3, nullptr, L[6].wf, bias(6), 1, n.t4, nullptr, nullptr, s, tc, true);  // up2(t3) ++ s2
    conv_launch<48, 16, 32>(B, N, N, n.s1, n.t4, nullptr, L[7].wf, bias(7), 1, n.a5, nullptr, nullptr, s, tc, true);    // up2(t4) ++ s1
    // the output: channel 0 in FP32 (the tensor-core kernel also writes its
    // BF16 tile)
    conv_launch<16, 16>(B, N, N, n.a5, nullptr, nullptr, L[8].wf, bias(8), 0, tc == 2 ? n.y : nullptr, nullptr, n.y32, s, tc, true);
}

// Loss and gradients of every parameter (into n.g, master layout).  A layer's
// weight gradient waits only for its output gradient, and nothing but the
// final reduction waits for it: the weight gradients (192 CTAs of a few warps,
// bound by latency) run on side streams next to the chain of input gradients
// and to one another (8 x 256^2, the whole call: 750 us one after another, 621
// so).  A buffer that a
// weight gradient may still be reading is not written again: where the chain
// needs one more it takes the target's or the output's (read by the loss
// alone), t4's or a5's (after the weight gradients that read them) or gup's.
void cnn_backward(Cnn &n, int B, int N, cudaStream_t s)
{
    const int N2 = N * N, H2 = N / 2, H4 = N / 4;
    const long P = (long)B * N2;
    auto &L = n.L;
    // the partial sums in the statistics' scratch (free by now)
    float2 *means = (float2 *)n.rpart, *sums = means + (size_t)B * kLossBlk;
    const float sc = 2.0f / ((float)B * (float)N2);
    const dim3 gl(kLossBlk, B);
    note_launch(3);
    k_loss_means<<<gl, 256, 0, s>>>(N2, n.y32, n.t, means);
    k_loss_sums<<<gl, 256, 0, s>>>(N2, sc, n.y32, n.t, means, sums);
    k_loss_grad<<<gl, 256, 0, s>>>(N2, B, sc, n.y32, n.t, means, sums, n.gbig, n.lsum);
    ReduceArgs ra;
    // layer k's weight gradient, from the output gradient that s has just formed
    auto side = [&](int k, auto launch) {
        cudaStream_t q = n.side[k % Cnn::kSide];
        cudaEventRecord(n.ev_gy[k], s);
        cudaStreamWaitEvent(q, n.ev_gy[k], 0);
        launch(q);
        cudaEventRecord(n.ev_dw[k], q);
    };
    // a layer's input gradient: convolution with the flipped weights
    const bf16 *none = nullptr;
    bf16 *gp2 = (bf16 *)n.t, *ga2 = n.t4, *gp1 = n.gup, *gs1 = n.y, *ga1 = n.a5;
    // c6 (linear): input a5, grad gbig (channel 0 of two stored)
    side(8, [&](cudaStream_t q) { conv_dw<16, 16, 0, 16, 2>(n, ra, 8, B, N, N, n.a5, n.gbig, q); });
    conv_launch<16, 16, 0, 2>(B, N, N, n.gbig, none, n.a5, L[8].wb, nullptr, 0, n.gbig2, nullptr, nullptr, s);  // grad a5, masked
    // c5: in up2(t4) ++ s1; the input gradient split into grad t4 (masked) and s1's skip part
    side(7, [&](cudaStream_t q) { conv_dw<48, 16, 32>(n, ra, 7, B, N, N, n.s1, n.gbig2, q, n.t4); });
    conv_launch<16, 48, 0, 16, kEpiSplit>(B, N, N, n.gbig2, none, n.t4, L[7].wb, nullptr, 0, n.gcat, n.gmid, nullptr, s);
    // c4: in up2(t3) ++ s2
    side(6, [&](cudaStream_t q) { conv_dw<64, 32, 32>(n, ra, 6, B, H2, H2, n.s2, n.gmid, q, n.t3); });
    conv_launch<32, 64, 0, 32, kEpiSplit>(B, H2, H2, n.gmid, none, n.t3, L[6].wb, nullptr, 0, n.gup, n.gsmall, nullptr, s);
    // c3b: in a3
    side(5, [&](cudaStream_t q) { conv_dw<32, 32>(n, ra, 5, B, H4, H4, n.a3, n.gsmall, q); });
    conv_launch<32, 32>(B, H4, H4, n.gsmall, none, n.a3, L[5].wb, nullptr, 0, n.gsmall2, nullptr, nullptr, s);  // grad a3, masked
    // c3a: in p2
    side(4, [&](cudaStream_t q) { conv_dw<32, 32>(n, ra, 4, B, H4, H4, n.p2, n.gsmall2, q); });
    conv_launch<32, 32>(B, H4, H4, n.gsmall2, none, nullptr, L[4].wb, nullptr, 0, gp2, nullptr, nullptr, s);  // grad p2
    // grad s2 = skip part of the c4 input grad + pool2 backward, masked
    note_launch();
    k_skip_grad<<<cdiv((long)B * H2 * H2 * 4, 256), 256, 0, s>>>(B * H2 * H2 * 4, H2, H2, 32, n.gup, gp2, n.s2, n.gmid2);
    // c2b: in a2
    side(3, [&](cudaStream_t q) { conv_dw<32, 32>(n, ra, 3, B, H2, H2, n.a2, n.gmid2, q); });
    cudaStreamWaitEvent(s, n.ev_dw[7], 0);  // which reads t4
    conv_launch<32, 32>(B, H2, H2, n.gmid2, none, n.a2, L[3].wb, nullptr, 0, ga2, nullptr, nullptr, s);   // grad a2, masked
    // c2a: in p1
    side(2, [&](cudaStream_t q) { conv_dw<16, 32>(n, ra, 2, B, H2, H2, n.p1, ga2, q); });
    conv_launch<32, 16>(B, H2, H2, ga2, none, nullptr, L[2].wb, nullptr, 0, gp1, nullptr, nullptr, s);  // grad p1
    // grad s1 = skip part of the c5 input grad + pool2 backward, masked
    note_launch();
    k_skip_grad<<<cdiv(P * 2, 256), 256, 0, s>>>((int)(P * 2), N, N, 16, n.gcat, gp1, n.s1, gs1);
    // c1b: in a1
    side(1, [&](cudaStream_t q) { conv_dw<16, 16>(n, ra, 1, B, N, N, n.a1, gs1, q); });
    cudaStreamWaitEvent(s, n.ev_dw[8], 0);  // which reads a5
    conv_launch<16, 16>(B, N, N, gs1, none, n.a1, L[1].wb, nullptr, 0, ga1, nullptr, nullptr, s);     // grad a1, masked
    // c1a: in x
    side(0, [&](cudaStream_t q) { conv_dw<16, 16, 0, 2, 16>(n, ra, 0, B, N, N, n.x, ga1, q); });
    for (int k = 0; k < kLayers; k++) cudaStreamWaitEvent(s, n.ev_dw[k], 0);
    int ctas = 0;
    for (int k = 0; k < kLayers; k++) {
        ra.gw[k] = n.g + L[k].woff; ra.gb[k] = n.g + L[k].boff;
        ra.ci[k] = L[k].ci; ra.co[k] = L[k].co; ra.cip[k] = L[k].cip; ra.cop[k] = L[k].cop;
        ra.first[k] = ctas;
        ctas += (int)cdiv(L[k].cop * 9 * L[k].cip + L[k].cop, 128);
    }
    ra.first[kLayers] = ctas;
    note_launch();
    k_reduce_grads<<<ctas, 128, 0, s>>>(ra);
}

void cnn_adam(Cnn &n, float lr, cudaStream_t s)
{
    n.step++;
    const float b1 = 0.9f, b2 = 0.999f;
    const float c1 = 1.0f - powf(b1, (float)n.step), c2 = 1.0f - powf(b2, (float)n.step);
    note_launch();
    k_adam<<<cdiv((long)n.nparam, 256), 256, 0, s>>>((long)n.nparam, n.w, n.m, n.v, n.g, lr, b1, b2,
                                                    1e-8f, c1, c2);
    cnn_pack(n, s);
}

void cnn_output(Cnn &n, int B, int N, double h, double *p0, cudaStream_t s)
{
    const int N2 = N * N;
    const long P = (long)B * N2;
    note_launch();
    launch_pdl(k_ysum_part, dim3(kRedBlocks, B), 256, 0, s, N2, n.y32, n.rpart);
    note_launch();
    launch_pdl(k_ymean_final, B, 256, 0, s, N2, n.rpart, n.stats);
    note_launch();
    launch_pdl(k_output, cdiv(P, 256), 256, 0, s, P, N2, n.y32, n.stats, h * h * n.out_scale, p0);
}

// Inference with the inputs averaged over 2^levels x 2^levels blocks, the
// network run on the coarse grid (cell size h 2^levels) and its estimate
// interpolated back (bilinear, once per level); levels = 0 is plain
// inference.  N must be a multiple of 4 * 2^levels.
cudaError_t cnn_infer_levels(Cnn &n, int B, int N, double h, const double *rhs, const double *rho,
                             double *p0, int levels, cudaStream_t s)
{
    const int Nc = N >> levels;
    if (levels < 0 || levels > 6 || (Nc << levels) != N || Nc < 4 || Nc % 4) return cudaErrorInvalidValue;
    cudaError_t e = cnn_workspace(n, B, Nc);
    if (e != cudaSuccess) return e;
    if (levels == 0) {
        cnn_forward(n, B, N, h, rhs, rho, nullptr, s);
        cnn_output(n, B, N, h, p0, s);
        return cudaGetLastError();
    }
    // per level k = 1..levels: b_k, rho_k, p_k (B (N >> k)^2 each)
    size_t need = 0;
    for (int k = 1; k <= levels; k++) need += 3 * (size_t)B * (N >> k) * (N >> k);
    if (need > n.cbuf_cap) {
        if (n.cbuf) cudaFree(n.cbuf);
        n.cbuf = nullptr;
        n.cbuf_cap = 0;
        e = cudaMalloc(&n.cbuf, need * 8);
        if (e != cudaSuccess) return e;
        n.cbuf_cap = need;
    }
    double *bk[8], *rk[8], *pk[8];
    double *q = n.cbuf;
    for (int k = 1; k <= levels; k++) {
        const size_t m = (size_t)B * (N >> k) * (N >> k);
        bk[k] = q; rk[k] = q + m; pk[k] = q + 2 * m;
        q += 3 * m;
    }
    bk[0] = const_cast<double *>(rhs);
    rk[0] = const_cast<double *>(rho);
    pk[0] = p0;
    for (int k = 1; k <= levels; k++) {
        const long m = (long)B * (N >> k) * (N >> k);
        note_launch();
        k_restrict2<<<cdiv(m, 256), 256, 0, s>>>(m, N >> k, bk[k - 1], bk[k]);
        note_launch();
        k_restrict2<<<cdiv(m, 256), 256, 0, s>>>(m, N >> k, rk[k - 1], rk[k]);
    }
    const double hc = h * (double)(1 << levels);
    cnn_forward(n, B, Nc, hc, bk[levels], rk[levels], nullptr, s);
    cnn_output(n, B, Nc, hc, pk[levels], s);
    for (int k = levels; k >= 1; k--) {
        const long m = (long)B * (N >> (k - 1)) * (N >> (k - 1));
        note_launch();
        k_prolong2<<<cdiv(m, 256), 256, 0, s>>>(m, N >> k, pk[k], pk[k - 1]);
    }
    return cudaGetLastError();
}

// The network's pressure scale from training data: c = the median over the
// samples of rms(p - mean p) / (rms(b - mean b) h^2) (samples with b = const
// skipped; the mean of the two middle values for an even count).  Sets it
// and returns it in *c.
cudaError_t cnn_fit_scale(Cnn &n, int B, int N, double h, const double *rhs, const double *p,
                          double *c, cudaStream_t s)
{
    const int N2 = N * N;
    double *d = nullptr;
    cudaError_t e = cudaMalloc(&d, (size_t)2 * B * 8);
    if (e != cudaSuccess) return e;
    note_launch(2);
    k_sample_rms<<<B, 256, 0, s>>>(N2, rhs, d);
    k_sample_rms<<<B, 256, 0, s>>>(N2, p, d + B);
    std::vector<double> hv((size_t)2 * B);
    e = cudaMemcpyAsync(hv.data(), d, (size_t)2 * B * 8, cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    cudaFree(d);
    if (e != cudaSuccess) return e;
    std::vector<double> r;
    for (int k = 0; k < B; k++)
        if (hv[k] > 0.0) r.push_back(hv[B + k] / (hv[k] * h * h));
    if (r.empty()) return cudaErrorInvalidValue;
    std::sort(r.begin(), r.end());
    const size_t m = r.size();
    const double med = m % 2 ? r[m / 2] : 0.5 * (r[m / 2 - 1] + r[m / 2]);
    if (!(med > 0.0)) return cudaErrorInvalidValue;
    n.out_scale = med;
    *c = med;
    return cudaSuccess;
}

// Training: the pressure scale from all samples, then `steps` Adam steps on
// mini-batches of `batch` samples drawn with replacement by a SplitMix64
// stream of `seed`, the learning rate decaying tenfold over the run
// (lr0 0.1^(k / steps)); the batch losses land in losses_host (steps floats)
// with one synchronisation at the end.
cudaError_t cnn_train_loop(Cnn &n, int ns, int N, double h, const double *rhs, const double *rho,
                           const double *p, int steps, int batch, float lr0, unsigned long long seed,
                           float *losses_host, cudaStream_t s)
{
    double c = 0.0;
    cudaError_t e = cnn_fit_scale(n, ns, N, h, rhs, p, &c, s);
    if (e != cudaSuccess) return e;
    e = cnn_workspace(n, batch, N);
    if (e != cudaSuccess) return e;
    const long N2 = (long)N * N, nb = (long)batch * N2;
    std::vector<int> idx((size_t)steps * batch);
    unsigned long long st = seed;
    for (auto &v : idx) {
        st += 0x9E3779B97F4A7C15ULL;
        unsigned long long z = st;
        z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ULL;
        z = (z ^ (z >> 27)) * 0x94D049BB133111EBULL;
        v = (int)((z ^ (z >> 31)) % (unsigned long long)ns);
    }
    char *mem = nullptr;
    const size_t bytes = al((size_t)nb * 8) * 3 + al(idx.size() * 4) + al((size_t)steps * 4);
    e = cudaMalloc(&mem, bytes);
    if (e != cudaSuccess) return e;
    double *gb = (double *)mem, *gr = (double *)(mem + al((size_t)nb * 8)),
           *gp = (double *)(mem + 2 * al((size_t)nb * 8));
    int *didx = (int *)(mem + 3 * al((size_t)nb * 8));
    float *dloss = (float *)(mem + 3 * al((size_t)nb * 8) + al(idx.size() * 4));
    e = cudaMemcpyAsync(didx, idx.data(), idx.size() * 4, cudaMemcpyHostToDevice, s);
    for (int k = 0; k < steps && e == cudaSuccess; k++) {
        note_launch();
        k_gather3<<<cdiv(nb, 256), 256, 0, s>>>(nb, (int)N2, didx + (size_t)k * batch, rhs, rho, p,
                                                gb, gr, gp);
        cnn_forward(n, batch, N, h, gb, gr, gp, s);
        cnn_backward(n, batch, N, s);
        note_launch();
        k_loss_record<<<1, 32, 0, s>>>(batch, n.lsum, dloss + k);
        cnn_adam(n, (float)((double)lr0 * pow(0.1, (double)k / (double)steps)), s);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(losses_host, dloss, (size_t)steps * 4, cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    int f = 0;
    if (e == cudaSuccess) e = cnn_take_fault(&f);
    if (e == cudaSuccess && f) e = cudaErrorLaunchFailure;  // a tensor-core completion wait ran out
    cudaFree(mem);
    return e;
}

void cnn_set_scale(Cnn &n, double c) { n.out_scale = c; }
void cnn_set_tc(Cnn &n, int mode) { n.tc = mode; }

// Reads and clears the tensor-core convolutions' fault word.
cudaError_t cnn_take_fault(int *f)
{
    int z = 0;
    cudaError_t e = cudaMemcpyFromSymbol(f, g_cnn_fault, sizeof(int));
    if (e == cudaSuccess && *f) e = cudaMemcpyToSymbol(g_cnn_fault, &z, sizeof(int));
    return e;
}
const void *cnn_workspace_ptr(const Cnn &n) { return n.amem; }
const void *cnn_cbuf_ptr(const Cnn &n) { return n.cbuf; }
double cnn_get_scale(const Cnn &n) { return n.out_scale; }

size_t cnn_nparam(const Cnn &n) { return n.nparam; }
float *cnn_weights(Cnn &n) { return n.w; }
float *cnn_grads(Cnn &n) { return n.g; }
float *cnn_lsum(Cnn &n) { return n.lsum; }
int cnn_steps(const Cnn &n) { return n.step; }
void cnn_reset_adam(Cnn &n) { n.step = 0; cudaMemset(n.m, 0, n.nparam * 8); }

}  // namespace ibk

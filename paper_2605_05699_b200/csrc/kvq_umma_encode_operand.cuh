// The B operand of the forward transform on the tensor cores, W = lambda M diag(s) 2^k in 16-bit terms (kvq_umma_encode.cu says why),
// built by the threads of a CTA out of the plan's table.  C describes the operand: kDim, kBf16 (the terms' type), kSplit (their number),
// kBBlock (bytes of a K block of 64, all rows), term(c) (bytes from a term's row of channel c to the next term's) and row(c), the row of
// a K block that channel c has (c modulo 8).
#pragma once

#include "kvq_umma.cuh"

namespace kvq {
namespace fwd {

// 2^k for a lambda row: the power of two that brings max_c lambda_c max|table entry| (sqrt(2 / D) without a rotation) into [2^13, 2^14), so that
// the first split term of W 2^k stays below fp16's maximum and the later ones above its subnormals.
// Every lane of the warp gets the same value.
template <int D>
__device__ __forceinline__ float lift_of(const float *__restrict__ lam, const float *__restrict__ e0, int lane)
{
    const float table_max = __ldg(e0 + D * D);   // largest |entry| of the table
    float mx = lam ? 0.0f : 1.0f;   // no lambda row (calibration): lambda = 1
#pragma unroll
    for (int p = 0; p < (D / 4 + 31) / 32; ++p) {
        const int i = lane + 32 * p;
        if (lam && i < D / 4) {
            const float4 l = load_input(reinterpret_cast<const float4 *>(lam) + i);
            mx = fmaxf(mx, fmaxf(fmaxf(fabsf(l.x), fabsf(l.y)), fmaxf(fabsf(l.z), fabsf(l.w))));
        }
    }
    if (lam) mx = __uint_as_float(__reduce_max_sync(0xFFFFFFFFu, __float_as_uint(mx)));   // non-negative: ordered like its bits
    else   // the same 1 everywhere, but without the shuffles the calibration's loop is laid out worse: 400,000 vectors at D = 128 33.4 -> 34.0 us
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xFFFFFFFFu, mx, o));
    mx = fminf(fmaxf(mx * table_max, 1e-30f), 1e30f);
    const int e = (int)((__float_as_uint(mx) >> 23) & 0xFFu) - 127;      // floor(log2 mx)
    return __uint_as_float((uint32_t)(127 + 13 - e) << 23);
}

// One quad of row c of every split term: the four table entries m scaled by f = lambda_c 2^k, 16-bit terms peeled
// off one after the other, 8 bytes of each term's swizzled row written.
template <class C>
__device__ __forceinline__ void build_b_quad(unsigned char *sB, float4 m, float f, int c, int i)
{
    constexpr bool BF16 = C::kBf16;
    float w[4] = {m.x * f, m.y * f, m.z * f, m.w * f};
    const int ch = i >> 1;   // 16-byte chunk of the K-major row: K block ch / 8, chunk ch % 8
    const uint32_t off = (uint32_t)((ch >> 3) * C::kBBlock + C::row(c) * 128 + (((ch & 7) ^ (c & 7)) << 4) + ((i & 1) ? 8 : 0));
#pragma unroll
    for (int t = 0; t < C::kSplit; ++t) {
        const uint32_t lo = narrow2<BF16>(w[0], w[1]), hi = narrow2<BF16>(w[2], w[3]);
        *reinterpret_cast<uint2 *>(sB + t * C::term(c) + off) = make_uint2(lo, hi);
        if (t + 1 < C::kSplit) {   // what the 16-bit term left behind (exact in fp32)
            const float2 a = widen2<BF16>(lo), b = widen2<BF16>(hi);
            w[0] -= a.x, w[1] -= a.y, w[2] -= b.x, w[3] -= b.y;
        }
    }
}

// The B operand by W warps: the table's quads, row after row, dealt out to all their lanes, so that no lane idles where a row is not
// a multiple of 32 quads, in batches of up to 16 that are requested together (load) and turned into B rows once the lift is
// known and the old operand is free (store): one round trip to L2 per batch, the first one before the wait.  The lambda entries of a
// batch are requested by one lane each (load_lambda, behind grid_wait) and handed round by shuffles: loads that cannot move across
// the stores to shared memory cost 100 cycles a quad in their place (5120 vectors under 160 lambda rows, D = 128: 9.5 and 11.4 us).
template <class C, int W>
struct BuildB {
    static constexpr int D = C::kDim;
    static constexpr int kQuads = D / 4, kTotal = D * kQuads;
    static constexpr int kPerLane = (kTotal + 32 * W - 1) / (32 * W);
    static constexpr int kBatches = (kPerLane + 15) / 16;
    static constexpr int kBatch = (kPerLane + kBatches - 1) / kBatches;
    static constexpr int kRowsPerPass = (31 + kQuads - 1) / kQuads + 1;   // table rows that 32 neighbouring quads can touch
    static_assert(kBatch * kRowsPerPass <= 32, "a lane per lambda entry of a batch");
    float4 m[kBatch];
    float l;   // lane k kRowsPerPass + d: lambda of the d-th table row of pass k
    static __device__ __forceinline__ int quad(int batch, int k, int w, int lane) { return ((batch * kBatch + k) * W + w) * 32 + lane; }
    __device__ __forceinline__ void load(const float *__restrict__ e0, int batch, int w, int lane)
    {
#pragma unroll
        for (int k = 0; k < kBatch; ++k) {
            const int f = quad(batch, k, w, lane);
            m[k] = f < kTotal ? __ldg(reinterpret_cast<const float4 *>(e0) + f) : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        }
    }
    __device__ __forceinline__ void load_lambda(const float *__restrict__ lam, int batch, int w, int lane)
    {
        const int k = lane / kRowsPerPass, c = quad(batch, k, w, 0) / kQuads + lane % kRowsPerPass;
        l = lam && k < kBatch && c < D ? load_input(lam + c) : 1.0f;
    }
    __device__ __forceinline__ void store(unsigned char *sB, float lift, int batch, int w, int lane) const
    {
        const float lifted = l * lift;
#pragma unroll
        for (int k = 0; k < kBatch; ++k) {
            const int f = quad(batch, k, w, lane), c = f / kQuads;
            const float lc = __shfl_sync(0xFFFFFFFFu, lifted, k * kRowsPerPass + c - quad(batch, k, w, 0) / kQuads);
            if (f < kTotal) build_b_quad<C>(sB, m[k], lc, c, f - c * kQuads);
        }
    }
    // batches from the second on, after store(0)
    __device__ __forceinline__ void rest(unsigned char *sB, const float *__restrict__ e0, const float *__restrict__ lam, float lift, int w, int lane)
    {
#pragma unroll
        for (int b = 1; b < kBatches; ++b) {
            load(e0, b, w, lane);
            load_lambda(lam, b, w, lane);
            store(sB, lift, b, w, lane);
        }
    }
};

}  // namespace fwd
}  // namespace kvq

// The B operand of the inverse transform on the tensor cores, W' = diag(s) M^T diag(1 / max(lambda, 1e-6)) / rho in fp16 terms
// (kvq_umma_decode.cu says why), built by the threads of a CTA out of the plan's table.  C describes the operand: kBits, kRadix2 (the
// form), kTerms, kBRows, kQuads (table rows it is built from, float4 per row) and the places of its parts (kBPartBlock, kBPart; kBBlock,
// kBTerm).
#pragma once

#include "kvq_umma.cuh"

namespace kvq {
namespace inv {

// One quad of the B operand, the table entries m of row n and channels 4 i .. 4 i + 3 times the reciprocals rc, and its place in the
// swizzled K-major row.  4-bit codes: neighbouring lanes hold the two quads of a word of eight codes and trade two values, so that
// each holds two K-ordered pairs of the dense form (K order of a word: 0, 4, 1, 5, 2, 6, 3, 7), or one pair of each parity of
// the radix-2 form (even lane 8w + p and 8w + p + 4, odd lane 8w + p + 2 and 8w + p + 6): the order in which the dequant threads
// write the codes.  Byte codes: the natural order, per parity pairs (c, c + 2).  Every lane calls it (shuffles); `live` ones store.
template <class C>
__device__ __forceinline__ void build_b_quad(unsigned char *sB, float4 m, float4 rc, int n, int i, bool live)
{
    constexpr int BITS = C::kBits;
    constexpr bool R2 = C::kRadix2;
    const bool odd = i & 1;
    // (The plain transform's entries are at most sqrt(2 / D) and the reciprocals below 2: only a rotated table could leave fp16's range.
    // Without the clamp 148, 296 and 592 tiles at D = 256 bf16 10.95 -> 10.5 us, 13.6 -> 13.2, 19.1 -> 18.75; D <= 160 up to 1 %.)
    auto sat = [](float v) { return R2 ? v : fminf(fmaxf(v, -65504.0f), 65504.0f); };
    const float v[4] = {sat(m.x * rc.x), sat(m.y * rc.y), sat(m.z * rc.z), sat(m.w * rc.w)};
    if constexpr (R2) {
        const int at = BITS == 4 ? 8 * (i >> 1) + (odd ? 4 : 0) : 4 * i;   // byte of the pair within a parity's K-major row
        unsigned char *dst = sB + (at >> 7) * C::kBPartBlock + n * 128 + ((((at >> 4) & 7) ^ (n & 7)) << 4) + (at & 15);
#pragma unroll
        for (int p = 0; p < 2; ++p) {
            float w0 = v[p], w1 = v[p + 2];
            if constexpr (BITS == 4) {
                const float got = __shfl_xor_sync(0xFFFFFFFFu, odd ? v[p] : v[p + 2], 1);
                w0 = odd ? got : v[p], w1 = odd ? v[p + 2] : got;
            }
#pragma unroll
            for (int t = 0; t < C::kTerms; ++t) {
                const uint32_t h = narrow2<false>(w0, w1);
                if (live) *reinterpret_cast<uint32_t *>(dst + p * C::kBPart + t * (2 * C::kBPart)) = h;
                if (t + 1 < C::kTerms) {   // what the fp16 term left behind (exact in fp32)
                    const float2 a = widen2<false>(h);
                    w0 -= a.x, w1 -= a.y;
                }
            }
        }
    } else {
        float vx = v[0], vy = v[1], vz = v[2], vw = v[3];
        const int w = i >> 1;   // 16-byte chunk w of the K-major row: K block w / 8, chunk w % 8
        unsigned char *dst = sB + (w >> 3) * C::kBBlock + n * 128 + (((w & 7) ^ (n & 7)) << 4) + (odd ? 8 : 0);
#pragma unroll
        for (int t = 0; t < C::kTerms; ++t) {
            uint2 o;
            if constexpr (BITS == 4) {
                const float r0 = __shfl_xor_sync(0xFFFFFFFFu, odd ? vx : vz, 1);
                const float r1 = __shfl_xor_sync(0xFFFFFFFFu, odd ? vy : vw, 1);
                o.x = odd ? narrow2<false>(r0, vz) : narrow2<false>(vx, r0);   // odd: (2, 6)   even: (0, 4)
                o.y = odd ? narrow2<false>(r1, vw) : narrow2<false>(vy, r1);   // odd: (3, 7)   even: (1, 5)
            } else {
                o.x = narrow2<false>(vx, vy);
                o.y = narrow2<false>(vz, vw);
            }
            if (live) *reinterpret_cast<uint2 *>(dst + t * C::kBTerm) = o;
            if (t + 1 < C::kTerms) {   // what the fp16 term left behind (exact in fp32)
                vx -= __half2float(__float2half_rn(vx)), vy -= __half2float(__float2half_rn(vy));
                vz -= __half2float(__float2half_rn(vz)), vw -= __half2float(__float2half_rn(vw));
            }
        }
    }
}

// The B operand by W warps: the table's quads, row after row, dealt out to all their lanes, so that no lane idles where a row is not
// a multiple of 32 quads, in batches of up to 16 that are requested together (load) and turned into B rows once the reciprocals
// are in shared memory and the old operand is free (store): one round trip to L2 per batch, the first one before the wait.
template <class C, int W>
struct BuildB {
    static constexpr int kTotal = C::kBRows * C::kQuads;
    static constexpr int kPerLane = (kTotal + 32 * W - 1) / (32 * W);
    static constexpr int kBatches = (kPerLane + 15) / 16;
    static constexpr int kBatch = (kPerLane + kBatches - 1) / kBatches;
    float4 m[kBatch];
    static __device__ __forceinline__ int quad(int batch, int k, int w, int lane) { return ((batch * kBatch + k) * W + w) * 32 + lane; }
    __device__ __forceinline__ void load(const float *__restrict__ b0, int batch, int w, int lane)
    {
#pragma unroll
        for (int k = 0; k < kBatch; ++k) {
            const int f = quad(batch, k, w, lane);
            m[k] = f < kTotal ? __ldg(reinterpret_cast<const float4 *>(b0) + f) : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        }
    }
    __device__ __forceinline__ void store(unsigned char *sB, const float *recip, int batch, int w, int lane) const
    {
#pragma unroll
        for (int k = 0; k < kBatch; ++k) {
            const int f = quad(batch, k, w, lane), n = f / C::kQuads, i = f - n * C::kQuads;   // kQuads is even: lane pairs stay in one row
            const bool live = f < kTotal;
            const float4 rc = *reinterpret_cast<const float4 *>(recip + 4 * i);
            build_b_quad<C>(sB, m[k], rc, live ? n : 0, i, live);
        }
    }
    // batches from the second on, after store(0)
    __device__ __forceinline__ void rest(unsigned char *sB, const float *__restrict__ b0, const float *recip, int w, int lane)
    {
#pragma unroll
        for (int b = 1; b < kBatches; ++b) {
            load(b0, b, w, lane);
            store(sB, recip, b, w, lane);
        }
    }
};

// every warp that builds writes the whole row itself (the same values) and so needs no more than its own lanes to be done
template <int D>
__device__ __forceinline__ void post_reciprocals(float *recip, const RecipLambda<D> &rl, int lane)
{
#pragma unroll
    for (int p = 0; p < RecipLambda<D>::kPasses; ++p)
        if (lane + 32 * p < D / 4) *reinterpret_cast<float4 *>(recip + 4 * (lane + 32 * p)) = rl.r[p];
    __syncwarp();
}

// The D / 32 fp16 group scales of one row, as packed 16-bit pairs.
template <int G>
__device__ __forceinline__ void load_row_scales(const uint16_t *__restrict__ sp, uint32_t (&sb)[(G + 1) / 2])
{
    if constexpr (G == 8) {
        const uint4 v = load_input(reinterpret_cast<const uint4 *>(sp));
        sb[0] = v.x, sb[1] = v.y, sb[2] = v.z, sb[3] = v.w;
    } else if constexpr (G == 4) {
        const uint2 v = load_input(reinterpret_cast<const uint2 *>(sp));
        sb[0] = v.x, sb[1] = v.y;
    } else if constexpr (G == 2) {
        sb[0] = load_input(reinterpret_cast<const uint32_t *>(sp));
    } else {   // rows of 6 or 10 bytes are only 2-byte aligned
#pragma unroll
        for (int j = 0; j < (G + 1) / 2; ++j) sb[j] = 0;
#pragma unroll
        for (int j = 0; j < G; ++j) sb[j / 2] |= (uint32_t)load_input(sp + j) << (16 * (j & 1));
    }
}

}  // namespace inv
}  // namespace kvq

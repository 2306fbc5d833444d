// The quantizer of the tensor-core encode kernels (Sec. 3.2 steps 3-4): one group of 32 accumulator values of a row, as
// tcgen05.ld delivers them -> largest magnitude -> fp16 scale -> round-to-nearest-even codes -> packed words.
//
// These kernels run at the board's power limit, where a warp instruction costs about a nanojoule, so the count is what matters:
// the magnitudes take half an instruction each (max.abs of three: the absolute values are free), sums and products of
// neighbouring values go in pairs (add / fma.f32x2, rounded like the single ones), the codes are gathered by byte permutes.
// Encode of 2,097,152 vectors at D = 128, back to back: 183.1 -> 180.2 us (another box: 182.7 -> 181.1, inside the spread); D = 160, 700,000:
// 97.5 -> 93.4; D = 256, 1,064,960: 269 -> 266.  The maxima three at a time instead of two are 17 instructions per
// group in place of 31; in time 1 % or less, inside the spread of repeated runs (2,097,152 at D = 128 179.5 -> 177.8).
#pragma once

#include "kvq_device.cuh"

namespace kvq {

// max(|a|, |b|, |c|); like fmaxf a NaN yields to the other operands
__device__ __forceinline__ float max_magnitude(uint32_t a, uint32_t b, uint32_t c)
{
    float d;
    asm("max.abs.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(__uint_as_float(a)), "f"(__uint_as_float(b)), "f"(__uint_as_float(c)));
    return d;
}

__device__ __forceinline__ float group_absmax(const uint32_t (&v)[32])
{
    float m[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) m[i] = max_magnitude(v[i], v[i + 4], v[i + 8]);   // four chains of eight
#pragma unroll
    for (int i = 12; i < 28; i += 8)
#pragma unroll
        for (int k = 0; k < 4; ++k) m[k] = max_magnitude(__float_as_uint(m[k]), v[i + k], v[i + 4 + k]);
    m[0] = max_magnitude(__float_as_uint(m[0]), v[28], v[29]);
    m[1] = max_magnitude(__float_as_uint(m[1]), v[30], v[31]);
    return fmaxf(max_magnitude(__float_as_uint(m[0]), __float_as_uint(m[1]), __float_as_uint(fmaxf(m[2], m[3]))), 0.0f);   // 0 where every value is a NaN
}

// v[i] += w[i], two at a time
__device__ __forceinline__ void add_group(uint32_t (&v)[32], const uint32_t (&w)[32])
{
#pragma unroll
    for (int i = 0; i < 32; i += 2)
        asm("{\n\t.reg .b64 a, b;\n\t"
            "mov.b64 a, {%0, %1};\n\tmov.b64 b, {%2, %3};\n\t"
            "add.rn.f32x2 a, a, b;\n\t"
            "mov.b64 {%0, %1}, a;\n\t}"
            : "+r"(v[i]), "+r"(v[i + 1])
            : "r"(w[i]), "r"(w[i + 1]));
}

// v[0 .. 3] *= l, two at a time
__device__ __forceinline__ void mul_quad(uint32_t *v, float4 l)
{
    const float2 a = unpack_f32x2(mul_f32x2(pack_f32x2(__uint_as_float(v[0]), __uint_as_float(v[1])), pack_f32x2(l.x, l.y)));
    const float2 b = unpack_f32x2(mul_f32x2(pack_f32x2(__uint_as_float(v[2]), __uint_as_float(v[3])), pack_f32x2(l.z, l.w)));
    v[0] = __float_as_uint(a.x), v[1] = __float_as_uint(a.y), v[2] = __float_as_uint(b.x), v[3] = __float_as_uint(b.y);
}

// bit patterns of v0 rs + magic, v1 rs + magic
__device__ __forceinline__ void fma_pair(uint32_t v0, uint32_t v1, uint64_t rs2, uint64_t magic2, uint32_t &t0, uint32_t &t1)
{
    asm("{\n\t.reg .b64 a;\n\t"
        "mov.b64 a, {%2, %3};\n\t"
        "fma.rn.f32x2 a, a, %4, %5;\n\t"
        "mov.b64 {%0, %1}, a;\n\t}"
        : "=r"(t0), "=r"(t1)
        : "r"(v0), "r"(v1), "l"(rs2), "l"(magic2));
}

struct GroupScale {
    uint16_t half;   // the stored scale, sigma = fp16(absmax / Q), saturating
    float rs;        // 1 / sigma, applied to the lifted accumulator values; codes are taken against the stored scale
    bool clamp;      // saturated or subnormal scale: codes could leave [-Q, Q]
};

// Q: the largest code, 7 or 127, inv_q = 1 / Q rounded.  The quotient is Markstein's: correctly rounded from a correctly rounded
// reciprocal, one residual and one correction (infinite maxima give a NaN, which fminf turns into the saturated scale).
__device__ __forceinline__ GroupScale group_scale(float amax_lifted, float unlift, float Q, float inv_q)
{
    const float amax = amax_lifted * unlift;
    const float q0 = amax * inv_q;
    const float quot = fmaf(fmaf(-Q, q0, amax), inv_q, q0);
    const __half hs = __float2half_rn(fminf(quot, 65504.0f));
    const float sg = __half2float(hs);
    const float rs1 = sg > 0.0f ? __frcp_rn(sg) : 0.0f;
    GroupScale s;
    s.half = __half_as_ushort(hs);
    s.rs = rs1 * unlift;
    s.clamp = !(amax * rs1 < Q + 0.25f);
    return s;
}

// Biased codes q + 8 (q + 128) sit in the low byte of v rs + magic.
template <int BITS>
__device__ __forceinline__ void round_four(const uint32_t *v, const GroupScale &s, uint64_t rs2, uint64_t magic2, uint32_t (&t)[4])
{
    constexpr float Q = BITS == 4 ? 7.0f : 127.0f, magic = BITS == 4 ? kMagicRound : kMagicRound8;
    if (!s.clamp) {
        fma_pair(v[0], v[1], rs2, magic2, t[0], t[1]);
        fma_pair(v[2], v[3], rs2, magic2, t[2], t[3]);
    } else {
#pragma unroll
        for (int e = 0; e < 4; ++e) t[e] = __float_as_uint(fminf(fmaxf(__uint_as_float(v[e]) * s.rs, -Q), Q) + magic);
    }
}

// 32 codes as nibble pairs: byte i = (q_{2i+1} << 4) | (q_{2i} & 15)
__device__ __forceinline__ uint4 pack_nibbles(const uint32_t (&v)[32], const GroupScale &s)
{
    const uint64_t rs2 = pack_f32x2(s.rs, s.rs), magic2 = pack_f32x2(kMagicRound, kMagicRound);
    uint32_t words[4];
#pragma unroll
    for (int w = 0; w < 4; ++w) {
        uint32_t a[4], b[4];
        round_four<4>(&v[8 * w], s, rs2, magic2, a);
        round_four<4>(&v[8 * w + 4], s, rs2, magic2, b);
        const uint32_t even = __byte_perm(__byte_perm(a[0], a[2], 0x0040), __byte_perm(b[0], b[2], 0x0040), 0x5410);
        const uint32_t odd = __byte_perm(__byte_perm(a[1], a[3], 0x0040), __byte_perm(b[1], b[3], 0x0040), 0x5410);
        words[w] = (even + (odd << 4)) ^ 0x88888888u;   // each byte of even and odd holds 1 .. 15
    }
    return make_uint4(words[0], words[1], words[2], words[3]);
}

// 16 codes (v[0 .. 15]) as two's-complement bytes
__device__ __forceinline__ uint4 pack_bytes(const uint32_t *v, const GroupScale &s)
{
    const uint64_t rs2 = pack_f32x2(s.rs, s.rs), magic2 = pack_f32x2(kMagicRound8, kMagicRound8);
    uint32_t words[4];
#pragma unroll
    for (int w = 0; w < 4; ++w) {
        uint32_t t[4];
        round_four<8>(v + 4 * w, s, rs2, magic2, t);
        words[w] = __byte_perm(__byte_perm(t[0], t[1], 0x0040), __byte_perm(t[2], t[3], 0x0040), 0x5410) ^ 0x80808080u;
    }
    return make_uint4(words[0], words[1], words[2], words[3]);
}

}  // namespace kvq

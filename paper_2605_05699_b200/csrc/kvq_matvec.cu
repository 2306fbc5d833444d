// Small-call kernels of libkvq: kvq_append, the window flush and other calls of a few thousand vectors at most.
//
// On such calls nothing is bandwidth-bound: what counts is the latency of one launch.  The register-FFT kernels
// give a whole vector to one thread (thousands of dependent instructions), the tensor-core kernels pay a fixed
// set-up per launch (operand build, pipeline fill); both take 10 us and more for 64 vectors.  Here the transform
// is a plain fp32 matrix-vector product with the plan's D x D table (Sec. 3.1 Eq. 1-2 written as a matrix, signs
// and, if the plan has one, the rotation of Sec. 5.1 item 2 folded in), spread over a whole CTA:
//
//   * a CTA takes 8 vectors; its 8 warps split the contraction index (K) into 8 slices;
//   * a lane owns four consecutive output coordinates (eight for D > 128): table rows are read as coalesced
//     float4 (all rows of a slice in flight at once: about one L2 round trip per CTA), the vectors' entries come
//     from shared memory as broadcasts;
//   * partial sums meet in shared memory; warp w then finishes vector w: lambda, group maxima by shuffles, scale,
//     rounding and packing (encode) or the conversion to half precision (decode).
//
// Every (group, bits) layout, both dtypes, rotated plans and row maps are served; group and bits are run-time
// (warp-uniform) values.  Arithmetic of the quantizer follows the register-FFT kernels (same operations in the
// same order), so the two families agree wherever fp32 rounding of the transform does not decide a code.
#include "kvq_internal.h"
#include "kvq_device.cuh"
#include "kvq_umma.cuh"

namespace kvq {

namespace {

constexpr int kWarps = 8;   // warps per CTA = slices of the contraction index
constexpr int kV = 8;       // vectors per CTA = one per warp in the finishing phase

struct MatvecParams {
    const void *in;        // encode: x [N, D] half precision
    const float *lambda;   // [n_lambda, D]
    void *packed;          // [*, D bits / 8]
    void *scales;          // [*, D / group] fp16
    void *out;             // decode: [*, D] half precision
    const float *table;    // encode: b0[n][c] (column c of the forward transform along a row); decode: e0[c][n]
    const float *table2;   // fused window flush: e0[c][n], for the way back
    int64_t N, n_lambda;
    FastDiv rows_per_lambda;
    RowMap map;            // where row r lives: encode of its output, decode of both sides (a cache view or the flat layout)
    int group, bits;
    // Position on the device: when pos_dev is set, the base row of map is *pos_dev, read when the kernel runs, and must
    // lie in [0, pos_limit]; otherwise the launch writes nothing and raises KVQ_DEV_POSITION in *status.
    const int64_t *pos_dev;
    int64_t pos_limit;
    uint32_t *status;
};

// The row map of this launch's output rows: as passed, or based at the position found in device memory.  False (for the
// whole grid alike) when that position is outside the cache.
__device__ __forceinline__ bool resolve_out_map(const MatvecParams &prm, RowMap &map)
{
    map = prm.map;
    if (prm.pos_dev) {
        const int64_t p = load_input(prm.pos_dev);
        if (p < 0 || p > prm.pos_limit) {
            if (blockIdx.x == 0 && threadIdx.x == 0) atomicOr(prm.status, KVQ_DEV_POSITION);
            return false;
        }
        map.base = p;
    }
    return true;
}

template <int D>
struct Geo {
    static constexpr int P = (D / 4 + 31) / 32;   // coordinate quads per lane
    static constexpr int KW = D / kWarps;         // contraction indices per warp
    // table rows a lane holds in flight per pass: the whole slice where registers allow (one L2 round trip per CTA)
    static constexpr int CH = P == 1 ? KW : (D == 160 ? 10 : 16);
    static_assert(D % (4 * kWarps) == 0 && KW % CH == 0, "slices must be whole quads and whole passes");
    static constexpr bool kLoops = CH == KW;      // the slice stays in registers: a CTA may take several batches of vectors
    static constexpr int kSmemBytes = (kV * D + kWarps * kV * D) * (int)sizeof(float);
};

__device__ __forceinline__ int64_t lambda_row(int64_t r, int64_t n_lambda, const FastDiv &rows_per_lambda)
{
    return n_lambda == 1 ? 0 : rows_per_lambda(r);
}

// Rows k0 .. k0 + CH - 1 of this warp's slice of the table into registers (coalesced float4 per row).
template <int D>
__device__ __forceinline__ void load_rows(const float *__restrict__ table, int warp, int lane, int k0, float4 (&t)[Geo<D>::CH][Geo<D>::P])
{
    using Gm = Geo<D>;
#pragma unroll
    for (int k = 0; k < Gm::CH; ++k)
#pragma unroll
        for (int p = 0; p < Gm::P; ++p) {
            const int i = lane + 32 * p;
            t[k][p] = i < D / 4 ? __ldg(reinterpret_cast<const float4 *>(table + (size_t)(warp * Gm::KW + k0 + k) * D) + i)
                                : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        }
}

// y_v[c] = sum_k table[k][c] xs[v][k] for the CTA's kV vectors: this warp's K slice into registers (its first pass
// of table rows, t, was fetched by the caller while the vectors were being staged), partial sums through shared
// memory, and the sums of vector `warp` back into y[P][4] (coordinates 4 i .. 4 i + 3, i = lane + 32 p).
template <int D>
__device__ __forceinline__ void matvec(const float *__restrict__ table, float4 (&t)[Geo<D>::CH][Geo<D>::P], const float *xs, float *red,
                                       int warp, int lane, float (&y)[Geo<D>::P][4])
{
    using Gm = Geo<D>;
    constexpr int P = Gm::P, KW = Gm::KW, CH = Gm::CH;
    float acc[kV][P][4];
#pragma unroll
    for (int v = 0; v < kV; ++v)
#pragma unroll
        for (int p = 0; p < P; ++p)
#pragma unroll
            for (int e = 0; e < 4; ++e) acc[v][p][e] = 0.0f;

#pragma unroll 1
    for (int k0 = 0; k0 < KW; k0 += CH) {
        if (k0 > 0) load_rows<D>(table, warp, lane, k0, t);
#pragma unroll
        for (int v = 0; v < kV; ++v) {
#pragma unroll
            for (int k = 0; k < CH; ++k) {
                const float xk = xs[v * D + warp * KW + k0 + k];   // broadcast
#pragma unroll
                for (int p = 0; p < P; ++p) {
                    acc[v][p][0] = fmaf(t[k][p].x, xk, acc[v][p][0]);
                    acc[v][p][1] = fmaf(t[k][p].y, xk, acc[v][p][1]);
                    acc[v][p][2] = fmaf(t[k][p].z, xk, acc[v][p][2]);
                    acc[v][p][3] = fmaf(t[k][p].w, xk, acc[v][p][3]);
                }
            }
        }
    }
#pragma unroll
    for (int v = 0; v < kV; ++v)
#pragma unroll
        for (int p = 0; p < P; ++p) {
            const int i = lane + 32 * p;
            if (i < D / 4)
                *reinterpret_cast<float4 *>(red + (size_t)(warp * kV + v) * D + 4 * i) =
                    make_float4(acc[v][p][0], acc[v][p][1], acc[v][p][2], acc[v][p][3]);
        }
    __syncthreads();
#pragma unroll
    for (int p = 0; p < P; ++p) {
        const int i = lane + 32 * p;
        float4 s = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        if (i < D / 4) {
#pragma unroll
            for (int w = 0; w < kWarps; ++w) {
                const float4 a = *reinterpret_cast<const float4 *>(red + (size_t)(w * kV + warp) * D + 4 * i);
                s.x += a.x, s.y += a.y, s.z += a.z, s.w += a.w;
            }
        }
        y[p][0] = s.x, y[p][1] = s.y, y[p][2] = s.z, y[p][3] = s.w;
    }
}

// ------------------------------------------------------------------------------------------------
// encode: x -> codes and scales  (Sec. 3.2 steps 1-4, lambda and group scales of Sec. 7.1)
// ------------------------------------------------------------------------------------------------
// FLUSH: the window flush in one launch (Sec. 7.2).  After the codes of a vector are stored, the warp that finished it puts
// q sigma / max(lambda, 1e-6) -- what kvq_decode would rebuild from the stored bytes -- back into shared memory, and the
// CTA runs the matrix-vector product once more with the inverse table: rows out_map(r) of prm.out get the dequantized
// vectors.
// One batch of kV vectors.  t: the first pass of this warp's table rows, requested by the caller.
template <int D, bool BF16, bool FLUSH>
__device__ __forceinline__ void encode_batch(const MatvecParams &prm, const RowMap &out_map, float4 (&t)[Geo<D>::CH][Geo<D>::P], float *xs,
                                             float *red, int warp, int lane, int64_t batch, bool last)
{
    using Gm = Geo<D>;
    constexpr int P = Gm::P;
    const int64_t v0 = batch * kV;
    const int64_t r = v0 + warp;   // the vector this warp finishes
    float4 lam4[P];
#pragma unroll
    for (int p = 0; p < P; ++p) {
        const int i = lane + 32 * p;
        lam4[p] = (r < prm.N && i < D / 4)
                      ? load_input(reinterpret_cast<const float4 *>(prm.lambda + lambda_row(r, prm.n_lambda, prm.rows_per_lambda) * D) + i)
                      : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    }

    // ---- the CTA's vectors, widened to fp32 (rows past the end are zeros)
    const uint32_t *x = static_cast<const uint32_t *>(prm.in);
    for (int idx = threadIdx.x; idx < kV * (D / 2); idx += kWarps * 32) {
        const int v = idx / (D / 2), j = idx % (D / 2);
        const int64_t r = v0 + v;
        const float2 f = widen2<BF16>(r < prm.N ? load_input(x + r * (D / 2) + j) : 0u);
        xs[v * D + 2 * j] = f.x, xs[v * D + 2 * j + 1] = f.y;
    }
    __syncthreads();
    if (last) grid_trigger();   // nothing but the tables is read from here on

    // The way back's table rows where registers hold both slices: requested here, their round trip to L2 runs under the product and the quantizer.
    constexpr bool kEarly = FLUSH && Gm::kLoops;
    float4 t2[kEarly ? Gm::CH : 1][P];
    if constexpr (kEarly) load_rows<D>(prm.table2, warp, lane, 0, t2);
    float z[P][4];
    matvec<D>(prm.table, t, xs, red, warp, lane, z);

    // ---- warp w finishes vector w
    const bool live = r < prm.N;
    if (!FLUSH && !live) return;   // only in a CTA's last batch, and no barrier follows
    const int64_t orow = live ? out_map(r) : 0;
    const bool per_vector = prm.group == D;
    const float Q = prm.bits == 4 ? 7.0f : 127.0f;
    float amax[P];
#pragma unroll
    for (int p = 0; p < P; ++p) {
        const int i = lane + 32 * p;
        amax[p] = 0.0f;
        if (i < D / 4) {
            const float4 l = lam4[p];
            z[p][0] *= l.x, z[p][1] *= l.y, z[p][2] *= l.z, z[p][3] *= l.w;
            amax[p] = fmaxf(fmaxf(fabsf(z[p][0]), fabsf(z[p][1])), fmaxf(fabsf(z[p][2]), fabsf(z[p][3])));
        }
    }
    // group maxima: a group of 32 coordinates is 8 neighbouring lanes of one p; one group over the vector is everything
    if (per_vector) {
        float m = amax[0];
#pragma unroll
        for (int p = 1; p < P; ++p) m = fmaxf(m, amax[p]);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xFFFFFFFFu, m, o));
#pragma unroll
        for (int p = 0; p < P; ++p) amax[p] = m;
    } else {
#pragma unroll
        for (int p = 0; p < P; ++p)
#pragma unroll
            for (int o = 4; o > 0; o >>= 1) amax[p] = fmaxf(amax[p], __shfl_xor_sync(0xFFFFFFFFu, amax[p], o));
    }
    uint16_t *scl = static_cast<uint16_t *>(prm.scales);
    unsigned char *pk = static_cast<unsigned char *>(prm.packed);
#pragma unroll
    for (int p = 0; p < P; ++p) {
        const int i = lane + 32 * p;
        // sigma = fp16(absmax / Q); codes are taken against the stored value
        const float sig = fminf(__fdiv_rn(amax[p], Q), 65504.0f);
        const __half hs = __float2half_rn(sig);
        const float sg = __half2float(hs);
        const float rs = sg > 0.0f ? __frcp_rn(sg) : 0.0f;
        const bool clamp = !(amax[p] * rs < Q + 0.25f);   // saturated or subnormal scale: codes could leave [-Q, Q]
        if (i >= D / 4) continue;
        if (live && (per_vector ? (lane == 0 && p == 0) : ((i & 7) == 0)))
            scl[orow * (D / prm.group) + (per_vector ? 0 : i >> 3)] = __half_as_ushort(hs);
        uint32_t code[4];
        float qf[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const float t = clamp ? fminf(fmaxf(z[p][e] * rs, -Q), Q) + 12582912.0f : fmaf(z[p][e], rs, 12582912.0f);
            code[e] = __float_as_uint(t);   // low bits: q in two's complement (1.5 * 2^23 + q)
            qf[e] = t - 12582912.0f;        // q itself, exactly
        }
        if (live) {
            if (prm.bits == 4) {
                const uint32_t w = (code[0] & 0xFu) | ((code[1] & 0xFu) << 4) | ((code[2] & 0xFu) << 8) | ((code[3] & 0xFu) << 12);
                *reinterpret_cast<uint16_t *>(pk + orow * (D / 2) + 2 * i) = (uint16_t)w;
            } else {
                const uint32_t w = (code[0] & 0xFFu) | ((code[1] & 0xFFu) << 8) | ((code[2] & 0xFFu) << 16) | (code[3] << 24);
                *reinterpret_cast<uint32_t *>(pk + orow * D + 4 * i) = w;
            }
        }
        if constexpr (FLUSH) {   // the way back starts from the stored values: q times the STORED scale over the clamped lambda
            const float4 l = lam4[p];
            const float4 o = make_float4(qf[0] * (sg * __frcp_rn(fmaxf(l.x, 1e-6f))), qf[1] * (sg * __frcp_rn(fmaxf(l.y, 1e-6f))),
                                         qf[2] * (sg * __frcp_rn(fmaxf(l.z, 1e-6f))), qf[3] * (sg * __frcp_rn(fmaxf(l.w, 1e-6f))));
            *reinterpret_cast<float4 *>(xs + warp * D + 4 * i) = live ? o : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        }
    }
    if constexpr (FLUSH) {
        float y[P][4];
        if constexpr (kEarly) {
            __syncthreads();                               // every warp's vector is back in shared memory; red is free again
            matvec<D>(prm.table2, t2, xs, red, warp, lane, y);
        } else {
            float4 t2[Gm::CH][P];
            load_rows<D>(prm.table2, warp, lane, 0, t2);   // in flight across the barrier
            __syncthreads();
            matvec<D>(prm.table2, t2, xs, red, warp, lane, y);
        }
        if (!live) return;
        unsigned char *out = static_cast<unsigned char *>(prm.out) + orow * (2 * D);
#pragma unroll
        for (int p = 0; p < P; ++p) {
            const int i = lane + 32 * p;
            if (i < D / 4)
                *reinterpret_cast<uint2 *>(out + 8 * i) = make_uint2(narrow2<BF16>(y[p][0], y[p][1]), narrow2<BF16>(y[p][2], y[p][3]));
        }
    }
}

// Where a warp's whole table slice fits its registers (D <= 128), a CTA takes batches blockIdx.x, blockIdx.x + gridDim.x,
// ... and the launch is one resident wave: on calls of more batches than the device holds CTAs the table crosses L2 once
// per CTA, not once per batch.  The barriers inside one batch also order the next batch's writes to xs and red after this
// batch's reads.  For D > 128 a CTA takes one batch.
template <int D, bool BF16, bool FLUSH>
__global__ void __launch_bounds__(kWarps * 32) kvq_encode_matvec_kernel(const __grid_constant__ MatvecParams prm)
{
    using Gm = Geo<D>;
    extern __shared__ __align__(16) float sm[];
    float *xs = sm, *red = sm + kV * D;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

    // ---- everything that does not depend on the vectors is requested first, so that one round trip covers it all
    float4 t[Gm::CH][Gm::P];
    load_rows<D>(prm.table, warp, lane, 0, t);
    grid_wait();
    RowMap out_map;
    if (!resolve_out_map(prm, out_map)) return;   // uniform over the grid: no barrier is left waiting
    if constexpr (Gm::kLoops) {
        const int64_t n_batches = (prm.N + kV - 1) / kV;
#pragma unroll 1
        for (int64_t batch = blockIdx.x; batch < n_batches; batch += gridDim.x)
            encode_batch<D, BF16, FLUSH>(prm, out_map, t, xs, red, warp, lane, batch, batch + gridDim.x >= n_batches);
    } else {
        encode_batch<D, BF16, FLUSH>(prm, out_map, t, xs, red, warp, lane, blockIdx.x, true);
    }
}

// ------------------------------------------------------------------------------------------------
// decode: codes and scales -> x^  (Sec. 3.1: Eq. 2 undone, inverse real DFT, signs last; 1 / max(lambda, 1e-6) of Sec. 5.1)
// ------------------------------------------------------------------------------------------------
// the CTA's stored vectors, dequantised: q sigma / max(lambda, 1e-6), four coordinates per thread and pass
template <int D>
__device__ __forceinline__ void dequantise_batch(const MatvecParams &prm, float *zs, int64_t batch)
{
    const int64_t v0 = batch * kV;
    const unsigned char *pk = static_cast<const unsigned char *>(prm.packed);
    const uint16_t *scl = static_cast<const uint16_t *>(prm.scales);
    const int G = D / prm.group;
    for (int idx = threadIdx.x; idx < kV * (D / 4); idx += kWarps * 32) {
        const int v = idx / (D / 4), i = idx % (D / 4);
        const int64_t r = v0 + v;
        float4 o = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        if (r < prm.N) {
            const int64_t irow = prm.map(r);
            int q[4];
            if (prm.bits == 4) {
                const uint32_t w = load_input(reinterpret_cast<const uint16_t *>(pk + irow * (D / 2) + 2 * i));
#pragma unroll
                for (int e = 0; e < 4; ++e) q[e] = (int)(((w >> (4 * e)) & 0xFu) ^ 8u) - 8;
            } else {
                const uint32_t w = load_input(reinterpret_cast<const uint32_t *>(pk + irow * D + 4 * i));
#pragma unroll
                for (int e = 0; e < 4; ++e) q[e] = (int)(signed char)((w >> (8 * e)) & 0xFFu);
            }
            const float sig = __half2float(__ushort_as_half(load_input(scl + irow * G + (4 * i) / prm.group)));
            const float4 l = load_input(reinterpret_cast<const float4 *>(prm.lambda + lambda_row(r, prm.n_lambda, prm.rows_per_lambda) * D) + i);
            o.x = (float)q[0] * (sig * __frcp_rn(fmaxf(l.x, 1e-6f)));
            o.y = (float)q[1] * (sig * __frcp_rn(fmaxf(l.y, 1e-6f)));
            o.z = (float)q[2] * (sig * __frcp_rn(fmaxf(l.z, 1e-6f)));
            o.w = (float)q[3] * (sig * __frcp_rn(fmaxf(l.w, 1e-6f)));
        }
        *reinterpret_cast<float4 *>(zs + v * D + 4 * i) = o;
    }
}

template <int D, bool BF16>
__device__ __forceinline__ void decode_batch(const MatvecParams &prm, float4 (&t)[Geo<D>::CH][Geo<D>::P], float *zs, float *red, int warp,
                                             int lane, int64_t batch, bool last)
{
    using Gm = Geo<D>;
    constexpr int P = Gm::P;
    const int64_t v0 = batch * kV;

    dequantise_batch<D>(prm, zs, batch);
    __syncthreads();
    if (last) grid_trigger();   // nothing but the table is read from here on

    float y[P][4];
    matvec<D>(prm.table, t, zs, red, warp, lane, y);

    const int64_t r = v0 + warp;
    if (r >= prm.N) return;
    unsigned char *out = static_cast<unsigned char *>(prm.out) + prm.map(r) * (2 * D);
#pragma unroll
    for (int p = 0; p < P; ++p) {
        const int i = lane + 32 * p;
        if (i < D / 4)
            *reinterpret_cast<uint2 *>(out + 8 * i) = make_uint2(narrow2<BF16>(y[p][0], y[p][1]), narrow2<BF16>(y[p][2], y[p][3]));
    }
}

template <int D, bool BF16>
__global__ void __launch_bounds__(kWarps * 32) kvq_decode_matvec_kernel(const __grid_constant__ MatvecParams prm)
{
    using Gm = Geo<D>;
    extern __shared__ __align__(16) float sm[];
    float *zs = sm, *red = sm + kV * D;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    float4 t[Gm::CH][Gm::P];
    load_rows<D>(prm.table, warp, lane, 0, t);   // in flight while the codes are fetched and dequantised
    grid_wait();
    if constexpr (Gm::kLoops) {   // as in the encode kernel
        const int64_t n_batches = (prm.N + kV - 1) / kV;
#pragma unroll 1
        for (int64_t batch = blockIdx.x; batch < n_batches; batch += gridDim.x)
            decode_batch<D, BF16>(prm, t, zs, red, warp, lane, batch, batch + gridDim.x >= n_batches);
    } else {
        decode_batch<D, BF16>(prm, t, zs, red, warp, lane, blockIdx.x, true);
    }
}

// ------------------------------------------------------------------------------------------------
// the smallest calls: the output coordinates of a batch over several CTAs
// ------------------------------------------------------------------------------------------------
// A call of a few batches leaves most of the chip idle while a CTA reads a whole table (64 KB at D = 128, 256 KB at D = 256, there in two
// passes) and makes 8 D^2 multiply-adds.  Here a CTA has 32 output coordinates of its batch, 64 at D = 256; 8 (16) lanes cover
// its part of a table row, and each quarter (half) of a warp takes two (four) of the eight vectors, so that every sum has the same terms
// in the same order: the results are those of the form above bit for bit.  Append of 64 vectors, back to
// back: D = 128 3.2 -> 2.6 us, 256 6.9 -> 3.6; 200 at D = 160 6.0 -> 3.0; 200 at D = 256 with one scale per vector 6.9 -> 4.4; decode of 64 at
// D = 256 6.8 -> 3.7; window flush of 8 x 15 rows at D = 256 12.3 -> 7.0.
// A group of 32 lies inside a slice.  What crosses slices, the row maximum of a plan with one scale per vector and the
// dequantized values of the window flush, goes through distributed shared memory; the CTAs of a batch are then a cluster (two or four:
// D = 96 and 160 would be three and five, and stay with the form above there).
// A CTA takes one batch, and the form is taken while the device holds all of them at once; beyond that the copies of
// the staging and the barriers cost more than they save.  sliced_tenths says where that is.
template <int D>
struct Slice {
    static constexpr int W = D == 256 ? 64 : 32, kSlices = D / W;   // coordinates per slice
    static constexpr bool kCluster = kSlices == 2 || kSlices == 4;
    static constexpr int Q = W / 4, kSub = 32 / Q, kSubV = kV / kSub;   // lanes per table row; parts of a warp, vectors of each
    static constexpr int KW = D / kWarps;                   // contraction indices per warp
    static constexpr int kSmemBytes = (2 * kV * D + kWarps * kV * W + kSlices * kV) * (int)sizeof(float);
};

template <int D>
__device__ __forceinline__ void slice_rows(const float *__restrict__ table, int slice, int warp, int lane, float4 (&t)[Slice<D>::KW])
{
    using S = Slice<D>;
#pragma unroll
    for (int k = 0; k < S::KW; ++k)
        t[k] = __ldg(reinterpret_cast<const float4 *>(table + (size_t)(warp * S::KW + k) * D + slice * S::W) + lane % S::Q);
}

// the sums of vector `warp`, coordinates 4 (lane % Q) .. + 3 of the slice, in every part of the warp
template <int D>
__device__ __forceinline__ float4 slice_matvec(const float4 (&t)[Slice<D>::KW], const float *xs, float *red, int warp, int lane)
{
    using S = Slice<D>;
    const int sub = lane / S::Q, i = lane % S::Q;
#pragma unroll
    for (int v = 0; v < S::kSubV; ++v) {
        const int vec = sub * S::kSubV + v;
        float4 a = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
#pragma unroll
        for (int k = 0; k < S::KW; ++k) {
            const float xk = xs[vec * D + warp * S::KW + k];
            a.x = fmaf(t[k].x, xk, a.x), a.y = fmaf(t[k].y, xk, a.y), a.z = fmaf(t[k].z, xk, a.z), a.w = fmaf(t[k].w, xk, a.w);
        }
        *reinterpret_cast<float4 *>(red + (warp * kV + vec) * S::W + 4 * i) = a;
    }
    __syncthreads();
    float4 y = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
#pragma unroll
    for (int w = 0; w < kWarps; ++w) {
        const float4 a = *reinterpret_cast<const float4 *>(red + (w * kV + warp) * S::W + 4 * i);
        y.x += a.x, y.y += a.y, y.z += a.z, y.w += a.w;
    }
    return y;
}

template <int D, bool BF16, bool FLUSH>
__global__ void __launch_bounds__(kWarps * 32, D == 256 ? 1 : 2) kvq_encode_matvec_sliced_kernel(const __grid_constant__ MatvecParams prm)
{
    using S = Slice<D>;
    extern __shared__ __align__(16) float sm[];
    float *xs = sm, *back = xs + kV * D, *red = back + kV * D, *peak = red + kWarps * kV * S::W;   // peak: [slice][vector]
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, i = lane % S::Q, sub = lane / S::Q;
    const int slice = (int)blockIdx.x % S::kSlices, c0 = slice * S::W + 4 * i;   // this lane's coordinates
    const bool per_vector = prm.group == D, cluster = FLUSH || per_vector;

    float4 t[S::KW];
    slice_rows<D>(prm.table, slice, warp, lane, t);
    if (cluster) cluster_arrive();   // all four have begun: waited for in front of the first access to a partner's memory
    grid_wait();
    RowMap out_map;
    const bool ok = resolve_out_map(prm, out_map);   // uniform over the grid
    if (cluster) cluster_wait();
    if (!ok) return;
    const int64_t batch = blockIdx.x / S::kSlices;
    const int64_t r = batch * kV + warp;   // the vector this warp finishes
    const bool live = r < prm.N;
    const float4 l = load_input(reinterpret_cast<const float4 *>(prm.lambda + lambda_row(live ? r : prm.N - 1, prm.n_lambda, prm.rows_per_lambda) * D + c0));
    const uint32_t *x = static_cast<const uint32_t *>(prm.in);
    for (int idx = threadIdx.x; idx < kV * (D / 2); idx += kWarps * 32) {
        const int64_t row = batch * kV + idx / (D / 2);
        const float2 f = widen2<BF16>(row < prm.N ? load_input(x + row * (D / 2) + idx % (D / 2)) : 0u);   // rows past the end are zeros
        xs[2 * idx] = f.x, xs[2 * idx + 1] = f.y;
    }
    __syncthreads();
    grid_trigger();   // nothing but the tables is read from here on
    float4 z = slice_matvec<D>(t, xs, red, warp, lane);

    // ---- warp w finishes this slice of vector w: the quantizer of encode_batch
    z.x *= l.x, z.y *= l.y, z.z *= l.z, z.w *= l.w;
    float amax = fmaxf(fmaxf(fabsf(z.x), fabsf(z.y)), fmaxf(fabsf(z.z), fabsf(z.w)));
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) amax = fmaxf(amax, __shfl_xor_sync(0xFFFFFFFFu, amax, o));   // 8 lanes are a group
    if (per_vector) {
#pragma unroll
        for (int o = 8; o < S::Q; o <<= 1) amax = fmaxf(amax, __shfl_xor_sync(0xFFFFFFFFu, amax, o));
        float *to = peak + slice * kV + warp;
        if (lane < S::kSlices) cluster_st_u32(cluster_map(smem_u32(to), (uint32_t)lane), __float_as_uint(amax));
        cluster_sync_all();
#pragma unroll
        for (int s = 0; s < S::kSlices; ++s) amax = fmaxf(amax, peak[s * kV + warp]);
    }
    const int64_t orow = live ? out_map(r) : 0;
    const float Q = prm.bits == 4 ? 7.0f : 127.0f;
    const __half hs = __float2half_rn(fminf(__fdiv_rn(amax, Q), 65504.0f));   // codes are taken against the stored value
    const float sg = __half2float(hs);
    const float rs = sg > 0.0f ? __frcp_rn(sg) : 0.0f;
    const bool clamp = !(amax * rs < Q + 0.25f);   // saturated or subnormal scale: codes could leave [-Q, Q]
    const bool stores = live && sub == 0;
    if (stores && (per_vector ? c0 == 0 : (i & 7) == 0)) static_cast<uint16_t *>(prm.scales)[orow * (D / prm.group) + (per_vector ? 0 : c0 >> 5)] = __half_as_ushort(hs);
    const float zz[4] = {z.x, z.y, z.z, z.w};
    uint32_t code[4];
    float qf[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        const float v = clamp ? fminf(fmaxf(zz[e] * rs, -Q), Q) + 12582912.0f : fmaf(zz[e], rs, 12582912.0f);
        code[e] = __float_as_uint(v);   // low bits: q in two's complement (1.5 * 2^23 + q)
        qf[e] = v - 12582912.0f;        // q itself, exactly
    }
    if (stores) {
        unsigned char *pk = static_cast<unsigned char *>(prm.packed);
        if (prm.bits == 4) {
            const uint32_t w = (code[0] & 0xFu) | ((code[1] & 0xFu) << 4) | ((code[2] & 0xFu) << 8) | ((code[3] & 0xFu) << 12);
            *reinterpret_cast<uint16_t *>(pk + orow * (D / 2) + c0 / 2) = (uint16_t)w;
        } else {
            const uint32_t w = (code[0] & 0xFFu) | ((code[1] & 0xFFu) << 8) | ((code[2] & 0xFFu) << 16) | (code[3] << 24);
            *reinterpret_cast<uint32_t *>(pk + orow * D + c0) = w;
        }
    }
    if constexpr (FLUSH) {   // the way back starts from the stored values
        const float o[4] = {qf[0] * (sg * __frcp_rn(fmaxf(l.x, 1e-6f))), qf[1] * (sg * __frcp_rn(fmaxf(l.y, 1e-6f))),
                            qf[2] * (sg * __frcp_rn(fmaxf(l.z, 1e-6f))), qf[3] * (sg * __frcp_rn(fmaxf(l.w, 1e-6f)))};
        float4 t2[S::KW];
        slice_rows<D>(prm.table2, slice, warp, lane, t2);   // in flight across the barrier
        for (int s = sub; s < S::kSlices; s += S::kSub) {   // every CTA of the cluster needs all of the vector
            const uint32_t to = cluster_map(smem_u32(back + warp * D + c0), (uint32_t)s);
#pragma unroll
            for (int e = 0; e < 4; ++e) cluster_st_u32(to + 4 * e, live ? __float_as_uint(o[e]) : 0u);
        }
        __syncwarp();
        cluster_sync_all();
        const float4 y = slice_matvec<D>(t2, back, red, warp, lane);
        if (stores)
            *reinterpret_cast<uint2 *>(static_cast<unsigned char *>(prm.out) + orow * (2 * D) + 2 * c0) = make_uint2(narrow2<BF16>(y.x, y.y), narrow2<BF16>(y.z, y.w));
    }
}

template <int D, bool BF16>
__global__ void __launch_bounds__(kWarps * 32, D == 256 ? 1 : 2) kvq_decode_matvec_sliced_kernel(const __grid_constant__ MatvecParams prm)
{
    using S = Slice<D>;
    extern __shared__ __align__(16) float sm[];
    float *zs = sm, *red = sm + 2 * kV * D;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int slice = (int)blockIdx.x % S::kSlices;
    float4 t[S::KW];
    slice_rows<D>(prm.table, slice, warp, lane, t);   // in flight while the codes are fetched and dequantised
    grid_wait();
    const int64_t batch = blockIdx.x / S::kSlices;
    dequantise_batch<D>(prm, zs, batch);
    __syncthreads();
    grid_trigger();   // nothing but the table is read from here on
    const float4 y = slice_matvec<D>(t, zs, red, warp, lane);
    const int64_t r = batch * kV + warp;
    if (r < prm.N && lane < S::Q)
        *reinterpret_cast<uint2 *>(static_cast<unsigned char *>(prm.out) + prm.map(r) * (2 * D) + 2 * (slice * S::W + 4 * lane)) =
            make_uint2(narrow2<BF16>(y.x, y.y), narrow2<BF16>(y.z, y.w));
}

// MODE: 0 decode, 1 encode, 2 encode + decode of the same rows (window flush)

// CTAs of the sliced form per ten SMs up to which a call takes it.  Two per SM fit (D = 256: one), and without clusters that is the
// limit but for the decode at D = 64, whose two halves share little (528 vectors 2.58 -> 2.21 us, 648 2.59 -> 2.52, 824 2.60 -> 2.69).  Clusters are
// placed inside a GPC and do not fill the last SMs; a second one on an SM waits for partners that run beside others: window flush at D = 64,
// 528 vectors 4.22 -> 3.95 us, 648 4.23 -> 4.31, 944 4.25 -> 5.39; D = 128, 176: 5.00 -> 4.85, 264: 4.99 -> 5.29, 592: 5.05 -> 10.4; D = 256, 264:
// 12.3 -> 8.0, 272: 12.3 -> 13.5; append with one scale per vector at D = 128, 264: 3.34 -> 3.28, 320: 3.34 -> 3.68; at D = 64 never (2.67 -> 2.85 at 112).
template <int D, int MODE>
constexpr int sliced_tenths(bool cluster, bool per_vector)
{
    return !cluster ? ((D == 64 && MODE == 0) || D == 256 ? 10 : 20) : D == 64 && per_vector ? 0 : D == 128 && MODE == 2 ? 6 : 9;
}

template <int D, bool BF16, int MODE>
constexpr auto sliced_kernel()
{
    if constexpr (MODE == 0) return &kvq_decode_matvec_sliced_kernel<D, BF16>;
    else return &kvq_encode_matvec_sliced_kernel<D, BF16, MODE == 2>;
}

template <int D, bool BF16, int MODE>
cudaError_t launch(const MatvecParams &prm, cudaStream_t stream)
{
    static DeviceSlots slots, sliced_slots;   // CTAs of the kernel that the device holds at once; its SMs, 0 where the sliced form does not fit as often as it is meant to
    int dev = 0;
    cudaError_t e = current_device_slot(&dev);
    if (e != cudaSuccess) return e;
    constexpr bool kSliced = MODE != 2 || Slice<D>::kCluster;
    auto kern = MODE == 0 ? kvq_decode_matvec_kernel<D, BF16> : MODE == 1 ? kvq_encode_matvec_kernel<D, BF16, false> : kvq_encode_matvec_kernel<D, BF16, true>;
    if (slots.sms[dev] == 0) {
        int sms = 0, per_sm = 0;
        if ((e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, Geo<D>::kSmemBytes)) != cudaSuccess) return e;
        if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
        if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kWarps * 32, Geo<D>::kSmemBytes)) != cudaSuccess) return e;
        if constexpr (kSliced) {
            int sliced_per_sm = 0;
            auto sliced = sliced_kernel<D, BF16, MODE>();
            if ((e = cudaFuncSetAttribute(sliced, cudaFuncAttributeMaxDynamicSharedMemorySize, Slice<D>::kSmemBytes)) != cudaSuccess) return e;
            if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&sliced_per_sm, sliced, kWarps * 32, Slice<D>::kSmemBytes)) != cudaSuccess) return e;
            sliced_slots.sms[dev] = sliced_per_sm >= (D == 256 ? 1 : 2) ? sms : 0;
        }
        slots.sms[dev] = sms * (per_sm > 0 ? per_sm : 1);
    }
    if (prm.N == 0) return cudaSuccess;   // kvq_plan_prepare: the launch attributes are set, there is nothing to run
    const int64_t batches = (prm.N + kV - 1) / kV;
    if (batches > 0x7FFFFFFF) return cudaErrorInvalidValue;
    if constexpr (kSliced) {
        constexpr int kSlices = Slice<D>::kSlices;
        const bool cluster = MODE == 2 || (MODE == 1 && prm.group == D);
        if (10 * batches * kSlices <= (int64_t)sliced_tenths<D, MODE>(cluster, prm.group == D) * sliced_slots.sms[dev] && (Slice<D>::kCluster || !cluster))
            return launch_kernel(sliced_kernel<D, BF16, MODE>(), (unsigned)(batches * kSlices), kWarps * 32, Slice<D>::kSmemBytes, stream, cluster ? kSlices : 1, prm);
    }
    // one resident wave of CTAs that loop over batches where the kernel does; else a CTA per batch
    const int ctas = (int)(Geo<D>::kLoops && batches > slots.sms[dev] ? slots.sms[dev] : batches);
    return launch_kernel(kern, (unsigned)ctas, kWarps * 32, Geo<D>::kSmemBytes, stream, 1, prm);
}

template <int MODE>
cudaError_t dispatch(int D, bool bf16, const MatvecParams &prm, cudaStream_t stream)
{
    switch (D) {
        case 64: return bf16 ? launch<64, true, MODE>(prm, stream) : launch<64, false, MODE>(prm, stream);
        case 96: return bf16 ? launch<96, true, MODE>(prm, stream) : launch<96, false, MODE>(prm, stream);
        case 128: return bf16 ? launch<128, true, MODE>(prm, stream) : launch<128, false, MODE>(prm, stream);
        case 160: return bf16 ? launch<160, true, MODE>(prm, stream) : launch<160, false, MODE>(prm, stream);
        case 256: return bf16 ? launch<256, true, MODE>(prm, stream) : launch<256, false, MODE>(prm, stream);
    }
    return cudaErrorInvalidValue;
}

MatvecParams from_fft(const FftParams &f, const float *table, int group, int bits)
{
    MatvecParams p;
    p.in = f.in, p.lambda = f.lambda, p.packed = f.packed, p.scales = f.scales, p.out = f.out;
    p.table = table;
    p.table2 = nullptr;
    p.N = f.N, p.n_lambda = f.n_lambda, p.rows_per_lambda = f.rows_per_lambda;
    p.map = f.out_map;
    p.group = group, p.bits = bits;
    p.pos_dev = nullptr, p.pos_limit = 0, p.status = f.status;
    return p;
}

}  // namespace

// b0: the plan's [n][c] table; e0: its transpose
cudaError_t matvec_encode(int D, int group, int bits, bool bf16, int64_t N, const FftParams &f, const float *b0, cudaStream_t stream,
                          const DevicePos *pos)
{
    (void)N;
    MatvecParams p = from_fft(f, b0, group, bits);
    if (pos) p.pos_dev = pos->ptr, p.pos_limit = pos->limit;
    return dispatch<1>(D, bf16, p, stream);
}

cudaError_t matvec_decode(int D, int group, int bits, bool bf16, int64_t N, const FftParams &f, const float *e0, cudaStream_t stream)
{
    (void)N;
    return dispatch<0>(D, bf16, from_fft(f, e0, group, bits), stream);
}

// The window flush in one launch: x rows -> codes and scales at rows out_map(r) of the caches, and the dequantized
// vectors at the same rows of f.out.
cudaError_t matvec_flush(int D, int group, int bits, bool bf16, int64_t N, const FftParams &f, const float *b0, const float *e0,
                         cudaStream_t stream, const DevicePos *pos)
{
    (void)N;
    MatvecParams p = from_fft(f, b0, group, bits);
    if (pos) p.pos_dev = pos->ptr, p.pos_limit = pos->limit;
    p.table2 = e0;
    return dispatch<2>(D, bf16, p, stream);
}

}  // namespace kvq

// Device-side building blocks shared by the libkvq kernels (sm_100a):
// compile-time trigonometry, compile-time loops, PTX wrappers for mbarrier and
// bulk asynchronous copies, and half-precision word helpers.
#pragma once

#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <stdint.h>

#include <type_traits>
#include <utility>

namespace kvq {

// Bits of the per-plan device status word.
enum : uint32_t {
    KVQ_DEV_LOAD_TIMEOUT = 1u,   // a bounded wait for a bulk load ran out
    KVQ_DEV_MMA_TIMEOUT = 2u,    // a bounded wait for a tensor-core commit ran out
    KVQ_DEV_SLOT_TIMEOUT = 4u,   // a bounded wait for a free pipeline slot ran out
    KVQ_DEV_RANGE = 8u,          // reserved: tiles outside the fp16 operands' range are redone in fp32 by the decode kernels themselves
    KVQ_DEV_POSITION = 16u,      // a cache position read from device memory was outside the cache: nothing was written
};

// ---------------------------------------------------------------------------
// compile-time loops: static_for<N>([&](auto i) { constexpr int I = decltype(i)::value; ... })
// ---------------------------------------------------------------------------
template <class F, int... I>
__device__ __forceinline__ void static_for_impl(F &&f, std::integer_sequence<int, I...>)
{
    (f(std::integral_constant<int, I>{}), ...);
}

template <int N, class F>
__device__ __forceinline__ void static_for(F &&f)
{
    static_for_impl(static_cast<F &&>(f), std::make_integer_sequence<int, N>{});
}

// ---------------------------------------------------------------------------
// compile-time trigonometry: cos / sin of 2 pi n / d with exact octant reduction
// on the integers and a Taylor series on [0, pi/4].  Evaluated by the compiler
// only; every twiddle factor becomes an immediate.
// ---------------------------------------------------------------------------
constexpr double kTwoPi = 6.283185307179586476925286766559;

constexpr double ct_cos_small(double x)
{
    double x2 = x * x, term = 1.0, sum = 1.0;
    for (int i = 1; i <= 13; ++i) {
        term *= -x2 / (double)((2 * i - 1) * (2 * i));
        sum += term;
    }
    return sum;
}

constexpr double ct_sin_small(double x)
{
    double x2 = x * x, term = x, sum = x;
    for (int i = 1; i <= 13; ++i) {
        term *= -x2 / (double)((2 * i) * (2 * i + 1));
        sum += term;
    }
    return sum;
}

constexpr double ct_cos2pi(long long n, long long d)
{
    n %= d;
    if (n < 0) n += d;
    long long a = 8 * n;            // angle = 2 pi a / (8 d); d <-> pi/4, 2d <-> pi/2, 4d <-> pi
    if (a > 4 * d) a = 8 * d - a;   // cos(2 pi - x) = cos x
    bool neg = false;
    if (a > 2 * d) {                // cos(pi - x) = -cos x
        a = 4 * d - a;
        neg = true;
    }
    double r = (a > d) ? ct_sin_small(kTwoPi * (double)(2 * d - a) / (double)(8 * d))   // cos x = sin(pi/2 - x)
                       : ct_cos_small(kTwoPi * (double)a / (double)(8 * d));
    return neg ? -r : r;
}

constexpr double ct_sin2pi(long long n, long long d) { return ct_cos2pi(4 * n - d, 4 * d); }

constexpr double ct_sqrt(double x)
{
    double r = x > 1.0 ? x : 1.0;
    for (int i = 0; i < 200; ++i) r = 0.5 * (r + x / r);
    return r;
}

// ---------------------------------------------------------------------------
// PTX wrappers
// ---------------------------------------------------------------------------
__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}

__device__ __forceinline__ void mbar_init_fence()
{
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

__device__ __forceinline__ void mbar_arrive(uint32_t bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}

__device__ __forceinline__ void mbar_arrive_expect_tx(uint32_t bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}

// takes `bytes` off what the barrier's current phase still expects, as a copy that landed would
__device__ __forceinline__ void mbar_complete_tx(uint32_t bar, uint32_t bytes)
{
    asm volatile("mbarrier.complete_tx.relaxed.cta.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}

// One look at an mbarrier's phase without the hardware's suspend window: true if the phase with this parity is complete.
__device__ __forceinline__ bool mbar_test_wait(uint32_t bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}

// Waits for the given phase of an mbarrier, but never for ever: after `limit` polls it
// gives up and returns false, so that a lost copy turns into an error code, not a hang.
__device__ __forceinline__ bool mbar_wait_bounded(uint32_t bar, uint32_t parity, uint32_t limit = (1u << 22))
{
    for (uint32_t it = 0; it < limit; ++it) {
        if (mbar_try_wait(bar, parity)) return true;
        if (it > 64) __nanosleep(64);
    }
    return false;
}

// global -> shared bulk copy (TMA, untiled); bytes % 16 == 0, both addresses 16-byte aligned.
__device__ __forceinline__ void bulk_load(uint32_t dst_smem, const void *src_gmem, uint32_t bytes, uint32_t bar)
{
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst_smem),
                 "l"(src_gmem), "r"(bytes), "r"(bar)
                 : "memory");
}

// shared -> global bulk copy (TMA, untiled); joins the thread's current bulk group.
__device__ __forceinline__ void bulk_store(void *dst_gmem, uint32_t src_smem, uint32_t bytes)
{
    asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(dst_gmem), "r"(src_smem), "r"(bytes)
                 : "memory");
}

// asks for a contiguous run to be brought into L2; bytes % 16 == 0, address 16-byte aligned
__device__ __forceinline__ void prefetch_l2(const void *src_gmem, uint32_t bytes)
{
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(src_gmem), "r"(bytes) : "memory");
}

__device__ __forceinline__ void bulk_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }

// Waits until the shared-memory sources of all this thread's bulk stores have been read.
__device__ __forceinline__ void bulk_wait_read_all() { asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory"); }

// Waits until all this thread's bulk stores have completed.
__device__ __forceinline__ void bulk_wait_all() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }

// Programmatic dependent launch.  The kernels of this library are launched with the attribute that lets a grid's blocks come up
// while its predecessor on the stream runs out (launch_kernel in kvq_internal.h): the launch, the set-up of barriers and tensor
// memory and the requests for table rows then run under the predecessor's last tiles.  grid_wait() returns once every grid ahead on
// the stream is complete and its writes are visible, and stands before the first access to anything but the plan's tables (which
// only host calls and kernels without an early trigger write).  Every thread takes the wait, so that no grid is complete before the
// grids ahead of it.  Results rest on that wait alone.  grid_trigger() only says when the successor's blocks may come up: once every
// block has had a thread there or has ended.  It stands where a block's last input is on its way or in, in the tensor-core kernels
// behind the producer's last load (a tile that is decoded again in fp32 is read later), in the register-FFT kernels where a block's
// first warp is done.  At entry it costs more than it hides, blocks then sit on SMs that a call leaves idle long before the
// rest of their grid (encode + decode of 99,993 vectors, D = 160, bf16: 78.7 us without any of this, 83.5 us with the trigger at entry,
// 76.5 us so; 5120 appends at D = 128, back to back: 12.3 -> 9.7 us).  Behind another program's kernel, which does not trigger early, a
// call gains less (those appends behind a small elementwise kernel: 12.3 -> 11.3 us).
__device__ __forceinline__ void grid_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void grid_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// Loads of what the grids ahead on the stream may have written (x, lambda, codes, scales, positions): coherent, and behind grid_wait(),
// which a volatile statement does not pass.  __ldg is neither: the non-coherent load is for memory that nobody writes
// while the kernel runs, from its launch on, and the compiler may move it past the wait.  It is for the plan's tables.
// (As ordinary loads of C++ the same reads hold up what stands around them more: 212,992 bf16 vectors decoded at D = 256 under 52
// lambda rows 54.9 us, so 54.3, through __ldg 54.3, alternating on one box; boxes and what ran before move that call between 53 and 59.)
__device__ __forceinline__ uint16_t load_input(const uint16_t *p)
{
    uint16_t v;
    asm volatile("ld.global.u16 %0, [%1];" : "=h"(v) : "l"(p));
    return v;
}
__device__ __forceinline__ uint32_t load_input(const uint32_t *p)
{
    uint32_t v;
    asm volatile("ld.global.u32 %0, [%1];" : "=r"(v) : "l"(p));
    return v;
}
__device__ __forceinline__ int64_t load_input(const int64_t *p)
{
    int64_t v;
    asm volatile("ld.global.s64 %0, [%1];" : "=l"(v) : "l"(p));
    return v;
}
__device__ __forceinline__ uint2 load_input(const uint2 *p)
{
    uint2 v;
    asm volatile("ld.global.v2.u32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "l"(p));
    return v;
}
__device__ __forceinline__ uint4 load_input(const uint4 *p)
{
    uint4 v;
    asm volatile("ld.global.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
    return v;
}
__device__ __forceinline__ float load_input(const float *p)
{
    float v;
    asm volatile("ld.global.f32 %0, [%1];" : "=f"(v) : "l"(p));
    return v;
}
__device__ __forceinline__ float4 load_input(const float4 *p)
{
    float4 v;
    asm volatile("ld.global.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "l"(p));
    return v;
}

// Makes generic-proxy writes to shared memory visible to the async proxy (TMA, tensor core).
__device__ __forceinline__ void fence_proxy_async() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

// ---------------------------------------------------------------------------
// Division by a number that the host knows.  The chip divides 64-bit integers in a chain of some hundred instructions, and every role of a
// persistent kernel began with several such chains, one behind the other: 1.0 us of an encode's 6.7 per launch at one tile per CTA
// (globaltimer marks in the kernel) stood between a CTA's start and its set-up barrier, 0.3 more in front of each role's first tile.
// With m = ceil(2^(31 + s) / d), s = ceil(log2 d): floor(n m / 2^(31 + s)) = floor(n / d) for n < 2^31, because m d - 2^(31 + s) < d <= 2^s
// (Granlund and Montgomery's multiplication by an invariant reciprocal).
// ---------------------------------------------------------------------------
struct FastDiv {
    int64_t d;
    uint32_t mul, shift;
    FastDiv() = default;
    __host__ FastDiv(int64_t divisor) : d(divisor < 1 ? 1 : divisor), mul(0x80000000u), shift(0)
    {
        if (d == 1) return;
        if (d >> 31) {   // 2^31 and more: 0 for every n < 2^31
            mul = 0;
            return;
        }
        shift = 32u - (uint32_t)__builtin_clz((uint32_t)(d - 1));
        mul = (uint32_t)((((uint64_t)1 << (31 + shift)) + (uint64_t)d - 1) / (uint64_t)d);
    }
    __host__ __device__ __forceinline__ uint32_t small(uint32_t n) const   // n < 2^31
    {
#ifdef __CUDA_ARCH__
        return __umulhi(2u * n, mul) >> shift;
#else
        return (uint32_t)(((uint64_t)n * mul) >> 31 >> shift);
#endif
    }
    __host__ __device__ __forceinline__ int64_t operator()(int64_t n) const { return n >> 31 ? n / d : (int64_t)small((uint32_t)n); }   // n >= 0
};

// ---------------------------------------------------------------------------
// Tiles of the tensor-core kernels.  Rows are cut into lambda segments of `rpl` rows, a segment into
// tiles of 128 rows (the last one of a segment may be short), tiles are numbered segment by segment.
//
// The contiguous share of a call's tiles that one CTA (or one CTA pair) of a persistent kernel takes: lambda segments of rpl
// rows are cut into tiles of 128 rows (256 where a CTA pair works on one tile) (a segment's last tile may be short), n_seg * tps tiles
// in all, `parts` shares.
// Contiguous, so that the B operand of a lambda row is rebuilt as rarely as possible.  `segs` consecutive segments have one
// lambda row (1, or the streams of a cache view that share theirs; the last row may have fewer).  A share that crosses into
// another lambda row pays a rebuild of B on its critical path, one to two tiles' time, so:
//   * where no more lambda rows than shares exist and the longest share grows by no more than that, every share stays inside one
//     lambda row (90,000 vectors under 30 rows, shares equal in tiles
//     against this: encode D = 160 25.2 and 18.1 us, decode D = 128 bf16 14.5 and 12.0, D = 256 31.2 and 28.9);
//   * else, with at least eight tiles per share, the shares are equal in COST, a lambda row counting one unit, the price's lower end,
//     more than its tiles (a share that would begin inside that unit begins at the row's first tile);
//   * else they are equal in tiles.
// TilePlan is the call's half of that, worked out by the host (fewer than 2^31 tiles); TileShare is a CTA's.
// Shares without a tile are not launched: the next call's blocks come up on the SMs they leave, and its last one does not wait for the
// last SM of this one (append + decode of 112 x 1152 rows, whose decode has 112 shares of nine tiles, 16.1 -> 15.8 us; D = 96 round trip
// of 65,536, 128 of four, 16.05 -> 15.9).
// ---------------------------------------------------------------------------
struct TilePlan {
    uint32_t tps;         // tiles per segment
    uint32_t n_tiles;
    uint32_t row_tiles;   // tiles per lambda row
    uint32_t n_rows;      // lambda rows
    uint32_t inside;      // shares stay inside lambda rows: per_row of them each
    uint32_t per;         // tiles (inside) or cost units per share
    uint32_t rebuild;     // cost units of a rebuild
    uint32_t shares;      // that have tiles, `parts` or fewer: the CTAs (CTA pairs) to launch
    FastDiv by_tps, by_per_row, by_cost;   // by_cost: units per lambda row
    TilePlan() = default;
    __host__ TilePlan(int64_t n_seg, int64_t rpl, unsigned parts, int tile_rows = 128, int64_t segs = 1)
    {
        const int64_t t = (rpl + tile_rows - 1) / tile_rows, tiles = n_seg * t;
        if (segs > n_seg) segs = n_seg;
        const int64_t rt = segs * t, rows = (n_seg + segs - 1) / segs, even = (tiles + parts - 1) / parts;
        tps = (uint32_t)t, n_tiles = (uint32_t)tiles, row_tiles = (uint32_t)rt, n_rows = (uint32_t)rows;
        inside = rebuild = 0;
        by_tps = FastDiv(t), by_per_row = by_cost = FastDiv(1);
        if (rows <= (int64_t)parts) {
            const int64_t k = parts / rows, p = (rt + k - 1) / k;   // shares per lambda row, tiles per share
            if (p <= even + 2 || rows == 1) {
                const int64_t used = (rt + p - 1) / p, last = tiles - (rows - 1) * rt;   // the last row may have fewer streams
                inside = 1, per = (uint32_t)p, shares = (uint32_t)((rows - 1) * used + (last + p - 1) / p), by_per_row = FastDiv(used);
                return;
            }
        }
        rebuild = tiles >= 8 * (int64_t)parts ? 1 : 0;
        by_cost = FastDiv(rt + rebuild);
        per = (uint32_t)((tiles + rows * rebuild + parts - 1) / parts);
        shares = (uint32_t)((tiles + rows * rebuild + per - 1) / per);
    }
};

struct TileShare {
    int64_t tps;     // tiles per segment
    int64_t begin;   // first tile of this share
    int n;           // tiles in this share
    uint32_t seg, tin;   // segment of the first tile, and its place there
    __host__ __device__ __forceinline__ TileShare(const TilePlan &p, uint32_t part) : tps(p.tps)
    {
        uint32_t from, to;
        if (p.inside) {
            const uint32_t row = p.by_per_row.small(part), r0 = row * p.row_tiles, at = (part - row * (uint32_t)p.by_per_row.d) * p.per;
            from = r0 + at, to = r0 + (p.row_tiles - at > p.per && at < p.row_tiles ? at + p.per : p.row_tiles);
            if (to > p.n_tiles) to = p.n_tiles;
            if (row >= p.n_rows) to = from;
        } else {
            const int64_t total = (int64_t)p.n_tiles + (int64_t)p.n_rows * p.rebuild, u = (int64_t)part * p.per;
            auto tile_of = [&](int64_t v) -> uint32_t {
                if (v >= total) return p.n_tiles;
                const int64_t row = p.by_cost(v);
                const uint32_t w = (uint32_t)(v - row * p.by_cost.d);
                return (uint32_t)row * p.row_tiles + (w > p.rebuild ? w - p.rebuild : 0u);
            };
            from = tile_of(u), to = tile_of(u + p.per);
        }
        n = to > from ? (int)(to - from) : 0;
        begin = from;
        if (n == 0) from = 0;
        seg = p.by_tps.small(from);
        tin = from - seg * p.tps;
    }
};

// Walks a CTA's tiles, from its first one on.
struct TileCursor {
    int seg;   // lambda segment of the current tile
    int tin;   // index of the tile within its segment
    int tps;   // tiles per segment
    __device__ __forceinline__ TileCursor(const TileShare &s) : seg((int)s.seg), tin((int)s.tin), tps((int)s.tps) {}
    __device__ __forceinline__ TileCursor(const TileShare &s, int step) : TileCursor(s) { advance(step); }
    __device__ __forceinline__ void advance(int step)
    {
        tin += step;
        while (tin >= tps) {
            tin -= tps;
            ++seg;
        }
    }
    __device__ __forceinline__ bool first_of_segment() const { return tin == 0; }
    __device__ __forceinline__ int64_t row_in_segment() const { return (int64_t)tin * 128; }
};

// ---------------------------------------------------------------------------
// half-precision words: two 16-bit values per 32-bit word, low half first
// ---------------------------------------------------------------------------
template <bool BF16>
__device__ __forceinline__ float2 widen2(uint32_t w)
{
    if constexpr (BF16) {
        return make_float2(__uint_as_float(w << 16), __uint_as_float(w & 0xFFFF0000u));
    } else {
        __half2 h = *reinterpret_cast<__half2 *>(&w);
        return __half22float2(h);
    }
}

template <bool BF16>
__device__ __forceinline__ uint32_t narrow2(float lo, float hi)
{
    if constexpr (BF16) {
        __nv_bfloat162 b = __floats2bfloat162_rn(lo, hi);
        return *reinterpret_cast<uint32_t *>(&b);
    } else {
        __half2 h = __floats2half2_rn(lo, hi);
        return *reinterpret_cast<uint32_t *>(&h);
    }
}

// ---------------------------------------------------------------------------
// two fp32 values in one 64-bit register: sums and differences of both in one instruction, each rounded like the single one
// ---------------------------------------------------------------------------
__device__ __forceinline__ uint64_t pack_f32x2(float lo, float hi)
{
    uint64_t d;
    asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "f"(lo), "f"(hi));
    return d;
}

__device__ __forceinline__ float2 unpack_f32x2(uint64_t v)
{
    float2 f;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(f.x), "=f"(f.y) : "l"(v));
    return f;
}

__device__ __forceinline__ uint64_t add_f32x2(uint64_t a, uint64_t b)
{
    uint64_t d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}

__device__ __forceinline__ uint64_t mul_f32x2(uint64_t a, uint64_t b)
{
    uint64_t d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}

__device__ __forceinline__ uint64_t fma_f32x2(uint64_t a, uint64_t b, uint64_t c)
{
    uint64_t d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}

__device__ __forceinline__ uint64_t sub_f32x2(uint64_t a, uint64_t b)
{
    uint64_t d;
    asm("fma.rn.f32x2 %0, %2, %3, %1;" : "=l"(d) : "l"(a), "l"(b), "l"(0xBF800000BF800000ull));   // a - 1 b, one rounding
    return d;
}

// ---------------------------------------------------------------------------
// round-to-nearest-even codes by the magic-number trick (Sec. 3.2 step 4): v / sigma + 1.5 * 2^23 (+ bias) has the
// biased code in its low mantissa bits, so eight nibbles (four bytes) are gathered with shifts and one subtraction
// ---------------------------------------------------------------------------
constexpr float kMagicRound = 12582912.0f + 8.0f;          // 1.5 * 2^23 + 8: (v + magic) has q + 8 in its low bits
constexpr uint32_t kMagicBits = 0x4B400000u;
constexpr uint32_t kMagicSum = kMagicBits * 0x11111111u;   // sum_i kMagicBits * 16^i  (mod 2^32)
constexpr float kMagicRound8 = 12582912.0f + 128.0f;       // byte codes: q + 128 in the low byte
constexpr uint32_t kMagicSum8 = kMagicBits * 0x01010101u;  // sum_i kMagicBits * 256^i (mod 2^32)

__device__ __forceinline__ uint32_t lop3_and_or(uint32_t a, uint32_t b, uint32_t c)
{
    uint32_t d;
    asm("lop3.b32 %0, %1, %2, %3, 0xEA;" : "=r"(d) : "r"(a), "r"(b), "r"(c));   // (a & b) | c
    return d;
}

}  // namespace kvq

// Building blocks shared by the tcgen05 (5th-generation tensor core) kernels of libkvq: PTX wrappers for
// tensor memory, the MMA, TMA tensor copies, the shared-memory matrix descriptor, and the bounded
// mbarrier wait that lets a role give up without hanging its CTA.
#pragma once

#include <cuda.h>

#include "kvq_device.cuh"

namespace kvq {

// K-major operand with the 128-byte swizzle: start address >> 4 | LBO 0 | SBO 1024 B (8 rows x 128 B) | version 1 | swizzle
__device__ __forceinline__ uint64_t smem_desc_sw128(uint32_t addr)
{
    return (uint64_t)((addr & 0x3FFFFu) >> 4) | ((uint64_t)(1024u >> 4) << 32) | (1ull << 46) | (2ull << 61);
}

// instruction descriptor of kind::f16: D = f32, A and B both f16 (bf16 = false) or both bf16, both K-major
__host__ __device__ constexpr uint32_t umma_idesc(int m, int n, bool bf16)
{
    return (1u << 4) | ((bf16 ? 1u : 0u) << 7) | ((bf16 ? 1u : 0u) << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(m >> 4) << 24);
}
__host__ __device__ constexpr uint32_t umma_idesc_m128(int n, bool bf16) { return umma_idesc(128, n, bf16); }

__device__ __forceinline__ void tmem_alloc(uint32_t smem_dst, uint32_t cols)   // one warp, its first thread perhaps out of the barriers' set-up
{
    __syncwarp();
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_dst), "r"(cols) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}

__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t cols)
{
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(cols) : "memory");
}

// one lane of a converged warp
__device__ __forceinline__ bool elect_one()
{
    uint32_t pred;
    asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(pred));
    return pred != 0;
}

__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// D[tmem] (+)= A[tmem] * B[smem]
template <bool ACCUMULATE>
__device__ __forceinline__ void umma_f16_ts(uint32_t d_tmem, uint32_t a_tmem, uint64_t bdesc, uint32_t idesc)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}" ::"r"(d_tmem),
        "r"(a_tmem), "l"(bdesc), "r"(idesc), "n"(ACCUMULATE ? 1 : 0)
        : "memory");
}

// D[tmem] (+)= A[smem] * B[smem]
template <bool ACCUMULATE>
__device__ __forceinline__ void umma_f16_ss(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
        "l"(adesc), "l"(bdesc), "r"(idesc), "n"(ACCUMULATE ? 1 : 0)
        : "memory");
}

// the mbarrier gets one arrival when every tcgen05 operation this thread issued so far is complete
__device__ __forceinline__ void umma_commit(uint32_t bar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}

// ---- a pair of CTAs (thread-block cluster of two) on one tile: M = 256, each CTA's shared memory holds its own 128 rows of A
// ---- and half of B's rows, its tensor memory its own 128 rows of the accumulator.  Rank 0, the leader, issues.
__device__ __forceinline__ uint32_t cluster_rank()
{
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ uint32_t cluster_map(uint32_t smem_addr, uint32_t cta_rank)   // the same object in CTA cta_rank
{
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(smem_addr), "r"(cta_rank));
    return r;
}
__device__ __forceinline__ void cluster_st_u32(uint32_t cluster_addr, uint32_t v)
{
    asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(cluster_addr), "r"(v) : "memory");
}
__device__ __forceinline__ void cluster_mbar_arrive(uint32_t cluster_addr)
{
    asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(cluster_addr) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait_cluster(uint32_t bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}
// The .aligned forms want the whole warp at the instruction together, and a branch that some lanes take may stand in front (a store by the
// first lanes, a status bit by one thread): __syncwarp brings them together.
__device__ __forceinline__ void cluster_arrive()
{
    __syncwarp();
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_wait()
{
    __syncwarp();
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_sync_all()
{
    __syncwarp();
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_alloc_pair(uint32_t smem_dst, uint32_t cols)   // one warp of each CTA
{
    __syncwarp();
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_dst), "r"(cols) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc_pair(uint32_t taddr, uint32_t cols)
{
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(cols) : "memory");
}
// D[tmem of both] (+)= A[smem of both] * B[smem of both]
template <bool ACCUMULATE>
__device__ __forceinline__ void umma_f16_ss_pair(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
        "l"(adesc), "l"(bdesc), "r"(idesc), "n"(ACCUMULATE ? 1 : 0)
        : "memory");
}
// the mbarrier at this offset in each CTA of the pair gets one arrival when every tcgen05 operation issued so far is complete
__device__ __forceinline__ void umma_commit_pair(uint32_t bar)
{
    asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(bar),
                 "h"((uint16_t)3)
                 : "memory");
}
// Both CTAs of a pair load block after block, in order, into the same ring of slots.  The leader's barrier of a slot counts the bytes
// of both: its producer arms it for two loads together with its own.  Where the producers have stopped early, after leader and partner
// blocks, the leader owes the barriers of the last `ring` blocks what follows, and each phase then ends when the
// loads that are under way have landed.  (A producer is at most one ring ahead of the other: a slot is free once block u - ring is used.)
struct PairDrain {
    int leader, partner, ring;
    __host__ __device__ __forceinline__ int end() const { return leader > partner ? leader : partner; }
    __host__ __device__ __forceinline__ int begin() const { return end() > ring ? end() - ring : 0; }
    __host__ __device__ __forceinline__ bool owes_arrival(int u) const { return u >= leader; }    // the partner's load alone: armed by nobody
    __host__ __device__ __forceinline__ bool owes_bytes(int u) const { return u >= partner; }     // the leader's load alone: armed for two
    __host__ __device__ __forceinline__ int slot(int u) const { return u % ring; }
    __host__ __device__ __forceinline__ uint32_t parity(int u) const { return (uint32_t)(u / ring) & 1u; }
};

// TMA tensor load into this CTA's shared memory that completes on an mbarrier of the leader (a shared::cluster address)
__device__ __forceinline__ void tma_load_2d_pair(uint32_t dst_smem, const CUtensorMap *tm, int c0, int c1, uint32_t leader_bar)
{
    asm volatile("cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::"r"(
                     dst_smem),
                 "l"(reinterpret_cast<uint64_t>(tm)), "r"(c0), "r"(c1), "r"(leader_bar)
                 : "memory");
}

// 32 consecutive accumulator columns of this thread's tensor-memory lane
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t (&r)[32])
{
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
        "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
          "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]),
          "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
          "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr)
        : "memory");
}

// 16 consecutive accumulator columns of this thread's tensor-memory lane
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t (&r)[16])
{
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
          "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr)
        : "memory");
}

// Says behind a tmem_ld_wait() that these values have arrived: what uses them stays behind it, also where other work stands between
// the request and the wait.
template <int N>
__device__ __forceinline__ void tmem_loaded(uint32_t (&r)[N])
{
#pragma unroll
    for (int i = 0; i < N; i += 4) asm volatile("" : "+r"(r[i]), "+r"(r[i + 1]), "+r"(r[i + 2]), "+r"(r[i + 3]));
}

__device__ __forceinline__ void tmem_ld_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

// 16 consecutive columns of this thread's tensor-memory lane
__device__ __forceinline__ void tmem_st16(uint32_t taddr, const uint32_t (&r)[16])
{
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], "
        "{%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16};" ::"r"(taddr),
        "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]), "r"(r[9]),
        "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15])
        : "memory");
}

// 8 consecutive columns of this thread's tensor-memory lane
__device__ __forceinline__ void tmem_st8(uint32_t taddr, const uint32_t (&r)[8])
{
    asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"r"(taddr), "r"(r[0]), "r"(r[1]),
                 "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7])
                 : "memory");
}

__device__ __forceinline__ void tmem_st_wait() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

// TMA tensor load, two coordinates, completion on an mbarrier: a per-CTA load of this GPU's own memory
__device__ __forceinline__ void tma_load_2d(uint32_t dst_smem, const CUtensorMap *tm, int c0, int c1, uint32_t bar)
{
    asm volatile("cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::"r"(
                     dst_smem),
                 "l"(reinterpret_cast<uint64_t>(tm)), "r"(c0), "r"(c1), "r"(bar)
                 : "memory");
}

// TMA tensor store, three coordinates; joins the thread's current bulk group
__device__ __forceinline__ void tma_store_3d(const CUtensorMap *tm, int c0, int c1, int c2, uint32_t src_smem)
{
    asm volatile("cp.async.bulk.tensor.3d.global.shared::cta.tile.bulk_group [%0, {%1, %2, %3}], [%4];" ::"l"(
                     reinterpret_cast<uint64_t>(tm)),
                 "r"(c0), "r"(c1), "r"(c2), "r"(src_smem)
                 : "memory");
}

// The A operand of the decode kernels, q sigma rho, is fp16.  A row whose G stored scales (packed 16-bit pairs in sc)
// would take it out of fp16's normal range -- sigma rho above max_t (the largest code times it must fit) or a non-zero
// sigma rho below 2^-14 -- is carried times a power of two instead: the function returns that factor (1 for every other
// row) and its inverse through inv, which the epilogue applies to the row's accumulators in fp32.  The factor takes
// 2^floor(log2(largest sigma rho)) to 2^7, so the largest operand lands in [7 * 128, 7 * 256) (byte codes: below 32512).
template <int G>
__device__ __forceinline__ float operand_rescue(const uint32_t (&sc)[(G + 1) / 2], float rho, float max_t, float &inv)
{
    uint32_t smax = 0u, smin = 0xFFFFu;
#pragma unroll
    for (int c = 0; c < G; ++c) {
        const uint32_t s = (sc[c >> 1] >> (16 * (c & 1))) & 0x7FFFu;   // fp16 bits of a non-negative number order like integers
        smax = max(smax, s);
        if (s != 0u) smin = min(smin, s);
    }
    const float tmax = __half2float(__ushort_as_half((unsigned short)smax)) * rho;
    const float tmin = __half2float(__ushort_as_half((unsigned short)(smin == 0xFFFFu ? 0u : smin))) * rho;
    inv = 1.0f;
    if (!(tmax > max_t || (tmin != 0.0f && tmin < 6.1035156e-5f))) return 1.0f;
    const int e = (int)((__float_as_uint(fminf(fmaxf(tmax, 1e-30f), 1e30f)) >> 23) & 0xFFu) - 127;
    inv = __uint_as_float((uint32_t)(127 - 7 + e) << 23);
    return __uint_as_float((uint32_t)(127 + 7 - e) << 23);
}

// sigma rho of a row with one scale per vector, sigma in the low half of `sc`: what its sums of codes are multiplied by.  An infinite
// sigma gives NaN, the sum that infinite products of both signs and 0 times infinity would have.
__device__ __forceinline__ float vector_factor(uint32_t sc, float rho)
{
    const float sigma = __half2float(__ushort_as_half((unsigned short)(sc & 0xFFFFu)));
    return fmaf(sigma, rho, sigma - sigma);
}

// 1 / max(lambda, 1e-6) for the channels this lane covers (4 i .. 4 i + 3, i = lane and, for D > 128, lane + 32; NEIGHBOURS: i = 2 lane and
// 2 lane + 1), divided by rho, the power of two that brings the row's largest reciprocal into [1, 2).  Every lane gets rho.
template <int D, bool NEIGHBOURS = false>
struct RecipLambda {
    static constexpr int kPasses = (D / 4 + 31) / 32;
    static_assert(!NEIGHBOURS || D == 256, "two quads for every lane");
    float4 r[kPasses];
    float rho;
    bool wide;   // the reciprocals span more than 2^8: B, which carries them in fp16 next to each other, loses bits on the small ones
    __device__ __forceinline__ RecipLambda(const float *__restrict__ lam, int lane)
    {
        float mx = 0.0f, mn = 3.0e38f;
#pragma unroll
        for (int p = 0; p < kPasses; ++p) {
            const int i = NEIGHBOURS ? 2 * lane + p : lane + 32 * p;
            r[p] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
            if (i < D / 4) {
                const float4 l = load_input(reinterpret_cast<const float4 *>(lam) + i);
                r[p] = make_float4(__frcp_rn(fmaxf(l.x, 1e-6f)), __frcp_rn(fmaxf(l.y, 1e-6f)), __frcp_rn(fmaxf(l.z, 1e-6f)),
                                   __frcp_rn(fmaxf(l.w, 1e-6f)));
            }
            mx = fmaxf(mx, fmaxf(fmaxf(r[p].x, r[p].y), fmaxf(r[p].z, r[p].w)));
            if (i < D / 4) mn = fminf(mn, fminf(fminf(r[p].x, r[p].y), fminf(r[p].z, r[p].w)));
        }
        // Positive: ordered like their bits, and one redux each in place of five dependent shuffles; the row is scaled by an exact
        // reciprocal, one division in place of four (eight).  This stands between lambda's arrival and the first MMA, and again at every lambda
        // row: decode of 1500 fp16 vectors at D = 256 10.0 -> 9.6 us, of 7100 under four rows at D = 128 6.4 -> 6.25 (one after another; with the D = 256
        // decode's first operand as it was before FirstRows).
        mx = __uint_as_float(__reduce_max_sync(0xFFFFFFFFu, __float_as_uint(mx)));
        mn = __uint_as_float(__reduce_min_sync(0xFFFFFFFFu, __float_as_uint(mn)));
        rho = __uint_as_float(__float_as_uint(mx) & 0x7F800000u);   // 2^floor(log2 max): exact to divide by
        wide = mn < rho * 0.00390625f;
        const float inv = rho > 0.0f ? 1.0f / rho : 0.0f;   // every entry infinite, or as good as: nothing comes out of such a row
#pragma unroll
        for (int p = 0; p < kPasses; ++p) r[p].x *= inv, r[p].y *= inv, r[p].z *= inv, r[p].w *= inv;
    }
};

// Bounded wait that also gives up when another role of the CTA has raised the abort flag.  On a
// time-out it raises the flag itself and records `reason` in the status word.
constexpr uint32_t kWaitPolls = 1u << 22;   // polls of a bounded wait before it gives up (seconds of wall time)

__device__ __forceinline__ bool wait_or_abort(uint32_t bar, uint32_t parity, volatile uint32_t *abort_flag, uint32_t *status,
                                              uint32_t reason, uint32_t limit = kWaitPolls)
{
    for (uint32_t it = 0; it < limit; ++it) {
        if (mbar_try_wait(bar, parity)) return true;
        if (it > 32) {
            if (*abort_flag) return false;
            __nanosleep(32);
        }
    }
    *abort_flag = 1u;
    atomicOr(status, reason);
    return false;
}

// The mma role's wait for a CTA's first B operand where the host has shortened its limit (kvq_plan_set_wait_limit): the one wait that can
// be shortened, because the waiting thread has issued nothing yet and can leave at once.  The looks at the barrier do not block, so that
// "one poll" is over before the operand can possibly be there.
__device__ __forceinline__ bool wait_first_operand(uint32_t bar, volatile uint32_t *abort_flag, uint32_t *status, uint32_t limit)
{
    for (uint32_t it = 0; it < limit; ++it)
        if (mbar_test_wait(bar, 0u)) return true;
    *abort_flag = 1u;
    atomicOr(status, (uint32_t)KVQ_DEV_SLOT_TIMEOUT);
    return false;
}

// wait_or_abort with cluster-scope acquire: what the partner CTA wrote before its arrival is visible afterwards
__device__ __forceinline__ bool wait_cluster_or_abort(uint32_t bar, uint32_t parity, volatile uint32_t *abort_flag, uint32_t *status,
                                                      uint32_t reason)
{
    for (uint32_t it = 0; it < kWaitPolls; ++it) {
        if (mbar_try_wait_cluster(bar, parity)) return true;
        if (it > 32) {
            if (*abort_flag) return false;
            __nanosleep(32);
        }
    }
    *abort_flag = 1u;
    atomicOr(status, reason);
    return false;
}

// ---- host side: cuTensorMapEncodeTiled through the runtime's driver entry point (no link against libcuda)
typedef CUresult (*TensorMapEncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                           const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                                           CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

inline TensorMapEncodeTiledFn tensor_map_encode_fn()
{
    // looked up once; the initialisation of a function-local static is thread-safe
    static const TensorMapEncodeTiledFn fn = [] {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult qres;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &qres) == cudaSuccess &&
            qres == cudaDriverEntryPointSuccess)
            return reinterpret_cast<TensorMapEncodeTiledFn>(p);
        (void)cudaGetLastError();
        return static_cast<TensorMapEncodeTiledFn>(nullptr);
    }();
    return fn;
}

// A tensor map over `rank` dimensions of `base`; strides in bytes for dimensions 1 .. rank - 1.
inline bool make_tensor_map(CUtensorMap *tm, CUtensorMapDataType type, int rank, const void *base, const cuuint64_t *dims,
                            const cuuint64_t *strides, const cuuint32_t *box, CUtensorMapSwizzle swizzle)
{
    TensorMapEncodeTiledFn enc = tensor_map_encode_fn();
    if (!enc) return false;
    const cuuint32_t es[5] = {1, 1, 1, 1, 1};
    return enc(tm, type, (cuuint32_t)rank, const_cast<void *>(base), dims, strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE, swizzle,
               CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

}  // namespace kvq

// Warp-specialised tcgen05 DFT-as-GEMM append kernel of libkvq (sm_100a): fp16 input, every D, calls above the matrix-vector limit.
//
// The same contraction as kvq_umma_encode.cu and kvq_umma_encode256.cu (v = lambda (.) M (s (.) x), Sec. 3.1 Eq. 1-2, Sec. 5.1 item 1) with
// the same two fp16 terms of a factor of 22 bits, for a call of one row of thousands of streams (every layer, head and sequence of a
// decode step, Sec. 7.2): a tile or two per CTA, and a lambda row for every few dozen of its vectors.  So lambda stands in the epilogue,
// half a multiply per channel (mul.f32x2), and not in the B operand:
//
//   * B = M diag(s) 2^14 is the plan's alone: split and swizzled once (build_encode_operands), fetched by bulk copies while the grid ahead
//     on the stream runs out.  The kernels above build it from the fp32 table and lambda at the start of every call and again at every
//     lambda row: 2 us of a call of one tile per CTA.
//   * A tile is any 128 consecutive vectors, whatever lambda rows they have: 160 lambda rows of 32 vectors are 40 full tiles, not 160.
//
// Back to back, before -> now, caches of 2 rows per stream: D = 128, 5120 vectors under 160 lambda rows 9.4 -> 3.9 us, 4096 under one 6.1 -> 3.9; D = 256,
// 4950 under two 9.5 -> 5.0.  Of 256 rows, each vector's bytes then on lines and pages of their own: 9.4 -> 4.4, 6.1 -> 4.4, 9.8 -> 5.3.
// What is left is the launch (2.2 us), one tile's way through the roles and the stores' drain.
// Appends alone take it.  Where lambda is rounded decides one to three codes in a million, those at a tie, and kvq_encode and the block
// flush, whose rows are also compared dequantized, keep the rounding they have.  bf16 stays with the kernels above: with two bf16
// terms, 16 bits, it would be ten times as many.
//
//   warp 0        producer   one TMA tensor load per K block of 64 columns (128-byte swizzle) into a ring of blocks
//   warp 1        mma        per tile the small term's K-steps over all blocks, then the large one's, in one accumulator: the small sums are
//                            complete before anything large is in it; a block is released in the second pass
//   warps 2-17    epilogue   all sixteen warps on every tile, thread = (row, every fourth group of 32 channels): tcgen05.ld, times
//                            lambda, abs-max, fp16 scale, round-to-nearest-even codes, nibble pack, direct global stores
//
// D = 256: B (256 KB) does not fit a CTA; a CTA has 128 of the channels of its tiles, B's 128 rows of them (128 KB) and all of x.
// Every wait on an mbarrier is bounded: on a time-out the role records the reason in the status word, raises the CTA's abort flag and
// leaves its loop; the CTA then frees its tensor memory and returns.
#include "kvq_internal.h"
#include "kvq_quantize.cuh"
#include "kvq_umma.cuh"

namespace kvq {

namespace {

constexpr int kTile = 128;                 // vectors per tile = MMA M
constexpr int kGroup = 32;
constexpr int kThreads = 576;              // producer, mma, 16 epilogue warps
constexpr int kParts = 4;                  // epilogue threads per row
constexpr int kBlockBytes = kTile * 128;   // one K block of the x tile: 128 rows x 128 B
constexpr int kMaxRing = 8;
constexpr int kSmemLimit = 232448;         // 227 KB of dynamic shared memory per CTA
constexpr uint32_t kTmemCols = 512;

template <int D>
struct Cfg {
    static constexpr int kCh = D == 256 ? 128 : D;              // channels per CTA = MMA N
    static constexpr int kHalves = D / kCh;
    static constexpr int G = D / kGroup, kGroups = kCh / kGroup;
    static constexpr int kPerThread = (kGroups + kParts - 1) / kParts;
    static constexpr int kKBlocks = (D + 63) / 64;              // K blocks of 64 elements (the last one may be half used)
    static constexpr int kBBlock = kCh * 128;                   // one K block of one term of B
    static constexpr int kBTerm = kKBlocks * kBBlock;
    static constexpr int kBBytes = 2 * kBTerm;
    static constexpr int kCtrlBytes = 256 + 2 * kParts * kTile * (int)sizeof(float);   // barriers, then the row maxima: [tile parity][part][row]
    static constexpr int kRoom = (kSmemLimit - 1024 - kCtrlBytes - kBBytes) / kBlockBytes;
    static constexpr int kRing = kRoom < kMaxRing ? kRoom : kMaxRing;
    static_assert(kRing > kKBlocks, "a whole tile stays in the ring for two passes over it");
    static constexpr int kSmemBytes = kBBytes + kRing * kBlockBytes + kCtrlBytes + 1024;
    static constexpr uint32_t kAccStride = kCh <= 128 ? 128 : 160;
    static constexpr int kAccStages = 512 / (int)kAccStride;    // accumulators in tensor memory
    static constexpr uint32_t kIdesc = umma_idesc_m128(kCh, false);
};

struct Ctrl {
    uint64_t in_full[kMaxRing], in_empty[kMaxRing];
    uint64_t acc_full[4], acc_empty[4];
    uint64_t b_full;
    uint64_t swap[4];           // one scale per vector: the warps that share 32 rows
    uint32_t tmem_base;
    volatile uint32_t abort;
};
static_assert(sizeof(Ctrl) <= 256, "control block too large");

// This CTA's rows of B: the plan's split terms, already swizzled, one bulk copy per term and K block.  One thread.
template <int D>
__device__ __forceinline__ void load_b(unsigned char *sB, const unsigned char *w, int half, uint32_t bar)
{
    using C = Cfg<D>;
    mbar_arrive_expect_tx(bar, C::kBBytes);
#pragma unroll
    for (int i = 0; i < 2 * C::kKBlocks; ++i)
        bulk_load(smem_u32(sB + i * C::kBBlock), w + (size_t)(i * C::kHalves + half) * C::kBBlock, C::kBBlock, bar);
}

}  // namespace

struct UmmaAppendParams {
    const float *lambda;   // [n_lambda, D] fp32
    const unsigned char *w;   // split terms of W 2^14: [term][K block][D rows][128 B], swizzled (build_encode_operands)
    unsigned char *packed; // [*, D bits / 8] bytes out
    uint16_t *scales;      // [*, D/32] (one scale per vector: [*, 1]) fp16 out
    uint32_t N;            // below 2^31
    FastDiv rpl;           // rows per lambda row
    int64_t n_lambda;
    RowMap out_map;        // output row of input row r
    float unlift;          // 1 / kOperandLift (as an immediate, or read from device memory: 5120 vectors at D = 128, calls one after another, 4.36 -> 4.41 us)
    int bits;              // 4: nibble pairs; 8: one two's-complement byte per code, scale = absmax / 127
    uint32_t *status;
    uint32_t first_wait_polls;  // polls the mma role gives the B operand before it gives up (kvq_plan_set_wait_limit)
};

// PERVEC: one scale per vector (group = D; Sec. 3.2 step 3, Sec. 4.1) instead of one per 32 channels.
template <int D, bool PERVEC>
__global__ void __launch_bounds__(kThreads, 1)
    kvq_append_umma_kernel(const __grid_constant__ UmmaAppendParams prm, const __grid_constant__ CUtensorMap tm_x)
{
    using C = Cfg<D>;
    static_assert(!PERVEC || C::kHalves == 1, "a row's maximum is traded inside a CTA");
    constexpr int kRing = C::kRing, kAccStages = C::kAccStages, kKBlocks = C::kKBlocks;
    extern __shared__ unsigned char smem_raw[];
    unsigned char *smem = reinterpret_cast<unsigned char *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    unsigned char *sB = smem;                                   // [term][K block][channel][128 B]
    unsigned char *sIn = sB + C::kBBytes;                       // ring of K blocks of x
    Ctrl *ctrl = reinterpret_cast<Ctrl *>(sIn + kRing * kBlockBytes);
    float *rowmax = reinterpret_cast<float *>(reinterpret_cast<unsigned char *>(ctrl) + 256);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int half = (int)blockIdx.x % C::kHalves;              // which channels
    const uint32_t part = blockIdx.x / C::kHalves, parts = gridDim.x / C::kHalves;
    // A limit shortened by the host (kvq_plan_set_wait_limit) is there to be run out of: B is then requested only when the wait begins.
    const bool short_wait = prm.first_wait_polls < kWaitPolls;

    if (threadIdx.x == 0) {
        for (int s = 0; s < kRing; ++s) {
            mbar_init(smem_u32(&ctrl->in_full[s]), 1);
            mbar_init(smem_u32(&ctrl->in_empty[s]), 1);
        }
        for (int s = 0; s < kAccStages; ++s) {
            mbar_init(smem_u32(&ctrl->acc_full[s]), 1);
            mbar_init(smem_u32(&ctrl->acc_empty[s]), 16);
        }
        mbar_init(smem_u32(&ctrl->b_full), 1);
        for (int q = 0; q < 4; ++q) mbar_init(smem_u32(&ctrl->swap[q]), kParts);
        ctrl->abort = 0u;
        mbar_init_fence();
        fence_proxy_async();
        if (!short_wait) load_b<D>(sB, prm.w, half, smem_u32(&ctrl->b_full));   // the plan's: in front of the grid wait
    }
    if (warp == 0) tmem_alloc(smem_u32(&ctrl->tmem_base), kTmemCols);

    // ---- tiles of 128 consecutive vectors: part, part + parts, ...
    const uint32_t N = prm.N, n_tiles = (N + kTile - 1) / kTile;
    const int n_my = (int)((n_tiles - part + parts - 1) / parts);
    auto first_row = [&](int j) -> uint32_t { return (part + (uint32_t)j * parts) * kTile; };

    fence_proxy_async();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    grid_wait();
    const uint32_t tmem_base = ctrl->tmem_base;
    volatile uint32_t *abort_flag = &ctrl->abort;
    uint32_t *status = prm.status;
    int issued = 0;   // producer thread: K blocks whose loads have been issued

    if (warp == 0) {
        // =========================== producer ===========================
        if (lane == 0) {
            bool ok = true;
            if (short_wait) load_b<D>(sB, prm.w, half, smem_u32(&ctrl->b_full));
            for (int j = 0; j < n_my && ok; ++j) {
#pragma unroll
                for (int kb = 0; kb < kKBlocks; ++kb) {   // columns past D (last block of D = 96, 160) are filled with zeros
                    const int u = kKBlocks * j + kb, s = u % kRing;
                    ok = wait_or_abort(smem_u32(&ctrl->in_empty[s]), ((uint32_t)(u / kRing) & 1u) ^ 1u, abort_flag, status, KVQ_DEV_SLOT_TIMEOUT);
                    if (!ok) break;
                    const uint32_t bar = smem_u32(&ctrl->in_full[s]);
                    mbar_arrive_expect_tx(bar, kBlockBytes);
                    tma_load_2d(smem_u32(sIn + s * kBlockBytes), &tm_x, 64 * kb, (int)first_row(j), bar);
                    issued = u + 1;
                }
            }
        }
        __syncwarp();
        grid_trigger();   // the last load is on its way
    } else if (warp == 1) {
        // =========================== mma issuer ===========================
        if (elect_one()) {
            // A limit shortened by the host is spent here, straight after the set-up barrier, when the copies have only just been asked
            // for: this thread has issued nothing yet and can leave at once.
            bool ok = true;
            if (short_wait) {   // looks that do not block, so that "one poll" is over before the operand can possibly be there
                ok = false;
                for (uint32_t it = 0; it < prm.first_wait_polls && !ok; ++it) ok = mbar_test_wait(smem_u32(&ctrl->b_full), 0u);
                if (!ok) {
                    *abort_flag = 1u;
                    atomicOr(status, (uint32_t)KVQ_DEV_SLOT_TIMEOUT);
                }
            }
            const uint64_t b_desc = smem_desc_sw128(smem_u32(sB));
            const uint64_t a_desc = smem_desc_sw128(smem_u32(sIn));
            const uint32_t b_lo = (uint32_t)b_desc, b_hi = (uint32_t)(b_desc >> 32);
            const uint32_t a_lo = (uint32_t)a_desc, a_hi = (uint32_t)(a_desc >> 32);
            ok = ok && wait_or_abort(smem_u32(&ctrl->b_full), 0u, abort_flag, status, KVQ_DEV_SLOT_TIMEOUT);
            for (int j = 0; j < n_my && ok; ++j) {
                const int sc = j % kAccStages;
                if (!wait_or_abort(smem_u32(&ctrl->acc_empty[sc]), ((uint32_t)(j / kAccStages) & 1u) ^ 1u, abort_flag, status, KVQ_DEV_SLOT_TIMEOUT)) break;
                const uint32_t d_tmem = tmem_base + (uint32_t)sc * C::kAccStride;
#pragma unroll
                for (int t = 1; t >= 0; --t) {   // the small term, then the large one
#pragma unroll
                    for (int kb = 0; kb < kKBlocks; ++kb) {
                        const int u = kKBlocks * j + kb, s = u % kRing;
                        if (t == 1 && ok) ok = wait_or_abort(smem_u32(&ctrl->in_full[s]), (uint32_t)(u / kRing) & 1u, abort_flag, status, KVQ_DEV_LOAD_TIMEOUT);
                        if (!ok) break;
                        tc_fence_after();
                        const uint32_t a_lo_s = a_lo + (uint32_t)s * (kBlockBytes >> 4);
#pragma unroll
                        for (int ks = 0; ks < (D - 64 * kb < 64 ? (D - 64 * kb) / 16 : 4); ++ks) {
                            const uint64_t ad = ((uint64_t)a_hi << 32) | (uint64_t)(a_lo_s + (uint32_t)ks * 2u);
                            const uint64_t bd = ((uint64_t)b_hi << 32) |
                                                (uint64_t)(b_lo + (uint32_t)t * (C::kBTerm >> 4) + (uint32_t)kb * (C::kBBlock >> 4) + (uint32_t)ks * 2u);
                            if (t == 0 || kb > 0 || ks > 0) umma_f16_ss<true>(d_tmem, ad, bd, C::kIdesc);
                            else umma_f16_ss<false>(d_tmem, ad, bd, C::kIdesc);
                        }
                        if (t == 0) umma_commit(smem_u32(&ctrl->in_empty[s]));   // the tensor core has read this block of x
                    }
                }
                if (ok) umma_commit(smem_u32(&ctrl->acc_full[sc]));
            }
        }
    } else {
        // =========================== epilogue: accumulator -> scales, codes, nibbles ===========================
        const int q = warp & 3;                 // tensor-memory lane quarter this warp may touch
        const int r = q * 32 + lane;            // tile row of this thread
        const int p = (warp - 2) >> 2;          // this thread's groups: p, p + 4
        const uint32_t t_addr = tmem_base + ((uint32_t)(q * 32) << 16);
        const float unlift = prm.unlift, Q = prm.bits == 4 ? 7.0f : 127.0f, inv_q = prm.bits == 4 ? 1.0f / 7.0f : 1.0f / 127.0f;
        // lambda of this thread's row and CTA's channels (the same for the whole warp where lambda rows are long: a broadcast out of L1)
        auto lambda_of = [&](uint32_t row) -> const float4 * {
            const uint32_t at = prm.n_lambda > 1 ? prm.rpl.small(row < N ? row : N - 1u) : 0u;
            return reinterpret_cast<const float4 *>(prm.lambda + (size_t)at * D + half * C::kCh);
        };
        const float4 *lam = lambda_of(first_row(0) + (uint32_t)r);
        if (p < C::kGroups && lane < 8) (void)load_input(lam + 8 * p + lane);   // the first tile's into L1 while its x is on the way
        auto load_group = [&](int sc, int g, uint32_t (&vb)[32]) {   // group g of accumulator stage sc, times lambda
            tmem_ld32(t_addr + (uint32_t)sc * C::kAccStride + (uint32_t)(g * kGroup), vb);
            float4 l[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) l[i] = load_input(lam + 8 * g + i);
            tmem_ld_wait();
            tmem_loaded(vb);
#pragma unroll
            for (int i = 0; i < 8; ++i) mul_quad(&vb[4 * i], l[i]);
        };
        for (int j = 0; j < n_my; ++j) {
            __syncwarp();
            const uint32_t row = first_row(j) + (uint32_t)r;
            const bool live = row < N;   // the tensor may end inside the tile
            const int64_t orow = prm.out_map(row);
            if (prm.n_lambda > 1) lam = lambda_of(row);
            const int sc = j % kAccStages;
            if (!wait_or_abort(smem_u32(&ctrl->acc_full[sc]), (uint32_t)(j / kAccStages) & 1u, abort_flag, status, KVQ_DEV_MMA_TIMEOUT)) break;
            tc_fence_after();
            // ---- one scale per vector: the row's maximum first (this thread's groups, then the others' through shared memory), then
            // ---- a second pass over the accumulator for the codes; buffers alternate with the tile parity, so a thread cannot
            // ---- overwrite what its partners still read
            GroupScale row_scale;
            if constexpr (PERVEC) {
                float m = 0.0f;
#pragma unroll
                for (int gi = 0; gi < C::kPerThread; ++gi) {
                    const int g = p + kParts * gi;   // warp-uniform
                    if (g < C::kGroups) {
                        uint32_t vb[32];
                        load_group(sc, g, vb);
                        m = fmaxf(m, group_absmax(vb));
                    }
                }
                float *slot = rowmax + (j & 1) * kParts * kTile;
                slot[p * kTile + r] = m;
                __syncwarp();
                if (lane == 0) mbar_arrive(smem_u32(&ctrl->swap[q]));
                if (!wait_or_abort(smem_u32(&ctrl->swap[q]), (uint32_t)j & 1u, abort_flag, status, KVQ_DEV_SLOT_TIMEOUT)) break;
#pragma unroll
                for (int i = 0; i < kParts; ++i) m = fmaxf(m, slot[i * kTile + r]);
                row_scale = group_scale(m, unlift, Q, inv_q);
                if (live && p == 0) prm.scales[orow] = row_scale.half;
            }
#pragma unroll
            for (int gi = 0; gi < C::kPerThread; ++gi) {
                const int g = p + kParts * gi, gd = half * C::kGroups + g;   // group of the CTA's channels, of the row
                uint32_t vb[32];
                if (g < C::kGroups) load_group(sc, g, vb);
                if (gi == C::kPerThread - 1) {   // this thread's last group is in registers: hand the accumulator back
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(smem_u32(&ctrl->acc_empty[sc]));
                }
                if (g < C::kGroups) {
                    const GroupScale gs = PERVEC ? row_scale : group_scale(group_absmax(vb), unlift, Q, inv_q);
                    if (prm.bits == 4) {
                        const uint4 codes = pack_nibbles(vb, gs);
                        if (live) *reinterpret_cast<uint4 *>(prm.packed + orow * (D / 2) + gd * 16) = codes;
                    } else {
                        const uint4 first = pack_bytes(vb, gs), second = pack_bytes(vb + 16, gs);
                        if (live) {
                            uint4 *dst = reinterpret_cast<uint4 *>(prm.packed + orow * D + gd * 32);
                            dst[0] = first, dst[1] = second;
                        }
                    }
                    if (!PERVEC && live) prm.scales[orow * C::G + gd] = gs.half;
                }
            }
        }
    }

    tc_fence_before();
    __syncthreads();
    if (warp == 0) {
        if (*abort_flag) {
            // Every role has left its loop.  The copies still in flight get a bounded chance to land, then tensor-core work that was
            // already issued to drain, before the shared and tensor memory go back.
            if (lane == 0) {
                for (int u = issued > kRing ? issued - kRing : 0; u < issued; ++u)
                    (void)mbar_wait_bounded(smem_u32(&ctrl->in_full[u % kRing]), (uint32_t)(u / kRing) & 1u, 1u << 16);
                (void)mbar_wait_bounded(smem_u32(&ctrl->b_full), 0u, 1u << 16);
            }
            __nanosleep(20000);
            __syncwarp();
        }
        tmem_dealloc(tmem_base, kTmemCols);
    }
}

// ------------------------------------------------------------------------------------------------
// host side
// ------------------------------------------------------------------------------------------------
namespace {

// The operands out of the forward table, once per plan (and rotation): 16 bytes of both terms' swizzled rows per thread.
__global__ void kvq_build_encode_operands_kernel(const float *e0, int D, unsigned char *out)
{
    const int chunks = (D + 63) / 64 * 8, i = (int)(blockIdx.x * blockDim.x + threadIdx.x);
    if (i >= D * chunks) return;
    const int c = i / chunks, ch = i - c * chunks;   // row, 16-byte chunk: K block ch / 8, chunk ch % 8
    unsigned char *dst = out + ((size_t)(ch >> 3) * D + c) * 128 + (((ch & 7) ^ (c & 7)) << 4);
    float w[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) w[k] = 8 * ch + k < D ? e0[(size_t)c * D + 8 * ch + k] * kOperandLift : 0.0f;
#pragma unroll
    for (int t = 0; t < 2; ++t) {
        uint32_t o[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            o[k] = narrow2<false>(w[2 * k], w[2 * k + 1]);
            const float2 f = widen2<false>(o[k]);
            w[2 * k] -= f.x, w[2 * k + 1] -= f.y;   // what the 16-bit term left behind (exact in fp32)
        }
        *reinterpret_cast<uint4 *>(dst + (t ? operand_bytes(D) / 2 : 0)) = make_uint4(o[0], o[1], o[2], o[3]);
    }
}

template <int D, bool PERVEC>
cudaError_t launch(int64_t N, const FftParams &f, cudaStream_t stream)
{
    using C = Cfg<D>;
    static DeviceSlots slots;
    int dev = 0;
    cudaError_t e = current_device_slot(&dev);
    if (e != cudaSuccess) return e;
    int &sms = slots.sms[dev];
    if (sms == 0) {
        int n = 0;
        if ((e = cudaFuncSetAttribute(kvq_append_umma_kernel<D, PERVEC>, cudaFuncAttributeMaxDynamicSharedMemorySize, C::kSmemBytes)) != cudaSuccess) return e;
        if ((e = cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
        sms = n;
    }
    if (N == 0) return cudaSuccess;   // kvq_plan_prepare: the launch attributes are set, there is nothing to run
    if (N >= (int64_t)1 << 31) return cudaErrorInvalidValue;   // tensor-map coordinates are 32-bit

    UmmaAppendParams prm;
    prm.lambda = f.lambda;
    prm.w = f.operands;
    prm.packed = static_cast<unsigned char *>(f.packed);
    prm.scales = static_cast<uint16_t *>(f.scales);
    prm.N = (uint32_t)N;
    prm.rpl = f.rows_per_lambda;
    prm.n_lambda = f.n_lambda;
    prm.out_map = f.out_map;
    prm.unlift = 1.0f / kOperandLift;
    prm.bits = f.bits;
    prm.status = f.status;
    prm.first_wait_polls = f.first_wait_polls ? f.first_wait_polls : kWaitPolls;

    CUtensorMap tm_x;
    const cuuint64_t dims[2] = {(cuuint64_t)D, (cuuint64_t)N};
    const cuuint64_t strides[1] = {(cuuint64_t)(2 * D)};
    const cuuint32_t box[2] = {64, (cuuint32_t)kTile};
    if (!make_tensor_map(&tm_x, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2, f.in, dims, strides, box, CU_TENSOR_MAP_SWIZZLE_128B)) return cudaErrorInvalidValue;

    const int64_t tiles = (N + kTile - 1) / kTile, fit = sms / C::kHalves;
    return launch_kernel(kvq_append_umma_kernel<D, PERVEC>, (unsigned)((tiles < fit ? tiles : fit) * C::kHalves), kThreads, C::kSmemBytes, stream, 1,
                         prm, tm_x);
}

}  // namespace

cudaError_t build_encode_operands(int D, const float *e0, unsigned char *out)
{
    const int n = D * ((D + 63) / 64 * 8);
    kvq_build_encode_operands_kernel<<<(n + 127) / 128, 128>>>(e0, D, out);
    const cudaError_t e = cudaGetLastError();
    return e != cudaSuccess ? e : cudaStreamSynchronize(nullptr);
}

// Where it pays: up to some tiles of 128 vectors per CTA under one lambda row (beyond, the multiplies by lambda cost more than the
// encode's one build), a few more under several, and for every further lambda row, whose build and short tile the encode kernels pay
// for, some tiles more.  Tiles per CTA: us of this kernel and (the encode), graphs of 20 calls (300 rows: streams), 148 CTAs; a stream
// of calls and calls alone change over at the same sizes:
//              one lambda row                          three                        52                300
//   D = 64     1: 3.6 (3.75), 2: 4.5 (4.1)             1: 3.6 (3.7), 2: 4.65 (4.5)  2: 4.6 (4.5)      7: 9.5 (10.3), 8: 10.6 (10.4)
//   D = 96     7: 10.0 (10.4), 10: 13.0 (12.8)         8: 11.4 (11.7)               9: 13.4 (13.6)    14: 18.7 (21.3), 20: 29 (27.5)
//   D = 128    5: 10.0 (10.2), 6: 11.4 (11.2)          7: 12.8 (12.9), 8: 14 (13.8)  10: 16.9 (17.9)  20: 35.4 (35.1)
//   D = 160    2: 8.0 (8.9), 2.5: 9.9 (9.7)            4: 12.5 (12.6), 5: 14 (14.2)  10: 25.2 (28.5)  14: 40.5 (43.9), 20: 59 (58)
//   D = 256    5: 22.0 (23.3), 6: 26.2 (26.2)          6: 26.1 (27.7)               10: 47.6 (49.2)   20: 101 (107)
//   one scale per vector:
//   D = 64     1: 4.3 (4.3), 2: 5.7 (4.9)              1: 4.15 (4.1)                2: 5.8 (5.15)     5: 10.2 (10.2)
//   D = 96     1: 4.7 (5.2), 2: 6.35 (5.9)             2: 6.5 (7.0), 2.5: 7.9 (7.1)  3: 8.0 (8.8)     9: 17.8 (18.4)
//   D = 128    4: 9.8 (10.0), 5: 11.4 (11.3)           6: 13.0 (13.2)               9: 18.4 (18.8)    14: 28 (31), 20: 41 (39)
//   D = 160    2: 8.7 (9.2), 2.5: 10.7 (10.0)          2: 8.8 (9.7), 2.5: 11 (10)   5: 15.8 (16.1)    12: 36.7 (37.1)
// (Under 52 rows at D = 160 the line lies at 6.75 tiles, and up to ten this kernel would be faster by 8 to 18 %.)
// N == 0 (kvq_plan_prepare): whether it is built.
bool umma_append_pays(int D, bool bf16, bool per_vector, int64_t N, const FftParams &f)
{
    if (bf16 || (D == 256 && per_vector)) return false;
    if (N == 0) return true;
    if (!f.append || !f.operands) return false;
    static DeviceSlots slots;
    int dev = 0;
    if (current_device_slot(&dev) != cudaSuccess) return false;
    if (slots.sms[dev] == 0) {
        int n = 0;
        if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return false;
        slots.sms[dev] = n;
    }
    struct Line { int one, several, more; };   // half tiles per CTA under one lambda row, under several; tiles for every further row
    const Line at = per_vector ? (D == 64 ? Line{2, 2, 1} : D == 96 ? Line{2, 4, 3} : D == 128 ? Line{8, 12, 5} : Line{4, 4, 5})
                               : (D == 64 ? Line{2, 2, 3} : D == 96 ? Line{14, 16, 4} : D == 128 ? Line{10, 14, 6} : D == 160 ? Line{4, 8, 8} : Line{12, 12, 8});
    const int64_t rows = f.n_lambda == 1 ? 1 : (N + f.rows_per_lambda.d - 1) / f.rows_per_lambda.d;
    return 2 * ((N + kTile - 1) / kTile) <= (int64_t)(rows == 1 ? at.one : at.several) * slots.sms[dev] + 2 * (int64_t)at.more * (rows - 1);
}

cudaError_t umma_append(int D, bool per_vector, int64_t N, const FftParams &f, cudaStream_t stream)
{
    if (!tensor_map_encode_fn()) return cudaErrorNotSupported;
    switch (D) {
        case 64: return per_vector ? launch<64, true>(N, f, stream) : launch<64, false>(N, f, stream);
        case 96: return per_vector ? launch<96, true>(N, f, stream) : launch<96, false>(N, f, stream);
        case 128: return per_vector ? launch<128, true>(N, f, stream) : launch<128, false>(N, f, stream);
        case 160: return per_vector ? launch<160, true>(N, f, stream) : launch<160, false>(N, f, stream);
        case 256: return per_vector ? cudaErrorInvalidValue : launch<256, false>(N, f, stream);
    }
    return cudaErrorInvalidValue;
}

}  // namespace kvq

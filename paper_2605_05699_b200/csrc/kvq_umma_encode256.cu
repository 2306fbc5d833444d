// Warp-specialised tcgen05 DFT-as-GEMM encode kernel of libkvq (sm_100a) for D = 256, fp16 or bf16 input.
//
// Same contraction and the same split of W into 16-bit terms as kvq_umma_encode.cu (v = lambda (.) M (s (.) x),
// Sec. 3.1 Eq. 1-2, Sec. 5.1 item 1; W 2^k = W1 + W2, a third term for bf16 in the calibration pass).  The split B operand
// (2 or 3 x 128 KB) does not fit one CTA's shared memory, so a PAIR of CTAs (a cluster of two) works on one tile of 256 vectors
// (128 on short calls) with cta_group::2 instructions: each CTA holds its own half of the vectors and one half of B's rows
// (channels), the leader's one thread issues MMAs of N = 256 over both, and each CTA's tensor memory receives all 256 channels
// of its own vectors.
//
// What bounds it: 32 MMAs of 128 cycles per tile (2.1 us per 128 vectors and SM at 1965 MHz; the bytes take 1.9), and, back to
// back, the board's power limit.  The form before this one gave each CTA 128 channels of the same 128 vectors: every x block was
// fetched by both CTAs, the ring beside B held less than the latency of its loads, and both split terms were added up in the
// epilogue.  Before -> now, back to back, both on one box (which vary by 5 %): 212,992 bf16 vectors under 52 lambda rows 63.7 -> 58.6 us,
// under one 59.6 -> 54.1, one scale per vector 69.7 -> 55.8; 9000 fp16 vectors 10.3 -> 9.7, 24,000: 14.4 -> 13.2, 42,000: 17.7 -> 17.0;
// 300 lambda rows of 300 vectors 47.1 -> 43.8.  Slower by 2 to 3 % where the last of many tall tiles is nearly
// empty (95,000 fp16 vectors 28.1 -> 28.8; 52 x 2048 31.6 -> 32.5).
//
//   warp 0        producer   (both CTAs) one TMA tensor load per K block of 64 columns into a ring of blocks; the
//                            loads of both CTAs complete on the leader's barrier
//   warp 1        mma        (leader) per tile every K step of the small term first, then of the large one: the small sums are
//                            then added up before anything large is in the accumulator, so that each rounding of the fp32
//                            accumulator is counted once per K step of the large term alone.  A block is released
//                            in the second pass.  (Three terms: block by block, all terms; the ring holds one tile.)
//   warps 2-17    epilogue   (both CTAs) all sixteen warps on every tile, thread = (row, two of the row's eight groups, or one)
//
// Byte codes (fp16 input) are a run-time switch of the epilogue.  Every wait is bounded.
#include "kvq_internal.h"
#include "kvq_quantize.cuh"
#include "kvq_umma.cuh"

namespace kvq {

namespace {

constexpr int kGroup = 32;
constexpr int kThreads = 576;              // producer, mma, 16 epilogue warps
constexpr int kEpiWarps = 16;
constexpr int kCtrlBytes = 512;
constexpr int kSmemLimit = 232448;         // 227 KB of dynamic shared memory per CTA
constexpr uint32_t kTmemCols = 512;

constexpr int kD = 256;
constexpr int kG = kD / kGroup;            // 8 scales per row
constexpr int kHalfN = 128;                // channels whose B rows a CTA holds
constexpr int kKBlocks = kD / 64;          // 4 K blocks per tile
constexpr int kBBlock = kHalfN * 128;      // one K block of one term of B: 128 rows x 128 B
constexpr int kBTerm = kKBlocks * kBBlock; // one split term of B: 128 rows x K = 256, 64 KB
constexpr int kMaxRing = 12;
constexpr int kMaxAcc = 4;

// CALIB: the calibration pass keeps a third bf16 term (it runs once; its result is compared at 1e-6 of the vector norm)
// PERVEC: one scale per vector: the four threads of a row trade their maxima through shared memory
// ROWS: vectors per CTA and tile; a pair's tile has twice as many = MMA M.  128, or 64 where that ends earlier (short_is_faster).
template <bool BF16, bool CALIB = false, bool PERVEC = false, int ROWS = 128>
struct Cfg {
    static_assert(ROWS == 64 || ROWS == 128, "tile heights");
    static constexpr int kBlockBytes = ROWS * 128;   // one K block of a CTA's x: ROWS x 128 B
    // tensor memory of an accumulator.  128 vectors: a lane per vector, 256 columns.  64: lanes 0-63 hold the vectors' channels
    // 0-127, lanes 64-127 the rest, 128 columns.
    static constexpr uint32_t kAccCols = 2 * ROWS;
    static constexpr int kAccStages = 512 / (int)kAccCols;
    static constexpr int kThreadGroups = ROWS / 64;  // groups of 32 channels per epilogue thread
    static constexpr int kSplit = (BF16 && CALIB) ? 3 : 2;
    static constexpr int kBBytes = kSplit * kBTerm;
    static constexpr int kParties = kG / kThreadGroups;   // threads that share a row
    static constexpr int kMaxBytes = PERVEC ? 2 * kParties * ROWS * (int)sizeof(float) : 0;   // one scale per vector: [tile parity][party][row]
    static constexpr int kRoom = (kSmemLimit - 1024 - kCtrlBytes - kMaxBytes - kBBytes) / kBlockBytes;
    static constexpr int kWant = 6 * 128 / ROWS;
    static constexpr int kRing = kRoom < kWant ? kRoom : kWant;   // K blocks of x in flight: 6 (12 short ones), one less with kMaxBytes, 4 short ones beside three terms
    static_assert(kRing >= 2, "no room for the x ring");
    static constexpr bool kSmallFirst = kRing > kKBlocks;   // a whole tile stays in the ring for two passes over it
    static constexpr int kSmemBytes = kBBytes + kRing * kBlockBytes + kCtrlBytes + kMaxBytes + 1024;
    static constexpr uint32_t kIdesc = umma_idesc(2 * ROWS, kD, BF16);
};

// Barriers that count arrivals of both CTAs (in_full, acc_empty, b_first, b_ready) are used in the leader's copy only.
struct Ctrl {
    uint64_t in_full[kMaxRing], in_empty[kMaxRing];
    uint64_t acc_full[kMaxAcc], acc_empty[kMaxAcc];
    uint64_t b_first, b_ready;
    uint64_t swap[4];           // one scale per vector: the warps that share 32 rows
    uint64_t drain;             // after an abort: every MMA issued is complete
    uint32_t tmem_base;
    volatile uint32_t abort;
    uint32_t mma_stopped;       // the mma role left its loop early (both CTAs' copies)
    uint32_t issued[2];         // leader's copy: K blocks that each CTA's producer asked for
};
static_assert(sizeof(Ctrl) <= kCtrlBytes, "control block too large");

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
    mx = __uint_as_float(__reduce_max_sync(0xFFFFFFFFu, __float_as_uint(mx)));   // non-negative: ordered like its bits
    mx = fminf(fmaxf(mx * table_max, 1e-30f), 1e30f);
    const int e = (int)((__float_as_uint(mx) >> 23) & 0xFFu) - 127;      // floor(log2 mx)
    return __uint_as_float((uint32_t)(127 + 13 - e) << 23);
}

// Eight rows from c0 on of every split term of this CTA's half of the B operand (channel 128 half + c), by one warp: a lane
// requests four table entries per pass and row, all at once (load), scales them by lambda_c 2^k, peels off 16-bit terms and
// writes 8 bytes of each term's swizzled row (store).
constexpr int kBuildRows = 8;
template <bool BF16, bool CALIB>
struct BuildRows {
    float4 m[kBuildRows][2];
    float l;   // lane k: lambda of row c0 + k (load_lambda, behind grid_wait)
    __device__ __forceinline__ void load(const float *__restrict__ e0, int half, int c0, int lane)
    {
#pragma unroll
        for (int k = 0; k < kBuildRows; ++k)
#pragma unroll
            for (int p = 0; p < 2; ++p) m[k][p] = __ldg(reinterpret_cast<const float4 *>(e0 + (size_t)(half * kHalfN + c0 + k) * kD) + lane + 32 * p);
    }
    __device__ __forceinline__ void load_lambda(const float *__restrict__ lam, int half, int c0, int lane)
    {
        l = lam ? load_input(lam + half * kHalfN + c0 + lane % kBuildRows) : 1.0f;
    }
    __device__ __forceinline__ void store(unsigned char *sB, float lift, int c0, int lane) const
    {
        using C = Cfg<BF16, CALIB>;
        const float lifted = l * lift;
#pragma unroll
        for (int k = 0; k < kBuildRows; ++k) {
            const int c = c0 + k;
            const float f = __shfl_sync(0xFFFFFFFFu, lifted, k);
#pragma unroll
            for (int p = 0; p < 2; ++p) {
                const int i = lane + 32 * p;
                float w[4] = {m[k][p].x * f, m[k][p].y * f, m[k][p].z * f, m[k][p].w * f};
                const int ch = i >> 1;   // 16-byte chunk of the K-major row: K block ch / 8, chunk ch % 8
                const uint32_t off = (uint32_t)((ch >> 3) * kBBlock + c * 128 + (((ch & 7) ^ (c & 7)) << 4) + ((i & 1) ? 8 : 0));
#pragma unroll
                for (int t = 0; t < C::kSplit; ++t) {
                    const uint32_t lo = narrow2<BF16>(w[0], w[1]), hi = narrow2<BF16>(w[2], w[3]);
                    *reinterpret_cast<uint2 *>(sB + t * kBTerm + off) = make_uint2(lo, hi);
                    if (t + 1 < C::kSplit) {   // what the 16-bit term left behind (exact in fp32)
                        const float2 a = widen2<BF16>(lo), b = widen2<BF16>(hi);
                        w[0] -= a.x, w[1] -= a.y, w[2] -= b.x, w[3] -= b.y;
                    }
                }
            }
        }
    }
};

}  // namespace

struct UmmaEncode256Params {
    const unsigned char *x;   // [N, D] 16-bit: for prefetches, the loads go through the tensor map
    const float *lambda;   // [n_lambda, D] fp32
    const float *e0;       // plan table [D, D] fp32: e0[c][n] = M[c][n] s_n
    unsigned char *packed; // [*, D/2] bytes out
    uint16_t *scales;      // [*, D/32] fp16 out
    int64_t N;
    int64_t n_lambda;
    int64_t rpl;           // rows per lambda segment (N when there is one lambda row)
    TilePlan plan;         // the call's tiles, cut into shares of the pairs
    RowMap out_map;        // output row of input row r
    uint32_t *status;
    uint32_t *amax_bits;        // calibration only: [D] running column maxima as fp32 bit patterns (start at zero)
    int bits;                   // 4: nibble pairs; 8 (fp16 input): one two's-complement byte per code, scale = absmax / 127
};

template <bool BF16, bool CALIB, bool PERVEC, int ROWS>
__global__ void __launch_bounds__(kThreads, 1)
    kvq_encode_umma_d256_kernel(const __grid_constant__ UmmaEncode256Params prm, const __grid_constant__ CUtensorMap tm_x)
{
    using C = Cfg<BF16, CALIB, PERVEC, ROWS>;
    constexpr int kRing = C::kRing, kAccStages = C::kAccStages, kBlockBytes = C::kBlockBytes;
    extern __shared__ unsigned char smem_raw[];
    unsigned char *smem = reinterpret_cast<unsigned char *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    unsigned char *sB = smem;                                   // [term][K block][128 rows][128 B]
    unsigned char *sIn = sB + C::kBBytes;                       // ring of K blocks of x
    Ctrl *ctrl = reinterpret_cast<Ctrl *>(sIn + kRing * kBlockBytes);
    float *rowmax = reinterpret_cast<float *>(reinterpret_cast<unsigned char *>(ctrl) + kCtrlBytes);   // PERVEC: [parity][party][row]

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int rank = (int)cluster_rank();       // which ROWS vectors of a tile, and which 128 rows of B, this CTA holds
    const int pair = blockIdx.x >> 1;

    if (threadIdx.x == 0) {
        for (int s = 0; s < kRing; ++s) {
            mbar_init(smem_u32(&ctrl->in_full[s]), 1);
            mbar_init(smem_u32(&ctrl->in_empty[s]), 1);
        }
        for (int s = 0; s < kAccStages; ++s) {
            mbar_init(smem_u32(&ctrl->acc_full[s]), 1);
            mbar_init(smem_u32(&ctrl->acc_empty[s]), 2 * kEpiWarps);
        }
        mbar_init(smem_u32(&ctrl->b_first), 2 * kEpiWarps);   // first B: all epilogue warps of both CTAs build it
        mbar_init(smem_u32(&ctrl->b_ready), 2 * kEpiWarps);   // later rebuilds
        for (int qq = 0; qq < 4; ++qq) mbar_init(smem_u32(&ctrl->swap[qq]), C::kParties);
        mbar_init(smem_u32(&ctrl->drain), 1);
        ctrl->abort = 0u;
        ctrl->mma_stopped = 0u;
        mbar_init_fence();
    }
    if (warp == 0) tmem_alloc_pair(smem_u32(&ctrl->tmem_base), kTmemCols);

    // ---- tiles: lambda segments of rpl rows, cut into tiles of 2 ROWS rows; a contiguous range per CTA pair
    const int64_t N = prm.N, rpl = prm.rpl;
    const TileShare share(prm.plan, (uint32_t)pair);
    const int tps = (int)share.tps;
    const int n_my = share.n;

    // ---- B for the pair's first lambda row: eight rows per epilogue warp, requested before the set-up barrier
    // The pair's set-up barrier in front of the grid wait for tall tiles, so that lambda and the first x loads follow the wait side by side
    // (592 128-row tiles bf16 20.7 -> 19.9 us, 1036: 30.2 -> 28.9, 1664: 51.5 -> 49.4); behind lambda for short ones, of which a pair has
    // one or two: one 128-row tile per CTA 11.0 us so, 11.7 the other way.
    constexpr bool kBarrierFirst = ROWS == 128;
    float first_lift = 1.0f;
    if (n_my > 0 && warp >= 2) {
        const float *lam = CALIB ? nullptr : prm.lambda + (prm.n_lambda == 1 ? 0 : (int64_t)share.seg) * kD;
        BuildRows<BF16, CALIB> rows;
        rows.load(prm.e0, rank, (warp - 2) * 8, lane);
        if constexpr (kBarrierFirst) {
            tc_fence_before();
            cluster_sync_all();   // both CTAs' barriers exist and both have their tensor memory
            tc_fence_after();
        }
        grid_wait();
        rows.load_lambda(lam, rank, (warp - 2) * 8, lane);
        first_lift = lift_of<kD>(lam, prm.e0, lane);
        if constexpr (!kBarrierFirst) {
            tc_fence_before();
            cluster_sync_all();
            tc_fence_after();
        }
        rows.store(sB, first_lift, (warp - 2) * 8, lane);
        fence_proxy_async();   // B is read by the tensor core through the async proxy
        __syncwarp();
        if (lane == 0) cluster_mbar_arrive(cluster_map(smem_u32(&ctrl->b_first), 0));
    } else {
        if constexpr (!kBarrierFirst) grid_wait();
        tc_fence_before();
        cluster_sync_all();
        tc_fence_after();
        if constexpr (kBarrierFirst) grid_wait();
    }
    const uint32_t tmem_base = ctrl->tmem_base;
    volatile uint32_t *abort_flag = &ctrl->abort;
    uint32_t *status = prm.status;

    if (warp == 0) {
        // =========================== producer ===========================
        if (lane == 0) {
            bool ok = true;
            int issued = 0;
            TileCursor cur(share), ahead(share, 1);
            for (int j = 0; j < n_my && ok; ++j, cur.advance(1), ahead.advance(1)) {
                const int64_t row0 = cur.seg * rpl + (int64_t)cur.tin * (2 * ROWS) + rank * ROWS;   // may lie past the end: zeros
                // The next tile's rows are one contiguous run: asked for as such, they come out of DRAM page by page, and the K block
                // loads, 128 bytes of each row at a time, find them in L2 (1,064,960 bf16 vectors: 278 -> 269 us; two tiles ahead: 273).
                if (j + 1 < n_my) {
                    const int64_t next = ahead.seg * rpl + (int64_t)ahead.tin * (2 * ROWS) + rank * ROWS;
                    const int64_t n = N - next < ROWS ? N - next : ROWS;
                    if (n > 0) prefetch_l2(prm.x + next * (2 * kD), (uint32_t)n * (2 * kD));
                }
#pragma unroll
                for (int kb = 0; kb < kKBlocks; ++kb) {
                    const int u = kKBlocks * j + kb, s = u % kRing;
                    ok = wait_or_abort(smem_u32(&ctrl->in_empty[s]), ((uint32_t)(u / kRing) & 1u) ^ 1u, abort_flag, status, KVQ_DEV_SLOT_TIMEOUT);
                    if (!ok) break;
                    if (rank == 0) mbar_arrive_expect_tx(smem_u32(&ctrl->in_full[s]), 2 * kBlockBytes);   // this CTA's block and the partner's
                    tma_load_2d_pair(smem_u32(sIn + s * kBlockBytes), &tm_x, 64 * kb, (int)row0, cluster_map(smem_u32(&ctrl->in_full[s]), 0));
                    issued = u + 1;
                }
            }
            cluster_st_u32(cluster_map(smem_u32(&ctrl->issued[rank]), 0), (uint32_t)issued);
        }
        __syncwarp();
        grid_trigger();   // the last load is on its way
    } else if (warp == 1) {
        // =========================== mma issuer (leader) ===========================
        if (rank == 0 && elect_one()) {
            // Descriptors differ only in their 14-bit start-address field (bytes >> 4): one base per operand, one add per MMA.
            const uint64_t b_desc = smem_desc_sw128(smem_u32(sB));
            const uint64_t a_desc = smem_desc_sw128(smem_u32(sIn));
            const uint32_t b_lo = (uint32_t)b_desc, b_hi = (uint32_t)(b_desc >> 32);
            const uint32_t a_lo = (uint32_t)a_desc, a_hi = (uint32_t)(a_desc >> 32);
            uint32_t builds = 0;
            bool ok = true;
            TileCursor cur(share);
            for (int j = 0; j < n_my && ok; ++j, cur.advance(1)) {
                const int sc = j % kAccStages;
                if (j == 0) {   // the epilogue warps build the first B while the first x blocks are in flight
                    ok = wait_cluster_or_abort(smem_u32(&ctrl->b_first), 0u, abort_flag, status, KVQ_DEV_SLOT_TIMEOUT);
                } else if (!CALIB && prm.n_lambda > 1 && cur.first_of_segment()) {   // the epilogue warps rebuild B for this lambda row
                    ok = wait_cluster_or_abort(smem_u32(&ctrl->b_ready), builds & 1u, abort_flag, status, KVQ_DEV_SLOT_TIMEOUT);
                    ++builds;
                }
                ok = ok && wait_cluster_or_abort(smem_u32(&ctrl->acc_empty[sc]), ((uint32_t)(j / kAccStages) & 1u) ^ 1u, abort_flag, status,
                                                 KVQ_DEV_SLOT_TIMEOUT);
                if (!ok) break;
                const uint32_t d_tmem = tmem_base + (uint32_t)sc * C::kAccCols;
                constexpr int kPasses = C::kSmallFirst ? C::kSplit : 1;   // passes over the tile's blocks
#pragma unroll
                for (int ps = 0; ps < kPasses && ok; ++ps) {
#pragma unroll
                    for (int kb = 0; kb < kKBlocks; ++kb) {
                        const int u = kKBlocks * j + kb, s = u % kRing;
                        if (ps == 0 && !wait_cluster_or_abort(smem_u32(&ctrl->in_full[s]), (uint32_t)(u / kRing) & 1u, abort_flag, status,
                                                              KVQ_DEV_LOAD_TIMEOUT)) {
                            ok = false;
                            break;
                        }
                        tc_fence_after();
                        const uint32_t a_lo_s = a_lo + (uint32_t)s * (kBlockBytes >> 4);
#pragma unroll
                        for (int tt = 0; tt < (C::kSmallFirst ? 1 : C::kSplit); ++tt) {
                            const int t = C::kSmallFirst ? C::kSplit - 1 - ps : tt;
#pragma unroll
                            for (int ks = 0; ks < 4; ++ks) {   // the four K steps of this block
                                const uint64_t ad = ((uint64_t)a_hi << 32) | (uint64_t)(a_lo_s + (uint32_t)ks * 2u);
                                const uint64_t bd = ((uint64_t)b_hi << 32) |
                                                    (uint64_t)(b_lo + (uint32_t)t * (kBTerm >> 4) + (uint32_t)kb * (kBBlock >> 4) + (uint32_t)ks * 2u);
                                if (ps > 0 || kb > 0 || tt > 0 || ks > 0) umma_f16_ss_pair<true>(d_tmem, ad, bd, C::kIdesc);
                                else umma_f16_ss_pair<false>(d_tmem, ad, bd, C::kIdesc);
                            }
                        }
                        if (ps == kPasses - 1) umma_commit_pair(smem_u32(&ctrl->in_empty[s]));   // the tensor core has read this block of x
                    }
                }
                if (ok) umma_commit_pair(smem_u32(&ctrl->acc_full[sc]));
            }
            if (!ok) {   // the abort flag is up: both CTAs take the drain below
                umma_commit_pair(smem_u32(&ctrl->drain));
                ctrl->mma_stopped = 1u;
                cluster_st_u32(cluster_map(smem_u32(&ctrl->mma_stopped), 1), 1u);
            }
        }
    } else {
        // =========================== epilogue: accumulator -> scales, codes, nibbles ===========================
        // All sixteen warps on every tile, thread = (row, ROWS / 64 of the row's eight groups): the accumulator goes back after
        // half the time that two sets on alternate tiles would hold it, and the tensor core has the other stages meanwhile.
        constexpr int kTG = C::kThreadGroups;
        const int q = warp & 3;                 // tensor-memory lane quarter this warp may touch
        const int q_rows = q % (ROWS / 32);     // the 32 rows those lanes hold
        const int r = q_rows * 32 + lane;       // row of this CTA's
        const int col0 = ((warp - 2) >> 2) * (kTG * kGroup);                              // first accumulator column of this thread
        const int g0 = (q / (ROWS / 32)) * (kG / 2) + ((warp - 2) >> 2) * kTG;            // and the group it belongs to
        const uint32_t t_addr = tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)col0;
        auto load_group = [&](int sc, int gi, uint32_t (&vb)[32]) {   // this thread's group g0 + gi out of accumulator stage sc
            tmem_ld32(t_addr + (uint32_t)sc * C::kAccCols + (uint32_t)(gi * kGroup), vb);
            tmem_ld_wait();
        };
        float lift_next = first_lift;
        float colmax[kTG] = {};   // calibration: lane i keeps the running maximum of column i of each of this thread's groups
        TileCursor cur(share);
        for (int j = 0; j < n_my; ++j, cur.advance(1)) {
            __syncwarp();
            const int64_t seg = cur.seg;
            const int64_t off = (int64_t)cur.tin * (2 * ROWS) + rank * ROWS;
            const float unlift = 1.0f / lift_next;

            // ---- this tile's accumulator.  Where the next tile begins a new lambda row, every MMA that read the old B is complete
            // ---- with it: B is rebuilt first, before this tile's own work, from table rows requested before the wait.
            const int sc = j % kAccStages;
            const bool rebuild = !CALIB && j + 1 < n_my && cur.tin + 1 == tps && prm.n_lambda > 1;
            if (rebuild) {
                const float *lam = prm.lambda + (seg + 1) * kD;
                BuildRows<BF16, CALIB> rows;
                rows.load(prm.e0, rank, (warp - 2) * 8, lane);
                rows.load_lambda(lam, rank, (warp - 2) * 8, lane);
                lift_next = lift_of<kD>(lam, prm.e0, lane);
                if (!wait_or_abort(smem_u32(&ctrl->acc_full[sc]), (uint32_t)(j / kAccStages) & 1u, abort_flag, status, KVQ_DEV_MMA_TIMEOUT)) break;
                rows.store(sB, lift_next, (warp - 2) * 8, lane);
                fence_proxy_async();   // B is read by the tensor core through the async proxy
                __syncwarp();
                if (lane == 0) cluster_mbar_arrive(cluster_map(smem_u32(&ctrl->b_ready), 0));
            } else {
                if (!wait_or_abort(smem_u32(&ctrl->acc_full[sc]), (uint32_t)(j / kAccStages) & 1u, abort_flag, status, KVQ_DEV_MMA_TIMEOUT)) break;
            }
            tc_fence_after();

            // ---- rows of the tile that exist: the segment (and with it the tensor) may end inside the tile
            int64_t seg_rows = N - seg * rpl;
            if (seg_rows > rpl) seg_rows = rpl;
            const bool live = off + r < seg_rows;
            const int64_t orow = prm.out_map(seg * rpl + off + r);
            const float Q = prm.bits == 4 ? 7.0f : 127.0f, inv_q = prm.bits == 4 ? 1.0f / 7.0f : 1.0f / 127.0f;   // largest code (warp-uniform)
            // ---- one scale per vector: the row's maximum first (this thread's groups, then the others' through
            // ---- shared memory), then a second pass over the accumulator for the codes; buffers alternate with the tile
            // ---- parity, so a thread cannot overwrite what its partners still read
            GroupScale row_scale;
            if constexpr (PERVEC) {
                float m = 0.0f;
#pragma unroll
                for (int gi = 0; gi < kTG; ++gi) {
                    uint32_t vb[32];
                    load_group(sc, gi, vb);
                    m = fmaxf(m, group_absmax(vb));
                }
                float *slot = rowmax + (j & 1) * C::kParties * ROWS;   // [party][row] of this buffer
                slot[(g0 / kTG) * ROWS + r] = m;
                __syncwarp();
                if (lane == 0) mbar_arrive(smem_u32(&ctrl->swap[q_rows]));
                if (!wait_or_abort(smem_u32(&ctrl->swap[q_rows]), (uint32_t)j & 1u, abort_flag, status, KVQ_DEV_SLOT_TIMEOUT)) break;
#pragma unroll
                for (int i = 0; i < C::kParties; ++i) m = fmaxf(m, slot[i * ROWS + r]);
                row_scale = group_scale(m, unlift, Q, inv_q);
                if (live && g0 == 0) prm.scales[orow] = row_scale.half;
            }
            uint32_t sc2 = 0u;   // the groups' fp16 scales
#pragma unroll
            for (int gi = 0; gi < kTG; ++gi) {
                const int g = g0 + gi;       // warp-uniform
                uint32_t vb[32];
                load_group(sc, gi, vb);
                if (gi == kTG - 1) {   // this thread's last group is in registers: hand the accumulator back
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) cluster_mbar_arrive(cluster_map(smem_u32(&ctrl->acc_empty[sc]), 0));
                }
                if constexpr (CALIB) {
                    // column maxima over the warp's 32 rows (rows past the end were filled with zeros by the TMA load)
#pragma unroll
                    for (int i = 0; i < 32; ++i) {
                        const uint32_t m = __reduce_max_sync(0xFFFFFFFFu, vb[i] & 0x7FFFFFFFu);   // |v| orders like its bits
                        if (lane == i) colmax[gi] = fmaxf(colmax[gi], __uint_as_float(m));
                    }
                    continue;
                }
                const GroupScale gs = PERVEC ? row_scale : group_scale(group_absmax(vb), unlift, Q, inv_q);
                sc2 |= (uint32_t)gs.half << (16 * gi);
                if (prm.bits == 4) {
                    const uint4 codes = pack_nibbles(vb, gs);
                    if (live) *reinterpret_cast<uint4 *>(prm.packed + orow * (kD / 2) + g * 16) = codes;
                } else {
                    const uint4 first = pack_bytes(vb, gs), second = pack_bytes(vb + 16, gs);
                    if (live) {
                        uint4 *dst = reinterpret_cast<uint4 *>(prm.packed + orow * kD + g * 32);
                        dst[0] = first, dst[1] = second;
                    }
                }
            }
            if constexpr (!CALIB && !PERVEC)
                if (live) {
                    if constexpr (kTG == 2) *reinterpret_cast<uint32_t *>(prm.scales + orow * kG + g0) = sc2;
                    else prm.scales[orow * kG + g0] = (uint16_t)sc2;
                }
        }
        if constexpr (CALIB) {   // this warp's maxima of its 32 rows of every tile -> the global column maxima
#pragma unroll
            for (int gi = 0; gi < kTG; ++gi) atomicMax(prm.amax_bits + (g0 + gi) * kGroup + lane, __float_as_uint(colmax[gi] * (1.0f / first_lift)));
        }
    }

    __syncwarp();
    if (lane == 0 && *abort_flag)   // tell the partner
        cluster_st_u32(cluster_map(smem_u32(const_cast<uint32_t *>(&ctrl->abort)), (uint32_t)(rank ^ 1)), 1u);
    __syncwarp();
    tc_fence_before();
    cluster_sync_all();   // neither CTA leaves, or gives its tensor memory back, while the other may still use it
    tc_fence_after();
    if (*abort_flag) {   // up in both CTAs or in neither: whoever raises it tells the other before the barrier
        if (threadIdx.x == 0) {
            // MMAs that were issued (they complete in order: after the last tile's, or the commit that the mma role left with, all
            // are) and loads that are under way get a bounded time to end before shared and tensor memory go back.
            if (ctrl->mma_stopped)
                (void)mbar_wait_bounded(smem_u32(&ctrl->drain), 0u, 1u << 16);
            else if (n_my > 0)
                (void)mbar_wait_bounded(smem_u32(&ctrl->acc_full[(n_my - 1) % kAccStages]), (uint32_t)((n_my - 1) / kAccStages) & 1u, 1u << 16);
            if (rank == 0) {
                const PairDrain d{(int)ctrl->issued[0], (int)ctrl->issued[1], kRing};
                for (int u = d.begin(); u < d.end(); ++u) {
                    const uint32_t bar = smem_u32(&ctrl->in_full[d.slot(u)]);
                    if (d.owes_arrival(u)) mbar_arrive_expect_tx(bar, kBlockBytes);
                    if (d.owes_bytes(u)) mbar_complete_tx(bar, kBlockBytes);
                    (void)mbar_wait_bounded(bar, d.parity(u), 1u << 16);
                }
            }
        }
        __syncwarp();
        cluster_sync_all();   // the partner stays until its loads, which arrive on the leader's barriers, have landed
    }
    if (warp == 0) tmem_dealloc_pair(tmem_base, kTmemCols);
}

// ------------------------------------------------------------------------------------------------
// host side
// ------------------------------------------------------------------------------------------------
namespace {

// Sets the kernel's launch attributes; fit: pairs resident at once (the SMs of a cluster share a GPC).  Looked up once per device.
template <bool BF16, bool CALIB, bool PERVEC, int ROWS>
cudaError_t resident_pairs(int *fit)
{
    using C = Cfg<BF16, CALIB, PERVEC, ROWS>;
    auto kern = kvq_encode_umma_d256_kernel<BF16, CALIB, PERVEC, ROWS>;
    static DeviceSlots slots;
    int dev = 0;
    cudaError_t e = current_device_slot(&dev);
    if (e != cudaSuccess) return e;
    if (slots.sms[dev] == 0) {
        int n = 0;
        if ((e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, C::kSmemBytes)) != cudaSuccess) return e;
        if ((e = cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
        cudaLaunchConfig_t cfg = {};
        cudaLaunchAttribute attr[1];
        cfg.gridDim = dim3((unsigned)(n & ~1), 1, 1);
        cfg.blockDim = dim3(kThreads, 1, 1);
        cfg.dynamicSmemBytes = C::kSmemBytes;
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = 2;
        attr[0].val.clusterDim.y = 1;
        attr[0].val.clusterDim.z = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        if ((e = cudaOccupancyMaxActiveClusters(&n, kern, &cfg)) != cudaSuccess) return e;
        if (n < 1) return cudaErrorLaunchOutOfResources;
        slots.sms[dev] = n;
    }
    *fit = slots.sms[dev];
    return cudaSuccess;
}

int64_t tiles_of(int64_t n_seg, int64_t rpl, int rows) { return n_seg * ((rpl + rows - 1) / rows); }

// Short tiles (128 vectors of a pair) cost a pair less each, tall ones (256) less per vector: short where 2 n_short <= 3 n_tall + 1, n the
// tiles of the longest share.  Back to back, us, short and tall:
//   fp16, one lambda row    9000: 9.3, 10.0   18,944: 11.1, 11.6   24,000: 12.6, 13.6   30,000: 14.5, 13.9   41,000: 16.2, 16.7
//                           46,000: 16.3, 16.7   50,000: 18.3, 16.8   60,000: 20.3, 19.5   212,992: 58.4, 48.8
//   bf16, one lambda row    9000: 9.4, 11.0   24,000: 13.6, 15.5   36,000: 15.4, 15.2   46,000: 16.7, 17.8   50,000: 18.3, 17.8
//   bf16, 52 lambda rows    9000: 11.5, 11.8   30,000: 17.7, 19.2   36,000: 19.8, 18.4   46,000: 21.5, 21.6   60,000: 26.5, 22.7
//                           70,000: 24.9, 25.2   110,000: 32.8, 33.9   130,000: 38.0, 38.0   160,000: 48.6, 40.1
// (the rule is wrong at 36,000 and 110,000 under 52 rows, by 8 and 3 %).  One scale per vector lies alike.
// Calibration from fp16: 9000 vectors 16.4 and 16.5, 57,000: 24.6, 28.2; 170,000: 39.7, 43.1; 200,000: 47.8, 46.8; 500,000: 106, 95.
// (From bf16 its three terms leave a tall tile two x blocks beside B, and short ones are as fast or faster throughout: 9000 vectors 16.5
// and 20.5, 57,000: 26.7, 30.8; 212,992: 63.9, 66.0; 500,000: 146.5, 145.1.  The tall form is not built.)
template <bool CALIB>
bool short_is_faster(int64_t n_seg, int64_t rpl, int fit)
{
    const int64_t n_short = (tiles_of(n_seg, rpl, 128) + fit - 1) / fit, n_tall = (tiles_of(n_seg, rpl, 256) + fit - 1) / fit;
    if (CALIB) return n_short <= 18;
    return 2 * n_short <= 3 * n_tall + 1;
}

template <bool BF16, bool CALIB, bool PERVEC, int ROWS>
cudaError_t launch(int64_t N, const FftParams &f, const float *e0, cudaStream_t stream, uint32_t *amax_bits)
{
    using C = Cfg<BF16, CALIB, PERVEC, ROWS>;
    int fit = 0;
    const cudaError_t e = resident_pairs<BF16, CALIB, PERVEC, ROWS>(&fit);
    if (e != cudaSuccess) return e;
    if (N == 0) return cudaSuccess;   // kvq_plan_prepare: the launch attributes are set, there is nothing to run
    if (N >= (int64_t)1 << 31) return cudaErrorInvalidValue;   // tensor-map coordinates are 32-bit

    UmmaEncode256Params prm;
    prm.x = static_cast<const unsigned char *>(f.in);
    prm.lambda = f.lambda;
    prm.e0 = e0;
    prm.packed = static_cast<unsigned char *>(f.packed);
    prm.scales = static_cast<uint16_t *>(f.scales);
    prm.N = N;
    prm.n_lambda = f.n_lambda;
    prm.rpl = f.n_lambda == 1 || f.rows_per_lambda.d > N ? N : f.rows_per_lambda.d;
    const int64_t n_seg = (N + prm.rpl - 1) / prm.rpl;
    prm.out_map = f.out_map;
    prm.status = f.status;
    prm.amax_bits = amax_bits;
    prm.bits = f.bits;

    CUtensorMap tm_x;
    const cuuint64_t dims[2] = {(cuuint64_t)kD, (cuuint64_t)N};
    const cuuint64_t strides[1] = {(cuuint64_t)(2 * kD)};
    const cuuint32_t box[2] = {64, (cuuint32_t)ROWS};
    if (!make_tensor_map(&tm_x, BF16 ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16 : CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2, f.in, dims, strides, box,
                         CU_TENSOR_MAP_SWIZZLE_128B))
        return cudaErrorInvalidValue;

    const int64_t tiles = tiles_of(n_seg, prm.rpl, 2 * ROWS);
    const unsigned pairs = (unsigned)(tiles < fit ? tiles : fit);
    prm.plan = TilePlan(n_seg, prm.rpl, pairs, 2 * ROWS);
    return launch_kernel(kvq_encode_umma_d256_kernel<BF16, CALIB, PERVEC, ROWS>, 2 * prm.plan.shares, kThreads, C::kSmemBytes, stream, 2, prm, tm_x);
}

template <bool BF16, bool CALIB, bool PERVEC>
cudaError_t launch_any(int64_t N, const FftParams &f, const float *e0, cudaStream_t stream, uint32_t *amax_bits = nullptr)
{
    if constexpr (BF16 && CALIB) {
        return launch<BF16, CALIB, PERVEC, 64>(N, f, e0, stream, amax_bits);
    } else {
        if (N == 0) {   // kvq_plan_prepare: both heights
            const cudaError_t e = launch<BF16, CALIB, PERVEC, 64>(N, f, e0, stream, amax_bits);
            return e != cudaSuccess ? e : launch<BF16, CALIB, PERVEC, 128>(N, f, e0, stream, amax_bits);
        }
        const int64_t rpl = f.n_lambda == 1 || f.rows_per_lambda.d > N ? N : f.rows_per_lambda.d;
        int fit = 0;
        const cudaError_t e = resident_pairs<BF16, CALIB, PERVEC, 128>(&fit);
        if (e != cudaSuccess) return e;
        return short_is_faster<CALIB>((N + rpl - 1) / rpl, rpl, fit) ? launch<BF16, CALIB, PERVEC, 64>(N, f, e0, stream, amax_bits)
                                                                     : launch<BF16, CALIB, PERVEC, 128>(N, f, e0, stream, amax_bits);
    }
}

}  // namespace

cudaError_t umma_encode_d256(bool bf16, bool per_vector, int64_t N, const FftParams &f, const float *e0, cudaStream_t stream)
{
    if (!tensor_map_encode_fn()) return cudaErrorNotSupported;
    if (per_vector) return bf16 ? launch_any<true, false, true>(N, f, e0, stream) : launch_any<false, false, true>(N, f, e0, stream);
    return bf16 ? launch_any<true, false, false>(N, f, e0, stream) : launch_any<false, false, false>(N, f, e0, stream);
}

cudaError_t umma_calibrate_d256(bool bf16, int64_t N, const FftParams &f, const float *e0, uint32_t *amax_bits, cudaStream_t stream)
{
    if (!tensor_map_encode_fn()) return cudaErrorNotSupported;
    return bf16 ? launch_any<true, true, false>(N, f, e0, stream, amax_bits) : launch_any<false, true, false>(N, f, e0, stream, amax_bits);
}

}  // namespace kvq

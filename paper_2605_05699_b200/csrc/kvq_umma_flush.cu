// The block flush in one launch (sm_100a): D = 64, 96, 128, fp16 and bf16, groups of 32, 4-bit codes, no rotation.
//
// A prefill block goes into the int4 caches and, dequantized, into the prefix cache (Sec. 7.2).  As an encode and a decode that is
// two starts, and the second kernel reads back and unpacks what a thread of the first had in registers.  Here the thread that has
// quantized a group writes it as the decode's A operand at once, and the tile goes on through the second contraction:
//
//   warp 0          producer   one TMA tensor load per K block of 64 elements and tile of 128 vectors, two to four tiles in flight
//   warp 1          mma        one elected thread: x B1 of tile j + 1, 64 channels and the rest into accumulators of their own, then
//                              A2 B2 of tile j, so that the first contraction of a tile runs under the quantizer of the one before
//   warps 2 ..      quantize   four warps per group of 32 channels, thread = (row, group), every tile: accumulator 1 -> scale,
//                              codes, caches (the quantizer and the arithmetic of kvq_umma_encode.cu: the same bits); the G threads
//                              of a row trade their scales, which decide the row's operand factor; codes -> A2 in tensor memory
//                              (the operands of kvq_umma_decode.cu: the same bits)
//   last 4 warps    output     thread = row: accumulator 2 -> E + O, E - O -> TMA store
//
//   tensor memory   accumulator 1 [128, 2 D] (two stacked terms) | A2, 64 columns per term | accumulator 2: E, O: all 512 columns at
//                   D = 128 with bf16
//   shared memory   B1 (two terms) | B2 | x tiles | output staging
//
// B1 and B2 carry lambda and are rebuilt at a new lambda row, B1 by the quantizing warps, B2 by the output warps, when the last MMA
// that reads the old one is complete.  Tiles do not cross streams: the output is clipped by its tensor map.  Waits, time-outs and wide
// lambda rows as in the two kernels that this one joins.
//
// Slower, 64 x 2000 and 128 x 4000 rows at D = 128 bf16 (27.3 and 79.9 us): two issuing threads, one per contraction 29.8 and 93;
// rows of the tiles ahead asked for in L2 28.7 and 85.
#include "kvq_decode_fp32.cuh"
#include "kvq_internal.h"
#include "kvq_quantize.cuh"
#include "kvq_umma.cuh"
#include "kvq_umma_decode_operand.cuh"
#include "kvq_umma_encode_operand.cuh"

namespace kvq {

namespace {

constexpr int kTile = 128;                 // vectors per tile = MMA M
constexpr int kBlockBytes = kTile * 128;   // one K block of the x tile
constexpr int kOutWarps = 4;
constexpr int kCtrlBytes = 5120;
constexpr uint32_t kTmemCols = 512;
constexpr int kFullBars = 4;   // ring of barriers, indexed by tile: the producer waits for tile j - kInStages's
constexpr int kSlots = 4;      // rows' output factors: tiles between the quantizing warps and the output warps (two)

template <int D, bool BF16>
struct Fwd {   // operand of the first contraction: two terms stacked along N
    static constexpr int kDim = D, kSplit = 2;
    static constexpr bool kBf16 = BF16;
    static constexpr int kKBlocks = (D + 63) / 64;
    // The channels in two parts, 64 and the rest, each with an accumulator of its own: [64 channels][first term, second term], and so
    // on.  One part is read and issued again while the tensor core is at the other.
    static constexpr int kParts = D > 64 ? 2 : 1;
    static __host__ __device__ constexpr int channels(int part) { return part == 0 ? 64 : D - 64; }
    static __device__ __forceinline__ int row(int c) { return c + (c < 64 ? 0 : 64); }   // the second term stands channels(part) rows behind
    static constexpr int kBBlock = 2 * D * 128, kBytes = kKBlocks * kBBlock;
    static __device__ __forceinline__ int term(int c) { return 128 * channels(c < 64 ? 0 : 1); }
    static __host__ __device__ constexpr uint32_t idesc(int part) { return umma_idesc_m128(2 * channels(part), BF16); }
};

template <int D, bool BF16>
struct Inv {   // operands of the second: [term][parity]
    static constexpr int kBits = 4, kTerms = BF16 ? 2 : 1, kQuads = D / 4, kBRows = D / 2;
    static constexpr bool kRadix2 = true;
    static constexpr int kBPartBlock = (D / 2) * 128, kBPart = kBPartBlock, kBytes = kTerms * 2 * kBPart;   // D / 2 <= 64: one K block
    static constexpr uint32_t kIdesc = umma_idesc_m128(D / 2, false);
};

template <int D, bool BF16>
struct Cfg {
    static_assert(D == 64 || D == 96 || D == 128, "head dim not built");
    using F = Fwd<D, BF16>;
    using I = Inv<D, BF16>;
    static constexpr int G = D / 32, kKSteps = D / 16;
    static constexpr int kQuantWarps = 4 * G;
    static constexpr int kThreads = 32 * (2 + kQuantWarps + kOutWarps);
    static constexpr int kXBytes = F::kKBlocks * kBlockBytes;
    static constexpr int kOutWarpBytes = 32 * 2 * D;
    // Output staging for two tiles with fp16 output (two x tiles still fit beside it): 128 x 4000 rows at D = 128 79.5 -> 75.6 us, at
    // D = 96 54.0 -> 50.7.  With bf16 output it is slower: D = 96 55.6 -> 57.7, D = 64 42.6 -> 44.3.
    static constexpr int kOutBufs = BF16 ? 1 : 2;
    static constexpr int kOutBytes = kOutBufs * kOutWarps * kOutWarpBytes;
    static constexpr int kRoom = (232448 - 1024 - kCtrlBytes - F::kBytes - I::kBytes - kOutBytes) / kXBytes;
    static constexpr int kInStages = kRoom < kFullBars ? kRoom : kFullBars;
    static_assert(kInStages >= 2, "too few x tiles in flight");
    static constexpr int kSmemBytes = F::kBytes + I::kBytes + kInStages * kXBytes + kOutBytes + kCtrlBytes + 1024;
    static constexpr uint32_t kACol = 2 * D, kALo = 64, kAcc2Col = kACol + 128, kOCol = D == 96 ? 64 : D / 2;
    static_assert(kAcc2Col + kOCol + D / 2 <= kTmemCols, "tensor memory");
};

struct Ctrl {
    uint64_t in_full[kFullBars];
    uint64_t acc1_full[2], acc1_empty[2];   // per part of the channels
    uint64_t x_free[kFullBars];  // ring by tile: the first contraction has read its x
    uint64_t swap[4];            // the G warps that share 32 rows have posted their scales
    uint64_t a2_full, a2_empty, acc2_full, acc2_empty;
    uint64_t b1_ready, b2_ready; // one phase per lambda row of the share
    uint32_t tmem_base;
    volatile uint32_t abort;
    volatile uint32_t any_wide;  // some lambda row of this CTA's tiles is too wide for the fp16 B2: redone in fp32 at the end
    alignas(16) float recip[160];               // 1 / (max(lambda, 1e-6) rho) of the row that B2 is built for
    alignas(16) uint16_t scale[2][kTile][4];    // [tile parity][row][group]
    alignas(16) float row_scale[kSlots][kTile]; // what the output multiplies a row by (1 unless its scales left fp16's comfort zone)
};
static_assert(sizeof(Ctrl) <= kCtrlBytes, "control block too large");

struct RowFactors {
    float unlift, rho;
};

// B1 of a lambda row by the quantizing warps, w of them.  first: from the kernel's entry, through the set-up barrier and the grid wait.
// Out of line, like the other build: the loops' registers are then their own.
template <int D, bool BF16>
__device__ __noinline__ RowFactors build_forward(unsigned char *sB, const float *__restrict__ e0, const float *lam, uint32_t ready, int w, int lane, bool first)
{
    fwd::BuildB<Fwd<D, BF16>, Cfg<D, BF16>::kQuantWarps> rows;
    rows.load(e0, 0, w, lane);
    if (first) {
        tc_fence_before();
        __syncthreads();
        tc_fence_after();
        grid_wait();
    }
    rows.load_lambda(lam, 0, w, lane);
    const float lift = fwd::lift_of<D>(lam, e0, lane);
    rows.store(sB, lift, 0, w, lane);
    rows.rest(sB, e0, lam, lift, w, lane);
    fence_proxy_async();   // B is read by the tensor core through the async proxy
    __syncwarp();
    if (lane == 0) mbar_arrive(ready);
    return {1.0f / lift, RecipLambda<D>(lam, lane).rho};
}

// B2 of a lambda row by the output warps.
template <int D, bool BF16>
__device__ __noinline__ void build_inverse(unsigned char *sB, Ctrl *ctrl, const float *__restrict__ b0, const float *lam, int w, int lane, bool first)
{
    inv::BuildB<Inv<D, BF16>, kOutWarps> rows;
    rows.load(b0, 0, w, lane);
    if (first) {
        tc_fence_before();
        __syncthreads();
        tc_fence_after();
        grid_wait();
    }
    const RecipLambda<D> rl(lam, lane);
    if (rl.wide) ctrl->any_wide = 1u;
    inv::post_reciprocals<D>(ctrl->recip, rl, lane);
    rows.store(sB, ctrl->recip, 0, w, lane);
    rows.rest(sB, b0, ctrl->recip, w, lane);
    fence_proxy_async();   // B is read by the tensor core through the async proxy
    __syncwarp();
    if (lane == 0) mbar_arrive(smem_u32(&ctrl->b2_ready));
}

}  // namespace

struct UmmaFlushParams {
    GemmParams g;          // the caches, lambda, the inverse table, where the rows live
    const float *e0;       // plan table [D, D] fp32: e0[c][n] = M[c][n] s_n, its largest |entry| behind it
    int64_t rows;          // per stream
    TilePlan plan;
    uint32_t flip2[32];    // sign-bit masks of s_n s_{n + D/2} for the output pairs (n, n + 1), n = 0, 2, .. D/2 - 2
    uint32_t first_wait_polls;   // SHORT: polls the mma role gives the first B1 before it gives up (kvq_plan_set_wait_limit)
};

struct UmmaFlushMaps {
    CUtensorMap x;         // [streams rows, D], boxes of 64 columns x 128 rows (128-byte swizzle)
    CUtensorMap wide;      // output, boxes of 64 columns x 32 rows (128-byte swizzle)
    CUtensorMap slim;      // output, boxes of 32 columns x 32 rows (64-byte swizzle), used when D / 32 is odd
};

// SHORT: the host has shortened the limit of the mma role's first wait.  A form of its own: the issuing loop answers to whatever stands
// beside it, and with the test in the one kernel 64 x 2000 rows took 25.3 us for 24.9 (D = 128 fp16) and 19.9 for 19.55 (D = 96 bf16).
template <int D, bool BF16, bool SHORT>
__global__ void __launch_bounds__(Cfg<D, BF16>::kThreads, 1)
    kvq_flush_umma_kernel(const __grid_constant__ UmmaFlushParams prm, const __grid_constant__ UmmaFlushMaps maps)
{
    using C = Cfg<D, BF16>;
    using F = typename C::F;
    using I = typename C::I;
    constexpr int G = C::G, kInStages = C::kInStages;
    extern __shared__ unsigned char smem_raw[];
    unsigned char *smem = reinterpret_cast<unsigned char *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    unsigned char *sB1 = smem;
    unsigned char *sB2 = sB1 + F::kBytes;
    unsigned char *sIn = sB2 + I::kBytes;
    unsigned char *sOut = sIn + kInStages * C::kXBytes;
    Ctrl *ctrl = reinterpret_cast<Ctrl *>(sOut + C::kOutBytes);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

    if (threadIdx.x == 0) {
        for (int s = 0; s < kInStages; ++s) mbar_init(smem_u32(&ctrl->in_full[s]), 1);
        for (int s = 0; s < kFullBars; ++s) mbar_init(smem_u32(&ctrl->x_free[s]), 1);
        for (int s = 0; s < F::kParts; ++s) {
            mbar_init(smem_u32(&ctrl->acc1_full[s]), 1);
            mbar_init(smem_u32(&ctrl->acc1_empty[s]), 4 * F::channels(s) / 32);
        }
        for (int s = 0; s < 4; ++s) mbar_init(smem_u32(&ctrl->swap[s]), G);
        mbar_init(smem_u32(&ctrl->a2_full), C::kQuantWarps);
        mbar_init(smem_u32(&ctrl->a2_empty), 1);
        mbar_init(smem_u32(&ctrl->acc2_full), 1);
        mbar_init(smem_u32(&ctrl->acc2_empty), kOutWarps);
        mbar_init(smem_u32(&ctrl->b1_ready), C::kQuantWarps);
        mbar_init(smem_u32(&ctrl->b2_ready), kOutWarps);
        ctrl->abort = 0u;
        ctrl->any_wide = 0u;
        mbar_init_fence();
        fence_proxy_async();
    }
    if (warp == 1) tmem_alloc(smem_u32(&ctrl->tmem_base), kTmemCols);

    const int64_t rows = prm.rows;
    const TileShare share(prm.plan, blockIdx.x);
    const int n_my = share.n;
    const int64_t row_first = prm.g.lambda_index(share.seg);
    auto lambda_row = [&](int64_t row) -> const float * { return prm.g.lambda + row * D; };

    RowFactors fac = {1.0f, 1.0f};
    if (n_my > 0 && warp >= 2 + C::kQuantWarps) {
        build_inverse<D, BF16>(sB2, ctrl, prm.g.b0, lambda_row(row_first), warp - 2 - C::kQuantWarps, lane, true);
    } else if (n_my > 0 && warp >= 2) {
        fac = build_forward<D, BF16>(sB1, prm.e0, lambda_row(row_first), smem_u32(&ctrl->b1_ready), warp - 2, lane, true);
    } else {
        tc_fence_before();
        __syncthreads();
        tc_fence_after();
        grid_wait();
    }
    const uint32_t tmem_base = ctrl->tmem_base;
    volatile uint32_t *abort_flag = &ctrl->abort;
    uint32_t *status = prm.g.status;
    int issued = 0;   // producer thread: x tiles whose loads have been issued

    if (warp == 0) {
        // =========================== producer ===========================
        if (lane == 0) {
            TileCursor cur(share);
            for (int j = 0; j < n_my; ++j, cur.advance(1)) {
                const int s = j % kInStages;
                if (j >= kInStages) {   // the first contraction of the tile that used the stage last is complete
                    const int jp = j - kInStages;
                    if (!wait_or_abort(smem_u32(&ctrl->x_free[jp % kFullBars]), (uint32_t)(jp / kFullBars) & 1u, abort_flag, status, KVQ_DEV_SLOT_TIMEOUT)) break;
                }
                const int64_t row0 = cur.seg * rows + cur.row_in_segment();   // rows past the stream's are read and never stored
                const uint32_t bar = smem_u32(&ctrl->in_full[s]);
                mbar_arrive_expect_tx(bar, C::kXBytes);
#pragma unroll
                for (int kb = 0; kb < F::kKBlocks; ++kb)   // columns past D (last block of D = 96) are filled with zeros
                    tma_load_2d(smem_u32(sIn + s * C::kXBytes + kb * kBlockBytes), &maps.x, 64 * kb, (int)row0, bar);
                issued = j + 1;
            }
        }
        __syncwarp();
        grid_trigger();   // the last load is on its way
    } else if (warp == 1) {
        // =========================== mma issuer ===========================
        if (elect_one()) {
            const uint64_t b1_desc = smem_desc_sw128(smem_u32(sB1)), b2_desc = smem_desc_sw128(smem_u32(sB2)), x_desc = smem_desc_sw128(smem_u32(sIn));
            const uint32_t b1_lo = (uint32_t)b1_desc, b2_lo = (uint32_t)b2_desc, x_lo = (uint32_t)x_desc, hi = (uint32_t)(b1_desc >> 32);   // the upper halves are alike
            TileCursor c1(share), c2(share);
            int64_t r1 = -1, r2 = -1;      // lambda rows of the contractions' last tiles
            uint32_t n1 = 0, n2 = 0;       // operands waited for
            auto first = [&](int j) -> bool {   // x B1 of tile j
                if (j > 0) c1.advance(1);
                if (j == 0 || (c1.first_of_segment() && prm.g.lambda_index(c1.seg) != r1)) {
                    r1 = prm.g.lambda_index(c1.seg);
                    if (!wait_or_abort(smem_u32(&ctrl->b1_ready), n1++ & 1u, abort_flag, status, KVQ_DEV_SLOT_TIMEOUT)) return false;
                }
                const int s = j % kInStages;
                if (!wait_or_abort(smem_u32(&ctrl->in_full[s]), (uint32_t)(j / kInStages) & 1u, abort_flag, status, KVQ_DEV_LOAD_TIMEOUT)) return false;
                const uint32_t x_s = x_lo + (uint32_t)s * (C::kXBytes >> 4);
#pragma unroll
                for (int part = 0; part < F::kParts; ++part) {
                    if (!wait_or_abort(smem_u32(&ctrl->acc1_empty[part]), ((uint32_t)j & 1u) ^ 1u, abort_flag, status, KVQ_DEV_SLOT_TIMEOUT)) return false;
                    tc_fence_after();
#pragma unroll
                    for (int ks = 0; ks < C::kKSteps; ++ks) {
                        const uint32_t a_off = (uint32_t)(ks >> 2) * (kBlockBytes >> 4) + (uint32_t)(ks & 3) * 2u;
                        const uint32_t b_off = (uint32_t)(ks >> 2) * (F::kBBlock >> 4) + (uint32_t)part * (128u * 128u >> 4) + (uint32_t)(ks & 3) * 2u;
                        const uint64_t ad = ((uint64_t)hi << 32) | (uint64_t)(x_s + a_off), bd = ((uint64_t)hi << 32) | (uint64_t)(b1_lo + b_off);
                        if (ks > 0) umma_f16_ss<true>(tmem_base + 128u * (uint32_t)part, ad, bd, F::idesc(part));
                        else umma_f16_ss<false>(tmem_base + 128u * (uint32_t)part, ad, bd, F::idesc(part));
                    }
                    umma_commit(smem_u32(&ctrl->acc1_full[part]));
                }
                umma_commit(smem_u32(&ctrl->x_free[j % kFullBars]));
                return true;
            };
            auto second = [&](int j) -> bool {   // A2 B2 of tile j
                if (j > 0) c2.advance(1);
                if (j == 0 || (c2.first_of_segment() && prm.g.lambda_index(c2.seg) != r2)) {
                    r2 = prm.g.lambda_index(c2.seg);
                    if (!wait_or_abort(smem_u32(&ctrl->b2_ready), n2++ & 1u, abort_flag, status, KVQ_DEV_SLOT_TIMEOUT)) return false;
                }
                if (!wait_or_abort(smem_u32(&ctrl->a2_full), (uint32_t)j & 1u, abort_flag, status, KVQ_DEV_SLOT_TIMEOUT)) return false;
                if (!wait_or_abort(smem_u32(&ctrl->acc2_empty), ((uint32_t)j & 1u) ^ 1u, abort_flag, status, KVQ_DEV_SLOT_TIMEOUT)) return false;
                tc_fence_after();
#pragma unroll
                for (int p = 0; p < 2; ++p)
#pragma unroll
                    for (int set = 0; set < (BF16 ? 3 : 1); ++set)   // bf16 output: a_hi W_hi + a_lo W_hi + a_hi W_lo
#pragma unroll
                        for (int ks = 0; ks < D / 32; ++ks) {
                            const uint32_t b_off = (uint32_t)((set == 2 ? 2 * I::kBPart : 0) + p * I::kBPart) / 16u + (uint32_t)ks * 2u;
                            const uint64_t bd = ((uint64_t)hi << 32) | (uint64_t)(b2_lo + b_off);
                            const uint32_t dp = tmem_base + C::kAcc2Col + (uint32_t)p * C::kOCol;
                            const uint32_t ap = tmem_base + C::kACol + (set == 1 ? C::kALo : 0u) + (uint32_t)p * (D / 4) + (uint32_t)ks * 8u;
                            if (set > 0 || ks > 0) umma_f16_ts<true>(dp, ap, bd, I::kIdesc);
                            else umma_f16_ts<false>(dp, ap, bd, I::kIdesc);
                        }
                umma_commit(smem_u32(&ctrl->acc2_full));
                umma_commit(smem_u32(&ctrl->a2_empty));
                return true;
            };
            bool ok = n_my > 0;
            if constexpr (SHORT) ok = ok && wait_first_operand(smem_u32(&ctrl->b1_ready), abort_flag, status, prm.first_wait_polls);
            ok = ok && first(0);
            for (int j = 0; j < n_my && ok; ++j) {
                if (j + 1 < n_my) ok = first(j + 1);
                ok = ok && second(j);
            }
        }
    } else if (warp < 2 + C::kQuantWarps) {
        // =========================== quantize: accumulator 1 -> scales, codes, A2 ===========================
        const int q = warp & 3;                 // tensor-memory lane quarter this warp may touch
        const int g = (warp - 2) >> 2;          // group of 32 channels
        const int part = g >> 1;
        const int r = q * 32 + lane;            // tile row and tensor-memory lane of this thread
        const uint32_t t_addr = tmem_base + ((uint32_t)(q * 32) << 16);
        unsigned char *packed = static_cast<unsigned char *>(const_cast<void *>(prm.g.packed));
        uint16_t *scales = static_cast<uint16_t *>(const_cast<void *>(prm.g.scales));
        int64_t cached_row = row_first;
        TileCursor cur(share);
        for (int j = 0; j < n_my; ++j, cur.advance(1)) {
            __syncwarp();
            // ---- a new lambda row, once every MMA that read the old B1 is complete
            if (cur.first_of_segment() && prm.g.lambda_index(cur.seg) != cached_row) {
                cached_row = prm.g.lambda_index(cur.seg);
                if (!wait_or_abort(smem_u32(&ctrl->x_free[(j - 1) % kFullBars]), (uint32_t)((j - 1) / kFullBars) & 1u, abort_flag, status, KVQ_DEV_MMA_TIMEOUT)) break;
                fac = build_forward<D, BF16>(sB1, prm.e0, lambda_row(cached_row), smem_u32(&ctrl->b1_ready), warp - 2, lane, false);
            }
            if (!wait_or_abort(smem_u32(&ctrl->acc1_full[part]), (uint32_t)j & 1u, abort_flag, status, KVQ_DEV_MMA_TIMEOUT)) break;
            tc_fence_after();
            const int64_t off = cur.row_in_segment() + r;
            const bool live = off < rows;   // the stream may end inside the tile
            const int64_t orow = prm.g.phys_row(cur.seg, off, rows);

            uint32_t vb[32];
            {
                uint32_t lo[32];
                const uint32_t at = t_addr + (uint32_t)(128 * part + 32 * (g & 1));
                tmem_ld32(at, vb);
                tmem_ld32(at + (uint32_t)F::channels(part), lo);
                tmem_ld_wait();
                add_group(vb, lo);
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&ctrl->acc1_empty[part]));   // the values are in registers
            const GroupScale gs = group_scale(group_absmax(vb), fac.unlift, 7.0f, 1.0f / 7.0f);
            uint16_t *slot = ctrl->scale[j & 1][r];   // buffers alternate: who writes the next but one has seen that all have read this one
            slot[g] = gs.half;
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&ctrl->swap[q]));
            const uint4 codes = pack_nibbles(vb, gs);
            if (live) *reinterpret_cast<uint4 *>(packed + orow * (D / 2) + g * 16) = codes;
            if (!wait_or_abort(smem_u32(&ctrl->swap[q]), (uint32_t)j & 1u, abort_flag, status, KVQ_DEV_SLOT_TIMEOUT)) break;
            const uint2 all = *reinterpret_cast<const uint2 *>(slot);
            uint32_t sc[(G + 1) / 2];
            sc[0] = all.x;
            if constexpr (G > 2) sc[1] = all.y;
            if (g == 0 && live) {
                if constexpr (G == 4) *reinterpret_cast<uint2 *>(scales + orow * G) = all;
                else if constexpr (G == 2) *reinterpret_cast<uint32_t *>(scales + orow * G) = all.x;
                else
#pragma unroll
                    for (int i = 0; i < G; ++i) scales[orow * G + i] = (uint16_t)(sc[i >> 1] >> (16 * (i & 1)));
            }

            // ---- the second contraction's operand, out of the codes and the STORED scale, as kvq_decode has it
            float inv;
            const float pw = operand_rescue<G>(sc, fac.rho, 9000.0f, inv);
            const __half2 s2 = __float2half2_rn(__half2float(__ushort_as_half(gs.half)) * fac.rho * pw);
            if (!wait_or_abort(smem_u32(&ctrl->a2_empty), ((uint32_t)j & 1u) ^ 1u, abort_flag, status, KVQ_DEV_MMA_TIMEOUT)) break;   // the tile before is through
            tc_fence_after();
            if (g == 0) ctrl->row_scale[j % kSlots][r] = inv;
            const __half2 h1032 = __float2half2_rn(1032.0f);
            const uint32_t words[4] = {codes.x, codes.y, codes.z, codes.w};
            uint32_t a[2][8], al[2][BF16 ? 8 : 1];   // [parity]
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const uint32_t u = words[i] ^ 0x88888888u;   // nibbles now hold q + 8
#pragma unroll
                for (int e = 0; e < 4; ++e) {   // pairs 0 and 2 of a word are even channels, 1 and 3 odd
                    const uint32_t m = lop3_and_or(u >> (4 * e), 0x000F000Fu, 0x64006400u);   // {1024 + n_e, 1024 + n_{e+4}}
                    const __half2 q2 = __hsub2(*reinterpret_cast<const __half2 *>(&m), h1032);
                    const __half2 h = __hmul2(q2, s2);
                    a[e & 1][2 * i + (e >> 1)] = *reinterpret_cast<const uint32_t *>(&h);
                    if constexpr (BF16) {   // q s2 - h, exact in fp16
                        const __half2 l = __hfma2(q2, s2, __hneg2(h));
                        al[e & 1][2 * i + (e >> 1)] = *reinterpret_cast<const uint32_t *>(&l);
                    }
                }
            }
#pragma unroll
            for (int p = 0; p < 2; ++p) {
                const uint32_t at = t_addr + C::kACol + (uint32_t)p * (D / 4) + 8u * (uint32_t)g;
                tmem_st8(at, a[p]);
                if constexpr (BF16) tmem_st8(at + C::kALo, al[p]);
            }
            tmem_st_wait();
            tc_fence_before();
            __threadfence_block();   // the rows' factors, for the output warps
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&ctrl->a2_full));
        }
    } else {
        // =========================== output: accumulator 2 -> TMA store ===========================
        const int w = warp - 2 - C::kQuantWarps, q = warp & 3;
        const uint32_t lane_addr = tmem_base + ((uint32_t)(q * 32) << 16) + C::kAcc2Col;
        int64_t cached_row = row_first;
        TileCursor cur(share);
        for (int j = 0; j < n_my; ++j, cur.advance(1)) {
            __syncwarp();
            if (cur.first_of_segment() && prm.g.lambda_index(cur.seg) != cached_row) {   // the last tile's accumulator has been here: nothing reads the old B2
                cached_row = prm.g.lambda_index(cur.seg);
                build_inverse<D, BF16>(sB2, ctrl, prm.g.b0, lambda_row(cached_row), w, lane, false);
            }
            if (!wait_or_abort(smem_u32(&ctrl->acc2_full), (uint32_t)j & 1u, abort_flag, status, KVQ_DEV_MMA_TIMEOUT)) break;
            tc_fence_after();
            unsigned char *stg = sOut + ((C::kOutBufs == 2 ? (j & 1) * kOutWarps : 0) + w) * C::kOutWarpBytes;   // this warp's staging tile
            if (lane == 0) {   // this warp's stores out of it have read it
                if constexpr (C::kOutBufs == 2) asm volatile("cp.async.bulk.wait_group.read 1;" ::: "memory");
                else bulk_wait_read_all();
            }
            __syncwarp();
            const float row_inv = ctrl->row_scale[j % kSlots][q * 32 + lane];
            const bool rescale = __any_sync(0xFFFFFFFFu, row_inv != 1.0f);   // rare: a row outside the operand's comfort zone
#pragma unroll
            for (int h = 0; h < D / 32; ++h) {   // E and O columns 16 h .. 16 h + 15 -> outputs 16 h .. and D / 2 + 16 h ..
                uint32_t ev[16], ov[16];
                tmem_ld16(lane_addr + (uint32_t)h * 16u, ev);
                tmem_ld16(lane_addr + C::kOCol + (uint32_t)h * 16u, ov);
                tmem_ld_wait();
                if (h == D / 32 - 1) {   // the last values are in registers: hand the accumulator back
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(smem_u32(&ctrl->acc2_empty));
                }
                if (rescale) {
#pragma unroll
                    for (int i = 0; i < 16; ++i) {
                        ev[i] = __float_as_uint(__uint_as_float(ev[i]) * row_inv);
                        ov[i] = __float_as_uint(__uint_as_float(ov[i]) * row_inv);
                    }
                }
#pragma unroll
                for (int k = 0; k < 2; ++k) {   // 16-byte chunk: 8 outputs
                    uint32_t lo[4], hi[4];
#pragma unroll
                    for (int p2 = 0; p2 < 4; ++p2) {
                        const int i = 8 * k + 2 * p2;
                        const uint64_t ep = pack_f32x2(__uint_as_float(ev[i]), __uint_as_float(ev[i + 1]));
                        const uint64_t op = pack_f32x2(__uint_as_float(ov[i]), __uint_as_float(ov[i + 1]));
                        const float2 sum = unpack_f32x2(add_f32x2(ep, op)), diff = unpack_f32x2(sub_f32x2(ep, op));
                        lo[p2] = narrow2<BF16>(sum.x, sum.y);                                          // s_n is already in E and O
                        hi[p2] = narrow2<BF16>(diff.x, diff.y) ^ prm.flip2[8 * h + 4 * k + p2];        // times s_n s_{n + D/2}
                    }
                    // 16-byte chunk c of the row: a 64-column box [32 rows][128 B] of 128-byte swizzle, or the last, 32-column one
                    auto at = [&](int c) -> uint4 * {
                        unsigned char *box = stg + (c >> 3) * (32 * 128);
                        return reinterpret_cast<uint4 *>((c >> 3) < G / 2 ? box + lane * 128 + (((c & 7) ^ (lane & 7)) << 4)
                                                                          : box + lane * 64 + (((c & 3) ^ ((lane >> 1) & 3)) << 4));
                    };
                    *at(2 * h + k) = make_uint4(lo[0], lo[1], lo[2], lo[3]);
                    *at(D / 16 + 2 * h + k) = make_uint4(hi[0], hi[1], hi[2], hi[3]);
                }
            }
            fence_proxy_async();
            __syncwarp();
            if (lane == 0) {
                const int row_in_seg = (int)cur.row_in_segment() + q * 32;
#pragma unroll
                for (int b = 0; b < G / 2; ++b) tma_store_3d(&maps.wide, 64 * b, row_in_seg, cur.seg, smem_u32(stg + b * (32 * 128)));
                if constexpr (G & 1) tma_store_3d(&maps.slim, 64 * (G / 2), row_in_seg, cur.seg, smem_u32(stg + (G / 2) * (32 * 128)));
                bulk_commit();
            }
        }
        if (lane == 0) bulk_wait_all();
    }

    tc_fence_before();
    __syncthreads();
    if (warp == 0) {
        if (*abort_flag) {
            // Every role has left its loop.  x tiles whose loads are still in flight get a bounded chance to land, then tensor-core work that
            // was already issued to drain, before the shared and tensor memory go back.
            if (lane == 0)
                for (int j = issued > kInStages ? issued - kInStages : 0; j < issued; ++j)
                    (void)mbar_wait_bounded(smem_u32(&ctrl->in_full[j % kInStages]), (uint32_t)(j / kInStages) & 1u, 1u << 16);
            __nanosleep(20000);
            __syncwarp();
        }
        tmem_dealloc(tmem_base, kTmemCols);
    }
    // ---- tiles of a lambda row too wide for the fp16 B2: decoded again in fp32 out of the caches, over what the pipeline stored
    if (ctrl->any_wide && !*abort_flag)
        redo_tiles_fp32<D, BF16, 4, kTile>(prm.g, share.begin, n_my, share.tps, rows, reinterpret_cast<float *>(smem));
}

// ------------------------------------------------------------------------------------------------
// host side
// ------------------------------------------------------------------------------------------------
namespace {

template <int D, bool BF16, bool SHORT>
cudaError_t launch_form(const void *x, int64_t N, const GemmParams &g, const float *e0, const uint32_t *sign_xor,
                        uint32_t first_wait_polls, cudaStream_t stream)
{
    using C = Cfg<D, BF16>;
    static DeviceSlots slots;
    int dev = 0;
    cudaError_t e = current_device_slot(&dev);
    if (e != cudaSuccess) return e;
    int &sms = slots.sms[dev];
    if (sms == 0) {
        int n = 0;
        if ((e = cudaFuncSetAttribute(kvq_flush_umma_kernel<D, BF16, SHORT>, cudaFuncAttributeMaxDynamicSharedMemorySize, C::kSmemBytes)) != cudaSuccess) return e;
        if ((e = cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
        sms = n;
    }
    if (N == 0) return cudaSuccess;   // kvq_plan_prepare: the launch attributes are set, there is nothing to run

    UmmaFlushParams prm;
    prm.g = g;
    prm.e0 = e0;
    prm.rows = g.view.rows;
    prm.first_wait_polls = first_wait_polls;
    const int64_t S = N / prm.rows;
    if (N >= (int64_t)1 << 31 || S * g.view.stride >= (int64_t)1 << 31) return cudaErrorInvalidValue;   // tensor-map coordinates are 32-bit
    for (int m = 0; m < D / 4; ++m) prm.flip2[m] = sign_xor[m] ^ sign_xor[m + D / 4];   // words hold two signs each

    UmmaFlushMaps maps;
    const CUtensorMapDataType type = BF16 ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16 : CU_TENSOR_MAP_DATA_TYPE_FLOAT16;
    {
        const cuuint64_t dims[2] = {(cuuint64_t)D, (cuuint64_t)N};
        const cuuint64_t strides[1] = {(cuuint64_t)(2 * D)};
        const cuuint32_t box[2] = {64, (cuuint32_t)kTile};
        if (!make_tensor_map(&maps.x, type, 2, x, dims, strides, box, CU_TENSOR_MAP_SWIZZLE_128B)) return cudaErrorInvalidValue;
    }
    {
        void *out = static_cast<unsigned char *>(g.out) + (size_t)g.view.base * (2 * D);
        const cuuint64_t dims[3] = {(cuuint64_t)D, (cuuint64_t)prm.rows, (cuuint64_t)S};
        const cuuint64_t strides[2] = {(cuuint64_t)(2 * D), (cuuint64_t)(2 * D) * (cuuint64_t)(S > 1 ? g.view.stride : prm.rows)};
        const cuuint32_t wide[3] = {64u, 32u, 1u}, slim[3] = {32u, 32u, 1u};
        if (!make_tensor_map(&maps.wide, type, 3, out, dims, strides, wide, CU_TENSOR_MAP_SWIZZLE_128B) ||
            !make_tensor_map(&maps.slim, type, 3, out, dims, strides, slim, CU_TENSOR_MAP_SWIZZLE_64B))
            return cudaErrorInvalidValue;
    }
    const int64_t tiles = S * ((prm.rows + kTile - 1) / kTile);
    const unsigned grid = (unsigned)(tiles < sms ? tiles : sms);
    prm.plan = TilePlan(S, prm.rows, grid, kTile, g.n_lambda == 1 ? S : g.view.streams_per_lambda.d);
    return launch_kernel(kvq_flush_umma_kernel<D, BF16, SHORT>, prm.plan.shares, C::kThreads, C::kSmemBytes, stream, 1, prm, maps);
}

template <int D, bool BF16>
cudaError_t launch(const void *x, int64_t N, const GemmParams &g, const float *e0, const uint32_t *sign_xor,
                   uint32_t first_wait_polls, cudaStream_t stream)
{
    // 0, and limits that are no shorter than the default: the default
    return first_wait_polls && first_wait_polls < kWaitPolls ? launch_form<D, BF16, true>(x, N, g, e0, sign_xor, first_wait_polls, stream)
                                                             : launch_form<D, BF16, false>(x, N, g, e0, sign_xor, 0, stream);
}

}  // namespace

bool umma_flush_supported(int D) { return D == 64 || D == 96 || D == 128; }

// Where it pays.  A tile takes the contractions, the quantizer and the output one behind the other through one stage each, so a tile
// more costs more than in the two kernels (D = 128 bf16 2.4 us and 2.0, D = 64 1.3 and 1.2; D = 96, with tensor memory to spare, less:
// 1.6 and 1.9), and what is saved is one start.  A call that is waited for pays the tile in full, calls in a stream overlap: the limits
// are the sizes up to which neither is slower.  Tiles per CTA: us per call in a stream over buffers in rotation, two launches -> one,
// and, where the limit is near, between two waits:
//   D = 64  bf16  7: 17.0 -> 15.0   16: 26.5 -> 26.9 (33.8 -> 34.3)   20: 31.5 -> 32.0 (39.0 -> 38.9)   28: 41.7 -> 42.1
//           fp16  7: 16.3 -> 14.3   16: 25.6 -> 25.4                  20: 30.4 -> 30.3 (37.2 -> 37.5)   28: 40.2 -> 40.0
//   D = 96  bf16  7: 23.7 -> 20.8   20: 46.5 -> 42.2   40: 86.5 -> 74.8;  fp16  7: 21.3 -> 17.6   40: 82.3 -> 68.4
//   D = 128 bf16  3: 20.3 -> 16.6   6: 26.7 -> 24.0 (34.8 -> 35.2)   7: 28.9 -> 26.4 (34.2 -> 38.5)   10: 34.4 -> 33.7   14: 42.7 -> 43.3
//           fp16  3: 19.7 -> 17.3   7: 27.5 -> 25.5 (34.3 -> 35.8)   8: 28.9 -> 27.7 (36.1 -> 36.7)   10: 32.5 -> 31.9   14: 40.0 -> 41.7
bool umma_flush_pays(int D, bool bf16, int64_t S, int64_t rows)
{
    static DeviceSlots slots;
    int dev = 0;
    if (!umma_flush_supported(D) || current_device_slot(&dev) != cudaSuccess) return false;
    if (slots.sms[dev] == 0) {
        int n = 0;
        if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return false;
        slots.sms[dev] = n;
    }
    const int64_t tiles = S * ((rows + kTile - 1) / kTile);
    return D == 96 || tiles <= (D == 64 ? 20 : bf16 ? 6 : 8) * (int64_t)slots.sms[dev];
}

cudaError_t umma_flush(int D, bool bf16, const void *x, int64_t N, const GemmParams &g, const float *e0, const uint32_t *sign_xor,
                       uint32_t first_wait_polls, cudaStream_t stream)
{
    if (!tensor_map_encode_fn()) return cudaErrorNotSupported;
    switch (D) {
        case 64: return bf16 ? launch<64, true>(x, N, g, e0, sign_xor, first_wait_polls, stream)
                             : launch<64, false>(x, N, g, e0, sign_xor, first_wait_polls, stream);
        case 96: return bf16 ? launch<96, true>(x, N, g, e0, sign_xor, first_wait_polls, stream)
                             : launch<96, false>(x, N, g, e0, sign_xor, first_wait_polls, stream);
        case 128: return bf16 ? launch<128, true>(x, N, g, e0, sign_xor, first_wait_polls, stream)
                              : launch<128, false>(x, N, g, e0, sign_xor, first_wait_polls, stream);
    }
    return cudaErrorInvalidValue;
}

}  // namespace kvq

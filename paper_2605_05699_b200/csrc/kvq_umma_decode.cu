// Warp-specialised tcgen05 DFT-as-GEMM decode kernel of libkvq (sm_100a): D = 64, 96, 128, 160, fp16 or bf16 output.
//
// The inverse path x^ = diag(s) M^T diag(1 / max(lambda, 1e-6)) (q (.) sigma) (Sec. 3.1: the packing of
// Eq. 2 undone, inverse real DFT, signs last; Sec. 5.1 item 1) is a dense D x D contraction per vector, for any even D (the mixed-radix
// head dims need no special case here).  A tile of 128 vectors is one 128 x D x D GEMM on the
// 5th-generation tensor core, a fraction of the time the tile's bytes need to cross HBM, so the kernel's
// job is to keep HBM busy: one persistent CTA per SM runs four roles that hand tiles to one another
// through mbarriers and never wait for one another's latency.
//
//   warp 0        producer   one TMA tensor load per tile: 128 packed rows into a ring of shared-memory
//                            stages, swizzled (or at a pitch) such that row-per-thread reads are free
//                            of bank conflicts
//   warps 2-9     dequant    two groups of four warps that take alternate tiles.  Thread t of a group
//                            owns row t: nibbles -> fp16 codes -> times sigma * rho, two codes per
//                            half2 instruction (one scale per vector: the codes as they are), stored
//                            straight into TENSOR MEMORY as the A operand (tcgen05.st); the scales
//                            come by plain loads, one tile ahead.
//                            The group that meets the first tile of a new lambda row rebuilds B.
//   warp 1        mma        one thread issues the K-steps of tcgen05.mma (A from tensor memory, B from shared memory; D / 16 of
//                            them, or D / 32 per parity of the radix-2 form) into an accumulator stage and commits
//   warps 10-17   epilogue   two groups of four warps, alternate tiles (both on every tile where there is
//                            one accumulator).  Thread t reads accumulator row t (tcgen05.ld; one scale per
//                            vector: times sigma * rho), rounds, writes a swizzled staging tile; one
//                            lane per warp issues the TMA tensor stores (32 rows x 128 B boxes, plus a
//                            64-byte one when D / 32 is odd).  The output tensor maps are
//                            three-dimensional (column, row within lambda segment, segment), so the
//                            hardware clips a tile that ends with its segment or with the tensor: no
//                            per-row tail code.
//
//   A [128 vectors, K = D]   fp16 in tensor memory: lane = vector, D / 2 columns of two codes each
//   B [N = D outputs, K]     fp16 in shared memory, K-major, 128-byte swizzle, K blocks of 64:
//                            W'[n, c] = s_n M[c, n] / max(lambda_c, 1e-6) / rho, rho a power of two
//   D [128, D]               fp32 accumulator in tensor memory, two stages (one at D = 160 with bf16 output in the radix-2 form)
//
// The K order inside a word of 8 codes is (0,4,1,5,2,6,3,7): that is how the half2 nibble trick
// delivers them, and B is built in the same order, so no instruction is spent on reordering.
//
// Precision: with fp16 output A and B are each rounded once to fp16 (one scale per vector: A is exact), accumulation
// is fp32: about 3e-4 relative L2 per vector before the output rounding.  Every wait on an mbarrier is bounded: on a time-out the role
// records the reason in the status word, raises the CTA's abort flag and leaves its loop; the CTA
// then frees its tensor memory and returns.
#include "kvq_decode_fp32.cuh"
#include "kvq_internal.h"
#include "kvq_umma.cuh"
#include "kvq_umma_decode_operand.cuh"

namespace kvq {

namespace {

constexpr int kTile = 128;       // vectors per tile = MMA M
constexpr int kThreads = 576;    // producer, mma, 2 x 4 dequant, 2 x 4 epilogue warps
constexpr int kBuilders = 12;    // warps that build the first B: the second dequant group and the epilogue
constexpr int kMaxInStages = 6;  // packed tiles in flight, at most
constexpr int kCtrlBytes = 5888;   // barriers and flags, eight tiles' worth of per-row output scales, two rows of reciprocals
constexpr int kRowScaleSlots = 8;  // a dequant group is never more than seven tiles ahead of the epilogue that reads its slot
constexpr uint32_t kTmemCols = 512;

// BF16OUT: bfloat16 output rounds 8x coarser than fp16, and a result that is off by 1e-4 of the vector's rms already
// lands on the other side of enough rounding boundaries to miss the 1e-3 tolerance.  Both operands are then carried
// in two fp16 terms: a = q sigma rho has 15 significant bits and splits exactly into a_hi + a_lo (one half2 FMA),
// W' = W_hi + W_lo, and x^ = a_hi W_hi + a_lo W_hi + a_hi W_lo accumulates in fp32 (a_lo W_lo is below 1e-7).
// BITS: 4 (nibble pairs) or 8 (one two's-complement byte per code; scale = absmax / 127).  The byte path dequantises
// pairs of neighbouring codes, so its K order is the natural one and the B operand is built to match.
// R2: one radix-2 step of the transform is taken out of the GEMM (plans without a rotation).  Rows of M are cos / sin(2 pi k n / D),
// so n -> n + D / 2 multiplies a row by (-1)^k, and in the packing of Eq. 2 the parity of k is the parity of the channel c.  With
// E_n / O_n the sums over the even / odd channels (n < D / 2),
//     x^_n = s_n (E_n + O_n),        x^_{n + D/2} = s_{n + D/2} (E_n - O_n):
// two 128 x D/2 x D/2 GEMMs per tile instead of one 128 x D x D, half the tensor work and half the B operand to build and to hold, for
// an add, a subtract and half a sign flip per output in the epilogue.  The half2 nibble trick yields pairs (c, c + 4) of equal
// parity, a byte permute pairs (c, c + 2), so routing codes to the two A operands is free.  2M vectors at D = 128 back to back: 147 ->
// 134 us (bf16 output: 215 -> 192).  At the other head dimensions, with the
// quads of the table dealt out evenly and elect.sync, dense form -> this: D = 160 bf16 500,000 vectors 87.9 -> 65.0, 99,993 under three
// lambda rows 37.9 -> 19.8; fp16 53.9 -> 45.9; D = 96 bf16 41.0 -> 34.9; D = 64 fp16 1M 42.7 -> 39.2; D = 128 bytes, bf16, 303,067: 36.2 -> 29.6.
// PV: one scale per vector (Sec. 3.2 step 3, Sec. 4.1), in the radix-2 form.  sigma rho is the same for all of a row, so it stands behind the
// contraction: the A operand is the code, exact in one fp16 term, the epilogue multiplies in fp32 (one product and two multiply-adds where it
// had a sum and a difference), and no row needs operand_rescue.  bf16 output then takes two operand sets instead of three and half the
// tensor-memory stores; fp16 output loses the rounding of q sigma rho to 11 bits.  Against the scaled operand, back to back, 592 and
// 2072 tiles: byte codes at D = 128 bf16 10.5 -> 8.5 us and 24.2 -> 20.4, 4-bit codes at D = 160 bf16 14.4 -> 10.6 and 34.4 -> 23.5 (two
// accumulators where two terms leave room for one), at D = 128 fp16 9.2 -> 8.3 and 19.4 -> 17.6.
template <int D, bool BF16OUT, int BITS = 4, bool R2 = false, bool PV = false>
struct Cfg {
    static_assert(D % 32 == 0 && D >= 64 && D <= 160, "head dim not built");
    static_assert(!BF16OUT || BITS == 4 || D <= 128, "two-term operands with byte codes: shared memory holds them for D <= 128 only");
    static_assert(BITS == 4 || BITS == 8, "code width not built");
    static constexpr int kBits = BITS;
    static constexpr bool kRadix2 = R2;
    static constexpr int kTerms = BF16OUT ? 2 : 1;         // W_hi (, W_lo)
    static constexpr int kATerms = BF16OUT && !PV ? 2 : 1; // a_hi (, a_lo)
    static constexpr int G = D / 32;                       // groups = 16-byte chunks of a packed row = 32-column accumulator chunks
    static constexpr int kKSteps = D / 16;
    static constexpr int kKBlocks = (D + 63) / 64;         // K blocks of 64 elements (the last one may be half used)
    static constexpr int kBBlock = D * 128;                // bytes of one K block: D rows x 128 B
    static constexpr int kBTerm = kKBlocks * kBBlock;
    static constexpr int kBPartBlock = (D / 2) * 128;      // R2: one K block of one parity's operand, D / 2 outputs x 64 channels
    static constexpr int kBPart = (D / 2 + 63) / 64 * kBPartBlock;   // D / 2 outputs x D / 2 channels
    static constexpr int kBBytes = R2 ? kTerms * 2 * kBPart : kTerms * kBTerm;   // R2: [term][parity]
    static constexpr int kInRow = D * BITS / 8;            // code bytes per row
    static constexpr int kInBytes = kTile * kInRow;        // bytes one TMA load brings
    static constexpr int kInPitch = (kInBytes + 1023) & ~1023;
    // The packed tile is read row per thread, 16 bytes at a time.  Row pitches of 48 and 80 bytes spread eight
    // consecutive rows over all banks by themselves (96 and 160 bytes over half of them); 32, 64 and 128 bytes need
    // the TMA swizzle of that width.
    static constexpr int kInSwizzleBits = kInRow == 32 ? 1 : kInRow == 64 ? 2 : kInRow == 128 ? 3 : 0;
    static constexpr int kOutWarpBytes = 32 * 2 * D;       // staging of one epilogue warp: G / 2 boxes of 4 KB (+ one of 2 KB)
    static constexpr int kOutBytes = 8 * kOutWarpBytes;
    static constexpr int kRoom = (232448 - 1024 - kCtrlBytes - kBBytes - kOutBytes) / kInPitch;
    static constexpr int kInStages = kRoom < kMaxInStages ? kRoom : kMaxInStages;
    static_assert(kInStages >= (D == 160 && BF16OUT ? 2 : 3), "too few packed tiles in flight");
    static constexpr int kSmemBytes = kBBytes + kInStages * kInPitch + kOutBytes + kCtrlBytes + 1024;
    // tensor memory, D <= 128: two accumulators of up to 128 columns, then the A stages of D / 2 columns per term (a_lo 64 columns
    // behind a_hi).  D = 160: an accumulator and an A term of 80 columns in each half of the 512 columns.  With two-term operands
    // the dense form has a_hi and a_lo of ONE stage there; the radix-2 form, whose MMAs take a third of the time, has two A stages
    // and one accumulator, which the epilogue hands back as soon as it is in registers.
    static constexpr bool kOneAcc = R2 && D == 160 && kATerms == 2;
    static constexpr int kAccStages = kOneAcc ? 1 : 2;
    static constexpr uint32_t kAccStride = D <= 128 ? 128 : 256;
    static constexpr uint32_t kOCol = D == 96 ? 64 : D == 160 ? 96 : D / 2;   // R2: the O columns of an accumulator (E at 0)
    static constexpr int kAStages = kOneAcc ? 2 : kATerms == 2 ? (D <= 128 ? 2 : 1) : D <= 128 ? 4 : 2;
    // The "A full" / "A free" barriers form a ring of at least two, indexed by tile: the two dequant groups take alternate
    // tiles, and a parity wait only tells a phase from its neighbours, so a barrier must not be shared by both groups.
    // Tile j writes A stage j % kAStages once the MMAs of tile j - kAStages have completed (barrier (j - kAStages) % kABars).
    // For the same reason the accumulator's barriers are a ring of two whatever the number of stages.
    static constexpr int kABars = kAStages < 2 ? 2 : kAStages;
    static constexpr uint32_t kALo = kOneAcc ? 80 : D <= 128 ? 64 : 256;
    __host__ __device__ static constexpr uint32_t acc_col(int s) { return (uint32_t)s * kAccStride; }
    __host__ __device__ static constexpr uint32_t a_col(int s)
    {
        return D <= 128 ? 256u + 64u * (uint32_t)kATerms * (uint32_t)s : kOneAcc ? 176u + 160u * (uint32_t)s : (R2 ? 176u : 160u) + 256u * (uint32_t)s;
    }
    static constexpr int kQuads = D / 4;                   // float4 per table row
    static constexpr uint32_t kIdesc = umma_idesc_m128(R2 ? D / 2 : D, false);
    static constexpr int kBRows = R2 ? D / 2 : D;          // rows of the plan table that B is built from
    // The radix-2 epilogue's sums and differences two at a time (add / fma.f32x2): 2,097,152 fp16 vectors at D = 128 128.3 -> 126.0 us,
    // 300,000: 21.0 -> 20.4.  With bf16 output, where a CTA waits for its operands and not for its instructions, single ones: 60,000 vectors
    // at D = 96 9.1, in pairs 9.3; 1,000,000 at D = 160 117 and 123.
    static constexpr bool kPairs = !BF16OUT;
    // The dequant and epilogue loops rolled: five unrolled groups of two-term operands stream a warp through more code than the instruction
    // caches hold beside the other roles' (a warp waits for an instruction 1.2 to 1.4 times per issue).  D = 160, bf16, 18,944 vectors
    // 10.9 -> 10.1 us, 300,000: 40.6 -> 39.4, 1,000,000: 117 -> 108; encode + decode of 99,993 under three lambda rows 38.0 -> 35.7.
    // (60,000 and 128,000 in a row of decodes alone: the same within 1 %.)  The other forms' loops are short enough: rolled they are 2 to 5 % slower.
    static constexpr bool kRolled = R2 && kATerms == 2 && D == 160;
};

struct Ctrl {
    uint64_t in_full[kMaxInStages], in_empty[kMaxInStages];
    uint64_t a_full[4], a_empty[4];
    uint64_t acc_full[2], acc_empty[2];
    uint64_t b_first;
    uint64_t meet[4];   // one accumulator: the two epilogue warps of 32 rows
    uint32_t tmem_base;
    volatile uint32_t abort;
    volatile uint32_t any_wide;   // some lambda row of this CTA's tiles is too wide for the fp16 B operand: redone in fp32 at the end
    alignas(16) float recip[2][160];                      // 1 / (max(lambda, 1e-6) rho) of the row a dequant group builds B for
    float row_scale[kRowScaleSlots][kTile];   // what the epilogue multiplies a row by (1 unless its scales left fp16's comfort zone)
};
static_assert(sizeof(Ctrl) <= kCtrlBytes, "control block too large");

}  // namespace

struct UmmaDecodeParams {
    GemmParams g;
    int64_t rpl;        // rows per lambda segment (N when there is one lambda row)
    TilePlan plan;      // the call's tiles, cut into shares
    int64_t n_full;     // segments of exactly rpl rows, covered by the main output maps; a shorter last one uses the tail maps
    int64_t phys_rows;  // rows of the packed / scales arrays (N, or the whole cache for a cache view)
    uint32_t flip2[40]; // radix-2 form: sign-bit masks of s_n s_{n + D/2} for the output pairs (n, n + 1), n = 0, 2, .. D/2 - 2
};

struct UmmaDecodeMaps {
    CUtensorMap packed;            // [N, D / 2] bytes, box 128 rows
    CUtensorMap wide, wide_tail;   // output, boxes of 64 columns x 32 rows (128-byte swizzle)
    CUtensorMap slim, slim_tail;   // output, boxes of 32 columns x 32 rows (64-byte swizzle), used when D / 32 is odd
};

// The group that meets a lambda row's first tile rebuilds B.  Kept out of line: rare, and the loop around it stays small.
template <int D, bool BF16OUT, int BITS, bool R2, bool PV>
__device__ __noinline__ bool rebuild_b(unsigned char *sB, Ctrl *ctrl, const float *__restrict__ b0, const RecipLambda<D> &rl, int grp, int q, int lane,
                                       int j, uint32_t *status)
{
    using C = Cfg<D, BF16OUT, BITS, R2, PV>;
    inv::BuildB<C, 4> rows;
    rows.load(b0, 0, q, lane);
    // Every MMA issued so far has read B: the commit of the previous tile (the other group's) covers them
    // all.  A parity wait can only tell a phase from its neighbours, and the other group may lag by more
    // than one of its tiles, so first wait for this group's own last tile (its barrier is at most one
    // phase behind, this group waited on it before writing that tile): MMAs complete in order, so after it
    // the previous tile's barrier is at most one phase behind too.
    if (j >= 2 && !wait_or_abort(smem_u32(&ctrl->a_empty[(j - 2) % C::kABars]), (uint32_t)((j - 2) / C::kABars) & 1u, &ctrl->abort, status,
                                 KVQ_DEV_MMA_TIMEOUT))
        return false;
    if (!wait_or_abort(smem_u32(&ctrl->a_empty[(j - 1) % C::kABars]), (uint32_t)((j - 1) / C::kABars) & 1u, &ctrl->abort, status,
                       KVQ_DEV_MMA_TIMEOUT))
        return false;
    // The reciprocals go to shared memory only now that nobody reads the ones before them: the MMAs of tile j - 2 were issued after
    // all four warps of this group had arrived for it, done with what they built there, and those of any tile after the first
    // build, by its builders, out of recip[0].
    inv::post_reciprocals<D>(ctrl->recip[grp], rl, lane);
    rows.store(sB, ctrl->recip[grp], 0, q, lane);
    rows.rest(sB, b0, ctrl->recip[grp], q, lane);
    fence_proxy_async();   // B is read by the tensor core through the async proxy
    return true;
}

// What the dequant warps take from the start: rho of the first lambda row and the scales of their first tile's row.
template <int G>
struct FirstOperand {
    float rho = 1.0f;
    uint32_t sc[(G + 1) / 2] = {};
};

// The way from the kernel's entry through the set-up barrier for warps 2 to 17, and B for the first tile's lambda row by the last
// kBuilders of them (w counts from the first builder on): table rows are requested in front of the grid wait, lambda and scales behind it
// and in front of the barrier.  The group that has the first tile does not build: it dequantises meanwhile, so that the first MMA waits
// for the longer of the two and not for their sum.  Out of line: its registers are then no part of the role loops' allocation.
// One tile per CTA, back to back, before (all sixteen warps build, then one group dequantises, in line) and now: D = 160 bf16
// 9.1 -> 8.2 us, fp16 9.1 -> 8.1, D = 96 fp16 5.7 -> 5.4, D = 128 bf16 7.4 -> 7.2; and for the registers 2072 tiles at D = 160 bf16
// 34.5 -> 32.8, D = 128 bf16 19.4 -> 19.0, fp16 17.3 -> 16.8.  (In line the same split made 2072 tiles at D = 128 bf16 20.5.)
template <int D, bool BF16OUT, int BITS, bool R2>
__device__ __noinline__ FirstOperand<D / 32> first_operand(unsigned char *sB, Ctrl *ctrl, const float *__restrict__ b0, const float *lam,
                                                           const uint16_t *row_scales, int per_vector, int w, int lane)
{
    constexpr int G = D / 32;
    FirstOperand<G> r;
    inv::BuildB<Cfg<D, BF16OUT, BITS, R2>, kBuilders> rows;
    if (w >= 0) rows.load(b0, 0, w, lane);
    grid_wait();
    if (row_scales) {
        if (per_vector) {
            const uint32_t s1 = (uint32_t)load_input(row_scales);
#pragma unroll
            for (int i = 0; i < (G + 1) / 2; ++i) r.sc[i] = s1 | (s1 << 16);
        } else {
            inv::load_row_scales<G>(row_scales, r.sc);
        }
    }
    const RecipLambda<D> rl(lam, lane);
    r.rho = rl.rho;
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (rl.wide) ctrl->any_wide = 1u;
    if (w >= 0) {
        inv::post_reciprocals<D>(ctrl->recip[0], rl, lane);
        rows.store(sB, ctrl->recip[0], 0, w, lane);
        rows.rest(sB, b0, ctrl->recip[0], w, lane);
        fence_proxy_async();   // B is read by the tensor core through the async proxy
        __syncwarp();
        if (lane == 0) mbar_arrive(smem_u32(&ctrl->b_first));
    }
    return r;
}

template <int D, bool BF16OUT, int BITS, bool R2, bool PV>
__global__ void __launch_bounds__(kThreads, 1)
    kvq_decode_umma_kernel(const __grid_constant__ UmmaDecodeParams prm, const __grid_constant__ UmmaDecodeMaps maps)
{
    using C = Cfg<D, BF16OUT, BITS, R2, PV>;
    constexpr int G = C::G, kInStages = C::kInStages, kAccStages = C::kAccStages;
    extern __shared__ unsigned char smem_raw[];
    unsigned char *smem = reinterpret_cast<unsigned char *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    unsigned char *sB = smem;
    unsigned char *sIn = sB + C::kBBytes;
    unsigned char *sOut = sIn + kInStages * C::kInPitch;
    Ctrl *ctrl = reinterpret_cast<Ctrl *>(sOut + C::kOutBytes);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

    if (threadIdx.x == 0) {
        for (int s = 0; s < kInStages; ++s) {
            mbar_init(smem_u32(&ctrl->in_full[s]), 1);
            mbar_init(smem_u32(&ctrl->in_empty[s]), 4);
        }
        for (int s = 0; s < C::kABars; ++s) {
            mbar_init(smem_u32(&ctrl->a_full[s]), 4);
            mbar_init(smem_u32(&ctrl->a_empty[s]), 1);
        }
        for (int s = 0; s < 2; ++s) {
            mbar_init(smem_u32(&ctrl->acc_full[s]), 1);
            mbar_init(smem_u32(&ctrl->acc_empty[s]), C::kOneAcc ? 8 : 4);
        }
        if constexpr (C::kOneAcc)
            for (int s = 0; s < 4; ++s) mbar_init(smem_u32(&ctrl->meet[s]), 2);
        mbar_init(smem_u32(&ctrl->b_first), kBuilders);
        ctrl->abort = 0u;
        ctrl->any_wide = 0u;
        mbar_init_fence();
        fence_proxy_async();
    }
    if (warp == 1) tmem_alloc(smem_u32(&ctrl->tmem_base), kTmemCols);

    // ---- tiles: lambda segments of rpl rows, cut into tiles of 128 rows; a contiguous range of tiles
    // ---- per CTA, so that the B operand is rebuilt as rarely as possible
    const int64_t rpl = prm.rpl;
    const TileShare share(prm.plan, blockIdx.x);
    const int n_my = share.n;
    const int64_t seg_first = share.seg;
    auto lambda_row = [&](int64_t seg) -> const float * { return prm.g.lambda + prm.g.lambda_index(seg) * D; };

    // ---- B for the first tile's lambda row (first_operand).  The dequant warps also request the scales of their first tile there and
    // ---- keep rho, so that neither costs a round trip to L2 afterwards.
    const bool per_vector = PV || (!R2 && prm.g.per_vector);
    FirstOperand<G> first;
    if (n_my > 0 && warp >= 2) {
        const uint16_t *row_scales = nullptr;
        if (warp < 10 && ((warp - 2) >> 2) < n_my) {   // dequant group g's first tile is the share's tile g
            const TileCursor at(share, (warp - 2) >> 2);
            const int64_t row = prm.g.phys_row(at.seg, at.row_in_segment(), rpl) + (warp & 3) * 32 + lane;
            if (row < prm.phys_rows) row_scales = static_cast<const uint16_t *>(prm.g.scales) + row * (per_vector ? 1 : G);
        }
        first = first_operand<D, BF16OUT, BITS, R2>(sB, ctrl, prm.g.b0, lambda_row(seg_first), row_scales, per_vector, warp - (18 - kBuilders), lane);
    } else {
        grid_wait();
        tc_fence_before();
        __syncthreads();
        tc_fence_after();
    }
    const uint32_t tmem_base = ctrl->tmem_base;
    volatile uint32_t *abort_flag = &ctrl->abort;
    uint32_t *status = prm.g.status;

    if (warp == 0) {
        // =========================== producer ===========================
        if (lane == 0) {
            int issued = 0;
            bool ok = true;
            TileCursor cur(share);
            for (int j = 0; j < n_my; ++j, cur.advance(1)) {
                const int s = j % kInStages;
                const uint32_t use = (uint32_t)(j / kInStages);
                ok = wait_or_abort(smem_u32(&ctrl->in_empty[s]), (use & 1u) ^ 1u, abort_flag, status, KVQ_DEV_SLOT_TIMEOUT);
                if (!ok) break;
                const int64_t row0 = prm.g.phys_row(cur.seg, cur.row_in_segment(), rpl);   // rows past the segment are read and never stored
                const uint32_t bar = smem_u32(&ctrl->in_full[s]);
                mbar_arrive_expect_tx(bar, C::kInBytes);
                tma_load_2d(smem_u32(sIn + s * C::kInPitch), &maps.packed, 0, (int)row0, bar);
                issued = j + 1;
            }
            if (!ok) {
                // give this thread's own copies in flight a bounded chance to land before the CTA goes away
                for (int j = issued > kInStages ? issued - kInStages : 0; j < issued; ++j)
                    (void)mbar_wait_bounded(smem_u32(&ctrl->in_full[j % kInStages]), (uint32_t)(j / kInStages) & 1u, 1u << 16);
            }
        }
        __syncwarp();
        grid_trigger();   // the last load is on its way
    } else if (warp == 1) {
        // =========================== mma issuer ===========================
        // (elect.sync, not lane 0: the compiler then knows that one thread issues.  128 x 64 x 16 with A in tensor memory: 32 cycles, else 45)
        if (elect_one()) {
            const uint64_t b_desc = smem_desc_sw128(smem_u32(sB));
            const uint32_t b_lo = (uint32_t)b_desc, b_hi = (uint32_t)(b_desc >> 32);
            int n_mma = n_my;
            if (n_my > 0 && !wait_or_abort(smem_u32(&ctrl->b_first), 0u, abort_flag, status, KVQ_DEV_SLOT_TIMEOUT)) n_mma = 0;
            for (int j = 0; j < n_mma; ++j) {
                const int sa = j % C::kAStages, sb = j % C::kABars, sc = j % kAccStages;
                if (!wait_or_abort(smem_u32(&ctrl->a_full[sb]), (uint32_t)(j / C::kABars) & 1u, abort_flag, status, KVQ_DEV_SLOT_TIMEOUT)) break;
                if (j >= kAccStages) {   // the epilogue has taken the tile that used this accumulator last
                    const int jp = j - kAccStages;
                    if (!wait_or_abort(smem_u32(&ctrl->acc_empty[jp & 1]), (uint32_t)(jp >> 1) & 1u, abort_flag, status, KVQ_DEV_SLOT_TIMEOUT)) break;
                }
                tc_fence_after();
                const uint32_t d_tmem = tmem_base + C::acc_col(sc);
                const uint32_t a_tmem = tmem_base + C::a_col(sa);
                if constexpr (R2) {   // E = A_even B_even into the first D / 2 accumulator columns, O = A_odd B_odd into the rest
#pragma unroll
                    for (int p = 0; p < 2; ++p) {
#pragma unroll
                        for (int set = 0; set < C::kATerms + C::kTerms - 1; ++set) {   // bf16 output: a_hi W_hi + a_lo W_hi + a_hi W_lo, or a W_hi + a W_lo
#pragma unroll
                            for (int ks = 0; ks < D / 32; ++ks) {
                                const uint32_t b_set = b_lo + (set == C::kATerms ? (uint32_t)((2 * C::kBPart) >> 4) : 0u) + (uint32_t)p * (C::kBPart >> 4);
                                const uint64_t bd = ((uint64_t)b_hi << 32) | (uint64_t)(b_set + (uint32_t)(ks >> 2) * (C::kBPartBlock >> 4) + (uint32_t)(ks & 3) * 2u);
                                const uint32_t dp = d_tmem + (uint32_t)p * C::kOCol;
                                const uint32_t ap = a_tmem + (C::kATerms == 2 && set == 1 ? C::kALo : 0u) + (uint32_t)p * (D / 4) + (uint32_t)ks * 8u;
                                if (set > 0 || ks > 0) umma_f16_ts<true>(dp, ap, bd, C::kIdesc);
                                else umma_f16_ts<false>(dp, ap, bd, C::kIdesc);
                            }
                        }
                    }
                }
                // bf16 output: a_hi W_hi + a_lo W_hi + a_hi W_lo
#pragma unroll
                for (int set = 0; set < (R2 ? 0 : BF16OUT ? 3 : 1); ++set) {
                    const uint32_t a_set = a_tmem + (set == 1 ? C::kALo : 0u);
                    const uint32_t b_set = b_lo + (set == 2 ? (uint32_t)(C::kBTerm >> 4) : 0u);
#pragma unroll
                    for (int ks = 0; ks < C::kKSteps; ++ks) {
                        const uint32_t koff = (uint32_t)(ks >> 2) * (C::kBBlock >> 4) + (uint32_t)(ks & 3) * 2u;   // (bytes >> 4) of K-step ks
                        const uint64_t bd = ((uint64_t)b_hi << 32) | (uint64_t)(b_set + koff);
                        if (set > 0 || ks > 0) umma_f16_ts<true>(d_tmem, a_set + (uint32_t)ks * 8u, bd, C::kIdesc);
                        else umma_f16_ts<false>(d_tmem, a_set, bd, C::kIdesc);
                    }
                }
                umma_commit(smem_u32(&ctrl->acc_full[j & 1]));
                umma_commit(smem_u32(&ctrl->a_empty[sb]));
            }
        }
    } else if (warp < 10) {
        // =========================== dequant: packed codes -> A in tensor memory ===========================
        const int grp = (warp - 2) >> 2;        // this group takes tiles grp, grp + 2, ...
        const int q = warp & 3;                 // tensor-memory lane quarter this warp may touch
        const int r = q * 32 + lane;            // tile row and tensor-memory lane of this thread
        const uint16_t *scales = static_cast<const uint16_t *>(prm.g.scales);   // D / 32 fp16 scales per row
        const uint32_t swz = C::kInSwizzleBits == 3   ? (uint32_t)(r & 7)
                             : C::kInSwizzleBits == 2 ? (uint32_t)((r >> 1) & 3)
                             : C::kInSwizzleBits == 1 ? (uint32_t)((r >> 2) & 1)
                                                      : 0u;
        int64_t cached_row = n_my > 0 ? prm.g.lambda_index(seg_first) : -1;   // the lambda row that B holds (built above)
        float rho = first.rho;

        TileCursor cur(share, grp), ahead = cur;   // this tile; the tile whose scales are fetched
        uint32_t sc_next[(G + 1) / 2];
        auto fetch_scales = [&](int j) {
#pragma unroll
            for (int i = 0; i < (G + 1) / 2; ++i) sc_next[i] = 0u;
            if (j < n_my) {
                const int64_t row = prm.g.phys_row(ahead.seg, ahead.row_in_segment(), rpl) + r;
                if (row < prm.phys_rows) {
                    if (per_vector) {   // one scale per vector: the same value in every group's slot
                        const uint32_t s1 = (uint32_t)load_input(scales + row);
#pragma unroll
                        for (int i = 0; i < (G + 1) / 2; ++i) sc_next[i] = s1 | (s1 << 16);
                    } else {
                        inv::load_row_scales<G>(scales + row * G, sc_next);
                    }
                }
            }
        };

#pragma unroll
        for (int i = 0; i < (G + 1) / 2; ++i) sc_next[i] = first.sc[i];   // requested before the first B build
        for (int j = grp; j < n_my; j += 2, cur.advance(2)) {
            uint32_t sc[(G + 1) / 2];
#pragma unroll
            for (int i = 0; i < (G + 1) / 2; ++i) sc[i] = sc_next[i];
            ahead.advance(2);
            fetch_scales(j + 2);
            const int64_t seg = cur.seg;

            // ---- a new lambda row: this group needs its rho; the group that meets the row's first tile rebuilds B
            const int64_t row_of_seg = prm.g.lambda_index(seg);
            if (row_of_seg != cached_row) {
                const RecipLambda<D> rl(lambda_row(seg), lane);
                rho = rl.rho;
                if (rl.wide) ctrl->any_wide = 1u;
                if (cur.first_of_segment() && prm.g.lambda_index(seg - 1) != row_of_seg) {
                    if (!rebuild_b<D, BF16OUT, BITS, R2, PV>(sB, ctrl, prm.g.b0, rl, grp, q, lane, j, status)) break;
                }
                cached_row = row_of_seg;
            }

            // ---- this tile's packed rows have landed; the A stage is free again
            const int s = j % kInStages, sa = j % C::kAStages, sb = j % C::kABars;
            if (!wait_or_abort(smem_u32(&ctrl->in_full[s]), (uint32_t)(j / kInStages) & 1u, abort_flag, status, KVQ_DEV_LOAD_TIMEOUT)) break;
            const unsigned char *row = sIn + s * C::kInPitch + r * C::kInRow;
            constexpr bool kAllCodes = BITS == 4 && !C::kRolled;   // the whole row's codes at once, or group by group
            uint4 pk[kAllCodes ? G : 1];
            if constexpr (kAllCodes) {
#pragma unroll
                for (int c = 0; c < G; ++c) pk[c] = *reinterpret_cast<const uint4 *>(row + (((uint32_t)c ^ swz) << 4));
                __syncwarp();
                if (lane == 0) mbar_arrive(smem_u32(&ctrl->in_empty[s]));   // the values are in registers
            }
            if (j >= C::kAStages) {   // the MMAs that read this A stage last
                const int jp = j - C::kAStages;
                if (!wait_or_abort(smem_u32(&ctrl->a_empty[jp % C::kABars]), (uint32_t)(jp / C::kABars) & 1u, abort_flag, status,
                                   KVQ_DEV_MMA_TIMEOUT))
                    break;
            }
            tc_fence_after();

            // ---- the A operand q sigma rho is fp16.  A row whose scales would take it out of fp16's normal range (a very
            // ---- small or very large vector) is carried times a power of two instead, which the epilogue takes out again
            // ---- in fp32; every other row has the factor 1 and costs the epilogue nothing.
            // ---- One scale per vector (PV): the operand is the code itself, and the epilogue multiplies by sigma rho.
            float inv, pw = 1.0f;
            if constexpr (PV) inv = vector_factor(sc[0], rho);
            else pw = operand_rescue<G>(sc, rho, BITS == 4 ? 9000.0f : 500.0f, inv);   // 7 (127) times this stays inside fp16
            ctrl->row_scale[j & (kRowScaleSlots - 1)][r] = inv;
            // ---- nibbles -> fp16 codes -> times sigma * rho, two codes per instruction
            const uint32_t a_row = tmem_base + ((uint32_t)(q * 32) << 16) + C::a_col(sa);
            const __half2 h1032 = __float2half2_rn(1032.0f);
#pragma unroll(C::kRolled ? 1 : G)
            for (int c = 0; c < G; ++c) {   // chunk c = group c: 32 codes, 16 tensor-memory columns
                uint32_t sc16 = sc[0];
                if constexpr (C::kRolled) {
#pragma unroll
                    for (int i = 0; i < (G + 1) / 2; ++i) sc[i] = (sc[i] >> 16) | (i + 1 < (G + 1) / 2 ? sc[i + 1] << 16 : 0u);   // the next group's to the front
                } else {
                    sc16 = sc[c >> 1] >> (16 * (c & 1));
                }
                const float sig = __half2float(__ushort_as_half((unsigned short)(sc16 & 0xFFFFu)));
                const __half2 s2 = __float2half2_rn(sig * rho * pw);
                uint32_t a[16], al[C::kATerms == 2 ? 16 : 1];
                auto put = [&](int k, __half2 q2) {   // K-pair k of the group: one rounding, and what it left behind
                    const __half2 h = PV ? q2 : __hmul2(q2, s2);
                    a[k] = *reinterpret_cast<const uint32_t *>(&h);
                    if constexpr (C::kATerms == 2) {   // q s2 - h, exact in fp16
                        const __half2 l = __hfma2(q2, s2, __hneg2(h));
                        al[k] = *reinterpret_cast<const uint32_t *>(&l);
                    }
                };
                if constexpr (BITS == 4) {
                    uint4 pc;
                    if constexpr (kAllCodes) pc = pk[c];
                    else pc = *reinterpret_cast<const uint4 *>(row + (((uint32_t)c ^ swz) << 4));
                    const uint32_t words[4] = {pc.x, pc.y, pc.z, pc.w};
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const uint32_t u = words[i] ^ 0x88888888u;   // nibbles now hold q + 8
#pragma unroll
                        for (int e = 0; e < 4; ++e) {
                            const uint32_t m = lop3_and_or(u >> (4 * e), 0x000F000Fu, 0x64006400u);   // {1024 + n_e, 1024 + n_{e+4}}
                            // radix-2 form: pairs 0 and 2 of a word are even channels (first half of a[]), 1 and 3 odd (second half)
                            put(R2 ? 8 * (e & 1) + 2 * i + (e >> 1) : 4 * i + e, __hsub2(*reinterpret_cast<const __half2 *>(&m), h1032));   // exact q
                        }
                    }
                } else {   // 32 byte codes: two 16-byte chunks of the row, pairs of neighbours
                    const __half2 h1152 = __float2half2_rn(1152.0f);
#pragma unroll
                    for (int hc = 0; hc < 2; ++hc) {
                        const uint4 pc = *reinterpret_cast<const uint4 *>(row + (((uint32_t)(2 * c + hc) ^ swz) << 4));
                        const uint32_t words[4] = {pc.x, pc.y, pc.z, pc.w};
#pragma unroll
                        for (int i = 0; i < 4; ++i) {
                            const uint32_t u = words[i] ^ 0x80808080u;                 // bytes now hold q + 128
                            // {1024 + b, 1024 + b'} as fp16 bit patterns: bytes 0, 1 and 2, 3, or 0, 2 (even channels) and 1, 3 (odd)
                            const uint32_t ma = __byte_perm(u, 0x64646464u, R2 ? 0x4240 : 0x4140);
                            const uint32_t mb = __byte_perm(u, 0x64646464u, R2 ? 0x4341 : 0x4342);
                            put(R2 ? 4 * hc + i : 8 * hc + 2 * i, __hsub2(*reinterpret_cast<const __half2 *>(&ma), h1152));       // exact q
                            put(R2 ? 8 + 4 * hc + i : 8 * hc + 2 * i + 1, __hsub2(*reinterpret_cast<const __half2 *>(&mb), h1152));
                        }
                    }
                }
                if constexpr (R2) {   // 8 columns of the even operand, 8 of the odd one
                    const uint32_t ae[8] = {a[0], a[1], a[2], a[3], a[4], a[5], a[6], a[7]};
                    const uint32_t ao[8] = {a[8], a[9], a[10], a[11], a[12], a[13], a[14], a[15]};
                    tmem_st8(a_row + 8u * (uint32_t)c, ae);
                    tmem_st8(a_row + (uint32_t)(D / 4) + 8u * (uint32_t)c, ao);
                    if constexpr (C::kATerms == 2) {
                        const uint32_t le[8] = {al[0], al[1], al[2], al[3], al[4], al[5], al[6], al[7]};
                        const uint32_t lo[8] = {al[8], al[9], al[10], al[11], al[12], al[13], al[14], al[15]};
                        tmem_st8(a_row + C::kALo + 8u * (uint32_t)c, le);
                        tmem_st8(a_row + C::kALo + (uint32_t)(D / 4) + 8u * (uint32_t)c, lo);
                    }
                } else {
                    tmem_st16(a_row + 16u * (uint32_t)c, a);
                    if constexpr (C::kATerms == 2) tmem_st16(a_row + C::kALo + 16u * (uint32_t)c, al);
                }
            }
            if constexpr (!kAllCodes) {   // the packed rows were read group by group: only now is their stage free
                __syncwarp();
                if (lane == 0) mbar_arrive(smem_u32(&ctrl->in_empty[s]));
            }
            tmem_st_wait();
            tc_fence_before();
            __threadfence_block();   // the row scales, for the epilogue that follows this tile's accumulator
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&ctrl->a_full[sb]));
        }
    } else {
        // =========================== epilogue: accumulator -> fp16 -> TMA store ===========================
        const int grp = (warp - 10) >> 2;
        const int q = warp & 3;
        const uint32_t lane_addr = tmem_base + ((uint32_t)(q * 32) << 16);
        // One accumulator: both groups take every tile, the first three fifths of its columns and the rest, so that it goes back sooner;
        // the two warps that share 32 rows fill one staging tile of two and meet before the first of them stores it.  bf16, 296, 1036 and
        // 2072 tiles 9.74 -> 9.64 us, 18.5 -> 17.8 and 32.7 -> 31.0.  (148, a tile per CTA, 8.1 -> 8.2; chosen at run time 8.5.)
        constexpr bool both = C::kOneAcc;
        constexpr int step = both ? 1 : 2;
        const int h0 = both && grp == 1 ? 3 : 0, h1 = both && grp == 0 ? 3 : D / 32;   // 16-column steps of each parity
        TileCursor cur(share, both ? 0 : grp);
        for (int j = both ? 0 : grp; j < n_my; j += step, cur.advance(step)) {
            const int sc = j % kAccStages;
            unsigned char *stg = sOut + (both ? (j & 1) * 4 + (warp - 10) % 4 : warp - 10) * C::kOutWarpBytes;   // this warp's staging tile
            if (!wait_or_abort(smem_u32(&ctrl->acc_full[j & 1]), (uint32_t)(j >> 1) & 1u, abort_flag, status, KVQ_DEV_MMA_TIMEOUT)) break;
            tc_fence_after();
            if (!both && lane == 0) bulk_wait_read_all();   // this warp's previous stores have read the staging tile
            __syncwarp();
            const float row_inv = ctrl->row_scale[j & (kRowScaleSlots - 1)][q * 32 + lane];
            const bool rescale = !PV && __any_sync(0xFFFFFFFFu, row_inv != 1.0f);   // rare: a row outside the operand's comfort zone
            const uint64_t rs2 = pack_f32x2(row_inv, row_inv), neg2 = pack_f32x2(-row_inv, -row_inv);   // PV: sigma rho
            if constexpr (R2) {
#pragma unroll(C::kRolled ? 1 : D / 32)
                for (int h = C::kOneAcc ? h0 : 0; h < (C::kOneAcc ? h1 : D / 32); ++h) {   // E and O columns 16 h .. 16 h + 15 -> outputs 16 h .. and D / 2 + 16 h ..
                    uint32_t ev[16], ov[16];
                    tmem_ld16(lane_addr + C::acc_col(sc) + (uint32_t)h * 16u, ev);
                    tmem_ld16(lane_addr + C::acc_col(sc) + C::kOCol + (uint32_t)h * 16u, ov);
                    tmem_ld_wait();
                    if (h == (C::kOneAcc ? h1 : D / 32) - 1) {   // the last values are in registers: hand the accumulator back
                        tc_fence_before();
                        __syncwarp();
                        if (lane == 0) mbar_arrive(smem_u32(&ctrl->acc_empty[j & 1]));
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
                            const float2 e = make_float2(__uint_as_float(ev[i]), __uint_as_float(ev[i + 1]));
                            const float2 o = make_float2(__uint_as_float(ov[i]), __uint_as_float(ov[i + 1]));
                            float2 sum, diff;
                            if constexpr (PV) {   // (E + O) sigma rho, (E - O) sigma rho
                                const uint64_t ep = mul_f32x2(pack_f32x2(e.x, e.y), rs2), op = pack_f32x2(o.x, o.y);
                                sum = unpack_f32x2(fma_f32x2(op, rs2, ep)), diff = unpack_f32x2(fma_f32x2(op, neg2, ep));
                            } else if constexpr (C::kPairs) {
                                const uint64_t ep = pack_f32x2(e.x, e.y), op = pack_f32x2(o.x, o.y);
                                sum = unpack_f32x2(add_f32x2(ep, op)), diff = unpack_f32x2(sub_f32x2(ep, op));
                            } else {
                                sum = make_float2(e.x + o.x, e.y + o.y), diff = make_float2(e.x - o.x, e.y - o.y);
                            }
                            lo[p2] = narrow2<BF16OUT>(sum.x, sum.y);                                          // s_n is already in E and O
                            hi[p2] = narrow2<BF16OUT>(diff.x, diff.y) ^ prm.flip2[8 * h + 4 * k + p2];       // times s_n s_{n + D/2}
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
            }
#pragma unroll
            for (int cc = 0; cc < (R2 ? 0 : G); ++cc) {   // 32 accumulator columns = 64 bytes of the output row
                uint32_t v[32];
                tmem_ld32(lane_addr + C::acc_col(sc) + (uint32_t)cc * 32u, v);
                tmem_ld_wait();
                if (rescale) {
#pragma unroll
                    for (int i = 0; i < 32; ++i) v[i] = __float_as_uint(__uint_as_float(v[i]) * row_inv);
                }
                constexpr int kWideBoxes = G / 2;
                const bool wide = (cc >> 1) < kWideBoxes;   // inside a 64-column box, or the last 32-column one
                unsigned char *box = stg + (cc >> 1) * (32 * 128);
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    uint4 o;
                    o.x = narrow2<BF16OUT>(__uint_as_float(v[8 * k]), __uint_as_float(v[8 * k + 1]));
                    o.y = narrow2<BF16OUT>(__uint_as_float(v[8 * k + 2]), __uint_as_float(v[8 * k + 3]));
                    o.z = narrow2<BF16OUT>(__uint_as_float(v[8 * k + 4]), __uint_as_float(v[8 * k + 5]));
                    o.w = narrow2<BF16OUT>(__uint_as_float(v[8 * k + 6]), __uint_as_float(v[8 * k + 7]));
                    if (wide) {   // [32 rows][128 B], 128-byte swizzle
                        const int chunk = (cc & 1) * 4 + k;
                        *reinterpret_cast<uint4 *>(box + lane * 128 + ((chunk ^ (lane & 7)) << 4)) = o;
                    } else {      // [32 rows][64 B], 64-byte swizzle
                        *reinterpret_cast<uint4 *>(box + lane * 64 + ((k ^ ((lane >> 1) & 3)) << 4)) = o;
                    }
                }
            }
            tc_fence_before();
            fence_proxy_async();
            __syncwarp();
            if (both) {
                if (lane == 0) {
                    if (grp == 0) bulk_wait_read_all();   // the tile before has left the other staging tile: its partner may fill that next
                    mbar_arrive(smem_u32(&ctrl->meet[q]));
                }
                if (!wait_or_abort(smem_u32(&ctrl->meet[q]), (uint32_t)j & 1u, abort_flag, status, KVQ_DEV_SLOT_TIMEOUT)) break;
            }
            if (lane == 0 && (!both || grp == 0)) {
                if constexpr (!R2) mbar_arrive(smem_u32(&ctrl->acc_empty[j & 1]));
                const int64_t seg = cur.seg;
                const int row_in_seg = (int)cur.row_in_segment() + q * 32;
                const bool tail = seg >= prm.n_full;
                const int segc = tail ? 0 : (int)seg;
                const CUtensorMap *tw = tail ? &maps.wide_tail : &maps.wide;
#pragma unroll
                for (int b = 0; b < G / 2; ++b) tma_store_3d(tw, 64 * b, row_in_seg, segc, smem_u32(stg + b * (32 * 128)));
                if constexpr (G & 1) {
                    const CUtensorMap *ts = tail ? &maps.slim_tail : &maps.slim;
                    tma_store_3d(ts, 64 * (G / 2), row_in_seg, segc, smem_u32(stg + (G / 2) * (32 * 128)));
                }
                bulk_commit();
            }
        }
        if (lane == 0) bulk_wait_all();
    }

    tc_fence_before();
    __syncthreads();
    if (warp == 0) {
        if (*abort_flag) __nanosleep(20000);   // let tensor-core work that was already issued drain
        tmem_dealloc(tmem_base, kTmemCols);
    }
    // ---- tiles of a lambda row too wide for the fp16 B operand: decoded again in fp32, over what the pipeline stored
    if (ctrl->any_wide && !*abort_flag)
        redo_tiles_fp32<D, BF16OUT, BITS, kTile>(prm.g, share.begin, n_my, share.tps, rpl, reinterpret_cast<float *>(smem));
}

// ------------------------------------------------------------------------------------------------
// host side
// ------------------------------------------------------------------------------------------------
namespace {

template <int D, bool BF16OUT, int BITS, bool R2, bool PV>
cudaError_t launch_form(int64_t N, const GemmParams &g, cudaStream_t stream, const uint32_t *sign_xor)
{
    using C = Cfg<D, BF16OUT, BITS, R2, PV>;
    static DeviceSlots slots;
    int dev = 0;
    cudaError_t e = current_device_slot(&dev);
    if (e != cudaSuccess) return e;
    int &sms = slots.sms[dev];
    if (sms == 0) {
        int n = 0;
        if ((e = cudaFuncSetAttribute(kvq_decode_umma_kernel<D, BF16OUT, BITS, R2, PV>, cudaFuncAttributeMaxDynamicSharedMemorySize, C::kSmemBytes)) != cudaSuccess) return e;
        if ((e = cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
        sms = n;
    }
    if (!tensor_map_encode_fn()) return cudaErrorNotSupported;
    if (N == 0) return cudaSuccess;   // kvq_plan_prepare: the launch attributes are set, there is nothing to run
    if (N >= (int64_t)1 << 31) return cudaErrorInvalidValue;   // tensor-map coordinates are 32-bit

    UmmaDecodeParams prm;
    prm.g = g;
    prm.rpl = g.view.rows ? g.view.rows : g.n_lambda == 1 || g.rows_per_lambda > N ? N : g.rows_per_lambda;   // a cache view: one segment per stream
    const int64_t n_seg = (N + prm.rpl - 1) / prm.rpl;
    const int64_t segs = g.n_lambda == 1 ? n_seg : g.view.rows ? g.view.streams_per_lambda.d : 1;   // consecutive segments with one lambda row
    prm.n_full = N / prm.rpl;
    prm.phys_rows = g.view.rows ? n_seg * g.view.stride : N;
    if (prm.phys_rows >= (int64_t)1 << 31) return cudaErrorInvalidValue;
    const int64_t seg_stride = g.view.rows ? g.view.stride : prm.rpl;   // rows from one segment's first row to the next's
    unsigned char *out0 = static_cast<unsigned char *>(g.out) + (size_t)(g.view.rows ? g.view.base : 0) * (2 * D);
    for (int m = 0; m < D / 4; ++m) prm.flip2[m] = R2 && sign_xor ? sign_xor[m] ^ sign_xor[m + D / 4] : 0u;   // words hold two signs each

    UmmaDecodeMaps maps;
    {
        const cuuint64_t dims[2] = {(cuuint64_t)C::kInRow, (cuuint64_t)prm.phys_rows};
        const cuuint64_t strides[1] = {(cuuint64_t)C::kInRow};
        const cuuint32_t box[2] = {(cuuint32_t)C::kInRow, (cuuint32_t)kTile};
        const CUtensorMapSwizzle sw = C::kInSwizzleBits == 3   ? CU_TENSOR_MAP_SWIZZLE_128B
                                      : C::kInSwizzleBits == 2 ? CU_TENSOR_MAP_SWIZZLE_64B
                                      : C::kInSwizzleBits == 1 ? CU_TENSOR_MAP_SWIZZLE_32B
                                                               : CU_TENSOR_MAP_SWIZZLE_NONE;
        if (!make_tensor_map(&maps.packed, CU_TENSOR_MAP_DATA_TYPE_UINT8, 2, g.packed, dims, strides, box, sw)) return cudaErrorInvalidValue;
    }
    auto out_map = [&](CUtensorMap *tm, void *base, int64_t rows, int64_t segs, bool wide) -> bool {
        const cuuint64_t dims[3] = {(cuuint64_t)D, (cuuint64_t)rows, (cuuint64_t)segs};
        const cuuint64_t strides[2] = {(cuuint64_t)(2 * D), (cuuint64_t)(2 * D) * (cuuint64_t)(segs > 1 ? seg_stride : rows)};
        const cuuint32_t box[3] = {wide ? 64u : 32u, 32u, 1u};
        return make_tensor_map(tm, BF16OUT ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16 : CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 3, base, dims, strides, box,
                               wide ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_64B);
    };
    const int64_t tail_rows = N - prm.n_full * prm.rpl;
    unsigned char *tail_base = out0 + (size_t)prm.n_full * seg_stride * (2 * D);
    if (prm.n_full > 0 && (!out_map(&maps.wide, out0, prm.rpl, prm.n_full, true) || !out_map(&maps.slim, out0, prm.rpl, prm.n_full, false)))
        return cudaErrorInvalidValue;
    if (tail_rows > 0 && (!out_map(&maps.wide_tail, tail_base, tail_rows, 1, true) || !out_map(&maps.slim_tail, tail_base, tail_rows, 1, false)))
        return cudaErrorInvalidValue;
    if (tail_rows == 0) maps.wide_tail = maps.wide, maps.slim_tail = maps.slim;
    if (prm.n_full == 0) maps.wide = maps.wide_tail, maps.slim = maps.slim_tail;

    const int64_t tiles = n_seg * ((prm.rpl + kTile - 1) / kTile);
    const int grid = (int)(tiles < sms ? tiles : sms);
    prm.plan = TilePlan(n_seg, prm.rpl, (unsigned)grid, kTile, segs);
    return launch_kernel(kvq_decode_umma_kernel<D, BF16OUT, BITS, R2, PV>, prm.plan.shares, kThreads, C::kSmemBytes, stream, 1, prm, maps);
}

template <int D, bool BF16OUT, int BITS = 4, bool R2 = false>
cudaError_t launch(int64_t N, const GemmParams &g, cudaStream_t stream, const uint32_t *sign_xor = nullptr)
{
    if constexpr (R2)
        if (g.per_vector) return launch_form<D, BF16OUT, BITS, R2, true>(N, g, stream, sign_xor);
    return launch_form<D, BF16OUT, BITS, R2, false>(N, g, stream, sign_xor);
}

}  // namespace

bool umma_decode_supported(int D, bool bf16)
{
    (void)bf16;
    return D == 256 || D == 64 || D == 96 || D == 128 || D == 160;
}

// byte codes: every kernel but the D = 160 bf16 form (and the dense D = 256 kernel of rotated plans, which the caller excludes)
bool umma_decode_bits8_supported(int D, bool bf16) { return !(D == 160 && bf16) && umma_decode_supported(D, bf16); }

cudaError_t umma_decode(int D, bool bf16, int bits, int64_t N, const GemmParams &g, const uint32_t *sign_xor, cudaStream_t stream,
                        bool radix2)
{
    if (D == 256 && sign_xor) return umma_decode_d256(bf16, bits, N, g, sign_xor, stream);   // its own kernel: radix-2 split, split operands for bf16
    // the radix-2 form needs the transform's even / odd structure: the caller asks for it on plans without a rotation
    if (radix2 && sign_xor) {
        if (bits == 8) {
            switch (D) {
                case 64: return bf16 ? launch<64, true, 8, true>(N, g, stream, sign_xor) : launch<64, false, 8, true>(N, g, stream, sign_xor);
                case 96: return bf16 ? launch<96, true, 8, true>(N, g, stream, sign_xor) : launch<96, false, 8, true>(N, g, stream, sign_xor);
                case 128: return bf16 ? launch<128, true, 8, true>(N, g, stream, sign_xor) : launch<128, false, 8, true>(N, g, stream, sign_xor);
                case 160: return bf16 ? cudaErrorInvalidValue : launch<160, false, 8, true>(N, g, stream, sign_xor);
            }
            return cudaErrorInvalidValue;
        }
        switch (D) {
            case 64: return bf16 ? launch<64, true, 4, true>(N, g, stream, sign_xor) : launch<64, false, 4, true>(N, g, stream, sign_xor);
            case 96: return bf16 ? launch<96, true, 4, true>(N, g, stream, sign_xor) : launch<96, false, 4, true>(N, g, stream, sign_xor);
            case 128: return bf16 ? launch<128, true, 4, true>(N, g, stream, sign_xor) : launch<128, false, 4, true>(N, g, stream, sign_xor);
            case 160: return bf16 ? launch<160, true, 4, true>(N, g, stream, sign_xor) : launch<160, false, 4, true>(N, g, stream, sign_xor);
        }
        return cudaErrorInvalidValue;
    }
    if (bits == 8) {
        switch (D) {
            case 64: return bf16 ? launch<64, true, 8>(N, g, stream) : launch<64, false, 8>(N, g, stream);
            case 96: return bf16 ? launch<96, true, 8>(N, g, stream) : launch<96, false, 8>(N, g, stream);
            case 128: return bf16 ? launch<128, true, 8>(N, g, stream) : launch<128, false, 8>(N, g, stream);
            case 160: return bf16 ? cudaErrorInvalidValue : launch<160, false, 8>(N, g, stream);
        }
        return cudaErrorInvalidValue;
    }
    switch (D) {
        case 64: return bf16 ? launch<64, true>(N, g, stream) : launch<64, false>(N, g, stream);
        case 96: return bf16 ? launch<96, true>(N, g, stream) : launch<96, false>(N, g, stream);
        case 128: return bf16 ? launch<128, true>(N, g, stream) : launch<128, false>(N, g, stream);
        case 160: return bf16 ? launch<160, true>(N, g, stream) : launch<160, false>(N, g, stream);
    }
    return cudaErrorInvalidValue;
}

}  // namespace kvq

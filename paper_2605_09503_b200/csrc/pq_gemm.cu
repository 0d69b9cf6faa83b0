// W4A4 NVFP4 block-scaled GEMM (right-hand side of Eq. 8) on the sm_100a tensor cores.
//
//   Y[m,n] = bf16( ts_x*ts_w * sum_k (qx[m,k]*sfx[m,k/16]) * (qw[n,k]*sfw[n,k/16]) )
//
// Design.  Thread-block clusters of two CTAs (one per SM) work as a pair on output tiles of
// 256 x 256, persistent over the tile list: tcgen05.mma.cta_group::2 lets each CTA hold 128 rows
// of the accumulator while the B operand is split between the two shared memories, so a CTA
// fetches 128 rows of X codes and 128 rows of W codes per 256-channel K step (38 KB with the
// scales, for 512 cycles of MMA).  Roles of the 10 warps of a CTA:
//   warp 0       producer: TMA loads of the packed E2M1 operand tiles (128-byte swizzle) and of the
//                scale-factor blocks into a 5-stage shared-memory ring.  The loads of both CTAs signal
//                the pair leader's barrier (cp.async.bulk.tensor with .cta_group::2).
//   warp 1       (leader CTA) copies the stage's scale blocks of both CTAs to tensor memory (tcgen05.cp) and
//                issues tcgen05.mma.kind::mxf4nvf4.block_scale, K = 64 per instruction, 4 per stage, into the
//                256-column fp32 accumulator in tensor memory.
//   warps 2..9   epilogue (lane quadrant x column half): tcgen05.ld the finished accumulator (own
//                CTA's 128 rows) 16 columns at a time, scale by ts_x*ts_w, round to bf16 and keep the
//                32 x 128 piece as 64 packed registers; hand the accumulator back; then stage 32 x 64
//                boxes in swizzled shared memory and write them with TMA stores (full 128-byte
//                lines), spread over the next tile's main loop.
// 256 divides every FLUX output width (3072, 9216, 12288).  The 512 tensor-memory columns hold one
// 256-column accumulator plus a scale slot of 48 columns per stage.
//
// What bounds it.  The main loop runs at 523 cycles per stage of 512 MMA cycles: waiting for the stage, issuing
// (about 340 cycles, a tcgen05.cp about 6 and an MMA about 50 of them) and the loop around it take that long, and a
// stage's loads land 700 to 1000 cycles after they were asked for with 2500 to spare.  A tile boundary costs about
// 1000 cycles (the last stage's MMAs, the read-out, the signals).  At that rate the chip is at its power limit:
// 1.55 GHz of 1.965.
//
// Measurements on B200 behind these choices (4608 x 3072 x 9216 / 4608 x 12288 x 3072 / 18432 x 3072 x 12288, us):
//   - scales by tcgen05.cp from the issuing warp 52.8 / 59.6 / 275; by eight more warps through registers (ld.shared +
//     tcgen05.st, three slots, 96 registers a thread) 55.9 / 62.7 / 289;
//   - stores spread over the next main loop (kPaceCycles, 30 to 32) 50.7 / 59.0 / 255.  All SMs finish their tiles together, and
//     while 16 stores of each went out at once the loads behind them took 2000 to 3500 cycles to land: the ring ran dry
//     for three or four stages of every tile.  24 cycles per box and stage 51.2 / 59.0 / 264, 14: 53.3 / 59.0 / 276,
//     40: 52.6 / 61.1 / 268 (the last store is then later than the next tile);
//   - two accumulators that overlap by 144 columns, so that a tile starts when those have been read: 51.4 / 59.0 / 265
//     against 51.2 / 59.0 / 264, not worth the fewer scale slots; four stages 53.3 / 62.5 / 271;
//   - tiles walked in groups of 6 to 16 rows of tiles: no better (50.9 to 51.1 / 59.1 to 59.4 / 257);
//   - TMA and tcgen05 instructions take their operands from uniform registers.  The issuing warps run their loops with
//     the whole warp, with the warp index from a shuffle so that the branch is known to be uniform, and single out one
//     lane with elect.sync around those instructions.  Predicated instructions instead of that branch: 56.1 / 67.6 / 283;
//   - all copies of a stage in front of its MMAs: 512 x 3072 x 3072 6.6, copies and MMAs in turn 6.9;
//   - a remote mbarrier arrive with cluster-scope release semantics costs 500 to 2500 cycles.  The only remote arrives here hand
//     the accumulator back, whose reads have completed (tcgen05.wait::ld) when they are issued, so they have the default semantics;
//   - the narrow tile's scales by plain bulk copies, which report to their own CTA, so that the other CTA has to pass them on to the
//     leader: by an arrive with default semantics 1 % slower (512 x 3072 x 3072 6.61 us, 6.57 by the pair's tensor loads) and of CTA
//     scope only; by release and acquire of the cluster, which is what it takes, 9.96.
//
// Scale factors live in global memory in 512-byte blocks of 128 rows x 4 groups (see pq.h); a
// block occupies 4 tensor-memory columns (row r of the block -> lane r%32, column r/32, the same
// in all four lane quadrants), which is the layout the MMA reads and what tcgen05.cp.32x128b.warpx4 makes of it.
// The 256 B-scale rows of a tile are two whole blocks: 8 columns per K block.
//
// Completion of a stage's MMAs and of a tile's accumulator is one tcgen05.commit by the pair leader's MMA warp, onto
// both CTAs' copies of the barrier; the epilogue warps hand the accumulator back by plain remote arrives.
// Every wait on an mbarrier is bounded.  If one
// expires the CTA records PQ_ERR_TIMEOUT in the status word, raises a shared abort flag that every role polls,
// and falls through to the common teardown (cluster barrier, tensor-memory release).
#include <cuda.h>

#include <mutex>

#include "pq_common.cuh"

namespace {

constexpr int BM = 256, BM_CTA = 128, BK = 256;
constexpr int kABytes = BM_CTA * BK / 2;   // 16384
constexpr int kSfBlock = 512;              // 128 rows x 4 groups
constexpr int kSfaBytes = 4 * kSfBlock;    // 4 K-blocks of one 128-row block
constexpr int kTmemCols = 512;
constexpr long long kWaitCycles = 4000000000ll;  // default limit of a wait: about two seconds of SM clock

constexpr int kEpiWarps = 8;               // lane quadrant x column half of the accumulator
constexpr int kBoxCols = 64;               // output staging box: 32 rows x 64 bf16, one TMA store
constexpr int kEpiBox = 32 * kBoxCols * 2;
constexpr int kEpiBytes = kEpiWarps * kEpiBox;      // one staging box per epilogue warp: 32 KB
// SM clock cycles per K step between the stores of a tile's 2 * kEpiWarps boxes: the last one starts at 15 / 17 of the
// next tile's main loop.
constexpr int kPaceCycles = 30;
constexpr int kThreads = 32 * (2 + kEpiWarps);      // producer, MMA issuer, 8 epilogue warps
// One 256-column accumulator, then the scale slots, one per stage: per 64-channel K block 4 columns of A scales (128
// rows) and 8 columns of B scales (256 rows).  A slot is written after the wait for its stage's data, which the producer
// asked for only when the MMAs that read the stage (and the slot) before had completed.
//
// Every wait here is a PARITY wait: it tells "phase n of this barrier has completed" from "it has not" only if the
// barrier cannot still be in phase n - 1, i.e. only if the waiter already knows that phase n - 1 has completed.  Every role
// waits on every phase of its barriers in turn (producer on stage_free, MMA issuer on stage_full and acc_empty, each
// epilogue warp on acc_full), so it knows it from its own previous wait.
//
// Two tile widths.  The wide tile (256 columns) needs the fewest operand bytes per flop and is what every
// product of more than one round of tiles runs on.  The narrow tile (128 columns) is for products that have at
// most one such tile per CTA pair: twice as many pairs work on them, half the MMA time per K step, and since a
// pair never has a next tile, the epilogue stages its boxes in the operand ring, which leaves room for eight stages.
template <int BN>
struct Tile {
    static constexpr int kNCta = BN / 2;
    static constexpr bool kOneTile = BN == 128;             // a pair computes one tile; the epilogue stages in the ring
    static constexpr int kStages = BN == 256 ? 5 : 8;
    static constexpr int kNB = BN / 128;                  // 128-row scale blocks of B per tile
    static constexpr int kBBytes = kNCta * BK / 2;
    static constexpr int kSfbBytes = kNB * kSfaBytes;     // the 128-row blocks of the tile's B rows
    static constexpr int kStageBytes = kABytes + kBBytes + kSfaBytes + kSfbBytes;  // 38 or 28 * 1024
    static constexpr uint32_t kSfSlotCol0 = BN, kSfbColsPerKb = 4 * kNB, kSfbOfs = 16;
    static constexpr uint32_t kSfSlotCols = 4 * (4 + kSfbColsPerKb);   // 48 or 32
    static constexpr int kNumBars = 2 * kStages + 2;      // stage_full[S] stage_free[S] acc_full acc_empty
    static constexpr int kRingBytes = kStages * kStageBytes, kEpi = kOneTile ? 0 : kRingBytes;  // where the boxes start
    static constexpr size_t kSmemBytes = kRingBytes + (kOneTile ? 0 : kEpiBytes) + 1024 /*alignment slack*/ + 8 * kNumBars + 64;
    // Instruction descriptor: E2M1 x E2M1, UE4M3 scales, both K-major, M = 256 (pair), N = BN, K = 64.
    static constexpr uint32_t kIdesc = (1u << 7) | (1u << 10) | (static_cast<uint32_t>(BN >> 3) << 17) | (0u << 23) |
                                       (static_cast<uint32_t>(BM >> 4) << 24);
    static_assert(kStageBytes % 1024 == 0, "swizzled operand tiles start on 1024-byte boundaries");
    static_assert(kSfSlotCol0 + kStages * kSfSlotCols <= 512, "tensor memory columns");
    static_assert(kSmemBytes <= 227 * 1024, "shared memory per CTA");
};

struct Maps {
    CUtensorMap a, b, y, sfa, sfb;
};

struct GemmParams {
    const float *ts_x, *ts_w;
    int M, N;
    int m_tiles, n_tiles, k_tiles, kb_total;
    long long wait_cycles;  // limit of every mbarrier wait, in SM clock cycles
    int *status;
};

// ---------------------------------------------------------------- PTX wrappers
__device__ __forceinline__ uint32_t smem_u32(const void *p) {
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}
__device__ __forceinline__ uint32_t cluster_ctarank() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
// Address of the same shared-memory location in CTA `rank` of the cluster.
__device__ __forceinline__ uint32_t mapa(uint32_t addr, uint32_t rank) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
    return r;
}
// One lane of a converged warp; the branch on it stays friendly to uniform registers.
__device__ __forceinline__ bool elect_one() {
    uint32_t pred = 0;
    asm volatile(
        "{\n"
        ".reg .b32 rx;\n"
        ".reg .pred px;\n"
        "elect.sync rx|px, %1;\n"
        "@px mov.s32 %0, 1;\n"
        "}\n"
        : "+r"(pred)
        : "r"(0xFFFFFFFFu));
    return pred != 0;
}
__device__ __forceinline__ void cluster_sync() {
    asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count));
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
// Arrive on the copy of a barrier in CTA `rank` of the pair.
__device__ __forceinline__ void mbar_arrive_remote(uint32_t bar, uint32_t rank) {
    asm volatile(
        "{\n"
        ".reg .b32 remote;\n"
        "mapa.shared::cluster.u32 remote, %0, %1;\n"
        "mbarrier.arrive.shared::cluster.b64 _, [remote];\n"
        "}\n" ::"r"(bar), "r"(rank)
        : "memory");
}
// Arrive on the pair leader's copy of a barrier.
__device__ __forceinline__ void mbar_arrive_leader(uint32_t bar, uint32_t rank) {
    if (rank == 0) mbar_arrive(bar);
    else mbar_arrive_remote(bar, 0);
}
__device__ __forceinline__ bool mbar_try(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n"
        ".reg .pred p;\n"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
        "selp.u32 %0, 1, 0, p;\n"
        "}\n"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}
// Bounded wait: polls until the phase completes, the abort flag goes up, or `limit` SM clock cycles
// have passed (then it raises the flag and records the timeout).
struct WaitCtx {
    volatile int *abort_flag;
    int *status;
    long long limit;
};
__device__ __noinline__ bool mbar_wait_slow(uint32_t bar, uint32_t parity, const WaitCtx w) {
    const long long t0 = clock64();
    for (uint32_t spins = 1;; ++spins) {
        if (mbar_try(bar, parity)) return true;
        if ((spins & 63u) == 0) {
            if (*w.abort_flag) return false;
            if (clock64() - t0 > w.limit) break;
        }
    }
    *w.abort_flag = 1;
    atomicExch(w.status, static_cast<int>(PQ_ERR_TIMEOUT));
    return false;
}
// Wait of a single thread (or of lanes that vote on the result themselves).
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, const WaitCtx w) {
    if (mbar_try(bar, parity)) return true;
    return mbar_wait_slow(bar, parity, w);
}
// Wait of a converged warp: every lane returns the same answer and the warp is converged again
// afterwards, so .sync.aligned instructions (elect, tcgen05.ld) may follow on either outcome.
__device__ __forceinline__ bool mbar_wait_warp(uint32_t bar, uint32_t parity, const WaitCtx w) {
    bool ok = mbar_try(bar, parity);
    if (__all_sync(0xFFFFFFFFu, ok)) return true;
    ok = ok || mbar_wait_slow(bar, parity, w);
    return __all_sync(0xFFFFFFFFu, ok);
}
__device__ __forceinline__ void prefetch_tensormap(const CUtensorMap *map) {
    asm volatile("prefetch.tensormap [%0];" ::"l"(map) : "memory");
}
// Operand tile load of a CTA pair: data lands in this CTA's shared memory, the byte count is
// credited to the barrier at `bar_cluster` (the pair leader's).
__device__ __forceinline__ void tma_load_2d_pair(uint32_t dst, const CUtensorMap *map, int x, int y,
                                                 uint32_t bar_cluster) {
    asm volatile(
        "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
        ::"r"(dst), "l"(map), "r"(x), "r"(y), "r"(bar_cluster)
        : "memory");
}
__device__ __forceinline__ void tma_store_2d(const CUtensorMap *map, int x, int y, uint32_t src) {
    asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.bulk_group [%0, {%1, %2}], [%3];"
                 ::"l"(map), "r"(x), "r"(y), "r"(src)
                 : "memory");
}
__device__ __forceinline__ void bulk_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void bulk_wait_read() {
    asm volatile("cp.async.bulk.wait_group.read %0;" ::"n"(N) : "memory");
}
__device__ __forceinline__ void bulk_wait_all() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }
__device__ __forceinline__ void fence_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
// Arrive on both CTAs' copies of `bar` once every tcgen05 operation issued so far by this thread has completed in the pair.
__device__ __forceinline__ void tc_commit_both(uint32_t bar) {
    asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;"
                 ::"r"(bar), "h"(static_cast<uint16_t>(3))
                 : "memory");
}
// Copies a 512-byte scale block of either CTA to four columns of its tensor memory, replicated over the lane quadrants.
__device__ __forceinline__ void tc_cp_scales(uint32_t tmem_col, uint64_t desc) {
    asm volatile("tcgen05.cp.cta_group::2.32x128b.warpx4 [%0], %1;" ::"r"(tmem_col), "l"(desc) : "memory");
}
__device__ __forceinline__ void tc_mma_pair(uint32_t d_tmem, uint64_t da, uint64_t db, uint32_t idesc, uint32_t sfa,
                                            uint32_t sfb, uint32_t accumulate) {
    asm volatile(
        "{\n"
        ".reg .pred p;\n"
        "setp.ne.b32 p, %4, 0;\n"
        "tcgen05.mma.cta_group::2.kind::mxf4nvf4.block_scale.block16 [%0], %1, %2, %3, [%5], [%6], p;\n"
        "}\n"
        ::"r"(d_tmem), "l"(da), "l"(db), "r"(idesc), "r"(accumulate), "r"(sfa), "r"(sfb)
        : "memory");
}
__device__ __forceinline__ void tc_ld16(uint32_t taddr, uint32_t (&v)[16]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];\n"
        : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
          "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
        : "r"(taddr)
        : "memory");
}
// The registers of a tcgen05.ld hold its result only after tcgen05.wait::ld.  The wait names them as
// in/out operands: whatever reads them afterwards then depends on the wait and cannot be scheduled in
// front of it (arithmetic on the loaded values has no other tie to the wait instruction; without it a
// tile was occasionally packed from registers the load had not written yet).
__device__ __forceinline__ void tc_wait_ld(uint32_t (&v)[16]) {
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+r"(v[0]), "+r"(v[1]), "+r"(v[2]), "+r"(v[3]), "+r"(v[4]), "+r"(v[5]), "+r"(v[6]), "+r"(v[7]),
                   "+r"(v[8]), "+r"(v[9]), "+r"(v[10]), "+r"(v[11]), "+r"(v[12]), "+r"(v[13]), "+r"(v[14]), "+r"(v[15])
                 :
                 : "memory");
}
__device__ __forceinline__ void sts128(uint32_t addr, uint32_t a, uint32_t b, uint32_t c, uint32_t d) {
    asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(a), "r"(b), "r"(c), "r"(d) : "memory");
}

// Shared-memory matrix descriptor of a K-major operand tile with 128-byte swizzle: rows of
// 128 bytes, 8-row groups 1024 bytes apart.
__device__ __forceinline__ uint64_t operand_desc(uint32_t smem_addr) {
    return static_cast<uint64_t>((smem_addr & 0x3FFFFu) >> 4) | (1ull << 16) | (64ull << 32) | (1ull << 46) |
           (2ull << 61);
}
// ... of scale blocks: no swizzle, 16-byte rows, 8-row groups 128 bytes apart.
__device__ __forceinline__ uint64_t scale_desc(uint32_t smem_addr) {
    return static_cast<uint64_t>((smem_addr & 0x3FFFFu) >> 4) | (1ull << 16) | (8ull << 32) | (1ull << 46);
}
// Two accumulator values times alpha, each rounded to bf16 (nearest even), packed low | high.
__device__ __forceinline__ uint32_t pack_bf16(uint32_t lo_bits, uint32_t hi_bits, float alpha) {
    uint32_t r;
    // one packed multiply (two IEEE products per issue slot), then the two-way convert
    asm("{\n"
        ".reg .b64 v, a;\n"
        ".reg .f32 lo, hi;\n"
        "mov.b64 v, {%1, %2};\n"
        "mov.b64 a, {%3, %3};\n"
        "mul.rn.f32x2 v, v, a;\n"
        "mov.b64 {lo, hi}, v;\n"
        "cvt.rn.bf16x2.f32 %0, hi, lo;\n"
        "}\n"
        : "=r"(r)
        : "r"(lo_bits), "r"(hi_bits), "f"(alpha));
    return r;
}

// ---------------------------------------------------------------- kernel
// Register budget: the register file is split over the four SM sub-partitions (16384 registers each) and two of them
// receive three of this CTA's ten warps: 3 x 32 x 128 = 12288.  The rest takes blocks of a 32-register kernel beside the GEMM.
constexpr int kMaxRegs = 128;
template <int BN>
__global__ void __cluster_dims__(2, 1, 1) __maxnreg__(kMaxRegs)
gemm_w4a4_kernel(const __grid_constant__ Maps maps, const GemmParams p) {
    using T = Tile<BN>;
    constexpr int kStages = T::kStages, kNB = T::kNB, BN_CTA = T::kNCta;
    constexpr int kBBytes = T::kBBytes, kStageBytes = T::kStageBytes, kNumBars = T::kNumBars;
    constexpr uint32_t kSfbOfs = T::kSfbOfs, kSfbColsPerKb = T::kSfbColsPerKb;
    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw = smem_u32(smem_raw);
    const uint32_t base = (raw + 1023u) & ~1023u;  // identical in both CTAs of the pair
    uint8_t *base_ptr = smem_raw + (base - raw);
    constexpr int kBarOfs = T::kRingBytes + (T::kOneTile ? 0 : kEpiBytes);
    const uint32_t epi = base + T::kEpi;
    const uint32_t bars = base + kBarOfs;
    uint8_t *bars_ptr = base_ptr + kBarOfs;
    // stage_full: operand and scale bytes of both CTAs have landed (1 arrival + transaction bytes); leader's copy only
    auto stage_full_bar = [&](int s) { return bars + 8u * s; };
    auto stage_free_bar = [&](int s) { return bars + 8u * (kStages + s); };  // the stage's MMAs have run
    const uint32_t acc_full_bar = bars + 8u * (2 * kStages);       // one copy per CTA, both signalled by the issuer
    const uint32_t acc_empty_bar = bars + 8u * (2 * kStages + 1);  // leader's copy only
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(bars_ptr + 8 * kNumBars);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(bars_ptr + 8 * kNumBars + 8);
    const WaitCtx wctx{abort_flag, p.status, p.wait_cycles};
    auto sf_slot_col = [](uint32_t t) { return T::kSfSlotCol0 + t * T::kSfSlotCols; };

    const int warp = __shfl_sync(0xFFFFFFFFu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
    const uint32_t rank = __shfl_sync(0xFFFFFFFFu, cluster_ctarank(), 0);  // 0 = pair leader
    const int pair = blockIdx.x >> 1, num_pairs = gridDim.x >> 1;

    if (threadIdx.x == 0) {
        for (int s = 0; s < kStages; ++s) {
            mbar_init(stage_full_bar(s), 1);
            mbar_init(stage_free_bar(s), 1);
        }
        mbar_init(acc_full_bar, 1);
        mbar_init(acc_empty_bar, 2 * kEpiWarps);  // the epilogue warps of both CTAs
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        prefetch_tensormap(&maps.a);
        prefetch_tensormap(&maps.b);
        prefetch_tensormap(&maps.sfa);
        prefetch_tensormap(&maps.sfb);
        prefetch_tensormap(&maps.y);
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                     "r"(kTmemCols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    cluster_sync();  // both CTAs' barriers are initialised before anyone signals across
    tc_fence_after();
    const uint32_t tmem_base = __shfl_sync(0xFFFFFFFFu, *tmem_slot, 0);
    // When launched as a programmatic dependent of the activation quantizer, everything above ran
    // while that kernel was finishing; its output (and any earlier work in the stream) is complete
    // and visible from here on.  A no-op for an ordinary launch.
    asm volatile("griddepcontrol.wait;" ::: "memory");
    // ... and a kernel launched as this one's programmatic dependent may start its own set-up as
    // soon as this kernel's CTAs leave their SMs.
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

    const int total_tiles = p.m_tiles * p.n_tiles;

    if (warp == 0) {
        // ------------------------------------------------------------ producer
        uint32_t it = 0;
        bool ok = true;
        for (int tile = pair; tile < total_tiles && ok; tile += num_pairs) {
            const int m_blk = tile % p.m_tiles, n_blk = tile / p.m_tiles;
            const int m0 = m_blk * BM + static_cast<int>(rank) * BM_CTA;
            const int n0 = n_blk * BN;
            for (int kt = 0; kt < p.k_tiles; ++kt, ++it) {
                const int s = it % kStages;
                const uint32_t par = (it / kStages) & 1u;
                ok = mbar_wait_warp(stage_free_bar(s), par ^ 1u, wctx);
                if (!ok) break;
                const uint32_t stage = base + s * kStageBytes;
                const uint32_t sf_stage = stage + kABytes + kBBytes;
                const uint32_t full_leader = mapa(stage_full_bar(s), 0);
                if (elect_one()) {
                    if (rank == 0) mbar_expect_tx(stage_full_bar(s), 2u * kStageBytes);
                    tma_load_2d_pair(sf_stage, &maps.sfa, kt * (4 * kSfBlock / 8), m0 >> 7, full_leader);
                    tma_load_2d_pair(sf_stage + kSfaBytes, &maps.sfb, kt * (4 * kSfBlock / 8), n0 >> 7, full_leader);
                    tma_load_2d_pair(stage, &maps.a, kt * (BK / 2), m0, full_leader);
                    tma_load_2d_pair(stage + kABytes, &maps.b, kt * (BK / 2), n0 + static_cast<int>(rank) * BN_CTA, full_leader);
                }
                __syncwarp();
            }
        }
        if (!ok && lane == 0 && rank == 0) {
            // give the copies already issued (they count on these barriers) a bounded chance to land before leaving
            const uint32_t first = it > kStages ? it - kStages : 0;
            for (uint32_t j = first; j < it; ++j)
                for (uint32_t i = 0; i < 4096 && !mbar_try(stage_full_bar(j % kStages), (j / kStages) & 1u); ++i) {}
        }
        __syncwarp();
    } else if (warp == 1) {
        // ------------------------------------------------------------ MMA issuer (pair leader)
        if (rank == 0) {
            // Ring positions are kept incrementally: stage (and scale slot) s with phase ph.
            uint32_t s = 0, ph = 0, tcount = 0;
            bool ok = true;
            for (int tile = pair; tile < total_tiles && ok; tile += num_pairs, ++tcount) {
                // the accumulator is free once the epilogue has read the previous tile out of it
                ok = mbar_wait_warp(acc_empty_bar, (tcount & 1u) ^ 1u, wctx);
                if (!ok) break;
                tc_fence_after();
                const uint32_t d_tmem = tmem_base;
                uint32_t acc = 0;
                for (int kt = 0; kt < p.k_tiles; ++kt) {
                    ok = mbar_wait_warp(stage_full_bar(s), ph, wctx);
                    if (!ok) break;
                    tc_fence_after();
                    const uint32_t stage = base + s * kStageBytes;
                    const uint64_t da = operand_desc(stage), db = operand_desc(stage + kABytes);
                    const uint64_t ds = scale_desc(stage + kABytes + kBBytes);
                    const uint32_t sfa_t = tmem_base + sf_slot_col(s), sfb_t = sfa_t + kSfbOfs;
                    const int kb_valid = min(4, p.kb_total - kt * 4);
                    if (elect_one()) {
                        // (what lies behind the last channel, zeros or an older stage, belongs to no MMA)
#pragma unroll
                        for (int kk = 0; kk < 4; ++kk) {
                            tc_cp_scales(sfa_t + 4 * kk, ds + kk * (kSfBlock / 16));
#pragma unroll
                            for (int j = 0; j < kNB; ++j)
                                tc_cp_scales(sfb_t + kSfbColsPerKb * kk + 4 * j, ds + ((1 + j) * kSfaBytes + kk * kSfBlock) / 16);
                        }
#pragma unroll
                        for (int kk = 0; kk < 4; ++kk) {
                            if (kk < kb_valid) {
                                const uint32_t accumulate = acc | static_cast<uint32_t>(kk);
                                tc_mma_pair(d_tmem, da + 2 * kk, db + 2 * kk, T::kIdesc, sfa_t + 4 * kk,
                                            sfb_t + kSfbColsPerKb * kk, accumulate);
                            }
                        }
                        // the stage (and its scale slot) is free in both CTAs once these MMAs have run
                        tc_commit_both(stage_free_bar(s));
                        if (kt == p.k_tiles - 1) tc_commit_both(acc_full_bar);  // ... and the tile's accumulator is complete
                    }
                    __syncwarp();
                    acc = 1u;
                    s = (s + 1 == kStages) ? 0u : s + 1;
                    ph ^= (s == 0) ? 1u : 0u;
                }
            }
        }
    } else {
        // ------------------------------------------------------------ epilogue
        // Eight warps: lane quadrant q x column half h.  A warp reads its 32 rows x BN / 2 columns out of
        // tensor memory, scales and rounds them to bf16 and keeps them packed in BN / 4 registers; the
        // accumulator goes back to the MMA issuer after those loads (a few hundred cycles), and the
        // 64-column boxes leave through one staging box and TMA stores, the warps and boxes one after the other over
        // the next tile's main loop (at once if there is none).
        constexpr int kCols = BN / 2, kBoxes = kCols / kBoxCols, kChunks = kBoxCols / 8;  // boxes per warp, 16-byte chunks per box row
        const int q = warp & 3;                // tensor-memory lane quadrant this warp may read
        const int h = (warp - 2) >> 2;         // column half
        const float alpha = __fmul_rn(__ldca(p.ts_x), __ldca(p.ts_w));
        const uint32_t buf = epi + static_cast<uint32_t>(warp - 2) * kEpiBox;
        // 128-byte swizzle of the staging box (what the store's tensor map expects): chunk ^ (row & 7)
        const uint32_t row_ofs = static_cast<uint32_t>(lane) * (kBoxCols * 2), sw = static_cast<uint32_t>(lane & 7);
        uint32_t tcount = 0;
        for (int tile = pair; tile < total_tiles; tile += num_pairs, ++tcount) {
            const int m_blk = tile % p.m_tiles, n_blk = tile / p.m_tiles;
            const int m0 = m_blk * BM + static_cast<int>(rank) * BM_CTA + q * 32, n0 = n_blk * BN + h * kCols;
            const bool got = mbar_wait(acc_full_bar, tcount & 1u, wctx);
            if (!__all_sync(0xFFFFFFFFu, got)) break;
            tc_fence_after();
            const bool more = tile + num_pairs < total_tiles;
            const long long t0 = clock64();
            const uint32_t acc = tmem_base + (static_cast<uint32_t>(q * 32) << 16) + h * kCols;
            uint32_t pk[kCols / 2];  // pk[8 c + i] = columns 16 c + 2 i, 16 c + 2 i + 1 of this lane's row
            // two loads in flight: chunk c + 1 is on its way while chunk c is scaled and packed
            uint32_t va[16], vb[16];
            tc_ld16(acc, va);
#pragma unroll
            for (int c = 0; c < kCols / 16; c += 2) {
                tc_wait_ld(va);
                tc_ld16(acc + (c + 1) * 16, vb);
#pragma unroll
                for (int i = 0; i < 8; ++i) pk[8 * c + i] = pack_bf16(va[2 * i], va[2 * i + 1], alpha);
                tc_wait_ld(vb);
                if (c + 2 < kCols / 16) tc_ld16(acc + (c + 2) * 16, va);
#pragma unroll
                for (int i = 0; i < 8; ++i) pk[8 * (c + 1) + i] = pack_bf16(vb[2 * i], vb[2 * i + 1], alpha);
            }
            // this warp's part of the accumulator has been read: hand it back to the MMA issuer
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive_leader(acc_empty_bar, rank);
#pragma unroll
            for (int c = 0; c < kBoxes; ++c) {
                if (more) {
                    const long long until = t0 + static_cast<long long>(c * kEpiWarps + warp - 2) * p.k_tiles * kPaceCycles;
                    while (clock64() < until) __nanosleep(64);
                }
                // the store that read the box before (previous box or previous tile) must be done with it
                if (lane == 0) bulk_wait_read<0>();
                __syncwarp();
#pragma unroll
                for (int i = 0; i < kChunks; ++i)
                    sts128(buf + row_ofs + ((static_cast<uint32_t>(i) ^ sw) << 4), pk[4 * kChunks * c + 4 * i],
                           pk[4 * kChunks * c + 4 * i + 1], pk[4 * kChunks * c + 4 * i + 2], pk[4 * kChunks * c + 4 * i + 3]);
                fence_async_smem();
                __syncwarp();
                if (lane == 0) {
                    if (m0 < p.M && n0 + c * kBoxCols < p.N) tma_store_2d(&maps.y, n0 + c * kBoxCols, m0, buf);
                    bulk_commit();
                }
            }
        }
        if (lane == 0) bulk_wait_all();  // shared memory must outlive the stores that read it
        __syncwarp();
    }

    // ---------------------------------------------------------------- teardown
    tc_fence_before();
    __syncthreads();
    cluster_sync();  // the peer may still signal this CTA's barriers or read its operands until here
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(kTmemCols) : "memory");
    }
}

// One warp waits, with the kernel's own bounded wait, on a barrier that nobody arrives at: the way
// the expiry path (status word, abort flag, orderly return) is exercised without a fault or a hang.
__global__ void __launch_bounds__(32) wait_expiry_kernel(int *status, long long limit, int *observed) {
    __shared__ __align__(8) unsigned long long bar;
    __shared__ int abort_word;
    if (threadIdx.x == 0) {
        mbar_init(smem_u32(&bar), 1);
        abort_word = 0;
    }
    __syncwarp();
    const WaitCtx w{&abort_word, status, limit};
    const bool ok = mbar_wait_warp(smem_u32(&bar), 0u, w);
    // every lane has the same answer and the warp is converged: what the roles of the GEMM rely on
    if (threadIdx.x == 0) {
        observed[0] = ok ? 1 : 0;
        observed[1] = abort_word;
    }
}

// ---------------------------------------------------------------- host side
typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                  const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_tiled() {
    static EncodeTiledFn fn = nullptr;
    if (!fn) {
        void *sym = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &sym, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<EncodeTiledFn>(sym);
    }
    return fn;
}

// A row-major 2-D tensor [rows, row_bytes / elem] cut into 128-byte-swizzled boxes of 128 bytes x
// box_rows rows; with elem = 8 (scale blocks, a row of blocks per row of the map) plain boxes of 2 KB x box_rows.  Loads read
// out-of-range rows / columns as zero, stores skip them.
bool encode_map(CUtensorMap *map, const void *ptr, int64_t rows, int64_t row_bytes, int64_t pitch, int box_rows, int elem) {
    EncodeTiledFn enc = encode_tiled();
    if (!enc) return false;
    const cuuint64_t dims[2] = {static_cast<cuuint64_t>(row_bytes / elem), static_cast<cuuint64_t>(rows)};
    const cuuint64_t strides[1] = {static_cast<cuuint64_t>(pitch)};
    const cuuint32_t box[2] = {static_cast<cuuint32_t>(elem == 8 ? 256 : 128 / elem), static_cast<cuuint32_t>(box_rows)};
    const cuuint32_t estr[2] = {1, 1};
    const CUtensorMapDataType dt = elem == 1   ? CU_TENSOR_MAP_DATA_TYPE_UINT8
                                   : elem == 2 ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16
                                               : CU_TENSOR_MAP_DATA_TYPE_UINT64;
    return enc(map, dt, 2, const_cast<void *>(ptr), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
               elem == 8 ? CU_TENSOR_MAP_SWIZZLE_NONE : CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// What the maps of an operand (ld = 0: codes and scale blocks; rows x K) or of the output (rows x K, ld) depend on.
struct MapKey {
    const void *ptr, *sf;
    int64_t rows, K, ld;
    int box_rows, sf_box_rows;
    bool operator==(const MapKey &o) const {
        return ptr == o.ptr && sf == o.sf && rows == o.rows && K == o.K && ld == o.ld && box_rows == o.box_rows && sf_box_rows == o.sf_box_rows;
    }
};
struct MapSlot {
    MapKey key;
    CUtensorMap map, scales;
    bool used;
};
// Encoding a tensor map costs several microseconds of host time; a layer calls the GEMM with the same buffers over and over, so
// a thread keeps the encodings of the last layers: three entries a call, each in one of four neighbouring slots found by a
// hash of its key.
const MapSlot *find_maps(const MapKey &key) {
    constexpr uint32_t kSlots = 64, kProbes = 4;
    static thread_local MapSlot cache[kSlots];
    static thread_local uint32_t next = 0;
    const uint64_t mix = (reinterpret_cast<uintptr_t>(key.ptr) >> 4) ^ (static_cast<uint64_t>(key.rows) << 20) ^
                         (static_cast<uint64_t>(key.K) << 40) ^ static_cast<uint64_t>(key.box_rows);
    const uint32_t home = static_cast<uint32_t>((mix * 0x9E3779B97F4A7C15ull) >> 58);
    uint32_t at = home + next % kProbes;  // an empty slot, or one of the four in turn
    for (uint32_t i = 0; i < kProbes; ++i) {
        const MapSlot &c = cache[(home + i) % kSlots];
        if (c.used && c.key == key) return &c;
        if (!c.used) {
            at = home + i;
            break;
        }
    }
    ++next;
    MapSlot &slot = cache[at % kSlots];
    slot.used = false;
    slot.key = key;
    if (key.ld) {
        slot.used = encode_map(&slot.map, key.ptr, key.rows, key.K * 2, key.ld * 2, key.box_rows, 2);
    } else {
        const int64_t sf_pitch = key.K / 64 * kSfBlock;
        slot.used = encode_map(&slot.map, key.ptr, key.rows, key.K / 2, key.K / 2, key.box_rows, 1) &&
                    encode_map(&slot.scales, key.sf, pq_ceil_div(key.rows, 128), sf_pitch, sf_pitch, key.sf_box_rows, 8);
    }
    return slot.used ? &slot : nullptr;
}

// Number of CTA pairs that can be resident at once on the current device (a cluster must fit inside
// one GPC), after opting the kernel in to its dynamic shared memory there.  Both are per device.
template <int BN>
int resident_pairs(int dev) {
    constexpr size_t kSmemBytes = Tile<BN>::kSmemBytes;
    static PqPerDevice cache;
    if (dev < 0) return 0;
    if (const int known = cache.value[dev]) return known;
    std::lock_guard<std::mutex> guard(cache.lock);
    if (const int known = cache.value[dev]) return known;
    if (cudaFuncSetAttribute(gemm_w4a4_kernel<BN>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             static_cast<int>(kSmemBytes)) != cudaSuccess) {
        (void)cudaGetLastError();
        return 0;
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(2, 1, 1);
    cfg.blockDim = dim3(kThreads, 1, 1);
    cfg.dynamicSmemBytes = kSmemBytes;
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = 2;
    attr.val.clusterDim.y = 1;
    attr.val.clusterDim.z = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, gemm_w4a4_kernel<BN>, &cfg) != cudaSuccess || n <= 0) {
        (void)cudaGetLastError();
        return 0;
    }
    cache.value[dev] = n;
    return n;
}

struct GemmArgs {
    const uint8_t *xq, *sfx, *wq, *sfw;
    const float *ts_x, *ts_w;
    int64_t M, N, K, ldy;
    void *Y, *ws;
    cudaStream_t st;
};

template <int BN>
pq_status launch_tiles(const GemmArgs &g, int pairs_max) {
    Maps maps;
    // copied one by one: a later entry may take an earlier one's slot
    auto find = [&](CUtensorMap &map, CUtensorMap *scales, const MapKey &key) {
        const MapSlot *slot = find_maps(key);
        if (!slot) return false;
        map = slot->map;
        if (scales) *scales = slot->scales;
        return true;
    };
    const bool found = find(maps.y, nullptr, MapKey{g.Y, nullptr, g.M, g.N, g.ldy, 32, 0}) &&
                       find(maps.a, &maps.sfa, MapKey{g.xq, g.sfx, g.M, g.K, 0, BM_CTA, 1}) &&
                       find(maps.b, &maps.sfb, MapKey{g.wq, g.sfw, g.N, g.K, 0, Tile<BN>::kNCta, Tile<BN>::kNB});
    if (!found) return PQ_ERR_CUDA;
    GemmParams p;
    p.ts_x = g.ts_x, p.ts_w = g.ts_w;
    p.M = static_cast<int>(g.M), p.N = static_cast<int>(g.N);
    p.m_tiles = static_cast<int>(pq_ceil_div(g.M, BM));
    p.n_tiles = static_cast<int>(pq_ceil_div(g.N, BN));
    p.k_tiles = static_cast<int>(pq_ceil_div(g.K, BK));
    p.kb_total = static_cast<int>(g.K / 64);
    p.wait_cycles = kWaitCycles;
    p.status = static_cast<int *>(g.ws);
    const int64_t tiles = static_cast<int64_t>(p.m_tiles) * p.n_tiles;
    PQ_REQUIRE(!Tile<BN>::kOneTile || tiles <= pairs_max, PQ_ERR_SHAPE);
    const int pairs = static_cast<int>(tiles < pairs_max ? tiles : pairs_max);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(2 * pairs, 1, 1);
    cfg.blockDim = dim3(kThreads, 1, 1);
    cfg.dynamicSmemBytes = Tile<BN>::kSmemBytes;
    cfg.stream = g.st;
    // Programmatic dependent launch: the kernel may start (barrier set-up, tensor-memory allocation,
    // tensor-map prefetch) while the kernel in front of it in the stream drains (the quantizer, or
    // the previous GEMM of a chain of layers); it waits for that kernel to complete with
    // griddepcontrol.wait before touching global memory, so stream order is what the caller sees.
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    PQ_CUDA_OK(cudaLaunchKernelEx(&cfg, gemm_w4a4_kernel<BN>, maps, p));
    return PQ_OK;
}

// One round of narrow tiles covers the product.  Measured on both sides of the line (M x N x K, narrow against wide, us):
// 128 x 3072 x 3072 6.2 / 7.6, 512 x 3072 x 3072 6.6 / 7.7, 512 x 3072 x 12288 16.1 / 19.3, 512 x 4736 x 3072 7.3 / 8.1; beyond one
// round, in a second wave of CTAs, the narrow tile loses by a third and more (512 x 4744 x 3072 12.0 / 8.2, 512 x 9216 x 3072 14.2 / 9.2,
// 1357 x 4744 x 1088 18.3 / 7.9, 2048 x 3072 x 12288 47.4 / 34.5).
// Few rows: the CTAs of all pairs fetch the same few lines of X at every K step, and with more than half of the pairs at that the
// narrow tile loses up to 16 rows (1 x 5120 x 3072 8.4 / 6.8, 4 x 9216 x 3072 7.7 / 7.1, 2 x 7168 x 12288 22.8 / 21.2, 16 x 9216 x 12288
// 22.2 / 21.4; 24 x 9216 x 12288 16.0 / 19.6).  It does so the later the fewer K steps there are and the more rows, as long as the rows of codes
// start on 128-byte lines: 3 to 16 rows of 256, 512 or 768 channels keep it up to two thirds of the pairs (wide 1.00 to 1.16 x the narrow
// time at 38 to 49 tiles), 8 to 16 rows of 1024 to 2048 for one tile more than half (wide 1.03 to 1.15 x; at 40 tiles 0.95 to 1.1 x).  Other
// row lengths do not (3 x 5120 x 960 5.2 narrow, 4.4 wide).
bool narrow_tiles(int64_t M, int64_t N, int64_t K, int pairs) {
    int most = pairs;
    if (M <= 2 || (M <= 16 && K > 3072)) most = pairs / 2;
    else if (M <= 16) most = K % 256 ? pairs / 2 : K < 1024 ? pairs * 2 / 3 : pairs / 2 + (M >= 8 && K <= 2048 ? 1 : 0);
    return pq_ceil_div(M, BM) * pq_ceil_div(N, 128) <= most;
}

pq_status gemm_launch(const uint8_t *xq, const uint8_t *sfx, const float *ts_x, const uint8_t *wq, const uint8_t *sfw,
                      const float *ts_w, int64_t M, int64_t N, int64_t K, void *Y, int64_t ldy, void *ws,
                      size_t ws_bytes, void *stream) {
    PQ_REQUIRE(xq && sfx && ts_x && wq && sfw && ts_w && Y, PQ_ERR_NULL);
    PQ_REQUIRE(M > 0 && N > 0 && K >= 64 && K % 64 == 0 && N % 8 == 0 && ldy >= N, PQ_ERR_SHAPE);
    PQ_REQUIRE(M < (1ll << 31) - 256 && N < (1ll << 31) - 256 && K < (1ll << 31), PQ_ERR_SHAPE);
    PQ_REQUIRE(pq_aligned16(xq) && pq_aligned16(sfx) && pq_aligned16(wq) && pq_aligned16(sfw) && pq_aligned16(Y) &&
                   ldy % 8 == 0,
               PQ_ERR_ALIGN);
    PQ_REQUIRE(ws && ws_bytes >= pq_workspace_bytes(PQ_OP_GEMM, M, K, N, 0), PQ_ERR_WORKSPACE);
    PQ_REQUIRE(pq_aligned256(ws), PQ_ERR_ALIGN);
    cudaStream_t st = static_cast<cudaStream_t>(stream);

    const int dev = pq_device_slot(), pairs_max = resident_pairs<256>(dev), pairs_narrow = resident_pairs<128>(dev);
    if (pairs_max <= 0 || pairs_narrow <= 0) return PQ_ERR_CUDA;
    const GemmArgs g{xq, sfx, wq, sfw, ts_x, ts_w, M, N, K, ldy, Y, ws, st};
    return narrow_tiles(M, N, K, pairs_narrow) ? launch_tiles<128>(g, pairs_narrow) : launch_tiles<256>(g, pairs_max);
}
}  // namespace

extern "C" pq_status pq_gemm_w4a4(const uint8_t *xq, const uint8_t *sfx, const float *ts_x, const uint8_t *wq,
                                  const uint8_t *sfw, const float *ts_w, int64_t M, int64_t N, int64_t K, void *Y,
                                  int64_t ldy, void *ws, size_t ws_bytes, void *stream) {
    return gemm_launch(xq, sfx, ts_x, wq, sfw, ts_w, M, N, K, Y, ldy, ws, ws_bytes, stream);
}

extern "C" pq_status pq_linear_w4a4(const void *X, int64_t M, int64_t K, int64_t ld, const float *ts_x, uint8_t *xq,
                                    uint8_t *sfx, const uint8_t *wq, const uint8_t *sfw, const float *ts_w, int64_t N,
                                    void *Y, int64_t ldy, void *ws, size_t ws_bytes, void *stream) {
    const pq_status rc = pq_quant_act_nvfp4(X, M, K, ld, ts_x, xq, sfx, PQ_SF_TCGEN05, stream);
    if (rc != PQ_OK) return rc;
    return gemm_launch(xq, sfx, ts_x, wq, sfw, ts_w, M, N, K, Y, ldy, ws, ws_bytes, stream);
}

extern "C" pq_status pq_linear_w4a4_host(const void *X_host, int64_t M, int64_t K, const float *ts_x, void *X_dev,
                                         uint8_t *xq, uint8_t *sfx, const uint8_t *wq, const uint8_t *sfw,
                                         const float *ts_w, int64_t N, void *Y_dev, void *Y_host, void *ws,
                                         size_t ws_bytes, void *stream) {
    PQ_REQUIRE(X_host && X_dev && Y_dev && Y_host, PQ_ERR_NULL);
    PQ_REQUIRE(M > 0 && K > 0 && N > 0, PQ_ERR_SHAPE);
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    PQ_CUDA_OK(cudaMemcpyAsync(X_dev, X_host, static_cast<size_t>(M) * K * 2, cudaMemcpyHostToDevice, st));
    const pq_status rc = pq_linear_w4a4(X_dev, M, K, K, ts_x, xq, sfx, wq, sfw, ts_w, N, Y_dev, N, ws, ws_bytes, stream);
    if (rc != PQ_OK) return rc;
    PQ_CUDA_OK(cudaMemcpyAsync(Y_host, Y_dev, static_cast<size_t>(M) * N * 2, cudaMemcpyDeviceToHost, st));
    return PQ_OK;
}

// ---------------------------------------------------------------- batches through one layer
namespace {
constexpr int kMaxSets = 8, kMaxPipeDevices = 64;

// Two internal streams and the events that order them, created once per device (host objects,
// no device memory).
struct Pipe {
    cudaStream_t q = nullptr, g = nullptr, up = nullptr, down = nullptr;
    cudaEvent_t fork = nullptr, join_q = nullptr, join_g = nullptr, join_up = nullptr, join_down = nullptr;
    cudaEvent_t q_done[kMaxSets] = {}, g_done[kMaxSets] = {}, up_done[kMaxSets] = {}, down_done[kMaxSets] = {};
    bool ready = false;
};

Pipe *pipe_for_current_device() {
    static std::mutex lock;
    static Pipe pipes[kMaxPipeDevices];
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxPipeDevices) return nullptr;
    std::lock_guard<std::mutex> guard(lock);
    Pipe &p = pipes[dev];
    if (!p.ready) {
        bool ok = cudaStreamCreateWithFlags(&p.q, cudaStreamNonBlocking) == cudaSuccess &&
                  cudaStreamCreateWithFlags(&p.g, cudaStreamNonBlocking) == cudaSuccess &&
                  cudaStreamCreateWithFlags(&p.up, cudaStreamNonBlocking) == cudaSuccess &&
                  cudaStreamCreateWithFlags(&p.down, cudaStreamNonBlocking) == cudaSuccess;
        auto make = [&](cudaEvent_t *e) { ok = ok && cudaEventCreateWithFlags(e, cudaEventDisableTiming) == cudaSuccess; };
        make(&p.fork), make(&p.join_q), make(&p.join_g), make(&p.join_up), make(&p.join_down);
        for (int i = 0; i < kMaxSets; ++i)
            make(&p.q_done[i]), make(&p.g_done[i]), make(&p.up_done[i]), make(&p.down_done[i]);
        if (!ok) {
            (void)cudaGetLastError();
            return nullptr;
        }
        p.ready = true;
    }
    return &p;
}
}  // namespace

extern "C" pq_status pq_linear_w4a4_batched(int n, const void *const *X, int64_t M, int64_t K, int64_t ld,
                                            const float *ts_x, uint8_t *const *xq, uint8_t *const *sfx, int n_sets,
                                            const uint8_t *wq, const uint8_t *sfw, const float *ts_w, int64_t N,
                                            void *const *Y, int64_t ldy, void *ws, size_t ws_bytes, void *stream) {
    PQ_REQUIRE(X && xq && sfx && Y, PQ_ERR_NULL);
    PQ_REQUIRE(n >= 1 && n_sets >= 2 && n_sets <= kMaxSets, PQ_ERR_SHAPE);
    for (int i = 0; i < n; ++i) PQ_REQUIRE(X[i] && Y[i], PQ_ERR_NULL);
    for (int s = 0; s < n_sets; ++s) PQ_REQUIRE(xq[s] && sfx[s], PQ_ERR_NULL);
    Pipe *pipe = pipe_for_current_device();
    if (!pipe) return PQ_ERR_CUDA;
    cudaStream_t user = static_cast<cudaStream_t>(stream);
    // fork: both internal streams start after everything already in the caller's stream
    PQ_CUDA_OK(cudaEventRecord(pipe->fork, user));
    PQ_CUDA_OK(cudaStreamWaitEvent(pipe->q, pipe->fork, 0));
    PQ_CUDA_OK(cudaStreamWaitEvent(pipe->g, pipe->fork, 0));
    pq_status rc = PQ_OK;
    // The GEMMs go out in pairs: both quantizer events are awaited in front of the pair, so the
    // second GEMM directly follows the first in its stream and may be its programmatic dependent
    // (its set-up overlaps the first one's last tiles).
    for (int i0 = 0; i0 < n && rc == PQ_OK; i0 += 2) {
        const int i1 = (i0 + 2 < n) ? i0 + 2 : n;
        for (int i = i0; i < i1 && rc == PQ_OK; ++i) {
            const int s = i % n_sets;
            // the GEMM that last read this set of intermediates has to be done with it
            if (i >= n_sets && cudaStreamWaitEvent(pipe->q, pipe->g_done[s], 0) != cudaSuccess) rc = PQ_ERR_CUDA;
            // 128-thread blocks: they fit on an SM beside the GEMM's CTA
            if (rc == PQ_OK) rc = pq_quant_act_nvfp4_shaped(X[i], M, K, ld, ts_x, xq[s], sfx[s], PQ_SF_TCGEN05, 1, pipe->q);
            if (rc == PQ_OK && cudaEventRecord(pipe->q_done[s], pipe->q) != cudaSuccess) rc = PQ_ERR_CUDA;
            if (rc == PQ_OK && cudaStreamWaitEvent(pipe->g, pipe->q_done[s], 0) != cudaSuccess) rc = PQ_ERR_CUDA;
        }
        for (int i = i0; i < i1 && rc == PQ_OK; ++i) {
            const int s = i % n_sets;
            rc = gemm_launch(xq[s], sfx[s], ts_x, wq, sfw, ts_w, M, N, K, Y[i], ldy, ws, ws_bytes, pipe->g);
            if (rc == PQ_OK && cudaEventRecord(pipe->g_done[s], pipe->g) != cudaSuccess) rc = PQ_ERR_CUDA;
        }
    }
    // join (also after an error, so that a stream capture in progress stays well-formed)
    bool joined = cudaEventRecord(pipe->join_q, pipe->q) == cudaSuccess &&
                  cudaEventRecord(pipe->join_g, pipe->g) == cudaSuccess &&
                  cudaStreamWaitEvent(user, pipe->join_q, 0) == cudaSuccess &&
                  cudaStreamWaitEvent(user, pipe->join_g, 0) == cudaSuccess;
    if (!joined) {
        (void)cudaGetLastError();
        return rc == PQ_OK ? PQ_ERR_CUDA : rc;
    }
    return rc;
}

extern "C" pq_status pq_linear_w4a4_host_batched(int n, const void *const *X_host, int64_t M, int64_t K,
                                                 const float *ts_x, void *const *X_dev, void *const *Y_dev, int n_sets,
                                                 uint8_t *xq, uint8_t *sfx, const uint8_t *wq, const uint8_t *sfw,
                                                 const float *ts_w, int64_t N, void *const *Y_host, void *ws,
                                                 size_t ws_bytes, void *stream) {
    PQ_REQUIRE(X_host && X_dev && Y_dev && Y_host, PQ_ERR_NULL);
    PQ_REQUIRE(n >= 1 && n_sets >= 2 && n_sets <= kMaxSets && M > 0 && K > 0 && N > 0, PQ_ERR_SHAPE);
    for (int i = 0; i < n; ++i) PQ_REQUIRE(X_host[i] && Y_host[i], PQ_ERR_NULL);
    for (int s = 0; s < n_sets; ++s) PQ_REQUIRE(X_dev[s] && Y_dev[s], PQ_ERR_NULL);
    Pipe *pipe = pipe_for_current_device();
    if (!pipe) return PQ_ERR_CUDA;
    cudaStream_t user = static_cast<cudaStream_t>(stream), up = pipe->up, run = pipe->g, down = pipe->down;
    const size_t x_bytes = static_cast<size_t>(M) * K * 2, y_bytes = static_cast<size_t>(M) * N * 2;
    PQ_CUDA_OK(cudaEventRecord(pipe->fork, user));
    PQ_CUDA_OK(cudaStreamWaitEvent(up, pipe->fork, 0));
    PQ_CUDA_OK(cudaStreamWaitEvent(run, pipe->fork, 0));
    PQ_CUDA_OK(cudaStreamWaitEvent(down, pipe->fork, 0));
    pq_status rc = PQ_OK;
    auto cuda_ok = [&](cudaError_t e) {
        if (e != cudaSuccess && rc == PQ_OK) rc = PQ_ERR_CUDA;
        return rc == PQ_OK;
    };
    for (int i = 0; i < n && rc == PQ_OK; ++i) {
        const int s = i % n_sets;
        // upload: the staging buffer is free once the quantizer of its previous batch has read it
        if (i >= n_sets && !cuda_ok(cudaStreamWaitEvent(up, pipe->q_done[s], 0))) break;
        if (!cuda_ok(cudaMemcpyAsync(X_dev[s], X_host[i], x_bytes, cudaMemcpyHostToDevice, up))) break;
        if (!cuda_ok(cudaEventRecord(pipe->up_done[s], up))) break;
        // compute: needs the upload, and the output buffer's previous download to have finished
        if (!cuda_ok(cudaStreamWaitEvent(run, pipe->up_done[s], 0))) break;
        if (i >= n_sets && !cuda_ok(cudaStreamWaitEvent(run, pipe->down_done[s], 0))) break;
        rc = pq_quant_act_nvfp4(X_dev[s], M, K, K, ts_x, xq, sfx, PQ_SF_TCGEN05, run);
        if (rc != PQ_OK || !cuda_ok(cudaEventRecord(pipe->q_done[s], run))) break;
        rc = gemm_launch(xq, sfx, ts_x, wq, sfw, ts_w, M, N, K, Y_dev[s], N, ws, ws_bytes, run);
        if (rc != PQ_OK || !cuda_ok(cudaEventRecord(pipe->g_done[s], run))) break;
        // download
        if (!cuda_ok(cudaStreamWaitEvent(down, pipe->g_done[s], 0))) break;
        if (!cuda_ok(cudaMemcpyAsync(Y_host[i], Y_dev[s], y_bytes, cudaMemcpyDeviceToHost, down))) break;
        if (!cuda_ok(cudaEventRecord(pipe->down_done[s], down))) break;
    }
    const bool joined = cudaEventRecord(pipe->join_up, up) == cudaSuccess &&
                        cudaEventRecord(pipe->join_g, run) == cudaSuccess &&
                        cudaEventRecord(pipe->join_down, down) == cudaSuccess &&
                        cudaStreamWaitEvent(user, pipe->join_up, 0) == cudaSuccess &&
                        cudaStreamWaitEvent(user, pipe->join_g, 0) == cudaSuccess &&
                        cudaStreamWaitEvent(user, pipe->join_down, 0) == cudaSuccess;
    if (!joined) {
        (void)cudaGetLastError();
        return rc == PQ_OK ? PQ_ERR_CUDA : rc;
    }
    return rc;
}

extern "C" pq_status pq_selftest_wait_expiry(void *ws, size_t ws_bytes, long long limit_cycles, int *observed,
                                             void *stream) {
    PQ_REQUIRE(ws && observed, PQ_ERR_NULL);
    PQ_REQUIRE(ws_bytes >= sizeof(int), PQ_ERR_WORKSPACE);
    PQ_REQUIRE(limit_cycles > 0 && limit_cycles <= 100000000ll, PQ_ERR_SHAPE);
    wait_expiry_kernel<<<1, 32, 0, static_cast<cudaStream_t>(stream)>>>(static_cast<int *>(ws), limit_cycles, observed);
    return pq_launch_status();
}

extern "C" pq_status pq_device_status(const void *ws, void *stream) {
    PQ_REQUIRE(ws, PQ_ERR_NULL);
    int word = 0;
    if (cudaStreamSynchronize(static_cast<cudaStream_t>(stream)) != cudaSuccess) {
        (void)cudaGetLastError();
        return PQ_ERR_CUDA;
    }
    PQ_CUDA_OK(cudaMemcpy(&word, ws, sizeof(int), cudaMemcpyDeviceToHost));
    return word == 0 ? PQ_OK : static_cast<pq_status>(word);
}

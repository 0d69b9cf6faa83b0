// Calibration quantization error per candidate order and group column (Eq. 3), the quantity
// the candidate selection (Sec. 3.3) and the acceptance rule (Eq. 10) compare.
//
// The original-order kernel leaves fp64 slab sums [slab][group column] in the workspace, the
// candidate kernel fp32 chunk partials [chunk][order][group column]; a second kernel, launched as a
// programmatic dependent, adds them to the fp64 totals in ascending order (for chunk partials:
// each slab's eight in fp64 from zero first).  No floating-point atomics.
//
//   original order (perms == NULL): a thread owns 16 adjacent channels (two 16-byte loads per
//     row) of one chunk, i.e. a whole NVFP4 group or 1/2 .. 1/8 of an integer group; it loads
//     eight rows at a time and walks them in order; a block covers the eight chunks of a slab.  The pass streams the tensor once from HBM;
//     its cost per element is arithmetic (about ten instructions), so it sits between the HBM and
//     the ALU roof.
//   candidate orders: persistent blocks of thread groups; a group stages a chunk's rows in shared memory four at a time,
//     interleaved per channel, for all orders of its share of the (chunk, order) pairs, and a lane gathers the 16 channels
//     of its run for four rows with 64-bit loads, two rows side by side in packed registers; the tensor is fetched from HBM
//     about once.  Few (chunk, order) pairs go to one block each instead (group_error_chunk).
#include <type_traits>

#include "pq_common.cuh"

namespace {

// ---------------------------------------------------------------- original order
constexpr int64_t kErrMaxK = 16384;
constexpr int kDirectThreads = 128;
constexpr int kDirectRows = 4;  // rows in flight per thread (2 x 16 bytes each)

// Decode scale d = sf * ts and its reciprocal for each of the 256 scale bytes (they depend on the
// byte only): built once per block, so a group costs one division, one convert and one 8-byte
// shared-memory load instead of a second convert, a multiply and an IEEE reciprocal.
__device__ __forceinline__ void build_scale_table(float2 *table, float ts) {
    for (int b = threadIdx.x; b < 256; b += blockDim.x) {
        const float d = __fmul_rn(pq::e4m3_to_f32(static_cast<uint32_t>(b)), ts);
        table[b] = make_float2(d, d > 0.0f ? __frcp_rn(d) : 0.0f);
    }
}

using pq::add2;
using pq::bf16_pattern;
using pq::fma2;
using pq::max_bf16x2;
using pq::max_u16x2;
using pq::min_u16x2;
using pq::mul2;
using pq::pack2;
using pq::unpack2;

// Error of one row's 16 channels held by this lane; TEAM16 = group / 16 adjacent lanes share a group.
// c6 = 6 * ts (NVFP4 only).  The lane's two 8-channel runs are carried side by side in packed
// registers: per run the operations and their order are those of the scalar definition (scale the
// magnitude by the reciprocal, round to a level, residual by one fused multiply-add, squares added in
// channel order), two results per instruction.  Magnitudes are taken on the bf16 pairs, which is exact.
template <int KIND, int TEAM16>
__device__ __forceinline__ float row_sse16(const uint4 &lo, const uint4 &hi, float c6, const float2 *table, float Qf) {
    const uint32_t m = 0x7FFF7FFFu;
    const uint4 la = make_uint4(lo.x & m, lo.y & m, lo.z & m, lo.w & m);
    const uint4 ha = make_uint4(hi.x & m, hi.y & m, hi.z & m, hi.w & m);
    float xa[8], xb[8];
    pq::unpack8(la, xa);
    pq::unpack8(ha, xb);
    // absmax of the 16 magnitudes on the bf16 pairs (exact: a maximum selects one of its inputs)
    const uint32_t mx = max_bf16x2(max_bf16x2(max_bf16x2(la.x, la.y), max_bf16x2(la.z, la.w)),
                                   max_bf16x2(max_bf16x2(ha.x, ha.y), max_bf16x2(ha.z, ha.w)));
    float amax = fmaxf(__uint_as_float(mx << 16), __uint_as_float(mx & 0xFFFF0000u));
    amax = pq::team_max<TEAM16>(amax);
    float d, r;
    if (KIND == 0) {
        const float2 dr = table[pq::f32_to_e4m3(__fdiv_rn(amax, c6))];
        d = dr.x, r = dr.y;
    } else {
        pq::int_scale(amax, Qf, d, r);
    }
    const uint64_t r2 = pack2(r, r), nd2 = pack2(-d, -d);
    uint64_t x2[8], q2[8];
    if (KIND == 0) {
        float ya[8], yb[8], qa[8], qb[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            x2[i] = pack2(xa[i], xb[i]);
            unpack2(mul2(x2[i], r2), ya[i], yb[i]);
        }
        pq::e2m1_levels(pq::f32x8_to_e2m1(ya), qa);
        pq::e2m1_levels(pq::f32x8_to_e2m1(yb), qb);
#pragma unroll
        for (int i = 0; i < 8; ++i) q2[i] = pack2(qa[i], qb[i]);
    } else {
        // min(rint(y), Q): adding and subtracting 1.5 * 2^23 rounds like rint for y < 2^22, beyond that the clamp decides
        // (the first addition is written as y * 1 + magic: a packed multiply directly followed by a packed
        // add was seen to come out as one fused operation, which rounds once instead of twice)
        const uint64_t magic = pack2(12582912.0f, 12582912.0f), unmagic = pack2(-12582912.0f, -12582912.0f);
        const uint64_t one2 = pack2(1.0f, 1.0f);
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            x2[i] = pack2(xa[i], xb[i]);
            float za, zb;
            unpack2(add2(fma2(mul2(x2[i], r2), one2, magic), unmagic), za, zb);
            q2[i] = pack2(fminf(za, Qf), fminf(zb, Qf));
        }
    }
    uint64_t acc2 = pack2(0.0f, 0.0f);
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const uint64_t delta = fma2(q2[i], nd2, x2[i]);
        acc2 = fma2(delta, delta, acc2);
    }
    float sa, sb;
    unpack2(acc2, sa, sb);
    // runs of 8 channels, then the balanced adjacent-pair tree: its first level is this lane's two runs
    return pq::team_sum<TEAM16>(__fadd_rn(sa, sb));
}

constexpr int kSlabChunks = PQ_SLAB_ROWS / PQ_CHUNK_ROWS;  // 8
constexpr int kDirectRuns = kDirectThreads / kSlabChunks;  // 16 runs of 16 channels per block
static_assert(kDirectRuns == 16, "a warp holds two chunks of 16 runs");

// One block = one 128-row slab x 256 channels: thread (c, j) owns chunk c of the slab and the
// j-th 16-channel run, so a warp reads 2 x 512 contiguous bytes per row step.  The eight chunk
// partials of a group meet in shared memory and one thread adds them in fp64 in chunk order;
// the workspace receives fp64 slab sums [slab][K/g].
template <int KIND, int TEAM16>
__global__ void __launch_bounds__(kDirectThreads, 8)
group_error_direct(const uint16_t *__restrict__ T, int64_t rows, int64_t K, int64_t ld,
                   const float *__restrict__ ts_ptr, float Qf, double *__restrict__ slab_part /*[slabs, K/g]*/) {
    __shared__ float part_s[kSlabChunks][kDirectRuns];
    __shared__ float2 scale_table[KIND == 0 ? 256 : 1];
    pq::dependents_may_launch();
    const int runs = static_cast<int>(K >> 4);  // K % (16 * TEAM16) == 0
    const int c = threadIdx.x / kDirectRuns, j = threadIdx.x % kDirectRuns;
    const int run = blockIdx.y * kDirectRuns + j;
    const int64_t slab = blockIdx.x;
    const int64_t r0 = slab * PQ_SLAB_ROWS + c * PQ_CHUNK_ROWS;
    // 16 % TEAM16 == 0 and runs % TEAM16 == 0: a team is live or dead as a whole, and the
    // shuffles below stay inside its 16-lane half of the warp
    const bool live = run < runs && r0 < rows;
    const int n = live ? static_cast<int>(min(static_cast<int64_t>(PQ_CHUNK_ROWS), rows - r0)) : 0;
    const float ts = (KIND == 0) ? __ldg(ts_ptr) : 1.0f;
    const float c6 = __fmul_rn(6.0f, ts);
    if (KIND == 0) {
        build_scale_table(scale_table, ts);
        __syncthreads();
    }
    const uint16_t *p = T + (live ? r0 * ld + static_cast<int64_t>(run) * 16 : 0);
    float acc = 0.0f;
#pragma unroll 1
    for (int t0 = 0; t0 < PQ_CHUNK_ROWS; t0 += kDirectRows) {
        uint4 lo[kDirectRows], hi[kDirectRows];
        const uint4 zero = make_uint4(0, 0, 0, 0);
#pragma unroll
        for (int u = 0; u < kDirectRows; ++u) {
            const bool have = t0 + u < n;
            const uint4 *src = reinterpret_cast<const uint4 *>(p + static_cast<int64_t>(t0 + u) * ld);
            lo[u] = have ? __ldg(src) : zero;
            hi[u] = have ? __ldg(src + 1) : zero;
        }
        // rows past the end are all-zero groups: their error is +0.0 and adding it changes nothing
#pragma unroll
        for (int u = 0; u < kDirectRows; ++u) acc = __fadd_rn(acc, row_sse16<KIND, TEAM16>(lo[u], hi[u], c6, scale_table, Qf));
    }
    part_s[c][j] = acc;
    __syncthreads();
    // chunks past the last row hold +0.0, which leaves the slab sum unchanged
    if (threadIdx.x < kDirectRuns && run < runs && (run % TEAM16) == 0) {
        double sum = 0.0;
#pragma unroll
        for (int k = 0; k < kSlabChunks; ++k) sum = __dadd_rn(sum, static_cast<double>(part_s[k][j]));
        slab_part[slab * (runs / TEAM16) + run / TEAM16] = sum;
    }
}

// ---------------------------------------------------------------- candidate orders
// A thread group (whole warps, one named barrier) owns a chunk of 16 rows.  It passes them through shared
// memory four at a time as magnitudes, interleaved per channel, and runs every order of its block over the
// staged rows before it fetches the next four: the staging is paid once for up to eight orders instead of
// once per order.  A lane takes a run of 16 positions: its slots come from a table of 16-bit indices the
// block prepared once per order, one 64-bit load per position brings that channel of four rows, and the
// error of TWO ROWS is carried side by side (row_pair_sse): the words the gather returns hold the same channel of
// two rows, so they are widened as they are; the one-row-at-a-time form
// had to re-pair them by byte permutes first (half an instruction per element), read the original-order
// kernel's decode tables (two per element; the hardware E2M1 -> f16 -> fp32 converts take one and a half)
// and divide once per group and row (the scale tables below take a clamp and two loads).
// Blocks are persistent, one per SM; the groups of a block only share the slot and scale tables.
//
// NVFP4 is scalar arithmetic but for the sums: packed f32x2 instructions save issue slots but run on one of the two FMA pipes only, and
// with the f16 converts there too it was 59 % busy (9216 x 3072, six orders, with an earlier fold: 79 us scalar, 84
// packed); only the sums of squares are packed, which leaves that pipe room (9216 x 3072 72.9 -> 71.6, 4608 x
// 12288 197.6 -> 194.7; the multiplication packed 81.2, the residual 74.6).  The integer formats, without converts, are packed (4608 x 3072,
// INT4 g64, with that fold: 53.4 us, 54.1 scalar).
// What bounds it: instruction issue (67 % of the slots busy at 23 warps per SM) and shared-memory wavefronts (a 64-bit gather
// through a random order takes about 6 of them where 2 would do: 0.069 per element and order).
// Registers: 80 per thread, of which 36 to 56 bytes are spilled.  The weights of the acceptance rule, two chains of K additions, have a
// block of their own and the gather one SM less: with a 25th warp on every SM for them the compiler had 72 (60 to 96 bytes), and
// the chain, among the gather's warps, outlasted short passes (3 x 500 x 2560 in INT3).
constexpr int kGatherThreads = 768;
constexpr int kMaxOrders = 9;      // eight candidates and the original order
constexpr int kMaxGroups = 15;                                           // named barriers 1..15
constexpr int kSfTabMax = 2624;  // bf16 magnitudes from "scale byte 0" to "saturated": 19 binades and the edges

// What a group's scale is looked up in, per side (activations / weight: they differ in the tensor scale).
//   NVFP4    {1 / d, -d} for the decode scale d, as a function of the group's absmax, a bf16 magnitude: every magnitude
//            up to `lo` gives scale byte 0 and every one from `hi` on the saturated byte, the ones between are
//            tabulated from the definition.
//   integer  by the mantissa of amax (pq::build_int_tab).
struct ScaleTab {
    float2 rd[kSfTabMax];
    uint32_t lo, hi, pad[2];
};
__device__ __forceinline__ void build_scale_tab(ScaleTab &tab, float ts) {
    const float c6 = __fmul_rn(6.0f, ts), mag = fabsf(c6);
    // (signed) byte 0 up to |c6| 2^-10, half the smallest subnormal (ties to even); saturated from 448 |c6| on.  A
    // zero c6 makes every quotient but 0 / 0 infinite; with an infinite or NaN one every decode scale is NaN.
    uint32_t lo = 0, hi = 0;
    if (mag == 0.0f) hi = 1;
    else if (mag < __uint_as_float(0x7F800000u)) {
        lo = __float_as_uint(__fmul_rz(mag, 0.0009765625f)) >> 16;
        hi = min(0x7F80u, (__float_as_uint(__fmul_rn(mag, 448.0f)) >> 16) + 2u);
    }
    if (threadIdx.x == 0) tab.lo = lo, tab.hi = hi;
#pragma unroll 4
    for (uint32_t i = threadIdx.x; i <= hi - lo && i < kSfTabMax; i += blockDim.x) {
        const float d = __fmul_rn(pq::e4m3_to_f32(pq::f32_to_e4m3(__fdiv_rn(bf16_pattern(lo + i), c6))), ts);
        tab.rd[i] = make_float2(d > 0.0f ? __frcp_rn(d) : 0.0f, -d);
    }
}
// E2M1 of two floats and back to fp32 (E2M1 -> f16 is exact, f16 -> f32 too).
__device__ __forceinline__ void e2m1_pair(float &y0, float &y1) {
    uint32_t h2;
    asm("{\n"
        ".reg .b8 c;\n"
        "cvt.rn.satfinite.e2m1x2.f32 c, %2, %1;\n"
        "cvt.rn.f16x2.e2m1x2 %0, c;\n"
        "}\n"
        : "=r"(h2)
        : "f"(y0), "f"(y1));
    y0 = __half2float(__ushort_as_half(static_cast<uint16_t>(h2 & 0xFFFFu)));
    y1 = __half2float(__ushort_as_half(static_cast<uint16_t>(h2 >> 16)));
}

// One row of a pair by the definition of the integer formats: for scales in subnormal or non-finite territory.
struct RunWords {
    uint32_t u[16];
};
template <int TEAM16>
__device__ __noinline__ float int_row_sse_words(const RunWords words, int row, float amax, float Qf) {
    float d, rc, run[2];
    pq::int_scale(amax, Qf, d, rc);
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        run[h] = 0.0f;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const uint32_t w = words.u[8 * h + i];
            const float x = __uint_as_float(row ? w & 0xFFFF0000u : w << 16);
            const float z = fminf(__fadd_rn(__fadd_rn(__fmul_rn(x, rc), 12582912.0f), -12582912.0f), Qf);
            const float delta = __fmaf_rn(-z, d, x);
            run[h] = __fmaf_rn(delta, delta, run[h]);
        }
    }
    return pq::team_sum<TEAM16>(__fadd_rn(run[0], run[1]));
}
template <int TEAM16>
__device__ __forceinline__ float int_row_sse(const uint32_t (&u)[16], int row, float amax, float Qf) {
    RunWords words;
#pragma unroll
    for (int i = 0; i < 16; ++i) words.u[i] = u[i];
    return int_row_sse_words<TEAM16>(words, row, amax, Qf);
}

// Errors of a run of 16 positions in two rows: u[i] = magnitudes of position i in row 0 (low half) and row 1
// (high half).  Per row the operations and their order are those of row_sse16.
template <int KIND, int TEAM16>
__device__ __forceinline__ void row_pair_sse(const uint32_t (&u)[16], const ScaleTab *tab, uint32_t lo2, uint32_t hi2,
                                             const uint2 *int_tab, float Qf, float &e0, float &e1) {
    // absmax of both rows at once (a maximum of magnitudes selects one of its inputs)
    uint32_t mx[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) mx[i] = max_bf16x2(u[i], u[i + 8]);
#pragma unroll
    for (int s = 4; s; s >>= 1)
#pragma unroll
        for (int i = 0; i < s; ++i) mx[i] = max_bf16x2(mx[i], mx[i + s]);
    uint32_t am = mx[0];
#pragma unroll
    for (int m = 1; m < TEAM16; m <<= 1) am = max_bf16x2(am, __shfl_xor_sync(0xFFFFFFFFu, am, m));
    float r0, r1, nd0, nd1;  // reciprocal and negated decode scale of either row
    if (KIND == 0) {
        const uint32_t cl = min_u16x2(max_u16x2(am, lo2), hi2);
        const float2 *rd = tab->rd - (lo2 & 0xFFFFu);
        const float2 d0 = rd[cl & 0xFFFFu], d1 = rd[cl >> 16];
        r0 = d0.x, r1 = d1.x, nd0 = d0.y, nd1 = d1.y;
    } else {
        const uint32_t a0 = am & 0xFFFFu, a1 = am >> 16;
        if (__any_sync(0xFFFFFFFFu, pq::int_scale_is_odd(a0) || pq::int_scale_is_odd(a1))) {
            e0 = int_row_sse<TEAM16>(u, 0, bf16_pattern(a0), Qf), e1 = int_row_sse<TEAM16>(u, 1, bf16_pattern(a1), Qf);
            return;
        }
        pq::int_scale_from_tab(int_tab, a0, r0, nd0);
        pq::int_scale_from_tab(int_tab, a1, r1, nd1);
    }

    float run0[2], run1[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        if (KIND == 0) {
            uint64_t acc2 = 0;  // {+0, +0}
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const uint32_t w = u[8 * h + i];
                const float x0 = __uint_as_float(w << 16), x1 = __uint_as_float(w & 0xFFFF0000u);
                float q0 = __fmul_rn(x0, r0), q1 = __fmul_rn(x1, r1);
                e2m1_pair(q0, q1);
                const float d0 = __fmaf_rn(q0, nd0, x0), d1 = __fmaf_rn(q1, nd1, x1);
                const uint64_t d2 = pack2(d0, d1);
                acc2 = fma2(d2, d2, acc2);
            }
            unpack2(acc2, run0[h], run1[h]);
        } else {
            const uint64_t r2 = pack2(r0, r1), nd2 = pack2(nd0, nd1), one2 = pack2(1.0f, 1.0f);
            const uint64_t magic = pack2(12582912.0f, 12582912.0f), unmagic = pack2(-12582912.0f, -12582912.0f);
            uint64_t acc2 = 0;  // {+0, +0}
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const uint32_t w = u[8 * h + i];
                const uint64_t x2 = pack2(__uint_as_float(w << 16), __uint_as_float(w & 0xFFFF0000u));
                // rint by adding and subtracting 1.5 * 2^23 (see row_sse16 for the form of the first addition).  No clamp:
                // |x| / s <= Q (1 + 2^-22) here, which rounds to Q at most.
                const uint64_t q2 = add2(fma2(mul2(x2, r2), one2, magic), unmagic);
                const uint64_t d2 = fma2(q2, nd2, x2);
                acc2 = fma2(d2, d2, acc2);
            }
            unpack2(acc2, run0[h], run1[h]);
        }
    }
    e0 = pq::team_sum<TEAM16>(__fadd_rn(run0[0], run0[1])), e1 = pq::team_sum<TEAM16>(__fadd_rn(run1[0], run1[1]));
}

struct GatherParams {
    PqTensorList list;
    const float *ts[2];        // tensor scale per side (NVFP4)
    int K, P, identity;        // P orders; identity != 0: order 0 is the original one and perms holds the others
    const int32_t *perms;      // [P - identity, K]
    int opb;                   // orders per block, a subset of them
    int groups, group_threads;
    int blocks;                // per subset of the orders; behind all of them one for the error weights, if they are asked for
    uint32_t base[2], rem[2];  // pairs of the first `split` chunks / shares and its remainder: subsets of opb orders, the last
    uint32_t split;
    int full;                  // whole chunks per share behind them
    int chunks;                // eight per slab; the chunks of a last slab that hold no rows may be left out
    float Qf;
    float *part;               // [chunks, P, K/g]
    PqErrorWeights weights;    // added up by a block of their own, beside the gather
};

constexpr size_t kGatherSmemMax = 226 * 1024;
constexpr int kTabBytes = (static_cast<int>(sizeof(ScaleTab)) + 15) / 16 * 16;

inline size_t gather_smem_bytes(int64_t K, int opb, int groups, int sides) {
    return static_cast<size_t>(groups) * K * 8 + static_cast<size_t>(opb) * K * 2 +
           static_cast<size_t>(groups) * opb * (K / 16) * 4 + static_cast<size_t>(sides) * kTabBytes;
}

// Eight channels of a staged row.  Both forms are coherent; which one the compiler schedules better differs (plain against .cg, us
// for 4608 x 12288 and six orders: NVFP4 180.1 / 180.8, INT g64 188.4 / 194.9, g128 194.4 / 202.8; g16 183.7 / 181.9, g32 188.3 / 186.2,
// g256 209.2 / 205.3).
template <int KIND, int TEAM16>
__device__ __forceinline__ uint4 load_row(const uint4 *p) {
    return KIND == 0 || TEAM16 == 4 || TEAM16 == 8 ? *p : __ldcg(p);
}

template <int KIND, int TEAM16>
__global__ void __launch_bounds__(kGatherThreads, 1) group_error_gather(const __grid_constant__ GatherParams p) {
    // [groups][K][4 rows] bf16 magnitudes | [opb][K] 16-bit slots | scale tables | [groups][opb][runs] fp32 chunk sums
    extern __shared__ __align__(16) unsigned char smem[];
    const int K = p.K, octs = K >> 3, runs = K >> 4;
    const uint32_t subset = blockIdx.x / static_cast<uint32_t>(p.blocks), block = blockIdx.x - subset * p.blocks;
    const int o0 = static_cast<int>(subset) * p.opb, no = min(p.opb, p.P - o0);
    uint16_t *slot_s = reinterpret_cast<uint16_t *>(smem + static_cast<size_t>(p.groups) * K * 8);
    unsigned char *tab_s = reinterpret_cast<unsigned char *>(slot_s + static_cast<size_t>(p.opb) * K);
    uint2 *int_tab = reinterpret_cast<uint2 *>(tab_s);
    if (KIND == 1) pq::build_int_tab(int_tab, p.Qf, true);  // needs nothing of the kernel in front
    pq::dependents_may_launch();
    pq::wait_for_prior_grid();

    if (o0 >= p.P) {  // the block of the error weights: a warp per side
        for (int s = threadIdx.x >> 5; s < 2; s += blockDim.x >> 5) {
            const double sum = pq::ordered_sum(s ? p.weights.sumsq_w : p.weights.sumsq_a, K);
            if ((threadIdx.x & 31) == 0) p.weights.lambda[s] = __ddiv_rn(1.0, sum);
        }
        return;
    }

    // Slots of the orders.  The two 16-byte halves of a run's lie in separate planes: lanes read consecutive 16-byte words.
    auto slots_at = [&](int j) { return slot_s + ((j >> 3) & 1) * (K >> 1) + (j >> 4) * 8 + (j & 7); };
    if (K <= static_cast<int>(blockDim.x) || (reinterpret_cast<uintptr_t>(p.perms) & 15u)) {
        for (int j = threadIdx.x; j < K; j += blockDim.x) {
            // the channel of every order at position j, all loads in flight (one after the other they cost 10 us a launch)
            uint32_t ch[kMaxOrders];
#pragma unroll
            for (int o = 0; o < kMaxOrders; ++o) {
                const int order = o0 + o - p.identity;
                ch[o] = o < no && order >= 0 ? static_cast<uint32_t>(__ldca(p.perms + static_cast<int64_t>(order) * K + j)) : static_cast<uint32_t>(j);
            }
#pragma unroll
            for (int o = 0; o < kMaxOrders; ++o)
                if (o < no) slots_at(j)[o * K] = static_cast<uint16_t>(pq::quad_channel(ch[o]));
        }
    } else {
        // four positions a thread, half of the orders at a time (3072 channels: 1.2 us, one position a thread 3.6)
        for (int j = 4 * threadIdx.x; j < K; j += 4 * blockDim.x) {
            constexpr int kHalf = (kMaxOrders + 1) / 2;
#pragma unroll
            for (int h = 0; h < kMaxOrders; h += kHalf) {
                int4 ch[kHalf];
#pragma unroll
                for (int u = 0; u < kHalf; ++u) {
                    const int order = o0 + h + u - p.identity;
                    ch[u] = h + u < no && order >= 0 ? __ldca(reinterpret_cast<const int4 *>(p.perms + static_cast<int64_t>(order) * K + j))
                                                     : make_int4(j, j + 1, j + 2, j + 3);
                }
#pragma unroll
                for (int u = 0; u < kHalf; ++u)
                    if (h + u < no)
                        *reinterpret_cast<uint2 *>(slots_at(j) + (h + u) * K) =
                            make_uint2(pq::quad_channel(static_cast<uint32_t>(ch[u].x)) | pq::quad_channel(static_cast<uint32_t>(ch[u].y)) << 16,
                                       pq::quad_channel(static_cast<uint32_t>(ch[u].z)) | pq::quad_channel(static_cast<uint32_t>(ch[u].w)) << 16);
            }
        }
    }
    const int sides = p.ts[1] ? 2 : 1;
    if (KIND == 0) {
        for (int s = 0; s < sides; ++s) build_scale_tab(reinterpret_cast<ScaleTab *>(tab_s + s * kTabBytes)[0], __ldca(p.ts[s]));
    }
    __syncthreads();

    const int grp = threadIdx.x / p.group_threads, tid = threadIdx.x - grp * p.group_threads;
    auto group_sync = [&]() {
        if (p.group_threads == 32) __syncwarp();
        else asm volatile("bar.sync %0, %1;" ::"r"(grp + 1), "r"(p.group_threads) : "memory");
    };
    uint4 *quad4 = reinterpret_cast<uint4 *>(smem + static_cast<size_t>(grp) * K * 8);
    const uint32_t quad_addr = static_cast<uint32_t>(__cvta_generic_to_shared(quad4));
    float *acc_s = reinterpret_cast<float *>(tab_s + (KIND == 0 ? sides : 1) * kTabBytes) + static_cast<size_t>(grp) * p.opb * runs;
    const uint4 *slot4 = reinterpret_cast<const uint4 *>(slot_s);
    const int64_t Kg = runs / TEAM16;

    // An equal part of the (chunk, order) pairs of the first p.split chunks, then p.full whole chunks.  Without the first
    // part a group that has work for a few chunks only would wait for the one that has a whole chunk more; without the
    // second a group would stage one more chunk of which it uses some orders (eight batches of 4608 x 3072 and a
    // 9216 x 3072 weight, with an earlier fold: 535 us a calibration all in pairs, 518 like this).
    const uint32_t shares = p.blocks * p.groups, share = block * p.groups + grp;
    const uint32_t base = p.base[o0 + no == p.P], rem = p.rem[o0 + no == p.P];
    const uint32_t first = share * base + min(share, rem);
    int pairs = static_cast<int>(base + (share < rem)), full = p.full * no;
    uint32_t chunk = first / static_cast<uint32_t>(no), step = 1;
    int ob = static_cast<int>(first - chunk * no);
    for (int oe;; pairs -= oe - ob, ob = 0, chunk += step) {
        if (pairs == 0) {
            if (full == 0) break;
            pairs = full, full = 0, ob = 0;
            chunk = p.split + share, step = shares;
        }
        oe = min(no, ob + pairs);
        const int slab = static_cast<int>(chunk / kSlabChunks), t = pq::tensor_of_slab(p.list, slab);
        const int64_t r0 = static_cast<int64_t>(slab - p.list.slab0[t]) * PQ_SLAB_ROWS + chunk % kSlabChunks * PQ_CHUNK_ROWS;
        const int64_t ld = p.list.ld[t], left = p.list.rows[t] - r0;
        const int n = left >= PQ_CHUNK_ROWS ? PQ_CHUNK_ROWS : (left > 0 ? static_cast<int>(left) : 0);
        const uint16_t *src = p.list.ptr[t] + r0 * ld;
        const ScaleTab *tab = reinterpret_cast<const ScaleTab *>(tab_s + (KIND == 0 && t >= p.list.n_x ? kTabBytes : 0));
        const uint32_t lo2 = KIND == 0 ? tab->lo * 0x10001u : 0u, hi2 = KIND == 0 ? tab->hi * 0x10001u : 0u;
#pragma unroll 1
        for (int quad = 0; quad < PQ_CHUNK_ROWS / 4; ++quad) {
            if (4 * quad >= n) break;  // no rows left: their error is +0.0
            group_sync();              // the previous four rows have been used
#pragma unroll 2
            for (int o = tid; o < octs; o += p.group_threads) {
                uint4 v[4];
#pragma unroll
                for (int r = 0; r < 4; ++r) {  // rows past the end are zeros: their error is +0.0 and adding it changes nothing
                    v[r] = 4 * quad + r < n ? load_row<KIND, TEAM16>(reinterpret_cast<const uint4 *>(src + (4 * quad + r) * ld) + o) : make_uint4(0, 0, 0, 0);
                    v[r].x &= 0x7FFF7FFFu, v[r].y &= 0x7FFF7FFFu, v[r].z &= 0x7FFF7FFFu, v[r].w &= 0x7FFF7FFFu;
                }
                pq::store_quad_octet(quad4, o, v);
            }
            group_sync();
#pragma unroll 1
            for (int o = ob; o < oe; ++o) {
#pragma unroll 1
                for (int q0 = 0; q0 < runs; q0 += p.group_threads) {
                    const int q = q0 + tid;
                    const bool live = q < runs;  // runs % TEAM16 == 0: a team is live or dead as a whole
                    const int at = o * (K >> 3) + (live ? q : 0);
                    const uint4 i0 = slot4[at], i1 = slot4[at + runs];
                    const uint32_t iw[8] = {i0.x, i0.y, i0.z, i0.w, i1.x, i1.y, i1.z, i1.w};
                    uint32_t lo[16], hi[16];
#pragma unroll
                    for (int w = 0; w < 8; ++w) {
                        // byte address 8 * slot + base of either half of the word: one dot product each
                        const uint32_t x = __dp2a_lo(iw[w], 0x0008u, quad_addr), y = __dp2a_lo(iw[w], 0x0800u, quad_addr);
                        asm("ld.shared.v2.b32 {%0, %1}, [%2];" : "=r"(lo[2 * w]), "=r"(hi[2 * w]) : "r"(x) : "memory");
                        asm("ld.shared.v2.b32 {%0, %1}, [%2];" : "=r"(lo[2 * w + 1]), "=r"(hi[2 * w + 1]) : "r"(y) : "memory");
                    }
                    float e0, e1, e2, e3;
                    row_pair_sse<KIND, TEAM16>(lo, tab, lo2, hi2, int_tab, p.Qf, e0, e1);
                    row_pair_sse<KIND, TEAM16>(hi, tab, lo2, hi2, int_tab, p.Qf, e2, e3);
                    if (live) {
                        float acc = quad ? acc_s[o * runs + q] : 0.0f;
                        acc = __fadd_rn(__fadd_rn(__fadd_rn(__fadd_rn(acc, e0), e1), e2), e3);
                        acc_s[o * runs + q] = acc;
                    }
                }
            }
        }
        // every thread writes out the sums it kept itself
        for (int o = ob; o < oe; ++o)
            for (int q = tid; q < runs; q += p.group_threads)
                if ((q % TEAM16) == 0) p.part[(static_cast<int64_t>(chunk) * p.P + o0 + o) * Kg + q / TEAM16] = n ? acc_s[o * runs + q] : 0.0f;
    }
}

// ---------------------------------------------------------------- candidate orders, few pairs
// One block per (chunk, order), several per SM.  The chunk goes through shared memory four rows at a time, interleaved per
// channel as above; a thread owns whole 16-channel runs (GPT of them, blockDim apart), keeps their slots packed in registers,
// and for every row rebuilds the two 16-byte words the original-order kernel loads, so the error of a run is computed by
// the same routine, in row order.  It prepares no tables, and the blocks of an SM fill each other's waits; what it costs is
// staging the chunk once per order.  While its blocks are all resident at once it is the faster one (chunk_kernel_serves).
constexpr int kChunkThreads = 256, kChunkMaxGpt = 4;  // 256 threads x 4 runs x 16 channels = 16384 channels

// one run per thread (up to 4096 channels): held to 64 registers, five 192-thread blocks per SM instead of four
template <int KIND, int TEAM16, int GPT>
__global__ void __launch_bounds__(kChunkThreads, GPT == 1 ? 4 : 1)
group_error_chunk(const uint16_t *__restrict__ T, int64_t rows, int64_t K, int64_t ld,
                  const float *__restrict__ ts_ptr, float Qf, const int32_t *__restrict__ perms, int P,
                  float *__restrict__ part /*[chunks, P, K/g]*/) {
    extern __shared__ __align__(16) uint16_t quad_s[];  // [K][4 rows]
    __shared__ float2 scale_table[KIND == 0 ? 256 : 1];
    pq::dependents_may_launch();
    const int64_t chunk = blockIdx.x;
    const int p = blockIdx.y;
    const int32_t *perm = perms + static_cast<int64_t>(p) * K;
    const int octs = static_cast<int>(K >> 3), runs = static_cast<int>(K >> 4);
    const int64_t r0 = chunk * PQ_CHUNK_ROWS;
    const float ts = (KIND == 0) ? __ldg(ts_ptr) : 1.0f;
    const float c6 = __fmul_rn(6.0f, ts);
    if (KIND == 0) build_scale_table(scale_table, ts);  // the first barrier below publishes it

    // positions of this thread's channels in the interleaved image, two per register
    uint32_t ch[GPT][8];
    float acc[GPT];
#pragma unroll
    for (int t = 0; t < GPT; ++t) {
        acc[t] = 0.0f;
        const int q = threadIdx.x + t * blockDim.x;
#pragma unroll
        for (int w = 0; w < 8; ++w) {
            uint32_t lo = 0, hi = 0;
            if (q < runs) {
                lo = pq::quad_channel(static_cast<uint32_t>(perm[q * 16 + 2 * w]));
                hi = pq::quad_channel(static_cast<uint32_t>(perm[q * 16 + 2 * w + 1]));
            }
            ch[t][w] = lo | (hi << 16);
        }
    }

    uint4 *quad4 = reinterpret_cast<uint4 *>(quad_s);
    const uint2 *quad2 = reinterpret_cast<const uint2 *>(quad_s);
#pragma unroll 1
    for (int quad = 0; quad < PQ_CHUNK_ROWS / 4; ++quad) {
        const int64_t row = r0 + 4 * quad;
        if (row >= rows) break;  // no rows left: their error is +0.0
        __syncthreads();         // the previous four rows have been used
        for (int o = threadIdx.x; o < octs; o += blockDim.x) {
            uint4 v[4];
#pragma unroll
            for (int r = 0; r < 4; ++r)  // rows past the end are zeros: their error is +0.0 and adding it changes nothing
                v[r] = row + r < rows ? __ldg(reinterpret_cast<const uint4 *>(T + (row + r) * ld) + o) : make_uint4(0, 0, 0, 0);
            pq::store_quad_octet(quad4, o, v);
        }
        __syncthreads();
#pragma unroll
        for (int t = 0; t < GPT; ++t) {
            if (t * static_cast<int>(blockDim.x) >= runs) break;  // uniform over the block
            uint2 g[16];
#pragma unroll
            for (int w = 0; w < 8; ++w) {
                g[2 * w] = quad2[ch[t][w] & 0xFFFFu];
                g[2 * w + 1] = quad2[ch[t][w] >> 16];
            }
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                uint32_t pr[8];
#pragma unroll
                for (int w = 0; w < 8; ++w) {
                    const uint32_t a = r < 2 ? g[2 * w].x : g[2 * w].y, b = r < 2 ? g[2 * w + 1].x : g[2 * w + 1].y;
                    pr[w] = __byte_perm(a, b, (r & 1) ? 0x7632 : 0x5410);
                }
                acc[t] = __fadd_rn(acc[t], row_sse16<KIND, TEAM16>(make_uint4(pr[0], pr[1], pr[2], pr[3]),
                                                                   make_uint4(pr[4], pr[5], pr[6], pr[7]), c6, scale_table, Qf));
            }
        }
    }
    const int64_t Kg = runs / TEAM16;
#pragma unroll
    for (int t = 0; t < GPT; ++t) {
        const int q = threadIdx.x + t * blockDim.x;
        if (q < runs && (q % TEAM16) == 0) part[(chunk * P + p) * Kg + q / TEAM16] = acc[t];
    }
}

// Orders per block, groups per block and threads per group for `chunks` chunks of K channels under P orders:
// the configuration with the shortest estimated schedule.  A group works through its share of the (chunk, order)
// pairs; a pair costs one unit per run of each lane, a chunk a quarter of a unit of staging per run (and a share
// touches one chunk more than it holds whole); an SM is taken to be saturated by 20 warps, fewer are
// proportionally slower.
struct GatherConfig {
    int opb = 0, groups = 0, group_threads = 0;
};
inline GatherConfig gather_config(int64_t chunks, int64_t K, int P, int sides, int sms) {
    GatherConfig best;
    double best_cost = 0.0;
    const int runs = static_cast<int>(K / 16);
    for (int per_lane = 1; per_lane <= 4; ++per_lane) {
        const int threads = static_cast<int>(pq_ceil_div(pq_ceil_div(runs, per_lane), 32)) * 32;
        if (threads > kGatherThreads) continue;
        for (int opb = 1; opb <= P; ++opb) {
            const int64_t subsets = pq_ceil_div(P, opb);
            for (int groups = 1; groups <= kMaxGroups && groups * threads <= kGatherThreads; ++groups) {
                if (gather_smem_bytes(K, opb, groups, sides) > kGatherSmemMax) break;
                const int64_t blocks = sms / subsets > 0 ? sms / subsets : 1;
                const double pairs = static_cast<double>(pq_ceil_div(chunks * opb, blocks * groups));
                const int warps = groups * threads / 32;
                const double cost = (pairs + 0.25 * (pairs / opb + 1.0)) * threads * groups * per_lane * (warps < 20 ? 20.0 / warps : 1.0);
                if (!best.groups || cost < best_cost) {
                    best_cost = cost;
                    best.opb = opb, best.groups = groups, best.group_threads = threads;
                }
            }
        }
        if (threads <= 32) break;
    }
    return best;
}

int sm_count() {
    int dev = 0, sms = 148;
    if (cudaGetDevice(&dev) == cudaSuccess) cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    return sms;
}

int chunk_threads(int64_t K) {
    const int64_t runs = K / 16;
    return static_cast<int>(runs >= kChunkThreads ? kChunkThreads : pq_ceil_div(runs, 32) * 32);
}
// Few (chunk, order) pairs: all blocks of the kernel for them resident at once.  One block per chunk and order / thread groups
// with tables, us with the fold, NVFP4: 37 x 3072 3 orders 12.6 / 21.5, 512 x 6400 3 orders 20.9 / 28.9, 4608 x 768 3 orders (864
// pairs) 20.4 / 27.5, 4608 x 6400 1 order (288) 36.3 / 63.9, 512 x 16384 3 orders (96) 37.7 / 48.4; past the line
// 4608 x 768 6 orders (1728) 29.2 / 25.9, 1357 x 6400 6 orders (510) 53.1 / 51.7, 512 x 16384 6 orders (192) 66.4 / 61.1,
// 4608 x 12288 8 orders 540 / 237.  704 threads of it per SM; above 8192 channels one block, by registers and shared memory.
bool chunk_kernel_serves(int64_t pairs, int64_t K) {
    return pairs <= static_cast<int64_t>(sm_count()) * (K > 2 * 16 * kChunkThreads ? 1 : 704 / chunk_threads(K));
}

template <typename PT, int PER_SLAB>
pq_status fold(const void *part, int64_t count, int64_t n, double *err, cudaStream_t st) {
    PQ_CUDA_OK((pq::launch_fold<PT, PER_SLAB, false>(static_cast<const PT *>(part), nullptr, count, n, err, nullptr, st)));
    return pq_launch_status();
}

// list, ts, identity, perms, chunks and weights of p are set by the caller.
template <int KIND, int TEAM>
pq_status launch_gather(GatherParams &p, int64_t K, int P, float Qf, float *part, cudaStream_t st) {
    const int weights = p.weights.lambda ? 1 : 0, sms = sm_count() - weights, sides = KIND == 0 && p.ts[1] ? 2 : 1;
    const GatherConfig cfg = gather_config(p.chunks, K, P, sides, sms);
    if (!cfg.groups) return PQ_ERR_SHAPE;
    p.K = static_cast<int>(K), p.P = P, p.Qf = Qf, p.part = part;
    p.opb = cfg.opb, p.groups = cfg.groups, p.group_threads = cfg.group_threads;
    const int64_t subsets = pq_ceil_div(P, cfg.opb), share = sms / subsets > 0 ? sms / subsets : 1;
    const int64_t want = pq_ceil_div(static_cast<int64_t>(p.chunks) * cfg.opb, cfg.groups);
    const int64_t blocks = want < share ? want : share;
    const int64_t shares = blocks * cfg.groups;
    p.full = static_cast<int>(p.chunks / shares), p.split = static_cast<uint32_t>(p.chunks % shares);
    for (int last = 0; last < 2; ++last) {
        const int64_t orders = last ? P - (subsets - 1) * cfg.opb : cfg.opb;
        const int64_t pairs = p.split * orders;
        p.base[last] = static_cast<uint32_t>(pairs / shares), p.rem[last] = static_cast<uint32_t>(pairs % shares);
    }
    const size_t smem = gather_smem_bytes(K, cfg.opb, cfg.groups, sides);
    auto kern = group_error_gather<KIND, TEAM / 2>;
    PQ_CUDA_OK(pq::allow_smem(kern, smem, kGatherSmemMax));
    p.blocks = static_cast<int>(blocks);
    PQ_CUDA_OK(pq::launch_dependent(kern, dim3(static_cast<unsigned>(blocks * subsets + weights)),
                                    dim3(static_cast<unsigned>(cfg.groups * cfg.group_threads)), smem, st, p));
    return pq_launch_status();
}

template <int KIND, int TEAM>  // TEAM = group / 8
pq_status launch(const uint16_t *T, int64_t rows, int64_t K, int64_t ld, const float *ts, float Qf,
                 const int32_t *perms, int P, void *ws, double *err, cudaStream_t st) {
    const int64_t chunks = pq_ceil_div(rows, PQ_CHUNK_ROWS), slabs = pq_ceil_div(rows, PQ_SLAB_ROWS);
    const int64_t Kg = K / (8 * TEAM);
    if (!perms) {
        dim3 grid(static_cast<unsigned>(slabs), static_cast<unsigned>(pq_ceil_div(K / 16, kDirectRuns)));
        group_error_direct<KIND, TEAM / 2><<<grid, kDirectThreads, 0, st>>>(T, rows, K, ld, ts, Qf, static_cast<double *>(ws));
        if (pq_launch_status() != PQ_OK) return PQ_ERR_CUDA;
        return fold<double, 1>(ws, slabs, Kg, err, st);
    }
    if (chunk_kernel_serves(chunks * P, K)) {
        const int runs = static_cast<int>(K >> 4), threads = chunk_threads(K);
        const size_t smem = static_cast<size_t>(K) * 8;  // four rows, interleaved per channel
        const dim3 grid(static_cast<unsigned>(chunks), static_cast<unsigned>(P));
        auto kern = runs <= threads       ? group_error_chunk<KIND, TEAM / 2, 1>
                    : runs <= 2 * threads ? group_error_chunk<KIND, TEAM / 2, 2>
                                          : group_error_chunk<KIND, TEAM / 2, kChunkMaxGpt>;
        PQ_CUDA_OK(pq::allow_smem(kern, smem, kErrMaxK * 8, 4096));
        kern<<<grid, threads, smem, st>>>(T, rows, K, ld, ts, Qf, perms, P, static_cast<float *>(ws));
        if (pq_launch_status() != PQ_OK) return PQ_ERR_CUDA;
        return fold<float, kSlabChunks>(ws, chunks, static_cast<int64_t>(P) * Kg, err, st);
    }
    GatherParams p;
    p.list.add(T, rows, ld);
    p.list.n_x = 1;
    p.ts[0] = ts, p.ts[1] = nullptr, p.identity = 0, p.perms = perms, p.chunks = static_cast<int>(chunks);
    p.weights = PqErrorWeights{};
    if (launch_gather<KIND, TEAM>(p, K, P, Qf, static_cast<float *>(ws), st) != PQ_OK) return PQ_ERR_CUDA;
    return fold<float, kSlabChunks>(ws, chunks, static_cast<int64_t>(P) * Kg, err, st);
}

// f(KIND, TEAM) for a format that has been checked.
template <typename F>
pq_status dispatch_format(pq_format fmt, F &&f) {
    using std::integral_constant;
    if (fmt.kind == 0) return f(integral_constant<int, 0>{}, integral_constant<int, 2>{});
    switch (fmt.group) {
        case 16: return f(integral_constant<int, 1>{}, integral_constant<int, 2>{});
        case 32: return f(integral_constant<int, 1>{}, integral_constant<int, 4>{});
        case 64: return f(integral_constant<int, 1>{}, integral_constant<int, 8>{});
        case 128: return f(integral_constant<int, 1>{}, integral_constant<int, 16>{});
        default: return f(integral_constant<int, 1>{}, integral_constant<int, 32>{});  // 256: a whole warp per group
    }
}
float level_max(pq_format fmt) { return fmt.kind == 1 ? static_cast<float>((1 << (fmt.bits - 1)) - 1) : 0.0f; }

}  // namespace

extern "C" pq_status pq_group_error(const void *T, int64_t rows, int64_t K, int64_t ld, pq_format fmt,
                                    const float *ts, const int32_t *perms, int P, double *err, void *ws,
                                    size_t ws_bytes, void *stream) {
    PQ_REQUIRE(T && err, PQ_ERR_NULL);
    PQ_REQUIRE(fmt.kind == 0 || fmt.kind == 1, PQ_ERR_FORMAT);
    const int group = fmt.kind == 0 ? 16 : fmt.group;
    if (fmt.kind == 1) {
        PQ_REQUIRE(fmt.bits >= 2 && fmt.bits <= 8, PQ_ERR_FORMAT);
        PQ_REQUIRE(group == 16 || group == 32 || group == 64 || group == 128 || group == 256, PQ_ERR_FORMAT);
    } else {
        PQ_REQUIRE(ts, PQ_ERR_NULL);
    }
    PQ_REQUIRE(rows > 0 && K > 0 && K % group == 0 && K <= kErrMaxK && ld >= K, PQ_ERR_SHAPE);
    PQ_REQUIRE(P >= 1 && P <= 8 && (perms || P == 1), PQ_ERR_SHAPE);
    PQ_REQUIRE(pq_aligned16(T) && ld % 8 == 0, PQ_ERR_ALIGN);
    const int64_t chunks = pq_ceil_div(rows, PQ_CHUNK_ROWS);
    PQ_REQUIRE(chunks < (1ll << 31), PQ_ERR_SHAPE);
    PQ_REQUIRE(ws && ws_bytes >= pq_workspace_bytes(PQ_OP_GROUP_ERROR, rows, K, 0, P), PQ_ERR_WORKSPACE);
    PQ_REQUIRE(pq_aligned256(ws), PQ_ERR_ALIGN);

    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const uint16_t *t = static_cast<const uint16_t *>(T);
    return dispatch_format(fmt, [&](auto kind, auto team) {
        return launch<decltype(kind)::value, decltype(team)::value>(t, rows, K, ld, ts, level_max(fmt), perms, P, ws, err, st);
    });
}

pq_status pq_errors_on_list(const PqTensorList &list, int64_t K, pq_format fmt, const float *const (&ts)[2], const int32_t *perms,
                            int P, const PqSide (&sides)[2], const PqErrorWeights &weights, void *ws, cudaStream_t st) {
    GatherParams p;
    p.list = list;
    p.ts[0] = ts[0], p.ts[1] = ts[1], p.identity = 1, p.perms = perms, p.chunks = list.slabs() * kSlabChunks;
    p.weights = weights;
    float *part = static_cast<float *>(ws);
    const pq_status rc = dispatch_format(fmt, [&](auto kind, auto team) {
        return launch_gather<decltype(kind)::value, decltype(team)::value>(p, K, P + 1, level_max(fmt), part, st);
    });
    if (rc != PQ_OK) return rc;
    const int64_t n = (P + 1) * (K / (fmt.kind == 0 ? 16 : fmt.group));
    const int64_t cx = static_cast<int64_t>(list.slabs_x()) * kSlabChunks, cw = p.chunks - cx;
    const pq::FoldRange rx{part, nullptr, cx, sides[0].total, nullptr, sides[0].from_zero};
    const pq::FoldRange rw{part + cx * n, nullptr, cw, sides[1].total, nullptr, sides[1].from_zero};
    PQ_CUDA_OK((pq::launch_fold<float, kSlabChunks, false>(sides[0].total ? rx : rw, sides[0].total ? rw : pq::FoldRange{}, n, st)));
    return pq_launch_status();
}

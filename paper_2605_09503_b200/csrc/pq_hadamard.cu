// PermuQuant-H producer (App. D): Hadamard transform of every token row, the channel reordering applied
// when the transformed row is read back (x H P: only the order in which transformed channels are
// consumed changes), and the NVFP4 quantizer of the runtime path (Eq. 8) attached, so the transformed
// activations never make a round trip through HBM.
//
// The transform.  K = m * 2^n with m = 1 or m = 12; y = x (H_m (x) H_{2^n}) / sqrt(K): with channel
// i = a * 2^n + b the matrix entry is H_m[a][a'] * (-1)^popcount(b & b').  H_12 is Paley's matrix for
// q = 11 (I + S, S skew, built from the quadratic character modulo 11).  All arithmetic is IEEE fp32 in
// a fixed order: the 12 segments are combined first (terms added one by one in ascending segment), then
// the butterflies of the fast Walsh-Hadamard transform run inside each segment with strides 1, 2, 4, ...,
// then one multiplication by fl(1 / sqrt(K)).  Within one stride the butterflies are independent, so how
// they are spread over threads does not change a bit of the result.
//
// Four kernels.  Widths of 768, 1024, 1536, 2048, 3072, 4096, 6144 and 12288 have rows that divide evenly over the lanes of
// one, two or four warps, which then carry a row through all phases by themselves (second half of this file).
// Every other width goes through the kernel described here.
// Work distribution.  A thread block keeps up to 8 rows as K fp32 values each in shared memory and walks
// over batches of rows (persistent grid):
//   phase 1  a thread takes one octet position of one row: m 16-byte loads (the same octet of every
//            segment), the segment combination and the strides 1, 2, 4 in registers, on PAIRS of
//            neighbouring channels in packed f32x2 instructions (two IEEE results per issue slot);
//   phase 2  the remaining strides in one to three passes over shared memory: a thread owns one channel
//            pair position and 2^LOG values of it at the pass's strides (up to 32 packed registers),
//            addressed through eight base pointers and immediate offsets;
//   phase 3  a lane takes one 16-channel group of the OUTPUT order: its 16 read-out positions (the
//            permutation with the shared-memory swizzle applied, as 16-bit byte offsets, prepared once
//            per block) come as two 16-byte loads, the values are gathered from shared memory and
//            quantized like pq_quant_act_nvfp4 (coalesced code stores, four scale bytes merged into a
//            word by shuffles).
// Shared-memory swizzle of a row image (fp32 index i): bits 3-4 are XORed with the two bits just above
// the first pass's window and bit 2 with bit 5.  The first spreads the strided accesses of phase 2 over
// all banks, the second lets the eight lanes of a 16-byte store wavefront of phase 1 hit distinct banks.
#include <algorithm>
#include <type_traits>
#include <utility>

#include "pq_common.cuh"

namespace {

#ifndef PQ_HAD_ROWS
#define PQ_HAD_ROWS 8
#endif
constexpr int kMaxRows = PQ_HAD_ROWS;   // rows per block (fewer when a row needs more than 24 KB of shared memory)
constexpr int kThreads = 32 * kMaxRows;
#ifndef PQ_HAD_BLOCKS
#define PQ_HAD_BLOCKS (512 / (32 * PQ_HAD_ROWS))
#endif
constexpr int kBlocksPerSm = PQ_HAD_BLOCKS;
constexpr size_t kSmemBudget = 192 * 1024;
constexpr int64_t kMaxK = 16384;

// ---- Paley's Hadamard matrix of order 12 (compile-time)
constexpr int quadratic_character_11(int r) {
    r = ((r % 11) + 11) % 11;
    if (r == 0) return 0;
    for (int t = 1; t < 11; ++t)
        if ((t * t) % 11 == r) return 1;
    return -1;
}
constexpr int paley12(int i, int j) {
    return i == j ? 1 : i == 0 ? 1 : j == 0 ? -1 : quadratic_character_11(i - j);
}
template <int I, int J>
struct Paley12 {
    static constexpr bool plus = paley12(I, J) > 0;
};

// ---- packed fp32 pairs
__device__ __forceinline__ uint64_t pack2(float lo, float hi) {
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ void unpack2(uint64_t v, float &lo, float &hi) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b) {
    uint64_t r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ uint64_t sub2(uint64_t a, uint64_t b) {
    uint64_t r;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ uint64_t mul2(uint64_t a, uint64_t b) {
    uint64_t r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
// (x, y) -> (x + y, x - y)
__device__ __forceinline__ uint64_t butterfly_in_pair(uint64_t v) {
    float x, y;
    unpack2(v, x, y);
    return pack2(__fadd_rn(x, y), __fsub_rn(x, y));
}

// fp32 index of a channel inside its row's shared-memory image
__device__ __forceinline__ int swz(int idx, int sw) { return idx ^ (((idx >> sw) & 3) << 3) ^ (((idx >> 5) & 1) << 2); }

struct HadParams {
    const uint16_t *X;
    int64_t rows, rows_pad, ld;
    int K, m, n;            // K = m * 2^n
    int log[3];             // bits taken by the passes of phase 2 (0 = no such pass)
    int sw;                 // swizzle source bit
    int rows_per_block;
    float scale;            // fl(1 / sqrt(K))
    const int32_t *perm;
    const float *ts;
    uint8_t *codes, *sf;
    uint16_t *y_out;
};

// ---- phase 1: one octet position of one row
template <int AP, int A>
__device__ __forceinline__ void combine_segments(uint64_t (&acc)[4], const uint64_t (&in)[12][4]) {
    if constexpr (A < 12) {
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            if constexpr (Paley12<A, AP>::plus) acc[e] = add2(acc[e], in[A][e]);
            else acc[e] = sub2(acc[e], in[A][e]);
        }
        combine_segments<AP, A + 1>(acc, in);
    }
}

// strides 1, 2, 4 on the four channel pairs of an octet, then the octet goes to shared memory
__device__ __forceinline__ void finish_octet(uint64_t (&v)[4], float *row_s, int idx, int sw) {
#pragma unroll
    for (int e = 0; e < 4; ++e) v[e] = butterfly_in_pair(v[e]);
    const uint64_t a0 = add2(v[0], v[1]), a1 = sub2(v[0], v[1]), a2 = add2(v[2], v[3]), a3 = sub2(v[2], v[3]);
    const uint64_t b0 = add2(a0, a2), b1 = add2(a1, a3), b2 = sub2(a0, a2), b3 = sub2(a1, a3);
    // two 16-byte stores; the swizzle swaps the halves of every other group of four octets, which keeps
    // the eight lanes of a store wavefront on distinct banks
    const int half = (idx >> 5) & 1;
    ulonglong2 *dst = reinterpret_cast<ulonglong2 *>(row_s + (idx ^ (((idx >> sw) & 3) << 3)));
    dst[half] = make_ulonglong2(b0, b1);
    dst[half ^ 1] = make_ulonglong2(b2, b3);
}

__device__ __forceinline__ void unpack_pairs(const uint4 &raw, uint64_t (&v)[4]) {
    const uint32_t w[4] = {raw.x, raw.y, raw.z, raw.w};
#pragma unroll
    for (int e = 0; e < 4; ++e) v[e] = pack2(__uint_as_float(w[e] << 16), __uint_as_float(w[e] & 0xFFFF0000u));
}

template <int AP>
__device__ __forceinline__ void column_12(const uint64_t (&in)[12][4], float *row_s, int seg, int o, int sw) {
    uint64_t acc[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) acc[e] = in[0][e];  // the first row of the matrix is all ones
    combine_segments<AP, 1>(acc, in);
    finish_octet(acc, row_s, AP * seg + o * 8, sw);
}
template <int... APs>
__device__ __forceinline__ void all_columns_12(std::integer_sequence<int, APs...>, const uint64_t (&in)[12][4], float *row_s,
                                               int seg, int o, int sw) {
    (column_12<APs>(in, row_s, seg, o, sw), ...);
}

// ---- phase 2: 2^LOG values of one channel-pair position, strides 2^S ... 2^(S+LOG-1)
// The swizzle reads two bits and bit 5 and writes bits 2-4; of the window's bits only the lowest three can
// be among those, so the address of value j is that of value j % 8 plus an immediate.
template <int LOG>
__device__ __forceinline__ void pass_item(float *row_s, int base, int S, int sw, bool last, uint64_t scale2) {
    constexpr int N = 1 << LOG, NB = N < 8 ? N : 8;
    uint64_t *slot[NB];
#pragma unroll
    for (int m = 0; m < NB; ++m) slot[m] = reinterpret_cast<uint64_t *>(row_s + swz(base + (m << S), sw));
    const int step = 4 << S;  // 64-bit words between value j and value j + 8
    uint64_t v[N];
#pragma unroll
    for (int j = 0; j < N; ++j) v[j] = slot[j % NB][(j / NB) * step];
#pragma unroll
    for (int l = 0; l < LOG; ++l) {
#pragma unroll
        for (int j = 0; j < N; ++j) {
            if ((j >> l) & 1) continue;
            const uint64_t p = v[j], q = v[j | (1 << l)];
            v[j] = add2(p, q);
            v[j | (1 << l)] = sub2(p, q);
        }
    }
    if (last) {
#pragma unroll
        for (int j = 0; j < N; ++j) v[j] = mul2(v[j], scale2);
    }
#pragma unroll
    for (int j = 0; j < N; ++j) slot[j % NB][(j / NB) * step] = v[j];
}

// One pass over the rows of the block: items = rows x (K / 2) channel pairs / 2^LOG.
template <int THREADS>
__device__ __forceinline__ void run_pass(float *smem, const HadParams &p, int nrows, int S, int LOG, bool last) {
    const uint64_t scale2 = pack2(p.scale, p.scale);
    const int per_row = (p.K >> 1) >> LOG;  // items per row
    const int low_mask = (1 << (S - 1)) - 1;  // pair-index bits below the window (a pair index is channel >> 1)
    for (int u = threadIdx.x; u < nrows * per_row; u += THREADS) {
        const int r = u / per_row, w = u - r * per_row;
        // w enumerates the pair positions with the window bits removed: low part below the window, the rest above
        const int pair = (w & low_mask) | ((w & ~low_mask) << LOG);
        float *row_s = smem + static_cast<size_t>(r) * p.K;
        const int base = pair << 1;
        switch (LOG) {
            case 1: pass_item<1>(row_s, base, S, p.sw, last, scale2); break;
            case 2: pass_item<2>(row_s, base, S, p.sw, last, scale2); break;
            case 3: pass_item<3>(row_s, base, S, p.sw, last, scale2); break;
            case 4: pass_item<4>(row_s, base, S, p.sw, last, scale2); break;
            default: pass_item<5>(row_s, base, S, p.sw, last, scale2); break;
        }
    }
}

// THREADS: 256 (two blocks per SM) while a block holds eight rows; 512 (one block) when rows wider than 6144
// channels leave room for fewer, so that an SM still has 16 warps at work on them
template <int SF_LAYOUT, int THREADS>
__global__ void __launch_bounds__(THREADS, 512 / THREADS) hadamard_quant_kernel(const HadParams p) {
    extern __shared__ __align__(16) float had_smem[];  // [rows_per_block][K] fp32, then K 16-bit read-out offsets
    const int kRows = p.rows_per_block;
    uint16_t *offset_s = reinterpret_cast<uint16_t *>(had_smem + static_cast<size_t>(kRows) * p.K);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int seg = p.K / p.m, octs = seg >> 3;
    const int gpr = p.K >> 4, chunks = (gpr + 31) >> 5;  // output groups per row, in chunks of one per lane
    const int64_t batches = (p.rows_pad + kRows - 1) / kRows;
    pq::wait_for_prior_grid();
    pq::dependents_may_launch();

    // where each output position reads its channel in a row's (swizzled) shared-memory image, as a byte
    // offset: the same for every row, so it is worked out once per block (K <= 16384: 16 bits)
    for (int j = threadIdx.x; j < p.K; j += THREADS)
        offset_s[j] = static_cast<uint16_t>(swz(p.perm ? p.perm[j] : j, p.sw) << 2);
    const pq::Nvfp4Scaler scaler = pq::nvfp4_scaler(p.codes ? __ldca(p.ts) : 1.0f);

    for (int64_t batch = blockIdx.x; batch < batches; batch += gridDim.x) {
        const int64_t row0 = batch * kRows;
        const int nrows = static_cast<int>(min(static_cast<int64_t>(kRows), max(static_cast<int64_t>(0), p.rows - row0)));
        __syncthreads();  // the previous batch has been read out (and the offsets are in place)

        // ---- phase 1
        for (int u = threadIdx.x; u < nrows * octs; u += THREADS) {
            const int r = u / octs, o = u - r * octs;
            const uint16_t *src = p.X + (row0 + r) * p.ld + o * 8;
            float *row_s = had_smem + static_cast<size_t>(r) * p.K;
            if (p.m == 12) {
                uint64_t in[12][4];
#pragma unroll
                for (int a = 0; a < 12; ++a) unpack_pairs(__ldcs(reinterpret_cast<const uint4 *>(src + a * seg)), in[a]);
                all_columns_12(std::make_integer_sequence<int, 12>{}, in, row_s, seg, o, p.sw);
            } else {
                uint64_t v[4];
                unpack_pairs(__ldcs(reinterpret_cast<const uint4 *>(src)), v);
                finish_octet(v, row_s, o * 8, p.sw);
            }
        }
        __syncthreads();
        // ---- phase 2 (the scaling rides on the last pass; without any pass it is applied in phase 3)
        int start = 3;
#pragma unroll 1
        for (int k = 0; k < 3 && p.log[k]; ++k) {
            run_pass<THREADS>(had_smem, p, nrows, start, p.log[k], k == 2 || p.log[k + 1] == 0);
            start += p.log[k];
            __syncthreads();
        }

        // ---- phase 3: a warp takes a chunk of 32 output groups of TWO rows at a time, one group per lane:
        // the read-out offsets are fetched once for both rows and the two quantizer chains interleave
        const int rows_here = static_cast<int>(min(static_cast<int64_t>(kRows), p.rows_pad - row0));
        const int row_pairs = (rows_here + 1) >> 1;
        auto read_out = [&](auto fast) {
            for (int c = warp; c < row_pairs * chunks; c += THREADS / 32) {
                const int rp = c / chunks, g = (c - rp * chunks) * 32 + lane;
                const bool have = g < gpr;
                uint32_t iw[8];
                if (have) {
                    const uint4 i0 = reinterpret_cast<const uint4 *>(offset_s)[2 * g], i1 = reinterpret_cast<const uint4 *>(offset_s)[2 * g + 1];
                    iw[0] = i0.x, iw[1] = i0.y, iw[2] = i0.z, iw[3] = i0.w, iw[4] = i1.x, iw[5] = i1.y, iw[6] = i1.z, iw[7] = i1.w;
                } else {
#pragma unroll
                    for (int j = 0; j < 8; ++j) iw[j] = 0;
                }
                float out[2][16];
                bool live[2], present[2];
                int64_t row[2];
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int r = 2 * rp + h;
                    row[h] = row0 + r;
                    present[h] = r < rows_here;
                    // the second row of the last pair does not exist when the block holds an odd number of rows (three
                    // at 16384 channels): that index is the first row of the NEXT batch and lies past this image
                    live[h] = present[h] && row[h] < p.rows;
                    const char *row_b = reinterpret_cast<const char *>(had_smem + static_cast<size_t>(r) * p.K);
#pragma unroll
                    for (int j = 0; j < 16; ++j) out[h][j] = 0.0f;
                    if (live[h] && have) {
#pragma unroll
                        for (int j = 0; j < 8; ++j) {
                            out[h][2 * j] = *reinterpret_cast<const float *>(row_b + (iw[j] & 0xFFFFu));
                            out[h][2 * j + 1] = *reinterpret_cast<const float *>(row_b + (iw[j] >> 16));
                        }
                        if (!p.log[0]) {  // no pass of phase 2 carried the scaling
#pragma unroll
                            for (int j = 0; j < 16; ++j) out[h][j] = __fmul_rn(out[h][j], p.scale);
                        }
                        if (p.y_out) {
                            uint32_t yw[8];
#pragma unroll
                            for (int j = 0; j < 8; ++j)
                                yw[j] = __bfloat16_as_ushort(__float2bfloat16_rn(out[h][2 * j])) |
                                        (static_cast<uint32_t>(__bfloat16_as_ushort(__float2bfloat16_rn(out[h][2 * j + 1]))) << 16);
                            uint4 *ydst = reinterpret_cast<uint4 *>(p.y_out + row[h] * p.K) + 2 * g;
                            ydst[0] = make_uint4(yw[0], yw[1], yw[2], yw[3]);
                            ydst[1] = make_uint4(yw[4], yw[5], yw[6], yw[7]);
                        }
                    }
                }
                if (!p.codes) continue;
                uint32_t sf8[2];
                float rcp[2];
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    float amax = 0.0f;
#pragma unroll
                    for (int j = 0; j < 16; ++j) amax = fmaxf(amax, fabsf(out[h][j]));
                    pq::nvfp4_scale<decltype(fast)::value>(amax, scaler, sf8[h], rcp[h]);
                }
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    if (live[h] && have) {
                        const uint64_t rcp2 = pack2(rcp[h], rcp[h]);
                        float ylo[8], yhi[8];
#pragma unroll
                        for (int j = 0; j < 4; ++j) {
                            unpack2(mul2(pack2(out[h][2 * j], out[h][2 * j + 1]), rcp2), ylo[2 * j], ylo[2 * j + 1]);
                            unpack2(mul2(pack2(out[h][8 + 2 * j], out[h][9 + 2 * j]), rcp2), yhi[2 * j], yhi[2 * j + 1]);
                        }
                        *reinterpret_cast<uint2 *>(p.codes + row[h] * (p.K >> 1) + g * 8) =
                            make_uint2(pq::f32x8_to_e2m1(ylo), pq::f32x8_to_e2m1(yhi));
                    }
                    // scale bytes: four neighbouring groups sit in neighbouring lanes (padding rows write zeros)
                    uint32_t word = sf8[h];
                    word |= __shfl_down_sync(0xFFFFFFFFu, sf8[h], 1) << 8;
                    word |= __shfl_down_sync(0xFFFFFFFFu, sf8[h], 2) << 16;
                    word |= __shfl_down_sync(0xFFFFFFFFu, sf8[h], 3) << 24;
                    if (!have || !present[h]) continue;
                    if (SF_LAYOUT == PQ_SF_TCGEN05) {
                        if ((g & 3) == 0) *reinterpret_cast<uint32_t *>(p.sf + pq::sf_tc_offset(row[h], g, gpr >> 2)) = word;
                    } else if (live[h]) {
                        if ((gpr & 3) == 0) {
                            if ((g & 3) == 0) *reinterpret_cast<uint32_t *>(p.sf + row[h] * gpr + g) = word;
                        } else {
                            p.sf[row[h] * gpr + g] = static_cast<uint8_t>(sf8[h]);
                        }
                    }
                }
            }
        };
        if (scaler.fast) read_out(std::true_type{});
        else read_out(std::false_type{});
    }
}

// ---- one warp per row (K = 12 * 256), or per two or four rows (12 * 128, 12 * 64)
// 32 octet positions of twelve segments are exactly one phase-1 item per lane, so a warp can carry its row(s)
// through all phases by itself: no block barrier, and the phases of the SM's sixteen warps, which load
// different units (fp32 pipe, shared memory, conversions), run beside each other.  The block version above
// holds its rows in step, and its second pass has 384 items for 256 threads: 32.6 us at 4608 x 3072 where this
// takes 23.5, 18.5 / 14.2 at 4608 x 1536, 26.7 / 13.8 at 9216 x 768, 11.3 / 8.8 at 512 x 3072.  The warp's 12 KB image stays conflict-free: octet b of segment a lies
// at octet b ^ (a & 3) (the strided column accesses of phase 2: four segments per half warp), its 16-byte halves
// swapped by bit 2 of b (the stores of phase 1).
constexpr int kRowWarps = 8;            // per block; two blocks per SM at 128 registers
constexpr int kRowImage = 3072;         // fp32 values per warp

template <int N>
__device__ __forceinline__ int row_octet(int a, int b) {  // where octet b of segment a lies inside its row's image
    return (a << N) + ((b ^ ((N > 8 ? b >> 3 : a) & 3)) << 3);
}
template <int N>
__device__ __forceinline__ int row_image_index(int channel) {  // of a channel inside its row's image
    const int a = channel >> N, b = (channel & ((1 << N) - 1)) >> 3, e = channel & 7;
    return row_octet<N>(a, b) + (e ^ (((b >> 2) & 1) << 2));
}

// The butterflies of NV values (of one channel, or of two neighbouring channels) in ascending stride.
template <int NV, typename T>
__device__ __forceinline__ void column_butterflies(T (&v)[NV]) {
#pragma unroll
    for (int l = 1; l < NV; l <<= 1) {
#pragma unroll
        for (int j = 0; j < NV; ++j) {
            if (j & l) continue;
            const T p = v[j], q = v[j | l];
            if constexpr (sizeof(T) == 8) {
                v[j] = add2(p, q);
                v[j | l] = sub2(p, q);
            } else {
                v[j] = __fadd_rn(p, q);
                v[j | l] = __fsub_rn(p, q);
            }
        }
    }
}
template <typename T>
__device__ __forceinline__ T column_scaled(T v, float scale) {
    if constexpr (sizeof(T) == 8) return mul2(v, pack2(scale, scale));
    else return __fmul_rn(v, scale);
}

// 2^LOG values of one column (of one channel, or of two neighbouring channels) at the octet stride, in place; LAST: and the scaling.
template <int LOG, typename T, bool LAST = true>
__device__ __forceinline__ void column_pass(float *image, int a_base, int s, int e, float scale) {
    constexpr int NV = 1 << LOG;
    T *slot[8];
#pragma unroll
    for (int b = 0; b < 8; ++b)
        slot[b] = reinterpret_cast<T *>(image + a_base + ((b ^ s) << 3) + (e ^ ((b >> 2) << 2)));
    constexpr int kStep = 64 * sizeof(float) / sizeof(T);  // eight octets further
    T v[NV];
#pragma unroll
    for (int b = 0; b < NV; ++b) v[b] = slot[b & 7][(b >> 3) * kStep];
    column_butterflies(v);
#pragma unroll
    for (int b = 0; b < NV; ++b) slot[b & 7][(b >> 3) * kStep] = LAST ? column_scaled(v[b], scale) : v[b];
}

// Column a' of the order-12 combination for one half of an octet (two channel pairs) and strides 1, 2.  The first half
// waits in the image; the second takes stride 4 with it and writes both.  Half an octet at a time keeps the inputs in
// 48 registers: with the whole octet (96) the compiler spilled 300 bytes per thread at 128 registers.
template <int AP, int A>
__device__ __forceinline__ void combine_segments_half(uint64_t (&acc)[2], const uint64_t (&in)[12][2]) {
    if constexpr (A < 12) {
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            if constexpr (Paley12<A, AP>::plus) acc[e] = add2(acc[e], in[A][e]);
            else acc[e] = sub2(acc[e], in[A][e]);
        }
        combine_segments_half<AP, A + 1>(acc, in);
    }
}
template <int N, int HALF, int AP>
__device__ __forceinline__ void row_column_12(const uint64_t (&in)[12][2], float *row_s, int b) {
    uint64_t v[2] = {in[0][0], in[0][1]};  // the first row of the matrix is all ones
    combine_segments_half<AP, 1>(v, in);
#pragma unroll
    for (int e = 0; e < 2; ++e) v[e] = butterfly_in_pair(v[e]);
    const uint64_t c0 = add2(v[0], v[1]), c1 = sub2(v[0], v[1]);
    const int half = (b >> 2) & 1;
    // row_octet<N>(AP, b) written out: through the call the warp-per-row kernel spilled more (23.8 against 23.1 us)
    ulonglong2 *dst = reinterpret_cast<ulonglong2 *>(row_s + (AP << N) + ((b ^ (N > 8 ? (b >> 3) & 3 : AP & 3)) << 3));
    if (HALF == 0) {
        dst[half] = make_ulonglong2(c0, c1);
    } else {
        const ulonglong2 f = dst[half];
        dst[half] = make_ulonglong2(add2(f.x, c0), add2(f.y, c1));
        dst[half ^ 1] = make_ulonglong2(sub2(f.x, c0), sub2(f.y, c1));
    }
}
template <int N, int HALF, int... APs>
__device__ __forceinline__ void row_columns_12(std::integer_sequence<int, APs...>, const uint4 (&raw)[12], float *row_s, int b) {
    uint64_t in[12][2];
#pragma unroll
    for (int a = 0; a < 12; ++a) {
        const uint32_t w0 = HALF ? raw[a].z : raw[a].x, w1 = HALF ? raw[a].w : raw[a].y;
        in[a][0] = pack2(__uint_as_float(w0 << 16), __uint_as_float(w0 & 0xFFFF0000u));
        in[a][1] = pack2(__uint_as_float(w1 << 16), __uint_as_float(w1 & 0xFFFF0000u));
    }
    (row_column_12<N, HALF, APs>(in, row_s, b), ...);
}

// The strides above a window of eight octets (segments of more than 256 channels): 2^LOG values, eight octets apart.
template <int LOG>
__device__ __forceinline__ void high_column_pass(float *segment, int k, int e, float scale) {
    constexpr int NV = 1 << LOG;
    uint64_t *slot[4];
#pragma unroll
    for (int j = 0; j < 4; ++j)
        slot[j] = reinterpret_cast<uint64_t *>(segment + ((k ^ j) << 3) + (e ^ ((k >> 2) << 2)));
    uint64_t v[NV];
#pragma unroll
    for (int j = 0; j < NV; ++j) v[j] = slot[j & 3][j * 32];
    column_butterflies(v);
#pragma unroll
    for (int j = 0; j < NV; ++j) slot[j & 3][j * 32] = column_scaled(v[j], scale);
}

// Phase 3 of a team of NT threads that holds ROWS transformed rows: one output group per lane.
template <int SF_LAYOUT, int K, int ROWS, int NT, bool FAST>
__device__ __forceinline__ void rows_read_out(const HadParams &p, const pq::Nvfp4Scaler &scaler, const float *image,
                                              const uint4 *offset4, int64_t row0, int tid) {
    constexpr int GPR = K / 16;
#pragma unroll 1
    for (int i = tid; i < ROWS * GPR; i += NT) {
        const int r = i / GPR, g = i - r * GPR;
        const int64_t row = row0 + r;
        const bool live = row < p.rows;
        float out[16];
#pragma unroll
        for (int j = 0; j < 16; ++j) out[j] = 0.0f;
        if (live) {
            const uint4 i0 = offset4[g], i1 = offset4[GPR + g];
            const uint32_t iw[8] = {i0.x, i0.y, i0.z, i0.w, i1.x, i1.y, i1.z, i1.w};
            const char *row_b = reinterpret_cast<const char *>(image + r * K);
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                out[2 * j] = *reinterpret_cast<const float *>(row_b + (iw[j] & 0xFFFFu));
                out[2 * j + 1] = *reinterpret_cast<const float *>(row_b + (iw[j] >> 16));
            }
            if (p.y_out) {
                uint32_t yw[8];
#pragma unroll
                for (int j = 0; j < 8; ++j)
                    yw[j] = __bfloat16_as_ushort(__float2bfloat16_rn(out[2 * j])) |
                            (static_cast<uint32_t>(__bfloat16_as_ushort(__float2bfloat16_rn(out[2 * j + 1]))) << 16);
                uint4 *ydst = reinterpret_cast<uint4 *>(p.y_out + row * K) + 2 * g;
                ydst[0] = make_uint4(yw[0], yw[1], yw[2], yw[3]);
                ydst[1] = make_uint4(yw[4], yw[5], yw[6], yw[7]);
            }
        }
        if (!p.codes) continue;
        float amax = 0.0f, rcp;
#pragma unroll
        for (int j = 0; j < 16; ++j) amax = fmaxf(amax, fabsf(out[j]));
        uint32_t sf8;
        pq::nvfp4_scale<FAST>(amax, scaler, sf8, rcp);
        if (live) {
            const uint64_t rcp2 = pack2(rcp, rcp);
            float ylo[8], yhi[8];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                unpack2(mul2(pack2(out[2 * j], out[2 * j + 1]), rcp2), ylo[2 * j], ylo[2 * j + 1]);
                unpack2(mul2(pack2(out[8 + 2 * j], out[9 + 2 * j]), rcp2), yhi[2 * j], yhi[2 * j + 1]);
            }
            *reinterpret_cast<uint2 *>(p.codes + row * (K / 2) + g * 8) = make_uint2(pq::f32x8_to_e2m1(ylo), pq::f32x8_to_e2m1(yhi));
        }
        // scale bytes: four neighbouring groups sit in neighbouring lanes (padding rows write zeros)
        uint32_t word = sf8;
        word |= __shfl_down_sync(0xFFFFFFFFu, sf8, 1) << 8;
        word |= __shfl_down_sync(0xFFFFFFFFu, sf8, 2) << 16;
        word |= __shfl_down_sync(0xFFFFFFFFu, sf8, 3) << 24;
        if ((g & 3) || row >= p.rows_pad) continue;
        if (SF_LAYOUT == PQ_SF_TCGEN05) *reinterpret_cast<uint32_t *>(p.sf + pq::sf_tc_offset(row, g, GPR >> 2)) = word;
        else if (live) *reinterpret_cast<uint32_t *>(p.sf + row * GPR + g) = word;
    }
}

template <int SF_LAYOUT, int N>
__global__ void __launch_bounds__(32 * kRowWarps, 2) hadamard_quant_rows_kernel(const HadParams p) {
    constexpr int SEG = 1 << N, K = 12 * SEG, OCTS = SEG / 8, RPW = 32 / OCTS, LOG = N - 3;
    extern __shared__ __align__(16) float had_smem[];  // [warps][3072] fp32, then K 16-bit read-out offsets in two planes
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    float *image = had_smem + warp * kRowImage;
    uint16_t *offset_s = reinterpret_cast<uint16_t *>(had_smem + kRowWarps * kRowImage);
    const uint4 *offset4 = reinterpret_cast<const uint4 *>(offset_s);
    pq::wait_for_prior_grid();
    pq::dependents_may_launch();
    // byte offset of the channel each output position reads; positions 0-7 and 8-15 of a group in separate planes,
    // so that the lanes' 16-byte reads are adjacent
    for (int j = threadIdx.x; j < K; j += 32 * kRowWarps)
        offset_s[((j >> 3) & 1) * (K / 2) + (j >> 4) * 8 + (j & 7)] =
            static_cast<uint16_t>(row_image_index<N>(p.perm ? p.perm[j] : j) << 2);
    const pq::Nvfp4Scaler scaler = pq::nvfp4_scaler(p.codes ? __ldca(p.ts) : 1.0f);
    __syncthreads();

    // warps of different blocks first, so that few rows spread over all SMs
    const int64_t batches = (p.rows_pad + RPW - 1) / RPW, step = static_cast<int64_t>(gridDim.x) * kRowWarps;
    for (int64_t batch = static_cast<int64_t>(warp) * gridDim.x + blockIdx.x; batch < batches; batch += step) {
        const int64_t row0 = batch * RPW;
        if (row0 < p.rows) {
            // ---- phase 1: lane = (row, octet); rows past the end are zeros
            const int r = lane / OCTS, b = lane % OCTS;
            const uint16_t *src = p.X + (row0 + r) * p.ld + b * 8;
            const bool have = row0 + r < p.rows;
            uint4 raw[12];
#pragma unroll
            for (int a = 0; a < 12; ++a)
                raw[a] = have ? __ldcs(reinterpret_cast<const uint4 *>(src + a * SEG)) : make_uint4(0, 0, 0, 0);
            __syncwarp();  // the previous rows have been read out
            row_columns_12<N, 0>(std::make_integer_sequence<int, 12>{}, raw, image + r * K, b);
            row_columns_12<N, 1>(std::make_integer_sequence<int, 12>{}, raw, image + r * K, b);
            // the next rows of this warp, into L2 while the remaining phases run
            if (row0 + step * RPW + r < p.rows) {
#pragma unroll
                for (int a = 0; a < 12; ++a)
                    if ((b & 7) == 0) asm volatile("prefetch.global.L2 [%0];" ::"l"(src + step * RPW * p.ld + a * SEG));
            }
            __syncwarp();
            // ---- phase 2: the remaining strides, column by column; 48 pair columns per row
            if constexpr (N == 8) {
                // 48 pair columns for 32 lanes: 32 of them as pairs, the other 16 as 32 single columns
                column_pass<LOG, uint64_t>(image, (lane >> 2) << N, (lane >> 2) & 3, (lane & 3) * 2, p.scale);
                const int a = 8 + (lane >> 3);
                column_pass<LOG, float>(image, a << N, a & 3, lane & 7, p.scale);
            } else {
#pragma unroll 1
                for (int i = lane; i < 48 * RPW; i += 32) {
                    const int row = i / 48, c = i - row * 48, a = c >> 2;
                    column_pass<LOG, uint64_t>(image, row * K + (a << N), a & 3, (c & 3) * 2, p.scale);
                }
            }
            __syncwarp();
        }
        // through a lambda: with the two calls written directly the 768- and 1536-channel kernels spilled
        auto read_out = [&](auto fast) {
            rows_read_out<SF_LAYOUT, K, RPW, 32, decltype(fast)::value>(p, scaler, image, offset4, row0, lane);
        };
        if (scaler.fast) read_out(std::true_type{});
        else read_out(std::false_type{});
    }
}

// ---- two or four warps per row (K = 12 * 512, 12 * 1024)
// A team's lanes take one phase-1 item each, as above, and meet at a barrier of their own, so the teams of an SM stay
// out of step with each other.  4608 x 6144 49.2 us (99.8 with the block kernel, whose rows move in step), 4608 x 12288
// 92.6 (161.6), 300 x 6144 9.9 (25.6), 200 x 12288 10.6 (21.6); instruction issue and shared memory bound it, as above.  The strides above 4 take two passes: 8 octets side by side, then the rest.  The image
// XORs an octet's two low bits with the two bits above the first window, which keeps the column accesses of both
// passes (four neighbouring windows, four neighbouring octets per half warp) and the stores of phase 1 conflict-free.
// One block of sixteen warps per SM: eight or four images of 24 or 48 KB.
template <int SF_LAYOUT, int N>
__global__ void __launch_bounds__(512, 1) hadamard_quant_team_kernel(const HadParams p) {
    constexpr int SEG = 1 << N, K = 12 * SEG, NT = SEG / 8, TEAMS = 512 / NT, WINDOWS = SEG / 64;
    extern __shared__ __align__(16) float had_smem[];  // [teams][K] fp32, then K 16-bit read-out offsets in two planes
    const int team = threadIdx.x / NT, tid = threadIdx.x % NT;
    float *image = had_smem + team * K;
    uint16_t *offset_s = reinterpret_cast<uint16_t *>(had_smem + TEAMS * K);
    const uint4 *offset4 = reinterpret_cast<const uint4 *>(offset_s);
    pq::wait_for_prior_grid();
    pq::dependents_may_launch();
    for (int j = threadIdx.x; j < K; j += 512)
        offset_s[((j >> 3) & 1) * (K / 2) + (j >> 4) * 8 + (j & 7)] =
            static_cast<uint16_t>(row_image_index<N>(p.perm ? p.perm[j] : j) << 2);
    const pq::Nvfp4Scaler scaler = pq::nvfp4_scaler(p.codes ? __ldca(p.ts) : 1.0f);
    __syncthreads();
    auto team_sync = [&] { asm volatile("bar.sync %0, %1;" ::"r"(1 + team), "n"(NT) : "memory"); };

    const int64_t step = static_cast<int64_t>(gridDim.x) * TEAMS;
    for (int64_t row = static_cast<int64_t>(team) * gridDim.x + blockIdx.x; row < p.rows_pad; row += step) {
        if (row < p.rows) {
            const uint16_t *src = p.X + row * p.ld + tid * 8;
            uint4 raw[12];
#pragma unroll
            for (int a = 0; a < 12; ++a) raw[a] = __ldcs(reinterpret_cast<const uint4 *>(src + a * SEG));
            team_sync();  // the previous row has been read out
            row_columns_12<N, 0>(std::make_integer_sequence<int, 12>{}, raw, image, tid);
            row_columns_12<N, 1>(std::make_integer_sequence<int, 12>{}, raw, image, tid);
            if (row + step < p.rows && (tid & 7) == 0) {  // this team's next row, into L2
#pragma unroll
                for (int a = 0; a < 12; ++a) asm volatile("prefetch.global.L2 [%0];" ::"l"(src + step * p.ld + a * SEG));
            }
            team_sync();
#pragma unroll 2
            for (int i = tid; i < 48 * WINDOWS; i += NT) {
                const int w = (i >> 2) % WINDOWS, a = (i >> 2) / WINDOWS;
                column_pass<3, uint64_t, false>(image, (a << N) + (w << 6), w & 3, (i & 3) * 2, 0.0f);
            }
            team_sync();
#pragma unroll 1
            for (int i = tid; i < 12 * 32; i += NT)
                high_column_pass<N - 6>(image + ((i >> 5) << N), (i >> 2) & 7, (i & 3) * 2, p.scale);
            team_sync();
        }
        if (scaler.fast) rows_read_out<SF_LAYOUT, K, 1, NT, true>(p, scaler, image, offset4, row, tid);
        else rows_read_out<SF_LAYOUT, K, 1, NT, false>(p, scaler, image, offset4, row, tid);
    }
}

// ---- one warp per row (K = 2048, 4096) or per two rows (1024), without the order-12 factor
// A lane holds blocks of 2^P1 neighbouring channels (strides 1 ... 2^(P1-1) in registers), then columns of 2^P2 values,
// one per block: a single pass over shared memory, packed where a lane's columns come in pairs.  16-byte chunk q of
// block u lies at chunk q ^ (u & 7): the stores of phase 1 (eight blocks per wavefront) and the column accesses (one
// block per instruction) are conflict-free.  Against the block kernel: 4608 x 1024 8.1 us (16.4), 9000 x 2048 29.8 (55.1),
// 4608 x 4096 33.0 (81.4), 300 x 1024 4.3 (5.8), 300 x 4096 7.7 (16.5).
template <int P1>
__device__ __forceinline__ int pow2_image_index(int channel) {
    const int u = channel >> P1, c = channel & ((1 << P1) - 1);
    return (u << P1) + (((c >> 2) ^ (u & 7)) << 2) + (c & 3);
}
template <int P1, int P2, typename T>
__device__ __forceinline__ void pow2_column(float *row_s, int c, float scale) {
    constexpr int NV = 1 << P2, kStep = (8 << P1) * sizeof(float) / sizeof(T);
    T *slot[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) slot[j] = reinterpret_cast<T *>(row_s + (j << P1) + (((c >> 2) ^ j) << 2) + (c & 3));
    T v[NV];
#pragma unroll
    for (int j = 0; j < NV; ++j) v[j] = slot[j & 7][(j >> 3) * kStep];
    column_butterflies(v);
#pragma unroll
    for (int j = 0; j < NV; ++j) slot[j & 7][(j >> 3) * kStep] = column_scaled(v[j], scale);
}

// RPW rows per warp; WARPS per block: two blocks' images fit an SM
template <int SF_LAYOUT, int P1, int P2, int RPW, int WARPS>
__global__ void __launch_bounds__(32 * WARPS, 2) hadamard_quant_pow2_kernel(const HadParams p) {
    constexpr int K = 1 << (P1 + P2), BL = 1 << P1, NB = 1 << P2;
    extern __shared__ __align__(16) float had_smem[];  // [warps][RPW][K] fp32, then K 16-bit read-out offsets in two planes
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    float *image = had_smem + warp * (RPW * K);
    uint16_t *offset_s = reinterpret_cast<uint16_t *>(had_smem + WARPS * RPW * K);
    const uint4 *offset4 = reinterpret_cast<const uint4 *>(offset_s);
    pq::wait_for_prior_grid();
    pq::dependents_may_launch();
    for (int j = threadIdx.x; j < K; j += 32 * WARPS)
        offset_s[((j >> 3) & 1) * (K / 2) + (j >> 4) * 8 + (j & 7)] =
            static_cast<uint16_t>(pow2_image_index<P1>(p.perm ? p.perm[j] : j) << 2);
    const pq::Nvfp4Scaler scaler = pq::nvfp4_scaler(p.codes ? __ldca(p.ts) : 1.0f);
    __syncthreads();

    const int64_t batches = (p.rows_pad + RPW - 1) / RPW, step = static_cast<int64_t>(gridDim.x) * WARPS;
    for (int64_t batch = static_cast<int64_t>(warp) * gridDim.x + blockIdx.x; batch < batches; batch += step) {
        const int64_t row0 = batch * RPW;
        if (row0 < p.rows) {
            __syncwarp();  // the previous rows have been read out
#pragma unroll 1
            for (int i = lane; i < RPW * NB; i += 32) {
                const int r = i / NB, u = i % NB;
                const uint4 *src = reinterpret_cast<const uint4 *>(p.X + (row0 + r) * p.ld + u * BL);
                const bool have = row0 + r < p.rows;  // rows past the end are zeros
                uint4 raw[BL / 8];
#pragma unroll
                for (int q = 0; q < BL / 8; ++q) raw[q] = have ? __ldca(src + q) : make_uint4(0, 0, 0, 0);
                uint64_t v[BL / 2];
#pragma unroll
                for (int q = 0; q < BL / 8; ++q) {
                    uint64_t w[4];
                    unpack_pairs(raw[q], w);
#pragma unroll
                    for (int e = 0; e < 4; ++e) v[4 * q + e] = butterfly_in_pair(w[e]);
                }
                column_butterflies(v);
                ulonglong2 *dst = reinterpret_cast<ulonglong2 *>(image + r * K + u * BL);
#pragma unroll
                for (int q = 0; q < BL / 4; ++q) dst[q ^ (u & 7)] = make_ulonglong2(v[2 * q], v[2 * q + 1]);
            }
            __syncwarp();
            if constexpr (P2 == 5) {
                const int r = RPW == 2 ? lane >> 4 : 0, c = RPW == 2 ? lane & 15 : lane;
                pow2_column<P1, P2, uint64_t>(image + r * K, 2 * c, p.scale);
            } else {
#pragma unroll 1
                for (int c = lane; c < BL; c += 32) pow2_column<P1, P2, float>(image, c, p.scale);
            }
            __syncwarp();
        }
        if (scaler.fast) rows_read_out<SF_LAYOUT, K, RPW, 32, true>(p, scaler, image, offset4, row0, lane);
        else rows_read_out<SF_LAYOUT, K, RPW, 32, false>(p, scaler, image, offset4, row0, lane);
    }
}

// K = m * 2^n with m in {1, 12} and 2^n >= 8; returns false otherwise.
bool factor_width(int64_t K, int &m, int &n) {
    if (K <= 0) return false;
    int64_t seg;
    if ((K & (K - 1)) == 0) m = 1, seg = K;
    else if (K % 12 == 0 && ((K / 12) & (K / 12 - 1)) == 0) m = 12, seg = K / 12;
    else return false;
    n = 0;
    while ((static_cast<int64_t>(1) << n) < seg) ++n;
    return seg >= 8;
}

}  // namespace

extern "C" pq_status pq_hadamard_quant_nvfp4(const void *X, int64_t M, int64_t K, int64_t ld, const int32_t *perm,
                                             const float *ts_x, uint8_t *codes, uint8_t *sf, int sf_layout, void *y_out,
                                             void *stream) {
    PQ_REQUIRE(X, PQ_ERR_NULL);
    PQ_REQUIRE((codes == nullptr) == (sf == nullptr), PQ_ERR_NULL);
    PQ_REQUIRE(codes || y_out, PQ_ERR_NULL);
    PQ_REQUIRE(!codes || ts_x, PQ_ERR_NULL);
    PQ_REQUIRE(sf_layout == PQ_SF_LINEAR || sf_layout == PQ_SF_TCGEN05, PQ_ERR_FORMAT);
    int m = 0, n = 0;
    PQ_REQUIRE(M > 0 && K >= 16 && K % 16 == 0 && K <= kMaxK && ld >= K && factor_width(K, m, n), PQ_ERR_SHAPE);
    PQ_REQUIRE(sf_layout == PQ_SF_LINEAR || !codes || K % 64 == 0, PQ_ERR_SHAPE);
    PQ_REQUIRE(pq_aligned16(X) && ld % 8 == 0 && (!codes || (pq_aligned16(codes) && pq_aligned16(sf))) &&
                   (!perm || pq_aligned16(perm)) && (!y_out || pq_aligned16(y_out)),
               PQ_ERR_ALIGN);
    HadParams p;
    p.X = static_cast<const uint16_t *>(X);
    p.rows = M;
    p.rows_pad = (codes && sf_layout == PQ_SF_TCGEN05) ? pq_ceil_div(M, 128) * 128 : M;
    p.ld = ld;
    p.K = static_cast<int>(K), p.m = m, p.n = n;
    // strides 1, 2, 4 are taken in phase 1; the remaining n - 3 bits in up to three passes of at most 5
    const int rest = n - 3, passes = (rest + 4) / 5;
    PQ_REQUIRE(passes <= 3, PQ_ERR_SHAPE);
    for (int k = 0, left = rest; k < 3; ++k) {
        p.log[k] = k < passes ? (left + (passes - k) - 1) / (passes - k) : 0;
        left -= p.log[k];
    }
    p.sw = p.log[0] ? 3 + p.log[0] : 30;
    p.scale = static_cast<float>(1.0 / sqrt(static_cast<double>(K)));
    p.perm = perm, p.ts = ts_x, p.codes = codes, p.sf = sf, p.y_out = static_cast<uint16_t *>(y_out);
    int dev = 0, sms = 148;
    if (cudaGetDevice(&dev) == cudaSuccess) cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    // warps or teams of warps with rows of their own: `images` values per block, `units` units of work of all rows,
    // `per_sm` blocks of `threads` per SM
    auto launch_rows = [&](auto kern, int64_t images, int64_t units, int per_sm, int threads) -> pq_status {
        const size_t smem = static_cast<size_t>(images) * sizeof(float) + static_cast<size_t>(K) * sizeof(uint16_t);
        PQ_CUDA_OK(pq::allow_smem(kern, smem, smem));  // a kernel serves one width
        PQ_CUDA_OK(pq::launch_dependent(kern, dim3(static_cast<unsigned>(std::min<int64_t>(units, per_sm * sms))), dim3(threads), smem,
                                        static_cast<cudaStream_t>(stream), p));
        return pq_launch_status();
    };
    const bool tc = sf_layout == PQ_SF_TCGEN05;
    if (m == 12 && n >= 6 && n <= 8) {  // widths whose rows fit a warp's lanes exactly: 768, 1536, 3072
        auto go = [&](auto kern) { return launch_rows(kern, kRowWarps * kRowImage, pq_ceil_div(p.rows_pad, 1 << (8 - n)), 2, 32 * kRowWarps); };
        if (n == 8) return go(tc ? hadamard_quant_rows_kernel<PQ_SF_TCGEN05, 8> : hadamard_quant_rows_kernel<PQ_SF_LINEAR, 8>);
        if (n == 7) return go(tc ? hadamard_quant_rows_kernel<PQ_SF_TCGEN05, 7> : hadamard_quant_rows_kernel<PQ_SF_LINEAR, 7>);
        return go(tc ? hadamard_quant_rows_kernel<PQ_SF_TCGEN05, 6> : hadamard_quant_rows_kernel<PQ_SF_LINEAR, 6>);
    }
    if (m == 12 && (n == 9 || n == 10)) {  // two and four times as wide: 6144, 12288
        auto go = [&](auto kern) { return launch_rows(kern, 16 * kRowImage, p.rows_pad, 1, 512); };
        if (n == 9) return go(tc ? hadamard_quant_team_kernel<PQ_SF_TCGEN05, 9> : hadamard_quant_team_kernel<PQ_SF_LINEAR, 9>);
        return go(tc ? hadamard_quant_team_kernel<PQ_SF_TCGEN05, 10> : hadamard_quant_team_kernel<PQ_SF_LINEAR, 10>);
    }
    if (m == 1 && n >= 10 && n <= 12) {  // 1024, 2048, 4096
        auto go = [&](auto kern, int rows, int warps) {
            return launch_rows(kern, warps * rows * K, pq_ceil_div(p.rows_pad, rows), 2, 32 * warps);
        };
        if (n == 10) return go(tc ? hadamard_quant_pow2_kernel<PQ_SF_TCGEN05, 5, 5, 2, 8> : hadamard_quant_pow2_kernel<PQ_SF_LINEAR, 5, 5, 2, 8>, 2, 8);
        if (n == 11) return go(tc ? hadamard_quant_pow2_kernel<PQ_SF_TCGEN05, 6, 5, 1, 8> : hadamard_quant_pow2_kernel<PQ_SF_LINEAR, 6, 5, 1, 8>, 1, 8);
        return go(tc ? hadamard_quant_pow2_kernel<PQ_SF_TCGEN05, 6, 6, 1, 6> : hadamard_quant_pow2_kernel<PQ_SF_LINEAR, 6, 6, 1, 6>, 1, 6);
    }
    // Every other width.  8192 and 16384 too: 4608 rows take 144 and 304 us where 4096 channels take 36; a warp-per-row form like
    // the one for 4096, whose image is 32 or 64 KB a row there, was not tried.  The kernel holds the order-12 inputs in registers
    // whatever the width (128 registers, 300 bytes spilled).
    const size_t row_bytes = static_cast<size_t>(K) * sizeof(float);
    p.rows_per_block = static_cast<int>(kSmemBudget / row_bytes < kMaxRows ? kSmemBudget / row_bytes : kMaxRows);
    const int kRows = p.rows_per_block;
    const size_t smem = static_cast<size_t>(kRows) * row_bytes + static_cast<size_t>(K) * sizeof(uint16_t);
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    // persistent grid: as many blocks as fit on the device at once, walking over the batches of rows
    const bool wide_block = kRows < kMaxRows;  // fewer rows per block: twice the threads on them, one block per SM
    const int per_sm = static_cast<int>(std::min<size_t>(wide_block ? 1 : kBlocksPerSm, (227 * 1024) / (smem + 1024)));
    const int64_t batches = pq_ceil_div(p.rows_pad, kRows);
    const int64_t blocks = std::min<int64_t>(batches, static_cast<int64_t>(sms) * (per_sm > 0 ? per_sm : 1));
    auto launch = [&](auto kern) -> pq_status {
        PQ_CUDA_OK(pq::allow_smem(kern, smem, kSmemBudget + kMaxK * sizeof(uint16_t)));
        PQ_CUDA_OK(pq::launch_dependent(kern, dim3(static_cast<unsigned>(blocks)), dim3(wide_block ? 2 * kThreads : kThreads),
                                        smem, st, p));
        return pq_launch_status();
    };
    if (wide_block)
        return sf_layout == PQ_SF_TCGEN05 ? launch(hadamard_quant_kernel<PQ_SF_TCGEN05, 2 * kThreads>)
                                          : launch(hadamard_quant_kernel<PQ_SF_LINEAR, 2 * kThreads>);
    return sf_layout == PQ_SF_TCGEN05 ? launch(hadamard_quant_kernel<PQ_SF_TCGEN05, kThreads>)
                                      : launch(hadamard_quant_kernel<PQ_SF_LINEAR, kThreads>);
}

// Sort candidates of the joint second-moment criterion (Eq. 9, Prop. 3.2) and the
// selection / acceptance rule (Eq. 10).
//
// Sorting: a thread-block cluster per order.  The channels are cut into chunks of 512 keys; a CTA sorts
// its chunks (bitonic, one key per thread: strides below a warp by shuffles, the others through shared
// memory), fetches the neighbours' sorted chunks out of their shared memory, and every key finds its rank by
// binary search in them.  The position of a channel is the number of channels that precede it under the total order
// (key descending, channel ascending), so the result is unique, hence identical to any comparison sort.
// Counting ranks against all K keys instead is K^2 comparisons: 38.9 us for six orders of 3072 channels and
// 517 us at 12288 on B200, where this takes 8.7 us at 3072.
// Keys are 64-bit patterns that order like the doubles they stand for: a non-negative double orders
// like its own bits; a signed one after flipping all bits of a negative value and the sign bit of
// the others.
#include "pq_common.cuh"

namespace {

// Where the keys of an order come from.
enum KeyKind { kKeyJoint, kKeyAbsmax, kKeyVariance, kKeyPlain };
struct SortParams {
    KeyKind kind;
    const double *a, *b;   // joint: second moments of activations, weight; variance: sum, sum of squares; plain: values
    const float *f;        // absmax: maxima
    double rows_a, rows_b;
    int J;                 // joint: blockIdx.y = j = 0..J
    int K, deal_groups, group;
    int32_t *perms;        // [orders, K]
    int orders;
    // rows of the grid past the orders: *scale_out[s] = tensor scale from the column maxima scale_max[s]
    const float *scale_max[2];
    float *scale_out[2];
};

__device__ __forceinline__ unsigned long long sort_key(const SortParams &p, int j, int i) {
    if (p.kind == kKeyJoint) {
        // bit pattern of (a_i)^j (w_i)^(J-j), multiplied left to right in fp64
        const double a = __ddiv_rn(p.a[i], p.rows_a), w = __ddiv_rn(p.b[i], p.rows_b);
        double key = 1.0;
        for (int f = 0; f < j; ++f) key = __dmul_rn(key, a);
        for (int f = 0; f < p.J - j; ++f) key = __dmul_rn(key, w);
        return static_cast<unsigned long long>(__double_as_longlong(key));
    }
    if (p.kind == kKeyAbsmax)  // the channel's absmax widened to fp64 (exact; non-negative)
        return static_cast<unsigned long long>(__double_as_longlong(static_cast<double>(fabsf(p.f[i]))));
    if (p.kind == kKeyVariance) {
        // sumsq_i / rows - (sum_i / rows)^2 in fp64 (two divisions, one multiplication, one subtraction); the value
        // may be slightly negative for a constant channel
        const double mean = __ddiv_rn(p.a[i], p.rows_a);
        const double second = __ddiv_rn(p.b[i], p.rows_a);
        const double var = __dadd_rn(__dsub_rn(second, __dmul_rn(mean, mean)), 0.0);  // + 0.0: a zero is +0
        const long long bits = __double_as_longlong(var);
        return bits < 0 ? ~static_cast<unsigned long long>(bits) : static_cast<unsigned long long>(bits) | (1ull << 63);
    }
    return static_cast<unsigned long long>(__double_as_longlong(fabs(p.a[i])));
}

constexpr int kSortChunk = 512, kSortMaxChunks = 32, kSortMaxCluster = 8;
constexpr int kSortPerCta = kSortMaxChunks / kSortMaxCluster;  // chunks a CTA may hold

// (okey, oidx) precedes (key, idx): larger key, or equal key and lower index.  The borrow of a 96-bit subtraction.
__device__ __forceinline__ bool precedes(unsigned long long okey, uint32_t oidx, unsigned long long key, uint32_t idx) {
    uint32_t borrow;
    asm("{\n"
        ".reg .u32 t;\n"
        "sub.cc.u32 t, %1, %2;\n"
        "subc.cc.u32 t, %3, %4;\n"
        "subc.cc.u32 t, %5, %6;\n"
        "subc.u32 %0, 0, 0;\n"
        "}\n"
        : "=r"(borrow)
        : "r"(oidx), "r"(idx), "r"(static_cast<uint32_t>(key)), "r"(static_cast<uint32_t>(okey)),
          "r"(static_cast<uint32_t>(key >> 32)), "r"(static_cast<uint32_t>(okey >> 32)));
    return borrow != 0;
}

// Key of the neighbour: shared memory of CTA `rank` of the cluster.
__device__ __forceinline__ uint32_t cluster_addr(const void *p, uint32_t rank) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(static_cast<uint32_t>(__cvta_generic_to_shared(p))), "r"(rank));
    return r;
}
__device__ __forceinline__ unsigned long long cluster_load(uint32_t addr) {
    unsigned long long v;
    asm volatile("ld.shared::cluster.b64 %0, [%1];" : "=l"(v) : "r"(addr) : "memory");
    return v;
}
__device__ __forceinline__ void cluster_barrier() {
    asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// gridDim.x = cluster size; CTA r holds the chunks r, r + cluster size, ...
// The searches go four chunks at a time in a loop: with all of them unrolled (up to 31) the kernel took 32 us at 512
// channels, where it has nothing to search, against 4.4 us (instruction fetches).
__global__ void __launch_bounds__(kSortChunk) order_sort_kernel(const __grid_constant__ SortParams p) {
    extern __shared__ unsigned long long all_s[];  // [chunks][512] sorted keys of the whole cluster
    __shared__ unsigned long long sorted[kSortPerCta][kSortChunk];
    __shared__ unsigned long long key_x[2][kSortChunk];
    __shared__ uint16_t idx_x[2][kSortChunk], channel_s[kSortPerCta][kSortChunk];
    const int j = blockIdx.y, rank = blockIdx.x, ctas = gridDim.x, tid = threadIdx.x;
    const int chunks = (p.K + kSortChunk - 1) / kSortChunk;
    pq::dependents_may_launch();
    pq::wait_for_prior_grid();
    if (j >= p.orders) {  // the whole cluster: nobody waits for it at a cluster barrier
        if (rank) return;
        const float a = pq::block_max(p.scale_max[j - p.orders], p.K);
        if (tid == 0) *p.scale_out[j - p.orders] = (a == 0.0f) ? 1.0f : __fdiv_rn(a, 2688.0f);
        return;
    }
#pragma unroll 1
    for (int t = 0; t < kSortPerCta; ++t) {
        const int chunk = rank + t * ctas;
        if (chunk >= chunks) break;  // uniform over the CTA
        const int base = chunk * kSortChunk;
        // a slot past the end holds key 0 at an index above every channel: it precedes nothing
        unsigned long long key = base + tid < p.K ? sort_key(p, j, base + tid) : 0ull;
        uint32_t idx = tid;
        int buf = 0;
#pragma unroll
        for (int k = 2; k <= kSortChunk; k <<= 1) {
#pragma unroll
            for (int d = k >> 1; d; d >>= 1) {
                unsigned long long okey;
                uint32_t oidx;
                if (d >= 32) {
                    key_x[buf][tid] = key, idx_x[buf][tid] = static_cast<uint16_t>(idx);
                    __syncthreads();  // one barrier per exchange: the other buffer is written next
                    okey = key_x[buf][tid ^ d], oidx = idx_x[buf][tid ^ d];
                    buf ^= 1;
                } else {
                    okey = __shfl_xor_sync(0xFFFFFFFFu, key, d), oidx = __shfl_xor_sync(0xFFFFFFFFu, idx, d);
                }
                const bool want_first = ((tid & d) == 0) == ((tid & k) == 0);
                if (want_first == precedes(okey, oidx, key, idx)) key = okey, idx = oidx;
            }
        }
        sorted[t][tid] = key;
        channel_s[t][tid] = static_cast<uint16_t>(base + idx);
        __syncthreads();  // the exchange buffers may be written again
    }
    cluster_barrier();
#pragma unroll 4
    for (int c = 0; c < chunks; ++c)
        all_s[c * kSortChunk + tid] = cluster_load(cluster_addr(&sorted[c / ctas][tid], static_cast<uint32_t>(c % ctas)));
    __syncthreads();
#pragma unroll 1
    for (int t = 0; t < kSortPerCta; ++t) {
        const int chunk = rank + t * ctas;
        if (chunk >= chunks) break;
        const unsigned long long mine = sorted[t][tid];
        // keys of an earlier chunk precede mine when they are not smaller, of a later one when larger
        int place = tid;
#pragma unroll 1
        for (int c0 = 0; c0 < chunks; c0 += 4) {
            int pos[4];
            const unsigned long long *keys[4];
            bool earlier[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int c = min(c0 + u, chunks - 1);
                pos[u] = 0, keys[u] = all_s + c * kSortChunk, earlier[u] = c < chunk;
            }
#pragma unroll
            for (int s = kSortChunk / 2; s; s >>= 1) {
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const unsigned long long other = keys[u][pos[u] + s - 1];
                    if (other > mine || (earlier[u] && other == mine)) pos[u] += s;
                }
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const unsigned long long other = keys[u][pos[u]];
                if (other > mine || (earlier[u] && other == mine)) ++pos[u];
                if (c0 + u < chunks && c0 + u != chunk) place += pos[u];
            }
        }
        // deal_groups == 0: the channel of rank r is read at position r; otherwise the sorted channels are dealt
        // to deal_groups groups in turn: rank r goes to group r % deal_groups, slot r / deal_groups
        const int at = p.deal_groups ? (place % p.deal_groups) * p.group + place / p.deal_groups : place;
        const int ch = channel_s[t][tid];
        if (ch < p.K) p.perms[static_cast<int64_t>(j) * p.K + at] = ch;
    }
    cluster_barrier();  // the neighbours may still be reading this CTA's keys
}

SortParams sort_params(KeyKind kind, int orders, const double *a, const double *b, const float *f, int64_t rows_a, int64_t rows_b, int J, int64_t K,
                       int32_t *perms) {
    SortParams p;
    p.kind = kind, p.a = a, p.b = b, p.f = f;
    p.rows_a = static_cast<double>(rows_a), p.rows_b = static_cast<double>(rows_b), p.J = J;
    p.K = static_cast<int>(K), p.deal_groups = 0, p.group = 0, p.perms = perms, p.orders = orders;
    p.scale_max[0] = p.scale_max[1] = nullptr, p.scale_out[0] = p.scale_out[1] = nullptr;
    return p;
}

pq_status launch_sort(const SortParams &p, cudaStream_t st) {
    const int chunks = static_cast<int>(pq_ceil_div(p.K, kSortChunk));
    const int ctas = chunks < kSortMaxCluster ? chunks : kSortMaxCluster;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(static_cast<unsigned>(ctas), static_cast<unsigned>(p.orders + (p.scale_out[0] ? 2 : 0)));
    cfg.blockDim = dim3(kSortChunk), cfg.stream = st;
    cfg.dynamicSmemBytes = static_cast<size_t>(chunks) * kSortChunk * sizeof(unsigned long long);
    PQ_CUDA_OK(pq::allow_smem(order_sort_kernel, cfg.dynamicSmemBytes, kSortMaxChunks * kSortChunk * sizeof(unsigned long long), 32 * 1024));
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = static_cast<unsigned>(ctas), attr[0].val.clusterDim.y = 1, attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr, cfg.numAttrs = 2;
    PQ_CUDA_OK(cudaLaunchKernelEx(&cfg, order_sort_kernel, p));
    return pq_launch_status();
}

// A warp per (order p = 0..P, side) adds up that error row in ascending order; thread 0 then applies Eq. 10.  One thread per order with its loads
// inside the chain took 22 us for 7 orders of 192 groups.
constexpr int kAcceptWarps = 16;
__global__ void __launch_bounds__(32 * kAcceptWarps)
accept_kernel(const double *ex, const double *ew, const double *lambda, int P, int64_t Kg,
              double tau, int32_t *best, int32_t *accept, double *E_out) {
    __shared__ double sums[2][32], E[32];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    pq::dependents_may_launch();
    pq::wait_for_prior_grid();
    for (int w = warp; w < 2 * (P + 1); w += kAcceptWarps) {
        const int p = w >> 1, side = w & 1;
        const double s = pq::ordered_sum((side ? ew : ex) + p * Kg, Kg);
        if (lane == 0) sums[side][p] = s;
    }
    __syncthreads();
    const int p = threadIdx.x;
    if (p <= P) {
        const double lx = lambda ? lambda[0] : 1.0, lw = lambda ? lambda[1] : 1.0;
        E[p] = __dadd_rn(__dmul_rn(lx, sums[0][p]), __dmul_rn(lw, sums[1][p]));
        if (E_out) E_out[p] = E[p];
    }
    __syncthreads();
    if (p == 0) {
        int b = 1;
        for (int q = 2; q <= P; ++q)
            if (E[q] < E[b]) b = q;
        const double gain = __dadd_rn(E[0], -E[b]);
        const double need = __dmul_rn(tau, E[0]);
        *best = b;
        *accept = (gain > need) ? 1 : 0;
    }
}

}  // namespace

pq_status pq_orders_and_scales(const double *sumsq_a, int64_t rows_a, const double *sumsq_w, int64_t rows_w, int64_t K, int J,
                               int32_t *perms, const float *amax_a, const float *amax_w, float *ts_x, float *ts_w, cudaStream_t st) {
    SortParams p = sort_params(kKeyJoint, J + 1, sumsq_a, sumsq_w, nullptr, rows_a, rows_w, J, K, perms);
    p.scale_max[0] = amax_a, p.scale_max[1] = amax_w;
    p.scale_out[0] = ts_x, p.scale_out[1] = ts_w;
    return launch_sort(p, st);
}

extern "C" pq_status pq_select_perm(const double *sumsq_a, int64_t rows_a, const double *sumsq_w,
                                    int64_t rows_w, int64_t K, int J, int32_t *perms, void *ws,
                                    size_t ws_bytes, void *stream) {
    PQ_REQUIRE(sumsq_a && sumsq_w && perms, PQ_ERR_NULL);
    PQ_REQUIRE(K > 0 && K <= 16384 && J >= 1 && J <= 16 && rows_a > 0 && rows_w > 0, PQ_ERR_SHAPE);
    const size_t need = pq_workspace_bytes(PQ_OP_SELECT_PERM, 0, K, 0, J + 1);
    PQ_REQUIRE(ws && ws_bytes >= need, PQ_ERR_WORKSPACE);
    PQ_REQUIRE(pq_aligned256(ws), PQ_ERR_ALIGN);
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    return launch_sort(sort_params(kKeyJoint, J + 1, sumsq_a, sumsq_w, nullptr, rows_a, rows_w, J, K, perms), st);
}

extern "C" pq_status pq_order_by_absmax(const float *amax, int64_t K, int32_t *perm, void *ws, size_t ws_bytes,
                                        void *stream) {
    PQ_REQUIRE(amax && perm, PQ_ERR_NULL);
    PQ_REQUIRE(K > 0 && K <= 16384, PQ_ERR_SHAPE);
    PQ_REQUIRE(ws && ws_bytes >= pq_workspace_bytes(PQ_OP_SELECT_PERM, 0, K, 0, 1), PQ_ERR_WORKSPACE);
    PQ_REQUIRE(pq_aligned256(ws), PQ_ERR_ALIGN);
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    return launch_sort(sort_params(kKeyAbsmax, 1, nullptr, nullptr, amax, 1, 1, 0, K, perm), st);
}

extern "C" pq_status pq_order_by_variance(const double *sum, const double *sumsq, int64_t rows, int64_t K, int32_t *perm,
                                          void *ws, size_t ws_bytes, void *stream) {
    PQ_REQUIRE(sum && sumsq && perm, PQ_ERR_NULL);
    PQ_REQUIRE(K > 0 && K <= 16384 && rows > 0, PQ_ERR_SHAPE);
    PQ_REQUIRE(ws && ws_bytes >= pq_workspace_bytes(PQ_OP_SELECT_PERM, 0, K, 0, 1), PQ_ERR_WORKSPACE);
    PQ_REQUIRE(pq_aligned256(ws), PQ_ERR_ALIGN);
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    return launch_sort(sort_params(kKeyVariance, 1, sum, sumsq, nullptr, rows, 1, 0, K, perm), st);
}

extern "C" pq_status pq_order_round_robin(const double *sumsq, int64_t K, int group, int32_t *perm, void *ws,
                                          size_t ws_bytes, void *stream) {
    PQ_REQUIRE(sumsq && perm, PQ_ERR_NULL);
    PQ_REQUIRE(K > 0 && K <= 16384 && group > 0 && K % group == 0, PQ_ERR_SHAPE);
    PQ_REQUIRE(ws && ws_bytes >= pq_workspace_bytes(PQ_OP_SELECT_PERM, 0, K, 0, 1), PQ_ERR_WORKSPACE);
    PQ_REQUIRE(pq_aligned256(ws), PQ_ERR_ALIGN);
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    SortParams p = sort_params(kKeyPlain, 1, sumsq, nullptr, nullptr, 1, 1, 0, K, perm);
    p.deal_groups = static_cast<int>(K / group), p.group = group;
    return launch_sort(p, st);
}

extern "C" pq_status pq_accept(const double *err_x, const double *err_w, const double *lambda, int P,
                               int64_t Kg, double tau, int32_t *best, int32_t *accept, double *E,
                               void *stream) {
    PQ_REQUIRE(err_x && err_w && best && accept, PQ_ERR_NULL);
    PQ_REQUIRE(P >= 1 && P <= 31 && Kg > 0, PQ_ERR_SHAPE);
    PQ_CUDA_OK(pq::launch_dependent(accept_kernel, dim3(1), dim3(32 * kAcceptWarps), 0, static_cast<cudaStream_t>(stream), err_x,
                                    err_w, lambda, P, Kg, tau, best, accept, E));
    return pq_launch_status();
}

// The whole offline pass of a layer in one call: statistics, candidate orders, errors, decision, quantized weight.
//
// What a pass over small tensors costs is launches: one call per step and batch was 45 launches with their host work
// (420 us for four batches of 256 x 512 and a 512 x 512 weight, of which 160 us device time), and on large ones the
// same structure left every batch a partly filled last wave and two ordered folds.  Here every step runs over all
// batches and the weight at once (PqTensorList): seven launches, each a programmatic dependent of the one before.  The
// partial sums of the tensors lie one behind the other in call order and no slab straddles two of them, so the folds
// add in the same order as one call per batch and the results are the same bits.
#include "pq_common.cuh"

namespace {
size_t round256(size_t b) { return (b + 255) / 256 * 256; }

// The batches of a round and whether the weight closes it: as many tensors as a list holds and as the partial sums have room
// for, one at least.  Without the second limit the sums of up to 64 tensors lie side by side, 400 MB for 64 batches of
// 4608 x 12288; 64 MiB hold the sums of 600 million elements in NVFP4, whose pass takes milliseconds.
constexpr size_t kPartialBytes = 64u << 20;
struct Round {
    int end;
    bool with_weight;
    int64_t slabs;
};
Round next_round(int i, int n, const int64_t *rows, int64_t N, int64_t most) {
    Round r{i, false, 0};
    int count = 0;
    for (; r.end < n && count < kPqListMax; ++r.end, ++count) {
        const int64_t slabs = rows[r.end] > 0 ? pq_ceil_div(rows[r.end], PQ_SLAB_ROWS) : 0;
        if (count && r.slabs + slabs > most) break;
        r.slabs += slabs;
    }
    const int64_t slabs = pq_ceil_div(N, PQ_SLAB_ROWS);
    r.with_weight = r.end == n && count < kPqListMax && (!count || r.slabs + slabs <= most);
    if (r.with_weight) r.slabs += slabs;
    return r;
}

size_t partial_bytes(int64_t slabs, int64_t K, int group, int P) {
    const size_t a = pq_stats_list_bytes(slabs, K), b = pq_errors_list_bytes(slabs, K, group, P);
    return round256(a > b ? a : b);
}
int64_t slabs_per_round(int64_t K, int group, int P) { return static_cast<int64_t>(kPartialBytes / partial_bytes(1, K, group, P)); }

// What can be told from the sizes alone; the caller's outputs and the workspace are sized by these.
pq_status sizes_status(int n, int64_t N, int64_t K, pq_format fmt, int J) {
    PQ_REQUIRE(fmt.kind == 0 || (fmt.kind == 1 && fmt.bits >= 2 && fmt.bits <= 8 &&
                                 (fmt.group == 16 || fmt.group == 32 || fmt.group == 64 || fmt.group == 128 || fmt.group == 256)),
               PQ_ERR_FORMAT);
    const int group = fmt.kind == 0 ? 16 : fmt.group;
    PQ_REQUIRE(n >= 1 && N > 0 && K > 0 && K % group == 0 && K % 16 == 0 && K <= 16384, PQ_ERR_SHAPE);
    PQ_REQUIRE(J >= 1 && J <= 7, PQ_ERR_SHAPE);
    return PQ_OK;
}
}  // namespace

extern "C" size_t pq_calibrate_workspace_bytes(int n, const int64_t *rows, int64_t N, int64_t K, pq_format fmt, int J) {
    if (!rows || sizes_status(n, N, K, fmt, J) != PQ_OK) return 0;
    const int group = fmt.kind == 0 ? 16 : fmt.group;
    const int64_t limit = slabs_per_round(K, group, J + 1);
    size_t most = 0;
    for (Round r{0, false, 0}; !r.with_weight;) {
        r = next_round(r.end, n, rows, N, limit);
        const size_t b = partial_bytes(r.slabs, K, group, J + 1);
        if (b > most) most = b;
    }
    return most + round256(static_cast<size_t>(K) * sizeof(float));
}

extern "C" pq_status pq_calibrate(int n, const void *const *X, const int64_t *rows, const int64_t *ld, const void *Wt, int64_t N,
                                  int64_t K, int64_t ldw, pq_format fmt, int J, double tau, int sf_layout, double *sumsq_a,
                                  double *sumsq_w, float *amax_a, float *ts_x, float *ts_w, int32_t *perms, double *err_x,
                                  double *err_w, double *lambda, double *E, int32_t *select, uint8_t *codes, uint8_t *sf,
                                  void *ws, size_t ws_bytes, void *stream) {
    const pq_status sizes = sizes_status(n, N, K, fmt, J);
    PQ_REQUIRE(sizes == PQ_OK, sizes);
    PQ_REQUIRE(sf_layout == PQ_SF_LINEAR || sf_layout == PQ_SF_TCGEN05, PQ_ERR_FORMAT);
    PQ_REQUIRE(X && rows && ld && Wt && sumsq_a && sumsq_w && amax_a && ts_x && ts_w && perms && err_x && err_w && lambda &&
                   select && codes && sf,
               PQ_ERR_NULL);
    const int group = fmt.kind == 0 ? 16 : fmt.group;
    PQ_REQUIRE(ldw >= K && (sf_layout == PQ_SF_LINEAR || K % 64 == 0), PQ_ERR_SHAPE);
    PQ_REQUIRE(pq_aligned16(Wt) && ldw % 8 == 0 && pq_aligned16(codes) && pq_aligned16(sf), PQ_ERR_ALIGN);
    int64_t rows_a = 0, slabs = pq_ceil_div(N, PQ_SLAB_ROWS);
    for (int i = 0; i < n; ++i) {
        PQ_REQUIRE(X[i], PQ_ERR_NULL);
        PQ_REQUIRE(rows[i] > 0 && ld[i] >= K, PQ_ERR_SHAPE);
        PQ_REQUIRE(pq_aligned16(X[i]) && ld[i] % 8 == 0, PQ_ERR_ALIGN);
        rows_a += rows[i], slabs += pq_ceil_div(rows[i], PQ_SLAB_ROWS);
    }
    PQ_REQUIRE(slabs < (1ll << 27), PQ_ERR_SHAPE);
    const size_t need = pq_calibrate_workspace_bytes(n, rows, N, K, fmt, J);
    PQ_REQUIRE(ws && ws_bytes >= need, PQ_ERR_WORKSPACE);
    PQ_REQUIRE(pq_aligned256(ws), PQ_ERR_ALIGN);
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    float *amax_w = reinterpret_cast<float *>(static_cast<unsigned char *>(ws) + need - round256(static_cast<size_t>(K) * sizeof(float)));

    const int64_t limit = slabs_per_round(K, group, J + 1);
    // f(list, first round, the weight is in the list) for every round of tensors
    auto each_round = [&](auto &&f) -> pq_status {
        for (Round r{0, false, 0}; !r.with_weight;) {
            PqTensorList list;
            int i = r.end;
            const bool first = i == 0;
            r = next_round(i, n, rows, N, limit);
            for (; i < r.end; ++i) list.add(X[i], rows[i], ld[i]);
            list.n_x = list.n;
            if (r.with_weight) list.add(Wt, N, ldw);
            const pq_status rc = f(list, first, r.with_weight);
            if (rc != PQ_OK) return rc;
        }
        return PQ_OK;
    };
    pq_status rc = each_round([&](const PqTensorList &list, bool first, bool with_w) {
        const PqSide sides[2] = {{list.n_x ? sumsq_a : nullptr, amax_a, first}, {with_w ? sumsq_w : nullptr, amax_w, true}};
        return pq_stats_on_list(list, K, sides, ws, st);
    });
    if (rc != PQ_OK) return rc;
    rc = pq_orders_and_scales(sumsq_a, rows_a, sumsq_w, N, K, J, perms, amax_a, amax_w, ts_x, ts_w, st);
    if (rc != PQ_OK) return rc;
    rc = each_round([&](const PqTensorList &list, bool first, bool with_w) {
        const float *const ts[2] = {ts_x, ts_w};
        const PqSide sides[2] = {{list.n_x ? err_x : nullptr, nullptr, first}, {with_w ? err_w : nullptr, nullptr, true}};
        return pq_errors_on_list(list, K, fmt, ts, perms, J + 1, sides, {sumsq_a, sumsq_w, first ? lambda : nullptr}, ws, st);
    });
    if (rc != PQ_OK) return rc;
    rc = pq_accept(err_x, err_w, lambda, J + 1, K / group, tau, select, select + 1, E, stream);
    if (rc != PQ_OK) return rc;
    return pq_quant_weight_scaled(Wt, N, K, ldw, perms, select, codes, sf, sf_layout, ts_w, st);
}

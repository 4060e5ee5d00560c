// FP64 block-sparse product C <- beta C + alpha mask_{P_C}(A.B) on FP64 FMAs.
//
// Work decomposition: an "item" is one scalar row r of one C block c; Q adjacent lanes of
// a warp share an item and split its task segment (lane q takes tasks q, q+Q, ...), each
// keeping the item's NB partial sums in registers; the Q partials are then combined by a
// fixed xor-shuffle tree, so every C row has exactly one writer (no atomics) and the
// summation order is fixed (deterministic).  Q is picked by pick_q.  The B block of a task is
// read by the NB lanes that own the rows of the same C block, so it is served from L1 after
// the first touch.
#include "cq_internal.cuh"

namespace {

// Threads per CTA: nothing is shared beyond the rows of a C block, and small CTAs fill the last
// wave better (U.X on 64 atoms: 32.9 us with 64 threads, 37.0 with 256 at the same lane split;
// large products do not change).
constexpr int F64_T = 64;

// One or two products over the same task list (blockIdx.y picks the operands): the pairs of an
// LNV evaluation that share their patterns go in one launch.  A 64-atom cell's product is one
// wave of short dependent chains (18 us alone), so its partner runs beside it for little: pairs
// and the lane split below took an LNV run at 64 atoms from 7.4 to 6.3 ms (it is 4.0 ms now, with
// the one-launch reductions and the small CTAs).
struct F64Ops {
    const double *A[2], *B[2];
    double *C[2];
};

// VEC: every array starts on a 16-byte boundary (and so does every block), so the B block and
// the rows of a 4-orbital basis move 16 bytes at a time (half the load instructions; the same
// FMAs in the same order).  Large products are FP64-bound and do not change; with 4 orbitals
// and 64 atoms U.X goes from 39 to 37 us.
template <int NB, int Q, bool VEC>
__global__ void __launch_bounds__(F64_T)
k_bsmm_f64_uniform(int64_t n_items, const int64_t *__restrict__ seg,
                   const int2 *__restrict__ tasks, const F64Ops ops, int stride, double alpha,
                   double beta)
{
    const bool two = blockIdx.y != 0;
    const double *__restrict__ A = two ? ops.A[1] : ops.A[0];
    const double *__restrict__ B = two ? ops.B[1] : ops.B[0];
    double *__restrict__ C = two ? ops.C[1] : ops.C[0];
    const int64_t gt = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t item = gt / Q;
    const int q = (int)(gt % Q);
    const bool active = item < n_items;
    const int64_t c = active ? item / NB : 0;
    const int r = (int)(item % NB);
    double acc[NB];
#pragma unroll
    for (int x = 0; x < NB; ++x) acc[x] = 0.0;
    if (active) {
        const int64_t t1 = seg[c + 1];
        int64_t t = seg[c] + q;
        int2 tk = t < t1 ? __ldg(&tasks[t]) : make_int2(0, 0);
        while (t < t1) {
            const double *a = A + (int64_t)tk.x * stride + r * NB;
            const double *b = B + (int64_t)tk.y * stride;
            t += Q;
            if (t < t1) tk = __ldg(&tasks[t]);  // the next task arrives under this one's FMAs
            double av[NB];
            if constexpr (VEC && NB % 2 == 0) {
#pragma unroll
                for (int m = 0; m < NB; m += 2) {
                    const double2 v = __ldg(reinterpret_cast<const double2 *>(a + m));
                    av[m] = v.x;
                    av[m + 1] = v.y;
                }
            } else {
#pragma unroll
                for (int m = 0; m < NB; ++m) av[m] = __ldg(a + m);
            }
            if constexpr (VEC) {
#pragma unroll
                for (int e = 0; e < NB * NB; e += 2) {
                    const double2 v = __ldg(reinterpret_cast<const double2 *>(b + e));
                    acc[e % NB] = fma(av[e / NB], v.x, acc[e % NB]);
                    if (e + 1 < NB * NB)
                        acc[(e + 1) % NB] = fma(av[(e + 1) / NB], v.y, acc[(e + 1) % NB]);
                }
            } else {
#pragma unroll
                for (int m = 0; m < NB; ++m)
#pragma unroll
                    for (int x = 0; x < NB; ++x)
                        acc[x] = fma(av[m], __ldg(b + m * NB + x), acc[x]);
            }
        }
    }
#pragma unroll
    for (int o = Q >> 1; o > 0; o >>= 1)
#pragma unroll
        for (int x = 0; x < NB; ++x) acc[x] += __shfl_xor_sync(0xffffffffu, acc[x], o);
    if (active && q == 0) {
        double *cp = C + c * stride + r * NB;
        if (beta == 0.0) {
#pragma unroll
            for (int x = 0; x < NB; ++x) cp[x] = alpha * acc[x];
        } else {
#pragma unroll
            for (int x = 0; x < NB; ++x) cp[x] = beta * cp[x] + alpha * acc[x];
        }
    }
}

// One C row of the mixed-basis product with NJ columns: the Q lanes of the row's group take
// tasks q, q + Q, ..., keep NJ partial sums and combine them with a fixed xor tree over the
// group (gmask: the group's lanes, so that groups of different widths may branch apart).
// NJ == CQ_MAX_NB is the catch-all for widths without their own instance (nj_rt columns).
template <int NJ, int Q>
__device__ __forceinline__ void generic_row(unsigned gmask, int q, int64_t c, int r, int ni,
                                            int nj_rt, const int64_t *__restrict__ seg,
                                            const int2 *__restrict__ tasks,
                                            const int32_t *__restrict__ nb,
                                            const int32_t *__restrict__ a_col,
                                            const int64_t *__restrict__ a_off,
                                            const int64_t *__restrict__ b_off,
                                            const int64_t *__restrict__ c_off,
                                            const double *__restrict__ A,
                                            const double *__restrict__ B, double *__restrict__ C,
                                            double alpha, double beta)
{
    constexpr bool ANY = NJ == CQ_MAX_NB;
    const int nj = ANY ? nj_rt : NJ;
    double acc[NJ];
#pragma unroll
    for (int x = 0; x < NJ; ++x) acc[x] = 0.0;
    const int64_t t1 = seg[c + 1];
    for (int64_t t = seg[c] + q; t < t1; t += Q) {
        const int2 tk = __ldg(&tasks[t]);
        const int nk = nb[a_col[tk.x]];
        const double *a = A + a_off[tk.x] + (int64_t)r * nk;
        const double *b = B + b_off[tk.y];
        for (int m = 0; m < nk; ++m) {
            const double av = __ldg(a + m);
#pragma unroll
            for (int x = 0; x < NJ; ++x)
                if (!ANY || x < nj) acc[x] = fma(av, __ldg(b + m * nj + x), acc[x]);
        }
    }
#pragma unroll
    for (int o = Q >> 1; o > 0; o >>= 1)
#pragma unroll
        for (int x = 0; x < NJ; ++x) acc[x] += __shfl_xor_sync(gmask, acc[x], o);
    if (q == 0 && r < ni) {
        double *cp = C + c_off[c] + (int64_t)r * nj;
#pragma unroll
        for (int x = 0; x < NJ; ++x)
            if (!ANY || x < nj)
                cp[x] = (beta == 0.0) ? alpha * acc[x] : beta * cp[x] + alpha * acc[x];
    }
}

// Mixed orbital counts (1..16 per atom): item -> C block by a search over the prefix of block
// row counts; block offsets from the patterns' val_off.  The row's column count selects an
// instance with exactly that many accumulators (4, 5, 9, 13: the bases of the mixed-species
// cells), so no FMA slot or shuffle is spent on absent columns.  Bound by the FP64 pipe, whose
// time goes by warp: lanes that run different numbers of terms or different instances idle.
// So the blocks come sorted by width and a segment's tasks by the orbital count of k (S.X of
// four cells of 5/9/13 orbitals: 56.5 ms unsorted at q = 8, 45.0 with sorted tasks, 33.1 with
// both at q = 4; U.X 76.7 -> 50.2 ms, 0.97 of the pipe's 1.26 TFLOP/s).
template <int Q>
__global__ void __launch_bounds__(F64_T)
k_bsmm_f64_generic(int64_t n_items, int64_t n_c, const int64_t *__restrict__ rowitem,
                   const int32_t *__restrict__ order,
                   const int64_t *__restrict__ seg, const int2 *__restrict__ tasks,
                   const int32_t *__restrict__ nb, const int32_t *__restrict__ c_row,
                   const int32_t *__restrict__ c_col, const int32_t *__restrict__ a_col,
                   const int64_t *__restrict__ a_off, const int64_t *__restrict__ b_off,
                   const int64_t *__restrict__ c_off, const F64Ops ops, double alpha, double beta)
{
    const bool two = blockIdx.y != 0;
    const double *__restrict__ A = two ? ops.A[1] : ops.A[0];
    const double *__restrict__ B = two ? ops.B[1] : ops.B[0];
    double *__restrict__ C = two ? ops.C[1] : ops.C[0];
    const int64_t gt = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t item = gt / Q;
    const int q = (int)(gt % Q);
    // the block of the CTA's first item, then each thread's among the next F64_T / Q
    __shared__ int64_t first;
    if (threadIdx.x < 32) {
        const int64_t i0 = (int64_t)blockIdx.x * (blockDim.x / Q);
        int64_t lo = 0, hi = n_c;  // largest c with rowitem[c] <= i0: 32 probes at a time
        while (hi - lo > 1) {
            const int64_t step = (hi - lo + 31) / 32, at = lo + step * (threadIdx.x + 1);
            const bool le = at < hi && rowitem[at] <= i0;
            const int n = __popc(__ballot_sync(0xffffffffu, le));
            hi = min(hi, lo + step * (n + 1));
            lo += step * n;
        }
        if (threadIdx.x == 0) first = lo;
    }
    __syncthreads();
    if (item >= n_items) return;  // whole Q groups leave together (blockDim is a multiple of Q)
    int64_t lo = first, hi = min(n_c, first + blockDim.x / Q + 1);
    while (hi - lo > 1) {
        int64_t mid = (lo + hi) >> 1;
        if (rowitem[mid] <= item)
            lo = mid;
        else
            hi = mid;
    }
    const int64_t c = order[lo];
    const int r = (int)(item - rowitem[lo]);
    const int ni = nb[c_row[c]], nj = nb[c_col[c]];
    const unsigned gmask =
        Q == 32 ? 0xffffffffu : (((1u << Q) - 1u) << ((threadIdx.x & 31) & ~(Q - 1)));
#define CQ_ROW(NJ)                                                                           \
    generic_row<NJ, Q>(gmask, q, c, r, ni, nj, seg, tasks, nb, a_col, a_off, b_off, c_off, A, \
                       B, C, alpha, beta)
    switch (nj) {
    case 4: CQ_ROW(4); break;
    case 5: CQ_ROW(5); break;
    case 9: CQ_ROW(9); break;
    case 13: CQ_ROW(13); break;
    default: CQ_ROW(CQ_MAX_NB); break;
    }
#undef CQ_ROW
}

// Lanes per C row.  Neighbouring lanes of a row read different B blocks, so a load of a warp
// touches about q cache lines: at q = 16 and 32 the L1 serves one line per clock and the kernel
// runs at 0.6 of the FP64 pipe (T.V on 216 SZP atoms: 4.02 ms at q = 4, 8.19 at 16); at q = 1
// short segments end at different times (L.S on 512 atoms: 8.58 ms at q = 4, 9.94 at 1).  So four
// lanes, two on a 4-orbital basis (S.X on 512 sp atoms: 719 us at 2, 782 at 4).  Up to eight
// lanes where that still leaves less than 60 k threads, so that the SMs have warps to switch
// between (4 orbitals, U.X on 64 atoms: 32.8 us at 2, 29.0 at 4, 34.8 at 8; on 32 atoms 18.3, 12.2
// and 11.0), or less than 200 k if segments are long (U.X on 216 atoms: 264 us at 2, 246 at 4).
int pick_q(const TaskList *tl, int nb)
{
    const double avg = tl->n_c ? (double)tl->n_tasks / (double)tl->n_c : 0.0;
    int q = nb == 4 ? 2 : 4;
    while (q < 8 && (tl->n_items * q < 30000 || (tl->n_items * q < 100000 && avg >= 64.0 * q)))
        q <<= 1;
    return q;
}

template <int NB, bool VEC>
void launch_uniform(int q, dim3 grid, cudaStream_t s, int64_t n_items, const TaskList *tl,
                    const F64Ops &ops, int stride, double alpha, double beta)
{
    const int64_t *seg = tl->seg.as<int64_t>();
    const int2 *tk = tl->tasks.as<int2>();
#define CQ_LAUNCH(QQ) \
    k_bsmm_f64_uniform<NB, QQ, VEC><<<grid, F64_T, 0, s>>>(n_items, seg, tk, ops, stride, alpha, beta)
    switch (q) {
    case 1: CQ_LAUNCH(1); break;
    case 2: CQ_LAUNCH(2); break;
    case 4: CQ_LAUNCH(4); break;
    case 8: CQ_LAUNCH(8); break;
    case 16: CQ_LAUNCH(16); break;
    default: CQ_LAUNCH(32); break;
    }
#undef CQ_LAUNCH
}

}  // namespace

// One launch of the FP64 product (n = 1) or of two on the same patterns (n = 2) with lane split q.
static void launch_f64(cq_ctx *ctx, int q, const TaskList *tl, double alpha,
                       const cq_pattern *pA, const cq_pattern *pB, double beta,
                       const cq_pattern *pC, const F64Ops &ops, int n)
{
    const int nbu = pC->geo->uniform_nb;
    cudaStream_t s = ctx->stream;
    const int64_t n_items = tl->n_items;
    const dim3 grid((unsigned)((n_items * q + F64_T - 1) / F64_T), (unsigned)n);
    if (nbu == 9 || nbu == 4) {
        uintptr_t bits = 0;
        for (int e = 0; e < n; ++e)
            bits |= reinterpret_cast<uintptr_t>(ops.A[e]) | reinterpret_cast<uintptr_t>(ops.B[e]);
        const bool vec = (bits & 15) == 0;
        auto go = nbu == 9 ? (vec ? launch_uniform<9, true> : launch_uniform<9, false>)
                           : (vec ? launch_uniform<4, true> : launch_uniform<4, false>);
        go(q, grid, s, n_items, tl, ops, pC->uniform, alpha, beta);
        return;
    }
    const int64_t *rowitem = tl->c_rowitem.as<int64_t>();
    const int32_t *nb = pC->geo->nb.as<int32_t>();
#define CQ_GEN(QQ)                                                                            \
    k_bsmm_f64_generic<QQ><<<grid, F64_T, 0, s>>>(                                              \
        n_items, tl->n_c, rowitem, tl->c_order.as<int32_t>(), tl->seg.as<int64_t>(),          \
        tl->tasks.as<int2>(), nb, pC->row.as<int32_t>(), pC->col.as<int32_t>(),               \
        pA->col.as<int32_t>(), pA->val_off.as<int64_t>(), pB->val_off.as<int64_t>(),          \
        pC->val_off.as<int64_t>(), ops, alpha, beta)
    switch (q) {
    case 1: CQ_GEN(1); break;
    case 2: CQ_GEN(2); break;
    case 4: CQ_GEN(4); break;
    case 8: CQ_GEN(8); break;
    case 16: CQ_GEN(16); break;
    default: CQ_GEN(32); break;
    }
#undef CQ_GEN
}

// Autotuner: on the first product of a task list (with autotuning on and no capture open),
// time every lane split on the real operands into scratch (beta = 0, so the caller's C is
// untouched) and keep the fastest for this task list.
static cq_status tune_q(cq_ctx *ctx, const TaskList *tl, const cq_pattern *pA, const double *A,
                        const cq_pattern *pB, const double *B, const cq_pattern *pC)
{
    void *tmp;
    cq_status st = cq_scratch(ctx, "tune_C", sizeof(double) * pC->n_values, &tmp);
    if (st != CQ_OK) return st;
    const F64Ops ops = {{A, nullptr}, {B, nullptr}, {(double *)tmp, nullptr}};
    cudaEvent_t e0, e1;
    cudaEventCreate(&e0);
    cudaEventCreate(&e1);
    float best = 1e30f;
    int best_q = cq_lane_split(tl);
    for (int q = 1; q <= 32; q <<= 1) {
        launch_f64(ctx, q, tl, 1.0, pA, pB, 0.0, pC, ops, 1);  // warm
        cudaEventRecord(e0, ctx->stream);
        launch_f64(ctx, q, tl, 1.0, pA, pB, 0.0, pC, ops, 1);
        cudaEventRecord(e1, ctx->stream);
        cq_count_launch(2);
        st = cq_check_cuda(ctx, cudaEventSynchronize(e1), "autotune");
        if (st != CQ_OK) break;
        float ms = 0.f;
        cudaEventElapsedTime(&ms, e0, e1);
        if (ms < best) {
            best = ms;
            best_q = q;
        }
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    tl->q = best_q;
    return st;
}

int cq_lane_split(const TaskList *tl) { return tl->q ? tl->q : pick_q(tl, tl->uniform_nb); }

static cq_status run_f64(cq_ctx *ctx, const TaskList *tl, double alpha, const cq_pattern *pA,
                         const cq_pattern *pB, double beta, const cq_pattern *pC,
                         const F64Ops &ops, int n)
{
    if (tl->n_c == 0) return CQ_OK;
    if (!tl->filled) {
        if (ctx->capturing)
            return cq_fail(ctx, CQ_ERR_INVALID,
                           "bsmm: first FP64 product of a triple inside a graph capture");
        cq_status st = cq_fill_tasks(ctx, pA, pB, pC, const_cast<TaskList *>(tl));
        if (st != CQ_OK) return st;
    }
    if (ctx->autotune && tl->q == 0 && !ctx->capturing) {
        cq_status st = tune_q(ctx, tl, pA, ops.A[0], pB, ops.B[0], pC);
        if (st != CQ_OK) return st;
    }
    cq_timing_begin(ctx, n * tl->flops);
    launch_f64(ctx, cq_lane_split(tl), tl, alpha, pA, pB, beta, pC, ops, n);
    cq_timing_end(ctx);
    cq_count_launch();
    return cq_check_cuda(ctx, cudaGetLastError(), "bsmm_f64");
}

cq_status cq_bsmm_f64(cq_ctx *ctx, const TaskList *tl, double alpha, const cq_pattern *pA,
                      const double *A, const cq_pattern *pB, const double *B, double beta,
                      const cq_pattern *pC, double *C)
{
    return run_f64(ctx, tl, alpha, pA, pB, beta, pC, F64Ops{{A, nullptr}, {B, nullptr}, {C, nullptr}},
                   1);
}

cq_status cq_bsmm_f64_pair(cq_ctx *ctx, const TaskList *tl, double alpha, const cq_pattern *pA,
                           const double *A0, const double *A1, const cq_pattern *pB,
                           const double *B0, const double *B1, double beta, const cq_pattern *pC,
                           double *C0, double *C1)
{
    return run_f64(ctx, tl, alpha, pA, pB, beta, pC, F64Ops{{A0, A1}, {B0, B1}, {C0, C1}}, 2);
}

// Traces, inner products, norms, Gershgorin bounds (deterministic FP64 reductions) and the
// elementwise kernels on pattern values.
//
// A reduction is one launch for up to RED_Q quantities of one basis: every thread accumulates
// its share in a fixed order, each CTA combines its threads by a fixed tree into one partial,
// and the last CTA of a quantity (and cell) to arrive folds the partials, again by a fixed
// tree, and writes the scalar straight to pinned host memory together with the device error
// word.  Grid and order depend on sizes alone, so repeated runs are bitwise identical.
// Padding values at the end of odd-sized blocks are never read.
//
// Small cells: a two-kernel reduction followed by two 8-byte copies cost 10 us of launches for
// a few us of work.  With all the sums of an evaluation in one launch and no copies, the
// reductions of an LNV run of 4 steps at 64 atoms take 53 launches and 0.46 ms (280 launches and
// 1.4 ms before).
#include <algorithm>
#include <cfloat>

#include "cq_internal.cuh"

namespace {

constexpr int RED_T = 256;
// Partials of a quantity and cell.  The sums are those of this many CTAs of eight warps, warp w
// taking every (8 RED_G)th block from block w on; a CTA does the work of NV of them (below), and
// partials without blocks, which would add zeros, are left out.
constexpr int RED_G = 1024;   // one cell, or the whole of several
constexpr int RED_CELL = 64;  // each cell of a batch

enum Op { SUM = 0, MIN = 1, MAX = 2 };

template <int OP>
__device__ __forceinline__ double combine(double a, double b)
{
    if (OP == SUM) return a + b;
    if (OP == MIN) return fmin(a, b);
    return fmax(a, b);
}

template <int OP>
__device__ __forceinline__ double identity_of()
{
    return OP == SUM ? 0.0 : (OP == MIN ? DBL_MAX : -DBL_MAX);
}

// Fixed-shape CTA tree over RED_T values; result valid in thread 0.
template <int OP>
__device__ double cta_reduce(double v)
{
    __shared__ double sh[RED_T / 32];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = combine<OP>(v, __shfl_xor_sync(0xffffffffu, v, o));
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    __syncthreads();
    if (lane == 0) sh[wid] = v;
    __syncthreads();
    if (wid == 0) {
        v = lane < RED_T / 32 ? sh[lane] : identity_of<OP>();
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v = combine<OP>(v, __shfl_xor_sync(0xffffffffu, v, o));
    }
    return v;
}

// Where the partials meet and the scalars go (see red_sink).
struct RedSink {
    double *part;         // per quantity and cell: gridDim.x partials (of NV values)
    uint32_t *count;      // arrivals per quantity and cell, zero between launches
    double *out;          // pinned host scalars, from the first slot on
    const int32_t *flag;  // device error word and its pinned copy
    int32_t *flag_out;
};

// True in every thread of the last CTA of (blockIdx.z, blockIdx.y) to get here; the writers of
// the CTA's partials have fenced them.
__device__ bool last_arrival(const RedSink &k, int64_t unit)
{
    __shared__ int last;
    __syncthreads();
    if (threadIdx.x == 0) {
        last = atomicAdd(&k.count[unit], 1u) == gridDim.x - 1;
        if (last) k.count[unit] = 0;
    }
    __syncthreads();
    if (last) __threadfence();
    return last;
}

__device__ __forceinline__ void publish_flag(const RedSink &k)
{
    *k.flag_out = *k.flag;
}

template <int OP>
__device__ double fold(const double *part, int n, int stride)
{
    double v = identity_of<OP>();
    for (int e = threadIdx.x; e < n; e += RED_T)
        v = combine<OP>(v, __ldcg(part + (int64_t)e * stride));
    return cta_reduce<OP>(v);
}

struct RedItem {
    int kind;  // RedKind
    int64_t nblk;
    const int64_t *seg;  // block ranges of the cells (null: one range)
    const int64_t *a_off, *b_off, *bmap;
    const int32_t *row, *col;
    const double *A, *B;
};

struct RedArgs {
    RedItem it[RED_Q];
    int nv;  // partials of a CTA
    const int32_t *nb;
    RedSink sink;
};

// One CTA's share of a quantity on a uniform basis of NB orbitals: warp per block, as on any basis,
// and the same sums to the bit.  Offsets need no index loads (the blocks of a uniform basis lie at
// a fixed stride) and a lane's elements, transposed ones included, have the same place in every
// block, so a warp keeps four blocks in flight (24 loads per lane for 9 orbitals) and the map of
// the next four arrives meanwhile.  Bound by HBM: a trace and a dot over 4.5 GB each at 4096 atoms
// take 0.73 ms, 6.1 TB/s (1.02 and 0.89 ms with a warp walking one block at a time through its
// index arrays).
template <int KIND, int NB, int NV>
__device__ void sum_uniform(const RedItem &it, int64_t b0, int64_t b1, double (&s)[4])
{
    constexpr int E = NB * NB, ST = (E + 1) & ~1, U = 4, EPL = (E + 31) / 32;
    const int sub = threadIdx.x & 31;
    int te[EPL];
#pragma unroll
    for (int k = 0; k < EPL; ++k) {
        const int e = sub + 32 * k;
        te[k] = KIND == RED_TRACE ? (e % NB) * NB + e / NB : e;
    }
    const int64_t W = (int64_t)gridDim.x * (RED_T / 32);
    const double *__restrict__ A = it.A;
    const double *__restrict__ B = it.B;
    int64_t b = b0 + (int64_t)blockIdx.x * (RED_T / 32) + (threadIdx.x >> 5);
    int64_t t[U];
    auto partner = [&](int64_t x) -> int64_t {
        if (x >= b1) return -1;
        if (KIND == RED_TRACE) return __ldg(it.bmap + x);
        if (KIND == RED_FROB_MI) return it.row[x] == it.col[x];
        return x;
    };
#pragma unroll
    for (int u = 0; u < U; ++u) t[u] = partner(b + u * W);
    while (b < b1) {
        double av[U][EPL], bv[U][EPL];
#pragma unroll
        for (int u = 0; u < U; ++u)
#pragma unroll
            for (int k = 0; k < EPL; ++k) {
                const bool ok = t[u] >= 0 && sub + 32 * k < E;
                av[u][k] = ok ? __ldg(A + (b + u * W) * ST + sub + 32 * k) : 0.0;
                if (KIND == RED_FROB_MI)
                    bv[u][k] = ok && t[u] && (sub + 32 * k) % (NB + 1) == 0 ? 1.0 : 0.0;
                else
                    bv[u][k] = ok ? __ldg(B + t[u] * ST + te[k]) : 0.0;
            }
        b += U * W;
#pragma unroll
        for (int u = 0; u < U; ++u) t[u] = partner(b + u * W);
#pragma unroll
        for (int u = 0; u < U; ++u)
#pragma unroll
            for (int k = 0; k < EPL; ++k) {
                if (KIND == RED_FROB_MI) {
                    const double v = av[u][k] - bv[u][k];
                    s[u % NV] = fma(v, v, s[u % NV]);
                } else {
                    s[u % NV] = fma(av[u][k], bv[u][k], s[u % NV]);
                }
            }
    }
}

// The same on any basis: a warp per block.
template <int KIND>
__device__ double sum_mixed(const RedItem &it, const int32_t *nb, int64_t b0, int64_t b1)
{
    const int lane = threadIdx.x & 31;
    double s = 0.0;
    for (int64_t b = b0 + (int64_t)blockIdx.x * (RED_T / 32) + (threadIdx.x >> 5); b < b1;
         b += (int64_t)gridDim.x * (RED_T / 32)) {
        const int i = it.row[b], j = it.col[b];
        const int ni = nb[i], nj = nb[j];
        const double *a = it.A + it.a_off[b];
        const double *bb = it.B;
        if (KIND == RED_TRACE) {
            const int64_t t = it.bmap[b];
            if (t < 0) continue;
            bb += it.b_off[t];
        } else if (KIND == RED_DOT) {
            bb += it.a_off[b];
        }
        for (int e = lane; e < ni * nj; e += 32) {
            if (KIND == RED_TRACE) {
                const int r = e / nj, q = e - r * nj;
                s = fma(a[e], bb[q * ni + r], s);
            } else if (KIND == RED_DOT) {
                s = fma(a[e], bb[e], s);
            } else {
                double v = a[e];
                if (i == j && (e / nj) == (e % nj)) v -= 1.0;
                s = fma(v, v, s);
            }
        }
    }
    return s;
}

// The sums s[0 .. nv) of the CTA's nv partials: partial i takes the i-th, (i + nv)-th, ... block of
// every warp.
template <int KIND, int NB>
__device__ __forceinline__ void sums_of(const RedArgs &a, const RedItem &it, int64_t b0, int64_t b1,
                                        double (&s)[4])
{
    if constexpr (NB == 0) {
        s[0] = sum_mixed<KIND>(it, a.nb, b0, b1);
    } else {
        if (a.nv == 4)
            sum_uniform<KIND, NB, 4>(it, b0, b1, s);
        else
            sum_uniform<KIND, NB, 1>(it, b0, b1, s);
    }
}

// Quantity blockIdx.z of cell blockIdx.y, NB orbitals per atom (0: any).
template <int NB>
__global__ void __launch_bounds__(RED_T, NB == 9 ? 3 : 4) k_reduce(const __grid_constant__ RedArgs a)
{
    __shared__ double sh[4][RED_T / 32];
    const RedItem &it = a.it[blockIdx.z];
    const int64_t unit = (int64_t)blockIdx.z * gridDim.y + blockIdx.y;
    const int64_t b0 = it.seg ? it.seg[blockIdx.y] : 0;
    const int64_t b1 = it.seg ? it.seg[blockIdx.y + 1] : it.nblk;
    double s[4] = {0.0, 0.0, 0.0, 0.0};
    if (it.kind == RED_TRACE)
        sums_of<RED_TRACE, NB>(a, it, b0, b1, s);
    else if (it.kind == RED_DOT)
        sums_of<RED_DOT, NB>(a, it, b0, b1, s);
    else
        sums_of<RED_FROB_MI, NB>(a, it, b0, b1, s);
    // the tree of cta_reduce for the nv sums side by side (16 lanes hold nothing for 4 orbitals)
#pragma unroll
    for (int o = NB == 4 ? 8 : 16; o > 0; o >>= 1)
#pragma unroll
        for (int i = 0; i < 4; ++i)
            if (i < a.nv) s[i] += __shfl_xor_sync(0xffffffffu, s[i], o);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (lane == 0)
#pragma unroll
        for (int i = 0; i < 4; ++i) sh[i][warp] = s[i];
    __syncthreads();
    double *part = a.sink.part + unit * (gridDim.x * a.nv);
    if (warp < a.nv) {
        double v = lane < RED_T / 32 ? sh[warp][lane] : 0.0;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if (lane == 0) {
            part[blockIdx.x + gridDim.x * warp] = v;
            __threadfence();
        }
    }
    if (!last_arrival(a.sink, unit)) return;
    const double v = fold<SUM>(part, gridDim.x * a.nv, 1);
    if (threadIdx.x == 0) {
        a.sink.out[unit] = v;
        if (unit == 0) publish_flag(a.sink);
    }
}

// Gershgorin data per scalar row: 32 / n_i atom rows per warp (two on a mixed basis), one lane
// per scalar row, which adds its values in the order of the columns (the sums are those of a
// plain loop to the bit).  Bound by the FP64 pipe (an add occupies it 16 clocks a warp) and by
// latency: the values of the next three 9-orbital blocks (six of 4 orbitals, one of a mixed
// basis) are fetched under the sums of these, and the first warps of all CTAs get work before
// the second ones do.  S of 216 atoms: 166 us with a warp per row and a plain loop, 128 with
// the prefetch on 27 CTAs, some 60 spread over 72.
template <int NB>
__global__ void __launch_bounds__(RED_T)
k_row_bounds(int n_atoms, const int32_t *cell_start, const int64_t *rp, const int32_t *col,
             const int32_t *nb, const int64_t *off, const double *M, const RedSink sink)
{
    constexpr int W = NB ? NB : 16, U = NB ? 27 / NB : 1, ST = (NB * NB + 1) & ~1, PER = 32 / W;
    const int sub = (threadIdx.x & 31) / W, lane = (threadIdx.x & 31) % W;
    const int i1 = cell_start ? cell_start[blockIdx.y + 1] : n_atoms;
    double lo = DBL_MAX, hi = -DBL_MAX, amax = 0.0;
    for (int i = (cell_start ? cell_start[blockIdx.y] : 0) +
                 PER * (blockIdx.x + gridDim.x * (threadIdx.x >> 5)) + sub;
         i < i1 && sub < PER; i += PER * gridDim.x * (RED_T / 32)) {
        const int ni = NB ? NB : nb[i];
        if (lane >= ni) continue;
        const int64_t b1 = rp[i + 1];
        double v[U][W], w[U][W];
        int j[U], nj[U], jw[U], njw[U];  // column atom, its orbitals (0 past the row's end)
        auto load = [&](int64_t b, double (&x)[U][W], int (&jx)[U], int (&nx)[U]) {
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const bool ok = b + u < b1;
                jx[u] = ok ? __ldg(col + b + u) : -1;
                nx[u] = !ok ? 0 : NB ? NB : __ldg(nb + jx[u]);
                const double *m = M + (!ok ? 0 : (NB ? (b + u) * ST : __ldg(off + b + u)) +
                                                     lane * nx[u]);
#pragma unroll
                for (int q = 0; q < W; ++q) x[u][q] = q < nx[u] ? __ldg(m + q) : 0.0;
            }
        };
        double centre = 0.0, rad = 0.0, tot = 0.0;
        int64_t b = rp[i];
        load(b, v, j, nj);
        while (b < b1) {
            b += U;
            load(b, w, jw, njw);
#pragma unroll
            for (int u = 0; u < U; ++u)
#pragma unroll
                for (int q = 0; q < W; ++q) {
                    if (q < nj[u]) {
                        tot += fabs(v[u][q]);
                        if (j[u] == i && q == lane)
                            centre = v[u][q];
                        else
                            rad += fabs(v[u][q]);
                    }
                }
#pragma unroll
            for (int u = 0; u < U; ++u) {
                j[u] = jw[u];
                nj[u] = njw[u];
#pragma unroll
                for (int q = 0; q < W; ++q) v[u][q] = w[u][q];
            }
        }
        lo = fmin(lo, centre - rad);
        hi = fmax(hi, centre + rad);
        amax = fmax(amax, tot);
    }
    lo = cta_reduce<MIN>(lo);
    hi = cta_reduce<MAX>(hi);
    amax = cta_reduce<MAX>(amax);
    double *part = sink.part + 3 * (int64_t)blockIdx.y * gridDim.x;
    if (threadIdx.x == 0) {
        part[3 * blockIdx.x + 0] = lo;
        part[3 * blockIdx.x + 1] = hi;
        part[3 * blockIdx.x + 2] = amax;
        __threadfence();
    }
    if (!last_arrival(sink, blockIdx.y)) return;
    lo = fold<MIN>(part + 0, gridDim.x, 3);
    hi = fold<MAX>(part + 1, gridDim.x, 3);
    amax = fold<MAX>(part + 2, gridDim.x, 3);
    if (threadIdx.x == 0) {
        double *o = sink.out + 3 * blockIdx.y;
        o[0] = lo;
        o[1] = hi;
        o[2] = amax;
        if (blockIdx.y == 0) publish_flag(sink);
    }
}

// y <- a x + b z (y may be x or z; b == 0: z not read)
__global__ void k_lincomb(int64_t n, double a, const double *x, double b, const double *z,
                          double *y)
{
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < n;
         e += (int64_t)gridDim.x * blockDim.x)
        y[e] = (b == 0.0) ? a * x[e] : a * x[e] + b * z[e];
}

// dst_b = s * (src_ij or src_ji^T) + bb * dst_b; warp per destination block.
__global__ void k_gather(int64_t nblk, const int32_t *row, const int32_t *col,
                         const int32_t *nb, const int64_t *d_off, const int64_t *s_off,
                         const int64_t *map, int transpose, const double *src, double *dst,
                         double s, double bb)
{
    const int64_t b = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    const int lane = threadIdx.x & 31;
    if (b >= nblk) return;
    const int ni = nb[row[b]], nj = nb[col[b]];
    const int64_t m = map[b];
    double *d = dst + d_off[b];
    for (int e = lane; e < ni * nj; e += 32) {
        double v = 0.0;
        if (m >= 0) {
            const int r = e / nj, q = e - r * nj;
            v = transpose ? src[s_off[m] + q * ni + r] : src[s_off[m] + e];
        }
        d[e] = (bb == 0.0) ? s * v : s * v + bb * d[e];
    }
}

__global__ void k_identity(int n_atoms, const int64_t *rp, const int32_t *col,
                           const int32_t *nb, const int64_t *off, double *M, double s)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n_atoms) return;
    int64_t lo = rp[i], hi = rp[i + 1];
    while (lo < hi) {
        int64_t mid = (lo + hi) >> 1;
        if (col[mid] < i)
            lo = mid + 1;
        else
            hi = mid;
    }
    const int ni = nb[i];
    for (int r = 0; r < ni; ++r) M[off[lo] + r * ni + r] = s;
}

__global__ void k_lnv_grad_n(int64_t nblk, const int32_t *row, const int32_t *col,
                             const int32_t *nb, const int64_t *l_off, const int64_t *u_off,
                             const int64_t *map_u, const double *U, const double *R3,
                             double *GN)
{
    const int64_t b = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    const int lane = threadIdx.x & 31;
    if (b >= nblk) return;
    const int sz = nb[row[b]] * nb[col[b]];
    const int64_t lb = l_off[b], zb = map_u[b];
    for (int e = lane; e < sz; e += 32) {
        const double u = zb >= 0 ? U[u_off[zb] + e] : 0.0;
        GN[lb + e] = 12.0 * (u - R3[lb + e]);
    }
}

__global__ void k_lnv_grad_e(int64_t nblk, const int32_t *row, const int32_t *col,
                             const int32_t *nb, const int64_t *l_off, const int64_t *l_tr,
                             const int64_t *u_off, const int64_t *map_u, const int64_t *map_ut,
                             const double *Z, const double *R1, const double *R2, double *GE)
{
    const int64_t b = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    const int lane = threadIdx.x & 31;
    if (b >= nblk) return;
    const int ni = nb[row[b]], nj = nb[col[b]];
    const int64_t lb = l_off[b], lt = l_off[l_tr[b]];
    const int64_t zb = map_u[b], zt = map_ut[b];
    for (int e = lane; e < ni * nj; e += 32) {
        const int r = e / nj, q = e - r * nj;
        const double z = zb >= 0 ? Z[u_off[zb] + e] : 0.0;
        const double zT = zt >= 0 ? Z[u_off[zt] + q * ni + r] : 0.0;
        const double t = (R1[lb + e] + R1[lt + q * ni + r]) + R2[lb + e];
        GE[lb + e] = 2.0 * (3.0 * (z + zT) - 2.0 * t);
    }
}

// ---------------- per-cell versions: blockIdx.y = cell

__global__ void k_lincomb_seg(const int64_t *seg_val, const double *coef, int n_cells,
                              const double *x, const double *z, double *y)
{
    const int c = blockIdx.y;
    const double a = coef[c], b = coef[n_cells + c];
    const int64_t v1 = seg_val[c + 1];
    for (int64_t e = seg_val[c] + (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < v1;
         e += (int64_t)gridDim.x * blockDim.x)
        y[e] = (b == 0.0) ? a * x[e] : a * x[e] + b * z[e];
}

__global__ void k_identity_seg(int n_atoms, const int32_t *cell_of, const int64_t *rp,
                               const int32_t *col, const int32_t *nb, const int64_t *off,
                               const double *scale, double *M)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n_atoms) return;
    int64_t lo = rp[i], hi = rp[i + 1];
    while (lo < hi) {
        int64_t mid = (lo + hi) >> 1;
        if (col[mid] < i)
            lo = mid + 1;
        else
            hi = mid;
    }
    const int ni = nb[i];
    const double s = scale[cell_of[i]];
    for (int r = 0; r < ni; ++r) M[off[lo] + r * ni + r] = s;
}

// Sink of a reduction over `cells` units per quantity whose scalars start at `slot`, and the
// CTAs of a unit with `work` CTAs' worth of items.
cq_status red_sink(cq_ctx *ctx, int cells, int64_t work, int slot, RedSink *k, unsigned *ctas)
{
    const int64_t cap = cells == 1 ? RED_G : RED_CELL;
    void *p;
    cq_status st = cq_scratch(ctx, "red_part", sizeof(double) * RED_Q * cap * cells, &p);
    k->part = (double *)p;
    k->count = ctx->red_count.as<uint32_t>();
    k->out = ctx->host_out + slot;
    k->flag = ctx->flag.as<int32_t>();
    k->flag_out = reinterpret_cast<int32_t *>(ctx->host_out + CQ_RED_SLOTS - 1);
    *ctas = (unsigned)std::min(cap, std::max<int64_t>(1, work));
    return st;
}

}  // namespace

cq_status cq_reduce(cq_ctx *ctx, int nq, const RedQ *q, bool per_cell, int slot)
{
    const int nc = per_cell ? q[0].pA->n_cells() : 1;
    const int nbu = q[0].pA->geo->uniform_nb;
    RedArgs a = {};
    int64_t nblk = 0;
    for (int e = 0; e < nq; ++e) {
        RedItem &it = a.it[e];
        const cq_pattern *pA = q[e].pA;
        it.kind = q[e].kind;
        it.nblk = pA->n_blocks;
        it.seg = nc > 1 ? pA->seg_blk_dev.as<int64_t>() : nullptr;
        it.a_off = pA->val_off.as<int64_t>();
        it.row = pA->row.as<int32_t>();
        it.col = pA->col.as<int32_t>();
        it.A = q[e].A;
        it.B = q[e].B;
        if (it.kind == RED_TRACE) {
            cq_status st = cq_get_map(ctx, q[e].pB, pA, 1, &it.bmap);
            if (st != CQ_OK) return st;
            it.b_off = q[e].pB->val_off.as<int64_t>();
        }
        nblk = std::max(nblk, it.nblk);
    }
    a.nb = q[0].pA->geo->nb.as<int32_t>();
    unsigned ctas;
    cq_status st = red_sink(ctx, nc, nc > 1 ? RED_CELL : (nblk + 7) / 8, slot, &a.sink, &ctas);
    if (st != CQ_OK) return st;
    // one cell on a kernel of its basis: four partials per CTA, so that all CTAs (256 at most) are
    // resident and a warp has four blocks in flight even if it has no more than four; the kernel
    // for any basis makes one
    a.nv = nc == 1 && (nbu == 9 || nbu == 4) ? 4 : 1;
    ctas = (ctas + a.nv - 1) / a.nv;
    const dim3 grid(ctas, (unsigned)nc, (unsigned)nq);
    if (nbu == 9)
        k_reduce<9><<<grid, RED_T, 0, ctx->stream>>>(a);
    else if (nbu == 4)
        k_reduce<4><<<grid, RED_T, 0, ctx->stream>>>(a);
    else
        k_reduce<0><<<grid, RED_T, 0, ctx->stream>>>(a);
    cq_count_launch();
    return cq_check_cuda(ctx, cudaGetLastError(), "reduction");
}

cq_status cq_row_bounds_dev(cq_ctx *ctx, const cq_pattern *p, const double *M, bool per_cell,
                            int slot)
{
    const int nc = per_cell ? p->n_cells() : 1;
    const int nbu = p->geo->uniform_nb;
    const int per = nbu == 9 ? 3 : nbu == 4 ? 8 : 2;  // atom rows of a warp
    RedSink sink;
    unsigned ctas;
    cq_status st = red_sink(ctx, nc, (p->geo->n_atoms / nc + per - 1) / per, slot, &sink, &ctas);
    if (st != CQ_OK) return st;
    auto kernel = nbu == 9 ? k_row_bounds<9> : nbu == 4 ? k_row_bounds<4> : k_row_bounds<0>;
    kernel<<<dim3(ctas, (unsigned)nc), RED_T, 0, ctx->stream>>>(
        p->geo->n_atoms, nc > 1 ? p->geo->cell_start_dev.as<int32_t>() : nullptr,
        p->row_ptr.as<int64_t>(), p->col.as<int32_t>(), p->geo->nb.as<int32_t>(),
        p->val_off.as<int64_t>(), M, sink);
    cq_count_launch();
    return cq_check_cuda(ctx, cudaGetLastError(), "row bounds");
}

cq_status cq_lincomb(cq_ctx *ctx, int64_t n, double a, const double *x, double b, const double *z,
                     double *y)
{
    if (n == 0) return CQ_OK;
    int64_t blocks = (n + 255) / 256;
    const int64_t cap = (int64_t)ctx->num_sms * 16;
    if (blocks > cap) blocks = cap;
    k_lincomb<<<(unsigned)blocks, 256, 0, ctx->stream>>>(n, a, x, b, z, y);
    cq_count_launch();
    return cq_check_cuda(ctx, cudaGetLastError(), "lincomb");
}

cq_status cq_gather(cq_ctx *ctx, const cq_pattern *pSrc, const double *src,
                    const cq_pattern *pDst, double *dst, int transpose, double s, double b)
{
    const int64_t *map;
    cq_status st = cq_get_map(ctx, pSrc, pDst, transpose, &map);
    if (st != CQ_OK) return st;
    if (pDst->n_blocks == 0) return CQ_OK;
    k_gather<<<(unsigned)((pDst->n_blocks + 7) / 8), 256, 0, ctx->stream>>>(
        pDst->n_blocks, pDst->row.as<int32_t>(), pDst->col.as<int32_t>(),
        pDst->geo->nb.as<int32_t>(), pDst->val_off.as<int64_t>(), pSrc->val_off.as<int64_t>(), map,
        transpose, src, dst, s, b);
    cq_count_launch();
    return cq_check_cuda(ctx, cudaGetLastError(), "gather");
}

cq_status cq_set_identity(cq_ctx *ctx, const cq_pattern *p, double *M, double s)
{
    cq_status st = cq_check_cuda(ctx, cudaMemsetAsync(M, 0, sizeof(double) * p->n_values,
                                                      ctx->stream), "identity");
    if (st != CQ_OK) return st;
    const int n = p->geo->n_atoms;
    k_identity<<<(n + 127) / 128, 128, 0, ctx->stream>>>(n, p->row_ptr.as<int64_t>(),
                                                        p->col.as<int32_t>(),
                                                        p->geo->nb.as<int32_t>(),
                                                        p->val_off.as<int64_t>(), M, s);
    cq_count_launch();
    return cq_check_cuda(ctx, cudaGetLastError(), "identity");
}

// ---------------------------------------------------------------- per-cell host wrappers

cq_status cq_lincomb_seg(cq_ctx *ctx, const cq_pattern *p, const double *a, const double *x,
                         const double *b, const double *z, double *y)
{
    const int nc = p->n_cells();
    void *v;
    cq_status st = cq_scratch(ctx, "seg_coef", sizeof(double) * 2 * nc, &v);
    if (st != CQ_OK) return st;
    std::vector<double> coef(a, a + nc);
    coef.insert(coef.end(), b, b + nc);
    cudaMemcpyAsync(v, coef.data(), sizeof(double) * 2 * nc, cudaMemcpyHostToDevice, ctx->stream);
    k_lincomb_seg<<<dim3(64, nc), 256, 0, ctx->stream>>>(p->seg_val_dev.as<int64_t>(), (double *)v,
                                                         nc, x, z, y);
    cq_count_launch();
    return cq_check_cuda(ctx, cudaGetLastError(), "lincomb (cells)");
}

cq_status cq_set_identity_seg(cq_ctx *ctx, const cq_pattern *p, double *M, const double *s)
{
    const int nc = p->n_cells();
    cq_status st = cq_check_cuda(ctx, cudaMemsetAsync(M, 0, sizeof(double) * p->n_values,
                                                      ctx->stream), "identity");
    if (st != CQ_OK) return st;
    void *v;
    if ((st = cq_scratch(ctx, "seg_scale", sizeof(double) * nc, &v)) != CQ_OK) return st;
    cudaMemcpyAsync(v, s, sizeof(double) * nc, cudaMemcpyHostToDevice, ctx->stream);
    const int n = p->geo->n_atoms;
    k_identity_seg<<<(n + 127) / 128, 128, 0, ctx->stream>>>(
        n, p->geo->cell_of.as<int32_t>(), p->row_ptr.as<int64_t>(), p->col.as<int32_t>(),
        p->geo->nb.as<int32_t>(), p->val_off.as<int64_t>(), (const double *)v, M);
    cq_count_launch();
    return cq_check_cuda(ctx, cudaGetLastError(), "identity (cells)");
}

cq_status cq_lnv_gradient_n(cq_ctx *ctx, const cq_pattern *pL, const cq_pattern *pU,
                            const double *U, const double *R3, double *GN)
{
    const int64_t *mu;
    cq_status st = cq_get_map(ctx, pU, pL, 0, &mu);
    if (st != CQ_OK) return st;
    if (pL->n_blocks == 0) return CQ_OK;
    k_lnv_grad_n<<<(unsigned)((pL->n_blocks + 7) / 8), 256, 0, ctx->stream>>>(
        pL->n_blocks, pL->row.as<int32_t>(), pL->col.as<int32_t>(), pL->geo->nb.as<int32_t>(),
        pL->val_off.as<int64_t>(), pU->val_off.as<int64_t>(), mu, U, R3, GN);
    cq_count_launch();
    return cq_check_cuda(ctx, cudaGetLastError(), "lnv gradient N");
}

cq_status cq_lnv_gradient_e(cq_ctx *ctx, const cq_pattern *pL, const cq_pattern *pU,
                            const double *Z, const double *R1, const double *R2, double *GE)
{
    const int64_t *mu, *mut;
    cq_status st = cq_get_map(ctx, pU, pL, 0, &mu);
    if (st != CQ_OK) return st;
    if ((st = cq_get_map(ctx, pU, pL, 1, &mut)) != CQ_OK) return st;
    if (pL->n_blocks == 0) return CQ_OK;
    k_lnv_grad_e<<<(unsigned)((pL->n_blocks + 7) / 8), 256, 0, ctx->stream>>>(
        pL->n_blocks, pL->row.as<int32_t>(), pL->col.as<int32_t>(), pL->geo->nb.as<int32_t>(),
        pL->val_off.as<int64_t>(), pL->transpose.as<int64_t>(), pU->val_off.as<int64_t>(), mu,
        mut, Z, R1, R2, GE);
    cq_count_launch();
    return cq_check_cuda(ctx, cudaGetLastError(), "lnv gradient E");
}

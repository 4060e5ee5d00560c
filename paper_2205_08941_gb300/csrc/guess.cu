// Learned initial guess for the density matrix L: a small MLP maps a descriptor of each atom
// pair's local environment to the pair's L block expressed in a pair frame; the block is
// rotated back to the global orbital frame.  Hand-written kernels: descriptors and frames,
// target extraction (global -> frame), MLP forward/backward (BF16 weights, FP32
// accumulation), Adam, and the apply step (frame -> global, both (i,j) and (j,i) blocks).
//
// Pair frame (i, j), i != j: e3 along r_j - r_i; e1 toward the atom nearest to the bond
// midpoint (other than i, j; ties: lowest index), made orthogonal to e3; e2 = e3 x e1.
// On-site (i, i): e3 toward i's nearest neighbour, e1 toward its second nearest.  Only
// blocks with i <= j are predicted; (j, i) is the transpose.  Uniform 9- or 4-orbital bases.
//
// Descriptor (64 numbers): 10 Gaussians of the pair distance (centres 1.6 p bohr, width
// 1.6) and, for the atoms k within 8 bohr of the midpoint m (k != i, j), sum_k h_n(|r_k - m|)
// Y_a(unit(r_k - m) in the pair frame) for 6 radial Gaussians h_n (centres 1.6 n, width
// 1.2, cosine cut at 8) and the 9 real harmonics Y_a up to l = 2.
#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>
#include <random>

#include "cq_internal.cuh"

#define CQ_TRY(x)                          \
    do {                                   \
        cq_status _st = (x);               \
        if (_st != CQ_OK) return _st;      \
    } while (0)

namespace {

constexpr int NDESC = 64;
constexpr int NOUT = 81;
constexpr float R_ENV = 8.0f;

struct Box3 {
    double v[3];
};

__device__ __forceinline__ void min_image(const double *pos, const Box3 &box, int i, int j,
                                          double d[3])
{
    for (int c = 0; c < 3; ++c) {
        double x = pos[3 * j + c] - pos[3 * i + c];
        d[c] = x - box.v[c] * rint(x / box.v[c]);
    }
}

__device__ __forceinline__ void normalize3(double v[3])
{
    const double n = sqrt(v[0] * v[0] + v[1] * v[1] + v[2] * v[2]);
    for (int c = 0; c < 3; ++c) v[c] /= n;
}

// Real d orbitals as unit-Frobenius quadratic forms (xy, yz, zx, x2-y2, 3z2-r2).
__device__ void dform(int a, double q[3][3])
{
    for (int r = 0; r < 3; ++r)
        for (int c = 0; c < 3; ++c) q[r][c] = 0.0;
    const double h = 0.70710678118654752440, s6 = 0.40824829046386301637;
    switch (a) {
    case 0: q[0][1] = q[1][0] = h; break;
    case 1: q[1][2] = q[2][1] = h; break;
    case 2: q[2][0] = q[0][2] = h; break;
    case 3: q[0][0] = h; q[1][1] = -h; break;
    default: q[0][0] = q[1][1] = -s6; q[2][2] = 2.0 * s6; break;
    }
}

// Orbital rotation D (local <- global) for a frame with rows R = (e1, e2, e3):
// s -> 1, p -> R, d -> D2[a][b] = <Q_b, R^T Q_a R>_F.
__device__ void orbital_rotation(const double R[3][3], int nb, double D[9][9])
{
    for (int a = 0; a < 9; ++a)
        for (int b = 0; b < 9; ++b) D[a][b] = 0.0;
    D[0][0] = 1.0;
    for (int a = 0; a < 3; ++a)
        for (int b = 0; b < 3; ++b) D[1 + a][1 + b] = R[a][b];
    if (nb < 9) return;
    for (int a = 0; a < 5; ++a) {
        double qa[3][3], t[3][3];
        dform(a, qa);
        for (int r = 0; r < 3; ++r)
            for (int c = 0; c < 3; ++c) {
                double acc = 0.0;
                for (int u = 0; u < 3; ++u)
                    for (int v = 0; v < 3; ++v) acc += R[u][r] * qa[u][v] * R[v][c];
                t[r][c] = acc;
            }
        for (int b = 0; b < 5; ++b) {
            double qb[3][3];
            dform(b, qb);
            double acc = 0.0;
            for (int r = 0; r < 3; ++r)
                for (int c = 0; c < 3; ++c) acc += qb[r][c] * t[r][c];
            D[4 + a][4 + b] = acc;
        }
    }
}

constexpr float R_ENV2_F = R_ENV * R_ENV + 0.1f;  // FP32 distances that may be within R_ENV
// upper word of R_ENV^2 as a double: a squared distance is below it when its upper word is (a compare
// of integers, off the FP64 pipe: 8 of the 1456 us of an apply on 1728 atoms)
constexpr int R_ENV2_HI = 0x40500000;
static_assert(R_ENV * R_ENV == 64.0f, "the upper word of 64.0");

// Radial and angular values of an atom at w from the midpoint (distance rho) in the frame
// (e1, e2, e3)
__device__ __forceinline__ void env_values(const double (&w)[3], const double (&e1)[3],
                                           const double (&e2)[3], const double (&e3)[3], float rho,
                                           float (&h)[6], float (&ang)[9])
{
    const float x = (float)((w[0] * e1[0] + w[1] * e1[1] + w[2] * e1[2]) / rho);
    const float y = (float)((w[0] * e2[0] + w[1] * e2[1] + w[2] * e2[2]) / rho);
    const float z = (float)((w[0] * e3[0] + w[1] * e3[1] + w[2] * e3[2]) / rho);
    ang[0] = 1.f;
    ang[1] = z;
    ang[2] = x;
    ang[3] = y;
    ang[4] = 0.5f * (3.f * z * z - 1.f);
    ang[5] = x * z;
    ang[6] = y * z;
    ang[7] = 0.5f * fmaf(x, x, -__fmul_rn(y, y));
    ang[8] = x * y;
    const float fc = 0.5f * (1.f + __cosf(3.14159265f * rho / R_ENV));
#pragma unroll
    for (int n = 0; n < 6; ++n) {
        const float t = (rho - 1.6f * n) / 1.2f;
        h[n] = __expf(-0.5f * t * t) * fc;
    }
}

// Neighbour e of an atom row: displacement from the row's atom and atom index, from shared memory
// (CACHED: filled once per row) or computed from the positions (rows too long to cache).
template <bool CACHED>
struct RowAtoms {
    int i, n;                 // the row's atom, its neighbours
    const int32_t *cols;      // neighbour atoms
    const double *d;          // cached displacements (n x 3)
    const float *df;          // the same in FP32
    const double *pos;
    Box3 box;
    __device__ __forceinline__ void disp(int e, double (&v)[3]) const
    {
        if (CACHED) {
            v[0] = d[3 * e];
            v[1] = d[3 * e + 1];
            v[2] = d[3 * e + 2];
        } else {
            min_image(pos, box, i, cols[e], v);
        }
    }
    __device__ __forceinline__ void dispf(int e, float (&v)[3]) const
    {
        if (CACHED) {
            v[0] = df[3 * e];
            v[1] = df[3 * e + 1];
            v[2] = df[3 * e + 2];
        } else {
            double w[3];
            min_image(pos, box, i, cols[e], w);
            for (int c = 0; c < 3; ++c) v[c] = (float)w[c];
        }
    }
};

constexpr int DESC_T = 256, DESC_PAIRS = 64;  // threads and pairs at a time of k_descriptors
constexpr int DESC_SMEM = 96 * 1024;  // its shared memory at most (two CTAs per SM)

struct DescShared {
    double e1[DESC_PAIRS][3], e2[DESC_PAIRS][3], e3[DESC_PAIRS][3], m[DESC_PAIRS][3];
    float rij[DESC_PAIRS];
    int je[DESC_PAIRS];              // the pair's second atom as a neighbour of the row (or -1)
    int sel[DESC_PAIRS];             // third atom (neighbour index, -1: none)
    int near;                        // nearest neighbour of the row's atom
    int queue[DESC_T / 32][64];      // neighbours waiting for a warp's next batch
    float hb[DESC_T / 32][32][17];   // per batch entry: 6 radial and 9 angular values
};

// Calls f(e, k) for the neighbours e (k = their atom) that pass `want`, a full warp of
// them at a time in ascending order (lanes without one get e = -1).
template <bool CACHED, class W, class F>
__device__ __forceinline__ void for_neighbours(const RowAtoms<CACHED> &row, int *queue, W want, F f)
{
    const int lane = threadIdx.x & 31;
    int held = 0;
    for (int base = 0; base < row.n; base += 32) {
        const int e = base + lane;
        const bool hit = e < row.n && want(e);
        const unsigned mask = __ballot_sync(0xffffffffu, hit);
        if (hit) queue[held + __popc(mask & ((1u << lane) - 1u))] = e;
        held += __popc(mask);
        __syncwarp();
        if (held >= 32) {
            f(queue[lane]);
            __syncwarp();
            held -= 32;
            const int rest = lane < held ? queue[32 + lane] : 0;
            __syncwarp();
            queue[lane] = rest;
            __syncwarp();
        }
    }
    if (held > 0) f(lane < held ? queue[lane] : -1);
    __syncwarp();
}

// smallest (r2, atom) over a warp; returns its neighbour index (-1 when no lane has one)
__device__ __forceinline__ int warp_nearest(double r2, int atom, int e)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const double r = __shfl_xor_sync(0xffffffffu, r2, o);
        const int a = __shfl_xor_sync(0xffffffffu, atom, o), q = __shfl_xor_sync(0xffffffffu, e, o);
        if (q >= 0 && (e < 0 || r < r2 || (r == r2 && a < atom))) {
            r2 = r;
            atom = a;
            e = q;
        }
    }
    return e;
}

// Frames and descriptors of the pair blocks (i, j), i <= j, of one atom row i of P_L (one CTA).
// pair0[b] counts the pair blocks before block b.
//
// Bound by the FP64 pipe (two lanes per clock and SM), on which one thread per pair spent 5.0
// ms for a 1728-atom cell: two minimum images with divisions per (pair, atom), distances and
// square roots of all of the row's atoms.  Here the displacements are made once per row, an
// FP32 distance keeps the sixth of the atoms that can lie within 8 bohr of the midpoint, and
// only they get the FP64 geometry; normalisations run a lane per pair, the sums over atoms a
// lane per (radial, angular) entry in the order of the atoms.
template <bool CACHED>
__global__ void __launch_bounds__(DESC_T)
k_descriptors(const int64_t *pair0, const int32_t *pairs, const int32_t *col, const int64_t *rp,
              const double *pos, Box3 box, float *desc, float *frames)
{
    extern __shared__ __align__(16) uint8_t dyn[];
    DescShared &sh = *reinterpret_cast<DescShared *>(dyn);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    RowAtoms<CACHED> row;
    row.i = blockIdx.x;
    const int64_t b0 = rp[row.i];
    row.n = (int)(rp[row.i + 1] - b0);
    row.pos = pos;
    row.box = box;
    row.cols = col + b0;
    if (CACHED) {
        double *d = reinterpret_cast<double *>(dyn + sizeof(DescShared));
        float *df = reinterpret_cast<float *>(d + 3 * row.n);
        int32_t *cols = reinterpret_cast<int32_t *>(df + 3 * row.n);
        for (int e = threadIdx.x; e < row.n; e += DESC_T) {
            const int k = col[b0 + e];
            double v[3];
            min_image(pos, box, row.i, k, v);
            for (int c = 0; c < 3; ++c) {
                d[3 * e + c] = v[c];
                df[3 * e + c] = (float)v[c];
            }
            cols[e] = k;
        }
        row.d = d;
        row.df = df;
        row.cols = cols;
        __syncthreads();
    }
    const int i = row.i;
    if (warp == 0) {  // nearest neighbour of i: e3 of the on-site pair
        double best = 1e300;
        int kb = -1, eb = -1;
        for (int e = lane; e < row.n; e += 32) {
            const int k = row.cols[e];
            if (k == i) continue;
            double d[3];
            row.disp(e, d);
            const double r2 = d[0] * d[0] + d[1] * d[1] + d[2] * d[2];
            if (r2 < best || (r2 == best && k < kb)) {
                best = r2;
                kb = k;
                eb = e;
            }
        }
        eb = warp_nearest(best, kb, eb);
        if (lane == 0) sh.near = eb;
    }
    __syncthreads();
    const int64_t p1 = pair0[rp[i + 1]];
    for (int64_t p0 = pair0[b0]; p0 < p1; p0 += DESC_PAIRS) {
        const int np = (int)min((int64_t)DESC_PAIRS, p1 - p0);
        if (threadIdx.x < np) {  // a lane per pair: bond direction and midpoint
            const int t = threadIdx.x, je = (int)(pairs[p0 + t] - b0);
            double e3[3] = {0.0, 0.0, 1.0}, dij[3] = {0.0, 0.0, 0.0};
            if (row.cols[je] != i) {
                row.disp(je, dij);
                for (int c = 0; c < 3; ++c) e3[c] = dij[c];
            } else if (sh.near >= 0) {
                row.disp(sh.near, e3);
            }
            normalize3(e3);
            for (int c = 0; c < 3; ++c) {
                sh.e3[t][c] = e3[c];
                sh.m[t][c] = 0.5 * dij[c];
            }
            sh.rij[t] = (float)sqrt(dij[0] * dij[0] + dij[1] * dij[1] + dij[2] * dij[2]);
            sh.je[t] = je;
        }
        __syncthreads();
        // a warp per pair: the third atom, nearest to the midpoint and off the axis
        for (int t = warp; t < np; t += DESC_T / 32) {
            const int je = sh.je[t];
            const double m[3] = {sh.m[t][0], sh.m[t][1], sh.m[t][2]};
            const double e3[3] = {sh.e3[t][0], sh.e3[t][1], sh.e3[t][2]};
            const float mf[3] = {(float)m[0], (float)m[1], (float)m[2]};
            double best = 1e300;
            int kb = -1, eb = -1;
            auto look = [&](int e) {
                if (e < 0) return;
                double d[3];
                row.disp(e, d);
                const double w[3] = {d[0] - m[0], d[1] - m[1], d[2] - m[2]};
                const double along = w[0] * e3[0] + w[1] * e3[1] + w[2] * e3[2];
                const double perp[3] = {w[0] - along * e3[0], w[1] - along * e3[1],
                                        w[2] - along * e3[2]};
                if (perp[0] * perp[0] + perp[1] * perp[1] + perp[2] * perp[2] < 1e-12) return;
                const double r2 = w[0] * w[0] + w[1] * w[1] + w[2] * w[2];
                const int k = row.cols[e];
                if (r2 < best || (r2 == best && k < kb)) {
                    best = r2;
                    kb = k;
                    eb = e;
                }
            };
            for_neighbours(row, sh.queue[warp],
                           [&](int e) {
                               float v[3];
                               row.dispf(e, v);
                               const float x = v[0] - mf[0], y = v[1] - mf[1], z = v[2] - mf[2];
                               return x * x + y * y + z * z < R_ENV2_F && e != je && row.cols[e] != i;
                           },
                           look);
            // none within R_ENV for certain (the FP32 filter decides beyond it): look at all of them
            if (!__any_sync(0xffffffffu, __double2hiint(best) < R_ENV2_HI))
                for (int base = 0; base < row.n; base += 32) {
                    const int e = base + lane;
                    look(e < row.n && e != je && row.cols[e] != i ? e : -1);
                }
            eb = warp_nearest(best, kb, eb);
            if (lane == 0) sh.sel[t] = eb;
        }
        __syncthreads();
        if (threadIdx.x < np) {  // a lane per pair: the frame
            const int t = threadIdx.x, sel = sh.sel[t];
            double e3[3], e1[3];
            for (int c = 0; c < 3; ++c) e3[c] = sh.e3[t][c];
            if (sel >= 0) {
                double d[3];
                row.disp(sel, d);
                const double w[3] = {d[0] - sh.m[t][0], d[1] - sh.m[t][1], d[2] - sh.m[t][2]};
                const double along = w[0] * e3[0] + w[1] * e3[1] + w[2] * e3[2];
                const double perp[3] = {w[0] - along * e3[0], w[1] - along * e3[1],
                                        w[2] - along * e3[2]};
                const double pn = sqrt(perp[0] * perp[0] + perp[1] * perp[1] + perp[2] * perp[2]);
                for (int c = 0; c < 3; ++c) e1[c] = perp[c] / pn;
            } else {  // no off-axis atom: any perpendicular
                const double h[3] = {fabs(e3[0]) < 0.9 ? 1.0 : 0.0, fabs(e3[0]) < 0.9 ? 0.0 : 1.0, 0.0};
                const double along = h[0] * e3[0] + h[1] * e3[1] + h[2] * e3[2];
                for (int c = 0; c < 3; ++c) e1[c] = h[c] - along * e3[c];
                normalize3(e1);
            }
            const double e2[3] = {e3[1] * e1[2] - e3[2] * e1[1], e3[2] * e1[0] - e3[0] * e1[2],
                                  e3[0] * e1[1] - e3[1] * e1[0]};
            float *fr = frames + (p0 + t) * 9;
            for (int c = 0; c < 3; ++c) {
                fr[c] = (float)e1[c];
                fr[3 + c] = (float)e2[c];
                fr[6 + c] = (float)e3[c];
                sh.e1[t][c] = e1[c];
                sh.e2[t][c] = e2[c];
            }
        }
        __syncthreads();
        // a warp per pair: the descriptor; lane c sums the (radial, angular) entries c and c + 32
        for (int t = warp; t < np; t += DESC_T / 32) {
            const int je = sh.je[t];
            const double m[3] = {sh.m[t][0], sh.m[t][1], sh.m[t][2]};
            const float mf[3] = {(float)m[0], (float)m[1], (float)m[2]};
            const int n0 = lane / 9, a0 = lane % 9, c1 = min(lane + 32, 53), n1 = c1 / 9, a1 = c1 % 9;
            float f0 = 0.f, f1 = 0.f;
            for_neighbours(
                row, sh.queue[warp],
                [&](int e) {
                    float v[3];
                    row.dispf(e, v);
                    const float x = v[0] - mf[0], y = v[1] - mf[1], z = v[2] - mf[2];
                    return x * x + y * y + z * z < R_ENV2_F && e != je && row.cols[e] != i;
                },
                [&](int e) {
                    float *o = sh.hb[warp][lane];
                    float h[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
                    float ang[9] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
                    if (e >= 0) {
                        double d[3];
                        row.disp(e, d);
                        const double w[3] = {d[0] - m[0], d[1] - m[1], d[2] - m[2]};
                        const float rho = (float)sqrt(w[0] * w[0] + w[1] * w[1] + w[2] * w[2]);
                        if (!(rho >= R_ENV || rho < 1e-6f))
                            env_values(w, sh.e1[t], sh.e2[t], sh.e3[t], rho, h, ang);
                    }
#pragma unroll
                    for (int n = 0; n < 6; ++n) o[n] = h[n];
#pragma unroll
                    for (int a = 0; a < 9; ++a) o[6 + a] = ang[a];
                    __syncwarp();
                    const int cnt = __popc(__ballot_sync(0xffffffffu, e >= 0));
                    for (int q = 0; q < cnt; ++q) {
                        const float *v = sh.hb[warp][q];
                        f0 = fmaf(v[n0], v[6 + a0], f0);
                        f1 = fmaf(v[n1], v[6 + a1], f1);
                    }
                });
            float *o = desc + (p0 + t) * NDESC;
            if (lane < 10) {
                const float x = (sh.rij[t] - __fmul_rn(1.6f, (float)lane)) / 1.6f;
                o[lane] = __expf(-0.5f * x * x);
            }
            o[10 + lane] = f0;
            if (lane + 32 < 54) o[42 + lane] = f1;
        }
        __syncthreads();
    }
}

// targets: the (i, j) block of L in the pair frame, L_loc = D L D^T (row-major nb x nb,
// zero-padded to 81)
__global__ void k_targets(int64_t n_pairs, int nb, int stride, const int32_t *pairs,
                          const float *frames, const double *L, float *targets)
{
    const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= n_pairs) return;
    double R[3][3], D[9][9], T[9][9];
    for (int r = 0; r < 3; ++r)
        for (int c = 0; c < 3; ++c) R[r][c] = frames[p * 9 + 3 * r + c];
    orbital_rotation(R, nb, D);
    const double *blk = L + (int64_t)pairs[p] * stride;
    for (int a = 0; a < nb; ++a)
        for (int c = 0; c < nb; ++c) {
            double acc = 0.0;
            for (int u = 0; u < nb; ++u) acc += D[a][u] * blk[u * nb + c];
            T[a][c] = acc;
        }
    float *o = targets + p * NOUT;
    for (int a = 0; a < 9; ++a)
        for (int c = 0; c < 9; ++c) {
            double acc = 0.0;
            if (a < nb && c < nb)
                for (int v = 0; v < nb; ++v) acc += T[a][v] * D[c][v];
            o[a * 9 + c] = (float)acc;
        }
}

// The d-shell rotation D2[a][b] = <Q_b, R^T Q_a R>_F of frame rows R, with the forms' few
// non-zero entries only (the terms and their order are orbital_rotation's)
__device__ __forceinline__ void d_rotation(const double (&R)[3][3], double (*D2)[5])
{
    const double h = 0.70710678118654752440, s6 = 0.40824829046386301637;
#pragma unroll
    for (int a = 0; a < 5; ++a) {
        double t[3][3];
#pragma unroll
        for (int r = 0; r < 3; ++r)
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                double acc = 0.0;
                if (a == 0) {
                    acc += R[0][r] * h * R[1][c];
                    acc += R[1][r] * h * R[0][c];
                } else if (a == 1) {
                    acc += R[1][r] * h * R[2][c];
                    acc += R[2][r] * h * R[1][c];
                } else if (a == 2) {
                    acc += R[0][r] * h * R[2][c];
                    acc += R[2][r] * h * R[0][c];
                } else if (a == 3) {
                    acc += R[0][r] * h * R[0][c];
                    acc += R[1][r] * -h * R[1][c];
                } else {
                    acc += R[0][r] * -s6 * R[0][c];
                    acc += R[1][r] * -s6 * R[1][c];
                    acc += R[2][r] * (2.0 * s6) * R[2][c];
                }
                t[r][c] = acc;
            }
        D2[a][0] = h * t[0][1] + h * t[1][0];
        D2[a][1] = h * t[1][2] + h * t[2][1];
        D2[a][2] = h * t[0][2] + h * t[2][0];
        D2[a][3] = h * t[0][0] + -h * t[1][1];
        D2[a][4] = (-s6 * t[0][0] + -s6 * t[1][1]) + 2.0 * s6 * t[2][2];
    }
}

// apply: block (i, j) = D^T L_loc D and block (j, i) = its transpose.  32 pairs per CTA, nine
// threads each: a column of T = D^T L_loc, then a row of T D.  Bound by the FP64 pipe; D is
// block diagonal (1, 3 and 5 orbitals), so a sum has one, three or five terms in place of
// nine, predictions are widened by their bits, and the blocks leave through shared memory.
constexpr int APPLY_P = 32, APPLY_T = 9 * APPLY_P;

__global__ void __launch_bounds__(APPLY_T)
k_apply(int64_t n_pairs, int nb, int stride, const int32_t *pairs, const int64_t *tr,
        const int32_t *row, const int32_t *col, const float *frames, const float *pred,
        const float *mean, const float *scale, double *L)
{
    __shared__ double R[APPLY_P][3][3], D2[APPLY_P][5][5], T[APPLY_P][9][9];
    const int64_t p0 = (int64_t)blockIdx.x * APPLY_P;
    const int np = (int)min((int64_t)APPLY_P, n_pairs - p0);
    for (int e = threadIdx.x; e < np * 9; e += APPLY_T)
        R[e / 9][e % 9 / 3][e % 3] = f32_to_f64(frames[p0 * 9 + e]);
    __syncthreads();
    if (threadIdx.x < np && nb == 9) d_rotation(R[threadIdx.x], D2[threadIdx.x]);
    __syncthreads();
    const int q = threadIdx.x % APPLY_P, x = threadIdx.x / APPLY_P;  // pair, column or row
    const bool on = q < np && x < nb;
    double v[9];
    if (on) {
        // column x of L_loc, then of D^T L_loc
        const float *y = pred + (p0 + q) * NOUT;
        double loc[9];
#pragma unroll
        for (int u = 0; u < 9; ++u)
            if (u < nb)
                loc[u] = f32_to_f64(y[u * 9 + x]) * f32_to_f64(scale[u * 9 + x]) +
                         f32_to_f64(mean[u * 9 + x]);
        T[q][0][x] = loc[0];
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            double acc = 0.0;
#pragma unroll
            for (int u = 0; u < 3; ++u) acc += R[q][u][a] * loc[1 + u];
            T[q][1 + a][x] = acc;
        }
        if (nb == 9)
#pragma unroll
            for (int a = 0; a < 5; ++a) {
                double acc = 0.0;
#pragma unroll
                for (int u = 0; u < 5; ++u) acc += D2[q][u][a] * loc[4 + u];
                T[q][4 + a][x] = acc;
            }
    }
    __syncthreads();
    if (on) {
        // row x of T D
        double w[9];
#pragma unroll
        for (int u = 0; u < 9; ++u)
            if (u < nb) w[u] = T[q][x][u];
        v[0] = w[0];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            double acc = 0.0;
#pragma unroll
            for (int u = 0; u < 3; ++u) acc += w[1 + u] * R[q][u][c];
            v[1 + c] = acc;
        }
        if (nb == 9)
#pragma unroll
            for (int c = 0; c < 5; ++c) {
                double acc = 0.0;
#pragma unroll
                for (int u = 0; u < 5; ++u) acc += w[4 + u] * D2[q][u][c];
                v[4 + c] = acc;
            }
    }
    __syncthreads();
    if (on)
#pragma unroll
        for (int c = 0; c < 9; ++c)
            if (c < nb) T[q][x][c] = v[c];
    __syncthreads();
    // a warp per pair writes both blocks; an on-site block is its own transpose: its lower
    // triangle stands for both
    const int lane = threadIdx.x & 31;
    for (int t = threadIdx.x >> 5; t < np; t += APPLY_T / 32) {
        const int b = pairs[p0 + t];
        const bool site = row[b] == col[b];
        double *blk = L + (int64_t)b * stride, *blt = L + tr[b] * stride;
        for (int e = lane; e < nb * nb; e += 32) {
            const int a = e / nb, c = e - a * nb;
            const double lo = T[t][a > c ? a : c][a > c ? c : a], here = T[t][a][c];
            blk[e] = site ? lo : here;
            if (!site) blt[e] = T[t][c][a];
        }
    }
}

__global__ void k_pair_flags(int64_t nblk, const int32_t *row, const int32_t *col, int64_t *f)
{
    const int64_t b = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (b < nblk) f[b] = row[b] <= col[b] ? 1 : 0;
}

__global__ void k_pair_fill(int64_t nblk, const int32_t *row, const int32_t *col,
                            const int64_t *pos, int32_t *pairs)
{
    const int64_t b = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (b < nblk && row[b] <= col[b]) pairs[pos[b]] = (int32_t)b;
}

// ---------------------------------------------------------------- MLP kernels

// C[M x N] (+)= op(A) op(B) in FP32 with 64 x 64 tiles, 16 x 16 threads, 4 x 4 outputs each.
// A: FP32, op(A)[m][k] = TA ? A[k * lda + m] : A[m * lda + k];
// B: BT (float or bf16), op(B)[k][n] = TB ? B[n * ldb + k] : B[k * ldb + n].
// The K range [k0, k1) lets callers split a long reduction into deterministic partials.
template <bool TA, bool TB, typename BT>
__global__ void __launch_bounds__(256)
k_gemm(int M, int N, const float *A, int lda, const BT *B, int ldb, float *C, int ldc,
       int64_t k0, int64_t k1, int64_t c_stride_z, int64_t k_chunk)
{
    __shared__ float As[16][65];
    __shared__ float Bs[16][65];
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
    const int m0 = blockIdx.y * 64, n0 = blockIdx.x * 64;
    const int64_t kb = k0 + (int64_t)blockIdx.z * k_chunk;
    const int64_t ke = min(k1, kb + k_chunk);
    float acc[4][4] = {};
    for (int64_t kt = kb; kt < ke; kt += 16) {
        for (int e = threadIdx.x; e < 16 * 64; e += 256) {
            const int kk = e / 64, mm = e % 64;
            const int64_t k = kt + kk;
            const int m = m0 + mm;
            float va = 0.f;
            if (k < ke && m < M) va = TA ? A[k * lda + m] : A[(int64_t)m * lda + k];
            As[kk][mm] = va;
            const int n = n0 + mm;
            float vb = 0.f;
            if (k < ke && n < N) vb = (float)(TB ? B[(int64_t)n * ldb + k] : B[k * ldb + n]);
            Bs[kk][mm] = vb;
        }
        __syncthreads();
#pragma unroll
        for (int kk = 0; kk < 16; ++kk) {
            float a[4], b[4];
#pragma unroll
            for (int r = 0; r < 4; ++r) a[r] = As[kk][ty * 4 + r];
#pragma unroll
            for (int c = 0; c < 4; ++c) b[c] = Bs[kk][tx * 4 + c];
#pragma unroll
            for (int r = 0; r < 4; ++r)
#pragma unroll
                for (int c = 0; c < 4; ++c) acc[r][c] = fmaf(a[r], b[c], acc[r][c]);
        }
        __syncthreads();
    }
    float *Cz = C + (int64_t)blockIdx.z * c_stride_z;
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const int m = m0 + ty * 4 + r, n = n0 + tx * 4 + c;
            if (m < M && n < N) Cz[(int64_t)m * ldc + n] = acc[r][c];
        }
}

#include "mlp_tc.cuh"

// Z += bias; H = silu(Z) (hidden) or H = Z (output)
__global__ void k_bias_act(int64_t M, int N, const float *bias, float *Z, float *H, int act)
{
    const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= M * N) return;
    const float z = Z[e] + bias[e % N];
    Z[e] = z;
    H[e] = act ? z / (1.f + __expf(-z)) : z;
}

// dZ = dH * silu'(Z)
__global__ void k_act_back(int64_t n, const float *Z, const float *dH, float *dZ)
{
    const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= n) return;
    const float z = Z[e], s = 1.f / (1.f + __expf(-z));
    dZ[e] = dH[e] * (s * (1.f + z * (1.f - s)));
}

// loss = mean (Y - T)^2 over n x 81 (per-CTA partials), dY = 2 (Y - T) / (n * 81)
__global__ void k_mse(int64_t n, const float *Y, const float *T, float *dY, float *part)
{
    __shared__ float sh[256];
    const int64_t tot = n * NOUT;
    float s = 0.f;
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < tot;
         e += (int64_t)gridDim.x * blockDim.x) {
        const float d = Y[e] - T[e];
        s += d * d;
        dY[e] = 2.f * d / (float)tot;
    }
    sh[threadIdx.x] = s;
    __syncthreads();
    for (int o = 128; o > 0; o >>= 1) {
        if (threadIdx.x < o) sh[threadIdx.x] += sh[threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0) part[blockIdx.x] = sh[0];
}

// adds the 256 block partials of k_mse (fixed order) and the batch's row count to the
// running sums acc[0], acc[1] (one CTA of 256 threads)
__device__ void loss_accum(const float *part, int64_t rows, double *acc)
{
    __shared__ double sh[256];
    sh[threadIdx.x] = (double)part[threadIdx.x];
    __syncthreads();
    for (int o = 128; o > 0; o >>= 1) {
        if (threadIdx.x < o) sh[threadIdx.x] += sh[threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        acc[0] += sh[0];
        acc[1] += (double)rows;
    }
}

__global__ void k_loss_accum(const float *part, int64_t rows, double *acc)
{
    loss_accum(part, rows, acc);
}

// sum of `parts` partial matrices (deterministic order) + column sums for bias gradients
__global__ void k_sum_parts(int64_t n, int parts, int64_t stride, const float *src, float *dst)
{
    const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= n) return;
    float s = 0.f;
    for (int q = 0; q < parts; ++q) s += src[q * stride + e];
    dst[e] = s;
}

__global__ void k_colsum(int64_t M, int N, const float *dZ, float *db)
{
    const int n = blockIdx.x * blockDim.x + threadIdx.x;
    if (n >= N) return;
    float s = 0.f;
    for (int64_t m = 0; m < M; ++m) s += dZ[m * N + n];
    db[n] = s;
}

struct AdamArgs {
    float lr, b1, b2, eps, c1, c2;
};

// Adam on one FP32 master weight (w, moments mo and ve, gradient gr): the updated weight
__device__ __forceinline__ float adam(float *w, float gr, float *mo, float *ve, const AdamArgs &a)
{
    // one rounding order wherever this is inlined: the gradient's term joins by FMA
    const float m = fmaf(1.f - a.b1, gr, __fmul_rn(a.b1, *mo));
    const float v = fmaf(__fmul_rn(1.f - a.b2, gr), gr, __fmul_rn(a.b2, *ve));
    *mo = m;
    *ve = v;
    const float nw = *w - a.lr * (m / a.c1) / (sqrtf(v / a.c2) + a.eps);
    *w = nw;
    return nw;
}

__global__ void k_adam(int64_t n, float *w, const float *g, float *mo, float *ve, AdamArgs a)
{
    const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e < n) adam(w + e, g[e], mo + e, ve + e, a);
}

// The network's shape: weights of layer l are K x N at offset W0, biases at B0.
constexpr int NHID = 256, NOUT_PAD = 96;
constexpr int W1 = NDESC * NHID, W2 = W1 + NHID * NHID, W3 = W2 + NHID * NHID;
constexpr int NW = W3 + NHID * NOUT, NB_ALL = 3 * NHID + NOUT;

// BF16 copies of one weight: wb (as the master, K x N), wt (transposed, N x K) and for the output
// layer also w4 (K x NOUT_PAD, so that its rows start on 16-byte boundaries)
__device__ __forceinline__ void put_weight(int e, float w, __nv_bfloat16 *wb, __nv_bfloat16 *wt,
                                           __nv_bfloat16 *w4)
{
    const __nv_bfloat16 v = __float2bfloat16(w);
    const int w0 = e >= W3 ? W3 : e >= W2 ? W2 : e >= W1 ? W1 : 0;
    const int K = w0 ? NHID : NDESC, N = w0 == W3 ? NOUT : NHID;
    const int k = (e - w0) / N, n = (e - w0) % N;
    wb[e] = v;
    wt[w0 + n * K + k] = v;
    if (w0 == W3) w4[k * NOUT_PAD + n] = v;
}

__global__ void k_tc_weights(const float *w, __nv_bfloat16 *wb, __nv_bfloat16 *wt,
                             __nv_bfloat16 *w4)
{
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e < NW) put_weight(e, w[e], wb, wt, w4);
}

// Normalised BF16 network inputs (32 rows per CTA of 256 threads, eight values per thread) and,
// if xt is not null, their transpose (ld_t apart).
__global__ void __launch_bounds__(256)
k_tc_input(int64_t rows, const float *x, const float *mean, const float *scale, __nv_bfloat16 *xb,
           __nv_bfloat16 *xt, int64_t ld_t)
{
    __shared__ __nv_bfloat16 tile[NDESC][34];
    const int64_t r0 = (int64_t)blockIdx.x * 32;
    const int r = threadIdx.x / 8, f0 = threadIdx.x % 8 * 8;
    if (r0 + r < rows) {
        const float *src = x + (r0 + r) * NDESC + f0;
        float v[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) v[q] = (src[q] - mean[f0 + q]) / scale[f0 + q];
        uint32_t u[4];
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            const __nv_bfloat16 b = __float2bfloat16(v[q]);
            tile[f0 + q][r] = b;
            u[q >> 1] = q & 1 ? u[q >> 1] | ((uint32_t)__bfloat16_as_ushort(b) << 16)
                              : (uint32_t)__bfloat16_as_ushort(b);
        }
        *reinterpret_cast<uint4 *>(xb + (r0 + r) * NDESC + f0) = make_uint4(u[0], u[1], u[2], u[3]);
    }
    if (!xt) return;
    __syncthreads();
    const int lane = threadIdx.x & 31;
    for (int f = threadIdx.x >> 5; f < NDESC; f += 8)
        if (r0 + lane < rows) xt[f * ld_t + r0 + lane] = tile[f][lane];
}

// k_mse on raw targets (normalised here), with dY also as BF16 rows of NOUT_PAD values (the
// padding is zero from the start) and transposed.
__global__ void __launch_bounds__(256)
k_tc_mse(int64_t n, const float *Y, const float *T, const float *mean, const float *scale,
         float *dY, __nv_bfloat16 *dYb, __nv_bfloat16 *dYt, int64_t ld_t, float *part)
{
    __shared__ float sh[256];
    const int64_t tot = n * NOUT;
    float s = 0.f;
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < tot;
         e += (int64_t)gridDim.x * blockDim.x) {
        const int64_t r = e / NOUT;
        const int f = (int)(e - r * NOUT);
        const float t = (T[e] - mean[f]) / scale[f];
        const float d = Y[e] - t;
        s += d * d;
        const float g = 2.f * d / (float)tot;
        dY[e] = g;
        const __nv_bfloat16 v = __float2bfloat16(g);
        dYb[r * NOUT_PAD + f] = v;
        dYt[f * ld_t + r] = v;
    }
    sh[threadIdx.x] = s;
    __syncthreads();
    for (int o = 128; o > 0; o >>= 1) {
        if (threadIdx.x < o) sh[threadIdx.x] += sh[threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0) part[blockIdx.x] = sh[0];
}

// End of a tensor-core training step: weight gradients as the ordered sums of their partial
// products, Adam on weights and biases (up.lr > 0) with the BF16 copies refreshed, and the
// batch's loss added to the running sums (last CTA).
struct TcUpdate {
    int parts;
    const float *part;      // per layer: parts x K x N, layers one after another
    float *gw, *w, *mw, *vw;
    float *gb, *b, *mb, *vb;
    __nv_bfloat16 *wb, *wt, *w4;
    const float *loss;
    double *acc;
    int64_t rows;
    AdamArgs up;
};

__global__ void __launch_bounds__(256) k_tc_update(const TcUpdate p)
{
    if (blockIdx.x == gridDim.x - 1) {
        loss_accum(p.loss, p.rows, p.acc);
        return;
    }
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e < NW) {
        const int w0 = e >= W3 ? W3 : e >= W2 ? W2 : e >= W1 ? W1 : 0;
        const int size = (w0 ? NHID : NDESC) * (w0 == W3 ? NOUT : NHID);
        const float *src = p.part + (int64_t)w0 * p.parts + (e - w0);
        float s = 0.f;
        for (int q = 0; q < p.parts; ++q) s += src[(int64_t)q * size];
        p.gw[e] = s;
        if (p.up.lr > 0.f)
            put_weight(e, adam(p.w + e, s, p.mw + e, p.vw + e, p.up), p.wb, p.wt, p.w4);
    } else if (e - NW < NB_ALL && p.up.lr > 0.f) {
        const int q = e - NW;
        adam(p.b + q, p.gb[q], p.mb + q, p.vb + q, p.up);
    }
}

inline unsigned blocks_for(int64_t n, int t = 256) { return (unsigned)((n + t - 1) / t); }

// per-column mean and standard deviation (FP64 sums; a floor keeps constant columns finite)
__global__ void k_colstats(int64_t M, int N, const float *X, float *mean, float *scale)
{
    const int n = blockIdx.x * blockDim.x + threadIdx.x;
    if (n >= N) return;
    double s = 0.0, s2 = 0.0;
    for (int64_t m = 0; m < M; ++m) {
        const double v = X[m * N + n];
        s += v;
        s2 += v * v;
    }
    const double mu = s / (double)M;
    const double var = fmax(s2 / (double)M - mu * mu, 0.0);
    mean[n] = (float)mu;
    scale[n] = (float)fmax(sqrt(var), 1e-6);
}

__global__ void k_norm_out(int64_t n, const float *t, const float *mean, const float *scale,
                           float *y)
{
    const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= n) return;
    const int f = (int)(e % NOUT);
    y[e] = (t[e] - mean[f]) / scale[f];
}

}  // namespace

// ---------------------------------------------------------------- host side

struct cq_guess {
    cq_ctx *ctx = nullptr;
    int n_layers = 4;                 // 3 hidden + output
    int dims[5] = {NDESC, 256, 256, 256, NOUT};
    bool fp32_weights = false;        // test mode: forward reads the FP32 weights
    DevBuf w, wb, b, gw, gb, mw, vw, mb, vb;  // all layers packed (NW weights, NB_ALL biases)
    std::vector<int64_t> w_off, b_off;
    int64_t n_w = 0, n_b = 0;
    int64_t step = 0;
    DevBuf mean, scale;               // target normalisation (81 each)
    DevBuf in_mean, in_scale;         // descriptor normalisation (64 each)
    DevBuf xin;                       // normalised inputs of the current batch
    int64_t xin_rows = 0;
    DevBuf act;                       // Z and H per layer for a batch
    int64_t act_rows = 0;
    // tensor-core path (BF16 weights): W^T per layer (BF16, N x K), the padded output layer,
    // the BF16 layer inputs of a batch, and what a training step keeps besides
    DevBuf wt, w4, hb, tr;
    int64_t hb_rows = 0, tr_rows = 0;
    DevBuf loss_acc;                  // running squared-error sum and row count (2 doubles)
};

namespace {

cq_status ensure_act(cq_guess *g, int64_t rows)
{
    int64_t per = 0;
    for (int l = 1; l <= g->n_layers; ++l) per += 2 * g->dims[l];
    per += g->dims[g->n_layers];  // dY
    per += 256;                   // dH scratch of the widest layer
    per += 256;
    return cq_grow_rows(g->act_rows, rows, [&] {
        return cq_alloc(g->ctx, g->act, sizeof(float) * per * rows);
    });
}

int64_t pad16(int64_t x) { return (x + 15) & ~(int64_t)15; }

// BF16 inputs of the layers for up to hb_rows rows: rows x 64, then three times rows x 256
__nv_bfloat16 *tc_hb(cq_guess *g, int l)
{
    return g->hb.as<__nv_bfloat16>() + (l ? g->hb_rows * (NDESC + (int64_t)(l - 1) * NHID) : 0);
}

// Buffers of a training step for up to tr_rows rows (ld_t = the transposes' leading dimension)
struct TrainBufs {
    int64_t ld_t;
    float *Z[3], *Y, *dZ[TC_LAYERS];           // hidden Z, output, dZ of every layer
    __nv_bfloat16 *Ht[TC_LAYERS], *dZt[TC_LAYERS];  // transposes: layer inputs, dZ
    __nv_bfloat16 *dZb[TC_LAYERS];             // dZ of layers 2-4 as rows of 256 (4: NOUT_PAD)
};

cq_status tc_rows(cq_guess *g, int64_t rows, bool train)
{
    CQ_TRY(cq_grow_rows(g->hb_rows, rows, [&] {
        return cq_alloc(g->ctx, g->hb, sizeof(__nv_bfloat16) * (size_t)(rows * (NDESC + 3 * NHID)));
    }));
    if (!train) return CQ_OK;
    return cq_grow_rows(g->tr_rows, rows, [&] {
        const int64_t ld = pad16(rows);
        const size_t f32 = sizeof(float) * (size_t)(ld * (6 * NHID + 2 * NOUT_PAD));
        const size_t b16 = sizeof(__nv_bfloat16) * (size_t)(ld * ((NDESC + 3 * NHID) + (3 * NHID + NOUT_PAD) +
                                                                  (2 * NHID + NOUT_PAD)));
        CQ_TRY(cq_alloc(g->ctx, g->tr, f32 + b16));
        // the padding columns of the output layer's dZ rows stay zero
        return cq_check_cuda(g->ctx, cudaMemsetAsync(g->tr.ptr, 0, f32 + b16, g->ctx->stream),
                             "training buffers");
    });
}

TrainBufs tc_train_bufs(cq_guess *g)
{
    TrainBufs t;
    const int64_t ld = t.ld_t = pad16(g->tr_rows);
    float *f = g->tr.as<float>();
    for (int l = 0; l < 3; ++l, f += ld * NHID) t.Z[l] = f;
    for (int l = 0; l < 3; ++l, f += ld * NHID) t.dZ[l] = f;
    t.Y = f;
    t.dZ[3] = f + ld * NOUT_PAD;
    __nv_bfloat16 *b = reinterpret_cast<__nv_bfloat16 *>(f + 2 * ld * NOUT_PAD);
    auto take = [&](int n) { __nv_bfloat16 *r = b; b += ld * n; return r; };
    for (int l = 0; l < TC_LAYERS; ++l) t.Ht[l] = take(l ? NHID : NDESC);
    for (int l = 0; l < TC_LAYERS; ++l) t.dZt[l] = take(l < 3 ? NHID : NOUT_PAD);
    t.dZb[0] = nullptr;
    for (int l = 1; l < TC_LAYERS; ++l) t.dZb[l] = take(l < 3 ? NHID : NOUT_PAD);
    return t;
}

cq_status tc_attr(cq_ctx *ctx)
{
    static bool done[64] = {};
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev < 0 || dev >= 64) return cq_fail(ctx, CQ_ERR_INVALID, "guess: device index");
    if (done[dev]) return CQ_OK;
    auto set = [&](const void *k) {
        return cq_check_cuda(ctx, cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                       TC_SMEM), "mlp attribute");
    };
    CQ_TRY(set((const void *)k_tc_hidden));
    CQ_TRY(set((const void *)k_tc_output));
    CQ_TRY(set((const void *)k_tc_back));
    CQ_TRY(set((const void *)k_tc_grads));
    done[dev] = true;
    return CQ_OK;
}

// BF16 copies of the weights (after every change of the master weights from the host)
void refresh_weights(cq_guess *g, cudaStream_t s)
{
    k_tc_weights<<<blocks_for(NW), 256, 0, s>>>(g->w.as<float>(), g->wb.as<__nv_bfloat16>(),
                                                g->wt.as<__nv_bfloat16>(), g->w4.as<__nv_bfloat16>());
    cq_count_launch();
}

// Tensor-core forward pass of `rows` descriptors into Y (rows x 81); t: the buffers a training
// step needs (pre-activations and transposes), or null.
cq_status tc_forward(cq_guess *g, const float *X, int64_t rows, float *Y, const TrainBufs *t)
{
    cq_ctx *ctx = g->ctx;
    cudaStream_t s = ctx->stream;
    CQ_TRY(tc_attr(ctx));
    const __nv_bfloat16 *wt = g->wt.as<__nv_bfloat16>();
    const float *b = g->b.as<float>();
    const unsigned mt = (unsigned)((rows + TC_MT - 1) / TC_MT);
    const int64_t ld = t ? t->ld_t : 0;
    k_tc_input<<<blocks_for(rows, 32), 256, 0, s>>>(rows, X, g->in_mean.as<float>(),
                                                    g->in_scale.as<float>(), tc_hb(g, 0),
                                                    t ? t->Ht[0] : nullptr, ld);
    const int w0[4] = {0, W1, W2, W3};
    for (int l = 0; l < 3; ++l)
        k_tc_hidden<<<dim3(mt, NHID / TC_NT), TC_T, TC_SMEM, s>>>(
            (int)rows, NHID, l ? NHID : NDESC, tc_hb(g, l), wt + w0[l], b + l * NHID,
            t ? t->Z[l] : nullptr, tc_hb(g, l + 1), t ? t->Ht[l + 1] : nullptr, ld,
            ctx->flag.as<int32_t>());
    k_tc_output<<<dim3(mt, (NOUT + TC_NT - 1) / TC_NT), TC_T, TC_SMEM, s>>>(
        (int)rows, NOUT, NHID, tc_hb(g, 3), wt + W3, b + 3 * NHID, Y, ctx->flag.as<int32_t>());
    cq_count_launch(5);
    return cq_check_cuda(ctx, cudaGetLastError(), "mlp forward");
}

__global__ void k_norm_in(int64_t n, const float *x, const float *mean, const float *scale,
                          float *y)
{
    const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= n) return;
    const int f = (int)(e % NDESC);
    y[e] = (x[e] - mean[f]) / scale[f];
}

// FP32 forward (test mode) on `rows` descriptors (normalised first): H[n_layers] is the output
// (rows x 81)
cq_status mlp_forward(cq_guess *g, const float *X, int64_t rows, std::vector<float *> &Z,
                      std::vector<float *> &H)
{
    cq_ctx *ctx = g->ctx;
    CQ_TRY(ensure_act(g, rows));
    CQ_TRY(cq_grow_rows(g->xin_rows, rows,
                        [&] { return cq_alloc(ctx, g->xin, sizeof(float) * NDESC * rows); }));
    k_norm_in<<<blocks_for(rows * NDESC), 256, 0, ctx->stream>>>(
        rows * NDESC, X, g->in_mean.as<float>(), g->in_scale.as<float>(), g->xin.as<float>());
    cq_count_launch();
    float *base = g->act.as<float>();
    Z.assign(g->n_layers + 1, nullptr);
    H.assign(g->n_layers + 1, nullptr);
    H[0] = g->xin.as<float>();
    int64_t off = 0;
    for (int l = 1; l <= g->n_layers; ++l) {
        Z[l] = base + off;
        off += rows * g->dims[l];
        H[l] = base + off;
        off += rows * g->dims[l];
        const int K = g->dims[l - 1], N = g->dims[l];
        dim3 grid((N + 63) / 64, (unsigned)((rows + 63) / 64), 1);
        k_gemm<false, false, float><<<grid, 256, 0, ctx->stream>>>(
            (int)rows, N, H[l - 1], K, g->w.as<float>() + g->w_off[l - 1], N, Z[l], N, 0, K, 0, K);
        k_bias_act<<<blocks_for(rows * N), 256, 0, ctx->stream>>>(
            rows, N, g->b.as<float>() + g->b_off[l - 1], Z[l], H[l], l < g->n_layers ? 1 : 0);
        cq_count_launch(2);
    }
    return cq_check_cuda(ctx, cudaGetLastError(), "mlp forward");
}

}  // namespace

extern "C" cq_status cq_guess_create(cq_ctx *ctx, uint64_t seed, int32_t fp32_weights,
                                     cq_guess **out)
{
    if (!ctx || !out) return CQ_ERR_INVALID;
    std::unique_ptr<cq_guess> g(new cq_guess());
    g->ctx = ctx;
    g->fp32_weights = fp32_weights != 0;
    g->w_off.push_back(0);
    g->b_off.push_back(0);
    for (int l = 0; l < g->n_layers; ++l) {
        g->w_off.push_back(g->w_off.back() + (int64_t)g->dims[l] * g->dims[l + 1]);
        g->b_off.push_back(g->b_off.back() + g->dims[l + 1]);
    }
    g->n_w = g->w_off.back();
    g->n_b = g->b_off.back();
    for (DevBuf *b : {&g->w, &g->gw, &g->mw, &g->vw})
        CQ_TRY(cq_alloc(ctx, *b, sizeof(float) * g->n_w));
    for (DevBuf *b : {&g->b, &g->gb, &g->mb, &g->vb})
        CQ_TRY(cq_alloc(ctx, *b, sizeof(float) * g->n_b));
    CQ_TRY(cq_alloc(ctx, g->wb, sizeof(__nv_bfloat16) * g->n_w));
    CQ_TRY(cq_alloc(ctx, g->wt, sizeof(__nv_bfloat16) * g->n_w));
    CQ_TRY(cq_alloc(ctx, g->w4, sizeof(__nv_bfloat16) * NHID * NOUT_PAD));
    CQ_TRY(cq_alloc(ctx, g->mean, sizeof(float) * NOUT));
    CQ_TRY(cq_alloc(ctx, g->scale, sizeof(float) * NOUT));
    CQ_TRY(cq_alloc(ctx, g->in_mean, sizeof(float) * NDESC));
    CQ_TRY(cq_alloc(ctx, g->in_scale, sizeof(float) * NDESC));
    // He-style initialisation from a seeded generator (host), zero biases and moments
    std::mt19937_64 rng(seed);
    std::vector<float> w(g->n_w);
    for (int l = 0; l < g->n_layers; ++l) {
        std::normal_distribution<float> nd(0.f, std::sqrt(2.f / g->dims[l]) *
                                                    (l + 1 == g->n_layers ? 0.1f : 1.f));
        for (int64_t e = g->w_off[l]; e < g->w_off[l + 1]; ++e) w[e] = nd(rng);
    }
    cudaStream_t s = ctx->stream;
    cudaMemcpyAsync(g->w.ptr, w.data(), sizeof(float) * g->n_w, cudaMemcpyHostToDevice, s);
    for (DevBuf *b : {&g->mw, &g->vw}) cudaMemsetAsync(b->ptr, 0, sizeof(float) * g->n_w, s);
    for (DevBuf *b : {&g->b, &g->mb, &g->vb}) cudaMemsetAsync(b->ptr, 0, sizeof(float) * g->n_b, s);
    std::vector<float> zero(NOUT, 0.f), one(NOUT, 1.f);
    cudaMemcpyAsync(g->mean.ptr, zero.data(), sizeof(float) * NOUT, cudaMemcpyHostToDevice, s);
    cudaMemcpyAsync(g->scale.ptr, one.data(), sizeof(float) * NOUT, cudaMemcpyHostToDevice, s);
    cudaMemcpyAsync(g->in_mean.ptr, zero.data(), sizeof(float) * NDESC, cudaMemcpyHostToDevice, s);
    cudaMemcpyAsync(g->in_scale.ptr, one.data(), sizeof(float) * NDESC, cudaMemcpyHostToDevice, s);
    cudaMemsetAsync(g->w4.ptr, 0, sizeof(__nv_bfloat16) * NHID * NOUT_PAD, s);
    refresh_weights(g.get(), s);
    CQ_TRY(cq_check_cuda(ctx, cudaStreamSynchronize(s), "guess create"));
    ctx->live_guess.push_back(g.get());
    *out = g.release();
    return CQ_OK;
}

void cq_guess_detach(cq_guess *g)
{
    g->ctx = nullptr;
    for (DevBuf *b : {&g->w, &g->wb, &g->b, &g->gw, &g->gb, &g->mw, &g->vw, &g->mb, &g->vb, &g->mean,
                      &g->scale, &g->in_mean, &g->in_scale, &g->xin, &g->act, &g->wt, &g->w4, &g->hb,
                      &g->tr, &g->loss_acc})
        b->ctx = nullptr;
}

extern "C" void cq_guess_destroy(cq_guess *g)
{
    if (!g) return;
    if (g->ctx) {
        cudaStreamSynchronize(g->ctx->stream);
        auto &v = g->ctx->live_guess;
        v.erase(std::find(v.begin(), v.end(), g));
    }
    delete g;
}

extern "C" cq_status cq_guess_params(cq_guess *g, float *w_host, float *b_host, int64_t *n_w,
                                     int64_t *n_b, int32_t set)
{
    if (!g || !g->ctx) return CQ_ERR_INVALID;
    if (n_w) *n_w = g->n_w;
    if (n_b) *n_b = g->n_b;
    cudaStream_t s = g->ctx->stream;
    if (set) {
        if (w_host) cudaMemcpyAsync(g->w.ptr, w_host, 4 * g->n_w, cudaMemcpyHostToDevice, s);
        if (b_host) cudaMemcpyAsync(g->b.ptr, b_host, 4 * g->n_b, cudaMemcpyHostToDevice, s);
        refresh_weights(g, s);
    } else {
        if (w_host) cudaMemcpyAsync(w_host, g->w.ptr, 4 * g->n_w, cudaMemcpyDeviceToHost, s);
        if (b_host) cudaMemcpyAsync(b_host, g->b.ptr, 4 * g->n_b, cudaMemcpyDeviceToHost, s);
    }
    return cq_check_cuda(g->ctx, cudaStreamSynchronize(s), "guess params");
}

extern "C" cq_status cq_guess_fit_scale(cq_guess *g, const float *desc, const float *targets,
                                        int64_t rows)
{
    if (!g || !g->ctx || !desc || !targets || rows <= 0) return CQ_ERR_INVALID;
    cudaStream_t s = g->ctx->stream;
    k_colstats<<<1, 128, 0, s>>>(rows, NDESC, desc, g->in_mean.as<float>(), g->in_scale.as<float>());
    k_colstats<<<1, 128, 0, s>>>(rows, NOUT, targets, g->mean.as<float>(), g->scale.as<float>());
    cq_count_launch(2);
    return cq_check_cuda(g->ctx, cudaStreamSynchronize(s), "fit scale");
}

extern "C" cq_status cq_guess_set_scale(cq_guess *g, const float *in_mean_host,
                                        const float *in_scale_host, const float *out_mean_host,
                                        const float *out_scale_host)
{
    if (!g || !g->ctx || !in_mean_host || !in_scale_host || !out_mean_host || !out_scale_host)
        return CQ_ERR_INVALID;
    cudaStream_t s = g->ctx->stream;
    cudaMemcpyAsync(g->in_mean.ptr, in_mean_host, 4 * NDESC, cudaMemcpyHostToDevice, s);
    cudaMemcpyAsync(g->in_scale.ptr, in_scale_host, 4 * NDESC, cudaMemcpyHostToDevice, s);
    cudaMemcpyAsync(g->mean.ptr, out_mean_host, 4 * NOUT, cudaMemcpyHostToDevice, s);
    cudaMemcpyAsync(g->scale.ptr, out_scale_host, 4 * NOUT, cudaMemcpyHostToDevice, s);
    return cq_check_cuda(g->ctx, cudaStreamSynchronize(s), "guess scale");
}

static cq_status pair_list(cq_ctx *ctx, const cq_pattern *pL, int32_t **pairs, int64_t *n,
                           int64_t **pair0 = nullptr)
{
    const int64_t nblk = pL->n_blocks;
    void *vf, *vp, *vl;
    CQ_TRY(cq_scratch(ctx, "gs_flags", 8 * (nblk + 1), &vf));
    CQ_TRY(cq_scratch(ctx, "gs_pos", 8 * (nblk + 1), &vp));
    k_pair_flags<<<blocks_for(nblk), 256, 0, ctx->stream>>>(nblk, pL->row.as<int32_t>(),
                                                            pL->col.as<int32_t>(), (int64_t *)vf);
    cq_count_launch();
    CQ_TRY(cq_scan_i64(ctx, (int64_t *)vf, (int64_t *)vp, nblk));
    cudaMemcpyAsync(n, (int64_t *)vp + nblk, 8, cudaMemcpyDeviceToHost, ctx->stream);
    CQ_TRY(cq_check_cuda(ctx, cudaStreamSynchronize(ctx->stream), "pairs"));
    CQ_TRY(cq_scratch(ctx, "gs_pairs", 4 * (*n + 1), &vl));
    k_pair_fill<<<blocks_for(nblk), 256, 0, ctx->stream>>>(nblk, pL->row.as<int32_t>(),
                                                           pL->col.as<int32_t>(), (int64_t *)vp,
                                                           (int32_t *)vl);
    cq_count_launch();
    *pairs = (int32_t *)vl;
    if (pair0) *pair0 = (int64_t *)vp;
    return cq_check_cuda(ctx, cudaGetLastError(), "pairs");
}

extern "C" cq_status cq_guess_pairs(cq_ctx *ctx, const cq_pattern *pL, int64_t *n_pairs_host)
{
    if (!ctx || !pL || !n_pairs_host) return CQ_ERR_INVALID;
    int32_t *pairs;
    return pair_list(ctx, pL, &pairs, n_pairs_host);
}

extern "C" cq_status cq_guess_descriptors(cq_ctx *ctx, const cq_pattern *pL, float *desc,
                                          float *frames, int32_t *pairs_out)
{
    if (!ctx || !pL || !desc || !frames) return CQ_ERR_INVALID;
    if (pL->n_cells() != 1)
        return cq_fail(ctx, CQ_ERR_INVALID, "guess: single-cell patterns only");
    int32_t *pairs;
    int64_t n, *pair0;
    CQ_TRY(pair_list(ctx, pL, &pairs, &n, &pair0));
    if (n == 0) return CQ_OK;
    Box3 box;
    for (int c = 0; c < 3; ++c) box.v[c] = pL->geo->box[c];
    // a row's displacements and atoms are cached in shared memory while they fit DESC_SMEM: about
    // 1800 atoms; the rows of the method's P_L hold about 130.  The kernel's limit is that of the
    // longest row whatever this row needs: it belongs to the process, and another thread's call
    // may come between setting it and the launch.
    const size_t cache = (size_t)pL->max_row * (3 * sizeof(double) + 3 * sizeof(float) + sizeof(int32_t));
    const bool cached = sizeof(DescShared) + cache <= DESC_SMEM;
    auto k = cached ? k_descriptors<true> : k_descriptors<false>;
    const size_t smem = sizeof(DescShared) + (cached ? cache : 0);
    CQ_TRY(cq_check_cuda(ctx, cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                   DESC_SMEM), "descriptors"));
    k<<<pL->geo->n_atoms, DESC_T, smem, ctx->stream>>>(pair0, pairs, pL->col.as<int32_t>(),
                                                       pL->row_ptr.as<int64_t>(),
                                                       pL->geo->pos.as<double>(), box, desc, frames);
    cq_count_launch();
    if (pairs_out)
        cudaMemcpyAsync(pairs_out, pairs, 4 * n, cudaMemcpyDeviceToDevice, ctx->stream);
    return cq_check_cuda(ctx, cudaGetLastError(), "descriptors");
}

extern "C" cq_status cq_guess_targets(cq_ctx *ctx, const cq_pattern *pL, const double *L,
                                      const float *frames, float *targets)
{
    if (!ctx || !pL || !L || !frames || !targets) return CQ_ERR_INVALID;
    const int nb = pL->geo->uniform_nb;
    if (nb != 9 && nb != 4) return cq_fail(ctx, CQ_ERR_INVALID, "guess: uniform 4 or 9 orbitals");
    int32_t *pairs;
    int64_t n;
    CQ_TRY(pair_list(ctx, pL, &pairs, &n));
    if (n == 0) return CQ_OK;
    k_targets<<<blocks_for(n, 128), 128, 0, ctx->stream>>>(n, nb, pL->uniform, pairs, frames, L,
                                                           targets);
    cq_count_launch();
    return cq_check_cuda(ctx, cudaGetLastError(), "targets");
}

extern "C" cq_status cq_guess_forward(cq_guess *g, const float *desc, int64_t rows, float *out)
{
    if (!g || !g->ctx || !desc || !out || rows < 0) return CQ_ERR_INVALID;
    if (rows == 0) return CQ_OK;
    if (!g->fp32_weights) {
        CQ_TRY(tc_rows(g, rows, false));
        return tc_forward(g, desc, rows, out, nullptr);
    }
    std::vector<float *> Z, H;
    CQ_TRY(mlp_forward(g, desc, rows, Z, H));
    return cq_check_cuda(g->ctx, cudaMemcpyAsync(out, H[g->n_layers], 4 * rows * NOUT,
                                                 cudaMemcpyDeviceToDevice, g->ctx->stream),
                         "forward copy");
}

// Forward, loss and gradients of a minibatch in the FP32 test mode (deterministic: the
// weight-gradient reduction over rows is split into fixed chunks and summed in order), then Adam
// if up.lr > 0.
static cq_status train_fp32(cq_guess *g, const float *desc, const float *targets, int64_t rows,
                            float *loss, double *acc, const AdamArgs &up)
{
    cq_ctx *ctx = g->ctx;
    cudaStream_t s = ctx->stream;
    std::vector<float *> Z, H;
    CQ_TRY(mlp_forward(g, desc, rows, Z, H));
    const int L = g->n_layers;
    void *vdy, *vdh, *vpart;
    int64_t maxw = 0;
    for (int l = 0; l <= L; ++l) maxw = std::max<int64_t>(maxw, g->dims[l]);
    CQ_TRY(cq_scratch(ctx, "gs_dy", 4 * rows * maxw, &vdy));
    CQ_TRY(cq_scratch(ctx, "gs_dh", 4 * rows * maxw, &vdh));
    const int parts = 16;
    CQ_TRY(cq_scratch(ctx, "gs_part", 4 * (int64_t)parts * NW, &vpart));
    float *dY = (float *)vdy, *dH = (float *)vdh;
    void *vt;
    CQ_TRY(cq_scratch(ctx, "gs_tnorm", 4 * rows * NOUT, &vt));
    k_norm_out<<<blocks_for(rows * NOUT), 256, 0, s>>>(rows * NOUT, targets, g->mean.as<float>(),
                                                      g->scale.as<float>(), (float *)vt);
    k_mse<<<256, 256, 0, s>>>(rows, H[L], (float *)vt, dY, loss);
    k_loss_accum<<<1, 256, 0, s>>>(loss, rows, acc);
    cq_count_launch(3);
    // dY holds dLoss/dZ_L (output layer is linear)
    float *dZ = dY;
    for (int l = L; l >= 1; --l) {
        const int K = g->dims[l - 1], N = g->dims[l];
        // dW_l = H_{l-1}^T dZ  (K x N), reduction over rows in `parts` fixed chunks
        const int64_t chunk = ((rows + parts - 1) / parts + 15) / 16 * 16;
        dim3 grid((N + 63) / 64, (K + 63) / 64, parts);
        k_gemm<true, false, float><<<grid, 256, 0, s>>>(K, N, H[l - 1], K, dZ, N, (float *)vpart, N,
                                                        0, rows, (int64_t)K * N, chunk);
        k_sum_parts<<<blocks_for((int64_t)K * N), 256, 0, s>>>((int64_t)K * N, parts,
                                                             (int64_t)K * N, (float *)vpart,
                                                             g->gw.as<float>() + g->w_off[l - 1]);
        k_colsum<<<blocks_for(N), 256, 0, s>>>(rows, N, dZ, g->gb.as<float>() + g->b_off[l - 1]);
        cq_count_launch(3);
        if (l > 1) {
            // dH_{l-1} = dZ W_l^T (rows x K), then dZ_{l-1} = dH * silu'(Z_{l-1}); the next
            // layer's dZ reuses the buffer
            dim3 g2((K + 63) / 64, (unsigned)((rows + 63) / 64), 1);
            k_gemm<false, true, float><<<g2, 256, 0, s>>>(
                (int)rows, K, dZ, N, g->w.as<float>() + g->w_off[l - 1], N, dH, K, 0, N, 0, N);
            k_act_back<<<blocks_for(rows * K), 256, 0, s>>>(rows * K, Z[l - 1], dH, dY);
            cq_count_launch(2);
        }
    }
    if (up.lr > 0.f) {
        k_adam<<<blocks_for(g->n_w), 256, 0, s>>>(g->n_w, g->w.as<float>(), g->gw.as<float>(),
                                                  g->mw.as<float>(), g->vw.as<float>(), up);
        k_adam<<<blocks_for(g->n_b), 256, 0, s>>>(g->n_b, g->b.as<float>(), g->gb.as<float>(),
                                                  g->mb.as<float>(), g->vb.as<float>(), up);
        cq_count_launch(2);
        refresh_weights(g, s);
    }
    return cq_check_cuda(ctx, cudaGetLastError(), "train step (FP32)");
}

// The same on the tensor cores: the same operations in the same order (sixteen row ranges per
// weight gradient, summed in order; column sums in row order) in eleven launches.
static cq_status train_tc(cq_guess *g, const float *desc, const float *targets, int64_t rows,
                          float *loss, double *acc, const AdamArgs &up)
{
    cq_ctx *ctx = g->ctx;
    cudaStream_t s = ctx->stream;
    CQ_TRY(tc_rows(g, rows, true));
    const int parts = 16;
    void *vpart;
    CQ_TRY(cq_scratch(ctx, "gs_part", 4 * (int64_t)parts * NW, &vpart));
    const TrainBufs t = tc_train_bufs(g);
    CQ_TRY(tc_forward(g, desc, rows, t.Y, &t));
    k_tc_mse<<<256, 256, 0, s>>>(rows, t.Y, targets, g->mean.as<float>(), g->scale.as<float>(),
                                 t.dZ[3], t.dZb[3], t.dZt[3], t.ld_t, loss);
    int32_t *flag = ctx->flag.as<int32_t>();
    const __nv_bfloat16 *wb = g->wb.as<__nv_bfloat16>();
    const unsigned mt = (unsigned)((rows + TC_MT - 1) / TC_MT);
    // dZ of layer l from dZ of layer l + 1 (layers counted from 0)
    for (int l = 2; l >= 0; --l)
        k_tc_back<<<dim3(mt, NHID / TC_NT), TC_T, TC_SMEM, s>>>(
            (int)rows, NHID, l == 2 ? NOUT : NHID, t.dZb[l + 1], l == 2 ? NOUT_PAD : NHID,
            l == 2 ? g->w4.as<__nv_bfloat16>() : wb + (l == 1 ? W2 : W1), l == 2 ? NOUT_PAD : NHID,
            t.Z[l], t.dZ[l], t.dZb[l], t.dZt[l], t.ld_t, flag);
    TcGrads q;
    q.rows = (int)rows;
    q.parts = parts;
    q.chunk = pad16((rows + parts - 1) / parts);
    q.ld_t = t.ld_t;
    q.flag = flag;
    const int w0[4] = {0, W1, W2, W3};
    q.tile0[0] = q.col0[0] = 0;
    for (int l = 0; l < TC_LAYERS; ++l) {
        q.K[l] = l ? NHID : NDESC;
        q.N[l] = l == 3 ? NOUT : NHID;
        q.Ht[l] = t.Ht[l];
        q.dZt[l] = t.dZt[l];
        q.dZ[l] = t.dZ[l];
        q.part[l] = (float *)vpart + (int64_t)w0[l] * parts;
        q.gb[l] = g->gb.as<float>() + l * NHID;
        q.tile0[l + 1] = q.tile0[l] + parts * ((q.K[l] + TC_MT - 1) / TC_MT) *
                                          ((q.N[l] + TC_NT - 1) / TC_NT);
        q.col0[l + 1] = q.col0[l] + (q.N[l] + 31) / 32;
    }
    k_tc_grads<<<q.tile0[TC_LAYERS] + q.col0[TC_LAYERS], TC_T, TC_SMEM, s>>>(q);
    TcUpdate u;
    u.parts = parts;
    u.part = (const float *)vpart;
    u.gw = g->gw.as<float>();
    u.w = g->w.as<float>();
    u.mw = g->mw.as<float>();
    u.vw = g->vw.as<float>();
    u.gb = g->gb.as<float>();
    u.b = g->b.as<float>();
    u.mb = g->mb.as<float>();
    u.vb = g->vb.as<float>();
    u.wb = g->wb.as<__nv_bfloat16>();
    u.wt = g->wt.as<__nv_bfloat16>();
    u.w4 = g->w4.as<__nv_bfloat16>();
    u.loss = loss;
    u.acc = acc;
    u.rows = rows;
    u.up = up;
    k_tc_update<<<blocks_for(NW + NB_ALL) + 1, 256, 0, s>>>(u);
    cq_count_launch(6);
    return cq_check_cuda(ctx, cudaGetLastError(), "train step");
}

// One optimisation step on a minibatch: forward, MSE against normalised targets, backward,
// Adam.  lr = 0 computes the loss and gradients without an update.
extern "C" cq_status cq_guess_train_step(cq_guess *g, const float *desc, const float *targets,
                                         int64_t rows, float lr, float *loss_host,
                                         float *grad_w_host, float *grad_b_host)
{
    if (!g || !g->ctx || !desc || !targets || rows <= 0) return CQ_ERR_INVALID;
    cq_ctx *ctx = g->ctx;
    cudaStream_t s = ctx->stream;
    void *vloss;
    CQ_TRY(cq_scratch(ctx, "gs_loss", 4 * 256, &vloss));
    if (!g->loss_acc.ptr) {
        CQ_TRY(cq_alloc(ctx, g->loss_acc, 2 * sizeof(double)));
        CQ_TRY(cq_check_cuda(ctx, cudaMemsetAsync(g->loss_acc.ptr, 0, 2 * sizeof(double), s),
                             "loss sums"));
    }
    AdamArgs up = {lr > 0.f ? lr : 0.f, 0.9f, 0.999f, 1e-8f, 1.f, 1.f};
    const int64_t step = g->step + (lr > 0.f ? 1 : 0);  // (a step that is refused does not count)
    if (lr > 0.f) {
        up.c1 = 1.f - std::pow(up.b1, (float)step);
        up.c2 = 1.f - std::pow(up.b2, (float)step);
    }
    CQ_TRY((g->fp32_weights ? train_fp32 : train_tc)(g, desc, targets, rows, (float *)vloss,
                                                     g->loss_acc.as<double>(), up));
    g->step = step;
    if (loss_host) {
        float part[256];
        cudaMemcpyAsync(part, vloss, sizeof(part), cudaMemcpyDeviceToHost, s);
        CQ_TRY(cq_check_cuda(ctx, cudaStreamSynchronize(s), "loss"));
        double tot = 0.0;
        for (int q = 0; q < 256; ++q) tot += part[q];
        *loss_host = (float)(tot / ((double)rows * NOUT));
    }
    if (grad_w_host)
        cudaMemcpyAsync(grad_w_host, g->gw.ptr, 4 * g->n_w, cudaMemcpyDeviceToHost, s);
    if (grad_b_host)
        cudaMemcpyAsync(grad_b_host, g->gb.ptr, 4 * g->n_b, cudaMemcpyDeviceToHost, s);
    if (!loss_host && !grad_w_host && !grad_b_host)
        return cq_check_cuda(ctx, cudaGetLastError(), "train step");
    return cq_check_cuda(ctx, cudaStreamSynchronize(s), "train step");
}

extern "C" cq_status cq_guess_loss_sum(cq_guess *g, double *sq_sum_host, int64_t *rows_host,
                                       int32_t reset)
{
    if (!g || !g->ctx) return CQ_ERR_INVALID;
    cq_ctx *ctx = g->ctx;
    double v[2] = {0.0, 0.0};
    if (g->loss_acc.ptr) {
        cudaMemcpyAsync(v, g->loss_acc.ptr, sizeof(v), cudaMemcpyDeviceToHost, ctx->stream);
        if (reset) cudaMemsetAsync(g->loss_acc.ptr, 0, sizeof(v), ctx->stream);
        CQ_TRY(cq_check_cuda(ctx, cudaStreamSynchronize(ctx->stream), "loss sums"));
    }
    if (sq_sum_host) *sq_sum_host = v[0];
    if (rows_host) *rows_host = (int64_t)v[1];
    return CQ_OK;
}

// Predict every block of P_L: descriptors -> MLP -> un-normalise -> rotate to the global
// frame; writes all (i, j) and (j, i) blocks of L.
extern "C" cq_status cq_guess_apply(cq_guess *g, const cq_pattern *pL, double *L)
{
    if (!g || !g->ctx || !pL || !L) return CQ_ERR_INVALID;
    cq_ctx *ctx = g->ctx;
    const int nb = pL->geo->uniform_nb;
    if (nb != 9 && nb != 4) return cq_fail(ctx, CQ_ERR_INVALID, "guess: uniform 4 or 9 orbitals");
    int64_t n;
    int32_t *pairs;
    CQ_TRY(pair_list(ctx, pL, &pairs, &n));
    void *vd, *vf, *vo, *vp;
    CQ_TRY(cq_scratch(ctx, "ga_desc", 4 * (n + 1) * NDESC, &vd));
    CQ_TRY(cq_scratch(ctx, "ga_frames", 4 * (n + 1) * 9, &vf));
    CQ_TRY(cq_scratch(ctx, "ga_out", 4 * (n + 1) * NOUT, &vo));
    CQ_TRY(cq_scratch(ctx, "ga_pairs", 4 * (n + 1), &vp));
    CQ_TRY(cq_guess_descriptors(ctx, pL, (float *)vd, (float *)vf, (int32_t *)vp));
    // forward in row chunks that keep the activations modest
    const int64_t chunk = 1 << 18;
    for (int64_t r0 = 0; r0 < n; r0 += chunk) {
        const int64_t rows = std::min(chunk, n - r0);
        CQ_TRY(cq_guess_forward(g, (float *)vd + r0 * NDESC, rows, (float *)vo + r0 * NOUT));
    }
    CQ_TRY(cq_check_cuda(ctx, cudaMemsetAsync(L, 0, sizeof(double) * pL->n_values, ctx->stream),
                         "apply"));
    if (n > 0)
        k_apply<<<blocks_for(n, APPLY_P), APPLY_T, 0, ctx->stream>>>(
            n, nb, pL->uniform, (int32_t *)vp, pL->transpose.as<int64_t>(), pL->row.as<int32_t>(),
            pL->col.as<int32_t>(), (float *)vf, (float *)vo, g->mean.as<float>(),
            g->scale.as<float>(), L);
    cq_count_launch();
    return cq_check_cuda(ctx, cudaGetLastError(), "apply");
}

// Tensor-core GEMMs of the learned-guess network (included by guess.cu): BF16 operands and FP32
// accumulation in tensor memory (tcgen05.mma kind::f16) for the three contractions of the MLP --
// the forward layer Z = H W, the backward dH = dZ W^T and the weight gradient dW = H^T dZ --
// with everything that follows an element in its own epilogue: bias and SiLU, silu', the BF16
// copies the next GEMM reads, and their transposes for the weight gradient.
//
// A tile is 128 rows and 64 columns of C = A Bt^T (an MMA of the tile's width rounded up to
// 16).  A (M x K) and Bt (N x K) are row-major BF16; K runs in chunks of up to 256 staged in
// shared memory in the canonical no-swizzle K-major layout (core matrices of 8 rows x 16
// bytes, adjacent along K, 8-row groups 4 KB apart; eight lanes fill one core matrix, so the
// stores have no bank conflicts); two CTAs of 256 threads fit one SM.
//
// What bounds a training step of 4096 rows: launches and latency (a layer is 0.5 GFLOP and
// 4 MB).  In 48 launches of separate passes, with column sums of one thread per column, it
// took 806 us; in these 11 launches about 154 us.
//
// The MMA completion wait is bounded (about two seconds); a CTA that gives up sets bit 16
// of the flag word, frees its tensor memory and returns.
constexpr int TC_MT = 128;      // rows of C per CTA
constexpr int TC_NT = 64;       // columns of C per CTA
constexpr int TC_KC = 256;      // K values per staged chunk
constexpr int TC_T = 256;       // threads per CTA
constexpr int TC_SBO = (TC_KC / 8) * 128;
constexpr int TC_SMEM = TC_MT * TC_KC * 2 + TC_NT * TC_KC * 2 + 64;
constexpr long long TC_WAIT = 4000000000LL;

__device__ __forceinline__ uint32_t tc_smem_u32(const void *p)
{
    return (uint32_t)__cvta_generic_to_shared(p);
}

__device__ __forceinline__ uint64_t tc_desc(uint32_t saddr)
{
    uint64_t d = (uint64_t)((saddr >> 4) & 0x3FFF);
    d |= (uint64_t)(128 >> 4) << 16;
    d |= (uint64_t)(TC_SBO >> 4) << 32;
    d |= (uint64_t)1 << 46;
    return d;
}

// rows [r0, r0 + rows) (rows a multiple of 8) of a row-major BF16 matrix, K range [k0, k0 + kn),
// into the staged layout (zeros outside the matrix or the range); kn16 = kn rounded up to 16
__device__ __forceinline__ void tc_stage(uint8_t *dst, int rows, const __nv_bfloat16 *src,
                                         int64_t ld, int r0, int rmax, int64_t k0, int64_t kend,
                                         int kn16)
{
    const int groups = kn16 / 8;
#pragma unroll 4
    for (int e = threadIdx.x; e < rows * groups; e += TC_T) {
        const int q = e >> 3, g = q % groups, r = (q / groups) * 8 + (e & 7);
        const int64_t k = k0 + 8 * g;
        uint8_t *o = dst + (r >> 3) * TC_SBO + g * 128 + (r & 7) * 16;
        const __nv_bfloat16 *p = src + (int64_t)(r0 + r) * ld + k;
        if (r0 + r < rmax && k + 8 <= kend && (reinterpret_cast<uintptr_t>(p) & 15) == 0) {
            // eight values, in flight until tc_staged
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(tc_smem_u32(o)), "l"(p)
                         : "memory");
        } else {
            uint32_t u[4] = {0u, 0u, 0u, 0u};
            if (r0 + r < rmax)
#pragma unroll
                for (int x = 0; x < 8; ++x)
                    if (k + x < kend)
                        u[x >> 1] |= (uint32_t)__bfloat16_as_ushort(p[x]) << (16 * (x & 1));
            *reinterpret_cast<uint4 *>(o) = make_uint4(u[0], u[1], u[2], u[3]);
        }
    }
}

// This thread's staged copies have landed and are visible to the tensor cores.
__device__ __forceinline__ void tc_staged()
{
    asm volatile("cp.async.wait_all;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

// One tile of C = A Bt^T: rows m0.., columns n0.., K range [kb, ke) of row-major operands.  The
// epilogue epi(row, col, v) receives 16 columns at a time of each row below M (values of columns
// past N are zeros or padding).
template <class Epi>
__device__ __forceinline__ void tc_tile(int M, int N, const __nv_bfloat16 *A, int64_t lda,
                                        const __nv_bfloat16 *Bt, int64_t ldb, int m0, int n0,
                                        int64_t kb, int64_t ke, int32_t *flag, Epi epi)
{
    extern __shared__ __align__(1024) uint8_t smem[];
    uint8_t *sa = smem, *sb = smem + TC_MT * TC_KC * 2;
    uint64_t *bar = reinterpret_cast<uint64_t *>(sb + TC_NT * TC_KC * 2);
    uint32_t *tslot = reinterpret_cast<uint32_t *>(bar + 1);
    const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
    if (t == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(tc_smem_u32(bar)), "r"(1));
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                         tc_smem_u32(tslot)),
                     "r"(TC_NT));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = *tslot;
    const int Npad = ((min(TC_NT, N - n0) + 15) / 16) * 16;  // this tile's MMA width
    // kind::f16: D = F32, A = B = BF16, both K-major, N = Npad, M = 128
    const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(Npad >> 3) << 17) |
                           ((uint32_t)(TC_MT >> 4) << 24);
    uint32_t phase = 0;
    bool issued = false, ok = true;
    for (int64_t kc = kb; kc < ke && ok; kc += TC_KC) {
        const int kn = (int)min((int64_t)TC_KC, ke - kc);
        const int kn16 = (kn + 15) & ~15;
        tc_stage(sa, TC_MT, A, lda, m0, M, kc, ke, kn16);
        tc_stage(sb, Npad, Bt, ldb, n0, N, kc, ke, kn16);
        tc_staged();
        __syncthreads();
        if (t == 0) {
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const uint64_t da = tc_desc(tc_smem_u32(sa)), db = tc_desc(tc_smem_u32(sb));
            for (int ks = 0; ks < kn16 / 16; ++ks) {
                const uint32_t acc = (issued || ks > 0) ? 1u : 0u;
                asm volatile(
                    "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
                    "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}\n" ::"r"(tmem),
                    "l"(da + (uint64_t)((ks * 256) >> 4)), "l"(db + (uint64_t)((ks * 256) >> 4)),
                    "r"(idesc), "r"(acc));
            }
            asm volatile(
                "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                    tc_smem_u32(bar))
                : "memory");
        }
        issued = true;
        // every thread waits for the chunk's MMAs before the next staging overwrites them;
        // past the limit the call has failed, but the wait goes on (bounded again) so that
        // no MMA is still writing when the tensor memory is freed
        const long long t0 = clock64();
        for (;;) {
            uint32_t done;
            asm volatile(
                "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
                "selp.u32 %0, 1, 0, p;\n\t}\n"
                : "=r"(done)
                : "r"(tc_smem_u32(bar)), "r"(phase)
                : "memory");
            if (done) break;
            const long long dt = clock64() - t0;
            if (dt > TC_WAIT) ok = false;
            if (dt > 2 * TC_WAIT) break;
        }
        phase ^= 1u;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        ok = __syncthreads_and(ok);  // uniform: every thread leaves the loop together
    }
    if (ok) {
        // epilogue: warp w holds rows m0 + 32 (w % 4) + lane, columns from 32 (w / 4)
        const int row = m0 + (warp & 3) * 32 + lane, c0 = (warp >> 2) * 32;
        for (int cb = c0; cb < min(Npad, c0 + 32); cb += 16) {
            uint32_t v[16];
            if (issued) {
                asm volatile(
                    "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,"
                    "%11,%12,%13,%14,%15}, [%16];"
                    : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]),
                      "=r"(v[6]), "=r"(v[7]), "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]),
                      "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
                    : "r"(tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)cb));
                asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
            } else {
#pragma unroll
                for (int x = 0; x < 16; ++x) v[x] = 0u;
            }
            if (row < M) {
                float f[16];
#pragma unroll
                for (int x = 0; x < 16; ++x) f[x] = __uint_as_float(v[x]);
                epi(row, n0 + cb, f);
            }
        }
    } else if (t == 0) {
        atomicOr(flag, 16);
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 0) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TC_NT));
    }
}

// 16 values of a row as BF16 (row-major, 32-byte aligned, if row is not null) and, if t is not
// null, into the transposed copy at t (t[x * ld], neighbouring rows in neighbouring lanes)
__device__ __forceinline__ void tc_put_bf16(__nv_bfloat16 *row, __nv_bfloat16 *t, int64_t ld,
                                            const float (&f)[16])
{
    uint32_t u[8];
    __nv_bfloat16 b[16];
#pragma unroll
    for (int x = 0; x < 16; ++x) b[x] = __float2bfloat16(f[x]);
#pragma unroll
    for (int x = 0; x < 8; ++x)
        u[x] = (uint32_t)__bfloat16_as_ushort(b[2 * x]) |
               ((uint32_t)__bfloat16_as_ushort(b[2 * x + 1]) << 16);
    if (row) {
        uint4 *o = reinterpret_cast<uint4 *>(row);
        o[0] = make_uint4(u[0], u[1], u[2], u[3]);
        o[1] = make_uint4(u[4], u[5], u[6], u[7]);
    }
    if (t)
#pragma unroll
        for (int x = 0; x < 16; ++x) t[x * ld] = b[x];
}

__device__ __forceinline__ void tc_put_f32(float *row, const float (&f)[16])
{
    float4 *o = reinterpret_cast<float4 *>(row);
#pragma unroll
    for (int x = 0; x < 4; ++x)
        o[x] = make_float4(f[4 * x], f[4 * x + 1], f[4 * x + 2], f[4 * x + 3]);
}

// Hidden layer: Z = A W + bias (stored if Z is not null), Hb = bf16(silu(Z)) and, if Ht is not
// null, its transpose (ld_t apart).  N is a multiple of 64.
__global__ void __launch_bounds__(TC_T, 2)
k_tc_hidden(int M, int N, int K, const __nv_bfloat16 *A, const __nv_bfloat16 *Wt,
            const float *bias, float *Z, __nv_bfloat16 *Hb, __nv_bfloat16 *Ht, int64_t ld_t,
            int32_t *flag)
{
    tc_tile(M, N, A, K, Wt, K, blockIdx.x * TC_MT, blockIdx.y * TC_NT, 0, K, flag,
            [&](int row, int col, float (&f)[16]) {
#pragma unroll
                for (int x = 0; x < 16; ++x) f[x] = f[x] + bias[col + x];
                if (Z) tc_put_f32(Z + (int64_t)row * N + col, f);
#pragma unroll
                for (int x = 0; x < 16; ++x) f[x] = f[x] / (1.f + __expf(-f[x]));
                tc_put_bf16(Hb + (int64_t)row * N + col, Ht ? Ht + col * ld_t + row : nullptr, ld_t,
                            f);
            });
}

// Output layer: Y = A W + bias (linear), row-major with N columns
__global__ void __launch_bounds__(TC_T, 2)
k_tc_output(int M, int N, int K, const __nv_bfloat16 *A, const __nv_bfloat16 *Wt,
            const float *bias, float *Y, int32_t *flag)
{
    tc_tile(M, N, A, K, Wt, K, blockIdx.x * TC_MT, blockIdx.y * TC_NT, 0, K, flag,
            [&](int row, int col, float (&f)[16]) {
#pragma unroll
                for (int x = 0; x < 16; ++x)
                    if (col + x < N) Y[(int64_t)row * N + col + x] = f[x] + bias[col + x];
            });
}

// Backward through a hidden layer of N units: dZ = (dZ' W^T) silu'(Z) as FP32, as BF16 (if dZb
// is not null) and transposed BF16.  dZ' is M x K (leading dimension lda), W N x K (ldw).
__global__ void __launch_bounds__(TC_T, 2)
k_tc_back(int M, int N, int K, const __nv_bfloat16 *dZn, int64_t lda, const __nv_bfloat16 *W,
          int64_t ldw, const float *Z, float *dZ, __nv_bfloat16 *dZb, __nv_bfloat16 *dZt,
          int64_t ld_t, int32_t *flag)
{
    tc_tile(M, N, dZn, lda, W, ldw, blockIdx.x * TC_MT, blockIdx.y * TC_NT, 0, K, flag,
            [&](int row, int col, float (&f)[16]) {
                const float4 *zr = reinterpret_cast<const float4 *>(Z + (int64_t)row * N + col);
                float z[16];
#pragma unroll
                for (int x = 0; x < 4; ++x) {
                    const float4 q = zr[x];
                    z[4 * x] = q.x;
                    z[4 * x + 1] = q.y;
                    z[4 * x + 2] = q.z;
                    z[4 * x + 3] = q.w;
                }
#pragma unroll
                for (int x = 0; x < 16; ++x) {
                    const float s = 1.f / (1.f + __expf(-z[x]));
                    f[x] = f[x] * (s * (1.f + z[x] * (1.f - s)));
                }
                tc_put_f32(dZ + (int64_t)row * N + col, f);
                tc_put_bf16(dZb ? dZb + (int64_t)row * N + col : nullptr, dZt + col * ld_t + row, ld_t, f);
            });
}

// All weight gradients of a step, dW_l = H_{l-1}^T dZ_l split over the rows into `parts` partial
// products (summed in order by k_tc_update), and the bias gradients, in one launch: first the
// blocks of the column sums (32 columns of one layer each: they take longest), then those of
// the layers' tiles (tile, then part); col0 and tile0 count the blocks before each layer's.
constexpr int TC_LAYERS = 4;
struct TcGrads {
    int rows, parts;
    int64_t chunk;                          // rows per part (a multiple of 16)
    int64_t ld_t;                           // leading dimension of the transposes
    int K[TC_LAYERS], N[TC_LAYERS];         // layer l: weights K x N
    const __nv_bfloat16 *Ht[TC_LAYERS], *dZt[TC_LAYERS];
    const float *dZ[TC_LAYERS];             // rows x N
    float *part[TC_LAYERS];                 // parts x K x N
    float *gb[TC_LAYERS];
    int tile0[TC_LAYERS + 1], col0[TC_LAYERS + 1];
    int32_t *flag;
};

// Column sums over the rows in ascending order (one chain of additions per column, so the
// order is that of a plain loop): 32 columns per CTA; eight warps stage 256 rows in shared
// memory (by column, so that one warp's lanes read four rows at a time) while the first warp
// adds the 256 before.  The chain itself is four clocks per row.
__device__ __forceinline__ void tc_colsum(int rows, int N, int c0, const float *dZ, float *db)
{
    extern __shared__ __align__(1024) uint8_t smem[];
    constexpr int R = 256, PER = R / (TC_T / 32), LD = R + 4;
    static_assert(2 * 32 * LD * 4 <= TC_SMEM, "column buffers");
    float *buf = reinterpret_cast<float *>(smem);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, c = c0 + lane;
    float reg[PER];
    auto fetch = [&](int r0) {
#pragma unroll
        for (int x = 0; x < PER; ++x) {
            const int r = r0 + warp * PER + x;
            reg[x] = (r < rows && c < N) ? __ldg(dZ + (int64_t)r * N + c) : 0.f;
        }
    };
    fetch(0);
    float s = 0.f;
    for (int r0 = 0, b = 0; r0 < rows; r0 += R, b ^= 1) {
        float *col = buf + (b * 32 + lane) * LD;
#pragma unroll
        for (int x = 0; x < PER; x += 4)
            *reinterpret_cast<float4 *>(col + warp * PER + x) =
                make_float4(reg[x], reg[x + 1], reg[x + 2], reg[x + 3]);
        __syncthreads();
        fetch(r0 + R);
        if (warp == 0) {
            const int n = min(R, rows - r0);
            if (n == R) {
#pragma unroll 16
                for (int r = 0; r < R; r += 4) {
                    const float4 v = *reinterpret_cast<const float4 *>(col + r);
                    s += v.x;
                    s += v.y;
                    s += v.z;
                    s += v.w;
                }
            } else {
                for (int r = 0; r < n; ++r) s += col[r];
            }
        }
    }
    if (warp == 0 && c < N) db[c] = s;
}

__global__ void __launch_bounds__(TC_T, 2) k_tc_grads(const TcGrads p)
{
    int b = blockIdx.x, l = 0;
    if (b < p.col0[TC_LAYERS]) {
        while (b >= p.col0[l + 1]) ++l;
        tc_colsum(p.rows, p.N[l], (b - p.col0[l]) * 32, p.dZ[l], p.gb[l]);
        return;
    }
    b -= p.col0[TC_LAYERS];
    while (b >= p.tile0[l + 1]) ++l;
    const int K = p.K[l], N = p.N[l], q = b - p.tile0[l], tm = (K + TC_MT - 1) / TC_MT;
    const int z = q % p.parts, tile = q / p.parts;
    const int64_t kb = (int64_t)z * p.chunk, ke = min((int64_t)p.rows, kb + p.chunk);
    float *out = p.part[l] + (int64_t)z * K * N;
    tc_tile(K, N, p.Ht[l], p.ld_t, p.dZt[l], p.ld_t, (tile % tm) * TC_MT, (tile / tm) * TC_NT, kb,
            ke, p.flag, [&](int row, int col, float (&f)[16]) {
#pragma unroll
                for (int x = 0; x < 16; ++x)
                    if (col + x < N) out[(int64_t)row * N + col + x] = f[x];
            });
}

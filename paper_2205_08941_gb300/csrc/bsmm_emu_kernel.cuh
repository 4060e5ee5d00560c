// The tile kernel of the emulated-FP64 product (included by bsmm_split.cu after the split
// kernel, whose barrier, copy, queue, epilogue and timeout helpers it shares).
//
// Operands are eight BF16 digit planes per value (emu_digits.cuh): A_p, B_q with planes
// pre-scaled by 2^(-8p), so the product of planes p and q lands at level p + q.  The planes of
// a B piece follow one another, so its eight planes of 64 columns are one operand of 512
// columns, and A_p times planes 0 .. 7 - p of B fills the levels p .. 7, which lie next to one
// another in tensor memory (64 columns each): the 36 products of a K step are twelve MMAs of
// up to 256 columns.  Over one scale period a level-l sum is an integer times 2^(-8 l) of
// magnitude at most (l + 1) * 144 * 128^2 (at most 144 K values per period), below 2^24 and
// so exact for l <= 6; level 7's rounding is 2^-56 below level 0.  A scale period is one
// tail group of K (16 consecutive atoms in Morton order for 9 orbitals, 4 for 4): the main K
// steps pairing the tile's K atoms of the group, then the group's tail step.
//
// At a period's end the drain warps compress every element's eight level sums into three
// floats (x0, x1, x2) and add them, scaled by 2^(E_A(row) + E_B(column) - 14), into a
// three-float sum (h, m, l) in registers: 45 FP32 operations per element (84 when each level was
// scaled and added by itself).  Levels 0-4 are compressed without error; levels 5-7 are added in
// FP32 first, which loses at most 2^-65 of level 0's bound (2^-65.0 in a CPU emulation of sums
// spread over their whole ranges, 2^-68 with Gaussian ones): the digits resolve 2^-64.
// After a tile's last period C = beta C + alpha (h + m + l) is written in FP64.
//
// Warp roles: as in the split kernel, with 16 drain warps (four to a scheduler, sixteen columns
// each).  A stage holds one K step (main step: two A main pieces of 8 planes x 128 rows x 8 K,
// 16 KB each, and two B main pieces of 8 KB; tail step: one A tail piece, 32 KB, and one B tail
// piece, 16 KB; both kinds with their second column one main piece further).  The levels take
// all 512 columns of tensor memory, so the MMAs wait while a period drains.
//
// What bounds it: per K step 1185 clocks of MMA (N = 256 runs at 128 clocks per MMA, the
// tensor cores' own rate; N = 64 took 58 for 32 clocks of work), then the drain, about 5000
// clocks per period of three to nine K steps.  Measured, U.X kept on P_L: 512 atoms 12.6 ms
// (36 MMAs of 64 columns per step) -> 11.1 with the cheaper waits -> 6.1 (wide MMAs, queue,
// levels compressed before they are scaled, sums in registers) -> 5.1 with 16 drain warps in
// place of 8 -> 4.8 ms with the scale factors made once per row and column; 1728 atoms 152 ->
// 56 ms, L.S on 1728 atoms (three steps per period) 30.7 -> 12.9 ms.
//
// Every wait is bounded as in the split kernel; a CTA that gives up retires its copies and
// MMAs, frees its tensor memory and sets bit 16 of the context flag.
constexpr int NSE = 4;                       // shared-memory stages (one K step each)
constexpr int E_AMAIN = EMU_P * COLB_A;      // 16 KB: an A main piece (planes x one column)
constexpr int E_BMAIN = EMU_P * COLB_B;      // 8 KB
constexpr int E_ATAIL = 2 * E_AMAIN;         // 32 KB: an A tail piece (two columns of planes)
constexpr int E_BTAIL = 2 * E_BMAIN;         // 16 KB
constexpr int E_STAGE = E_ATAIL + E_BTAIL;   // one K step: A at 0, B at E_ATAIL
constexpr int E_TMEM_COLS = EMU_P * NT;      // 512: one accumulator per level
constexpr int E_DRAIN = 16;                  // drain warps: four per scheduler hide each other's
                                             // tensor-memory reads and FP32 chains
constexpr int E_W = 4 * NT / E_DRAIN;        // columns of a drain warp
constexpr int EW_PROD = E_DRAIN, EW_MMA = EW_PROD + NPROD, EW_SCHED = EW_MMA + 1;
constexpr int E_ST = 32 * (EW_SCHED + 1);    // threads per CTA (20 warps)
constexpr int E_READERS = NPROD + 1 + E_DRAIN;
constexpr int E_MMAS = EMU_P * (EMU_P + 1) / 2;  // 36 plane products per K step

struct EBars {
    uint64_t full[NSE], empty[NSE], acc_full, acc_empty, done;
    static constexpr int TQ = 2;  // tiles queued ahead
    uint64_t tile_full[TQ], tile_empty[TQ];
    TileRec rec[TQ];
    uint32_t tmem_slot;
    int abort_flag;
};
static_assert(sizeof(EBars) <= BAR_BYTES, "barrier block");
static_assert(NSE * E_STAGE + BAR_BYTES <= 227 * 1024, "shared memory per CTA");

struct EmuArgs {
    int n_tiles;
    const int64_t *kstart;     // K-step range of each tile (n_tiles + 1)
    const int4 *steps;         // piece entries of every K step; second entries TAIL_STEP in the
                               // tail step that ends a scale period
    const int32_t *cidx;       // C block of each (M slot, N slot) pair of each tile
    const uint8_t *a_main;     // A main pieces of entries [am0, ...)
    int64_t am0;
    const uint8_t *a_tail;     // A tail pieces of entries [at0, ...)
    int64_t at0;
    const uint8_t *b_main;     // all B main pieces
    const uint8_t *b_tail;     // all B tail pieces
    const uint8_t *zero;       // an all-zero A main piece
    const int16_t *scale_a;    // group exponent of every (A tail entry, row): n_at x 128
    const int16_t *scale_b;    // group exponent of every (B tail entry, column): n_bt x 64
    double *C;
    int c_stride;
    double alpha, beta;
    int32_t *flag;
    uint32_t *counter;         // two zero words of the tile queue (left at zero)
};

// x 2^e for exponents outside one FP32 scale factor's range, exact while the result stays a
// normal FP32 number (rare, and out of line: the drain's straight-line code has to stay in
// the instruction cache)
__device__ __noinline__ float3 mul_pow2(float3 x, int e)
{
    auto times = [&](float f) { x = make_float3(x.x * f, x.y * f, x.z * f); };
    for (; e > 127; e -= 127) times(1.7014118e38f);    // 2^127
    for (; e < -126; e += 126) times(1.1754944e-38f);  // 2^-126
    times(__uint_as_float((uint32_t)(e + 127) << 23));
    return x;
}

// a + b c as a rounded sum and its error, for an exact product b c (c a power of two)
__device__ __forceinline__ float two_sum(float a, float b, float c, float &err)
{
    const float s = fmaf(b, c, a), bp = s - a;
    err = (a - (s - bp)) + fmaf(b, c, -bp);
    return s;
}

// a + b as a rounded sum and its error where a is a multiple of b's last place (or larger than b)
__device__ __forceinline__ float fast_two_sum(float a, float b, float &err)
{
    const float s = a + b;
    err = b - (s - a);
    return s;
}

// Eight level sums (level l a multiple of 2^(-8 l) below 2^(24 - 8 l)) as x0 + x1 + x2.  From
// the bottom up, each level is a multiple of the last place of the sum of those below it, so
// the fast sums are exact; e0 is a multiple of s1's last place and e1 half of it at most, so
// theirs is too.
__device__ __forceinline__ void emu_compress(const uint32_t (&v)[EMU_P], float &x0, float &x1,
                                             float &x2)
{
    static_assert(EMU_P == 8, "levels");
    float e0, e1, e2, e3, e4, r;
    const float w = __uint_as_float(v[5]) + (__uint_as_float(v[6]) + __uint_as_float(v[7]));
    const float s4 = fast_two_sum(__uint_as_float(v[4]), w, e4);
    const float s3 = fast_two_sum(__uint_as_float(v[3]), s4, e3);
    const float s2 = fast_two_sum(__uint_as_float(v[2]), s3, e2);
    const float s1 = fast_two_sum(__uint_as_float(v[1]), s2, e1);
    x0 = fast_two_sum(__uint_as_float(v[0]), s1, e0);
    x1 = fast_two_sum(e0, e1, r);
    x2 = r + (e2 + (e3 + e4));
}

constexpr int E_C = 4;  // columns drained together

__device__ __forceinline__ void tm_ld(uint32_t addr, uint32_t (&v)[4])
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];"
                 : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3])
                 : "r"(addr));
}

constexpr int TAIL_STEP = -2;  // second entry of a tail step (-1: no second atom)

// Columns [COL, COL + N) of plane PA's product with planes 0 .. 7 - PA of B (COL counted from
// the plane's first level), a and b the low words of the plane-0 descriptors.
template <int PA, int COL, int N>
__device__ __forceinline__ void emu_mma(uint32_t tmem, uint32_t a, uint32_t b, uint32_t acc)
{
    static_assert(N % 16 == 0 && N <= 256 && COL + N <= (EMU_P - PA) * NT, "MMA width");
    constexpr uint32_t hi = (uint32_t)(128 >> 4) | (1u << 14);  // piece_desc's high word
    constexpr uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) |
                               ((uint32_t)(MT >> 4) << 24);
    asm volatile(
        "{\n\t.reg .pred p;\n\t.reg .b64 da, db;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "mov.b64 da, {%1, %5};\n\tmov.b64 db, {%2, %5};\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %3, p;\n\t}\n" ::"r"(
            tmem + (uint32_t)(PA * NT + COL)),
        "r"(a + (uint32_t)(PA * COLB_A / 16)), "r"(b + (uint32_t)COL), "r"(idesc), "r"(acc), "r"(hi));
}

// The 36 plane products of one K step; acc = 0 overwrites every level (plane 0 reaches all).
__device__ __forceinline__ void emu_step(uint32_t tmem, uint32_t a, uint32_t b, uint32_t acc)
{
    emu_mma<0, 0, 256>(tmem, a, b, acc);
    emu_mma<0, 256, 256>(tmem, a, b, acc);
    emu_mma<1, 0, 224>(tmem, a, b, 1u);
    emu_mma<1, 224, 224>(tmem, a, b, 1u);
    emu_mma<2, 0, 192>(tmem, a, b, 1u);
    emu_mma<2, 192, 192>(tmem, a, b, 1u);
    emu_mma<3, 0, 160>(tmem, a, b, 1u);
    emu_mma<3, 160, 160>(tmem, a, b, 1u);
    emu_mma<4, 0, 256>(tmem, a, b, 1u);
    emu_mma<5, 0, 192>(tmem, a, b, 1u);
    emu_mma<6, 0, 128>(tmem, a, b, 1u);
    emu_mma<7, 0, 64>(tmem, a, b, 1u);
}

// One producer warp (SIDE 0: A pieces, 1: B pieces) over all K steps of the CTA's tiles.
template <int SIDE>
__device__ __forceinline__ void emu_produce(const EmuArgs &p, uint32_t sm0, EBars *bars,
                                            volatile int *abort_flag, int lane)
{
    constexpr int MAIN = SIDE ? E_BMAIN : E_AMAIN;
    const uint8_t *mains = SIDE ? p.b_main : p.a_main - p.am0 * E_AMAIN;
    const uint8_t *tails = SIDE ? p.b_tail : p.a_tail - p.at0 * E_ATAIL;
    const uint32_t dst0 = sm0 + (SIDE ? E_ATAIL : 0);
    // K steps come 32 at a time, one per lane, loaded one batch ahead
    auto load = [&](const TileRec &t, int base) {
        return base + lane < t.nks
                   ? __ldg(reinterpret_cast<const int2 *>(p.steps + t.s0 + base + lane) + SIDE)
                   : make_int2(0, 0);
    };
    const uint64_t policy = SIDE ? l2_evict_first() : l2_evict_last();
    uint32_t sg = 0;  // running stage (K step) counter
    bool ok = true;
    TileRec t = next_tile(bars, 0, abort_flag, lane);
    int2 cur = load(t, 0);
    for (uint32_t n = 1; t.tile >= 0 && ok; ++n) {
        TileRec tn = t;
        for (int base = 0; base == 0 || base < t.nks; base += 32) {
            int2 nxt;
            if (base + 32 < t.nks) {
                nxt = load(t, base + 32);
            } else {
                tn = next_tile(bars, n, abort_flag, lane);
                nxt = load(tn, 0);
            }
            for (int q = base; q < min(t.nks, base + 32); ++q, ++sg) {
                const uint32_t s = sg % NSE, fb = smem_u32(&bars->full[s]);
                const int ex = __shfl_sync(0xffffffffu, cur.x, q - base);
                const int ey = __shfl_sync(0xffffffffu, cur.y, q - base);
                if (!warp_wait_lane0(sg >= (uint32_t)NSE, smem_u32(&bars->empty[s]),
                                     ((sg / NSE) + 1) & 1u, abort_flag, lane)) {
                    ok = false;
                    break;
                }
                if (lane == 0) {
                    const uint32_t dst = dst0 + s * E_STAGE;
                    const bool tail = ey == TAIL_STEP, pair = ey == ex + 1;
                    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(fb),
                                 "r"((uint32_t)(2 * MAIN))
                                 : "memory");
                    bulk_copy(dst, tail ? tails + (int64_t)ex * (2 * MAIN) : mains + (int64_t)ex * MAIN,
                              tail || pair ? 2 * MAIN : MAIN, fb, policy);
                    if (!tail && !pair)
                        bulk_copy(dst + MAIN, ey < 0 ? p.zero : mains + (int64_t)ey * MAIN, MAIN, fb,
                                  policy);
                }
                __syncwarp();
            }
            if (!ok) break;
            cur = nxt;
        }
        t = tn;
    }
    // every copy lands before the CTA's shared memory is released (both sides arm the same
    // stages, as in the split kernel)
    if (lane == 0)
        for (uint32_t k = 0; k < (uint32_t)NSE && k < sg; ++k) {
            const uint32_t c = sg - 1 - k;
            if (!bar_wait_plain(smem_u32(&bars->full[c % NSE]), (c / NSE) & 1u)) *abort_flag = 1;
        }
    __syncwarp();
}

// The scheduler warp: hands out the launch's tiles in order, so that the tiles in flight on the
// GPU stay neighbours (they share the A pieces of one or two M groups) and no CTA idles while
// others hold several tiles.
__device__ __forceinline__ void schedule(const EmuArgs &p, EBars *bars, volatile int *abort_flag,
                                         int lane)
{
    if (lane == 0) {
        int i = blockIdx.x;
        for (uint32_t n = 0;; ++n) {
            TileRec r;
            r.tile = -1;
            r.s0 = 0;
            r.nks = r.nm = 0;
            if (i < p.n_tiles) {
                r.tile = i;
                r.s0 = p.kstart[i];
                r.nks = (int)(p.kstart[i + 1] - r.s0);
                r.nm = 0;
            }
            if (n >= (uint32_t)EBars::TQ &&
                !bar_wait(smem_u32(&bars->tile_empty[n % EBars::TQ]), ((n / EBars::TQ) + 1) & 1u, abort_flag))
                break;
            bars->rec[n % EBars::TQ] = r;
            bar_arrive(smem_u32(&bars->tile_full[n % EBars::TQ]));
            if (r.tile < 0) break;
            i = (int)gridDim.x + (int)atomicAdd(&p.counter[0], 1u);
        }
        // the last CTA to finish handing out resets the counters for the next launch
        __threadfence();
        if (atomicInc(&p.counter[1], gridDim.x - 1) == gridDim.x - 1) atomicExch(&p.counter[0], 0u);
    }
    __syncwarp();
}

template <int NB>
__global__ void __launch_bounds__(E_ST, 1) k_bsmm_emu(const EmuArgs p)
{
    constexpr int GI = MT / NB, GJ = NT / NB;
    extern __shared__ __align__(1024) uint8_t smem[];
    EBars *bars = reinterpret_cast<EBars *>(smem + NSE * E_STAGE);
    volatile int *abort_flag = &bars->abort_flag;
    const int t = threadIdx.x, warp = __shfl_sync(0xffffffffu, t >> 5, 0), lane = t & 31;
    const uint32_t sm0 = smem_u32(smem);

    if (t == 0) {
        auto init = [](uint64_t *b, int n) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(b)), "r"(n));
        };
        for (int s = 0; s < NSE; ++s) {
            init(&bars->full[s], NPROD);
            init(&bars->empty[s], 1);
        }
        init(&bars->acc_full, 1);
        init(&bars->acc_empty, 32 * E_DRAIN);
        for (int r = 0; r < EBars::TQ; ++r) {
            init(&bars->tile_full[r], 1);
            init(&bars->tile_empty[r], E_READERS);
        }
        init(&bars->done, 1);
        bars->abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == EW_MMA) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                         smem_u32(&bars->tmem_slot)),
                     "r"(E_TMEM_COLS));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = bars->tmem_slot;

    if (warp == EW_PROD) {
        emu_produce<0>(p, sm0, bars, abort_flag, lane);
    } else if (warp == EW_PROD + 1) {
        emu_produce<1>(p, sm0, bars, abort_flag, lane);
    } else if (warp == EW_MMA) {
        // ------------------------------------------------------------ MMA issue
        const bool el = elect_one();
        uint32_t sg = 0, pg = 0;  // running K step and period counters
        bool ok = true;
        const uint32_t da = (uint32_t)piece_desc(sm0, E_AMAIN);
        const uint32_t db = (uint32_t)piece_desc(sm0 + E_ATAIL, E_BMAIN);
        for (uint32_t n = 0; ok; ++n) {
            const TileRec tr = next_tile(bars, n, abort_flag, lane);
            if (tr.tile < 0) break;
            auto tails = [&](int base) {  // which of 32 K steps end a period
                return __ballot_sync(0xffffffffu,
                                     base + lane < tr.nks &&
                                         __ldg(&p.steps[tr.s0 + base + lane].y) == TAIL_STEP);
            };
            uint32_t ends = tails(0), ends_next = 0;
            bool first = true;
            for (int q = 0; q < tr.nks; ++q, ++sg) {
                if ((q & 31) == 0) {
                    if (q) ends = ends_next;
                    if (q + 32 < tr.nks) ends_next = tails(q + 32);
                }
                const bool last = ends >> (q & 31) & 1u;
                if (first && pg > 0 &&
                    !warp_wait(smem_u32(&bars->acc_empty), (pg - 1) & 1u, abort_flag)) {
                    ok = false;
                    break;
                }
                const uint32_t s = sg % NSE;
                if (!warp_wait(smem_u32(&bars->full[s]), (sg / NSE) & 1u, abort_flag)) {
                    ok = false;
                    break;
                }
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                if (el) {
                    const uint32_t o = s * (E_STAGE >> 4);
                    emu_step(tmem, da + o, db + o, first ? 0u : 1u);
                    bar_commit(smem_u32(&bars->empty[s]));
                    if (last) bar_commit(smem_u32(&bars->acc_full));
                }
                __syncwarp();
                first = last;
                pg += last;
            }
        }
        // retire every MMA before the tensor memory is released
        if (sg > 0 && el) {
            bar_commit(smem_u32(&bars->done));
            if (!bar_wait_plain(smem_u32(&bars->done), 0u)) *abort_flag = 1;
        }
        __syncwarp();
    } else if (warp == EW_SCHED) {
        schedule(p, bars, abort_flag, lane);
    } else {
        // ------------------------------------------------------------ drain and epilogue
        // at every tail step the warp drains the levels with the scales of the step's tail
        // pieces (the period's group exponents); the K-step entries come 32 at a time
        const int quarter = warp & 3, c0 = (warp >> 2) * E_W;  // lanes and first column
        const int arow = quarter * 32 + lane;
        const uint32_t lane_addr = tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)c0;
        uint32_t pg = 0;
        bool ok = true;
        for (uint32_t n = 0; ok; ++n) {
            const TileRec tr = next_tile(bars, n, abort_flag, lane);
            if (tr.tile < 0) break;
            // this row's C blocks, loaded now and used after the tile's last period
            constexpr int NJ = epi_slots<NB, E_W>(), G = E_W / E_C;
            int32_t cid[NJ];
            const int si = arow / NB, j0 = c0 / NB;
#pragma unroll
            for (int u = 0; u < NJ; ++u)
                cid[u] = (arow < GI * NB && j0 + u < GJ)
                             ? __ldg(&p.cidx[((int64_t)tr.tile * GI + si) * GJ + j0 + u])
                             : -1;
            // groups of E_C columns in which a row of this warp has a block of P_C: only they
            // are drained (on the 4096-atom cell's U.X a tile's slots are 17 % full)
            uint32_t need = 0;
#pragma unroll
            for (int g = 0; g < G; ++g) {
                bool any = false;
#pragma unroll
                for (int u = 0; u < NJ; ++u) {
                    const int s0 = (j0 + u) * NB - c0;  // the slot's first column of this warp's
                    any = any || (cid[u] >= 0 && s0 < E_C * (g + 1) && s0 + NB > E_C * g);
                }
                need |= (uint32_t)__any_sync(0xffffffffu, any) << g;
            }
            float h[E_W], m[E_W], l[E_W];
#pragma unroll
            for (int x = 0; x < E_W; ++x) h[x] = m[x] = l[x] = 0.f;
            for (int base = 0; base < tr.nks && ok; base += 32) {
                const int4 ent = base + lane < tr.nks ? __ldg(&p.steps[tr.s0 + base + lane])
                                                      : make_int4(0, 0, 0, 0);
                uint32_t ends = __ballot_sync(0xffffffffu, base + lane < tr.nks && ent.y == TAIL_STEP);
                for (; ends; ends &= ends - 1, ++pg) {
                    const int q = __ffs(ends) - 1;
                    const int ea_ent = __shfl_sync(0xffffffffu, ent.x, q);
                    const int eb_ent = __shfl_sync(0xffffffffu, ent.z, q);
                    // scales first, so their loads overlap the wait for the accumulators: this
                    // row's 2^(E_A - 14), and in lane x column x's 2^E_B.  Groups without a
                    // nonzero value have zero sums and a poisoned group's are NaN: any scale
                    // will do.  2^ea 2^eb has to be finite (0 x infinity would be NaN), so at most
                    // 2^127: E_A from -60 to 81 and E_B from -60 to 60 take the single factor,
                    // anything beyond the general path.
                    auto plain = [](int e) { return (e ^ (e >> 31)) == EMU_POISON ? 0 : e; };
                    const int ea = plain(p.scale_a[(int64_t)ea_ent * MT + arow]) - 14;
                    const int eb = plain(p.scale_b[(int64_t)eb_ent * NT + c0 + (lane % E_W)]);
                    const bool fast = __all_sync(0xffffffffu, ea >= -74 && ea <= 67 && abs(eb) <= 60);
                    const float fa = __uint_as_float((uint32_t)(ea + 127) << 23);
                    const float fb = __uint_as_float((uint32_t)(eb + 127) << 23);
                    if (!warp_wait(smem_u32(&bars->acc_full), pg & 1u, abort_flag)) {
                        ok = false;
                        break;
                    }
                    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll
                    for (int g = 0; g < G; ++g) {
                        uint32_t v[EMU_P][E_C];
                        if (need >> g & 1u) {
#pragma unroll
                            for (int lev = 0; lev < EMU_P; ++lev)
                                tm_ld(lane_addr + (uint32_t)(lev * NT + g * E_C), v[lev]);
                            asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
                        }
                        if (g == G - 1) {  // all levels read: the next period's MMAs may start
                            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                            bar_arrive(smem_u32(&bars->acc_empty));
                        }
                        if (!(need >> g & 1u)) continue;
#pragma unroll
                        for (int c = 0; c < E_C; ++c) {
                            const int x = g * E_C + c;
                            const uint32_t lv[EMU_P] = {v[0][c], v[1][c], v[2][c], v[3][c],
                                                        v[4][c], v[5][c], v[6][c], v[7][c]};
                            float x0, x1, x2, r1, r2, r3;
                            emu_compress(lv, x0, x1, x2);
                            float sc = fa * __shfl_sync(0xffffffffu, fb, x);
                            if (!fast) {
                                const float3 f = mul_pow2(make_float3(x0, x1, x2),
                                                          ea + __shfl_sync(0xffffffffu, eb, x));
                                x0 = f.x;
                                x1 = f.y;
                                x2 = f.z;
                                sc = 1.0f;
                            }
                            h[x] = two_sum(h[x], x0, sc, r1);
                            m[x] = two_sum(m[x], x1, sc, r2);
                            m[x] = two_sum(m[x], r1, 1.0f, r3);
                            l[x] = fmaf(x2, sc, l[x]) + (r2 + r3);
                        }
                    }
                }
            }
            if (!ok) break;
            auto v = [&](int x) {
                return (f32_to_f64(h[x]) + f32_to_f64(m[x])) + f32_to_f64(l[x]);
            };
            static_assert(E_W == 16, "four column ranges");
            switch (warp >> 2) {
            case 0: write_rows<NB, 0, E_W>(p.C, p.c_stride, p.alpha, p.beta, cid, arow, v); break;
            case 1: write_rows<NB, 16, E_W>(p.C, p.c_stride, p.alpha, p.beta, cid, arow, v); break;
            case 2: write_rows<NB, 32, E_W>(p.C, p.c_stride, p.alpha, p.beta, cid, arow, v); break;
            default: write_rows<NB, 48, E_W>(p.C, p.c_stride, p.alpha, p.beta, cid, arow, v); break;
            }
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (t == 0 && *abort_flag) atomicOr(p.flag, 16);
    if (warp == EW_MMA) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem),
                     "r"(E_TMEM_COLS));
    }
}

// The tile kernel of the split-BF16 product (included by bsmm_split.cu).
//
// Warp roles (12 warps, one CTA per SM):
//   warps 0-7   drain: every DRAIN chunks they read the FP32 accumulator (warp w: TMEM lane
//               quarter w % 4, columns 32 * (w / 4) ..) into double-float (hi, lo) sums in
//               registers, release the accumulator, and write C after a tile's last period;
//   warps 8, 9  producers of the A and of the B pieces: a chunk is up to three consecutive K
//               steps of a tile; its pieces (main step: two A and two B main pieces; tail step:
//               one A and one B tail piece; 18 KB either way) go into the step's slot of a
//               free stage with TMA bulk copies that complete on the stage's "full" barrier.
//               Lane 0 of warp 8 also takes the launch's tiles from a global counter and queues
//               them for the other warps (TileFeed);
//   warps 10, 11  MMA: each takes every second drain period; one elected lane issues the MMAs
//               of a chunk (6 split products per K step) into one of NACC TMEM accumulators
//               (one per drain period, in rotation) and commits them to the stage's "empty"
//               barrier, and at the end of a drain period to the accumulator's "full" barrier.
// The stages form one ring per MMA warp, each with a running chunk counter across all tiles of
// the CTA (one warp alone waits on a stage, phase after phase); the chunks of two consecutive
// periods of a tile are sent in turns.  Accumulators rotate over one running period counter;
// every wait computes its parity from those counters.
//
// What bounds it, on the 4096-atom SZP cell's U.X kept on P_L (25.7 M K steps of 169 K per
// SM, 18 KB each): the issue of copies and MMAs, then shared memory (the operands of an MMA
// of N = 64 take 48 clocks at 128 B per clock, a K step 150 ns).
//  * A bulk copy costs its issuing thread 70-126 clocks whatever its size when its operands sit
//    in per-lane registers, much less when they are warp-uniform (entries and tile records
//    broadcast by shuffles, one elected lane).  Two producer warps share a chunk, and the two
//    pieces of a step that are neighbours in memory move in one copy.  Chunks of one or two K
//    steps cost more waits and barriers than they save (307 and 185 ns per step against 181).
//  * tcgen05.mma (N = 64) issues at 68 clocks from a single-lane branch with descriptors in
//    ordinary registers, at 58 from warp-uniform code with an elected lane, and a chunk's
//    waits and commits add 140 during which nothing is issued: two warps on different
//    accumulators cover each other.
//  * With tiles dealt round-robin the CTAs drifted apart until the tiles in flight spanned
//    ten M groups: 345 GB of DRAM reads, 7.2 TB/s.  The queue keeps them neighbours, and the
//    B pieces (read once per tile) are evicted first, so the A pieces of one or two M groups
//    (9 MB each) stay in L2.  Pairing periods across tiles, which needs tiles taken further
//    ahead, cost more than it gave (L.S on 1728 atoms: 343 ns per step against 289).
// Measured on that product, ns per K step and SM: 316 with two producers (360 with one), 282
// with warp-uniform MMA issue, 253 with the eviction policies, 204 with the queue, 188 with two
// MMA warps, 181 with warp-uniform copies (30.5 ms; 60.8 at first).  S.X on 512 atoms 214 -> 201 by
// the last two; L.S on 1728 atoms, 36 steps a tile, 272 -> 289 (its odd third period is alone).
//
// Every wait is bounded (about two seconds) and also ends when another role has given up:
// the CTA then stops issuing work, retires its own copies and MMAs (bounded), frees its
// tensor memory and returns with bit 16 of the context flag set.
constexpr int NS = 4;                  // shared-memory stages, NR of each MMA warp
constexpr int N_DRAIN = 256;           // drain threads
constexpr int NPROD = 2;               // producer warps
constexpr int NMMA = 2;                // MMA warps
constexpr int W_PROD = 8, W_MMA = W_PROD + NPROD;  // first producer and MMA warp (0-7 drain)
constexpr int ST = 32 * (W_MMA + NMMA);            // threads per CTA (12 warps)
constexpr int NTQ = 4;                 // slots of the tile queue
constexpr int TILE_READERS = NPROD + NMMA + N_DRAIN / 32;  // warps that read each queued tile
constexpr int PERIOD = KSTEPS * DRAIN; // K steps of a drain period
constexpr int NR = NS / NMMA;

// A queued tile: its index, first K step, K steps and main K steps (tile < 0: no more tiles)
struct TileRec {
    int64_t s0;
    int32_t tile, nks, nm;
};

struct Bars {
    uint64_t full[NS], empty[NS], acc_full[NACC], acc_empty[NACC], done[NMMA];
    static constexpr int TQ = NTQ;
    uint64_t tile_full[TQ], tile_empty[TQ];
    TileRec rec[TQ];
    uint64_t never;  // no thread ever arrives here: the test-only wait on it must run out
    uint32_t tmem_slot;
    int abort_flag;
};
static_assert(sizeof(Bars) <= BAR_BYTES, "barrier block");
static_assert(NS * STAGE + BAR_BYTES <= 227 * 1024, "shared memory per CTA");

__device__ __forceinline__ bool bar_try(uint32_t addr, uint32_t parity)
{
    uint32_t done;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}\n"
        : "=r"(done)
        : "r"(addr), "r"(parity)
        : "memory");
    return done != 0;
}

__device__ __forceinline__ void bar_arrive(uint32_t addr)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(addr) : "memory");
}

// Bounded wait on an mbarrier phase; gives up when another role has set the abort flag.
__device__ __forceinline__ bool bar_wait(uint32_t addr, uint32_t parity, volatile int *abort_flag)
{
    if (bar_try(addr, parity)) return true;
    const long long t0 = clock64();
    while (!bar_try(addr, parity)) {
        if (*abort_flag) return false;
        if (clock64() - t0 > WAIT_CYCLES) {
            *abort_flag = 1;
            return false;
        }
    }
    return true;
}

// bar_wait by a whole warp: its lanes go on together or give up together
__device__ __forceinline__ bool warp_wait(uint32_t addr, uint32_t parity, volatile int *abort_flag)
{
    return __all_sync(0xffffffffu, bar_wait(addr, parity, abort_flag));
}

// bar_wait by lane 0 alone, its outcome for the whole warp
__device__ __forceinline__ bool warp_wait_lane0(bool need, uint32_t addr, uint32_t parity,
                                                volatile int *abort_flag, int lane)
{
    int go = 1;
    if (need && lane == 0) go = bar_wait(addr, parity, abort_flag);
    return __shfl_sync(0xffffffffu, go, 0) != 0;
}

// The n-th tile of this CTA from the queue, read by a whole warp (tile -1: none, or given up)
template <class B>
__device__ __forceinline__ TileRec next_tile(B *bars, uint32_t n, volatile int *abort_flag, int lane)
{
    TileRec r;
    r.tile = -1;
    r.s0 = 0;
    r.nks = r.nm = 0;
    if (warp_wait(smem_u32(&bars->tile_full[n % B::TQ]), (n / B::TQ) & 1u, abort_flag)) {
        // broadcast, so that what follows from it is warp-uniform
        const TileRec q = bars->rec[n % B::TQ];
        r.tile = __shfl_sync(0xffffffffu, q.tile, 0);
        r.nks = __shfl_sync(0xffffffffu, q.nks, 0);
        r.nm = __shfl_sync(0xffffffffu, q.nm, 0);
        r.s0 = __shfl_sync(0xffffffffu, q.s0, 0);
        if (lane == 0) bar_arrive(smem_u32(&bars->tile_empty[n % B::TQ]));
    }
    return r;
}

// Bounded wait with its own limit in cycles (the test-only short wait).
__device__ __forceinline__ bool bar_wait_for(uint32_t addr, uint32_t parity,
                                             volatile int *abort_flag, long long limit)
{
    const long long t0 = clock64();
    while (!bar_try(addr, parity)) {
        if (*abort_flag) return false;
        if (clock64() - t0 > limit) {
            *abort_flag = 1;
            return false;
        }
    }
    return true;
}

// Bounded wait that ignores the abort flag (retiring work already issued).
__device__ __forceinline__ bool bar_wait_plain(uint32_t addr, uint32_t parity)
{
    const long long t0 = clock64();
    while (!bar_try(addr, parity))
        if (clock64() - t0 > WAIT_CYCLES) return false;
    return true;
}

__device__ __forceinline__ bool elect_one()
{
    uint32_t p;
    asm volatile("{\n\t.reg .pred q;\n\telect.sync _|q, 0xffffffff;\n\tselp.u32 %0, 1, 0, q;\n\t}\n" : "=r"(p));
    return p != 0;
}

__device__ __forceinline__ void bar_commit(uint32_t addr)
{
    asm volatile(
        "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(addr)
        : "memory");
}

// TMA bulk copy global -> shared completing `bytes` of transaction count on mbarrier bar
__device__ __forceinline__ void bulk_copy(uint32_t dst, const void *src, uint32_t bytes,
                                          uint32_t bar)
{
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
            dst),
        "l"(src), "r"(bytes), "r"(bar)
        : "memory");
}

// The same with an L2 eviction policy
__device__ __forceinline__ void bulk_copy(uint32_t dst, const void *src, uint32_t bytes,
                                          uint32_t bar, uint64_t policy)
{
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], "
        "[%1], %2, [%3], %4;" ::"r"(dst),
        "l"(src), "r"(bytes), "r"(bar), "l"(policy)
        : "memory");
}

__device__ __forceinline__ uint64_t l2_evict_first()
{
    uint64_t p;
    asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(p));
    return p;
}

__device__ __forceinline__ uint64_t l2_evict_last()
{
    uint64_t p;
    asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(p));
    return p;
}

// Writes one row's columns of a block, values w[b] for b in [B0, B1) (b a column of the
// block), at dst = the row's first column: 16-byte stores where two neighbours share one.
// odd: whether dst is an odd multiple of eight bytes.
template <int NB, int B0, int B1>
__device__ __forceinline__ void put_row(double *dst, bool odd, const double (&w)[NB])
{
    constexpr int N = B1 - B0;
    if constexpr (N <= 0) return;
    const bool s = odd != (bool)(B0 & 1);  // a single value comes first
#pragma unroll
    for (int t = 0; t < (N - 1) / 2; ++t) {
        const int b = B0 + 2 * t;
        *reinterpret_cast<double2 *>(dst + b + s) =
            make_double2(s ? w[b + 1] : w[b], s ? w[b + 2] : w[b + 1]);
    }
    if constexpr (N & 1) {
        dst[s ? B0 : B1 - 1] = s ? w[B0] : w[B1 - 1];
    } else if (!s) {
        *reinterpret_cast<double2 *>(dst + B1 - 2) = make_double2(w[B1 - 2], w[B1 - 1]);
    } else {
        dst[B0] = w[B0];
        dst[B1 - 1] = w[B1 - 1];
    }
}

// Epilogue of one drain thread: accumulator row arow = (atom of M slot si, orbital a),
// columns H0 .. H0 + W - 1 = (atom of N slot, orbital); cid[u] is the P_C block of slot pair
// (si, H0 / NB + u) or -1; each present block gets beta*C + alpha*v(column).  The plain case
// (alpha 1, beta 0, C on a 16-byte boundary) costs one FP64 addition per value and stores 16
// bytes at a time; the general one is bound by its four FP64-pipe operations per value.
template <int NB, int W> __host__ __device__ constexpr int epi_slots()
{
    return NB ? (W + NB - 2) / NB + 1 : 1;
}

template <int NB, int H0, int W, class V>
__device__ __forceinline__ void write_rows(double *C, int c_stride, double alpha, double beta,
                                           const int32_t (&cid)[epi_slots<NB, W>()], int arow, V v)
{
    constexpr int GI = MT / NB, GJ = NT / NB;
    constexpr int J0 = H0 / NB, J1 = (H0 + W - 1) / NB;
    if (arow >= GI * NB) return;
    const int a = arow % NB;
    const bool plain = alpha == 1.0 && beta == 0.0 && (reinterpret_cast<uintptr_t>(C) & 15) == 0;
    const bool odd = (a * NB) & 1;
    auto block = [&](auto jc) {
        constexpr int jl = J0 + decltype(jc)::value;
        if constexpr (jl <= J1 && jl < GJ) {
            const int32_t blk = cid[jl - J0];
            if (blk < 0) return;
            constexpr int B0 = jl * NB < H0 ? H0 - jl * NB : 0;
            constexpr int B1 = (jl + 1) * NB > H0 + W ? H0 + W - jl * NB : NB;
            double *dst = C + (int64_t)blk * c_stride + a * NB;
            double w[NB];
#pragma unroll
            for (int b = B0; b < B1; ++b) w[b] = v(jl * NB + b - H0);
            if (plain) {
                put_row<NB, B0, B1>(dst, odd, w);
            } else {
#pragma unroll
                for (int b = B0; b < B1; ++b)
                    dst[b] = beta == 0.0 ? alpha * w[b] : beta * dst[b] + alpha * w[b];
            }
        }
    };
    static_assert(J1 - J0 < 9 && J1 - J0 < epi_slots<NB, W>(), "slots of a thread's columns");
    block(std::integral_constant<int, 0>());
    block(std::integral_constant<int, 1>());
    block(std::integral_constant<int, 2>());
    block(std::integral_constant<int, 3>());
    block(std::integral_constant<int, 4>());
    block(std::integral_constant<int, 5>());
    block(std::integral_constant<int, 6>());
    block(std::integral_constant<int, 7>());
    block(std::integral_constant<int, 8>());
}

// The six split products of one K step into the accumulator at acc_addr: a, b are the low
// words of the step's plane-0 descriptors, PA and PB the plane strides in 16-byte units; acc
// = 0 overwrites the accumulator.
template <int PA, int PB>
__device__ __forceinline__ void mma_step(uint32_t acc_addr, uint32_t a, uint32_t b, uint32_t acc)
{
    constexpr int pq[6][2] = {{0, 0}, {0, 1}, {1, 0}, {0, 2}, {1, 1}, {2, 0}};
    constexpr uint32_t hi = (uint32_t)(128 >> 4) | (1u << 14);  // piece_desc's high word
#pragma unroll
    for (int x = 0; x < 6; ++x)
        asm volatile(
            "{\n\t.reg .pred p;\n\t.reg .b64 da, db;\n\tsetp.ne.b32 p, %4, 0;\n\t"
            "mov.b64 da, {%1, %5};\n\tmov.b64 db, {%2, %5};\n\t"
            "tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %3, p;\n\t}\n" ::"r"(acc_addr),
            "r"(a + pq[x][0] * PA), "r"(b + pq[x][1] * PB), "r"(IDESC), "r"(x == 0 ? acc : 1u), "r"(hi));
}

// The chunks of a pair of drain periods that starts at K step `base` of a tile of nks: n0 of the
// first period, n1 of the second (0: none).  They go through the stages in turns -- chunk j of
// the first, chunk j of the second -- as long as the second has any.
struct PairChunks {
    int n0, n1;
    __device__ __forceinline__ PairChunks(int nks, int base)
        : n0((min(PERIOD, nks - base) + KSTEPS - 1) / KSTEPS),
          n1((max(0, min(PERIOD, nks - base - PERIOD)) + KSTEPS - 1) / KSTEPS)
    {
    }
};

// Hands out the launch's tiles in order from a global counter, so that the tiles in flight on the
// GPU stay neighbours (they share the A pieces of one or two M groups) and no CTA idles while
// others hold several tiles.  Lane 0 of the A producer runs it between tiles; a record is fetched
// one tile before it is queued, so its latency is not seen.  Queueing record n + 1 waits until
// all warps have read record n + 1 - NTQ, whose predecessors' chunks are all sent by then.
struct TileFeed {
    TileRec rec;   // the next record to queue
    uint32_t n;    // records queued
    bool open;

    __device__ __forceinline__ void load(const SplitArgs &p, int i)
    {
        rec.tile = -1;
        rec.s0 = 0;
        rec.nks = rec.nm = 0;
        if (i < p.n_tiles) {
            rec.tile = i;
            rec.s0 = p.kstart[i];
            rec.nks = (int)(p.kstart[i + 1] - rec.s0);
            rec.nm = p.nmain[i];
        }
    }
    __device__ __forceinline__ int take(const SplitArgs &p)
    {
        return (int)gridDim.x + (int)atomicAdd(&p.counter[0], 1u);
    }
    // queues the CTA's first two records
    __device__ __forceinline__ void start(const SplitArgs &p, Bars *bars, volatile int *abort_flag)
    {
        n = 0;
        open = true;
        load(p, blockIdx.x);
        post(p, bars, abort_flag);
        post(p, bars, abort_flag);
    }
    // queues the next record and fetches the one after
    __device__ __forceinline__ void post(const SplitArgs &p, Bars *bars, volatile int *abort_flag)
    {
        if (!open) return;
        if (n >= (uint32_t)NTQ &&
            !bar_wait(smem_u32(&bars->tile_empty[n % NTQ]), ((n / NTQ) + 1) & 1u, abort_flag)) {
            open = false;
            return;
        }
        bars->rec[n % NTQ] = rec;
        bar_arrive(smem_u32(&bars->tile_full[n % NTQ]));
        ++n;
        open = rec.tile >= 0;
        if (!open) return;
        load(p, take(p));
    }
    // the last CTA to finish handing out resets the counters for the next launch
    __device__ __forceinline__ void close(const SplitArgs &p)
    {
        __threadfence();
        if (atomicInc(&p.counter[1], gridDim.x - 1) == gridDim.x - 1) atomicExch(&p.counter[0], 0u);
    }
};

// One producer warp (SIDE 0: A pieces, 1: B pieces) over all chunks of the CTA's tiles.
template <int SIDE>
__device__ __forceinline__ void produce(const SplitArgs &p, uint32_t sm0, Bars *bars,
                                        volatile int *abort_flag, int lane)
{
    constexpr int MAIN = SIDE ? B_MAIN : A_MAIN, TAIL = SIDE ? B_TAIL : A_TAIL;
    constexpr int SLOT = SIDE ? B_SLOT : A_SLOT;
    const uint8_t *mains = SIDE ? p.b_main : p.a_main - p.am0 * A_MAIN;
    const uint8_t *tails = SIDE ? p.b_tail : p.a_tail - p.at0 * A_TAIL;
    const uint32_t dst0 = sm0 + (SIDE ? B_SLOTS : 0);
    static_assert(TAIL == 2 * MAIN, "a tail piece fills a step's slot like two main pieces");
    const bool el = elect_one();
    // K steps come a pair of periods at a time, one per lane, loaded one pair ahead (the next
    // tile's first pair during this tile's last)
    constexpr int PB = 2 * PERIOD;
    static_assert(PB <= 32, "a lane per K step of a pair of periods");
    auto load = [&](const TileRec &t, int base) {
        return lane < PB && base + lane < t.nks
                   ? __ldg(reinterpret_cast<const int2 *>(p.steps + t.s0 + base + lane) + SIDE)
                   : make_int2(0, 0);
    };
    const uint64_t policy = SIDE ? l2_evict_first() : l2_evict_last();
    uint32_t cm[NMMA] = {0, 0};  // running chunk counters of the MMA warps
    uint32_t pg0 = 0;            // running period counter
    bool ok = true;
    TileFeed feed;
    if (SIDE == 0 && lane == 0) feed.start(p, bars, abort_flag);
    __syncwarp();
    TileRec t = next_tile(bars, 0, abort_flag, lane);
    int2 cur = load(t, 0);
    for (uint32_t n = 1; t.tile >= 0 && ok; ++n) {
        TileRec tn = t;
        for (int base = 0; base == 0 || base < t.nks; base += PB) {
            int2 nxt;
            if (base + PB < t.nks) {
                nxt = load(t, base + PB);
            } else {
                tn = next_tile(bars, n, abort_flag, lane);
                if (SIDE == 0 && lane == 0) feed.post(p, bars, abort_flag);
                __syncwarp();
                nxt = load(tn, 0);
            }
            const PairChunks pc(t.nks, base);
            for (int c = 0; c < pc.n0 + pc.n1; ++c) {
                // chunks in turns while the second period has any, then the first's rest
                const int second = c < 2 * pc.n1 ? c & 1 : 0, j = c < 2 * pc.n1 ? c >> 1 : c - pc.n1;
                const int q0 = base + second * PERIOD + j * KSTEPS;
                const uint32_t m = (pg0 + second) & 1u, k = m ? cm[1] : cm[0];
                const uint32_t s = NMMA * (k % NR) + m, fb = smem_u32(&bars->full[s]);
                // broadcast entries, so that the copies' operands are warp-uniform
                int ex[KSTEPS], ey[KSTEPS];
#pragma unroll
                for (int ks = 0; ks < KSTEPS; ++ks) {
                    ex[ks] = __shfl_sync(0xffffffffu, cur.x, q0 - base + ks);
                    ey[ks] = __shfl_sync(0xffffffffu, cur.y, q0 - base + ks);
                }
                if (k >= (uint32_t)NR &&
                    !warp_wait(smem_u32(&bars->empty[s]), ((k / NR) + 1) & 1u, abort_flag)) {
                    ok = false;
                    break;
                }
                const int nk = min(KSTEPS, t.nks - q0);
                if (el) {
                    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(fb),
                                 "r"((uint32_t)(nk * SLOT))
                                 : "memory");
#pragma unroll
                    for (int ks = 0; ks < KSTEPS; ++ks) {
                        if (ks >= nk) break;
                        const uint32_t dst = dst0 + s * STAGE + ks * SLOT;
                        if (q0 + ks >= t.nm) {
                            bulk_copy(dst, tails + (int64_t)ex[ks] * TAIL, TAIL, fb, policy);
                        } else if (ey[ks] == ex[ks] + 1) {
                            bulk_copy(dst, mains + (int64_t)ex[ks] * MAIN, 2 * MAIN, fb, policy);
                        } else {
                            bulk_copy(dst, mains + (int64_t)ex[ks] * MAIN, MAIN, fb, policy);
                            bulk_copy(dst + MAIN, ey[ks] < 0 ? p.zero : mains + (int64_t)ey[ks] * MAIN,
                                      MAIN, fb, policy);
                        }
                    }
                }
                __syncwarp();
                cm[0] += 1 - m;
                cm[1] += m;
            }
            if (!ok) break;
            pg0 += (pc.n0 > 0) + (pc.n1 > 0);  // (a tile without K steps has no period)
            cur = nxt;
        }
        t = tn;
    }
    // every copy lands before the CTA's shared memory is released.  A stage's barrier needs both
    // sides.  They arm the same chunks unless the CTA is giving up: then one side may have found a
    // stage busy and left, and the other finds it free and arms it.  Its wait below runs out after
    // two seconds (the flag is set already), and its own copies have long landed by then.
    if (lane == 0)
        for (uint32_t m = 0; m < NMMA; ++m)
            for (uint32_t k = 0; k < (uint32_t)NR && k < cm[m]; ++k) {
                const uint32_t c = cm[m] - 1 - k;
                if (!bar_wait_plain(smem_u32(&bars->full[NMMA * (c % NR) + m]), (c / NR) & 1u))
                    *abort_flag = 1;
            }
    if (SIDE == 0 && lane == 0) feed.close(p);
    __syncwarp();
}

// NB = 0: mixed basis (groups, rows and columns through the tables of bsmm_mixed.cuh)
template <int NB>
__global__ void __launch_bounds__(ST, 1) k_bsmm_split(const SplitArgs p)
{
    constexpr int GI = NB ? MT / NB : GI_MIX, GJ = NB ? NT / NB : GJ_MIX;
    extern __shared__ __align__(1024) uint8_t smem[];
    Bars *bars = reinterpret_cast<Bars *>(smem + NS * STAGE);
    volatile int *abort_flag = &bars->abort_flag;
    const int t = threadIdx.x, warp = __shfl_sync(0xffffffffu, t >> 5, 0), lane = t & 31;
    const uint32_t sm0 = smem_u32(smem);

    if (t == 0) {
        for (int s = 0; s < NS; ++s) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(&bars->full[s])),
                         "r"(NPROD));
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(&bars->empty[s])),
                         "r"(1));
        }
        for (int b = 0; b < NACC; ++b) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(
                             smem_u32(&bars->acc_full[b])),
                         "r"(1));
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(
                             smem_u32(&bars->acc_empty[b])),
                         "r"(N_DRAIN));
        }
        for (int r = 0; r < NTQ; ++r) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(&bars->tile_full[r])),
                         "r"(1));
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(&bars->tile_empty[r])),
                         "r"(TILE_READERS));
        }
        for (int m = 0; m < NMMA; ++m)
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(&bars->done[m])),
                         "r"(1));
        asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(&bars->never)), "r"(1));
        bars->abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == W_MMA) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                         smem_u32(&bars->tmem_slot)),
                     "r"(TMEM_COLS));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = bars->tmem_slot;

    if (warp == W_PROD || warp == W_PROD + 1) {
        // ------------------------------------------------------------ producers
        // warp W_PROD copies the A pieces of every chunk, the next warp the B pieces (one elected
        // lane issues them).  The two main pieces of a step are neighbours in memory when no atom
        // of the group's list lies between the two, and then one copy moves both.
        if (warp == W_PROD)
            produce<0>(p, sm0, bars, abort_flag, lane);
        else
            produce<1>(p, sm0, bars, abort_flag, lane);
    } else if (warp >= W_MMA) {
        // ------------------------------------------------------------ MMA issue
        // MMA warp m takes the periods of parity m.  The whole warp walks the
        // chunks (uniform control flow keeps the descriptors in uniform registers: 58 clocks
        // per MMA against 68 from a single-lane branch); one elected lane issues.
        const int m = warp - W_MMA;
        const bool el = elect_one();
        uint32_t cm = 0, pg0 = 0;  // chunks consumed, first period of the current pair
        bool ok = true, issued = false;
        // test mode: the first wait is on a barrier nothing completes, with a short limit,
        // so it runs out; the CTA then takes the same abort path as a real timeout
        if (p.test_wait_cycles > 0) {
            bar_wait_for(smem_u32(&bars->never), 0u, abort_flag, p.test_wait_cycles);
            ok = false;
        }
        // low words of the descriptors of slot 0 of stage 0 for both kinds of K step (main:
        // the second column is the second atom's piece, A_MAIN / B_MAIN further; tail: the
        // piece's second column); a stage, slot or plane only moves the 14-bit start address
        // field (shared addresses stay below 256 KB, so no carry leaves it)
        const uint32_t dam = (uint32_t)piece_desc(sm0, A_MAIN);
        const uint32_t dat = (uint32_t)piece_desc(sm0, COLB_A);
        const uint32_t dbm = (uint32_t)piece_desc(sm0 + B_SLOTS, B_MAIN);
        const uint32_t dbt = (uint32_t)piece_desc(sm0 + B_SLOTS, COLB_B);
        const uint32_t bar0 = smem_u32(bars);
        for (uint32_t n = 0; ok; ++n) {
            const TileRec tr = next_tile(bars, n, abort_flag, lane);
            if (tr.tile < 0) break;
            const int nks = tr.nks, nm = tr.nm;
            for (int base = 0; base < nks && ok; base += 2 * PERIOD) {
                const PairChunks pc(nks, base);
                const int second = (m ^ pg0) & 1, nc = second ? pc.n1 : pc.n0;
                const uint32_t pg = pg0 + second, b = pg % NACC;
                const uint32_t acc_addr = tmem + b * NT;
                for (int j = 0; j < nc; ++j, ++cm) {
                    if (j == 0 && pg >= (uint32_t)NACC &&
                        !warp_wait(bar0 + (uint32_t)offsetof(Bars, acc_empty) + 8 * b,
                                   ((pg / NACC) + 1) & 1u, abort_flag)) {
                        ok = false;
                        break;
                    }
                    const uint32_t s = NMMA * (cm % NR) + m;
                    const int q0 = base + second * PERIOD + j * KSTEPS;
                    if (!warp_wait(bar0 + (uint32_t)offsetof(Bars, full) + 8 * s, (cm / NR) & 1u,
                                   abort_flag)) {
                        ok = false;
                        break;
                    }
                    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                    if (el) {
#pragma unroll
                        for (int ks = 0; ks < KSTEPS; ++ks) {
                            if (q0 + ks >= nks) break;
                            const uint32_t oa = s * (STAGE >> 4) + ks * (A_SLOT >> 4);
                            const uint32_t ob = s * (STAGE >> 4) + ks * (B_SLOT >> 4);
                            const uint32_t acc = j == 0 && ks == 0 ? 0u : 1u;
                            // plane strides in 16-byte units: main pieces hold one column per
                            // plane, tail pieces two
                            if (q0 + ks < nm)
                                mma_step<COLB_A / 16, COLB_B / 16>(acc_addr, dam + oa, dbm + ob, acc);
                            else
                                mma_step<2 * COLB_A / 16, 2 * COLB_B / 16>(acc_addr, dat + oa,
                                                                           dbt + ob, acc);
                        }
                        bar_commit(bar0 + (uint32_t)offsetof(Bars, empty) + 8 * s);
                        if (j == nc - 1)
                            bar_commit(bar0 + (uint32_t)offsetof(Bars, acc_full) + 8 * b);
                    }
                    __syncwarp();
                    issued = true;
                }
                pg0 += pc.n1 ? 2 : 1;
            }
        }
        // retire every MMA before the tensor memory is released
        if (issued && el) {
            bar_commit(smem_u32(&bars->done[m]));
            if (!bar_wait_plain(smem_u32(&bars->done[m]), 0u)) *abort_flag = 1;
        }
        __syncwarp();
    } else {
        // ------------------------------------------------------------ drain and epilogue
        const int quarter = warp & 3, half = warp >> 2;
        const int arow = quarter * 32 + lane;
        const uint32_t lane_addr = tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(half * 32);
        uint32_t pg = 0;
        bool ok = true;
        for (uint32_t n = 0; ok; ++n) {
            const TileRec tr = next_tile(bars, n, abort_flag, lane);
            if (tr.tile < 0) break;
            const int tile = tr.tile;
            const int np = (tr.nks + PERIOD - 1) / PERIOD;
            // this row's C blocks, loaded now and used after the tile's last period
            constexpr int NJ = epi_slots<NB, 32>();
            int32_t cid[NJ];
            if constexpr (NB > 0) {
                const int si = arow / NB, j0 = (half * 32) / NB;
#pragma unroll
                for (int u = 0; u < NJ; ++u)
                    cid[u] = (arow < GI * NB && j0 + u < GJ)
                                 ? __ldg(&p.cidx[((int64_t)tile * GI + si) * GJ + j0 + u])
                                 : -1;
            }
            float hi[32], lo[32];
#pragma unroll
            for (int x = 0; x < 32; ++x) hi[x] = lo[x] = 0.f;
            for (int d = 0; d < np; ++d, ++pg) {
                const uint32_t b = pg % NACC;
                if (!warp_wait(smem_u32(&bars->acc_full[b]), (pg / NACC) & 1u, abort_flag)) {
                    ok = false;
                    break;
                }
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll
                for (int q = 0; q < 2; ++q) {
                    uint32_t v[16];
                    asm volatile(
                        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,"
                        "%10,%11,%12,%13,%14,%15}, [%16];"
                        : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]),
                          "=r"(v[6]), "=r"(v[7]), "=r"(v[8]), "=r"(v[9]), "=r"(v[10]),
                          "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
                        : "r"(lane_addr + b * NT + q * 16));
                    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
                    for (int x = 0; x < 16; ++x)
                        two_sum_add(hi[q * 16 + x], lo[q * 16 + x], __uint_as_float(v[x]));
                }
                asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                bar_arrive(smem_u32(&bars->acc_empty[b]));
            }
            if (!ok) break;
            if constexpr (NB > 0) {
                auto v = [&](int x) { return f32_to_f64(hi[x]) + f32_to_f64(lo[x]); };
                if (half == 0)
                    write_rows<NB, 0, 32>(p.C, p.c_stride, p.alpha, p.beta, cid, arow, v);
                else
                    write_rows<NB, 32, 32>(p.C, p.c_stride, p.alpha, p.beta, cid, arow, v);
            } else {
                write_rows_mixed(p, tile, arow, half, hi, lo);
            }
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (t == 0 && *abort_flag) atomicOr(p.flag, 16);
    if (warp == W_MMA) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem),
                     "r"(TMEM_COLS));
    }
}

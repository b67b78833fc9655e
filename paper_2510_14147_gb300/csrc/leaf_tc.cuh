// leaf_tc.cuh -- the tensor-core leaf stage (precision 1), included by
// query.cu inside its namespaces: k_filter_tc finds the (query, point) pairs
// that may be edges, k_pairs decides them and writes the edges.
//
// Filter: per work item, the group's 32 queries (B, N = 32) against 128-row
// tiles of packed candidate points (A, M = 128), both as fp16 rows prepared
// once per query, multiplied by tcgen05 MMAs (K = 16 per instruction) into a
// 128 x 32 fp32 accumulator in tensor memory.  The accumulator, the rows'
// squared norms and a rigorous bound on the fp16 and fp32 rounding keep every
// edge; kept pairs go to a list.
// Decision: the canonical fp32 direct-difference sum of the original rows
// (decide32), the pinned FP64 sum where that cannot decide.
//
// The two used to be one kernel (two CTAs of 8 warps per SM, each tile
// filtered, barrier, rechecked, barrier): every kept pair cost about 60 SM
// clocks, because a tile's rechecks were a chain of round trips to memory with
// 16 warps to hide it, and a tile without any cost 2500.  As two kernels each
// has its own bound: the filter the 16-byte copies of its operands and the
// issue slots of its epilogue, the decisions the L1 reads of both rows.
// Count stage, 1M x 128 at 70 / 500 neighbours: 27.5 / 78.0 -> 10.8 / 28.7 ms;
// two-pass count + emit of 20 clouds (3 to 64 floats per row): 35.8 -> 10.3 ms.

constexpr int TC_ROWS = 128;
constexpr int TC_NB = kItemTC;            // candidate blocks of one item
constexpr uint32_t TC_HINT = 1u << 16;    // ns a suspended poll may sleep (woken by the phase)
constexpr uint32_t TC_SLEEPS = 1u << 14;  // suspended polls before a wait gives up (about a second)

constexpr int FT_STAGES = 5;   // tiles in flight (operand buffer, accumulator, row map)
constexpr int FT_ITEMS = 3;    // items in flight, one scout warp each
constexpr int FT_CHUNK = 1024; // pair-list entries an epilogue warp reserves at a time (>= 32 x 32)
// warps: 0-7 two producer groups, 8-10 scouts, 11-15 MMA issue (one per stage), 16-27 three epilogue groups
constexpr int FT_PGROUPS = 2, FT_EGROUPS = 3;
constexpr int FT_SCOUT = 4 * FT_PGROUPS, FT_MMA = FT_SCOUT + FT_ITEMS, FT_EPI = FT_MMA + FT_STAGES;
constexpr int FT_EWARPS = 4 * FT_EGROUPS, FT_T = 32 * (FT_EPI + FT_EWARPS);
static_assert(FT_EPI % 4 == 0, "an epilogue warp reads the tensor-memory lanes of its index mod 4");

struct FtItem {
    int ntiles;   // -1: no more items in this buffer
    int T, qfirst, nqr, qb, qe, cloud, rbase;
};
struct __align__(1024) FtShared {
    unsigned char A[FT_STAGES][2][TC_ROWS * 128];  // fp16 candidate rows: K half (64 halves), 128-byte swizzle
    unsigned char B[FT_ITEMS][2][32 * 128];        // fp16 query rows, the same layout
    float pn[FT_STAGES][TC_ROWS];                  // squared norms of a tile's rows
    int pos[FT_STAGES][TC_ROWS];                   // their tree positions
    int bbeg[FT_ITEMS][TC_NB], bpre[FT_ITEMS][TC_NB];  // an item's blocks: first position, row prefix
    int bco[FT_ITEMS][32];                             // the prefix of every 32nd block (a row of its own: no bank conflicts)
    float4 qhg[FT_ITEMS][16];                      // filter terms of two queries: (h_q, h_q+1, g_q, g_q+1)
    FtItem item[FT_ITEMS];
    uint64_t full[FT_STAGES], done[FT_STAGES], free_[FT_STAGES];  // rows copied; MMAs complete; epilogue has read
    uint64_t ifull[FT_ITEMS], ifree[FT_ITEMS];                    // item published; item no longer read
    uint32_t tslot;
    int fail;
};
constexpr size_t kFtSmem = sizeof(FtShared) + 1024;
static_assert(kFtSmem <= 227 * 1024, "k_filter_tc: shared memory of one CTA");
static_assert(FT_STAGES * 32 <= 256 && TC_NB == 1024, "accumulator columns; block searches of 32 x 32");

// A bounded wait of a whole warp; false (in every lane) once any wait of the
// CTA has given up.
__device__ __forceinline__ bool ft_wait(FtShared &S, uint64_t *bar, uint32_t parity) {
    bool ok = false;
    for (uint32_t i = 0; i < TC_SLEEPS && !ok; ++i) {
        ok = tc::mbar_wait_sleep(bar, parity, 1, TC_HINT);
        if (!ok && *(volatile int *)&S.fail) break;
    }
    if (!ok) *(volatile int *)&S.fail = 1;
    return __all_sync(0xffffffffu, ok);
}

// Persistent, one CTA of 28 warps per SM; the wave's items are taken
// dynamically.  Roles, connected by mbarriers (no CTA barrier between tiles):
//  scout warp b -- takes an item, lays out its blocks' row prefix, its query
//     rows (MMA layout) and filter terms in item buffer b;
//  producer warps -- two groups of four take alternate tiles: a warp maps 32
//     rows to positions (two ballot searches over the prefix and a popcount of
//     block starts) and copies them with coalesced 16-byte cp.async into the
//     swizzled operand layout, five tiles deep in all; the copies arrive on
//     the tile's mbarrier as they land (a producer that waited for them, to
//     fence before arriving, spent two thirds of its time there);
//  MMA warp m -- waits for a tile of stage m, makes the copies visible to the
//     tensor core and issues its MMA chain (the proxy fence takes about 700
//     clocks whoever executes it, more than a tile: one per stage hides it);
//  epilogue warps -- three groups of four take every third tile: thread = row,
//     32 accumulator columns, packed FMA, add and subtract for two queries and
//     a shift of the sign; kept pairs go to the warp's chunk of the pair list.
// A warp issues one instruction every three or four clocks here, so the roles
// are as wide as their instruction counts ask (about 170 per producer warp
// and tile, 200 per epilogue warp and tile), which bounds the kernel with the
// L2 reads of the rows.
// Every wait is bounded; a wait that gives up ends all roles (CT_ETIMEOUT).
// 290 M candidate rows of 128 floats (2.2 M tiles): 7.5 ms, about 980 clocks a
// tile and SM, of which the epilogue's warps are busy 650 and the producers'
// 800; 292 M rows of 16 floats: 6.3 ms.  (28 warps leave 72 registers a thread;
// -Xptxas -v: 28 bytes of them spilled, 32 read back.)
__global__ void __launch_bounds__(FT_T, 1) k_filter_tc(const __grid_constant__ Views V, Items items,
                                                       ItemWave wave, const uint32_t *__restrict__ cand, PairList out,
                                                       unsigned long long *__restrict__ next,
                                                       int32_t *__restrict__ err) {
    extern __shared__ unsigned char ft_raw[];
    FtShared &S = *reinterpret_cast<FtShared *>(((uintptr_t)ft_raw + 1023) & ~(uintptr_t)1023);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    if (warp == 0) tc::tmem_alloc(&S.tslot, 256);
    if (tid == 0) {
        for (int i = 0; i < FT_STAGES; ++i) {
            tc::mbar_init(&S.full[i], 256);  // per producer thread: its copies, and its other writes
            tc::mbar_init(&S.done[i], 1);
            tc::mbar_init(&S.free_[i], 4);
        }
        for (int i = 0; i < FT_ITEMS; ++i) {
            tc::mbar_init(&S.ifull[i], 32);
            tc::mbar_init(&S.ifree[i], FT_EWARPS + 4 * FT_PGROUPS + FT_STAGES);  // every warp that may not see the last tile
        }
        S.fail = 0;
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    }
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    const uint32_t tmem = S.tslot;
    const int64_t n_items = *items.count;
    constexpr int ST = FT_STAGES;

    if (warp >= FT_SCOUT && warp < FT_SCOUT + FT_ITEMS) {
        // ---- scout of item buffer b
        const int b = warp - FT_SCOUT;
        uint32_t use = 0;  // publications of this buffer
        bool ok = true;
        auto wait_free = [&]() { return use == 0 || ft_wait(S, &S.ifree[b], (use - 1) & 1u); };
        for (; ok;) {
            unsigned long long k = 0;
            if (lane == 0) k = atomicAdd(next, 1ull);
            const int64_t it = wave.item((int64_t)__shfl_sync(0xffffffffu, k, 0));
            if (it >= n_items) {
                if (wait_free()) {
                    if (lane == 0) S.item[b].ntiles = -1;
                    __syncwarp();
                    tc::mbar_arrive(&S.ifull[b]);
                }
                break;
            }
            const int gg = items.group[it];
            const int c = cloud_of_group(V, gg);
            const TreeView &tv = V.tv[c];
            const int g = gg - V.gbase[c];
            const int qb = tv.group_begin[g], qn = tv.group_count[g];
            const int64_t c0 = items.begin[it];
            const int nb = (int)(items.end[it] - c0);  // <= TC_NB
            const int halves = (tv.dp + 63) >> 6, kc = 8 * halves;
            const uint4 *h16 = V.h16[c];
            const float *n16 = V.n16[c];
            for (int q0 = 0; q0 < qn; q0 += 32) {  // groups hold at most 32 queries (loaded trees may not)
                const int nqr = min(32, qn - q0), qfirst = qb + q0;
                if (!wait_free()) {
                    ok = false;
                    break;
                }
                // block table: 32 blocks at a time, the loads of eight such steps
                // together (two round trips to memory for 256 blocks)
                int run = 0;
                for (int j0 = 0; j0 < TC_NB; j0 += 256) {
                    int beg[8], cnt[8];
#pragma unroll
                    for (int u = 0; u < 8; ++u) {
                        const int i = j0 + 32 * u + lane;
                        beg[u] = i < nb ? (int)__ldg(cand + c0 + i) : -1;
                    }
#pragma unroll
                    for (int u = 0; u < 8; ++u) {
                        const int v = beg[u];
                        cnt[u] = v >= 0 ? __ldg(tv.node_count + v) : 0;
                        beg[u] = v >= 0 ? __ldg(tv.node_begin + v) : 0;
                    }
#pragma unroll
                    for (int u = 0; u < 8; ++u) {
                        const int i0 = j0 + 32 * u;
                        int incl = cnt[u];
                        if (i0 < nb) {  // warp-uniform
#pragma unroll
                            for (int o = 1; o < 32; o <<= 1) {
                                const int y = __shfl_up_sync(0xffffffffu, incl, o);
                                if (lane >= o) incl += y;
                            }
                        }
                        S.bbeg[b][i0 + lane] = beg[u];
                        S.bpre[b][i0 + lane] = run + incl - cnt[u];
                        if (lane == 0) S.bco[b][i0 >> 5] = run;
                        if (i0 < nb) run += __shfl_sync(0xffffffffu, incl, 31);
                    }
                }
                // query rows (past the group's queries: its last one again) and filter terms
                for (int i = lane; i < 32 * kc; i += 32) {
                    const int r = i / kc, ch = i - r * kc, h = ch >> 3, j = ch & 7;
                    cp_async16(S.B[b][h] + r * 128 + ((j ^ (r & 7)) << 4),
                               h16 + (size_t)(qfirst + min(r, nqr - 1)) * kc + ch, true);
                }
                cp_async_commit();
                const float qn2 = lane < nqr ? __ldg(n16 + qfirst + lane) : 0.f;
                const float qa = sqrtf(qn2) * H16_NORM_UP;
                const float E = fmaf(H16_REL, qa, V.s16[c][1]) + H16_ABS;
                const float hq = 0.5f * (qn2 - fmaf(E, E, fmaf(H16_ABS2 * qa, qa, 0x1p-60f))) - 0x1p-20f * (E * E);
                float *hg = reinterpret_cast<float *>(&S.qhg[b][lane >> 1]) + (lane & 1);
                hg[0] = hq;
                hg[2] = -H16_REL * E;
                if (lane == 0)
                    S.item[b] = FtItem{(run + TC_ROWS - 1) / TC_ROWS, run, qfirst, nqr, qb, qb + qn, c,
                                       (int)V.rbase[c]};
                cp_async_wait<0>();
                tc::fence_smem_to_async();
                __syncwarp();
                if (run == 0) continue;  // no rows: nothing to publish (every block holds points)
                tc::mbar_arrive(&S.ifull[b]);  // every lane: its own writes and copies
                ++use;
            }
        }
        cp_async_wait<0>();
    } else if (warp < FT_SCOUT) {
        // ---- producers: rows 32 pw .. + 31 of the group's tiles
        const int pg = warp >> 2, pw = warp & 3;
        uint32_t iph = 0;  // next phase parity of each item buffer (bit b)
        uint32_t k = 0;    // tiles so far
        unsigned alive = (1u << FT_ITEMS) - 1u;
        bool ok = true;
        for (int b = 0; alive && ok; b = b + 1 == FT_ITEMS ? 0 : b + 1) {
            if (!((alive >> b) & 1u)) continue;
            if (!ft_wait(S, &S.ifull[b], (iph >> b) & 1u)) break;
            iph ^= 1u << b;
            const FtItem I = S.item[b];
            if (I.ntiles < 0) {
                alive &= ~(1u << b);
                continue;
            }
            const uint4 *h16 = V.h16[I.cloud];
            const float *n16 = V.n16[I.cloud];
            const bool two = V.tv[I.cloud].dp > 64;  // two K halves per row
            const int *bpre = S.bpre[b], *bbeg = S.bbeg[b];
            for (int t = 0; t < I.ntiles; ++t, ++k) {
                if (k % FT_PGROUPS != (uint32_t)pg) continue;
                const int s = k % ST;
                // the block b0 holding the window's first row R0 (the largest with
                // bpre[b0] <= R0) from two 32-wide ballots; blocks b0 + 1 .. b0 + 31
                // start inside the window or after it, and a row's block is b0 plus
                // the number of block starts in (R0, R]
                const int R0 = t * TC_ROWS + 32 * pw;
                int pos = I.qfirst;  // rows past the last one: any row
                if (R0 < I.T) {
                    const unsigned mc = __ballot_sync(0xffffffffu, S.bco[b][lane] <= R0);  // bit 0 set: bco[0] = 0
                    const int cb = 31 - __clz(mc);
                    const unsigned mf = __ballot_sync(0xffffffffu, bpre[32 * cb + lane] <= R0);
                    const int b0 = 32 * cb + 31 - __clz(mf);
                    const int j = b0 + 1 + lane;
                    const int v = j < TC_NB ? bpre[j] : INT_MAX;
                    const unsigned m = __reduce_or_sync(0xffffffffu, v < R0 + 32 ? 1u << (v - R0) : 0u);  // v > R0
                    const int R = R0 + lane;
                    if (R < I.T) {
                        const int blk = b0 + __popc(m & (0xffffffffu >> (31 - lane)));
                        pos = bbeg[blk] + (R - bpre[blk]);
                    }
                }
                if (k >= ST && !ft_wait(S, &S.free_[s], (k / ST - 1) & 1u)) {
                    ok = false;
                    break;
                }
                S.pos[s][32 * pw + lane] = pos;
                cp_async4(&S.pn[s][32 * pw + lane], n16 + pos);
                // whole rows: 2 per step of the warp with two K halves (16 chunks of 16
                // bytes each), else 4; a lane's chunk and the swizzle of its row's low
                // bits are the same in every step
                unsigned char *base = S.A[s][0] + 32 * pw * 128;
                if (two) {
                    const int ch = lane & 15, hi = lane >> 4;
                    const uint32_t dst = tc::smem_u32(base) + (ch >> 3) * (TC_ROWS * 128) + hi * 128;
                    const uint32_t sw = (uint32_t)((ch & 7) ^ hi) << 4;
                    const uint4 *src = h16 + ch;
#pragma unroll
                    for (int i = 0; i < 16; ++i) {
                        const int p = __shfl_sync(0xffffffffu, pos, 2 * i + hi);
                        cp_async16_at(dst + 256 * i + (sw ^ (((2 * i) & 7) << 4)), src + (size_t)(uint32_t)p * 16);
                    }
                } else {
                    const int ch = lane & 7, hi = lane >> 3;
                    const uint32_t dst = tc::smem_u32(base) + hi * 128;
                    const uint32_t sw = (uint32_t)(ch ^ hi) << 4;
                    const uint4 *src = h16 + ch;
#pragma unroll
                    for (int i = 0; i < 8; ++i) {
                        const int p = __shfl_sync(0xffffffffu, pos, 4 * i + hi);
                        cp_async16_at(dst + 512 * i + (sw ^ (((4 * i) & 7) << 4)), src + (size_t)(uint32_t)p * 8);
                    }
                }
                tc::mbar_arrive_copies(&S.full[s]);
                tc::mbar_arrive(&S.full[s]);
            }
            __syncwarp();
            if (ok && lane == 0) tc::mbar_arrive(&S.ifree[b]);  // this warp is past the item
        }
        cp_async_wait_all();
    } else if (warp < FT_EPI) {
        // ---- MMA issue of stage s (lane 0 issues; the warp waits together)
        const int s = warp - FT_MMA;
        const uint64_t adesc0 = tc::smem_desc_sw128(tc::smem_u32(S.A[0][0]));
        uint32_t iph = 0;  // next phase parity of each item buffer (bit b)
        uint32_t k = 0;
        int64_t last = -1;  // the last tile issued
        unsigned alive = (1u << FT_ITEMS) - 1u;
        bool ok = true;
        for (int b = 0; alive && ok; b = b + 1 == FT_ITEMS ? 0 : b + 1) {
            if (!((alive >> b) & 1u)) continue;
            if (!ft_wait(S, &S.ifull[b], (iph >> b) & 1u)) break;
            iph ^= 1u << b;
            const FtItem I = S.item[b];
            if (I.ntiles < 0) {
                alive &= ~(1u << b);
                continue;
            }
            const bool two = V.tv[I.cloud].dp > 64;  // two K halves per row
            const uint64_t bdesc = tc::smem_desc_sw128(tc::smem_u32(S.B[b][0]));
            for (int t = 0; t < I.ntiles; ++t, ++k) {
                if (k % ST != (uint32_t)s) continue;
                if (!ft_wait(S, &S.full[s], (k / ST) & 1u)) {
                    ok = false;
                    break;
                }
                last = (int64_t)k;
                tc::fence_smem_to_async();  // the copies, acquired from their barrier
                tc::fence_after_sync();
                if (lane == 0) {
                    constexpr uint32_t idesc = tc::idesc_f16_f32(TC_ROWS, 32);
                    // descriptors count 16-byte units: K half h at 16 KB (A) or 4 KB (B), a
                    // 16-half step inside it at 32 bytes
                    const uint64_t ad = adesc0 + (uint64_t)(s * (int)(sizeof(S.A[0]) >> 4));
                    const uint32_t d = tmem + (uint32_t)(32 * s);
#pragma unroll
                    for (int j = 0; j < 4; ++j) tc::mma_f16(d, ad + 2 * j, bdesc + 2 * j, idesc, j > 0);
                    if (two) {
#pragma unroll
                        for (int j = 0; j < 4; ++j)
                            tc::mma_f16(d, ad + (sizeof(S.A[0][0]) >> 4) + 2 * j, bdesc + (sizeof(S.B[0][0]) >> 4) + 2 * j,
                                        idesc, true);
                    }
                    tc::mma_commit(&S.done[s]);
                }
                __syncwarp();
            }
            if (ok && lane == 0) tc::mbar_arrive(&S.ifree[b]);  // this warp is past the item
        }
        // the stage's MMAs in flight complete before tensor memory is freed (bounded)
        if (last >= 0) tc::mbar_wait_sleep(&S.done[s], (uint32_t)(last / ST) & 1u, TC_SLEEPS, TC_HINT);
    } else if (warp >= FT_EPI) {
        // ---- epilogue group e: every FT_EGROUPS-th tile
        const int e = (warp - FT_EPI) >> 2, quarter = warp & 3, row = 32 * quarter + lane;
        uint32_t turn = 0;  // the group whose tile it is
        uint32_t iph = 0;  // next phase parity of each item buffer (bit b)
        uint32_t k = 0, pairs = 0, kept = 0, rows_ld = 0;
        int64_t cur = 0, lim = 0;  // the warp's chunk of the list: [cur, lim) is free
        unsigned alive = (1u << FT_ITEMS) - 1u;
        bool ok = true;
        for (int b = 0; alive && ok; b = b + 1 == FT_ITEMS ? 0 : b + 1) {
            if (!((alive >> b) & 1u)) continue;
            if (!ft_wait(S, &S.ifull[b], (iph >> b) & 1u)) break;
            iph ^= 1u << b;
            const FtItem I = S.item[b];
            if (I.ntiles < 0) {
                alive &= ~(1u << b);
                continue;
            }
            const bool half = V.qp[I.cloud].half != 0, self_ok = V.qp[I.cloud].include_self != 0;
            const unsigned qmask = I.nqr >= 32 ? 0xffffffffu : (1u << I.nqr) - 1u;
            for (int t = 0; t < I.ntiles; ++t, ++k) {
                const bool mine = turn == (uint32_t)e;
                turn = turn + 1 == FT_EGROUPS ? 0 : turn + 1;
                if (!mine) continue;
                const int s = k % ST;
                if (!ft_wait(S, &S.full[s], (k / ST) & 1u) || !ft_wait(S, &S.done[s], (k / ST) & 1u)) {
                    ok = false;
                    break;
                }
                tc::fence_after_sync();
                const int pos = S.pos[s][row];
                const float pn = S.pn[s][row];
                // kept iff d^2 = n^_q + n^_p - 2 dot <= (E_q + rel |p^|)^2 + abs2 (|q^|^2 + |p^|^2)
                // + 2^-60 with E_q = s eps + rel |q^| + 2^-20, i.e. iff dot >= h_q + g_q |p^| + w_p
                // with h_q = (n^_q - E_q^2 - abs2 |q^|^2 - 2^-60) / 2, g_q = -rel E_q,
                // w_p = (n^_p - (rel^2 + abs2) |p^|^2) / 2.  The rounding of this form stays
                // below 2^-21 (n^_q + n^_p + 2 E_q^2): the first part is inside the abs2
                // term's slack over the other fp32 errors, the second is covered by the
                // 2^-20 E_q^2 taken off h_q.  The sign of dot minus the right-hand side
                // decides (exact for a subtraction); NaN (positive) keeps the pair.
                const float pa = sqrtf(pn) * H16_NORM_UP;
                const float wp = 0.5f * fmaf(-(H16_REL * H16_REL + H16_ABS2) * pa, pa, pn);
                const unsigned long long pa2 = f2_pack(pa, pa), wp2 = f2_pack(wp, wp);
                uint32_t drop = 0u;
                const uint32_t acc = tmem + ((uint32_t)(32 * quarter) << 16) + (uint32_t)(32 * s);
#pragma unroll
                for (int half16 = 1; half16 >= 0; --half16) {  // queries 31 .. 0: bit q of drop is query q's sign
                    float dot[16];
                    tc::tmem_ld16(acc + (uint32_t)(16 * half16), dot);
#pragma unroll
                    for (int j = 7; j >= 0; --j) {
                        const float4 hg = S.qhg[b][8 * half16 + j];
                        const unsigned long long thr =
                            f2_add(f2_fma(f2_pack(hg.z, hg.w), pa2, f2_pack(hg.x, hg.y)), wp2);
                        const unsigned long long df = f2_sub(f2_pack(dot[2 * j], dot[2 * j + 1]), thr);
                        drop = __funnelshift_l((uint32_t)(df >> 32), drop, 1);
                        drop = __funnelshift_l((uint32_t)df, drop, 1);
                    }
                }
                tc::fence_before_sync();
                __syncwarp();
                if (lane == 0) tc::mbar_arrive(&S.free_[s]);
                uint32_t keep = ~drop;
                const int rows = I.T - t * TC_ROWS;  // rows of the tile (and more)
                if (row < rows) {
                    uint32_t valid = qmask;
                    const int self = pos - I.qfirst;
                    if (!self_ok && (unsigned)self < 32u) valid &= ~(1u << self);
                    if (half && pos < I.qb) valid = 0u;
                    keep &= valid;
                    pairs += __popc(valid);
                } else {
                    keep = 0u;
                }
                if (quarter == 0 && lane == 0) rows_ld += min(rows, TC_ROWS);
                if (!__any_sync(0xffffffffu, keep != 0u)) continue;
                const int c = __popc(keep);
                kept += c;
                int incl = c;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const int y = __shfl_up_sync(0xffffffffu, incl, o);
                    if (lane >= o) incl += y;
                }
                const int n = __shfl_sync(0xffffffffu, incl, 31);
                // entries fill the rest of the chunk, then a new one
                const int64_t old = cur;
                const int room = (int)(lim - cur);
                int64_t nxt = 0;
                if (n > room) {
                    unsigned long long a = 0;
                    if (lane == 0) a = atomicAdd(out.n, (unsigned long long)FT_CHUNK);
                    nxt = (int64_t)__shfl_sync(0xffffffffu, a, 0);
                    lim = nxt + FT_CHUNK;
                    cur = nxt + (n - room);
                } else {
                    cur += n;
                }
                const uint32_t gp = (uint32_t)(I.rbase + pos) | (half && pos >= I.qe ? PAIR_MIRROR : 0u);
                for (int i = incl - c; keep; ++i) {
                    const int q = __ffs(keep) - 1;
                    keep &= keep - 1u;
                    const int64_t at = i < room ? old + i : nxt + (i - room);
                    if (at < out.cap) out.e[at] = make_uint2((uint32_t)(I.rbase + I.qfirst + q), gp);
                }
            }
            if (ok && lane == 0) tc::mbar_arrive(&S.ifree[b]);  // this warp is past the item
        }
        for (int64_t i = cur + lane; i < min(lim, out.cap); i += 32) out.e[i] = make_uint2(PAIR_NONE, 0u);
        unsigned long long p64 = pairs, k64 = kept;
        for (int o = 16; o > 0; o >>= 1) {
            p64 += __shfl_xor_sync(0xffffffffu, p64, o);
            k64 += __shfl_xor_sync(0xffffffffu, k64, o);
        }
        if (lane == 0) {
            stat_add(out.stat, 0, p64);
            stat_add(out.stat, 1, k64);
            stat_add(out.stat, 2, rows_ld);
        }
    }
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    if (tid == 0 && S.fail) atomicOr(err, 32);
    if (warp == 0) tc::tmem_dealloc(tmem, 256);
}

// What k_pairs does with the edges of a list.
enum {
    PAIRS_COUNT = 0,  // degrees; entries that are no edge become PAIR_NONE
    PAIRS_PLACE = 1,  // one-pass emit: each edge into its row's capacity (co.fill counts the degrees)
    PAIRS_EMIT = 2    // into the CSR (rowsel: the selected rows only)
};

// Eight consecutive floats: one 256-bit load where the address allows (al),
// else two 16-byte loads.
__device__ __forceinline__ void ld_f8(const float4 *p, bool al, float4 &a, float4 &b) {
    if (al) {
        asm("ld.global.nc.v8.f32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
            : "=f"(a.x), "=f"(a.y), "=f"(a.z), "=f"(a.w), "=f"(b.x), "=f"(b.y), "=f"(b.z), "=f"(b.w)
            : "l"(p));
    } else {
        a = __ldg(p);
        b = __ldg(p + 1);
    }
}

__device__ __forceinline__ float4 f4_sub(float4 a, float4 b) {
    return make_float4(a.x - b.x, a.y - b.y, a.z - b.z, a.w - b.w);
}
// A warp's batch of 32 pairs: positions, clouds, the pairs' eight chunk sums.
struct PairShared {
    float sum[32 * 8];
    uint2 pos[32];
    int cloud[32];
};

// Decides a list's pairs.  A warp takes 32 entries at a time: the eight lanes
// of an octet read both fp32 rows of a pair, lane j eight floats of every 64
// (contiguous 256-byte reads; a lane per 16-float chunk would touch four times
// the lines per load), and form the canonical sum (l2dist.cuh) in its order --
// a chunk of 16 coordinates lies in two neighbouring lanes, and its two FMA
// chains pass from one to the other: in the first 64 coordinates from the even
// lane to the odd one, in the second the other way round, so one exchange
// serves both and every lane ends with one chunk sum.  The chunk sums of the 32
// pairs go through shared memory, lane i adds up pair i's, decides and writes
// it.  Rows of at most 16 floats take one lane per pair.  Bound by the L1 data
// path: 1 KB of rows per pair at 128 floats, and the shuffles, which share it
// (13 per four pairs when the sums were gathered by shuffles too, 2 now).
// 256 M pairs of 128 floats and their 478 M entries placed in 17.7 ms (19.0
// before), 39 M in 3.2.
template <int MODE>
__global__ void __launch_bounds__(256, 4) k_pairs(const __grid_constant__ Views V, PairList list,
                                                  int32_t *__restrict__ deg, CapOut co,
                                                  const int64_t *__restrict__ row_ptr, int32_t *__restrict__ rowcur,
                                                  int32_t *__restrict__ col, float *__restrict__ dist,
                                                  const uint8_t *__restrict__ rowsel,
                                                  unsigned long long *__restrict__ st, int32_t *__restrict__ err) {
    const int lane = threadIdx.x & 31;
    // the entries: all of cap, or the device's count of a list that did not run out
    const int64_t total = !list.n ? list.cap : (int64_t)*list.n <= list.cap ? (int64_t)*list.n : 0;
    const int64_t warps = (int64_t)gridDim.x * (blockDim.x >> 5);
    __shared__ PairShared shared[8];  // one per warp
    PairShared &sh = shared[threadIdx.x >> 5];
    unsigned long long guard = 0, band = 0;
    uint32_t done = 0;  // emit: pairs decided; one-pass: entries of the edges found
    for (int64_t base = ((int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5)) * 32; base < total;
         base += warps * 32) {
        const uint2 e = base + lane < total ? list.e[base + lane] : make_uint2(PAIR_NONE, 0u);
        const bool valid = e.x != PAIR_NONE;
        const uint32_t gp = e.y & ~PAIR_MIRROR;
        int c = 0;
        if (V.nc > 1 && valid) {
            int lo = 0, hi = V.nc;
            while (hi - lo > 1) {
                const int mid = (lo + hi) >> 1;
                if (V.rbase[mid] <= (int64_t)e.x) lo = mid; else hi = mid;
            }
            c = lo;
        }
        const TreeView &tv = V.tv[c];
        const int dp4 = tv.dp >> 2;
        const int64_t rb = V.rbase[c];
        const float4 *qrow = reinterpret_cast<const float4 *>(tv.pts) + ((int64_t)e.x - rb) * dp4;
        const float4 *prow = reinterpret_cast<const float4 *>(tv.pts) + ((int64_t)gp - rb) * dp4;
        float sv = 0.f;
        if (valid && dp4 <= 4) sv = pair_sqdist(qrow, prow, dp4);
        const unsigned wide = __ballot_sync(0xffffffffu, valid && dp4 > 4);
        if (wide) {
            const int j = lane & 7;
            const bool odd = lane & 1;
            const int nu = (int)__reduce_max_sync(0xffffffffu, valid ? (unsigned)((dp4 + 15) >> 4) : 0u);
            __syncwarp();  // the last batch's sums are read
            sh.pos[lane] = make_uint2(e.x, gp);
            if (V.nc > 1) sh.cloud[lane] = c;
            __syncwarp();
            for (int r = 0; r < 8; ++r) {
                if (!((wide >> (4 * r)) & 0xfu)) continue;
                const int src = 4 * r + (lane >> 3);
                const bool on = (wide >> src) & 1u;
                const uint2 sp = sh.pos[src];
                const int cs = V.nc > 1 ? sh.cloud[src] : 0;
                const int n4 = V.tv[cs].dp >> 2;
                const float4 *pts = reinterpret_cast<const float4 *>(V.tv[cs].pts);
                const float4 *x = pts + (int64_t)(sp.x - (uint32_t)V.rbase[cs]) * n4;
                const float4 *y = pts + (int64_t)(sp.y - (uint32_t)V.rbase[cs]) * n4;
                const bool al = ((n4 & 1) | (int)(reinterpret_cast<uintptr_t>(pts) & 31)) == 0;
                float4 a[2][2], d[2][2];
#pragma unroll
                for (int u = 0; u < 2; ++u) {  // dp <= 128: at most two times eight floats per lane
                    const int f = 16 * u + 2 * (j ^ u);  // float4s f and f + 1
                    a[u][0] = a[u][1] = d[u][0] = d[u][1] = make_float4(0.f, 0.f, 0.f, 0.f);
                    if (on && f + 1 < n4) {
                        ld_f8(x + f, al, a[u][0], a[u][1]);
                        ld_f8(y + f, al, d[u][0], d[u][1]);
                    } else if (on && f < n4) {
                        a[u][0] = __ldg(x + f);
                        d[u][0] = __ldg(y + f);
                    }
                }
                // the chains of a chunk's first eight floats (u = 0: even lanes, 1: odd lanes) go to
                // the neighbour, which has its last eight
                float lo[2], hi[2];
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                    a[u][0] = f4_sub(a[u][0], d[u][0]);
                    a[u][1] = f4_sub(a[u][1], d[u][1]);
                    const float4 p = a[u][0], q = a[u][1];
                    lo[u] = fmaf(q.z, q.z, fmaf(q.x, q.x, fmaf(p.z, p.z, p.x * p.x)));
                    hi[u] = fmaf(q.w, q.w, fmaf(q.y, q.y, fmaf(p.w, p.w, p.y * p.y)));
                }
                const float lo_in = __shfl_xor_sync(0xffffffffu, odd ? lo[1] : lo[0], 1);
                const float hi_in = __shfl_xor_sync(0xffffffffu, odd ? hi[1] : hi[0], 1);
                float chunk[2];
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                    const float4 p = a[u][0], q = a[u][1];
                    chunk[u] = fmaf(q.z, q.z, fmaf(q.x, q.x, fmaf(p.z, p.z, fmaf(p.x, p.x, lo_in)))) +
                               fmaf(q.w, q.w, fmaf(q.y, q.y, fmaf(p.w, p.w, fmaf(p.y, p.y, hi_in))));
                }
                // chunk j / 2 in odd lanes, 4 + j / 2 in even ones; odd rounds swap the halves (banks)
                sh.sum[8 * src + ((odd ? j >> 1 : 4 + (j >> 1)) ^ ((r & 1) << 2))] = odd ? chunk[0] : chunk[1];
            }
            __syncwarp();
            if ((wide >> lane) & 1u) {
                const float4 *ss = reinterpret_cast<const float4 *>(sh.sum + 8 * lane);
                const int sw = (lane >> 2) & 1;
                const float4 s0 = ss[sw];
                sv = ((s0.x + s0.y) + s0.z) + s0.w;
                if (nu > 1) {
                    const float4 s1 = ss[1 - sw];
                    sv = (((sv + s1.x) + s1.y) + s1.z) + s1.w;
                }
            }
        }
        if (!valid) continue;
        const QParams &qp = V.qp[c];
        if (MODE == PAIRS_EMIT) ++done;
        const int edge = decide32(qp, sv, band);
        bool is_edge = edge > 0;
        float d = sqrtf(sv);
        const int64_t o = rb + tv.perm[(int64_t)e.x - rb], p = rb + tv.perm[(int64_t)gp - rb];
        if (edge < 0) {
            if (MODE != PAIRS_EMIT) {
                ++guard;
                note_guard_rows((int32_t)o, (int32_t)p);
            }
            const double s64 = sq_l2_exact4(qrow, prow, tv.dim);
            is_edge = s64 <= qp.eps2_64;
            d = (float)sqrt(s64);
        }
        if (!is_edge) {
            if (MODE == PAIRS_COUNT) list.e[base + lane] = make_uint2(PAIR_NONE, 0u);
            continue;
        }
        const bool mir = (e.y & PAIR_MIRROR) != 0u;
        if (MODE == PAIRS_COUNT) {
            atomicAdd(&deg[o], 1);
            if (mir) atomicAdd(&deg[p], 1);
        } else if (MODE == PAIRS_PLACE) {
            done += mir ? 2u : 1u;
            cap_put(co, (int)o, (int)(p - rb), d);
            if (mir) cap_put(co, (int)p, (int)(o - rb), d);
        } else {
            auto put = [&](int64_t row, int32_t v) {
                if (rowsel && !rowsel[row]) return;
                const int64_t at = row_ptr[row] + atomicAdd(&rowcur[row], 1);
                if (at < row_ptr[row + 1]) {
                    col[at] = v;
                    dist[at] = d;
                } else {
                    atomicOr(err, 4);
                }
            };
            put(o, (int32_t)(p - rb));
            if (mir) put(p, (int32_t)(o - rb));
        }
    }
    unsigned long long done64 = done;
    for (int o = 16; o > 0; o >>= 1) {
        guard += __shfl_xor_sync(0xffffffffu, guard, o);
        band += __shfl_xor_sync(0xffffffffu, band, o);
        done64 += __shfl_xor_sync(0xffffffffu, done64, o);
    }
    if (lane == 0) {
        if (MODE == PAIRS_EMIT) {
            stat_add(st, ST_EMIT, done64);
        } else {
            stat_add(st, ST_GUARD, guard);
            stat_add(st, ST_BAND, band);
            if (MODE == PAIRS_PLACE) stat_add(st, ST_PLACED, done64);
        }
    }
}

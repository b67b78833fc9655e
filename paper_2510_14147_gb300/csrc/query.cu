// query.cu -- the batched ε query (Algorithm 3 with the batching of Sec. IV-B)
// as a count -> scan -> emit pipeline, plus the CSR row sort.
//
// Query groups are runs of sibling leaf blocks (at most 32 points, contiguous
// in tree order, centre c_g, radius r_g).  Stages:
//   1. traversal (k_traverse_*): one warp per group walks the tree from the
//      root with a stack of sibling ranges; 32 vertices are tested at a time,
//      one per lane.  A vertex v survives iff d(c_g, v) <= r(v) + eps + r_g
//      (every query q of the group has d(q, c_g) <= r_g, so no descendant of a
//      pruned v is within eps of any q: triangle inequality).  Survivors are
//      compacted with ballots: leaf blocks are candidates, internal vertices
//      push their child range.  One pass into a pool that grows when it runs
//      out, then one range of candidates per group.
//   2. leaf stage: slices of a group's candidates (work items) decide d(q, p) <=
//      eps exactly (see QParams) for every (query, candidate point) pair.  Count
//      pass: per-query degrees and, for L2 points, a list of the edges (or, from
//      the tensor-core filter, of the pairs that may be edges); the learned form
//      places the edges right away.  Emit pass: the list's entries, or the
//      blocks flagged by the count pass; writes col/dist at the row offsets.
//   3. scan of degrees to row_ptr (int64), then a per-row sort by column.
#include <cfloat>
#include <climits>
#include <cmath>
#include <cstring>
#include <mutex>
#include <type_traits>

#include "f32x2.cuh"
#include "lev.cuh"
#include "profile.cuh"
#include "query.cuh"
#include "reserve.cuh"
#include "tc.cuh"
#include "l2dist.cuh"

namespace ct {

namespace {

constexpr int TRAV_WARPS = 4;              // warps per traversal block
constexpr size_t kTravSmemMost = TRAV_WARPS * 4096 * sizeof(float);  // the group centres at the longest rows
constexpr size_t kLevSmemMost = 96 * 1024;                           // match masks of an edit-distance leaf block
constexpr int LEAF_T = 128;                // threads per leaf-tile block
constexpr int KC = 128;                    // floats per K chunk of a tile
// padded row stride of a tile in float4 (odd: rows 8 apart share no bank), for
// rows of at most 64 floats and for longer ones (in chunks of KC)
constexpr int KS_SHORT = 64 / 4 + 1, KS_LONG = KC / 4 + 1;
constexpr bool short_rows(int dp) { return dp <= 64; }
constexpr uint32_t FLAG = 0x80000000u;     // candidate produced an edge
constexpr float PRUNE_REL = 1.0f + 0x1p-10f;
constexpr float PRUNE_ABS = 0x1p-60f;


// Diagnostic (off unless a test sets it): the CSR rows of both ends of every
// pair a count pass decides by the FP64 sum, appended to a caller's buffer.
__device__ int32_t *g_guard_rows = nullptr;
__device__ unsigned long long *g_guard_n = nullptr;
__device__ long long g_guard_cap = 0;

__device__ __forceinline__ void note_guard_rows(int32_t a, int32_t b) {
    int32_t *r = g_guard_rows;
    if (!r) return;
    const unsigned long long k = atomicAdd(g_guard_n, 2ull);
    if ((long long)k + 1 < g_guard_cap) {
        r[k] = a;
        r[k + 1] = b;
    }
}

__device__ __forceinline__ void stat_add(unsigned long long *st, int slot, unsigned long long v) {
    if (v) atomicAdd(st + slot, v);
}

struct TreeView {
    const float *pts, *node_ctr, *radius, *dcen, *group_radius;
    const uint32_t *bits;  // Hamming rows (wp words each)
    const int32_t *perm, *node_begin, *node_count, *child_begin, *child_count, *leaf_ids;
    const int32_t *group_begin, *group_count, *group_order;
    const uint8_t *sdata;
    const int64_t *soff;
    int dp, dim, n_leaves, n_groups, wp;
};

TreeView view_of(const ct_tree *t) {
    TreeView v;
    v.pts = t->pts; v.node_ctr = t->node_ctr; v.radius = t->radius; v.dcen = t->dcen;
    v.perm = t->perm; v.node_begin = t->node_begin; v.node_count = t->node_count;
    v.child_begin = t->child_begin; v.child_count = t->child_count; v.leaf_ids = t->leaf_ids;
    v.sdata = t->sdata; v.soff = t->soff; v.dp = t->dp; v.dim = t->dim; v.n_leaves = t->n_leaves;
    v.group_begin = t->group_begin; v.group_count = t->group_count; v.group_radius = t->group_radius;
    v.group_order = t->group_order;
    v.n_groups = t->n_groups;
    v.bits = t->bits;
    v.wp = t->wp;
    return v;
}

// Up to kMaxClouds trees queried by the same launches (in the kernel parameter
// bank): global group gg of cloud c is gbase[c] + g, global row rbase[c] + o.
// A single query is the case nc = 1.
constexpr int kMaxClouds = kBatchClouds;
struct Views {
    int nc;
    int32_t gbase[kMaxClouds + 1];
    int64_t rbase[kMaxClouds + 1];
    TreeView tv[kMaxClouds];
    QParams qp[kMaxClouds];
    int16_t item_len[kMaxClouds];  // candidate blocks per work item
    uint8_t use_tc[kMaxClouds];    // leaf kernel of the count pass: tensor-core tiles (1) or FP32 tiles (0)
    // tensor-core filter rows: the fp16 rows, their squared norms, {s, s eps_up}
    const uint4 *h16[kMaxClouds];
    const float *n16[kMaxClouds];
    const float *s16[kMaxClouds];
};
static_assert(sizeof(Views) <= 32000, "Views exceeds the kernel parameter space");
__device__ __forceinline__ int cloud_of_group(const Views &V, int gg) {
    int lo = 0, hi = V.nc;
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (V.gbase[mid] <= gg) lo = mid; else hi = mid;
    }
    return lo;
}

// ------------------------------------------------------------ traversal
//
// One pass: every warp appends the candidate leaf blocks of its groups to
// private chunks of a shared pool; a group's candidates form one or more
// segments (group, pool offset, count).  If the pool runs out, the walks stop
// where they are: a warp that finds no chunk for its next step stores the
// ranges on its stack, and the work it takes after that, in the resume list;
// the host grows the pool and walks the list on.  (The pass used to be rerun
// from the start: 19.5 of 63 ms on 121k x 16 uniform points and 23 of 60 ms
// on a million codes went into two full passes.)

constexpr int POOL_CHUNK = 2048;

struct Pool {
    uint32_t *data;
    int64_t cap;
    unsigned long long *next;  // chunk allocator
    int32_t *seg_group, *seg_count;
    int64_t *seg_begin;
    int32_t *nseg;
    int64_t seg_cap;
    unsigned long long *total;  // candidates of all groups
    int32_t *overflow;          // 1: out of chunks; 2: out of segments or of the resume list
    // work left when the pool ran out, as items (group, first vertex, count or
    // -1: the whole group); null: walks go on, counting without writing
    int4 *resume = nullptr;
    unsigned long long *n_resume = nullptr;
    int32_t *n_whole = nullptr;  // whole groups among them
    int resume_cap = 0;
};
constexpr int POOL_STOPPED = 1;

// Walks stopped at a step limit leave their stack's ranges here, as items
// (global group, first vertex, count, -) that the next round walks.
struct Spill {
    int4 *items;
    unsigned long long *count;  // entries asked for: may exceed cap (see reserve.cuh)
    int cap;
    int limit;       // steps before a walk stops
};
// Rounds after the groups' round; the last one has no step limit, and walks
// that are long when it begins set its time.  L2 walks are done by the third
// or fourth.  Of edit-distance walks, whose vertices can have thousands of
// children, 6.0 of 7.3 ms were spent in the last of 4 rounds (50k reads of 96);
// with long ranges cut up they are done by the fourth, 1.5 ms in all, and two
// spare rounds stand against other data.  A round that finds no work takes 6 us.
constexpr int TRAV_ROUNDS = 4, TRAV_ROUNDS_LEV = 6;
constexpr int TRAV_LIMIT0 = 256;   // step limit of the groups' round
constexpr int TRAV_LIMIT = 128;    // step limit of the next rounds
// edit distance: a step (32 bit-parallel recurrences) costs about a hundred
// L2 steps, so its walks stop much sooner
constexpr int TRAV_LIMIT0_LEV = 8, TRAV_LIMIT_LEV = 8;

// Warp-uniform write cursor: current chunk, its fill, the open segment.
struct PoolCursor {
    int64_t cur;
    int fill;
    int64_t seg_begin;
    int seg_count;
};

__device__ __forceinline__ void pool_close(const Pool &P, int g, PoolCursor &pc) {
    if (pc.seg_count > 0 && (threadIdx.x & 31) == 0) {
        int idx = atomicAdd(P.nseg, 1);
        if (idx < P.seg_cap) {
            P.seg_group[idx] = g;
            P.seg_begin[idx] = pc.seg_begin;
            P.seg_count[idx] = pc.seg_count;
        } else {
            atomicOr(P.overflow, 2);
        }
    }
    pc.seg_count = 0;
}

// A new chunk for the next step's 32 vertices; false when the pool is out.
__device__ __forceinline__ bool pool_more(const Pool &P, int g, PoolCursor &pc) {
    pool_close(P, g, pc);
    unsigned long long c = 0ull;
    if ((threadIdx.x & 31) == 0) {
        c = atomicAdd(P.next, (unsigned long long)POOL_CHUNK);
        if ((int64_t)c + POOL_CHUNK > P.cap) {
            atomicOr(P.overflow, 1);
            c = ~0ull;
        }
    }
    c = __shfl_sync(0xffffffffu, c, 0);
    if (c == ~0ull) {
        pc.cur = -1;
        pc.fill = POOL_CHUNK;
        return false;
    }
    pc.cur = (int64_t)c;
    pc.fill = 0;
    pc.seg_begin = pc.cur;
    return true;
}
__device__ __forceinline__ void resume_put(const Pool &P, unsigned long long at, int4 item) {
    if (at < (unsigned long long)P.resume_cap) P.resume[at] = item;
    else atomicOr(P.overflow, 2);
}
// Leaves one work item (group, range; count 0: the whole group) for the next pass.
__device__ __forceinline__ void resume_item(const Pool &P, int g, int2 start) {
    if ((threadIdx.x & 31) == 0) {
        if (start.y == 0) atomicAdd(P.n_whole, 1);
        resume_put(P, atomicAdd(P.n_resume, 1ull), make_int4(g, start.x, start.y ? start.y : -1, 0));
    }
}

// Appends the values of the lanes with `flag` set, in lane order.
__device__ __forceinline__ void pool_append(const Pool &P, int g, PoolCursor &pc, bool flag, uint32_t v) {
    const int lane = threadIdx.x & 31;
    const unsigned m = __ballot_sync(0xffffffffu, flag);
    const int n = __popc(m);
    if (!n) return;
    const int rank = __popc(m & lanemask_lt());
    const int room = pc.cur >= 0 ? POOL_CHUNK - pc.fill : 0;
    if (n <= room) {
        if (flag) P.data[pc.cur + pc.fill + rank] = v;
        pc.fill += n;
        pc.seg_count += n;
        return;
    }
    if (flag && rank < room) P.data[pc.cur + pc.fill + rank] = v;
    pc.seg_count += room;
    pool_close(P, g, pc);
    unsigned long long c = 0ull;
    if (lane == 0) c = atomicAdd(P.next, (unsigned long long)POOL_CHUNK);
    c = __shfl_sync(0xffffffffu, c, 0);
    if ((int64_t)c + POOL_CHUNK > P.cap) {  // out of pool: keep counting, write nothing
        if (lane == 0) atomicOr(P.overflow, 1);
        pc.cur = -1;
        pc.fill = POOL_CHUNK;
        pc.seg_begin = 0;
        pc.seg_count = 0;
        return;
    }
    pc.cur = (int64_t)c;
    pc.fill = n - room;
    pc.seg_begin = pc.cur;
    pc.seg_count = n - room;
    if (flag && rank >= room) P.data[pc.cur + rank - room] = v;
}

// DFS over ranges of sibling vertices from `start` (count 0: the root's
// children): up to 32 vertices are tested per step, vertex i of the step by
// lane i (`tester(v, n)` returns the keep flag of the lane's vertex v, for
// lanes below n); a top range shorter than 32 is completed from the range
// below it, so that fewer lanes idle; survivors are
// compacted with ballots -- leaf blocks are appended to the pool, internal
// vertices push their child range.  The vertices' child ranges are loaded
// before the test, so that their loads overlap the test's.  With `sp`, a walk
// that reaches sp->limit steps stores the ranges left on its stack in
// sp->items and stops (if they do not fit it goes on).
// A vertex's points are the positions from node_begin on, node_count of them;
// vertices whose points all lie before `qlo` are left out with everything
// below them (upper-triangle form: a group takes the pairs from its own first
// row on; 0: none).  (They used to be walked and dropped when the candidates
// were gathered.  Walk of 1M x 128: 11.2 -> 6.9 ms at 70 neighbours, 15.5 ->
// 8.2 at 500; 1M codes 8.7 -> 5.5, with the gather 15 ms less in all.)
template <class Tester>
__device__ __forceinline__ int walk_group(const TreeView &tv, int2 *__restrict__ stack, int cap, int g, int qlo,
                                          int2 start, const Pool &P, PoolCursor &pc, unsigned long long &evals,
                                          int32_t *__restrict__ err, const Spill *sp, Tester tester) {
    const int lane = threadIdx.x & 31;
    int n_cand = 0, status = 0;
    pc.seg_begin = pc.cur + pc.fill;
    pc.seg_count = 0;
    if (P.resume && pc.fill > POOL_CHUNK - 32 && !pool_more(P, g, pc)) {
        resume_item(P, g, start);
        return POOL_STOPPED;
    }
    if (start.y == 0 && tv.child_count[0] == 0) {  // the root is a leaf block: it is the only candidate
        pool_append(P, g, pc, lane == 0, 0u);
        n_cand = 1;
    } else {
        int top = 0;
        if (lane == 0) stack[0] = start.y ? start : make_int2(tv.child_begin[0], tv.child_count[0]);
        top = 1;
        __syncwarp();
        int limit = sp ? sp->limit : INT_MAX;
        for (int steps = 0; top > 0; ++steps) {
            if (steps >= limit) {
                // long ranges are stored in pieces that a quarter of the limit walks: a
                // vertex can have tens of thousands of children
                const int piece = max(32, 8 * sp->limit);
                int total = 0;
                for (int i = lane; i < top; i += 32) total += (stack[i].y + piece - 1) / piece;
                total = (int)__reduce_add_sync(0xffffffffu, (unsigned)total);
                unsigned long long first = 0;
                if (lane == 0) first = atomicAdd(sp->count, (unsigned long long)total);
                const ListRoom room = list_room(__shfl_sync(0xffffffffu, first, 0), total, sp->cap);
                if (room.fits) {
                    int base = room.begin;
                    for (int i0 = 0; i0 < top; i0 += 32) {
                        const int2 r = i0 + lane < top ? stack[i0 + lane] : make_int2(0, 0);
                        const int c = (r.y + piece - 1) / piece;
                        int incl = c;
#pragma unroll
                        for (int o = 1; o < 32; o <<= 1) {
                            const int y = __shfl_up_sync(0xffffffffu, incl, o);
                            if (lane >= o) incl += y;
                        }
                        for (int j = 0; j < c; ++j)
                            sp->items[base + incl - c + j] =
                                make_int4(g, r.x + j * piece, min(piece, r.y - j * piece), 0);
                        base += __shfl_sync(0xffffffffu, incl, 31);
                    }
                    break;
                }
                // no room: what was asked for below the end holds empty ranges (count 0,
                // skipped), and the walk is finished here
                for (int i = room.begin + lane; i < sp->cap; i += 32) sp->items[i] = make_int4(g, 0, 0, 0);
                limit = INT_MAX;
            }
            // resumable walks have room for every vertex of a step before it begins
            if (P.resume && pc.fill > POOL_CHUNK - 32 && !pool_more(P, g, pc)) {
                unsigned long long base = 0;
                if (lane == 0) base = atomicAdd(P.n_resume, (unsigned long long)top);
                base = __shfl_sync(0xffffffffu, base, 0);
                for (int i = lane; i < top; i += 32) {
                    const int2 r = stack[i];
                    resume_put(P, base + i, make_int4(g, r.x, r.y, 0));
                }
                status = POOL_STOPPED;
                break;
            }
            // the step's vertices: the top ranges of the stack, newest first,
            // until the 32 lanes are filled (lane i reads the i-th range from
            // the top; ranges are never empty); the last range drawn on may be
            // taken in part and keeps its rest on the stack.  A step reaches an
            // older block of ranges only when the newer ones are used up, so
            // the least deep vertex of each block on the stack is deeper than
            // the block below's: at most depth + 1 blocks of at most 32 ranges.
            const int nr = top < 32 ? top : 32;
            const int2 ri = lane < nr ? stack[top - 1 - lane] : make_int2(0, 0);
            int incl = ri.y;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int y = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += y;
            }
            const int excl = incl - ri.y;
            const int total = __shfl_sync(0xffffffffu, incl, 31);
            const int n = total < 32 ? total : 32;
            const int nfull = __popc(__ballot_sync(0xffffffffu, lane < nr && incl <= 32));
            // the first lane of each range drawn on, then each lane's range
            const unsigned smask = __reduce_or_sync(0xffffffffu, (lane < nr && excl < 32) ? 1u << excl : 0u);
            const int k = __popc(smask & (0xffffffffu >> (31 - lane))) - 1;
            const int kx = __shfl_sync(0xffffffffu, ri.x, k);
            const int ke = __shfl_sync(0xffffffffu, excl, k);
            const int px = __shfl_sync(0xffffffffu, ri.x, nfull & 31), py = __shfl_sync(0xffffffffu, ri.y, nfull & 31);
            const int pe = __shfl_sync(0xffffffffu, excl, nfull & 31);
            __syncwarp();
            top -= nfull;
            if (nfull < nr && pe < 32 && lane == 0) stack[top - 1] = make_int2(px + (32 - pe), py - (32 - pe));
            if (lane < n) ++evals;
            const int v = lane < n ? kx + (lane - ke) : 0;
            int ccount = 0, cbegin = 0, end = INT_MAX;
            if (lane < n) {
                ccount = tv.child_count[v];
                cbegin = tv.child_begin[v];
                if (qlo > 0) end = tv.node_begin[v] + tv.node_count[v];
            }
            const bool keep = tester(v, n) && end > qlo;
            const bool leaf = keep && ccount == 0;
            pool_append(P, g, pc, keep && leaf, (uint32_t)v);
            n_cand += __popc(__ballot_sync(0xffffffffu, keep && leaf));
            const unsigned mi = __ballot_sync(0xffffffffu, keep && !leaf);
            const int np = __popc(mi);
            if (top + np > cap) {  // cannot happen for a stack of 32 * (depth + 2) ranges (above)
                if (lane == 0) atomicOr(err, 2);
                return -1;
            }
            if (keep && !leaf) {
                // reverse lane order so the lowest lane's children are on top (DFS order)
                int slot = top + __popc(mi & ~lanemask_lt() & ~(1u << lane));
                stack[slot] = make_int2(cbegin, ccount);
            }
            top += np;
            __syncwarp();
        }
    }
    pool_close(P, g, pc);
    if (lane == 0) atomicAdd(P.total, (unsigned long long)n_cand);
    return status;
}

// Vertices the warp tested for group g (for fitting the predictor; the rounds
// of one group's walk add up).
__device__ __forceinline__ void group_visits(int32_t *gvisit, int g, unsigned long long mine) {
    unsigned long long v = mine;
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if ((threadIdx.x & 31) == 0) atomicAdd(gvisit + g, (int32_t)(v < 0x7fffffffull ? v : 0x7fffffffull));
}

// L2 test of `take` vertices (lane i's: vid) against the group centre (shared
// memory): TPD lanes share one vertex and read its centre row in coalesced
// 16-byte pieces.  The TPD rounds' partial sums are reduced together -- each
// exchange halves the sums a lane holds, 7 shuffles instead of 8 x 4 at 8 lanes
// a vertex -- and lane i gets vertex i's squared distance.  Keep v unless
// d > (r(v) + eps + r_g)(1 + 2^-10).  Bound by the latency of a step's loads
// (L2 hits) and its issue slots: walk of 1M x 128 6.85 -> 6.4 ms with the packed
// arithmetic and the joint reduction.
template <int TPD>
__device__ __forceinline__ bool l2_keep(const TreeView &tv, const float4 *cen, int nq4, int vid, int take,
                                        float add) {
    constexpr int NPR = 32 / TPD;  // vertices per round; TPD rounds cover a step of 32
    const int lane = threadIdx.x & 31, sub = lane / TPD, j = lane % TPD;
    const float rad = lane < take ? tv.radius[vid] : 0.f;  // issued with the centre rows
    // all rounds' partial sums first (their loads overlap), then the reductions
    float part[TPD];
#pragma unroll
    for (int u = 0; u < TPD; ++u) {
        const int i = u * NPR + sub;
        const int vi = __shfl_sync(0xffffffffu, vid, i);  // vertex of lane i
        unsigned long long acc = 0ull;
        if (u * NPR < take && i < take) {
            const ulonglong2 *row = reinterpret_cast<const ulonglong2 *>(tv.node_ctr) + (size_t)vi * nq4;
            const ulonglong2 *c = reinterpret_cast<const ulonglong2 *>(cen);
#pragma unroll 4
            for (int k = j; k < nq4; k += TPD) {
                const ulonglong2 a = c[k], b = __ldg(row + k);
                const unsigned long long dx = f2_sub(a.x, b.x), dy = f2_sub(a.y, b.y);
                acc = f2_sqacc(dx, acc);
                acc = f2_sqacc(dy, acc);
            }
        }
        part[u] = f2_sum(acc);
    }
#pragma unroll
    for (int o = TPD / 2; o > 0; o >>= 1) {  // lane j keeps the sums of the rounds u with bit o of j
        const bool upper = (j & o) != 0;
#pragma unroll
        for (int i = 0; i < o; ++i) {
            const float send = upper ? part[i] : part[i + o], own = upper ? part[i + o] : part[i];
            part[i] = own + __shfl_xor_sync(0xffffffffu, send, o);
        }
    }
    // lane (sub, j) holds vertex j NPR + sub
    const float mine = __shfl_sync(0xffffffffu, part[0], (lane & (NPR - 1)) * TPD + lane / NPR);
    if (lane >= take) return false;
    const float bound = fmaf(rad + add, PRUNE_REL, PRUNE_ABS);
    return !(sqrtf(mine) > bound);
}

// Warp per group over all clouds' groups, taken dynamically in `order`
// (global group ids), or -- in the later rounds -- per stored range of a
// walk that reached the step limit; the lanes per vertex test follow the
// cloud's row length.  Walks stop at out.limit steps (no limit without
// out.items) and store the rest of their stack in `out`.  (Eight blocks an SM
// leave 64 registers a thread; -Xptxas -v: 124 bytes of them spilled, 100 read
// back.)
__global__ void __launch_bounds__(TRAV_WARPS * 32, 8) k_traverse_l2(
    const __grid_constant__ Views V, const int32_t *__restrict__ order, int n_order,
    const int4 *__restrict__ in_items, const unsigned long long *__restrict__ in_count, int in_cap, Spill out, Pool P,
    longlong2 *__restrict__ cursors, int2 *__restrict__ stacks, int cap, unsigned long long *__restrict__ st,
    int32_t *__restrict__ err, int32_t *__restrict__ next_group, int32_t *__restrict__ gvisit, int max_nq4) {
    extern __shared__ float4 sc[];  // TRAV_WARPS x (largest dp / 4)
    const int wib = threadIdx.x >> 5, lane = threadIdx.x & 31;
    float4 *cen = sc + wib * max_nq4;
    const int gw = blockIdx.x * TRAV_WARPS + wib;
    int2 *stack = stacks + (int64_t)gw * cap;
    unsigned long long evals = 0;
    // the warp's pool chunk carries over from the previous round
    PoolCursor pc{-1, POOL_CHUNK, 0, 0};
    if (in_items) {
        const longlong2 c = cursors[gw];
        pc.cur = c.x;
        pc.fill = (int)c.y;
    }
    const int n_work = in_items ? list_length(*in_count, in_cap) : n_order;
    const Spill *sp = out.items ? &out : nullptr;
    bool full = false;  // the pool had no chunk for this warp
    for (;;) {
        // work is taken dynamically: walks differ widely in length
        int gi = 0;
        if (lane == 0) gi = atomicAdd(next_group, 1);
        gi = __shfl_sync(0xffffffffu, gi, 0);
        if (gi >= n_work) break;
        int gg;
        int2 start = make_int2(0, 0);
        if (in_items) {
            const int4 w = in_items[gi];
            if (w.z == 0) continue;  // an empty range (a stop that did not fit)
            gg = w.x;
            if (w.z > 0) start = make_int2(w.y, w.z);
        } else {
            gg = order[gi];
        }
        if (full) {
            resume_item(P, gg, start);
            continue;
        }
        const int c = cloud_of_group(V, gg);
        const TreeView &tv = V.tv[c];
        const int g = gg - V.gbase[c];
        const int nq4 = tv.dp >> 2;
        const int tpd = nq4 >= 16 ? 8 : nq4 >= 8 ? 4 : nq4 >= 4 ? 2 : 1;
        const float4 *crow = reinterpret_cast<const float4 *>(tv.pts + (size_t)tv.group_begin[g] * tv.dp);
        for (int k = lane; k < nq4; k += 32) cen[k] = crow[k];
        __syncwarp();
        const float add = V.qp[c].eps_up + tv.group_radius[g];
        auto tester = [&](int v, int take) {
            switch (tpd) {
                case 8: return l2_keep<8>(tv, cen, nq4, v, take, add);
                case 4: return l2_keep<4>(tv, cen, nq4, v, take, add);
                case 2: return l2_keep<2>(tv, cen, nq4, v, take, add);
                default: return l2_keep<1>(tv, cen, nq4, v, take, add);
            }
        };
        const unsigned long long e0 = evals;
        const int qlo = V.qp[c].half ? tv.group_begin[g] : 0;
        const int ws = walk_group(tv, stack, cap, gg, qlo, start, P, pc, evals, err, sp, tester);
        if (ws < 0) return;
        full = ws == POOL_STOPPED;
        if (gvisit) group_visits(gvisit, gg, evals - e0);
        __syncwarp();
    }
    if (lane == 0) cursors[gw] = make_longlong2(pc.cur, pc.fill);
    for (int o = 16; o > 0; o >>= 1) evals += __shfl_xor_sync(0xffffffffu, evals, o);
    if (lane == 0) stat_add(st, ST_TRAV, evals);
}

// Edit distance: a vertex survives iff lev(c_g, v) <= r(v) + eps + r_g
// (integers, exact).  One warp per block; the group centre's match masks are
// in shared memory.
template <int W>
__global__ void __launch_bounds__(32) k_traverse_lev(
    TreeView tv, QParams qp, const int4 *__restrict__ in_items, const unsigned long long *__restrict__ in_count, int in_cap,
    Spill out, Pool P, longlong2 *__restrict__ cursors, int2 *__restrict__ stacks, int cap,
    unsigned long long *__restrict__ st, int32_t *__restrict__ err, int32_t *__restrict__ next_group,
    int32_t *__restrict__ gvisit) {
    __shared__ uint64_t peq[256 * W];
    const int lane = threadIdx.x;
    int2 *stack = stacks + (int64_t)blockIdx.x * cap;
    unsigned long long evals = 0;
    // the warp's pool chunk carries over from the previous round
    PoolCursor pc{-1, POOL_CHUNK, 0, 0};
    if (in_items) {
        const longlong2 c = cursors[blockIdx.x];
        pc.cur = c.x;
        pc.fill = (int)c.y;
    }
    const int n_work = in_items ? list_length(*in_count, in_cap) : tv.n_groups;
    const Spill *sp = out.items ? &out : nullptr;
    bool full = false;  // the pool had no chunk for this warp
    for (;;) {
        int gi = 0;
        if (lane == 0) gi = atomicAdd(next_group, 1);
        gi = __shfl_sync(0xffffffffu, gi, 0);
        if (gi >= n_work) break;
        int g;
        int2 start = make_int2(0, 0);
        if (in_items) {
            const int4 w = in_items[gi];
            if (w.z == 0) continue;  // an empty range (a stop that did not fit)
            g = w.x;
            if (w.z > 0) start = make_int2(w.y, w.z);
        } else {
            g = tv.group_order[gi];
        }
        if (full) {
            resume_item(P, g, start);
            continue;
        }
        int cpos = tv.group_begin[g];
        const uint8_t *pat = tv.sdata + tv.soff[cpos];
        int m = (int)(tv.soff[cpos + 1] - tv.soff[cpos]);
        __syncwarp();
        lev_build_peq<W>(peq, pat, m);
        __syncwarp();
        const int add = qp.lev_k + (int)tv.group_radius[g];
        auto tester = [&](int v, int take) {
            if (lane >= take) return false;
            const int vp = tv.node_begin[v];
            const int k = add + (int)tv.radius[v];
            const uint8_t *txt = tv.sdata + tv.soff[vp];
            const int n = (int)(tv.soff[vp + 1] - tv.soff[vp]);
            return lev_myers<W>(peq, m, txt, n, k) <= k;
        };
        const unsigned long long e0 = evals;
        const int qlo = qp.half ? tv.group_begin[g] : 0;
        const int ws = walk_group(tv, stack, cap, g, qlo, start, P, pc, evals, err, sp, tester);
        if (ws < 0) return;
        full = ws == POOL_STOPPED;
        if (gvisit) group_visits(gvisit, g, evals - e0);
        __syncwarp();
    }
    if (lane == 0) cursors[blockIdx.x] = make_longlong2(pc.cur, pc.fill);
    for (int o = 16; o > 0; o >>= 1) evals += __shfl_xor_sync(0xffffffffu, evals, o);
    if (lane == 0) stat_add(st, ST_TRAV, evals);
}

// Hamming: a vertex survives iff ham(c_g, v) <= r(v) + eps + r_g (integers,
// exact).  One warp per block, lane i tests vertex i of a step against the
// group centre's row in shared memory.
// Distance of a row in shared memory (a) to a row in global memory (b, read
// through the read-only path).
__device__ __forceinline__ int ham_rows(const uint4 *a, const uint4 *__restrict__ b, int nq) {
    int d = 0;
    for (int k = 0; k < nq; ++k) {
        const uint4 x = a[k], y = __ldg(b + k);
        d += __popc(x.x ^ y.x) + __popc(x.y ^ y.y) + __popc(x.z ^ y.z) + __popc(x.w ^ y.w);
    }
    return d;
}
// Both rows in shared memory (plain loads).
__device__ __forceinline__ int ham_rows_smem(const uint4 *a, const uint4 *b, int nq) {
    int d = 0;
    for (int k = 0; k < nq; ++k) {
        const uint4 x = a[k], y = b[k];
        d += __popc(x.x ^ y.x) + __popc(x.y ^ y.y) + __popc(x.z ^ y.z) + __popc(x.w ^ y.w);
    }
    return d;
}

__global__ void __launch_bounds__(32) k_traverse_ham(
    TreeView tv, QParams qp, const int4 *__restrict__ in_items, const unsigned long long *__restrict__ in_count, int in_cap,
    Spill out, Pool P, longlong2 *__restrict__ cursors, int2 *__restrict__ stacks, int cap,
    unsigned long long *__restrict__ st, int32_t *__restrict__ err, int32_t *__restrict__ next_group,
    int32_t *__restrict__ gvisit) {
    __shared__ uint4 cen[32];  // up to 4096 bits
    const int lane = threadIdx.x;
    const int nq = tv.wp >> 2;
    int2 *stack = stacks + (int64_t)blockIdx.x * cap;
    unsigned long long evals = 0;
    // the warp's pool chunk carries over from the previous round
    PoolCursor pc{-1, POOL_CHUNK, 0, 0};
    if (in_items) {
        const longlong2 c = cursors[blockIdx.x];
        pc.cur = c.x;
        pc.fill = (int)c.y;
    }
    const int n_work = in_items ? list_length(*in_count, in_cap) : tv.n_groups;
    const Spill *sp = out.items ? &out : nullptr;
    bool full = false;  // the pool had no chunk for this warp
    for (;;) {
        int gi = 0;
        if (lane == 0) gi = atomicAdd(next_group, 1);
        gi = __shfl_sync(0xffffffffu, gi, 0);
        if (gi >= n_work) break;
        int g;
        int2 start = make_int2(0, 0);
        if (in_items) {
            const int4 w = in_items[gi];
            if (w.z == 0) continue;  // an empty range (a stop that did not fit)
            g = w.x;
            if (w.z > 0) start = make_int2(w.y, w.z);
        } else {
            g = tv.group_order[gi];
        }
        if (full) {
            resume_item(P, g, start);
            continue;
        }
        const uint4 *crow = reinterpret_cast<const uint4 *>(tv.bits + (size_t)tv.group_begin[g] * tv.wp);
        __syncwarp();
        for (int k = lane; k < nq; k += 32) cen[k] = crow[k];
        __syncwarp();
        const int add = qp.lev_k + (int)tv.group_radius[g];
        auto tester = [&](int v, int take) {
            if (lane >= take) return false;
            const int k = add + (int)tv.radius[v];
            const uint4 *row = reinterpret_cast<const uint4 *>(tv.bits + (size_t)tv.node_begin[v] * tv.wp);
            return ham_rows(cen, row, nq) <= k;
        };
        const unsigned long long e0 = evals;
        const int qlo = qp.half ? tv.group_begin[g] : 0;
        const int ws = walk_group(tv, stack, cap, g, qlo, start, P, pc, evals, err, sp, tester);
        if (ws < 0) return;
        full = ws == POOL_STOPPED;
        if (gvisit) group_visits(gvisit, g, evals - e0);
        __syncwarp();
    }
    if (lane == 0) cursors[blockIdx.x] = make_longlong2(pc.cur, pc.fill);
    for (int o = 16; o > 0; o >>= 1) evals += __shfl_xor_sync(0xffffffffu, evals, o);
    if (lane == 0) stat_add(st, ST_TRAV, evals);
}

// ------------------------------------------------------------ leaf tiles

// Packs the next run of candidate points into a tile of up to 32 rows, with one
// warp.  The candidates of a group are leaf blocks of a few points each; rows
// of consecutive candidates are concatenated so that every tile is full.
// (ci, off) is the cursor: candidate index and the number of its points already
// consumed.  Returns the rows; lane r < rows gets row r's position and
// candidate.  In the emit pass, candidates without the "produced an edge" flag
// are skipped.
__device__ __forceinline__ int tile_rows(const TreeView &tv, const uint32_t *__restrict__ cand, int64_t c1,
                                         bool flagged_only, int64_t &ci, int &off, int &pos, int64_t &pcand) {
    const int lane = threadIdx.x & 31;
    const int64_t c = ci + lane;
    int beg = 0, cnt = 0;
    if (c < c1) {
        uint32_t e = cand[c];
        if (!flagged_only || (e & FLAG)) {
            int v = (int)(e & ~FLAG);
            beg = tv.node_begin[v];
            cnt = tv.node_count[v];
        }
    }
    if (lane == 0) {
        beg += off;
        cnt -= off;
    }
    int incl = cnt;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        int y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
    }
    const int excl = incl - cnt;
    const int total = __shfl_sync(0xffffffffu, incl, 31);
    const int rows = total < 32 ? total : 32;
    // owner of row r = lane: number of candidates whose inclusive end is <= r
    int L = 0;
#pragma unroll
    for (int step = 16; step >= 1; step >>= 1) {
        int probe = __shfl_sync(0xffffffffu, incl, L + step - 1);
        if (probe <= lane) L += step;
    }
    const int bl = __shfl_sync(0xffffffffu, beg, L);
    const int el = __shfl_sync(0xffffffffu, excl, L);
    pos = bl + (lane - el);
    pcand = ci + L;
    const int L31 = __shfl_sync(0xffffffffu, L, 31);
    const int e31 = __shfl_sync(0xffffffffu, excl, L31);
    const int n31 = __shfl_sync(0xffffffffu, cnt, L31);
    if (total <= 32) {
        ci = ci + 32 < c1 ? ci + 32 : c1;
        off = 0;
    } else {
        const int used = 32 - e31;
        if (used == n31) {
            ci += L31 + 1;
            off = 0;
        } else {
            off = (L31 == 0 ? off : 0) + used;
            ci += L31;
        }
    }
    return rows;
}

// The same by warp 0 for a block: the cursor and the tile in shared memory.
__device__ __forceinline__ void fill_tile(const TreeView &tv, const uint32_t *__restrict__ cand, int64_t c1,
                                          bool flagged_only, int64_t *s_ci, int *s_off, int *s_rows,
                                          int *tpos, int64_t *tcand) {
    const int lane = threadIdx.x & 31;
    int64_t ci = *s_ci, pc;
    int off = *s_off, pos;
    __syncwarp();
    const int rows = tile_rows(tv, cand, c1, flagged_only, ci, off, pos, pc);
    if (lane < rows) {
        tpos[lane] = pos;
        tcand[lane] = pc;
    }
    if (lane == 0) {
        *s_ci = ci;
        *s_off = off;
        *s_rows = rows;
    }
}

// Loads rows (K chunk kc0 .. kc0 + 4 kq floats) into a padded shared tile;
// row r comes from position pos[r] (or first + r when pos is null); rows
// beyond `rows` are zero.
template <int KS4>
__device__ __forceinline__ void load_rows(float4 *__restrict__ tile, const float *__restrict__ pts, int dp,
                                          const int *pos, int first, int rows, int kc0, int kq) {
    for (int i = threadIdx.x; i < 32 * kq; i += LEAF_T) {
        int r = i / kq, k = i - r * kq;
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
        if (r < rows) {
            int p = pos ? pos[r] : first + r;
            v = __ldg(reinterpret_cast<const float4 *>(pts + (size_t)p * dp + kc0) + k);
        }
        tile[r * KS4 + k] = v;
    }
}

constexpr int NB = 128;       // candidate leaf blocks per batch
constexpr int GQ_CAP = 1088;  // guard-band queue: <= 63 carried + 1024 from one tile
constexpr int RCAP = 512;     // packed rows mapped to positions at a time

__device__ __forceinline__ void cp_async16(void *smem, const void *gmem, bool valid) {
    unsigned sa = (unsigned)__cvta_generic_to_shared(smem);
    int n = valid ? 16 : 0;  // 0: the 16 bytes are zero-filled, nothing is read
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(sa), "l"(gmem), "r"(n));
}
__device__ __forceinline__ void cp_async16_at(uint32_t smem, const void *gmem) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(smem), "l"(gmem));
}
// 4-byte copy through L1 (cp.async.cg takes 16-byte copies only)
__device__ __forceinline__ void cp_async4(void *smem, const void *gmem) {
    unsigned sa = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(sa), "l"(gmem));
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::); }
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;\n" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;\n" ::"n"(N)); }

// Squared distances of the 2 x 4 pairs owned by this thread: queries qi and
// qi + 16 of the Q tile against rows pj, pj+8, pj+16, pj+24 of the P tile,
// whose positions are prow[0..npr).  Coordinates are summed in chunks of 16
// (FMA per term) and the chunk sums added into the total.  Contains barriers;
// every thread of the block calls it.  On return the P tile is loaded and
// every thread is past its last read of Qs/Ps for this call.
template <int KS4>
__device__ __forceinline__ void tile_accumulate(const float4 *Qs, const float4 *Ps, int kq, float (&tot)[2][4]);

template <int KS4>
__device__ __forceinline__ void tile_sqdist(const TreeView &tv, float4 *Qs, float4 *Ps, const int *prow, int npr,
                                            int qfirst, int nqr, int nkc, float (&tot)[2][4]) {
    const int dp = tv.dp;
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) tot[i][j] = 0.f;
    for (int kc = 0; kc < nkc; ++kc) {
        const int k0 = kc * KC;
        const int kq = min(KC, dp - k0) >> 2;
        if (kc > 0) __syncthreads();
        if (nkc > 1) load_rows<KS4>(Qs, tv.pts, dp, nullptr, qfirst, nqr, k0, kq);
        load_rows<KS4>(Ps, tv.pts, dp, prow, 0, npr, k0, kq);
        __syncthreads();
        tile_accumulate<KS4>(Qs, Ps, kq, tot);  // KC is a multiple of 16: chunks line up across K chunks
    }
}

// 2 x 4 micro-tile from tiles already in shared memory (rows of kq float4).
// Per chunk of 16 coordinates two packed partial sums of 8 terms each (even
// and odd coordinates) are formed with FMA, added, and the chunk sum is added
// into the running total: fp32 error of the squared distance <= ~19 u for
// rows of 128 floats (u = 2^-24).
template <int KS4>
__device__ __forceinline__ void tile_accumulate(const float4 *Qs, const float4 *Ps, int kq, float (&tot)[2][4]) {
    const int tid = threadIdx.x, qi = tid >> 3, pj = tid & 7;
    const ulonglong2 *qa[2] = {reinterpret_cast<const ulonglong2 *>(Qs + qi * KS4),
                               reinterpret_cast<const ulonglong2 *>(Qs + (qi + 16) * KS4)};
    const ulonglong2 *pr[4] = {reinterpret_cast<const ulonglong2 *>(Ps + pj * KS4),
                               reinterpret_cast<const ulonglong2 *>(Ps + (pj + 8) * KS4),
                               reinterpret_cast<const ulonglong2 *>(Ps + (pj + 16) * KS4),
                               reinterpret_cast<const ulonglong2 *>(Ps + (pj + 24) * KS4)};
    int k4 = 0;
    for (; k4 + 4 <= kq; k4 += 4) {
        unsigned long long acc[2][4];
#pragma unroll
        for (int i = 0; i < 2; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) acc[i][j] = 0ull;
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const ulonglong2 a0 = qa[0][k4 + u], a1 = qa[1][k4 + u];
            const ulonglong2 b[4] = {pr[0][k4 + u], pr[1][k4 + u], pr[2][k4 + u], pr[3][k4 + u]};
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                acc[0][j] = f2_sqacc(f2_sub(a0.x, b[j].x), acc[0][j]);
                acc[0][j] = f2_sqacc(f2_sub(a0.y, b[j].y), acc[0][j]);
                acc[1][j] = f2_sqacc(f2_sub(a1.x, b[j].x), acc[1][j]);
                acc[1][j] = f2_sqacc(f2_sub(a1.y, b[j].y), acc[1][j]);
            }
        }
#pragma unroll
        for (int i = 0; i < 2; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) tot[i][j] += f2_sum(acc[i][j]);
    }
    if (k4 < kq) {  // rows whose length is not a multiple of 16 floats
        unsigned long long acc[2][4];
#pragma unroll
        for (int i = 0; i < 2; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) acc[i][j] = 0ull;
        for (int k = k4; k < kq; ++k) {
            const ulonglong2 a0 = qa[0][k], a1 = qa[1][k];
            const ulonglong2 b[4] = {pr[0][k], pr[1][k], pr[2][k], pr[3][k]};
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                acc[0][j] = f2_sqacc(f2_sub(a0.x, b[j].x), acc[0][j]);
                acc[0][j] = f2_sqacc(f2_sub(a0.y, b[j].y), acc[0][j]);
                acc[1][j] = f2_sqacc(f2_sub(a1.x, b[j].x), acc[1][j]);
                acc[1][j] = f2_sqacc(f2_sub(a1.y, b[j].y), acc[1][j]);
            }
        }
#pragma unroll
        for (int i = 0; i < 2; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) tot[i][j] += f2_sum(acc[i][j]);
    }
}

template <int KS4>
__device__ __forceinline__ void tile_sqdist_smem(const float4 *Qs, const float4 *Ps, int kq, float (&tot)[2][4]) {
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) tot[i][j] = 0.f;
    tile_accumulate<KS4>(Qs, Ps, kq, tot);
}

// pair_sqdist with both rows in shared memory (plain loads).
__device__ __forceinline__ float pair_sqdist_smem(const float4 *x, const float4 *y, int nq4) {
    float tot = 0.f;
    int k = 0;
    for (; k + 4 <= nq4; k += 4) {
        float lo = 0.f, hi = 0.f;
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const float4 a = x[k + u], b = y[k + u];
            const float dx = a.x - b.x, dy = a.y - b.y, dz = a.z - b.z, dw = a.w - b.w;
            lo = fmaf(dx, dx, lo);
            hi = fmaf(dy, dy, hi);
            lo = fmaf(dz, dz, lo);
            hi = fmaf(dw, dw, hi);
        }
        tot += lo + hi;
    }
    if (k < nq4) {
        float lo = 0.f, hi = 0.f;
        for (; k < nq4; ++k) {
            const float4 a = x[k], b = y[k];
            const float dx = a.x - b.x, dy = a.y - b.y, dz = a.z - b.z, dw = a.w - b.w;
            lo = fmaf(dx, dx, lo);
            hi = fmaf(dy, dy, hi);
            lo = fmaf(dz, dz, lo);
            hi = fmaf(dw, dw, hi);
        }
        tot += lo + hi;
    }
    return tot;
}

template <int KS4>
struct LeafShared {
    float4 Qs[32 * KS4];
    float4 Ps[2][32 * KS4];
    int bbeg[NB], bcnt[NB], bpre[NB + 1];
    uint32_t bmask[NB], bem[NB];
    float brad[NB];
    int64_t bci[NB];
    int rpos[RCAP];
    uint8_t rli[RCAP];
    int64_t rowb[32], rowe[32];
    int cursor[32], qcnt[32];
    int gpos[GQ_CAP];
    uint8_t gq[GQ_CAP], gb[GQ_CAP];
    int gn, nb_fill, scan_tmp[LEAF_T / 32];
    uint32_t selm;
    int64_t next_ci;
    int tpre[33];  // emit pass: pairs per row of the current tile (exclusive prefix)
};
constexpr size_t leaf_smem(bool shorts) {
    return shorts ? sizeof(LeafShared<KS_SHORT>) : sizeof(LeafShared<KS_LONG>);
}

// One CTA per query group; queries in chunks of 32 (Q tile), candidate leaf
// blocks in batches of NB.  Per batch:
//  stage 1 (count pass) -- Algorithm 3's own test per query,
//             d(q, c_v) <= r(v) + eps, for every (query, candidate block) pair,
//             as dense 32 x 32 tiles of query rows against block centres; it
//             gives each block the mask of queries that still need it (a
//             pruned pair cannot hold an edge);
//  stage 2 -- the points of blocks with a non-empty mask, packed into 32-row
//             tiles (double buffered with cp.async); pairs outside the block's
//             mask are skipped.
// The emit pass skips stage 1: the count pass leaves, per candidate block,
// the mask of queries that found an edge in it, and the emit pass batches only
// blocks whose mask is non-empty.  Pairs that the fp32 value cannot decide
// (decide32) are queued and decided in FP64 by whole warps.
// A work item: a slice of at most kItem candidate blocks of one query group.
// Heavy groups (large candidate lists) are spread over several CTAs.
constexpr int kItem = 512;
constexpr int kItemTC = 1024;  // the tensor-core leaf kernel's work items (precision 1)
struct Items {
    const int32_t *group;
    const int64_t *begin, *end;
    const int32_t *count;  // device: number of items
};

// The items of a wave, in increasing order: part `part` of `parts` interleaved
// parts of all items, of every WAVE_SAMPLE-th (the sample that sizes the other
// waves), or of those not in the sample.
constexpr int WAVE_SAMPLE = 32;
struct ItemWave {
    int sampled;  // 0: of all items; 1: the sample; 2: of the rest
    int part, parts;
    __host__ __device__ int64_t item(int64_t i) const {
        const int64_t j = i * parts + part;
        if (sampled == 1) return j * WAVE_SAMPLE;
        return sampled == 2 ? j + j / (WAVE_SAMPLE - 1) + 1 : j;
    }
};

// One-pass emit (learned form): the count pass also writes every edge into a
// per-row capacity region sized from the predicted degree.  A row's entries
// past its capacity go to an overflow arena as (row, slot, col, dist); once
// the arena is full the row is marked lost and re-emitted exactly later.
// off == nullptr: plain count pass.
struct CapOut {
    const int64_t *off;      // n + 1 capacity offsets by original id
    int32_t *fill;           // entries produced per row (ends equal to the degree)
    uint2 *ent;              // capacity region: (col, distance bits)
    uint4 *ovf;              // arena: (row, slot, col, distance bits)
    unsigned long long *ovf_n;
    int64_t ovf_cap;
    uint8_t *lost;
};

// Writes entry `slot` of row o: in the row's capacity, else in the arena.
__device__ __forceinline__ void cap_place(const CapOut &co, int o, int slot, int32_t c, float d) {
    const int64_t b = co.off[o];
    if (slot < co.off[o + 1] - b) {
        co.ent[b + slot] = make_uint2((uint32_t)c, __float_as_uint(d));
        return;
    }
    const unsigned long long k = atomicAdd(co.ovf_n, 1ull);
    if ((int64_t)k < co.ovf_cap) co.ovf[k] = make_uint4((uint32_t)o, (uint32_t)slot, (uint32_t)c, __float_as_uint(d));
    else co.lost[o] = 1;
}
__device__ __forceinline__ void cap_put(const CapOut &co, int o, int32_t c, float d) {
    cap_place(co, o, atomicAdd(&co.fill[o], 1), c, d);
}

// A pair (global positions: the cloud's first row + tree position; the top
// bit of y: a mirrored edge of the upper-triangle form).
constexpr uint32_t PAIR_NONE = 0xffffffffu, PAIR_MIRROR = 0x80000000u;
struct PairList {
    uint2 *e;
    int64_t cap;
    unsigned long long *n;      // entries reserved (may exceed cap: the rest was not stored)
    unsigned long long *stat;   // tensor-core filter: valid pairs, kept pairs, rows
};
// A warp's part of the list: it reserves l2_chunk entries at a time and marks
// what it leaves of the last ones (k_leaf_l2).
constexpr int l2_chunk(bool shorts) { return shorts ? 128 : 32; }
struct PairCursor {
    int64_t cur = 0, lim = 0;
};
// Appends n entries of the warp (each lane's from `at` of them on); room(i)
// gives entry i's place.
struct PairPlaces {
    int64_t old, nxt;
    int room;
    __device__ __forceinline__ int64_t operator()(int i) const { return i < room ? old + i : nxt + (i - room); }
};
template <int CHUNK>
__device__ __forceinline__ PairPlaces pair_reserve(const PairList &pl, PairCursor &pc, int n) {
    PairPlaces p{pc.cur, 0, (int)(pc.lim - pc.cur)};
    if (n > p.room) {
        const int more = ((n - p.room + CHUNK - 1) / CHUNK) * CHUNK;
        unsigned long long a = 0;
        if ((threadIdx.x & 31) == 0) a = atomicAdd(pl.n, (unsigned long long)more);
        p.nxt = (int64_t)__shfl_sync(0xffffffffu, a, 0);
        pc.lim = p.nxt + more;
        pc.cur = p.nxt + (n - p.room);
    } else {
        pc.cur += n;
    }
    return p;
}
__device__ __forceinline__ void pair_close(const PairList &pl, const PairCursor &pc) {
    for (int64_t i = pc.cur + (threadIdx.x & 31); i < pc.lim && i < pl.cap; i += 32)
        pl.e[i] = make_uint2(PAIR_NONE, 0u);
}

// One work item of the FP32 tiles (count or emit pass), by the whole CTA.
template <bool EMIT, int KS4>
__device__ __forceinline__ void leaf_l2_item(
    const Views &V, const Items &items, const int it, const uint32_t *__restrict__ cand,
    uint32_t *__restrict__ emask, int32_t *__restrict__ deg, const int64_t *__restrict__ row_ptr,
    int32_t *__restrict__ rowcur, int32_t *__restrict__ col, float *__restrict__ dist,
    unsigned long long *__restrict__ st, int32_t *__restrict__ err, const CapOut &co,
    const uint8_t *__restrict__ rowsel, const PairList &pl, PairCursor &pc, LeafShared<KS4> &S) {
    if (it >= *items.count) return;
    const int gg = items.group[it];
    const int cloud = cloud_of_group(V, gg);
    const TreeView &tv = V.tv[cloud];
    const QParams &qp = V.qp[cloud];
    const int g = gg - V.gbase[cloud];
    const int64_t rbase = V.rbase[cloud];  // CSR rows of this cloud start here
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int qi = tid >> 3, pj = tid & 7;
    const int dp = tv.dp, dim = tv.dim;
    const int nkc = (dp + KC - 1) / KC;
    const int kq = dp >> 2;  // float4 per row when nkc == 1
    const unsigned kq_inv = (65536u + kq - 1) / kq;  // i / kq = i * kq_inv >> 16: the excess stays below 1024 / 65536 < 1 / kq
    const bool fp32_dist_ok = dp <= 128;
    const int qb = tv.group_begin[g], qn = tv.group_count[g];
    const int qe = qb + qn;       // the group's positions: [qb, qe)
    const bool half = qp.half != 0;
    const int64_t c0 = items.begin[it], c1 = items.end[it];
    unsigned long long pairs = 0, s1evals = 0, guard = 0, band = 0, rows_ld = 0;  // rows_ld: thread 0
    // upper-triangle form: an edge (q, p) with p in a later group is also the
    // edge (p, q) of p's row -- its degree (count pass, with the one-pass
    // emit's entry) or its entry (emit pass; only a selected row when rows
    // are emitted again)
    auto mirror = [&](int qpos, int ppos, float d) {
        const int64_t o = rbase + tv.perm[ppos];
        if (!EMIT) {
            atomicAdd(&deg[o], 1);
            if (co.off) cap_put(co, (int)o, tv.perm[qpos], d);
        } else {
            if (rowsel && !rowsel[o]) return;
            const int slot = atomicAdd(&rowcur[o], 1);
            const int64_t at = row_ptr[o] + slot;
            if (at < row_ptr[o + 1]) {
                col[at] = tv.perm[qpos];
                dist[at] = d;
            } else {
                atomicOr(err, 4);
            }
        }
    };

    for (int q0 = 0; q0 < qn; q0 += 32) {
        const int nqr = min(32, qn - q0);
        const int qfirst = qb + q0;
        auto pair_of = [&](int q, int ppos) {
            return make_uint2((uint32_t)(rbase + qfirst + q),
                              (uint32_t)(rbase + ppos) | (half && ppos >= qe ? PAIR_MIRROR : 0u));
        };
        __syncthreads();
        if (tid < 32) {
            S.qcnt[tid] = 0;
            bool sel = false;
            if (tid < nqr) {
                const int64_t o = rbase + tv.perm[qfirst + tid];
                S.cursor[tid] = (int)o;  // row of the query in the (concatenated) CSR
                if (EMIT) {
                    S.rowb[tid] = row_ptr[o];
                    S.rowe[tid] = row_ptr[o + 1];
                    sel = rowsel == nullptr || rowsel[o] != 0;
                }
            }
            // emit pass: queries whose rows are written (all, or the selected ones)
            const unsigned sm = __ballot_sync(0xffffffffu, sel);
            if (tid == 0) S.selm = sm;
        }
        if (tid == 0) S.gn = 0;
        int cnt0 = 0, cnt1 = 0;
        if (nkc == 1) load_rows<KS4>(S.Qs, tv.pts, dp, nullptr, qfirst, nqr, 0, kq);

        // decides the queued guard-band pairs; `all` drains everything, else
        // whole warps' worth and keeps the rest
        auto drain = [&](bool all) {
            __syncthreads();
            const int n = S.gn;
            const int m = all ? n : (n & ~31);
            for (int i = tid; i < m; i += LEAF_T) {
                const int q = S.gq[i], ppos = S.gpos[i], li = S.gb[i];
                if (!EMIT) {
                    ++guard;
                    note_guard_rows(S.cursor[q], (int32_t)(rbase + tv.perm[ppos]));
                }
                double s64 = sq_l2_exact(tv.pts + (size_t)(qfirst + q) * dp, tv.pts + (size_t)ppos * dp, dim);
                if (s64 <= qp.eps2_64) {
                    if (half && ppos >= qe) mirror(qfirst + q, ppos, (float)sqrt(s64));
                    if (!EMIT) {
                        atomicAdd(&S.qcnt[q], 1);
                        atomicOr(&S.bem[li], 1u << q);
                        if (pl.e) {  // few: an entry of its own each
                            const int64_t at = (int64_t)atomicAdd(pl.n, 1ull);
                            if (at < pl.cap) pl.e[at] = pair_of(q, ppos);
                        }
                        if (co.off) cap_put(co, S.cursor[q], tv.perm[ppos], (float)sqrt(s64));
                    } else if ((S.selm >> q) & 1u) {
                        int slot = atomicAdd(&rowcur[S.cursor[q]], 1);
                        int64_t at = S.rowb[q] + slot;
                        if (at < S.rowe[q]) {
                            col[at] = tv.perm[ppos];
                            dist[at] = (float)sqrt(s64);
                        } else {
                            atomicOr(err, 4);
                        }
                    }
                }
            }
            __syncthreads();
            const int rest = n - m;
            int rp = 0, rq = 0, rb = 0;
            if (tid < rest) {
                rp = S.gpos[m + tid];
                rq = S.gq[m + tid];
                rb = S.gb[m + tid];
            }
            __syncthreads();
            if (tid < rest) {
                S.gpos[tid] = rp;
                S.gq[tid] = (uint8_t)rq;
                S.gb[tid] = (uint8_t)rb;
            }
            if (tid == 0) S.gn = rest;
            __syncthreads();
        };

        // issues the cp.async copies of tile t (rows rowsrc[32t ..]) into buffer buf
        auto issue = [&](int t, int buf, const int *rowsrc, int nrows) {
            if (nkc != 1) return;
            const int r0 = 32 * t;
            const int rows = min(32, nrows - r0);
            float4 *dst = S.Ps[buf];
            for (int i = tid; i < 32 * kq; i += LEAF_T) {
                const int r = (int)(((unsigned)i * kq_inv) >> 16), k = i - r * kq;  // i / kq (i < 1024, kq <= 32)
                const bool valid = r < rows;
                const int pos = valid ? rowsrc[r0 + r] : qfirst;
                cp_async16(dst + r * KS4 + k, tv.pts + (size_t)pos * dp + 4 * k, valid);
            }
            cp_async_commit();
        };
        auto compute = [&](int t, int buf, const int *rowsrc, int nrows, float (&tot)[2][4]) {
            if (nkc == 1) {
                tile_sqdist_smem<KS4>(S.Qs, S.Ps[buf], kq, tot);
            } else {
                const int r0 = 32 * t;
                tile_sqdist<KS4>(tv, S.Qs, S.Ps[0], rowsrc + r0, min(32, nrows - r0), qfirst, nqr, nkc, tot);
            }
        };

        int64_t ci = c0;
        while (ci < c1) {
            // ---- batch of candidate blocks
            int bn;
            if (EMIT) {
                __syncthreads();
                if (tid == 0) S.nb_fill = 0;
                __syncthreads();
                for (;;) {
                    const int nf = S.nb_fill;
                    if (nf >= NB || ci >= c1) break;
                    const int64_t idx = ci + tid;
                    // (rows emitted again in the upper-triangle form: every query, as a
                    // selected row can be the mirror of another query's edge)
                    const uint32_t m = idx < c1 ? (emask[idx] & (half && rowsel ? 0xffffffffu : S.selm)) : 0u;
                    const bool f = m != 0u;
                    const unsigned bal = __ballot_sync(0xffffffffu, f);
                    if (lane == 0) S.scan_tmp[warp] = __popc(bal);
                    __syncthreads();
                    int off = 0, tot = 0;
#pragma unroll
                    for (int w = 0; w < LEAF_T / 32; ++w) {
                        if (w < warp) off += S.scan_tmp[w];
                        tot += S.scan_tmp[w];
                    }
                    const int rank = off + __popc(bal & lanemask_lt());
                    const int room = NB - nf;
                    if (f && rank < room) {
                        S.bci[nf + rank] = idx;
                        S.bmask[nf + rank] = m;
                    }
                    if (f && rank == room) S.next_ci = idx;
                    __syncthreads();
                    if (tot <= room) ci = ci + LEAF_T < c1 ? ci + LEAF_T : c1;
                    else ci = S.next_ci;
                    if (tid == 0) S.nb_fill = nf + (tot < room ? tot : room);
                    __syncthreads();
                }
                bn = S.nb_fill;
                if (bn == 0) break;
            } else {
                bn = (int)((c1 - ci) < NB ? (c1 - ci) : NB);
                if (tid < NB) S.bci[tid] = ci + tid;
                ci += bn;
            }
            __syncthreads();
            for (int i = tid; i < bn; i += LEAF_T) {
                const int v = (int)cand[S.bci[i]];
                S.bbeg[i] = tv.node_begin[v];
                S.bcnt[i] = tv.node_count[v];
                S.brad[i] = tv.radius[v];
                if (!EMIT) S.bmask[i] = 0u;
                S.bem[i] = 0u;
            }
            __syncthreads();

            // ---- stage 1 (count pass): per-query test against the block centres
            if (!EMIT) {
                const int nt = (bn + 31) >> 5;
                if (tid == 0) rows_ld += bn;
                issue(0, 0, S.bbeg, bn);
                for (int t = 0; t < nt; ++t) {
                    if (t + 1 < nt) {
                        issue(t + 1, (t + 1) & 1, S.bbeg, bn);
                        cp_async_wait<1>();
                    } else {
                        cp_async_wait<0>();
                    }
                    __syncthreads();
                    float tot[2][4];
                    compute(t, t & 1, S.bbeg, bn, tot);
                    const int rows = min(32, bn - 32 * t);
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const int p = pj + 8 * j;
                        if (p >= rows) continue;
                        const int li = 32 * t + p;
                        const float bound = fmaf(S.brad[li] + qp.eps_up, PRUNE_REL, PRUNE_ABS);
                        uint32_t m = 0u;
#pragma unroll
                        for (int i = 0; i < 2; ++i) {
                            const int q = qi + 16 * i;
                            if (q >= nqr) continue;
                            ++s1evals;
                            if (!(sqrtf(tot[i][j]) > bound)) m |= 1u << q;
                        }
                        if (m) atomicOr(&S.bmask[li], m);
                    }
                    __syncthreads();
                }
            }

            // ---- prefix over the batch (warp 0): count pass -- points of the
            // surviving blocks; emit pass -- (query, point) pairs to evaluate
            const uint32_t qvalid = nqr >= 32 ? 0xffffffffu : ((1u << nqr) - 1u);
            if (warp == 0) {
                int loc[4], sum = 0;
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const int i = 4 * lane + k;
                    if (EMIT && nkc > 1) loc[k] = i < bn ? __popc(S.bmask[i] & qvalid) * S.bcnt[i] : 0;
                    else loc[k] = (i < bn && (S.bmask[i] & qvalid) != 0u) ? S.bcnt[i] : 0;
                    sum += loc[k];
                }
                int incl = sum;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    int y = __shfl_up_sync(0xffffffffu, incl, o);
                    if (lane >= o) incl += y;
                }
                int run = incl - sum;
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    S.bpre[4 * lane + k] = run;
                    run += loc[k];
                }
                if (lane == 31) S.bpre[NB] = incl;
            }
            __syncthreads();
            const int T = S.bpre[NB];

            // ---- emit pass: one thread per (query, point) pair of the blocks in
            // which the query found an edge; same arithmetic as the tiles;
            // undecided pairs go through the FP64 queue
            if (EMIT && nkc > 1) {
                for (int r0 = 0; r0 < T; r0 += LEAF_T) {
                    const int r = r0 + tid;
                    if (r < T) {
                        int lo = 0, hi = NB;
                        while (hi - lo > 1) {
                            const int mid = (lo + hi) >> 1;
                            if (S.bpre[mid] <= r) lo = mid; else hi = mid;
                        }
                        const int idx = r - S.bpre[lo], cnt = S.bcnt[lo];
                        const int qr = idx / cnt, pidx = idx - qr * cnt;
                        const int q = (int)__fns(S.bmask[lo] & qvalid, 0u, qr + 1);
                        const int qpos = qfirst + q, ppos = S.bbeg[lo] + pidx;
                        if ((qpos != ppos || qp.include_self) && !(half && ppos < qb)) {
                            ++pairs;
                            const float4 *qrow = reinterpret_cast<const float4 *>(tv.pts + (size_t)qpos * dp);
                            const float sv = pair_sqdist(qrow, reinterpret_cast<const float4 *>(tv.pts + (size_t)ppos * dp),
                                                         dp >> 2);
                            const int edge = decide32(qp, sv, band);
                            if (edge < 0) {
                                const int slot = atomicAdd(&S.gn, 1);
                                S.gpos[slot] = ppos;
                                S.gq[slot] = (uint8_t)q;
                                S.gb[slot] = (uint8_t)lo;
                            } else if (edge) {
                                const float d = fp32_dist_ok ? sqrtf(sv)
                                                             : (float)sqrt(sq_l2_exact(tv.pts + (size_t)qpos * dp,
                                                                                       tv.pts + (size_t)ppos * dp, dim));
                                if (half && ppos >= qe) mirror(qpos, ppos, d);
                                if ((S.selm >> q) & 1u) {
                                    const int slot = atomicAdd(&rowcur[S.cursor[q]], 1);
                                    const int64_t at = S.rowb[q] + slot;
                                    if (at < S.rowe[q]) {
                                        col[at] = tv.perm[ppos];
                                        dist[at] = d;
                                    } else {
                                        atomicOr(err, 4);
                                    }
                                }
                            }
                        }
                    }
                    __syncthreads();
                    if (S.gn >= 64) drain(false);
                }
            }

            // ---- stage 2: packed points of the surviving blocks (count pass: dense
            // 32 x 32 tiles; emit pass: only the (query, row) pairs of each tile
            // whose block holds an edge of the query)
            for (int R0 = 0; (!EMIT || nkc == 1) && R0 < T; R0 += RCAP) {
                const int RN = min(RCAP, T - R0);
                if (!EMIT && tid == 0) rows_ld += RN;
                __syncthreads();
                for (int r = tid; r < RN; r += LEAF_T) {
                    const int R = R0 + r;
                    int lo = 0, hi = NB;  // last li with bpre[li] <= R (and a non-empty block)
                    while (hi - lo > 1) {
                        const int mid = (lo + hi) >> 1;
                        if (S.bpre[mid] <= R) lo = mid; else hi = mid;
                    }
                    S.rpos[r] = S.bbeg[lo] + (R - S.bpre[lo]);
                    S.rli[r] = (uint8_t)lo;
                }
                __syncthreads();
                const int nt = (RN + 31) >> 5;
                issue(0, 0, S.rpos, RN);
                for (int t = 0; t < nt; ++t) {
                    if (t + 1 < nt) {
                        issue(t + 1, (t + 1) & 1, S.rpos, RN);
                        cp_async_wait<1>();
                    } else {
                        cp_async_wait<0>();
                    }
                    __syncthreads();
                    const int npr = min(32, RN - 32 * t);
                    if (EMIT) {
                        // pairs of this tile: row r pairs with the queries of its block's mask
                        if (warp == 0) {
                            const int c = lane < npr ? __popc(S.bmask[S.rli[32 * t + lane]] & qvalid) : 0;
                            int incl = c;
#pragma unroll
                            for (int o = 1; o < 32; o <<= 1) {
                                int y = __shfl_up_sync(0xffffffffu, incl, o);
                                if (lane >= o) incl += y;
                            }
                            S.tpre[lane] = incl - c;
                            if (lane == 31) S.tpre[32] = incl;
                        }
                        __syncthreads();
                        const int TP = S.tpre[32];
                        const float4 *Pb = S.Ps[t & 1];
                        for (int pi = tid; pi < TP; pi += LEAF_T) {
                            int lo = 0, hi = 32;
                            while (hi - lo > 1) {
                                const int mid = (lo + hi) >> 1;
                                if (S.tpre[mid] <= pi) lo = mid; else hi = mid;
                            }
                            const int r = 32 * t + lo;
                            const int li = S.rli[r];
                            const int q = (int)__fns(S.bmask[li] & qvalid, 0u, pi - S.tpre[lo] + 1);
                            const int qpos = qfirst + q, ppos = S.rpos[r];
                            if (qpos == ppos && !qp.include_self) continue;
                            if (half && ppos < qb) continue;
                            ++pairs;
                            const float sv = pair_sqdist_smem(S.Qs + q * KS4, Pb + lo * KS4, kq);
                            const int edge = decide32(qp, sv, band);
                            if (edge < 0) {
                                const int slot = atomicAdd(&S.gn, 1);
                                S.gpos[slot] = ppos;
                                S.gq[slot] = (uint8_t)q;
                                S.gb[slot] = (uint8_t)li;
                            } else if (edge) {
                                if (half && ppos >= qe) mirror(qpos, ppos, sqrtf(sv));
                                if ((S.selm >> q) & 1u) {
                                    const int slot = atomicAdd(&rowcur[S.cursor[q]], 1);
                                    const int64_t at = S.rowb[q] + slot;
                                    if (at < S.rowe[q]) {
                                        col[at] = tv.perm[ppos];
                                        dist[at] = sqrtf(sv);
                                    } else {
                                        atomicOr(err, 4);
                                    }
                                }
                            }
                        }
                        __syncthreads();
                        if (S.gn >= 64) drain(false);
                        continue;
                    }
                    float tot[2][4];
                    compute(t, t & 1, S.rpos, RN, tot);
                    uint32_t hitrow = 0u;
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const int p = pj + 8 * j;
                        if (p >= npr) continue;
                        const int r = 32 * t + p;
                        const int li = S.rli[r];
                        const uint32_t mask = S.bmask[li];
                        const int ppos = S.rpos[r];
#pragma unroll
                        for (int i = 0; i < 2; ++i) {
                            const int q = qi + 16 * i;
                            if (q >= nqr || !((mask >> q) & 1u)) continue;
                            const int qpos = qfirst + q;
                            if (qpos == ppos && !qp.include_self) continue;
                            if (half && ppos < qb) continue;
                            if (!EMIT) ++pairs;
                            const float sv = tot[i][j];
                            const int edge = decide32(qp, sv, band);
                            if (edge < 0) {  // undecided in fp32: queue for the FP64 decision
                                const int slot = atomicAdd(&S.gn, 1);
                                S.gpos[slot] = ppos;
                                S.gq[slot] = (uint8_t)q;
                                S.gb[slot] = (uint8_t)li;
                                continue;
                            }
                            if (!edge) continue;
                            const bool want_d = co.off || EMIT || (half && ppos >= qe);
                            const float d = !want_d ? 0.f
                                            : fp32_dist_ok ? sqrtf(sv)
                                                           : (float)sqrt(sq_l2_exact(tv.pts + (size_t)qpos * dp,
                                                                                     tv.pts + (size_t)ppos * dp, dim));
                            if (half && ppos >= qe) mirror(qpos, ppos, d);
                            if (!EMIT) {
                                if (i == 0) ++cnt0; else ++cnt1;
                                hitrow |= 1u << (4 * j + i);
                                if (co.off) cap_put(co, S.cursor[q], tv.perm[ppos], d);
                            } else if ((S.selm >> q) & 1u) {
                                const int slot = atomicAdd(&rowcur[S.cursor[q]], 1);
                                const int64_t at = S.rowb[q] + slot;
                                if (at < S.rowe[q]) {
                                    col[at] = tv.perm[ppos];
                                    dist[at] = d;
                                } else {
                                    atomicOr(err, 4);
                                }
                            }
                        }
                    }
                    if (!EMIT && pl.e && __any_sync(0xffffffffu, hitrow != 0u)) {  // the edges, for the emit pass
                        const int c = __popc(hitrow);
                        int incl = c;
#pragma unroll
                        for (int o = 1; o < 32; o <<= 1) {
                            const int y = __shfl_up_sync(0xffffffffu, incl, o);
                            if (lane >= o) incl += y;
                        }
                        const PairPlaces place =
                            pair_reserve<l2_chunk(KS4 == KS_SHORT)>(pl, pc, __shfl_sync(0xffffffffu, incl, 31));
                        uint32_t m = hitrow;
                        for (int i = incl - c; m; ++i) {
                            const int x = __ffs(m) - 1, j = x >> 2;
                            m &= m - 1u;
                            const int64_t at = place(i);
                            if (at < pl.cap) pl.e[at] = pair_of(qi + 16 * (x & 1), S.rpos[32 * t + pj + 8 * j]);
                        }
                    }
                    if (!EMIT && hitrow) {
#pragma unroll
                        for (int j = 0; j < 4; ++j) {
                            const uint32_t qm = (hitrow >> (4 * j)) & 3u;
                            if (!qm) continue;
                            uint32_t bits = 0u;
                            if (qm & 1u) bits |= 1u << qi;
                            if (qm & 2u) bits |= 1u << (qi + 16);
                            atomicOr(&S.bem[S.rli[32 * t + pj + 8 * j]], bits);
                        }
                    }
                    __syncthreads();
                    if (S.gn >= 64) drain(false);
                }
            }
            drain(true);
            // count pass: queries that found an edge in each block (all queries
            // for a group above 32 points), read by the emit pass
            if (!EMIT && emask) {
                for (int i = tid; i < bn; i += LEAF_T) emask[S.bci[i]] = qn <= 32 ? S.bem[i] : ~0u;
            }
        }
        if (!EMIT) {
            for (int o = 1; o < 8; o <<= 1) {
                cnt0 += __shfl_xor_sync(0xffffffffu, cnt0, o);
                cnt1 += __shfl_xor_sync(0xffffffffu, cnt1, o);
            }
            __syncthreads();
            if (pj == 0) {
                if (qi < nqr && cnt0 + S.qcnt[qi]) atomicAdd(&deg[S.cursor[qi]], cnt0 + S.qcnt[qi]);
                if (qi + 16 < nqr && cnt1 + S.qcnt[qi + 16])
                    atomicAdd(&deg[S.cursor[qi + 16]], cnt1 + S.qcnt[qi + 16]);
            }
        }
    }
    for (int o = 16; o > 0; o >>= 1) {
        pairs += __shfl_xor_sync(0xffffffffu, pairs, o);
        s1evals += __shfl_xor_sync(0xffffffffu, s1evals, o);
        guard += __shfl_xor_sync(0xffffffffu, guard, o);
        band += __shfl_xor_sync(0xffffffffu, band, o);
    }
    if ((tid & 31) == 0) {
        if (!EMIT) {
            stat_add(st, ST_PAIRS, pairs);
            stat_add(st, ST_TRAV, s1evals);
            stat_add(st, ST_GUARD, guard);
            stat_add(st, ST_BAND, band);
            if (tid == 0) stat_add(st, ST_ROWS, rows_ld);
        } else {
            stat_add(st, ST_EMIT, pairs);
        }
    }
}

// The wave's items.  Rows of at most 64 floats: taken dynamically by a grid of
// resident CTAs (leaf_l2_ctas), so that a warp's place in the edge list outlives
// an item.  (With a CTA per item every warp that found an edge left up to 127
// entries of its own behind: 240 thousand warps of 121k x 16 uniform points asked
// for 31 M entries to list 2.5 M edges, more than the list had.)  Longer rows,
// whose items take longer: a CTA per item, which the hardware schedules better
// (1M x 128, upper triangle: 91.5 ms, 93.9 with resident CTAs), and reservations
// of 32 entries (l2_chunk), whose leavings the list has room for.
// Rows of at most 64 floats take a shorter tile stride and fewer registers, so
// that five CTAs share an SM instead of three (a tile is a chain of copy,
// barrier, arithmetic, barrier: more of them in flight; -Xptxas -v: 96
// registers, the count form spills 32 bytes of them and reads 28 back).
// 174k x 64 at 87 neighbours: count 16.3 -> 13.7 ms, bound by the shared-memory
// reads of the micro-tiles (71 % of that pipe, four wavefronts per 16-byte
// read whatever is broadcast) and the FP32 pipe (58 %).  The emit pass reads
// the list of edges instead of the blocks' pairs: 4.8 -> 0.8 ms.
constexpr int leaf_l2_ctas(bool shorts) { return shorts ? 5 : 3; }  // of an SM
// CTAs of a launch over a wave of at most max_items items, and the list entries
// that the warps of all waves of a call (two at most) may leave unused.
int64_t leaf_l2_grid(bool shorts, int64_t max_items) {
    return shorts ? std::min<int64_t>(max_items, (int64_t)num_sms() * leaf_l2_ctas(true)) : max_items;
}
int64_t leaf_l2_slack(bool shorts, int64_t max_items) {
    return (shorts ? 2 : 1) * leaf_l2_grid(shorts, max_items) * (LEAF_T / 32) * l2_chunk(shorts);
}
template <bool EMIT, int KS4>
__global__ void __launch_bounds__(LEAF_T, leaf_l2_ctas(KS4 == KS_SHORT)) k_leaf_l2(
    const __grid_constant__ Views V, Items items, ItemWave wave, unsigned long long *__restrict__ next,
    const uint32_t *__restrict__ cand,
    uint32_t *__restrict__ emask, int32_t *__restrict__ deg, const int64_t *__restrict__ row_ptr,
    int32_t *__restrict__ rowcur, int32_t *__restrict__ col, float *__restrict__ dist,
    unsigned long long *__restrict__ st, int32_t *__restrict__ err, CapOut co, const uint8_t *__restrict__ rowsel,
    PairList pl) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    LeafShared<KS4> &S = *reinterpret_cast<LeafShared<KS4> *>(smem_raw);
    PairCursor pc;
    if constexpr (KS4 == KS_LONG) {
        // the wave's items from the block index alone (uniform registers): a CTA for every
        // 32nd item, or for every item but those, which leave at once
        const int it = (int)blockIdx.x * (wave.sampled == 1 ? WAVE_SAMPLE : 1);
        if (wave.sampled == 2 && it % WAVE_SAMPLE == 0) return;
        leaf_l2_item<EMIT, KS4>(V, items, it, cand, emask, deg, row_ptr, rowcur, col, dist, st, err, co, rowsel, pl,
                                pc, S);
    } else {
        __shared__ int64_t s_it;
        for (;;) {
            __syncthreads();  // the last item is done
            if (threadIdx.x == 0) s_it = wave.item((int64_t)atomicAdd(next, 1ull));
            __syncthreads();
            const int64_t it = s_it;
            if (it >= *items.count) break;
            leaf_l2_item<EMIT, KS4>(V, items, (int)it, cand, emask, deg, row_ptr, rowcur, col, dist, st, err, co,
                                    rowsel, pl, pc, S);
        }
    }
    if (!EMIT && pl.e) pair_close(pl, pc);
}

// Work items: every pool segment split into slices of at most kItem blocks.
// The walk rounds leave a group's candidates in several pool segments; these
// copy them into one contiguous range per group (longer work items, fewer
// CTAs in the leaf pass): counts per group, then a warp per segment copies it
// to its group's range at a place taken from the group's fill counter.
__global__ void k_group_cand_counts(int nseg, const int32_t *__restrict__ seg_group,
                                    const int32_t *__restrict__ seg_count, int32_t *__restrict__ gcnt) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < nseg && seg_count[i] > 0) atomicAdd(gcnt + seg_group[i], seg_count[i]);
}
__global__ void k_group_cand_copy(int nseg, const int32_t *__restrict__ seg_group,
                                  const int64_t *__restrict__ seg_begin, const int32_t *__restrict__ seg_count,
                                  const int64_t *__restrict__ goff, int32_t *__restrict__ gfill,
                                  const uint32_t *__restrict__ pool, uint32_t *__restrict__ gcand) {
    const int i = (int)(((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5), lane = threadIdx.x & 31;
    if (i >= nseg) return;
    const int g = seg_group[i], c = seg_count[i];
    int64_t base = 0;
    if (lane == 0) base = goff[g] + atomicAdd(gfill + g, c);
    base = __shfl_sync(0xffffffffu, base, 0);
    const uint32_t *src = pool + seg_begin[i];
    for (int k = lane; k < c; k += 32) gcand[base + k] = src[k];
}

__global__ void k_iota(int n, int32_t *__restrict__ out) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) out[i] = i;
}

__global__ void k_item_counts(const __grid_constant__ Views V, int nseg, const int32_t *__restrict__ seg_group,
                              const int32_t *__restrict__ seg_count, int32_t *__restrict__ icnt) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= nseg) return;
    const int len = V.item_len[cloud_of_group(V, seg_group[i])];
    icnt[i] = (seg_count[i] + len - 1) / len;
}
__global__ void k_item_fill(const __grid_constant__ Views V, int nseg, const int32_t *__restrict__ seg_group,
                            const int64_t *__restrict__ seg_begin, const int32_t *__restrict__ seg_count,
                            const int64_t *__restrict__ ioff, int32_t *__restrict__ ig, int64_t *__restrict__ ib,
                            int64_t *__restrict__ ie, int32_t *__restrict__ nitems) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i == 0) *nitems = (int32_t)ioff[nseg];
    if (i >= nseg) return;
    const int len = V.item_len[cloud_of_group(V, seg_group[i])];
    const int64_t a = seg_begin[i], b = a + seg_count[i];
    int64_t k = ioff[i];
    for (int64_t c = a; c < b; c += len, ++k) {
        ig[k] = seg_group[i];
        ib[k] = c;
        ie[k] = c + len < b ? c + len : b;
    }
}
// Splits the items between the two count kernels by their cloud's choice.
__global__ void k_item_split(const __grid_constant__ Views V, Items all, int32_t *__restrict__ tg,
                             int64_t *__restrict__ tb, int64_t *__restrict__ te, int32_t *__restrict__ tn,
                             int32_t *__restrict__ fg, int64_t *__restrict__ fb, int64_t *__restrict__ fe,
                             int32_t *__restrict__ fn) {
    const int it = blockIdx.x * blockDim.x + threadIdx.x;
    if (it >= *all.count) return;
    const int gg = all.group[it];
    if (V.use_tc[cloud_of_group(V, gg)]) {
        const int k = atomicAdd(tn, 1);
        tg[k] = gg;
        tb[k] = all.begin[it];
        te[k] = all.end[it];
    } else {
        const int k = atomicAdd(fn, 1);
        fg[k] = gg;
        fb[k] = all.begin[it];
        fe[k] = all.end[it];
    }
}
__global__ void k_check_rows(int64_t n, const int64_t *__restrict__ row_ptr, const int32_t *__restrict__ rowcur,
                             int32_t *__restrict__ err) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n && row_ptr[i] + rowcur[i] != row_ptr[i + 1]) atomicOr(err, 8);
}
// rowsel != nullptr: only the selected rows were written.
__global__ void k_check_rows_sel(int64_t n, const int64_t *__restrict__ row_ptr, const int32_t *__restrict__ rowcur,
                                 const uint8_t *__restrict__ rowsel, int32_t *__restrict__ err) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n && rowsel[i] && row_ptr[i] + rowcur[i] != row_ptr[i + 1]) atomicOr(err, 8);
}

// One-pass emit, after the count pass: every row's produced entries must equal
// its degree (tensor-core clouds have no degrees of their own: the entries are
// the degrees, and their total is compared with the edges that k_pairs found);
// counts rows past their capacity (cnt[0]) and lost rows (cnt[1]).
__global__ void k_cap_rows(int64_t n, const int64_t *__restrict__ row_ptr, const int64_t *__restrict__ off,
                           const int32_t *__restrict__ fill, const uint8_t *__restrict__ lost,
                           unsigned long long *__restrict__ cnt, int32_t *__restrict__ err) {
    const int64_t o = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    bool ov = false, ls = false;
    if (o < n) {
        const int64_t deg = row_ptr[o + 1] - row_ptr[o];
        if ((int64_t)fill[o] != deg) atomicOr(err, 64);
        ov = deg > off[o + 1] - off[o];
        ls = lost[o] != 0;
    }
    const unsigned a = __ballot_sync(0xffffffffu, ov), b = __ballot_sync(0xffffffffu, ls);
    if ((threadIdx.x & 31) == 0) {
        if (a) atomicAdd(cnt, (unsigned long long)__popc(a));
        if (b) atomicAdd(cnt + 1, (unsigned long long)__popc(b));
    }
}

// Copies each kept row's capacity-region entries into the CSR (warp per row).
__global__ void k_compact(int64_t n, const int64_t *__restrict__ row_ptr, const int64_t *__restrict__ off,
                          const uint8_t *__restrict__ lost, const uint2 *__restrict__ ent, int32_t *__restrict__ col,
                          float *__restrict__ dist) {
    const int64_t w = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (w >= n || lost[w]) return;
    const int64_t b = off[w], cap = off[w + 1] - b, d0 = row_ptr[w], deg = row_ptr[w + 1] - d0;
    const int64_t m = deg < cap ? deg : cap;
    for (int64_t j = lane; j < m; j += 32) {
        const uint2 e = ent[b + j];
        col[d0 + j] = (int32_t)e.x;
        dist[d0 + j] = __uint_as_float(e.y);
    }
}

// Places the overflow arena's entries of kept rows at their slots.
__global__ void k_ovf_scatter(int64_t used, const uint4 *__restrict__ ovf, const uint8_t *__restrict__ lost,
                              const int64_t *__restrict__ row_ptr, int32_t *__restrict__ col,
                              float *__restrict__ dist, int32_t *__restrict__ err) {
    const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= used) return;
    const uint4 e = ovf[k];
    if (lost[e.x]) return;
    const int64_t at = row_ptr[e.x] + e.y;
    if (at >= row_ptr[e.x + 1]) {
        atomicOr(err, 128);
        return;
    }
    col[at] = (int32_t)e.z;
    dist[at] = __uint_as_float(e.w);
}

// ---------------------------------------------------------------------------
// FP16 rows for the tensor-core filter.  Each cloud's points are stored once
// per query as x^ = fp16(s fl(x - m)) (m: the column means, s: a power of two
// with s |x_k - m_k| < 2^14), rows of kp = 64 ceil(dp / 64) halves, zero
// padded, with n^ = the fp32 sum of their squares.  Rounding to nearest gives
// |x^_k - s (x_k - m_k)| <= 2^-11 (1 + 2^-10) |x^_k| + 2^-25 (the last for
// subnormal halves), so with |x^| <= sqrt(n^) (1 + 2^-16) =: a_x
//   ||x^ - y^|| <= s d(x, y) + rel (a_x + a_y) + 2^-20,  rel = 2^-11 (1 + 2^-8).
// d^2 = n^_x + n^_y - 2 x^.y^ is formed from exact fp16 products with fp32
// sums: the MMA's accumulation (K <= 128 terms, below 2^-17 (n^_x + n^_y)),
// the norms (2^-17 each) and the formula (2^-22) stay below 2^-15.9 (n^_x +
// n^_y).  A pair is kept iff
//   d^2 <= (s eps + rel (a_x + a_y) + 2^-20)^2 + 2^-14 (a_x^2 + a_y^2) + 2^-60,
// which keeps every edge with a 4x margin on the fp32 terms.  The slack
// relative to eps grows with |x - m| / eps (about 2^-10 of it); rows are
// copied into the MMA's layout unchanged, so the count pass converts nothing.
//
// Any m keeps the bound; the column means only keep |x - m| small, so they are
// taken from a strided sample of at most H16_SAMPLE points.  The three
// launches serve every cloud of a batch (a serial sum of 1024 partials per
// cloud used to take 83 us each: 1.9 ms for 20 clouds, 5.0 ms for 60, now
// 0.1 and 0.2; 1M x 128: 0.36 -> 0.17 ms, bound by its 0.77 GB of traffic).
constexpr int H16_MB = 64;        // blocks of a cloud's column sums
constexpr int H16_SAMPLE = 16384; // points of a cloud's column sums
constexpr int H16_T = 256;
constexpr float H16_REL = 0x1.01p-11f, H16_ABS = 0x1p-20f, H16_ABS2 = 0x1p-14f;
constexpr float H16_NORM_UP = 1.0f + 0x1p-16f;

// Per cloud: its fp16 rows, norms, means and {s, s eps_up} (null: FP32 tiles).
struct H16Out {
    uint4 *h16[kMaxClouds];
    float *n16[kMaxClouds], *mean[kMaxClouds], *scal[kMaxClouds];
};

// Partial column sums of a cloud's sample: block (b, cloud) adds the sampled
// points b R, b R + 1, ... (R rows of dp / 4 threads at a time; dp <= 128).
__global__ void __launch_bounds__(H16_T) k_h16_sums(const __grid_constant__ Views V, float *__restrict__ partial) {
    const int c = blockIdx.y;
    if (!V.h16[c]) return;
    const int64_t n = V.rbase[c + 1] - V.rbase[c];
    const int64_t ns = n < H16_SAMPLE ? n : H16_SAMPLE, step = n / ns;
    const int nq = V.tv[c].dp >> 2, R = H16_T / nq, r = threadIdx.x / nq, q = threadIdx.x % nq;
    __shared__ float4 sh[H16_T];
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
    if (r < R) {
        for (int64_t i = (int64_t)blockIdx.x * R + r; i < ns; i += (int64_t)gridDim.x * R) {
            const float4 x = __ldg(reinterpret_cast<const float4 *>(V.tv[c].pts) + i * step * nq + q);
            acc.x += x.x;
            acc.y += x.y;
            acc.z += x.z;
            acc.w += x.w;
        }
    }
    sh[threadIdx.x] = acc;
    __syncthreads();
    if (r == 0) {
        for (int k = 1; k < R; ++k) {
            const float4 x = sh[k * nq + q];
            acc.x += x.x;
            acc.y += x.y;
            acc.z += x.z;
            acc.w += x.w;
        }
        reinterpret_cast<float4 *>(partial)[((size_t)c * H16_MB + blockIdx.x) * 32 + q] = acc;
    }
}

// Column means and the scale of each cloud: every point is within r_root of
// the root centre, and so is the sample's mean, so |x_k - m_k| <= |x - m| <=
// 2 r_root; s = 2^(14 - e) with max(2 r_root, eps) < 2^e.  scal = {s, s eps_up}.
__global__ void __launch_bounds__(128) k_h16_means(const __grid_constant__ Views V,
                                                   const __grid_constant__ H16Out out,
                                                   const float *__restrict__ partial) {
    const int c = blockIdx.x, k = threadIdx.x;
    if (!V.h16[c]) return;
    const int64_t n = V.rbase[c + 1] - V.rbase[c];
    const int64_t ns = n < H16_SAMPLE ? n : H16_SAMPLE;
    if (k < V.tv[c].dp) {
        double acc = 0.0;
#pragma unroll 16
        for (int b = 0; b < H16_MB; ++b) acc += (double)partial[((size_t)c * H16_MB + b) * 128 + k];
        out.mean[c][k] = (float)(acc / (double)ns);
    }
    if (k == 0) {
        const float eps_up = V.qp[c].eps_up;
        const float M = fmaxf(2.0f * V.tv[c].radius[0] * (1.0f + 0x1p-10f), eps_up);
        float s = 0x1p-100f;
        if (M <= 0x1p100f) {
            int e;
            frexpf(fmaxf(M, 0x1p-100f), &e);  // M < 2^e
            s = ldexpf(1.0f, 14 - e);
        }
        out.scal[c][0] = s;
        out.scal[c][1] = s * eps_up;
    }
}

// Rows in tree order -> fp16 rows and their squared norms; sixteen lanes per
// row (of all clouds, concatenated), lane j converts halves 8j .. 8j + 7 (one
// 16-byte chunk).
__global__ void __launch_bounds__(H16_T) k_to_h16(const __grid_constant__ Views V,
                                                  const __grid_constant__ H16Out out) {
    const int64_t gid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t grow = gid >> 4;
    const int j = (int)(gid & 15);
    int c = 0;
    if (V.nc > 1) {
        int lo = 0, hi = V.nc;
        while (hi - lo > 1) {
            const int mid = (lo + hi) >> 1;
            if (V.rbase[mid] <= grow) lo = mid; else hi = mid;
        }
        c = lo;
    }
    const bool on = grow < V.rbase[V.nc] && V.h16[c];
    const int64_t row = grow - V.rbase[c];
    const int dp = V.tv[c].dp, kc = 8 * ((dp + 63) >> 6);
    float sq = 0.f;
    if (on && j < kc) {
        const float s = out.scal[c][0];
        float v[8];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int k = 8 * j + 4 * h;
            float4 x = make_float4(0.f, 0.f, 0.f, 0.f), m = x;
            if (k < dp) {  // dp is a multiple of 4
                x = __ldg(reinterpret_cast<const float4 *>(V.tv[c].pts + row * dp + k));
                m = __ldg(reinterpret_cast<const float4 *>(out.mean[c] + k));
            }
            v[4 * h + 0] = (x.x - m.x) * s;
            v[4 * h + 1] = (x.y - m.y) * s;
            v[4 * h + 2] = (x.z - m.z) * s;
            v[4 * h + 3] = (x.w - m.w) * s;
        }
        uint32_t w[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const __half2 hh = __floats2half2_rn(v[2 * u], v[2 * u + 1]);
            w[u] = *reinterpret_cast<const uint32_t *>(&hh);
            const float2 f = __half22float2(hh);
            sq = fmaf(f.x, f.x, sq);
            sq = fmaf(f.y, f.y, sq);
        }
        out.h16[c][row * kc + j] = make_uint4(w[0], w[1], w[2], w[3]);
    }
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) sq += __shfl_xor_sync(0xffffffffu, sq, o, 16);
    if (on && j == 0) out.n16[c][row] = sq;
}

#include "leaf_tc.cuh"

// Dynamic shared memory of the L2 leaf kernels (set once per process).
void leaf_l2_prepare() {
    static bool done = false;
    if (done) return;
    auto allow = [](auto kern, bool shorts) {
        CT_CHECK_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)leaf_smem(shorts)));
    };
    allow(k_leaf_l2<true, KS_SHORT>, true);
    allow(k_leaf_l2<false, KS_SHORT>, true);
    allow(k_leaf_l2<true, KS_LONG>, false);
    allow(k_leaf_l2<false, KS_LONG>, false);
    done = true;
}

// Upper-triangle form, integer metrics (one cloud): the edge (q, p) with p in
// a later group is also the edge (p, q) of p's row: its degree and one-pass
// entry (count pass) or its entry (emit pass; a selected row only when rows
// are emitted again).
__device__ __forceinline__ void mirror_int(const TreeView &tv, int32_t *deg, const int64_t *row_ptr, int32_t *rowcur,
                                           int32_t *col, float *dist, int32_t *err, const CapOut &co,
                                           const uint8_t *rowsel, bool emit, int qpos, int ppos, int d) {
    const int o = tv.perm[ppos];
    if (!emit) {
        atomicAdd(&deg[o], 1);
        if (co.off) cap_put(co, o, tv.perm[qpos], (float)d);
        return;
    }
    if (rowsel && !rowsel[o]) return;
    const int slot = atomicAdd(&rowcur[o], 1);
    const int64_t at = row_ptr[o] + slot;
    if (at < row_ptr[o + 1]) {
        col[at] = tv.perm[qpos];
        dist[at] = (float)d;
    } else {
        atomicOr(err, 4);
    }
}

// Edit distance of one (pattern, text) pair over alphabet-mapped symbols;
// the distance if <= k, else k + 1.
template <int W>
__device__ __forceinline__ int lev_mapped(const uint64_t *__restrict__ pq, const uint8_t *__restrict__ amap, int m,
                                          const uint8_t *__restrict__ txt, int n, int k,
                                          unsigned long long &cols) {
    if (k < 0) return (m == 0 && n == 0) ? 0 : k + 1;
    if ((m > n ? m - n : n - m) > k) return k + 1;
    if (m == 0) return n;
    if (n == 0) return m;
    if (W > 1 && k < 64) {
        int done;
        auto sym = [amap](int s) { return (int)amap[s]; };
        const int d = k < 32 ? lev_band<uint32_t, W>(pq, sym, m, txt, n, k, done)
                             : lev_band<uint64_t, W>(pq, sym, m, txt, n, k, done);
        cols += (unsigned)done;
        return d;
    }
    const int nw = (m + 63) >> 6, hw = (m - 1) >> 6;
    const uint64_t hbit = 1ull << ((m - 1) & 63);
    uint64_t Pv[W], Mv[W];
#pragma unroll
    for (int w = 0; w < W; ++w) {
        Pv[w] = ~0ull;
        Mv[w] = 0ull;
    }
    int score = m;
    for (int j = 0; j < n; ++j) {
        const uint64_t *eqr = pq + (int)amap[txt[j]] * W;
        uint64_t carry = 0ull, hp_in = 1ull, hn_in = 0ull;
#pragma unroll
        for (int w = 0; w < W; ++w) {
            if (w < nw) {
                uint64_t Eq = eqr[w], pv = Pv[w], mv = Mv[w];
                uint64_t Xv = Eq | mv, tt = Eq & pv;
                uint64_t s1 = tt + pv, c1b = s1 < tt ? 1ull : 0ull;
                uint64_t s2 = s1 + carry, c2b = s2 < s1 ? 1ull : 0ull;
                carry = c1b | c2b;
                uint64_t Xh = (s2 ^ pv) | Eq;
                uint64_t Ph = mv | ~(Xh | pv), Mh = pv & Xh;
                if (w == hw) {
                    if (Ph & hbit) ++score;
                    else if (Mh & hbit) --score;
                }
                uint64_t po = Ph >> 63, mo = Mh >> 63;
                Ph = (Ph << 1) | hp_in;
                Mh = (Mh << 1) | hn_in;
                hp_in = po;
                hn_in = mo;
                Pv[w] = Mh | ~(Xv | Ph);
                Mv[w] = Ph & Xv;
            }
        }
        if (score - (n - 1 - j) > k) {
            cols += (unsigned long long)(j + 1) * nw;
            return k + 1;
        }
    }
    cols += (unsigned long long)n * nw;
    return score;
}

// Edit distance leaf stage: one CTA per group; packed candidate tiles as in
// the L2 kernel; each thread decides (query, candidate point) pairs with the
// query as the bit-parallel pattern.  The queries' match masks cover only the
// bytes that occur in the data (alphabet map amap, A symbols).
template <bool EMIT, int W>
__global__ void __launch_bounds__(LEAF_T) k_leaf_lev(
    TreeView tv, QParams qp, const uint8_t *__restrict__ amap_g, int A, int qchunk, Items items,
    uint32_t *__restrict__ cand, int32_t *__restrict__ deg, const int64_t *__restrict__ row_ptr,
    int32_t *__restrict__ rowcur, int32_t *__restrict__ col, float *__restrict__ dist,
    unsigned long long *__restrict__ st, int32_t *__restrict__ err, CapOut co, const uint8_t *__restrict__ rowsel) {
    extern __shared__ uint64_t speq[];  // qchunk x A x W
    __shared__ uint8_t amap[256];
    __shared__ int cnt[32], cursor[32], qlen[32], sel[32];
    __shared__ int64_t rowb[32], rowe[32];
    __shared__ int tpos[32];
    __shared__ int64_t tcand[32];
    __shared__ int64_t s_ci;
    __shared__ int s_off, s_rows;
    __shared__ unsigned s_hit;
    const int tid = threadIdx.x, warp = tid >> 5;
    const int it = blockIdx.x;
    if (it >= *items.count) return;
    const int g = items.group[it];
    const int qb = tv.group_begin[g], qn = tv.group_count[g], qe = qb + qn;
    const int64_t c0 = items.begin[it], c1 = items.end[it];
    const int k = qp.lev_k;
    for (int i = tid; i < 256; i += LEAF_T) amap[i] = amap_g[i];
    unsigned long long pairs = 0, cols = 0;
    for (int q0 = 0; q0 < qn; q0 += qchunk) {
        const int nqr = min(qchunk, qn - q0);
        __syncthreads();
        for (int i = tid; i < qchunk * A * W; i += LEAF_T) speq[i] = 0ull;
        if (tid < 32) {
            cnt[tid] = 0;
            if (tid < nqr) {
                int qpos = qb + q0 + tid;
                qlen[tid] = (int)(tv.soff[qpos + 1] - tv.soff[qpos]);
                int o = tv.perm[qpos];
                cursor[tid] = o;  // original id of the query (row of the CSR)
                sel[tid] = rowsel == nullptr || rowsel[o] != 0;
                if (EMIT) {
                    rowb[tid] = row_ptr[o];
                    rowe[tid] = row_ptr[o + 1];
                }
            }
        }
        if (tid == 0) {
            s_ci = c0;
            s_off = 0;
            s_hit = 0u;
        }
        __syncthreads();
        for (int q = 0; q < nqr; ++q) {
            int qpos = qb + q0 + q;
            const uint8_t *sq = tv.sdata + tv.soff[qpos];
            int m = qlen[q];
            for (int j = tid; j < m; j += LEAF_T)
                atomicOr((unsigned long long *)&speq[((size_t)q * A + amap[sq[j]]) * W + (j >> 6)], 1ull << (j & 63));
        }
        for (;;) {
            __syncthreads();
            if (warp == 0) fill_tile(tv, cand, c1, EMIT, &s_ci, &s_off, &s_rows, tpos, tcand);
            __syncthreads();
            const int npr = s_rows;
            const bool last = s_ci >= c1;
            if (npr > 0) {
                unsigned hit = 0u;
                for (int t = tid; t < nqr * npr; t += LEAF_T) {
                    int q = t / npr, p = t - q * npr;
                    int qpos = qb + q0 + q, ppos = tpos[p];
                    if (qpos == ppos && !qp.include_self) continue;
                    if (qp.half && ppos < qb) continue;
                    const bool mir = qp.half && ppos >= qe;
                    if (EMIT && !sel[q] && !(mir && rowsel)) continue;
                    if (!EMIT) ++pairs;
                    const uint8_t *txt = tv.sdata + tv.soff[ppos];
                    int n = (int)(tv.soff[ppos + 1] - tv.soff[ppos]);
                    int d = lev_mapped<W>(speq + (size_t)q * A * W, amap, qlen[q], txt, n, k, cols);
                    if (d > k) continue;
                    if (mir) mirror_int(tv, deg, row_ptr, rowcur, col, dist, err, co, rowsel, EMIT, qpos, ppos, d);
                    if (!EMIT) {
                        hit |= 1u << p;
                        atomicAdd(&cnt[q], 1);
                        if (co.off) cap_put(co, cursor[q], tv.perm[ppos], (float)d);
                    } else if (sel[q]) {
                        int slot = atomicAdd(&rowcur[cursor[q]], 1);
                        int64_t at = rowb[q] + slot;
                        if (at < rowe[q]) {
                            col[at] = tv.perm[ppos];
                            dist[at] = (float)d;
                        } else {
                            atomicOr(err, 4);
                        }
                    }
                }
                if (!EMIT) {
                    if (hit) atomicOr(&s_hit, hit);
                    __syncthreads();
                    if (tid < npr && ((s_hit >> tid) & 1u)) atomicOr(&cand[tcand[tid]], FLAG);
                    __syncthreads();
                    if (tid == 0) s_hit = 0u;
                }
            }
            if (last) break;
        }
        __syncthreads();
        if (!EMIT && tid < nqr && cnt[tid]) atomicAdd(&deg[cursor[tid]], cnt[tid]);
    }
    if (!EMIT) {
        for (int o = 16; o > 0; o >>= 1) {
            pairs += __shfl_xor_sync(0xffffffffu, pairs, o);
            cols += __shfl_xor_sync(0xffffffffu, cols, o);
        }
        if ((tid & 31) == 0) {
            stat_add(st, ST_PAIRS, pairs);
            stat_add(st, ST_COLS, cols);
        }
    }
}

// Set bits of eight words: four full adders leave the ones in two words and the
// twos and fours in one each, so four population counts instead of eight.
__device__ __forceinline__ int popc8(const uint4 x, const uint4 y) {
    const uint32_t s1 = x.x ^ x.y ^ x.z, c1 = (x.x & x.y) | (x.x & x.z) | (x.y & x.z);
    const uint32_t s2 = x.w ^ y.x ^ y.y, c2 = (x.w & y.x) | (x.w & y.y) | (y.x & y.y);
    const uint32_t s3 = s1 ^ s2 ^ y.z, c3 = (s1 & s2) | (s1 & y.z) | (s2 & y.z);
    const uint32_t t = c1 ^ c2 ^ c3, u = (c1 & c2) | (c1 & c3) | (c2 & c3);
    return (__popc(s3) + __popc(y.w)) + 2 * __popc(t) + 4 * __popc(u);
}
__device__ __forceinline__ int popc4(const uint4 x) {
    const uint32_t s1 = x.x ^ x.y ^ x.z, c1 = (x.x & x.y) | (x.x & x.z) | (x.y & x.z);
    return (__popc(s1) + __popc(x.w)) + 2 * __popc(c1);
}
__device__ __forceinline__ uint4 xor4(const uint4 a, const uint4 b) {
    return make_uint4(a.x ^ b.x, a.y ^ b.y, a.z ^ b.z, a.w ^ b.w);
}

// Hamming leaf stage, integer distances: one CTA per work item, the group's
// query rows (zero padded to nch x NQ uint4) in shared memory.  Each warp takes
// a quarter of the item's candidates by itself (handing out 32 at a time to the
// four was slower: 16.1 against 14.7 ms) and packs 32 rows at a time: lane p keeps
// row p in registers (NQ uint4; longer rows in nch chunks, eight queries at a
// time) and the queries are read as broadcasts, so a pair costs no shared
// bandwidth and the tiles no barriers.  The hits of a lane are a mask over the
// queries; they are written after the tile, two rounds or so for all lanes
// together instead of a divergent branch per hit.
// Bound by the population counts (16 per clock and SM) and the logic before
// them: 6.6e9 pairs of 256 bits took 23.4 ms as 32 x 32 tiles of two shared rows per
// pair and a count per word, 14.7 ms now.
template <bool EMIT, int NQ>
__global__ void __launch_bounds__(LEAF_T) k_leaf_ham(
    TreeView tv, QParams qp, Items items, uint32_t *__restrict__ cand, int32_t *__restrict__ deg,
    const int64_t *__restrict__ row_ptr, int32_t *__restrict__ rowcur, int32_t *__restrict__ col,
    float *__restrict__ dist, unsigned long long *__restrict__ st, int32_t *__restrict__ err, CapOut co,
    const uint8_t *__restrict__ rowsel) {
    constexpr int QB = 8;
    extern __shared__ uint4 Qs[];  // 32 query rows
    __shared__ int cnt[32], cursor[32];
    __shared__ int64_t rowb[32], rowe[32];
    __shared__ unsigned s_sel;
    const int tid = threadIdx.x, lane = tid & 31;
    const int it = blockIdx.x;
    if (it >= *items.count) return;
    const int g = items.group[it];
    const int qb = tv.group_begin[g], qn = tv.group_count[g], qe = qb + qn;  // at most 32 queries
    const int k = qp.lev_k, nq = tv.wp >> 2, nch = (nq + NQ - 1) / NQ, qs = nch * NQ;
    const uint4 *rows = reinterpret_cast<const uint4 *>(tv.bits);
    if (tid < 32) {
        cnt[tid] = 0;
        bool sel = false;
        if (tid < qn) {
            const int o = tv.perm[qb + tid];
            cursor[tid] = o;
            sel = rowsel == nullptr || rowsel[o] != 0;
            if (EMIT) {
                rowb[tid] = row_ptr[o];
                rowe[tid] = row_ptr[o + 1];
            }
        }
        const unsigned m = __ballot_sync(0xffffffffu, sel);
        if (tid == 0) s_sel = m;
    }
    for (int i = tid; i < 32 * qs; i += LEAF_T) {
        const int q = i / qs, j = i - q * qs;
        Qs[i] = q < qn && j < nq ? rows[(size_t)(qb + q) * nq + j] : make_uint4(0u, 0u, 0u, 0u);
    }
    __syncthreads();
    const unsigned selm = s_sel, qmask = 0xffffffffu >> (32 - qn);
    // the warp's part: whole steps of 32 candidates
    const int64_t c0 = items.begin[it], c1 = items.end[it];
    const int64_t part = ((c1 - c0 + LEAF_T - 1) / LEAF_T) * 32;
    int64_t ci = c0 + (tid >> 5) * part;
    const int64_t ce = min(ci + part, c1);
    int off = 0;
    unsigned long long pairs = 0;
    while (ci < ce) {
        int pos;
        int64_t pcand;
        const int npr = tile_rows(tv, cand, ce, EMIT, ci, off, pos, pcand);
        if (npr == 0) continue;
        const int ppos = lane < npr ? pos : qb;
        const bool mir = qp.half && ppos >= qe;
        // the queries this row is paired with
        unsigned want = lane < npr && !(qp.half && ppos < qb) ? qmask : 0u;
        if (!qp.include_self && ppos >= qb && ppos < qe) want &= ~(1u << (ppos - qb));
        if (EMIT && !(mir && rowsel)) want &= selm;
        if (!EMIT) pairs += __popc(want);
        const uint4 *prow = rows + (size_t)ppos * nq;
        uint4 x[NQ];
        unsigned hits = 0u;
        for (int q0 = 0; q0 < qn; q0 += QB) {
            int acc[QB];
#pragma unroll
            for (int j = 0; j < QB; ++j) acc[j] = 0;
            for (int c = 0; c < nch; ++c) {
                if (q0 == 0 || nch > 1) {
#pragma unroll
                    for (int i = 0; i < NQ; ++i)
                        x[i] = c * NQ + i < nq ? __ldg(prow + c * NQ + i) : make_uint4(0u, 0u, 0u, 0u);
                }
#pragma unroll
                for (int j = 0; j < QB; ++j) {
                    const uint4 *a = Qs + (q0 + j) * qs + c * NQ;
                    if (NQ == 1) acc[j] += popc4(xor4(a[0], x[0]));
#pragma unroll
                    for (int i = 0; i + 1 < NQ; i += 2) acc[j] += popc8(xor4(a[i], x[i]), xor4(a[i + 1], x[i + 1]));
                }
            }
#pragma unroll
            for (int j = 0; j < QB; ++j) hits |= (acc[j] <= k ? 1u : 0u) << (q0 + j);
        }
        hits &= want;
        const int o = hits ? tv.perm[ppos] : 0;
        if (!EMIT && hits) atomicOr(&cand[pcand], FLAG);
        int mslot = 0;  // the lane's first entry of its own (mirrored) row
        if (!EMIT && mir && hits) {
            atomicAdd(&deg[o], __popc(hits));
            if (co.off) mslot = atomicAdd(&co.fill[o], __popc(hits));
        }
        const bool mrow = EMIT && mir && hits && (!rowsel || rowsel[o]);
        const int64_t mb = mrow ? row_ptr[o] : 0, me = mrow ? row_ptr[o + 1] : 0;
        if (mrow) mslot = atomicAdd(&rowcur[o], __popc(hits));
        for (; hits; hits &= hits - 1u) {
            const int q = __ffs(hits) - 1, oq = cursor[q];
            int di = 0;
            if (EMIT || co.off) di = ham_rows_smem(Qs + q * qs, prow, nq);
            const float d = (float)di;
            if (!EMIT) {
                atomicAdd(&cnt[q], 1);
                if (co.off) {
                    cap_put(co, oq, o, d);
                    if (mir) cap_place(co, o, mslot++, oq, d);
                }
                continue;
            }
            if (mrow) {
                const int64_t at = mb + mslot++;
                if (at < me) {
                    col[at] = oq;
                    dist[at] = d;
                } else {
                    atomicOr(err, 4);
                }
            }
            if ((selm >> q) & 1u) {
                const int64_t at = rowb[q] + atomicAdd(&rowcur[oq], 1);
                if (at < rowe[q]) {
                    col[at] = o;
                    dist[at] = d;
                } else {
                    atomicOr(err, 4);
                }
            }
        }
        __syncwarp();
    }
    if (EMIT) return;
    __syncthreads();
    if (tid < qn && cnt[tid]) atomicAdd(&deg[cursor[tid]], cnt[tid]);
    for (int o = 16; o > 0; o >>= 1) pairs += __shfl_xor_sync(0xffffffffu, pairs, o);
    if (lane == 0) stat_add(st, ST_PAIRS, pairs);
}

// ------------------------------------------------------------- row sort

constexpr int SORT_MID = 4096;  // rows up to this length are sorted in one CTA

// Row classes by length: 0 <= 32, 1 <= 64, 2 <= 128, 3 <= 256, 4 <= 512 (one
// warp per row), 5 <= 1024, 6 <= 2048, 7 <= SORT_MID (one CTA per row), 8 longer.
constexpr int kSortClasses = 9;
__global__ void k_row_classes(const int64_t *__restrict__ row_ptr, int64_t n, int32_t *__restrict__ lists,
                              int32_t *__restrict__ counts) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    int64_t len = row_ptr[i + 1] - row_ptr[i];
    if (len <= 1) return;
    int cls = kSortClasses - 1;
    for (int c = 0; c < kSortClasses - 1; ++c)
        if (len <= (int64_t)32 << c) {
            cls = c;
            break;
        }
    // one atomic per class present in the warp (the lanes still here)
    const unsigned peers = __match_any_sync(__activemask(), cls);
    const int lane = threadIdx.x & 31, leader = __ffs(peers) - 1;
    int base = 0;
    if (lane == leader) base = atomicAdd(&counts[cls], __popc(peers));
    base = __shfl_sync(peers, base, leader);
    lists[(int64_t)cls * n + base + __popc(peers & ((1u << lane) - 1))] = (int32_t)i;
}

// Bitonic network over the 32 lanes of a warp: (key, val) pairs ascending by
// key, lane i ending with the i-th smallest.
__device__ __forceinline__ void warp_sort32(int &key, float &val, int lane) {
#pragma unroll
    for (int k = 2; k <= 32; k <<= 1) {
#pragma unroll
        for (int j = k >> 1; j > 0; j >>= 1) {
            const int ok = __shfl_xor_sync(0xffffffffu, key, j);
            const float ov = __shfl_xor_sync(0xffffffffu, val, j);
            const bool up = (lane & k) == 0, lower = (lane & j) == 0;
            if ((lower == up) ? (ok < key) : (ok > key)) {
                key = ok;
                val = ov;
            }
        }
    }
}

// A warp's 32 E entries in the blocked layout: lane l holds entries l E ..
// l E + E - 1 in registers.  In shared memory entry i sits at swz<E>(i), its
// low bits XORed with bits 5.., so that a warp's striped access (entries
// c 32 + lane, coalesced in global memory) and its blocked access (entries
// lane E + e) both hit 32 distinct banks.
template <int E>
__device__ __forceinline__ int swz(int i) {
    return i ^ ((i >> 5) & (E - 1));
}

// Bitonic sorting network over 32 E (key, val) pairs in the blocked layout,
// ascending by key.  Exchanges at distances below E pair entries of one lane
// (registers only); the others pair lane l with lane l ^ (distance / E) at
// the same register (one shuffle of key and of val).  The low distances,
// which the network visits most often, are thus the register ones.
template <int E>
__device__ __forceinline__ void warp_sort_blocked(int (&key)[E], float (&val)[E], int lane) {
    constexpr int N = 32 * E;
#pragma unroll
    for (int k = 2; k <= N; k <<= 1) {
#pragma unroll
        for (int j = k >> 1; j > 0; j >>= 1) {
            if (j < E) {
#pragma unroll
                for (int e = 0; e < E; ++e) {
                    if (e & j) continue;
                    const int f = e | j;
                    const bool up = ((lane * E + e) & k) == 0;
                    // selects, not a branch: lanes disagree on the swap
                    const int a = key[e], c = key[f];
                    const float va = val[e], vc = val[f];
                    const bool sw = (a > c) == up;
                    key[e] = sw ? c : a;
                    key[f] = sw ? a : c;
                    val[e] = sw ? vc : va;
                    val[f] = sw ? va : vc;
                }
            } else {
                const int lj = j / E;
                const bool keep_min = (((lane * E) & k) == 0) == ((lane & lj) == 0);
#pragma unroll
                for (int e = 0; e < E; ++e) {
                    const int ok = __shfl_xor_sync(0xffffffffu, key[e], lj);
                    const float ov = __shfl_xor_sync(0xffffffffu, val[e], lj);
                    const bool take = (ok < key[e]) == keep_min;  // equal keys: padding only
                    key[e] = take ? ok : key[e];
                    val[e] = take ? ov : val[e];
                }
            }
        }
    }
}

// One warp's blocked registers from / to its swizzled shared slice sh
// (entries at or past len read as INT_MAX keys).
template <int E>
__device__ __forceinline__ void take_blocked(const int *sh, const float *sv, int len, int lane, int (&key)[E],
                                             float (&val)[E]) {
#pragma unroll
    for (int e = 0; e < E; ++e) {
        const int i = lane * E + e;
        key[e] = i < len ? sh[swz<E>(i)] : INT_MAX;
        val[e] = i < len ? sv[swz<E>(i)] : 0.f;
    }
}
template <int E>
__device__ __forceinline__ void put_blocked(int *sh, float *sv, int lane, const int (&key)[E], const float (&val)[E]) {
#pragma unroll
    for (int e = 0; e < E; ++e) {
        sh[swz<E>(lane * E + e)] = key[e];
        sv[swz<E>(lane * E + e)] = val[e];
    }
}

constexpr int SORT_WARPS = 8;  // warps per CTA of k_sort_warp

// Warp per row of 16 E + 1 .. 32 E entries (E = 2 .. 16): the row is read
// coalesced into the warp's shared slice (all its loads issued before the
// first store), taken into registers in the blocked layout, sorted by
// warp_sort_blocked and written back the same way.
template <int E>
__global__ void __launch_bounds__(32 * SORT_WARPS, 3) k_sort_warp(const int32_t *__restrict__ rows,
                                                               const int32_t *__restrict__ count,
                                                               const int64_t *__restrict__ row_ptr,
                                                               int32_t *__restrict__ col, float *__restrict__ dist) {
    __shared__ int s_key[SORT_WARPS][32 * E];
    __shared__ float s_val[SORT_WARPS][32 * E];
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    int *sk = s_key[wib];
    float *sv = s_val[wib];
    const int nrows = *count;
    for (int w = blockIdx.x * SORT_WARPS + wib; w < nrows; w += gridDim.x * SORT_WARPS) {
        const int r = rows[w];
        const int64_t b = row_ptr[r];
        const int len = (int)min(row_ptr[r + 1] - b, (int64_t)(32 * E));  // rows of this class fit
        int key[E];
        float val[E];
#pragma unroll
        for (int c = 0; c < E; ++c) {
            const int i = c * 32 + lane;
            key[c] = i < len ? col[b + i] : 0;
            val[c] = i < len ? dist[b + i] : 0.f;
        }
        __syncwarp();  // the previous row's write-back has read the slice
#pragma unroll
        for (int c = 0; c < E; ++c) {
            const int i = c * 32 + lane;
            if (i < len) {
                sk[swz<E>(i)] = key[c];
                sv[swz<E>(i)] = val[c];
            }
        }
        __syncwarp();
        take_blocked<E>(sk, sv, len, lane, key, val);
        warp_sort_blocked<E>(key, val, lane);
        __syncwarp();
        put_blocked<E>(sk, sv, lane, key, val);
        __syncwarp();
#pragma unroll
        for (int c = 0; c < E; ++c) {
            const int i = c * 32 + lane;
            if (i < len) {
                col[b + i] = sk[swz<E>(i)];
                dist[b + i] = sv[swz<E>(i)];
            }
        }
    }
}

// One merge round of a row's sorted runs of length run >= 512 (the last may
// be shorter or alone): the pair (A, B) = runs 2 m, 2 m + 1 goes to the
// outputs [2 m run, ...) of buffers (kn, vn).  Thread tid writes the SEG = 16
// outputs from 16 tid: one binary search along its diagonal finds how many of
// them come from A (merge path), then it merges them one by one.  Every
// buffer holds entry i at swz<16>(i) (runs start at multiples of 512, so a
// run's entry x sits at its start + swz<16>(x)): the warp's stores of its
// 16 consecutive outputs then hit 32 distinct banks.
template <int SEG>
__device__ __forceinline__ void merge_round(const int *__restrict__ kc, const float *__restrict__ vc,
                                            int *__restrict__ kn, float *__restrict__ vn, int len, int run,
                                            int tid) {
    const int o = tid * SEG;
    if (o >= len) return;
    const int s0 = o & ~(2 * run - 1);
    const int na = min(run, len - s0), nb = max(0, min(run, len - s0 - run));
    const int *A = kc + s0, *B = A + run;
    const float *Av = vc + s0, *Bv = Av + run;
    auto at = [](int i) { return swz<16>(i); };
    const int d = o - s0;  // outputs of the pair before this thread's
    int lo = max(0, d - nb), hi = min(d, na);
    while (lo < hi) {  // entries of A among the pair's d smallest
        const int mid = (lo + hi) >> 1;
        if (A[at(mid)] < B[at(d - 1 - mid)]) lo = mid + 1; else hi = mid;
    }
    // An exhausted run's head reads INT_MAX, above every column, so the other
    // run is taken; each step selects, no branch.
    int ia = lo, ib = d - lo;
    int ka = ia < na ? A[at(ia)] : INT_MAX, kb = ib < nb ? B[at(ib)] : INT_MAX;
    const int cnt = min(SEG, len - o);
#pragma unroll 4
    for (int t = 0; t < cnt; ++t) {
        const bool ta = ka < kb;
        kn[swz<16>(o + t)] = ta ? ka : kb;
        vn[swz<16>(o + t)] = ta ? Av[at(ia)] : Bv[at(ib)];
        ia += ta;
        ib += !ta;
        const int nx = ta ? ia : ib;
        const int nk = nx < (ta ? na : nb) ? (ta ? A : B)[at(nx)] : INT_MAX;
        ka = ta ? nk : ka;
        kb = ta ? kb : nk;
    }
}

// CTA of P = CAP / 16 threads per row of 513 .. CAP entries (16 CAP bytes of
// dynamic shared memory: keys and values, two buffers each).  Each warp sorts
// one 512-entry run in registers (warp_sort_blocked<16>) and leaves it in the
// swizzled layout (swz<16>, which every buffer keeps); then runs merge in
// pairs (merge_round) until one is left.
// The columns of a row are distinct, so the merged order is unique.
template <int CAP>
__global__ void __launch_bounds__(CAP / 16, 12288 / CAP) k_sort_merge(const int32_t *__restrict__ rows,
                                                                      const int32_t *__restrict__ count,
                                                                      const int64_t *__restrict__ row_ptr,
                                                                      int32_t *__restrict__ col,
                                                                      float *__restrict__ dist) {
    constexpr int P = CAP / 16, SEG = 16, RUN = 512;
    extern __shared__ int sort_smem[];
    int (*sk)[CAP] = reinterpret_cast<int (*)[CAP]>(sort_smem);
    float (*sv)[CAP] = reinterpret_cast<float (*)[CAP]>(sort_smem + 2 * CAP);
    const int tid = threadIdx.x, lane = tid & 31;
    const int nrows = *count;
    for (int w = blockIdx.x; w < nrows; w += gridDim.x) {
        const int r = rows[w];
        const int64_t b = row_ptr[r];
        const int len = (int)min(row_ptr[r + 1] - b, (int64_t)CAP);  // rows of this class fit
        {  // coalesced read: SEG loads a thread, then the stores
            int key[SEG];
            float val[SEG];
#pragma unroll
            for (int c = 0; c < SEG; ++c) {
                const int i = c * P + tid;
                key[c] = i < len ? col[b + i] : 0;
                val[c] = i < len ? dist[b + i] : 0.f;
            }
            __syncthreads();  // the previous row's write-back has read sk / sv
#pragma unroll
            for (int c = 0; c < SEG; ++c) {
                const int i = c * P + tid;
                if (i < len) {
                    sk[0][swz<16>(i)] = key[c];
                    sv[0][swz<16>(i)] = val[c];
                }
            }
        }
        __syncthreads();
        const int base = (tid >> 5) * RUN;
        if (base < len) {  // the warp's run, sorted in place
            int key[16];
            float val[16];
            take_blocked<16>(sk[0] + base, sv[0] + base, len - base, lane, key, val);
            warp_sort_blocked<16>(key, val, lane);
            __syncwarp();
            put_blocked<16>(sk[0] + base, sv[0] + base, lane, key, val);
        }
        __syncthreads();
        int cur = 0;
        for (int run = RUN; run < len; run <<= 1) {
            merge_round<SEG>(sk[cur], sv[cur], sk[cur ^ 1], sv[cur ^ 1], len, run, tid);
            __syncthreads();
            cur ^= 1;
        }
#pragma unroll
        for (int c = 0; c < SEG; ++c) {
            const int i = c * P + tid;
            if (i < len) {
                col[b + i] = sk[cur][swz<16>(i)];
                dist[b + i] = sv[cur][swz<16>(i)];
            }
        }
    }
}

// Rows of a graph with fewer than 2^20 columns sort one 32-bit key per
// entry, (column << PACK_BITS) | (the entry's position in the row, below
// SORT_MID): a row's keys are distinct and order as its columns do, so the
// network moves keys alone (min / max, no selects of values) and each value
// is fetched by its position once the keys are sorted.
constexpr int PACK_BITS = 12;
constexpr uint32_t PACK_POS = (1u << PACK_BITS) - 1;
constexpr int64_t PACK_MAX_COLS = int64_t(1) << (32 - PACK_BITS);  // packed when n (columns < n) is below
static_assert(SORT_MID <= (1 << PACK_BITS), "positions must fit the packed keys");

// Sorting network over 32 E packed keys in the blocked layout (padding:
// 0xffffffff, above every key): bitonic merges in the form whose first step
// of each merge compares entry i with its mirror i ^ (k - 1) in the block of
// k, the rest comparing i with i ^ j -- every comparator puts the minimum at
// the lower index, so a pair in one lane costs one min and one max.  Across
// lanes (distances of E and more) each lane keeps the minimum or the maximum
// of its key and its partner's, shuffled over.
template <int E>
__device__ __forceinline__ void warp_sort_keys(uint32_t (&key)[E], int lane) {
    constexpr int N = 32 * E;
#pragma unroll
    for (int k = 2; k <= N; k <<= 1) {
        if (k <= E) {  // the mirror step inside a lane
#pragma unroll
            for (int e = 0; e < E; ++e) {
                if (e & (k >> 1)) continue;
                const int f = e ^ (k - 1);
                const uint32_t lo = min(key[e], key[f]), hi = max(key[e], key[f]);
                key[e] = lo;
                key[f] = hi;
            }
        } else {  // mirror partner: lane ^ (k / E - 1), register E - 1 - e
            const int m = k / E - 1;
            const bool keep_min = (lane & (k / (2 * E))) == 0;
#pragma unroll
            for (int t = 0; t < E / 2; ++t) {
                const uint32_t o1 = __shfl_xor_sync(0xffffffffu, key[E - 1 - t], m);
                const uint32_t o2 = __shfl_xor_sync(0xffffffffu, key[t], m);
                key[t] = keep_min ? min(key[t], o1) : max(key[t], o1);
                key[E - 1 - t] = keep_min ? min(key[E - 1 - t], o2) : max(key[E - 1 - t], o2);
            }
        }
#pragma unroll
        for (int j = k >> 2; j > 0; j >>= 1) {
            if (j < E) {
#pragma unroll
                for (int e = 0; e < E; ++e) {
                    if (e & j) continue;
                    const int f = e | j;
                    const uint32_t lo = min(key[e], key[f]), hi = max(key[e], key[f]);
                    key[e] = lo;
                    key[f] = hi;
                }
            } else {
                const int lj = j / E;
                const bool keep_min = (lane & lj) == 0;
#pragma unroll
                for (int e = 0; e < E; ++e) {
                    const uint32_t o = __shfl_xor_sync(0xffffffffu, key[e], lj);
                    key[e] = keep_min ? min(key[e], o) : max(key[e], o);
                }
            }
        }
    }
}

// merge_round on packed keys alone.
template <int SEG>
__device__ __forceinline__ void merge_round_keys(const uint32_t *__restrict__ kc, uint32_t *__restrict__ kn,
                                                 int len, int run, int tid) {
    const int o = tid * SEG;
    if (o >= len) return;
    const int s0 = o & ~(2 * run - 1);
    const int na = min(run, len - s0), nb = max(0, min(run, len - s0 - run));
    const uint32_t *A = kc + s0, *B = A + run;
    auto at = [](int i) { return swz<16>(i); };
    const int d = o - s0;
    int lo = max(0, d - nb), hi = min(d, na);
    while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (A[at(mid)] < B[at(d - 1 - mid)]) lo = mid + 1; else hi = mid;
    }
    int ia = lo, ib = d - lo;
    uint32_t ka = ia < na ? A[at(ia)] : 0xffffffffu, kb = ib < nb ? B[at(ib)] : 0xffffffffu;
    const int cnt = min(SEG, len - o);
#pragma unroll 4
    for (int t = 0; t < cnt; ++t) {
        const bool ta = ka < kb;
        kn[swz<16>(o + t)] = min(ka, kb);
        ia += ta;
        ib += !ta;
        const int nx = ta ? ia : ib;
        const uint32_t nk = nx < (ta ? na : nb) ? (ta ? A : B)[at(nx)] : 0xffffffffu;
        ka = ta ? nk : ka;
        kb = ta ? kb : nk;
    }
}

// k_sort_warp on packed keys: the values wait in shared memory in row order.
template <int E>
__global__ void __launch_bounds__(32 * SORT_WARPS, 4) k_sort_warp_packed(const int32_t *__restrict__ rows,
                                                                         const int32_t *__restrict__ count,
                                                                         const int64_t *__restrict__ row_ptr,
                                                                         int32_t *__restrict__ col,
                                                                         float *__restrict__ dist) {
    __shared__ uint32_t s_key[SORT_WARPS][32 * E];
    __shared__ float s_val[SORT_WARPS][32 * E];
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    uint32_t *sk = s_key[wib];
    float *sv = s_val[wib];
    const int nrows = *count;
    for (int w = blockIdx.x * SORT_WARPS + wib; w < nrows; w += gridDim.x * SORT_WARPS) {
        const int r = rows[w];
        const int64_t b = row_ptr[r];
        const int len = (int)min(row_ptr[r + 1] - b, (int64_t)(32 * E));  // rows of this class fit
        uint32_t key[E];
        float val[E];
#pragma unroll
        for (int c = 0; c < E; ++c) {
            const int i = c * 32 + lane;
            key[c] = i < len ? ((uint32_t)col[b + i] << PACK_BITS) | (uint32_t)i : 0u;
            val[c] = i < len ? dist[b + i] : 0.f;
        }
        __syncwarp();  // the previous row's write-back has read the slice
#pragma unroll
        for (int c = 0; c < E; ++c) {
            const int i = c * 32 + lane;
            if (i < len) {
                sk[swz<E>(i)] = key[c];
                sv[i] = val[c];
            }
        }
        __syncwarp();
#pragma unroll
        for (int e = 0; e < E; ++e) {
            const int i = lane * E + e;
            key[e] = i < len ? sk[swz<E>(i)] : 0xffffffffu;
        }
        warp_sort_keys<E>(key, lane);
        __syncwarp();
#pragma unroll
        for (int e = 0; e < E; ++e) sk[swz<E>(lane * E + e)] = key[e];
        __syncwarp();
#pragma unroll
        for (int c = 0; c < E; ++c) {
            const int i = c * 32 + lane;
            if (i < len) {
                const uint32_t kk = sk[swz<E>(i)];
                col[b + i] = (int32_t)(kk >> PACK_BITS);
                dist[b + i] = sv[kk & PACK_POS];
            }
        }
    }
}

// k_sort_merge on packed keys (12 CAP bytes of dynamic shared memory: two
// key buffers and the values in row order).
template <int CAP>
__global__ void __launch_bounds__(CAP / 16, 16384 / CAP) k_sort_merge_packed(const int32_t *__restrict__ rows,
                                                                             const int32_t *__restrict__ count,
                                                                             const int64_t *__restrict__ row_ptr,
                                                                             int32_t *__restrict__ col,
                                                                             float *__restrict__ dist) {
    constexpr int P = CAP / 16, SEG = 16, RUN = 512;
    extern __shared__ uint32_t sort_smem_packed[];
    uint32_t (*sk)[CAP] = reinterpret_cast<uint32_t (*)[CAP]>(sort_smem_packed);
    float *sv = reinterpret_cast<float *>(sort_smem_packed + 2 * CAP);
    const int tid = threadIdx.x, lane = tid & 31;
    const int nrows = *count;
    for (int w = blockIdx.x; w < nrows; w += gridDim.x) {
        const int r = rows[w];
        const int64_t b = row_ptr[r];
        const int len = (int)min(row_ptr[r + 1] - b, (int64_t)CAP);  // rows of this class fit
        {
            uint32_t key[SEG];
            float val[SEG];
#pragma unroll
            for (int c = 0; c < SEG; ++c) {
                const int i = c * P + tid;
                key[c] = i < len ? ((uint32_t)col[b + i] << PACK_BITS) | (uint32_t)i : 0u;
                val[c] = i < len ? dist[b + i] : 0.f;
            }
            __syncthreads();  // the previous row's write-back has read sk / sv
#pragma unroll
            for (int c = 0; c < SEG; ++c) {
                const int i = c * P + tid;
                if (i < len) {
                    sk[0][swz<16>(i)] = key[c];
                    sv[i] = val[c];
                }
            }
        }
        __syncthreads();
        const int base = (tid >> 5) * RUN;
        if (base < len) {
            uint32_t key[16];
#pragma unroll
            for (int e = 0; e < 16; ++e) {
                const int i = lane * 16 + e;
                key[e] = base + i < len ? sk[0][base + swz<16>(i)] : 0xffffffffu;
            }
            warp_sort_keys<16>(key, lane);
            __syncwarp();
#pragma unroll
            for (int e = 0; e < 16; ++e) sk[0][base + swz<16>(lane * 16 + e)] = key[e];
        }
        __syncthreads();
        int cur = 0;
        for (int run = RUN; run < len; run <<= 1) {
            merge_round_keys<SEG>(sk[cur], sk[cur ^ 1], len, run, tid);
            __syncthreads();
            cur ^= 1;
        }
#pragma unroll
        for (int c = 0; c < SEG; ++c) {
            const int i = c * P + tid;
            if (i < len) {
                const uint32_t kk = sk[cur][swz<16>(i)];
                col[b + i] = (int32_t)(kk >> PACK_BITS);
                dist[b + i] = sv[kk & PACK_POS];
            }
        }
    }
}

// Warp per row, <= 32 entries: bitonic network across lanes.
__global__ void k_sort_small(const int32_t *__restrict__ rows, const int32_t *__restrict__ count,
                             const int64_t *__restrict__ row_ptr, int32_t *__restrict__ col,
                             float *__restrict__ dist) {
    int w = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    if (w >= *count) return;
    int r = rows[w];
    int64_t b = row_ptr[r];
    int len = (int)(row_ptr[r + 1] - b);
    int key = lane < len ? col[b + lane] : INT_MAX;
    float val = lane < len ? dist[b + lane] : 0.f;
    warp_sort32(key, val, lane);
    if (lane < len) {
        col[b + lane] = key;
        dist[b + lane] = val;
    }
}
// Long rows: gather (row rank, col) keys and sort them globally.
__global__ void k_big_gather(const int32_t *__restrict__ rows, int nbig, const int64_t *__restrict__ row_ptr,
                             const int64_t *__restrict__ big_off, const int32_t *__restrict__ col,
                             uint64_t *__restrict__ keys, uint32_t *__restrict__ vals) {
    int w = blockIdx.x;
    if (w >= nbig) return;
    int r = rows[w];
    int64_t b = row_ptr[r], len = row_ptr[r + 1] - b, o = big_off[w];
    for (int64_t i = threadIdx.x; i < len; i += blockDim.x) {
        keys[o + i] = ((uint64_t)w << 32) | (uint32_t)col[b + i];
        vals[o + i] = (uint32_t)i;
    }
}
__global__ void k_big_apply(const int32_t *__restrict__ rows, int nbig, const int64_t *__restrict__ row_ptr,
                            const int64_t *__restrict__ big_off, const uint64_t *__restrict__ keys,
                            const uint32_t *__restrict__ vals, int32_t *__restrict__ col, float *__restrict__ dist,
                            float *__restrict__ tmpd) {
    int w = blockIdx.x;
    if (w >= nbig) return;
    int r = rows[w];
    int64_t b = row_ptr[r], len = row_ptr[r + 1] - b, o = big_off[w];
    for (int64_t i = threadIdx.x; i < len; i += blockDim.x) tmpd[o + i] = dist[b + vals[o + i]];
    __syncthreads();
    for (int64_t i = threadIdx.x; i < len; i += blockDim.x) {
        col[b + i] = (int32_t)(uint32_t)(keys[o + i] & 0xffffffffull);
        dist[b + i] = tmpd[o + i];
    }
}
__global__ void k_big_lengths(const int32_t *__restrict__ rows, int nbig, const int64_t *__restrict__ row_ptr,
                              int64_t *__restrict__ lens) {
    int w = blockIdx.x * blockDim.x + threadIdx.x;
    if (w < nbig) lens[w] = row_ptr[rows[w] + 1] - row_ptr[rows[w]];
}

inline unsigned grid_for(int64_t n, int t) { return (unsigned)ceil_div(n > 0 ? n : 1, t); }

// Row-sort kernels: dynamic shared memory allowed and CTAs resident per SM,
// found once (before any capture) and kept.  [0]: (key, value) kernels, [1]:
// packed keys.
struct SortGrids {
    int warp_per_sm[2][5] = {};   // k_sort_warp<2 .. 16> for classes 1 .. 4
    int merge_per_sm[2][8] = {};  // k_sort_merge for classes 5 .. 7
};
const SortGrids &sort_grids() {
    static const SortGrids g = [] {
        SortGrids r;
        auto warp = [&](int pk, int c, auto kern) {
            CT_CHECK_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&r.warp_per_sm[pk][c], kern,
                                                                        32 * SORT_WARPS, 0));
            r.warp_per_sm[pk][c] = std::max(r.warp_per_sm[pk][c], 1);
        };
        auto merge = [&](int pk, int c, auto kern, int cap) {
            const int smem = (pk ? 12 : 16) * cap;
            if (smem > 48 * 1024)
                CT_CHECK_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
            CT_CHECK_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&r.merge_per_sm[pk][c], kern, cap / 16, smem));
            r.merge_per_sm[pk][c] = std::max(r.merge_per_sm[pk][c], 1);
        };
        warp(0, 1, k_sort_warp<2>);
        warp(0, 2, k_sort_warp<4>);
        warp(0, 3, k_sort_warp<8>);
        warp(0, 4, k_sort_warp<16>);
        merge(0, 5, k_sort_merge<1024>, 1024);
        merge(0, 6, k_sort_merge<2048>, 2048);
        merge(0, 7, k_sort_merge<SORT_MID>, SORT_MID);
        warp(1, 1, k_sort_warp_packed<2>);
        warp(1, 2, k_sort_warp_packed<4>);
        warp(1, 3, k_sort_warp_packed<8>);
        warp(1, 4, k_sort_warp_packed<16>);
        merge(1, 5, k_sort_merge_packed<1024>, 1024);
        merge(1, 6, k_sort_merge_packed<2048>, 2048);
        merge(1, 7, k_sort_merge_packed<SORT_MID>, SORT_MID);
        return r;
    }();
    return g;
}

// The sorts of the rows in classes 0 .. kSortClasses - 2 (class lists of
// stride n, their counts on the device) of a graph whose columns are below
// ncols.  hc: the same counts on the host -- classes without rows are skipped
// and grids sized to the rows; null: every class launched on a full grid (the
// kernels loop over the rows the device counted).
void launch_class_sorts(const int32_t *lists, const int32_t *counts, const int32_t *hc, int64_t n, int64_t ncols,
                        const int64_t *row_ptr, int32_t *col, float *dist, cudaStream_t s) {
    const SortGrids &g = sort_grids();
    const int pk = ncols < PACK_MAX_COLS ? 1 : 0;
    if (!hc || hc[0]) {
        k_sort_small<<<grid_for((hc ? hc[0] : n) * 32, 256), 256, 0, s>>>(lists, counts, row_ptr, col, dist);
        CT_COUNT_LAUNCH();
    }
    auto launch = [&](int c, auto kern, int threads, int smem, int per_sm, int rows_per_cta) {
        if (hc && !hc[c]) return;
        const int64_t full = (int64_t)num_sms() * per_sm;
        const int64_t blocks = hc ? std::min<int64_t>(ceil_div((int64_t)hc[c], rows_per_cta), full) : full;
        kern<<<(unsigned)blocks, threads, smem, s>>>(lists + (int64_t)c * n, counts + c, row_ptr, col, dist);
        CT_COUNT_LAUNCH();
    };
    constexpr int WT = 32 * SORT_WARPS;
    if (pk) {
        launch(1, k_sort_warp_packed<2>, WT, 0, g.warp_per_sm[1][1], SORT_WARPS);
        launch(2, k_sort_warp_packed<4>, WT, 0, g.warp_per_sm[1][2], SORT_WARPS);
        launch(3, k_sort_warp_packed<8>, WT, 0, g.warp_per_sm[1][3], SORT_WARPS);
        launch(4, k_sort_warp_packed<16>, WT, 0, g.warp_per_sm[1][4], SORT_WARPS);
        launch(5, k_sort_merge_packed<1024>, 1024 / 16, 12 * 1024, g.merge_per_sm[1][5], 1);
        launch(6, k_sort_merge_packed<2048>, 2048 / 16, 12 * 2048, g.merge_per_sm[1][6], 1);
        launch(7, k_sort_merge_packed<SORT_MID>, SORT_MID / 16, 12 * SORT_MID, g.merge_per_sm[1][7], 1);
    } else {
        launch(1, k_sort_warp<2>, WT, 0, g.warp_per_sm[0][1], SORT_WARPS);
        launch(2, k_sort_warp<4>, WT, 0, g.warp_per_sm[0][2], SORT_WARPS);
        launch(3, k_sort_warp<8>, WT, 0, g.warp_per_sm[0][3], SORT_WARPS);
        launch(4, k_sort_warp<16>, WT, 0, g.warp_per_sm[0][4], SORT_WARPS);
        launch(5, k_sort_merge<1024>, 1024 / 16, 16 * 1024, g.merge_per_sm[0][5], 1);
        launch(6, k_sort_merge<2048>, 2048 / 16, 16 * 2048, g.merge_per_sm[0][6], 1);
        launch(7, k_sort_merge<SORT_MID>, SORT_MID / 16, 16 * SORT_MID, g.merge_per_sm[0][7], 1);
    }
}

}  // namespace

void sort_rows(const int64_t *row_ptr, int64_t n, int64_t ncols, int32_t *col, float *dist, int64_t nnz,
               cudaStream_t s) {
    if (n <= 0 || nnz <= 0) return;
    DBuf<int32_t> lists(kSortClasses * n, s), counts(kSortClasses, s);
    CT_CHECK_CUDA(cudaMemsetAsync(counts.p, 0, kSortClasses * sizeof(int32_t), s));
    k_row_classes<<<grid_for(n, 256), 256, 0, s>>>(row_ptr, n, lists.p, counts.p);
    CT_COUNT_LAUNCH();
    int32_t hc[kSortClasses];
    to_host(hc, counts.p, kSortClasses, s);
    launch_class_sorts(lists.p, counts.p, hc, n, ncols, row_ptr, col, dist, s);
    constexpr int BIG = kSortClasses - 1;
    if (hc[BIG]) {
        int nb = hc[BIG];
        const int32_t *big = lists.p + BIG * n;
        DBuf<int64_t> lens(nb, s), off(nb, s), tot(1, s);
        k_big_lengths<<<grid_for(nb, 256), 256, 0, s>>>(big, nb, row_ptr, lens.p);
        CT_COUNT_LAUNCH();
        exclusive_scan_i64(lens.p, off.p, nb, tot.p, s);
        int64_t total = 0;
        to_host(&total, tot.p, 1, s);
        DBuf<uint64_t> k1(total, s), k2(total, s);
        DBuf<uint32_t> v1(total, s), v2(total, s);
        DBuf<float> td(total, s);
        k_big_gather<<<nb, 256, 0, s>>>(big, nb, row_ptr, off.p, col, k1.p, v1.p);
        CT_COUNT_LAUNCH();
        int bits = 32;
        while ((int64_t(1) << (bits - 32)) < nb) ++bits;
        radix_sort_pairs64(k1.p, v1.p, k2.p, v2.p, total, bits, s);
        k_big_apply<<<nb, 256, 0, s>>>(big, nb, row_ptr, off.p, k1.p, v1.p, col, dist, td.p);
        CT_COUNT_LAUNCH();
    }
    CT_LAUNCH_CHECK();
}

QParams make_qparams(const ct_tree *t, double eps, int include_self) {
    QParams q;
    q.eps64 = eps;
    q.eps2_64 = eps * eps;
    q.include_self = include_self;
    float ef = (float)eps;
    if ((double)ef < eps) ef = nextafterf(ef, INFINITY);
    q.eps_up = ef;
    if (t->metric == CT_LEVENSHTEIN_U8 || t->metric == CT_HAMMING_B1) {
        double fl = floor(eps);
        q.lev_k = fl > 1e9 ? 1000000000 : (int)fl;
        return q;
    }
    const double e2 = q.eps2_64;
    if (eps == 0.0) {
        q.mode = 1;
    } else if (e2 >= 0x1p115) {
        q.mode = 3;
    } else if (e2 < 0x1p-100 || e2 > 0x1p100) {
        q.mode = 2;
    } else {
        q.mode = 0;
        double lo = eps * (1.0 - 1e-3), hi = eps * (1.0 + 1e-3);
        double lo2 = lo * lo, hi2 = hi * hi;
        float l = (float)lo2, h = (float)hi2;
        if ((double)l > lo2) l = nextafterf(l, 0.0f);
        if ((double)h < hi2) h = nextafterf(h, INFINITY);
        q.lo2 = l;
        q.hi2 = h;
        // error bound of the canonical fp32 sum: one rounding per FMA of a
        // 16-float chunk (8), the chunk sum, one per chunk of the running
        // total, the rounded differences; doubled
        const double m = 2.0 * ((double)(t->dp / 16) + 16.0) * 0x1p-24;
        const double cl = e2 * (1.0 - m), ch = e2 * (1.0 + m);
        float a = (float)cl, b = (float)ch;
        if ((double)a > cl) a = nextafterf(a, 0.0f);
        if ((double)b < ch) b = nextafterf(b, INFINITY);
        q.c_lo = a;
        q.c_hi = b;
    }
    return q;
}

// Traversal launch shape: L2 uses blocks of TRAV_WARPS warps, edit distance
// one warp per block; both are capped at a resident-sized grid.
struct TravLaunch {
    int blocks, warps;
};
TravLaunch trav_launch_config(bool l2, int64_t G) {
    TravLaunch tl;
    if (l2) {
        tl.blocks = (int)std::min<int64_t>(ceil_div(G, TRAV_WARPS), (int64_t)num_sms() * 8);
        tl.blocks = std::max(tl.blocks, 1);
        tl.warps = tl.blocks * TRAV_WARPS;
    } else {
        // a warp per block, as many as an SM holds: the later rounds' stored
        // ranges can outnumber the groups
        tl.blocks = (int)std::max<int64_t>(1, (int64_t)num_sms() * 32);
        tl.warps = tl.blocks;
    }
    return tl;
}

// First pool size: 256 candidate blocks per point (or 512 per group), at most
// a quarter of the free device memory, plus one chunk per warp.
int64_t pool_capacity_guess(int64_t n, int64_t G, const TravLaunch &tl) {
    int64_t want = std::max<int64_t>(256 * n, G * 512);
    size_t fr = 0, tot = 0;
    if (cudaMemGetInfo(&fr, &tot) == cudaSuccess) {
        int64_t lim = (int64_t)(fr / 4 / sizeof(uint32_t));
        if (lim > 0 && want > lim) want = lim;
    } else {
        cudaGetLastError();
    }
    return want + (int64_t)(tl.warps + 1) * POOL_CHUNK;
}

// Clears the pool counters and launches the traversal over `order` (global
// group ids; allocates nothing).  L2: a round over the groups with a step
// limit, then TRAV_ROUNDS rounds over the ranges the previous round stored
// (`spill`: two buffers of spill_cap items and two counters; the last round
// has no limit), so that no single long walk sets the time.  Each warp's
// pool chunk carries over between rounds (`cursors`: one per warp of the
// grid).  Hamming and edit distance: a single cloud, the same rounds (one
// warp per block; edit-distance walks stop sooner: their steps cost more).
void launch_traversal(const Views &V, int64_t G, int max_dp, int max_len, bool l2, const int32_t *order,
                      const Pool &P, int2 *stacks, int cap, const TravLaunch &tl, unsigned long long *st,
                      int32_t *err, int32_t *next_group, int4 *const spill[2], unsigned long long *spill_cnt, int spill_cap,
                      longlong2 *cursors, cudaStream_t s, int32_t *gvisit = nullptr, const int4 *resumed = nullptr,
                      const unsigned long long *n_resumed = nullptr, int resumed_cap = 0) {
    // P.next .. P.overflow are the four 64-bit words of one counter block
    // (kept when a resume list is walked on, as are gvisit and the cursors)
    CT_CHECK_CUDA(cudaMemsetAsync(next_group, 0, sizeof(int32_t), s));
    if (!resumed) {
        CT_CHECK_CUDA(cudaMemsetAsync(P.next, 0, 4 * sizeof(unsigned long long), s));
        if (gvisit && G > 0) CT_CHECK_CUDA(cudaMemsetAsync(gvisit, 0, (size_t)G * sizeof(int32_t), s));
    }
    if (G == 0) return;
    if (l2) {
        const size_t tsm = (size_t)TRAV_WARPS * max_dp * sizeof(float);
        if (tsm > 48 * 1024) allow_smem(k_traverse_l2, kTravSmemMost);
        CT_CHECK_CUDA(cudaMemsetAsync(spill_cnt, 0, 2 * sizeof(unsigned long long), s));
        for (int r = 0; r <= TRAV_ROUNDS; ++r) {
            const int4 *in = r ? spill[(r - 1) & 1] : resumed;
            const unsigned long long *in_cnt = r ? spill_cnt + ((r - 1) & 1) : n_resumed;
            const int in_cap = r ? spill_cap : resumed_cap;
            Spill out{nullptr, spill_cnt + (r & 1), spill_cap, INT_MAX};
            if (r < TRAV_ROUNDS) {
                out.items = spill[r & 1];
                out.limit = r ? TRAV_LIMIT : TRAV_LIMIT0;
            }
            if (r) {
                CT_CHECK_CUDA(cudaMemsetAsync(next_group, 0, sizeof(int32_t), s));
                CT_CHECK_CUDA(cudaMemsetAsync(spill_cnt + (r & 1), 0, sizeof(unsigned long long), s));
            }
            k_traverse_l2<<<tl.blocks, TRAV_WARPS * 32, tsm, s>>>(V, order, (int)G, in, in_cnt, in_cap, out, P,
                                                                   cursors, stacks, cap, st, err, next_group,
                                                                   gvisit, max_dp >> 2);
            CT_COUNT_LAUNCH();
            CT_LAUNCH_CHECK();
        }
    } else {  // Hamming or edit distance: one cloud, the same rounds (a warp per block)
        TreeView tv = V.tv[0];
        tv.group_order = order;
        const bool ham = tv.wp != 0;
        CT_CHECK_CUDA(cudaMemsetAsync(spill_cnt, 0, 2 * sizeof(unsigned long long), s));
        const int rounds = ham ? TRAV_ROUNDS : TRAV_ROUNDS_LEV;
        for (int r = 0; r <= rounds; ++r) {
            const int4 *in = r ? spill[(r - 1) & 1] : resumed;
            const unsigned long long *in_cnt = r ? spill_cnt + ((r - 1) & 1) : n_resumed;
            const int in_cap = r ? spill_cap : resumed_cap;
            Spill out{nullptr, spill_cnt + (r & 1), spill_cap, INT_MAX};
            if (r < rounds) {
                out.items = spill[r & 1];
                out.limit = ham ? (r ? TRAV_LIMIT : TRAV_LIMIT0) : (r ? TRAV_LIMIT_LEV : TRAV_LIMIT0_LEV);
            }
            if (r) {
                CT_CHECK_CUDA(cudaMemsetAsync(next_group, 0, sizeof(int32_t), s));
                CT_CHECK_CUDA(cudaMemsetAsync(spill_cnt + (r & 1), 0, sizeof(unsigned long long), s));
            }
            if (ham) {
                k_traverse_ham<<<tl.blocks, 32, 0, s>>>(tv, V.qp[0], in, in_cnt, in_cap, out, P, cursors, stacks,
                                                        cap, st, err, next_group, gvisit);
            } else {
                switch (lev_words_for(max_len)) {
#define CT_TL(WW) \
    case WW: k_traverse_lev<WW><<<tl.blocks, 32, 0, s>>>(tv, V.qp[0], in, in_cnt, in_cap, out, P, cursors, stacks, cap, st, err, next_group, gvisit); break;
                    CT_TL(1) CT_TL(2) CT_TL(4) CT_TL(8) CT_TL(16)
#undef CT_TL
                }
            }
            CT_COUNT_LAUNCH();
            CT_LAUNCH_CHECK();
        }
    }
}

// Leaf kernel and item length per cloud.  precision 0: FP32 tiles; 1: tensor-
// core tiles where the rows allow (L2, at most 128 floats); 2: the autotuned
// choice of the cloud's row-length class (a default until tuned).
std::mutex g_tune_mu;
LeafChoice g_tune[kDpClasses] = {{-1, kItem}, {-1, kItem}, {-1, kItem}, {-1, kItem}, {-1, kItem}, {-1, kItem}};

int dp_class(int dp) { return dp <= 4 ? 0 : dp <= 16 ? 1 : dp <= 32 ? 2 : dp <= 64 ? 3 : dp <= 128 ? 4 : 5; }

LeafChoice tuned_choice(int dp) {
    std::lock_guard<std::mutex> lk(g_tune_mu);
    LeafChoice e = g_tune[dp_class(dp)];
    if (e.use_tc < 0) e.use_tc = dp >= 32;
    return e;
}
void tune_set(int cls, LeafChoice c) {
    std::lock_guard<std::mutex> lk(g_tune_mu);
    g_tune[cls] = c;
}
void tune_reset() {
    std::lock_guard<std::mutex> lk(g_tune_mu);
    for (auto &e : g_tune) e = LeafChoice{-1, kItem};
}
LeafChoice leaf_choice(const ct_tree *t, int precision) {
    if (t->metric != CT_L2_F32 || t->dp > 128 || precision == 0) return LeafChoice{0, kItem};
    if (precision == 1) return LeafChoice{1, kItemTC};
    LeafChoice c = tuned_choice(t->dp);
    if (c.item_len < 32 || c.item_len > kItem) c.item_len = kItem;
    return c;
}

// Global walk order of several clouds: groups by decreasing radius relative
// to their cloud's eps.
__global__ void k_radius_keys(int G, const float *__restrict__ group_radius, float inv_eps, int gbase,
                              uint32_t *__restrict__ keys, uint32_t *__restrict__ vals) {
    const int g = blockIdx.x * blockDim.x + threadIdx.x;
    if (g >= G) return;
    keys[gbase + g] = ~__float_as_uint(fmaxf(group_radius[g] * inv_eps, 0.f));
    vals[gbase + g] = (uint32_t)(gbase + g);
}

// Relative row_ptr of one cloud from the concatenated one.
__global__ void k_rel_rows(int64_t n1, const int64_t *__restrict__ grow, int64_t *__restrict__ out) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n1) out[i] = grow[i] - grow[0];
}

void query_multi(int C, const ct_tree *const *trees, const QParams *qps, cudaStream_t s, QueryOut *outs,
                 int precision, const ct_predictor *pred, Probe *probe) {
    if (C < 1 || C > kMaxClouds) CT_FAIL(CT_EINVAL, "between 1 and %d clouds per batch", kMaxClouds);
    const bool l2 = trees[0]->metric == CT_L2_F32;
    const bool ham = trees[0]->metric == CT_HAMMING_B1;
    if (C > 1 && !l2) CT_FAIL(CT_EINVAL, "edit-distance and Hamming trees are queried one at a time");
    // the clouds' groups and rows, concatenated
    Views V;
    std::memset(&V, 0, sizeof(V));
    V.nc = C;
    int max_dp = 4, max_fp_dp = 4, max_depth = 0, max_len = 0, min_len = kItemTC;
    bool any_tc = false, any_fp = false;
    for (int c = 0; c < C; ++c) {
        const ct_tree *tc = trees[c];
        if ((tc->metric == CT_L2_F32) != l2) CT_FAIL(CT_EINVAL, "a batch mixes metrics");
        V.tv[c] = view_of(tc);
        V.qp[c] = qps[c];
        const LeafChoice ch = leaf_choice(tc, precision);
        V.use_tc[c] = (uint8_t)ch.use_tc;
        V.item_len[c] = (int16_t)ch.item_len;
        any_tc |= ch.use_tc != 0;
        any_fp |= ch.use_tc == 0;
        min_len = std::min(min_len, ch.item_len);
        V.gbase[c + 1] = V.gbase[c] + tc->n_groups;
        V.rbase[c + 1] = V.rbase[c] + tc->n;
        max_dp = std::max(max_dp, tc->dp);
        if (!ch.use_tc) max_fp_dp = std::max(max_fp_dp, tc->dp);
        max_depth = std::max(max_depth, tc->depth);
        max_len = std::max(max_len, tc->max_len);
    }
    if (V.rbase[C] >= 0x7fffffffLL) CT_FAIL(CT_EOVERFLOW, "a batch above 2^31 points");
    // fp16 rows of the clouds that take the tensor-core filter
    DBuf<uint4> h16s;
    DBuf<float> f16s;  // per cloud: means (dp), {s, s eps_up, -, -}, norms (n, rounded up to 4)
    if (any_tc) {
        ProfScope ps("rows_f16", s);
        int64_t rows = 0, floats = 0;
        for (int c = 0; c < C; ++c) {
            if (!V.use_tc[c]) continue;
            const int dp = trees[c]->dp;
            rows += trees[c]->n * (8 * ((dp + 63) / 64));  // rows of 64-half K blocks
            floats += dp + 4 + ceil_div(trees[c]->n, 4) * 4;
        }
        h16s = DBuf<uint4>((size_t)(rows ? rows : 1), s);
        f16s = DBuf<float>((size_t)(floats ? floats : 1), s);
        DBuf<float> partial((size_t)C * H16_MB * 128, s);
        H16Out ho{};
        rows = floats = 0;
        bool any = false;
        for (int c = 0; c < C; ++c) {
            if (!V.use_tc[c]) continue;
            const ct_tree *tc = trees[c];
            if (tc->n == 0) continue;  // no work items
            any = true;
            const int dp = tc->dp, kp = 64 * ((dp + 63) / 64);
            ho.h16[c] = h16s.p + rows;
            ho.mean[c] = f16s.p + floats;
            ho.scal[c] = ho.mean[c] + dp;
            ho.n16[c] = ho.scal[c] + 4;
            rows += tc->n * (kp / 8);
            floats += dp + 4 + ceil_div(tc->n, 4) * 4;
            V.h16[c] = ho.h16[c];
            V.n16[c] = ho.n16[c];
            V.s16[c] = ho.scal[c];
        }
        if (any) {
            k_h16_sums<<<dim3(H16_MB, (unsigned)C), H16_T, 0, s>>>(V, partial.p);
            CT_COUNT_LAUNCH();
            CT_LAUNCH_CHECK();
            k_h16_means<<<(unsigned)C, 128, 0, s>>>(V, ho, partial.p);
            CT_COUNT_LAUNCH();
            CT_LAUNCH_CHECK();
            k_to_h16<<<grid_for(V.rbase[C] * 16, H16_T), H16_T, 0, s>>>(V, ho);
            CT_COUNT_LAUNCH();
            CT_LAUNCH_CHECK();
        }
    }
    const int64_t n = V.rbase[C];
    const int G = V.gbase[C];
    const ct_tree *t = trees[0];  // edit distance: the only cloud
    DBuf<unsigned long long> st(ST_N, s);
    CT_CHECK_CUDA(cudaMemsetAsync(st.p, 0, ST_N * sizeof(unsigned long long), s));
    int32_t *err = reinterpret_cast<int32_t *>(st.p + ST_ERR);
    QueryOut all;  // the concatenated CSR of all clouds
    struct AllGuard {  // releases its arrays unless they were handed to the caller
        QueryOut &q;
        cudaStream_t s;
        bool armed = true;
        ~AllGuard() {
            if (!armed) return;
            dfree(q.row_ptr, s);
            dfree(q.col, s);
            dfree(q.dist, s);
        }
    } all_guard{all, s};

    // learned form: row capacities and the traversal order from the predictor
    LearnedPlan lp;
    if (pred && !probe && n > 0) {
        ProfScope ps("predict", s);
        learned_plan(pred, C, trees, qps, V.rbase, V.gbase, s, lp);
    }
    // walk order: predicted walk length, else decreasing radius (relative to eps)
    DBuf<uint32_t> okeys, ovals;
    const int32_t *order = lp.group_order.p;
    if (!order && C == 1) order = t->group_order;
    if (!order && G > 0) {
        okeys = DBuf<uint32_t>(G, s);
        ovals = DBuf<uint32_t>(G, s);
        for (int c = 0; c < C; ++c) {
            const int Gc = trees[c]->n_groups;
            if (!Gc) continue;
            k_radius_keys<<<grid_for(Gc, 256), 256, 0, s>>>(Gc, trees[c]->group_radius,
                                                            (float)(1.0 / std::max(qps[c].eps64, 1e-30)),
                                                            V.gbase[c], okeys.p, ovals.p);
            CT_COUNT_LAUNCH();
        }
        DBuf<uint32_t> tk(G, s), tvv(G, s);
        radix_sort_pairs(okeys.p, ovals.p, tk.p, tvv.p, G, 32, s);
        order = reinterpret_cast<const int32_t *>(ovals.p);
    }
    int32_t *gvisit = probe ? probe->gvisit : nullptr;

    const int W = l2 || ham ? 1 : lev_words_for(t->max_len);
    // 1. traversal into the candidate pool, which grows when it runs out
    const int cap = 32 * (max_depth + 2);
    TravLaunch tl = trav_launch_config(l2, G);
    DBuf<int2> stacks((size_t)tl.warps * cap, s);
    DBuf<unsigned long long> ctr(4, s);
    DBuf<int32_t> next_group(1, s);
    // ranges of step-limited walks: two buffers and their counters
    const int spill_cap = (int)std::min<int64_t>(std::max<int64_t>(4 * G, 1 << 16), 1 << 20);
    DBuf<int4> spill_a(spill_cap, s), spill_b(spill_cap, s);
    DBuf<unsigned long long> spill_cnt(2, s);
    int4 *const spills[2] = {spill_a.p, spill_b.p};
    DBuf<longlong2> cursors(tl.warps, s);
    // a pool of whole chunks; work left when it runs out goes to a resume list
    // (at most every group, a full spill buffer a round and the stacks of the
    // warps; a list that is too short restarts the walk with a larger pool).
    // Every pass at least doubles the pool while half of the free memory allows
    // it; passes that go on and those that restart are counted together.
    constexpr int kPoolPasses = 16;
    int64_t pool_cap = ceil_div(pool_capacity_guess(n, G, tl), POOL_CHUNK) * POOL_CHUNK;
    const int resume_cap = (int)std::min<int64_t>(G + 2LL * spill_cap + 65536, 1 << 26);
    DBuf<uint32_t> pool;
    DBuf<int4> resume[2];
    DBuf<unsigned long long> rctr(3, s);  // entries of the two lists, whole groups
    DBuf<int32_t> seg_group, seg_count;
    DBuf<int64_t> seg_begin;
    unsigned long long hc[4] = {0, 0, 0, 0};
    int64_t seg_cap = 0;
    Pool P{};
    for (int pass = 0, passes = 1;; ++pass, ++passes) {
        // a segment per walk (groups, stored ranges) and per chunk a walk crosses
        const int64_t old_seg = seg_cap, nseg0 = pass ? (int64_t)(uint32_t)hc[1] : 0;
        seg_cap = old_seg + G + (int64_t)(l2 || ham ? TRAV_ROUNDS : TRAV_ROUNDS_LEV) * spill_cap + pool_cap / POOL_CHUNK + tl.warps + 16 +
                  (pass ? resume_cap : 0);
        auto grown = [&](auto &buf, int64_t cap_new, int64_t used) {  // a larger copy
            std::decay_t<decltype(buf)> b((size_t)cap_new, s);
            if (used) CT_CHECK_CUDA(cudaMemcpyAsync(b.p, buf.p, (size_t)used * sizeof(*b.p), cudaMemcpyDeviceToDevice, s));
            buf = std::move(b);
        };
        grown(pool, pool_cap, pass ? P.cap : 0);
        grown(seg_group, seg_cap, nseg0);
        grown(seg_count, seg_cap, nseg0);
        grown(seg_begin, seg_cap, nseg0);
        const int cur = pass & 1;  // this pass writes list cur and reads the other
        if (!resume[cur].p) resume[cur] = DBuf<int4>(resume_cap, s);
        CT_CHECK_CUDA(cudaMemsetAsync(rctr.p + cur, 0, sizeof(unsigned long long), s));
        CT_CHECK_CUDA(cudaMemsetAsync(rctr.p + 2, 0, sizeof(unsigned long long), s));
        P = Pool{pool.p, pool_cap, ctr.p, seg_group.p, seg_count.p, seg_begin.p,
                 reinterpret_cast<int32_t *>(ctr.p + 1), seg_cap, ctr.p + 2, reinterpret_cast<int32_t *>(ctr.p + 3),
                 resume[cur].p, rctr.p + cur, reinterpret_cast<int32_t *>(rctr.p + 2), resume_cap};
        {
            ProfScope ps("traverse", s);
            launch_traversal(V, G, max_dp, max_len, l2, order, P, stacks.p, cap, tl, st.p, err, next_group.p, spills,
                             spill_cnt.p, spill_cap, cursors.p, s, gvisit, pass ? resume[cur ^ 1].p : nullptr,
                             rctr.p + (cur ^ 1), resume_cap);
        }
        to_host(hc, ctr.p, 4, s);
        const uint32_t full = (uint32_t)hc[3];
        if (!full) break;
        if (passes > kPoolPasses) CT_FAIL(CT_ECUDA, "the candidate pool overflowed %d times", passes);
        // the size the walked groups ask for (the longest walks come first), at
        // least double, within half of the free memory if that is still larger
        int32_t whole = 0;
        to_host(&whole, reinterpret_cast<int32_t *>(rctr.p + 2), 1, s);
        const double walked = std::max(1.0, (double)(G - whole));
        double want = std::max(2.0 * (double)pool_cap,
                               1.1 * (double)hc[2] * (double)G / walked + 2.0 * (double)tl.warps * POOL_CHUNK);
        size_t fr = 0, tot = 0;
        if (cudaMemGetInfo(&fr, &tot) == cudaSuccess) {
            const double lim = std::max(1.125 * (double)pool_cap, (double)fr / 2 / sizeof(uint32_t));
            want = std::min(want, lim);
        } else {
            cudaGetLastError();
        }
        const unsigned long long used = (unsigned long long)pool_cap;
        pool_cap = ceil_div((int64_t)want, POOL_CHUNK) * POOL_CHUNK;
        if (full & 2u) {  // work was lost: from the start
            pass = -1;
            pool.reset();
            seg_cap = 0;
            CT_CHECK_CUDA(cudaMemsetAsync(st.p, 0, ST_N * sizeof(unsigned long long), s));
            continue;
        }
        // every chunk below the old capacity is taken; the counters of the walked part stay
        CT_CHECK_CUDA(cudaMemcpyAsync(ctr.p, &used, sizeof(used), cudaMemcpyHostToDevice, s));
        CT_CHECK_CUDA(cudaMemsetAsync(ctr.p + 3, 0, sizeof(unsigned long long), s));
        CT_CHECK_CUDA(cudaStreamSynchronize(s));  // `used` is on the stack
    }
    stacks.reset();
    resume[0].reset();
    resume[1].reset();
    const int64_t n_cand = (int64_t)hc[2];
    int nseg = (int)(uint32_t)hc[1];
    // each group's candidates in one range (segments become one per group)
    DBuf<uint32_t> gcand(n_cand ? n_cand : 1, s);
    DBuf<int32_t> gseg_group, gseg_count;
    DBuf<int64_t> gseg_begin;
    if (nseg && G) {
        gseg_group = DBuf<int32_t>(G, s);
        gseg_count = DBuf<int32_t>(G, s);
        gseg_begin = DBuf<int64_t>(G + 1, s);
        DBuf<int32_t> gfill(G, s);
        CT_CHECK_CUDA(cudaMemsetAsync(gseg_count.p, 0, G * sizeof(int32_t), s));
        CT_CHECK_CUDA(cudaMemsetAsync(gfill.p, 0, G * sizeof(int32_t), s));
        k_group_cand_counts<<<grid_for(nseg, 256), 256, 0, s>>>(nseg, seg_group.p, seg_count.p, gseg_count.p);
        CT_COUNT_LAUNCH();
        exclusive_scan_i32_to_i64(gseg_count.p, gseg_begin.p, G, gseg_begin.p + G, s);
        k_group_cand_copy<<<grid_for((int64_t)nseg * 32, 256), 256, 0, s>>>(nseg, seg_group.p, seg_begin.p, seg_count.p,
                                                                          gseg_begin.p, gfill.p, pool.p, gcand.p);
        CT_COUNT_LAUNCH();
        k_iota<<<grid_for(G, 256), 256, 0, s>>>(G, gseg_group.p);
        CT_COUNT_LAUNCH();
        CT_LAUNCH_CHECK();
        nseg = G;
    }
    pool.reset();
    seg_group.reset();
    seg_count.reset();
    seg_begin.reset();
    DBuf<uint32_t> emask(l2 && any_fp ? (n_cand ? n_cand : 1) : 0, s);
    // work items: the groups' candidate ranges in slices of the clouds' item lengths
    const int64_t max_items = nseg + n_cand / min_len + 1;
    DBuf<int32_t> icnt(nseg + 1, s), igroup(max_items, s), nitems(1, s);
    DBuf<int64_t> ioff(nseg + 1, s), ibeg(max_items, s), iend(max_items, s);
    Items items{igroup.p, ibeg.p, iend.p, nitems.p};
    CT_CHECK_CUDA(cudaMemsetAsync(nitems.p, 0, sizeof(int32_t), s));
    if (nseg) {
        k_item_counts<<<grid_for(nseg, 256), 256, 0, s>>>(V, nseg, gseg_group.p, gseg_count.p, icnt.p);
        CT_COUNT_LAUNCH();
        exclusive_scan_i32_to_i64(icnt.p, ioff.p, nseg, ioff.p + nseg, s);
        k_item_fill<<<grid_for(nseg, 256), 256, 0, s>>>(V, nseg, gseg_group.p, gseg_begin.p, gseg_count.p, ioff.p,
                                                       igroup.p, ibeg.p, iend.p, nitems.p);
        CT_COUNT_LAUNCH();
        CT_LAUNCH_CHECK();
    }
    DBuf<int32_t> rowcur(n + 1, s);
    uint32_t *cand_p = gcand.p;

    // alphabet of the strings (edit distance)
    DBuf<uint8_t> amap;
    int A = 0, qchunk = 32;
    if (!l2 && !ham) {
        DBuf<int32_t> present(256, s);
        CT_CHECK_CUDA(cudaMemsetAsync(present.p, 0, 256 * sizeof(int32_t), s));
        if (t->sbytes) {
            mark_bytes(t->sdata, t->sbytes, present.p, s);
        }
        int32_t hp[256];
        to_host(hp, present.p, 256, s);
        uint8_t hm[256];
        for (int c = 0; c < 256; ++c) hm[c] = 0;
        int a = 1;  // slot 0: bytes absent from the data (never matched)
        for (int c = 0; c < 256; ++c)
            if (hp[c]) hm[c] = (uint8_t)std::min(a++, 255);
        A = std::min(a, 256);
        if (a > 256) {  // every byte value occurs: identity map
            for (int c = 0; c < 256; ++c) hm[c] = (uint8_t)c;
            A = 256;
        }
        amap = DBuf<uint8_t>(256, s);
        CT_CHECK_CUDA(cudaMemcpyAsync(amap.p, hm, 256, cudaMemcpyHostToDevice, s));
        CT_CHECK_CUDA(cudaStreamSynchronize(s));
        size_t per_q = (size_t)A * W * sizeof(uint64_t);
        qchunk = (int)std::max<size_t>(1, std::min<size_t>(32, kLevSmemMost / per_q));
    }
    size_t lsm = l2 || ham ? 0 : (size_t)qchunk * A * W * sizeof(uint64_t);

    // one-pass emit: capacity region and overflow arena
    const bool capmode = pred && !probe && lp.one_pass;
    CapOut co{};
    DBuf<int32_t> c_fill;
    DBuf<uint2> c_ent;
    DBuf<uint4> o_ent;
    DBuf<unsigned long long> o_n;
    DBuf<uint8_t> lost;
    if (capmode) {
        const int64_t ct = lp.cap_total > 0 ? lp.cap_total : 1, oc = lp.arena > 0 ? lp.arena : 1;
        c_fill = DBuf<int32_t>(n + 1, s);
        c_ent = DBuf<uint2>(ct, s);
        o_ent = DBuf<uint4>(oc, s);
        o_n = DBuf<unsigned long long>(3, s);
        lost = DBuf<uint8_t>(n + 1, s);
        CT_CHECK_CUDA(cudaMemsetAsync(c_fill.p, 0, (n + 1) * sizeof(int32_t), s));
        CT_CHECK_CUDA(cudaMemsetAsync(o_n.p, 0, 3 * sizeof(unsigned long long), s));
        CT_CHECK_CUDA(cudaMemsetAsync(lost.p, 0, n + 1, s));
        co = CapOut{lp.cap_off.p, c_fill.p, c_ent.p, o_ent.p, o_n.p, lp.arena > 0 ? lp.arena : 0, lost.p};
    }

    // counters of the FP32 leaf launches, each used once (count: one or two; emit; rows emitted again)
    DBuf<unsigned long long> fp_ctr(8, s);
    if (any_fp) CT_CHECK_CUDA(cudaMemsetAsync(fp_ctr.p, 0, 8 * sizeof(unsigned long long), s));
    int fp_launches = 0;
    unsigned long long *const fp_n = fp_ctr.p + 7;  // entries of the edge list
    DBuf<uint2> fp_e;
    PairList fp_list{};
    bool fp_listed = false;  // the list holds every edge of the FP32 items
    unsigned long long fp_entries = 0;

    // 2. count pass
    DBuf<int32_t> deg(n + 1, s);
    CT_CHECK_CUDA(cudaMemsetAsync(deg.p, 0, (n + 1) * sizeof(int32_t), s));
    auto leaf = [&](bool emit, int64_t *row_ptr, int32_t *col, float *dist, const uint8_t *rowsel,
                    const Items &items, const ItemWave &wave) {
        if (G == 0 || nseg == 0) return;
        const CapOut cw = emit ? CapOut{} : co;
        if (l2) {
            leaf_l2_prepare();
            const bool sh = short_rows(max_fp_dp);
            const unsigned ctas = (unsigned)leaf_l2_grid(sh, wave.sampled == 1 ? ceil_div(max_items, WAVE_SAMPLE) : max_items);
            unsigned long long *const next = fp_ctr.p + fp_launches++;
            auto go = [&](auto kern) {
                kern<<<ctas, LEAF_T, leaf_smem(sh), s>>>(V, items, wave, next, cand_p, emask.p, deg.p, row_ptr, rowcur.p, col, dist, st.p, err, cw, rowsel, emit ? PairList{} : fp_list);
            };
            if (emit && sh) go(k_leaf_l2<true, KS_SHORT>);
            else if (emit) go(k_leaf_l2<true, KS_LONG>);
            else if (sh) go(k_leaf_l2<false, KS_SHORT>);
            else go(k_leaf_l2<false, KS_LONG>);
        } else if (ham) {
            const int nq = t->wp / 4;
            auto go = [&](auto kern, int qreg) {  // qreg: uint4 of a row in registers
                const size_t hsm = (size_t)32 * ((nq + qreg - 1) / qreg * qreg) * sizeof(uint4);
                kern<<<(unsigned)max_items, LEAF_T, hsm, s>>>(V.tv[0], V.qp[0], items, cand_p, deg.p, row_ptr, rowcur.p, col, dist, st.p, err, cw, rowsel);
            };
            if (nq <= 1) emit ? go(k_leaf_ham<true, 1>, 1) : go(k_leaf_ham<false, 1>, 1);
            else if (nq <= 2) emit ? go(k_leaf_ham<true, 2>, 2) : go(k_leaf_ham<false, 2>, 2);
            else emit ? go(k_leaf_ham<true, 4>, 4) : go(k_leaf_ham<false, 4>, 4);
        } else {
            switch (W) {
#define CT_LL(WW)                                                                                                      \
    case WW:                                                                                                           \
        if (lsm > 48 * 1024) {                                                                                         \
            allow_smem(k_leaf_lev<true, WW>, kLevSmemMost);                                                            \
            allow_smem(k_leaf_lev<false, WW>, kLevSmemMost);                                                           \
        }                                                                                                              \
        if (emit) k_leaf_lev<true, WW><<<(unsigned)max_items, LEAF_T, lsm, s>>>(V.tv[0], V.qp[0], amap.p, A, qchunk, items, cand_p, deg.p, row_ptr, rowcur.p, col, dist, st.p, err, cw, rowsel); \
        else k_leaf_lev<false, WW><<<(unsigned)max_items, LEAF_T, lsm, s>>>(V.tv[0], V.qp[0], amap.p, A, qchunk, items, cand_p, deg.p, row_ptr, rowcur.p, col, dist, st.p, err, cw, rowsel);    \
        break;
                CT_LL(1) CT_LL(2) CT_LL(4) CT_LL(8) CT_LL(16)
#undef CT_LL
            }
        }
        CT_COUNT_LAUNCH();
        CT_LAUNCH_CHECK();
    };
    // each cloud's count kernel: the tensor-core filter and decisions (L2 rows
    // of at most 128 floats) or FP32 tiles -- the same output; a mixed batch
    // splits its work items
    DBuf<int32_t> tg, fg, cnt2;
    DBuf<int64_t> tb, te, fb, fe;
    Items items_tc = items, items_fp = items;
    if (l2 && any_tc && any_fp) {
        tg = DBuf<int32_t>(max_items, s);
        fg = DBuf<int32_t>(max_items, s);
        cnt2 = DBuf<int32_t>(2, s);
        for (DBuf<int64_t> *d : {&tb, &te, &fb, &fe}) *d = DBuf<int64_t>(max_items, s);
        CT_CHECK_CUDA(cudaMemsetAsync(cnt2.p, 0, 2 * sizeof(int32_t), s));
        if (nseg) {
            k_item_split<<<grid_for(max_items, 256), 256, 0, s>>>(V, items, tg.p, tb.p, te.p, cnt2.p, fg.p, fb.p, fe.p,
                                                                   cnt2.p + 1);
            CT_COUNT_LAUNCH();
            CT_LAUNCH_CHECK();
        }
        items_tc = Items{tg.p, tb.p, te.p, cnt2.p};
        items_fp = Items{fg.p, fb.p, fe.p, cnt2.p + 1};
    }
    // Tensor-core items in waves: a wave's kept pairs go to a list, which is
    // decided before the next wave.  With many items a first wave of every
    // 32nd gives the pairs per item; the rest is cut into interleaved parts
    // (every part like the whole) whose lists fit pair_budget with a quarter
    // to spare.  A list that runs out is sized again from what the filter
    // counted, or its wave cut in two.  The two-pass form keeps its lists for
    // the emit pass while they fit; else that filters again.
    struct Wave {
        ItemWave wave;
        int64_t n;         // entries reserved
        DBuf<uint2> list;  // kept list (its first n entries), or empty
    };
    std::vector<Wave> waves;
    unsigned long long tc_stats[3] = {0, 0, 0};
    DBuf<unsigned long long> fctr(5, s);  // next item, entries, {valid pairs, kept pairs, rows}
    bool lists_kept = !capmode && !probe;
    int64_t filtered = 0;  // entries of the last filter
    const int64_t pair_slack = (int64_t)num_sms() * FT_EWARPS * FT_CHUNK;  // partly filled chunks
    int64_t pair_budget = 64ll << 20;  // one-pass: half a GB of pairs at a time
    if (any_tc) {
        size_t fr = 0, tot = 0;
        if (cudaMemGetInfo(&fr, &tot) == cudaSuccess) {
            const int64_t lim = (int64_t)(fr / 4 / sizeof(uint2));
            // the two-pass form gains by one list (no second filter pass)
            pair_budget = std::max<int64_t>(1 << 20, lists_kept ? lim : std::min(lim, pair_budget));
        } else {
            cudaGetLastError();
        }
        if (capacity_budget() > 0) pair_budget = std::max<int64_t>(1, capacity_budget() / (int64_t)sizeof(uint2));
    }
    // filters a wave's items into a list of at least `want` entries (grown to
    // the need once that is known); false when the need exceeds `most`
    auto tc_filter = [&](const ItemWave &w, double want, DBuf<uint2> &list, bool stats, int64_t most) {
        for (;;) {
            const int64_t cap = ceil_div((int64_t)want, FT_CHUNK) * FT_CHUNK;
            if ((int64_t)list.n < cap) {
                list.reset();
                list = DBuf<uint2>((size_t)cap, s);
            }
            CT_CHECK_CUDA(cudaMemsetAsync(fctr.p, 0, 5 * sizeof(unsigned long long), s));
            const PairList pl{list.p, (int64_t)(list.n / FT_CHUNK * FT_CHUNK), fctr.p + 1, fctr.p + 2};
            const int ctas = (int)std::min<int64_t>(num_sms(), max_items);
            k_filter_tc<<<ctas, FT_T, kFtSmem, s>>>(V, items_tc, w, cand_p, pl, fctr.p, err);
            CT_COUNT_LAUNCH();
            CT_LAUNCH_CHECK();
            unsigned long long h[4];
            to_host(h, fctr.p + 1, 4, s);
            filtered = (int64_t)h[0];
            if (filtered <= pl.cap) {
                if (stats)
                    for (int k = 0; k < 3; ++k) tc_stats[k] += h[1 + k];
                return true;
            }
            const int64_t need = filtered + pair_slack;  // the next run's chunks may be filled differently
            if (need > most) return false;
            want = (double)need;
        }
    };
    auto tc_pairs = [&](int mode, uint2 *list, int64_t entries, const uint8_t *rowsel) {
        if (!entries) return;
        const PairList pl{list, entries, nullptr, nullptr};
        const int blocks = (int)std::min<int64_t>(ceil_div(entries, 256), (int64_t)num_sms() * 16);
        switch (mode) {
#define CT_KP(M) case M: k_pairs<M><<<blocks, 256, 0, s>>>(V, pl, deg.p, co, all.row_ptr, rowcur.p, all.col, all.dist, rowsel, st.p, err); break;
            CT_KP(PAIRS_COUNT) CT_KP(PAIRS_PLACE) CT_KP(PAIRS_EMIT)
#undef CT_KP
        }
        CT_COUNT_LAUNCH();
        CT_LAUNCH_CHECK();
    };
    auto count_tc = [&]() {
        ProfScope ps("leaf_count_tc", s);
        CT_CHECK_CUDA(cudaFuncSetAttribute(k_filter_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kFtSmem));
        if (!G || !nseg) return;
        int64_t kept_entries = 0;
        DBuf<uint2> list;
        // waves still to run (a stack); a wave whose list would exceed the
        // budget is cut in two interleaved halves
        std::vector<ItemWave> todo;
        const bool sample = max_items > 32ll * num_sms();
        todo.push_back(sample ? ItemWave{1, 0, 1} : ItemWave{0, 0, 1});
        const int64_t most = pair_budget + pair_slack;
        double want = std::min((double)most, (double)pair_slack + std::min(512.0 * (double)n, (double)(16 << 20)));
        bool sampled = !sample;
        while (!todo.empty()) {
            const ItemWave w = todo.back();
            todo.pop_back();
            const bool can_cut = w.parts < (1 << 20);
            if (!tc_filter(w, want, list, true, can_cut ? most : INT64_MAX)) {
                todo.push_back(ItemWave{w.sampled, w.part + w.parts, 2 * w.parts});
                todo.push_back(ItemWave{w.sampled, w.part, 2 * w.parts});
                want = (double)most;
                continue;
            }
            tc_pairs(capmode ? PAIRS_PLACE : PAIRS_COUNT, list.p, filtered, nullptr);
            waves.push_back(Wave{w, filtered, DBuf<uint2>()});
            kept_entries += filtered;
            if (lists_kept && kept_entries <= most) {
                waves.back().list = std::move(list);
            } else if (lists_kept) {
                lists_kept = false;
                for (auto &x : waves) x.list.reset();
            }
            if (!sampled && todo.empty()) {  // the rest, from the sample's pairs
                sampled = true;
                const double total = 1.25 * (WAVE_SAMPLE - 1) * std::max(1.0, (double)tc_stats[1]);
                const int parts = (int)std::min(65536.0, std::ceil(total / (double)pair_budget));
                for (int k = parts - 1; k >= 0; --k) todo.push_back(ItemWave{2, k, parts});
                want = total / parts + (double)pair_slack;
            }
        }
    };
    // Count pass of the other kernels.  FP32 tiles of the two-pass form list
    // their edges for the emit pass (8 bytes each; dp <= 128), which then decides
    // only those again instead of every pair of an edge-bearing block and query.
    // The list holds 192 edges per point at most, within an eighth of the free
    // memory (a denser graph's emit pass takes the blocks' masks).  Where that is
    // more than 2 GB (1.4 million points), every 32nd item is counted first and
    // its edges size the list, with half as much again to spare; a sample of
    // fewer points does not fill the chip (with a line at 64 MB, 130k x 3: 3.00 ->
    // 3.19 ms; at 1 GB, 1M x 128: 91.3 -> 92.2).
    // The list is no condition: without the memory for it, or when it runs out,
    // the emit pass takes the masks.
    auto count_other = [&](const Items &items) {
        ProfScope ps("leaf_count", s);
        const ItemWave every{0, 0, 1};
        auto count = [&](const ItemWave &w) { leaf(false, nullptr, nullptr, nullptr, nullptr, items, w); };
        if (!l2 || capmode || probe || max_fp_dp > 128 || n == 0) return count(every);
        const int64_t slack = leaf_l2_slack(short_rows(max_fp_dp), max_items);
        int64_t most = 192 * n + slack;
        size_t fr = 0, tot = 0;
        if (cudaMemGetInfo(&fr, &tot) == cudaSuccess) most = std::min(most, (int64_t)(fr / 8 / sizeof(uint2)));
        else cudaGetLastError();
        if (capacity_budget() > 0) most = std::min<int64_t>(most, capacity_budget() / (int64_t)sizeof(uint2));
        most = std::max<int64_t>(most, 1);
        auto room = [&](int64_t cap, int64_t used) {  // a list of cap entries with the first `used` of the last one
            DBuf<uint2> e;
            try {
                e = DBuf<uint2>((size_t)cap, s);
            } catch (const Error &x) {
                if (x.st != CT_ENOMEM) throw;
            }
            if (e.p && used) CT_CHECK_CUDA(cudaMemcpyAsync(e.p, fp_e.p, (size_t)used * sizeof(uint2), cudaMemcpyDeviceToDevice, s));
            fp_e = std::move(e);
            fp_list = fp_e.p ? PairList{fp_e.p, cap, fp_n, nullptr} : PairList{};
        };
        if (most <= (2ll << 30) / (int64_t)sizeof(uint2)) {
            room(most, 0);
            return count(every);
        }
        room(std::min(most, 192 * n / WAVE_SAMPLE + slack), 0);
        count(ItemWave{1, 0, 1});
        if (fp_list.e) {
            to_host(&fp_entries, fp_n, 1, s);
            const int64_t used = (int64_t)fp_entries, all = WAVE_SAMPLE * used + slack;
            if (used <= fp_list.cap && all <= most) {
                room(std::min(most, all + all / 2), used);
            } else {
                fp_e.reset();
                fp_list = PairList{};
            }
        }
        count(ItemWave{2, 0, 1});
    };
    if (!l2 || !any_tc) {
        count_other(items);
    } else {
        count_tc();
        if (any_fp) count_other(items_fp);
        if (capmode)  // the entries placed are the degrees
            for (int c = 0; c < C; ++c)
                if (V.use_tc[c] && trees[c]->n)
                    CT_CHECK_CUDA(cudaMemcpyAsync(deg.p + V.rbase[c], c_fill.p + V.rbase[c],
                                                  (size_t)trees[c]->n * sizeof(int32_t), cudaMemcpyDeviceToDevice, s));
    }
    // emit pass (rowsel: of the selected rows)
    auto emit = [&](const uint8_t *rowsel) {
        if (fp_listed) tc_pairs(PAIRS_EMIT, fp_e.p, (int64_t)fp_entries, rowsel);
        else if (!l2 || any_fp) leaf(true, all.row_ptr, all.col, all.dist, rowsel, items_fp, ItemWave{0, 0, 1});
        DBuf<uint2> list;
        for (auto &w : waves) {
            if (lists_kept) {
                tc_pairs(PAIRS_EMIT, w.list.p, w.n, rowsel);
                continue;
            }
            tc_filter(w.wave, (double)(w.n + pair_slack), list, false, INT64_MAX);
            tc_pairs(PAIRS_EMIT, list.p, filtered, rowsel);
        }
    };

    unsigned long long tc_placed = 0;  // one-pass form: entries of the tensor-core clouds' rows
    auto finish_stats = [&]() {
        unsigned long long hs[ST_N];
        to_host(hs, st.p, ST_N, s);
        prof_flush();
        if (hs[ST_ERR] & 32)
            CT_FAIL(CT_ETIMEOUT, "a bounded wait of the tensor-core leaf kernel gave up (code %llu)", hs[ST_ERR]);
        if (hs[ST_ERR]) CT_FAIL(CT_ECUDA, "internal consistency check failed in the query (code %llu)", hs[ST_ERR]);
        if (hs[ST_PLACED] != tc_placed)
            CT_FAIL(CT_ECUDA, "internal consistency check failed in the query (%llu entries of %llu found)", tc_placed, hs[ST_PLACED]);
        all.stats.traversal_evals = (int64_t)hs[ST_TRAV];
        all.stats.leaf_pairs = (int64_t)(hs[ST_PAIRS] + tc_stats[0]);
        all.stats.guard_fp64 = (int64_t)hs[ST_GUARD];
        all.stats.recheck_fp32 = (int64_t)tc_stats[1];
        all.stats.emit_pairs = (int64_t)hs[ST_EMIT];
        all.stats.leaf_rows = (int64_t)(hs[ST_ROWS] + tc_stats[2]);
        all.stats.guard_band = (int64_t)hs[ST_BAND];
        all.stats.lev_columns = (int64_t)hs[ST_COLS];
        all.stats.candidates = n_cand;
    };

    if (probe) {  // labels for fitting the predictor
        if (n && probe->deg) CT_CHECK_CUDA(cudaMemcpyAsync(probe->deg, deg.p, n * sizeof(int32_t), cudaMemcpyDeviceToDevice, s));
        finish_stats();
        return;
    }

    // 3. scan -> row_ptr, then emit
    int64_t *row_ptr = (int64_t *)dmalloc((size_t)(n + 1) * sizeof(int64_t), s);
    all.row_ptr = row_ptr;
    exclusive_scan_i32_to_i64(deg.p, row_ptr, n + 1, nullptr, s);
    int64_t nnz = 0;
    if (fp_list.e) to_host_async(&fp_entries, fp_n, 1, s);
    to_host(&nnz, row_ptr + n, 1, s);
    fp_listed = fp_list.e && (int64_t)fp_entries <= fp_list.cap;
    all.nnz = nnz;
    all.col = (int32_t *)dmalloc((size_t)(nnz ? nnz : 1) * sizeof(int32_t), s);
    all.dist = (float *)dmalloc((size_t)(nnz ? nnz : 1) * sizeof(float), s);
    if (capmode) {
        // one-pass emit: move the capacity region and the arena into the CSR;
        // rows that lost entries are emitted again, exactly
        unsigned long long hv[3] = {0, 0, 0};
        {
            ProfScope ps("compact", s);
            if (n) {
                k_cap_rows<<<grid_for(n, 256), 256, 0, s>>>(n, row_ptr, lp.cap_off.p, c_fill.p, lost.p, o_n.p + 1, err);
                CT_COUNT_LAUNCH();
                k_compact<<<grid_for(n * 32, 256), 256, 0, s>>>(n, row_ptr, lp.cap_off.p, lost.p, c_ent.p, all.col,
                                                                all.dist);
                CT_COUNT_LAUNCH();
                CT_LAUNCH_CHECK();
            }
            to_host(hv, o_n.p, 3, s);
            if (any_tc && any_fp) {
                std::vector<int64_t> first(C + 1);  // the clouds' first entries
                for (int c = 0; c <= C; ++c) to_host_async(&first[c], row_ptr + V.rbase[c], 1, s);
                CT_CHECK_CUDA(cudaStreamSynchronize(s));
                for (int c = 0; c < C; ++c)
                    if (V.use_tc[c]) tc_placed += (unsigned long long)(first[c + 1] - first[c]);
            } else if (any_tc) {
                tc_placed = (unsigned long long)nnz;
            }
            const int64_t used = std::min<int64_t>((int64_t)hv[0], co.ovf_cap);
            if (used > 0) {
                k_ovf_scatter<<<grid_for(used, 256), 256, 0, s>>>(used, o_ent.p, lost.p, row_ptr, all.col, all.dist,
                                                                  err);
                CT_COUNT_LAUNCH();
                CT_LAUNCH_CHECK();
            }
        }
        all.stats.overflow_rows = (int64_t)hv[1];
        all.stats.reemit_rows = (int64_t)hv[2];
        c_ent.reset();
        if (hv[2]) {
            ProfScope ps("reemit", s);
            CT_CHECK_CUDA(cudaMemsetAsync(rowcur.p, 0, (n + 1) * sizeof(int32_t), s));
            emit(lost.p);
            k_check_rows_sel<<<grid_for(n, 256), 256, 0, s>>>(n, row_ptr, rowcur.p, lost.p, err);
            CT_COUNT_LAUNCH();
        }
    } else if (nnz) {
        ProfScope ps("leaf_emit", s);
        CT_CHECK_CUDA(cudaMemsetAsync(rowcur.p, 0, (n + 1) * sizeof(int32_t), s));
        emit(nullptr);
        k_check_rows<<<grid_for(n, 256), 256, 0, s>>>(n, row_ptr, rowcur.p, err);
        CT_COUNT_LAUNCH();
    }
    {
        ProfScope ps("row_sort", s);
        int64_t ncols = 0;  // columns index points of their own cloud
        for (int c = 0; c < C; ++c) ncols = std::max<int64_t>(ncols, trees[c]->n);
        sort_rows(row_ptr, n, ncols, all.col, all.dist, nnz, s);
    }
    finish_stats();
    if (C == 1) {
        outs[0] = all;
        all_guard.armed = false;
        return;
    }
    // several clouds: CSRs that view one shared allocation each of row
    // offsets (relative to the cloud), columns and distances
    std::vector<int64_t> hb(C + 1);
    for (int c = 0; c <= C; ++c) to_host_async(&hb[c], row_ptr + V.rbase[c], 1, s);
    CT_CHECK_CUDA(cudaStreamSynchronize(s));
    auto blocks = std::make_shared<SharedBlocks>(s);
    blocks->p[0] = dmalloc((size_t)(n + C) * sizeof(int64_t), s);
    int64_t *rel = (int64_t *)blocks->p[0];
    int32_t *colp = all.col;
    float *distp = all.dist;
    blocks->p[1] = colp;
    blocks->p[2] = distp;
    all.col = nullptr;  // the blocks own them now
    all.dist = nullptr;
    for (int c = 0; c < C; ++c) {
        const int64_t nc1 = trees[c]->n + 1, o = V.rbase[c] + c;
        k_rel_rows<<<grid_for(nc1, 256), 256, 0, s>>>(nc1, row_ptr + V.rbase[c], rel + o);
        CT_COUNT_LAUNCH();
        QueryOut &q = outs[c];
        q.row_ptr = rel + o;
        q.col = colp + hb[c];
        q.dist = distp + hb[c];
        q.nnz = hb[c + 1] - hb[c];
        q.stats = all.stats;
        q.shared = blocks;
    }
    CT_LAUNCH_CHECK();
    all.row_ptr = nullptr;
    all_guard.armed = false;
    dfree(row_ptr, s);  // stream ordered: after the relative copies
}

void query_plain(const ct_tree *t, const QParams &qp, cudaStream_t s, QueryOut &out) {
    query_multi(1, &t, &qp, s, &out, 0, nullptr, nullptr);
}

void query_tc(const ct_tree *t, const QParams &qp, cudaStream_t s, QueryOut &out) {
    query_multi(1, &t, &qp, s, &out, 1, nullptr, nullptr);
}

void set_guard_rows(int32_t *rows, unsigned long long *count, int64_t cap) {
    long long c = rows ? (long long)cap : 0;
    int32_t *r = rows;
    unsigned long long *n = rows ? count : nullptr;
    CT_CHECK_CUDA(cudaDeviceSynchronize());
    CT_CHECK_CUDA(cudaMemcpyToSymbol(g_guard_rows, &r, sizeof(r)));
    CT_CHECK_CUDA(cudaMemcpyToSymbol(g_guard_n, &n, sizeof(n)));
    CT_CHECK_CUDA(cudaMemcpyToSymbol(g_guard_cap, &c, sizeof(c)));
}

// ---------------------------------------------------------------- plans
//
// A batch of L2 clouds queried again and again over the same trees (a served
// set of point clouds): every buffer is sized once, from a sizing query plus
// a margin, so that a run enqueues the whole query -- walk, candidate ranges,
// count pass, scan, emit, row sort -- without reading anything back to the
// host.  A run can therefore be captured in a CUDA graph and replayed.  The
// leaf stage is one persistent launch over every cloud's (cloud, group) work
// items: each CTA first produces the items of a chunk of groups into a device
// work queue (in the walk order, which the predictor sets when one is given),
// then consumes queue slots; a slot is waited for, with a bounded number of
// polls, until its producer has published it.  Sizes that outgrow the plan, a
// wait that gives up, and rows too long for the in-place sorts are reported
// by the run's status word.

namespace {

constexpr int32_t Q_ERR_OVERFLOW = 128;  // a run outgrew one of the plan's capacities
constexpr int32_t Q_ERR_TIMEOUT = 256;   // a queue wait gave up

__device__ __forceinline__ int ld_acquire_i32(const int32_t *p) {
    int v;
    asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void st_release_i32(int32_t *p, int v) {
    asm volatile("st.release.gpu.global.s32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

// The leaf stage's work queue.  Counters: claim (next group chunk to
// produce), tail (slots reserved), head (next slot to consume), published
// (groups whose items are all written).
struct Queue {
    int32_t *claim, *tail, *head, *published;
    int32_t *ready;  // per slot: 1 once its item is written
    int32_t *group;
    int64_t *begin, *end;
    const int32_t *order;   // production order (global group ids)
    const int32_t *gcount;  // candidate blocks per group
    const int64_t *gbegin;  // first candidate of each group
    const int32_t *ctl;     // ctl[0] != 0: producers publish nothing (a test); ctl[1]: polls before a wait gives up
    int64_t cand_cap;       // candidate ranges beyond it were not copied
    int G, cap, produce;
};

// Producer: chunks of LEAF_T groups, one thread per group; a group's items
// are its candidate range cut at its cloud's item length.
__device__ __forceinline__ void queue_produce(const Views &V, const Queue &Q, int32_t *err) {
    __shared__ int s_c0;
    for (;;) {
        __syncthreads();
        if (threadIdx.x == 0) s_c0 = atomicAdd(Q.claim, LEAF_T);
        __syncthreads();
        const int c0 = s_c0;
        if (c0 >= Q.G) break;
        if (Q.ctl[0]) continue;  // withheld: the chunk is taken and nothing is published
        const int i = c0 + threadIdx.x;
        if (i < Q.G) {
            const int gg = Q.order[i];
            const int cnt = Q.gcount[gg];
            const int len = V.item_len[cloud_of_group(V, gg)];
            int k = (cnt + len - 1) / len;
            if (Q.gbegin[gg] + cnt > Q.cand_cap) {  // its range was not copied: no items
                atomicOr(err, Q_ERR_OVERFLOW);
                k = 0;
            }
            if (k > 0) {
                const int base = atomicAdd(Q.tail, k);
                const int64_t b0 = Q.gbegin[gg];
                for (int j = 0; j < k; ++j) {
                    const int slot = base + j;
                    if (slot >= Q.cap) {  // slots past the plan's capacity are never consumed
                        atomicOr(err, Q_ERR_OVERFLOW);
                        break;
                    }
                    Q.group[slot] = gg;
                    Q.begin[slot] = b0 + (int64_t)j * len;
                    Q.end[slot] = min(b0 + (int64_t)(j + 1) * len, b0 + cnt);
                    __threadfence();
                    st_release_i32(Q.ready + slot, 1);
                }
            }
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            __threadfence();
            atomicAdd(Q.published, min(LEAF_T, Q.G - c0));
        }
    }
}

// Consumer: the next slot, once published; -1 when the queue is exhausted
// (or a wait gave up: Q_ERR_TIMEOUT).
__device__ __forceinline__ int queue_next(const Queue &Q, int32_t *err) {
    __shared__ int s_it;
    __syncthreads();
    if (threadIdx.x == 0) {
        const int slot = atomicAdd(Q.head, 1);
        int it = -1;
        if (slot < Q.cap) {
            const unsigned limit = (unsigned)Q.ctl[1];
            for (unsigned poll = 0;; ++poll) {
                if (ld_acquire_i32(Q.ready + slot)) {
                    it = slot;
                    break;
                }
                if (ld_acquire_i32(Q.published) >= Q.G && slot >= ld_acquire_i32(Q.tail)) break;
                if (poll >= limit) {
                    atomicOr(err, Q_ERR_TIMEOUT);
                    break;
                }
                __nanosleep(poll < 64 ? 64 : 1024);
            }
            __threadfence();
        }
        s_it = it;
    }
    __syncthreads();
    return s_it;
}

// The FP32 tiles as one persistent launch over the queue (count pass:
// produce, then consume; emit pass: consume the complete queue again).
template <bool EMIT, int KS4>
__global__ void __launch_bounds__(LEAF_T, leaf_l2_ctas(KS4 == KS_SHORT)) k_leaf_l2_queue(
    const __grid_constant__ Views V, Queue Q, const uint32_t *__restrict__ cand, uint32_t *__restrict__ emask,
    int32_t *__restrict__ deg, const int64_t *__restrict__ row_ptr, int32_t *__restrict__ rowcur,
    int32_t *__restrict__ col, float *__restrict__ dist, unsigned long long *__restrict__ st,
    int32_t *__restrict__ err, PairList pl) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    LeafShared<KS4> &S = *reinterpret_cast<LeafShared<KS4> *>(smem_raw);
    if (EMIT && pl.e && (int64_t)*pl.n <= pl.cap) return;  // the count pass listed every edge: k_pairs emits them
    PairCursor pc;
    if (Q.produce) queue_produce(V, Q, err);
    const Items items{Q.group, Q.begin, Q.end, Q.tail};
    for (;;) {
        const int it = queue_next(Q, err);
        if (it < 0) break;
        leaf_l2_item<EMIT, KS4>(V, items, it, cand, emask, deg, row_ptr, rowcur, col, dist, st, err, CapOut{}, nullptr,
                                EMIT ? PairList{} : pl, pc, S);
    }
    if (!EMIT && pl.e) pair_close(pl, pc);
}

// Candidate ranges per group from the walk's segments (segment count read on
// the device; destinations checked against the plan's capacity).
__global__ void k_plan_cand_counts(const int32_t *__restrict__ nseg_dev, int64_t seg_cap,
                                   const int32_t *__restrict__ seg_group, const int32_t *__restrict__ seg_count,
                                   int32_t *__restrict__ gcnt) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t nseg = min((int64_t)*nseg_dev, seg_cap);
    if (i < nseg && seg_count[i] > 0) atomicAdd(gcnt + seg_group[i], seg_count[i]);
}
__global__ void k_plan_cand_copy(const int32_t *__restrict__ nseg_dev, int64_t seg_cap,
                                 const int32_t *__restrict__ seg_group, const int64_t *__restrict__ seg_begin,
                                 const int32_t *__restrict__ seg_count, const int64_t *__restrict__ goff,
                                 int32_t *__restrict__ gfill, const uint32_t *__restrict__ pool,
                                 uint32_t *__restrict__ gcand, int64_t cand_cap, int32_t *__restrict__ err) {
    const int64_t i = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    const int64_t nseg = min((int64_t)*nseg_dev, seg_cap);
    if (i >= nseg) return;
    const int g = seg_group[i], c = seg_count[i];
    int64_t base = 0;
    if (lane == 0) base = goff[g] + atomicAdd(gfill + g, c);
    base = __shfl_sync(0xffffffffu, base, 0);
    if (base + c > cand_cap) {
        if (lane == 0) atomicOr(err, Q_ERR_OVERFLOW);
        return;
    }
    const uint32_t *src = pool + seg_begin[i];
    for (int k = lane; k < c; k += 32) gcand[base + k] = src[k];
}
// The walk's own overflow flag, and the candidate total against the plan.
__global__ void k_plan_walk_check(const int32_t *__restrict__ pool_ovf, const int64_t *__restrict__ total,
                                  int64_t cand_cap, int32_t *__restrict__ err) {
    if (*pool_ovf || *total > cand_cap) atomicOr(err, Q_ERR_OVERFLOW);
}
// Edges above the plan's capacity: flagged, and every row emptied so that the
// emit pass writes nothing.
__global__ void k_plan_nnz_check(const int64_t *__restrict__ row_ptr, int64_t n, int64_t nnz_cap,
                                 int32_t *__restrict__ flag, int32_t *__restrict__ err) {
    if (row_ptr[n] > nnz_cap) {
        *flag = 1;
        atomicOr(err, Q_ERR_OVERFLOW);
    } else {
        *flag = 0;
    }
}
__global__ void k_plan_empty_rows(int64_t n1, const int32_t *__restrict__ flag, int64_t *__restrict__ row_ptr) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n1 && *flag) row_ptr[i] = 0;
}
// Rows longer than the in-place sorts take: their count against the plan,
// their lengths (zero past the count), then (after a scan) their entries
// against the plan's capacity.
__global__ void k_plan_big_lengths(const int32_t *__restrict__ rows, const int32_t *__restrict__ nbig_dev,
                                   int cap_rows, const int64_t *__restrict__ row_ptr, int64_t *__restrict__ lens,
                                   int32_t *__restrict__ err) {
    const int w = blockIdx.x * blockDim.x + threadIdx.x;
    const int nbig = *nbig_dev;
    if (w == 0 && nbig > cap_rows) atomicOr(err, Q_ERR_OVERFLOW);
    if (w < cap_rows) lens[w] = w < nbig ? row_ptr[rows[w] + 1] - row_ptr[rows[w]] : 0;
}
__global__ void k_plan_big_check(const int64_t *__restrict__ total, int64_t big_cap, int32_t *__restrict__ err,
                                 int32_t *__restrict__ skip) {
    *skip = *total > big_cap;
    if (*skip) atomicOr(err, Q_ERR_OVERFLOW);
}
// Keys (rank of the row in the list, column) of the long rows, in the
// plan's buffer (prefilled with keys that sort last).
__global__ void k_plan_big_gather(const int32_t *__restrict__ rows, const int32_t *__restrict__ nbig_dev, int cap_rows,
                                  const int32_t *__restrict__ skip, const int64_t *__restrict__ row_ptr,
                                  const int64_t *__restrict__ big_off, const int32_t *__restrict__ col,
                                  uint64_t *__restrict__ keys, uint32_t *__restrict__ vals) {
    const int w = blockIdx.x;
    if (w >= min(*nbig_dev, cap_rows) || *skip) return;
    const int r = rows[w];
    const int64_t b = row_ptr[r], len = row_ptr[r + 1] - b, o = big_off[w];
    for (int64_t i = threadIdx.x; i < len; i += blockDim.x) {
        keys[o + i] = ((uint64_t)w << 32) | (uint32_t)col[b + i];
        vals[o + i] = (uint32_t)i;
    }
}
__global__ void k_plan_big_apply(const int32_t *__restrict__ rows, const int32_t *__restrict__ nbig_dev, int cap_rows,
                                 const int32_t *__restrict__ skip, const int64_t *__restrict__ row_ptr,
                                 const int64_t *__restrict__ big_off, const uint64_t *__restrict__ keys,
                                 const uint32_t *__restrict__ vals, int32_t *__restrict__ col,
                                 float *__restrict__ dist, float *__restrict__ tmpd) {
    const int w = blockIdx.x;
    if (w >= min(*nbig_dev, cap_rows) || *skip) return;
    const int r = rows[w];
    const int64_t b = row_ptr[r], len = row_ptr[r + 1] - b, o = big_off[w];
    for (int64_t i = threadIdx.x; i < len; i += blockDim.x) tmpd[o + i] = dist[b + vals[o + i]];
    __syncthreads();
    for (int64_t i = threadIdx.x; i < len; i += blockDim.x) {
        col[b + i] = (int32_t)(uint32_t)(keys[o + i] & 0xffffffffull);
        dist[b + i] = tmpd[o + i];
    }
}

}  // namespace

struct PlanImpl {
    int C = 0;
    std::vector<const ct_tree *> trees;
    Views V;
    int64_t n = 0, max_cols = 0;  // rows of all clouds; points of the largest cloud
    int G = 0;
    int max_dp = 4, cap_stack = 0, spill_cap = 0, leaf_grid = 1;
    TravLaunch tl{1, 1};
    int64_t pool_cap = 0, seg_cap = 0, cand_cap = 0, item_cap = 0, nnz_cap = 0;
    int big_rows = 0;       // rows above the in-place sorts' length the plan sorts by radix
    int64_t big_cap = 0;    // their entries
    cudaStream_t s0 = 0;
    DBuf<int32_t> order;
    DBuf<unsigned long long> st, ctr;
    DBuf<int32_t> next_group, ctl, qctr, ready, igroup, gcount, gfill, deg, rowcur, empty_flag;
    DBuf<int2> stacks;
    DBuf<int4> spill_a, spill_b;
    DBuf<longlong2> cursors;
    DBuf<uint32_t> pool, gcand, emask;
    DBuf<int32_t> seg_group, seg_count, col, sort_lists, sort_counts;
    DBuf<int64_t> seg_begin, gbegin, ibeg, iend, sums, row_ptr, rel;
    DBuf<float> dist, big_tmpd;
    DBuf<uint2> pair_e;               // edges of the count pass, for the emit pass (rows of at most 128 floats)
    DBuf<unsigned long long> spill_cnt;
    DBuf<unsigned long long> pair_n;  // entries reserved
    DBuf<int64_t> big_lens, big_off;
    DBuf<uint64_t> big_k1, big_k2;
    DBuf<uint32_t> big_v1, big_v2;
    DBuf<int32_t> big_skip;
    cudaGraph_t graph = nullptr;
    cudaGraphExec_t exec = nullptr;
    ~PlanImpl() {
        if (exec) cudaGraphExecDestroy(exec);
        if (graph) cudaGraphDestroy(graph);
    }
};

namespace {
// One run of a plan: every launch on `s`, nothing read back, nothing allocated.
void plan_enqueue(PlanImpl &p, cudaStream_t s) {
    const Views &V = p.V;
    const int64_t n = p.n;
    const int G = p.G;
    unsigned long long *st = p.st.p;
    int32_t *err = reinterpret_cast<int32_t *>(st + ST_ERR);
    CT_CHECK_CUDA(cudaMemsetAsync(st, 0, ST_N * sizeof(unsigned long long), s));
    if (G == 0) {  // empty clouds only
        CT_CHECK_CUDA(cudaMemsetAsync(p.row_ptr.p, 0, (size_t)(n + 1) * sizeof(int64_t), s));
        CT_CHECK_CUDA(cudaMemsetAsync(p.rel.p, 0, (size_t)(n + p.C) * sizeof(int64_t), s));
        return;
    }
    Pool P{p.pool.p, p.pool_cap, p.ctr.p, p.seg_group.p, p.seg_count.p, p.seg_begin.p,
           reinterpret_cast<int32_t *>(p.ctr.p + 1), p.seg_cap, p.ctr.p + 2, reinterpret_cast<int32_t *>(p.ctr.p + 3)};
    int4 *const spills[2] = {p.spill_a.p, p.spill_b.p};
    // 1. the walk over every cloud's groups
    launch_traversal(V, G, p.max_dp, 0, true, p.order.p, P, p.stacks.p, p.cap_stack, p.tl, st, err, p.next_group.p,
                     spills, p.spill_cnt.p, p.spill_cap, p.cursors.p, s);
    k_plan_walk_check<<<1, 1, 0, s>>>(P.overflow, reinterpret_cast<const int64_t *>(P.total), p.cand_cap, err);
    CT_COUNT_LAUNCH();
    // 2. each group's candidates in one range
    CT_CHECK_CUDA(cudaMemsetAsync(p.gcount.p, 0, (size_t)G * sizeof(int32_t), s));
    CT_CHECK_CUDA(cudaMemsetAsync(p.gfill.p, 0, (size_t)G * sizeof(int32_t), s));
    k_plan_cand_counts<<<grid_for(p.seg_cap, 256), 256, 0, s>>>(P.nseg, p.seg_cap, P.seg_group, P.seg_count,
                                                              p.gcount.p);
    CT_COUNT_LAUNCH();
    exclusive_scan_i32_to_i64_into(p.gcount.p, p.gbegin.p, G, p.gbegin.p + G, p.sums.p, s);
    k_plan_cand_copy<<<grid_for(p.seg_cap * 32, 256), 256, 0, s>>>(P.nseg, p.seg_cap, P.seg_group, P.seg_begin,
                                                                  P.seg_count, p.gbegin.p, p.gfill.p, P.data,
                                                                  p.gcand.p, p.cand_cap, err);
    CT_COUNT_LAUNCH();
    // 3. count pass: one persistent launch producing and consuming the work queue
    CT_CHECK_CUDA(cudaMemsetAsync(p.qctr.p, 0, 4 * sizeof(int32_t), s));
    CT_CHECK_CUDA(cudaMemsetAsync(p.ready.p, 0, (size_t)p.item_cap * sizeof(int32_t), s));
    CT_CHECK_CUDA(cudaMemsetAsync(p.deg.p, 0, (size_t)(n + 1) * sizeof(int32_t), s));
    Queue Q{p.qctr.p, p.qctr.p + 1, p.qctr.p + 2, p.qctr.p + 3, p.ready.p, p.igroup.p, p.ibeg.p, p.iend.p,
            p.order.p, p.gcount.p, p.gbegin.p, p.ctl.p, p.cand_cap, G, (int)p.item_cap, 1};
    // (it lists the edges; the emit pass decides those again, or walks the queue when the list ran out)
    const bool sh = short_rows(p.max_dp);
    const PairList pl{p.pair_e.p, (int64_t)p.pair_e.n, p.pair_n.p, nullptr};
    CT_CHECK_CUDA(cudaMemsetAsync(p.pair_n.p, 0, sizeof(unsigned long long), s));
    auto leaf_queue = [&](auto kern, int64_t *rp) {
        kern<<<p.leaf_grid, LEAF_T, leaf_smem(sh), s>>>(V, Q, p.gcand.p, p.emask.p, p.deg.p, rp, p.rowcur.p, p.col.p,
                                                        p.dist.p, st, err, pl);
        CT_COUNT_LAUNCH();
    };
    if (sh) leaf_queue(k_leaf_l2_queue<false, KS_SHORT>, nullptr);
    else leaf_queue(k_leaf_l2_queue<false, KS_LONG>, nullptr);
    // 4. scan; a run above the plan's edge capacity empties every row
    exclusive_scan_i32_to_i64_into(p.deg.p, p.row_ptr.p, n + 1, nullptr, p.sums.p, s);
    k_plan_nnz_check<<<1, 1, 0, s>>>(p.row_ptr.p, n, p.nnz_cap, p.empty_flag.p, err);
    CT_COUNT_LAUNCH();
    k_plan_empty_rows<<<grid_for(n + 1, 256), 256, 0, s>>>(n + 1, p.empty_flag.p, p.row_ptr.p);
    CT_COUNT_LAUNCH();
    // 5. emit pass over the complete queue
    CT_CHECK_CUDA(cudaMemsetAsync(p.qctr.p + 2, 0, sizeof(int32_t), s));
    CT_CHECK_CUDA(cudaMemsetAsync(p.rowcur.p, 0, (size_t)(n + 1) * sizeof(int32_t), s));
    Q.produce = 0;
    if (sh) leaf_queue(k_leaf_l2_queue<true, KS_SHORT>, p.row_ptr.p);
    else leaf_queue(k_leaf_l2_queue<true, KS_LONG>, p.row_ptr.p);
    if (pl.e) {
        k_pairs<PAIRS_EMIT><<<num_sms() * 8, 256, 0, s>>>(V, pl, p.deg.p, CapOut{}, p.row_ptr.p, p.rowcur.p, p.col.p,
                                                          p.dist.p, nullptr, st, err);
        CT_COUNT_LAUNCH();
    }
    k_check_rows<<<grid_for(n, 256), 256, 0, s>>>(n, p.row_ptr.p, p.rowcur.p, err);
    CT_COUNT_LAUNCH();
    // 6. rows sorted in place (rows above the in-place sorts' length are reported)
    CT_CHECK_CUDA(cudaMemsetAsync(p.sort_counts.p, 0, kSortClasses * sizeof(int32_t), s));
    k_row_classes<<<grid_for(n, 256), 256, 0, s>>>(p.row_ptr.p, n, p.sort_lists.p, p.sort_counts.p);
    CT_COUNT_LAUNCH();
    launch_class_sorts(p.sort_lists.p, p.sort_counts.p, nullptr, n, p.max_cols, p.row_ptr.p, p.col.p, p.dist.p, s);
    {  // longer rows: one radix sort of (row rank, column) keys over the plan's capacity
        const int32_t *big = p.sort_lists.p + (int64_t)(kSortClasses - 1) * n;
        const int32_t *nbig = p.sort_counts.p + (kSortClasses - 1);
        k_plan_big_lengths<<<grid_for(p.big_rows, 256), 256, 0, s>>>(big, nbig, p.big_rows, p.row_ptr.p,
                                                                     p.big_lens.p, err);
        CT_COUNT_LAUNCH();
        exclusive_scan_i64(p.big_lens.p, p.big_off.p, p.big_rows, p.big_off.p + p.big_rows, s);
        k_plan_big_check<<<1, 1, 0, s>>>(p.big_off.p + p.big_rows, p.big_cap, err, p.big_skip.p);
        CT_COUNT_LAUNCH();
        CT_CHECK_CUDA(cudaMemsetAsync(p.big_k1.p, 0xff, (size_t)p.big_cap * sizeof(uint64_t), s));
        k_plan_big_gather<<<p.big_rows, 256, 0, s>>>(big, nbig, p.big_rows, p.big_skip.p, p.row_ptr.p, p.big_off.p,
                                                     p.col.p, p.big_k1.p, p.big_v1.p);
        CT_COUNT_LAUNCH();
        int bits = 32;
        while ((int64_t(1) << (bits - 32)) < p.big_rows) ++bits;
        radix_sort_pairs64(p.big_k1.p, p.big_v1.p, p.big_k2.p, p.big_v2.p, p.big_cap, bits, s);
        k_plan_big_apply<<<p.big_rows, 256, 0, s>>>(big, nbig, p.big_rows, p.big_skip.p, p.row_ptr.p, p.big_off.p,
                                                    p.big_k1.p, p.big_v1.p, p.col.p, p.dist.p, p.big_tmpd.p);
        CT_COUNT_LAUNCH();
    }
    // 7. each cloud's row offsets relative to its first row
    for (int c = 0; c < p.C; ++c) {
        const int64_t nc1 = p.trees[c]->n + 1;
        k_rel_rows<<<grid_for(nc1, 256), 256, 0, s>>>(nc1, p.row_ptr.p + V.rbase[c], p.rel.p + V.rbase[c] + c);
        CT_COUNT_LAUNCH();
    }
    CT_LAUNCH_CHECK();
}
}  // namespace

PlanImpl *plan_create(int C, const ct_tree *const *trees, const QParams *qps, int precision,
                      const ct_predictor *pred, float margin, bool use_graph, cudaStream_t s) {
    if (C < 1 || C > kMaxClouds) CT_FAIL(CT_EINVAL, "between 1 and %d clouds per plan", kMaxClouds);
    std::unique_ptr<PlanImpl> pp(new PlanImpl());
    PlanImpl &p = *pp;
    p.C = C;
    p.s0 = s;
    std::memset(&p.V, 0, sizeof(p.V));
    p.V.nc = C;
    int max_depth = 0, min_len = kItem;
    for (int c = 0; c < C; ++c) {
        const ct_tree *t = trees[c];
        if (t->metric != CT_L2_F32) CT_FAIL(CT_EINVAL, "plans take L2 trees only");
        p.trees.push_back(t);
        p.V.tv[c] = view_of(t);
        p.V.qp[c] = qps[c];
        p.V.use_tc[c] = 0;  // the persistent launch runs the FP32 tiles
        const int len = precision == 2 ? leaf_choice(t, 2).item_len : kItem;
        p.V.item_len[c] = (int16_t)len;
        min_len = std::min(min_len, len);
        p.V.gbase[c + 1] = p.V.gbase[c] + t->n_groups;
        p.V.rbase[c + 1] = p.V.rbase[c] + t->n;
        p.max_cols = std::max<int64_t>(p.max_cols, t->n);
        p.max_dp = std::max(p.max_dp, t->dp);
        max_depth = std::max(max_depth, t->depth);
    }
    if (p.V.rbase[C] >= 0x7fffffffLL) CT_FAIL(CT_EOVERFLOW, "a plan above 2^31 points");
    p.n = p.V.rbase[C];
    p.G = p.V.gbase[C];
    const int64_t n = p.n;
    const int G = p.G;
    // sizing query (the batch's own exact query, FP32 tiles)
    std::vector<QueryOut> outs((size_t)C);
    struct OutsGuard {  // the sizing query's CSRs are released on every path
        std::vector<QueryOut> &o;
        cudaStream_t s;
        ~OutsGuard() {
            for (auto &q : o) {
                if (!q.shared) {
                    dfree(q.row_ptr, s);
                    dfree(q.col, s);
                    dfree(q.dist, s);
                }
                q = QueryOut();
            }
        }
    } outs_guard{outs, s};
    query_multi(C, trees, qps, s, outs.data(), 0, pred, nullptr);
    const int64_t n_cand = outs[0].stats.candidates;
    int64_t nnz = 0, nbig = 0, big_entries = 0;
    {
        std::vector<int64_t> hrp;
        for (int c = 0; c < C; ++c) {
            nnz += outs[c].nnz;
            hrp.resize((size_t)trees[c]->n + 1);
            to_host(hrp.data(), outs[c].row_ptr, hrp.size(), s);
            for (size_t i = 0; i + 1 < hrp.size(); ++i) {
                const int64_t len = hrp[i + 1] - hrp[i];
                if (len > SORT_MID) {
                    ++nbig;
                    big_entries += len;
                }
            }
        }
    }
    const double m = std::max(0.0, (double)margin);
    p.big_rows = (int)std::min<int64_t>((int64_t)std::ceil((double)nbig * (1.0 + m)) + 16, 0x7fffffff);
    p.big_cap = (int64_t)std::ceil((double)big_entries * (1.0 + m)) + 4096;
    p.tl = trav_launch_config(true, G);
    p.cap_stack = 32 * (max_depth + 2);
    p.spill_cap = (int)std::min<int64_t>(std::max<int64_t>(4 * (int64_t)G, 1 << 16), 1 << 20);
    p.cand_cap = (int64_t)std::ceil((double)n_cand * (1.0 + m)) + 4096;
    p.pool_cap = p.cand_cap + (int64_t)(p.tl.warps + 1) * POOL_CHUNK;
    p.seg_cap = G + (int64_t)TRAV_ROUNDS * p.spill_cap + p.pool_cap / POOL_CHUNK + p.tl.warps + 16;
    p.item_cap = std::min<int64_t>(G + p.cand_cap / min_len + 1, 0x7fffffff);
    p.nnz_cap = (int64_t)std::ceil((double)nnz * (1.0 + m)) + 4096;
    // walk order: the predictor's (groups by decreasing predicted walk
    // length), else decreasing radius relative to eps
    p.order = DBuf<int32_t>(G ? G : 1, s);
    if (G) {
        LearnedPlan lp;
        if (pred) learned_plan(pred, C, trees, qps, p.V.rbase, p.V.gbase, s, lp);
        if (lp.group_order.p) {
            CT_CHECK_CUDA(cudaMemcpyAsync(p.order.p, lp.group_order.p, (size_t)G * sizeof(int32_t),
                                          cudaMemcpyDeviceToDevice, s));
        } else {
            DBuf<uint32_t> k1(G, s), v1(G, s), k2(G, s), v2(G, s);
            for (int c = 0; c < C; ++c) {
                const int Gc = trees[c]->n_groups;
                if (!Gc) continue;
                k_radius_keys<<<grid_for(Gc, 256), 256, 0, s>>>(Gc, trees[c]->group_radius,
                                                                (float)(1.0 / std::max(qps[c].eps64, 1e-30)),
                                                                p.V.gbase[c], k1.p, v1.p);
                CT_COUNT_LAUNCH();
            }
            radix_sort_pairs(k1.p, v1.p, k2.p, v2.p, G, 32, s);
            CT_CHECK_CUDA(cudaMemcpyAsync(p.order.p, v1.p, (size_t)G * sizeof(int32_t), cudaMemcpyDeviceToDevice, s));
        }
    }
    // buffers
    p.st = DBuf<unsigned long long>(ST_N, s);
    p.ctr = DBuf<unsigned long long>(4, s);
    p.next_group = DBuf<int32_t>(1, s);
    p.spill_cnt = DBuf<unsigned long long>(2, s);
    p.ctl = DBuf<int32_t>(2, s);
    p.qctr = DBuf<int32_t>(4, s);
    p.empty_flag = DBuf<int32_t>(1, s);
    p.stacks = DBuf<int2>((size_t)p.tl.warps * p.cap_stack, s);
    p.spill_a = DBuf<int4>(p.spill_cap, s);
    p.spill_b = DBuf<int4>(p.spill_cap, s);
    p.cursors = DBuf<longlong2>(p.tl.warps, s);
    p.pool = DBuf<uint32_t>(p.pool_cap, s);
    p.seg_group = DBuf<int32_t>(p.seg_cap, s);
    p.seg_count = DBuf<int32_t>(p.seg_cap, s);
    p.seg_begin = DBuf<int64_t>(p.seg_cap, s);
    p.gcand = DBuf<uint32_t>(p.cand_cap, s);
    p.emask = DBuf<uint32_t>(p.cand_cap, s);
    p.gcount = DBuf<int32_t>(G ? G : 1, s);
    p.gfill = DBuf<int32_t>(G ? G : 1, s);
    p.gbegin = DBuf<int64_t>(G + 1, s);
    p.sums = DBuf<int64_t>(std::max<int64_t>(scan_scratch_entries(std::max<int64_t>(n + 1, G)), 1), s);
    p.ready = DBuf<int32_t>(p.item_cap, s);
    p.igroup = DBuf<int32_t>(p.item_cap, s);
    p.ibeg = DBuf<int64_t>(p.item_cap, s);
    p.iend = DBuf<int64_t>(p.item_cap, s);
    p.deg = DBuf<int32_t>(n + 1, s);
    p.rowcur = DBuf<int32_t>(n + 1, s);
    p.row_ptr = DBuf<int64_t>(n + 1, s);
    p.rel = DBuf<int64_t>(n + C, s);
    p.col = DBuf<int32_t>(p.nnz_cap, s);
    p.dist = DBuf<float>(p.nnz_cap, s);
    p.sort_lists = DBuf<int32_t>((size_t)kSortClasses * (n ? n : 1), s);
    p.sort_counts = DBuf<int32_t>(kSortClasses, s);
    p.big_lens = DBuf<int64_t>(p.big_rows, s);
    p.big_off = DBuf<int64_t>(p.big_rows + 1, s);
    p.big_k1 = DBuf<uint64_t>(p.big_cap, s);
    p.big_k2 = DBuf<uint64_t>(p.big_cap, s);
    p.big_v1 = DBuf<uint32_t>(p.big_cap, s);
    p.big_v2 = DBuf<uint32_t>(p.big_cap, s);
    p.big_tmpd = DBuf<float>(p.big_cap, s);
    p.big_skip = DBuf<int32_t>(1, s);
    const int32_t ctl0[2] = {0, 1 << 20};  // about a second of polls
    CT_CHECK_CUDA(cudaMemcpyAsync(p.ctl.p, ctl0, sizeof(ctl0), cudaMemcpyHostToDevice, s));
    // persistent grid: the FP32 tiles' resident CTAs on every SM
    leaf_l2_prepare();
    {
        int per_sm = 0;
        const bool sh = short_rows(p.max_dp);
        auto resident = [&](auto kern) {
            int b = 0;
            CT_CHECK_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)leaf_smem(sh)));
            CT_CHECK_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, kern, LEAF_T, leaf_smem(sh)));
            per_sm = per_sm ? std::min(per_sm, b) : b;
        };
        if (sh) {
            resident(k_leaf_l2_queue<false, KS_SHORT>);
            resident(k_leaf_l2_queue<true, KS_SHORT>);
        } else {
            resident(k_leaf_l2_queue<false, KS_LONG>);
            resident(k_leaf_l2_queue<true, KS_LONG>);
        }
        p.leaf_grid = std::max(1, num_sms() * std::max(per_sm, 1));
        p.pair_n = DBuf<unsigned long long>(1, s);
        if (p.max_dp <= 128) {  // the edges, and what each warp leaves of its last entries; without room, none
            try {
                p.pair_e = DBuf<uint2>((size_t)(p.nnz_cap + (int64_t)p.leaf_grid * (LEAF_T / 32) * l2_chunk(sh)), s);
            } catch (const Error &x) {
                if (x.st != CT_ENOMEM) throw;
            }
        }
    }
    {
        const size_t tsm = (size_t)TRAV_WARPS * p.max_dp * sizeof(float);
        if (tsm > 48 * 1024) allow_smem(k_traverse_l2, kTravSmemMost);
        sort_grids();  // row-sort attributes set outside the capture
    }
    CT_CHECK_CUDA(cudaStreamSynchronize(s));
    if (use_graph) {
        // captured on a private stream (the caller's may be the legacy
        // default stream, which cannot be captured); launched on any stream
        cudaStream_t cs = nullptr;
        CT_CHECK_CUDA(cudaStreamCreateWithFlags(&cs, cudaStreamNonBlocking));
        struct StreamGuard {
            cudaStream_t s;
            ~StreamGuard() { cudaStreamDestroy(s); }
        } sg{cs};
        CT_CHECK_CUDA(cudaStreamBeginCapture(cs, cudaStreamCaptureModeRelaxed));
        try {
            plan_enqueue(p, cs);
        } catch (...) {
            cudaGraph_t g = nullptr;
            cudaStreamEndCapture(cs, &g);
            if (g) cudaGraphDestroy(g);
            cudaGetLastError();
            throw;
        }
        CT_CHECK_CUDA(cudaStreamEndCapture(cs, &p.graph));
        CT_CHECK_CUDA(cudaGraphInstantiate(&p.exec, p.graph, 0));
    }
    return pp.release();
}

void plan_launch(PlanImpl *p, cudaStream_t s) {
    if (p->exec)
        CT_CHECK_CUDA(cudaGraphLaunch(p->exec, s));
    else
        plan_enqueue(*p, s);
}

void plan_set_wait(PlanImpl *p, int withhold, int max_polls) {
    const int32_t v[2] = {withhold ? 1 : 0, max_polls};
    CT_CHECK_CUDA(cudaDeviceSynchronize());  // no run of the plan is in flight
    CT_CHECK_CUDA(cudaMemcpy(p->ctl.p, v, sizeof(v), cudaMemcpyHostToDevice));
}

int plan_clouds(const PlanImpl *p) { return p->C; }
int64_t plan_rows(const PlanImpl *p, int c) { return p->trees[c]->n; }

// Status of the last run (synchronises `s`): CT_OK and the clouds' CSR views
// into the plan's buffers, or the failure.
ct_status plan_result(PlanImpl *p, cudaStream_t s, QueryOut *outs) {
    unsigned long long hs[ST_N];
    to_host(hs, p->st.p, ST_N, s);
    const int32_t e = (int32_t)hs[ST_ERR];
    if (e & Q_ERR_TIMEOUT) {
        set_error("a work-queue wait of the plan's leaf stage gave up (its producer never published)");
        return CT_ETIMEOUT;
    }
    if (e & Q_ERR_OVERFLOW) {
        set_error("the run outgrew the plan's capacities (candidates, work items, edges or row length); "
                  "create a new plan");
        return CT_EOVERFLOW;
    }
    if (e) {
        set_error("internal consistency check failed in the plan's run (code %d)", e);
        return CT_ECUDA;
    }
    std::vector<int64_t> hb((size_t)p->C + 1);
    for (int c = 0; c <= p->C; ++c) to_host_async(&hb[c], p->row_ptr.p + p->V.rbase[c], 1, s);
    CT_CHECK_CUDA(cudaStreamSynchronize(s));
    auto blocks = std::make_shared<SharedBlocks>(s);  // views: the plan keeps the memory
    for (int c = 0; c < p->C; ++c) {
        QueryOut &q = outs[c];
        q.row_ptr = p->rel.p + p->V.rbase[c] + c;
        q.col = p->col.p + hb[c];
        q.dist = p->dist.p + hb[c];
        q.nnz = hb[c + 1] - hb[c];
        q.stats = ct_query_stats{};
        q.stats.traversal_evals = (int64_t)hs[ST_TRAV];
        q.stats.leaf_pairs = (int64_t)hs[ST_PAIRS];
        q.stats.guard_fp64 = (int64_t)hs[ST_GUARD];
        q.stats.emit_pairs = (int64_t)hs[ST_EMIT];
        q.stats.leaf_rows = (int64_t)hs[ST_ROWS];
        q.stats.guard_band = (int64_t)hs[ST_BAND];
        q.shared = blocks;
    }
    return CT_OK;
}

void plan_free(PlanImpl *p) {
    if (!p) return;
    cudaStream_t s = p->s0;
    cudaStreamSynchronize(s);
    delete p;
    cudaStreamSynchronize(s);
}

}  // namespace ct

// ----------------------------------------------------------------------
// Degrees without device allocation.
//
// Some callers cannot let a library allocate device memory: an application
// whose own allocator owns the whole device and hands out fixed budgets, or a
// latency-bound loop where an allocation's implicit synchronisation, or its
// possible failure, is not acceptable.  For them the count pass (tree walk +
// FP32 leaf tiles with the FP64 guard band) also runs with every temporary
// buffer placed in one fixed device array of this translation unit.
static __device__ __align__(256) unsigned char g_noalloc_scratch[CT_NOALLOC_SCRATCH_BYTES];

namespace ct {

namespace {
std::mutex g_noalloc_mu;
void *g_noalloc_addr[64] = {};

// Device address of the fixed array on the current device, looked up once per
// device (the host-side symbol is not a device address).
unsigned char *noalloc_scratch() {
    int dev = 0;
    CT_CHECK_CUDA(cudaGetDevice(&dev));
    if (dev < 0 || dev >= 64) CT_FAIL(CT_EUNSUPPORTED, "device ordinal %d above 63", dev);
    std::lock_guard<std::mutex> lk(g_noalloc_mu);
    if (!g_noalloc_addr[dev]) {
        void *p = nullptr;
        cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
        if (e != cudaSuccess || !p) {
            cudaGetLastError();
            CT_FAIL(CT_ECUDA, "cudaGetSymbolAddress of the fixed scratch failed: %s", cudaGetErrorString(e));
        }
        g_noalloc_addr[dev] = p;
    }
    return (unsigned char *)g_noalloc_addr[dev];
}

size_t align256(size_t x) { return (x + 255) & ~(size_t)255; }
}  // namespace

void degrees_noalloc(const ct_tree *t, const QParams &qp, int32_t *degrees, cudaStream_t s) {
    if (t->metric != CT_L2_F32) CT_FAIL(CT_EUNSUPPORTED, "the allocation-free degree count supports L2 trees only");
    const int64_t n = t->n;
    if (n == 0) return;
    unsigned char *base = noalloc_scratch();
    const size_t cap_bytes = CT_NOALLOC_SCRATCH_BYTES;
    const int cap = 32 * (t->depth + 2);
    size_t off = 0;
    auto take = [&](size_t bytes) {
        unsigned char *p = base + off;
        off = align256(off + bytes);
        return p;
    };
    // fixed part: counters, scan tile sums, traversal stacks
    unsigned long long *st = (unsigned long long *)take(ST_N * sizeof(unsigned long long));
    unsigned long long *ctr = (unsigned long long *)take(4 * sizeof(unsigned long long));
    int32_t *next_group = (int32_t *)take(sizeof(int32_t));
    int32_t *nitems = (int32_t *)take(sizeof(int32_t));
    constexpr int kSpillCap = 1 << 15;  // ranges of step-limited walks per round (a full buffer only ends the limit)
    unsigned long long *spill_cnt = (unsigned long long *)take(2 * sizeof(unsigned long long));
    int4 *const spills[2] = {(int4 *)take(kSpillCap * sizeof(int4)), (int4 *)take(kSpillCap * sizeof(int4))};
    TravLaunch tl = trav_launch_config(true, t->n_groups);
    const size_t stack_per_block = (size_t)TRAV_WARPS * cap * sizeof(int2);
    if (off + stack_per_block > cap_bytes / 2)
        CT_FAIL(CT_EUNSUPPORTED, "a tree of depth %d needs more than the fixed %zu-byte scratch", t->depth, cap_bytes);
    // stacks take at most a quarter of the array, and the warps' partly filled
    // pool chunks (POOL_CHUNK entries each) at most a quarter of it: with a
    // 16 MiB array that caps the walk at 64 blocks of TRAV_WARPS warps, fewer
    // than the main path's resident grid (the walk is slower, not different)
    const int64_t chunk_blocks = (int64_t)(cap_bytes / 4 / sizeof(uint32_t)) / ((int64_t)TRAV_WARPS * POOL_CHUNK);
    tl.blocks = (int)std::max<int64_t>(
        1, std::min<int64_t>(std::min<int64_t>(tl.blocks, (cap_bytes / 4) / stack_per_block), chunk_blocks));
    tl.warps = tl.blocks * TRAV_WARPS;
    int2 *stacks = (int2 *)take((size_t)tl.blocks * stack_per_block);
    longlong2 *cursors = (longlong2 *)take((size_t)tl.warps * sizeof(longlong2));
    // the rest: segments (a sixth of it: 16 bytes each, one per walk and per
    // pool chunk a walk crosses) and the pool
    const size_t rest = cap_bytes > off ? cap_bytes - off : 0;
    const int64_t seg_cap = (int64_t)(rest / 6 / (sizeof(int32_t) * 2 + sizeof(int64_t)));
    int32_t *seg_group = (int32_t *)take((size_t)seg_cap * sizeof(int32_t));
    int32_t *seg_count = (int32_t *)take((size_t)seg_cap * sizeof(int32_t));
    int64_t *seg_begin = (int64_t *)take((size_t)seg_cap * sizeof(int64_t));
    if (off >= cap_bytes) CT_FAIL(CT_EUNSUPPORTED, "problem too large for the fixed scratch");
    const int64_t pool_cap = (int64_t)((cap_bytes - off) / sizeof(uint32_t));
    uint32_t *pool = (uint32_t *)take((size_t)pool_cap * sizeof(uint32_t));
    Pool P{pool, pool_cap, ctr, seg_group, seg_count, seg_begin, reinterpret_cast<int32_t *>(ctr + 1), seg_cap,
           ctr + 2, reinterpret_cast<int32_t *>(ctr + 3)};

    Views V;
    std::memset(&V, 0, sizeof(V));
    V.nc = 1;
    V.tv[0] = view_of(t);
    V.qp[0] = qp;
    V.gbase[1] = t->n_groups;
    V.rbase[1] = n;
    V.item_len[0] = kItem;
    int32_t *err = reinterpret_cast<int32_t *>(st + ST_ERR);
    // the array keeps the previous call's contents: clear what must start at zero
    CT_CHECK_CUDA(cudaMemsetAsync(st, 0, ST_N * sizeof(unsigned long long), s));
    launch_traversal(V, t->n_groups, t->dp, 0, true, t->group_order, P, stacks, cap, tl, st, err, next_group, spills,
                     spill_cnt, kSpillCap, cursors, s);
    unsigned long long hc[4] = {0, 0, 0, 0};
    CT_CHECK_CUDA(cudaMemcpyAsync(hc, ctr, sizeof(hc), cudaMemcpyDeviceToHost, s));
    CT_CHECK_CUDA(cudaStreamSynchronize(s));
    if ((uint32_t)hc[3])
        CT_FAIL(CT_EUNSUPPORTED, "%llu candidate blocks do not fit the fixed %zu-byte scratch (room for %lld); use eps_graph_query",
                hc[2], cap_bytes, (long long)pool_cap);
    const int nseg = (int)(uint32_t)hc[1];
    // work items live in the unused tail of the pool
    const int64_t used = (int64_t)hc[0] < pool_cap ? (int64_t)hc[0] : pool_cap;
    const int64_t max_items = nseg + (int64_t)hc[2] / kItem + 1;
    size_t toff = align256((size_t)used * sizeof(uint32_t));
    auto ttake = [&](size_t bytes) {
        unsigned char *p = (unsigned char *)pool + toff;
        toff = align256(toff + bytes);
        return p;
    };
    int32_t *icnt = (int32_t *)ttake((size_t)(nseg + 1) * sizeof(int32_t));
    int64_t *ioff = (int64_t *)ttake((size_t)(nseg + 1) * sizeof(int64_t));
    int64_t *sums = (int64_t *)ttake((size_t)std::max<int64_t>(scan_scratch_entries(nseg), 1) * sizeof(int64_t));
    int32_t *igroup = (int32_t *)ttake((size_t)max_items * sizeof(int32_t));
    int64_t *ibeg = (int64_t *)ttake((size_t)max_items * sizeof(int64_t));
    int64_t *iend = (int64_t *)ttake((size_t)max_items * sizeof(int64_t));
    if (toff > (size_t)pool_cap * sizeof(uint32_t))
        CT_FAIL(CT_EUNSUPPORTED, "work items of %llu candidate blocks do not fit the fixed scratch; use eps_graph_query",
                hc[2]);
    CT_CHECK_CUDA(cudaMemsetAsync(degrees, 0, (size_t)n * sizeof(int32_t), s));
    CT_CHECK_CUDA(cudaMemsetAsync(nitems, 0, sizeof(int32_t), s));
    if (nseg) {
        k_item_counts<<<grid_for(nseg, 256), 256, 0, s>>>(V, nseg, seg_group, seg_count, icnt);
        CT_COUNT_LAUNCH();
        exclusive_scan_i32_to_i64_into(icnt, ioff, nseg, ioff + nseg, sums, s);
        k_item_fill<<<grid_for(nseg, 256), 256, 0, s>>>(V, nseg, seg_group, seg_begin, seg_count, ioff, igroup, ibeg,
                                                       iend, nitems);
        CT_COUNT_LAUNCH();
        Items items{igroup, ibeg, iend, nitems};
        leaf_l2_prepare();
        CT_CHECK_CUDA(cudaMemsetAsync(ctr, 0, sizeof(unsigned long long), s));  // the walk's counters have been read
        auto go = [&](auto kern, bool sh) {
            const unsigned ctas = (unsigned)leaf_l2_grid(sh, max_items);
            kern<<<ctas, LEAF_T, leaf_smem(sh), s>>>(V, items, ItemWave{0, 0, 1}, ctr, pool, nullptr, degrees, nullptr,
                                                     nullptr, nullptr, nullptr, st, err, CapOut{}, nullptr,
                                                     PairList{});
        };
        if (short_rows(t->dp)) go(k_leaf_l2<false, KS_SHORT>, true);
        else go(k_leaf_l2<false, KS_LONG>, false);
        CT_COUNT_LAUNCH();
    }
    CT_LAUNCH_CHECK();
    unsigned long long e = 0;
    CT_CHECK_CUDA(cudaMemcpyAsync(&e, st + ST_ERR, sizeof(e), cudaMemcpyDeviceToHost, s));
    CT_CHECK_CUDA(cudaStreamSynchronize(s));
    if (e) CT_FAIL(CT_ECUDA, "internal consistency check failed in the degree count (code %llu)", e);
}

}  // namespace ct

// build.cu -- cover-tree construction on the GPU (Algorithm 1 SplitVertex and
// Algorithm 2 BuildLevel of the paper, Sec. IV-A).
//
// All hubs created in one round are split together, in passes over every hub
// of the round that each take a batch of centres (see k_net_update_l2):
// farthest-first among the farthest points that the blocks of the pass report,
// while they lie beyond 2^(l-1); every point keeps the distance D and the
// label L of its nearest centre so far (strict <).  Small hubs (L2) are split
// whole in one CTA each.
// When every hub has stopped, the round's points are partitioned by
// (hub, label) with a stable radix sort; each child's centre is moved to the
// front of its range, its radius is the max of D over its range, and a child
// with more than zeta points and positive radius becomes a hub of the next
// round at level ceil(log2 r) (levels with a single nested child are skipped);
// the others become leaf blocks.  Radii are stored rounded up so that they
// bound every descendant's exact distance.
//
// Distances are fp32 for L2 (direct differences) and exact integers for edit
// distance (bit-parallel, lev.cuh).
#include <climits>
#include <cstdio>
#include <memory>
#include <mutex>
#include <type_traits>
#include <vector>
#include <algorithm>

#include "common.cuh"
#include "lev.cuh"
#include "profile.cuh"

namespace ct {

namespace {

constexpr int BT = 256;  // threads per block in the build kernels
constexpr int32_t kNone = 0x7f7f7f7f;  // byte-fill 0x7f: "no position yet"

// ceil(log2 r) for finite r > 0 (exact at powers of two).
__device__ __forceinline__ int ceil_log2f(float r) {
    int e;
    float m = frexpf(r, &e);  // r = m * 2^e, m in [0.5, 1)
    return m == 0.5f ? e - 1 : e;
}

// Rounded-up radius: bounds the exact distance of every point whose fp32
// distance was at most r (fp32 relative error of the distance sums here is
// below 2^-17 for rows up to 4096 floats; absolute slack covers underflow).
__device__ __forceinline__ float round_radius_up(float r, int metric) {
    if (metric != CT_L2_F32) return r;
    if (r == 0.0f) return 0.0f;
    float t = __fmul_ru(r, 1.0f + 0x1p-16f);
    return __fadd_ru(t, 0x1p-64f);
}

// ---- L2 distances of a row held in registers.  TPD lanes share one row:
// lane j holds its float4s j, j + TPD, ... (NV of them; NV = 0: rows too long
// for registers, read again for every distance).  The other row comes from
// shared or global memory.  Callers run whole warps converged.
template <int TPD, int NV>
struct RowRegs {
    float4 v[NV ? NV : 1];
    const float4 *row;
    __device__ __forceinline__ void load(const float4 *r, int nq, int j) {
        row = r;
#pragma unroll
        for (int u = 0; u < NV; ++u) {
            const int k = j + u * TPD;
            v[u] = k < nq ? __ldg(r + k) : make_float4(0.f, 0.f, 0.f, 0.f);
        }
    }
    __device__ __forceinline__ void zero() {
        row = nullptr;
#pragma unroll
        for (int u = 0; u < NV; ++u) v[u] = make_float4(0.f, 0.f, 0.f, 0.f);
    }
    // squared distance to `other`, the same in all TPD lanes
    __device__ __forceinline__ float sqdist(const float4 *other, int nq, int j) const {
        float acc = 0.f;
        auto add = [&](const float4 a, const float4 b) {
            const float dx = a.x - b.x, dy = a.y - b.y, dz = a.z - b.z, dw = a.w - b.w;
            acc = fmaf(dx, dx, acc);
            acc = fmaf(dy, dy, acc);
            acc = fmaf(dz, dz, acc);
            acc = fmaf(dw, dw, acc);
        };
        if (NV) {
#pragma unroll
            for (int u = 0; u < NV; ++u) {
                const int k = j + u * TPD;
                if (k < nq) add(v[u], other[k]);
            }
        } else if (row) {
#pragma unroll 4
            for (int k = j; k < nq; k += TPD) add(__ldg(row + k), other[k]);
        }
#pragma unroll
        for (int o = TPD / 2; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o, TPD);
        return acc;
    }
};

struct Hubs {
    int32_t *begin, *count, *node, *nc, *m, *done, *level;
    int32_t *flat;  // 1: the split stopped early and every child is a leaf block
    float *thr;
};

// A split that has taken FLAT_MIN_CENTRES centres while they cover on average
// fewer than 1 + 1/8 points each is making almost every point its own child
// (in high-dimensional data where all distances lie above the threshold):
// the triangle inequality can then prune nothing below this hub, and the
// farthest-first iterations would grow quadratically with its size.  Such a
// hub keeps the centres taken so far (a net of its own: separated, within
// 2^l of the hub's centre) and its children become leaf blocks whatever their
// size; their stored radii keep the query exact.
constexpr int FLAT_MIN_CENTRES = 256;
__device__ __forceinline__ bool flat_split(int nc, int covered) {
    return nc >= FLAT_MIN_CENTRES && covered <= nc + (nc >> 3);
}

// ---- Splitting in batches of centres.
//
// A hub's split takes centres until every point lies within the threshold
// 2^(l-1) of one.  Taken one at a time, the farthest point first, that is a
// chain of as many dependent passes as the hub has children (1250 launches
// for 121k uniform points in 16-D, 480 for 50k DNA strings, 700 a level for a
// million 256-bit codes), each as long as a launch and a round trip to memory
// (about 15 us) whatever its work.  Here a pass takes up to NET_M centres:
//   update -- every point of the hub against the batch (its row is read
//             once); each warp then reports its farthest point;
//   select -- one CTA per hub reduces the reports to NET_C candidates and
//             takes the next batch from them farthest-first: the first is the
//             hub's farthest point, each next one the candidate farthest from
//             every centre including those just taken, while above the
//             threshold;
//   dists  -- distances of the batch to the hub's centres, for the triangle-
//             inequality test of the next update.
// The centres are a net as before (pairwise farther apart than the threshold,
// every point within it); only their order among near-equals differs.
// Measured (build stage, before -> after): see k_net_update_l2.
constexpr int NET_M = 32;    // centres of a batch
constexpr int NET_C = 128;   // candidates of a selection
constexpr int NET_KEYS = 8;  // farthest-point reports of a chunk

// A chunk of a hub's points: {hub, first position, index of its reports}.
struct Chunks {
    const int4 *list;
    int len;                     // points per chunk
    unsigned long long *keys;    // NET_KEYS per chunk: (distance, position) of a part's farthest point
    int32_t *cov;                // NET_KEYS per chunk: points of the part within the threshold
};
// A hub's batch.  The arrays are laid out by position, so that a hub's part
// grows with its points: it has at most as many centres.
struct Batch {
    int32_t *pos;     // begin + i: position of the batch's centre i (label nc - m + i)
    int32_t *cpos;    // begin + label: position of the label's centre
    float *dcc;       // DCC_PP floats per point, see Dcc
};
// Distances of a hub's labels to its batch, a row per label: 32 columns (8 to 24
// in hubs of one to three chunks: a batch has at most NET_KEYS centres a chunk)
// and the rows that fit 8 floats a point.  Labels past them, where more than a
// quarter of a hub's points are centres, are not pruned.  (A row of 32 for every
// point is as much memory as a row of 32 floats, and builds no faster.)
constexpr int DCC_PP = NET_KEYS;
struct Dcc {
    float *p;
    int rows, cols;
    __device__ __forceinline__ Dcc(const Batch &bt, int begin, int count, int chunk_len) {
        const int c = min(NET_M / NET_KEYS, (count + chunk_len - 1) / chunk_len);
        p = bt.dcc + (size_t)begin * DCC_PP;
        cols = c * NET_KEYS;
        rows = count / c;
    }
    __device__ __forceinline__ float *row(int label) const { return p + (size_t)label * cols; }
};

template <int TPD>
constexpr int net_passes() { return TPD == 1 ? 1 : TPD == 2 ? 2 : 4; }

// The farthest point and the number of covered points of a warp's points.
__device__ __forceinline__ void net_report(unsigned long long best, int cov, const Chunks &ch, int slot) {
    for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long v = __shfl_xor_sync(0xffffffffu, best, o);
        best = v > best ? v : best;
        cov += __shfl_xor_sync(0xffffffffu, cov, o);
    }
    if ((threadIdx.x & 31) == 0) {
        ch.keys[slot] = best;
        ch.cov[slot] = cov;
    }
}

// L2 update pass: TPD lanes per point, its row in registers, the batch's
// centres in shared memory.  PRUNE: a point labelled L cannot come closer to
// centre c than its distance D when d(c, centre L) >= 2 D (triangle
// inequality, with a margin for the fp32 errors); each point computes only
// the distances its mask leaves, and the row is not read when none is left.
// The test costs one 128-byte read per point, so it pays for rows longer than
// that (dp > 16); shorter rows compute every distance.  root: the first pass
// (D infinite) also reduces each hub's farthest point into root[hub].
// Bound by the centres' shared-memory reads and the FP32 pipe where little is
// pruned, by the latency of one chunk where the hub is small.
// Build stage of 1M x 128 (mixture), 121k x 16 (uniform), 174k x 64 (mixture):
// 18.6 / 22.7 / 9.6 ms with one centre per pass -> 10.3 / 2.6 / 3.6 ms
// (with the selection from all distances at once, k_net_select_l2).
template <int TPD, int NV, bool PRUNE>
__global__ void __launch_bounds__(BT) k_net_update_l2(const float *__restrict__ X, int dp,
                                                      const int32_t *__restrict__ ids, float *__restrict__ D,
                                                      int32_t *__restrict__ lab, Chunks ch, Hubs hb, Batch bt,
                                                      unsigned long long *__restrict__ root) {
    extern __shared__ float4 cen[];  // m x nq
    constexpr int P = net_passes<TPD>(), G = BT / TPD;
    const int4 ck = ch.list[blockIdx.x];
    const int h = ck.x, start = ck.y;
    if (hb.done[h]) return;
    const int hbeg = hb.begin[h], m = hb.m[h], lbl0 = hb.nc[h] - m, nq = dp >> 2;
    const int end = min(start + ch.len, hbeg + hb.count[h]);
    const float thr = hb.thr[h];
    const int32_t *bpos = bt.pos + hbeg;
    for (int i = threadIdx.x; i < m * nq; i += BT) {
        const int c = i / nq, k = i - c * nq;
        cen[i] = __ldg(reinterpret_cast<const float4 *>(X + (size_t)ids[bpos[c]] * dp) + k);
    }
    const int g = threadIdx.x / TPD, j = threadIdx.x % TPD, lane = threadIdx.x & 31;
    float cur[P];
    int lb[P], pid[P];
    unsigned mask[P];
#pragma unroll
    for (int p = 0; p < P; ++p) {
        const int pos = start + p * G + g;
        const bool valid = pos < end;
        cur[p] = valid ? D[pos] : 0.f;
        lb[p] = valid && PRUNE ? lab[pos] : 0;
        pid[p] = valid ? ids[pos] : 0;
        mask[p] = valid && m ? 0xffffffffu >> (32 - m) : 0u;
    }
    if (PRUNE && m && !root) {
        const Dcc dcc(bt, hbeg, hb.count[h], ch.len);
#pragma unroll
        for (int p = 0; p < P; ++p) {
            if (!mask[p] || lb[p] >= dcc.rows) continue;
            const float lim = 2.0f * cur[p] * (1.0f + 0x1p-12f) + 0x1p-60f;
            const float4 *row = reinterpret_cast<const float4 *>(dcc.row(lb[p]));
            unsigned near = 0u;
            for (int q = j; 4 * q < m; q += TPD) {  // entries at and past m are masked out
                const float4 d = row[q];
                near |= ((d.x < lim ? 1u : 0u) | (d.y < lim ? 2u : 0u) | (d.z < lim ? 4u : 0u) |
                         (d.w < lim ? 8u : 0u)) << (4 * q);
            }
            mask[p] &= near;  // this lane's part; the group's parts are combined below
        }
#pragma unroll
        for (int p = 0; p < P; ++p)
#pragma unroll
            for (int o = TPD / 2; o > 0; o >>= 1) mask[p] |= __shfl_xor_sync(0xffffffffu, mask[p], o, TPD);
    }
    __syncthreads();  // the centres
    unsigned long long best = 0ull;
    int cov = 0;
#pragma unroll
    for (int p = 0; p < P; ++p) {
        const int pos = start + p * G + g;
        unsigned mk = mask[p];
        if (__any_sync(0xffffffffu, mk != 0u)) {
            RowRegs<TPD, NV> r;
            if (mk) r.load(reinterpret_cast<const float4 *>(X + (size_t)pid[p] * dp), nq, j);
            else r.zero();
            float sb = INFINITY;
            int ib = 0;
            if (PRUNE) {
                do {  // each group its next centre
                    const int i = mk ? __ffs(mk) - 1 : 0;
                    const float s = r.sqdist(cen + i * nq, nq, j);
                    if (mk && s < sb) {
                        sb = s;
                        ib = i;
                    }
                    mk &= mk - 1u;
                } while (__any_sync(0xffffffffu, mk != 0u));
            } else {
                for (int i = 0; i < m; ++i) {
                    const float s = r.sqdist(cen + i * nq, nq, j);
                    if (s < sb) {
                        sb = s;
                        ib = i;
                    }
                }
                if (!mk) sb = INFINITY;
            }
            const float d = sqrtf(sb);
            if (d < cur[p]) {
                cur[p] = d;
                if (j == 0) {
                    D[pos] = d;
                    lab[pos] = lbl0 + ib;
                }
            }
        }
        if (pos < end && j == 0) {
            const unsigned long long k = pack_max_key(cur[p], (uint32_t)pos);
            best = k > best ? k : best;
            cov += cur[p] <= thr;
        }
    }
    net_report(best, cov, ch, ck.z * NET_KEYS + (threadIdx.x >> 5));
    if (root) {
        for (int o = 16; o > 0; o >>= 1) {
            const unsigned long long v = __shfl_xor_sync(0xffffffffu, best, o);
            best = v > best ? v : best;
        }
        if (lane == 0) atomicMax(root + h, best);
    }
}

// Reduces the reports of a hub's chunks to at most C candidates above the
// threshold (slot s: the farthest of the reports s, s + C, ...), in cd / cp
// (distance, position); returns their number, and the hub's covered points in
// *covered.  Called by a whole block of at least C threads; ends with a barrier.
template <int C>
__device__ __forceinline__ int net_candidates(const Chunks &ch, int64_t first, int n_rep, float thr, float *cd,
                                              int32_t *cp, int *covered) {
    __shared__ unsigned long long slot[C];
    __shared__ int s_n[C / 32], s_cov[32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
    for (int i = threadIdx.x; i < C; i += blockDim.x) slot[i] = 0ull;
    __syncthreads();
    int cov = 0;
    unsigned long long best = 0ull;  // blockDim.x is a multiple of C: a thread's reports share a slot
    // eight loads in flight: a hub of a million points has 62k reports (build of
    // 1M x 128: 10.3 -> 10.0 ms)
    for (int i0 = threadIdx.x; i0 < n_rep; i0 += 8 * blockDim.x) {
        unsigned long long k[8];
        int c[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const int i = i0 + u * blockDim.x;
            k[u] = i < n_rep ? ch.keys[first + i] : 0ull;
            c[u] = i < n_rep ? ch.cov[first + i] : 0;
        }
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            best = k[u] > best ? k[u] : best;
            cov += c[u];
        }
    }
    if (best && key_value(best) > thr) atomicMax(&slot[threadIdx.x % C], best);
    for (int o = 16; o > 0; o >>= 1) cov += __shfl_xor_sync(0xffffffffu, cov, o);
    if (lane == 0) s_cov[w] = cov;
    __syncthreads();
    unsigned long long k = 0ull;
    unsigned bal = 0u;
    if (threadIdx.x < C) {
        k = slot[threadIdx.x];
        bal = __ballot_sync(0xffffffffu, k != 0ull);
        if (lane == 0) s_n[w] = __popc(bal);
    }
    __syncthreads();
    int total = 0, base = 0;
#pragma unroll
    for (int i = 0; i < C / 32; ++i) {
        if (i < w) base += s_n[i];
        total += s_n[i];
    }
    if (k) {
        const int at = base + __popc(bal & lanemask_lt());
        cd[at] = key_value(k);
        cp[at] = (int32_t)key_pos(k);
    }
    int c = 0;
    for (int i = 0; i < nw; ++i) c += s_cov[i];
    *covered = c;
    __syncthreads();
    return total;
}

// The candidate farthest from every centre so far (lowest index among equals;
// lane l of the warp holds candidates l, l + 32, ...), or -1: none lies beyond
// the threshold.
template <int C>
__device__ __forceinline__ int net_farthest(const float (&d)[C / 32], float thr) {
    const int lane = threadIdx.x & 31;
    float best = d[0];
#pragma unroll
    for (int k = 1; k < C / 32; ++k) best = fmaxf(best, d[k]);
    // distances are not negative: their bits order as they do
    const unsigned top = __reduce_max_sync(0xffffffffu, __float_as_uint(best));
    if (!(__uint_as_float(top) > thr)) return -1;
    unsigned at = 0xffffffffu;
#pragma unroll
    for (int k = C / 32 - 1; k >= 0; --k)
        if (__float_as_uint(d[k]) == top) at = (unsigned)(lane + 32 * k);
    return (int)__reduce_min_sync(0xffffffffu, at);
}

// The picks of one warp from n <= C candidates, farthest-first: each time the
// candidate farthest from every centre so far, while it lies beyond the
// threshold; pd(i, j): their mutual distances.  Two warp reductions and a row
// of pd per pick.  Returns the number of picks.
template <int C, class Pd>
__device__ __forceinline__ int net_greedy(const float *cd, int n, float thr, int mcap, int *picks, Pd pd) {
    const int lane = threadIdx.x & 31;
    float d[C / 32];
#pragma unroll
    for (int k = 0; k < C / 32; ++k) d[k] = lane + 32 * k < n ? cd[lane + 32 * k] : 0.f;
    int m = 0;
    for (; m < mcap; ++m) {
        const int pick = net_farthest<C>(d, thr);
        if (pick < 0) break;
        if (lane == 0) picks[m] = pick;
#pragma unroll
        for (int k = 0; k < C / 32; ++k)
            if (lane + 32 * k < n) d[k] = fminf(d[k], pd(pick, lane + 32 * k));
    }
    __syncwarp();
    return m;
}

// Tile idx of the upper triangle (with its diagonal) of T x T tiles, rows
// rp and T - 1 - rp folded into one row of T + 1; false: none.
__device__ __forceinline__ bool upper_tile(int idx, int T, int &ti, int &tj) {
    const int rp = idx / (T + 1), c = idx - rp * (T + 1);
    ti = rp;
    tj = rp + c;
    if (c < T - rp) return true;
    ti = T - 1 - rp;
    tj = ti + (c - (T - rp));
    return ti > rp;
}

// A hub's batch taken (thread 0): m centres after the nc it had, or done.
__device__ __forceinline__ void net_take(Hubs hb, int h, int m, bool flat, int32_t *active) {
    hb.m[h] = m;
    hb.nc[h] += m;
    if (m == 0) hb.done[h] = 1;
    if (flat) hb.flat[h] = 1;
    if (m) atomicAdd(active, 1);
}

// Picks from candidates whose rows are too long to stage: after each pick its
// distances alone, TPD lanes per candidate, a group's candidates together (so
// that their loads overlap).  A batch of such rows has few centres (3 at 4096
// floats), so that m n distances are far fewer than the n^2 / 2 of all pairs:
// build of 20000 x 4096 27.8 -> 8.1 ms (9.3 to 11.2 with a launch per centre).
template <int C, int TPD>
__device__ __forceinline__ int net_pick_long(const float *__restrict__ X, int dp, const int32_t *__restrict__ ids,
                                             float *cd, const int32_t *cp, int n, float thr, int mcap, int *picks) {
    constexpr int G = BT / TPD, U = C / G;  // groups; candidates of a group
    __shared__ int s_pick;
    const int lane = threadIdx.x & 31, g = threadIdx.x / TPD, j = threadIdx.x % TPD, nq = dp >> 2;
    int m = 0;
    for (; m < mcap; ++m) {
        if (threadIdx.x < 32) {
            float d[C / 32];
#pragma unroll
            for (int k = 0; k < C / 32; ++k) d[k] = lane + 32 * k < n ? cd[lane + 32 * k] : 0.f;
            const int p = net_farthest<C>(d, thr);
            if (lane == 0) s_pick = picks[m] = p;
        }
        __syncthreads();
        const int p = s_pick;
        if (p < 0) break;
        if (m + 1 < mcap) {
            const float4 *x = reinterpret_cast<const float4 *>(X + (size_t)ids[cp[p]] * dp);
            const float4 *y[U];
            float acc[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                y[u] = reinterpret_cast<const float4 *>(X + (size_t)ids[cp[min(g + u * G, n - 1)]] * dp);
                acc[u] = 0.f;
            }
            for (int k = j; k < nq; k += TPD) {
                const float4 a = __ldg(x + k);
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const float4 b = __ldg(y[u] + k);
                    const float dx = a.x - b.x, dy = a.y - b.y, dz = a.z - b.z, dw = a.w - b.w;
                    acc[u] = fmaf(dx, dx, acc[u]);
                    acc[u] = fmaf(dy, dy, acc[u]);
                    acc[u] = fmaf(dz, dz, acc[u]);
                    acc[u] = fmaf(dw, dw, acc[u]);
                }
            }
#pragma unroll
            for (int u = 0; u < U; ++u) {
#pragma unroll
                for (int o = TPD / 2; o > 0; o >>= 1) acc[u] += __shfl_xor_sync(0xffffffffu, acc[u], o, TPD);
                const int c = g + u * G;
                if (j == 0 && c < n) cd[c] = fminf(cd[c], sqrtf(acc[u]));
            }
        }
        __syncthreads();  // the distances; s_pick has been read
    }
    return m;
}

// The next batch of a hub (one CTA per listed hub {hub, slot}): at most C
// candidates, all their mutual distances at once (4 x 4 micro-tiles from rows
// staged in shared memory), then one warp picks.  (Picking with a block-wide
// distance update per pick, two barriers each, took 29 us at 121k x 16: 13 now;
// 15 at 100k x 64: 8.)  Rows too long to stage: net_pick_long.
// 128 candidates up to 32 floats per row, 64 above: the distances grow with both.
template <int C, int TPD>
__global__ void __launch_bounds__(BT) k_net_select_l2(const float *__restrict__ X, int dp,
                                                      const int32_t *__restrict__ ids, const int2 *__restrict__ hlist,
                                                      Hubs hb, const int64_t *__restrict__ coff, Chunks ch, Batch bt,
                                                      int mcap, int staged, int32_t *__restrict__ active) {
    extern __shared__ float4 rows[];  // staged: C x (nq + 1), then C x C distances
    __shared__ float cd[C];
    __shared__ int32_t cp[C];
    __shared__ int picks[NET_M];
    const int2 hs = hlist[blockIdx.x];
    const int h = hs.x;
    if (hb.done[h]) return;
    const int b = hb.begin[h], nc = hb.nc[h], nq = dp >> 2, rs = nq + 1;
    float *pd = reinterpret_cast<float *>(rows + C * rs);
    const float thr = hb.thr[h];
    const int n_rep = (hb.count[h] + ch.len - 1) / ch.len * NET_KEYS;
    int covered;
    const int n = net_candidates<C>(ch, coff[hs.y] * NET_KEYS, n_rep, thr, cd, cp, &covered);
    const bool flat = n > 0 && flat_split(nc, covered);
    if (n == 0 || flat) {
        if (threadIdx.x == 0) net_take(hb, h, 0, flat, active);
        return;
    }
    const int T = (n + 3) >> 2;
    if (staged) {
        for (int i = threadIdx.x; i < 4 * T * nq; i += BT) {
            const int c = i / nq, k = i - c * nq;
            rows[c * rs + k] = c < n ? __ldg(reinterpret_cast<const float4 *>(X + (size_t)ids[cp[c]] * dp) + k)
                                     : make_float4(0.f, 0.f, 0.f, 0.f);
        }
        __syncthreads();
        for (int idx = threadIdx.x; idx < ((T + 1) >> 1) * (T + 1); idx += BT) {
            int ti, tj;
            if (!upper_tile(idx, T, ti, tj)) continue;
            float acc[4][4] = {};
            for (int k = 0; k < nq; ++k) {
                float4 x[4], y[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    x[u] = rows[(4 * ti + u) * rs + k];
                    y[u] = rows[(4 * tj + u) * rs + k];
                }
#pragma unroll
                for (int u = 0; u < 4; ++u)
#pragma unroll
                    for (int v = 0; v < 4; ++v) {
                        const float dx = x[u].x - y[v].x, dy = x[u].y - y[v].y, dz = x[u].z - y[v].z,
                                    dw = x[u].w - y[v].w;
                        acc[u][v] = fmaf(dx, dx, acc[u][v]);
                        acc[u][v] = fmaf(dy, dy, acc[u][v]);
                        acc[u][v] = fmaf(dz, dz, acc[u][v]);
                        acc[u][v] = fmaf(dw, dw, acc[u][v]);
                    }
            }
#pragma unroll
            for (int u = 0; u < 4; ++u)
#pragma unroll
                for (int v = 0; v < 4; ++v) {
                    const float dd = sqrtf(acc[u][v]);
                    pd[(4 * ti + u) * C + 4 * tj + v] = dd;
                    pd[(4 * tj + v) * C + 4 * ti + u] = dd;
                }
        }
    }
    int m;
    if constexpr (TPD >= 16) {  // staged up to 256 floats: shorter rows have fewer lanes
        if (!staged) m = net_pick_long<C, TPD>(X, dp, ids, cd, cp, n, thr, mcap, picks);
    }
    __syncthreads();
    if (threadIdx.x >= 32) return;
    if (staged) m = net_greedy<C>(cd, n, thr, mcap, picks, [&](int i, int j) { return pd[i * C + j]; });
    for (int i = threadIdx.x; i < m; i += 32) {
        bt.pos[b + i] = cp[picks[i]];
        bt.cpos[b + nc + i] = cp[picks[i]];
    }
    if (threadIdx.x == 0) {
        if (nc == 1) bt.cpos[b] = b;  // label 0: the hub's own centre
        net_take(hb, h, m, false, active);
    }
}

// its dynamic shared memory where the rows are staged
constexpr size_t net_select_smem(int cands, int dp) {
    return ((size_t)cands * cands + (size_t)cands * (dp + 4)) * sizeof(float);
}

// Distances of a hub's centres (labels below nc) to its new batch: blocks
// (hub, y) over the labels, TPD lanes per label.
template <int TPD, int NV>
__global__ void __launch_bounds__(BT) k_net_dists_l2(const float *__restrict__ X, int dp,
                                                     const int32_t *__restrict__ ids, const int2 *__restrict__ hlist,
                                                     Hubs hb, Batch bt, int chunk_len) {
    extern __shared__ float4 cen[];  // m x nq
    const int h = hlist[blockIdx.x].x;
    if (hb.done[h]) return;
    const int b = hb.begin[h], m = hb.m[h], nq = dp >> 2;
    const Dcc dcc(bt, b, hb.count[h], chunk_len);
    const int nc = min(hb.nc[h], dcc.rows);
    constexpr int G = BT / TPD;
    if ((int)blockIdx.y * G >= nc) return;
    const int32_t *bpos = bt.pos + b;
    for (int i = threadIdx.x; i < m * nq; i += BT) {
        const int c = i / nq, k = i - c * nq;
        cen[i] = __ldg(reinterpret_cast<const float4 *>(X + (size_t)ids[bpos[c]] * dp) + k);
    }
    __syncthreads();
    const int g = threadIdx.x / TPD, j = threadIdx.x % TPD;
    for (int L0 = blockIdx.y * G; L0 < nc; L0 += gridDim.y * G) {  // the same number of steps in every group
        const int L = L0 + g;
        RowRegs<TPD, NV> r;
        r.load(reinterpret_cast<const float4 *>(X + (size_t)ids[bt.cpos[b + min(L, nc - 1)]] * dp), nq, j);
        float *out = dcc.row(L);
        for (int i = 0; i < m; ++i) {
            const float s = r.sqdist(cen + i * nq, nq, j);
            if (L < nc && j == 0) out[i] = sqrtf(s);
        }
    }
}

// ---- Edit distance: the same passes.  Strings are re-coded to the A bytes
// that occur (match masks of A entries), and each update block compacts the
// (point, centre) pairs that the triangle inequality leaves, so that its
// threads run the recurrence on full warps.
constexpr int LEV_P = 64;     // points per chunk
constexpr int LEV_C = 64;     // candidates of a selection
// Long strings of many symbols (masks above 10 KB a centre, so that 40 KB hold
// fewer than four): a pass lasts as long as the full recurrences that follow one
// another in it, however few centres it takes.  It takes six centres and chunks
// of 42 points (a pair per thread), and compares them all: two recurrences, not
// the three of a pass that prunes (update, pairs, distances to the centres so
// far).  5000 / 20000 strings of 1000 symbols out of 256 (32 KB a centre), ms:
// 276 / 532 with a launch per centre, 625 / - pruned with a centre per pass,
// 148 / 490 this way.
constexpr int LEV_WIDE_M = 6, LEV_WIDE_P = BT / LEV_WIDE_M;

// code[byte] = its rank among the bytes that occur; *A = their number.
__global__ void k_codes(const int32_t *__restrict__ present, uint8_t *__restrict__ code, int32_t *__restrict__ A) {
    __shared__ int s_w[8];
    const int t = threadIdx.x, lane = t & 31;
    const bool p = present[t] != 0;
    const unsigned bal = __ballot_sync(0xffffffffu, p);
    if (lane == 0) s_w[t >> 5] = __popc(bal);
    __syncthreads();
    int base = 0, total = 0;
    for (int w = 0; w < 8; ++w) {
        if (w < (t >> 5)) base += s_w[w];
        total += s_w[w];
    }
    code[t] = (uint8_t)(p ? base + __popc(bal & lanemask_lt()) : 0);
    if (t == 0) *A = total;
}
__global__ void k_recode(const uint8_t *__restrict__ s, int64_t nbytes, const uint8_t *__restrict__ code,
                         uint8_t *__restrict__ out) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < nbytes) out[i] = code[s[i]];
}

struct Strings {
    const uint8_t *s;    // codes below A
    const int64_t *off;
    int A;
};

// Match masks of one string over A codes, by the whole block (barriers inside).
template <int W>
__device__ __forceinline__ void lev_masks(uint64_t *peq, const uint8_t *pat, int m, int A) {
    for (int i = threadIdx.x; i < A * W; i += blockDim.x) peq[i] = 0ull;
    __syncthreads();
    for (int i = threadIdx.x; i < m; i += blockDim.x)
        atomicOr((unsigned long long *)&peq[pat[i] * W + (i >> 6)], 1ull << (i & 63));
    __syncthreads();
}

template <int W>
__global__ void __launch_bounds__(BT) k_net_update_lev(Strings S, const int32_t *__restrict__ ids,
                                                       float *__restrict__ D, int32_t *__restrict__ lab, Chunks ch,
                                                       Hubs hb, Batch bt, int prune,
                                                       unsigned long long *__restrict__ root) {
    extern __shared__ uint64_t speq[];  // m x A x W
    __shared__ int sd[LEV_P], sid[LEV_P], clen[NET_M];
    __shared__ unsigned skey[LEV_P];    // (distance << 8) | centre of the point's best so far
    __shared__ uint16_t pairs[LEV_P * NET_M];
    __shared__ int s_n;
    const int4 ck = ch.list[blockIdx.x];
    const int h = ck.x, start = ck.y;
    if (hb.done[h]) return;
    const int hbeg = hb.begin[h], m = hb.m[h], lbl0 = hb.nc[h] - m;
    const int np = min(ch.len, hbeg + hb.count[h] - start);
    const int32_t *bpos = bt.pos + hbeg;
    const int t = threadIdx.x;
    for (int i = t; i < m * S.A * W; i += BT) speq[i] = 0ull;
    float cur = 0.f;
    if (t < LEV_P) {
        if (t < np) {
            cur = D[start + t];
            sid[t] = ids[start + t];
        }
        sd[t] = isinf(cur) ? INT_MAX / 4 : (int)cur;
        skey[t] = 0xffffffffu;
    }
    if (t < m) {
        const int c = ids[bpos[t]];
        clen[t] = (int)(S.off[c + 1] - S.off[c]);
    }
    if (t == 0) s_n = 0;
    __syncthreads();
    for (int c = 0; c < m; ++c) {
        const uint8_t *pat = S.s + S.off[ids[bpos[c]]];
        for (int i = t; i < clen[c]; i += BT)
            atomicOr((unsigned long long *)&speq[((size_t)c * S.A + pat[i]) * W + (i >> 6)], 1ull << (i & 63));
    }
    // the pairs left by the triangle inequality: d(c, p) >= d(c, centre of p) - D(p)
    const Dcc dcc(bt, hbeg, hb.count[h], ch.len);
    for (int i0 = 0; i0 < m * LEV_P; i0 += BT) {
        const int i = i0 + t, c = i / LEV_P, p = i % LEV_P;
        bool keep = c < m && p < np;
        if (keep && prune) {
            const int L = lab[start + p];
            keep = L >= dcc.rows || dcc.row(L)[c] < 2.0f * (float)sd[p];
        }
        const unsigned bal = __ballot_sync(0xffffffffu, keep);
        int base = 0;
        if ((t & 31) == 0 && bal) base = atomicAdd(&s_n, __popc(bal));
        base = __shfl_sync(0xffffffffu, base, 0);
        if (keep) pairs[base + __popc(bal & lanemask_lt())] = (uint16_t)(c * LEV_P + p);
    }
    __syncthreads();
    const int n = s_n;
    for (int i = t; i < n; i += BT) {
        const int c = pairs[i] / LEV_P, p = pairs[i] % LEV_P;
        const int id = sid[p];
        // a distance above the best so far cannot win; an equal one wins by its lower centre
        const unsigned seen = *(volatile unsigned *)&skey[p];
        const int k = min(sd[p] - 1, (int)(seen >> 8));
        const int d = lev_myers<W>(speq + (size_t)c * S.A * W, clen[c], S.s + S.off[id],
                                   (int)(S.off[id + 1] - S.off[id]), k);
        if (d <= k) atomicMin(&skey[p], ((unsigned)d << 8) | (unsigned)c);
    }
    __syncthreads();
    if (t < LEV_P) {  // two warps: reports of eight points each
        unsigned long long best = 0ull;
        if (t < np) {
            const unsigned k = skey[t];
            if (k != 0xffffffffu) {
                cur = (float)(k >> 8);
                D[start + t] = cur;
                lab[start + t] = lbl0 + (int)(k & 255u);
            }
            best = pack_max_key(cur, (uint32_t)(start + t));
        }
#pragma unroll
        for (int o = LEV_P / NET_KEYS / 2; o > 0; o >>= 1) {
            const unsigned long long v = __shfl_xor_sync(0xffffffffu, best, o);
            best = v > best ? v : best;
        }
        if (t % (LEV_P / NET_KEYS) == 0) {
            ch.keys[ck.z * NET_KEYS + t / (LEV_P / NET_KEYS)] = best;
            ch.cov[ck.z * NET_KEYS + t / (LEV_P / NET_KEYS)] = 0;  // no flat-split test for edit distance
            if (root) atomicMax(root + h, best);
        }
    }
}

// Selection in three launches: the candidates, all their mutual distances
// (one block per candidate: a distance takes tens of microseconds, so they
// are not left to the picks' chain), and the picks.
// Laid out by position, as the batches.
struct LevCands {
    int32_t *n;          // per listed hub
    float *d;            // begin + i
    int32_t *pos;
    uint16_t *pair;      // LEV_PAIR_PP per point: K x K, K = lev_most_cands
};
// Candidates of a hub at most: its chunks' reports (one per eight points, or
// part of eight, of a chunk).  K^2 <= 10 count for chunks of 64 and 42 points.
// (64 x 64 pairs for every hub took 8 KB a hub, and with a leaf size of 1 there
// is a hub for every few strings.)
constexpr int LEV_PAIR_PP = 10;
__device__ __forceinline__ int lev_most_cands(int count, int chunk_len) {
    constexpr int pts = LEV_P / NET_KEYS;  // of a report
    return min(min(count, LEV_C), (count + chunk_len - 1) / chunk_len * ((chunk_len + pts - 1) / pts));
}
__global__ void __launch_bounds__(BT) k_net_cands_lev(const int2 *__restrict__ hlist, Hubs hb,
                                                      const int64_t *__restrict__ coff, Chunks ch, LevCands lc) {
    __shared__ float cd[LEV_C];
    __shared__ int32_t cp[LEV_C];
    const int2 hs = hlist[blockIdx.x];
    if (hb.done[hs.x]) return;
    const int n_rep = (hb.count[hs.x] + ch.len - 1) / ch.len * NET_KEYS;
    int covered;
    const int n = net_candidates<LEV_C>(ch, coff[hs.y] * NET_KEYS, n_rep, hb.thr[hs.x], cd, cp, &covered);
    if (threadIdx.x < n) {
        lc.d[hb.begin[hs.x] + threadIdx.x] = cd[threadIdx.x];
        lc.pos[hb.begin[hs.x] + threadIdx.x] = cp[threadIdx.x];
    }
    if (threadIdx.x == 0) lc.n[blockIdx.x] = n;
}
template <int W>
__global__ void __launch_bounds__(LEV_C) k_net_pairs_lev(Strings S, const int32_t *__restrict__ ids,
                                                         const int2 *__restrict__ hlist, Hubs hb, LevCands lc,
                                                         int chunk_len) {
    extern __shared__ uint64_t speq[];  // A x W
    const int i = blockIdx.x, a = blockIdx.y, t = threadIdx.x, h = hlist[i].x;
    if (hb.done[h]) return;
    const int n = lc.n[i], b = hb.begin[h], K = lev_most_cands(hb.count[h], chunk_len);
    if (a >= n) return;
    const int32_t *pos = lc.pos + b;
    const int ia = ids[pos[a]];
    const int la = (int)(S.off[ia + 1] - S.off[ia]);
    lev_masks<W>(speq, S.s + S.off[ia], la, S.A);
    if (t < n && t >= a) {
        const int ib = ids[pos[t]];
        const int d = t == a ? 0 : lev_myers<W>(speq, la, S.s + S.off[ib], (int)(S.off[ib + 1] - S.off[ib]), INT_MAX / 2);
        uint16_t *pr = lc.pair + (size_t)b * LEV_PAIR_PP;
        pr[a * K + t] = (uint16_t)d;
        pr[t * K + a] = (uint16_t)d;
    }
}
__global__ void __launch_bounds__(128) k_net_pick_lev(const int2 *__restrict__ hlist, Hubs hb, Batch bt, LevCands lc,
                                                      int mcap, int chunk_len, int32_t *__restrict__ active) {
    __shared__ float cd[LEV_C];
    __shared__ __align__(4) uint16_t pd[LEV_C * LEV_C];
    __shared__ int picks[NET_M];
    const int2 hs = hlist[blockIdx.x];
    const int h = hs.x;
    if (hb.done[h]) return;
    const int n = lc.n[blockIdx.x], b = hb.begin[h], nc = hb.nc[h], K = lev_most_cands(hb.count[h], chunk_len);
    for (int i = threadIdx.x; i < n; i += blockDim.x) cd[i] = lc.d[b + i];
    // rows below n, two entries at a time (those at and past n, and one past an odd end, are not read)
    const uint32_t *pair = reinterpret_cast<const uint32_t *>(lc.pair + (size_t)b * LEV_PAIR_PP);
#pragma unroll 4
    for (int i = threadIdx.x; i < (n * K + 1) >> 1; i += 128) reinterpret_cast<uint32_t *>(pd)[i] = pair[i];
    __syncthreads();
    if (threadIdx.x >= 32) return;
    const int m = n ? net_greedy<LEV_C>(cd, n, hb.thr[h], mcap, picks,
                                        [&](int i, int j) { return (float)pd[i * K + j]; })
                    : 0;
    for (int i = threadIdx.x; i < m; i += 32) {
        bt.pos[b + i] = lc.pos[b + picks[i]];
        bt.cpos[b + nc + i] = lc.pos[b + picks[i]];
    }
    if (threadIdx.x == 0) {
        if (nc == 1) bt.cpos[b] = b;  // label 0: the hub's own centre
        net_take(hb, h, m, false, active);
    }
}
// Distances of a hub's centres to its new batch: block (hub, batch centre).
template <int W>
__global__ void __launch_bounds__(128) k_net_dists_lev(Strings S, const int32_t *__restrict__ ids,
                                                       const int2 *__restrict__ hlist, Hubs hb, Batch bt,
                                                       int chunk_len) {
    extern __shared__ uint64_t speq[];  // A x W
    const int h = hlist[blockIdx.x].x, c = blockIdx.y;
    if (hb.done[h] || c >= hb.m[h]) return;
    const int b = hb.begin[h];
    const Dcc dcc(bt, b, hb.count[h], chunk_len);
    const int nc = min(hb.nc[h], dcc.rows);
    const int id = ids[bt.pos[b + c]];
    const int m = (int)(S.off[id + 1] - S.off[id]);
    lev_masks<W>(speq, S.s + S.off[id], m, S.A);
    for (int L = threadIdx.x; L < nc; L += blockDim.x) {
        const int il = ids[bt.cpos[b + L]];
        dcc.row(L)[c] =
            (float)lev_myers<W>(speq, m, S.s + S.off[il], (int)(S.off[il + 1] - S.off[il]), INT_MAX / 2);
    }
}

// ---- Hamming distance: rows of wp 32-bit words (wp a multiple of 4),
// compared four words at a time.
__device__ __forceinline__ int ham_dist4(const uint4 *__restrict__ a, const uint4 *b, int nq) {
    int d = 0;
    for (int k = 0; k < nq; ++k) {
        const uint4 x = a[k], y = b[k];
        d += __popc(x.x ^ y.x) + __popc(x.y ^ y.y) + __popc(x.z ^ y.z) + __popc(x.w ^ y.w);
    }
    return d;
}

// Input rows of ceil(dim/8) bytes (bit j = bit j % 8 of byte j / 8) into
// words of 32 bits (bit j = bit j % 32 of word j / 32); bits past dim cleared.
__global__ void k_pack_bits(const uint8_t *__restrict__ src, int64_t n, int dim, int wp, uint32_t *__restrict__ dst) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n * wp) return;
    const int64_t r = i / wp;
    const int w = (int)(i - r * wp);
    const int nbytes = (dim + 7) >> 3;
    uint32_t v = 0u;
    for (int b = 0; b < 4; ++b) {
        const int byte = 4 * w + b;
        if (byte < nbytes) v |= (uint32_t)src[r * nbytes + byte] << (8 * b);
    }
    const int lo = 32 * w;
    if (lo >= dim) v = 0u;
    else if (dim - lo < 32) v &= (1u << (dim - lo)) - 1u;
    dst[i] = v;
}

// Hamming update pass: one thread per point, its row in registers (NQ 16-byte
// pieces; 0: longer rows, read again for every centre), the batch's centres in
// shared memory.  A distance is a few population counts, so nothing is pruned.
template <int NQ>
__global__ void __launch_bounds__(BT) k_net_update_ham(const uint32_t *__restrict__ X, int wp,
                                                       const int32_t *__restrict__ ids, float *__restrict__ D,
                                                       int32_t *__restrict__ lab, Chunks ch, Hubs hb, Batch bt,
                                                       unsigned long long *__restrict__ root) {
    extern __shared__ uint4 hcen[];  // m x nq
    const int4 ck = ch.list[blockIdx.x];
    const int h = ck.x, start = ck.y;
    if (hb.done[h]) return;
    const int hbeg = hb.begin[h], m = hb.m[h], lbl0 = hb.nc[h] - m, nq = NQ ? NQ : wp >> 2;
    const int end = min(start + ch.len, hbeg + hb.count[h]);
    const int32_t *bpos = bt.pos + hbeg;
    for (int i = threadIdx.x; i < m * nq; i += BT) {
        const int c = i / nq, k = i - c * nq;
        hcen[i] = reinterpret_cast<const uint4 *>(X + (size_t)ids[bpos[c]] * wp)[k];
    }
    const int pos = start + threadIdx.x;  // ch.len = BT
    const bool valid = pos < end;
    float cur = valid ? D[pos] : 0.f;
    const uint4 *row = reinterpret_cast<const uint4 *>(X + (size_t)(valid ? ids[pos] : 0) * wp);
    uint4 v[NQ ? NQ : 1];
#pragma unroll
    for (int k = 0; k < NQ; ++k) v[k] = m ? __ldg(row + k) : make_uint4(0u, 0u, 0u, 0u);
    __syncthreads();
    int db = INT_MAX, ib = 0;
    for (int c = 0; c < m; ++c) {
        int d = 0;
        if (NQ) {
#pragma unroll
            for (int k = 0; k < NQ; ++k) {
                const uint4 y = hcen[c * nq + k];
                d += __popc(v[k].x ^ y.x) + __popc(v[k].y ^ y.y) + __popc(v[k].z ^ y.z) + __popc(v[k].w ^ y.w);
            }
        } else {
            d = ham_dist4(row, hcen + c * nq, nq);
        }
        if (d < db) {
            db = d;
            ib = c;
        }
    }
    unsigned long long best = 0ull;
    int cov = 0;
    if (valid) {
        if (m && (float)db < cur) {
            cur = (float)db;
            D[pos] = cur;
            lab[pos] = lbl0 + ib;
        }
        best = pack_max_key(cur, (uint32_t)pos);
        cov = cur <= hb.thr[h];
    }
    net_report(best, cov, ch, ck.z * NET_KEYS + (threadIdx.x >> 5));
    if (root) {
        for (int o = 16; o > 0; o >>= 1) {
            const unsigned long long k = __shfl_xor_sync(0xffffffffu, best, o);
            best = k > best ? k : best;
        }
        if ((threadIdx.x & 31) == 0) atomicMax(root + h, best);
    }
}

// The next batch of a hub (one CTA per listed hub), as k_net_select_l2.
__global__ void __launch_bounds__(BT) k_net_select_ham(const uint32_t *__restrict__ X, int wp,
                                                       const int32_t *__restrict__ ids, const int2 *__restrict__ hlist,
                                                       Hubs hb, const int64_t *__restrict__ coff, Chunks ch, Batch bt,
                                                       int32_t *__restrict__ active) {
    extern __shared__ uint4 hrows[];  // NET_C x (nq + 1), then NET_C x NET_C distances
    __shared__ float cd[NET_C];
    __shared__ int32_t cp[NET_C];
    __shared__ int picks[NET_M];
    const int2 hs = hlist[blockIdx.x];
    const int h = hs.x;
    if (hb.done[h]) return;
    const int b = hb.begin[h], nc = hb.nc[h], nq = wp >> 2;
    const float thr = hb.thr[h];
    const int n_rep = (hb.count[h] + ch.len - 1) / ch.len * NET_KEYS;
    int covered;
    const int n = net_candidates<NET_C>(ch, coff[hs.y] * NET_KEYS, n_rep, thr, cd, cp, &covered);
    const bool flat = n > 0 && flat_split(nc, covered);
    if (n == 0 || flat) {
        if (threadIdx.x == 0) net_take(hb, h, 0, flat, active);
        return;
    }
    const int rs = nq + 1;
    uint16_t *pd = reinterpret_cast<uint16_t *>(hrows + NET_C * rs);
    for (int i = threadIdx.x; i < n * nq; i += BT) {
        const int c = i / nq, k = i - c * nq;
        hrows[c * rs + k] = reinterpret_cast<const uint4 *>(X + (size_t)ids[cp[c]] * wp)[k];
    }
    __syncthreads();
    for (int idx = threadIdx.x; idx < ((n + 1) >> 1) * (n + 1); idx += BT) {
        int i, j;
        if (!upper_tile(idx, n, i, j)) continue;
        const uint16_t d = (uint16_t)ham_dist4(hrows + i * rs, hrows + j * rs, nq);
        pd[i * NET_C + j] = d;
        pd[j * NET_C + i] = d;
    }
    __syncthreads();
    if (threadIdx.x >= 32) return;
    const int m = net_greedy<NET_C>(cd, n, thr, NET_M, picks, [&](int i, int j) { return (float)pd[i * NET_C + j]; });
    for (int i = threadIdx.x; i < m; i += 32) bt.pos[b + i] = cp[picks[i]];
    if (threadIdx.x == 0) net_take(hb, h, m, false, active);
}

constexpr size_t net_select_ham_smem(int wp) {
    return (size_t)NET_C * (wp + 4) * sizeof(uint32_t) + (size_t)NET_C * NET_C * sizeof(uint16_t);
}

__global__ void k_gather_bits(const uint32_t *__restrict__ Xb, int wp, const int32_t *__restrict__ perm, int64_t n,
                              uint32_t *__restrict__ out) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int nq = wp >> 2;
    if (i >= n * nq) return;
    const int64_t r = i / nq;
    const int k = (int)(i - r * nq);
    reinterpret_cast<uint4 *>(out)[r * nq + k] = reinterpret_cast<const uint4 *>(Xb)[(int64_t)perm[r] * nq + k];
}

// Radius of each query group (Hamming): warp per group, lane per point.
__global__ void k_group_radius_ham(int ng, const int32_t *__restrict__ gbeg, const int32_t *__restrict__ gcnt,
                                   const uint32_t *__restrict__ bits, int wp, float *__restrict__ grad) {
    const int g = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    if (g >= ng) return;
    const int nq = wp >> 2;
    const uint4 *c = reinterpret_cast<const uint4 *>(bits + (size_t)gbeg[g] * wp);
    int r = 0;
    for (int i = lane; i < gcnt[g]; i += 32)
        r = max(r, ham_dist4(reinterpret_cast<const uint4 *>(bits + (size_t)(gbeg[g] + i) * wp), c, nq));
    for (int o = 16; o > 0; o >>= 1) r = max(r, __shfl_xor_sync(0xffffffffu, r, o));
    if (lane == 0) grad[g] = (float)r;
}

// Chunks per listed hub.
__global__ void k_chunk_counts(int nl, const int2 *__restrict__ hlist, const int32_t *__restrict__ count,
                               int chunk_len, int32_t *__restrict__ out) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= nl) return;
    out[i] = (count[hlist[i].x] + chunk_len - 1) / chunk_len;
}

// The whole split of one small hub (at most SPLIT_SMALL points) in one CTA,
// in the same batched passes: every warp's farthest point is a candidate, the
// candidates' mutual distances are taken at once (a group of TPD lanes per
// pair), one thread picks from them farthest-first, and a pass compares every
// point (its row read once) with the picks.  Distances and labels stay in
// shared memory; no launch per pass.  Larger hubs exit.
// Bound by the latency of a pass (about 2 us); before the batches each pass
// took one centre: 3.2 -> 1.6 ms for the small hubs of 1M x 128.
constexpr int SPLIT_SMALL = 512;
constexpr int SMALL_M = BT / 32;  // candidates, and centres of a pass
template <int TPD, int NV>
__global__ void __launch_bounds__(BT) k_split_small(const float *__restrict__ X, int dp,
                                                    const int32_t *__restrict__ ids, float *__restrict__ D,
                                                    int32_t *__restrict__ lab, Hubs hb) {
    __shared__ float Ds[SPLIT_SMALL], pd[SMALL_M * SMALL_M];
    __shared__ int32_t labs[SPLIT_SMALL];
    __shared__ float4 cen[SMALL_M * 32];  // dp <= 128
    __shared__ unsigned long long cand[SMALL_M];
    __shared__ int s_pick[SMALL_M], s_m;
    const int h = blockIdx.x;
    if (hb.done[h] || hb.count[h] > SPLIT_SMALL) return;  // a large hub: the level-wide passes
    const int b = hb.begin[h], cnt = hb.count[h], nq = dp >> 2;
    const float thr = hb.thr[h];
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    constexpr int G = BT / TPD;
    const int g = threadIdx.x / TPD, j = threadIdx.x % TPD;
    unsigned long long best = 0ull;
    for (int i = threadIdx.x; i < cnt; i += BT) {
        Ds[i] = D[b + i];
        labs[i] = lab[b + i];
        const unsigned long long k = pack_max_key(Ds[i], (uint32_t)i);
        best = k > best ? k : best;
    }
    int nc = hb.nc[h];
    for (;;) {
        for (int o = 16; o > 0; o >>= 1) {
            const unsigned long long v = __shfl_xor_sync(0xffffffffu, best, o);
            best = v > best ? v : best;
        }
        // candidates in cand / cen: the farthest point of every warp
        if (lane == 0) cand[w] = best;
        const int wpos = best ? (int)key_pos(best) : 0;
        const float4 *crow = reinterpret_cast<const float4 *>(X + (size_t)ids[b + wpos] * dp);
        for (int k = lane; k < nq; k += 32) cen[w * nq + k] = __ldg(crow + k);
        __syncthreads();
        // their mutual distances
        for (int q0 = 0; q0 < SMALL_M * SMALL_M; q0 += G) {
            const int q = min(q0 + g, SMALL_M * SMALL_M - 1);
            float acc = 0.f;
            const float4 *x = cen + (q / SMALL_M) * nq, *y = cen + (q % SMALL_M) * nq;
#pragma unroll 4
            for (int k = j; k < nq; k += TPD) {
                const float4 u = x[k], v = y[k];
                const float dx = u.x - v.x, dy = u.y - v.y, dz = u.z - v.z, dw = u.w - v.w;
                acc = fmaf(dx, dx, acc);
                acc = fmaf(dy, dy, acc);
                acc = fmaf(dz, dz, acc);
                acc = fmaf(dw, dw, acc);
            }
#pragma unroll
            for (int o = TPD / 2; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o, TPD);
            if (j == 0) pd[q] = sqrtf(acc);
        }
        __syncthreads();
        // the picks, farthest-first (lane c of warp 0 follows candidate c)
        if (w == 0) {
            const unsigned long long mine = lane < SMALL_M ? cand[lane] : 0ull;
            float d = mine ? key_value(mine) : 0.f;
            int m = 0;
            for (; m < SMALL_M; ++m) {
                unsigned long long f = lane < SMALL_M ? pack_max_key(d, (uint32_t)lane) : 0ull;
#pragma unroll
                for (int o = SMALL_M / 2; o > 0; o >>= 1) {
                    const unsigned long long v = __shfl_xor_sync(0xffffffffu, f, o);
                    f = v > f ? v : f;
                }
                f = __shfl_sync(0xffffffffu, f, 0);
                if (!(key_value(f) > thr)) break;
                const int pick = (int)key_pos(f);
                if (lane == 0) s_pick[m] = pick;
                if (lane < SMALL_M) d = fminf(d, pd[pick * SMALL_M + lane]);
            }
            if (lane == 0) s_m = m;
        }
        __syncthreads();
        const int m = s_m;
        if (m == 0) break;
        // every point against the picks
        best = 0ull;
        for (int i0 = 0; i0 < cnt; i0 += G) {
            const int i = i0 + g;
            const bool valid = i < cnt;
            RowRegs<TPD, NV> r;
            r.load(reinterpret_cast<const float4 *>(X + (size_t)ids[b + (valid ? i : 0)] * dp), nq, j);
            float sb = INFINITY;
            int ib = 0;
            for (int c = 0; c < m; ++c) {
                const float s = r.sqdist(cen + s_pick[c] * nq, nq, j);
                if (s < sb) {
                    sb = s;
                    ib = c;
                }
            }
            if (valid && j == 0) {
                float cur = Ds[i];
                const float d = sqrtf(sb);
                if (d < cur) {
                    cur = d;
                    Ds[i] = d;
                    labs[i] = nc + ib;
                }
                const unsigned long long k = pack_max_key(cur, (uint32_t)i);
                best = k > best ? k : best;
            }
        }
        nc += m;
        __syncthreads();  // cen and s_pick have been read
    }
    for (int i = threadIdx.x; i < cnt; i += BT) {
        D[b + i] = Ds[i];
        lab[b + i] = labs[i];
    }
    if (threadIdx.x == 0) {
        hb.nc[h] = nc;
        hb.done[h] = 1;
    }
}

// The listed hubs not yet done, and their chunks, for the next passes (the
// order within the lists is immaterial).  cnt: {hubs, chunks}.
__device__ __forceinline__ int append_slot(bool a, int32_t *cnt) {
    const unsigned m = __ballot_sync(0xffffffffu, a);
    if (!m) return 0;
    const int lane = threadIdx.x & 31, leader = __ffs(m) - 1;
    int base = 0;
    if (lane == leader) base = atomicAdd(cnt, __popc(m));
    base = __shfl_sync(0xffffffffu, base, leader);
    return base + __popc(m & lanemask_lt());
}
__global__ void k_active(int nl, const int2 *__restrict__ hl, int64_t nck, const int4 *__restrict__ cl,
                         const int32_t *__restrict__ done, int2 *__restrict__ hl2, int4 *__restrict__ cl2,
                         int32_t *__restrict__ cnt) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const bool ah = i < nl && !done[hl[i < nl ? i : 0].x];
    int k = append_slot(ah, cnt);
    if (ah) hl2[k] = hl[i];
    const bool ac = i < nck && !done[cl[i < nck ? i : 0].x];
    k = append_slot(ac, cnt + 1);
    if (ac) cl2[k] = cl[i];
}

// Chunk table of the listed hubs, one thread per chunk: its hub is the last
// one whose chunk offset is at most the chunk's index.
__global__ void k_chunk_fill(int64_t nchunks, int nl, const int2 *__restrict__ hlist,
                             const int32_t *__restrict__ begin, const int64_t *__restrict__ coff, int chunk_len,
                             int4 *__restrict__ chunks) {
    const int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= nchunks) return;
    int lo = 0, hi = nl;  // coff[lo] <= c, and c < coff[hi] unless hi = nl
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (__ldg(coff + mid) <= c) lo = mid; else hi = mid;
    }
    const int h = hlist[lo].x;
    chunks[c] = make_int4(h, begin[h] + (int)(c - coff[lo]) * chunk_len, (int)c, 0);
}

// Partition keys for the round: key = child_base[hub] + label, value = round
// index.  One thread per point of the round; its hub is the last one whose
// round offset is at most the index (hubs without points share an offset with
// the next hub and are skipped by the search).
__global__ void k_part_keys(int64_t R, int nh, const int32_t *__restrict__ begin,
                            const int64_t *__restrict__ round_off, const int64_t *__restrict__ child_base,
                            const int32_t *__restrict__ lab, uint32_t *__restrict__ keys,
                            uint32_t *__restrict__ vals, int32_t *__restrict__ rpos) {
    const int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= R) return;
    int lo = 0, hi = nh;  // round_off[lo] <= r, and r < round_off[hi] unless hi = nh
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (__ldg(round_off + mid) <= r) lo = mid; else hi = mid;
    }
    const int pos = begin[lo] + (int)(r - round_off[lo]);
    keys[r] = (uint32_t)(child_base[lo] + lab[pos]);
    vals[r] = (uint32_t)r;
    rpos[r] = pos;
}

// Gather the round in sorted order into temporaries; per child: count, first
// position, first zero-distance position (its centre or a duplicate of it).
// The sorted keys put each child's points in one run, so a warp combines its
// lanes of the same run (their destinations increase along the run) and one
// lane per run updates the child's count, first position and zero point.
__global__ void k_part_gather(int64_t R, const uint32_t *__restrict__ skeys, const uint32_t *__restrict__ svals,
                              const int32_t *__restrict__ rpos, const int32_t *__restrict__ ids,
                              const float *__restrict__ D, int32_t *__restrict__ tids,
                              float *__restrict__ tD, int32_t *__restrict__ ccount,
                              int32_t *__restrict__ cbegin, int32_t *__restrict__ czero) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const bool valid = i < R;
    uint32_t gc = 0xffffffffu;
    int dst = 0;
    int zero = INT_MAX;
    if (valid) {
        const int src = rpos[svals[i]];
        dst = rpos[i];
        gc = skeys[i];
        const float d = D[src];
        tids[i] = ids[src];
        tD[i] = d;
        if (d == 0.0f) zero = dst;
    }
    const unsigned same = __match_any_sync(0xffffffffu, gc);
    const int lane = threadIdx.x & 31;
    const int zmin = __reduce_min_sync(same, (unsigned)zero);
    if (valid && lane == __ffs(same) - 1) {  // the run's first lane: the smallest destination
        atomicAdd(&ccount[gc], __popc(same));
        atomicMin(&cbegin[gc], dst);
        if (zmin != INT_MAX) atomicMin(&czero[gc], zmin);
    }
}

// Writes the sorted round back; every point starts the next round labelled 0
// (the centre of the child it now belongs to).
__global__ void k_part_scatter(int64_t R, const int32_t *__restrict__ rpos, const int32_t *__restrict__ tids,
                               const float *__restrict__ tD, int32_t *__restrict__ ids,
                               float *__restrict__ D, int32_t *__restrict__ lab) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= R) return;
    int dst = rpos[i];
    ids[dst] = tids[i];
    D[dst] = tD[i];
    lab[dst] = 0;
}

// Move each child's centre to the front of its range.
__global__ void k_centre_front(int64_t T, const int32_t *__restrict__ cbegin, const int32_t *__restrict__ czero,
                               int32_t *__restrict__ ids, float *__restrict__ D, int32_t *__restrict__ err) {
    int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= T) return;
    int b = cbegin[c], z = czero[c];
    if (z == kNone) { atomicOr(err, 1); return; }
    if (z != b) {
        int ti = ids[b]; ids[b] = ids[z]; ids[z] = ti;
        float td = D[b]; D[b] = D[z]; D[z] = td;
    }
}

// Per child, the largest (distance, position) key: a prefix maximum along each
// run of equal keys in the warp, then one atomic per run (its last lane).
__global__ void k_child_keys(int64_t R, const uint32_t *__restrict__ skeys, const int32_t *__restrict__ rpos,
                             const float *__restrict__ D, unsigned long long *__restrict__ ckey) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const bool valid = i < R;
    const int lane = threadIdx.x & 31;
    uint32_t gc = 0xffffffffu;
    unsigned long long v = 0ull;
    if (valid) {
        const int pos = rpos[i];
        gc = skeys[i];
        v = pack_max_key(D[pos], (uint32_t)pos);
    }
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned long long ov = __shfl_up_sync(0xffffffffu, v, o);
        const uint32_t og = __shfl_up_sync(0xffffffffu, gc, o);
        if (lane >= o && og == gc && ov > v) v = ov;
    }
    const uint32_t next = __shfl_down_sync(0xffffffffu, gc, 1);
    if (valid && (lane == 31 || next != gc)) atomicMax(&ckey[gc], v);
}

// Link every hub to its children (consecutive node ids): one thread per child
// finds its hub (the last one whose child base is at most the child's index;
// every hub has children), the hub's first child writes the hub's record.
__global__ void k_link_children(int64_t T, int nh, Hubs hb, const int64_t *__restrict__ child_base, int node_base,
                                int32_t *__restrict__ child_begin, int32_t *__restrict__ child_count,
                                int32_t *__restrict__ node_level, int32_t *__restrict__ parent,
                                int32_t *__restrict__ leafy) {
    const int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= T) return;
    int lo = 0, hi = nh;
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (__ldg(child_base + mid) <= c) lo = mid; else hi = mid;
    }
    const int u = hb.node[lo];
    parent[node_base + c] = u;
    leafy[c] = hb.flat[lo];
    if (c == child_base[lo]) {
        child_begin[u] = node_base + (int32_t)c;
        child_count[u] = hb.nc[lo];
        node_level[u] = hb.level[lo];
    }
}

// New vertices of the round; flags children that become next-round hubs.
__global__ void k_make_nodes(int64_t T, int node_base, int zeta, int metric,
                             const int32_t *__restrict__ cbegin, const int32_t *__restrict__ ccount,
                             const unsigned long long *__restrict__ ckey, int32_t *__restrict__ node_begin,
                             int32_t *__restrict__ node_count, int32_t *__restrict__ child_begin,
                             int32_t *__restrict__ child_count, float *__restrict__ radius,
                             int32_t *__restrict__ level, const int32_t *__restrict__ leafy,
                             int32_t *__restrict__ is_hub) {
    int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= T) return;
    int v = node_base + (int)c;
    float r = key_value(ckey[c]);
    node_begin[v] = cbegin[c];
    node_count[v] = ccount[c];
    child_begin[v] = 0;
    child_count[v] = 0;
    radius[v] = round_radius_up(r, metric);
    level[v] = r > 0.0f ? ceil_log2f(r) : INT_MIN;
    is_hub[c] = (ccount[c] > zeta && r > 0.0f && !leafy[c]) ? 1 : 0;
}

// Next round's hubs from the flagged children (order preserved); the hubs of
// more than small_max points are listed for the level-wide passes (cnt: listed
// hubs, their chunks).
__global__ void k_next_hubs(int64_t T, int node_base, const int32_t *__restrict__ is_hub,
                            const int64_t *__restrict__ hub_off, const int32_t *__restrict__ cbegin,
                            const int32_t *__restrict__ ccount, const int32_t *__restrict__ level, Hubs nh, int small_max, int chunk_len,
                            int2 *__restrict__ hlist, int32_t *__restrict__ cnt) {
    int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const bool hub = c < T && is_hub[c];
    const bool listed = hub && ccount[c] > small_max;
    const int k = append_slot(listed, cnt);
    const int chunks = __reduce_add_sync(0xffffffffu, listed ? (ccount[c] + chunk_len - 1) / chunk_len : 0);
    if ((threadIdx.x & 31) == 0 && chunks) atomicAdd(cnt + 2, chunks);
    if (!hub) return;
    int64_t h = hub_off[c];
    if (listed) hlist[k] = make_int2((int)h, k);
    int v = node_base + (int)c;
    nh.begin[h] = cbegin[c];
    nh.count[h] = ccount[c];
    nh.node[h] = v;
    nh.nc[h] = 1;
    nh.m[h] = 0;
    nh.done[h] = 0;
    nh.flat[h] = 0;
    int l = level[v];
    nh.level[h] = l;
    nh.thr[h] = ldexpf(1.0f, l - 1);
}

// rbegin, rcount: the range of the only tree, or null.
__global__ void k_root_init(int64_t n, int root, int32_t *__restrict__ ids, float *__restrict__ D,
                            int32_t *__restrict__ lab, int32_t *__restrict__ rbegin, int32_t *__restrict__ rcount) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    if (i == 0 && rbegin) {
        *rbegin = 0;
        *rcount = (int32_t)n;
    }
    ids[i] = i == 0 ? root : (i <= root ? (int32_t)i - 1 : (int32_t)i);
    D[i] = INFINITY;
    lab[i] = 0;
}

// The roots' first pass: hub c holds every point of tree c, its batch is its
// first position with label 0.
__global__ void k_root_hubs(int R, const int32_t *__restrict__ rbegin, const int32_t *__restrict__ rcount, Hubs hb,
                            int32_t *__restrict__ bpos, int2 *__restrict__ hlist,
                            unsigned long long *__restrict__ rkey) {
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= R) return;
    hb.begin[c] = rbegin[c];
    hb.count[c] = rcount[c];
    hb.nc[c] = 1;
    hb.m[c] = 1;
    hb.done[c] = 0;
    hb.thr[c] = 0.0f;
    rkey[c] = 0ull;
    bpos[rbegin[c]] = rbegin[c];
    hlist[c] = make_int2(c, c);
}

// Rows already of dp = dim floats (dim a multiple of 4, 16-byte aligned
// source): a float4 copy with the same coordinate-range check.
__global__ void k_copy_rows4(const float4 *__restrict__ src, int64_t nq, float4 *__restrict__ dst,
                             int32_t *__restrict__ bad) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= nq) return;
    const float4 v = src[i];
    if (!(fabsf(v.x) <= 0x1p50f && fabsf(v.y) <= 0x1p50f && fabsf(v.z) <= 0x1p50f && fabsf(v.w) <= 0x1p50f))
        atomicOr(bad, 1);
    dst[i] = v;
}

// Pad rows to dp floats (original order) and check the coordinate range.
__global__ void k_pad_rows(const float *__restrict__ src, int64_t n, int dim, int dp,
                           float *__restrict__ dst, int32_t *__restrict__ bad) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n * dp) return;
    int64_t r = i / dp;
    int k = (int)(i - r * dp);
    float v = k < dim ? src[r * dim + k] : 0.0f;
    if (!(fabsf(v) <= 0x1p50f)) atomicOr(bad, 1);
    dst[i] = v;
}

__global__ void k_gather_rows(const float *__restrict__ Xp, int dp, const int32_t *__restrict__ perm,
                              int64_t n, float *__restrict__ out) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    int nq = dp >> 2;
    if (i >= n * nq) return;
    int64_t r = i / nq;
    int k = (int)(i - r * nq);
    reinterpret_cast<float4 *>(out)[i] = reinterpret_cast<const float4 *>(Xp + (size_t)perm[r] * dp)[k];
}

__global__ void k_node_centres(int nn, const int32_t *__restrict__ node_begin, const float *__restrict__ pts,
                               int dp, float *__restrict__ ctr) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    int nq = dp >> 2;
    if (i >= (int64_t)nn * nq) return;
    int64_t v = i / nq;
    int k = (int)(i - v * nq);
    reinterpret_cast<float4 *>(ctr)[i] =
        reinterpret_cast<const float4 *>(pts + (size_t)node_begin[v] * dp)[k];
}

__global__ void k_leaf_keys(int nn, const int32_t *__restrict__ child_count, const int32_t *__restrict__ node_begin,
                            const int32_t *__restrict__ node_count, uint32_t *__restrict__ keys,
                            uint32_t *__restrict__ vals, int32_t *__restrict__ nleaf,
                            int32_t *__restrict__ maxcnt) {
    int v = blockIdx.x * blockDim.x + threadIdx.x;
    if (v >= nn || child_count[v] != 0) return;
    int slot = atomicAdd(nleaf, 1);
    keys[slot] = (uint32_t)node_begin[v];
    vals[slot] = (uint32_t)v;
    atomicMax(maxcnt, node_count[v]);
}

__global__ void k_string_lengths(int64_t n, const int32_t *__restrict__ perm, const int64_t *__restrict__ off,
                                 int64_t *__restrict__ len_out, int32_t *__restrict__ maxlen) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    int64_t id = perm ? perm[i] : i;
    int64_t l = off[id + 1] - off[id];
    len_out[i] = l;
    atomicMax(maxlen, (int32_t)(l < INT_MAX ? l : INT_MAX));
}

__global__ void k_gather_strings(int64_t n, const int32_t *__restrict__ perm, const uint8_t *__restrict__ S,
                                 const int64_t *__restrict__ off, const int64_t *__restrict__ noff,
                                 uint8_t *__restrict__ out) {
    int64_t i = blockIdx.x;
    if (i >= n) return;
    int64_t id = perm[i];
    int64_t b = off[id], l = off[id + 1] - b, o = noff[i];
    for (int64_t k = threadIdx.x; k < l; k += blockDim.x) out[o + k] = S[b + k];
}

// Query groups: greedy runs of consecutive sibling leaf blocks of at most
// kGroupSize points in total; a larger block is cut into groups of kGroupSize
// consecutive points (the last one shorter) that hold no other block.  The
// leaf blocks are in position order; k_group_prep lays out each block's size
// and parent in that order, a run of siblings starts where the parent
// changes, and one thread walks each run (sequential reads), marking how many
// groups start at each block and recording the size of a merged group there.
__global__ void k_group_prep(int L, const int32_t *__restrict__ leaf_ids, const int32_t *__restrict__ node_count,
                             const int32_t *__restrict__ parent, int32_t *__restrict__ lcount,
                             int32_t *__restrict__ lpar) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= L) return;
    const int v = leaf_ids[i];
    lcount[i] = node_count[v];
    lpar[i] = parent[v];
}

__global__ void k_group_marks(int L, const int32_t *__restrict__ lcount, const int32_t *__restrict__ lpar,
                              int32_t *__restrict__ gstart, int32_t *__restrict__ gsize,
                              unsigned long long *__restrict__ maxc) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= L) return;
    const int p = lpar[i];
    if (i > 0 && lpar[i - 1] == p) return;  // not the first block of its sibling run
    int first = -1, acc = 0, big = 0;
    for (int j = i; j < L && lpar[j] == p; ++j) {
        const int c = lcount[j];
        if (c > kGroupSize) {  // groups of its own
            if (first >= 0) gsize[first] = acc;
            gstart[j] = (c + kGroupSize - 1) / kGroupSize;
            gsize[j] = c;
            big = kGroupSize;
            first = -1;
            acc = 0;
        } else if (first >= 0 && acc + c <= kGroupSize) {
            acc += c;
            gstart[j] = 0;
        } else {
            if (first >= 0) gsize[first] = acc;
            big = max(big, acc);
            first = j;
            acc = c;
            gstart[j] = 1;
        }
    }
    if (first >= 0) gsize[first] = acc;
    big = max(big, acc);
    atomicMax(maxc, (unsigned long long)big);
}

__global__ void k_group_scatter(int L, const int32_t *__restrict__ leaf_ids, const int32_t *__restrict__ node_begin,
                                const int32_t *__restrict__ gstart, const int32_t *__restrict__ gsize,
                                const int64_t *__restrict__ gidx, int32_t *__restrict__ group_begin,
                                int32_t *__restrict__ group_count) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= L || !gstart[i]) return;
    const int64_t g = gidx[i];
    const int b = node_begin[leaf_ids[i]], c = gsize[i];
    for (int k = 0; k < gstart[i]; ++k) {  // one group, or the cuts of a large block
        group_begin[g + k] = b + k * kGroupSize;
        group_count[g + k] = min(kGroupSize, c - k * kGroupSize);
    }
}

// Sort keys putting larger radii first (radii are non-negative floats).
__global__ void k_radius_desc_keys(int ng, const float *__restrict__ r, uint32_t *__restrict__ keys,
                                   uint32_t *__restrict__ vals) {
    int g = blockIdx.x * blockDim.x + threadIdx.x;
    if (g >= ng) return;
    keys[g] = 0xFFFFFFFFu - __float_as_uint(r[g]);
    vals[g] = (uint32_t)g;
}

// Radius of each query group: max distance from its first point (rounded up).
// One warp per group, one lane per point.
__global__ void k_group_radius_l2(int ng, const int32_t *__restrict__ gbeg, const int32_t *__restrict__ gcnt,
                                  const float *__restrict__ pts, int dp, float *__restrict__ grad) {
    int g = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    if (g >= ng) return;
    const float4 *c = reinterpret_cast<const float4 *>(pts + (size_t)gbeg[g] * dp);
    float r = 0.f;
    for (int i = lane; i < gcnt[g]; i += 32) {
        const float4 *p = reinterpret_cast<const float4 *>(pts + (size_t)(gbeg[g] + i) * dp);
        float acc = 0.f;
        for (int k = 0; k < dp / 4; ++k) {
            float4 a = __ldg(c + k), b = __ldg(p + k);
            float dx = a.x - b.x, dy = a.y - b.y, dz = a.z - b.z, dw = a.w - b.w;
            acc = fmaf(dx, dx, acc); acc = fmaf(dy, dy, acc); acc = fmaf(dz, dz, acc); acc = fmaf(dw, dw, acc);
        }
        r = fmaxf(r, sqrtf(acc));
    }
    for (int o = 16; o > 0; o >>= 1) r = fmaxf(r, __shfl_xor_sync(0xffffffffu, r, o));
    if (lane == 0) grad[g] = round_radius_up(r, CT_L2_F32);
}

template <int W>
__global__ void __launch_bounds__(32) k_group_radius_lev(int ng, const int32_t *__restrict__ gbeg,
                                                         const int32_t *__restrict__ gcnt,
                                                         const uint8_t *__restrict__ S,
                                                         const int64_t *__restrict__ off, float *__restrict__ grad) {
    __shared__ uint64_t peq[256 * W];
    int g = blockIdx.x;
    if (g >= ng) return;
    int cpos = gbeg[g];
    const uint8_t *pat = S + off[cpos];
    int m = (int)(off[cpos + 1] - off[cpos]);
    lev_build_peq<W>(peq, pat, m);
    __syncthreads();
    int r = 0;
    for (int i = threadIdx.x; i < gcnt[g]; i += 32) {
        int p = cpos + i;
        int d = lev_myers<W>(peq, m, S + off[p], (int)(off[p + 1] - off[p]), INT_MAX / 2);
        r = max(r, d);
    }
    for (int o = 16; o > 0; o >>= 1) r = max(r, __shfl_xor_sync(0xffffffffu, r, o));
    if (threadIdx.x == 0) grad[g] = (float)r;
}

inline unsigned grid_for(int64_t n, int t = BT) { return (unsigned)ceil_div(n > 0 ? n : 1, t); }

int bits_for(int64_t v) {
    int b = 0;
    while ((int64_t(1) << b) <= v && b < 62) ++b;
    return b;
}

}  // namespace

// Builds the tree; on failure throws ct::Error after freeing what it allocated.
void free_tree(ct_tree *t);

namespace {
struct TreeGuard {
    ct_tree *t;
    ~TreeGuard() { if (t) free_tree(t); }
};
}  // namespace

namespace {
void finish_forest(const ct_tree &proto, const std::vector<int64_t> &off, int N, DBuf<int32_t> &ids, DBuf<float> &D,
                   DBuf<int32_t> &nb, DBuf<int32_t> &ncnt, DBuf<int32_t> &cbeg, DBuf<int32_t> &ccnt,
                   DBuf<int32_t> &lvl, DBuf<int32_t> &par, DBuf<float> &rad, const float *Xp, const uint32_t *Xb,
                   std::vector<ct_tree *> &out, cudaStream_t s);

// A tree of all points; or, with `off` (the first position of each tree, and
// the end), a tree per range of points in `out`, all split together: their
// levels share every launch.
ct_tree *build_impl(const ct_points *pts, int zeta, int root, cudaStream_t s, const std::vector<int64_t> *off,
                    std::vector<ct_tree *> *out) {
    const int64_t n = pts->n;
    std::vector<int64_t> hroot;  // first position of each tree that has points
    if (off) {
        for (size_t c = 0; c + 1 < off->size(); ++c)
            if ((*off)[c] < (*off)[c + 1]) hroot.push_back((*off)[c]);
    } else if (n > 0) {
        hroot.push_back(0);
    }
    TreeGuard tg{new ct_tree()};
    ct_tree *t = tg.t;
    struct Flush { ~Flush() { prof_flush(); } } flush_at_exit;
    ProfScope prof_all("build", s, off ? (int64_t)off->size() - 1 : 1);
    t->metric = pts->metric;
    t->n = n;
    t->leaf_size = zeta;
    t->stream = s;
    CT_CHECK_CUDA(cudaGetDevice(&t->device));
    const bool l2 = pts->metric == CT_L2_F32;
    const bool ham = pts->metric == CT_HAMMING_B1;
    const bool lev = pts->metric == CT_LEVENSHTEIN_U8;
    t->dim = l2 || ham ? pts->dim : 0;
    t->dp = l2 ? (int)ceil_div(pts->dim, 4) * 4 : 0;
    t->wp = ham ? (int)ceil_div(pts->dim, 128) * 4 : 0;
    const int dp = t->dp, wp = t->wp;

    DBuf<int32_t> err(2, s);
    CT_CHECK_CUDA(cudaMemsetAsync(err.p, 0, 2 * sizeof(int32_t), s));
    int64_t sspan[2] = {0, 0};  // edit distance: first and past-the-end byte of the strings

    // padded copy of the input (original order) / string lengths
    DBuf<float> Xp;
    DBuf<uint32_t> Xb;
    DBuf<uint8_t> codes, scode;  // edit distance: the strings re-coded to the bytes that occur
    int W = 1, A = 1;
    if (ham) {
        Xb = DBuf<uint32_t>((size_t)(n ? n : 1) * wp, s);
        if (n) {
            k_pack_bits<<<grid_for(n * wp), BT, 0, s>>>((const uint8_t *)pts->data, n, pts->dim, wp, Xb.p);
            CT_COUNT_LAUNCH();
        }
    } else if (l2) {
        Xp = DBuf<float>((size_t)n * dp, s);
        if (n && dp == pts->dim && (reinterpret_cast<uintptr_t>(pts->data) & 15) == 0) {
            const int64_t nq = n * dp / 4;
            k_copy_rows4<<<grid_for(nq), BT, 0, s>>>((const float4 *)pts->data, nq, (float4 *)Xp.p, err.p);
            CT_COUNT_LAUNCH();
        } else if (n) {
            k_pad_rows<<<grid_for(n * dp), BT, 0, s>>>((const float *)pts->data, n, pts->dim, dp, Xp.p, err.p);
            CT_COUNT_LAUNCH();
        }
    } else {
        DBuf<int64_t> lens(n > 0 ? n : 1, s);
        if (n) {
            k_string_lengths<<<grid_for(n), BT, 0, s>>>(n, nullptr, pts->offsets, lens.p, err.p + 1);
            CT_COUNT_LAUNCH();
            to_host_async(sspan, pts->offsets, 1, s);
            to_host_async(sspan + 1, pts->offsets + n, 1, s);
        }
    }
    CT_LAUNCH_CHECK();
    int32_t herr[2] = {0, 0};
    to_host(herr, err.p, 2, s);
    if (herr[0]) CT_FAIL(CT_EUNSUPPORTED, "coordinates must be finite with |x| <= 2^50");
    if (lev) {
        if (herr[1] > CT_MAX_STRING_LEN)
            CT_FAIL(CT_EUNSUPPORTED, "string of length %d above the limit %d", herr[1], CT_MAX_STRING_LEN);
        t->max_len = herr[1];
        W = lev_words_for(t->max_len);
        const int64_t bytes = sspan[1] - sspan[0];
        DBuf<int32_t> present(257, s);  // per byte value; their number
        CT_CHECK_CUDA(cudaMemsetAsync(present.p, 0, 257 * sizeof(int32_t), s));
        codes = DBuf<uint8_t>(256, s);
        scode = DBuf<uint8_t>(bytes > 0 ? bytes : 1, s);
        const uint8_t *src = (const uint8_t *)pts->data + sspan[0];
        if (bytes > 0) {
            mark_bytes(src, bytes, present.p, s);
            k_codes<<<1, 256, 0, s>>>(present.p, codes.p, present.p + 256);
            CT_COUNT_LAUNCH();
            k_recode<<<grid_for(bytes), BT, 0, s>>>(src, bytes, codes.p, scode.p);
            CT_COUNT_LAUNCH();
        }
        CT_LAUNCH_CHECK();
        int32_t a = 0;
        to_host(&a, present.p + 256, 1, s);
        A = std::max(a, 1);
    }

    // tree arrays: a tree whose internal vertices have >= 2 children has < 2n vertices
    const int64_t cap = 2 * n + 1 + (int64_t)hroot.size();
    DBuf<int32_t> nb(cap, s), ncnt(cap, s), cbeg(cap, s), ccnt(cap, s), lvl(cap, s), par(cap, s);
    CT_CHECK_CUDA(cudaMemsetAsync(par.p, 0xff, cap * sizeof(int32_t), s));
    DBuf<float> rad(cap, s);
    DBuf<int32_t> ids(n ? n : 1, s), lab(n ? n : 1, s);
    DBuf<float> D(n ? n : 1, s);

    int n_nodes = 0, depth = 0;
    if (n > 0) {
        if (root < 0 || root >= n) CT_FAIL(CT_EINVAL, "root %d out of range", root);
        // ---- round 0: distances to the root
        const int64_t cap_h = n;  // hubs per round never exceed n / (zeta+1) + 1
        DBuf<int32_t> hbuf(8 * (cap_h + 1), s);
        DBuf<float> hthr(cap_h + 1, s);
        DBuf<int32_t> hbuf2(8 * (cap_h + 1), s);
        DBuf<float> hthr2(cap_h + 1, s);
        auto make_hubs = [&](DBuf<int32_t> &b, DBuf<float> &th) {
            Hubs h;
            int64_t st = cap_h + 1;
            h.begin = b.p; h.count = b.p + st; h.node = b.p + 2 * st; h.nc = b.p + 3 * st;
            h.m = b.p + 4 * st; h.done = b.p + 5 * st; h.level = b.p + 6 * st;
            h.flat = b.p + 7 * st;
            h.thr = th.p;
            return h;
        };
        Hubs H = make_hubs(hbuf, hthr), H2 = make_hubs(hbuf2, hthr2);

        const int R0 = (int)hroot.size();
        DBuf<int32_t> rbegin(R0, s), rcount(R0, s);
        k_root_init<<<grid_for(n), BT, 0, s>>>(n, root, ids.p, D.p, lab.p, R0 == 1 ? rbegin.p : nullptr, rcount.p);
        CT_COUNT_LAUNCH();
        // lanes per distance: four 16-byte loads each (at most eight for row
        // lengths between two powers of two, more above 1024 floats)
        int tpd = 1;  // a power of two
        while (l2 && tpd < 32 && 2 * tpd * 16 <= dp) tpd *= 2;
        const int nv = (dp / 4 + tpd - 1) / tpd;  // float4s per lane
        const int passes = tpd == 1 ? net_passes<1>() : tpd == 2 ? net_passes<2>() : net_passes<4>();
        const int mask_bytes = A * W * (int)sizeof(uint64_t);  // of a centre (edit distance)
        const bool wide = lev && 40960 / mask_bytes < 4;
        const int chunk_len = l2 ? passes * (BT / tpd) : ham ? BT : wide ? LEV_WIDE_P : LEV_P;
        // hubs of at most small_max points are split whole in one CTA each
        const int small_max = l2 && dp <= 128 ? SPLIT_SMALL : 0;
        // centres of a batch: what 48 KB of shared memory hold
        const int mcap = l2 ? std::max(1, std::min(NET_M, 12288 / std::max(dp, 1)))
                       : wide ? LEV_WIDE_M : lev ? std::min(NET_M, 40960 / mask_bytes) : NET_M;
        const bool prune = l2 ? dp > 16 : lev && !wide;
        const Strings S{scode.p - sspan[0], pts->offsets, A};
        DBuf<int32_t> cpos(l2 || lev ? n : 1, s);
        DBuf<float> dcc(prune ? (size_t)n * DCC_PP : 1, s);
        DBuf<int32_t> bpos(n, s);
        DBuf<int4> chunks_a, chunks_b;
        DBuf<int2> hl_a(cap_h + 1, s), hl_b(cap_h + 1, s);
        DBuf<unsigned long long> keys;
        DBuf<int32_t> cov;
        DBuf<int32_t> lcn, lcpos(lev ? n : 0, s);
        DBuf<float> lcd(lev ? n : 0, s);
        DBuf<uint16_t> lcpair(lev ? (size_t)n * LEV_PAIR_PP : 0, s);
        LevCands lc{nullptr, lcd.p, lcpos.p, lcpair.p};
        auto dispatch = [&](auto f) {  // f(lanes per distance, float4s per lane) as compile-time constants
#define CT_TN(T, V) f(std::integral_constant<int, T>(), std::integral_constant<int, V>())
#define CT_T48(T) case T: if (nv <= 4) CT_TN(T, 4); else CT_TN(T, 8); break;
            switch (tpd) {
                case 1: if (nv <= 1) CT_TN(1, 1); else if (nv <= 2) CT_TN(1, 2); else if (nv <= 4) CT_TN(1, 4); else CT_TN(1, 8); break;
                CT_T48(2) CT_T48(4) CT_T48(8) CT_T48(16)
                case 32: if (nv <= 4) CT_TN(32, 4); else if (nv <= 8) CT_TN(32, 8); else CT_TN(32, 0); break;
            }
#undef CT_T48
#undef CT_TN
            CT_COUNT_LAUNCH();
            CT_LAUNCH_CHECK();
        };
        // one update pass over the listed chunks
        auto update = [&](const Hubs &hb, int64_t nck, const int4 *list, const Batch &bt, unsigned long long *root) {
            const Chunks ch{list, chunk_len, keys.p, cov.p};
            if (l2) {
                const size_t sm = (size_t)mcap * dp * sizeof(float);
                dispatch([&](auto T, auto V) {
                    if (prune)
                        k_net_update_l2<T(), V(), true><<<(unsigned)nck, BT, sm, s>>>(Xp.p, dp, ids.p, D.p, lab.p, ch, hb, bt, root);
                    else
                        k_net_update_l2<T(), V(), false><<<(unsigned)nck, BT, sm, s>>>(Xp.p, dp, ids.p, D.p, lab.p, ch, hb, bt, root);
                });
                return;
            }
            if (ham) {
                const size_t sm = (size_t)NET_M * wp * sizeof(uint32_t);
                switch (wp / 4) {
#define CT_UH(Q) k_net_update_ham<Q><<<(unsigned)nck, BT, sm, s>>>(Xb.p, wp, ids.p, D.p, lab.p, ch, hb, bt, root)
                    case 1: CT_UH(1); break;
                    case 2: CT_UH(2); break;
                    case 3: CT_UH(3); break;
                    case 4: CT_UH(4); break;
                    default: CT_UH(0); break;
#undef CT_UH
                }
            } else {
                const size_t sm = (size_t)mcap * mask_bytes;
                switch (W) {
#define CT_UL(WW) case WW: if (wide) allow_smem(k_net_update_lev<WW>, (size_t)LEV_WIDE_M * 256 * WW * sizeof(uint64_t)); k_net_update_lev<WW><<<(unsigned)nck, BT, sm, s>>>(S, ids.p, D.p, lab.p, ch, hb, bt, prune && !root, root); break;
                    CT_UL(1) CT_UL(2) CT_UL(4) CT_UL(8) CT_UL(16)
#undef CT_UL
                }
            }
            CT_COUNT_LAUNCH();
            CT_LAUNCH_CHECK();
        };
        // the listed hubs' next batches and, where updates prune, their distances to the hubs' centres
        auto select = [&](const Hubs &hb, int nlist, const int2 *list, const int64_t *coff, const Batch &bt,
                          int32_t *active) {
            const Chunks ch{nullptr, chunk_len, keys.p, cov.p};
            if (l2) {
                const int cands = dp <= 32 ? NET_C : NET_C / 2, staged = dp <= 256;
                const size_t sm = staged ? net_select_smem(cands, dp) : 0;
                const size_t dsm = (size_t)mcap * dp * sizeof(float);
                dispatch([&](auto T, auto V) {
                    auto kern = T() <= 2 ? k_net_select_l2<NET_C, T()> : k_net_select_l2<NET_C / 2, T()>;
                    if (cands == NET_C / 2) kern = k_net_select_l2<NET_C / 2, T()>;
                    if (sm > 40 * 1024)
                        allow_smem(kern, cands == NET_C ? net_select_smem(NET_C, 32) : net_select_smem(NET_C / 2, 256));
                    kern<<<(unsigned)nlist, BT, sm, s>>>(Xp.p, dp, ids.p, list, hb, coff, ch, bt, mcap, staged, active);
                    if (prune) {
                        CT_COUNT_LAUNCH();
                        k_net_dists_l2<T(), V()><<<dim3((unsigned)nlist, nlist >= 64 ? 4 : 32), BT, dsm, s>>>(Xp.p, dp, ids.p, list, hb, bt, chunk_len);
                    }
                });
                return;
            }
            if (ham) {
                const size_t sm = net_select_ham_smem(wp);
                if (sm > 40 * 1024) allow_smem(k_net_select_ham, net_select_ham_smem(128));  // 4096 bits
                k_net_select_ham<<<(unsigned)nlist, BT, sm, s>>>(Xb.p, wp, ids.p, list, hb, coff, ch, bt, active);
            } else {
                const size_t sm = mask_bytes;
                k_net_cands_lev<<<(unsigned)nlist, BT, 0, s>>>(list, hb, coff, ch, lc);
                CT_COUNT_LAUNCH();
                switch (W) {
#define CT_PL(WW) case WW: k_net_pairs_lev<WW><<<dim3((unsigned)nlist, LEV_C), LEV_C, sm, s>>>(S, ids.p, list, hb, lc, chunk_len); break;
                    CT_PL(1) CT_PL(2) CT_PL(4) CT_PL(8) CT_PL(16)
#undef CT_PL
                }
                CT_COUNT_LAUNCH();
                k_net_pick_lev<<<(unsigned)nlist, 128, 0, s>>>(list, hb, bt, lc, mcap, chunk_len, active);
                if (prune) CT_COUNT_LAUNCH();
                if (prune) switch (W) {
#define CT_DL(WW) case WW: k_net_dists_lev<WW><<<dim3((unsigned)nlist, (unsigned)mcap), 128, sm, s>>>(S, ids.p, list, hb, bt, chunk_len); break;
                    CT_DL(1) CT_DL(2) CT_DL(4) CT_DL(8) CT_DL(16)
#undef CT_DL
                }
            }
            CT_COUNT_LAUNCH();
            CT_LAUNCH_CHECK();
        };
        int64_t nchunks = ceil_div(n, chunk_len);
        auto grow_chunks = [&]() {
            for (DBuf<int4> *c : {&chunks_a, &chunks_b})
                if ((int64_t)c->n < nchunks) *c = DBuf<int4>(nchunks, s);
            if ((int64_t)cov.n < nchunks * NET_KEYS) {
                keys = DBuf<unsigned long long>(nchunks * NET_KEYS, s);
                cov = DBuf<int32_t>(nchunks * NET_KEYS, s);
            }
        };
        // the roots: vertices 0 .. R - 1, one hub each, with a batch of one centre (its first position)
        if (R0 > 1) {
            std::vector<int32_t> hb(R0), hn(R0);
            nchunks = 0;
            for (int c = 0; c < R0; ++c) {
                hb[c] = (int32_t)hroot[c];
                hn[c] = (int32_t)((c + 1 < R0 ? hroot[c + 1] : n) - hroot[c]);
                nchunks += ceil_div(hn[c], chunk_len);
            }
            CT_CHECK_CUDA(cudaMemcpyAsync(rbegin.p, hb.data(), R0 * sizeof(int32_t), cudaMemcpyHostToDevice, s));
            CT_CHECK_CUDA(cudaMemcpyAsync(rcount.p, hn.data(), R0 * sizeof(int32_t), cudaMemcpyHostToDevice, s));
            CT_CHECK_CUDA(cudaStreamSynchronize(s));  // the host arrays are on the stack
        }
        DBuf<int64_t> i64tmp(4, s);
        DBuf<int32_t> rhub(R0, s), rleafy(R0, s);
        DBuf<int64_t> roff(R0, s);
        DBuf<unsigned long long> rkey(R0, s);  // each root's farthest point
        CT_CHECK_CUDA(cudaMemsetAsync(i64tmp.p, 0, 4 * sizeof(int64_t), s));
        CT_CHECK_CUDA(cudaMemsetAsync(rleafy.p, 0, R0 * sizeof(int32_t), s));
        grow_chunks();
        k_root_hubs<<<grid_for(R0), BT, 0, s>>>(R0, rbegin.p, rcount.p, H, bpos.p, hl_a.p, rkey.p);
        CT_COUNT_LAUNCH();
        k_chunk_counts<<<grid_for(R0), BT, 0, s>>>(R0, hl_a.p, H.count, chunk_len, rhub.p);
        CT_COUNT_LAUNCH();
        exclusive_scan_i32_to_i64(rhub.p, roff.p, R0, nullptr, s);
        k_chunk_fill<<<grid_for(nchunks), BT, 0, s>>>(nchunks, R0, hl_a.p, H.begin, roff.p, chunk_len, chunks_a.p);
        CT_COUNT_LAUNCH();
        update(H, nchunks, chunks_a.p, Batch{bpos.p, cpos.p, dcc.p}, rkey.p);
        k_make_nodes<<<grid_for(R0), BT, 0, s>>>(R0, 0, zeta, pts->metric, rbegin.p, rcount.p, rkey.p, nb.p, ncnt.p,
                                                 cbeg.p, ccnt.p, rad.p, lvl.p, rleafy.p, rhub.p);
        CT_COUNT_LAUNCH();
        exclusive_scan_i32_to_i64(rhub.p, roff.p, R0, i64tmp.p, s);
        k_next_hubs<<<grid_for(R0), BT, 0, s>>>(R0, 0, rhub.p, roff.p, rbegin.p, rcount.p, lvl.p, H2, small_max,
                                                chunk_len, hl_a.p, reinterpret_cast<int32_t *>(i64tmp.p + 1));
        CT_COUNT_LAUNCH();
        CT_LAUNCH_CHECK();
        int64_t first[3] = {0, 0, 0};
        to_host(first, i64tmp.p, 3, s);
        std::swap(H, H2);
        n_nodes = R0;
        int64_t nh = first[0];
        int nl = (int32_t)first[1];  // hubs of the level-wide passes
        nchunks = (int32_t)first[2];

        // scratch for partitioning
        DBuf<uint32_t> pk(n, s), pv(n, s), tk(n, s), tv(n, s);
        DBuf<int32_t> rpos(n, s), tids(n, s);
        DBuf<float> tD(n, s);
        DBuf<int32_t> active(3, s);  // batches taken in a burst; hubs and chunks left

        while (nh > 0) {
            ++depth;
            {
                ProfScope prof_split("build_split", s);
                if (small_max && (nl < nh)) {
                    dispatch([&](auto T, auto V) {
                        if constexpr (T() <= 8)
                            k_split_small<T(), V()><<<(unsigned)nh, BT, 0, s>>>(Xp.p, dp, ids.p, D.p, lab.p, H);
                    });
                }
                if (nl) {
                    // the listed hubs' chunk table
                    DBuf<int32_t> ccounts(nl, s);
                    DBuf<int64_t> coff(nl, s);
                    grow_chunks();
                    if (lev && (int64_t)lcn.n < nl) lcn = DBuf<int32_t>(nl, s);
                    lc.n = lcn.p;
                    k_chunk_counts<<<grid_for(nl), BT, 0, s>>>(nl, hl_a.p, H.count, chunk_len, ccounts.p);
                    CT_COUNT_LAUNCH();
                    exclusive_scan_i32_to_i64(ccounts.p, coff.p, nl, nullptr, s);
                    k_chunk_fill<<<grid_for(nchunks), BT, 0, s>>>(nchunks, nl, hl_a.p, H.begin, coff.p, chunk_len,
                                                                  chunks_a.p);
                    CT_COUNT_LAUNCH();
                    CT_LAUNCH_CHECK();
                    const Batch bt{bpos.p, cpos.p, dcc.p};
                    int2 *hl = hl_a.p, *hl2 = hl_b.p;
                    int4 *cl = chunks_a.p, *cl2 = chunks_b.p;
                    int64_t nck = nchunks;
                    // bursts of passes (the first compares nothing: it reports the farthest points), then the
                    // hubs and chunks still splitting
                    int64_t done_passes = 0;
                    for (int burst = 2; nl > 0; burst = std::min(2 * burst, 8)) {
                        // every pass gives each hub left a new centre: none is left after n + 1 passes
                        if (done_passes > n + 2) CT_FAIL(CT_ECUDA, "split loop did not terminate");
                        done_passes += burst;
                        CT_CHECK_CUDA(cudaMemsetAsync(active.p, 0, 3 * sizeof(int32_t), s));
                        for (int it = 0; it < burst; ++it) {
                            update(H, nck, cl, bt, nullptr);
                            select(H, nl, hl, coff.p, bt, active.p);
                        }
                        k_active<<<grid_for(std::max<int64_t>(nl, nck)), BT, 0, s>>>(nl, hl, nck, cl, H.done, hl2, cl2,
                                                                                    active.p + 1);
                        CT_COUNT_LAUNCH();
                        CT_LAUNCH_CHECK();
                        int32_t act[3] = {0, 0, 0};
                        to_host(act, active.p, 3, s);
                        nl = act[1];
                        nck = act[2];
                        std::swap(hl, hl2);
                        std::swap(cl, cl2);
                    }
                }
            }

            // partition the round's points by (hub, label)
            DBuf<int32_t> ncs(nh, s);
            DBuf<int64_t> child_base(nh, s), round_off(nh, s);
            CT_CHECK_CUDA(cudaMemcpyAsync(ncs.p, H.nc, nh * sizeof(int32_t), cudaMemcpyDeviceToDevice, s));
            exclusive_scan_i32_to_i64(ncs.p, child_base.p, nh, i64tmp.p, s);
            exclusive_scan_i32_to_i64(H.count, round_off.p, nh, i64tmp.p + 1, s);
            int64_t tot[2];
            to_host(tot, i64tmp.p, 2, s);
            const int64_t T = tot[0], R = tot[1];
            if (n_nodes + T > cap) CT_FAIL(CT_ECUDA, "vertex capacity exceeded");
            k_part_keys<<<grid_for(R), BT, 0, s>>>(R, (int)nh, H.begin, round_off.p, child_base.p, lab.p, pk.p,
                                                   pv.p, rpos.p);
            CT_COUNT_LAUNCH();
            radix_sort_pairs(pk.p, pv.p, tk.p, tv.p, R, bits_for(T), s);
            DBuf<int32_t> ccount(T, s), cbegin(T, s), czero(T, s), is_hub(T, s), leafy(T, s);
            DBuf<unsigned long long> ckey(T, s);
            CT_CHECK_CUDA(cudaMemsetAsync(ccount.p, 0, T * sizeof(int32_t), s));
            CT_CHECK_CUDA(cudaMemsetAsync(cbegin.p, 0x7f, T * sizeof(int32_t), s));
            CT_CHECK_CUDA(cudaMemsetAsync(czero.p, 0x7f, T * sizeof(int32_t), s));
            CT_CHECK_CUDA(cudaMemsetAsync(ckey.p, 0, T * sizeof(unsigned long long), s));
            k_part_gather<<<grid_for(R), BT, 0, s>>>(R, pk.p, pv.p, rpos.p, ids.p, D.p, tids.p, tD.p, ccount.p,
                                                     cbegin.p, czero.p);
            CT_COUNT_LAUNCH();
            k_part_scatter<<<grid_for(R), BT, 0, s>>>(R, rpos.p, tids.p, tD.p, ids.p, D.p, lab.p);
            CT_COUNT_LAUNCH();
            k_centre_front<<<grid_for(T), BT, 0, s>>>(T, cbegin.p, czero.p, ids.p, D.p, err.p);
            CT_COUNT_LAUNCH();
            k_child_keys<<<grid_for(R), BT, 0, s>>>(R, pk.p, rpos.p, D.p, ckey.p);
            CT_COUNT_LAUNCH();
            k_link_children<<<grid_for(T), BT, 0, s>>>(T, (int)nh, H, child_base.p, n_nodes, cbeg.p, ccnt.p, lvl.p,
                                                       par.p, leafy.p);
            CT_COUNT_LAUNCH();
            k_make_nodes<<<grid_for(T), BT, 0, s>>>(T, n_nodes, zeta, pts->metric, cbegin.p, ccount.p, ckey.p,
                                                    nb.p, ncnt.p, cbeg.p, ccnt.p, rad.p, lvl.p, leafy.p, is_hub.p);
            CT_COUNT_LAUNCH();
            DBuf<int64_t> hub_off(T, s);
            CT_CHECK_CUDA(cudaMemsetAsync(i64tmp.p + 1, 0, 2 * sizeof(int64_t), s));
            exclusive_scan_i32_to_i64(is_hub.p, hub_off.p, T, i64tmp.p, s);
            // a hub has more than zeta points: at most n / (zeta + 1) of them, within cap_h
            k_next_hubs<<<grid_for(T), BT, 0, s>>>(T, n_nodes, is_hub.p, hub_off.p, cbegin.p, ccount.p, lvl.p,
                                                   H2, small_max, chunk_len, hl_a.p,
                                                   reinterpret_cast<int32_t *>(i64tmp.p + 1));
            CT_COUNT_LAUNCH();
            CT_LAUNCH_CHECK();
            int64_t next[3] = {0, 0, 0};  // hubs; listed hubs (int32); their chunks (int32)
            to_host(next, i64tmp.p, 3, s);
            n_nodes += (int)T;
            std::swap(H, H2);
            nh = next[0];
            nl = (int32_t)next[1];
            nchunks = (int32_t)next[2];
        }
        int32_t e2 = 0;
        to_host(&e2, err.p, 1, s);
        if (e2) CT_FAIL(CT_ECUDA, "internal: a child without a zero-distance centre");
    }

    // ---- final layout
    t->n_nodes = n_nodes;
    t->depth = depth;
    if (off) {
        finish_forest(*t, *off, n_nodes, ids, D, nb, ncnt, cbeg, ccnt, lvl, par, rad, Xp.p, Xb.p, *out, s);
        return nullptr;
    }
    t->perm = ids.release();
    t->dcen = D.release();
    lab.reset();
    if (n == 0) {
        // empty tree: keep valid (non-null) small allocations
        t->perm = (int32_t *)dmalloc(sizeof(int32_t), s);
        t->dcen = (float *)dmalloc(sizeof(float), s);
    }
    if (l2) {
        t->pts = (float *)dmalloc((size_t)(n ? n : 1) * dp * sizeof(float) + 16, s);
        if (n) {
            k_gather_rows<<<grid_for(n * (dp / 4)), BT, 0, s>>>(Xp.p, dp, t->perm, n, t->pts);
            CT_COUNT_LAUNCH();
        }
        Xp.reset();
    } else if (ham) {
        t->bits = (uint32_t *)dmalloc((size_t)(n ? n : 1) * wp * sizeof(uint32_t) + 16, s);
        if (n) {
            k_gather_bits<<<grid_for(n * (wp / 4)), BT, 0, s>>>(Xb.p, wp, t->perm, n, t->bits);
            CT_COUNT_LAUNCH();
        }
        Xb.reset();
    } else {
        DBuf<int64_t> lens(n + 1, s);
        DBuf<int32_t> ml(1, s);
        CT_CHECK_CUDA(cudaMemsetAsync(ml.p, 0, sizeof(int32_t), s));
        if (n) {
            k_string_lengths<<<grid_for(n), BT, 0, s>>>(n, t->perm, pts->offsets, lens.p, ml.p);
            CT_COUNT_LAUNCH();
        }
        t->soff = (int64_t *)dmalloc((size_t)(n + 1) * sizeof(int64_t), s);
        DBuf<int64_t> tot(1, s);
        exclusive_scan_i64(lens.p, t->soff, n, tot.p, s);
        CT_CHECK_CUDA(cudaMemcpyAsync(t->soff + n, tot.p, sizeof(int64_t), cudaMemcpyDeviceToDevice, s));
        int64_t total = 0;
        to_host(&total, tot.p, 1, s);
        t->sbytes = total;
        t->sdata = (uint8_t *)dmalloc((size_t)total + 16, s);
        if (n) {
            k_gather_strings<<<(unsigned)n, 128, 0, s>>>(n, t->perm, (const uint8_t *)pts->data, pts->offsets,
                                                         t->soff, t->sdata);
            CT_COUNT_LAUNCH();
        }
    }
    // shrink vertex arrays to n_nodes
    auto shrink_i = [&](DBuf<int32_t> &b) {
        int32_t *p = (int32_t *)dmalloc(sizeof(int32_t) * (size_t)(n_nodes ? n_nodes : 1), s);
        if (n_nodes) CT_CHECK_CUDA(cudaMemcpyAsync(p, b.p, sizeof(int32_t) * n_nodes, cudaMemcpyDeviceToDevice, s));
        b.reset();
        return p;
    };
    t->node_begin = shrink_i(nb);
    t->node_count = shrink_i(ncnt);
    t->child_begin = shrink_i(cbeg);
    t->child_count = shrink_i(ccnt);
    t->level = shrink_i(lvl);
    t->parent = shrink_i(par);
    t->radius = (float *)dmalloc(sizeof(float) * (size_t)(n_nodes ? n_nodes : 1), s);
    if (n_nodes) CT_CHECK_CUDA(cudaMemcpyAsync(t->radius, rad.p, sizeof(float) * n_nodes, cudaMemcpyDeviceToDevice, s));
    rad.reset();
    if (l2) {
        t->node_ctr = (float *)dmalloc(sizeof(float) * (size_t)(n_nodes ? n_nodes : 1) * dp + 16, s);
        if (n_nodes) {
            k_node_centres<<<grid_for((int64_t)n_nodes * (dp / 4)), BT, 0, s>>>(n_nodes, t->node_begin, t->pts, dp,
                                                                               t->node_ctr);
            CT_COUNT_LAUNCH();
        }
    }
    // leaf blocks in position order
    {
        int64_t nn = n_nodes ? n_nodes : 1;
        DBuf<uint32_t> k1(nn, s), v1(nn, s), k2(nn, s), v2(nn, s);
        DBuf<int32_t> cnts(2, s);
        CT_CHECK_CUDA(cudaMemsetAsync(cnts.p, 0, 2 * sizeof(int32_t), s));
        if (n_nodes) {
            k_leaf_keys<<<grid_for(n_nodes), BT, 0, s>>>(n_nodes, t->child_count, t->node_begin, t->node_count, k1.p,
                                                         v1.p, cnts.p, cnts.p + 1);
            CT_COUNT_LAUNCH();
        }
        int32_t hc[2];
        to_host(hc, cnts.p, 2, s);
        t->n_leaves = hc[0];
        t->max_leaf_count = hc[1];
        radix_sort_pairs(k1.p, v1.p, k2.p, v2.p, hc[0], bits_for(n), s);
        t->leaf_ids = (int32_t *)dmalloc(sizeof(int32_t) * (size_t)(hc[0] ? hc[0] : 1), s);
        if (hc[0]) CT_CHECK_CUDA(cudaMemcpyAsync(t->leaf_ids, v1.p, sizeof(int32_t) * hc[0], cudaMemcpyDeviceToDevice, s));
    }
    // query groups: greedy runs of consecutive sibling leaf blocks (k_group_marks)
    {
        const int L = t->n_leaves;
        DBuf<int32_t> gstart(L ? L : 1, s), gsize(L ? L : 1, s), lcount(L ? L : 1, s), lpar(L ? L : 1, s);
        DBuf<int64_t> gidx(L ? L : 1, s), tot(2, s);  // tot: group count, largest group
        CT_CHECK_CUDA(cudaMemsetAsync(tot.p, 0, 2 * sizeof(int64_t), s));
        if (L) {
            k_group_prep<<<grid_for(L), BT, 0, s>>>(L, t->leaf_ids, t->node_count, t->parent, lcount.p, lpar.p);
            CT_COUNT_LAUNCH();
            k_group_marks<<<grid_for(L), BT, 0, s>>>(L, lcount.p, lpar.p, gstart.p, gsize.p,
                                                     reinterpret_cast<unsigned long long *>(tot.p + 1));
            CT_COUNT_LAUNCH();
            exclusive_scan_i32_to_i64(gstart.p, gidx.p, L, tot.p, s);
        }
        int64_t gh[2] = {0, 0};
        to_host(gh, tot.p, 2, s);
        const int G = (int)gh[0];
        t->n_groups = G;
        t->max_group_count = (int)gh[1];
        t->group_begin = (int32_t *)dmalloc(sizeof(int32_t) * (size_t)(G ? G : 1), s);
        t->group_count = (int32_t *)dmalloc(sizeof(int32_t) * (size_t)(G ? G : 1), s);
        if (G) {
            k_group_scatter<<<grid_for(L), BT, 0, s>>>(L, t->leaf_ids, t->node_begin, gstart.p, gsize.p, gidx.p,
                                                       t->group_begin, t->group_count);
            CT_COUNT_LAUNCH();
        }
        t->group_radius = (float *)dmalloc(sizeof(float) * (size_t)(G ? G : 1), s);
        if (G) {
            if (ham) {
                k_group_radius_ham<<<grid_for((int64_t)G * 32), BT, 0, s>>>(G, t->group_begin, t->group_count,
                                                                           t->bits, wp, t->group_radius);
            } else if (l2) {
                k_group_radius_l2<<<grid_for((int64_t)G * 32), BT, 0, s>>>(G, t->group_begin, t->group_count, t->pts,
                                                                          dp, t->group_radius);
            } else {
                switch (W) {
#define CT_GR(WW) case WW: k_group_radius_lev<WW><<<G, 32, 0, s>>>(G, t->group_begin, t->group_count, t->sdata, t->soff, t->group_radius); break;
                    CT_GR(1) CT_GR(2) CT_GR(4) CT_GR(8) CT_GR(16)
#undef CT_GR
                }
            }
            CT_COUNT_LAUNCH();
        }
        // traversal order: groups with larger balls walk more of the tree; taking
        // them first shortens the tail of the dynamically scheduled walk
        t->group_order = (int32_t *)dmalloc(sizeof(int32_t) * (size_t)(G ? G : 1), s);
        if (G) {
            DBuf<uint32_t> ok(G, s), ov(G, s), tk2(G, s), tv2(G, s);
            k_radius_desc_keys<<<grid_for(G), BT, 0, s>>>(G, t->group_radius, ok.p, ov.p);
            CT_COUNT_LAUNCH();
            radix_sort_pairs(ok.p, ov.p, tk2.p, tv2.p, G, 32, s);
            CT_CHECK_CUDA(cudaMemcpyAsync(t->group_order, ov.p, sizeof(int32_t) * G, cudaMemcpyDeviceToDevice, s));
        }
    }
    CT_LAUNCH_CHECK();
    CT_CHECK_CUDA(cudaStreamSynchronize(s));
    tg.t = nullptr;
    return t;
}

// ---- Forests: trees built one after another cost their launches and
// read-backs each (60 cells of 96820 x 64: 113 ms, 125 launches a tree); split
// together they cost one tree's (5.2 ms).  The trees' vertices are created
// level by level in one array;
// a stable sort by tree gives each tree its own consecutive vertices (its root
// first, siblings still consecutive), and every array is made relative to its
// tree.

// The tree (of R, by first position) that holds a position.
__device__ __forceinline__ int tree_of(const int32_t *__restrict__ rbegin, int R, int pos) {
    int lo = 0, hi = R;
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (__ldg(rbegin + mid) <= pos) lo = mid; else hi = mid;
    }
    return lo;
}
__global__ void k_tree_keys(int64_t n, const int32_t *__restrict__ pos, const uint32_t *__restrict__ order, int R,
                            const int32_t *__restrict__ rbegin, uint32_t *__restrict__ keys,
                            uint32_t *__restrict__ vals) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const uint32_t v = order ? order[i] : (uint32_t)i;
    keys[i] = (uint32_t)tree_of(rbegin, R, pos[v]);
    vals[i] = v;
}
// base[r] = first index of the (ascending) keys not below bound[r]; base[R] = n.
__global__ void k_bounds(int R, int64_t n, const uint32_t *__restrict__ keys, const int32_t *__restrict__ bound,
                         int32_t *__restrict__ base) {
    const int r = blockIdx.x * blockDim.x + threadIdx.x;
    if (r > R) return;
    const uint32_t want = r == R ? 0xffffffffu : bound ? (uint32_t)bound[r] : (uint32_t)r;
    int64_t lo = 0, hi = n;
    while (lo < hi) {
        const int64_t mid = (lo + hi) >> 1;
        if (r < R && keys[mid] >= want) hi = mid; else lo = mid + 1;
    }
    base[r] = (int32_t)lo;
}
__global__ void k_invert(int64_t n, const uint32_t *__restrict__ order, int32_t *__restrict__ inv) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) inv[order[i]] = (int32_t)i;
}
struct NodeArrays {
    int32_t *begin, *count, *cbegin, *ccount, *level, *parent;
    float *radius;
};
// Vertex j of the sorted order from its old record: indices in the sorted
// order (children, parents; a root's parent becomes -2 - tree, so that
// neighbouring trees' roots are no siblings).
__global__ void k_forest_nodes(int64_t N, const uint32_t *__restrict__ order, const uint32_t *__restrict__ tree,
                               const int32_t *__restrict__ inv, NodeArrays a, NodeArrays b) {
    const int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= N) return;
    const uint32_t v = order[j];
    b.begin[j] = a.begin[v];
    b.count[j] = a.count[v];
    const int cc = a.ccount[v], p = a.parent[v];
    b.ccount[j] = cc;
    b.cbegin[j] = cc ? inv[a.cbegin[v]] : 0;
    b.parent[j] = p >= 0 ? inv[p] : -2 - (int)tree[j];
    b.level[j] = a.level[v];
    b.radius[j] = a.radius[v];
}
// Everything relative to its tree.
__global__ void k_forest_local(int64_t N, int64_t L, int64_t G, int64_t n, int R,
                               const int32_t *__restrict__ rbegin, const int32_t *__restrict__ nbase,
                               const int32_t *__restrict__ gbase, const uint32_t *__restrict__ ntree, NodeArrays b,
                               const uint32_t *__restrict__ leaf_keys, const uint32_t *__restrict__ leaves,
                               int32_t *__restrict__ leaf_ids, int32_t *__restrict__ group_begin,
                               const uint32_t *__restrict__ gtree, const uint32_t *__restrict__ gsorted,
                               int32_t *__restrict__ group_order, int32_t *__restrict__ perm) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < N) {
        const int t = (int)ntree[i];
        b.begin[i] -= rbegin[t];
        if (b.ccount[i]) b.cbegin[i] -= nbase[t];
        b.parent[i] = b.parent[i] >= 0 ? b.parent[i] - nbase[t] : -1;
    }
    if (i < L) leaf_ids[i] = (int32_t)leaves[i] - nbase[tree_of(rbegin, R, (int)leaf_keys[i])];
    if (i < G) {
        group_order[i] = (int32_t)gsorted[i] - gbase[gtree[i]];
        group_begin[i] -= rbegin[tree_of(rbegin, R, group_begin[i])];
    }
    if (i < n) perm[i] -= rbegin[tree_of(rbegin, R, (int)i)];
}

void finish_forest(const ct_tree &proto, const std::vector<int64_t> &off, int N, DBuf<int32_t> &ids, DBuf<float> &D,
                   DBuf<int32_t> &nb, DBuf<int32_t> &ncnt, DBuf<int32_t> &cbeg, DBuf<int32_t> &ccnt,
                   DBuf<int32_t> &lvl, DBuf<int32_t> &par, DBuf<float> &rad, const float *Xp, const uint32_t *Xb,
                   std::vector<ct_tree *> &out, cudaStream_t s) {
    const int64_t n = proto.n;
    const int C = (int)off.size() - 1, dp = proto.dp, wp = proto.wp;
    const bool l2 = proto.metric == CT_L2_F32;
    std::vector<int> tree_cell;  // the trees with points
    std::vector<int32_t> hb;
    for (int c = 0; c < C; ++c)
        if (off[c] < off[c + 1]) {
            tree_cell.push_back(c);
            hb.push_back((int32_t)off[c]);
        }
    const int R = (int)hb.size();
    // the arrays of all trees, released with the last tree
    struct Blocks {
        cudaStream_t s;
        std::vector<void *> p;
        ~Blocks() {
            for (void *q : p) cudaFreeAsync(q, s);
            cudaStreamSynchronize(s);
        }
    };
    auto blocks = std::make_shared<Blocks>();
    blocks->s = s;
    auto take = [&](size_t bytes) {
        void *q = dmalloc(bytes + 16, s);
        blocks->p.push_back(q);
        return q;
    };
    auto take_i = [&](int64_t k) { return (int32_t *)take((size_t)std::max<int64_t>(k, 1) * sizeof(int32_t)); };
    DBuf<int32_t> rbegin(std::max(R, 1), s), nbase(R + 1, s), lbase(R + 1, s), gbase(R + 1, s);
    if (R) CT_CHECK_CUDA(cudaMemcpyAsync(rbegin.p, hb.data(), R * sizeof(int32_t), cudaMemcpyHostToDevice, s));
    const int tbits = bits_for(R);
    // vertices by tree
    DBuf<uint32_t> nk(std::max(N, 1), s), nv(std::max(N, 1), s), tk(std::max(N, 1), s), tv(std::max(N, 1), s);
    DBuf<int32_t> inv(std::max(N, 1), s);
    NodeArrays a{nb.p, ncnt.p, cbeg.p, ccnt.p, lvl.p, par.p, rad.p}, b{};
    b.begin = take_i(N);
    b.count = take_i(N);
    b.cbegin = take_i(N);
    b.ccount = take_i(N);
    b.level = take_i(N);
    b.parent = take_i(N);
    b.radius = (float *)take_i(N);
    float *pts = nullptr, *ctr = nullptr;
    uint32_t *bits = nullptr;
    int32_t *perm = take_i(n);
    float *dcen = (float *)take_i(n);
    if (l2) {
        pts = (float *)take((size_t)std::max<int64_t>(n, 1) * dp * sizeof(float));
        ctr = (float *)take((size_t)std::max(N, 1) * dp * sizeof(float));
    } else {
        bits = (uint32_t *)take((size_t)std::max<int64_t>(n, 1) * wp * sizeof(uint32_t));
    }
    int32_t hc[2] = {0, 0};
    DBuf<uint32_t> lk(std::max(N, 1), s), lv(std::max(N, 1), s);
    DBuf<int32_t> cnts(2, s);
    CT_CHECK_CUDA(cudaMemsetAsync(cnts.p, 0, 2 * sizeof(int32_t), s));
    if (N) {
        k_tree_keys<<<grid_for(N), BT, 0, s>>>(N, nb.p, nullptr, R, rbegin.p, nk.p, nv.p);
        CT_COUNT_LAUNCH();
        radix_sort_pairs(nk.p, nv.p, tk.p, tv.p, N, tbits, s);
        k_bounds<<<grid_for(R + 1), BT, 0, s>>>(R, N, nk.p, nullptr, nbase.p);
        CT_COUNT_LAUNCH();
        k_invert<<<grid_for(N), BT, 0, s>>>(N, nv.p, inv.p);
        CT_COUNT_LAUNCH();
        k_forest_nodes<<<grid_for(N), BT, 0, s>>>(N, nv.p, nk.p, inv.p, a, b);
        CT_COUNT_LAUNCH();
        CT_CHECK_CUDA(cudaMemcpyAsync(perm, ids.p, n * sizeof(int32_t), cudaMemcpyDeviceToDevice, s));
        CT_CHECK_CUDA(cudaMemcpyAsync(dcen, D.p, n * sizeof(float), cudaMemcpyDeviceToDevice, s));
        if (l2) {
            k_gather_rows<<<grid_for(n * (dp / 4)), BT, 0, s>>>(Xp, dp, perm, n, pts);
            CT_COUNT_LAUNCH();
            k_node_centres<<<grid_for((int64_t)N * (dp / 4)), BT, 0, s>>>(N, b.begin, pts, dp, ctr);
        } else {
            k_gather_bits<<<grid_for(n * (wp / 4)), BT, 0, s>>>(Xb, wp, perm, n, bits);
        }
        CT_COUNT_LAUNCH();
        k_leaf_keys<<<grid_for(N), BT, 0, s>>>(N, b.ccount, b.begin, b.count, lk.p, lv.p, cnts.p, cnts.p + 1);
        CT_COUNT_LAUNCH();
        CT_LAUNCH_CHECK();
    }
    to_host(hc, cnts.p, 2, s);
    const int L = hc[0];
    // leaf blocks in position order, groups as in a single tree
    int32_t *leaf_ids = take_i(L);
    DBuf<int32_t> gstart(std::max(L, 1), s), gsize(std::max(L, 1), s), lcount(std::max(L, 1), s), lpar(std::max(L, 1), s);
    DBuf<int64_t> gidx(std::max(L, 1), s), tot(2, s);
    CT_CHECK_CUDA(cudaMemsetAsync(tot.p, 0, 2 * sizeof(int64_t), s));
    if (L) {
        radix_sort_pairs(lk.p, lv.p, tk.p, tv.p, L, bits_for(n), s);
        k_bounds<<<grid_for(R + 1), BT, 0, s>>>(R, L, lk.p, rbegin.p, lbase.p);
        CT_COUNT_LAUNCH();
        const int32_t *leaves = reinterpret_cast<const int32_t *>(lv.p);
        k_group_prep<<<grid_for(L), BT, 0, s>>>(L, leaves, b.count, b.parent, lcount.p, lpar.p);
        CT_COUNT_LAUNCH();
        k_group_marks<<<grid_for(L), BT, 0, s>>>(L, lcount.p, lpar.p, gstart.p, gsize.p,
                                                 reinterpret_cast<unsigned long long *>(tot.p + 1));
        CT_COUNT_LAUNCH();
        exclusive_scan_i32_to_i64(gstart.p, gidx.p, L, tot.p, s);
    }
    int64_t gh[2] = {0, 0};
    to_host(gh, tot.p, 2, s);
    const int G = (int)gh[0];
    int32_t *gbeg = take_i(G), *gcnt = take_i(G), *gord = take_i(G);
    float *grad = (float *)take_i(G);
    std::vector<int32_t> hn(R + 1, 0), hl(R + 1, 0), hg(R + 1, 0);
    if (G) {
        k_group_scatter<<<grid_for(L), BT, 0, s>>>(L, reinterpret_cast<const int32_t *>(lv.p), b.begin, gstart.p,
                                                   gsize.p, gidx.p, gbeg, gcnt);
        CT_COUNT_LAUNCH();
        if (l2)
            k_group_radius_l2<<<grid_for((int64_t)G * 32), BT, 0, s>>>(G, gbeg, gcnt, pts, dp, grad);
        else
            k_group_radius_ham<<<grid_for((int64_t)G * 32), BT, 0, s>>>(G, gbeg, gcnt, bits, wp, grad);
        CT_COUNT_LAUNCH();
        // walk order: by decreasing radius, then (stably) by tree
        DBuf<uint32_t> ok(G, s), ov(G, s), ok2(G, s), ov2(G, s), sk(G, s), sv(G, s);
        k_radius_desc_keys<<<grid_for(G), BT, 0, s>>>(G, grad, ok.p, ov.p);
        CT_COUNT_LAUNCH();
        radix_sort_pairs(ok.p, ov.p, sk.p, sv.p, G, 32, s);
        k_tree_keys<<<grid_for(G), BT, 0, s>>>(G, gbeg, ov.p, R, rbegin.p, ok2.p, ov2.p);
        CT_COUNT_LAUNCH();
        radix_sort_pairs(ok2.p, ov2.p, sk.p, sv.p, G, tbits, s);
        k_bounds<<<grid_for(R + 1), BT, 0, s>>>(R, G, ok2.p, nullptr, gbase.p);
        CT_COUNT_LAUNCH();
        const int64_t most = std::max<int64_t>(std::max<int64_t>(N, L), std::max<int64_t>(G, n));
        k_forest_local<<<grid_for(most), BT, 0, s>>>(N, L, G, n, R, rbegin.p, nbase.p, gbase.p, nk.p, b, lk.p, lv.p,
                                                     leaf_ids, gbeg, ok2.p, ov2.p, gord, perm);
        CT_COUNT_LAUNCH();
        CT_LAUNCH_CHECK();
        to_host_async(hn.data(), nbase.p, R + 1, s);
        to_host_async(hl.data(), lbase.p, R + 1, s);
        to_host_async(hg.data(), gbase.p, R + 1, s);
        CT_CHECK_CUDA(cudaStreamSynchronize(s));
    }
    // the trees: views of the arrays
    std::vector<std::unique_ptr<ct_tree>> made;
    for (int c = 0, r = 0; c < C; ++c) {
        made.emplace_back(new ct_tree(proto));  // proto: metric, dimensions, leaf size, depth
        ct_tree *t = made.back().get();
        t->shared = blocks;
        t->n = off[c + 1] - off[c];
        const bool has = t->n > 0;
        const int64_t p0 = has ? off[c] : 0, n0 = has ? hn[r] : 0, l0 = has ? hl[r] : 0, g0 = has ? hg[r] : 0;
        t->n_nodes = has ? hn[r + 1] - hn[r] : 0;
        t->n_leaves = has ? hl[r + 1] - hl[r] : 0;
        t->n_groups = has ? hg[r + 1] - hg[r] : 0;
        t->max_leaf_count = has ? hc[1] : 0;  // of the forest
        t->max_group_count = has ? (int)gh[1] : 0;
        t->perm = perm + p0;
        t->dcen = dcen + p0;
        if (l2) {
            t->pts = pts + p0 * dp;
            t->node_ctr = ctr + n0 * dp;
        } else {
            t->bits = bits + p0 * wp;
        }
        t->node_begin = b.begin + n0;
        t->node_count = b.count + n0;
        t->child_begin = b.cbegin + n0;
        t->child_count = b.ccount + n0;
        t->level = b.level + n0;
        t->parent = b.parent + n0;
        t->radius = b.radius + n0;
        t->leaf_ids = leaf_ids + l0;
        t->group_begin = gbeg + g0;
        t->group_count = gcnt + g0;
        t->group_radius = grad + g0;
        t->group_order = gord + g0;
        r += has ? 1 : 0;
    }
    for (auto &m : made) out.push_back(m.release());
}

}  // namespace

ct_tree *build_tree(const ct_points *pts, int zeta, int root, cudaStream_t s) {
    return build_impl(pts, zeta, root, s, nullptr, nullptr);
}

// A tree per consecutive range off[c] .. off[c + 1] - 1 of the points (the
// root of each its first point); the trees share their device memory.
std::vector<ct_tree *> build_forest(const ct_points *pts, const std::vector<int64_t> &off, int zeta, cudaStream_t s) {
    std::vector<ct_tree *> out;
    build_impl(pts, zeta, 0, s, &off, &out);
    return out;
}

void free_tree(ct_tree *t) {
    if (!t) return;
    if (t->shared) {  // a forest's memory goes with the last of its trees
        delete t;
        return;
    }
    cudaStream_t s = t->stream;
    void *ptrs[] = {t->pts, t->bits, t->sdata, t->soff, t->perm, t->dcen, t->node_begin, t->node_count,
                    t->child_begin, t->child_count, t->radius, t->level, t->node_ctr, t->leaf_ids,
                    t->parent, t->group_begin, t->group_count, t->group_radius, t->group_order};
    for (void *p : ptrs)
        if (p) cudaFreeAsync(p, s);
    cudaStreamSynchronize(s);
    delete t;
}

}  // namespace ct

// landmark.cu -- the ε-graph through landmarks on one GPU (Sec. IV-D; the
// paper's Algorithms 5 and 6 with the processors replaced by one batch):
//   1. Voronoi cells of the caller's centres C (each point's nearest centre,
//      the lowest index among equals);
//   2. the ε-ghosts of every cell by Lemma 1: a point p outside cell k whose
//      neighbours could lie in it, d(p, c_k) <= d(p, C) + 2 eps;
//   3. one cover tree per cell over its points and ghosts (Algorithms 1-2),
//      built together and queried together (a forest whose levels, and a batch
//      whose stages, share their launches);
//   4. every point's row taken from its own cell's CSR: by Lemma 1 each of
//      its neighbours in another cell is a ghost of its own cell, so the row
//      is complete there.
// The output is the CSR eps_graph_query returns (same entries and stored
// distances: each pair is decided by the same kernels).  A cell's members are
// kept in increasing original id, so the local-to-original map is increasing
// and rows stay sorted.
#include <algorithm>
#include <climits>
#include <cmath>
#include <vector>

#include "common.cuh"
#include "profile.cuh"
#include "query.cuh"

namespace ct {

std::vector<ct_tree *> build_forest(const ct_points *pts, const std::vector<int64_t> &off, int zeta, cudaStream_t s);
void free_tree(ct_tree *t);
void query_batched(int n_clouds, const ct_tree *const *trees, const QParams *qps, const ct_query_opts *opts,
                   cudaStream_t s, QueryOut *outs);

namespace {

constexpr int LM_T = 256;

struct LmInput {
    int metric, dim;
    const float *X;      // L2: n x dim
    const uint8_t *B;    // Hamming: n x ceil(dim/8)
    const int64_t *cid;  // m centre ids
    int m;
};

// Lemma 1's ghost test of point p (nearest-centre distance dmin) for cell k:
// exact for Hamming (integers); for L2 with a relative margin of 2^-10 over
// fp32 distances whose error is below 2^-12 (a row's terms in one chain, up to
// 4096 of them; more ghosts never change rows).
__device__ __forceinline__ bool lm_ghost(const LmInput &in, float d, float dmin, float eps_up, int lev_k) {
    if (in.metric == CT_HAMMING_B1) return d <= dmin + 2.0f * (float)lev_k;
    return d <= fmaf(dmin + eps_up, 1.0f + 0x1p-10f, eps_up) + 0x1p-60f;
}

// Distances of LM_P points to LM_C centres at a time: fp32 direct differences,
// a term after the other (L2; the ghost test carries a margin far above their
// error), or exact popcounts (Hamming).  A block has LM_P points; the rows of
// both sides go through shared memory in chunks of 32 words, coalesced, and
// every thread forms 4 x 4 of the distances.
// k_lm_cells<false>: nearest centre and distance of each point, then its number
// of memberships (its own cell and the cells it is a ghost of); a single tile
// of centres is evaluated once for both.  k_lm_cells<true>: the membership keys
// (cell << 32 | p) at moff[p], in increasing cell.
// Bound by the shared-memory reads (8 words per 16 terms).  97k x 64 against 60
// centres: both kernels together took 4.5 ms with a thread per point that read
// its row and the centres' a word at a time, 0.1 ms now.
constexpr int LM_P = 64, LM_C = 64, LM_KC = 32;

struct LmTile {
    uint32_t x[LM_P][LM_KC + 1], c[LM_C][LM_KC + 1];
    float d[LM_P][LM_C + 1];
};

// Word w of a row: a float's bits, or 32 bits of a code (bits past dim cleared).
__device__ __forceinline__ uint32_t lm_word(const LmInput &in, int64_t p, int w) {
    if (in.metric == CT_L2_F32) return __float_as_uint(in.X[p * in.dim + w]);
    const int nb = (in.dim + 7) >> 3;
    const uint8_t *r = in.B + p * nb;
    uint32_t v = 0u;
    for (int i = 0; i < 4; ++i)
        if (4 * w + i < nb) v |= (uint32_t)r[4 * w + i] << (8 * i);
    const int bits = in.dim - 32 * w;
    return bits < 32 ? v & ((1u << bits) - 1u) : v;
}

// S.d[i][j] = distance of point p0 + i and centre k0 + j (i < np, j < nc).
__device__ __forceinline__ void lm_tile(const LmInput &in, LmTile &S, int64_t p0, int np, int k0, int nc) {
    const int tid = threadIdx.x, ty = tid >> 4, tx = tid & 15;
    const bool l2 = in.metric == CT_L2_F32;
    const int words = l2 ? in.dim : (in.dim + 31) >> 5;
    float acc[4][4] = {};
    int bits[4][4] = {};
    for (int w0 = 0; w0 < words; w0 += LM_KC) {
        const int kn = min(LM_KC, words - w0);
        __syncthreads();
        for (int i = tid; i < (LM_P + LM_C) * LM_KC; i += LM_T) {
            const int r = i / LM_KC, w = i % LM_KC;
            if (w >= kn) continue;
            if (r < LM_P) S.x[r][w] = r < np ? lm_word(in, p0 + r, w0 + w) : 0u;
            else S.c[r - LM_P][w] = r - LM_P < nc ? lm_word(in, in.cid[k0 + r - LM_P], w0 + w) : 0u;
        }
        __syncthreads();
        if (l2) {
            for (int w = 0; w < kn; ++w) {
                float c[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) c[j] = __uint_as_float(S.c[tx + 16 * j][w]);
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const float x = __uint_as_float(S.x[ty + 16 * i][w]);
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const float t = x - c[j];
                        acc[i][j] = fmaf(t, t, acc[i][j]);
                    }
                }
            }
        } else {
            for (int w = 0; w < kn; ++w)
#pragma unroll
                for (int i = 0; i < 4; ++i)
#pragma unroll
                    for (int j = 0; j < 4; ++j) bits[i][j] += __popc(S.x[ty + 16 * i][w] ^ S.c[tx + 16 * j][w]);
        }
    }
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) S.d[ty + 16 * i][tx + 16 * j] = l2 ? sqrtf(acc[i][j]) : (float)bits[i][j];
    __syncthreads();
}

template <bool FILL>
__global__ void __launch_bounds__(LM_T) k_lm_cells(LmInput in, int64_t n, float eps_up, int lev_k,
                                                   int32_t *__restrict__ cell, float *__restrict__ dmin,
                                                   int32_t *__restrict__ mcount, const int64_t *__restrict__ moff,
                                                   uint64_t *__restrict__ keys) {
    static_assert(LM_T == 4 * LM_P, "four threads per point");
    __shared__ LmTile S;
    __shared__ int s_cell[LM_P];
    __shared__ float s_dmin[LM_P];
    const int tid = threadIdx.x;
    const int64_t p0 = (int64_t)blockIdx.x * LM_P;
    const int np = (int)min((int64_t)LM_P, n - p0);
    if (tid < np && FILL) {
        s_cell[tid] = cell[p0 + tid];
        s_dmin[tid] = dmin[p0 + tid];
    }
    if (!FILL) {
        int best = 0;
        float bd = 0.f;
        for (int k0 = 0; k0 < in.m; k0 += LM_C) {
            const int nc = min(LM_C, in.m - k0);
            __syncthreads();
            lm_tile(in, S, p0, np, k0, nc);
            if (tid < np) {
                for (int j = 0; j < nc; ++j) {
                    const float d = S.d[tid][j];
                    if (d < bd || k0 + j == 0) {  // the lowest index among equals
                        bd = d;
                        best = k0 + j;
                    }
                }
            }
        }
        if (tid < np) {
            cell[p0 + tid] = s_cell[tid] = best;
            dmin[p0 + tid] = s_dmin[tid] = bd;
        }
    }
    // memberships: four threads per point, 16 centres of a tile each
    const int r = tid >> 2, part = tid & 3;
    int64_t at = FILL && r < np ? moff[p0 + r] : 0;
    for (int k0 = 0; k0 < in.m; k0 += LM_C) {
        const int nc = min(LM_C, in.m - k0);
        __syncthreads();
        if (FILL || in.m > LM_C) lm_tile(in, S, p0, np, k0, nc);
        uint32_t mem = 0u;
        if (r < np) {
            const int own = s_cell[r];
            const float dm = s_dmin[r];
            for (int j = 16 * part; j < min(16 * part + 16, nc); ++j)
                if (k0 + j == own || lm_ghost(in, S.d[r][j], dm, eps_up, lev_k)) mem |= 1u << (j & 15);
        }
        const int c = __popc(mem);
        const int c1 = __shfl_up_sync(0xffffffffu, c, 1, 4), c2 = __shfl_up_sync(0xffffffffu, c, 2, 4),
                  c3 = __shfl_up_sync(0xffffffffu, c, 3, 4);
        const int before = (part > 0 ? c1 : 0) + (part > 1 ? c2 : 0) + (part > 2 ? c3 : 0);
        if (FILL) {
            for (int64_t a = at + before; mem; mem &= mem - 1u)
                keys[a++] = ((uint64_t)(k0 + 16 * part + __ffs(mem) - 1) << 32) | (uint64_t)(p0 + r);
        }
        at += __shfl_sync(0xffffffffu, before + c, 3, 4);
    }
    if (!FILL && r < np && part == 0) mcount[p0 + r] = (int32_t)at;
}

// First member of each cell in the sorted keys (k in [0, m]).
__global__ void k_lm_cell_offsets(const uint64_t *__restrict__ keys, int64_t M, int m, int64_t *__restrict__ off) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k > m) return;
    int64_t lo = 0, hi = M;
    while (lo < hi) {
        const int64_t mid = (lo + hi) >> 1;
        if ((int64_t)(keys[mid] >> 32) < k) lo = mid + 1; else hi = mid;
    }
    off[k] = lo;
}

// Rows of the members, cell by cell, in member order.
__global__ void k_lm_gather_l2(const uint64_t *__restrict__ keys, int64_t M, const float *__restrict__ X, int dim,
                               float *__restrict__ out) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= M * dim) return;
    const int64_t j = i / dim;
    const int k = (int)(i - j * dim);
    out[i] = X[(int64_t)(uint32_t)keys[j] * dim + k];
}
__global__ void k_lm_gather_bytes(const uint64_t *__restrict__ keys, int64_t M, const uint8_t *__restrict__ B, int nb,
                                  uint8_t *__restrict__ out) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= M * nb) return;
    const int64_t j = i / nb;
    const int k = (int)(i - j * nb);
    out[i] = B[(int64_t)(uint32_t)keys[j] * nb + k];
}

// Per cell: its CSR (local row offsets, columns as local member indices).
struct CellCsr {
    const int64_t *const *rp;
    const int32_t *const *col;
    const float *const *dist;
};

// Degree of each point: the length of its row in its own cell.
__global__ void k_lm_degrees(const uint64_t *__restrict__ keys, int64_t M, const int64_t *__restrict__ cell_off,
                             const int32_t *__restrict__ cell, CellCsr cc, int32_t *__restrict__ deg) {
    const int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= M) return;
    const int k = (int)(keys[j] >> 32);
    const int64_t p = (int64_t)(uint32_t)keys[j];
    if (cell[p] != k) return;  // a ghost here
    const int64_t l = j - cell_off[k];
    deg[p] = (int32_t)(cc.rp[k][l + 1] - cc.rp[k][l]);
}

// Warp per membership of an own point: its row, columns mapped to original ids.
__global__ void k_lm_fill(const uint64_t *__restrict__ keys, int64_t M, const int64_t *__restrict__ cell_off,
                          const int32_t *__restrict__ cell, CellCsr cc, const int64_t *__restrict__ row_ptr,
                          int32_t *__restrict__ col, float *__restrict__ dist) {
    const int64_t j = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (j >= M) return;
    const int k = (int)(keys[j] >> 32);
    const int64_t p = (int64_t)(uint32_t)keys[j];
    if (cell[p] != k) return;
    const int64_t l = j - cell_off[k];
    const int64_t a = cc.rp[k][l], b = cc.rp[k][l + 1], o = row_ptr[p];
    const uint64_t *mk = keys + cell_off[k];
    for (int64_t e = a + lane; e < b; e += 32) {
        col[o + (e - a)] = (int32_t)(uint32_t)mk[cc.col[k][e]];
        dist[o + (e - a)] = cc.dist[k][e];
    }
}

inline unsigned grid_of(int64_t n, int t) { return (unsigned)ceil_div(n > 0 ? n : 1, t); }

}  // namespace

void landmark_query(const ct_points *pts, const int64_t *centres_h, int m, double eps, int zeta,
                    const ct_query_opts *opts, cudaStream_t s, QueryOut &out, ct_landmark_info *info) {
    const int64_t n = pts->n;
    const bool l2 = pts->metric == CT_L2_F32;
    if (info) *info = ct_landmark_info{};
    if (n == 0) {  // the empty graph
        out.row_ptr = (int64_t *)dmalloc(sizeof(int64_t), s);
        CT_CHECK_CUDA(cudaMemsetAsync(out.row_ptr, 0, sizeof(int64_t), s));
        out.col = (int32_t *)dmalloc(sizeof(int32_t), s);
        out.dist = (float *)dmalloc(sizeof(float), s);
        out.nnz = 0;
        return;
    }
    if (!l2 && pts->metric != CT_HAMMING_B1)
        CT_FAIL(CT_EUNSUPPORTED, "the landmark form takes L2 points or Hamming rows");
    if (m < 1 || (int64_t)m > std::max<int64_t>(n, 1)) CT_FAIL(CT_EINVAL, "m must be in [1, n] (got %d)", m);
    for (int k = 0; k < m; ++k)
        if (centres_h[k] < 0 || centres_h[k] >= n) CT_FAIL(CT_EINVAL, "centre %d out of range", k);
    const int dim = pts->dim, nb = (dim + 7) / 8;
    // QParams of the metric for the ghost bound (an empty tree stands in)
    ct_tree shape;
    shape.metric = pts->metric;
    shape.dp = l2 ? (int)ceil_div(dim, 4) * 4 : 0;
    QParams qp = make_qparams(&shape, eps, opts->include_self);
    qp.half = opts->upper_triangle;
    DBuf<int64_t> cid(m, s);
    CT_CHECK_CUDA(cudaMemcpyAsync(cid.p, centres_h, (size_t)m * sizeof(int64_t), cudaMemcpyHostToDevice, s));
    const LmInput in{pts->metric, dim, l2 ? (const float *)pts->data : nullptr,
                     l2 ? nullptr : (const uint8_t *)pts->data, cid.p, m};
    // 1. Voronoi cells, 2. memberships (own cell and ghost cells), cell-major and id-minor
    DBuf<int32_t> cell(n, s), mcount(n + 1, s);
    DBuf<float> dmin(n, s);
    DBuf<int64_t> moff(n + 1, s);
    CT_CHECK_CUDA(cudaMemsetAsync(mcount.p + n, 0, sizeof(int32_t), s));
    k_lm_cells<false><<<grid_of(n, LM_P), LM_T, 0, s>>>(in, n, qp.eps_up, qp.lev_k, cell.p, dmin.p, mcount.p, nullptr,
                                                        nullptr);
    CT_COUNT_LAUNCH();
    exclusive_scan_i32_to_i64(mcount.p, moff.p, n + 1, nullptr, s);
    int64_t M = 0;
    to_host(&M, moff.p + n, 1, s);
    DBuf<uint64_t> keys(M, s), tk(M, s);
    DBuf<uint32_t> vals(M, s), tv(M, s);
    k_lm_cells<true><<<grid_of(n, LM_P), LM_T, 0, s>>>(in, n, qp.eps_up, qp.lev_k, cell.p, dmin.p, mcount.p, moff.p,
                                                       keys.p);
    CT_COUNT_LAUNCH();
    CT_CHECK_CUDA(cudaMemsetAsync(vals.p, 0, (size_t)M * sizeof(uint32_t), s));
    int bits = 32;
    while ((int64_t(1) << (bits - 32)) < m) ++bits;
    radix_sort_pairs64(keys.p, vals.p, tk.p, tv.p, M, bits, s);
    tk.reset();
    tv.reset();
    vals.reset();
    DBuf<int64_t> coff(m + 1, s);
    k_lm_cell_offsets<<<grid_of(m + 1, LM_T), LM_T, 0, s>>>(keys.p, M, m, coff.p);
    CT_COUNT_LAUNCH();
    std::vector<int64_t> hoff(m + 1);
    to_host(hoff.data(), coff.p, m + 1, s);
    // 3. member rows gathered cell by cell; a tree per cell
    DBuf<float> gx(l2 ? (size_t)M * dim : 0, s);
    DBuf<uint8_t> gb(l2 ? 0 : (size_t)M * nb, s);
    if (l2) {
        k_lm_gather_l2<<<grid_of(M * dim, LM_T), LM_T, 0, s>>>(keys.p, M, (const float *)pts->data, dim, gx.p);
    } else {
        k_lm_gather_bytes<<<grid_of(M * nb, LM_T), LM_T, 0, s>>>(keys.p, M, (const uint8_t *)pts->data, nb, gb.p);
    }
    CT_COUNT_LAUNCH();
    CT_LAUNCH_CHECK();
    struct Trees {
        std::vector<ct_tree *> t;
        ~Trees() {
            for (ct_tree *x : t) free_tree(x);
        }
    } trees;
    std::vector<QueryOut> outs((size_t)m);
    struct OutsGuard {
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
    } og{outs, s};
    int64_t largest = 0;
    {
        ProfScope ps("landmark_build", s);
        for (int k = 0; k < m; ++k) largest = std::max(largest, hoff[k + 1] - hoff[k]);
        ct_points cp{};
        cp.metric = pts->metric;
        cp.dim = dim;
        // forests of consecutive cells, within a bound on their points (scratch memory)
        constexpr int64_t kForest = 1 << 24;
        for (int k = 0; k < m;) {
            int e = k + 1;
            while (e < m && hoff[e + 1] - hoff[k] <= kForest) ++e;
            ct_points fp = cp;
            fp.n = hoff[e] - hoff[k];
            fp.data = l2 ? (const void *)(gx.p + hoff[k] * dim) : (const void *)(gb.p + hoff[k] * nb);
            std::vector<int64_t> off(hoff.begin() + k, hoff.begin() + e + 1);
            for (int64_t &o : off) o -= hoff[k];
            for (ct_tree *x : build_forest(&fp, off, zeta, s)) trees.t.push_back(x);
            k = e;
        }
    }
    std::vector<QParams> qps((size_t)m, qp);
    {
        ProfScope ps("landmark_query", s);
        query_batched(m, trees.t.data(), qps.data(), opts, s, outs.data());
    }
    // 4. rows of the own points from their cells
    DBuf<const int64_t *> prp(m, s);
    DBuf<const int32_t *> pcol(m, s);
    DBuf<const float *> pdist(m, s);
    {
        std::vector<const int64_t *> a((size_t)m);
        std::vector<const int32_t *> b((size_t)m);
        std::vector<const float *> c((size_t)m);
        for (int k = 0; k < m; ++k) {
            a[k] = outs[k].row_ptr;
            b[k] = outs[k].col;
            c[k] = outs[k].dist;
        }
        CT_CHECK_CUDA(cudaMemcpyAsync(prp.p, a.data(), (size_t)m * sizeof(void *), cudaMemcpyHostToDevice, s));
        CT_CHECK_CUDA(cudaMemcpyAsync(pcol.p, b.data(), (size_t)m * sizeof(void *), cudaMemcpyHostToDevice, s));
        CT_CHECK_CUDA(cudaMemcpyAsync(pdist.p, c.data(), (size_t)m * sizeof(void *), cudaMemcpyHostToDevice, s));
        CT_CHECK_CUDA(cudaStreamSynchronize(s));  // the host arrays above are on the stack
    }
    const CellCsr cc{prp.p, pcol.p, pdist.p};
    DBuf<int32_t> deg(n + 1, s);
    CT_CHECK_CUDA(cudaMemsetAsync(deg.p, 0, (size_t)(n + 1) * sizeof(int32_t), s));
    k_lm_degrees<<<grid_of(M, LM_T), LM_T, 0, s>>>(keys.p, M, coff.p, cell.p, cc, deg.p);
    CT_COUNT_LAUNCH();
    out.row_ptr = (int64_t *)dmalloc((size_t)(n + 1) * sizeof(int64_t), s);
    exclusive_scan_i32_to_i64(deg.p, out.row_ptr, n + 1, nullptr, s);
    int64_t nnz = 0;
    to_host(&nnz, out.row_ptr + n, 1, s);
    out.nnz = nnz;
    out.col = (int32_t *)dmalloc((size_t)(nnz ? nnz : 1) * sizeof(int32_t), s);
    out.dist = (float *)dmalloc((size_t)(nnz ? nnz : 1) * sizeof(float), s);
    k_lm_fill<<<grid_of(M * 32, LM_T), LM_T, 0, s>>>(keys.p, M, coff.p, cell.p, cc, out.row_ptr, out.col, out.dist);
    CT_COUNT_LAUNCH();
    CT_LAUNCH_CHECK();
    CT_CHECK_CUDA(cudaStreamSynchronize(s));
    prof_flush();
    out.stats = ct_query_stats{};
    // the batches' counters (every CSR of an L2 batch carries that batch's;
    // Hamming cells are queried one at a time)
    for (int k = 0; k < m; k += l2 ? kBatchClouds : 1) {
        const ct_query_stats &b = outs[k].stats;
        out.stats.traversal_evals += b.traversal_evals;
        out.stats.leaf_pairs += b.leaf_pairs;
        out.stats.guard_fp64 += b.guard_fp64;
        out.stats.recheck_fp32 += b.recheck_fp32;
        out.stats.candidates += b.candidates;
        out.stats.leaf_rows += b.leaf_rows;
        out.stats.guard_band += b.guard_band;
    }
    if (info) {
        info->members = M;
        info->ghosts = M - n;
        info->largest_cell = largest;
        info->cells = m;
    }
}

}  // namespace ct

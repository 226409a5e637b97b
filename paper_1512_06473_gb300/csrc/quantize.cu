// quantize.cu -- learning the PQ parameters: k-means in every sub-space
// (Sec. 3.1, Eq. 4 for FC weights; Sec. 3.2, Eq. 6 for conv kernels).
//
// For sub-space m the points are the m-th sub-vectors of all weight vectors
// (FC: one per c_t; conv: one per (c_t, p_k), index p = c_t * kh*kw + p_k).
// All M sub-spaces run at once.  One Lloyd round is two launches:
//   1. assign: every point to its nearest centroid.  Squared distances are
//      evaluated term by term in binary32 (subtract, square, add, each
//      rounded, no fused multiply-add), ties to the smallest index -- the
//      integer decision is taken in one stated precision, so it can be
//      checked bit for bit.
//   2. update: one thread per (m, k, j) sums its cluster's coordinates in
//      double in index order, divides by the count and rounds to binary32;
//      a cluster without points keeps its centroid.  The fixed order makes
//      the centroids reproducible bit for bit.
// After `iters` rounds a last assignment writes the codes in the layer's
// layout.  Points are padded to CSP4 = 4 or 8 coordinates with zeros, which
// adds exact zeros to the distances.
#include "qcnn_internal.cuh"

#include <algorithm>
#include <climits>

namespace qcnn {

constexpr int kSortThreads = 1024;

// points[m][p][0..CSP4) from W viewed as [Ct][Cs][kk] (kk = 1 for FC).
__global__ void pq_points_kernel(const float *__restrict__ W, int Ct, int Cs, int kk, int Csp,
                                 int csp4, int M, float *__restrict__ pts) {
    const long long P = (long long)Ct * kk;
    const long long total = (long long)M * P * csp4;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < total;
         i += (long long)gridDim.x * blockDim.x) {
        const int j = (int)(i % csp4);
        const long long r = i / csp4;
        const long long p = r % P;
        const int m = (int)(r / P);
        const long long ct = p / kk, pk = p % kk;
        pts[i] = j < Csp ? W[(ct * Cs + (long long)m * Csp + j) * kk + pk] : 0.f;
    }
}

// cen[m][k][0..CSP4) from a dense [M][K][Csp] array (zero padding), or back.
__global__ void pad_centroids_kernel(const float *__restrict__ in, int M, int K, int Csp,
                                     int csp4, float *__restrict__ out, int to_padded) {
    const int total = M * K * csp4;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < total; i += gridDim.x * blockDim.x) {
        const int j = i % csp4, mk = i / csp4;
        if (to_padded)
            out[i] = j < Csp ? in[mk * Csp + j] : 0.f;
        else if (j < Csp)
            out[mk * Csp + j] = in[i];
    }
}

// Nearest centroid of every point of sub-space blockIdx.y.  assign[m][p];
// codes (if given) at codes[m * code_sm + p * code_sp].
// Bound by the instructions of a distance and its comparison (a pair of point
// and centroid is 8 CSP4 / 4 + 3 + CSP4 / 4 of them one at a time) and by their
// latency.  So a thread has two points, side by side in the packed binary32
// operations (each half rounded as on its own; a coordinate is in shared memory
// twice, negated: x + -c is x - c), four centroids at a time, and the CTA's
// upper half takes the upper half of the centroids.  64 sub-spaces of 3,456
// points, 128 centroids: 19.8 us with a point a thread, 17.2 with two, 15.8
// with the centroids in halves.  (Comparing four distances' minimum instead, and
// finding the index at the end, was slower: 22.)
template <int CSP4>
__global__ void __launch_bounds__(256) kmeans_assign_kernel(const float *__restrict__ pts, int P,
                                                            int K, const float *cen,
                                                            uint8_t *__restrict__ assign,
                                                            uint8_t *__restrict__ codes,
                                                            long long code_sm, long long code_sp) {
    __shared__ __align__(16) float2 cs[kMaxK * CSP4];
    __shared__ float2 upper_d[128];
    __shared__ int2 upper_k[128];
    const int m = blockIdx.y, t = threadIdx.x & 127;
    const bool upper = threadIdx.x >= 128;
    const int p0 = blockIdx.x * 256 + t;
    for (int e = threadIdx.x; e < K * CSP4; e += 256) {
        const float c = -cen[(size_t)m * K * CSP4 + e];
        cs[e] = make_float2(c, c);
    }
    float2 x[CSP4];
    const float4 *xp = reinterpret_cast<const float4 *>(pts + (size_t)m * P * CSP4);
#pragma unroll
    for (int q = 0; q < CSP4 / 4; ++q) {
        const float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
        const float4 u = p0 < P ? xp[(size_t)p0 * (CSP4 / 4) + q] : z;
        const float4 v = p0 + 128 < P ? xp[(size_t)(p0 + 128) * (CSP4 / 4) + q] : z;
        x[4 * q] = make_float2(u.x, v.x);
        x[4 * q + 1] = make_float2(u.y, v.y);
        x[4 * q + 2] = make_float2(u.z, v.z);
        x[4 * q + 3] = make_float2(u.w, v.w);
    }
    __syncthreads();
    auto dist = [&](int k) {
        const float4 *c = reinterpret_cast<const float4 *>(cs + k * CSP4);
        float2 d;
#pragma unroll
        for (int j = 0; j < CSP4; j += 2) {
            const float4 cc = c[j / 2];
            const float2 e = __fadd2_rn(x[j], make_float2(cc.x, cc.y));
            const float2 f = __fadd2_rn(x[j + 1], make_float2(cc.z, cc.w));
            // (0 + a square is the square)
            d = j ? __fadd2_rn(d, __fmul2_rn(e, e)) : __fmul2_rn(e, e);
            d = __fadd2_rn(d, __fmul2_rn(f, f));
        }
        return d;
    };
    const int half = (K + 1) / 2, k1 = upper ? K : half;
    int k = upper ? half : 0;
    // (the first centroid stands even at a distance that is no number; the upper
    // half has to be nearer than what it has not seen)
    int best0 = k, best1 = k;
    float2 best_d = make_float2(INFINITY, INFINITY);
    if (!upper) best_d = dist(k++);
    auto take = [&](int k, const float2 &d) {
        const bool l0 = d.x < best_d.x, l1 = d.y < best_d.y;
        best_d.x = l0 ? d.x : best_d.x;
        best0 = l0 ? k : best0;
        best_d.y = l1 ? d.y : best_d.y;
        best1 = l1 ? k : best1;
    };
    for (; k + 4 <= k1; k += 4) {
        float2 d[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) d[i] = dist(k + i);
#pragma unroll
        for (int i = 0; i < 4; ++i) take(k + i, d[i]);
    }
    for (; k < k1; ++k) take(k, dist(k));
    if (upper) {
        upper_d[t] = best_d;
        upper_k[t] = make_int2(best0, best1);
    }
    __syncthreads();
    if (upper || p0 >= P) return;
    const float2 ud = upper_d[t];
    const int2 uk = upper_k[t];
    if (ud.x < best_d.x) best0 = uk.x;
    if (ud.y < best_d.y) best1 = uk.y;
    assign[(size_t)m * P + p0] = (uint8_t)best0;
    if (codes) codes[(size_t)m * code_sm + (size_t)p0 * code_sp] = (uint8_t)best0;
    if (p0 + 128 < P) {
        assign[(size_t)m * P + p0 + 128] = (uint8_t)best1;
        if (codes) codes[(size_t)m * code_sm + (size_t)(p0 + 128) * code_sp] = (uint8_t)best1;
    }
}

// One CTA per label array: order[m][*] = its point indices grouped
// by cluster, index order inside a cluster; starts[m][k] = first slot of
// cluster k (starts[m][K] = P).
__global__ void __launch_bounds__(kSortThreads) kmeans_order_kernel(
    const uint8_t *__restrict__ assign, int P, int K, int *__restrict__ order,
    int *__restrict__ starts) {
    constexpr int NW = kSortThreads / 32;
    __shared__ int wcount[NW][kMaxK];  // per-warp counts of one round, then offsets
    __shared__ int base[kMaxK + 1];    // running start of each cluster
    const int m = blockIdx.x;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint8_t *a = assign + (size_t)m * P;
    // cluster sizes -> exclusive starts
    for (int k = tid; k <= K; k += kSortThreads) base[k] = 0;
    __syncthreads();
    for (int p = tid; p < P; p += kSortThreads) atomicAdd(&base[a[p] + 1], 1);
    __syncthreads();
    if (tid == 0)
        for (int k = 1; k <= K; ++k) base[k] += base[k - 1];
    __syncthreads();
    for (int k = tid; k <= K; k += kSortThreads) starts[(size_t)m * (K + 1) + k] = base[k];
    // stable scatter, kSortThreads points per round
    for (int p0 = 0; p0 < P; p0 += kSortThreads) {
        for (int e = tid; e < NW * K; e += kSortThreads) wcount[e / K][e % K] = 0;
        __syncthreads();
        const int p = p0 + tid;
        const int k = p < P ? a[p] : -1;
        const unsigned same = __match_any_sync(0xffffffffu, k);
        const int rank = __popc(same & ((1u << lane) - 1u));
        if (k >= 0 && rank == 0) wcount[warp][k] = __popc(same);
        __syncthreads();
        for (int c = tid; c < K; c += kSortThreads) {  // offsets over the warps, in order
            int run = base[c];
            for (int w = 0; w < NW; ++w) {
                const int v = wcount[w][c];
                wcount[w][c] = run;
                run += v;
            }
            base[c] = run;
        }
        __syncthreads();
        if (k >= 0) order[(size_t)m * P + wcount[warp][k] + rank] = p;
        __syncthreads();
    }
}

// A float's value in double, by integer operations where it is a normal number
// or zero: the conversion instruction shares the double units.
__device__ __forceinline__ double widen(float f) {
    const unsigned b = __float_as_uint(f), t = b & 0x7fffffffu;
    if (t != 0u && t - 0x00800000u >= 0x7f000000u) return (double)f;
    const unsigned hi = t ? (t >> 3) + 0x38000000u : 0u;
    return __hiloint2double((int)((b & 0x80000000u) | hi), (int)(b << 29));
}

// The means of clusters 8 blockIdx.x .. + 7 of sub-space blockIdx.y, summed in
// double in point-index order; unchanged when a cluster is empty.  Of
// kUpdateLabels labels at a time a thread looks at 16 in a row, and the CTA
// lists those of its eight clusters; a warp per cluster lists its own of these;
// then a lane per cluster and coordinate adds up its list, all in index order.
// The double units do two lanes a clock, whatever lanes of a warp are in use:
// one warp per cluster with four lanes adding took 47 us for 64 sub-spaces of
// 3,456 points and 128 clusters, this 18.6.  (Before: a counting sort by one CTA
// per sub-space, 13 us, then a thread per coordinate that waited for each point
// in turn, 17 us.)
constexpr int kUpdateClusters = 8, kUpdateLabels = 4096;

template <int CSP4>
__global__ void __launch_bounds__(kUpdateClusters * 32) kmeans_update_kernel(
    const float *__restrict__ pts, int P, int K, int Csp, const uint8_t *assign, float *cen) {
    static_assert(kUpdateClusters * 32 * 16 == kUpdateLabels, "16 labels a thread");
    __shared__ unsigned short cand[kUpdateLabels];  // labels of these clusters,
    __shared__ uint8_t cand_k[kUpdateLabels];       // and which of the eight
    __shared__ unsigned short list[kUpdateLabels];
    __shared__ int sizes[kUpdateClusters], warp_cand[kUpdateClusters];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int m = blockIdx.y, k0 = blockIdx.x * kUpdateClusters;
    // this thread's cluster and coordinate when adding (the first warps)
    const int wk = tid / CSP4, wj = tid % CSP4;
    const uint8_t *a = assign + (size_t)m * P;
    const bool vec = reinterpret_cast<uintptr_t>(a) % 16 == 0;
    const float *pm = pts + (size_t)m * P * CSP4 + wj;
    const unsigned key = (unsigned)k0 * 0x01010101u;
    double s = 0.0;
    int count = 0;
    for (int p0 = 0; p0 < P; p0 += kUpdateLabels) {
        const int here = min(kUpdateLabels, P - p0);
        unsigned w[4] = {0u, 0u, 0u, 0u};
        const int left = here - tid * 16;
        if (vec && left >= 16) {
            const uint4 v = *reinterpret_cast<const uint4 *>(a + p0 + tid * 16);
            w[0] = v.x, w[1] = v.y, w[2] = v.z, w[3] = v.w;
        } else {
#pragma unroll
            for (int i = 0; i < 16; ++i)
                if (i < left) w[i / 4] |= (unsigned)a[p0 + tid * 16 + i] << (i % 4 * 8);
        }
        unsigned hit = 0;  // which of them are of these eight clusters
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            // (a byte of x is zero where the label is; its bit 7, then, of z)
            const unsigned x = (w[i] & 0xf8f8f8f8u) ^ key;
            const unsigned z = ~(((x & 0x7f7f7f7fu) + 0x7f7f7f7fu) | x | 0x7f7f7f7fu) >> 7;
            hit |= ((z | z >> 7 | z >> 14 | z >> 21) & 15u) << (i * 4);
        }
        if (left < 16) hit &= left > 0 ? (1u << left) - 1u : 0u;
        const int mine = __popc(hit);
        int upto = mine;  // of this lane and those below
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int v = __shfl_up_sync(0xffffffffu, upto, o);
            if (lane >= o) upto += v;
        }
        if (lane == 31) warp_cand[warp] = upto;
        __syncthreads();
        int at = upto - mine, all = 0;
        for (int v = 0; v < kUpdateClusters; ++v) {
            if (v < warp) at += warp_cand[v];
            all += warp_cand[v];
        }
        for (unsigned h = hit; h; h &= h - 1, ++at) {
            const int i = __ffs((int)h) - 1;
            const unsigned word = i < 8 ? (i < 4 ? w[0] : w[1]) : (i < 12 ? w[2] : w[3]);
            cand[at] = (unsigned short)(tid * 16 + i);
            cand_k[at] = (uint8_t)(word >> (i % 4 * 8) & 7u);
        }
        __syncthreads();
        // the warp's own: counted, then listed behind the warps' before
        int n = 0;
        for (int c = lane; c < all; c += 32) n += cand_k[c] == warp;
        n = __reduce_add_sync(0xffffffffu, n);
        if (lane == 0) sizes[warp] = n;
        __syncthreads();
        int to = 0;
        for (int v = 0; v < warp; ++v) to += sizes[v];
        for (int c0 = 0; c0 < all; c0 += 32) {
            const int c = c0 + lane;
            const bool is = c < all && cand_k[c] == warp;
            const unsigned vote = __ballot_sync(0xffffffffu, is);
            if (is) list[to + __popc(vote & ((1u << lane) - 1u))] = cand[c];
            to += __popc(vote);
        }
        __syncthreads();
        if (wk < kUpdateClusters && wj < Csp) {
            int i = 0;
            for (int v = 0; v < wk; ++v) i += sizes[v];
            const int end = i + sizes[wk];
            count += sizes[wk];
            const float *src = pm + (size_t)p0 * CSP4;
            for (; i < end; i += 8) {
                float v[8];
#pragma unroll
                for (int e = 0; e < 8; ++e) v[e] = i + e < end ? src[list[i + e] * CSP4] : 0.f;
#pragma unroll
                for (int e = 0; e < 8; ++e)
                    if (i + e < end) s += widen(v[e]);
            }
        }
        __syncthreads();
    }
    const int k = k0 + wk;
    if (wk < kUpdateClusters && k < K && wj < Csp && count > 0)
        cen[((size_t)m * K + k) * CSP4 + wj] = __double2float_rn(s / (double)count);
}

// ------------------------------------------------------------------ host --
struct KmeansWs {
    size_t pts, cen, assign, total;
};

KmeansWs kmeans_ws_layout(int M, long long P, int Csp, int K, bool with_points) {
    const int csp4 = Csp <= 4 ? 4 : 8;
    KmeansWs w;
    size_t off = 0;
    w.pts = off;
    if (with_points) off += align_up((size_t)M * P * csp4 * sizeof(float), kWsAlign);
    w.cen = off;
    off += align_up((size_t)M * K * csp4 * sizeof(float), kWsAlign);
    w.assign = off;
    off += align_up((size_t)M * P, kWsAlign);
    w.total = off;
    return w;
}

qcnn_status run_kmeans(const float *pts, int M, int P, int Csp, int K, const float *init,
                       int iters, float *D, uint8_t *codes, long long code_sm,
                       long long code_sp, void *ws, const KmeansWs &L, cudaStream_t st) {
    const int csp4 = Csp <= 4 ? 4 : 8;
    uint8_t *base = static_cast<uint8_t *>(ws);
    float *cen = reinterpret_cast<float *>(base + L.cen);
    uint8_t *assign = base + L.assign;
    const int sms = num_sms();
    const int cen_blocks = std::max(1, std::min(cdiv(M * K * csp4, 256), sms * 8));
    pad_centroids_kernel<<<cen_blocks, 256, 0, st>>>(init, M, K, Csp, csp4, cen, 1);
    qcnn_status rc = after_launch();
    if (rc != QCNN_OK) return rc;
    const dim3 agrid(cdiv(P, 256), M), ugrid(cdiv(K, kUpdateClusters), M);
    const auto assign_k = csp4 == 4 ? kmeans_assign_kernel<4> : kmeans_assign_kernel<8>;
    const auto update_k = csp4 == 4 ? kmeans_update_kernel<4> : kmeans_update_kernel<8>;
    // (plain launches: as programmatic ones ten rounds took 507 us, so 390)
    for (int it = 0; it <= iters; ++it) {
        const bool last = it == iters;
        assign_k<<<agrid, 256, 0, st>>>(pts, P, K, cen, assign, last ? codes : nullptr, code_sm,
                                        code_sp);
        if ((rc = after_launch()) != QCNN_OK) return rc;
        if (last) break;
        update_k<<<ugrid, kUpdateClusters * 32, 0, st>>>(pts, P, K, Csp, assign, cen);
        if ((rc = after_launch()) != QCNN_OK) return rc;
    }
    pad_centroids_kernel<<<cen_blocks, 256, 0, st>>>(cen, M, K, Csp, csp4, D, 0);
    return after_launch();
}

}  // namespace qcnn

using namespace qcnn;

namespace {

bool kmeans_args_ok(int M, long long P, int Csp, int K, int iters) {
    return M > 0 && P > 0 && Csp >= 1 && Csp <= kMaxCsp && K >= 1 && K <= kMaxK &&
           iters >= 0 && (long long)M * P * 8 < (long long)INT_MAX &&
           (long long)M * K * 8 < (long long)INT_MAX;
}

}  // namespace

extern "C" {

qcnn_status qcnn_kmeans_workspace_size(int M, int P, int Csp, int K, size_t *bytes) {
    if (!bytes || !kmeans_args_ok(M, P, Csp, K, 0)) return QCNN_ERR_INVALID_ARG;
    *bytes = kmeans_ws_layout(M, P, Csp, K, true).total;
    return QCNN_OK;
}

qcnn_status qcnn_kmeans(const float *points, int M, int P, int Csp, int K, const float *init,
                        int iters, float *D, uint8_t *assign, void *workspace,
                        size_t workspace_bytes, void *stream) {
    if (!points || !init || !D || !assign || !kmeans_args_ok(M, P, Csp, K, iters))
        return QCNN_ERR_INVALID_ARG;
    const KmeansWs L = kmeans_ws_layout(M, P, Csp, K, true);
    if (!workspace || workspace_bytes < L.total ||
        reinterpret_cast<uintptr_t>(workspace) % kWsAlign != 0)
        return QCNN_ERR_WORKSPACE;
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    const int csp4 = Csp <= 4 ? 4 : 8;
    float *pts = reinterpret_cast<float *>(static_cast<uint8_t *>(workspace) + L.pts);
    // points [M][P][Csp] -> zero-padded [M][P][csp4] (same pass as for centroids)
    const long long total = (long long)M * P * csp4;
    const int blocks = (int)std::min<long long>((total + 255) / 256, (long long)num_sms() * 16);
    pad_centroids_kernel<<<blocks, 256, 0, st>>>(points, M, P, Csp, csp4, pts, 1);
    qcnn_status rc = after_launch();
    if (rc != QCNN_OK) return rc;
    return run_kmeans(pts, M, P, Csp, K, init, iters, D, assign, P, 1, workspace, L, st);
}

qcnn_status qcnn_pq_quantize_workspace_size(int kind, int Ct, int Cs, int kh, int kw, int Csp,
                                            int K, size_t *bytes) {
    if (!bytes || Ct <= 0 || Cs <= 0 || Csp < 1 || Cs % Csp != 0) return QCNN_ERR_INVALID_ARG;
    if (kind == QCNN_LAYER_FC) kh = kw = 1;
    else if (kind != QCNN_LAYER_CONV || kh <= 0 || kw <= 0) return QCNN_ERR_INVALID_ARG;
    const long long P = (long long)Ct * kh * kw;
    if (P >= INT_MAX || !kmeans_args_ok(Cs / Csp, P, Csp, K, 0)) return QCNN_ERR_INVALID_ARG;
    *bytes = kmeans_ws_layout(Cs / Csp, P, Csp, K, true).total;
    return QCNN_OK;
}

qcnn_status qcnn_pq_quantize(int kind, const float *W, int Ct, int Cs, int kh, int kw, int Csp,
                             int K, const float *init, int iters, float *D, uint8_t *codes,
                             void *workspace, size_t workspace_bytes, void *stream) {
    size_t need = 0;
    qcnn_status rc = qcnn_pq_quantize_workspace_size(kind, Ct, Cs, kh, kw, Csp, K, &need);
    if (rc != QCNN_OK) return rc;
    if (!W || !init || !D || !codes || iters < 0) return QCNN_ERR_INVALID_ARG;
    if (!workspace || workspace_bytes < need ||
        reinterpret_cast<uintptr_t>(workspace) % kWsAlign != 0)
        return QCNN_ERR_WORKSPACE;
    if (kind == QCNN_LAYER_FC) kh = kw = 1;
    const int M = Cs / Csp, kk = kh * kw, csp4 = Csp <= 4 ? 4 : 8;
    const int P = Ct * kk;
    const KmeansWs L = kmeans_ws_layout(M, P, Csp, K, true);
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    float *pts = reinterpret_cast<float *>(static_cast<uint8_t *>(workspace) + L.pts);
    const long long total = (long long)M * P * csp4;
    const int blocks = (int)std::min<long long>((total + 255) / 256, (long long)num_sms() * 16);
    pq_points_kernel<<<blocks, 256, 0, st>>>(W, Ct, Cs, kk, Csp, csp4, M, pts);
    rc = after_launch();
    if (rc != QCNN_OK) return rc;
    // codes: FC [M][Ct] (m stride P, p stride 1); conv [Ct][kk][M] (m stride 1, p stride M)
    const long long sm = kind == QCNN_LAYER_FC ? P : 1, sp = kind == QCNN_LAYER_FC ? 1 : M;
    return run_kmeans(pts, M, P, Csp, K, init, iters, D, codes, sm, sp, workspace, L, st);
}

}  // extern "C"

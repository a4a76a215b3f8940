// Freivalds integrity check of the server's answer (Sec. 3.2 box, Init W
// step 4 and Online step 4; appendix "Computational integrity"):
//   setup:  Ychk = a W'            (k check vectors, one-time per matrix)
//   online: a^T Y' == Ychk X'      per token, over Z_{2^32}
// The online check streams Z and X' once, in one launch for up to about 1200
// tokens and as two streaming ring products and a comparison beyond; the
// setup's column sums run here too.
#include <cooperative_groups.h>

#include "mosaic_internal.cuh"

namespace cg = cooperative_groups;

namespace mosaic {
namespace {

constexpr int kMaxK = 16;

// Y[v][c] += sum_{i in [i0, i1)} a[v][i] W[i][c] for one column c per thread
// (a warp reads 32 consecutive words of a row of W; a[v][i] is the same for
// the whole warp).  Partial sums of the row chunks meet with atomic adds,
// which wrap mod 2^32 like the sums themselves.
__global__ void colsum_kernel(const uint32_t *a, int k, const uint32_t *W, int64_t ldw, int64_t m,
                              int64_t ncols, int64_t rows_per_block, uint32_t *Y) {
    const int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t i0 = (int64_t)blockIdx.y * rows_per_block;
    const int64_t i1 = i0 + rows_per_block < m ? i0 + rows_per_block : m;
    if (c >= ncols) return;
    uint32_t acc[kMaxK];
#pragma unroll
    for (int v = 0; v < kMaxK; v++) acc[v] = 0u;
    for (int64_t i = i0; i < i1; i++) {
        const uint32_t w = W[i * ldw + c];
#pragma unroll
        for (int v = 0; v < kMaxK; v++)
            if (v < k) acc[v] += __ldg(a + (int64_t)v * m + i) * w;
    }
#pragma unroll
    for (int v = 0; v < kMaxK; v++)
        if (v < k) atomicAdd(Y + (int64_t)v * ncols + c, acc[v]);
}

// acc[v][t] += (or -=) sum_{c in [c0, c1)} A[v][c] B[t][c] over this block's
// threads (A: k rows with leading dimension lda, B: T token rows with leading
// dimension ldb, `tn` of them in range).
template <int KV, int T, bool MINUS>
__device__ __forceinline__ void dot_rows(uint32_t (&acc)[KV][T], const uint32_t *A, int64_t lda, int k,
                                         const uint32_t *B, int64_t ldb, int tn, int64_t c0, int64_t c1, bool vec) {
    auto mac = [&](int v, int t, uint32_t x, uint32_t y) {
        if (MINUS) acc[v][t] -= x * y;
        else acc[v][t] += x * y;
    };
    // From 8 vectors on, the loads of four rows of A are in flight at once: one
    // after another, their latencies made up most of a share.
    constexpr int G = KV >= 8 ? 4 : 1;
    int64_t c = c0;
    if (vec) {   // 16-byte loads; c0 is a multiple of 4
        const int64_t quads = (c1 - c0) >> 2;
#pragma unroll 2
        for (int64_t i = threadIdx.x; i < quads; i += blockDim.x) {
            uint4 x[T];
#pragma unroll
            for (int t = 0; t < T; t++)
                x[t] = t < tn ? __ldcg(reinterpret_cast<const uint4 *>(B + t * ldb + c0) + i) : make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
            for (int v0 = 0; v0 < KV; v0 += G) {
                if (v0 >= k) break;
                uint4 y[G];
#pragma unroll
                for (int g = 0; g < G; g++)
                    y[g] = G == 1 || v0 + g < k ? __ldca(reinterpret_cast<const uint4 *>(A + (v0 + g) * lda + c0) + i)
                                                : make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
                for (int g = 0; g < G; g++)
#pragma unroll
                    for (int t = 0; t < T; t++) {
                        mac(v0 + g, t, y[g].x, x[t].x);
                        mac(v0 + g, t, y[g].y, x[t].y);
                        mac(v0 + g, t, y[g].z, x[t].z);
                        mac(v0 + g, t, y[g].w, x[t].w);
                    }
            }
        }
        c = c0 + 4 * quads;
    }
    for (int64_t i = c + threadIdx.x; i < c1; i += blockDim.x) {
        uint32_t x[T];
#pragma unroll
        for (int t = 0; t < T; t++) x[t] = t < tn ? __ldcg(B + t * ldb + i) : 0u;
#pragma unroll
        for (int v0 = 0; v0 < KV; v0 += G) {
            if (v0 >= k) break;
            uint32_t y[G];
#pragma unroll
            for (int g = 0; g < G; g++) y[g] = G == 1 || v0 + g < k ? __ldca(A + (v0 + g) * lda + i) : 0u;
#pragma unroll
            for (int g = 0; g < G; g++)
#pragma unroll
                for (int t = 0; t < T; t++) mac(v0 + g, t, y[g], x[t]);
        }
    }
}

// The whole online check in one launch: a cluster of `S` blocks takes T
// tokens, block s of it the s-th share of the columns of Z and of X'; each
// thread keeps the k x T differences a Y' - Ychk X' of its columns, summed by
// warp reductions, in shared memory across warps and through the cluster's
// shared memory across blocks, and the first block counts the vectors that
// differ from zero.  Bound by reading Z and X' once (HBM) and a and Ychk once
// per cluster (L2).  T = 4 tokens share each read of a and Ychk; the cluster
// splits the columns where the tokens alone would leave SMs idle.  512 tokens,
// m = n_pad = 8192, k = 4: 10.2 us (3.3 TB/s of Z and X'); two streaming ring
// products on 18 blocks each and a comparison took 18.1 + 17.9 + 2.0 us.
constexpr int kChkThreads = 256;
template <int KV, int T>
__global__ void __launch_bounds__(kChkThreads, KV >= 8 && T > 1 ? 2 : 4)
    check_kernel(int k, const uint32_t *a, const uint32_t *Ychk, int64_t m, int64_t n_pad, int64_t l,
                 const uint32_t *Z, int64_t ldz, const uint32_t *Xp, int64_t ldx, uint32_t *bad, uint32_t *n_bad,
                 int vec_z, int vec_x) {
    pdl_enter();
    __shared__ uint32_t part[kChkThreads / 32][KV * T];
    __shared__ uint32_t sums[KV * T];
    cg::cluster_group cluster = cg::this_cluster();
    const int S = (int)cluster.num_blocks(), s = (int)cluster.block_rank();
    const int64_t j0 = (int64_t)(blockIdx.x / S) * T;
    const int tn = l - j0 < T ? (int)(l - j0) : T;
    uint32_t acc[KV][T];
#pragma unroll
    for (int v = 0; v < KV; v++)
#pragma unroll
        for (int t = 0; t < T; t++) acc[v][t] = 0u;
    auto share = [&](int64_t cols, int i) {   // start of share i: a multiple of 4 columns
        const int64_t c = (cols * i / S + 3) & ~(int64_t)3;
        return c < cols ? c : cols;
    };
    dot_rows<KV, T, false>(acc, a, m, k, Z + j0 * ldz, ldz, tn, share(m, s), share(m, s + 1), vec_z != 0);
    dot_rows<KV, T, true>(acc, Ychk, n_pad, k, Xp + j0 * ldx, ldx, tn, share(n_pad, s), share(n_pad, s + 1),
                          vec_x != 0);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
#pragma unroll
    for (int v = 0; v < KV; v++)
#pragma unroll
        for (int t = 0; t < T; t++) {
            const uint32_t w = __reduce_add_sync(0xffffffffu, acc[v][t]);
            if (lane == 0) part[warp][v * T + t] = w;
        }
    __syncthreads();
    for (int i = threadIdx.x; i < KV * T; i += kChkThreads) {
        uint32_t w = 0u;
#pragma unroll
        for (int q = 0; q < kChkThreads / 32; q++) w += part[q][i];
        sums[i] = w;
    }
    cluster.sync();   // every block's sums are in place
    if (s == 0 && threadIdx.x < tn) {
        uint32_t b = 0u;
        for (int v = 0; v < k; v++) {
            uint32_t w = 0u;
            for (int q = 0; q < S; q++) w += cluster.map_shared_rank(sums, q)[v * T + threadIdx.x];
            b += w != 0u ? 1u : 0u;
        }
        bad[j0 + threadIdx.x] = b;
        if (b) atomicAdd(n_bad, 1u);
    }
    cluster.sync();   // the first block has read the others' shared memory
}

__global__ void compare_kernel(const uint32_t *lhs, const uint32_t *rhs, int k, int64_t l, uint32_t *bad,
                               uint32_t *n_bad) {
    const int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= l) return;
    uint32_t b = 0u;
    for (int v = 0; v < k; v++) b += lhs[(int64_t)v * l + j] != rhs[(int64_t)v * l + j] ? 1u : 0u;
    bad[j] = b;
    if (b) atomicAdd(n_bad, 1u);
}

// Clusters of S = 2^s blocks of check_kernel<KV, T> that are resident at once on
// device `dev`, looked up once (0 on failure).
template <int KV, int T>
int check_resident(int dev, int s) {
    static std::atomic<int> cache[64][4];
    std::atomic<int> &at = cache[dev & 63][s];
    int n = at.load(std::memory_order_relaxed);
    if (n > 0) return n;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(1u << s);
    cfg.blockDim = dim3(kChkThreads);
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = 1u << s;
    attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    if (cudaOccupancyMaxActiveClusters(&n, check_kernel<KV, T>, &cfg) != cudaSuccess) return 0;
    at.store(n, std::memory_order_relaxed);
    return n;
}

// The check by one launch of token clusters, or, where their blocks no longer
// fit on the device at once, by two streaming products (k x l words each in
// lhs and rhs) and a comparison: every further wave of clusters reads a and
// Ychk again and leaves no other warps to hide its latencies behind, while the
// streaming kernel takes 60 tokens a CTA.  From 8 vectors a second wave still
// pays where the columns are many.  Inside a CUDA graph, microseconds, clusters
// / products, by k vectors, l tokens and m = n_pad:
//   m        4, 2048     4, 4096     8, 1024     8, 2048     8, 4096    16, 4096
//   64      5.1 /  4.8  9.7 /  5.0  5.0 /  5.7   10 /  5.8       -           -
//   1024    7.0 /  8.7   12 /  8.7  5.9 / 11.7   11 / 11.8   22 / 11.7       -
//   8192     37 / 38.7   74 / 50.6   19 / 56.5   43 / 58.3   88 / 58.1  151 / 96.9
template <int KV, int T>
mosaic_status launch_check(int k, const uint32_t *a, const uint32_t *Ychk, int64_t m, int64_t n_pad, int64_t l,
                           const uint32_t *Z, int64_t ldz, const uint32_t *Xp, int64_t ldx, uint32_t *bad,
                           uint32_t *n_bad, uint32_t *lhs, uint32_t *rhs, cudaStream_t st) {
    const int64_t groups = (l + T - 1) / T;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || check_resident<KV, T>(dev, 0) < 1) return MOSAIC_ERR_CUDA;
    const int64_t one = check_resident<KV, T>(dev, 0), waves = (groups + one - 1) / one;
    if (waves > (KV >= 8 && m + n_pad >= 2048 ? 2 : 1) && skinny_ok(a, m, Z, ldz, k, m) &&
        skinny_ok(Ychk, n_pad, Xp, ldx, k, n_pad)) {
        MOSAIC_TRY(ring_gemm_skinny(a, m, Z, ldz, lhs, l, nullptr, 0, 1, k, l, m, st));
        MOSAIC_TRY(ring_gemm_skinny(Ychk, n_pad, Xp, ldx, rhs, l, nullptr, 0, 1, k, l, n_pad, st));
        {
            KernelSpan span("freivalds_compare", st);
            compare_kernel<<<(unsigned)((l + 255) / 256), 256, 0, st>>>(lhs, rhs, k, l, bad, n_bad);
        }
        return launch_status();
    }
    // The columns are split over as many blocks as are all resident at once and
    // have a quad of columns for every thread.
    int s = 0;
    while (s < 3 && m + n_pad >= ((int64_t)2048 << s) && groups <= check_resident<KV, T>(dev, s + 1)) ++s;
    const int S = 1 << s;
    if (groups * S > 0x7fffffff) return MOSAIC_ERR_SHAPE;
    const int vec_z = aligned16(a) && aligned16(Z) && m % 4 == 0 && ldz % 4 == 0;
    const int vec_x = aligned16(Ychk) && aligned16(Xp) && n_pad % 4 == 0 && ldx % 4 == 0;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(groups * S));
    cfg.blockDim = dim3(kChkThreads);
    cfg.stream = st;
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)S;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 2;
    {
        KernelSpan span("freivalds_check", st);
        if (cudaLaunchKernelEx(&cfg, check_kernel<KV, T>, k, a, Ychk, m, n_pad, l, Z, ldz, Xp, ldx, bad, n_bad, vec_z,
                               vec_x) != cudaSuccess)
            return MOSAIC_ERR_CUDA;
    }
    return launch_status();
}

}  // namespace

mosaic_status freivalds_colsum(const uint32_t *a, int k, const uint32_t *W, int64_t ldw, int64_t m,
                               int64_t ncols, uint32_t *Y, cudaStream_t st) {
    if (k < 1 || k > kMaxK) return MOSAIC_ERR_ARG;
    if (cudaMemsetAsync(Y, 0, sizeof(uint32_t) * (size_t)k * (size_t)ncols, st) != cudaSuccess)
        return MOSAIC_ERR_CUDA;
    if (m == 0 || ncols == 0) return MOSAIC_OK;
    // About four resident blocks per SM: split the rows so that the grid has
    // ~600 blocks, each summing at least 64 rows.
    const int64_t xblocks = (ncols + 255) / 256;
    int64_t yblocks = (608 + xblocks - 1) / xblocks;
    int64_t rows = (m + yblocks - 1) / yblocks;
    if (rows < 64) rows = 64;
    yblocks = (m + rows - 1) / rows;
    if (xblocks > 0x7fffffff || yblocks > 65535) return MOSAIC_ERR_SHAPE;
    {
        KernelSpan span("freivalds_colsum", st);
        colsum_kernel<<<dim3((unsigned)xblocks, (unsigned)yblocks), 256, 0, st>>>(a, k, W, ldw, m, ncols, rows, Y);
    }
    return launch_status();
}

mosaic_status freivalds_check(int k, const uint32_t *a, const uint32_t *Ychk, int64_t m, int64_t n_pad,
                              int64_t l, const uint32_t *Z, int64_t ldz, const uint32_t *Xp, int64_t ldx,
                              uint32_t *bad, uint32_t *n_bad, uint32_t *lhs, uint32_t *rhs, cudaStream_t st) {
    if (k < 1 || k > kMaxK) return MOSAIC_ERR_ARG;
    if (l == 0) return MOSAIC_OK;
    // Four tokens a cluster once that still fills the SMs with clusters of 8.
    int dev = 0;
    const bool four = cudaGetDevice(&dev) == cudaSuccess && 2 * l >= sm_count(dev);
#define MOSAIC_CHECK(KV)                                                                                         \
    (four ? launch_check<KV, 4>(k, a, Ychk, m, n_pad, l, Z, ldz, Xp, ldx, bad, n_bad, lhs, rhs, st)              \
          : launch_check<KV, 1>(k, a, Ychk, m, n_pad, l, Z, ldz, Xp, ldx, bad, n_bad, lhs, rhs, st))
    if (k <= 2) return MOSAIC_CHECK(2);
    if (k <= 4) return MOSAIC_CHECK(4);
    if (k <= 8) return MOSAIC_CHECK(8);
    return MOSAIC_CHECK(16);
#undef MOSAIC_CHECK
}

}  // namespace mosaic

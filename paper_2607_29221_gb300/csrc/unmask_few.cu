// Unmask and decode of a few tokens (one decode step or a small batch) in one
// launch (Sec. 3.2 box, Online step 5; Pi_Sec-Linear Online step 3):
//   Y_hat = Y' - K - L Q_d - sum_i S_{i+1} Q_i,  Y = Y_hat s_w s_x + bias.
//
// With l <= 16 tokens the step is bound by reading the client's rows once:
// per output row j, L's row (r_d words) and the row's S lists ((position,
// value) pairs), about 3.9 KB at the Example 3.1 ranks against 3212 l words of
// Q that every row shares.  So each block stages all of Q once, [position][token]
// so that one position's tokens are one vector load, and its warps walk output
// rows: a warp issues its row's loads of L, lists, Y' and K up front (everything
// it needs from HBM is in flight at once), then multiplies out of shared
// memory and sums the lanes with a halving exchange.  The dense segment Q_d
// is stored quad-transposed (position k at (k mod 4) quads + k / 4), so the
// lanes of a warp, which hold four consecutive K values each, read consecutive
// vectors.  With one or two tokens a lane keeps every token of its share of a
// row and two blocks share an SM (unmask_few_kernel); with more, the
// shared-memory reads of Q would bind, so the tokens are split over 1, 2 or 4
// lanes of four tokens each and a warp takes four rows at a time, which share
// its dense reads of Q (unmask_rows_kernel).
//
// Whole call on output rows x tokens, microseconds (ranks (1536, 1024, 652), t =
// 80): the preparation, CUDA-core product and two gather passes that it replaced,
// and one launch of this kernel; "flushed": L2 flushed before each call, events
// around it, else back to back inside a CUDA graph, where 8192 rows of L and S
// (33 MB) stay in L2:
//                       57344 x 1   57344 x 8  57344 x 16   8192 x 1  8192 x 8  8192 x 16
//   before, graph          81.9        113.2      139.2        14.8      33.7      38.3
//   one launch, graph      42.6         94.6      140.0         7.5      14.0      22.6
//   before, flushed        98.3        129.0      155.7        32.8      51.2      55.3
//   one launch, flushed    55.3        106.5      149.5        16.4      28.7      38.9
// (42.6 us = 5.2 TB/s of L and S lists; with more tokens the shared-memory reads
// and multiply-adds of a row bind instead: unmask_few_loses() tells where a call
// is better off on the general path, as 57344 x 16 is, 103 us in a graph.)
#include "mosaic_internal.cuh"

namespace mosaic {
namespace {

constexpr int kUfThreads = 512;
constexpr int kUfWarps = kUfThreads / 32;
constexpr int kUfDense = 6;    // quads of L a lane loads ahead (768 words)
constexpr int kUfSparse = 3;   // pairs of a list a lane loads ahead (96 pairs)

struct UfArgs {
    const uint32_t *Z;
    int64_t ldz;
    const uint32_t *K, *L;
    int l, m, rd, quads;       // quads: stride of the quad-transposed dense segment
    int vec_l;                 // L rows take 16-byte loads
    int nlev;
    const uint32_t *idx[2], *val[2];
    int t[2], r[2];
    int vec_s[2];              // lists take 16-byte loads
    int64_t col[2];            // first column of Q_i in Z
    int64_t dcol;              // first column of Q_d in Z
    const float *s_w, *s_x, *bias;
    float *Y;
    uint32_t *Yhat;
    int64_t ldy;
};

template <int NT>
struct Toks {
    uint32_t v[NT];
};
// The NT tokens of staged index i.
template <int NT>
__device__ __forceinline__ Toks<NT> toks(const uint32_t *sm, int i) {
    Toks<NT> q;
    if constexpr (NT == 2) {
        const uint2 x = *reinterpret_cast<const uint2 *>(sm + i * 2);
        q.v[0] = x.x; q.v[1] = x.y;
    } else {
        q.v[0] = sm[i];
    }
    return q;
}

template <int NT>
__device__ __forceinline__ void mac(uint32_t (&acc)[NT], uint32_t x, const Toks<NT> &q) {
#pragma unroll
    for (int t = 0; t < NT; t++) acc[t] += x * q.v[t];
}

template <int NT>
__global__ void __launch_bounds__(kUfThreads, 2) unmask_few_kernel(UfArgs a) {
    extern __shared__ __align__(16) uint32_t sm[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    // Stage Q: the dense segment quad-transposed first, then each level's positions.
    const int dense = 4 * a.quads;
    auto put = [&](int i, int64_t col) {
        Toks<NT> q;
#pragma unroll
        for (int t = 0; t < NT; t++) q.v[t] = t < a.l ? __ldg(a.Z + t * a.ldz + col) : 0u;
#pragma unroll
        for (int t = 0; t < NT; t++) sm[i * NT + t] = q.v[t];
    };
    for (int k = threadIdx.x; k < a.rd; k += kUfThreads) put((k & 3) * a.quads + (k >> 2), a.dcol + k);
    int base[2];
    base[0] = dense;
    base[1] = dense + (a.nlev > 0 ? a.r[0] : 0);
    for (int i = 0; i < a.nlev; i++)
        for (int p = threadIdx.x; p < a.r[i]; p += kUfThreads) put(base[i] + p, a.col[i] + p);
    __syncthreads();

    const int nq = a.rd >> 2;   // whole quads of an L row
    for (int j = blockIdx.x * kUfWarps + warp; j < a.m; j += gridDim.x * kUfWarps) {
        const uint32_t *Lr = a.L + (int64_t)j * a.rd;
        // Everything row j needs from HBM, issued before the first use.
        uint4 d[kUfDense];
        if (a.vec_l) {
#pragma unroll
            for (int i = 0; i < kUfDense; i++) {
                const int q = lane + 32 * i;
                d[i] = q < nq ? __ldg(reinterpret_cast<const uint4 *>(Lr) + q) : make_uint4(0u, 0u, 0u, 0u);
            }
        }
        uint32_t sp[2][kUfSparse], sv[2][kUfSparse];
#pragma unroll
        for (int i = 0; i < 2; i++)
#pragma unroll
            for (int e = 0; e < kUfSparse; e++) {
                const int q = lane + 32 * e;
                const bool ok = i < a.nlev && q < a.t[i];
                sp[i][e] = ok ? __ldg(a.idx[i] + (int64_t)j * a.t[i] + q) : 0u;
                sv[i][e] = ok ? __ldg(a.val[i] + (int64_t)j * a.t[i] + q) : 0u;
            }
        // Lane layout of the sums after the exchange below: token t on the lanes t (32 / NT) ..
        const int tok = lane / (32 / NT);
        const bool writes = lane % (32 / NT) == 0 && tok < a.l;
        uint32_t base_y = 0u;
        if (writes) base_y = __ldg(a.Z + tok * a.ldz + j) - __ldg(a.K + (int64_t)tok * a.m + j);

        uint32_t acc[NT];
#pragma unroll
        for (int t = 0; t < NT; t++) acc[t] = 0u;
        if (a.vec_l) {
#pragma unroll
            for (int i = 0; i < kUfDense; i++) {
                const int q = lane + 32 * i;
                if (q < nq) {
                    mac<NT>(acc, d[i].x, toks<NT>(sm, q));
                    mac<NT>(acc, d[i].y, toks<NT>(sm, a.quads + q));
                    mac<NT>(acc, d[i].z, toks<NT>(sm, 2 * a.quads + q));
                    mac<NT>(acc, d[i].w, toks<NT>(sm, 3 * a.quads + q));
                }
            }
            for (int q = lane + 32 * kUfDense; q < nq; q += 32) {
                const uint4 x = __ldg(reinterpret_cast<const uint4 *>(Lr) + q);
                mac<NT>(acc, x.x, toks<NT>(sm, q));
                mac<NT>(acc, x.y, toks<NT>(sm, a.quads + q));
                mac<NT>(acc, x.z, toks<NT>(sm, 2 * a.quads + q));
                mac<NT>(acc, x.w, toks<NT>(sm, 3 * a.quads + q));
            }
        } else {
            for (int k = lane; k < a.rd; k += 32) mac<NT>(acc, __ldg(Lr + k), toks<NT>(sm, (k & 3) * a.quads + (k >> 2)));
        }
#pragma unroll
        for (int i = 0; i < 2; i++) {
            if (i >= a.nlev) break;
            const uint32_t last = (uint32_t)a.r[i] - 1u;   // malformed positions stay inside the segment
#pragma unroll
            for (int e = 0; e < kUfSparse; e++)
                if (lane + 32 * e < a.t[i]) mac<NT>(acc, sv[i][e], toks<NT>(sm, base[i] + (int)min(sp[i][e], last)));
            for (int q = lane + 32 * kUfSparse; q < a.t[i]; q += 32)
                mac<NT>(acc, __ldg(a.val[i] + (int64_t)j * a.t[i] + q),
                        toks<NT>(sm, base[i] + (int)min(__ldg(a.idx[i] + (int64_t)j * a.t[i] + q), last)));
        }
        // Sum the lanes: log2(NT) halving exchanges leave each lane with one
        // token, whose 32 / NT lanes then meet in plain butterflies.
        int off = 16;
#pragma unroll
        for (int half = NT / 2; half >= 1; half >>= 1, off >>= 1) {
            const bool upper = (lane & off) != 0;
#pragma unroll
            for (int i = 0; i < half; i++) {
                const uint32_t send = upper ? acc[i] : acc[half + i];
                const uint32_t keep = upper ? acc[half + i] : acc[i];
                acc[i] = keep + __shfl_xor_sync(0xffffffffu, send, off);
            }
        }
        for (; off >= 1; off >>= 1) acc[0] += __shfl_xor_sync(0xffffffffu, acc[0], off);
        if (writes) {
            const uint32_t y = base_y - acc[0];
            if (a.Yhat) a.Yhat[tok * a.ldy + j] = y;
            float f = __fmul_rn(__fmul_rn(__int2float_rn((int32_t)y), a.s_w[j]), a.s_x[tok]);
            if (a.bias) f = __fadd_rn(f, a.bias[j]);
            a.Y[tok * a.ldy + j] = f;
        }
    }
}

// 3 to 16 tokens: CH = 1, 2 or 4 lanes of four tokens each share a position, so
// that a warp holds 32 / CH positions ("slots") at a time and every phase of a
// shared-memory access reads whole positions; a warp takes R rows, whose dense
// products use each vector of Q it reads R times.
template <int CH, int R>
__global__ void __launch_bounds__(kUfThreads, 1) unmask_rows_kernel(UfArgs a) {
    constexpr int NT = 4 * CH, SLOTS = 32 / CH;
    constexpr int V = 4 * R;                              // sums a lane holds
    constexpr int HMAX = SLOTS == 32 ? 5 : SLOTS == 16 ? 4 : 3, VMAX = R == 4 ? 4 : 2;
    constexpr int H = HMAX < VMAX ? HMAX : VMAX;          // halving exchanges
    constexpr int VL = V >> H;                            // sums a lane holds after them
    extern __shared__ __align__(16) uint32_t sm[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int slot = lane / CH, ch = lane % CH;
    auto put = [&](int i, int64_t col) {
        uint32_t q[NT];
#pragma unroll
        for (int t = 0; t < NT; t++) q[t] = t < a.l ? __ldg(a.Z + t * a.ldz + col) : 0u;
#pragma unroll
        for (int t = 0; t < NT; t += 4)
            *reinterpret_cast<uint4 *>(sm + i * NT + t) = make_uint4(q[t], q[t + 1], q[t + 2], q[t + 3]);
    };
    for (int k = threadIdx.x; k < a.rd; k += kUfThreads) put((k & 3) * a.quads + (k >> 2), a.dcol + k);
    const int base0 = 4 * a.quads, base1 = base0 + (a.nlev > 0 ? a.r[0] : 0);
    for (int i = 0; i < a.nlev; i++)
        for (int p = threadIdx.x; p < a.r[i]; p += kUfThreads) put((i ? base1 : base0) + p, a.col[i] + p);
    __syncthreads();
    const uint32_t *smc = sm + 4 * ch;   // this lane's four tokens of index i: smc[i NT ..]

    const int nq = a.rd >> 2;
    for (int j0 = (blockIdx.x * kUfWarps + warp) * R; j0 < a.m; j0 += gridDim.x * kUfWarps * R) {
        // Row of local index r: rows past the end repeat the last one and are not written.
        auto row = [&](int r) { return (int64_t)(j0 + r < a.m ? j0 + r : a.m - 1); };
        // After the exchanges lane (slot, ch) holds sums v0 .. v0 + VL - 1, v = 4 r + token of the chunk.
        int v0 = 0;
        {
            int off = SLOTS / 2;
#pragma unroll
            for (int h = 0; h < H; h++, off >>= 1)
                if (slot & off) v0 += V >> (h + 1);
        }
        const bool writer = (slot & ((SLOTS >> H) - 1)) == 0;
        uint32_t base_y[VL];
#pragma unroll
        for (int i = 0; i < VL; i++) {
            const int j = j0 + ((v0 + i) >> 2), t = 4 * ch + ((v0 + i) & 3);
            base_y[i] = writer && j < a.m && t < a.l ? __ldg(a.Z + t * a.ldz + j) - __ldg(a.K + (int64_t)t * a.m + j) : 0u;
        }
        uint32_t acc[R][4];
#pragma unroll
        for (int r = 0; r < R; r++)
#pragma unroll
            for (int t = 0; t < 4; t++) acc[r][t] = 0u;
        auto mac4 = [&](int r, uint32_t x, const uint4 &q) {
            acc[r][0] += x * q.x;
            acc[r][1] += x * q.y;
            acc[r][2] += x * q.z;
            acc[r][3] += x * q.w;
        };
        if (a.vec_l) {
#pragma unroll 3
            for (int q0 = 0; q0 < nq; q0 += SLOTS) {
                const int q = q0 + slot;
                uint4 x[R];
#pragma unroll
                for (int r = 0; r < R; r++)
                    x[r] = q < nq ? __ldg(reinterpret_cast<const uint4 *>(a.L + row(r) * a.rd) + q) : make_uint4(0u, 0u, 0u, 0u);
                const int qs = q < nq ? q : 0;   // in bounds; its products are with zeros
#pragma unroll
                for (int k = 0; k < 4; k++) {
                    const uint4 y = *reinterpret_cast<const uint4 *>(smc + (k * a.quads + qs) * NT);
#pragma unroll
                    for (int r = 0; r < R; r++) mac4(r, k == 0 ? x[r].x : k == 1 ? x[r].y : k == 2 ? x[r].z : x[r].w, y);
                }
            }
        } else {
            for (int k = slot; k < a.rd; k += SLOTS) {
                const uint4 y = *reinterpret_cast<const uint4 *>(smc + ((k & 3) * a.quads + (k >> 2)) * NT);
#pragma unroll
                for (int r = 0; r < R; r++) mac4(r, __ldg(a.L + row(r) * a.rd + k), y);
            }
        }
#pragma unroll
        for (int i = 0; i < 2; i++) {
            if (i >= a.nlev) break;
            const uint32_t last = (uint32_t)a.r[i] - 1u;   // malformed positions stay inside the segment
            const uint32_t *sml = smc + (i ? base1 : base0) * NT;
            const int t = a.t[i];
            if (a.vec_s[i]) {
#pragma unroll
                for (int r = 0; r < R; r++) {
                    const uint4 *ip = reinterpret_cast<const uint4 *>(a.idx[i] + row(r) * t);
                    const uint4 *vp = reinterpret_cast<const uint4 *>(a.val[i] + row(r) * t);
#pragma unroll 3
                    for (int q = slot; q < t >> 2; q += SLOTS) {
                        const uint4 p = __ldg(ip + q), v = __ldg(vp + q);
                        mac4(r, v.x, *reinterpret_cast<const uint4 *>(sml + min(p.x, last) * NT));
                        mac4(r, v.y, *reinterpret_cast<const uint4 *>(sml + min(p.y, last) * NT));
                        mac4(r, v.z, *reinterpret_cast<const uint4 *>(sml + min(p.z, last) * NT));
                        mac4(r, v.w, *reinterpret_cast<const uint4 *>(sml + min(p.w, last) * NT));
                    }
                }
            } else {
#pragma unroll
                for (int r = 0; r < R; r++)
                    for (int q = slot; q < t; q += SLOTS)
                        mac4(r, __ldg(a.val[i] + row(r) * t + q),
                             *reinterpret_cast<const uint4 *>(sml + min(__ldg(a.idx[i] + row(r) * t + q), last) * NT));
            }
        }
        uint32_t sum[V];
#pragma unroll
        for (int v = 0; v < V; v++) sum[v] = acc[v >> 2][v & 3];
        int off = 16;
#pragma unroll
        for (int h = 0; h < H; h++, off >>= 1) {
            const int half = V >> (h + 1);
            const bool upper = (lane & off) != 0;
#pragma unroll
            for (int i = 0; i < half; i++) {
                const uint32_t send = upper ? sum[i] : sum[half + i];
                const uint32_t keep = upper ? sum[half + i] : sum[i];
                sum[i] = keep + __shfl_xor_sync(0xffffffffu, send, off);
            }
        }
#pragma unroll
        for (; off >= CH; off >>= 1)
#pragma unroll
            for (int i = 0; i < VL; i++) sum[i] += __shfl_xor_sync(0xffffffffu, sum[i], off);
        if (writer) {
#pragma unroll
            for (int i = 0; i < VL; i++) {
                const int j = j0 + ((v0 + i) >> 2), t = 4 * ch + ((v0 + i) & 3);
                if (j < a.m && t < a.l) {
                    const uint32_t y = base_y[i] - sum[i];
                    if (a.Yhat) a.Yhat[t * a.ldy + j] = y;
                    float f = __fmul_rn(__fmul_rn(__int2float_rn((int32_t)y), a.s_w[j]), a.s_x[t]);
                    if (a.bias) f = __fadd_rn(f, a.bias[j]);
                    a.Y[t * a.ldy + j] = f;
                }
            }
        }
    }
}

template <class Kernel>
mosaic_status launch(Kernel kern, std::atomic<unsigned long long> &attr_set, int rows, const UfArgs &a, size_t smem,
                     int per_sm, cudaStream_t st) {
    int dev = 0, sms = 0;
    if (!ensure_smem_limit(attr_set, kern, kUnmaskFewSmem, &dev) ||
        (sms = sm_count(dev)) < 1)
        return MOSAIC_ERR_CUDA;
    const int need = (a.m + kUfWarps * rows - 1) / (kUfWarps * rows);
    const int slots = sms * per_sm;
    {
        KernelSpan span("unmask_few", st);
        kern<<<need < slots ? need : slots, kUfThreads, smem, st>>>(a);
    }
    return launch_status();
}
template <int NT>
mosaic_status launch_few(const UfArgs &a, size_t smem, cudaStream_t st) {
    static std::atomic<unsigned long long> attr_set{0};   // one bit per device ordinal
    return launch(unmask_few_kernel<NT>, attr_set, 1, a, smem, smem <= 113 * 1024 ? 2 : 1, st);
}
// Four rows a warp where one row a warp would take three rounds or more over the
// SMs' warps (4865 rows on 152 SMs), else one.  Ratio of the two, 8 tokens, by
// (r_d, t, t): rows 2048 4096 6144 8191: (652, 80, 80) 1.65 1.15 0.89 0.73;
// (1536) 1.59 1.00 0.74 0.59; (64, 8, 8) 1.41 1.07 0.89 0.76.
template <int CH>
mosaic_status launch_rows(const UfArgs &a, size_t smem, cudaStream_t st) {
    static std::atomic<unsigned long long> attr1{0}, attr4{0};   // one bit per device ordinal
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return MOSAIC_ERR_CUDA;
    if (a.m > 2 * kUfWarps * sm_count(dev)) return launch(unmask_rows_kernel<CH, 4>, attr4, 4, a, smem, 1, st);
    return launch(unmask_rows_kernel<CH, 1>, attr1, 1, a, smem, 1, st);
}

size_t smem_bytes(int64_t l, int64_t rd, int nlev, const SparseLevel *lev) {
    const int64_t nt = l <= 1 ? 1 : l <= 2 ? 2 : l <= 4 ? 4 : l <= 8 ? 8 : 16;
    int64_t words = 4 * ((rd + 3) / 4);
    for (int i = 0; i < nlev; i++) words += lev[i].r;
    return (size_t)(4 * nt * words);
}

}  // namespace

bool unmask_few_ok(int64_t l, int64_t m, int64_t rd, int nlev, const SparseLevel *lev) {
    return l >= 1 && l <= 16 && m <= (int64_t)INT32_MAX / 2 && nlev <= 2 &&
           smem_bytes(l, rd, nlev, lev) <= kUnmaskFewSmem;
}

// When the general path (a product that streams L, then the gathers) is the
// faster one.  It costs about 2 us a launch and a gather pass a level; what it
// gains lies in the dense words r_d of a row, which the product streams at 7
// TB/s where the one launch reads L at 5.2 (one or two tokens) or is bound by the
// shared-memory reads and multiply-adds of its rows (more tokens).  The latter
// go up with every round of rows over the warps: 2432 rows (152 x 16), and, with
// four rows a warp from 4865 rows on, 9728.  The lines were drawn through the
// ratios one launch / general of r_d from 64 to 14000, one to three levels of t
// = 8, 80, 128 and 400, and 16 to 57344 rows; the lists' words (sum_t = t_2 +
// t_3) move a line up since the gathers then cost more.  Examples, ratio of the
// whole call inside a CUDA graph, one launch / general (with L2 flushed before
// every call the ratios cross 1 at the same places):
//   1 token, d = 1:  r_d 2048 x 57344 rows 1.00, 4096 x 4096 0.64, 4096 x 57344 1.18
//   1 token, d = 3, t = 80:  4096 x 57344 0.99, 8192 x 8192 1.15
//   4 tokens, d = 1:  8192 x 20480 1.14, 12000 x 2448 1.36, 12000 x 1024 0.69
//   8 tokens, d = 1:  2048 x 4096 1.01, 4096 x 1024 0.74, 4096 x 4096 1.24,
//                     4096 x 8192 0.94, 4096 x 20480 1.26, 4096 x 28672 0.87
//   8 tokens, d = 3, t = 80:  4096 x 4096 0.73, 4096 x 12000 1.13
//   16 tokens, d = 1:  1024 x 2400 0.64, 1536 x 16 1.20, 1536 x 2448 1.38, 2048 x 4864 1.44
//   16 tokens, d = 3, t = 80:  1536 x 16 0.93, 2700 x 16 1.42, 1536 x 4096 1.08, 2700 x 2448 1.64
// Beyond 9728 rows, 9 to 16 tokens stream L wherever a row holds enough words
// (r_d + sum_t); whole call at 16 tokens, L2 flushed before each, events
// around it (about 10 us of them are launch and events), one launch /
// streamed, microseconds, by words a row:
//   rows     812 (652, 80, 80)   1536 (one level)   732 (652, 80)   280 (200, 40, 40)
//    8192      38.9 / 49.2          30.7 / 33.8       28.7 / 36.9      22.5 / 36.9
//   10240      59.4 / 49.2          49.2 / 39.9       45.1 / 36.9      32.8 / 36.9
//   20480      86.0 / 73.7          69.6 / 52.2       61.4 / 53.3      45.1 / 53.3
//   57344     149.5 / 116.7        124.9 / 105.4      108.5 / 88.0     82.0 / 73.7
constexpr int64_t kFewRowWords = 512;
bool unmask_few_loses(int64_t l, int64_t m, int64_t rd, int nlev, const SparseLevel *lev) {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return false;
    int64_t sum_t = 0;
    bool tiled = true;   // the general path's gathers take every level in tiles
    for (int i = 0; i < nlev; i++) {
        tiled = tiled && pgather_takes(l, lev[i].r, lev[i].t) && aligned16(lev[i].idx) && aligned16(lev[i].val);
        sum_t += lev[i].t;
    }
    const int64_t rows = (int64_t)sm_count(dev) * kUfWarps;   // one row a warp; 4 rows from 2 rounds on
    if (l <= 2) {
        if (nlev == 0 && rd < 512) return m > 10 * rows;      // little to read: the rows' own overhead
        return m * rd >= (int64_t)(nlev ? 20 : 24) << 20 && rd > 2560 + 1024 * nlev;
    }
    if (l <= 4) return m > rows && rd > 8192;
    if (l <= 8) {
        if (m <= rows) return false;
        if (m <= 2 * rows) return rd > 2048 + 16 * sum_t;
        const int64_t rounds = (m + 4 * rows - 1) / (4 * rows);   // the last one may be nearly empty
        return 2 * m > (rd > 3072 ? 8 : 9) * rows && m < 3 * rounds * rows && rd > 1792 + 4 * sum_t;
    }
    if (!tiled) return false;
    if (m > 4 * rows) return rd + sum_t >= kFewRowWords;
    if (m <= rows) return rd > (nlev || m < 128 ? 1280 : 1600) + 5 * sum_t;   // a few rows leave SMs idle
    return rd > (m <= 2 * rows ? 850 : nlev ? 1350 : 1600) + 3 * sum_t;
}

mosaic_status unmask_few(int64_t l, int64_t m, const uint32_t *Z, int64_t ldz, int64_t dcol, int64_t rd,
                         const uint32_t *K_tm, const uint32_t *L, int nlev, const SparseLevel *lev, const float *s_w,
                         const float *s_x, const float *bias, float *Y, uint32_t *Yhat, int64_t ldy,
                         cudaStream_t st) {
    if (!unmask_few_ok(l, m, rd, nlev, lev)) return MOSAIC_ERR_SHAPE;
    UfArgs a{};
    a.Z = Z; a.ldz = ldz; a.K = K_tm; a.L = L;
    a.l = (int)l; a.m = (int)m; a.rd = (int)rd; a.quads = (int)((rd + 3) / 4);
    a.vec_l = rd % 4 == 0 && aligned16(L);
    a.nlev = nlev;
    for (int i = 0; i < nlev; i++) {
        a.idx[i] = lev[i].idx; a.val[i] = lev[i].val;
        a.vec_s[i] = lev[i].t % 4 == 0 && aligned16(lev[i].idx) && aligned16(lev[i].val);
        a.t[i] = lev[i].t; a.r[i] = (int)lev[i].r; a.col[i] = lev[i].off;
    }
    a.dcol = dcol;
    a.s_w = s_w; a.s_x = s_x; a.bias = bias; a.Y = Y; a.Yhat = Yhat; a.ldy = ldy;
    const size_t smem = smem_bytes(l, rd, nlev, lev);
    if (l == 1) return launch_few<1>(a, smem, st);
    if (l == 2) return launch_few<2>(a, smem, st);
    if (l <= 4) return launch_rows<1>(a, smem, st);
    if (l <= 8) return launch_rows<2>(a, smem, st);
    return launch_rows<4>(a, smem, st);
}

}  // namespace mosaic

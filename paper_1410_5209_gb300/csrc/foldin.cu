// Fold-in of a new row against frozen factors: the ALS row solve of Eq. (2),
// a = (B + lambda I_K)^{-1} c with B = sum_e h_e h_e^T, c = sum_e x_e h_e and
// h_e,k = prod_{l != mode} a^(l)_{i_l k}, over the request's m entries.
// Float contexts (K < 128) refine every solve once: the residual of the normal equations
// is formed from the entries to twice the working precision and the correction solved with
// the FP32 factor, which takes the row to FP32 accuracy whatever the rounding of the FP32
// Gram sums.
//
// K >= 128: one block per request.  Entries are taken in tiles of kTileE: the tile's H rows
// are built in shared memory, then each thread adds the tile's contribution to its own
// entries of the lower triangle of B (kept in shared memory) and of c.  The K x K
// system is factored in place by a right-looking Cholesky (one column per step), and
// warp 0 does the two triangular solves.  K < 128: further down.
#include <algorithm>

#include "float_pair.cuh"
#include "sweep.cuh"

namespace tfs {
namespace {

constexpr int kFoldThreads = 256;
constexpr int kTileE = 32;

template <class T>
__global__ void __launch_bounds__(kFoldThreads) k_foldin(const FoldArgs<T> a) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int K = a.K;
    T *B = reinterpret_cast<T *>(smem_raw);  // K*K, lower triangle used
    T *cv = B + (size_t)K * K;                // K (c, then y, then x)
    T *H = cv + K;                            // kTileE*K
    T *xs = H + (size_t)kTileE * K;           // kTileE
    __shared__ int bad;
    const int tid = threadIdx.x;
    if (tid == 0) bad = 0;
    for (int q = tid; q < K * K; q += blockDim.x) B[q] = T(0);
    for (int q = tid; q < K; q += blockDim.x) cv[q] = T(0);
    __syncthreads();

    for (int64_t e0 = 0; e0 < a.m; e0 += kTileE) {
        const int ne = (int)(a.m - e0 < kTileE ? a.m - e0 : kTileE);
        for (int q = tid; q < ne * K; q += blockDim.x) {
            const int e = q / K, k = q - e * K;
            T p = T(1);
            int t = 0;
            for (int l = 0; l < a.N; ++l) {
                if (l == a.mode) continue;
                const int32_t idx = a.other[(e0 + e) * (a.N - 1) + t];
                ++t;
                if (idx < 0 || idx >= a.I[l]) {
                    bad = 1;
                    p = T(0);
                } else {
                    p *= a.A[l][(int64_t)idx * K + k];
                }
            }
            H[e * K + k] = p;
        }
        for (int q = tid; q < ne; q += blockDim.x) xs[q] = a.x[e0 + q];
        __syncthreads();
        for (int q = tid; q < K * K; q += blockDim.x) {
            const int i = q / K, j = q - i * K;
            if (j > i) continue;
            T s = T(0);
            for (int e = 0; e < ne; ++e) s += H[e * K + i] * H[e * K + j];
            B[q] += s;
        }
        for (int q = tid; q < K; q += blockDim.x) {
            T s = T(0);
            for (int e = 0; e < ne; ++e) s += H[e * K + q] * xs[e];
            cv[q] += s;
        }
        __syncthreads();
    }
    for (int q = tid; q < K; q += blockDim.x) B[q * K + q] += a.lambda;
    __syncthreads();

    // right-looking Cholesky, lower triangle
    __shared__ int pivot_bad;
    if (tid == 0) pivot_bad = 0;
    for (int j = 0; j < K; ++j) {
        __syncthreads();
        if (tid == 0) {
            T d = B[j * K + j];
            if (!(d > T(0))) {
                pivot_bad = 1;
                d = T(1);
            }
            B[j * K + j] = sqrt(d);
        }
        __syncthreads();
        const T ljj = B[j * K + j];
        for (int i = j + 1 + tid; i < K; i += blockDim.x) B[i * K + j] /= ljj;
        __syncthreads();
        const int rem = K - j - 1;
        for (int q = tid; q < rem * rem; q += blockDim.x) {
            const int i = j + 1 + q / rem, k = j + 1 + q % rem;
            if (k <= i) B[i * K + k] -= B[i * K + j] * B[k * K + j];
        }
    }
    __syncthreads();
    if (tid < kWarp) {
        const int lane = tid;
        for (int i = 0; i < K; ++i) {  // L y = c (y overwrites c)
            T s = T(0);
            for (int k = lane; k < i; k += kWarp) s += B[i * K + k] * cv[k];
            for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xFFFFFFFFu, s, o);
            if (lane == 0) cv[i] = (cv[i] - s) / B[i * K + i];
            __syncwarp();
        }
        for (int i = K - 1; i >= 0; --i) {  // L^T x = y (x overwrites y)
            T s = T(0);
            for (int k = i + 1 + lane; k < K; k += kWarp) s += B[k * K + i] * cv[k];
            for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xFFFFFFFFu, s, o);
            if (lane == 0) cv[i] = (cv[i] - s) / B[i * K + i];
            __syncwarp();
        }
    }
    __syncthreads();
    if (tid == 0) {
        if (bad) atomicOr(&a.stat->bits, kStatFoldRange);
        if (pivot_bad) atomicOr(&a.stat->bits, kStatFoldPivot);
    }
    if (!bad && !pivot_bad)
        for (int q = tid; q < K; q += blockDim.x) a.out[q] = cv[q];
}

// ---------------------------------------------------------------------------- K < 128
// Two kernels for any number of requests.  Both take blocks of consecutive entries of one
// request (foldin_plan_blocks; the cut depends on the request alone, so a row does not
// depend on the batch it arrives in), write a partial result each, and the block that
// finishes a request last (a counter per request) sums the partials in block order and
// solves.  What bounds them is latency for one request and issue for a batch.  On GB300, one
// request of 317 entries at K = 100 took 123 (gram) + 304 (solve) + 198 (residual) + 71
// (refine) us as four kernels with one warp per solve, and takes 54 + 26 us; 256 requests,
// 337,568 entries: 505 + 605 + 1,550 + 79 us before, 290 + 165 us now.
//   k_fold_gram: tiles of 32 entries build H' = [H | x] in shared memory (8 threads per
//     entry, 16-byte loads of the factor rows where K allows), and threads hold R x R tiles
//     of the lower triangle of H'^T H' (B and, in row K, c).  Only the tiles that exist
//     are handed out, and where they are fewer than the threads, several groups of threads
//     take every G-th entry and add up at the end: the old 16 x 16 thread grid left 47% of
//     the threads idle above the diagonal.
//   The solve is a blocked Cholesky of [B + lambda I, c] by the whole block (panels of 16
//     columns: diagonal block in one warp's registers, the rows below one per thread, the
//     rest 4 x 4 tiles); c travels as one more row, so the forward substitution comes with
//     the factor.
//   k_fold_resid (float): sum_e h_e (x_e - h_e . x0) in pairs of floats (float_pair.cuh,
//     ~48 bits; in FP64 it took 8 times as long), 8 lanes per entry, then the correction
//     solved with the stored factor.  One step of refinement leaves 2^-48 times the square of
//     the condition, so pairs do for it what FP64 does (condition 2e0 to 6e4: errors of the
//     rows 2e-8 to 9e-8, with the former FP64 residual 2e-8 to 3e-7) as long as no bits fall
//     out of the float range: a block that meets a nonzero product or value below 2^-40, or
//     whose sums are not finite, forms its sums in FP64.
// Bad indices and non-positive pivots are flagged per request in req_status (1 and 2).
constexpr int kFoldTile = 32;
constexpr int kFoldBlock = 256;  // two blocks an SM at 128 registers
constexpr int kFoldPanel = 16;

// Register tile edge for K: 16 R columns hold H'.
__host__ __device__ constexpr int fold_edge(int K) { return K + 1 <= 32 ? 2 : (K + 1 <= 64 ? 4 : 8); }
__host__ __device__ constexpr int fold_tiles(int K) {
    const int n = (K + fold_edge(K)) / fold_edge(K);
    return n * (n + 1) / 2;
}
// Row stride of the solved matrix: rows read one per lane in 16-byte vectors do not conflict.
template <class T>
__host__ __device__ constexpr int fold_ld(int K) {
    return sizeof(T) == 4 ? (K + 32) / 32 * 32 + 4 : (K + 16) / 16 * 16 + 2;
}
__host__ __device__ constexpr int fold_fac_ld(int K) { return (K + 3) / 4 * 4; }

template <class T>
struct FoldVec;  // 16 bytes
template <>
struct FoldVec<float> {
    using type = float4;
};
template <>
struct FoldVec<double> {
    using type = double2;
};

// N values from 16-byte aligned (8-byte for N = 2 floats) shared or global memory.
template <class T, int N>
__device__ __forceinline__ void fold_load(const T *p, T (&v)[N]) {
    constexpr int V = 16 / (int)sizeof(T);
    if constexpr (N % V == 0) {
        using Q = typename FoldVec<T>::type;
#pragma unroll
        for (int k = 0; k < N / V; ++k) {
            const Q q = reinterpret_cast<const Q *>(p)[k];
            const T *w = reinterpret_cast<const T *>(&q);
#pragma unroll
            for (int u = 0; u < V; ++u) v[k * V + u] = w[u];
        }
    } else {
        const float2 q = *reinterpret_cast<const float2 *>(p);
        v[0] = q.x, v[1] = q.y;
    }
}

// Place of column c in a row of H'.  With 8-wide float tiles the odd 4-column chunks go to
// the upper half of the row, so that neighbouring lanes' 16-byte reads are neighbours.
template <class T, int R>
__device__ __forceinline__ int fold_pos(int c) {
    if constexpr (R == 8 && sizeof(T) == 4) return (c >> 3) * 4 + ((c >> 2) & 1) * 64 + (c & 3);
    return c;
}
template <class T, int R>
__device__ __forceinline__ void fold_tile_load(const T *h, int I, T (&v)[R]) {
    if constexpr (R == 8 && sizeof(T) == 4) {
        T lo[4], hi[4];
        fold_load<T, 4>(h + 4 * I, lo);
        fold_load<T, 4>(h + 64 + 4 * I, hi);
#pragma unroll
        for (int u = 0; u < 4; ++u) v[u] = lo[u], v[4 + u] = hi[u];
    } else {
        fold_load<T, R>(h + R * I, v);
    }
}

// Row t of lower-triangle element number t counted row by row.
__device__ __forceinline__ int tri_row(int t) {
    int i = (int)((sqrtf(8.f * (float)t + 1.f) - 1.f) * 0.5f);
    while ((i + 1) * (i + 2) / 2 <= t) ++i;
    while (i * (i + 1) / 2 > t) --i;
    return i;
}

// Columns of entry e's H row held by lane g of its 8 lanes, in registers: with 16-byte rows
// (K a multiple of the vector) vectors g, g + 8, ..., else columns g, g + 8, ....
template <class T, int R>
struct FoldCols {
    static constexpr int V = 16 / (int)sizeof(T);
    static constexpr int N = 2 * R;  // columns per lane (16 R / 8)
    static constexpr bool kVec = N >= V;
    __device__ static __forceinline__ int col(int j, int g, bool vec) {
        return vec ? V * (g + 8 * (j / V)) + j % V : g + 8 * j;
    }
    // the lane's columns of one factor row; zero from K on
    __device__ static __forceinline__ void row(const T *r, int K, int g, bool vec, T (&v)[N]) {
        if (vec) {
            if constexpr (kVec) {
#pragma unroll
                for (int k = 0; k < N / V; ++k) {
                    const int c = V * (g + 8 * k);
                    T w[V];
#pragma unroll
                    for (int u = 0; u < V; ++u) w[u] = T(0);
                    if (c < K) fold_load<T, V>(r + c, w);
#pragma unroll
                    for (int u = 0; u < V; ++u) v[k * V + u] = w[u];
                }
            }
        } else {
#pragma unroll
            for (int j = 0; j < N; ++j) v[j] = g + 8 * j < K ? r[g + 8 * j] : T(0);
        }
    }
};

template <class T, int R>
__device__ __forceinline__ bool fold_vec(int K) {
    return FoldCols<T, R>::kVec && K % FoldCols<T, R>::V == 0;
}

// This block was the last of the request's blocks to get here.
__device__ __forceinline__ bool fold_last_block(int32_t *count, int blocks, int *flag) {
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) *flag = atomicAdd(count, 1) == blocks - 1;
    __syncthreads();
    const bool last = *flag != 0;
    __threadfence();
    return last;
}

// Backward substitution L^T x = y, L in A (rows 0 .. K-1, stride LD), inverse diagonal in
// invd; y is replaced by x (shared memory).  red: 8 * kFoldPanel values.  Whole block.
template <class T>
__device__ void fold_back(const T *A, int LD, int K, const T *invd, T *y, T *red) {
    const int tid = threadIdx.x, lane = tid & 31;
    for (int p = (K - 1) / kFoldPanel * kFoldPanel; p >= 0; p -= kFoldPanel) {
        const int nb = K - p < kFoldPanel ? K - p : kFoldPanel;
        const int c = tid & 15, g = tid >> 4;
        T s = T(0);
        if (c < nb)
            for (int r = p + nb + g; r < K; r += 16) s += A[r * LD + p + c] * y[r];
        s += __shfl_xor_sync(0xFFFFFFFFu, s, 16);
        if (lane < 16) red[(tid >> 5) * kFoldPanel + c] = s;
        __syncthreads();
        if (tid < 32) {
            T a[kFoldPanel];
#pragma unroll
            for (int j = 0; j < kFoldPanel; ++j)
                a[j] = (lane < j && j < nb) ? A[(p + j) * LD + p + lane] : T(0);
            T v = T(0);
            if (lane < nb) {
                v = y[p + lane];
#pragma unroll
                for (int w = 0; w < 8; ++w) v -= red[w * kFoldPanel + lane];
            }
            const T inv = lane < nb ? invd[p + lane] : T(0);
#pragma unroll
            for (int j = kFoldPanel - 1; j >= 0; --j) {
                if (lane == j) v *= inv;
                const T xj = __shfl_sync(0xFFFFFFFFu, v, j);
                v -= a[j] * xj;
            }
            if (lane < nb) y[p + lane] = v;
        }
        __syncthreads();
    }
}

// Forward substitution L y = d in place (shared memory).  t: kFoldPanel values.
template <class T>
__device__ void fold_forward(const T *A, int LD, int K, const T *invd, T *d, T *t) {
    const int tid = threadIdx.x, lane = tid & 31;
    for (int p = 0; p < K; p += kFoldPanel) {
        const int nb = K - p < kFoldPanel ? K - p : kFoldPanel;
        const int c = tid & 15, r = tid >> 4;
        T s = T(0);
        if (r < nb)
            for (int cc = c; cc < p; cc += 16) s += A[(p + r) * LD + cc] * d[cc];
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) s += __shfl_xor_sync(0xFFFFFFFFu, s, o);
        if (c == 0 && r < nb) t[r] = d[p + r] - s;
        __syncthreads();
        if (tid < 32) {
            T a[kFoldPanel];
#pragma unroll
            for (int j = 0; j < kFoldPanel; ++j)
                a[j] = (lane > j && lane < nb) ? A[(p + lane) * LD + p + j] : T(0);
            T v = lane < nb ? t[lane] : T(0);
            const T inv = lane < nb ? invd[p + lane] : T(0);
#pragma unroll
            for (int j = 0; j < kFoldPanel; ++j) {
                if (lane == j) v *= inv;
                const T yj = __shfl_sync(0xFFFFFFFFu, v, j);
                v -= a[j] * yj;
            }
            if (lane < nb) d[p + lane] = v;
        }
        __syncthreads();
    }
}

// Cholesky of the K x K system in A (lower triangle, lambda already on the diagonal) with
// the right-hand side as row K: on return rows 0 .. K-1 hold L, row K holds L^-1 c.
// Pt: kFoldPanel x LD values.  Returns false when a pivot was not positive.  Whole block;
// A has its rows rounded up to a multiple of four.
template <class T>
__device__ bool fold_cholesky(T *A, int LD, int K, T *invd, T *Pt, int *bad) {
    const int tid = threadIdx.x, lane = tid & 31;
    if (tid == 0) *bad = 0;
    for (int p = 0; p < K; p += kFoldPanel) {
        const int nb = K - p < kFoldPanel ? K - p : kFoldPanel;
        if (tid < 32) {  // the diagonal block: lane i holds row i
            T a[kFoldPanel];
#pragma unroll
            for (int j = 0; j < kFoldPanel; ++j)
                a[j] = lane < nb ? (j <= lane ? A[(p + lane) * LD + p + j] : T(0))
                                 : (j == lane ? T(1) : T(0));
            bool ok = true;
            T mine = T(1);
#pragma unroll
            for (int j = 0; j < kFoldPanel; ++j) {
                T d = __shfl_sync(0xFFFFFFFFu, a[j], j);
                ok = ok && (d > T(0));
                d = d > T(0) ? d : T(1);
                const T l = sqrt(d), inv = T(1) / l;
                if (lane == j) mine = inv;
                a[j] = lane == j ? l : a[j] * inv;
#pragma unroll
                for (int k = j + 1; k < kFoldPanel; ++k)
                    a[k] -= a[j] * __shfl_sync(0xFFFFFFFFu, a[j], k);
            }
#pragma unroll
            for (int j = 0; j < kFoldPanel; ++j)
                if (lane < nb && j <= lane) A[(p + lane) * LD + p + j] = a[j];
            if (lane < nb) invd[p + lane] = mine;
            if (lane == 0 && !ok) *bad = 1;
        }
        __syncthreads();
        const int q = p + nb, M = K + 1 - q;  // rows below, the right-hand side among them
        if (tid < M) {
            T a[kFoldPanel];
            T *r = A + (q + tid) * LD + p;
            fold_load<T, kFoldPanel>(r, a);
#pragma unroll
            for (int j = 0; j < kFoldPanel; ++j) {
                if (j < nb) {
                    T v = a[j];
#pragma unroll
                    for (int k = 0; k < j; ++k) v -= a[k] * A[(p + j) * LD + p + k];
                    a[j] = v * invd[p + j];
                    r[j] = a[j];
                    Pt[j * LD + tid] = a[j];
                }
            }
        }
        __syncthreads();
        if (q >= K) break;
        const int mt = (M + 3) / 4, nt = mt * (mt + 1) / 2;
        for (int t = tid; t < nt; t += kFoldBlock) {
            const int I = tri_row(t), J = t - I * (I + 1) / 2;
            T acc[4][4];
            T *c = A + (q + 4 * I) * LD + q + 4 * J;
#pragma unroll
            for (int i = 0; i < 4; ++i) fold_load<T, 4>(c + i * LD, acc[i]);
#pragma unroll
            for (int k = 0; k < kFoldPanel; ++k) {
                T x[4], y[4];
                fold_load<T, 4>(Pt + k * LD + 4 * I, x);
                fold_load<T, 4>(Pt + k * LD + 4 * J, y);
#pragma unroll
                for (int i = 0; i < 4; ++i)
#pragma unroll
                    for (int j = 0; j < 4; ++j) acc[i][j] -= x[i] * y[j];
            }
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) c[i * LD + j] = acc[i][j];
        }
        __syncthreads();
    }
    return *bad == 0;
}

// Shared memory of k_fold_gram: the tile of H' and the groups' sums, or the solve.
template <class T, int R>
__host__ __device__ constexpr size_t fold_gram_smem(int K) {
    const size_t h = sizeof(T) * (size_t)kFoldTile * (16 * R + 16 / sizeof(T));
    const size_t red = sizeof(T) * (size_t)fold_tiles(K) * R * R;
    const size_t solve = sizeof(T) * ((size_t)((K + 4) / 4 * 4) * fold_ld<T>(K) +
                                      (size_t)kFoldPanel * fold_ld<T>(K) + 128 + 8 * kFoldPanel);
    const size_t a = h > red ? h : red;
    return a > solve ? a : solve;
}

template <class T, int R, int NO>
__global__ void __launch_bounds__(kFoldBlock, sizeof(T) == 4 ? 2 : 1)
    k_fold_gram(const FoldArgs<T> a) {
    using FC = FoldCols<T, R>;
    constexpr int HS = 16 * R + 16 / (int)sizeof(T);
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ unsigned char tile_i[136], tile_j[136];
    __shared__ int bad, flag;
    T *H = reinterpret_cast<T *>(smem_raw);
    const int tid = threadIdx.x, K = a.K;
    const int ntiles = fold_tiles(K), groups = kFoldBlock / ntiles;
    const int grp = tid / ntiles, tile = tid - grp * ntiles;
    const bool active = grp < groups, vec = fold_vec<T, R>(K);
    if (tid < ntiles) {
        const int I = tri_row(tid);
        tile_i[tid] = (unsigned char)I;
        tile_j[tid] = (unsigned char)(tid - I * (I + 1) / 2);
    }
    if (tid == 0) bad = 0;
    for (int q = tid; q < kFoldTile * HS; q += kFoldBlock) H[q] = T(0);  // columns past K stay 0
    __syncthreads();
    const int I = tile_i[tile < ntiles ? tile : 0], J = tile_j[tile < ntiles ? tile : 0];
    T acc[R][R];
#pragma unroll
    for (int i = 0; i < R; ++i)
#pragma unroll
        for (int j = 0; j < R; ++j) acc[i][j] = T(0);
    const int blk = a.blk0 + blockIdx.x, req = a.blk_req[blk];
    const int64_t b0 = a.blk_range[2 * blk], b1 = a.blk_range[2 * blk + 1];
    for (int64_t e0 = b0; e0 < b1; e0 += kFoldTile) {
        const int ne = (int)(b1 - e0 < kFoldTile ? b1 - e0 : kFoldTile);
        const int e = tid >> 3, g = tid & 7;
        if (e < ne) {
            T hv[FC::N];
            bool ok = true;
            const int no = NO > 0 ? NO : a.N - 1;
#pragma unroll
            for (int j = 0; j < FC::N; ++j) hv[j] = T(1);
#pragma unroll(NO > 0 ? NO : 1)
            for (int t = 0; t < no; ++t) {
                const int l = t < a.mode ? t : t + 1;
                const int32_t idx = a.other[(e0 + e) * (a.N - 1) + t];
                const bool in = idx >= 0 && idx < a.I[l];
                ok = ok && in;
                T v[FC::N];
                FC::row(a.A[l] + (int64_t)(in ? idx : 0) * K, K, g, vec, v);
#pragma unroll
                for (int j = 0; j < FC::N; ++j) hv[j] = t == 0 ? v[j] : hv[j] * v[j];
            }
            T *h = H + e * HS;
#pragma unroll
            for (int j = 0; j < FC::N; ++j) {
                const int c = FC::col(j, g, vec);
                if (c < K) h[fold_pos<T, R>(c)] = ok ? hv[j] : T(0);
            }
            if (g == 0) {
                h[fold_pos<T, R>(K)] = ok ? a.x[e0 + e] : T(0);
                if (!ok) bad = 1;
            }
        }
        __syncthreads();
        if (active) {
#pragma unroll 2
            for (int q = grp; q < ne; q += groups) {
                T x[R], y[R];
                fold_tile_load<T, R>(H + q * HS, I, x);
                fold_tile_load<T, R>(H + q * HS, J, y);
#pragma unroll
                for (int i = 0; i < R; ++i)
#pragma unroll
                    for (int j = 0; j < R; ++j) acc[i][j] += x[i] * y[j];
            }
        }
        __syncthreads();
    }
    for (int o = 1; o < groups; ++o) {  // the groups' sums, in group order
        if (active && grp == o)
#pragma unroll
            for (int i = 0; i < R; ++i)
#pragma unroll
                for (int j = 0; j < R; ++j) H[(i * R + j) * ntiles + tile] = acc[i][j];
        __syncthreads();
        if (grp == 0)
#pragma unroll
            for (int i = 0; i < R; ++i)
#pragma unroll
                for (int j = 0; j < R; ++j) acc[i][j] += H[(i * R + j) * ntiles + tile];
        __syncthreads();
    }
    const int PB = ntiles * R * R;
    if (grp == 0) {
        T *p = a.part + (int64_t)blockIdx.x * PB;
#pragma unroll
        for (int i = 0; i < R; ++i)
#pragma unroll
            for (int j = 0; j < R; ++j) p[(i * R + j) * ntiles + tile] = acc[i][j];
    }
    if (tid == 0 && bad) atomicOr(&a.req_status[req], 1);
    const int bb = a.req_blk[req], be = a.req_blk[req + 1];
    if (!fold_last_block(a.req_count + req, be - bb, &flag)) return;

    const int LD = fold_ld<T>(K);
    T *A = H, *Pt = A + (K + 4) / 4 * 4 * LD, *invd = Pt + kFoldPanel * LD, *red = invd + 128;
    for (int q0 = tid; q0 < PB; q0 += 4 * kFoldBlock) {
        T s[4] = {T(0), T(0), T(0), T(0)};
        for (int b = bb; b < be; ++b) {
            const T *p = a.part + (int64_t)(b - a.blk0) * PB;
#pragma unroll
            for (int u = 0; u < 4; ++u)
                if (q0 + u * kFoldBlock < PB) s[u] += __ldcg(p + q0 + u * kFoldBlock);
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int q = q0 + u * kFoldBlock;
            if (q < PB) {
                const int ij = q / ntiles, t = q - ij * ntiles;
                const int r = R * tile_i[t] + ij / R, c = R * tile_j[t] + ij % R;
                if (r <= K && c <= r && c < K) A[r * LD + c] = r == c ? s[u] + a.lambda : s[u];
            }
        }
    }
    __syncthreads();
    if (!fold_cholesky<T>(A, LD, K, invd, Pt, &flag)) {
        if (tid == 0) atomicOr(&a.req_status[req], 2);
        return;
    }
    T *y = A + K * LD;
    fold_back<T>(A, LD, K, invd, y, red);
    for (int k = tid; k < K; k += kFoldBlock) a.out[(int64_t)req * K + k] = y[k];
    if (a.refine) {
        const int LF = fold_fac_ld(K), V = 16 / (int)sizeof(T), nv = LF / V;
        T *f = a.fac + (int64_t)(req - a.req0) * K * LF;
        using Q = typename FoldVec<T>::type;
        for (int q = tid; q < K * nv; q += kFoldBlock) {
            const int r = q / nv, v = q - r * nv;
            if (v * V <= r)
                *reinterpret_cast<Q *>(f + r * LF + v * V) =
                    *reinterpret_cast<const Q *>(A + r * LD + v * V);
        }
    }
}

// Shared memory of k_fold_resid: the warps' sums (8 doubles per column), or the factor and
// the correction.
__host__ __device__ constexpr size_t fold_resid_smem(int K) {
    const size_t red = sizeof(double) * (size_t)8 * K;
    const size_t solve =
        sizeof(float) * ((size_t)K * fold_ld<float>(K) + 2 * 128 + 9 * (size_t)kFoldPanel);
    return red > solve ? red : solve;
}

// With |h| and |x| from here on (or zero), an error term lost below 2^-149 is at most 2^-69 of
// h x.
constexpr float kFoldLeast = 0x1p-40f;

// The warps' sums of h_e (x_e - h_e . x0) in FP64, lanes and columns as in k_fold_resid; x: the
// lane's columns of x0.
template <int R>
__device__ __noinline__ void fold_resid_f64(const FoldArgs<float> &a,
                                            const float (&x)[FoldCols<float, R>::N], int64_t b0,
                                            int64_t b1, double *sums) {
    using FC = FoldCols<float, R>;
    const int K = a.K, grp = threadIdx.x >> 3, g = threadIdx.x & 7;
    const bool vec = fold_vec<float, R>(K);
    double acc[FC::N];
#pragma unroll
    for (int j = 0; j < FC::N; ++j) acc[j] = 0.0;
    for (int64_t e0 = b0; e0 < b1; e0 += 32) {
        const bool valid = e0 + grp < b1;
        const int64_t es = valid ? e0 + grp : b0;
        double h[FC::N], dot = 0.0;
#pragma unroll
        for (int j = 0; j < FC::N; ++j) h[j] = 1.0;
        for (int t = 0; t < a.N - 1; ++t) {
            const int l = t < a.mode ? t : t + 1;
            float v[FC::N];
            FC::row(a.A[l] + (int64_t)a.other[es * (a.N - 1) + t] * K, K, g, vec, v);
#pragma unroll
            for (int j = 0; j < FC::N; ++j) h[j] *= (double)v[j];
        }
#pragma unroll
        for (int j = 0; j < FC::N; ++j)
            if (FC::col(j, g, vec) < K) dot += h[j] * (double)x[j];
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) dot += __shfl_xor_sync(0xFFFFFFFFu, dot, o);
        const double rho = (double)a.x[es] - dot;
        if (valid)
#pragma unroll
            for (int j = 0; j < FC::N; ++j) acc[j] += h[j] * rho;
    }
#pragma unroll
    for (int j = 0; j < FC::N; ++j) {
        const int c = FC::col(j, g, vec);
#pragma unroll
        for (int o = 8; o < 32; o <<= 1) acc[j] += __shfl_xor_sync(0xFFFFFFFFu, acc[j], o);
        if ((grp & 3) == 0 && c < K) sums[(grp >> 2) * K + c] = acc[j];
    }
}

template <int R, int NO>
__global__ void __launch_bounds__(kFoldBlock) k_fold_resid(const FoldArgs<float> a) {
    using FC = FoldCols<float, R>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ int flag;
    const int tid = threadIdx.x, K = a.K;
    const int blk = a.blk0 + blockIdx.x, req = a.blk_req[blk];
    if (a.req_status[req] != 0) return;  // bad index or pivot: every block of it leaves
    const bool vec = fold_vec<float, R>(K);
    const float *x0 = a.out + (int64_t)req * K;
    double *sums = reinterpret_cast<double *>(smem_raw);
    const int64_t b0 = a.blk_range[2 * blk], b1 = a.blk_range[2 * blk + 1];
    const int grp = tid >> 3, g = tid & 7;
    const int no = NO > 0 ? NO : a.N - 1;
    float x[FC::N];
#pragma unroll
    for (int j = 0; j < FC::N; ++j) {
        const int c = FC::col(j, g, vec);
        x[j] = c < K ? x0[c] : 0.f;
    }
    FloatPair acc[FC::N];
    bool lost = false;  // a product or value outside the pairs' range
#pragma unroll
    for (int j = 0; j < FC::N; ++j) acc[j].h = acc[j].l = 0.f;
    for (int64_t e0 = b0; e0 < b1; e0 += 32) {
        const int64_t e = e0 + grp;
        const bool valid = e < b1;
        // h of the entry as pairs; an idle group works on entry b0 and adds nothing
        const int64_t es = valid ? e : b0;
        FloatPair h[FC::N];
#pragma unroll
        for (int j = 0; j < FC::N; ++j) h[j].h = 1.f, h[j].l = 0.f;
#pragma unroll(NO > 0 ? NO : 1)
        for (int t = 0; t < no; ++t) {
            const int l = t < a.mode ? t : t + 1;
            const int32_t idx = a.other[es * (a.N - 1) + t];  // checked by k_fold_gram
            float v[FC::N];
            FC::row(a.A[l] + (int64_t)idx * K, K, g, vec, v);
#pragma unroll
            for (int j = 0; j < FC::N; ++j) {
                if (t == 0) {
                    h[j].h = v[j];
                    lost = lost || (no == 1 && fabsf(v[j]) < kFoldLeast && v[j] != 0.f);
                } else {
                    const float before = h[j].h;
                    h[j] = pair_mul(h[j], v[j]);
                    lost = lost || (fabsf(h[j].h) < kFoldLeast && before != 0.f && v[j] != 0.f);
                }
            }
        }
        const float xe = a.x[es];
        lost = lost || (fabsf(xe) < kFoldLeast && xe != 0.f);
        FloatPair dot = {0.f, 0.f};
#pragma unroll
        for (int j = 0; j < FC::N; ++j)
            if (FC::col(j, g, vec) < K) {
                const FloatPair p = pair_mul(h[j], x[j]);
                pair_add(dot, p.h, p.l);
            }
        dot = pair_group_sum(dot, 8, 0xFFFFFFFFu);
        FloatPair rho;
        rho.h = two_sum(xe, -dot.h, rho.l);
        rho.l = __fsub_rn(rho.l, dot.l);
        if (valid)
#pragma unroll
            for (int j = 0; j < FC::N; ++j) {
                FloatPair p = pair_mul(h[j], rho.h);
                p.l = __fmaf_rn(h[j].h, rho.l, p.l);
                pair_add(acc[j], p.h, p.l);
            }
    }
#pragma unroll
    for (int j = 0; j < FC::N; ++j)
        lost = lost || !(fabsf(acc[j].h) + fabsf(acc[j].l) < INFINITY);
    if (!__syncthreads_or(lost)) {
#pragma unroll
        for (int j = 0; j < FC::N; ++j) {
            // the warp's four groups, still as pairs; then one row of doubles per warp
            const int c = FC::col(j, g, vec);
#pragma unroll
            for (int o = 8; o < 32; o <<= 1)
                pair_add(acc[j], __shfl_xor_sync(0xFFFFFFFFu, acc[j].h, o),
                         __shfl_xor_sync(0xFFFFFFFFu, acc[j].l, o));
            if ((grp & 3) == 0 && c < K)
                sums[(grp >> 2) * K + c] = (double)acc[j].h + (double)acc[j].l;
        }
    } else {
        fold_resid_f64<R>(a, x, b0, b1, sums);
    }
    __syncthreads();
    for (int k = tid; k < K; k += kFoldBlock) {
        double s = 0.0;
        for (int w = 0; w < 8; ++w) s += sums[w * K + k];
        a.rpart[(int64_t)blockIdx.x * K + k] = s;
    }
    const int bb = a.req_blk[req], be = a.req_blk[req + 1];
    if (!fold_last_block(a.req_count + a.n_req + req, be - bb, &flag)) return;

    const int LD = fold_ld<float>(K), LF = fold_fac_ld(K), nv = LF / 4;
    float *A = reinterpret_cast<float *>(smem_raw), *d = A + K * LD, *invd = d + 128,
          *red = invd + 128;
    const float *f = a.fac + (int64_t)(req - a.req0) * K * LF;
    for (int q = tid; q < K * nv; q += kFoldBlock) {
        const int r = q / nv, v = q - r * nv;
        if (4 * v <= r)
            *reinterpret_cast<float4 *>(A + r * LD + 4 * v) =
                *reinterpret_cast<const float4 *>(f + r * LF + 4 * v);
    }
    for (int k = tid; k < K; k += kFoldBlock) {
        double s = 0.0;
        for (int b = bb; b < be; ++b) s += __ldcg(a.rpart + (int64_t)(b - a.blk0) * K + k);
        d[k] = (float)(s - (double)a.lambda * (double)x0[k]);
    }
    __syncthreads();
    for (int k = tid; k < K; k += kFoldBlock) invd[k] = 1.f / A[k * LD + k];
    __syncthreads();
    fold_forward<float>(A, LD, K, invd, d, red);
    fold_back<float>(A, LD, K, invd, d, red);
    for (int k = tid; k < K; k += kFoldBlock) a.out[(int64_t)req * K + k] = x0[k] + d[k];
}

template <class T, int R, int NO>
void launch_foldin_edge(const FoldArgs<T> &a, int blocks, cudaStream_t st) {
    const size_t smem = fold_gram_smem<T, R>(a.K);
    TFS_CUDA(raise_smem_limit((const void *)k_fold_gram<T, R, NO>, (int)smem));
    k_fold_gram<T, R, NO><<<blocks, kFoldBlock, smem, st>>>(a);
    TFS_CUDA(cudaGetLastError());
    if constexpr (sizeof(T) == 4) {
        if (a.refine) {
            const size_t rs = fold_resid_smem(a.K);
            TFS_CUDA(raise_smem_limit((const void *)k_fold_resid<R, NO>, (int)rs));
            k_fold_resid<R, NO><<<blocks, kFoldBlock, rs, st>>>(a);
            TFS_CUDA(cudaGetLastError());
        }
    }
}

}  // namespace

bool foldin_tiled_ok(int K) { return K + 1 <= 128; }

// Blocks of a request of m entries: 64 entries each up to 1,024 (a lone request then spreads
// over up to 16 SMs), 256 beyond (fewer partial systems to write and sum): up to 370 KB of
// partial systems a request of 1,024 entries at K = 100.  A request
// without entries has one empty block, which solves lambda I x = 0.
int foldin_plan_blocks(const int64_t *offsets, int n_req, std::vector<int64_t> &blk_range,
                       std::vector<int32_t> &blk_req, std::vector<int32_t> &req_blk) {
    blk_range.clear();
    blk_req.clear();
    req_blk.assign((size_t)n_req + 1, 0);
    for (int r = 0; r < n_req; ++r) {
        req_blk[r] = (int32_t)blk_req.size();
        const int64_t m = offsets[r + 1] - offsets[r], step = m <= 1024 ? 64 : 256;
        int64_t b = offsets[r];
        do {
            blk_range.push_back(b);
            blk_range.push_back(std::min<int64_t>(b + step, offsets[r + 1]));
            blk_req.push_back(r);
            b += step;
        } while (b < offsets[r + 1]);
    }
    req_blk[n_req] = (int32_t)blk_req.size();
    return (int)blk_req.size();
}

size_t foldin_part_elems(int K, int blocks) {
    return (size_t)std::max(blocks, 1) * (size_t)fold_tiles(K) * fold_edge(K) * fold_edge(K);
}

template <class T>
void launch_foldin_tiled(const FoldArgs<T> &a, int blocks, cudaStream_t st) {
    if (blocks <= 0) return;
    const bool two = a.N == 3;  // two other modes: the loop over them unrolled
    switch (fold_edge(a.K)) {
        case 2:
            two ? launch_foldin_edge<T, 2, 2>(a, blocks, st) : launch_foldin_edge<T, 2, 0>(a, blocks, st);
            return;
        case 4:
            two ? launch_foldin_edge<T, 4, 2>(a, blocks, st) : launch_foldin_edge<T, 4, 0>(a, blocks, st);
            return;
        default:
            two ? launch_foldin_edge<T, 8, 2>(a, blocks, st) : launch_foldin_edge<T, 8, 0>(a, blocks, st);
            return;
    }
}

size_t foldin_refine_elems(int K, int blocks, int n_req, size_t *fac_elems) {
    *fac_elems = (size_t)std::max(n_req, 1) * (size_t)K * fold_fac_ld(K);
    return (size_t)std::max(blocks, 1) * (size_t)K;
}

template <class T>
size_t foldin_smem_bytes(int K) {
    return sizeof(T) * ((size_t)K * K + K + (size_t)kTileE * K + kTileE);
}

template <class T>
void launch_foldin(const FoldArgs<T> &a, cudaStream_t st) {
    const size_t smem = foldin_smem_bytes<T>(a.K);
    TFS_CUDA(raise_smem_limit((const void *)k_foldin<T>, (int)smem));
    k_foldin<T><<<1, kFoldThreads, smem, st>>>(a);
    TFS_CUDA(cudaGetLastError());
}

template size_t foldin_smem_bytes<float>(int);
template size_t foldin_smem_bytes<double>(int);
template void launch_foldin<float>(const FoldArgs<float> &, cudaStream_t);
template void launch_foldin<double>(const FoldArgs<double> &, cudaStream_t);
template void launch_foldin_tiled<float>(const FoldArgs<float> &, int, cudaStream_t);
template void launch_foldin_tiled<double>(const FoldArgs<double> &, int, cudaStream_t);

}  // namespace tfs

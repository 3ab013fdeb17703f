// Per-split and per-sweep helper kernels: slice packing (the C columns of a split,
// Theorem 3's "only C columns need to be resident"), residual reconstruction and
// loss reduction (Eq. 1, accumulated in double in a fixed order), residual
// initialisation (Section 3.1) and the default factor initialisation (Algorithm 1).
#include <math.h>

#include <algorithm>

#include <map>
#include <mutex>

#include <type_traits>

#include "float_pair.cuh"
#include "sweep.cuh"

namespace tfs {

cudaError_t raise_smem_limit(const void *kern, int bytes) {
    static std::mutex mu;
    static std::map<std::pair<int, const void *>, int> limit;  // (device, kernel) -> bytes
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    std::lock_guard<std::mutex> g(mu);
    int &cur = limit[{dev, kern}];
    if (bytes <= cur) return cudaSuccess;
    e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    if (e == cudaSuccess) cur = bytes;
    return e;
}

int pick_cm(int C) {
    static const int cms[] = {1, 2, 4, 6, 8, 10, 12, 16};
    for (int cm : cms)
        if (C <= cm) return cm;
    if (wide_tile_width(C) > 0) return (C + 3) / 4 * 4;
    return 0;
}

namespace {

constexpr int kResThreads = 256;

// Slice pack of a split: one thread per (slice row, column), so that a row's regions are
// written by neighbouring lanes.  Bound: the factor rows are read a column (one 32-byte
// sector) at a time.  Regions are CM = off_prev wide; columns beyond C (cur, old) and Cq
// (prev) are zero, so products over a full region need no column mask.  Within a sweep the
// previous split's final values are the slice's own cur region (prev_in_cur), read as they
// lie instead of column by column from the factors.  201,000 rows, C = 10, K = 100: 64 us
// with a thread per row.
constexpr int kPackThreads = 256;

template <class T>
__global__ void __launch_bounds__(kPackThreads) k_pack(const PackArgs<T> a) {
    __shared__ uint32_t mx[kMaxModes * kGateCols];
    const int CM = a.off_prev, rows = kPackThreads / CM;
    const int w = (int)threadIdx.x / CM, c = (int)threadIdx.x - w * CM;
    if (a.mx) {
        for (int q = threadIdx.x; q < a.N * kGateCols; q += kPackThreads) mx[q] = 0u;
        __syncthreads();
    }
    int l = 0;
    uint32_t most = 0u;  // of this thread's column in mode l
    for (int64_t r = (int64_t)blockIdx.x * rows + w; w < rows && r < a.row_base[a.N];
         r += (int64_t)gridDim.x * rows) {
        while (r >= a.row_base[l + 1]) {
            if (a.mx && most) atomicMax(&mx[l * kGateCols + c], most);
            most = 0u;
            ++l;
        }
        const int64_t i = r - a.row_base[l];  // slice row (rank)
        const T *Ar = a.A[l] + (int64_t)a.id_of[l][i] * a.K;
        T *z = a.Z[l] + i * a.W;
        const T v = c < a.C ? Ar[a.S[c]] : T(0);
        const T p = c >= a.Cq ? T(0) : (a.prev_in_cur ? z[c] : Ar[a.Q[c]]);
        z[c] = v;
        z[a.off_old + c] = v;
        z[CM + c] = p;
        if (a.mx) most = max(most, __float_as_uint((float)v) & 0x7FFFFFFFu);
    }
    if (!a.mx) return;
    if (most) atomicMax(&mx[l * kGateCols + c], most);
    __syncthreads();
    for (int q = threadIdx.x; q < a.N * kGateCols; q += kPackThreads)
        record_max(a.mx + q, __uint_as_float(mx[q]));
}

template <class T>
__global__ void __launch_bounds__(kResThreads) k_init_res(const InitArgs<T> a) {
    const int lane = threadIdx.x & 31;
    const int bin = (int)(((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5);
    if (bin >= a.P) return;
    for (int64_t it = a.bin_ptr[bin]; it < a.bin_ptr[bin + 1]; ++it) {
        const tf_item item = a.items[it];
        const T *An = a.An + (int64_t)item.row * a.K;
        const int64_t jend = item.begin + item.len;
        for (int64_t j = item.begin + lane; j < jend; j += kWarp) {
            T model = T(0);
            if (!a.model_zero) {
                for (int k = 0; k < a.K; ++k) {
                    T q = An[k];
                    for (int t = 0; t < a.N - 1; ++t)
                        q *= a.Ao[t][(int64_t)a.id_o[t][a.oidx[t][j]] * a.K + k];
                    model += q;
                }
            }
            a.res[j] = a.x[a.perm[j]] - model;
        }
    }
}

// Sum of squares of a factor matrix, each row weighted by its entries if off is given; one
// double per block.  Float values: squares and sums as pairs of floats (float_pair.cuh; in
// FP64 the conversions and sums bound it), a double taking the pair after every eight values: a
// pair's low word rounds at its own size, so a chain of 2,000 equal values was 2^-33 off its
// sum, where eight at a time is 2^-47 and FP64 throughout 2^-44.  The FP64 form remains for a
// thread whose largest value lies outside 2^-40 .. 2^50.  Without weights the matrix is one
// flat array; with them a thread takes a row at a time.
constexpr int kPairChain = 8;

template <class T>
__device__ __forceinline__ double sum_squares(const T *p, int64_t n, int64_t first, int64_t step) {
    double s = 0.0;
    if constexpr (sizeof(T) == 4) {
        float big = 0.f;
        for (int64_t i = first; i < n; i += kPairChain * step) {
            float v[kPairChain];
#pragma unroll
            for (int u = 0; u < kPairChain; ++u) v[u] = i + u * step < n ? p[i + u * step] : 0.f;
            FloatPair acc = {0.f, 0.f};
#pragma unroll
            for (int u = 0; u < kPairChain; ++u) {
                FloatPair q;
                q.h = two_prod(v[u], v[u], q.l);
                pair_add(acc, q.h, q.l);
                big = fmaxf(big, fabsf(v[u]));
            }
            s += (double)acc.h + (double)acc.l;
        }
        if (big == 0.f || (big > 0x1p-40f && big < 0x1p50f && s == s)) return s;
        s = 0.0;
    }
    for (int64_t i = first; i < n; i += step) s += (double)p[i] * (double)p[i];
    return s;
}

template <class T>
__global__ void __launch_bounds__(kResThreads) k_reg(const T *A, int64_t I, int K,
                                                     const int64_t *off, double *block_out) {
    __shared__ double wsum[kResThreads / kWarp];
    const int64_t first = (int64_t)blockIdx.x * blockDim.x + threadIdx.x,
                  step = (int64_t)gridDim.x * blockDim.x;
    double acc = 0.0;
    if (off) {
        for (int64_t i = first; i < I; i += step)
            acc += sum_squares(A + i * K, K, 0, 1) * (double)(off[i + 1] - off[i]);
    } else {
        acc = sum_squares(A, I * K, first, step);
    }
    acc = warp_sum_d(acc);
    if ((threadIdx.x & 31) == 0) wsum[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x == 0) {
        double s = 0.0;
        for (int w = 0; w < kResThreads / kWarp; ++w) s += wsum[w];
        block_out[blockIdx.x] = s;
    }
}

// Sum of n doubles in a fixed order, one block: 97,000 item sums took 104 us with 256 threads
// and one load in flight each.
constexpr int kSumThreads = 1024;

__global__ void __launch_bounds__(kSumThreads) k_sum_blocks(const double *in, int n, double *out) {
    constexpr int U = 8;
    __shared__ double sh[kSumThreads];
    double s = 0.0;
    for (int64_t i = threadIdx.x; i < n; i += U * kSumThreads) {
        double v[U];
#pragma unroll
        for (int u = 0; u < U; ++u) v[u] = i + u * kSumThreads < n ? in[i + u * kSumThreads] : 0.0;
#pragma unroll
        for (int u = 0; u < U; ++u) s += v[u];
    }
    sh[threadIdx.x] = s;
    __syncthreads();
    for (int w = blockDim.x / 2; w > 0; w >>= 1) {
        if ((int)threadIdx.x < w) sh[threadIdx.x] += sh[threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x == 0) *out = sh[0];
}

__device__ __forceinline__ uint64_t mix64(uint64_t z) {
    z += 0x9E3779B97F4A7C15ull;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}

// Box-Muller from two counter-based uniforms per element.  Float factors take 24-bit
// uniforms and float arithmetic (FP64 transcendentals run at a small fraction of the
// FP32 rate on this GPU and made the draw a millisecond per 1e7 values).
template <class T>
__global__ void k_init_normal(T *A, int64_t count, uint64_t key, double std) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= count) return;
    if constexpr (std::is_same<T, float>::value) {
        const float u1 = (float)(mix64(key + 2 * (uint64_t)i) >> 40) * 0x1.0p-24f;
        const float u2 = (float)(mix64(key + 2 * (uint64_t)i + 1) >> 40) * 0x1.0p-24f;
        A[i] = (float)std * sqrtf(-2.0f * log1pf(-u1)) * cospif(2.0f * u2);
    } else {
        const double u1 = (double)(mix64(key + 2 * (uint64_t)i) >> 11) * 0x1.0p-53;
        const double u2 = (double)(mix64(key + 2 * (uint64_t)i + 1) >> 11) * 0x1.0p-53;
        A[i] = (T)(std * sqrt(-2.0 * log1p(-u1)) * cospi(2.0 * u2));
    }
}

// Model values: LP lanes per coordinate, lanes over the K columns.  Float contexts carry the
// products and the sum as pairs of floats (float_pair.cuh), double contexts in FP64.
//   Bound: gathering the factor rows (N rows of K values per coordinate, mostly from L2).
//   The former form, a warp per coordinate with FP64 products and sums, was bound by the
//   FP64 unit (three conversions, two products and a sum per column at 1/64 of the FP32
//   rate) and left 22% of its lanes idle at K = 100.  8 lanes per coordinate with 16-byte
//   loads take four steps at K = 100.  3,000,017 coordinates, N = 3,
//   K = 100 on GB300: 6.11 ms before, 0.41 ms now
//   (8.8 TB/s of gathered rows).
// A pair loses bits where a product or its error leaves the float range, and a sum of pairs
// keeps (n 2^-24)^2 of the terms' magnitudes at worst, n additions in a chain (Ogita, Rump and
// Oishi; 2^-46 is usual), where FP64 keeps 2^-53.  So a coordinate is formed again in FP64 whose
// values reach a.big (2^(56 / (N - 1)): no product overflows), whose sum is below 2^-40 or not
// finite, or whose terms' magnitudes are more than a.cancel = 2^21 / n^2 of it: up to there the
// worst error is an eighth of the result's rounding (n = 10 at K = 100: 3 of 10,000 coordinates
// with terms of random sign are formed again).  A sum all of whose terms have a zero factor
// (rows without entries solve to zero) is exact as it is, which a second look at the factors
// shows where the magnitudes' sum is zero: with 30% of the rows of one mode zero 0.49 ms, and
// 3.39 when those took the FP64 form too.
template <class T>
struct PredictVec;
template <>
struct PredictVec<float> {
    using type = float4;
};
template <>
struct PredictVec<double> {
    using type = double2;
};

// One coordinate in FP64 by the whole warp (c the same in every lane): eight lanes took 6 us of
// a batch of 3,000 for the few coordinates that come here.
template <class T, int NM>
__device__ __forceinline__ double predict_f64(const PredictArgs<T> &a, const int32_t *c, int lane) {
    const int N = NM > 0 ? NM : a.N;
    double s = 0.0;
    for (int k = lane; k < a.K; k += 32) {
        double p = 1.0;
#pragma unroll(NM > 0 ? NM : 1)
        for (int n = 0; n < N; ++n) p *= (double)a.A[n][(int64_t)c[n] * a.K + k];
        s += p;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xFFFFFFFFu, s, o);
    return s;
}

// NM: number of modes when it is a compile-time constant (rows of all modes loaded
// together), 0 for any; VEC: 16-byte loads (K a multiple of the vector).
template <class T, int LP, int NM, bool VEC>
__global__ void __launch_bounds__(256) k_predict(const PredictArgs<T> a) {
    constexpr int V = VEC ? 16 / (int)sizeof(T) : 1;
    constexpr unsigned kGroup = LP == 32 ? 0xFFFFFFFFu : (1u << LP) - 1u;
    const int lane = threadIdx.x & 31, sub = lane & (LP - 1), first = lane - sub;
    const int64_t e = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) / LP;
    const unsigned mask = kGroup << first;
    const int N = NM > 0 ? NM : a.N;
    const int32_t *c = a.coords + e * a.N;
    const bool there = e < a.m;
    bool ok = there;
    const T *row[NM > 0 ? NM : 1];
#pragma unroll(NM > 0 ? NM : 1)
    for (int n = 0; n < N; ++n) {
        const int32_t i = there ? c[n] : 0;
        ok = ok && i >= 0 && i < a.I[n];
        if (NM > 0) row[NM > 0 ? n : 0] = a.A[n] + (int64_t)i * a.K;
    }
    if (there && !ok && sub == 0) {
        a.out[e] = T(0);
        atomicOr(&a.stat->bits, kStatPredictRange);
    }
    auto load = [&](int n, int k, T (&v)[V]) {
        const T *p = (NM > 0 ? row[NM > 0 ? n : 0] : a.A[n] + (int64_t)c[n] * a.K) + k;
        if constexpr (VEC) {
            using Q = typename PredictVec<T>::type;
            const Q q = __ldg(reinterpret_cast<const Q *>(p));
            const T *w = reinterpret_cast<const T *>(&q);
#pragma unroll
            for (int u = 0; u < V; ++u) v[u] = w[u];
        } else {
            v[0] = __ldg(p);
        }
    };
    if constexpr (sizeof(T) == 4) {
        FloatPair sum[V];
        float big = 0.f, mag = 0.f;  // largest factor, sum of the terms' magnitudes
        const int K = ok ? a.K : 0;
#pragma unroll
        for (int u = 0; u < V; ++u) sum[u].h = sum[u].l = 0.f;
        // (few steps at once: the other warps hide the loads, and the registers of four steps'
        // rows leave fewer of them: 3e6 coordinates, K = 100 / 64 / 25: 0.41 / 0.29 / 0.24 ms,
        // with four steps 0.66 / 0.37 / 0.29)
#pragma unroll(VEC ? 1 : 2)
        for (int k = sub * V; k < K; k += LP * V) {
            T v[V];
            FloatPair p[V];
            load(0, k, v);
#pragma unroll
            for (int u = 0; u < V; ++u) {
                p[u].h = v[u], p[u].l = 0.f;
                big = fmaxf(big, fabsf(v[u]));
            }
#pragma unroll(NM > 0 ? NM : 1)
            for (int n = 1; n < N; ++n) {
                load(n, k, v);
#pragma unroll
                for (int u = 0; u < V; ++u) {
                    p[u] = pair_mul(p[u], v[u]);
                    big = fmaxf(big, fabsf(v[u]));
                }
            }
#pragma unroll
            for (int u = 0; u < V; ++u) pair_add(sum[u], p[u].h, p[u].l);
            if constexpr (V == 4)
                mag += (fabsf(p[0].h) + fabsf(p[1].h)) + (fabsf(p[2].h) + fabsf(p[3].h));
            else
                mag += fabsf(p[0].h);
        }
#pragma unroll
        for (int u = 1; u < V; ++u) pair_add(sum[0], sum[u].h, sum[u].l);
        const FloatPair s = pair_group_sum(sum[0], LP, mask);
#pragma unroll
        for (int o = LP / 2; o > 0; o >>= 1) mag += __shfl_xor_sync(mask, mag, o);
        float r = __fadd_rn(s.h, s.l);
        bool fine = big < a.big && fabsf(r) >= 0x1p-40f && fabsf(r) < 0x1p126f &&
                    mag <= a.cancel * fabsf(r);
        if (mag == 0.f) {  // zero factors, or products that vanished?
            fine = true;
            for (int k = sub * V; k < K; k += LP * V) {
                float v[V], least[V];
                load(0, k, least);
                for (int n = 1; n < N; ++n) {
                    load(n, k, v);
#pragma unroll
                    for (int u = 0; u < V; ++u) least[u] = fminf(fabsf(least[u]), fabsf(v[u]));
                }
#pragma unroll
                for (int u = 0; u < V; ++u) fine = fine && least[u] == 0.f;
            }
        }
        for (unsigned redo = __ballot_sync(0xFFFFFFFFu, !fine); redo;) {
            const int of = (__ffs(redo) - 1) & ~(LP - 1);  // the first group that asks for it
            const int64_t er = __shfl_sync(0xFFFFFFFFu, e, of);
            const double s64 = predict_f64<T, NM>(a, a.coords + er * a.N, lane);
            if (first == of) r = (float)s64;
            redo &= ~(kGroup << of);
        }
        if (ok && sub == 0) a.out[e] = r;
    } else {
        double s = 0.0;
        if (!ok) return;
#pragma unroll 4
        for (int k = sub * V; k < a.K; k += LP * V) {
            T v[V], p[V];
            load(0, k, p);
#pragma unroll(NM > 0 ? NM : 1)
            for (int n = 1; n < N; ++n) {
                load(n, k, v);
#pragma unroll
                for (int u = 0; u < V; ++u) p[u] *= v[u];
            }
#pragma unroll
            for (int u = 0; u < V; ++u) s += p[u];
        }
#pragma unroll
        for (int o = LP / 2; o > 0; o >>= 1) s += __shfl_xor_sync(mask, s, o);
        if (sub == 0) a.out[e] = s;
    }
}

template <class T, int LP, int NM>
void launch_predict_lanes(const PredictArgs<T> &a, cudaStream_t st) {
    const int64_t blocks = (a.m + 256 / LP - 1) / (256 / LP);
    if (a.K % (16 / (int)sizeof(T)) == 0)
        k_predict<T, LP, NM, true><<<(unsigned)blocks, 256, 0, st>>>(a);
    else
        k_predict<T, LP, NM, false><<<(unsigned)blocks, 256, 0, st>>>(a);
    TFS_CUDA(cudaGetLastError());
}

inline unsigned blocks_for(int64_t n, int threads) {
    return (unsigned)((n > 0 ? n : 1) + threads - 1) / threads;
}

}  // namespace

template <class T>
void launch_pack(const PackArgs<T> &a, cudaStream_t st) {
    const int64_t rows = a.row_base[a.N];
    if (rows <= 0) return;
    // with maxima few blocks, each over many rows: a block ends with up to N kGateCols atomics
    unsigned blocks = blocks_for(rows, kPackThreads / a.off_prev);
    if (a.mx) blocks = std::min(blocks, 1024u);
    k_pack<T><<<blocks, kPackThreads, 0, st>>>(a);
    TFS_CUDA(cudaGetLastError());
}

template <class T>
void launch_init_res(const InitArgs<T> &a, cudaStream_t st) {
    k_init_res<T><<<(unsigned)((a.P * kWarp + kResThreads - 1) / kResThreads), kResThreads, 0, st>>>(a);
    TFS_CUDA(cudaGetLastError());
}

template <class T>
void launch_reg(const T *A, int64_t I, int K, const int64_t *off, double *block_out, int blocks,
                cudaStream_t st) {
    k_reg<T><<<blocks, kResThreads, 0, st>>>(A, I, K, off, block_out);
    TFS_CUDA(cudaGetLastError());
}

void launch_sum_blocks(const double *in, int n, double *out, cudaStream_t st) {
    k_sum_blocks<<<1, kSumThreads, 0, st>>>(in, n, out);
    TFS_CUDA(cudaGetLastError());
}

template <class T>
void launch_predict(const PredictArgs<T> &a, cudaStream_t st) {
    if (a.m <= 0) return;
    PredictArgs<T> b = a;
    b.big = exp2f(56.f / (float)std::max(a.N - 1, 1));
    if (a.N == 1) b.big = INFINITY;  // no products
    // additions in a lane's chain, over its vector and over the lanes
    const int V = a.K % 4 == 0 ? 4 : 1;
    const float n = (float)((a.K + 8 * V - 1) / (8 * V) + V - 1 + 3);
    b.cancel = 0x1p21f / (n * n);
    if (a.N == 3)
        launch_predict_lanes<T, 8, 3>(b, st);
    else
        launch_predict_lanes<T, 8, 0>(b, st);
}

// Bfloat16 copy of a slice's columns, two values per thread (round to nearest even).
__global__ void k_slice_bf16(const float *__restrict__ Z, uint32_t *__restrict__ Zb, int64_t rows,
                             int W, int Wb, int col0, int npairs) {
    const int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= rows * npairs) return;
    const int64_t i = q / npairs;
    const int c = col0 + 2 * (int)(q - i * npairs);
    const float2 v = *reinterpret_cast<const float2 *>(Z + i * W + c);
    uint32_t packed;
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(packed) : "f"(v.y), "f"(v.x));
    Zb[(i * Wb + c) / 2] = packed;
}

void launch_slice_bf16(const float *Z, uint16_t *Zb, int64_t rows, int W, int Wb, int col0,
                       int ncols, cudaStream_t st) {
    if (rows <= 0 || ncols <= 0) return;
    if ((col0 | ncols | W | Wb) & 1) throw ApiError{TF_EINVAL, "bfloat16 slice copy: odd column"};
    const int npairs = ncols / 2;
    k_slice_bf16<<<blocks_for(rows * npairs, 256), 256, 0, st>>>(
        Z, reinterpret_cast<uint32_t *>(Zb), rows, W, Wb, col0, npairs);
    TFS_CUDA(cudaGetLastError());
}

template <class T>
void launch_init_normal(T *A, int64_t count, uint64_t seed, uint64_t stream_id, double std,
                        cudaStream_t st) {
    if (count <= 0) return;
    const uint64_t key = mix64_host(seed ^ mix64_host(stream_id + 0x51A5ull));
    k_init_normal<T><<<blocks_for(count, 256), 256, 0, st>>>(A, count, key, std);
    TFS_CUDA(cudaGetLastError());
}

#define TFS_INST(T)                                                                        \
    template void launch_pack<T>(const PackArgs<T> &, cudaStream_t);                       \
    template void launch_init_res<T>(const InitArgs<T> &, cudaStream_t);                   \
    template void launch_reg<T>(const T *, int64_t, int, const int64_t *, double *, int,   \
                                cudaStream_t);                                             \
    template void launch_init_normal<T>(T *, int64_t, uint64_t, uint64_t, double, cudaStream_t); \
    template void launch_predict<T>(const PredictArgs<T> &, cudaStream_t);
TFS_INST(float)
TFS_INST(double)
#undef TFS_INST

}  // namespace tfs

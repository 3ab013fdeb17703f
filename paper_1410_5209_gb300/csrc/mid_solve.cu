// Row solves of float contexts for subsets of 17 to 63 columns without solve options: one warp
// per row, the factor of [B + lambda I, c] in registers (lane i holds rows i and, past 31
// columns, i + 32; the right-hand side is row C, so the forward substitution comes with the
// factor), whose column j reaches the other lanes through shared memory as 16-byte broadcasts.
//
// Bound: the chain of C columns (pivot, broadcast, update: about 170 cycles each) with 12 warps
// per SM in flight, and issue: 1,300 packed FMAs and 520 broadcasts a row at C = 63.  The form it
// replaces (k_solve_wide, wide.cu, still used for wider subsets, FP64 and the solve options)
// walks a packed triangle in shared memory, two loads per multiply-add and a warp reduction
// per column: 50,021 rows at C = 50 took it 1.06 ms (0.60 here), 30,011 at C = 20 0.26 (0.062).
//   Precision: the products to take off an element are summed first and taken off once, as there.
// Taking each off the element (right-looking; 0.44 and 0.052 ms) rounds at the element's size
// every time: factors of a weighted-lambda fit 4.1e-7 / 6.1e-7 / 1.3e-6 off 64 bits, where this
// form and the old one are 2.7e-7 / 4.2e-7 / 7e-7 off.  Quotients by the pivot keep what its
// rounded inverse leaves (0.02 ms of 2.4; without it up to 8.8e-7).
//   Rows held by one item: four per block.  Split rows: one block each, whose threads first
// add the row's slots (or sums of kSlotGroup slots) in order, eight loads in flight each.
#include <algorithm>

#include "sweep.cuh"

namespace tfs {
namespace {

typedef unsigned long long u64;

constexpr int kMidThreads = 128;

__device__ __forceinline__ u64 mid_pack(float lo, float hi) {
    u64 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ float mid_get(u64 v, int hi) {
    float a, b;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
    return hi ? b : a;
}
__device__ __forceinline__ u64 mid_set(u64 v, int hi, float x) {
    return hi ? mid_pack(mid_get(v, 0), x) : mid_pack(x, mid_get(v, 1));
}
// a += l * m, two columns at once
__device__ __forceinline__ u64 mid_fma(u64 l, u64 m, u64 a) {
    u64 d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(l), "l"(m), "l"(a));
    return d;
}

// KM: columns held (C + 1 <= KM, a multiple of eight): 24 or 32 with one row per lane, up to 64
// with two.  The work grows with KM^2 and the unrolled code with it.
__host__ __device__ constexpr int mid_rows(int KM) { return KM <= 32 ? 1 : 2; }
// Row stride of the factor in shared memory: 16-byte stores one row per lane do not conflict.
__host__ __device__ constexpr int mid_ld(int KM) { return 32 * mid_rows(KM) + 4; }
// Per warp: the factor's rows (the packed system before), and two column buffers.
__host__ __device__ constexpr int mid_warp_floats(int KM) {
    return 32 * mid_rows(KM) * mid_ld(KM) + 64 * mid_rows(KM);
}

// Solves the system whose packed lower triangle is P[ntc] followed by the right-hand side [C]
// (shared memory, overwritten).  x0 / x1: the solution's values lane and lane + 32.
template <int KM>
__device__ __forceinline__ bool mid_solve(float *P, float *col, int C, float lam, int lane,
                                          float &x0, float &x1) {
    constexpr int R = mid_rows(KM), LD = mid_ld(KM);
    constexpr int K0 = KM < 32 ? KM : 32;
    const int ntc = C * (C + 1) / 2;
    for (int i = lane; i < C; i += 32) P[i * (i + 1) / 2 + i] += lam;
    __syncwarp();
    // Of rows lane (columns 0 .. 31) and lane + 32 (0 .. KM - 1), in pairs: the sums of products
    // that column j's elements will have taken off when it comes up (one subtraction at the
    // element's size, as in a left-looking factorisation, instead of one per column before it),
    // then L.  The elements themselves wait in shared memory: triangular numbers differ modulo
    // 32, so lanes reading column j do not conflict.  What is read past a row's end (the next
    // rows, the rest of the buffer) ends up above the diagonal, in columns from C on or in rows
    // past C, none of which reach the factor or the solution.
    const float *p0 = P + (lane < C ? lane * (lane + 1) / 2 : ntc);
    const float *p1 = P + (lane + 32 < C ? (lane + 32) * (lane + 33) / 2 : ntc);
    u64 a0[K0 / 2], a1[R == 2 ? KM / 2 : 1];
#pragma unroll
    for (int p = 0; p < K0 / 2; ++p) a0[p] = 0ull;
#pragma unroll
    for (int p = 0; p < (R == 2 ? KM / 2 : 1); ++p) a1[p] = 0ull;
    bool ok = true;
    float inv0 = 1.f, inv1 = 1.f, rest0 = 0.f, rest1 = 0.f;  // inverse pivots of the lane's rows
#pragma unroll
    for (int j = 0; j < KM - 1; ++j) {
        if (j < C) {
            float *c = col + (j & 1) * 32 * R;
            const float m0 = j < 32 ? p0[j] - mid_get(a0[j < K0 ? j / 2 : 0], j & 1) : 0.f;
            const float m1 = R == 2 ? p1[j] - mid_get(a1[R == 2 ? j / 2 : 0], j & 1) : 0.f;
            const float mine = j < 32 ? m0 : m1;
            float d = __shfl_sync(0xFFFFFFFFu, mine, j & 31);
            ok = ok && (d > 0.f);
            d = d > 0.f ? d : 1.f;
            // square roots and quotients by fused corrections (Markstein, "Computation of
            // elementary functions on the IBM RISC System/6000 processor", IBM J. Res. Dev. 34,
            // 1990): a quotient is the product with the pivot's inverse and with what that
            // leaves, since a rounded inverse alone would scale the whole column
            float root, inv;
            if (d > 0x1p-60f && d < 0x1p120f) {
                // d^1/2 and its inverse from the approximate d^-1/2 by one correction each,
                // where no step leaves the float range
                inv = rsqrtf(d);
                root = d * inv;
                root = fmaf(fmaf(-root, root, d), 0.5f * inv, root);
                inv = fmaf(inv, fmaf(-root, inv, 1.f), inv);
            } else {
                root = sqrtf(d);
                inv = 1.f / root;
            }
            const float rest = fmaf(-inv, root, 1.f) * inv;
            float l0 = 0.f, l1 = 0.f;
            if (j < 32) {
                l0 = lane == j ? root : fmaf(m0, inv, m0 * rest);
                if (lane == j) inv0 = inv, rest0 = rest;
                a0[j < K0 ? j / 2 : 0] = mid_set(a0[j < K0 ? j / 2 : 0], j & 1, l0);
                c[lane] = l0;
            }
            if constexpr (R == 2) {
                l1 = j >= 32 && lane == j - 32 ? root : fmaf(m1, inv, m1 * rest);
                if (j >= 32 && lane == j - 32) inv1 = inv, rest1 = rest;
                a1[j / 2] = mid_set(a1[j / 2], j & 1, l1);
                c[lane + 32] = l1;
            }
            __syncwarp();
            const u64 n0 = mid_pack(l0, l0), n1 = mid_pack(l1, l1);
#pragma unroll
            for (int q = 0; q < KM / 4; ++q) {
                if (4 * q + 3 > j) {
                    const float4 v = *reinterpret_cast<const float4 *>(c + 4 * q);
                    const float w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const int k = 4 * q + 2 * h;
                        if (k + 1 <= j) continue;
                        // column j itself is finished: its half of the pair takes no update
                        const u64 l = mid_pack(k > j ? w[2 * h] : 0.f, w[2 * h + 1]);
                        if (j < 32 && k < 32) a0[k < K0 ? k / 2 : 0] = mid_fma(l, n0, a0[k < K0 ? k / 2 : 0]);
                        if constexpr (R == 2) a1[k / 2] = mid_fma(l, n1, a1[k / 2]);
                    }
                }
            }
        }
    }
    // the factor's rows, L^-1 c as row C, over the system
    __syncwarp();
    float *L = P;
#pragma unroll
    for (int p = 0; p < K0 / 4; ++p)
        *reinterpret_cast<float4 *>(L + lane * LD + 4 * p) =
            make_float4(mid_get(a0[2 * p], 0), mid_get(a0[2 * p], 1), mid_get(a0[2 * p + 1], 0),
                        mid_get(a0[2 * p + 1], 1));
    if constexpr (R == 2) {
#pragma unroll
        for (int p = 0; p < KM / 4; ++p)
            *reinterpret_cast<float4 *>(L + (lane + 32) * LD + 4 * p) =
                make_float4(mid_get(a1[2 * p], 0), mid_get(a1[2 * p], 1), mid_get(a1[2 * p + 1], 0),
                            mid_get(a1[2 * p + 1], 1));
    }
    __syncwarp();
    float y0 = L[C * LD + lane], y1 = R == 2 ? L[C * LD + lane + 32] : 0.f;
    float s0 = 0.f, s1 = 0.f;  // sums to take off, as above
    x0 = x1 = 0.f;
#pragma unroll 4
    for (int j = C - 1; j >= 0; --j) {
        const float r0 = lane < j ? L[j * LD + lane] : 0.f;
        const float r1 = R == 2 && lane + 32 < j ? L[j * LD + lane + 32] : 0.f;
        const float m = R == 2 && j >= 32 ? y1 - s1 : y0 - s0;
        const float mine = R == 2 && j >= 32 ? fmaf(m, inv1, m * rest1) : fmaf(m, inv0, m * rest0);
        const float xj = __shfl_sync(0xFFFFFFFFu, mine, j & 31);
        if (lane == (j & 31)) {
            if (R == 2 && j >= 32)
                x1 = xj;
            else
                x0 = xj;
        }
        s0 += r0 * xj;
        s1 += r1 * xj;
    }
    return ok;
}

template <int KM>
__global__ void __launch_bounds__(kMidThreads) k_solve_mid(const PassArgs<float> a,
                                                           const SplitRow *split, int n_split,
                                                           const SplitRow *single, int n_single,
                                                           int CM, int W) {
    constexpr int R = mid_rows(KM);
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, C = a.C;
    const int NT = CM * (CM + 1) / 2, NB = NT + CM, ntc = C * (C + 1) / 2;
    float *P = reinterpret_cast<float *>(smem_raw) + warp * mid_warp_floats(KM);
    float *col = P + 32 * R * mid_ld(KM);
    SplitRow sr;
    if ((int)blockIdx.x < n_split) {
        sr = split[blockIdx.x];
        const int step = sr.n_slots > kSlotGroup ? kSlotGroup : 1;
        const float *src = a.partials + (int64_t)sr.first_slot * NB;
        float *sum = reinterpret_cast<float *>(smem_raw);  // the first warp's system
        for (int q = threadIdx.x; q < ntc + C; q += kMidThreads) {
            const float *p = src + (q < ntc ? q : NT + (q - ntc));
            float s = 0.f;
            for (int k = 0; k < sr.n_slots; k += 8 * step) {
                float v[8];
#pragma unroll
                for (int u = 0; u < 8; ++u)
                    v[u] = k + u * step < sr.n_slots ? p[(int64_t)(k + u * step) * NB] : 0.f;
#pragma unroll
                for (int u = 0; u < 8; ++u) s += v[u];
            }
            sum[q] = s;
        }
        __syncthreads();
        if (warp != 0) return;
    } else {
        const int r = ((int)blockIdx.x - n_split) * (kMidThreads / 32) + warp;
        if (r >= n_single) return;
        sr = single[r];
        // the slot's first C rows are the packed C-triangle; pairs are 8-byte aligned (NB and
        // NT are even for CM a multiple of four)
        const float *src = a.partials + (int64_t)sr.first_slot * NB;
#pragma unroll 8
        for (int q = 2 * lane; q < ntc; q += 64) {
            const unsigned dst = (unsigned)__cvta_generic_to_shared(P + q);
            if (q + 1 < ntc)
                asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(dst), "l"(src + q) : "memory");
            else
                asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(dst), "l"(src + q) : "memory");
        }
        for (int q = lane; q < C; q += 32) {
            const unsigned dst = (unsigned)__cvta_generic_to_shared(P + ntc + q);
            asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(dst), "l"(src + NT + q) : "memory");
        }
        asm volatile("cp.async.commit_group;\ncp.async.wait_group 0;\n" ::: "memory");
        __syncwarp();
    }
    const float lam = a.weighted ? a.lambda * (float)sr.len : a.lambda;
    float x0, x1;
    const bool ok = mid_solve<KM>(P, col, C, lam, lane, x0, x1);
    float *z = a.Zn + (int64_t)a.rank_n[sr.row] * W;
    float *Ar = a.A_n + (int64_t)sr.row * a.K;
    const bool in0 = lane < C, in1 = R == 2 && lane + 32 < C;
    if (!ok) {
        if (lane == 0) atomicAdd(&a.stat->singular_rows, 1ull);
        x0 = in0 ? z[lane] : 0.f;
        x1 = in1 ? z[lane + 32] : 0.f;
    } else {
        if (in0) {
            z[lane] = x0;
            Ar[a.S[lane]] = x0;
        }
        if (in1) {
            z[lane + 32] = x1;
            Ar[a.S[lane + 32]] = x1;
        }
    }
    if (a.mx_out) {
        if (in0) record_max(a.mx_out + lane, x0);
        if (in1) record_max(a.mx_out + lane + 32, x1);
    }
}

template <int KM>
void launch_solve_mid_km(const PassArgs<float> &a, const SplitRow *split, int n_split,
                         const SplitRow *single, int n_single, int CM, int W, cudaStream_t st) {
    constexpr int wpb = kMidThreads / 32;
    const size_t smem = sizeof(float) * wpb * (size_t)mid_warp_floats(KM);
    TFS_CUDA(raise_smem_limit((const void *)k_solve_mid<KM>, (int)smem));
    k_solve_mid<KM><<<n_split + (n_single + wpb - 1) / wpb, kMidThreads, smem, st>>>(
        a, split, n_split, single, n_single, CM, W);
    TFS_CUDA(cudaGetLastError());
}

}  // namespace

bool solve_mid_supported(int C, bool options) { return C <= 63 && !options; }

void launch_solve_mid(const PassArgs<float> &a, const SplitRow *split, int n_split,
                      const SplitRow *single, int n_single, int CM, int W, cudaStream_t st) {
    if (n_split + n_single <= 0) return;
    auto launch = a.C < 24   ? launch_solve_mid_km<24>
                  : a.C < 32 ? launch_solve_mid_km<32>
                  : a.C < 40 ? launch_solve_mid_km<40>
                  : a.C < 48 ? launch_solve_mid_km<48>
                  : a.C < 56 ? launch_solve_mid_km<56>
                             : launch_solve_mid_km<64>;
    launch(a, split, n_split, single, n_single, CM, W, st);
}

}  // namespace tfs

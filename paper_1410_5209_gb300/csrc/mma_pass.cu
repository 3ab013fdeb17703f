// Mode pass of float three-way tensors for column subsets of 17 to 63 columns (Eq. 4 with the
// lazy R-hat refresh of Algorithm 1): a warp per item, the Gram matrix H'^T H' of
// H' = [H | r_hat] on the tensor cores by mma.sync, with operands that never leave registers.
//
// Why this form.  Per entry the pass gathers two slice rows of up to three regions, forms C
// products and adds a C x C outer product.  The block-wide forms (wide.cu) build H' in shared
// memory for the Gram: at C = 50 about 190 warp instructions an entry (stores of both TF32
// halves one value at a time, two block barriers per 32 entries, an own-row load per column),
// issue-bound with the tensor pipe 17% busy.  In the m16n8k8 fragment layout lane 4 g + t
// holds row g (a feature) of columns t and t + 4 (entries), for A and B alike, and since the
// features may be numbered at will, lane 4 g + t takes features 32 q + 4 g + 0..3 of entries
// t and t + 4: one 16-byte load per region brings them, the eight lanes of an entry read 128
// bytes of its row, and the products are the A and the B fragments as they are.  No barrier,
// no shared memory until the end of an item, all of it left to the L1 cache for the gathers.
//
// Precision.  C <= 31: h = b1 + b2 + b3 in bfloat16 (24 bits), the six products of rank up to
// b1 b3; b1 b1 (16 bits) is summed apart from the rest, so that the tensor core, which truncates
// what it adds, has nothing to cut off there.  C >= 32 (two chunks, no registers for that):
// h = hi + lo in TF32, lo hi + hi lo + hi hi.  Either way the products of one step are summed
// from zero and added to FP32 sums with ordinary rounding.  With one chunk the right-hand side
// and B's diagonal are summed by FMAs on the same registers instead (no cost beside the loads:
// 0.14 ms a pass either way); over six seeds of a weighted-lambda fit at C = 20 the largest
// error of a factor against 64 bits is then 6.6e-7, with the diagonal on the tensor cores
// 2.0e-6, and 1.5e-6 with FP32 throughout.  With two chunks the FMAs' registers cost 0.2 ms of
// 1.6, and the errors are a third of FP32's without them (dispatch in api.cu).
//   Range.  Below 2^-100 the split of h would lose its last parts, and collapsed columns
// (weighted lambda) do get there.  The pack and the solves record the largest value of each of
// every mode's current columns (PassArgs::mx); a pass in which some column's product lies
// outside 2^-80 .. 2^60 and is not zero is left to the block-wide kernel, launched behind this
// one with the opposite gate (one of the two returns at once).  No cost beside one maximum
// over all columns (C = 20 and 50: solves and passes as they were, the pack 0.13 -> 0.08 ms).
#include <algorithm>

#include "entry_steps.h"
#include "sweep.cuh"

namespace tfs {
namespace {

typedef unsigned long long u64;

__device__ __forceinline__ float tf32_round(float x) {
    uint32_t r;
    asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(r) : "f"(x));
    return __uint_as_float(r);
}
// d = A B: the first product of a chain (no zeros to move into place)
__device__ __forceinline__ void mma8z(float (&d)[4], float a0, float a1, float a2, float a3, float b0,
                                      float b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k8.row.col.f32.tf32.tf32.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, "
        "{%8, %9}, {%10, %10, %10, %10};"
        : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
        : "r"(__float_as_uint(a0)), "r"(__float_as_uint(a1)), "r"(__float_as_uint(a2)),
          "r"(__float_as_uint(a3)), "r"(__float_as_uint(b0)), "r"(__float_as_uint(b1)), "f"(0.f));
}
// d += A B: A 16 x 8, B 8 x 8, TF32
__device__ __forceinline__ void mma8(float (&d)[4], float a0, float a1, float a2, float a3, float b0,
                                     float b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k8.row.col.f32.tf32.tf32.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, "
        "{%8, %9}, {%0, %1, %2, %3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(__float_as_uint(a0)), "r"(__float_as_uint(a1)), "r"(__float_as_uint(a2)),
          "r"(__float_as_uint(a3)), "r"(__float_as_uint(b0)), "r"(__float_as_uint(b1)));
}
__device__ __forceinline__ u64 add2(u64 a, float lo, float hi) {
    u64 b, d;
    asm("mov.b64 %0, {%1, %2};" : "=l"(b) : "f"(lo), "f"(hi));
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ u64 mul2(u64 a, u64 b) {
    u64 d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ u64 fma2(u64 a, u64 b, u64 c) {
    u64 d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ u64 pair(float x, float y) {
    u64 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(x), "f"(y));
    return r;
}
__device__ __forceinline__ void halves(u64 v, float &x, float &y) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(x), "=f"(y) : "l"(v));
}
// four columns of a row as two pairs, or zeros
__device__ __forceinline__ void ld4(const float *p, bool ok, u64 (&v)[2]) {
    ulonglong2 q = make_ulonglong2(0ull, 0ull);
    if (ok) q = *reinterpret_cast<const ulonglong2 *>(p);
    v[0] = q.x, v[1] = q.y;
}

// bfloat16 pair of (x, y), x in the lower half, and what it leaves of them
__device__ __forceinline__ uint32_t bf16_part(float &x, float &y) {
    uint32_t r;
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(y), "f"(x));
    x -= __uint_as_float(r << 16);
    y -= __uint_as_float(r & 0xFFFF0000u);
    return r;
}
// d += A B: A 16 x 16, B 16 x 8, bfloat16
__device__ __forceinline__ void mma16(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2,
                                      uint32_t a3, uint32_t b0, uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, "
        "{%8, %9}, {%0, %1, %2, %3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

__device__ __forceinline__ void mma16z(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2,
                                       uint32_t a3, uint32_t b0, uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, "
        "{%8, %9}, {%10, %10, %10, %10};"
        : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1), "f"(0.f));
}

// Entries per step: 16 (two halves of 8) for one chunk, 8 for two.
__host__ __device__ constexpr int mma_step(int CH) { return CH == 1 ? 16 : 8; }
__host__ __device__ constexpr int mma_tiles(int CH) { return 2 * CH * (2 * CH + 1); }
// Warps per block (one block per SM).  CH = 1: 16 at 128 registers (12: 0.29, 16: 0.28, 20:
// 0.32 ms for a mode's two passes at 5e6 entries, C = 20).  CH = 2: 8, whose 255 registers hold the 80 sums and
// a step's operands and loads without spilling (1e7 entries, C = 50: 12 warps 1.62 / 1.87 /
// 2.34, 10 warps 1.64 / 1.85 / 1.91, 8 warps 1.54 / 1.60 / 1.65 ms, each the pass that refreshes
// R-hat and the one that does not together).
__host__ __device__ constexpr int mma_warps(int CH) { return CH == 1 ? 16 : 8; }

// CH: 32-feature chunks (C < 32 CH; chunk features past C are zero).  FIRST: the split's
// first inner iteration; NLO other modes precede mode n (already updated in this split: their
// old columns differ from cur).  Lane 4 g + t works on entries t, t + 4 (and t + 8, t + 12: the
// second half of a 16-entry step); which of a step's entries is which index of the product's
// inner dimension does not matter.
template <int CH, bool FIRST, int NLO>
__global__ void __launch_bounds__(mma_warps(CH) * kWarp, 1)
    k_pass_mma(const PassArgs<float> a, int CM, int W) {
    constexpr int J = 4 * CH, TILES = mma_tiles(CH), NV = TILES * 4;
    constexpr int STEP = mma_step(CH), E = STEP / 4;  // entries per step and per lane
    if (!wide_gate(a)) return;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    uint16_t *place = reinterpret_cast<uint16_t *>(smem_raw);  // [NV][32]: value -> partial slot
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, g = lane >> 2, t = lane & 3;
    const int C = a.C, NT = CM * (CM + 1) / 2, NB = NT + CM;
    float *buf = reinterpret_cast<float *>(smem_raw + NV * 32 * sizeof(uint16_t)) +
                 warp * ((NB + 4) / 4 * 4);
    // Tile (m, n) holds the products of feature rows 2 m (values 0, 1) and 2 m + 1 (2, 3) with
    // feature column n, where row j of lane group g is feature 32 (j / 4) + 4 g + j % 4.  Each
    // pair is written once: tiles of row j < n, half of row j = n and padding go nowhere (NB).
    for (int q = threadIdx.x; q < NV * 32; q += blockDim.x) {
        const int l = q & 31, i = (q >> 5) & 3, tile = q >> 7;
        int m = 0;
        while ((m + 1) * (m + 2) <= tile) ++m;
        const int n = tile - m * (m + 1), j = 2 * m + (i >> 1);
        const int r = 32 * (j >> 2) + 4 * (l >> 2) + (j & 3);
        const int c = 32 * (n >> 2) + 4 * (2 * (l & 3) + (i & 1)) + (n & 3);
        const int hi = r > c ? r : c, lo = r > c ? c : r;
        int at = NB;
        if (j > n || (j == n && r >= c)) {
            if (hi < C && (CH > 1 || lo < hi))
                at = hi * (hi + 1) / 2 + lo;
            else if (CH > 1 && hi == C && lo < C)
                at = NT + lo;
        }
        place[q] = (uint16_t)at;
    }
    for (int q = lane; q < NB; q += 32) buf[q] = 0.f;  // rows and columns from C on stay zero
    __syncthreads();

    bool in[CH], inq[CH];  // the lane's columns of a chunk exist in this / the previous subset
    unsigned is_res = 0u;  // two chunks: bit j, the lane's feature j is column C of H' (r_hat)
#pragma unroll
    for (int q = 0; q < CH; ++q) {
        in[q] = 32 * q + 4 * g < CM;
        inq[q] = 32 * q + 4 * g < a.Cq;
#pragma unroll
        for (int u = 0; u < 4; ++u)
            if (CH > 1 && 32 * q + 4 * g + u == C) is_res |= 1u << (4 * q + u);
    }
    const float *Z0 = a.Zo[0] + 4 * g, *Z1 = a.Zo[1] + 4 * g;
    const int32_t *ix0 = a.oidx[0], *ix1 = a.oidx[1];
    u64 acc[TILES][2];
#pragma unroll
    for (int k = 0; k < TILES; ++k) acc[k][0] = acc[k][1] = 0ull;
    // one chunk: the lane's entries' part of the right-hand side and of B's diagonal, by feature
    constexpr int JF = CH == 1 ? J / 2 : 1;
    u64 csum[JF], dsum[JF];
#pragma unroll
    for (int j = 0; j < JF; ++j) csum[j] = dsum[j] = 0ull;
    u64 own_old[J / 2], own_prev[J / 2];  // own row: old columns, and prev ones negated
#pragma unroll
    for (int j = 0; j < J / 2; ++j) own_old[j] = own_prev[j] = 0ull;

    for (;;) {
        unsigned long long tk = 0;
        if (lane == 0) tk = atomicAdd(a.ticket, 1ull) - a.ticket_base;
        tk = __shfl_sync(0xFFFFFFFFu, tk, 0);
        if (tk >= (unsigned long long)a.P) break;
        int64_t it = a.bin_ptr[tk];
        const int64_t it_end = a.bin_ptr[tk + 1];
        if (it >= it_end) continue;
        tf_item item = a.items[it];
        int j0 = (int)item.begin, jend = (int)(item.begin + item.len);
        bool fresh = true;
        // indices and residuals of the lane's entries (t, t + 4, ...), one step ahead
        int32_t i0[E], i1[E];
        float rv[E];
        auto load_entries = [&](int j, int end, int32_t (&x0)[E], int32_t (&x1)[E], float (&r)[E]) {
#pragma unroll
            for (int e = 0; e < E; ++e) {
                x0[e] = x1[e] = -1;
                r[e] = 0.f;
                if (has_entry(j, t + 4 * e, end)) {
                    const int at = j + (t + 4 * e);
                    x0[e] = ix0[at];
                    x1[e] = ix1[at];
                    r[e] = a.res[at];
                }
            }
        };
        load_entries(j0, jend, i0, i1, rv);
        for (;;) {
            if (FIRST && fresh) {
                const float *z = a.Zn + (int64_t)a.rank_n[item.row] * W + 4 * g;
                const u64 sign = 0x8000000080000000ull;
#pragma unroll
                for (int q = 0; q < CH; ++q) {
                    u64 o[2], p[2];
                    ld4(z + CM + 32 * q, in[q], p);
                    ld4(z + 2 * CM + 32 * q, in[q], o);
#pragma unroll
                    for (int u = 0; u < 2; ++u) {
                        own_prev[2 * q + u] = p[u] ^ sign;
                        own_old[2 * q + u] = o[u];
                    }
                }
            }
            // the next step's entries
            const bool last = last_step(j0, STEP, jend);
            const bool more = !last || it + 1 < it_end;
            tf_item next = item;
            int nj = last ? jend : j0 + STEP, nend = jend;  // none after the bin's last step
            if (last && more) {
                next = a.items[it + 1];
                nj = (int)next.begin;
                nend = (int)(next.begin + next.len);
            }
            int32_t n0[E], n1[E];
            float nr[E];
            load_entries(nj, nend, n0, n1, nr);

            // products of this step
            float h[E][J], d[E];
#pragma unroll
            for (int e = 0; e < E; ++e) {
                const bool valid = i0[e] >= 0;
                const float *z0 = Z0 + (int64_t)(valid ? i0[e] : 0) * W;
                const float *z1 = Z1 + (int64_t)(valid ? i1[e] : 0) * W;
                u64 da = 0ull, db = 0ull;
#pragma unroll
                for (int q = 0; q < CH; ++q) {
                    u64 x0[2], x1[2];
                    const bool ok = valid && in[q], okq = valid && inq[q];
                    ld4(z0 + 32 * q, ok, x0);
                    ld4(z1 + 32 * q, ok, x1);
                    if (FIRST) {
                        u64 o0[2], o1[2], p0[2], p1[2];
                        if (NLO > 0) ld4(z0 + 2 * CM + 32 * q, ok, o0);
                        if (NLO > 1) ld4(z1 + 2 * CM + 32 * q, ok, o1);
                        ld4(z0 + CM + 32 * q, okq, p0);  // zero from Cq on
                        ld4(z1 + CM + 32 * q, okq, p1);
#pragma unroll
                        for (int u = 0; u < 2; ++u) {
                            da = fma2(own_old[2 * q + u],
                                      mul2(NLO > 0 ? o0[u] : x0[u], NLO > 1 ? o1[u] : x1[u]), da);
                            db = fma2(own_prev[2 * q + u], mul2(p0[u], p1[u]), db);
                        }
                    }
#pragma unroll
                    for (int u = 0; u < 2; ++u) {
                        halves(mul2(x0[u], x1[u]), h[e][4 * q + 2 * u], h[e][4 * q + 2 * u + 1]);
                    }
                }
                float s0, s1, r0, r1;
                halves(da, s0, s1);
                halves(db, r0, r1);
                d[e] = (s0 + s1) + (r0 + r1);
            }
            if (FIRST) {
#pragma unroll
                for (int o = 4; o < 32; o <<= 1)
#pragma unroll
                    for (int e = 0; e < E; ++e) d[e] += __shfl_xor_sync(0xFFFFFFFFu, d[e], o);
            }
#pragma unroll
            for (int e = 0; e < E; ++e) {
                const float v = FIRST ? rv[e] + d[e] : rv[e];
                if (FIRST && g == 0 && i0[e] >= 0) a.res[j0 + t + 4 * e] = v;
                if constexpr (CH == 1) {
                    const u64 vv = pair(v, v);
#pragma unroll
                    for (int j = 0; j < J / 2; ++j) {
                        const u64 hp = pair(h[e][2 * j], h[e][2 * j + 1]);
                        csum[j] = fma2(hp, vv, csum[j]);
                        dsum[j] = fma2(hp, hp, dsum[j]);
                    }
                } else {
#pragma unroll
                    for (int j = 0; j < J; ++j)
                        if ((is_res >> j) & 1u) h[e][j] = i0[e] >= 0 ? v : 0.f;
                }
            }
            if constexpr (CH == 1) {
                uint32_t b1[J][2], b2[J][2], b3[J][2];
#pragma unroll
                for (int j = 0; j < J; ++j)
#pragma unroll
                    for (int k = 0; k < 2; ++k) {
                        b1[j][k] = bf16_part(h[2 * k][j], h[2 * k + 1][j]);
                        b2[j][k] = bf16_part(h[2 * k][j], h[2 * k + 1][j]);
                        b3[j][k] = bf16_part(h[2 * k][j], h[2 * k + 1][j]);
                    }
#pragma unroll
                for (int m = 0; m < J / 2; ++m)
#pragma unroll
                    for (int n = 0; n < 2 * m + 2; ++n) {
                        float s[4], r[4];
                        const int j = 2 * m, k = m * (m + 1) + n;
                        auto mul = [&](float (&d)[4], uint32_t (&x)[J][2], uint32_t (&y)[J][2]) {
                            mma16(d, x[j][0], x[j + 1][0], x[j][1], x[j + 1][1], y[n][0], y[n][1]);
                        };
                        mma16z(s, b1[j][0], b1[j + 1][0], b1[j][1], b1[j + 1][1], b1[n][0], b1[n][1]);
                        mma16z(r, b3[j][0], b3[j + 1][0], b3[j][1], b3[j + 1][1], b1[n][0], b1[n][1]);
                        mul(r, b1, b3);
                        mul(r, b2, b2);
                        mul(r, b2, b1);
                        mul(r, b1, b2);
                        acc[k][0] = add2(acc[k][0], s[0] + r[0], s[1] + r[1]);
                        acc[k][1] = add2(acc[k][1], s[2] + r[2], s[3] + r[3]);
                    }
            } else {
                float lo[2][J];
#pragma unroll
                for (int e = 0; e < 2; ++e)
#pragma unroll
                    for (int j = 0; j < J; ++j) {
                        const float hi = tf32_round(h[e][j]);
                        lo[e][j] = tf32_round(h[e][j] - hi);
                        h[e][j] = hi;
                    }
#pragma unroll
                for (int m = 0; m < J / 2; ++m)
#pragma unroll
                    for (int n = 0; n < 2 * m + 2; ++n) {
                        float s[4];
                        const int j = 2 * m, k = m * (m + 1) + n;
                        mma8z(s, lo[0][j], lo[0][j + 1], lo[1][j], lo[1][j + 1], h[0][n], h[1][n]);
                        mma8(s, h[0][j], h[0][j + 1], h[1][j], h[1][j + 1], lo[0][n], lo[1][n]);
                        mma8(s, h[0][j], h[0][j + 1], h[1][j], h[1][j + 1], h[0][n], h[1][n]);
                        acc[k][0] = add2(acc[k][0], s[0], s[1]);
                        acc[k][1] = add2(acc[k][1], s[2], s[3]);
                    }
            }
            if (last) {  // the item's sums, through shared memory into its packed partial
#pragma unroll
                for (int k = 0; k < TILES; ++k)
#pragma unroll
                    for (int i = 0; i < 2; ++i) {
                        float x, y;
                        asm("mov.b64 {%0, %1}, %2;" : "=f"(x), "=f"(y) : "l"(acc[k][i]));
                        buf[place[(4 * k + 2 * i) * 32 + lane]] = x;
                        buf[place[(4 * k + 2 * i + 1) * 32 + lane]] = y;
                        acc[k][i] = 0ull;
                    }
                if constexpr (CH == 1) {
#pragma unroll
                    for (int j = 0; j < J; ++j) {  // the FMAs' sums over the lanes of a feature
                        const int f = 4 * g + j;
                        auto over_lanes = [&](u64 v) {
                            float x, y;
                            halves(v, x, y);
                            float c = j & 1 ? y : x;
                            c += __shfl_xor_sync(0xFFFFFFFFu, c, 1);
                            return c + __shfl_xor_sync(0xFFFFFFFFu, c, 2);
                        };
                        const float c = over_lanes(csum[j / 2]), b = over_lanes(dsum[j / 2]);
                        if (t == 0 && f < C) buf[NT + f] = c;
                        if (t == 1 && f < C) buf[f * (f + 1) / 2 + f] = b;
                    }
#pragma unroll
                    for (int j = 0; j < J / 2; ++j) csum[j] = dsum[j] = 0ull;
                }
                __syncwarp();
                float *p = a.partials + (int64_t)item.slot * NB;
                for (int q = lane; q < NB; q += 32) p[q] = buf[q];
                __syncwarp();
                if (!more) break;
                ++it;
            }
            fresh = last;
            item = next;
            j0 = nj;
            jend = nend;
#pragma unroll
            for (int e = 0; e < E; ++e) i0[e] = n0[e], i1[e] = n1[e], rv[e] = nr[e];
        }
    }
}

size_t mma_smem(int CH, int CM) {
    const size_t nb = (size_t)CM * (CM + 1) / 2 + CM;
    return (size_t)mma_tiles(CH) * 4 * 32 * sizeof(uint16_t) +
           sizeof(float) * (size_t)mma_warps(CH) * ((nb + 4) / 4 * 4);
}

template <int CH>
void launch_pass_mma_ch(const PassArgs<float> &a, int CM, int W, int grid, cudaStream_t st) {
    auto kern = !a.first ? k_pass_mma<CH, false, 0>
                         : (a.n == 0 ? k_pass_mma<CH, true, 0>
                                     : (a.n == 1 ? k_pass_mma<CH, true, 1> : k_pass_mma<CH, true, 2>));
    const size_t smem = mma_smem(CH, CM);
    TFS_CUDA(raise_smem_limit((const void *)kern, (int)smem));
    kern<<<grid, mma_warps(CH) * kWarp, smem, st>>>(a, CM, W);
    TFS_CUDA(cudaGetLastError());
}

}  // namespace

bool pass_mma_supported(int N, int C, int CM) { return N == 3 && std::max(C + 1, CM) <= 64; }

PassPlan pass_mma_plan(int C, int CM, int num_sms, int P) {
    PassPlan plan;
    plan.warps = mma_warps(std::max(C + 1, CM) <= 32 ? 1 : 2);
    plan.grid = std::max(1, std::min(num_sms, (P + plan.warps - 1) / plan.warps));
    return plan;
}

void launch_pass_mma(const PassArgs<float> &a, int CM, int W, int grid, cudaStream_t st) {
    if (std::max(a.C + 1, CM) <= 32)
        launch_pass_mma_ch<1>(a, CM, W, grid, st);
    else
        launch_pass_mma_ch<2>(a, CM, W, grid, st);
}

}  // namespace tfs

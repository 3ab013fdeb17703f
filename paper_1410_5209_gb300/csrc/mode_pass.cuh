// The fused mode pass of a SALS split (Algorithm 1, inner loop over rows; Eq. (4)),
// and the residual / loss pass that shares its gather machinery.
//
// One warp works through the items of one bin.  For an item (a row, or a chunk of a
// row split across bins) the warp walks the row's entries 32 at a time:
//   1. each lane reads its entry's N-1 other-mode indices and its residual-copy value
//      (coalesced streams);
//   2. the warp stages the 32 entries' packed slice rows of every other mode into
//      shared memory cooperatively: 16-byte vector loads, consecutive lanes covering
//      one row, so each gathered row costs one L1 wavefront instead of one per element;
//   3. each lane forms h = prod_{l != n} a^(l)_{i_l, S} (the Hadamard product of Eq. 4)
//      from shared memory, refreshes its residual copy to this split's R-hat on the
//      first inner iteration (Algorithm 1; done lazily per copy, see PassArgs) and
//      accumulates B += h h^T (lower triangle) and c += r_hat h in registers.
// The warp then sums B and c by halving exchanges and writes them to the item's slot.
// k_solve_rows sums the slots of each row in a fixed order and solves B + lambda I_C (lambda
// * |Omega_i| when weighted) by a register Cholesky (Section 3.1); the new C parameters go to
// the packed slice and to A^(n).
#pragma once

#include <algorithm>
#include <type_traits>

#include "entry_steps.h"
#include "sweep.cuh"

namespace tfs {

__host__ __device__ constexpr int tri(int i, int j) { return i * (i + 1) / 2 + j; }

template <class T>
struct Vec16;
template <>
struct Vec16<float> {
    using type = float4;
};
template <>
struct Vec16<double> {
    using type = double2;
};

// Compile-time geometry of the packed slices and of the shared-memory staging.
template <class T, int CM>
struct Geo {
    static constexpr int V = 16 / (int)sizeof(T);               // elements per 16-byte vector
    static constexpr int W = slice_stride_elems(CM, sizeof(T));  // slice row stride
    static constexpr int NV = W / V;                             // vectors per row (power of 2)
    static constexpr int RS = W + V;                             // staged row stride: odd in
                                                                 // vectors -> conflict-free
    static constexpr int NV_CUR = (CM + V - 1) / V;              // vectors covering cur
    static constexpr int NV_CP = (2 * CM + V - 1) / V;           // cur|prev
    static constexpr int NV_ALL = (3 * CM + V - 1) / V;          // cur|prev|old
    static constexpr int OFF_PREV = CM, OFF_OLD = 2 * CM;
    static constexpr int NT = CM * (CM + 1) / 2;
    static_assert((NV & (NV - 1)) == 0 && NV <= 32, "slice rows must be 2^k vectors");
};

// Reads elements [OFF, OFF + CNT) of a 16-byte aligned shared-memory row with vector
// loads (the covering vectors; all offsets are compile-time).
template <class T, int OFF, int CNT>
__device__ __forceinline__ void lds_range(T (&r)[CNT], const T *row) {
    constexpr int V = 16 / (int)sizeof(T);
    constexpr int v0 = OFF / V, v1 = (OFF + CNT - 1) / V;
    T tmp[(v1 - v0 + 1) * V];
#pragma unroll
    for (int k = v0; k <= v1; ++k) {
        if constexpr (sizeof(T) == 4) {
            const float4 v = reinterpret_cast<const float4 *>(row)[k];
            tmp[(k - v0) * 4 + 0] = v.x;
            tmp[(k - v0) * 4 + 1] = v.y;
            tmp[(k - v0) * 4 + 2] = v.z;
            tmp[(k - v0) * 4 + 3] = v.w;
        } else {
            const double2 v = reinterpret_cast<const double2 *>(row)[k];
            tmp[(k - v0) * 2 + 0] = v.x;
            tmp[(k - v0) * 2 + 1] = v.y;
        }
    }
#pragma unroll
    for (int e = 0; e < CNT; ++e) r[e] = tmp[OFF - v0 * V + e];
}

template <class T>
__device__ __forceinline__ T warp_sum(T v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, o);
    return v;
}

// v / pivot.  Float: the division.  Double: an FP64 division is a dozen instructions of the
// FP64 unit, which issues a warp's instruction over 64 cycles, so the pivot is inverted once
// per column and a quotient is the product with the rounded inverse, corrected by what it
// leaves of v (three instructions; Markstein, "Computation of elementary functions on the IBM
// RISC System/6000 processor", IBM J. Res. Dev. 34, 1990), which rounds as the division does.
// The product alone took factors of a weighted-lambda fit from 1.6e-17 to 1.2e-15 off 64-bit
// results.  Quotients that are zero, subnormal or not finite stay as the product gives them.
template <class T>
__device__ __forceinline__ T chol_over(T v, T pivot, T inverse) {
    if constexpr (sizeof(T) == 8) {
        const T q = v * inverse;
        const unsigned e = (unsigned)__double2hiint(q) & 0x7FF00000u;
        return e - 0x00100000u < 0x7FE00000u ? fma(fma(-q, pivot, v), inverse, q) : q;
    }
    return v / pivot;
}

// Cholesky factor, in place, of B + lam I for the leading C x C block of a CM x CM packed
// lower triangle; rows/columns >= C are replaced by the identity.  inv: inverses of the
// factor's diagonal (double only).  min_ratio receives the smallest pivot ratio d_j / (B_jj +
// lam) over the leading block (1 when perfectly conditioned, near 0 when a column is nearly a
// combination of the earlier ones).  Returns false when a pivot is <= 0.
template <class T, int CM>
__device__ __forceinline__ bool chol_factor(T (&B)[CM * (CM + 1) / 2], T (&inv)[CM], int C, T lam,
                                            T &min_ratio) {
#pragma unroll
    for (int i = 0; i < CM; ++i) {
#pragma unroll
        for (int j = 0; j <= i; ++j) {
            T v = B[tri(i, j)];
            if (i >= C || j >= C)
                v = (i == j) ? T(1) : T(0);
            else if (i == j)
                v += lam;
            B[tri(i, j)] = v;
        }
    }
    bool ok = true;
    min_ratio = T(1);
    // (trip counts independent of the outer index: with triangular loops the compiler left
    // the matrix of CM = 6 and 8 in local memory)
#pragma unroll
    for (int j = 0; j < CM; ++j) {
        // double: nothing to do for the identity's rows (a root, a division and their products
        // on a unit that takes 64 cycles a step; 1,000 rows, C = 5: 21 us, 19.5 without them)
        if (sizeof(T) == 8 && j >= C) {
            inv[j] = T(1);
            continue;
        }
        const T a_jj = B[tri(j, j)];
        T d = a_jj;
#pragma unroll
        for (int k = 0; k < CM; ++k)
            if (k < j) d -= B[tri(j, k)] * B[tri(j, k)];
        ok = ok && (d > T(0));
        if (a_jj > T(0)) min_ratio = fmin(min_ratio, d / a_jj);
        const T piv = sqrt(d > T(0) ? d : T(1));
        B[tri(j, j)] = piv;
        inv[j] = sizeof(T) == 8 ? T(1) / piv : T(0);
#pragma unroll
        for (int i = 0; i < CM; ++i) {
            if (i <= j || (sizeof(T) == 8 && i >= C)) continue;
            T s = B[tri(i, j)];
#pragma unroll
            for (int k = 0; k < CM; ++k)
                if (k < j) s -= B[tri(i, k)] * B[tri(j, k)];
            B[tri(i, j)] = chol_over<T>(s, piv, inv[j]);
        }
    }
    return ok;
}

// x = (L L^T)^-1 r with the factor of chol_factor (r beyond C is ignored).
template <class T, int CM>
__device__ __forceinline__ void chol_apply(const T (&L)[CM * (CM + 1) / 2], const T (&inv)[CM],
                                           const T (&r)[CM], int C, T (&x)[CM]) {
    T y[CM];
#pragma unroll
    for (int i = 0; i < CM; ++i) {
        T s = (i < C) ? r[i] : T(0);
#pragma unroll
        for (int k = 0; k < i; ++k) s -= L[tri(i, k)] * y[k];
        y[i] = chol_over<T>(s, L[tri(i, i)], inv[i]);
    }
#pragma unroll
    for (int i = CM - 1; i >= 0; --i) {
        T s = y[i];
#pragma unroll
        for (int k = i + 1; k < CM; ++k) s -= L[tri(k, i)] * x[k];
        x[i] = chol_over<T>(s, L[tri(i, i)], inv[i]);
    }
}

// Solves (B + lam I) x = c for the leading C x C block of a CM x CM packed lower
// triangle; rows/columns >= C are replaced by the identity (their x is 0).  B is
// overwritten by its factor.  Returns false when a pivot is <= 0 (x is then meaningless).
template <class T, int CM>
__device__ __forceinline__ bool chol_solve(T (&B)[CM * (CM + 1) / 2], const T (&c)[CM], int C,
                                           T lam, T (&x)[CM]) {
    T ratio, inv[CM];
    const bool ok = chol_factor<T, CM>(B, inv, C, lam, ratio);
    chol_apply<T, CM>(B, inv, c, C, x);
    return ok;
}

// The row solve of the mode passes (Eq. 4).  Double contexts: the Cholesky above.  Float
// contexts with a.cond_limit > 0: a row whose smallest pivot ratio is below 1 / cond_limit
// (or that has a non-positive pivot) is solved again in FP64 from the same sums; with
// a.refine: one step of iterative refinement, x += (L L^T)^-1 (c - (B + lam I) x) with the
// residual formed in FP64.  B and c are the row's sums as accumulated; B is not modified.
template <class T, int CM>
__device__ __forceinline__ bool row_solve(const PassArgs<T> &a, const T (&B)[CM * (CM + 1) / 2],
                                          const T (&c)[CM], T lam, T (&x)[CM]) {
    constexpr int NT = CM * (CM + 1) / 2;
    const int C = a.C;
    T L[NT];
#pragma unroll
    for (int q = 0; q < NT; ++q) L[q] = B[q];
    T ratio, inv[CM];
    bool ok = chol_factor<T, CM>(L, inv, C, lam, ratio);
    if constexpr (sizeof(T) == 4) {
        if (a.cond_limit > 0.f && (!ok || ratio * a.cond_limit < 1.f)) {
            double Bd[NT], cd[CM], xd[CM];
#pragma unroll
            for (int q = 0; q < NT; ++q) Bd[q] = (double)B[q];
#pragma unroll
            for (int q = 0; q < CM; ++q) cd[q] = (double)c[q];
            if (!chol_solve<double, CM>(Bd, cd, C, (double)lam, xd)) return false;
#pragma unroll
            for (int q = 0; q < CM; ++q) x[q] = (T)xd[q];
            atomicAdd(&a.stat->fp64_rows, 1ull);
            return true;
        }
        if (!ok) return false;
        chol_apply<T, CM>(L, inv, c, C, x);
        if (a.refine) {
            T r[CM], dx[CM];
#pragma unroll
            for (int i = 0; i < CM; ++i) {
                double s = (i < C) ? (double)c[i] - (double)lam * (double)x[i] : 0.0;
#pragma unroll
                for (int j = 0; j < CM; ++j) {
                    const T b = j <= i ? B[tri(i, j)] : B[tri(j, i)];
                    if (i < C && j < C) s -= (double)b * (double)x[j];
                }
                r[i] = (T)s;
            }
            chol_apply<T, CM>(L, inv, r, C, dx);
#pragma unroll
            for (int i = 0; i < CM; ++i) x[i] += dx[i];
        }
        return true;
    } else {
        if (ok) chol_apply<T, CM>(L, inv, c, C, x);
        return ok;
    }
}

template <class T, int CM>
__device__ __forceinline__ void write_row(const PassArgs<T> &a, int row, const T (&x)[CM]) {
    T *z = a.Zn + (int64_t)a.rank_n[row] * Geo<T, CM>::W;
    T *Ar = a.A_n + (int64_t)row * a.K;
#pragma unroll
    for (int c = 0; c < CM; ++c) {
        if (c < a.C) {
            z[c] = x[c];
            Ar[a.S[c]] = x[c];
        }
    }
}

// ----------------------------------------------------------------- warp pipeline
//
// Per warp, steps of up to 32 entries (one item, i.e. one row or row chunk, per step)
// flow through a ring in shared memory:
//   lead kLeadIdx: the other-mode indices, residual values and (first step of an item)
//                  the own row are copied in with 4/8-byte cp.async;
//   lead kLeadRows: the slice rows of the other modes are gathered with 16-byte
//                  cp.async, one fixed vector column per lane, skipping rows equal to
//                  the previous entry's (entries are sorted, so equal indices form runs);
//   lead 0: the step is computed.
// One commit group per iteration; since kLeadIdx >= 2 kLeadRows, waiting for all but
// the newest kLeadRows - 1 groups makes both this step's rows and the indices of the
// step whose rows are issued next available.
// The ring is kept shallow (rows one step ahead): the shared memory it leaves is the
// SM's L1, which serves the gathers of the hot (high-degree) slice rows; deeper rings
// and explicit row caches measured slower on Zipf-skewed tensors.

// SLOTS (row slots per warp): kRowSlots, or 1 where rings of four staged modes would leave few
// warps on an SM; a step's rows are then gathered when it comes up and the other warps hide
// the wait (mode_pass_plan_cm).
constexpr int kLeadRows = 1;
constexpr int kLeadIdx = 2;
constexpr int kRowSlots = kLeadRows + 1;
constexpr int kIdxSlots = kLeadIdx + 1;

__device__ __forceinline__ unsigned smem_addr(const void *p) {
    return (unsigned)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ void cp_async16(void *dst, const void *src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 16;\n" ::"r"(smem_addr(dst)), "l"(src)
                 : "memory");
}
__device__ __forceinline__ void cp_async16_l2(void *dst, const void *src) {  // past the L1
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(smem_addr(dst)), "l"(src)
                 : "memory");
}
template <int BYTES>
__device__ __forceinline__ void cp_async_small(void *dst, const void *src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2;\n" ::"r"(smem_addr(dst)), "l"(src),
                 "n"(BYTES)
                 : "memory");
}
__device__ __forceinline__ void cp_async_commit() {
    asm volatile("cp.async.commit_group;\n" ::: "memory");
}
template <int N>
__device__ __forceinline__ void cp_async_wait() {
    asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory");
}

__host__ __device__ constexpr size_t align16(size_t b) { return (b + 15) / 16 * 16; }
// A step's indices and residuals are staged as the aligned 16-byte vectors that cover them:
// 32 values from anywhere in a vector of `per` values, and where the step's first one lies.
__host__ __device__ constexpr int window(int per) { return 32 / per * per + per; }
// NO > 2 only: the vectors' bookkeeping costs three-way passes more than the narrower copies
// (C = 4: 0.70 against 0.66 ms).
template <class T, int NO>
__host__ __device__ constexpr int window_skew(int j0) {
    return NO > 2 ? j0 & (16 / (int)sizeof(T) - 1) : 0;
}
constexpr int kIdxWin = window(4);
__host__ __device__ constexpr int odd_up(int v) { return v | 1; }

__device__ __forceinline__ Step step_at_item(const tf_item *items, int64_t it, int64_t it_end) {
    return it < it_end ? first_step(items[it], it) : no_step(it);
}

__device__ __forceinline__ Step step_next(const Step &s, const tf_item *items, int64_t it_end) {
    if (!(s.flags & 1)) return s;
    if (!(s.flags & 4)) return step_on(s);
    return step_at_item(items, (int64_t)s.it + 1, it_end);
}

// Geometry of one pipeline flavour: NV_LO / NV_HI vectors fetched for other modes before
// / after mode n (n_lo of them are "before"); staged row strides are odd numbers of
// vectors, so 32 lanes reading one vector each of their own rows never conflict.
template <class T, int CM, int NV_LO, int NV_HI>
struct PipeGeo {
    static constexpr int V = 16 / (int)sizeof(T);
    static constexpr int RS_LO = odd_up(NV_LO) * V;
    static constexpr int RS_HI = odd_up(NV_HI) * V;
    static __host__ __device__ int lo_count(int no, int n_lo) { return no < n_lo ? no : n_lo; }
    static __host__ __device__ size_t slot_elems(int no, int n_lo) {
        const int nl = lo_count(no, n_lo);
        return (size_t)32 * (nl * RS_LO + (no - nl) * RS_HI);
    }
    static __host__ __device__ size_t mode_off(int t, int n_lo) {  // elements within a slot
        const int nl = t < n_lo ? t : n_lo;
        return (size_t)32 * (nl * RS_LO + (t - nl) * RS_HI);
    }
    static __host__ __device__ size_t rows_bytes(int no, int n_lo) {
        return align16(slot_elems(no > 0 ? no : 1, n_lo) * sizeof(T));
    }
    static __host__ __device__ size_t ridx_bytes(int no) {
        return align16((size_t)(no > 0 ? no : 1) * kIdxWin * 4);
    }
    static constexpr size_t RV_BYTES = align16(window(V) * sizeof(T));
    static constexpr size_t OWN_BYTES = align16(2 * CM * sizeof(T));
    static __host__ __device__ size_t heads_bytes(int no) {
        return align16((size_t)(no > 0 ? no : 1) * 4);
    }
    static __host__ __device__ size_t warp_bytes(int no, int n_lo, int slots = kRowSlots) {
        return slots * (rows_bytes(no, n_lo) + heads_bytes(no)) +
               kIdxSlots * (ridx_bytes(no) + RV_BYTES + OWN_BYTES + sizeof(Step)) + OWN_BYTES;
    }
};

// Warp-private views of the ring (slot pointers are computed, not stored in arrays).
template <class T, int CM, int NV_LO, int NV_HI, int SLOTS = kRowSlots>
struct PipeSmem {
    using PG = PipeGeo<T, CM, NV_LO, NV_HI>;
    unsigned char *rows0, *heads0, *ridx0, *rv0, *ownr0, *steps0;
    unsigned rows_b, heads_b, ridx_b;
    T *own;
    __device__ PipeSmem(unsigned char *base, int no, int n_lo) {
        rows_b = (unsigned)PG::rows_bytes(no, n_lo);
        heads_b = (unsigned)PG::heads_bytes(no);
        ridx_b = (unsigned)PG::ridx_bytes(no);
        rows0 = base;
        heads0 = rows0 + SLOTS * rows_b;
        ridx0 = heads0 + SLOTS * heads_b;
        rv0 = ridx0 + kIdxSlots * ridx_b;
        ownr0 = rv0 + kIdxSlots * PG::RV_BYTES;
        own = reinterpret_cast<T *>(ownr0 + kIdxSlots * PG::OWN_BYTES);
        steps0 = reinterpret_cast<unsigned char *>(own) + PG::OWN_BYTES;
    }
    __device__ __forceinline__ T *rows(int b) const {
        return reinterpret_cast<T *>(rows0 + b * rows_b);
    }
    __device__ __forceinline__ uint32_t *heads(int b) const {
        return reinterpret_cast<uint32_t *>(heads0 + b * heads_b);
    }
    __device__ __forceinline__ int32_t *ridx(int r) const {
        return reinterpret_cast<int32_t *>(ridx0 + r * ridx_b);
    }
    __device__ __forceinline__ T *rv(int r) const {
        return reinterpret_cast<T *>(rv0 + r * PG::RV_BYTES);
    }
    __device__ __forceinline__ T *ownring(int r) const {
        return reinterpret_cast<T *>(ownr0 + r * PG::OWN_BYTES);
    }
    __device__ __forceinline__ Step *step(int r) const {
        return reinterpret_cast<Step *>(steps0) + r;
    }
};

// Where the other modes' index streams and slices are: read from the kernel
// parameters when the number of other modes is a compile-time constant (every index
// is then a constant), from a shared-memory table otherwise (no local-memory copy of
// the parameter arrays).
template <class T, int NO>
struct OtherModes {
    const int32_t *const *oidx;
    const T *const *Zo;
    int no;
    __device__ __forceinline__ int count() const { return NO > 0 ? NO : no; }
};

// Indices, residual values, and (first step of an item) the own row's elements
// [own_off, own_off + own_len) of the own slice.
template <class T, int CM, int NO>
__device__ __forceinline__ void issue_idx(const Step &s, int32_t *ridx, T *rv, T *ownring,
                                          const OtherModes<T, NO> &om, const T *res,
                                          const tf_item *items, const T *Zn, const int32_t *rank_n,
                                          int own_off, int own_len, int lane) {
    if (!(s.flags & 1)) return;
    if constexpr (NO > 2) {
        constexpr int V = 16 / (int)sizeof(T);
        // a 16-byte copy per lane, in two rounds, instead of a 4-byte one per lane and array;
        // the arrays end in padding
        const int si = window_skew<int32_t, NO>(s.j0), sr = window_skew<T, NO>(s.j0);
        constexpr int VI = kIdxWin / 4, VR = window(V) / V, ALL = NO * VI + VR;
        const int n = min(s.jend - s.j0, kWarp);
#pragma unroll
        for (int q0 = 0; q0 < ALL; q0 += kWarp) {
            const int q = q0 + lane, t = q / VI, v = q - t * VI;
            if (t < NO) {
                const int32_t *src = om.oidx[0];
#pragma unroll
                for (int k = 1; k < NO; ++k) src = t == k ? om.oidx[k] : src;
                if (4 * v < n + si) cp_async16_l2(ridx + t * kIdxWin + 4 * v, src + (s.j0 - si) + 4 * v);
            } else {
                const int w = q - NO * VI;
                if (w < VR && V * w < n + sr) cp_async16_l2(rv + V * w, res + (s.j0 - sr) + V * w);
            }
        }
    } else {
        if (has_entry(s.j0, lane, s.jend)) {
            const int j = s.j0 + lane;
            const int no = om.count();
#pragma unroll(NO > 0 ? NO : 1)
            for (int t = 0; t < no; ++t) cp_async_small<4>(ridx + t * kIdxWin + lane, om.oidx[t] + j);
            cp_async_small<sizeof(T)>(rv + lane, res + j);
        }
    }
    if ((s.flags & 2) && lane < own_len) {
        const int64_t row = rank_n[items[s.it].row];
        cp_async_small<sizeof(T)>(ownring + lane, Zn + row * Geo<T, CM>::W + own_off + lane);
    }
}

// The slice rows of a step: for each other mode, entry r's row unless it equals entry
// r-1's (then entry r reads the run head's staged row).  Records the run heads.
template <class T, int CM, int NV_LO, int NV_HI, int NO>
__device__ __forceinline__ void issue_rows(const Step &s, T *rows, uint32_t *heads,
                                           const int32_t *ridx, const OtherModes<T, NO> &om,
                                           int n_lo, int lane) {
    using G = Geo<T, CM>;
    using PG = PipeGeo<T, CM, NV_LO, NV_HI>;
    constexpr int RPR = 32 / G::NV;  // rows per round
    if (!(s.flags & 1)) return;
    const int nvalid = min(s.jend - s.j0, kWarp);
    const int no = om.count();
    const int part = lane & (G::NV - 1), rsub = lane / G::NV;
#pragma unroll(NO > 0 ? NO : 1)
    for (int t = 0; t < no; ++t) {
        const int32_t *ri = ridx + t * kIdxWin + window_skew<int32_t, NO>(s.j0);
        const int mine = ri[lane], before = lane > 0 ? ri[lane - 1] : -1;
        const uint32_t hm =
            __ballot_sync(0xFFFFFFFFu, lane < nvalid && (lane == 0 || mine != before));
        if (lane == 0) heads[t] = hm;
        const bool lo = t < n_lo;
        const int need = lo ? NV_LO : NV_HI, rs = lo ? PG::RS_LO : PG::RS_HI;
        if (part >= need) continue;
        T *dst = rows + PG::mode_off(t, n_lo) + rsub * rs + part * G::V;
        const T *Z = om.Zo[t] + part * G::V;
#pragma unroll
        for (int k = 0; k < G::NV; ++k) {
            const int row = k * RPR + rsub;
            if ((hm >> row) & 1u) {
                // through the L1, which holds hot rows; four other modes' rows leave it no
                // room for that (five-way, 2e7 entries: last mode 2.80 ms, 2.52 past it; 256
                // small three-way tensors the other way, 0.67 and 0.74)
                if (NO > 2)
                    cp_async16_l2(dst + k * RPR * rs, Z + (int64_t)ri[row] * G::W);
                else
                    cp_async16(dst + k * RPR * rs, Z + (int64_t)ri[row] * G::W);
            }
        }
    }
}

// Staged row of other mode t that entry `lane` reads: the head of its run.
__device__ __forceinline__ int run_head(uint32_t heads, int lane) {
    const uint32_t upto = heads & (0xFFFFFFFFu >> (31 - lane));
    return 31 - __clz(upto);
}

// End of an item: the warp's sums of (B, c) to the item's partial slot (the solves run
// afterwards, all rows in parallel: k_solve_rows).  A reduce-scatter by halving exchanges
// (lane distances 16 .. 1): 67 shuffles for C = 10 where a butterfly per value took 325, with
// the same additions in the same order; lane segments of the packed values are written.  Rows
// of few entries spend much of their step here (five-way, five entries a row: 1,900 warp
// instructions per item before).
template <class T, int CM>
__device__ __forceinline__ void finish_item(const PassArgs<T> &a, const Step &s,
                                            T (&Bacc)[CM * (CM + 1) / 2], T (&cacc)[CM],
                                            int lane) {
    constexpr int NT = CM * (CM + 1) / 2, NB = NT + CM;
    constexpr int L1 = (NB + 1) / 2, L2 = (L1 + 1) / 2, L3 = (L2 + 1) / 2, L4 = (L3 + 1) / 2,
                  L5 = (L4 + 1) / 2;
    T *p = a.partials + (int64_t)a.items[s.it].slot * NB;
    T f[NB];
#pragma unroll
    for (int v = 0; v < NB; ++v) f[v] = v < NT ? Bacc[v < NT ? v : 0] : cacc[v < NT ? 0 : v - NT];
    int base = 0, cnt = NB;  // the lane's segment of the sums, in f[0 .. cnt)
    auto level = [&](auto nconst, auto hconst, int o) {
        constexpr int n = decltype(nconst)::value, hh = decltype(hconst)::value;
        const bool up = (lane & o) != 0;
#pragma unroll
        for (int k = 0; k < hh; ++k) {
            const T lo = f[k], hi = k + hh < n ? f[k + hh < n ? k + hh : 0] : T(0);
            const T send = up ? lo : hi, keep = up ? hi : lo;
            f[k] = keep + __shfl_xor_sync(0xFFFFFFFFu, send, o);
        }
        if (up) {
            base += hh;
            cnt = cnt > hh ? cnt - hh : 0;
        } else {
            cnt = cnt < hh ? cnt : hh;
        }
    };
    level(std::integral_constant<int, NB>{}, std::integral_constant<int, L1>{}, 16);
    level(std::integral_constant<int, L1>{}, std::integral_constant<int, L2>{}, 8);
    level(std::integral_constant<int, L2>{}, std::integral_constant<int, L3>{}, 4);
    level(std::integral_constant<int, L3>{}, std::integral_constant<int, L4>{}, 2);
    level(std::integral_constant<int, L4>{}, std::integral_constant<int, L5>{}, 1);
#pragma unroll
    for (int k = 0; k < L5; ++k)
        if (k < cnt) p[base + k] = f[k];
#pragma unroll
    for (int v = 0; v < NT; ++v) Bacc[v] = T(0);
#pragma unroll
    for (int c = 0; c < CM; ++c) cacc[c] = T(0);
}

// Per-entry arithmetic of the mode pass on staged rows.  rowp[t] points at the staged
// row of other mode t that this entry reads.  Returns h (zero beyond C) and, on the
// first inner iteration, the products that refresh R-hat: po = sum_{c<C} prod_l old_l[c]
// (own old included) and pp = sum_{c<Cq} prod_l prev_l[c].  Other modes t >= n_lo come
// after mode n and have not been updated in this split: their "old" is their "cur".
// own is 16-byte aligned; its prev / old regions start at OWN_PREV / OWN_OLD.
template <class T, int CM, int NO, bool FIRST, int OWN_PREV = 0, int OWN_OLD = CM>
__device__ __forceinline__ void entry_products(const T *const (&rowp)[(NO > 0 ? NO : kMaxModes - 1)],
                                               const T *own, int no, int n_lo, int C, int Cq,
                                               T (&h)[CM], T &po, T &pp) {
    using G = Geo<T, CM>;
    constexpr int OP = G::OFF_PREV, OO = G::OFF_OLD;
    if constexpr (NO == 2) {
        const T *r0 = rowp[0], *r1 = rowp[1];
        {
            T x[CM], y[CM];
            lds_range<T, 0, CM>(x, r0);
            lds_range<T, 0, CM>(y, r1);
#pragma unroll
            for (int c = 0; c < CM; ++c) h[c] = (c < C) ? x[c] * y[c] : T(0);
        }
        if constexpr (FIRST) {
            {
                T x[CM], y[CM], o[CM];
                lds_range<T, OP, CM>(x, r0);
                lds_range<T, OP, CM>(y, r1);
                lds_range<T, OWN_PREV, CM>(o, own);
                pp = T(0);
#pragma unroll
                for (int c = 0; c < CM; ++c)
                    if (c < Cq) pp += o[c] * (x[c] * y[c]);
            }
            {
                T o[CM];
                lds_range<T, OWN_OLD, CM>(o, own);
                po = T(0);
                if (n_lo == 0) {  // both other modes after n: old == cur, so po = own_old . h
#pragma unroll
                    for (int c = 0; c < CM; ++c) po += o[c] * h[c];
                } else {
                    T x[CM], y[CM];
                    lds_range<T, OO, CM>(x, r0);
                    if (n_lo > 1)
                        lds_range<T, OO, CM>(y, r1);
                    else
                        lds_range<T, 0, CM>(y, r1);
#pragma unroll
                    for (int c = 0; c < CM; ++c)
                        if (c < C) po += o[c] * (x[c] * y[c]);
                }
            }
        }
    } else {
        T x[CM];
#pragma unroll
        for (int c = 0; c < CM; ++c) h[c] = T(1);
#pragma unroll(NO > 0 ? NO : 1)
        for (int t = 0; t < (NO > 0 ? NO : no); ++t) {
            lds_range<T, 0, CM>(x, rowp[t]);
#pragma unroll
            for (int c = 0; c < CM; ++c) h[c] *= x[c];
        }
#pragma unroll
        for (int c = 0; c < CM; ++c)
            if (c >= C) h[c] = T(0);
        if constexpr (FIRST) {
            T q[CM];
            lds_range<T, OWN_PREV, CM>(q, own);  // own prev
#pragma unroll(NO > 0 ? NO : 1)
            for (int t = 0; t < (NO > 0 ? NO : no); ++t) {
                lds_range<T, OP, CM>(x, rowp[t]);
#pragma unroll
                for (int c = 0; c < CM; ++c) q[c] *= x[c];
            }
            pp = T(0);
#pragma unroll
            for (int c = 0; c < CM; ++c)
                if (c < Cq) pp += q[c];
            lds_range<T, OWN_OLD, CM>(q, own);  // own old
#pragma unroll(NO > 0 ? NO : 1)
            for (int t = 0; t < (NO > 0 ? NO : no); ++t) {
                if (t < n_lo)
                    lds_range<T, OO, CM>(x, rowp[t]);
                else
                    lds_range<T, 0, CM>(x, rowp[t]);
#pragma unroll
                for (int c = 0; c < CM; ++c) q[c] *= x[c];
            }
            po = T(0);
#pragma unroll
            for (int c = 0; c < CM; ++c)
                if (c < C) po += q[c];
        }
    }
}

// Drives one bin through the ring; Consumer does the per-step work:
//   c.item_begin(sm, step, idx_slot)   first step of an item (own row is in the ring)
//   c.entry(sm, step, row_slot, idx_slot, lane)
//   c.item_end(step)                   last step of an item
template <class T, int CM, int NV_LO, int NV_HI, int NO, int SLOTS, class Consumer>
__device__ __forceinline__ void run_bin(const tf_item *items, int64_t it0, int64_t it1,
                                        const OtherModes<T, NO> &om, const T *res, const T *Zn,
                                        const int32_t *rank_n, int n_lo, int own_off, int own_len,
                                        bool fetch_rows,
                                        PipeSmem<T, CM, NV_LO, NV_HI, SLOTS> &sm,
                                        Consumer &cons,
                                        int lane) {
    // prologue: steps 0 .. kLeadIdx-1 (indices), then rows of steps 0 .. kLeadRows-1
    Step gen = step_at_item(items, it0, it1);
#pragma unroll
    for (int k = 0; k < kLeadIdx; ++k) {
        if (lane == 0) *sm.step(k) = gen;
        issue_idx<T, CM, NO>(gen, sm.ridx(k), sm.rv(k), sm.ownring(k), om, res, items, Zn, rank_n,
                             own_off, own_len, lane);
        gen = step_next(gen, items, it1);
    }
    cp_async_commit();
    cp_async_wait<0>();
    __syncwarp();
    if constexpr (SLOTS == 1) {
        for (int is = 0;; is = (is + 1) % kIdxSlots) {
            const Step cur = *sm.step(is);
            if (!(cur.flags & 1)) break;
            if (fetch_rows)
                issue_rows<T, CM, NV_LO, NV_HI, NO>(cur, sm.rows(0), sm.heads(0), sm.ridx(is), om,
                                                    n_lo, lane);
            cp_async_commit();
            const int ia = (is + kLeadIdx) % kIdxSlots;
            if (lane == 0) *sm.step(ia) = gen;
            issue_idx<T, CM, NO>(gen, sm.ridx(ia), sm.rv(ia), sm.ownring(ia), om, res, items, Zn,
                                 rank_n, own_off, own_len, lane);
            gen = step_next(gen, items, it1);
            cp_async_commit();
            cp_async_wait<1>();  // this step's rows, and the next one's indices
            __syncwarp();
            if (cur.flags & 2) cons.item_begin(sm, cur, is, lane);
            cons.entry(sm, cur, 0, is, lane);
            if (cur.flags & 4) cons.item_end(cur, lane);
            __syncwarp();
        }
        cp_async_wait<0>();
        __syncwarp();
        return;
    }
#pragma unroll
    for (int k = 0; k < kLeadRows; ++k) {
        if (fetch_rows) {
            const Step sk = *sm.step(k);
            issue_rows<T, CM, NV_LO, NV_HI, NO>(sk, sm.rows(k), sm.heads(k), sm.ridx(k), om, n_lo,
                                                lane);
        }
        cp_async_commit();
    }
    int is = 0, rs = 0;  // ring slots of the step computed now
    for (;;) {
        cp_async_wait<kLeadRows - 1>();
        __syncwarp();
        const Step cur = *sm.step(is);
        if (!(cur.flags & 1)) break;
        // rows of step +kLeadRows, indices of step +kLeadIdx
        {
            const int ib = (is + kLeadRows) % kIdxSlots, rb = (rs + kLeadRows) % kRowSlots;
            if (fetch_rows) {
                const Step sb = *sm.step(ib);
                issue_rows<T, CM, NV_LO, NV_HI, NO>(sb, sm.rows(rb), sm.heads(rb), sm.ridx(ib), om,
                                                    n_lo, lane);
            }
            const int ia = (is + kLeadIdx) % kIdxSlots;
            __syncwarp();  // everyone has read slot ia's step before it is replaced
            if (lane == 0) *sm.step(ia) = gen;
            issue_idx<T, CM, NO>(gen, sm.ridx(ia), sm.rv(ia), sm.ownring(ia), om, res, items, Zn,
                                 rank_n, own_off, own_len, lane);
            gen = step_next(gen, items, it1);
            cp_async_commit();
        }
        if (cur.flags & 2) cons.item_begin(sm, cur, is, lane);
        cons.entry(sm, cur, rs, is, lane);
        if (cur.flags & 4) cons.item_end(cur, lane);
        __syncwarp();
        is = (is + 1) % kIdxSlots;
        rs = (rs + 1) % kRowSlots;
    }
    cp_async_wait<0>();
    __syncwarp();
}

template <class T, int CM, int NO, bool FIRST, int SLOTS>
struct PassConsumer {
    using G = Geo<T, CM>;
    static constexpr int NV_LO = FIRST ? G::NV_ALL : G::NV_CUR;  // cur|prev|old
    static constexpr int NV_HI = FIRST ? G::NV_CP : G::NV_CUR;   // cur|prev
    using PG = PipeGeo<T, CM, NV_LO, NV_HI>;
    using SM = PipeSmem<T, CM, NV_LO, NV_HI, SLOTS>;
    const PassArgs<T> &a;
    int no, n_lo;
    T Bacc[G::NT], cacc[CM];
    __device__ PassConsumer(const PassArgs<T> &a_, int no_, int n_lo_) : a(a_), no(no_), n_lo(n_lo_) {
#pragma unroll
        for (int v = 0; v < G::NT; ++v) Bacc[v] = T(0);
#pragma unroll
        for (int c = 0; c < CM; ++c) cacc[c] = T(0);
    }
    __device__ __forceinline__ void item_begin(const SM &sm, const Step &, int is, int lane) {
        if (FIRST) {
            if (lane < 2 * CM) sm.own[lane] = sm.ownring(is)[lane];
            __syncwarp();
        }
    }
    __device__ __forceinline__ void entry(const SM &sm, const Step &st, int rs, int is, int lane) {
        if (!has_entry(st.j0, lane, st.jend)) return;
        const int j = st.j0 + lane;
        const T *slot = sm.rows(rs);
        const uint32_t *hd = sm.heads(rs);
        constexpr int NP = NO > 0 ? NO : kMaxModes - 1;
        const T *rowp[NP];
#pragma unroll
        for (int t = 0; t < NP; ++t) {
            if (t < no) {
                const int rsz = t < n_lo ? PG::RS_LO : PG::RS_HI;
                rowp[t] = slot + PG::mode_off(t, n_lo) + run_head(hd[t], lane) * rsz;
            } else {
                rowp[t] = slot;
            }
        }
        T h[CM], po = T(0), pp = T(0);
        entry_products<T, CM, NO, FIRST>(rowp, sm.own, no, n_lo, a.C, a.Cq, h, po, pp);
        T v = sm.rv(is)[window_skew<T, NO>(st.j0) + lane];
        if (FIRST) {
            v = v - pp + po;
            a.res[j] = v;
        }
#pragma unroll
        for (int c1 = 0; c1 < CM; ++c1) {
            cacc[c1] += v * h[c1];
#pragma unroll
            for (int c2 = 0; c2 <= c1; ++c2) Bacc[tri(c1, c2)] += h[c1] * h[c2];
        }
    }
    __device__ __forceinline__ void item_end(const Step &st, int lane) {
        finish_item<T, CM>(a, st, Bacc, cacc, lane);
    }
};

template <class T, int NO>
__device__ __forceinline__ OtherModes<T, NO> other_modes(const int32_t *const *p_oidx,
                                                         const T *const *p_Zo, int N,
                                                         const int32_t **s_oidx,
                                                         const T **s_Zo) {
    OtherModes<T, NO> om;
    om.no = N - 1;
    if constexpr (NO > 0) {
        om.oidx = p_oidx;
        om.Zo = p_Zo;
    } else {
        if (threadIdx.x < kMaxModes - 1) {
            s_oidx[threadIdx.x] = p_oidx[threadIdx.x];
            s_Zo[threadIdx.x] = p_Zo[threadIdx.x];
        }
        __syncthreads();
        om.oidx = s_oidx;
        om.Zo = s_Zo;
    }
    return om;
}

// Bytes of one warp's ring for a mode pass of mode n (n_lo = n other modes before it).
template <class T, int CM, bool FIRST>
__host__ __device__ size_t pass_warp_bytes(int N, int n, int slots) {
    using G = Geo<T, CM>;
    using PG = PipeGeo<T, CM, FIRST ? G::NV_ALL : G::NV_CUR, FIRST ? G::NV_CP : G::NV_CUR>;
    return PG::warp_bytes(N - 1, n, slots);
}

// Warps per block of the mode pass (one block per SM): as many as the registers of the
// per-lane Gram accumulators allow without spilling (the accumulators grow as CM^2).
template <class T, int CM>
constexpr int pass_max_warps() {
    return sizeof(T) == 4 ? (CM <= 2 ? 24 : (CM <= 4 ? 20 : (CM <= 8 ? 16 : 12))) : (CM <= 4 ? 12 : 8);
}

// NO: number of other modes (N - 1) when specialised, 0 for any N (runtime loops).
// FIRST: the split's first inner iteration (R-hat refresh) or a later one.
// One block per SM (the staging rings are small, so most of the SM's shared memory
// stays L1 cache: the hottest slice rows are served from there).
template <class T, int CM, int NO, bool FIRST, int SLOTS>
__global__ void __launch_bounds__(pass_max_warps<T, CM>() * kWarp, 1)
    k_mode_pass(const PassArgs<T> a) {
    using Cons = PassConsumer<T, CM, NO, FIRST, SLOTS>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ const int32_t *s_oidx[kMaxModes - 1];
    __shared__ const T *s_Zo[kMaxModes - 1];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const OtherModes<T, NO> om = other_modes<T, NO>(a.oidx, a.Zo, a.N, s_oidx, s_Zo);
    const int no = a.N - 1, n_lo = a.n;
    typename Cons::SM sm(smem_raw + warp * pass_warp_bytes<T, CM, FIRST>(a.N, a.n, SLOTS), no, n_lo);
    Cons cons(a, no, n_lo);
    // own row: prev|old regions, [CM, 3 CM) of the own slice row (first iteration only)
    const int own_len = FIRST ? 2 * CM : 0;
    // Bins are fetched dynamically (one ticket per fetch): which warp runs a bin does
    // not change any result, only the load balance.
    for (;;) {
        unsigned long long tk = 0;
        if (lane == 0) tk = atomicAdd(a.ticket, 1ull) - a.ticket_base;
        tk = __shfl_sync(0xFFFFFFFFu, tk, 0);
        if (tk >= (unsigned long long)a.P) break;
        const int bin = (int)tk;
        run_bin<T, CM, Cons::NV_LO, Cons::NV_HI, NO, SLOTS>(a.items, a.bin_ptr[bin], a.bin_ptr[bin + 1],
                                                     om, a.res, a.Zn, a.rank_n, n_lo, CM, own_len,
                                                     true, sm, cons, lane);
    }
}

// Mode pass of three-way tensors for C = 1 (CDTF): a slice row is one 16-byte vector (32 bytes
// for doubles) of cur, prev and old, so each lane reads its entries' rows directly, four
// entries in flight, instead of staging them for the warp; lane and entry pairing and every
// sum are those of the staged pass.  Bound: the row gathers (L1 lookups, one line per lane).
// 1e7 entries, modes of 30,011 / 20,021 / 503 rows: 0.112 ms a pass staged, 0.060 now.
template <class T>
struct RowOne {
    T cur, prev, old;
};
template <class T, bool ALL>
__device__ __forceinline__ RowOne<T> load_row_one(const T *z) {
    RowOne<T> r{};
    if constexpr (!ALL) {
        r.cur = z[0];
    } else if constexpr (sizeof(T) == 4) {
        const float4 v = *reinterpret_cast<const float4 *>(z);
        r.cur = v.x, r.prev = v.y, r.old = v.z;
    } else {
        const double2 v = *reinterpret_cast<const double2 *>(z);
        r.cur = v.x, r.prev = v.y, r.old = z[2];
    }
    return r;
}

constexpr int kOneWarps = 32;

template <class T, bool FIRST>
__global__ void __launch_bounds__(kOneWarps * kWarp, 1) k_pass_one(const PassArgs<T> a) {
    constexpr int W = Geo<T, 1>::W, U = 4;
    const int lane = threadIdx.x & 31, n_lo = a.n, Cq = a.Cq;
    const T *Z0 = a.Zo[0], *Z1 = a.Zo[1];
    const int32_t *ix0 = a.oidx[0], *ix1 = a.oidx[1];
    for (;;) {
        unsigned long long tk = 0;
        if (lane == 0) tk = atomicAdd(a.ticket, 1ull) - a.ticket_base;
        tk = __shfl_sync(0xFFFFFFFFu, tk, 0);
        if (tk >= (unsigned long long)a.P) break;
        for (int64_t it = a.bin_ptr[tk]; it < a.bin_ptr[tk + 1]; ++it) {
            const tf_item item = a.items[it];
            RowOne<T> own{};
            if (FIRST) own = load_row_one<T, true>(a.Zn + (int64_t)a.rank_n[item.row] * W);
            T B[1] = {T(0)}, c[1] = {T(0)};
            const int end = (int)(item.begin + item.len);
            int j0 = (int)item.begin;
            while (j0 < end) {
                int32_t i0[U], i1[U];
                T rv[U];
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const int k = u * kWarp + lane;
                    const bool in = has_entry(j0, k, end);
                    i0[u] = in ? ix0[j0 + k] : -1;
                    i1[u] = in ? ix1[j0 + k] : 0;
                    rv[u] = in ? a.res[j0 + k] : T(0);
                }
                RowOne<T> r0[U], r1[U];
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    r0[u] = load_row_one<T, FIRST>(Z0 + (int64_t)(i0[u] < 0 ? 0 : i0[u]) * W);
                    r1[u] = load_row_one<T, FIRST>(Z1 + (int64_t)i1[u] * W);
                }
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    if (i0[u] < 0) continue;
                    const T h = r0[u].cur * r1[u].cur;
                    T v = rv[u];
                    if (FIRST) {
                        T pp = T(0), po = T(0);
                        if (Cq > 0) pp += own.prev * (r0[u].prev * r1[u].prev);
                        if (n_lo == 0)
                            po += own.old * h;
                        else
                            po += own.old * (r0[u].old * (n_lo > 1 ? r1[u].old : r1[u].cur));
                        v = v - pp + po;
                        a.res[j0 + (u * kWarp + lane)] = v;
                    }
                    c[0] += v * h;
                    B[0] += h * h;
                }
                if (last_step(j0, U * kWarp, end)) break;
                j0 += U * kWarp;
            }
            Step st{};
            st.it = (int32_t)it;
            finish_item<T, 1>(a, st, B, c, lane);
        }
    }
}

// Row solves of a mode: (B + lambda I) a = c (Eq. 4) for every row, by the register Cholesky
// of Section 3.1 with one lane per row, in one launch.  A row with several slots is summed as
// G = kSlotSums / NB sums of every G-th slot, added in order (plain order up to G slots).
//   Heavy rows (more than kHeavySlots partial slots): one block each; a thread advances up to
//   four of the G * NB sums together, 32 loads in flight.
//   Medium rows: eight per block, two per warp, lanes over the values.
//   Light rows (up to kLightSlots): 32 per warp, brought into shared memory with consecutive
//   lanes on consecutive values; where the 32 slots lie together, as 16-byte cp.async.
// Bound: latency, reading the slots (C = 10: 260 B a row) and the scattered columns of the
// factor rows written (one 32-byte sector per value where K is large).  Before, one launch
// solved the single-slot rows, each thread reading its row's slot at a stride of NB values,
// and a second took 512 threads per split row: 44 + 55 us per mode of 1e5 rows (1e8 entries,
// C = 10), now 61; 1,000 FP64 rows of two slots, C = 5: 127 us (a lone lane's FP64
// instructions take the unit as long as a full warp's), now 19.5.
// XS: the solve options of float contexts (refinement / FP64 fallback) are on; the plain
// Cholesky otherwise, so that the default kernels carry none of their registers.
template <class T, int CM, bool XS>
__device__ __forceinline__ void solve_and_write(const PassArgs<T> &a, const SplitRow &sr,
                                                const T *sum) {
    constexpr int NT = CM * (CM + 1) / 2;
    T B[NT], c[CM], x[CM];
#pragma unroll
    for (int q = 0; q < NT; ++q) B[q] = sum[q];
#pragma unroll
    for (int q = 0; q < CM; ++q) c[q] = sum[NT + q];
    const T lam = a.weighted ? a.lambda * (T)sr.len : a.lambda;
    if (XS ? row_solve<T, CM>(a, B, c, lam, x) : chol_solve<T, CM>(B, c, a.C, lam, x))
        write_row<T, CM>(a, sr.row, x);
    else
        atomicAdd(&a.stat->singular_rows, 1ull);
}

constexpr int kSolveThreads = 128;

// Sum of a heavy row's slots at p into tot[NB]; red: G * NB values (both shared memory).
template <class T, int NB>
__device__ __forceinline__ void sum_slots(const T *p, int count, T *red, T *tot) {
    // a thread's sums (every kSolveThreads-th of the G * NB) advance together
    constexpr int G = kSlotSums / NB, PT = (G * NB + kSolveThreads - 1) / kSolveThreads, U = 32 / PT;
    const int tid = threadIdx.x;
    T s[PT];
#pragma unroll
    for (int i = 0; i < PT; ++i) s[i] = T(0);
    for (int k = 0; k < count; k += U * G) {
        T w[PT][U];
#pragma unroll
        for (int i = 0; i < PT; ++i) {
            const int t = tid + i * kSolveThreads, g = t / NB, v = t - g * NB;
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int slot = k + g + u * G;
                w[i][u] = t < G * NB && slot < count ? p[(int64_t)slot * NB + v] : T(0);
            }
        }
#pragma unroll
        for (int i = 0; i < PT; ++i)
#pragma unroll
            for (int u = 0; u < U; ++u) s[i] += w[i][u];
    }
#pragma unroll
    for (int i = 0; i < PT; ++i)
        if (tid + i * kSolveThreads < G * NB) red[tid + i * kSolveThreads] = s[i];
    __syncthreads();
    for (int v = tid; v < NB; v += kSolveThreads) {
        T s = T(0);
        for (int g = 0; g < G; ++g) s += red[g * NB + v];
        tot[v] = s;
    }
    __syncthreads();
}

// Sum of a medium row's slots at p into tot[NB] (shared memory) by one warp.
template <class T, int NB>
__device__ __forceinline__ void sum_slots_warp(const T *p, int count, T *tot, int lane) {
    constexpr int G = kSlotSums / NB, VL = (NB + 31) / 32, U = VL > 2 ? 4 : 8;
    T sum[VL];
#pragma unroll
    for (int i = 0; i < VL; ++i) sum[i] = T(0);
    for (int g = 0; g < G && g < count; g += U) {
        T s[VL][U];
#pragma unroll
        for (int i = 0; i < VL; ++i)
#pragma unroll
            for (int u = 0; u < U; ++u) s[i][u] = T(0);
        for (int k = g; k < count; k += G) {
            T w[VL][U];
#pragma unroll
            for (int i = 0; i < VL; ++i)
#pragma unroll
                for (int u = 0; u < U; ++u)
                    w[i][u] = g + u < G && k + u < count && lane + 32 * i < NB
                                  ? p[(int64_t)(k + u) * NB + lane + 32 * i]
                                  : T(0);
#pragma unroll
            for (int i = 0; i < VL; ++i)
#pragma unroll
                for (int u = 0; u < U; ++u) s[i][u] += w[i][u];
        }
#pragma unroll
        for (int i = 0; i < VL; ++i)
#pragma unroll
            for (int u = 0; u < U; ++u) sum[i] += s[i][u];
    }
#pragma unroll
    for (int i = 0; i < VL; ++i)
        if (lane + 32 * i < NB) tot[lane + 32 * i] = sum[i];
}

// Values of a warp's 32 light rows in shared memory, and their row stride: flat where NB is
// odd (lanes reading their rows do not conflict) or the conflicts are few, else one more.
template <int NB>
constexpr int solve_stride() {
    return NB % 8 == 0 ? NB + 1 : NB;
}
template <class T, int CM>
constexpr size_t solve_rows_smem() {
    constexpr int NB = CM * (CM + 1) / 2 + CM;
    constexpr int light = kSolveThreads / 32 * ((32 * solve_stride<NB>() + 7) / 4 * 4);
    constexpr int heavy = kSlotSums + NB, medium = kMediumRows * NB;
    constexpr int most = light > heavy ? light : heavy;
    return sizeof(T) * (size_t)(most > medium ? most : medium);
}

template <class T, int CM, bool XS>
__global__ void __launch_bounds__(kSolveThreads) k_solve_rows(const PassArgs<T> a,
                                                              const SolveRows r) {
    constexpr int NT = CM * (CM + 1) / 2, NB = NT + CM, NBP = solve_stride<NB>();
    constexpr int V = 16 / (int)sizeof(T);
    extern __shared__ __align__(16) unsigned char smem_raw[];
    T *sm = reinterpret_cast<T *>(smem_raw);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int blk = (int)blockIdx.x;
    if (blk < r.n_heavy) {  // first, the longest
        const SplitRow sr = r.split[r.n_light + r.n_medium + blk];
        T *tot = sm + kSlotSums;
        sum_slots<T, NB>(a.partials + (int64_t)sr.first_slot * NB, sr.n_slots, sm, tot);
        if (threadIdx.x == 0) solve_and_write<T, CM, XS>(a, sr, tot);
        return;
    }
    blk -= r.n_heavy;
    if (blk < (r.n_medium + kMediumRows - 1) / kMediumRows) {
        const SplitRow *rows = r.split + r.n_light + blk * kMediumRows;
        const int n = min(kMediumRows, r.n_medium - blk * kMediumRows);
        for (int q = warp; q < n; q += kSolveThreads / 32)
            sum_slots_warp<T, NB>(a.partials + (int64_t)rows[q].first_slot * NB, rows[q].n_slots,
                                  sm + q * NB, lane);
        __syncthreads();
        if ((int)threadIdx.x < n)
            solve_and_write<T, CM, XS>(a, rows[threadIdx.x], sm + threadIdx.x * NB);
        return;
    }
    blk -= (r.n_medium + kMediumRows - 1) / kMediumRows;
    const int i = blk * kSolveThreads + (int)threadIdx.x;
    SplitRow sr{};
    if (i < r.n_single)
        sr = r.single[i];
    else if (i < r.n_single + r.n_light)
        sr = r.split[i - r.n_single];
    T *buf = sm + warp * ((32 * NBP + 7) / 4 * 4);
    const int first0 = __shfl_sync(0xFFFFFFFFu, sr.first_slot, 0);
    if (NBP == NB && __all_sync(0xFFFFFFFFu, sr.n_slots == 1 && sr.first_slot == first0 + lane)) {
        // 32 slots in a row: copied as they lie, in whole vectors but for the ends
        const int64_t e0 = (int64_t)first0 * NB;
        const int skew = (int)(e0 % V), lead = skew ? V - skew : 0;
        const T *src = a.partials + e0;
        buf += skew;
        const int nv = (32 * NB - lead) / V, tail = 32 * NB - lead - nv * V;
        for (int q = lane; q < nv; q += 32) cp_async16(buf + lead + q * V, src + lead + q * V);
        if (lane < lead) cp_async_small<sizeof(T)>(buf + lane, src + lane);
        if (lane < tail) {
            const int q = 32 * NB - tail + lane;
            cp_async_small<sizeof(T)>(buf + q, src + q);
        }
        cp_async_commit();
        cp_async_wait<0>();
    } else {
        constexpr int U = 8;
        for (int q0 = lane; q0 < 32 * NB; q0 += 32 * U) {
            T s[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int q = q0 + 32 * u, w = q / NB, v = q - w * NB;
                const int first = __shfl_sync(0xFFFFFFFFu, sr.first_slot, w & 31);
                const int n = __shfl_sync(0xFFFFFFFFu, sr.n_slots, w & 31);
                const T *p = a.partials + (int64_t)first * NB + v;
                const int ns = q < 32 * NB ? n : 0;
                T t[kLightSlots];
#pragma unroll
                for (int k = 0; k < kLightSlots; ++k) t[k] = k < ns ? p[k * NB] : T(0);
                s[u] = t[0];
#pragma unroll
                for (int k = 1; k < kLightSlots; ++k) s[u] += t[k];
            }
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int q = q0 + 32 * u, w = q / NB, v = q - w * NB;
                if (q < 32 * NB) buf[w * NBP + v] = s[u];
            }
        }
    }
    __syncwarp();
    if (sr.n_slots > 0) solve_and_write<T, CM, XS>(a, sr, buf + lane * NBP);
}

// Residual of copy n against the columns held in the slices' "cur" region (the last
// split's final values): r = res - sum_{c < Cq} prod_l Z_l[i_l, c].  One warp per bin,
// every bin launched (the per-block double sums are then in a fixed order); the same
// warp pipeline as the mode pass feeds it.
template <class T, int CM, int NO>
struct ResConsumer {
    using G = Geo<T, CM>;
    static constexpr int NV_LO = G::NV_CUR, NV_HI = G::NV_CUR;
    static constexpr int SLOTS = NO > 2 ? 1 : kRowSlots;  // as the passes of four other modes
    using PG = PipeGeo<T, CM, NV_LO, NV_HI>;
    using SM = PipeSmem<T, CM, NV_LO, NV_HI, SLOTS>;
    const ResArgs<T> &a;
    int no;
    double acc = 0.0;
    __device__ ResConsumer(const ResArgs<T> &a_, int no_) : a(a_), no(no_) {}
    __device__ __forceinline__ void item_begin(const SM &sm, const Step &, int is, int lane) {
        if (a.Cq > 0) {
            if (lane < CM) sm.own[lane] = sm.ownring(is)[lane];
            __syncwarp();
        }
    }
    __device__ __forceinline__ void entry(const SM &sm, const Step &st, int rs, int is, int lane) {
        if (!has_entry(st.j0, lane, st.jend)) return;
        const int j = st.j0 + lane;
        T p = T(0);
        if (a.Cq > 0) {
            const T *slot = sm.rows(rs);
            const uint32_t *hd = sm.heads(rs);
            T q[CM], x[CM];
            lds_range<T, 0, CM>(q, sm.own);
#pragma unroll(NO > 0 ? NO : 1)
            for (int t = 0; t < (NO > 0 ? NO : no); ++t) {
                lds_range<T, 0, CM>(x, slot + PG::mode_off(t, no) + run_head(hd[t], lane) * PG::RS_LO);
#pragma unroll
                for (int c = 0; c < CM; ++c) q[c] *= x[c];
            }
#pragma unroll
            for (int c = 0; c < CM; ++c)
                if (c < a.Cq) p += q[c];
        }
        const T r = sm.rv(is)[window_skew<T, NO>(st.j0) + lane] - p;
        if (a.what == 0)
            acc += (double)r * (double)r;
        else if (a.what == 1)
            a.out[a.perm[j]] = r;
        else
            a.res[j] = r;
    }
    __device__ __forceinline__ void item_end(const Step &, int) {}
};

// Number of other modes as a compile-time constant: five-way float tensors, any (0).  Orders 4 and
// 6 to 8 and double run the generic kernel; the constant, the 16-byte windows and the single row
// slot were not measured for them.
template <class T>
__host__ __device__ constexpr int res_no(int N) {
    return sizeof(T) == 4 && N == 5 ? 4 : 0;
}
template <class T, int CM>
__host__ __device__ size_t res_warp_bytes(int N) {
    using G = Geo<T, CM>;
    return PipeGeo<T, CM, G::NV_CUR, G::NV_CUR>::warp_bytes(N - 1, N - 1,
                                                            res_no<T>(N) > 2 ? 1 : kRowSlots);
}

template <class T, int CM, int NO>
__global__ void __launch_bounds__(kPassThreads) k_res(const ResArgs<T> a) {
    using Cons = ResConsumer<T, CM, NO>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ double wsum[kPassThreads / kWarp];
    __shared__ const int32_t *s_oidx[kMaxModes - 1];
    __shared__ const T *s_Zo[kMaxModes - 1];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int no = a.N - 1;
    const OtherModes<T, NO> om = other_modes<T, NO>(a.oidx, a.Zo, a.N, s_oidx, s_Zo);
    typename Cons::SM sm(smem_raw + warp * res_warp_bytes<T, CM>(a.N), no, no);
    Cons cons(a, no);
    const int bin = (int)(((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5);
    if (bin < a.P)
        run_bin<T, CM, Cons::NV_LO, Cons::NV_HI, NO, Cons::SLOTS>(
            a.items, a.bin_ptr[bin], a.bin_ptr[bin + 1], om, a.res, a.Zn, a.rank_n, no, 0,
            a.Cq > 0 ? CM : 0, a.Cq > 0, sm, cons, lane);
    if (a.what != 0) return;
    const double acc = warp_sum_d(cons.acc);
    if (lane == 0) wsum[warp] = acc;
    __syncthreads();
    if (threadIdx.x == 0) {
        double s = 0.0;
        for (int w = 0; w < (int)(blockDim.x / kWarp); ++w) s += wsum[w];
        a.block_out[blockIdx.x] = s;
    }
}

// Warps per block of the pipelined kernels: the count (1, 2 or 4) that puts the most
// warps on an SM given the per-warp ring size (at least one).
inline int best_warps_per_block(size_t warp_bytes) {
    int dev = 0, smem_sm = 0, smem_blk = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&smem_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev);
    cudaDeviceGetAttribute(&smem_blk, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    int best = 1, best_total = 0;
    for (int w = kPassThreads / kWarp; w >= 1; w /= 2) {
        const size_t blk = w * warp_bytes + 1024;  // + static shared memory / reserve
        if (blk > (size_t)smem_blk) continue;
        const int total = w * std::min(32 / w, (int)(smem_sm / blk));
        if (total > best_total) {
            best_total = total;
            best = w;
        }
    }
    return best;
}

// Three- and five-way tensors get the number of other modes as a compile-time constant
// (fully unrolled mode loops); other orders run the generic kernel.
template <class T, int CM>
auto mode_pass_kernel(int N, bool first, int slots) {
    constexpr int S = kRowSlots;
    if constexpr (CM > 1)  // CM = 1: k_pass_one
        if (N == 3) return first ? k_mode_pass<T, CM, 2, true, S> : k_mode_pass<T, CM, 2, false, S>;
    if constexpr (sizeof(T) == 4)
        if (N == 5) {
            if (slots == 1)
                return first ? k_mode_pass<T, CM, 4, true, 1> : k_mode_pass<T, CM, 4, false, 1>;
            return first ? k_mode_pass<T, CM, 4, true, S> : k_mode_pass<T, CM, 4, false, S>;
        }
    return first ? k_mode_pass<T, CM, 0, true, S> : k_mode_pass<T, CM, 0, false, S>;
}

// Plan of a mode-n pass: one block per SM with as many warps as fit (up to
// pass_max_warps); the shared memory the rings leave is L1 cache.  Float five-way tensors
// take one row slot per warp where two would leave fewer than pass_max_warps: C = 10, modes
// of 1e6 rows, 2e7 entries, passes with 9 to 5 warps of two slots 3.5 to 5.1 ms, 2.35 to 2.8
// ms with 12 to 10 warps of one (and the cheaper ends of items, finish_item).
template <class T, int CM, bool FIRST>
PassPlan mode_pass_plan_cm(int N, int n, int num_sms, int P) {
    constexpr size_t kReserve = 1024;  // static shared memory of the kernel
    int dev = 0, smem_blk = 0;
    TFS_CUDA(cudaGetDevice(&dev));
    TFS_CUDA(cudaDeviceGetAttribute(&smem_blk, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev));
    PassPlan plan;
    if (CM == 1 && N == 3) {  // k_pass_one
        // fewer bins than warps: spread over the SMs (300 x 200 x 100, 20,000 entries, 313 bins:
        // a sweep 71 us in ten blocks of 32 warps, 65 now, 60 with the staged pass and its solves)
        plan.warps = std::min(kOneWarps, std::max(1, (P + num_sms - 1) / num_sms));
        plan.grid = std::max(1, std::min(num_sms, (P + plan.warps - 1) / plan.warps));
        return plan;
    }
    const size_t room = (size_t)smem_blk - kReserve;
    auto fit = [&](int slots) {
        return (int)std::min<size_t>(pass_max_warps<T, CM>(),
                                     room / pass_warp_bytes<T, CM, FIRST>(N, n, slots));
    };
    plan.warps = fit(kRowSlots);
    if (sizeof(T) == 4 && N == 5 && fit(1) > plan.warps) {
        plan.slots = 1;
        plan.warps = fit(1);
    }
    if (plan.warps < 1) throw ApiError{TF_EINVAL, "mode pass does not fit in shared memory"};
    plan.smem = (size_t)plan.warps * pass_warp_bytes<T, CM, FIRST>(N, n, plan.slots);
    plan.grid = std::max(1, std::min(num_sms, (P + plan.warps - 1) / plan.warps));
    return plan;
}

template <class T, int CM>
void launch_mode_pass_cm(const PassArgs<T> &a, const PassPlan &plan, cudaStream_t st) {
    if constexpr (CM == 1) {
        if (a.N == 3) {
            if (a.first)
                k_pass_one<T, true><<<plan.grid, plan.warps * kWarp, 0, st>>>(a);
            else
                k_pass_one<T, false><<<plan.grid, plan.warps * kWarp, 0, st>>>(a);
            TFS_CUDA(cudaGetLastError());
            return;
        }
    }
    auto kern = mode_pass_kernel<T, CM>(a.N, a.first != 0, plan.slots);
    TFS_CUDA(raise_smem_limit((const void *)kern, (int)plan.smem));
    kern<<<plan.grid, plan.warps * kWarp, plan.smem, st>>>(a);
    TFS_CUDA(cudaGetLastError());
}

template <class T, int CM>
void launch_solve_rows_cm(const PassArgs<T> &a, const SolveRows &rows, cudaStream_t st) {
    SolveRows r = rows;
    if (CM * (CM + 1) / 2 + CM < 32) {
        // fewer values than lanes: a warp would leave lanes idle and walk the slots in more
        // rounds than a block (C = 1, 2,000 medium rows: 10 against 8 us; C = 5 in FP64, 100
        // rows: 18 against 14.5; the other way at C = 10, 1,500 rows: 60 against 70)
        r.n_heavy += r.n_medium;
        r.n_medium = 0;
    }
    const int64_t blocks = r.n_heavy + (r.n_medium + kMediumRows - 1) / kMediumRows +
                           ((int64_t)r.n_single + r.n_light + kSolveThreads - 1) / kSolveThreads;
    if (blocks <= 0) return;
    const bool xs = sizeof(T) == 4 && (a.refine || a.cond_limit > 0.f);
    auto kern = xs ? k_solve_rows<T, CM, true> : k_solve_rows<T, CM, false>;
    constexpr size_t smem = solve_rows_smem<T, CM>();
    TFS_CUDA(raise_smem_limit((const void *)kern, (int)smem));
    kern<<<(unsigned)blocks, kSolveThreads, smem, st>>>(a, r);
    TFS_CUDA(cudaGetLastError());
}

template <class T, int CM>
int res_warps(int N) {
    return best_warps_per_block(res_warp_bytes<T, CM>(N));
}

template <class T, int CM>
void launch_res_cm(const ResArgs<T> &a, cudaStream_t st) {
    const int wpb = res_warps<T, CM>(a.N);
    const size_t smem = wpb * res_warp_bytes<T, CM>(a.N);
    auto kern = k_res<T, CM, 0>;
    if constexpr (res_no<T>(5) == 4)
        if (a.N == 5) kern = k_res<T, CM, 4>;
    TFS_CUDA(raise_smem_limit((const void *)kern, (int)smem));
    kern<<<res_blocks(a.P, wpb), wpb * kWarp, smem, st>>>(a);
    TFS_CUDA(cudaGetLastError());
}

template <class T, int CM>
int res_blocks_cm(int P, int N) {
    return res_blocks(P, res_warps<T, CM>(N));
}

#define TFS_FOR_EACH_CM(X) X(1) X(2) X(4) X(6) X(8) X(10) X(12) X(16)

template <class T>
void launch_mode_pass_impl(const PassArgs<T> &a, int CM, const PassPlan &plan, cudaStream_t st) {
    switch (CM) {
#define TFS_CASE(cm)                             \
    case cm:                                     \
        launch_mode_pass_cm<T, cm>(a, plan, st); \
        return;
        TFS_FOR_EACH_CM(TFS_CASE)
#undef TFS_CASE
        default:
            throw ApiError{TF_EINVAL, "no mode-pass instance for this C"};
    }
}

template <class T>
PassPlan mode_pass_plan_impl(int CM, int N, int n, bool first, int num_sms, int P) {
    switch (CM) {
#define TFS_CASE(cm)                                                       \
    case cm:                                                               \
        return first ? mode_pass_plan_cm<T, cm, true>(N, n, num_sms, P)    \
                     : mode_pass_plan_cm<T, cm, false>(N, n, num_sms, P);
        TFS_FOR_EACH_CM(TFS_CASE)
#undef TFS_CASE
        default:
            throw ApiError{TF_EINVAL, "no mode-pass instance for this C"};
    }
}

template <class T>
void launch_solve_rows_impl(const PassArgs<T> &a, int CM, const SolveRows &r, cudaStream_t st) {
    switch (CM) {
#define TFS_CASE(cm)                             \
    case cm:                                     \
        launch_solve_rows_cm<T, cm>(a, r, st);   \
        return;
        TFS_FOR_EACH_CM(TFS_CASE)
#undef TFS_CASE
        default:
            throw ApiError{TF_EINVAL, "no solve instance for this C"};
    }
}

template <class T>
void launch_res_impl(const ResArgs<T> &a, int CM, cudaStream_t st) {
    switch (CM) {
#define TFS_CASE(cm)                 \
    case cm:                         \
        launch_res_cm<T, cm>(a, st); \
        return;
        TFS_FOR_EACH_CM(TFS_CASE)
#undef TFS_CASE
        default:
            if (CM > 16) {
                launch_res_wide<T>(a, slice_stride_elems(CM, (int)sizeof(T)), st);
                return;
            }
            throw ApiError{TF_EINVAL, "no residual instance for this C"};
    }
}

template <class T>
int res_blocks_impl(int CM, int P, int N) {
    switch (CM) {
#define TFS_CASE(cm) \
    case cm:         \
        return res_blocks_cm<T, cm>(P, N);
        TFS_FOR_EACH_CM(TFS_CASE)
#undef TFS_CASE
        default:
            if (CM > 16) return res_wide_blocks(P);
            throw ApiError{TF_EINVAL, "no residual instance for this C"};
    }
}

}  // namespace tfs

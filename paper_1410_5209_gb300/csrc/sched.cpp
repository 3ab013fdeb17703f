// Host-side row scheduling: the GPU counterpart of the paper's greedy row assignment
// (Algorithm 3, Section 3.3).  The paper balances |mOmega^(n)| (entries per machine)
// because the slowest machine sets each step's time; here the "machines" are bins of
// warps on the GPU.  The default policy is LPT without the paper's row cap (the cap
// only bounded the parameter broadcast of the MapReduce design) and with rows longer
// than a cap split into chunks whose partial Gram/rhs are summed before the solve.
// The paper's own policy (row cap and both tie-breaks) and its SEQ / RAN baselines
// (Section 5.5) are kept for comparison.
#include <stdint.h>

#include <algorithm>
#include <numeric>
#include <queue>
#include <tuple>
#include <vector>

#include "../../include/tf_sals.h"

namespace tfs {
namespace {

uint64_t splitmix(uint64_t z) {
    z += 0x9E3779B97F4A7C15ull;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}

// Bin key in the order the paper's Algorithm 3 prefers machines: fewest entries of
// this mode, then fewest rows of this mode, then fewest entries over all modes so far,
// then the lowest index.
struct BinKey {
    int64_t load, rows, total;
    int32_t bin;
    bool operator>(const BinKey &o) const {
        return std::tie(load, rows, total, bin) > std::tie(o.load, o.rows, o.total, o.bin);
    }
};
using MinHeap = std::priority_queue<BinKey, std::vector<BinKey>, std::greater<BinKey>>;

// (complemented length << 32 | index) of len[0 .. n) in increasing order: decreasing length,
// equal lengths in increasing index.  Short lengths take one counting sort; otherwise a
// least-significant-digit radix sort of the length (11-bit digits, all counted in the pass
// that builds the keys), skipping digits that every key shares.
constexpr int64_t key_index(uint64_t key) { return (int64_t)(uint32_t)key; }
constexpr int64_t key_length(uint64_t key) { return (int64_t)(UINT32_MAX - (uint32_t)(key >> 32)); }

template <class Len>
std::vector<uint64_t> keys_by_length(const Len *len, size_t n) {
    auto key_of = [&](size_t i) {
        return (uint64_t)(UINT32_MAX - (uint32_t)len[i]) << 32 | (uint32_t)i;
    };
    std::vector<uint64_t> key(n);
    uint32_t max_len = 0;
    for (size_t i = 0; i < n; ++i) max_len = std::max(max_len, (uint32_t)len[i]);
    if ((uint64_t)max_len <= 4 * (uint64_t)n + 1024) {
        std::vector<uint32_t> start((size_t)max_len + 2, 0);
        for (size_t i = 0; i < n; ++i) start[max_len - (uint32_t)len[i] + 1] += 1;
        for (size_t v = 0; v <= max_len; ++v) start[v + 1] += start[v];
        for (size_t i = 0; i < n; ++i) key[start[max_len - (uint32_t)len[i]]++] = key_of(i);
        return key;
    }
    constexpr int kBits = 11, kBuckets = 1 << kBits;
    std::vector<uint64_t> other(n);
    std::vector<uint32_t> cnt(3 * (kBuckets + 1), 0);
    for (size_t i = 0; i < n; ++i) {
        key[i] = key_of(i);
        for (int d = 0; d < 3; ++d)
            cnt[(size_t)(d * (kBuckets + 1)) + ((key[i] >> (32 + d * kBits)) & (kBuckets - 1)) + 1] += 1;
    }
    for (int d = 0; d < 3; ++d) {
        uint32_t *c = cnt.data() + d * (kBuckets + 1);
        bool one_bucket = false;
        for (int q = 0; q < kBuckets; ++q) one_bucket = one_bucket || c[q + 1] == n;
        if (one_bucket) continue;
        for (int q = 0; q < kBuckets; ++q) c[q + 1] += c[q];
        for (size_t i = 0; i < n; ++i) other[c[(key[i] >> (32 + d * kBits)) & (kBuckets - 1)]++] = key[i];
        key.swap(other);
    }
    return key;
}

// Rows in decreasing length, equal lengths in increasing index; lengths or rows beyond 32
// bits take a comparison sort.
std::vector<int64_t> rows_by_length(const int64_t *len, int64_t I) {
    std::vector<int64_t> order((size_t)I);
    bool narrow = I <= (int64_t)UINT32_MAX;
    for (int64_t i = 0; i < I; ++i) narrow = narrow && len[i] >= 0 && len[i] <= (int64_t)UINT32_MAX;
    if (narrow) {
        const std::vector<uint64_t> keys = keys_by_length(len, (size_t)I);
        for (int64_t i = 0; i < I; ++i) order[(size_t)i] = key_index(keys[(size_t)i]);
        return order;
    }
    std::iota(order.begin(), order.end(), 0);
    std::stable_sort(order.begin(), order.end(), [&](int64_t a, int64_t b) { return len[a] > len[b]; });
    return order;
}

// LPT: every job, longest first, to the bin with the least load (lowest index on ties).
// A job's load is its entries plus kItemCost: every item has a fixed cost in the mode
// pass (its first step, its partial write), so the many short or empty rows of a tensor
// spread over the bins instead of piling into whichever bin is least loaded last.
//   The loads of all bins lie within the longest job's cost of each other, so they are kept in
// a ring of buckets, one per load: the bins of the lowest bucket take the next jobs in index
// order (a job's cost is positive, so the bucket gains no bin meanwhile) and move on.  A heap
// (4-ary, packed keys) took 7.6 ms for 114,000 jobs on 19,456 bins on the GPU's host, the
// slowest part of a build of 3e7 entries.
constexpr int64_t kItemCost = 32;
// len(k): entries of the k-th job, longest first; put(k, bin) receives its bin.
template <class Len, class Put>
void lpt_bins(int64_t jobs, int64_t longest, int M, Len len, Put put) {
    const int64_t ring = longest + kItemCost + 1;
    if (ring <= (int64_t(1) << 20)) {
        std::vector<int32_t> head((size_t)ring, -1), next((size_t)M), now((size_t)M);
        std::vector<uint64_t> bits((size_t)(M + 63) / 64, 0);
        for (int m = 0; m < M; ++m) now[(size_t)m] = m;
        int64_t k = 0, load = 0;  // load: the lowest bucket's place in the ring
        size_t n = (size_t)M;
        for (;;) {
            for (size_t i = 0; i < n; ++i) {
                if (k == jobs) return;
                const int32_t m = now[i];
                int64_t at = load + len(k) + kItemCost;
                if (at >= ring) at -= ring;
                put(k++, m);
                next[(size_t)m] = head[(size_t)at];
                head[(size_t)at] = m;
            }
            do
                if (++load == ring) load = 0;
            while (head[(size_t)load] < 0);
            // the bucket's bins in index order: through a bit per bin where they are many,
            // sorted (last in first out: often decreasing) where they are few
            n = 0;
            for (int32_t m = head[(size_t)load]; m >= 0; m = next[(size_t)m]) now[n++] = m;
            head[(size_t)load] = -1;
            if (n > bits.size()) {
                for (size_t i = 0; i < n; ++i) bits[(size_t)now[i] / 64] |= uint64_t(1) << (now[i] % 64);
                n = 0;
                for (size_t w = 0; w < bits.size(); ++w) {
                    for (uint64_t v = bits[w]; v; v &= v - 1)
                        now[n++] = (int32_t)(64 * w + (size_t)__builtin_ctzll(v));
                    bits[w] = 0;
                }
            } else if (n > 1) {
                std::reverse(now.begin(), now.begin() + (ptrdiff_t)n);
                std::sort(now.begin(), now.begin() + (ptrdiff_t)n);
            }
        }
    }
    // jobs too long for the ring: a min-heap of (load, bin), half the levels of a binary one
    std::vector<std::pair<int64_t, int32_t>> heap((size_t)M);
    for (int m = 0; m < M; ++m) heap[(size_t)m] = {0, m};  // already a min-heap
    for (int64_t k = 0; k < jobs; ++k) {
        auto v = heap[0];
        put(k, v.second);
        v.first += len(k) + kItemCost;
        size_t i = 0;
        for (;;) {
            const size_t c0 = 4 * i + 1, cend = std::min(c0 + 4, heap.size());
            if (c0 >= heap.size()) break;
            size_t c = c0;
            for (size_t q = c0 + 1; q < cend; ++q)
                if (heap[q] < heap[c]) c = q;
            if (!(heap[c] < v)) break;
            heap[i] = heap[c];
            i = c;
        }
        heap[i] = v;
    }
}

// Greedy assignment of one mode's jobs to M bins.  cap_rows < 0 means no row cap.
// totals (size M) carries |mOmega| across modes and is updated.
void greedy_bins(const std::vector<int64_t> &job_len, const std::vector<int64_t> &order, int M,
                 int64_t cap_rows, std::vector<int64_t> &totals, std::vector<int32_t> &bin_of_job) {
    std::vector<int64_t> load(M, 0), rows(M, 0);
    MinHeap heap;
    for (int m = 0; m < M; ++m) heap.push({0, 0, totals[m], m});
    bin_of_job.assign(job_len.size(), -1);
    for (int64_t j : order) {
        BinKey k = heap.top();
        heap.pop();
        const int m = k.bin;
        bin_of_job[j] = m;
        load[m] += job_len[j];
        rows[m] += 1;
        totals[m] += job_len[j];
        if (cap_rows < 0 || rows[m] < cap_rows) heap.push({load[m], rows[m], totals[m], m});
    }
}

}  // namespace

tf_status assign_rows_impl(tf_sched_policy policy, int N, const int64_t *dims,
                           const int64_t *const *row_nnz, int M, uint64_t seed,
                           int32_t *const *assign) {
    if (N < 1 || M < 1 || !dims || !row_nnz || !assign) return TF_EINVAL;
    std::vector<int64_t> totals(M, 0);
    for (int n = 0; n < N; ++n) {
        const int64_t I = dims[n];
        if (I < 0) return TF_EINVAL;
        switch (policy) {
            case TF_SCHED_GREEDY:
            case TF_SCHED_LPT: {
                std::vector<int64_t> len(row_nnz[n], row_nnz[n] + I);
                std::vector<int64_t> order = rows_by_length(len.data(), I);
                std::vector<int32_t> bin;
                const int64_t cap = policy == TF_SCHED_GREEDY ? (I + M - 1) / M : -1;
                greedy_bins(len, order, M, cap, totals, bin);
                for (int64_t i = 0; i < I; ++i) assign[n][i] = bin[i];
                break;
            }
            case TF_SCHED_SEQ:
                // m-th range: I*m/M <= i < I*(m+1)/M (0-based form of the paper's SEQ)
                for (int m = 0; m < M; ++m)
                    for (int64_t i = I * m / M; i < I * (m + 1) / M; ++i) assign[n][i] = m;
                break;
            case TF_SCHED_RAN:
                for (int64_t i = 0; i < I; ++i)
                    assign[n][i] = (int32_t)(splitmix(seed ^ splitmix((uint64_t)n << 40 ^ i)) % M);
                break;
            default:
                return TF_EINVAL;
        }
    }
    return TF_OK;
}

std::vector<int64_t> rows_by_degree(const std::vector<int64_t> &count) {
    return rows_by_length(count.data(), (int64_t)count.size());
}

tf_status plan_mode(const int64_t *off, int64_t I, int P, int64_t cap, tf_sched_policy policy,
                    uint64_t seed, std::vector<tf_item> &items, int64_t &n_slots,
                    std::vector<int64_t> &bin_ptr) {
    if (I < 0 || P < 1 || cap < 0) return TF_EINVAL;
    const int64_t nnz = I > 0 ? off[I] : 0;
    if (cap == 0) cap = std::max<int64_t>(1, (nnz + P - 1) / P);

    // an item's length is 32 bits: a whole row's, or that of a long row's chunks
    for (int64_t i = 0; i < I; ++i) {
        const int64_t len = off[i + 1] - off[i];
        const int64_t chunks = policy == TF_SCHED_LPT && len > cap ? (len + cap - 1) / cap : 1;
        if (len > INT32_MAX && (len + chunks - 1) / chunks > INT32_MAX) return TF_EINVAL;
    }
    if (policy == TF_SCHED_LPT) {
        // jobs: whole rows, or near-equal chunks of rows longer than cap; one slot each, in
        // row order, so a job's number is its slot
        auto each_job = [&](auto f) {
            int64_t job = 0;
            for (int64_t i = 0; i < I; ++i) {
                const int64_t len = off[i + 1] - off[i];
                if (len <= cap) {
                    f(job++, i, off[i], (int32_t)len);
                    continue;
                }
                const int64_t k = (len + cap - 1) / cap, base = len / k, rem = len % k;
                for (int64_t c = 0, at = off[i]; c < k; ++c) {
                    const int64_t l = base + (c < rem ? 1 : 0);
                    f(job++, i, at, (int32_t)l);
                    at += l;
                }
            }
            return job;
        };
        std::vector<int32_t> len;
        len.reserve((size_t)I + (size_t)P + 16);
        n_slots = each_job([&](int64_t, int64_t, int64_t, int32_t l) { len.push_back(l); });
        const std::vector<uint64_t> keys = keys_by_length(len.data(), len.size());
        // a job's bin and its place in it: bins receive jobs longest first
        std::vector<uint64_t> place(len.size());
        std::vector<uint32_t> count((size_t)P, 0);
        auto put = [&](int64_t k, int32_t m) {
            place[(size_t)key_index(keys[(size_t)k])] = (uint64_t)m << 32 | count[(size_t)m]++;
        };
        if (P < (1 << 21)) {
            lpt_bins(n_slots, n_slots > 0 ? key_length(keys[0]) : 0, P,
                     [&](int64_t k) { return key_length(keys[(size_t)k]); }, put);
        } else {  // without the cost per item
            std::vector<int64_t> len64(len.begin(), len.end()), order, totals((size_t)P, 0);
            for (uint64_t k : keys) order.push_back(key_index(k));
            std::vector<int32_t> bin;
            greedy_bins(len64, order, P, -1, totals, bin);
            for (int64_t k = 0; k < n_slots; ++k) put(k, bin[(size_t)order[(size_t)k]]);
        }
        bin_ptr.assign((size_t)P + 1, 0);
        for (int p = 0; p < P; ++p) bin_ptr[(size_t)p + 1] = bin_ptr[(size_t)p] + count[(size_t)p];
        items.resize(len.size());
        each_job([&](int64_t job, int64_t row, int64_t begin, int32_t l) {
            const uint64_t at = place[(size_t)job];
            const int32_t m = (int32_t)(at >> 32);
            items[(size_t)bin_ptr[(size_t)m] + (uint32_t)at] = {begin, l, (int32_t)row, (int32_t)job, m};
        });
        return TF_OK;
    }
    std::vector<tf_item> jobs;
    jobs.reserve((size_t)I);
    n_slots = 0;
    for (int64_t i = 0; i < I; ++i)
        jobs.push_back({off[i], (int32_t)(off[i + 1] - off[i]), (int32_t)i, (int32_t)n_slots++, -1});
    std::vector<int32_t> bin(jobs.size(), 0);
    switch (policy) {
        case TF_SCHED_GREEDY: {
            std::vector<int64_t> len(jobs.size());
            for (size_t j = 0; j < jobs.size(); ++j) len[j] = jobs[j].len;
            std::vector<int64_t> order = rows_by_length(len.data(), (int64_t)len.size());
            std::vector<int64_t> totals(P, 0);
            greedy_bins(len, order, P, (I + P - 1) / P, totals, bin);
            // bins receive jobs longest first: keep that order inside each bin (grouped
            // by bin in the same pass)
            bin_ptr.assign((size_t)P + 1, 0);
            for (size_t j = 0; j < jobs.size(); ++j) bin_ptr[bin[j] + 1] += 1;
            for (int p = 0; p < P; ++p) bin_ptr[p + 1] += bin_ptr[p];
            std::vector<int64_t> fill(bin_ptr.begin(), bin_ptr.end() - 1);
            items.resize(jobs.size());
            for (int64_t j : order) {
                tf_item it = jobs[j];
                it.bin = bin[j];
                items[(size_t)fill[it.bin]++] = it;
            }
            return TF_OK;
        }
        case TF_SCHED_SEQ:
            for (auto &it : jobs) it.bin = (int32_t)(((int64_t)it.row * P) / std::max<int64_t>(I, 1));
            break;
        case TF_SCHED_RAN:
            for (auto &it : jobs) it.bin = (int32_t)(splitmix(seed ^ (uint64_t)it.row) % P);
            break;
        default:
            return TF_EINVAL;
    }
    // group by bin, keeping the assignment order within a bin (a counting sort)
    bin_ptr.assign((size_t)P + 1, 0);
    for (const auto &it : jobs) bin_ptr[it.bin + 1] += 1;
    for (int p = 0; p < P; ++p) bin_ptr[p + 1] += bin_ptr[p];
    std::vector<int64_t> fill(bin_ptr.begin(), bin_ptr.end() - 1);
    items.resize(jobs.size());
    for (const auto &it : jobs) items[(size_t)fill[it.bin]++] = it;
    return TF_OK;
}

}  // namespace tfs

extern "C" {

tf_status tf_assign_rows(tf_sched_policy policy, int N, const int64_t *dims,
                         const int64_t *const *row_nnz, int M, uint64_t seed,
                         int32_t *const *assign) {
    try {
        return tfs::assign_rows_impl(policy, N, dims, row_nnz, M, seed, assign);
    } catch (...) {
        return TF_ENOMEM;
    }
}

tf_status tf_plan_mode(const int64_t *off, int64_t I, int P, int64_t cap,
                       tf_sched_policy policy, uint64_t seed, tf_item *items,
                       int64_t max_items, int64_t *n_items, int64_t *n_slots,
                       int64_t *bin_ptr) {
    if (!off || !n_items || !n_slots) return TF_EINVAL;
    try {
        std::vector<tf_item> v;
        std::vector<int64_t> bp;
        int64_t slots = 0;
        tf_status st = tfs::plan_mode(off, I, P, cap, policy, seed, v, slots, bp);
        if (st != TF_OK) return st;
        *n_items = (int64_t)v.size();
        *n_slots = slots;
        if ((int64_t)v.size() > max_items || !items) return TF_ENOMEM;
        std::copy(v.begin(), v.end(), items);
        if (bin_ptr) std::copy(bp.begin(), bp.end(), bin_ptr);
        return TF_OK;
    } catch (...) {
        return TF_ENOMEM;
    }
}

const char *tf_version(void) { return "sals-gb300 0.1"; }

}  // extern "C"

// hpd_build_meta: per-step int32 bookkeeping tables and the attention work list (device side).
//
// On the caller's stream, no host synchronisation.  Steps with up to 4096 documents and 65536 slots take one
// launch (meta_step_kernel); larger ones three:
//   doc_scan_kernel   exclusive scans over documents (prefix tokens, slots)
//   compact_kernel    stable compaction of live slots -> row tables, rows-per-document CSR
//   plan_kernel       split-KV policy + work list for the attention kernel; -1 fill of table tails
#include "common.cuh"

namespace hpd {

namespace {

constexpr int kScanThreads = 1024;
constexpr int kCompactThreads = 256;
constexpr int kPlanThreads = 1024;

__device__ __forceinline__ int warp_incl_scan(int v) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        int t = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += t;
    }
    return v;
}

// Block-wide exclusive scan of one int per thread; returns the exclusive prefix and the block total.
template <int THREADS>
__device__ __forceinline__ int block_excl_scan(int v, int* smem /* THREADS/32 + 1 */, int& total) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int incl = warp_incl_scan(v);
    if (lane == 31) smem[warp] = incl;
    __syncthreads();
    if (warp == 0) {
        int w = (lane < THREADS / 32) ? smem[lane] : 0;
        int wi = warp_incl_scan(w);
        if (lane < THREADS / 32) smem[lane] = wi - w;
        if (lane == 31) smem[THREADS / 32] = wi;
    }
    __syncthreads();
    int res = incl - v + smem[warp];
    total = smem[THREADS / 32];
    __syncthreads();
    return res;
}

__global__ void __launch_bounds__(kScanThreads)
doc_scan_kernel(int n_docs, const int32_t* __restrict__ doc_prefix_len, const int32_t* __restrict__ doc_branch_cnt,
                int32_t* __restrict__ doc_kv_start, int32_t* __restrict__ doc_slot_start)
{
    __shared__ int sm[kScanThreads / 32 + 1];
    int run_kv = 0, run_sl = 0;
    for (int base = 0; base < n_docs; base += kScanThreads) {
        int d = base + threadIdx.x;
        int l = d < n_docs ? doc_prefix_len[d] : 0;
        int c = d < n_docs ? doc_branch_cnt[d] : 0;
        int tot;
        int el = block_excl_scan<kScanThreads>(l, sm, tot);
        int tl = tot;
        int ec = block_excl_scan<kScanThreads>(c, sm, tot);
        if (d < n_docs) {
            doc_kv_start[d] = run_kv + el;
            doc_slot_start[d] = run_sl + ec;
        }
        run_kv += tl;
        run_sl += tot;
    }
    if (threadIdx.x == 0) {
        doc_kv_start[n_docs] = run_kv;
        doc_slot_start[n_docs] = run_sl;
    }
}

// Each block owns kCompactThreads consecutive slots.  The number of live slots before the block is
// recounted by the block itself (reads at most n_slots bytes from L2), which keeps the kernel free of
// any inter-block dependency.
__global__ void __launch_bounds__(kCompactThreads)
compact_kernel(int n_docs, int n_slots, int32_t suffix_cap, int32_t pos_gap,
               const int32_t* __restrict__ doc_prefix_len, const int32_t* __restrict__ doc_branch_cnt,
               const int32_t* __restrict__ doc_slot_start,
               const int32_t* __restrict__ slot_depth, const uint8_t* __restrict__ slot_alive,
               const int32_t* __restrict__ slot_vis /* nullable: anchor = document length */,
               int32_t* __restrict__ doc_active_start, int32_t* __restrict__ active_slot,
               int32_t* __restrict__ doc_id, int32_t* __restrict__ branch_start, int32_t* __restrict__ pos_id,
               int32_t* __restrict__ suffix_off, int32_t* __restrict__ suffix_len,
               int32_t* __restrict__ prefix_vis /* nullable */, int32_t* __restrict__ n_active)
{
    __shared__ int sm[kCompactThreads / 32 + 1];
    const int first = blockIdx.x * kCompactThreads;

    // live slots in [0, first)
    int cnt = 0;
    {
        const uintptr_t addr = reinterpret_cast<uintptr_t>(slot_alive);
        int head = static_cast<int>((16 - (addr & 15)) & 15);
        if (head > first) head = first;
        for (int i = threadIdx.x; i < head; i += kCompactThreads) cnt += slot_alive[i] != 0;
        const int n_vec = (first - head) / 16;
        const uint4* v = reinterpret_cast<const uint4*>(slot_alive + head);
        for (int i = threadIdx.x; i < n_vec; i += kCompactThreads) {
            uint4 w = v[i];
            cnt += __popc(__vcmpne4(w.x, 0u) & 0x01010101u) + __popc(__vcmpne4(w.y, 0u) & 0x01010101u) +
                   __popc(__vcmpne4(w.z, 0u) & 0x01010101u) + __popc(__vcmpne4(w.w, 0u) & 0x01010101u);
        }
        for (int i = head + n_vec * 16 + threadIdx.x; i < first; i += kCompactThreads) cnt += slot_alive[i] != 0;
    }
    int before;
    {
        int tot;
        block_excl_scan<kCompactThreads>(cnt, sm, tot);
        before = tot;
    }

    const int s = first + threadIdx.x;
    const int alive = (s < n_slots) && slot_alive[s] != 0;
    int tot;
    const int excl = before + block_excl_scan<kCompactThreads>(alive, sm, tot);
    const int block_end = before + tot;

    if (s < n_slots) {
        // document of slot s: last d with doc_slot_start[d] <= s (documents without slots are skipped
        // automatically because their start equals the next document's start)
        int lo = 0, hi = n_docs;           // invariant: doc_slot_start[lo] <= s < doc_slot_start[hi]
        while (hi - lo > 1) {
            int mid = (lo + hi) >> 1;
            if (doc_slot_start[mid] <= s) lo = mid; else hi = mid;
        }
        const int d = lo;
        const int j = s - doc_slot_start[d];
        if (j == 0) {
            // first slot of document d: rows before it; empty documents just before d share the value
            doc_active_start[d] = excl;
            for (int e = d - 1; e >= 0 && doc_branch_cnt[e] == 0; --e) doc_active_start[e] = excl;
        }
        if (alive) {
            const int depth = slot_depth[s];
            const int anchor = slot_vis ? slot_vis[s] : doc_prefix_len[d];
            const int bs = anchor + j * pos_gap;
            active_slot[excl] = s;
            doc_id[excl] = d;
            branch_start[excl] = bs;
            pos_id[excl] = bs + depth;
            suffix_off[excl] = s * suffix_cap;
            suffix_len[excl] = depth;
            if (prefix_vis) prefix_vis[excl] = anchor;
        }
    }
    if (blockIdx.x == gridDim.x - 1 && threadIdx.x == 0) {
        *n_active = block_end;
        doc_active_start[n_docs] = block_end;
        for (int e = n_docs - 1; e >= 0 && doc_branch_cnt[e] == 0; --e) doc_active_start[e] = block_end;
    }
}

// Split-KV policy.  A work item is (document, chunk of prefix tokens, block of <= 128/G branches).
// Documents are left whole unless the step has fewer items than SMs; then the largest chunk size
// 128 * 2^k that yields at least n_sm * Hkv^-1 items is taken, subject to the partial-result and
// work-list capacities of the workspace.  Chunks below 512 tokens are never taken: a chunk's fp32
// partial result and its merge then cost more than the chunk's keys (measured: batches of 2 to 4
// prompts with 512-token documents ran 10 % faster whole than in 128- or 256-token chunks).
constexpr int kCand = 9;             // chunk sizes 128 << 0..7, then "whole document"
constexpr int kMinCand = 2;          // smallest chunk size taken: 128 << 2 tokens

__device__ __forceinline__ int chunks_of(int L, int cand) {
    if (cand == kCand - 1 || L <= 0) return 1;
    constexpr int kShift = 7;                           // kTileN = 1 << 7
    static_assert(kTileN == 1 << kShift, "chunk sizes are powers of two");
    return static_cast<int>((static_cast<long long>(L) + (kTileN << cand) - 1) >> (kShift + cand));
}

// Longest units first.  The attention kernel hands units out in list order, a few per pipeline, so a long unit drawn
// late leaves one pipeline running after the others have finished.  Lists of up to kSortItems items (from up to
// kSortDocs documents) whose items differ in length are therefore written in descending order of an estimate of
// their duration: one per prefix key, a constant per branch-cache column of the rows (the cached lengths are not
// looked at: one pass over every row would cost more than it saves) and a constant per unit.  Ties keep document
// order, so the list is reproducible.  Longer lists stay in document order: their units are short against the launch.
constexpr int kSortItems = 2048;
constexpr int kSortDocs = 2048;
constexpr int kPlanScratchInts = kSortItems;                  // the sort keys
constexpr uint32_t kCostMax = 0xFFFFFu;                       // 20 bits of cost above 12 bits of item index
constexpr int kUnitCost = 2 * kTileN;                         // a unit's fixed part, in key columns
constexpr int kBranchCost = 16;                               // per row and q head of the group: its cached tokens' columns

// estimate of a unit's duration, in key columns: keys of the prefix chunk, rows whose branch caches the unit visits
__device__ __forceinline__ int unit_cost(int keys, int branch_rows, int G) {
    return min(kUnitCost + keys + branch_rows * G * kBranchCost, static_cast<int>(kCostMax));
}

// Bitonic sort by 1024 threads, ascending.  A thread holds the keys t and t + 1024 in registers: distances below 32 go
// through shuffles and 1024 through the thread itself, only 32..512 through shared memory (15 of the 55 stages of 1024
// keys; with every stage in shared memory behind a barrier of its own the sort was half of the table kernel's time).
// key: n2 keys (n2 a power of two, at most 2048); on return rank[key & 0xFFF] = place for the first n_items keys.
__device__ __forceinline__ uint32_t bitonic_keep(uint32_t mine, uint32_t other, int i, int j, int k)
{
    const bool low = (i & j) == 0, up = (i & k) == 0;
    return low == up ? min(mine, other) : max(mine, other);
}

__device__ __forceinline__ void rank_keys(uint32_t* key, int n2, int n_items, uint16_t* rank)
{
    const int t = threadIdx.x;
    const bool two = n2 > 1024;
    uint32_t e0 = t < n2 ? key[t] : 0xFFFFFFFFu, e1 = two ? key[t + 1024] : 0xFFFFFFFFu;
    for (int k = 2; k <= n2; k <<= 1) {
        for (int j = k >> 1; j > 0; j >>= 1) {
            if (j == 1024) {
                const uint32_t a = e0, b = e1;
                e0 = bitonic_keep(a, b, t, j, k);
                e1 = bitonic_keep(b, a, t + 1024, j, k);
            } else {
                uint32_t o0, o1 = 0;
                if (j < 32) {
                    o0 = __shfl_xor_sync(0xffffffffu, e0, j);
                    if (two) o1 = __shfl_xor_sync(0xffffffffu, e1, j);
                } else {
                    __syncthreads();                     // the previous exchange has been read
                    if (t < n2) key[t] = e0;
                    if (two) key[t + 1024] = e1;
                    __syncthreads();
                    o0 = t < n2 ? key[t ^ j] : 0xFFFFFFFFu;
                    if (two) o1 = key[(t ^ j) + 1024];
                }
                e0 = bitonic_keep(e0, o0, t, j, k);
                if (two) e1 = bitonic_keep(e1, o1, t + 1024, j, k);
            }
        }
    }
    __syncthreads();                                     // rank may share memory with nothing, but its readers wait here
    if (t < n_items) rank[e0 & 0xFFFu] = static_cast<uint16_t>(t);
    if (two && t + 1024 < n_items) rank[e1 & 0xFFFu] = static_cast<uint16_t>(t + 1024);
    __syncthreads();
}

// The same by counting, for short lists: a key's place is the number of smaller ones.  1024 / n2 threads share a key and compare it with
// an equal part of the others (n2^2 / 1024 comparisons a thread, read four at a time by all lanes of a warp alike), so nothing
// waits for anything but two barriers, where the bitonic network is 21 to 45 dependent stages.
// key: n2 keys (a power of two, 64 to kCountItems), key[w] being that of item w; cnt: n2 counters.
constexpr int kCountItems = 512;

__device__ __forceinline__ void count_ranks(const uint32_t* key, int n2, int n_items, uint32_t* cnt, uint16_t* rank)
{
    const int t = threadIdx.x, i = t & (n2 - 1), part = t / n2, len = n2 * n2 / kPlanThreads;
    if (t < n2) cnt[t] = 0;
    __syncthreads();
    const uint32_t mine = key[i];
    const uint4* other = reinterpret_cast<const uint4*>(key + part * len);
    uint32_t smaller = 0;
#pragma unroll 4
    for (int j = 0; j < len / 4; ++j) {
        const uint4 k = other[j];
        smaller += (k.x < mine) + (k.y < mine) + (k.z < mine) + (k.w < mine);
    }
    atomicAdd(&cnt[i], smaller);
    __syncthreads();
    if (t < n_items) rank[t] = static_cast<uint16_t>(cnt[t]);
    __syncthreads();
}

// Block-wide exclusive scan of one 64-bit word per thread (two packed ints) by 1024 threads behind ONE barrier: every warp
// scans the 32 warp totals for itself.  buf alternates between consecutive calls.
__device__ __forceinline__ long long scan_words(long long v, long long* buf, long long& total)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    long long incl = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const long long u = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += u;
    }
    if (lane == 31) buf[warp] = incl;
    __syncthreads();
    const long long w = buf[lane];
    long long wi = w;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const long long u = __shfl_up_sync(0xffffffffu, wi, o);
        if (lane >= o) wi += u;
    }
    total = __shfl_sync(0xffffffffu, wi, 31);
    return incl - v + __shfl_sync(0xffffffffu, wi - w, warp);
}
__device__ __forceinline__ long long words(int lo, int hi) { return static_cast<long long>(static_cast<unsigned>(lo)) | (static_cast<long long>(hi) << 32); }
__device__ __forceinline__ int word_lo(long long v) { return static_cast<int>(v & 0xffffffffll); }
__device__ __forceinline__ int word_hi(long long v) { return static_cast<int>(v >> 32); }

// The split-KV plan, run by ONE block of 1024 threads; the two document tables may be in shared or global memory.
// scratch: kPlanScratchInts ints of shared memory, rank: kSortItems entries.
// A serial chain of barriers and shuffles with little work in between: sums go through warp reductions, one candidate chunk
// size per warp, and one-barrier scans (the same sums as 64-bit shuffles and shared-memory atomics of all 32 warps took 5 us of
// the 12 us this kernel needed for a step of few documents).
__device__ __forceinline__ void plan_block(int n_docs, int G, int Hkv, int n_sm,
                                           const int32_t* doc_prefix_len, const int32_t* doc_active_start,
                                           int* scratch, uint16_t* rank,
                                           WsHeader* __restrict__ hdr, WorkItem* __restrict__ work, DocSplit* __restrict__ split,
                                           int work_cap, int part_cap)
{
    __shared__ long long buf[2][32];
    __shared__ long long s_items[kCand], s_prow[kCand];
    __shared__ int s_whole, s_cost_min, s_cost_max, s_choice;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int rows_per_block = kTileM / G;               // a power of two
    const int rb_shift = 31 - __clz(rows_per_block);
    auto rows_of = [&](int d) { return doc_active_start[d + 1] - doc_active_start[d]; };
    auto blocks_of = [&](int rows) { return (rows + rows_per_block - 1) >> rb_shift; };

    // the usual case first: whole documents already give one unit per SM or more -> nothing to weigh
    // (the same pass weighs the whole documents' units: only lists whose units differ in length are put in order below)
    if (threadIdx.x == 0) { s_whole = 0; s_cost_min = 0x7fffffff; s_cost_max = 0; }
    __syncthreads();
    for (int base = warp * 32; base < n_docs; base += kPlanThreads) {
        const int d = base + lane;
        int whole = 0, cmin = 0x7fffffff, cmax = 0;
        if (d < n_docs) {
            const int rows = rows_of(d);
            if (rows > 0) {
                whole = blocks_of(rows);
                const int L = min(max(doc_prefix_len[d], 0), static_cast<int>(kCostMax));
                cmin = unit_cost(L, rows - (whole - 1) * rows_per_block, G);
                cmax = unit_cost(L, min(rows, rows_per_block), G);
            }
        }
        whole = __reduce_add_sync(0xffffffffu, whole);
        cmin = __reduce_min_sync(0xffffffffu, cmin);
        cmax = __reduce_max_sync(0xffffffffu, cmax);
        if (lane == 0 && whole) { atomicAdd(&s_whole, whole); atomicMin(&s_cost_min, cmin); atomicMax(&s_cost_max, cmax); }
    }
    __syncthreads();
    const bool enough = static_cast<long long>(s_whole) * Hkv >= n_sm;
    // worth the sort only when the units differ: more than a quarter between the shortest and the longest, or the chunks of a split list
    bool differ = s_cost_max > s_cost_min && (s_cost_max - s_cost_min) * 4 > s_cost_max;
    int cand = kCand - 1;                                // whole documents
    if (!enough) {
        if (warp < kCand) {                              // warp c weighs chunk size c
            long long items = 0, prow = 0;
            for (int d = lane; d < n_docs; d += 32) {
                const int rows = rows_of(d);
                if (rows <= 0) continue;
                const int ch = chunks_of(doc_prefix_len[d], warp);
                items += static_cast<long long>(ch) * blocks_of(rows);
                if (ch > 1) prow += static_cast<long long>(ch) * rows;
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                items += __shfl_down_sync(0xffffffffu, items, o);
                prow += __shfl_down_sync(0xffffffffu, prow, o);
            }
            if (lane == 0) { s_items[warp] = items; s_prow[warp] = prow; }
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            int c = kCand - 1;
            while (c > kMinCand && s_items[c] * Hkv < n_sm) {
                const int nc = c - 1;
                if (s_items[nc] > work_cap || s_prow[nc] > part_cap) break;
                c = nc;
            }
            s_choice = c;
        }
        __syncthreads();
        cand = s_choice;
        differ |= s_prow[cand] > 0;
    }

    int parity = 0;
    // ---- order of the list: rank[item in document order] = its place, longest first ----
    bool sorted = false;
    if (n_docs <= kSortDocs && differ) {
        uint32_t* s_key = reinterpret_cast<uint32_t*>(scratch);
        int n_items = 0;
        for (int base = 0; base < n_docs; base += kPlanThreads) {
            const int d = base + threadIdx.x;
            int rows = 0, L = 0, mb = 0, ch = 0;
            if (d < n_docs) {
                rows = rows_of(d);
                L = doc_prefix_len[d];
                if (rows > 0) { mb = blocks_of(rows); ch = chunks_of(L, cand); }
            }
            long long tot;
            const int ei = n_items + word_lo(scan_words(ch * mb, buf[parity], tot));
            parity ^= 1;
            if (d < n_docs) {
                const int S = (cand == kCand - 1) ? L : (kTileN << cand);
                for (int c = 0, w = ei; c < ch; ++c) {
                    const int kc = max(min(S, L - c * S), 0);
                    for (int m = 0; m < mb; ++m, ++w) {
                        const int nr = min(rows_per_block, rows - m * rows_per_block);
                        const int cost = unit_cost(min(kc, static_cast<int>(kCostMax)), c == ch - 1 ? nr : 0, G);
                        if (w < kSortItems) s_key[w] = ((kCostMax - static_cast<uint32_t>(cost)) << 12) | static_cast<uint32_t>(w);
                    }
                }
            }
            n_items += word_lo(tot);
        }
        if (n_items > 1 && n_items <= kSortItems) {
            sorted = true;
            int n2 = 64;
            while (n2 < n_items) n2 <<= 1;
            for (int w = n_items + threadIdx.x; w < n2; w += kPlanThreads) s_key[w] = 0xFFFFFFFFu;
            __syncthreads();
            if (n2 <= kCountItems) count_ranks(s_key, n2, n_items, s_key + kCountItems, rank);
            else rank_keys(s_key, n2, n_items, rank);
        }
    }

    // emit the work list: exclusive scans of items and partial rows per document give an item's place in document
    // order, rank[] its place in the list
    int run_items = 0, run_part = 0, any_split = 0;
    for (int base = 0; base < n_docs; base += kPlanThreads) {
        const int d = base + threadIdx.x;
        int rows = 0, L = 0, mb = 0, ch = 0;
        if (d < n_docs) {
            rows = rows_of(d);
            L = doc_prefix_len[d];
            if (rows > 0) { mb = blocks_of(rows); ch = chunks_of(L, cand); }
        }
        long long tot;
        const long long ex = scan_words(words(ch * mb, ch > 1 ? ch * rows : 0), buf[parity], tot);
        parity ^= 1;
        const int ei = run_items + word_lo(ex), ep = run_part + word_hi(ex);
        if (d < n_docs) {
            split[d].part_base = ch > 1 ? ep : -1;
            split[d].n_chunks = ch;
            if (ch > 1) any_split = 1;
            const int S = (cand == kCand - 1) ? L : (kTileN << cand);
            int w = ei;
            for (int c = 0; c < ch; ++c) {
                const int kb = c * S;
                const int kc = min(S, L - kb);
                for (int m = 0; m < mb; ++m, ++w) {
                    WorkItem it;
                    it.doc = d;
                    it.key_begin = kb;
                    it.key_count = kc > 0 ? kc : 0;
                    it.row_begin = m * rows_per_block;
                    it.row_count = min(rows_per_block, rows - it.row_begin);
                    it.part_base = ch > 1 ? ep + c * rows : -1;
                    it.with_suffix = (c == ch - 1);
                    it.doc_row = doc_active_start[d];
                    work[sorted ? static_cast<int>(rank[w]) : w] = it;
                }
            }
        }
        run_items += word_lo(tot);
        run_part += word_hi(tot);
    }
    const int split_any = __syncthreads_or(any_split);
    if (threadIdx.x == 0) {
        hdr->n_work = run_items;
        hdr->chunk_tokens = (cand == kCand - 1) ? 0 : (kTileN << cand);
        hdr->n_part_rows = run_part;
        hdr->any_split = split_any;
        hdr->longest_first = sorted ? 1 : 0;
        hdr->ticket = 0;
        hdr->work_cap = work_cap;
        hdr->part_cap = part_cap;
    }
}

__global__ void __launch_bounds__(kPlanThreads)
plan_kernel(int n_docs, int n_slots, int G, int Hkv, int n_sm,
            const int32_t* __restrict__ doc_prefix_len, const int32_t* __restrict__ doc_active_start,
            const int32_t* __restrict__ n_active,
            int32_t* __restrict__ active_slot, int32_t* __restrict__ doc_id, int32_t* __restrict__ branch_start,
            int32_t* __restrict__ pos_id, int32_t* __restrict__ suffix_off, int32_t* __restrict__ suffix_len,
            int32_t* __restrict__ prefix_vis /* nullable */,
            WsHeader* __restrict__ hdr, WorkItem* __restrict__ work, DocSplit* __restrict__ split,
            int work_cap, int part_cap)
{
    if (blockIdx.x > 0) {
        // tail fill: entries past n_active read -1 in every per-row table
        const int na = *n_active;
        for (int i = na + (blockIdx.x - 1) * kPlanThreads + threadIdx.x; i < n_slots; i += (gridDim.x - 1) * kPlanThreads) {
            active_slot[i] = -1; doc_id[i] = -1; branch_start[i] = -1;
            pos_id[i] = -1; suffix_off[i] = -1; suffix_len[i] = -1;
            if (prefix_vis) prefix_vis[i] = -1;
        }
        return;
    }
    __shared__ __align__(16) int s_scratch[kPlanScratchInts];
    __shared__ uint16_t s_rank[kSortItems];
    plan_block(n_docs, G, Hkv, n_sm, doc_prefix_len, doc_active_start, s_scratch, s_rank,
                             hdr, work, split, work_cap, part_cap);
}

// ---------------------------------------------------------------------------------------------------------------
// All of the above in ONE launch without any dependency between blocks, for steps of at most kStepDocs documents and
// kStepSlots slots (the usual case).  The kernel is a chain of memory and barrier latencies, not of bytes, so every block
// repeats the cheap global steps for itself: the scans over documents, and the live flags of ALL slots as a bit mask with
// a prefix count per 32 slots, both in shared memory.  From there "live slots before s" is one lookup for any s: the row
// blocks place their 1024 slots' rows and -1 tail entries with it, and block 0 derives every document's row range and
// writes the split-KV plan from shared memory alone.  One round trip to memory in all; the earlier form, in which the
// last row block to finish (a counter in the workspace, cleared by a memset) wrote the plan, took four.
// ---------------------------------------------------------------------------------------------------------------
constexpr int kStepDocs = 4096;
constexpr int kStepSlots = 65536;                    // two mask words per thread
constexpr int kStepWords = kStepSlots / 32;

// bit i of the result: byte i of the word is not zero
__device__ __forceinline__ uint32_t nonzero_bytes(uint32_t w) {
    return ((__vcmpne4(w, 0u) & 0x08040201u) * 0x01010101u) >> 24;
}

// SHIFTED: the live flags do not begin on a 16-byte address (a slice of a larger buffer).  A kernel of its own, because the
// other form lost 1 to 7 % with both in one; single bytes took 29 us at 65536 slots, the pieces take 14.
template <bool SHIFTED>
__global__ void __launch_bounds__(kPlanThreads)
meta_step_kernel(int n_docs, int n_slots, int32_t suffix_cap, int32_t pos_gap, int G, int Hkv, int n_sm,
                 const int32_t* doc_prefix_len, const int32_t* doc_branch_cnt,
                 const int32_t* slot_depth, const uint8_t* slot_alive,
                 const int32_t* slot_vis /* nullable */,
                 int32_t* doc_kv_start, int32_t* doc_slot_start, int32_t* doc_active_start,
                 int32_t* active_slot, int32_t* doc_id, int32_t* branch_start,
                 int32_t* pos_id, int32_t* suffix_off, int32_t* suffix_len,
                 int32_t* prefix_vis /* nullable */,
                 int32_t* n_active, WsHeader* hdr, WorkItem* work, DocSplit* split,
                 int work_cap, int part_cap)
{
    __shared__ int s_start[kStepDocs + 1];           // first slot of every document; block 0 turns it into its first row
    __shared__ int s_len[kStepDocs];
    __shared__ __align__(16) uint32_t s_bits[kStepWords + kStepWords / 2];      // live mask, then the 16-bit prefix counts
    __shared__ long long s_scan[2][32];
    __shared__ int s_cnt[32];
    uint32_t* s_mask = s_bits;
    uint16_t* s_pre = reinterpret_cast<uint16_t*>(s_bits + kStepWords);
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const bool planner = blockIdx.x == 0;
    const int s = (static_cast<int>(blockIdx.x) - 1) * kPlanThreads + t;
    const bool mine = !planner && s < n_slots;

    start_dependents();
    await_predecessors();
    // ---- everything that is read from memory is asked for here ----
    const int depth = mine ? slot_depth[s] : 0;
    const int my_vis = (slot_vis && mine) ? slot_vis[s] : 0;
    int l = t < n_docs ? doc_prefix_len[t] : 0, c = t < n_docs ? doc_branch_cnt[t] : 0;
    uint32_t m[2] = {0u, 0u};                        // live flags of slots [64 t, 64 t + 64)
    if constexpr (SHIFTED) {
        // five pieces of 16 slots, the first from sh slots earlier, one load each where they lie inside the flags and single bytes at the two ends
        const int sh = static_cast<int>(reinterpret_cast<uintptr_t>(slot_alive) & 15), q0 = t * 64 - sh;
        if (q0 < n_slots) {
            uint4 w[5];
            unsigned long long lo = 0;                   // slots q0 .. q0 + 63
            uint32_t hi = 0, ends = 0;                   // slots from q0 + 64; pieces that lie inside in part
#pragma unroll
            for (int i = 0; i < 5; ++i) {
                const int q = q0 + 16 * i;
                w[i] = make_uint4(0, 0, 0, 0);
                if (q >= 0 && q + 16 <= n_slots) w[i] = *reinterpret_cast<const uint4*>(slot_alive + q);
                else if (q < n_slots) ends |= 1u << i;
            }
#pragma unroll 1
            while (ends) {
                const int i = __ffs(ends) - 1, q = q0 + 16 * i;
                ends &= ends - 1;
                uint32_t f = 0;
#pragma unroll
                for (int b = 0; b < 16; ++b)
                    if (q + b >= 0 && q + b < n_slots && slot_alive[q + b]) f |= 1u << b;
                if (i < 4) lo |= static_cast<unsigned long long>(f) << (16 * i); else hi |= f;
            }
#pragma unroll
            for (int i = 0; i < 5; ++i) {
                const uint32_t f = nonzero_bytes(w[i].x) | nonzero_bytes(w[i].y) << 4 | nonzero_bytes(w[i].z) << 8 | nonzero_bytes(w[i].w) << 12;
                if (i < 4) lo |= static_cast<unsigned long long>(f) << (16 * i); else hi |= f;
            }
            lo = lo >> sh | static_cast<unsigned long long>(hi) << (64 - sh);
            m[0] = static_cast<uint32_t>(lo); m[1] = static_cast<uint32_t>(lo >> 32);
        }
    } else if ((t + 1) * 64 <= n_slots) {
        const uint4* v = reinterpret_cast<const uint4*>(slot_alive) + t * 4;
        uint4 w[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) w[i] = v[i];
#pragma unroll
        for (int i = 0; i < 4; ++i)
            m[i >> 1] |= (nonzero_bytes(w[i].x) | nonzero_bytes(w[i].y) << 4 | nonzero_bytes(w[i].z) << 8 | nonzero_bytes(w[i].w) << 12) << (16 * (i & 1));
    } else {
        const int n = min(max(n_slots - t * 64, 0), 64);
#pragma unroll 8
        for (int i = 0; i < n; ++i)
            if (slot_alive[t * 64 + i]) m[i >> 5] |= 1u << (i & 31);
    }

    // ---- scans: live slots, and prefix tokens and slots per document (1024 documents at a time) ----
    const int pop = __popc(m[0]) + __popc(m[1]);
    int pop_incl = warp_incl_scan(pop);
    int run_kv = 0, run_sl = 0, total = 0;
    for (int base = 0; base == 0 || base < n_docs; base += kPlanThreads) {
        if (base > 0) {
            const int d = base + t;
            l = d < n_docs ? doc_prefix_len[d] : 0;
            c = d < n_docs ? doc_branch_cnt[d] : 0;
        }
        if (base == 0 && lane == 31) s_cnt[warp] = pop_incl;
        long long tot;
        // a count outside [0, n_slots] cannot be right and is clamped: the first slots index shared memory below
        const long long ex = scan_words(words(l, min(max(c, 0), n_slots)), s_scan[(base / kPlanThreads) & 1], tot);
        const int d = base + t;
        if (d < n_docs) {
            const int kv0 = run_kv + word_lo(ex), sl0 = run_sl + word_hi(ex);
            s_start[d] = sl0;
            s_len[d] = l;
            if (planner) { doc_kv_start[d] = kv0; doc_slot_start[d] = sl0; }
        }
        run_kv += word_lo(tot); run_sl += word_hi(tot);
        if (base == 0) {
            const int ct = s_cnt[lane];
            const int ci = warp_incl_scan(ct);
            const int excl = pop_incl - pop + __shfl_sync(0xffffffffu, ci - ct, warp);
            total = __shfl_sync(0xffffffffu, ci, 31);
            s_mask[2 * t] = m[0]; s_mask[2 * t + 1] = m[1];
            s_pre[2 * t] = static_cast<uint16_t>(excl);               // at most 65535 wherever a live slot may follow
            s_pre[2 * t + 1] = static_cast<uint16_t>(excl + __popc(m[0]));
        }
    }
    if (t == 0) {
        s_start[n_docs] = run_sl;
        if (planner) { doc_kv_start[n_docs] = run_kv; doc_slot_start[n_docs] = run_sl; }
    }
    __syncthreads();
    auto live_before = [&](int x) {                  // live slots below x
        if (x >= n_slots) return total;
        return static_cast<int>(s_pre[x >> 5]) + __popc(s_mask[x >> 5] & ((1u << (x & 31)) - 1u));
    };

    if (!planner) {
        if (!mine) return;
        int lo = 0, hi = n_docs;           // invariant: start[lo] <= s < start[hi]; documents without slots share a start and are skipped
        while (hi - lo > 1) {
            const int mid = (lo + hi) >> 1;
            if (s_start[mid] <= s) lo = mid; else hi = mid;
        }
        const int d = lo;
        const int j = s - s_start[d];
        const int excl = live_before(s);
        if ((s_mask[s >> 5] >> (s & 31)) & 1u) {
            const int anchor = slot_vis ? my_vis : (n_docs > 0 ? s_len[d] : 0);
            const int bs = anchor + j * pos_gap;
            active_slot[excl] = s;
            doc_id[excl] = d;
            branch_start[excl] = bs;
            pos_id[excl] = bs + depth;
            suffix_off[excl] = s * suffix_cap;
            suffix_len[excl] = depth;
            if (prefix_vis) prefix_vis[excl] = anchor;
        } else {
            const int x = total + (s - excl);        // the dead slots fill the tail of every row table with -1
            active_slot[x] = -1; doc_id[x] = -1; branch_start[x] = -1;
            pos_id[x] = -1; suffix_off[x] = -1; suffix_len[x] = -1;
            if (prefix_vis) prefix_vis[x] = -1;
        }
        return;
    }

    // ---- block 0: rows per document, then the plan ----
    for (int d = t; d <= n_docs; d += kPlanThreads) {
        const int r = d == n_docs ? total : live_before(s_start[d]);
        s_start[d] = r;
        doc_active_start[d] = r;
    }
    if (t == 0) *n_active = total;
    __syncthreads();                                 // the mask is not read any more: its memory serves the plan's sort
    static_assert(kPlanScratchInts * 4 + kSortItems * 2 <= sizeof(s_bits), "the sort's keys and ranks take the mask's place");
    plan_block(n_docs, G, Hkv, n_sm, s_len, s_start, reinterpret_cast<int*>(s_bits), reinterpret_cast<uint16_t*>(s_bits + kPlanScratchInts),
               hdr, work, split, work_cap, part_cap);
}

// ---------------------------------------------------------------------------------------------------------------
// First inference step (Sec. 4.3.2): the rows are the prompt tokens themselves.  One launch writes, per token, its
// group, Algorithm 2's position ID (a gap of pos_gap behind every attribute key: t + pos_gap * #{slots whose key ends
// before t}) and its causal bound t + 1; and the attention's work list: (group, block of 128/G tokens) against the
// keys [0, end of the block) -- later keys are masked for every row of the block, so they are not visited at all.
// ---------------------------------------------------------------------------------------------------------------
constexpr int kPrefillDocs = 2048;
constexpr int kPrefillThreads = 256;

__global__ void __launch_bounds__(kPrefillThreads)
prefill_meta_kernel(int n_docs, int G, int32_t pos_gap,
                    const int32_t* doc_prefix_len, const int32_t* doc_branch_cnt,
                    const int32_t* slot_vis,
                    int32_t* doc_kv_start, int32_t* doc_slot_start,
                    int32_t* tok_doc, int32_t* tok_pos, int32_t* tok_vis,
                    int32_t* n_tokens, WsHeader* hdr, WorkItem* work,
                    DocSplit* split, int work_cap, int part_cap)
{
    __shared__ int sm[kPrefillThreads / 32 + 1];
    __shared__ int s_kv[kPrefillDocs + 1], s_slot[kPrefillDocs + 1], s_item[kPrefillDocs + 1];
    const int rpb = kTileM / G;                      // tokens per row block
    start_dependents();
    await_predecessors();
    int run_kv = 0, run_sl = 0, run_it = 0;
    for (int base = 0; base < n_docs; base += kPrefillThreads) {
        const int d = base + threadIdx.x;
        const int l = d < n_docs ? doc_prefix_len[d] : 0;
        const int c = d < n_docs ? doc_branch_cnt[d] : 0;
        const int it = (l + rpb - 1) / rpb;
        int tl, tc, ti;
        const int el = block_excl_scan<kPrefillThreads>(l, sm, tl);
        const int ec = block_excl_scan<kPrefillThreads>(c, sm, tc);
        const int ei = block_excl_scan<kPrefillThreads>(it, sm, ti);
        if (d < n_docs) { s_kv[d] = run_kv + el; s_slot[d] = run_sl + ec; s_item[d] = run_it + ei; }
        run_kv += tl; run_sl += tc; run_it += ti;
    }
    if (threadIdx.x == 0) { s_kv[n_docs] = run_kv; s_slot[n_docs] = run_sl; s_item[n_docs] = run_it; }
    __syncthreads();
    const int n_tok = run_kv, n_items = min(run_it, work_cap);
    auto doc_of = [&](const int* start, int x) {      // last d with start[d] <= x (empty groups share a start and are skipped)
        int lo = 0, hi = n_docs;
        while (hi - lo > 1) {
            const int mid = (lo + hi) >> 1;
            if (start[mid] <= x) lo = mid; else hi = mid;
        }
        return lo;
    };
    const int stride = gridDim.x * kPrefillThreads;
    for (int x = blockIdx.x * kPrefillThreads + threadIdx.x; x < n_tok; x += stride) {
        const int d = doc_of(s_kv, x);
        const int t = x - s_kv[d];
        int lo = s_slot[d], hi = s_slot[d + 1];       // slots of the group whose key ends before token t: slot_vis <= t
        while (lo < hi) {
            const int mid = (lo + hi) >> 1;
            if (slot_vis[mid] <= t) lo = mid + 1; else hi = mid;
        }
        tok_doc[x] = d;
        tok_pos[x] = t + pos_gap * (lo - s_slot[d]);
        tok_vis[x] = t + 1;
    }
    for (int x = blockIdx.x * kPrefillThreads + threadIdx.x; x < n_items; x += stride) {
        const int d = doc_of(s_item, x);
        const int m = s_item[d + 1] - 1 - x;         // a prompt's last block has the most keys: longest first (step of 1 prompt 81 -> 71 us)
        const int L = s_kv[d + 1] - s_kv[d];
        WorkItem it;
        it.doc = d; it.key_begin = 0; it.key_count = min(L, (m + 1) * rpb);
        it.part_base = -1; it.row_begin = m * rpb; it.row_count = min(rpb, L - m * rpb);
        it.with_suffix = 0; it.doc_row = s_kv[d];
        work[x] = it;
    }
    if (blockIdx.x == 0) {
        for (int d = threadIdx.x; d <= n_docs; d += kPrefillThreads) {
            doc_kv_start[d] = s_kv[d];
            doc_slot_start[d] = s_slot[d];
            if (d < n_docs) { split[d].part_base = -1; split[d].n_chunks = 1; }
        }
        if (threadIdx.x == 0) {
            *n_tokens = n_tok;
            hdr->n_work = n_items; hdr->chunk_tokens = 0; hdr->n_part_rows = 0; hdr->any_split = 0;
            hdr->ticket = 0; hdr->work_cap = work_cap; hdr->part_cap = part_cap; hdr->longest_first = n_docs == 1;
        }
    }
}

}  // namespace

int launch_prefill_meta(const hpd_geom& g, int n_docs, int total_tokens, int32_t pos_gap, const int32_t* doc_prefix_len,
                        const int32_t* doc_branch_cnt, const int32_t* slot_vis, int32_t* doc_kv_start, int32_t* doc_slot_start,
                        int32_t* tok_doc, int32_t* tok_pos, int32_t* tok_vis, int32_t* n_tokens, void* workspace,
                        const WsLayout& lay, int n_sm, cudaStream_t stream)
{
    if (n_docs > kPrefillDocs) return HPD_E_CAPACITY;
    char* ws = static_cast<char*>(workspace);
    int blocks = (total_tokens + kPrefillThreads - 1) / kPrefillThreads;
    if (blocks < 1) blocks = 1;
    if (blocks > 4 * n_sm) blocks = 4 * n_sm;
    HPD_CUDA_TRY(launch_chained(prefill_meta_kernel, blocks, kPrefillThreads, 0, stream,
        n_docs, g.Hq / g.Hkv, pos_gap, doc_prefix_len, doc_branch_cnt, slot_vis, doc_kv_start, doc_slot_start, tok_doc, tok_pos,
        tok_vis, n_tokens, reinterpret_cast<WsHeader*>(ws), reinterpret_cast<WorkItem*>(ws + lay.off_work),
        reinterpret_cast<DocSplit*>(ws + lay.off_split), lay.work_cap, lay.part_cap));
    return HPD_OK;
}

WsLayout ws_layout(const hpd_geom& g, int max_docs, int max_slots, int n_sm)
{
    WsLayout l{};
    const int G = g.Hq / g.Hkv;
    const long long blocks = (static_cast<long long>(max_slots) * G + kTileM - 1) / kTileM;
    long long work_cap = 2ll * max_docs + 4 * (blocks + 1) + 2ll * n_sm + 64;
    long long part_cap = 2ll * max_slots + 1024;
    if (work_cap > 0x7fffffffll) work_cap = 0x7fffffffll;
    if (part_cap > 0x7fffffffll) part_cap = 0x7fffffffll;
    l.work_cap = static_cast<int32_t>(work_cap);
    l.part_cap = static_cast<int32_t>(part_cap);
    auto up = [](size_t x) { return (x + 255) & ~static_cast<size_t>(255); };
    size_t off = up(sizeof(WsHeader));
    l.off_work = off;  off = up(off + sizeof(WorkItem) * static_cast<size_t>(l.work_cap));
    l.off_split = off; off = up(off + sizeof(DocSplit) * static_cast<size_t>(max_docs > 0 ? max_docs : 1));
    l.off_ml = off;    off = up(off + sizeof(float) * 2 * static_cast<size_t>(l.part_cap) * g.Hq);
    l.off_o = off;     off = up(off + sizeof(float) * static_cast<size_t>(l.part_cap) * g.Hq * g.D);
    l.total = off;
    return l;
}

int launch_build_meta(const hpd_geom& g, int n_docs, int n_slots, const int32_t* doc_prefix_len,
                      const int32_t* doc_branch_cnt, const int32_t* slot_depth, const uint8_t* slot_alive,
                      int32_t pos_gap, int32_t* doc_kv_start, int32_t* doc_slot_start, int32_t* doc_active_start,
                      int32_t* active_slot, int32_t* doc_id, int32_t* branch_start, int32_t* pos_id,
                      int32_t* suffix_off, int32_t* suffix_len, int32_t* n_active, void* workspace,
                      const WsLayout& lay, int n_sm, int32_t* /*dev_status*/, cudaStream_t stream,
                      const int32_t* slot_vis, int32_t* prefix_vis)
{
    char* ws = static_cast<char*>(workspace);
    WsHeader* hdr = reinterpret_cast<WsHeader*>(ws);
    WorkItem* work = reinterpret_cast<WorkItem*>(ws + lay.off_work);
    DocSplit* split = reinterpret_cast<DocSplit*>(ws + lay.off_split);

    // one launch up to 4096 documents and 65536 slots: what a block can hold in shared memory (45 KB) and count in 16 bits
    if (n_docs <= kStepDocs && n_slots <= kStepSlots) {
        const int blocks = 1 + (n_slots + kPlanThreads - 1) / kPlanThreads;
        HPD_CUDA_TRY(launch_chained(aligned16(slot_alive) ? meta_step_kernel<false> : meta_step_kernel<true>, blocks, kPlanThreads, 0, stream,
            n_docs, n_slots, g.suffix_cap, pos_gap, g.Hq / g.Hkv, g.Hkv, n_sm, doc_prefix_len, doc_branch_cnt, slot_depth,
            slot_alive, slot_vis, doc_kv_start, doc_slot_start, doc_active_start, active_slot, doc_id, branch_start, pos_id,
            suffix_off, suffix_len, prefix_vis, n_active, hdr, work, split, lay.work_cap, lay.part_cap));
        return HPD_OK;
    }
    doc_scan_kernel<<<1, kScanThreads, 0, stream>>>(n_docs, doc_prefix_len, doc_branch_cnt, doc_kv_start, doc_slot_start);
    const int cblocks = n_slots > 0 ? (n_slots + kCompactThreads - 1) / kCompactThreads : 1;
    compact_kernel<<<cblocks, kCompactThreads, 0, stream>>>(
        n_docs, n_slots, g.suffix_cap, pos_gap, doc_prefix_len, doc_branch_cnt, doc_slot_start, slot_depth, slot_alive,
        slot_vis, doc_active_start, active_slot, doc_id, branch_start, pos_id, suffix_off, suffix_len, prefix_vis, n_active);
    int fill_blocks = (n_slots + kPlanThreads * 4 - 1) / (kPlanThreads * 4);
    if (fill_blocks < 1) fill_blocks = 1;
    if (fill_blocks > 64) fill_blocks = 64;
    plan_kernel<<<1 + fill_blocks, kPlanThreads, 0, stream>>>(
        n_docs, n_slots, g.Hq / g.Hkv, g.Hkv, n_sm, doc_prefix_len, doc_active_start, n_active, active_slot, doc_id,
        branch_start, pos_id, suffix_off, suffix_len, prefix_vis, hdr, work, split, lay.work_cap, lay.part_cap);
    HPD_CUDA_TRY(cudaGetLastError());
    return HPD_OK;
}

}  // namespace hpd

// Offline construction of a frozen table from a token corpus on the GPU (Section 4: the most frequent LC n-grams of
// length LL become the leaders; each keeps the FC most frequent n-grams of length FL that follow it).
//
// A window is LL + FL consecutive tokens; the corpus of N tokens has M = N - LL - FL + 1 of them.  Everything is counting
// and selection on integers, done without sorting:
//   1. leader counts: every window inserts-or-increments its leader in an open-addressing table whose slots hold the
//      position of one occurrence (keys are compared by reading the corpus there) and, in the same 8 bytes, a counter; a
//      window remembers its leader's slot for step 3;
//   2. the LC best leaders under the order (count falling, tokens rising) are found by a most-significant-digit-first
//      radix select over the distinct leaders (one histogram pass per 12 bits of the composite key; the block that comes
//      last picks the digit), then written into the frozen table's entries and hashed into its index;
//   3. follower counts: windows whose leader was selected insert-or-increment the whole window in a second table; a distinct
//      window takes its ordinal among its leader's when it is created, every leader takes a range of the group array, and
//      position and count of the distinct windows go there, grouped by leader;
//   4. a warp per leader (a block for those with more than 32 distinct windows) picks the FC best of its group under
//      (count falling, follower tokens rising): a threshold by bisection on the count, then on the tokens of the windows that
//      tie with it where those are many, and ranks what is left.
// What bounds it is random access to the two hash tables (8 bytes a slot, 2 to 4 slots a window) and the counting of frequent
// keys; a block gathers its counts of repeated slots in shared memory, so that a key that makes up a tenth of the corpus costs
// an atomic per block and not one per occurrence.  4 M tokens, LL = 2, LC = 65,536, FC = 8: 3.1 ms with a scan of the whole group per
// distinct window (1.57 ms of it), 37 launches and a one-block scan, 0.75 ms with this form; 8 M tokens, LL = 1, FC = 128: 26.9 and 2.8 ms.
// Which occurrence represents a key, and which entry id a leader gets, depends on timing; the table's content (and
// cb_frozen_dump's output) does not.
#include <algorithm>

#include "cb_common.cuh"

namespace {

constexpr uint32_t kEmpty = 0xFFFFFFFFu;
constexpr unsigned long long kEmptySlot = 0x00000000FFFFFFFFull;   // low word: position, high word: count
constexpr int kMaxWords = 1 + CB_MAX_LL;      // composite selection key: count (complemented), then the leader's tokens
constexpr int kDigitBits = 12, kBins = 1 << kDigitBits;
constexpr uint32_t kMidGroup = 1024;          // distinct windows of one leader up to which a block of 128 threads does the selection
constexpr int kCand = 512;                    // candidates ranked against one another (at least FC)
static_assert(kCand >= 2 * CB_MAX_FC, "the FC best and as many ties fit");

struct BuildState {                           // head of the scratch buffer
    uint32_t status;
    uint32_t n_uniq;                          // distinct leaders
    uint32_t n_sel;                           // entry ids handed out
    uint32_t n_mid, n_big;                    // leaders with groups of more than 32, of more than kMidGroup windows
    uint32_t n_ties;                          // leaders whose count is exactly that of the LC-th best
    uint32_t count_known;                     // word 0 of the prefix is resolved
    uint32_t k_rem;                           // radix select: rank still to be resolved inside the current prefix
    uint32_t cursor;                          // next free place of the group array
    uint32_t arrived;                         // blocks of the running histogram pass that are done
    uint32_t max_token;                       // largest token of a leader
    uint32_t prefix[kMaxWords];               // composite key of the LC-th best leader, resolved digit by digit
    uint32_t hist[kBins];
};

struct BuildView {
    BuildState* st;
    unsigned long long* h1; int32_t* h1_eid;                      // [S] leaders: position and count; entry id or -1
    unsigned long long* h2; uint32_t* h2_ord;                     // [S] windows of selected leaders; ordinal in the leader's group
    uint32_t* lslot;                                              // [M] leader slot of every window (kEmpty: left out)
    uint2* group;                                                 // [S] distinct windows grouped by leader: position, count
    uint32_t* uniq; uint32_t* ties;                               // [M] slots of the distinct leaders, of those that tie with the LC-th best
                                                                  // (both share group's memory: dead before that is filled)
    uint32_t* grp_n; uint32_t* grp_off; uint32_t* listed;         // [LC] group size, start; leaders with middling groups from the front, large from the back
    uint32_t S;                                                   // slots of each hash table (a power of two)
    const int32_t* corpus;
    uint32_t M;
    int LL, FL, LC, FC;
};

__device__ __forceinline__ uint64_t hash_tokens(const int32_t* p, int n) {
    uint64_t h = 0x9E3779B97F4A7C15ull ^ (uint64_t)n;
    for (int j = 0; j < n; ++j) { h = (h ^ (uint32_t)p[j]) * 0xFF51AFD7ED558CCDull; h ^= h >> 32; }
    h ^= h >> 33; h *= 0xC4CEB9FE1A85EC53ull; h ^= h >> 33;
    return h;
}
__device__ __forceinline__ bool same_tokens(const int32_t* a, const int32_t* b, int n) {
    for (int j = 0; j < n; ++j) if (a[j] != b[j]) return false;
    return true;
}
// Finds or creates the slot of the n-token key at corpus position i.  Returns the slot, or kEmpty when every slot was
// visited (cannot happen at the load factor the tables are sized for; reported as CB_ERR_PROBE_LIMIT).  A slot's position never
// changes once it is set, so an ordinary load will do; one that still shows an empty slot is put right by the compare-and-swap.
__device__ __forceinline__ uint32_t find_or_claim(unsigned long long* slots, uint32_t S, const int32_t* corpus, uint32_t i, int n, bool* created) {
    uint32_t s = (uint32_t)(hash_tokens(corpus + i, n) >> 20) & (S - 1);
    *created = false;
    for (uint32_t p = 0; p < S; ++p) {
        uint32_t pos = *reinterpret_cast<const uint32_t*>(&slots[s]);
        if (pos == kEmpty) {
            const unsigned long long was = atomicCAS(&slots[s], kEmptySlot, (1ull << 32) | i);   // the creator counts itself
            if (was == kEmptySlot) { *created = true; return s; }
            pos = (uint32_t)was;
        }
        if (same_tokens(corpus + pos, corpus + i, n)) return s;
        s = (s + 1) & (S - 1);
    }
    return kEmpty;
}
__device__ __forceinline__ uint32_t* count_of(unsigned long long* slots, uint32_t s) { return reinterpret_cast<uint32_t*>(&slots[s]) + 1; }

// A block's counts of the slots it meets first in each of 512 places; other slots are counted in memory right away.
struct CountCache {
    uint32_t key[512], cnt[512];
    __device__ __forceinline__ void clear() {
        for (int i = threadIdx.x; i < 512; i += blockDim.x) { key[i] = kEmpty; cnt[i] = 0u; }
        __syncthreads();
    }
    __device__ __forceinline__ void add(unsigned long long* slots, uint32_t s) {
        const uint32_t at = (s * 0x9E3779B1u) >> 23;
        uint32_t k = key[at];
        if (k == kEmpty) {
            k = atomicCAS(&key[at], kEmpty, s);
            if (k == kEmpty) k = s;
        }
        if (k == s) atomicAdd(&cnt[at], 1u);
        else atomicAdd(count_of(slots, s), 1u);
    }
    __device__ __forceinline__ void flush(unsigned long long* slots) {
        __syncthreads();
        for (int i = threadIdx.x; i < 512; i += blockDim.x)
            if (key[i] != kEmpty && cnt[i]) atomicAdd(count_of(slots, key[i]), cnt[i]);
    }
};

// Items that threads of a block append to a list in memory: gathered in shared memory, so that the list's counter takes an atomic
// per thousand or so (one address takes one atomic in about 2 ns: an atomic per warp was 260 of 310 us of the leader count).
struct Appender {
    static constexpr uint32_t kCap = 1536;
    uint32_t item[kCap], n, at;
    __device__ __forceinline__ void clear() { if (threadIdx.x == 0) n = 0u; __syncthreads(); }
    // all threads of the block together
    __device__ __forceinline__ void add(bool has, uint32_t x, uint32_t* list, uint32_t* counter) {
        const uint32_t m = __ballot_sync(CB_FULL, has), lane = threadIdx.x & 31;
        uint32_t k = 0;
        if (m && lane == 0) k = atomicAdd(&n, (uint32_t)__popc(m));
        k = __shfl_sync(CB_FULL, k, 0) + __popc(m & ((1u << lane) - 1u));
        if (has) item[k] = x;
        // The block decides as one: every warp reads the count before it arrives at the barrier (the last to add sees all of it), and
        // nobody adds again before all have.  Read after a barrier, the count could already hold the next call's additions.
        if (__syncthreads_or(n > kCap - 256u)) flush(list, counter);
    }
    __device__ __forceinline__ void flush(uint32_t* list, uint32_t* counter) {
        __syncthreads();
        if (threadIdx.x == 0) at = n ? atomicAdd(counter, n) : 0u;
        __syncthreads();
        for (uint32_t i = threadIdx.x; i < n; i += blockDim.x) list[at + i] = item[i];
        __syncthreads();
        if (threadIdx.x == 0) n = 0u;
        __syncthreads();
    }
};

__global__ void fb_init_kernel(BuildView v, CbTables t) {
    const size_t g = (size_t)blockIdx.x * blockDim.x + threadIdx.x, stride = (size_t)gridDim.x * blockDim.x;
    ulonglong2* a = reinterpret_cast<ulonglong2*>(v.h1);
    ulonglong2* b = reinterpret_cast<ulonglong2*>(v.h2);
    for (size_t i = g; i < v.S / 2; i += stride) { a[i] = make_ulonglong2(kEmptySlot, kEmptySlot); b[i] = make_ulonglong2(kEmptySlot, kEmptySlot); }
    for (size_t i = g; i < (size_t)v.LC; i += stride) { v.grp_n[i] = 0u; t.lstamp[i] = 0u; }
    for (size_t i = g; i < t.nslots; i += stride) t.index[i] = CB_IDX_EMPTY;
    for (size_t i = g; i < (size_t)v.LC * t.E; i += stride) t.entries[i] = 0u;
    for (size_t i = g; i < sizeof(BuildState) / 4; i += stride) reinterpret_cast<uint32_t*>(v.st)[i] = 0u;
    if (g < 4) t.hdr[g] = 0u;
}

// 1. leader counts
__global__ void __launch_bounds__(256) fb_count_leaders_kernel(BuildView v) {
    __shared__ CountCache cache;
    __shared__ Appender made;
    cache.clear();
    made.clear();
    const size_t stride = (size_t)gridDim.x * blockDim.x;
    uint32_t mx = 0;
    for (size_t i0 = (size_t)blockIdx.x * blockDim.x; i0 < v.M; i0 += stride) {
        const size_t i = i0 + threadIdx.x;
        uint32_t s = kEmpty;
        bool created = false;
        if (i < v.M) {
            bool neg = false;
            for (int j = 0; j < v.LL + v.FL; ++j) neg |= v.corpus[i + j] < 0;
            if (neg) {
                atomicCAS(&v.st->status, 0u, (uint32_t)CB_ERR_INVALID_ARG);
            } else {
                for (int j = 0; j < v.LL; ++j) mx = max(mx, (uint32_t)v.corpus[i + j]);
                s = find_or_claim(v.h1, v.S, v.corpus, (uint32_t)i, v.LL, &created);
                if (s == kEmpty) atomicCAS(&v.st->status, 0u, (uint32_t)CB_ERR_PROBE_LIMIT);
                else if (!created) cache.add(v.h1, s);
            }
            v.lslot[i] = s;
        }
        made.add(created, s, v.uniq, &v.st->n_uniq);
    }
    made.flush(v.uniq, &v.st->n_uniq);
    mx = __reduce_max_sync(CB_FULL, mx);
    if ((threadIdx.x & 31) == 0) atomicMax(&v.st->max_token, mx);
    cache.flush(v.h1);
}

// Word w of a leader's composite key: the count so that more comes first (counts are at most M < 2^cbits), then its tokens.
__device__ __forceinline__ uint32_t sel_word(const BuildView& v, unsigned long long slot, int w, uint32_t cmask) {
    return w == 0 ? cmask - (uint32_t)(slot >> 32) : (uint32_t)v.corpus[(uint32_t)slot + (w - 1)];
}

// The last block of a histogram pass picks the bin in which the k-th smallest key lies and clears the histogram.  Every thread of
// the block gets the bin; *rest is the rank inside it.
__device__ __forceinline__ uint32_t pick_bin(const BuildView& v, uint32_t k, uint32_t* s_part, uint32_t* s_pick, uint32_t* rest) {
    constexpr int PER = kBins / 256;
    uint32_t c[PER], sum = 0;
#pragma unroll
    for (int j = 0; j < PER; ++j) { c[j] = __ldcg(&v.st->hist[threadIdx.x * PER + j]); sum += c[j]; v.st->hist[threadIdx.x * PER + j] = 0u; }
    s_part[threadIdx.x] = sum;
    __syncthreads();
    for (int o = 1; o < 256; o <<= 1) {
        const uint32_t add = (int)threadIdx.x >= o ? s_part[threadIdx.x - o] : 0u;
        __syncthreads();
        s_part[threadIdx.x] += add;
        __syncthreads();
    }
    uint32_t cum = s_part[threadIdx.x] - sum;
    if (cum < k && k <= cum + sum) {
#pragma unroll
        for (int j = 0; j < PER; ++j) {
            if (cum < k && k <= cum + c[j]) { s_pick[0] = (uint32_t)(threadIdx.x * PER + j); s_pick[1] = k - cum; }
            cum += c[j];
        }
    }
    __syncthreads();
    *rest = s_pick[1];
    return s_pick[0];
}
// All threads of a block: true in the block that comes last to this point of a launch.
__device__ __forceinline__ bool last_block(const BuildView& v, uint32_t* s_last) {
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) {
        *s_last = atomicAdd(&v.st->arrived, 1u) == gridDim.x - 1u ? 1u : 0u;
        if (*s_last) v.st->arrived = 0u;
    }
    __syncthreads();
    __threadfence();
    return *s_last != 0u;
}
// one shared atomic per warp and bin (most counts are 1); kEmpty: none
__device__ __forceinline__ void add_bin(uint32_t* sh, uint32_t bin) {
    const uint32_t peers = __match_any_sync(CB_FULL, bin);
    if (bin != kEmpty && (int)(threadIdx.x & 31) == __ffs(peers) - 1) atomicAdd(&sh[bin], (uint32_t)__popc(peers));
}

// 2a. The count of the LC-th best leader, one pass where it is below 4,095: a bin per count, the last one for all above.
__global__ void __launch_bounds__(256) fb_select_count_kernel(BuildView v, uint32_t cmask) {
    __shared__ uint32_t sh[kBins];
    __shared__ uint32_t s_last, s_part[256], s_pick[2];
    const uint32_t n = v.st->n_uniq;
    if (n <= (uint32_t)v.LC) return;          // all of them are taken
    for (int i = threadIdx.x; i < kBins; i += 256) sh[i] = 0u;
    __syncthreads();
    for (size_t i0 = (size_t)blockIdx.x * 256; i0 < n; i0 += (size_t)gridDim.x * 256) {
        const size_t i = i0 + threadIdx.x;
        add_bin(sh, i < n ? kBins - 1 - min((uint32_t)(v.h1[v.uniq[i]] >> 32), (uint32_t)(kBins - 1)) : kEmpty);
    }
    __syncthreads();
    for (int i = threadIdx.x; i < kBins; i += 256)
        if (sh[i]) atomicAdd(&v.st->hist[i], sh[i]);
    if (!last_block(v, &s_last)) return;
    uint32_t rest;
    const uint32_t bin = pick_bin(v, (uint32_t)v.LC, s_part, s_pick, &rest);
    if (threadIdx.x == 0) {
        v.st->k_rem = bin > 0u ? rest : (uint32_t)v.LC;
        v.st->count_known = bin > 0u ? 1u : 0u;
        v.st->prefix[0] = bin > 0u ? cmask - (kBins - 1 - bin) : 0u;
    }
}

// 2b. Histogram of the digit at `shift` of word `w` over the leaders that match the prefix resolved so far; the last
// block to finish picks the digit in which the k-th smallest composite key lies.  Word 0 goes over all leaders and only where
// the pass above did not settle it, the tokens over the leaders that tie with its count; leading digits that are zero in
// every token are passed over.
__global__ void __launch_bounds__(256) fb_select_kernel(BuildView v, int w, int shift, uint32_t cmask) {
    __shared__ uint32_t sh[kBins];
    __shared__ uint32_t s_last, s_part[256], s_pick[2];
    if (v.st->n_uniq <= (uint32_t)v.LC) return;
    if (w == 0 && v.st->count_known) return;
    if (w > 0 && shift > 0 && (v.st->max_token >> shift) == 0u) return;
    const uint32_t n = w == 0 ? v.st->n_uniq : v.st->n_ties;
    const uint32_t* const list = w == 0 ? v.uniq : v.ties;
    for (int i = threadIdx.x; i < kBins; i += 256) sh[i] = 0u;
    __syncthreads();
    const uint32_t hi_mask = shift + kDigitBits >= 32 ? 0u : (0xFFFFFFFFu << (shift + kDigitBits));
    uint32_t prefix[kMaxWords];
#pragma unroll
    for (int k = 0; k < kMaxWords; ++k) prefix[k] = v.st->prefix[k];
    for (size_t i0 = (size_t)blockIdx.x * 256; i0 < n; i0 += (size_t)gridDim.x * 256) {
        const size_t i = i0 + threadIdx.x;
        uint32_t bin = kEmpty;
        if (i < n) {
            const unsigned long long slot = v.h1[list[i]];
            bool ok = true;
            for (int k = 1; k < w && ok; ++k) ok = sel_word(v, slot, k, cmask) == prefix[k];
            if (ok) {
                const uint32_t x = sel_word(v, slot, w, cmask);
                if ((x & hi_mask) == (prefix[w] & hi_mask)) bin = (x >> shift) & (kBins - 1);
            }
        }
        add_bin(sh, bin);
    }
    __syncthreads();
    for (int i = threadIdx.x; i < kBins; i += 256)
        if (sh[i]) atomicAdd(&v.st->hist[i], sh[i]);
    if (!last_block(v, &s_last)) return;
    uint32_t rest;
    const uint32_t bin = pick_bin(v, v.st->k_rem, s_part, s_pick, &rest);
    if (threadIdx.x == 0) { v.st->k_rem = rest; v.st->prefix[w] |= bin << shift; }
}

// The leader in slot `at` of the first table gets the next entry (take; all threads of a block together, one atomic for all of
// them); its key goes into the frozen table's index.
__device__ __forceinline__ void place_leader(const BuildView& v, const CbTables& t, bool take, uint32_t at, unsigned long long slot, uint32_t* s_cnt /* [9] */) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t m = __ballot_sync(CB_FULL, take);
    __syncthreads();
    if (lane == 0) s_cnt[warp] = (uint32_t)__popc(m);
    __syncthreads();
    if (threadIdx.x == 0) {
        uint32_t total = 0;
        for (int k = 0; k < 8; ++k) { const uint32_t c = s_cnt[k]; s_cnt[k] = total; total += c; }
        s_cnt[8] = total ? atomicAdd(&v.st->n_sel, total) : 0u;
    }
    __syncthreads();
    if (!take) return;
    const uint32_t eid = s_cnt[8] + s_cnt[warp] + __popc(m & ((1u << lane) - 1u));
    if (eid >= (uint32_t)v.LC) { atomicCAS(&v.st->status, 0u, (uint32_t)CB_ERR_PROBE_LIMIT); v.h1_eid[at] = -1; return; }
    v.h1_eid[at] = (int32_t)eid;
    const int32_t* key = v.corpus + (uint32_t)slot;
    uint32_t* e = t.entries + (size_t)eid * t.E;
    int32_t k4[4] = {0, 0, 0, 0};
    for (int j = 0; j < v.LL; ++j) { k4[j] = key[j]; e[j] = (uint32_t)key[j]; }
    t.lstamp[eid] = (uint32_t)(slot >> 32);
    const uint64_t h = cb_hash4(k4[0], k4[1], k4[2], k4[3], v.LL);
    const uint32_t nb = t.nslots >> 5, word = (cb_hash_tag(h) << CB_EID_BITS) | eid;
    uint32_t bucket = cb_hash_bucket(h, t.nslots);
    for (uint32_t p = 0; p < nb; ++p) {
        // the bucket's 32 words at once; only those seen empty are tried
        const uint4* bp = reinterpret_cast<const uint4*>(t.index + (size_t)bucket * 32);
        uint32_t empty = 0u;
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            const uint4 x = __ldcg(bp + q);
            empty |= ((x.x == CB_IDX_EMPTY ? 1u : 0u) | (x.y == CB_IDX_EMPTY ? 2u : 0u) | (x.z == CB_IDX_EMPTY ? 4u : 0u) | (x.w == CB_IDX_EMPTY ? 8u : 0u)) << (4 * q);
        }
        for (; empty; empty &= empty - 1u)
            if (atomicCAS(&t.index[bucket * 32 + __ffs(empty) - 1], CB_IDX_EMPTY, word) == CB_IDX_EMPTY) return;
        bucket = (bucket + 1) & (nb - 1);
    }
    atomicCAS(&v.st->status, 0u, (uint32_t)CB_ERR_PROBE_LIMIT);
}

// 2c. the leaders with a larger count than the LC-th best are placed, those with the same count listed
__global__ void __launch_bounds__(256) fb_place_leaders_kernel(BuildView v, CbTables t, uint32_t cmask) {
    const uint32_t n = v.st->n_uniq;
    const bool all = n <= (uint32_t)v.LC;
    const uint32_t cut = cmask - v.st->prefix[0];
    __shared__ uint32_t s_cnt[9];
    __shared__ Appender tied;
    tied.clear();
    for (size_t i0 = (size_t)blockIdx.x * 256; i0 < n; i0 += (size_t)gridDim.x * 256) {
        const size_t i = i0 + threadIdx.x;
        bool take = false, tie = false;
        uint32_t at = 0;
        unsigned long long slot = 0;
        if (i < n) {
            at = v.uniq[i];
            slot = v.h1[at];
            take = all || (uint32_t)(slot >> 32) > cut;
            tie = !take && (uint32_t)(slot >> 32) == cut;
            if (!take) v.h1_eid[at] = -1;
        }
        tied.add(tie, at, v.ties, &v.st->n_ties);
        place_leader(v, t, take, at, slot, s_cnt);
    }
    tied.flush(v.ties, &v.st->n_ties);
    if (blockIdx.x == 0 && threadIdx.x == 0) t.hdr[1] = min(n, (uint32_t)v.LC);
}
// 2d. of the tied leaders those whose tokens come no later than the LC-th best's
__global__ void __launch_bounds__(256) fb_place_ties_kernel(BuildView v, CbTables t, uint32_t cmask) {
    const uint32_t n = v.st->n_ties;
    __shared__ uint32_t s_cnt[9];
    for (size_t i0 = (size_t)blockIdx.x * 256; i0 < n; i0 += (size_t)gridDim.x * 256) {
        const size_t i = i0 + threadIdx.x;
        bool take = i < n;
        uint32_t at = 0;
        unsigned long long slot = 0;
        if (take) {
            at = v.ties[i];
            slot = v.h1[at];
            for (int k = 1; k <= v.LL; ++k) {
                const uint32_t x = sel_word(v, slot, k, cmask), y = v.st->prefix[k];
                if (x != y) { take = x < y; break; }
            }
        }
        place_leader(v, t, take, at, slot, s_cnt);
    }
}

// 3a. follower counts of the selected leaders; a new window takes its ordinal in its leader's group
__global__ void __launch_bounds__(256) fb_count_followers_kernel(BuildView v) {
    __shared__ CountCache cache;
    cache.clear();
    const int lane = threadIdx.x & 31;
    const size_t stride = (size_t)gridDim.x * blockDim.x;
    for (size_t i0 = (size_t)blockIdx.x * blockDim.x; i0 < v.M; i0 += stride) {
        const size_t i = i0 + threadIdx.x;
        bool created = false;
        uint32_t s = kEmpty;
        int32_t eid = -1;
        if (i < v.M) {
            const uint32_t ls = v.lslot[i];
            if (ls != kEmpty) eid = v.h1_eid[ls];
            if (eid >= 0) {
                s = find_or_claim(v.h2, v.S, v.corpus, (uint32_t)i, v.LL + v.FL, &created);
                if (s == kEmpty) atomicCAS(&v.st->status, 0u, (uint32_t)CB_ERR_PROBE_LIMIT);
                else if (!created) cache.add(v.h2, s);
            }
        }
        // the new windows of one leader in a warp take their ordinals with one atomic
        if (__any_sync(CB_FULL, created)) {
            const uint32_t peers = __match_any_sync(CB_FULL, created ? eid : -1 - lane);
            const int head = __ffs(peers) - 1;
            uint32_t at = 0;
            if (created && lane == head) at = atomicAdd(&v.grp_n[eid], (uint32_t)__popc(peers));
            at = __shfl_sync(CB_FULL, at, head) + __popc(peers & ((1u << lane) - 1u));
            if (created) v.h2_ord[s] = at;
        }
    }
    cache.flush(v.h2);
}
// 3b. every leader takes a range of the group array (an atomic per block of 256: their ranges lie side by side); the leaders with
// more than 32 distinct windows are listed
__global__ void __launch_bounds__(256) fb_group_ranges_kernel(BuildView v) {
    const uint32_t n = min(v.st->n_sel, (uint32_t)v.LC);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    __shared__ uint32_t s_tot[8], s_start;
    for (uint32_t e0 = blockIdx.x * 256u; e0 < n; e0 += gridDim.x * 256u) {
        const uint32_t e = e0 + threadIdx.x, c = e < n ? v.grp_n[e] : 0u;
        uint32_t incl = c;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t up = __shfl_up_sync(CB_FULL, incl, o);
            if (lane >= o) incl += up;
        }
        if (lane == 31) s_tot[warp] = incl;
        __syncthreads();
        if (threadIdx.x == 0) {
            uint32_t total = 0;
            for (int k = 0; k < 8; ++k) { const uint32_t x = s_tot[k]; s_tot[k] = total; total += x; }
            s_start = total ? atomicAdd(&v.st->cursor, total) : 0u;
        }
        __syncthreads();
        if (e < n) {
            v.grp_off[e] = s_start + s_tot[warp] + incl - c;
            if (c > kMidGroup) v.listed[v.LC - 1 - atomicAdd(&v.st->n_big, 1u)] = e;
            else if (c > 32) v.listed[atomicAdd(&v.st->n_mid, 1u)] = e;
        }
        __syncthreads();                                         // the shared words are rewritten by the next round
    }
}
// 3c. the distinct windows, grouped by leader: position and count
__global__ void __launch_bounds__(256) fb_group_scatter_kernel(BuildView v) {
    const size_t stride = (size_t)gridDim.x * blockDim.x;
    for (size_t s = (size_t)blockIdx.x * blockDim.x + threadIdx.x; s < v.S; s += stride) {
        const unsigned long long x = v.h2[s];
        if ((uint32_t)x == kEmpty) continue;
        const int32_t eid = v.h1_eid[v.lslot[(uint32_t)x]];
        v.group[v.grp_off[eid] + v.h2_ord[s]] = make_uint2((uint32_t)x, (uint32_t)(x >> 32));
    }
}

// 4. The FC best of a leader's group.  A block of NT threads works on one leader.
template <int NT>
struct Crew {
    uint32_t* red;            // [NT / 32] shared words
    __device__ __forceinline__ uint32_t gather(uint32_t x) const {   // the warps' values, one per lane
        __syncthreads();
        if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = x;
        __syncthreads();
        return (threadIdx.x & 31) < NT / 32 ? red[threadIdx.x & 31] : 0u;
    }
    __device__ __forceinline__ uint32_t sum(uint32_t x) const { return __reduce_add_sync(CB_FULL, gather(__reduce_add_sync(CB_FULL, x))); }
    __device__ __forceinline__ uint32_t max(uint32_t x) const { return __reduce_max_sync(CB_FULL, gather(__reduce_max_sync(CB_FULL, x))); }
};

// The windows that may be among the FC best, with their followers, in shared memory.
struct Candidates {
    uint32_t n, cnt[kCand];
    int32_t tok[kCand * CB_MAX_FL];           // [kCand][FL]
    // true if candidate a comes before candidate b
    __device__ __forceinline__ bool before(uint32_t a, uint32_t b, int FL) const {
        if (cnt[a] != cnt[b]) return cnt[a] > cnt[b];
        for (int j = 0; j < FL; ++j)
            if (tok[a * FL + j] != tok[b * FL + j]) return tok[a * FL + j] < tok[b * FL + j];
        return false;
    }
};

template <int NT>
__device__ void pick_followers(const BuildView& v, const CbTables& t, uint32_t eid, Candidates& cand, const Crew<NT>& crew) {
    const uint32_t n = v.grp_n[eid];
    const uint2* g = v.group + v.grp_off[eid];
    const int me = (int)threadIdx.x;
    uint32_t cmin = 1;                        // candidates have at least this count
    uint32_t ties = 0;                        // resolved tokens: candidates with exactly cmin come no later than lim[0 .. ties)
    uint32_t lim[CB_MAX_FL];
    uint32_t have = n;
    if (n > (uint32_t)v.FC) {
        // the largest count that FC windows reach
        uint32_t top = 0;
        for (uint32_t k = me; k < n; k += NT) top = ::max(top, g[k].y);
        uint32_t lo = 1, hi = crew.max(top);
        have = n;
        while (lo < hi) {
            const uint32_t mid = lo + (hi - lo + 1u) / 2u;
            uint32_t c = 0;
            for (uint32_t k = me; k < n; k += NT) c += g[k].y >= mid ? 1u : 0u;
            c = crew.sum(c);
            if (c >= (uint32_t)v.FC) { lo = mid; have = c; } else hi = mid - 1u;
        }
        cmin = lo;
    }
    if (have > (uint32_t)kCand) {
        // too many windows tie at that count: of those only the first by tokens, token by token, until the rest fits
        uint32_t above = 0;
        for (uint32_t k = me; k < n; k += NT) above += g[k].y > cmin ? 1u : 0u;
        uint32_t need = (uint32_t)v.FC - crew.sum(above);       // ties to be taken, at least one
        for (int lev = 0; lev < v.FL && have > (uint32_t)kCand; ++lev) {
            auto token = [&](const uint2& x, uint32_t* tok) {    // this level's token of a tie that matches the limits so far
                if (x.y != cmin) return false;
                const int32_t* f = v.corpus + x.x + v.LL;
                for (int j = 0; j < lev; ++j) if ((uint32_t)f[j] != lim[j]) return false;
                *tok = (uint32_t)f[lev];
                return true;
            };
            uint32_t top = 0, tok = 0;
            for (uint32_t k = me; k < n; k += NT) if (token(g[k], &tok)) top = ::max(top, tok);
            uint32_t lo = 0, hi = crew.max(top);                // the smallest token that `need` of them do not exceed
            while (lo < hi) {
                const uint32_t mid = lo + (hi - lo) / 2u;
                uint32_t c = 0;
                for (uint32_t k = me; k < n; k += NT) c += token(g[k], &tok) && tok <= mid ? 1u : 0u;
                if (crew.sum(c) >= need) hi = mid; else lo = mid + 1u;
            }
            uint32_t below = 0, equal = 0;
            for (uint32_t k = me; k < n; k += NT)
                if (token(g[k], &tok)) { below += tok < lo ? 1u : 0u; equal += tok == lo ? 1u : 0u; }
            lim[lev] = lo;
            ties = lev + 1;
            need -= crew.sum(below);
            have = (uint32_t)v.FC - need + crew.sum(equal);
        }
    }
    // the candidates, then each one's rank among them
    if (me == 0) cand.n = 0u;
    __syncthreads();
    for (uint32_t k = me; k < n; k += NT) {
        const uint2 x = g[k];
        bool in = x.y > cmin;
        if (x.y == cmin) {
            in = true;
            const int32_t* f = v.corpus + x.x + v.LL;
            for (uint32_t j = 0; j < ties; ++j)
                if ((uint32_t)f[j] != lim[j]) { in = (uint32_t)f[j] < lim[j]; break; }
        }
        if (in) {
            const uint32_t at = atomicAdd(&cand.n, 1u);
            if (at < (uint32_t)kCand) {
                cand.cnt[at] = x.y;
                for (int j = 0; j < v.FL; ++j) cand.tok[at * v.FL + j] = v.corpus[x.x + v.LL + j];
            }
        }
    }
    __syncthreads();
    const uint32_t nc = min(cand.n, (uint32_t)kCand);
    uint32_t* e = t.entries + (size_t)eid * t.E;
    for (uint32_t i = me; i < nc; i += NT) {
        int rank = 0;
        for (uint32_t k = 0; k < nc && rank < v.FC; ++k) rank += cand.before(k, i, v.FL) ? 1 : 0;
        if (rank >= v.FC) continue;
        for (int j = 0; j < v.FL; ++j) e[v.LL + v.FC + rank * v.FL + j] = (uint32_t)cand.tok[i * v.FL + j];
        e[v.LL + rank] = (uint32_t)(v.FC - rank);
    }
    __syncthreads();                                             // the candidates are overwritten by the next leader
}

// the common case, up to 32 distinct windows: a warp per leader; the next leader's group is looked up while this one is ranked
__global__ void __launch_bounds__(256) fb_rank_kernel(BuildView v, CbTables t) {
    const int lane = threadIdx.x & 31;
    const uint32_t n = min(v.st->n_sel, (uint32_t)v.LC), nw = gridDim.x * 8;
    uint32_t eid = blockIdx.x * 8 + (threadIdx.x >> 5);
    uint32_t ng_next = eid < n ? v.grp_n[eid] : 0u, off_next = eid < n ? v.grp_off[eid] : 0u;
    for (; eid < n; eid += nw) {
        const uint32_t ng = ng_next, off = off_next;
        if (eid + nw < n) { ng_next = v.grp_n[eid + nw]; off_next = v.grp_off[eid + nw]; }
        if (ng > 32) continue;
        // a lane per window, ranked against one another by shuffles
        uint2 x = make_uint2(0u, 0u);
        int32_t f[CB_MAX_FL];
#pragma unroll
        for (int j = 0; j < CB_MAX_FL; ++j) f[j] = 0;
        if ((uint32_t)lane < ng) {
            x = v.group[off + lane];
#pragma unroll
            for (int j = 0; j < CB_MAX_FL; ++j) if (j < v.FL) f[j] = v.corpus[x.x + v.LL + j];
        }
        int rank = 0;
        for (uint32_t k = 0; k < ng; ++k) {
            const uint32_t oc = __shfl_sync(CB_FULL, x.y, k);
            int cmp = oc > x.y ? -1 : (oc < x.y ? 1 : 0);        // -1: the other one comes before
#pragma unroll
            for (int j = 0; j < CB_MAX_FL; ++j) {
                if (j >= v.FL) break;
                const int32_t o = __shfl_sync(CB_FULL, f[j], k);
                if (cmp == 0 && o != f[j]) cmp = o < f[j] ? -1 : 1;
            }
            rank += cmp < 0 ? 1 : 0;
        }
        if ((uint32_t)lane < ng && rank < v.FC) {
            uint32_t* e = t.entries + (size_t)eid * t.E;
#pragma unroll
            for (int j = 0; j < CB_MAX_FL; ++j) if (j < v.FL) e[v.LL + v.FC + rank * v.FL + j] = (uint32_t)f[j];
            e[v.LL + rank] = (uint32_t)(v.FC - rank);
        }
    }
}
// the others, a block per leader: NT = 128 up to kMidGroup distinct windows, 1,024 above
template <int NT>
__global__ void __launch_bounds__(NT) fb_rank_listed_kernel(BuildView v, CbTables t) {
    __shared__ Candidates cand;
    __shared__ uint32_t red[NT / 32];
    const Crew<NT> crew = {red};
    const uint32_t n = NT == 1024 ? v.st->n_big : v.st->n_mid;
    for (uint32_t k = blockIdx.x; k < n; k += gridDim.x) pick_followers<NT>(v, t, v.listed[NT == 1024 ? (uint32_t)v.LC - 1 - k : k], cand, crew);
}

size_t fb_align(size_t x) { return (x + 255) / 256 * 256; }

struct BuildLayout {
    uint32_t S;
    size_t off_h1, off_h1_eid, off_h2, off_h2_ord, off_lslot, off_group, off_grp, total;
};

cb_status fb_layout(const cb_frozen_config* c, int64_t n_tokens, BuildLayout* B) {
    if (n_tokens < 0 || n_tokens > (int64_t)1 << 30) return CB_ERR_INVALID_ARG;
    const int64_t M = n_tokens - c->LL - c->FL + 1 > 0 ? n_tokens - c->LL - c->FL + 1 : 0;
    uint64_t S = 1024;
    while (S < 2ull * (uint64_t)M) S <<= 1;
    B->S = (uint32_t)S;
    size_t o = fb_align(sizeof(BuildState));
    B->off_h1 = o;      o = fb_align(o + S * 8);
    B->off_h1_eid = o;  o = fb_align(o + S * 4);
    B->off_h2 = o;      o = fb_align(o + S * 8);
    B->off_h2_ord = o;  o = fb_align(o + S * 4);
    B->off_lslot = o;   o = fb_align(o + (size_t)(M > 0 ? M : 1) * 4);
    B->off_group = o;   o = fb_align(o + S * 8);
    B->off_grp = o;     o = fb_align(o + (size_t)c->LC * 4 * 3);
    B->total = o;
    return CB_OK;
}

}  // namespace

extern "C" cb_status cb_frozen_build_bytes(const cb_frozen_config* cfg, int64_t n_tokens, size_t* scratch_bytes) {
    CbFrozenLayout L;
    BuildLayout B;
    if (!scratch_bytes) return CB_ERR_INVALID_ARG;
    cb_status s = cb_frozen_layout(cfg, &L);
    if (s != CB_OK) return s;
    s = fb_layout(cfg, n_tokens, &B);
    if (s != CB_OK) return s;
    *scratch_bytes = B.total;
    return CB_OK;
}

extern "C" cb_status cb_frozen_build(const cb_frozen_config* cfg, const int32_t* dev_corpus, int64_t n_tokens, void* dev_table,
                                     size_t table_bytes, void* dev_scratch, size_t scratch_bytes, void* stream) {
    CbFrozenLayout L;
    BuildLayout B;
    cb_status s = cb_frozen_layout(cfg, &L);
    if (s != CB_OK) return s;
    s = fb_layout(cfg, n_tokens, &B);
    if (s != CB_OK) return s;
    CB_CHECK_ARG(dev_table && ((uintptr_t)dev_table & 255) == 0 && dev_scratch && ((uintptr_t)dev_scratch & 255) == 0);
    CB_CHECK_ARG(dev_corpus || n_tokens == 0);
    if (table_bytes < L.total || scratch_bytes < B.total) return CB_ERR_WORKSPACE_TOO_SMALL;
    cudaStream_t st = (cudaStream_t)stream;
    CbTables t = cb_frozen_view(cfg, L, dev_table);
    char* base = (char*)dev_scratch;
    BuildView v;
    v.st = (BuildState*)base;
    v.h1 = (unsigned long long*)(base + B.off_h1); v.h1_eid = (int32_t*)(base + B.off_h1_eid);
    v.h2 = (unsigned long long*)(base + B.off_h2); v.h2_ord = (uint32_t*)(base + B.off_h2_ord);
    v.lslot = (uint32_t*)(base + B.off_lslot);
    v.group = (uint2*)(base + B.off_group); v.uniq = (uint32_t*)(base + B.off_group); v.ties = v.uniq + B.S / 2;   // M <= S / 2
    v.grp_n = (uint32_t*)(base + B.off_grp); v.grp_off = v.grp_n + cfg->LC; v.listed = v.grp_off + cfg->LC;
    v.S = B.S;
    v.corpus = dev_corpus;
    const int64_t M = n_tokens - cfg->LL - cfg->FL + 1;
    v.M = (uint32_t)(M > 0 ? M : 0);
    v.LL = cfg->LL; v.FL = cfg->FL; v.LC = cfg->LC; v.FC = cfg->FC;
    int dev = 0, sms = 0;
    CB_CUDA(cudaGetDevice(&dev));
    CB_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    const dim3 grid((unsigned)(sms * 8)), block(256);
    fb_init_kernel<<<grid, block, 0, st>>>(v, t);
    if (v.M > 0) {
        int cbits = 1;                                        // counts are at most M
        while (cbits < 31 && (v.M >> cbits) != 0) ++cbits;
        const uint32_t cmask = (1u << cbits) - 1u;
        int passes = 0;
        auto select = [&](int w, int bits) {
            for (int shift = (bits - 1) / kDigitBits * kDigitBits; shift >= 0; shift -= kDigitBits, ++passes)
                fb_select_kernel<<<grid, block, 0, st>>>(v, w, shift, cmask);
        };
        fb_count_leaders_kernel<<<grid, block, 0, st>>>(v);
        fb_select_count_kernel<<<grid, block, 0, st>>>(v, cmask);
        if (cbits > kDigitBits) select(0, cbits);             // counts of 4,095 and more can occur
        fb_place_leaders_kernel<<<grid, block, 0, st>>>(v, t, cmask);
        for (int w = 1; w <= cfg->LL; ++w) select(w, 31);
        fb_place_ties_kernel<<<grid, block, 0, st>>>(v, t, cmask);
        fb_count_followers_kernel<<<grid, block, 0, st>>>(v);
        fb_group_ranges_kernel<<<dim3((unsigned)std::min(4 * sms, (cfg->LC + 255) / 256)), block, 0, st>>>(v);
        fb_group_scatter_kernel<<<grid, block, 0, st>>>(v);
        fb_rank_kernel<<<grid, block, 0, st>>>(v, t);
        fb_rank_listed_kernel<128><<<dim3((unsigned)(sms * 8)), dim3(128), 0, st>>>(v, t);
        fb_rank_listed_kernel<1024><<<dim3((unsigned)sms), dim3(1024), 0, st>>>(v, t);
        cb_count_launch(10 + passes);
    }
    cb_count_launch(1);
    CB_CUDA(cudaGetLastError());
    uint32_t status = 0;
    CB_CUDA(cudaMemcpyAsync(&status, &v.st->status, 4, cudaMemcpyDeviceToHost, st));
    CB_CUDA(cudaStreamSynchronize(st));
    return (cb_status)status;
}

// Offline construction of a frozen table from a token corpus on the GPU (Section 4: the most frequent LC n-grams of
// length LL become the leaders; each keeps the FC most frequent n-grams of length FL that follow it).
//
// A window is LL + FL consecutive tokens; the corpus of N tokens has M = N - LL - FL + 1 of them.  Everything is counting
// and selection on integers, done without sorting:
//   1. leader counts: every window inserts-or-increments its leader in an open-addressing table whose slots hold the leader's tokens as
//      one number (or, where they do not fit 63 bits, the position of one occurrence), with the counters in an array beside it; a
//      window remembers its leader's slot for step 3;
//   2. the LC best leaders under the order (count falling, tokens rising) are found by a most-significant-digit-first
//      radix select over the table (one histogram pass per 12 bits of the composite key; every block picks the digit for
//      itself), then take a range for their windows and are written into the frozen table's entries and hashed into its index;
//   3. the windows of the selected leaders go into the leaders' ranges of one array (a counting sort: the leader counts are known
//      from step 1), all but those of the few leaders with more than kBigGroup windows: these insert-or-increment the whole window in
//      a second hash table, and the distinct ones are grouped by leader afterwards;
//   4. a leader's windows are told apart, counted and the FC best picked under (count falling, follower tokens rising) by a warp
//      (up to 32 windows: the lanes match their tokens against one another) or by a block with a table in shared memory; of a
//      big leader's distinct windows a block picks the FC best from memory.  The pick: a threshold by bisection on the count, then on
//      the tokens of the windows that tie with it where those are many; what is left is ranked.
// What bounds it is random access: to the leader table (four slots for three windows) and to the ranges.  The frequent
// keys' counts and the lists are gathered per block in shared memory, so that a key that makes up a tenth of the corpus costs
// an atomic per block and not one per occurrence.  Counting every selected window in a second hash table took 212 us of a build from 4 M
// tokens (LL = 2, LC = 65,536, FC = 8: 167 MB of tables at random, more than the L2 holds), grouping its slots 49 us, ranking 187 us.
// The whole call with the draft that follows it: 763 us that way, 508 with windows in ranges, 453 with keys in the leader table, read from
// end to end by the selection, and ranges taken as the leaders are placed (a table of positions with a list of its used slots: the same
// call from 302 k tokens 218, so 178; 949 k, LL = 3: 256 and 198).  Of the 453: leader counts 72, windows into ranges 106, selection 60,
// ranking some 150 with its kernels side by side.
// Which occurrence represents a key, and which entry id a leader gets, depends on timing; the table's content (and
// cb_frozen_dump's output) does not.
#include <algorithm>
#include <type_traits>

#include "cb_common.cuh"

namespace {

constexpr uint32_t kEmpty = 0xFFFFFFFFu;
constexpr unsigned long long kNoLeader = ~0ull;                    // first table: a free slot
constexpr unsigned long long kEmptySlot = 0x00000000FFFFFFFFull;   // second table; low word: position, high word: count
constexpr int kMaxWords = 1 + CB_MAX_LL;      // composite selection key: count (complemented), then the leader's tokens
constexpr int kDigitBits = 12, kBins = 1 << kDigitBits;
constexpr int kMaxPasses = 1 + 3 * kMaxWords;  // leader counts below 4,095, then three digits for each word of the key
constexpr uint32_t kWarpGroup = 128;          // windows of one leader that a warp takes (up to 32: a lane each)
constexpr uint32_t kMidGroup = 512;           // windows of one leader that a block of 128 threads takes
constexpr uint32_t kBigGroup = 4096;          // windows of one leader that a block of 512 threads takes; above: the second hash table
constexpr int kCand = 256;                    // candidates ranked against one another (at least FC)
static_assert(kCand >= 2 * CB_MAX_FC, "the FC best and as many ties fit");

struct BuildState {                           // head of the scratch buffer
    uint32_t status;                          // (the state is cleared before the first launch)
    uint32_t n_once;                          // leaders that occur once (counted where that matters)
    uint32_t n_sel;                           // entry ids handed out
    uint32_t n_warp, n_mid, n_large, n_big;   // leaders with more than 32, kWarpGroup, kMidGroup, kBigGroup windows
    uint32_t n_ties;                          // leaders whose count is exactly that of the LC-th best
    uint32_t cursor, big_cursor;              // next free place of the window array, of the group array (the big leaders' windows)
    uint32_t arrived;                         // blocks of the selection that have come to its barriers so far
    uint32_t aborted;                         // a block has given up on such a barrier: what the later kernels read is incomplete
    uint32_t grouped;                         // kGo: step 3 is over and can be read (kGaveUp: it was not done)
    uint32_t max_token;                       // largest token of the corpus
    uint32_t has_neg;                         // some token is negative
    alignas(16) uint32_t hist[kMaxPasses][kBins];   // one histogram per pass of the selection (read 16 bytes at a time)
};

static_assert(offsetof(BuildState, hist) % 16 == 0, "histograms are read 16 bytes at a time");

struct BuildView {
    BuildState* st;
    unsigned long long* h1;                                       // [S1] leaders: the tokens as one number where they fit, else the position of an occurrence
    uint32_t* h1_cnt;                                             // [S1] occurrences but one; of a selected one later kTaken | next free place of its range,
                                                                  // with more than kBigGroup windows kTaken | kBigLeader | entry id
    unsigned long long* h2; uint32_t* h2_ord;                     // [S] windows of big leaders (big_slots in use); ordinal in the leader's group
    uint32_t* lslot;                                              // [M] leader slot of every window (kEmpty: left out)
    uint2* group;                                                 // [M] distinct windows of the big leaders, grouped by leader: position, count
    uint32_t* ties;                                               // [M] slots of the leaders that tie with the LC-th best (in group's memory: dead before that is filled)
    uint32_t* wpos;                                               // [M] windows of the other selected leaders, grouped by leader
    uint32_t* grp_n; uint32_t* grp_off;                           // [LC] windows placed (big: distinct ones); start, kBigFlag: of group, else of wpos
    uint32_t* listed; uint32_t* listed_big;                       // [LC] each: middling leaders from the front, large ones from the back; big ones
                                                                  // from the front, those that a warp takes from the back
    uint32_t S1, S;                                               // slots of the first table (any number), of the second (a power of two)
    const int32_t* corpus;
    uint32_t M, n_tokens;
    uint32_t wait_limit;                                          // looks at the selection's barriers before a block gives up
    int LL, FL, LC, FC;
};

constexpr uint32_t kTaken = 0x80000000u, kBigLeader = 0x40000000u, kBigFlag = 0x80000000u;   // counts, positions and entry ids stay below 2^30

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
// A leader's tokens as one number, the first one highest, so that the numbers' order is that of the tokens: bits each, as many as the
// corpus' largest token has.  0: they do not fit 63 bits (four tokens of 16 bits or more); the table then holds positions.  With
// positions, every look at a slot is followed by one at the corpus (4 M windows, LL = 2: count of the leaders 94 us).
__device__ __forceinline__ int key_bits(const BuildView& v) {
    const int bits = max(32 - __clz((int)v.st->max_token), 1);
    return bits * v.LL <= 63 ? bits : 0;
}
__device__ __forceinline__ uint64_t hash_key(uint64_t k) {
    k *= 0xFF51AFD7ED558CCDull; k ^= k >> 32;
    k *= 0xC4CEB9FE1A85EC53ull; return k ^ (k >> 29);
}
// Token j of the leader in a slot that holds x.
__device__ __forceinline__ int32_t leader_token(const BuildView& v, int bits, uint64_t x, int j) {
    return bits ? (int32_t)((x >> (bits * (v.LL - 1 - j))) & ((1ull << bits) - 1ull)) : v.corpus[(uint32_t)x + j];
}
// The first table keeps keys and counts apart and has four slots for three windows.  Home slots are the hash's share of the table.
__device__ __forceinline__ uint32_t home_leader(uint64_t h, uint32_t S1) { return __umulhi((uint32_t)(h >> 20), S1); }
// Finds or creates the slot of leader `me` (same(x): the one that a slot holds is this), from slot s on, whose word is x; kEmpty when every
// slot was visited.
template <typename Same>
__device__ __forceinline__ uint32_t claim_leader(unsigned long long* slots, uint32_t S1, uint32_t s, unsigned long long x, unsigned long long me, bool* created, Same&& same) {
    *created = false;
    for (uint32_t p = 0; p < S1; ++p) {
        if (x == kNoLeader) {
            x = atomicCAS(&slots[s], kNoLeader, me);
            if (x == kNoLeader) { *created = true; return s; }
        }
        if (same(x)) return s;
        s = s + 1 == S1 ? 0u : s + 1;
        x = slots[s];
    }
    return kEmpty;
}
// Finds or creates the slot of the n-token key at corpus position i, from slot s on.  Returns the slot, or kEmpty when every slot was
// visited (cannot happen at the load factor the tables are sized for; reported as CB_ERR_PROBE_LIMIT).  A slot's position never
// changes once it is set, so an ordinary load will do; one that still shows an empty slot is put right by the compare-and-swap.
__device__ __forceinline__ uint32_t find_or_claim(unsigned long long* slots, uint32_t S, uint32_t s, const int32_t* corpus, uint32_t i, int n, bool* created) {
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
__device__ __forceinline__ uint32_t home_slot(const int32_t* key, int n, uint32_t S) { return (uint32_t)(hash_tokens(key, n) >> 20) & (S - 1); }
// Slots of the second table that this corpus needs: a power of two, at least twice the windows that go there.
__device__ __forceinline__ uint32_t big_slots(const BuildView& v) {
    uint32_t s = 1024;
    while (s < 2u * __ldcg(&v.st->big_cursor) && s < v.S) s <<= 1;
    return s;
}
__device__ __forceinline__ uint32_t* counts_of(unsigned long long* slots) { return reinterpret_cast<uint32_t*>(slots) + 1; }   // two words apart

// A block's counts of the slots it meets first in each of 512 places; other slots are counted in memory right away.  The count of
// slot s is the word counts[s * STRIDE].
template <int STRIDE>
struct CountCache {
    uint32_t key[512], cnt[512];
    __device__ __forceinline__ void clear() {
        for (int i = threadIdx.x; i < 512; i += blockDim.x) { key[i] = kEmpty; cnt[i] = 0u; }
        __syncthreads();
    }
    __device__ __forceinline__ void add(uint32_t* counts, uint32_t s) {
        const uint32_t at = (s * 0x9E3779B1u) >> 23;
        uint32_t k = key[at];
        if (k == kEmpty) {
            k = atomicCAS(&key[at], kEmpty, s);
            if (k == kEmpty) k = s;
        }
        if (k == s) atomicAdd(&cnt[at], 1u);
        else atomicAdd(counts + (size_t)s * STRIDE, 1u);
    }
    __device__ __forceinline__ void flush(uint32_t* counts) {
        __syncthreads();
        for (int i = threadIdx.x; i < 512; i += blockDim.x)
            if (key[i] != kEmpty && cnt[i]) atomicAdd(counts + (size_t)key[i] * STRIDE, cnt[i]);
    }
};

// Items that threads of a block append to a list in memory: gathered in shared memory, so that the list's counter takes an atomic
// per thousand or so (one address takes one atomic in about 2 ns: an atomic per warp was 260 of 310 us of the leader count).
template <typename T, uint32_t CAP = 2048>
struct Appender {
    static constexpr uint32_t kCap = CAP;
    T item[kCap];
    uint32_t n, at;
    __device__ __forceinline__ void clear() { if (threadIdx.x == 0) n = 0u; __syncthreads(); }
    // All threads of the block together, U items each at most.
    template <int U>
    __device__ __forceinline__ void put(const bool (&has)[U], const T (&x)[U]) {
        const uint32_t lane = threadIdx.x & 31;
        uint32_t m[U], k = 0, total = 0;
#pragma unroll
        for (int q = 0; q < U; ++q) { m[q] = __ballot_sync(CB_FULL, has[q]); total += (uint32_t)__popc(m[q]); }
        if (total && lane == 0) k = atomicAdd(&n, total);
        k = __shfl_sync(CB_FULL, k, 0);
#pragma unroll
        for (int q = 0; q < U; ++q) {
            if (has[q]) item[k + __popc(m[q] & ((1u << lane) - 1u))] = x[q];
            k += (uint32_t)__popc(m[q]);
        }
        __syncwarp();
    }
    __device__ __forceinline__ bool near_full(uint32_t u) const { return *(volatile const uint32_t*)&n > kCap - blockDim.x * u; }
    // The same; true (in all threads) if there may be no room for as many again.  The block decides as one: every warp reads the count
    // before it arrives at the barrier (the last to add sees all of it), and nobody adds again before all have.  Read after a barrier, the
    // count could already hold the next call's additions.
    template <int U>
    __device__ __forceinline__ bool gather(const bool (&has)[U], const T (&x)[U]) {
        put(has, x);
        return __syncthreads_or(near_full(U)) != 0;
    }
    __device__ __forceinline__ void flush(T* list, uint32_t* counter) {
        __syncthreads();
        if (threadIdx.x == 0) at = n ? atomicAdd(counter, n) : 0u;
        __syncthreads();
        for (uint32_t i = threadIdx.x; i < n; i += blockDim.x) list[at + i] = item[i];
        __syncthreads();
        if (threadIdx.x == 0) n = 0u;
        __syncthreads();
    }
};

__global__ void __launch_bounds__(256) fb_init_kernel(BuildView v, CbTables t) {
    CB_PDL_ENTRY();
    const size_t g = (size_t)blockIdx.x * blockDim.x + threadIdx.x, stride = (size_t)gridDim.x * blockDim.x;
    for (size_t i = g; i < (size_t)v.LC; i += stride) { v.grp_n[i] = 0u; t.lstamp[i] = 0u; }
    for (size_t i = g; i < t.nslots; i += stride) t.index[i] = CB_IDX_EMPTY;
    uint4* const e = reinterpret_cast<uint4*>(t.entries);      // E is a multiple of four words
    for (size_t i = g; i < (size_t)v.LC * t.E / 4; i += stride) e[i] = make_uint4(0u, 0u, 0u, 0u);
    if (g < 4) t.hdr[g] = 0u;
    // what the passes want to know of the corpus (the state was cleared before this launch)
    int32_t lo = 0, hi = 0;
    for (size_t i = g; i < v.n_tokens; i += stride) { const int32_t x = v.corpus[i]; lo = min(lo, x); hi = max(hi, x); }
    const bool neg = __syncthreads_or(lo < 0) != 0;
    hi = __reduce_max_sync(CB_FULL, hi);
    __shared__ int32_t s_hi[8];
    if ((threadIdx.x & 31) == 0) s_hi[threadIdx.x >> 5] = hi;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int k = 1; k < 8; ++k) hi = max(hi, s_hi[k]);
        atomicMax(&v.st->max_token, (uint32_t)hi);
        if (neg) { v.st->has_neg = 1u; if (v.M > 0) atomicCAS(&v.st->status, 0u, (uint32_t)CB_ERR_INVALID_ARG); }
    }
    // last, so that it is in L2 when the leaders are counted
    uint4* const key = reinterpret_cast<uint4*>(v.h1);
    uint4* const cnt = reinterpret_cast<uint4*>(v.h1_cnt);
    for (size_t i = g; i < v.S1 / 4; i += stride) cnt[i] = make_uint4(0u, 0u, 0u, 0u);
    for (size_t i = g; i < v.S1 / 2; i += stride) key[i] = make_uint4(kEmpty, kEmpty, kEmpty, kEmpty);
}

// 1. leader counts.  A window a thread at a time, so that eight blocks of 256 fit an SM (32 registers); four at a time, whose chains overlap,
// leave room for four: 4 M windows, LL = 2, 472 us the whole build, 450 with two windows and eight blocks, 446 with one.
// What a block has met lies in shared memory, a key to each place: the windows with such a key are counted there and never look at the
// table, and where the corpus begins, a frequent key's free slot is tried once a block and not by every thread that has it (733 k
// windows, LL = 1: 38 us, 75 without it).
struct KeyCache {
    static constexpr uint32_t N = 1024;
    unsigned long long key[N];
    uint32_t slot[N], cnt[N];
};
// The window at i as one number; false where it has a negative token, which leaves it out.
template <int LL>
__device__ __forceinline__ bool packed_key(const BuildView& v, int bits, bool has_neg, size_t i, unsigned long long* key) {
    *key = 0ull;
#pragma unroll
    for (int j = 0; j < LL; ++j) *key = *key << bits | (uint32_t)v.corpus[i + j];
    bool ok = true;
    for (int j = 0; has_neg && j < LL + v.FL && ok; ++j) ok = v.corpus[i + j] >= 0;
    return ok;
}
template <int LL>
__device__ __forceinline__ void count_packed(const BuildView& v, int bits, KeyCache& cache) {
    for (uint32_t i = threadIdx.x; i < KeyCache::N; i += 256) { cache.key[i] = kNoLeader; cache.cnt[i] = 0u; }
    __syncthreads();
    const bool has_neg = v.st->has_neg != 0u;
    for (size_t i0 = (size_t)blockIdx.x * 256; i0 < v.M; i0 += (size_t)gridDim.x * 256) {
        const size_t i = i0 + threadIdx.x;
        unsigned long long me = kNoLeader;
        const bool ok = i < v.M && packed_key<LL>(v, bits, has_neg, i, &me);
        uint32_t s = kEmpty, at = 0u;
        bool look = false;                                      // this thread finds or makes the slot
        if (ok) {
            const uint64_t h = hash_key(me);
            at = (uint32_t)h & (KeyCache::N - 1);
            unsigned long long k = *reinterpret_cast<volatile unsigned long long*>(&cache.key[at]);
            bool first = false;                                 // and has a place in the cache
            if (k == kNoLeader) {
                k = atomicCAS(&cache.key[at], kNoLeader, me);
                first = k == kNoLeader;
            }
            look = k != me;
            if (!look) {
                atomicAdd(&cache.cnt[at], 1u);
            } else {
                // A slot never changes once it is set, so an ordinary load will do; one that still shows a free slot is put right by
                // the compare-and-swap.
                bool created = false;
                s = home_leader(h, v.S1);
                s = claim_leader(v.h1, v.S1, s, v.h1[s], me, &created, [&](unsigned long long y) { return y == me; });
                if (s == kEmpty) atomicCAS(&v.st->status, 0u, (uint32_t)CB_ERR_PROBE_LIMIT);
                if (first) cache.slot[at] = s;
                if (!created && s != kEmpty) atomicAdd(first ? &cache.cnt[at] : &v.h1_cnt[s], 1u);
            }
        }
        __syncthreads();                                        // the new places' slots are known
        if (i < v.M) v.lslot[i] = !ok ? kEmpty : (look ? s : cache.slot[at]);
    }
    __syncthreads();
    for (uint32_t i = threadIdx.x; i < KeyCache::N; i += 256)
        if (cache.cnt[i] && cache.slot[i] != kEmpty) atomicAdd(&v.h1_cnt[cache.slot[i]], cache.cnt[i]);
}
// The same for longer leaders, most of which a block meets once: no places for keys, the counts alone are gathered.
template <int LL>
__device__ __forceinline__ void count_packed(const BuildView& v, int bits, CountCache<1>& cache) {
    cache.clear();
    const bool has_neg = v.st->has_neg != 0u;
    for (size_t i = (size_t)blockIdx.x * 256 + threadIdx.x; i < v.M; i += (size_t)gridDim.x * 256) {
        unsigned long long me;
        uint32_t s = kEmpty;
        if (packed_key<LL>(v, bits, has_neg, i, &me)) {
            bool created = false;
            s = home_leader(hash_key(me), v.S1);
            s = claim_leader(v.h1, v.S1, s, v.h1[s], me, &created, [&](unsigned long long y) { return y == me; });
            if (s == kEmpty) atomicCAS(&v.st->status, 0u, (uint32_t)CB_ERR_PROBE_LIMIT);
            else if (!created) cache.add(v.h1_cnt, s);
        }
        v.lslot[i] = s;
    }
    cache.flush(v.h1_cnt);
}
// The same with positions in the table: every look at a slot is followed by one at the tokens there.
template <int LL>
__device__ __forceinline__ void count_positions(const BuildView& v, CountCache<1>& cache) {
    cache.clear();
    const bool has_neg = v.st->has_neg != 0u;
    for (size_t i = (size_t)blockIdx.x * 256 + threadIdx.x; i < v.M; i += (size_t)gridDim.x * 256) {
        bool ok = true, created = false;
        for (int j = 0; has_neg && j < LL + v.FL; ++j) ok = ok && v.corpus[i + j] >= 0;
        uint32_t s = kEmpty;
        if (ok) {
            s = home_leader(hash_tokens(v.corpus + i, LL), v.S1);
            s = claim_leader(v.h1, v.S1, s, v.h1[s], i, &created, [&](unsigned long long y) { return same_tokens(v.corpus + (uint32_t)y, v.corpus + i, LL); });
            if (s == kEmpty) atomicCAS(&v.st->status, 0u, (uint32_t)CB_ERR_PROBE_LIMIT);
            else if (!created) cache.add(v.h1_cnt, s);
        }
        v.lslot[i] = s;
    }
    cache.flush(v.h1_cnt);
}
// Up to that many tokens a leader's keys are kept, of the longer ones the counts alone (4 M windows: LL = 2 75 us with keys, 90 with counts; LL = 3
// 101 and 92; 700 k windows: 24 and 29, 30 and 28).
constexpr int kCachedKeys = 2;
template <int LL>
__global__ void __launch_bounds__(256, 8) fb_count_leaders_kernel(BuildView v) {
    CB_PDL_ENTRY();
    __shared__ std::conditional_t<LL <= kCachedKeys, KeyCache, CountCache<1>> cache;
    const int bits = key_bits(v);
    if constexpr (LL * 31 <= 63) {                              // a token has 31 bits at most: one and two of them always fit
        count_packed<LL>(v, bits, cache);
    } else {
        if (bits) count_packed<LL>(v, bits, cache);
        else count_positions<LL>(v, cache);
    }
}

// ---------------------------------------------------------------------------------------------------
// 2. Selection of the LC best leaders and what follows from it, as one cooperative launch: its steps are a few microseconds each
// and every one needs the result of the one before (13 launches otherwise, for 60,000 tokens most of the build's time).
constexpr int kSelThreads = 1024;
struct SelSmem {
    uint32_t bins[kBins], part[32], pick[2], last, start, range, made[4], from[4];
    Appender<uint2, 12288> taken;             // slot and count
    Appender<uint32_t, 12288> tied;           // slot
};

// All blocks of the launch; false after a wait that ran out (the others run out too).  The call then returns CB_ERR_TIMEOUT, whatever
// was recorded before, and the kernels behind this launch do nothing: a leader may have been selected by then without a range.
__device__ __forceinline__ bool grid_barrier(const BuildView& v, uint32_t* round, uint32_t* s_flag) {
    __syncthreads();
    if (threadIdx.x == 0) {
        *round += gridDim.x;
        __threadfence();
        atomicAdd(&v.st->arrived, 1u);
        uint32_t ok = 0u;
        for (uint32_t k = 0; k < v.wait_limit && !ok; ++k) {
            uint32_t x;
            asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(x) : "l"(&v.st->arrived) : "memory");
            ok = x >= *round ? 1u : 0u;
        }
        if (!ok) { v.st->aborted = 1u; atomicExch(&v.st->status, (uint32_t)CB_ERR_TIMEOUT); }
        *s_flag = ok;
    }
    __syncthreads();
    return *s_flag != 0u;
}
// Asked by the kernels after that one, by every thread: a load that L1 serves (past it, thousands of warps at one word cost a kernel 2 us).
__device__ __forceinline__ bool fb_aborted(const BuildView& v) { return v.st->aborted != 0u; }
__device__ __forceinline__ uint32_t sel_scan(uint32_t x, uint32_t* part, uint32_t* total) {   // exclusive, over the block
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t incl = x;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t up = __shfl_up_sync(CB_FULL, incl, o);
        if (lane >= o) incl += up;
    }
    __syncthreads();
    if (lane == 31) part[warp] = incl;
    __syncthreads();
    uint32_t y = part[lane];
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t up = __shfl_up_sync(CB_FULL, y, o);
        if (lane >= o) y += up;
    }
    *total = __shfl_sync(CB_FULL, y, 31);
    const uint32_t before = __shfl_sync(CB_FULL, y, warp > 0 ? warp - 1 : 0);
    return incl - x + (warp > 0 ? before : 0u);
}
// The bin of a finished histogram in which the k-th smallest key lies; *rest: its rank inside the bin.  Every block for itself.
__device__ __forceinline__ uint32_t pick_bin(const uint32_t* hist, uint32_t k, SelSmem& S, uint32_t* rest, uint32_t* all = nullptr) {
    const uint4 c = __ldcg(reinterpret_cast<const uint4*>(hist) + threadIdx.x);      // four bins a thread
    const uint32_t cs[4] = {c.x, c.y, c.z, c.w};
    uint32_t total;
    uint32_t cum = sel_scan(cs[0] + cs[1] + cs[2] + cs[3], S.part, &total);
    if (all) *all = total;                                      // (fewer than k keys: the bin means nothing)
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        if (cum < k && k <= cum + cs[j]) { S.pick[0] = threadIdx.x * 4 + j; S.pick[1] = k - cum; }
        cum += cs[j];
    }
    __syncthreads();
    const uint32_t bin = S.pick[0];
    *rest = S.pick[1];
    __syncthreads();
    return bin;
}
static_assert(kBins == 4 * kSelThreads, "four bins a thread");
// Most counts are the same: the lanes with the first one's bin take one shared atomic, the others one each (__match_any_sync, for one
// per bin, takes some 500 cycles).  kEmpty: none.
__device__ __forceinline__ void add_bin(uint32_t* sh, uint32_t bin) {
    const uint32_t some = __ballot_sync(CB_FULL, bin != kEmpty);
    if (some == 0u) return;
    const int head = __ffs(some) - 1;
    const uint32_t with = __ballot_sync(CB_FULL, bin == __shfl_sync(CB_FULL, bin, head));
    if ((int)(threadIdx.x & 31) == head) atomicAdd(&sh[bin], (uint32_t)__popc(with));
    else if (bin != kEmpty && !((with >> (threadIdx.x & 31)) & 1u)) atomicAdd(&sh[bin], 1u);
}
// Histogram of bin_of(i) over items [0, n) into hist; blocks without an item have nothing to clear and to add.
template <typename F>
__device__ __forceinline__ void sel_histogram(uint32_t n, uint32_t* hist, SelSmem& S, F&& bin_of) {
    if (blockIdx.x * (uint32_t)kSelThreads >= n) return;
    for (int i = threadIdx.x; i < kBins; i += kSelThreads) S.bins[i] = 0u;
    __syncthreads();
    constexpr int U = 4;                                        // items of a thread whose look-ups overlap
    const uint32_t step = gridDim.x * kSelThreads;
    for (uint32_t i0 = blockIdx.x * kSelThreads; i0 < n; i0 += U * step) {
        uint32_t bin[U];
#pragma unroll
        for (int q = 0; q < U; ++q) {
            const uint32_t i = i0 + q * step + threadIdx.x;
            bin[q] = i < n ? bin_of(i) : kEmpty;
        }
#pragma unroll
        for (int q = 0; q < U; ++q) if (i0 + q * step < n) add_bin(S.bins, bin[q]);
    }
    __syncthreads();
    for (int i = threadIdx.x; i < kBins; i += kSelThreads)
        if (S.bins[i]) atomicAdd(&hist[i], S.bins[i]);
}

// The same over the counts of the first table, four slots a load: bin_of(count, slot), for counts of two or more.
template <typename F>
__device__ __forceinline__ void sel_count_histogram(const BuildView& v, uint32_t* hist, SelSmem& S, F&& bin_of) {
    for (int i = threadIdx.x; i < kBins; i += kSelThreads) S.bins[i] = 0u;
    __syncthreads();
    const uint4* const cnt = reinterpret_cast<const uint4*>(v.h1_cnt);
    constexpr int U = 4;
    const uint32_t n = v.S1 / 4, step = gridDim.x * kSelThreads;
    for (uint32_t i0 = blockIdx.x * kSelThreads; i0 < n; i0 += U * step) {
        uint4 c[U];
#pragma unroll
        for (int q = 0; q < U; ++q) { const uint32_t i = i0 + q * step + threadIdx.x; c[q] = i < n ? cnt[i] : make_uint4(0u, 0u, 0u, 0u); }
#pragma unroll
        for (int q = 0; q < U; ++q) {
            const uint32_t x[4] = {c[q].x, c[q].y, c[q].z, c[q].w};
#pragma unroll
            for (int j = 0; j < 4; ++j) add_bin(S.bins, x[j] ? bin_of(x[j] + 1u) : kEmpty);
        }
    }
    __syncthreads();
    for (int i = threadIdx.x; i < kBins; i += kSelThreads)
        if (S.bins[i]) atomicAdd(&hist[i], S.bins[i]);
}

// The leader in slot `at` of the first table, which says `word` from now on, gets entry eid; its key goes into the frozen table's index.
__device__ __forceinline__ void place_leader(const BuildView& v, const CbTables& t, int bits, uint32_t eid, uint32_t at, uint32_t count, uint32_t word) {
    v.h1_cnt[at] = word;
    const uint64_t key = v.h1[at];
    uint32_t* e = t.entries + (size_t)eid * t.E;
    int32_t k4[4] = {0, 0, 0, 0};
#pragma unroll
    for (int j = 0; j < CB_MAX_LL; ++j) if (j < v.LL) { k4[j] = leader_token(v, bits, key, j); e[j] = (uint32_t)k4[j]; }
    t.lstamp[eid] = count;
    const uint64_t h = cb_hash4(k4[0], k4[1], k4[2], k4[3], v.LL);
    const uint32_t nb = t.nslots >> 5, tagged = (cb_hash_tag(h) << CB_EID_BITS) | eid;
    // From a place of its own on through the bucket, then through the next one: with the bucket's first free slot tried first, the eight leaders
    // that it gets at once took eight rounds of a compare-and-swap each (placing 65,536 leaders 27 us).
    uint32_t bucket = cb_hash_bucket(h, t.nslots);
    for (uint32_t p = 0; p < nb; ++p) {
        for (uint32_t j = 0; j < 32u; ++j)
            if (atomicCAS(&t.index[bucket * 32 + (((uint32_t)(h >> 20) + j) & 31u)], CB_IDX_EMPTY, tagged) == CB_IDX_EMPTY) return;
        bucket = (bucket + 1) & (nb - 1);
    }
    atomicCAS(&v.st->status, 0u, (uint32_t)CB_ERR_PROBE_LIMIT);
}


// All leaders gathered so far (slot and count) take entries and ranges for their windows, an atomic for the entries and one per 1,024
// ranges, which lie side by side; those with more than 32 windows are listed by size.  All threads of the block together.  They are
// gathered first because a placement is a chain of some 4 k cycles that the few threads with a leader would otherwise take between two
// barriers of all.
__device__ __forceinline__ void place_taken(const BuildView& v, const CbTables& t, int bits, SelSmem& S) {
    __syncthreads();
    const uint32_t n = S.taken.n;
    if (threadIdx.x == 0) S.start = n ? atomicAdd(&v.st->n_sel, n) : 0u;
    for (uint32_t j0 = 0; j0 < n; j0 += kSelThreads) {
        const uint32_t j = j0 + threadIdx.x;
        const bool has = j < n;
        const uint2 item = has ? S.taken.item[j] : make_uint2(0u, 0u);
        const bool big = item.y > kBigGroup;
        const uint32_t c = big ? 0u : item.y;
        uint32_t total;
        const uint32_t before = sel_scan(c, S.part, &total);
        if (threadIdx.x == 0) S.range = total ? atomicAdd(&v.st->cursor, total) : 0u;
        if (threadIdx.x < 4) S.made[threadIdx.x] = 0u;
        __syncthreads();
        const uint32_t eid = S.start + j;
        const bool fits = has && eid < (uint32_t)v.LC;
        if (has && !fits) atomicCAS(&v.st->status, 0u, (uint32_t)CB_ERR_PROBE_LIMIT);
        // the listed kinds take their places in the block first (one address takes one atomic in about 2 ns)
        const int kind = !fits ? -1 : big ? 3 : c > kMidGroup ? 2 : c > kWarpGroup ? 1 : c > 32u ? 0 : -1;
        const uint32_t place = kind >= 0 ? atomicAdd(&S.made[kind], 1u) : 0u;
        __syncthreads();
        if (threadIdx.x < 4) {
            uint32_t* const lists[4] = {&v.st->n_warp, &v.st->n_mid, &v.st->n_large, &v.st->n_big};
            S.from[threadIdx.x] = S.made[threadIdx.x] ? atomicAdd(lists[threadIdx.x], S.made[threadIdx.x]) : 0u;
        }
        __syncthreads();
        const uint32_t at = kind >= 0 ? S.from[kind] + place : 0u;
        if (kind == 0) v.listed_big[v.LC - 1 - at] = eid;
        else if (kind == 1) v.listed[at] = eid;
        else if (kind == 2) v.listed[v.LC - 1 - at] = eid;
        else if (kind == 3) v.listed_big[at] = eid;
        if (!fits) continue;
        const uint32_t start = S.range + before;
        if (big) {
            v.grp_off[eid] = kBigFlag | atomicAdd(&v.st->big_cursor, item.y);   // no more distinct windows than windows
        } else {
            v.grp_off[eid] = start;
            v.grp_n[eid] = c;
        }
        place_leader(v, t, bits, eid, item.x, item.y, kTaken | (big ? kBigLeader | eid : start));
    }
    __syncthreads();
    if (threadIdx.x == 0) S.taken.n = 0u;
    __syncthreads();
}

__global__ void __launch_bounds__(kSelThreads, 1) fb_select_kernel(BuildView v, CbTables t, int cbits) {
    extern __shared__ __align__(16) unsigned char sel_smem[];
    SelSmem& S = *reinterpret_cast<SelSmem*>(sel_smem);
    const uint32_t LC = (uint32_t)v.LC, cmask = (1u << cbits) - 1u;
    const int bits = key_bits(v);
    bool all = false;                                           // all of them are taken
    uint32_t round = 0, pass = 0, cut = 1, k = LC, n = LC;
    // 2a. the count of the LC-th best leader: a bin per count from two to 4,094 (most comes first), the last one for all above.  The table is
    // read from one end to the other; by a list of its used slots every look was one at random (and the list took the count
    // kernel's blocks a barrier for every four windows of a thread).
    sel_count_histogram(v, v.st->hist[pass], S, [&](uint32_t c) { return kBins - 1 - min(c, (uint32_t)(kBins - 1)); });
    if (!grid_barrier(v, &round, &S.last)) return;
    uint32_t rest, more, bin = pick_bin(v.st->hist[pass++], k, S, &rest, &more);
    if (more < LC) {
        // not enough occur twice: those that occur once tie, or all are taken
        const uint4* const cnt = reinterpret_cast<const uint4*>(v.h1_cnt);
        const ulonglong2* const key = reinterpret_cast<const ulonglong2*>(v.h1);
        uint32_t once = 0;
        for (uint32_t i = blockIdx.x * kSelThreads + threadIdx.x; i < v.S1 / 4; i += gridDim.x * kSelThreads) {
            const uint4 c = cnt[i];
            const ulonglong2 a = key[2 * i], b = key[2 * i + 1];
            once += (c.x == 0u && a.x != kNoLeader) + (c.y == 0u && a.y != kNoLeader) + (c.z == 0u && b.x != kNoLeader) + (c.w == 0u && b.y != kNoLeader);
        }
        once = __reduce_add_sync(CB_FULL, once);
        if ((threadIdx.x & 31) == 0 && once) atomicAdd(&v.st->n_once, once);
        if (!grid_barrier(v, &round, &S.last)) return;
        n = more + __ldcg(&v.st->n_once);
        all = n <= LC;
        k = LC - more;
    } else if (bin > 0u) {
        cut = kBins - 1 - bin;
        k = rest;
    } else {
        // 4,095 or more: digit by digit over the complemented count
        uint32_t prefix = 0;
        for (int shift = (cbits - 1) / kDigitBits * kDigitBits; shift >= 0; shift -= kDigitBits) {
            const uint32_t hi_mask = shift + kDigitBits >= 32 ? 0u : (0xFFFFFFFFu << (shift + kDigitBits));
            sel_count_histogram(v, v.st->hist[pass], S, [&](uint32_t c) {
                const uint32_t x = cmask - c;
                return (x & hi_mask) == (prefix & hi_mask) ? (x >> shift) & (kBins - 1) : kEmpty;
            });
            if (!grid_barrier(v, &round, &S.last)) return;
            bin = pick_bin(v.st->hist[pass++], k, S, &k);
            prefix |= bin << shift;
        }
        cut = cmask - prefix;
    }
    // 2b. the leaders with a larger count are placed, those with the same count listed
    S.taken.clear();
    S.tied.clear();
    const uint32_t step = gridDim.x * kSelThreads;
    {
        constexpr int U = 8;                                    // slots of a thread between two barriers
        const uint4* const cnt = reinterpret_cast<const uint4*>(v.h1_cnt);
        const uint32_t n4 = v.S1 / 4;
        for (uint32_t i0 = blockIdx.x * kSelThreads; i0 < n4; i0 += U / 4 * step) {
            uint4 c4[U / 4];
#pragma unroll
            for (int h = 0; h < U / 4; ++h) { const uint32_t i = i0 + h * step + threadIdx.x; c4[h] = i < n4 ? cnt[i] : make_uint4(0u, 0u, 0u, 0u); }
            uint32_t at[U];
            bool take[U], tie[U];
            uint2 x[U];
#pragma unroll
            for (int q = 0; q < U; ++q) {
                const uint32_t i = i0 + (q / 4) * step + threadIdx.x, c = (q % 4 == 0 ? c4[q / 4].x : q % 4 == 1 ? c4[q / 4].y : q % 4 == 2 ? c4[q / 4].z : c4[q / 4].w) + 1u;
                at[q] = 4 * i + q % 4;
                // a count of one may be a free slot's
                const bool there = c > 1u || (cut == 1u && i < n4 && v.h1[at[q]] != kNoLeader);
                take[q] = there && (all || c > cut);
                tie[q] = there && !take[q] && c == cut;
                x[q] = make_uint2(at[q], c);
            }
            S.taken.put(take, x);
            S.tied.put(tie, at);
            if (__syncthreads_or(S.taken.near_full(U) || S.tied.near_full(U))) {
                place_taken(v, t, bits, S);
                S.tied.flush(v.ties, &v.st->n_ties);
            }
        }
    }
    // (what is gathered by now is placed with the ties that are taken)
    if (all) place_taken(v, t, bits, S);
    S.tied.flush(v.ties, &v.st->n_ties);
    if (blockIdx.x == 0 && threadIdx.x == 0) t.hdr[1] = min(n, LC);
    if (!grid_barrier(v, &round, &S.last)) return;
    if (!all) {
        // 2c. of those the k first by tokens, digit by digit: over the whole number that the slot holds, or token by token
        const uint32_t n_ties = __ldcg(&v.st->n_ties);
        const int words = bits ? 1 : v.LL, wbits = bits ? bits * v.LL : max(32 - __clz((int)v.st->max_token), 1);
        uint64_t prefix[CB_MAX_LL] = {0ull, 0ull, 0ull, 0ull};
        // a thread's first tie stays in its registers: most have no other
        const uint32_t i_mine = blockIdx.x * kSelThreads + threadIdx.x, at_mine = i_mine < n_ties ? __ldcg(&v.ties[i_mine]) : 0u;
        const uint64_t x_mine = v.h1[at_mine];
        auto word = [&](uint64_t x, int w) { return bits ? x : (uint64_t)(uint32_t)v.corpus[(uint32_t)x + w]; };
        auto before_or_in = [&](uint64_t x, int upto) {         // -1, 0, 1: the leader's first words against the prefix
            for (int j = 0; j < upto; ++j) {
                const uint64_t y = word(x, j);
                if (y != prefix[j]) return y < prefix[j] ? -1 : 1;
            }
            return 0;
        };
        for (int w = 0; w < words; ++w)
            for (int shift = (wbits - 1) / kDigitBits * kDigitBits; shift >= 0; shift -= kDigitBits) {
                const uint64_t hi_mask = shift + kDigitBits >= 64 ? 0ull : (~0ull << (shift + kDigitBits));
                sel_histogram(n_ties, v.st->hist[pass], S, [&](uint32_t i) {
                    const uint64_t x = i == i_mine ? x_mine : v.h1[__ldcg(&v.ties[i])];
                    if (before_or_in(x, w) != 0) return kEmpty;
                    const uint64_t y = word(x, w);
                    return (y & hi_mask) == (prefix[w] & hi_mask) ? (uint32_t)(y >> shift) & (kBins - 1) : kEmpty;
                });
                if (!grid_barrier(v, &round, &S.last)) return;
                const uint32_t digit = pick_bin(v.st->hist[pass++], k, S, &k);
                prefix[w] |= (uint64_t)digit << shift;
            }
        // 2d. placed like the others
        for (uint32_t i0 = blockIdx.x * kSelThreads; i0 < n_ties; i0 += step) {
            const uint32_t i = i0 + threadIdx.x, at = i == i_mine ? at_mine : i < n_ties ? __ldcg(&v.ties[i]) : 0u;
            const bool take[1] = {i < n_ties && before_or_in(i == i_mine ? x_mine : v.h1[at], words) <= 0};
            const uint2 item[1] = {make_uint2(at, cut)};
            if (S.taken.gather(take, item)) place_taken(v, t, bits, S);
        }
        place_taken(v, t, bits, S);
        if (!grid_barrier(v, &round, &S.last)) return;
    }
    // 3a. the part of the second table that the big leaders' windows need
    if (__ldcg(&v.st->n_big) == 0u) return;
    const uint32_t S2 = big_slots(v);
    ulonglong2* a = reinterpret_cast<ulonglong2*>(v.h2);
    for (size_t i = (size_t)blockIdx.x * kSelThreads + threadIdx.x; i < S2 / 2; i += (size_t)gridDim.x * kSelThreads) a[i] = make_ulonglong2(kEmptySlot, kEmptySlot);
}

// 3b. every window of a selected leader goes into its leader's range; a big leader's window is counted in the second table, where a
// new one takes its ordinal in its leader's group.  Four windows a thread, whose chains (leader slot, leader, place) overlap.
__global__ void __launch_bounds__(256) fb_windows_kernel(BuildView v) {
    CB_PDL_ENTRY();
    if (fb_aborted(v)) return;
    __shared__ CountCache<2> cache;
    constexpr int U = 4;
    const bool any_big = v.st->n_big != 0u;
    const uint32_t S2 = any_big ? big_slots(v) : 0u;
    if (any_big) cache.clear();
    __shared__ uint2 s_big[8][160];                             // by warp: position and entry id
    const int lane = threadIdx.x & 31;
    uint2* const list = s_big[threadIdx.x >> 5];
    uint32_t n_list = 0;
    auto count_big = [&](bool has) {                            // the last 32 of the list
        const uint2 x = has ? list[n_list + lane] : make_uint2(0u, 0u);
        __syncwarp();
        bool created = false;
        uint32_t s = kEmpty;
        if (has) {
            s = find_or_claim(v.h2, S2, home_slot(v.corpus + x.x, v.LL + v.FL, S2), v.corpus, x.x, v.LL + v.FL, &created);
            if (s == kEmpty) atomicCAS(&v.st->status, 0u, (uint32_t)CB_ERR_PROBE_LIMIT);
            else if (!created) cache.add(counts_of(v.h2), s);
        }
        // the new windows of one leader in a warp take their ordinals with one atomic
        if (__any_sync(CB_FULL, created)) {
            const uint32_t peers = __match_any_sync(CB_FULL, created ? (int)x.y : -1 - lane);
            const int head = __ffs(peers) - 1;
            uint32_t o = 0;
            if (created && lane == head) o = atomicAdd(&v.grp_n[x.y], (uint32_t)__popc(peers));
            o = __shfl_sync(CB_FULL, o, head) + __popc(peers & ((1u << lane) - 1u));
            if (created) v.h2_ord[s] = o;
        }
    };
    const size_t stride = (size_t)gridDim.x * blockDim.x * U;
    for (size_t i0 = (size_t)blockIdx.x * blockDim.x * U; i0 < v.M; i0 += stride) {
        uint32_t slot[U], word[U];
#pragma unroll
        for (int q = 0; q < U; ++q) {
            const size_t i = i0 + (size_t)q * blockDim.x + threadIdx.x;
            slot[q] = i < v.M ? v.lslot[i] : kEmpty;
        }
#pragma unroll
        for (int q = 0; q < U; ++q) word[q] = slot[q] != kEmpty ? v.h1_cnt[slot[q]] : 0u;    // (the flags and an entry id do not change here)
#pragma unroll
        for (int q = 0; q < U; ++q) slot[q] = (word[q] & kTaken) && !(word[q] & kBigLeader) ? atomicAdd(&v.h1_cnt[slot[q]], 1u) & ~kTaken : kEmpty;
#pragma unroll
        for (int q = 0; q < U; ++q) if (slot[q] != kEmpty) v.wpos[slot[q]] = (uint32_t)(i0 + (size_t)q * blockDim.x + threadIdx.x);
        if (!any_big) continue;
        // The big leaders' windows are gathered and counted with full warps: they are a seventh of the windows here, some in every warp.
#pragma unroll
        for (int q = 0; q < U; ++q) {
            const bool is_big = (word[q] & kTaken) && (word[q] & kBigLeader);
            const uint32_t m = __ballot_sync(CB_FULL, is_big);
            if (is_big) list[n_list + __popc(m & ((1u << lane) - 1u))] = make_uint2((uint32_t)(i0 + (size_t)q * blockDim.x + threadIdx.x), word[q] & (kBigLeader - 1u));
            n_list += (uint32_t)__popc(m);
        }
        __syncwarp();
        while (n_list >= 32u) { n_list -= 32u; count_big(true); }
    }
    if (any_big) {
        const uint32_t n = n_list;
        n_list = 0;
        count_big((uint32_t)lane < n);
        cache.flush(counts_of(v.h2));
    }
}
// 3c. the distinct windows of the big leaders, grouped by leader: position and count
__global__ void __launch_bounds__(256) fb_group_scatter_kernel(BuildView v) {
    CB_PDL_ENTRY();
    if (fb_aborted(v) || v.st->n_big == 0u) return;
    const uint32_t S2 = big_slots(v);
    const size_t stride = (size_t)gridDim.x * blockDim.x;
    for (size_t s = (size_t)blockIdx.x * blockDim.x + threadIdx.x; s < S2; s += stride) {
        const unsigned long long x = v.h2[s];
        if ((uint32_t)x == kEmpty) continue;
        const uint32_t eid = v.h1_cnt[v.lslot[(uint32_t)x]] & (kBigLeader - 1u);
        v.group[(v.grp_off[eid] & ~kBigFlag) + v.h2_ord[s]] = make_uint2((uint32_t)x, (uint32_t)(x >> 32));
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

// The distinct windows of a leader: in memory (big leaders), or in shared memory (index of one occurrence + 1 and count in a word, the
// occurrences' follower tokens).
struct MemoryGroup {
    const uint2* g; const int32_t* corpus; int LL;
    __device__ __forceinline__ uint32_t count(uint32_t k) const { return g[k].y; }
    __device__ __forceinline__ const int32_t* tokens(uint32_t k) const { return corpus + g[k].x + LL; }
};
struct SharedGroup {
    const uint32_t* d; const int32_t* tok; int FL;
    __device__ __forceinline__ uint32_t count(uint32_t k) const { return d[k] & 0xFFFFu; }
    __device__ __forceinline__ const int32_t* tokens(uint32_t k) const { return tok + ((d[k] >> 16) - 1u) * FL; }
};

template <int NT, typename Group>
__device__ void pick_followers(const BuildView& v, const CbTables& t, uint32_t eid, const Group& g, uint32_t n, Candidates& cand, const Crew<NT>& crew) {
    // Ties are left in while ranking everything against everything is cheap: FC places and as many windows again, or 64.
    const uint32_t few = (uint32_t)::max(2 * v.FC, 64);
    const int me = (int)threadIdx.x;
    uint32_t cmin = 1;                        // candidates have at least this count
    uint32_t ties = 0;                        // resolved tokens: candidates with exactly cmin come no later than lim[0 .. ties)
    uint32_t lim[CB_MAX_FL];
    uint32_t have = n;
    if (n > (uint32_t)v.FC) {
        // the largest count that FC windows reach
        uint32_t top = 0;
        for (uint32_t k = me; k < n; k += NT) top = ::max(top, g.count(k));
        uint32_t lo = 1, hi = crew.max(top);
        have = n;
        while (lo < hi) {
            const uint32_t mid = lo + (hi - lo + 1u) / 2u;
            uint32_t c = 0;
            for (uint32_t k = me; k < n; k += NT) c += g.count(k) >= mid ? 1u : 0u;
            c = crew.sum(c);
            if (c >= (uint32_t)v.FC) { lo = mid; have = c; } else hi = mid - 1u;
        }
        cmin = lo;
    }
    if (have > few) {
        // too many windows tie at that count: of those only the first by tokens, token by token, until the rest fits
        uint32_t above = 0;
        for (uint32_t k = me; k < n; k += NT) above += g.count(k) > cmin ? 1u : 0u;
        uint32_t need = (uint32_t)v.FC - crew.sum(above);       // ties to be taken, at least one
        for (int lev = 0; lev < v.FL && have > few; ++lev) {
            auto token = [&](uint32_t k, uint32_t* tok) {         // this level's token of a tie that matches the limits so far
                if (g.count(k) != cmin) return false;
                const int32_t* f = g.tokens(k);
                for (int j = 0; j < lev; ++j) if ((uint32_t)f[j] != lim[j]) return false;
                *tok = (uint32_t)f[lev];
                return true;
            };
            uint32_t top = 0, tok = 0;
            for (uint32_t k = me; k < n; k += NT) if (token(k, &tok)) top = ::max(top, tok);
            uint32_t lo = 0, hi = crew.max(top);                // the smallest token that `need` of them do not exceed
            while (lo < hi) {
                const uint32_t mid = lo + (hi - lo) / 2u;
                uint32_t c = 0;
                for (uint32_t k = me; k < n; k += NT) c += token(k, &tok) && tok <= mid ? 1u : 0u;
                if (crew.sum(c) >= need) hi = mid; else lo = mid + 1u;
            }
            uint32_t below = 0, equal = 0;
            for (uint32_t k = me; k < n; k += NT)
                if (token(k, &tok)) { below += tok < lo ? 1u : 0u; equal += tok == lo ? 1u : 0u; }
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
        const uint32_t c = g.count(k);
        const int32_t* const f = g.tokens(k);
        bool in = c > cmin;
        if (c == cmin) {
            in = true;
            for (uint32_t j = 0; j < ties; ++j)
                if ((uint32_t)f[j] != lim[j]) { in = (uint32_t)f[j] < lim[j]; break; }
        }
        if (in) {
            const uint32_t at = atomicAdd(&cand.n, 1u);
            if (at < (uint32_t)kCand) {
                cand.cnt[at] = c;
                for (int j = 0; j < v.FL; ++j) cand.tok[at * v.FL + j] = f[j];
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

// The five kernels of step 4 touch different leaders and depend on nothing but step 3, which is over when the first of them lets
// the others start: so each of them starts as SMs become free and waits for the one before it only at its end (the stream's next
// kernel is ordered behind the last of them only).  A kernel that has not waited yet is promised nothing of what ran before it, so the
// first one, which has, hands step 3 on with a release that every block of the others acquires; it is set when they start, but for a moment.
constexpr uint32_t kGo = 1u, kGaveUp = 2u;
__device__ __forceinline__ void fb_hand_on(const BuildView& v) {
    if (blockIdx.x == 0 && threadIdx.x == 0)
        asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(&v.st->grouped), "r"(fb_aborted(v) ? kGaveUp : kGo) : "memory");
}
__device__ __forceinline__ bool fb_rank_begin(const BuildView& v) {   // false: nothing to rank
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    __shared__ uint32_t s_go;
    if (threadIdx.x == 0) {
        uint32_t x = 0u;
        for (uint32_t k = 0; k < (1u << 24) && x == 0u; ++k)
            asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(x) : "l"(&v.st->grouped) : "memory");
        if (x == 0u) atomicExch(&v.st->status, (uint32_t)CB_ERR_TIMEOUT);
        s_go = x;
    }
    __syncthreads();
    return s_go == kGo;
}
__device__ __forceinline__ void fb_rank_end() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// The big leaders, a block each.  A frequent token of a large corpus has 100 k distinct windows and more, of which the few with the largest counts
// are wanted: a histogram of the counts says from which count on there are FC, and those from there on are copied to shared memory, two looks
// at memory where the bisections of pick_followers took one a step (3.7 M windows, LL = 1, FC = 64: 275 us for the longest leader).  Where too many
// tie, or fewer than FC occur twice, it goes over all of them as they are.
constexpr uint32_t kShort = 2048, kCountBins = 1024;
__global__ void __launch_bounds__(kCountBins) fb_rank_big_kernel(BuildView v, CbTables t) {
    CB_PDL_ENTRY();
    __shared__ Candidates cand;
    __shared__ uint32_t red[32], bins[kCountBins], n_short, from;
    __shared__ uint2 best[kShort];
    const Crew<kCountBins> crew = {red};
    fb_hand_on(v);
    const int me = (int)threadIdx.x, lane = me & 31;
    const uint32_t n_big = fb_aborted(v) ? 0u : v.st->n_big;
    for (uint32_t k = blockIdx.x; k < n_big; k += gridDim.x) {
        const uint32_t eid = v.listed_big[k], n = v.grp_n[eid];
        const uint2* const g = v.group + (v.grp_off[eid] & ~kBigFlag);
        bool few = false;
        if (n > kShort) {
            bins[me] = 0u;
            if (me == 0) { n_short = 0u; from = 0u; }
            __syncthreads();
            constexpr int U = 4;
            for (uint32_t i0 = 0; i0 < n; i0 += U * kCountBins) {
                uint32_t c[U];
#pragma unroll
                for (int q = 0; q < U; ++q) { const uint32_t i = i0 + q * kCountBins + me; c[q] = i < n ? g[i].y : 0u; }
#pragma unroll
                for (int q = 0; q < U; ++q) add_bin(bins, c[q] > 1u ? min(c[q], kCountBins - 1u) : kEmpty);
            }
            __syncthreads();
            uint32_t total;                                     // thread t: how many have the count kCountBins - 1 - t or more
            const uint32_t own = bins[kCountBins - 1 - me], above = sel_scan(own, red, &total);
            if (above < (uint32_t)v.FC && above + own >= (uint32_t)v.FC && above + own <= kShort) from = kCountBins - 1u - (uint32_t)me;
            __syncthreads();
            few = from != 0u;
            for (uint32_t i0 = 0; few && i0 < n; i0 += U * kCountBins) {
                uint2 x[U];
#pragma unroll
                for (int q = 0; q < U; ++q) { const uint32_t i = i0 + q * kCountBins + me; x[q] = i < n ? g[i] : make_uint2(0u, 0u); }
#pragma unroll
                for (int q = 0; q < U; ++q) {
                    const uint32_t m = __ballot_sync(CB_FULL, x[q].y >= from);
                    uint32_t at = 0;
                    if (m && lane == 0) at = atomicAdd(&n_short, (uint32_t)__popc(m));
                    at = __shfl_sync(CB_FULL, at, 0) + __popc(m & ((1u << lane) - 1u));
                    if (x[q].y >= from) best[at] = x[q];
                }
            }
            __syncthreads();
        }
        const MemoryGroup group = {few ? best : g, v.corpus, v.LL};
        pick_followers<kCountBins>(v, t, eid, group, few ? n_short : n, cand, crew);
    }
}

// A block per leader with up to CAP windows: their follower tokens come into shared memory, the distinct ones and their counts are found
// through a table there (a word per slot: index of the first claimant + 1, count).
template <int NT, int CAP>
__global__ void __launch_bounds__(NT) fb_rank_block_kernel(BuildView v, CbTables t, uint32_t n_leaders_at) {
    const bool go = fb_rank_begin(v);
    extern __shared__ uint32_t fb_smem[];
    uint32_t* const tab = fb_smem;                               // [2 CAP], then the distinct windows at its front
    int32_t* const tok = reinterpret_cast<int32_t*>(tab + 2 * CAP); // [CAP][FL]
    __shared__ Candidates cand;
    __shared__ uint32_t red[NT / 32], n_dist;
    const Crew<NT> crew = {red};
    const int me = (int)threadIdx.x, lane = me & 31;
    const uint32_t n = !go ? 0u : n_leaders_at ? v.st->n_large : v.st->n_mid;
    for (uint32_t k = blockIdx.x; k < n; k += gridDim.x) {
        const uint32_t eid = v.listed[n_leaders_at ? (uint32_t)v.LC - 1 - k : k], nw = v.grp_n[eid];
        const uint32_t* const wp = v.wpos + v.grp_off[eid];
        uint32_t slots = 64;                                     // a power of two, at least twice the windows
        while (slots < 2u * nw) slots <<= 1;
        for (uint32_t i = me; i < slots; i += NT) tab[i] = 0u;
        if (me == 0) n_dist = 0u;
        for (uint32_t i = me; i < nw; i += NT) {
            const int32_t* f = v.corpus + wp[i] + v.LL;
#pragma unroll
            for (int j = 0; j < CB_MAX_FL; ++j) if (j < v.FL) tok[i * v.FL + j] = f[j];
        }
        __syncthreads();
        for (uint32_t i = me; i < nw; i += NT) {
            const int32_t* const f = tok + i * v.FL;
            uint32_t x = 0x9E3779B9u;
            for (int j = 0; j < v.FL; ++j) { x = (x ^ (uint32_t)f[j]) * 0x85EBCA77u; x ^= x >> 15; }
            for (uint32_t p = 0, s = x & (slots - 1); p < slots; ++p, s = (s + 1) & (slots - 1)) {
                uint32_t y = *reinterpret_cast<volatile uint32_t*>(&tab[s]);
                if (y == 0u) {
                    y = atomicCAS(&tab[s], 0u, ((i + 1u) << 16) | 1u);
                    if (y == 0u) break;
                }
                const int32_t* const o = tok + ((y >> 16) - 1u) * v.FL;
                int32_t diff = 0;
                for (int j = 0; j < v.FL; ++j) diff |= o[j] ^ f[j];
                if (diff == 0) { atomicAdd(&tab[s], 1u); break; }
            }
        }
        __syncthreads();
        constexpr int PER = 2 * CAP / NT;
        uint32_t y[PER];
#pragma unroll
        for (int q = 0; q < PER; ++q) y[q] = (uint32_t)(q * NT) + me < slots ? tab[q * NT + me] : 0u;
        __syncthreads();
#pragma unroll
        for (int q = 0; q < PER; ++q) {
            const uint32_t m = __ballot_sync(CB_FULL, y[q] != 0u);
            uint32_t at = 0;
            if (m && lane == 0) at = atomicAdd(&n_dist, (uint32_t)__popc(m));
            at = __shfl_sync(CB_FULL, at, 0) + __popc(m & ((1u << lane) - 1u));
            if (y[q]) tab[at] = y[q];
        }
        __syncthreads();
        const SharedGroup g = {tab, tok, v.FL};
        pick_followers<NT>(v, t, eid, g, n_dist, cand, crew);    // ends with a barrier
    }
    fb_rank_end();
}

// Up to kWarpGroup windows, a warp per leader, four windows a lane: the same as the block kernel does with barriers, the warp's own
// table in shared memory and the counts in registers.  A block of 128 threads took 12 us a leader.
constexpr int kRankWarps = 8;
__global__ void __launch_bounds__(32 * kRankWarps) fb_rank_warp_kernel(BuildView v, CbTables t) {
    const bool go = fb_rank_begin(v);
    constexpr int PER = kWarpGroup / 32;
    extern __shared__ uint32_t fb_smem[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t* const tab = fb_smem + warp * (kWarpGroup * (2 + v.FL));      // [2 kWarpGroup]: index of the first claimant + 1, count
    int32_t* const tok = reinterpret_cast<int32_t*>(tab + 2 * kWarpGroup); // [kWarpGroup][FL]
    const uint32_t n = !go ? 0u : v.st->n_warp, below = (1u << lane) - 1u;
    for (uint32_t k = blockIdx.x * kRankWarps + warp; k < n; k += gridDim.x * kRankWarps) {
        const uint32_t eid = v.listed_big[(uint32_t)v.LC - 1 - k], nw = v.grp_n[eid];
        const uint32_t* const wp = v.wpos + v.grp_off[eid];
        uint32_t pos[PER];
#pragma unroll
        for (int q = 0; q < PER; ++q) pos[q] = q * 32 + lane < nw ? wp[q * 32 + lane] : 0u;
#pragma unroll
        for (int q = 0; q < 2 * PER; ++q) tab[q * 32 + lane] = 0u;
#pragma unroll
        for (int q = 0; q < PER; ++q)
            if (q * 32 + lane < nw) {
                const int32_t* f = v.corpus + pos[q] + v.LL;
#pragma unroll
                for (int j = 0; j < CB_MAX_FL; ++j) if (j < v.FL) tok[(q * 32 + lane) * v.FL + j] = f[j];
            }
        __syncwarp();
#pragma unroll 1
        for (uint32_t i = lane; i < nw; i += 32) {
            const int32_t* const f = tok + i * v.FL;
            uint32_t x = 0x9E3779B9u;
            for (int j = 0; j < v.FL; ++j) { x = (x ^ (uint32_t)f[j]) * 0x85EBCA77u; x ^= x >> 15; }
            for (uint32_t p = 0, s = x & (2 * kWarpGroup - 1); p < 2 * kWarpGroup; ++p, s = (s + 1) & (2 * kWarpGroup - 1)) {
                uint32_t y = *reinterpret_cast<volatile uint32_t*>(&tab[s]);
                if (y == 0u) {
                    y = atomicCAS(&tab[s], 0u, ((i + 1u) << 16) | 1u);
                    if (y == 0u) break;
                }
                const int32_t* const o = tok + ((y >> 16) - 1u) * v.FL;
                int32_t diff = 0;
                for (int j = 0; j < v.FL; ++j) diff |= o[j] ^ f[j];
                if (diff == 0) { atomicAdd(&tab[s], 1u); break; }
            }
        }
        __syncwarp();
        // the distinct ones to the front of the table (a slot is read before its group of 32 or an earlier one is written)
        uint32_t nd = 0;
#pragma unroll
        for (int q = 0; q < 2 * PER; ++q) {
            const uint32_t y = tab[q * 32 + lane], m = __ballot_sync(CB_FULL, y != 0u);
            __syncwarp();
            if (y) tab[nd + __popc(m & below)] = y;
            nd += (uint32_t)__popc(m);
            __syncwarp();
        }
        uint32_t cnt[PER];
        const int32_t* f[PER];
#pragma unroll
        for (int q = 0; q < PER; ++q) {
            const uint32_t y = q * 32 + lane < nd ? tab[q * 32 + lane] : 0u;
            cnt[q] = y & 0xFFFFu;
            f[q] = tok + (y ? (y >> 16) - 1u : 0u) * v.FL;
        }
        // in[q]: among the FC best.  First the largest count that FC of them reach, then the ties at it token by token.
        bool in[PER];
#pragma unroll
        for (int q = 0; q < PER; ++q) in[q] = cnt[q] > 0u;
        if (nd > (uint32_t)v.FC) {
            auto sum = [&](auto&& has) {
                uint32_t c = 0;
#pragma unroll
                for (int q = 0; q < PER; ++q) c += (uint32_t)__popc(__ballot_sync(CB_FULL, has(q)));
                return c;
            };
            uint32_t top = 0;
#pragma unroll
            for (int q = 0; q < PER; ++q) top = max(top, cnt[q]);
            uint32_t lo = 1, hi = __reduce_max_sync(CB_FULL, top);
            while (lo < hi) {
                const uint32_t mid = lo + (hi - lo + 1u) / 2u;
                if (sum([&](int q) { return cnt[q] >= mid; }) >= (uint32_t)v.FC) lo = mid; else hi = mid - 1u;
            }
            uint32_t need = (uint32_t)v.FC - sum([&](int q) { return cnt[q] > lo; });   // ties to be taken, at least one
            bool tie[PER];
#pragma unroll
            for (int q = 0; q < PER; ++q) { in[q] = cnt[q] > lo; tie[q] = cnt[q] == lo; }
            // the ties with the smallest first token, then the next ones; where one token has too many, those by their next token
            for (int lev = 0; lev < v.FL && sum([&](int q) { return tie[q]; }) > need; ++lev) {
                uint32_t x[PER], least = 0u, many = 0u;
#pragma unroll
                for (int q = 0; q < PER; ++q) x[q] = tie[q] ? (uint32_t)f[q][lev] : 0xFFFFFFFFu;
                for (uint32_t got = 0u;;) {                      // at most FC rounds: each takes one tie or more
                    uint32_t mn = 0xFFFFFFFFu;
#pragma unroll
                    for (int q = 0; q < PER; ++q) mn = min(mn, x[q]);
                    least = __reduce_min_sync(CB_FULL, mn);
                    many = sum([&](int q) { return x[q] == least; });
                    if (got + many >= need) { need -= got; break; }
                    got += many;
#pragma unroll
                    for (int q = 0; q < PER; ++q) if (x[q] == least) { in[q] = true; x[q] = 0xFFFFFFFFu; }
                }
#pragma unroll
                for (int q = 0; q < PER; ++q) tie[q] = x[q] == least;
            }
#pragma unroll
            for (int q = 0; q < PER; ++q) in[q] = in[q] || tie[q];
        }
        // those that are in, side by side at the front of the table, and each one's rank among them
        __syncwarp();
        uint32_t ni = 0;
        uint32_t keep[PER];
#pragma unroll
        for (int q = 0; q < PER; ++q) keep[q] = q * 32 + lane < nd ? tab[q * 32 + lane] : 0u;
        __syncwarp();
#pragma unroll
        for (int q = 0; q < PER; ++q) {
            const uint32_t m = __ballot_sync(CB_FULL, in[q]);
            if (in[q]) tab[ni + __popc(m & below)] = keep[q];
            ni += (uint32_t)__popc(m);
        }
        __syncwarp();
        uint32_t* e = t.entries + (size_t)eid * t.E;
        for (uint32_t i = lane; i < ni; i += 32) {
            const uint32_t y = tab[i];
            const int32_t* const g = tok + ((y >> 16) - 1u) * v.FL;
            uint32_t rank = 0;
            for (uint32_t o = 0; o < ni; ++o) {
                const uint32_t z = tab[o];
                bool before = (z & 0xFFFFu) > (y & 0xFFFFu);
                if ((z & 0xFFFFu) == (y & 0xFFFFu)) {
                    const int32_t* const h = tok + ((z >> 16) - 1u) * v.FL;
                    for (int j = 0; j < v.FL; ++j)
                        if (h[j] != g[j]) { before = h[j] < g[j]; break; }
                }
                rank += before ? 1u : 0u;
            }
            for (int j = 0; j < v.FL; ++j) e[v.LL + v.FC + rank * v.FL + j] = (uint32_t)g[j];
            e[v.LL + rank] = (uint32_t)v.FC - rank;
        }
        __syncwarp();                                           // the table is overwritten by the next leader
    }
    fb_rank_end();
}

// the common case, up to 32 windows: a warp per leader, a lane per window; the next leader's range is looked up while this one is ranked
__global__ void __launch_bounds__(256) fb_rank_kernel(BuildView v, CbTables t) {
    const bool go = fb_rank_begin(v);
    const int lane = threadIdx.x & 31;
    const uint32_t n = !go ? 0u : min(v.st->n_sel, (uint32_t)v.LC), nw = gridDim.x * 8;
    const bool short_tokens = go && v.st->max_token < (1u << 26);
    uint32_t eid = blockIdx.x * 8 + (threadIdx.x >> 5);
    // windows of leader e for this warp (0: another kernel's) and this lane's position
    auto range_of = [&](uint32_t e, uint32_t* pos) {
        const uint32_t c = e < n ? t.lstamp[e] : 0u, off = e < n ? v.grp_off[e] : 0u;
        *pos = 0u;
        if (c == 0u || c > 32u) return 0u;
        if ((uint32_t)lane < c) *pos = v.wpos[off + lane];
        return c;
    };
    uint32_t pos_next, ng_next = range_of(eid, &pos_next);
    for (; eid < n; eid += nw) {
        const uint32_t ng = ng_next, pos = pos_next;
        const bool mine = (uint32_t)lane < ng;
        int32_t f[CB_MAX_FL];
#pragma unroll
        for (int j = 0; j < CB_MAX_FL; ++j) f[j] = mine && j < v.FL ? v.corpus[pos + v.LL + j] : -1 - lane;
        ng_next = range_of(eid + nw, &pos_next);
        if (ng == 0u) continue;
        // the lanes with the same follower: its count; the first of them stands for it.  Compared by a hash, the hash by the tokens
        // (__match_any_sync on each token instead held every warp of an SM up for some 500 cycles a call).
        uint32_t x = 0x9E3779B9u;
#pragma unroll
        for (int j = 0; j < CB_MAX_FL; ++j) { if (j >= v.FL) break; x = (x ^ (uint32_t)f[j]) * 0x85EBCA77u; x ^= x >> 15; }
        uint32_t same = 0u;
        for (uint32_t k = 0; k < ng; ++k) same |= (__shfl_sync(CB_FULL, x, k) == x ? 1u : 0u) << k;
        const int rep = mine ? __ffs(same) - 1 : lane;
        bool differ = false;
#pragma unroll
        for (int j = 0; j < CB_MAX_FL; ++j) { if (j >= v.FL) break; differ = __shfl_sync(CB_FULL, f[j], rep) != f[j] || differ; }
        if (__any_sync(CB_FULL, differ)) {                      // two followers with one hash: token by token
            same = 0u;
            for (uint32_t k = 0; k < ng; ++k) {
                bool eq = true;
#pragma unroll
                for (int j = 0; j < CB_MAX_FL; ++j) { if (j >= v.FL) break; eq = __shfl_sync(CB_FULL, f[j], k) == f[j] && eq; }
                same |= (eq ? 1u : 0u) << k;
            }
        }
        const uint32_t cnt = (uint32_t)__popc(same);
        const bool stands = mine && (same & ((1u << lane) - 1u)) == 0u;
        const uint32_t standing = __ballot_sync(CB_FULL, stands);
        // Count and first token in one word, the second token in another (smaller comes first): seven instructions for each of the others
        // where the loop below, for two followers with the same words, takes twenty-five.
        const uint32_t key = (32u - cnt) << 26 | (uint32_t)f[0], key2 = v.FL > 1 ? (uint32_t)f[1] : 0u;
        int rank = 0, alike = 0;
        if (short_tokens)
            for (uint32_t m = standing; m; m &= m - 1u) {
                const int k = __ffs(m) - 1;
                const uint32_t o = __shfl_sync(CB_FULL, key, k), o2 = __shfl_sync(CB_FULL, key2, k);
                rank += o < key || (o == key && o2 < key2) ? 1 : 0;
                alike += o == key && o2 == key2 ? 1 : 0;
            }
        if (!short_tokens || __any_sync(CB_FULL, stands && alike > 1)) {
            rank = 0;
            for (uint32_t m = standing; m; m &= m - 1u) {
                const int k = __ffs(m) - 1;
                const uint32_t oc = __shfl_sync(CB_FULL, cnt, k);
                int cmp = oc > cnt ? -1 : (oc < cnt ? 1 : 0);    // -1: the other one comes before
#pragma unroll
                for (int j = 0; j < CB_MAX_FL; ++j) {
                    if (j >= v.FL) break;
                    const int32_t o = __shfl_sync(CB_FULL, f[j], k);
                    if (cmp == 0 && o != f[j]) cmp = o < f[j] ? -1 : 1;
                }
                rank += cmp < 0 ? 1 : 0;
            }
        }
        if (stands && rank < v.FC) {
            uint32_t* e = t.entries + (size_t)eid * t.E;
#pragma unroll
            for (int j = 0; j < CB_MAX_FL; ++j) if (j < v.FL) e[v.LL + v.FC + rank * v.FL + j] = (uint32_t)f[j];
            e[v.LL + rank] = (uint32_t)(v.FC - rank);
        }
    }
    fb_rank_end();
}

size_t fb_align(size_t x) { return (x + 255) / 256 * 256; }

struct BuildLayout {
    uint32_t S1, S;
    size_t off_cnt, off_h2, off_h2_ord, off_lslot, off_group, off_grp, total;
};

cb_status fb_layout(const cb_frozen_config* c, int64_t n_tokens, BuildLayout* B) {
    if (n_tokens < 0 || n_tokens > (int64_t)1 << 30) return CB_ERR_INVALID_ARG;
    const int64_t M = n_tokens - c->LL - c->FL + 1 > 0 ? n_tokens - c->LL - c->FL + 1 : 0;
    uint64_t S = 1024;
    while (S < 2ull * (uint64_t)M) S <<= 1;
    B->S = (uint32_t)S;
    size_t o = fb_align(sizeof(BuildState));
    uint64_t S1 = ((uint64_t)M + (uint64_t)M / 3 + 1024) / 4 * 4;
    B->S1 = (uint32_t)S1;
    B->off_cnt = o;     o = fb_align(o + S1 * 4);
    B->off_h2 = o;      o = fb_align(o + std::max(S, S1) * 8);   // until the selection's end it holds the first table's words
    B->off_h2_ord = o;  o = fb_align(o + S * 4);
    B->off_lslot = o;   o = fb_align(o + (size_t)(M > 0 ? M : 1) * 4);
    B->off_group = o;   o = fb_align(o + S * 6);   // M x 8 bytes, then M x 4
    B->off_grp = o;     o = fb_align(o + (size_t)c->LC * 4 * 4);
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

static cb_status frozen_build(const cb_frozen_config* cfg, const int32_t* dev_corpus, int64_t n_tokens, void* dev_table,
                              size_t table_bytes, void* dev_scratch, size_t scratch_bytes, void* stream, uint32_t wait_limit) {
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
    v.h1_cnt = (uint32_t*)(base + B.off_cnt);
    v.h2 = v.h1 = (unsigned long long*)(base + B.off_h2); v.h2_ord = (uint32_t*)(base + B.off_h2_ord);
    v.lslot = (uint32_t*)(base + B.off_lslot);
    v.group = (uint2*)(base + B.off_group); v.ties = (uint32_t*)(base + B.off_group);   // M <= S / 2
    v.wpos = (uint32_t*)(v.group + B.S / 2);                      // behind group's M places
    v.grp_n = (uint32_t*)(base + B.off_grp); v.grp_off = v.grp_n + cfg->LC; v.listed = v.grp_off + cfg->LC;
    v.listed_big = v.listed + cfg->LC;
    v.S1 = B.S1; v.S = B.S;
    v.corpus = dev_corpus;
    const int64_t M = n_tokens - cfg->LL - cfg->FL + 1;
    v.M = (uint32_t)(M > 0 ? M : 0);
    v.n_tokens = (uint32_t)n_tokens;
    v.wait_limit = wait_limit;
    v.LL = cfg->LL; v.FL = cfg->FL; v.LC = cfg->LC; v.FC = cfg->FC;
    int dev = 0, sms = 0;
    CB_CUDA(cudaGetDevice(&dev));
    CB_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    const dim3 grid((unsigned)(sms * 8)), block(256);
    CB_CUDA(cudaMemsetAsync(v.st, 0, sizeof(BuildState), st));
    CB_CUDA(cb_launch_pdl(fb_init_kernel, grid, block, 0, st, v, t));
    if (v.M > 0) {
        // shared memory of step 4's blocks: table, follower tokens
        auto block_smem = [&](uint32_t cap) { return (size_t)(2 + cfg->FL) * cap * 4; };
        auto* const mid = fb_rank_block_kernel<128, kMidGroup>;
        auto* const large = fb_rank_block_kernel<512, kBigGroup>;
        CB_CUDA(cudaFuncSetAttribute(large, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(2 + CB_MAX_FL) * kBigGroup * 4));
        int cbits = 1;                                        // counts are at most M
        while (cbits < 31 && (v.M >> cbits) != 0) ++cbits;
        CB_CUDA(cudaFuncSetAttribute(fb_select_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(SelSmem)));
        static_assert(CB_MAX_LL == 4, "a leader count for every leader length");
        auto* const count = cfg->LL == 1 ? fb_count_leaders_kernel<1> : cfg->LL == 2 ? fb_count_leaders_kernel<2>
                            : cfg->LL == 3 ? fb_count_leaders_kernel<3> : fb_count_leaders_kernel<4>;
        CB_CUDA(cb_launch_pdl(count, grid, block, 0, st, v));
        {
            // a block per SM, all resident at once: they wait for one another
            cudaLaunchConfig_t lc = {};
            lc.gridDim = dim3((unsigned)sms); lc.blockDim = dim3(kSelThreads); lc.dynamicSmemBytes = sizeof(SelSmem); lc.stream = st;
            cudaLaunchAttribute at[1];
            at[0].id = cudaLaunchAttributeCooperative;
            at[0].val.cooperative = 1;
            lc.attrs = at; lc.numAttrs = 1;
            CB_CUDA(cudaLaunchKernelEx(&lc, fb_select_kernel, v, t, cbits));
        }
        CB_CUDA(cb_launch_pdl(fb_windows_kernel, grid, block, 0, st, v));
        CB_CUDA(cb_launch_pdl(fb_group_scatter_kernel, grid, block, 0, st, v));
        CB_CUDA(cb_launch_pdl(fb_rank_big_kernel, dim3((unsigned)sms), dim3(kCountBins), 0, st, v, t));
        CB_CUDA(cb_launch_pdl(large, dim3((unsigned)(sms * 2)), dim3(512), block_smem(kBigGroup), st, v, t, 1u));
        CB_CUDA(cb_launch_pdl(mid, dim3((unsigned)(sms * 8)), dim3(128), block_smem(kMidGroup), st, v, t, 0u));
        const size_t warp_smem = (size_t)kRankWarps * kWarpGroup * (2 + cfg->FL) * 4;
        CB_CUDA(cb_launch_pdl(fb_rank_warp_kernel, dim3((unsigned)(sms * 8)), dim3(32 * kRankWarps), warp_smem, st, v, t));
        CB_CUDA(cb_launch_pdl(fb_rank_kernel, grid, block, 0, st, v, t));
        cb_count_launch(9);
    }
    cb_count_launch(1);
    uint32_t status = 0;
    CB_CUDA(cudaMemcpyAsync(&status, &v.st->status, 4, cudaMemcpyDeviceToHost, st));
    CB_CUDA(cudaStreamSynchronize(st));
    return (cb_status)status;
}

extern "C" cb_status cb_frozen_build(const cb_frozen_config* cfg, const int32_t* dev_corpus, int64_t n_tokens, void* dev_table,
                                     size_t table_bytes, void* dev_scratch, size_t scratch_bytes, void* stream) {
    return frozen_build(cfg, dev_corpus, n_tokens, dev_table, table_bytes, dev_scratch, scratch_bytes, stream, 1u << 24);
}

#ifdef CB_DEBUG
// Checking build only: the same with the number of looks that a block of the selection takes at a barrier (0: it gives up at once).
extern "C" cb_status cb_debug_frozen_build(const cb_frozen_config* cfg, const int32_t* dev_corpus, int64_t n_tokens, void* dev_table,
                                           size_t table_bytes, void* dev_scratch, size_t scratch_bytes, void* stream, uint32_t wait_limit) {
    return frozen_build(cfg, dev_corpus, n_tokens, dev_table, table_bytes, dev_scratch, scratch_bytes, stream, wait_limit);
}
#endif

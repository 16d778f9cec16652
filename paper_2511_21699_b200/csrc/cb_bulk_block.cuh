// Bulk update of runs whose reduction fits a block's shared memory (prompts of up to kBlkRun windows), one launch for the whole
// call.  Included by cb_table.cu after the table helpers.
//
// The reduction is the order-free one of cb_bulk_free.cuh (a leader's stamp is that of its last window, its followers are the FC
// distinct ones touched last), but a sequence is cut into parts by a hash of the leader and a block does one part alone: the tokens
// of the run, the table of the part's leaders and that of its (leader, follower) pairs lie in shared memory, so claims, "last
// index" maxima and the grouping of pairs by leader are shared-memory operations, and what is left in global memory is an atomic per
// new leader and the entry itself.  Through scratch in global memory the same run is six launches whose every step is a chain of L2
// round trips: batch 32 of 1,024 to 8,192 tokens (147 k windows), reset and first draft with it, 118 us against 30.0 us this way
// (some 17 of them this kernel's, 36 k cycles: lengths, parts and tokens 6 k, listing the part's windows 4 k, claims 7 k with the second
// turn of those beyond 1,024, ranges and grouping 2.5 k, entries and their index words 12 k, the rest at the end).  What bounds it is the chain of phases in a block, a thread or two per window: a quarter of the SM's issue
// rate, a fifth of the shared-memory pipe, 5 MB from DRAM; half of the stalled warps wait at a barrier.
//
// Parts: every block reads all lengths and deals gridDim.x parts to the sequences in proportion to their windows (at least one
// each, and no more than kBlkPart windows expected in one, so that the tables stay at most half full), so no plan kernel and no host
// knowledge of the lengths is needed.  A block that has a part of sequence b reads all of its tokens and hashes all of its windows
// (a few per thread) and keeps those of its part.
//
// What the blocks of a sequence share: hdr[0] and hdr[1] (clock, leaders) are read by all and not changed while any is at work;
// entry ids come from hdr[2], arrivals are counted in hdr[3] (both zero between calls), and the last block to arrive folds them
// into hdr[0] and hdr[1].  A sequence that does not qualify (fewer than 64 windows, or a leader could be evicted during the run) stays one
// (its leaders only grow in number) and is left to the kernels after this one, or, where there are none (`alone`), done in order
// by one warp of the block that has its first part, side by side with the block's others: such a run is a chain of 1 to 2.5 k cycles a
// window (batch 1,024 of 45 windows: 292 us with a block's one after the other, 64 so; batch 512 of 5,000 that evict, in the kernel
// behind: 52.4 ms and 7.2).
#pragma once

namespace {

constexpr int kBlkThreads = 1024;
constexpr int kBlkRun = 8192;          // windows of a run: positions fit 16 bits beside one another, and the tables hold them all
constexpr int kBlkPart = 4096;         // windows expected in a part
constexpr int kBlkSlots = 8192;        // slots of either table: a part that takes a whole run of distinct windows just fills them
constexpr int kBlkMaxBatch = 1024;     // a length per thread
static_assert(kBlkSlots >= kBlkRun && kBlkRun < 65535, "every window finds a slot");

struct BlkSmem {
    uint32_t pair[kBlkSlots];          // (first window + 1) << 16 | (last window + 1) of a distinct window, 0 = free
    uint32_t lead[kBlkSlots];          // the same of a distinct leader
    uint32_t cur[kBlkSlots];           // by leader slot: pairs, then next place of its range of group; then, by leader: entry + 1
    uint16_t pl[kBlkSlots];            // leader slot of a pair; then the list of leaders that take a whole warp
    uint16_t group[kBlkSlots];         // pair slots grouped by leader
    uint16_t lslot[kBlkSlots];         // the leaders' slots
    uint16_t pslot[kBlkSlots];         // the pairs' slots
    uint16_t gbase[kBlkSlots + 8];     // start of each leader's range of group
    int32_t tok[kBlkRun + CB_MAX_LL + CB_MAX_FL];
    uint32_t pre[kBlkMaxBatch + 1];    // parts of the sequences before b
    int32_t first[kBlkMaxBatch];       // first position, clock, leaders and windows of every sequence
    uint32_t clock[kBlkMaxBatch], count[kBlkMaxBatch];
    uint16_t nwin[kBlkMaxBatch];
    float inv;                         // one over the windows of a part
    uint32_t red[32], total, n_multi, n_own, n_lead, n_pair, n_fresh, n_list, base;
};
static_assert(sizeof(BlkSmem) <= 227 * 1024, "shared memory of one CTA");
constexpr uint32_t kBlkFresh = 0x80000000u;

// Sum over the block of x in the threads before this one; *total: over all of them.
__device__ __forceinline__ uint32_t blk_scan(uint32_t x, uint32_t* red, uint32_t* total) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t incl = x;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t up = __shfl_up_sync(CB_FULL, incl, o);
        if (lane >= o) incl += up;
    }
    __syncthreads();
    if (lane == 31) red[warp] = incl;
    __syncthreads();
    uint32_t w = red[lane];
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t up = __shfl_up_sync(CB_FULL, w, o);
        if (lane >= o) w += up;
    }
    *total = __shfl_sync(CB_FULL, w, 31);
    const uint32_t before = __shfl_sync(CB_FULL, w, warp > 0 ? warp - 1 : 0);
    return incl - x + (warp > 0 ? before : 0u);
}

// Finds or claims the slot of the N-token key (n of them in use, held in key) at window k in a shared table and raises its last window.
// All of a candidate's tokens are read at once: compared one by one they were a chain of shared-memory round trips.
template <int N>
__device__ __forceinline__ uint32_t blk_slot(uint32_t* slots, const int32_t* tok, const int32_t (&key)[N], int n, uint32_t h, uint32_t k, bool* created) {
    const uint32_t me = ((k + 1u) << 16) | (k + 1u);
    uint32_t s = h & (kBlkSlots - 1);
    *created = false;
    for (int p = 0; p < kBlkSlots; ++p) {
        uint32_t x = *reinterpret_cast<volatile uint32_t*>(&slots[s]);
        if (x == 0u) {
            x = atomicCAS(&slots[s], 0u, me);
            if (x == 0u) { *created = true; return s; }
        }
        const int32_t* q = tok + (x >> 16) - 1u;
        int32_t diff = 0;
#pragma unroll
        for (int j = 0; j < N; ++j) if (j < n) diff |= q[j] ^ key[j];
        if (diff == 0) {
            if ((x & 0xFFFFu) < k + 1u) atomicMax(&slots[s], (x & 0xFFFF0000u) | (k + 1u));
            return s;
        }
        s = (s + 1u) & (kBlkSlots - 1);
    }
    return 0u;                                                  // excluded: there are as many slots as windows
}

// Hash of a window: of the leader's tokens, carried on over the follower's.
template <int LL, int N>
__device__ __forceinline__ uint32_t blk_leader_hash(const int32_t (&key)[N]) {
    uint32_t x = 0x9E3779B9u;
#pragma unroll
    for (int j = 0; j < LL; ++j) { x = (x ^ (uint32_t)key[j]) * 0x85EBCA77u; x ^= x >> 15; }
    return x;
}
template <int LL, int N>
__device__ __forceinline__ uint32_t blk_pair_hash(uint32_t x, const int32_t (&key)[N], int n) {
#pragma unroll
    for (int j = LL; j < N; ++j) if (j < n) { x = (x ^ (uint32_t)key[j]) * 0x9E3779B1u; x ^= x >> 15; }
    return x;
}

// Followers that the part's windows displace one after the other, which the reduction itself cannot say (it stores the latest only):
// every listed leader that cannot keep all of its followers is marked, the marked ones' windows are listed in order, and a warp per
// leader goes through its own among them with the leader's list in registers: lane l keeps places l, l + 32, ...: the stamp (0: free) and
// the slot in `pair` of what is stored there.  All threads together; each warp gets its own share of the sum.  What it costs is some 300
// cycles for each window of the most frequent leader, one after the other: batch 32 of 1,024 to 8,192 tokens,
// reset and first draft included, 70 us where 32 do without (leaders of one token: 195 and 36).
constexpr uint32_t kBlkMark = 0x80000000u;      // of a leader's word; windows stay below 2^14
template <int LL, int FLX, int CH>
__device__ __noinline__ uint32_t blk_evictions(BlkSmem& S, const uint32_t* entries, uint32_t E, int FL, int FC, uint32_t count0, uint32_t clock0,
                                               uint32_t nwin, uint32_t part, uint32_t np) {
    constexpr uint32_t kNone = 0xFFFFFFFFu;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, w = LL + FL;
    auto find = [&](const uint32_t* slots, const int32_t (&key)[LL + FLX], int n, uint32_t h) {
        uint32_t at = h & (kBlkSlots - 1);
        for (int p = 0; p < kBlkSlots; ++p) {
            const uint32_t x = slots[at] & ~kBlkMark;
            if (x == 0u) break;
            const int32_t* q = S.tok + (x >> 16) - 1u;
            int32_t diff = 0;
#pragma unroll
            for (int j = 0; j < LL + FLX; ++j) if (j < n) diff |= q[j] ^ key[j];
            if (diff == 0) return at;
            at = (at + 1u) & (kBlkSlots - 1);
        }
        return kNone;
    };
    auto pair_of = [&](const int32_t (&key)[LL + FLX]) { return find(S.pair, key, w, blk_pair_hash<LL>(blk_leader_hash<LL>(key), key, w)); };
    uint32_t id[CH], st[CH];
    // Reads leader o's list as it was before the run; true if the run's followers do not all have room beside it.
    auto crowded = [&](uint32_t o) {
        const uint32_t at = ((S.lead[S.lslot[o]] & ~kBlkMark) >> 16) - 1u, x = count0 > 0u ? S.cur[o] : kBlkFresh;
        const uint32_t* e = entries + (size_t)((x & kBlkFresh) ? 0u : x - 1u) * E;
        uint32_t stored = 0, known = 0;
#pragma unroll
        for (int c = 0; c < CH; ++c) {
            const int f = c * 32 + lane;
            id[c] = kNone;
            st[c] = !(x & kBlkFresh) && f < FC ? e[LL + f] : 0u;
            if (st[c]) {
                int32_t key[LL + FLX];
#pragma unroll
                for (int j = 0; j < LL + FLX; ++j) key[j] = j < LL ? S.tok[at + j] : j < w ? (int32_t)e[LL + FC + f * FL + j - LL] : 0;
                id[c] = pair_of(key);
            }
            stored += __popc(__ballot_sync(CB_FULL, st[c] != 0u));
            known += __popc(__ballot_sync(CB_FULL, id[c] != kNone));
        }
        return stored + (S.gbase[o + 1] - S.gbase[o]) - known > (uint32_t)FC;
    };
    const uint32_t n_list = S.n_list;
    bool any = false;
    for (uint32_t i = warp; i < n_list; i += kBlkThreads / 32) {
        const uint32_t o = S.pl[i];
        if (!crowded(o)) continue;
        any = true;
        if (lane == 0) atomicOr(&S.lead[S.lslot[o]], kBlkMark);
    }
    if (!__syncthreads_or(any)) return 0u;
    uint32_t m = 0;
    for (uint32_t k0 = 0; k0 < nwin; k0 += kBlkThreads) {
        const uint32_t k = k0 + tid;
        bool in = false;
        if (k < nwin) {
            int32_t key[LL + FLX];
            uint32_t x = 0x85EBCA6Bu;
#pragma unroll
            for (int j = 0; j < LL + FLX; ++j) {
                key[j] = j < LL ? S.tok[k + j] : 0;
                if (j < LL) { x = (x ^ (uint32_t)key[j]) * 0x9E3779B1u; x ^= x >> 16; }
            }
            if (__umulhi(x * 0xC2B2AE35u, np) == part) {
                const uint32_t at = find(S.lead, key, LL, blk_leader_hash<LL>(key));
                in = at != kNone && (S.lead[at] & kBlkMark);
            }
        }
        uint32_t total;
        const uint32_t before = blk_scan(in ? 1u : 0u, S.red, &total);
        if (in) S.pslot[m + before] = (uint16_t)k;                // the pairs' list is not needed any more
        m += total;
    }
    __syncthreads();
    uint32_t out = 0;
    for (uint32_t i = warp; i < n_list; i += kBlkThreads / 32) {
        const uint32_t o = S.pl[i], lw = S.lead[S.lslot[o]];
        if (!(lw & kBlkMark)) continue;
        const uint32_t at = ((lw & ~kBlkMark) >> 16) - 1u;
        (void)crowded(o);
        uint32_t now = clock0;                                   // above every stored stamp; only their order matters here
        for (uint32_t k0 = 0; k0 < m; k0 += 32) {
            bool mine = k0 + lane < m;
            const uint32_t k = mine ? S.pslot[k0 + lane] : 0u;
#pragma unroll
            for (int j = 0; j < LL; ++j) mine = mine && S.tok[k + j] == S.tok[at + j];
            uint32_t ps = kNone;
            if (mine) {
                int32_t key[LL + FLX];
#pragma unroll
                for (int j = 0; j < LL + FLX; ++j) key[j] = j < w ? S.tok[k + j] : 0;
                ps = pair_of(key);
            }
            for (uint32_t todo = __ballot_sync(CB_FULL, mine); todo; todo &= todo - 1u) {
                const uint32_t x = __shfl_sync(CB_FULL, ps, __ffs(todo) - 1);
                ++now;
                bool hit = false;
                uint32_t oldest = kNone;
#pragma unroll
                for (int c = 0; c < CH; ++c) {
                    if (id[c] == x && st[c]) { st[c] = now; hit = true; }
                    if (c * 32 + lane < FC) oldest = min(oldest, st[c]);
                }
                if (__any_sync(CB_FULL, hit)) continue;
                // a free place has stamp 0 and there may be several; stamps in use are unique
                const uint32_t g = __reduce_min_sync(CB_FULL, oldest);
                out += g ? 1u : 0u;
                if (lane == __ffs(__ballot_sync(CB_FULL, oldest == g)) - 1) {
                    bool open = true;
#pragma unroll
                    for (int c = 0; c < CH; ++c)
                        if (open && c * 32 + lane < FC && st[c] == g) { st[c] = now; id[c] = x; open = false; }
                }
            }
        }
    }
    __syncthreads();                                             // the entries have been read
    return out;
}

// Parts of a run of n windows where a part is to have 1 / inv of them: no more than kBlkPart expected in one.
__device__ __forceinline__ uint32_t blk_parts(uint32_t n, float inv) {
    return n == 0u ? 0u : max((uint32_t)ceilf((float)n * inv), (n + kBlkPart - 1u) / kBlkPart);
}
// One warp: about the smallest number of windows a part with which the parts of all sequences are no more than the blocks (a part too many
// is a second turn for some block, and the longest part is what the launch waits for: shares rounded down left 16 of 148 blocks without a
// part at batch 32 and gave 1,270 windows to one where 1,050 do).
// At least 32 windows a part: batch 13 of 294 to 450 tokens 18.5 us, 19.0 with 48 or 64; batch 13 of 344 to 688 18.8, 18.9 and 19.3; longer runs are
// cut by the number of blocks.
constexpr int kBlkLeast = 32;
constexpr int kBlkSearch = 8;                                   // sequences a lane
__device__ __forceinline__ float blk_share(const uint16_t* nwin, int B, uint32_t blocks, int lane) {
    uint32_t n[kBlkSearch], all = 0;
#pragma unroll
    for (int q = 0; q < kBlkSearch; ++q) { n[q] = q * 32 + lane < B ? nwin[q * 32 + lane] : 0u; all += n[q]; }
    all = __reduce_add_sync(CB_FULL, all);
    float share = fmaxf((float)all / ((float)blocks - 0.5f * (float)B), (float)kBlkLeast), inv = 1.f / share;   // rounding up adds half a part a sequence
    for (int k = 0; k < 16; ++k) {
        uint32_t parts = 0;
#pragma unroll
        for (int q = 0; q < kBlkSearch; ++q) if (q * 32 < B) parts += blk_parts(n[q], inv);
        parts = __reduce_add_sync(CB_FULL, parts);
        if (parts <= blocks) break;
        share += share * (float)(parts - blocks) / (float)blocks + 1.f;
        inv = 1.f / share;
    }
    return inv;
}

// alone: no other kernel follows, so that no run may be longer than kBlkRun windows.  COUNT_ALL: every follower that the windows displace
// one after the other is counted, also those that the run itself brought (else those displaced from the lists as they were).
// LL: the leader's tokens, FLX: a bound of the follower's (4 or 8), so that the loops over a window's tokens are straight code.
template <int LL, int FLX, bool COUNT_ALL>
__global__ void __launch_bounds__(kBlkThreads, 1) cb_update_bulk_block_kernel(CbTables t, int B, const int32_t* __restrict__ tokens, int64_t row_stride,
                                                                           const int32_t* __restrict__ n_old, const int32_t* __restrict__ n_new,
                                                                           bool alone, uint32_t* status, unsigned long long* counters) {
    extern __shared__ __align__(16) unsigned char blk_smem[];
    BlkSmem& S = *reinterpret_cast<BlkSmem*>(blk_smem);
    auto clear_tables = [&] {
        uint4* z = reinterpret_cast<uint4*>(S.pair);            // pair, lead and cur lie behind one another
        for (int i = threadIdx.x; i < 3 * kBlkSlots / 4; i += kBlkThreads) z[i] = make_uint4(0u, 0u, 0u, 0u);
    };
    clear_tables();                                             // for the first part, while the kernels before this one end
    CB_PDL_ENTRY();
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int w = LL + t.FL;
    {
        // the parts of all sequences
        uint32_t nwin = 0, parts = 0;
        if (tid < B) {
            const uint2 h = *reinterpret_cast<const uint2*>(cb_seq(t, tid).hdr);
            const int first = max(0, n_old[tid] - w + 1);
            nwin = (uint32_t)max(0, n_new[tid] - w + 1 - first);
            if (nwin > (uint32_t)kBlkRun) {                     // left to the kernels after this one, or longer than its row
                nwin = 0;
                if (alone && blockIdx.x == 0) atomicCAS(status, 0u, (uint32_t)CB_ERR_INVALID_ARG);
            }
            if (!cb_dbg_in(h.y, (long long)t.LC + 1, t.dbg_status)) nwin = 0;
            S.nwin[tid] = (uint16_t)nwin; S.first[tid] = first; S.clock[tid] = h.x; S.count[tid] = h.y;
        }
        float inv = 1.f / (float)kBlkPart;
        if ((uint32_t)B < gridDim.x && B <= 32 * kBlkSearch) {
            __syncthreads();
            if (warp == 0) { const float x = blk_share(S.nwin, B, gridDim.x, lane); if (lane == 0) S.inv = x; }
            __syncthreads();
            inv = S.inv;
        }
        const uint32_t mine = blk_parts(nwin, inv);
        const uint32_t before = blk_scan(mine, S.red, &parts);
        if (tid < B) S.pre[tid] = before;
        if (tid == 0) { S.pre[B] = parts; S.total = parts; }
    }
    __syncthreads();
    const uint32_t n_parts = S.total;
    TblCounters cnt = {0, 0, 0, 0};
    auto sequence_of = [&](uint32_t u) {                        // the last sequence whose parts begin at or before u
        int b = 0;
        for (int hi = B - 1; b < hi;) {
            const int mid = (b + hi + 1) >> 1;
            if (S.pre[mid] <= u) b = mid; else hi = mid - 1;
        }
        return b;
    };
    auto reduced = [&](int b) { return S.nwin[b] >= 64u && (unsigned long long)S.count[b] + S.nwin[b] <= (unsigned long long)t.LC; };
    bool in_order = false;
    for (uint32_t u = blockIdx.x; u < n_parts; u += gridDim.x) {
        const int b = sequence_of(u);
        const uint32_t part = u - S.pre[b], np = S.pre[b + 1] - S.pre[b];
        const CbSeq s = cb_seq(t, b);
        const uint32_t clock0 = S.clock[b], count0 = S.count[b], nwin = S.nwin[b];
        const int first = S.first[b];
        const int32_t* row = tokens + (size_t)b * row_stride;
        if (!reduced(b)) {
            in_order = in_order || part == 0u;
            continue;
        }
        {
            // ---- the run's tokens
            {
                if (u != blockIdx.x) clear_tables();
                // all of a thread's loads at once (one after the other they were 3.6 k cycles)
                auto fetch = [&](auto loads) {
                    constexpr int U = decltype(loads)::value;
                    const uint32_t len = nwin + (uint32_t)w - 1u;
                    int32_t x[U];
#pragma unroll
                    for (int q = 0; q < U; ++q) x[q] = (uint32_t)(q * kBlkThreads + tid) < len ? row[first + q * kBlkThreads + tid] : 0;
#pragma unroll
                    for (int q = 0; q < U; ++q) if ((uint32_t)(q * kBlkThreads + tid) < len) S.tok[q * kBlkThreads + tid] = x[q];
                };
                constexpr int kMost = (kBlkRun + CB_MAX_LL + CB_MAX_FL + kBlkThreads - 1) / kBlkThreads;
                if (nwin + (uint32_t)w <= 2u * kBlkThreads) fetch(std::integral_constant<int, 2>{});
                else fetch(std::integral_constant<int, kMost>{});
                if (tid == 0) { S.n_multi = 0u; S.n_own = 0u; S.n_lead = 0u; S.n_pair = 0u; S.n_fresh = 0u; S.n_list = 0u; }
            }
            __syncthreads();
            // ---- the part's windows are listed first (in `group`), so that the claims below run with full warps
            auto leader_hash = [&](uint32_t k) {
                int32_t k4[4] = {0, 0, 0, 0};
#pragma unroll
                for (int j = 0; j < LL; ++j) k4[j] = S.tok[k + j];
                return cb_hash4(k4[0], k4[1], k4[2], k4[3], LL);
            };
            // (One atomic a warp, with the votes of all its rounds unrolled into registers, gains 1% on runs of some thousand windows and costs a run of
            // 300 a twentieth: code that it jumps over, 13 against 14 us.)
            for (uint32_t k0 = warp * 32; k0 < nwin; k0 += kBlkThreads) {
                const uint32_t k = k0 + lane;
                uint32_t x = 0x85EBCA6Bu;
#pragma unroll
                for (int j = 0; j < LL; ++j) { x = (x ^ (uint32_t)S.tok[k + j]) * 0x9E3779B1u; x ^= x >> 16; }
                const bool own = k < nwin && __umulhi(x * 0xC2B2AE35u, np) == part;
                const uint32_t m = __ballot_sync(CB_FULL, own);
                uint32_t at = 0;
                if (m && lane == 0) at = atomicAdd(&S.n_own, (uint32_t)__popc(m));
                at = __shfl_sync(CB_FULL, at, 0) + __popc(m & ((1u << lane) - 1u));
                if (own) S.group[at] = (uint16_t)k;
            }
            __syncthreads();
            const uint32_t n_own = S.n_own;
            // ---- the part's windows: leader and pair are found or claimed, their last window raised
            for (uint32_t i0 = warp * 32; i0 < n_own; i0 += kBlkThreads) {
                const uint32_t i = i0 + lane;
                bool new_l = false, new_p = false;
                uint32_t ls = 0, ps = 0;
                if (i < n_own) {
                    const uint32_t k = S.group[i];
                    int32_t lk[LL], wk[LL + FLX];
#pragma unroll
                    for (int j = 0; j < LL + FLX; ++j) wk[j] = j < w ? S.tok[k + j] : 0;
#pragma unroll
                    for (int j = 0; j < LL; ++j) lk[j] = wk[j];
                    const uint32_t x = blk_leader_hash<LL>(wk);
                    ls = blk_slot<LL>(S.lead, S.tok, lk, LL, x, k, &new_l);
                    ps = blk_slot<LL + FLX>(S.pair, S.tok, wk, w, blk_pair_hash<LL>(x, wk, w), k, &new_p);
                    if (new_p) { S.pl[ps] = (uint16_t)ls; atomicAdd(&S.cur[ls], 1u); }
                }
                // what is new goes into the lists
                const uint32_t ml = __ballot_sync(CB_FULL, new_l), mp = __ballot_sync(CB_FULL, new_p), below = (1u << lane) - 1u;
                uint32_t at = 0;
                if (lane == 0) at = atomicAdd(&S.n_lead, (uint32_t)__popc(ml));
                if (lane == 1) at = atomicAdd(&S.n_pair, (uint32_t)__popc(mp));
                const uint32_t al = __shfl_sync(CB_FULL, at, 0), ap = __shfl_sync(CB_FULL, at, 1);
                if (new_l) S.lslot[al + __popc(ml & below)] = (uint16_t)ls;
                if (new_p) S.pslot[ap + __popc(mp & below)] = (uint16_t)ps;
            }
            __syncthreads();
            // ---- every leader takes a range of the pairs
            const uint32_t nl = S.n_lead, n_pair = S.n_pair;
            // the ids of new leaders; where all are new, under way while the pairs are grouped
            uint32_t got = 0;
            if (tid == 0 && count0 == 0u && nl) got = atomicAdd(&s.hdr[2], nl);
            for (uint32_t o0 = 0, g0 = 0; o0 < nl; o0 += kBlkThreads) {
                const uint32_t o = o0 + tid, ls = o < nl ? S.lslot[o] : 0u, c = o < nl ? S.cur[ls] : 0u;
                uint32_t tot;
                const uint32_t g = g0 + blk_scan(c, S.red, &tot);
                if (o < nl) { S.gbase[o] = (uint16_t)g; S.cur[ls] = g; }
                g0 += tot;
            }
            if (tid == 0) S.gbase[nl] = (uint16_t)n_pair;
            __syncthreads();
            for (uint32_t i = tid; i < n_pair; i += kBlkThreads) {
                const uint32_t ps = S.pslot[i];
                S.group[atomicAdd(&S.cur[S.pl[ps]], 1u)] = (uint16_t)ps;
            }
            __syncthreads();
            // ---- which leaders are stored already: eight lanes per leader read its bucket.  Entries of other parts of this run are
            // not looked at (their ids begin at count0).  A table without leaders has nothing to find.
            const int sub = lane & 7, oct = lane >> 3;
            if (count0 > 0u) {
                const uint32_t nb = t.nslots >> 5;
                for (uint32_t o0 = warp * 4; o0 < nl; o0 += kBlkThreads / 8) {
                    const uint32_t o = o0 + oct;
                    bool open = o < nl;
                    uint32_t kpos = 0, tag = 0, bucket = 0, found = 0;
                    if (open) {
                        kpos = (S.lead[S.lslot[o]] >> 16) - 1u;
                        const uint64_t h = leader_hash(kpos);
                        tag = cb_hash_tag(h);
                        bucket = cb_hash_bucket(h, t.nslots);
                    }
                    for (uint32_t p = 0; p < nb && __any_sync(CB_FULL, open); ++p) {
                        bool empty = false;
                        if (open) {
                            const uint4 x = __ldcg(reinterpret_cast<const uint4*>(s.index + (size_t)bucket * 32) + sub);
                            const uint32_t xs[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
                            for (int q = 0; q < 4; ++q) {
                                empty = empty || xs[q] == CB_IDX_EMPTY;
                                const uint32_t eid = xs[q] & CB_EID_MASK;
                                if (xs[q] == CB_IDX_EMPTY || xs[q] == CB_IDX_TOMB || (xs[q] >> CB_EID_BITS) != tag) continue;
                                if (!cb_dbg_in(eid, t.LC, t.dbg_status) || eid >= count0) continue;   // (from count0 on: a leader of another part)
                                bool eq = true;
                                for (int j = 0; j < LL; ++j) eq = eq && (int32_t)__ldcg(&s.entries[(size_t)eid * t.E + j]) == S.tok[kpos + j];
                                if (eq) found = eid + 1u;
                            }
                        }
#pragma unroll
                        for (int m = 1; m < 8; m <<= 1) found = max(found, __shfl_xor_sync(CB_FULL, found, m));
                        const uint32_t em = __ballot_sync(CB_FULL, empty);
                        if (open) cnt.maxprobe = max(cnt.maxprobe, p + 1u);
                        if (found || ((em >> (oct * 8)) & 0xFFu)) open = false;
                        bucket = (bucket + 1) & (nb - 1);
                    }
                    const bool fresh = o < nl && sub == 0 && found == 0u;
                    const uint32_t fm = __ballot_sync(CB_FULL, fresh);
                    uint32_t at = 0;
                    if (fm && lane == 0) at = atomicAdd(&S.n_fresh, (uint32_t)__popc(fm));
                    at = __shfl_sync(CB_FULL, at, 0) + __popc(fm & ((1u << lane) - 1u));
                    if (o < nl && sub == 0) S.cur[o] = found ? found : kBlkFresh | at;
                }
                __syncthreads();
            }
            if (tid == 0) {
                if (count0 > 0u && S.n_fresh) got = atomicAdd(&s.hdr[2], S.n_fresh);
                S.base = count0 + got;
            }
            // (the hash of this thread's first leader, meanwhile)
            const uint64_t mine_h = (uint32_t)tid < nl ? leader_hash((S.lead[S.lslot[tid]] >> 16) - 1u) : 0ull;
            __syncthreads();
            const uint32_t base = S.base;
            // entry id of leader o: the plan excludes that ids run out
            auto entry_of = [&](uint32_t o, bool* fresh) {
                const uint32_t x = count0 > 0u ? S.cur[o] : kBlkFresh | o;
                *fresh = (x & kBlkFresh) != 0u;
                return *fresh ? base + (x & ~kBlkFresh) : x - 1u;
            };
            // ---- publication: each new leader takes a free slot of the first bucket that has one.  Nobody follows the word before this
            // launch is over (the look-up above passes over ids from count0 on), so it may go out before the entry is written, and
            // the entries are written while the first attempts are under way.
            struct Claim { uint64_t h; uint32_t word, tries; bool open; };
            auto claim_of = [&](uint32_t o, uint64_t h) {
                Claim c = {0, 0, 0, false};
                if (o < nl) {
                    const uint32_t eid = entry_of(o, &c.open);
                    c.open = c.open && eid < (uint32_t)t.LC;
                    c.h = h;
                    c.word = (cb_hash_tag(c.h) << CB_EID_BITS) | eid;
                }
                return c;
            };
            auto attempt = [&](const Claim& c) {
                const uint32_t nb = t.nslots >> 5, bucket = (cb_hash_bucket(c.h, t.nslots) + (c.tries >> 5)) & (nb - 1);
                return &s.index[bucket * 32u + (((uint32_t)(c.h >> 20) + c.tries) & 31u)];
            };
            Claim mine = claim_of((uint32_t)tid, mine_h);
            uint32_t mine_old = CB_IDX_EMPTY;
            if (mine.open) mine_old = atomicCAS(attempt(mine), CB_IDX_EMPTY, mine.word);
            auto finish = [&](Claim& c, uint32_t old) {              // old: what the first attempt met
                for (;;) {
                    if (old == CB_IDX_TOMB) old = atomicCAS(attempt(c), CB_IDX_TOMB, c.word) == CB_IDX_TOMB ? CB_IDX_EMPTY : 1u;
                    if (old == CB_IDX_EMPTY) break;
                    if (++c.tries == t.nslots) { atomicCAS(status, 0u, (uint32_t)CB_ERR_PROBE_LIMIT); break; }
                    old = atomicCAS(attempt(c), CB_IDX_EMPTY, c.word);
                }
                cnt.maxprobe = max(cnt.maxprobe, (c.tries >> 5) + 1u);
            };
            // ---- entries, 16 bytes at a time: key, stamps (0: free), tokens of the followers that there are; zeros behind them up to 16
            // bytes.  A new leader that has room for its followers is written by a team of lanes, the others are listed.
            const uint32_t fl_inv = 65536u / (uint32_t)t.FL + 1u;          // x * fl_inv >> 16 = x / FL for x < 8,192
            auto team_of = [](uint32_t n) { return n > kBlkThreads / 2 ? 0 : n > kBlkThreads / 4 ? 1 : n > kBlkThreads / 8 ? 2 : 3; };   // log2 of its lanes
            auto write_entry = [&](uint32_t o, uint32_t eid, int lg) {
                if (eid >= (uint32_t)t.LC) return;
                const uint32_t lw = S.lead[S.lslot[o]], kpos = (lw >> 16) - 1u, g = S.gbase[o], n = S.gbase[o + 1] - g, team = (uint32_t)tid & ((1u << lg) - 1u);
                uint32_t* e = s.entries + (size_t)eid * t.E;
                if (team == 0u) s.lstamp[eid] = clock0 + (lw & 0xFFFFu);
                // (most leaders have one follower, which is looked up once)
                const uint32_t end = (uint32_t)(LL + t.FC) + n * (uint32_t)t.FL, pw0 = S.pair[S.group[g]];
                for (uint32_t q0 = 4u * team; q0 < end; q0 += 4u << lg) {
                    uint32_t v[4];
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const int f = (int)q0 + j - LL, x = f - t.FC;       // follower of a stamp, place among the followers' tokens
                        const uint32_t fi = x >= 0 ? ((uint32_t)x * fl_inv) >> 16 : (uint32_t)max(f, 0);
                        uint32_t pw = pw0;
                        if (fi != 0u) pw = fi < n ? S.pair[S.group[g + fi]] : 0u;
                        const uint32_t at = f < 0 ? kpos + q0 + j : (pw >> 16) + (uint32_t)(LL - 1 + x) - fi * (uint32_t)t.FL;
                        v[j] = pw ? clock0 + (pw & 0xFFFFu) : 0u;
                        if (f < 0 || (x >= 0 && pw)) v[j] = (uint32_t)S.tok[at];
                    }
                    *reinterpret_cast<uint4*>(e + q0) = make_uint4(v[0], v[1], v[2], v[3]);
                }
            };
            if (nl > kBlkThreads / 2) {
                // A thread to a leader: those with one follower, as most are, are their first window's tokens and one stamp and need no look at
                // the pairs; the few with more come after them (all in one loop: 8.1 k cycles, so 6).  Shorter lists go to teams as they are:
                // a second loop and its barrier cost a part of 60 leaders more than it gains.
                for (uint32_t o = (uint32_t)tid; o < nl; o += kBlkThreads) {
                    const uint32_t lw = S.lead[S.lslot[o]], kpos = (lw >> 16) - 1u, n = S.gbase[o + 1] - S.gbase[o];
                    bool fresh;
                    const uint32_t eid = entry_of(o, &fresh);
                    if (!fresh || n > (uint32_t)t.FC) { S.pl[atomicAdd(&S.n_list, 1u)] = (uint16_t)o; continue; }
                    if (n > 1u) { S.pslot[atomicAdd(&S.n_multi, 1u)] = (uint16_t)o; continue; }       // the pairs' list is not needed any more
                    if (eid >= (uint32_t)t.LC) continue;
                    uint32_t* e = s.entries + (size_t)eid * t.E;
                    const uint32_t stamp = clock0 + (lw & 0xFFFFu);
                    s.lstamp[eid] = stamp;
                    for (int q0 = 0; q0 < LL + t.FC + t.FL; q0 += 4) {
                        uint32_t v[4];
#pragma unroll
                        for (int j = 0; j < 4; ++j) {
                            const int x = q0 + j, y = x < LL ? x : x - t.FC;    // its place among the window's tokens
                            v[j] = (x < LL || x >= LL + t.FC) && y < w ? (uint32_t)S.tok[kpos + y] : (x == LL ? stamp : 0u);
                        }
                        *reinterpret_cast<uint4*>(e + q0) = make_uint4(v[0], v[1], v[2], v[3]);
                    }
                }
                __syncthreads();
                const int lg = team_of(S.n_multi);
                for (uint32_t i = (uint32_t)tid >> lg; i < S.n_multi; i += (uint32_t)kBlkThreads >> lg) {
                    bool fresh;
                    write_entry(S.pslot[i], entry_of(S.pslot[i], &fresh), lg);
                }
            } else {
                const int lg = team_of(nl);
                for (uint32_t o = (uint32_t)tid >> lg; o < nl; o += (uint32_t)kBlkThreads >> lg) {
                    bool fresh;
                    const uint32_t eid = entry_of(o, &fresh);
                    if (fresh && S.gbase[o + 1] - S.gbase[o] <= (uint32_t)t.FC) write_entry(o, eid, lg);
                    else if (((uint32_t)tid & ((1u << lg) - 1u)) == 0u) S.pl[atomicAdd(&S.n_list, 1u)] = (uint16_t)o;
                }
            }
            __syncthreads();
            // ---- the listed ones by a warp each
            const uint32_t n_list = S.n_list;
            uint32_t displaced = cnt.fevict;
            if (COUNT_ALL && n_list)
                displaced += t.FC <= 32 ? blk_evictions<LL, FLX, 1>(S, s.entries, t.E, t.FL, t.FC, count0, clock0, nwin, part, np)
                                        : blk_evictions<LL, FLX, CB_MAX_FC / 32>(S, s.entries, t.E, t.FL, t.FC, count0, clock0, nwin, part, np);
            for (uint32_t i = warp; i < n_list; i += kBlkThreads / 32) {
                const uint32_t o = S.pl[i], lw = S.lead[S.lslot[o]] & ~kBlkMark, kpos = (lw >> 16) - 1u, g = S.gbase[o], n = S.gbase[o + 1] - g;
                bool fresh;
                const uint32_t eid = entry_of(o, &fresh);
                if (eid >= (uint32_t)t.LC) continue;
                uint32_t* e = s.entries + (size_t)eid * t.E;
                if (lane == 0) s.lstamp[eid] = clock0 + (lw & 0xFFFFu);
                if (fresh && lane < LL) e[lane] = (uint32_t)S.tok[kpos + lane];   // and every follower place below (n > FC)
                // with more than FC distinct followers only the FC latest count: the largest thr with FC pairs at or above it
                uint32_t thr = 0;
                if (n > (uint32_t)t.FC && n <= 32u) {
                    const uint32_t last = (uint32_t)lane < n ? S.pair[S.group[g + lane]] & 0xFFFFu : 0u;
                    int later = 0;
                    for (uint32_t j = 0; j < n; ++j) later += __shfl_sync(CB_FULL, last, j) > last ? 1 : 0;
                    thr = __reduce_max_sync(CB_FULL, (uint32_t)lane < n && later == t.FC - 1 ? last : 0u);
                } else if (n > (uint32_t)t.FC) {
                    uint32_t top = 0;
                    for (uint32_t j = lane; j < n; j += 32) top = max(top, S.pair[S.group[g + j]] & 0xFFFFu);
                    uint32_t lo = 1, hi = __reduce_max_sync(CB_FULL, top);
                    if (t.FC <= 32) {
                        // the FC-th largest of the lanes' maxima is reached by FC pairs
                        uint32_t rest = top;
                        for (int r = 1; r < t.FC; ++r) {
                            const uint32_t m = __reduce_max_sync(CB_FULL, rest);
                            if (rest == m) rest = 0u;           // last windows of different pairs differ
                        }
                        lo = max(lo, __reduce_max_sync(CB_FULL, rest));
                    }
                    while (lo < hi) {
                        const uint32_t mid = lo + (hi - lo + 1u) / 2u;
                        uint32_t c = 0;
                        for (uint32_t j = lane; j < n; j += 32) c += (S.pair[S.group[g + j]] & 0xFFFFu) >= mid ? 1u : 0u;
                        c = __reduce_add_sync(CB_FULL, c);
                        if (c >= (uint32_t)t.FC) lo = mid; else hi = mid - 1u;
                    }
                    thr = lo;
                }
                uint32_t placed = 0;
                for (uint32_t j0 = 0; j0 < n; j0 += 32) {
                    const uint32_t j = j0 + lane, x = j < n ? S.pair[S.group[g + j]] : 0u;
                    const uint32_t keep = __ballot_sync(CB_FULL, j < n && (x & 0xFFFFu) >= thr);
                    if (fresh) {
                        const uint32_t place = placed + __popc(keep & ((1u << lane) - 1u));
                        if (((keep >> lane) & 1u) && place < (uint32_t)t.FC) {
                            for (int f = 0; f < t.FL; ++f) e[LL + t.FC + place * t.FL + f] = (uint32_t)S.tok[(x >> 16) - 1u + LL + f];
                            e[LL + place] = clock0 + (x & 0xFFFFu);
                        }
                        placed += __popc(keep);
                    } else {
                        for (uint32_t k = keep; k; k &= k - 1) {
                            const uint32_t y = __shfl_sync(CB_FULL, x, __ffs(k) - 1);
                            const int32_t myfol = lane < t.FL ? S.tok[(y >> 16) - 1u + LL + lane] : 0;
                            tbl_put_follower(t, e, myfol, clock0 + (y & 0xFFFFu), lane, cnt);
                            __syncwarp();
                        }
                    }
                }
            }
            if (COUNT_ALL) cnt.fevict = displaced;
            // ---- the rest of the publication
            if (mine.open) finish(mine, mine_old);
            for (uint32_t o = tid + kBlkThreads; o < nl; o += kBlkThreads) {
                Claim c = claim_of(o, leader_hash(((S.lead[S.lslot[o]] & ~kBlkMark) >> 16) - 1u));
                if (c.open) finish(c, atomicCAS(attempt(c), CB_IDX_EMPTY, c.word));
            }
        }
        // ---- the last block of the sequence folds the run into its header
        __syncthreads();
        if (tid == 0) {
            if (add_acq_rel(&s.hdr[3], 1u) == np - 1u) {
                s.hdr[1] = count0 + __ldcg(&s.hdr[2]);
                s.hdr[0] = clock0 + nwin;
                s.hdr[2] = 0u;
                s.hdr[3] = 0u;
                atomicAdd(&counters[CB_CNT_INSERTS], (unsigned long long)nwin);
            }
        }
    }
    if (alone && in_order) {
        uint32_t k = 0;
        for (uint32_t u = blockIdx.x; u < n_parts; u += gridDim.x) {
            const int b = sequence_of(u);
            if (u != S.pre[b] || reduced(b) || (k++ & 31u) != (uint32_t)warp) continue;
            const CbSeq s = cb_seq(t, b);
            const int32_t* row = tokens + (size_t)b * row_stride;
            uint32_t clock = S.clock[b], count = S.count[b];
            for (int i = S.first[b], end = i + (int)S.nwin[b]; i < end; ++i) {
                const int32_t mykey = lane < LL ? row[i + lane] : 0;
                const int32_t myfol = lane < t.FL ? row[i + LL + lane] : 0;
                if (t.FC <= 32) tbl_insert<1>(t, s, mykey, myfol, clock, count, lane, status, cnt);
                else tbl_insert<0>(t, s, mykey, myfol, clock, count, lane, status, cnt);
            }
            if (lane == 0) { s.hdr[0] = clock; s.hdr[1] = count; }
        }
    }
    const uint32_t mp = __reduce_max_sync(CB_FULL, cnt.maxprobe);
    if (lane == 0) {
        if (cnt.inserts) atomicAdd(&counters[CB_CNT_INSERTS], (unsigned long long)cnt.inserts);
        if (cnt.levict) atomicAdd(&counters[CB_CNT_LEADER_EVICTIONS], (unsigned long long)cnt.levict);
        if (cnt.fevict) atomicAdd(&counters[CB_CNT_FOLLOWER_EVICTIONS], (unsigned long long)cnt.fevict);
        if (mp) atomicMax(&counters[CB_CNT_MAX_PROBE], (unsigned long long)mp);
    }
}

}  // namespace

// Per-sequence LRU cache table kernels: sliding-window update and batched draft-tree expansion.
//
// Every table operation is executed by one warp acting as a unit: the 32 lanes probe the 32 slots of an
// index bucket with one coalesced load, compare the FC followers of an entry in parallel, and scan the
// dense stamp array for the least recently used leader.  Recency is a per-sequence operation counter
// ("clock"); a leader or follower stamp is the clock value of the operation that last touched it.
#include <algorithm>
#include <mutex>

#include "cb_accept_dev.cuh"

namespace {

struct Probe {
    int eid;             // entry id, -1 absent, -2 probe limit
    uint32_t slot;       // index slot holding the entry (when found)
    uint32_t free_slot;  // first reusable slot on the probe path (when absent), 0xFFFFFFFF if none seen
    uint32_t probes;     // buckets visited
};

// Warp-wide lookup of a leader. mykey = key[lane] for lane < LL (0 otherwise), identical call in all lanes.
// SHARED: other SMs publish index words and entries while this warp probes (bulk update), so index and key are read
// through to L2 instead of from an L1 line that may be stale.
// FETCH (tables with FC <= 32, so that lane l owns follower l alone): the follower's stamp and tokens are loaded together
// with the key when an index word's tag matches, which saves the callers two dependent memory round trips.
// FETCH == 2 (larger FC): the stamps of all the lane's followers come with the key (one round trip saved); the tokens are
// loaded when they are known to be needed.
struct EntryRegs {
    uint32_t fs;
    int32_t tok[CB_MAX_FL];
    uint32_t fs4[CB_MAX_FC / 32];
};
template <bool SHARED = false, int FETCH = 0>
__device__ __forceinline__ Probe tbl_find(const CbTables& t, const CbSeq& s, int32_t mykey, uint64_t h, int lane, EntryRegs* er = nullptr) {
    Probe r;
    r.eid = -2; r.slot = 0; r.free_slot = 0xFFFFFFFFu; r.probes = 0;
    const uint32_t nb = t.nslots >> 5, tag = cb_hash_tag(h);
    uint32_t bucket = cb_hash_bucket(h, t.nslots);
    for (uint32_t p = 0; p < nb; ++p) {
        r.probes = p + 1;
        const uint32_t w = SHARED ? __ldcg(&s.index[bucket * 32 + lane]) : s.index[bucket * 32 + lane];
        uint32_t cand = __ballot_sync(CB_FULL, w != CB_IDX_EMPTY && w != CB_IDX_TOMB && (w >> CB_EID_BITS) == tag);
        while (cand) {
            const int l = __ffs(cand) - 1;
            cand &= cand - 1;
            const uint32_t eid = __shfl_sync(CB_FULL, w, l) & CB_EID_MASK;
            if (!cb_dbg_in(eid, t.LC, t.dbg_status)) continue;                // an index word naming an entry that cannot exist
            bool eq = true;
            if (FETCH == 2) {
                const uint32_t* e = s.entries + (size_t)eid * t.E;
                const uint32_t kv = lane < t.LL ? e[lane] : 0u;
#pragma unroll
                for (int c = 0; c < CB_MAX_FC / 32; ++c) er->fs4[c] = (c * 32 + lane) < t.FC ? e[t.LL + c * 32 + lane] : 0u;
                if (lane < t.LL) eq = (int32_t)kv == mykey;
            } else if (FETCH == 1) {
                const uint32_t* e = s.entries + (size_t)eid * t.E;
                const bool mine = lane < t.FC;
                const uint32_t kv = lane < t.LL ? e[lane] : 0u;
                er->fs = mine ? e[t.LL + lane] : 0u;
#pragma unroll
                for (int j = 0; j < CB_MAX_FL; ++j) er->tok[j] = (mine && j < t.FL) ? (int32_t)e[t.LL + t.FC + lane * t.FL + j] : -1;
                if (lane < t.LL) eq = (int32_t)kv == mykey;
            } else if (lane < t.LL) {
                const uint32_t* kp = &s.entries[(size_t)eid * t.E + lane];
                eq = ((int32_t)(SHARED ? __ldcg(kp) : *kp) == mykey);
            }
            if (__all_sync(CB_FULL, eq)) { r.eid = (int)eid; r.slot = bucket * 32 + l; return r; }
        }
        const uint32_t fr = __ballot_sync(CB_FULL, w == CB_IDX_EMPTY || w == CB_IDX_TOMB);
        if (r.free_slot == 0xFFFFFFFFu && fr) r.free_slot = bucket * 32 + (__ffs(fr) - 1);
        if (__ballot_sync(CB_FULL, w == CB_IDX_EMPTY)) { r.eid = -1; return r; }
        bucket = (bucket + 1) & (nb - 1);
    }
    return r;
}

__device__ __forceinline__ uint64_t warp_hash(const CbTables& t, int32_t mykey) {
    const int32_t k0 = __shfl_sync(CB_FULL, mykey, 0), k1 = __shfl_sync(CB_FULL, mykey, 1),
                  k2 = __shfl_sync(CB_FULL, mykey, 2), k3 = __shfl_sync(CB_FULL, mykey, 3);
    return cb_hash4(k0, k1, k2, k3, t.LL);
}

// Removes the least recently used leader from the index and returns its entry id for reuse.
__device__ int tbl_evict_lru(const CbTables& t, const CbSeq& s, int lane, uint32_t* status) {
    uint32_t minv = 0xFFFFFFFFu;
    int mine = 0;
#pragma unroll 4
    for (int i = lane; i < t.LC; i += 32) {
        const uint32_t v = s.lstamp[i];
        if (v < minv) { minv = v; mine = i; }
    }
    const uint32_t g = __reduce_min_sync(CB_FULL, minv);
    const int wl = __ffs(__ballot_sync(CB_FULL, minv == g)) - 1;   // stamps are unique
    const int eid = __shfl_sync(CB_FULL, mine, wl);
    const int32_t vkey = lane < t.LL ? (int32_t)s.entries[(size_t)eid * t.E + lane] : 0;
    const uint64_t h = warp_hash(t, vkey);
    const uint32_t nb = t.nslots >> 5, word = (cb_hash_tag(h) << CB_EID_BITS) | (uint32_t)eid;
    uint32_t bucket = cb_hash_bucket(h, t.nslots);
    for (uint32_t p = 0; p < nb; ++p) {
        const uint32_t w = s.index[bucket * 32 + lane];
        const uint32_t hit = __ballot_sync(CB_FULL, w == word);
        const uint32_t empties = __ballot_sync(CB_FULL, w == CB_IDX_EMPTY);
        if (hit) {
            // A bucket that still has an empty slot is the end of every probe path through it, so the
            // slot can simply become empty again; otherwise later buckets may hold keys that probed
            // past this one and the slot must stay marked as deleted.
            if (lane == __ffs(hit) - 1) s.index[bucket * 32 + lane] = empties ? CB_IDX_EMPTY : CB_IDX_TOMB;
            __syncwarp();
            return eid;
        }
        if (empties) break;
        bucket = (bucket + 1) & (nb - 1);
    }
    if (lane == 0) atomicCAS(status, 0u, (uint32_t)CB_ERR_PROBE_LIMIT);   // index and entries disagree
    return eid;
}

struct TblCounters { uint32_t inserts, levict, fevict, maxprobe; };

// Follower list of an existing leader (Section 3.1): a stored copy of the follower is refreshed, otherwise the follower takes
// the lowest free place or replaces the least recently inserted one.  e = the leader's entry, c = this operation's stamp.
// The same with the follower's stamp and tokens already in registers (FC <= 32).
__device__ __forceinline__ void tbl_put_follower_regs(const CbTables& t, uint32_t* e, const EntryRegs& er, int32_t myfol, uint32_t c, int lane,
                                                      TblCounters& cnt) {
    const bool mine = lane < t.FC;
    bool match = mine && er.fs != 0u;
#pragma unroll
    for (int j = 0; j < CB_MAX_FL; ++j) {
        const int32_t fj = __shfl_sync(CB_FULL, myfol, j);
        if (j < t.FL) match = match && (er.tok[j] == fj);
    }
    const uint32_t mm = __ballot_sync(CB_FULL, match);
    if (mm) {
        if (t.refresh && lane == 0) e[t.LL + (__ffs(mm) - 1)] = c;
        return;
    }
    const uint32_t freem = __ballot_sync(CB_FULL, mine && er.fs == 0u);
    int tgt;
    if (freem) {
        tgt = __ffs(freem) - 1;
    } else {
        const uint32_t g = __reduce_min_sync(CB_FULL, mine ? er.fs : 0xFFFFFFFFu);
        tgt = __ffs(__ballot_sync(CB_FULL, mine && er.fs == g)) - 1;
        cnt.fevict++;
    }
    if (lane < t.FL) e[t.LL + t.FC + tgt * t.FL + lane] = (uint32_t)myfol;
    if (lane == 0) e[t.LL + tgt] = c;
}

template <bool PRE = false>
__device__ __forceinline__ void tbl_put_follower(const CbTables& t, uint32_t* e, int32_t myfol, uint32_t c, int lane, TblCounters& cnt,
                                                 const EntryRegs* er = nullptr) {
    // Lane l looks after followers l, l + 32, ...: one pass finds a stored copy of the follower, the lowest free place
    // and the least recently inserted follower.  PRE: the stamps came with the lookup; the first tokens of all of the lane's
    // followers are then read at once, and the others only of those that match so far (read follower by follower and token by
    // token they were a chain of 12 memory round trips with FC = 128, FL = 3).
    constexpr int CH = CB_MAX_FC / 32;
    const int32_t f0 = __shfl_sync(CB_FULL, myfol, 0);
    int32_t t0[CH];
#pragma unroll
    for (int ch = 0; ch < CH; ++ch) t0[ch] = PRE && er->fs4[ch] != 0u ? (int32_t)e[t.LL + t.FC + (ch * 32 + lane) * t.FL] : 0;
    int match_f = -1, free_f = -1, lru_f = -1;
    uint32_t lru_stamp = 0xFFFFFFFFu;
#pragma unroll
    for (int ch = 0; ch < CH; ++ch) {
        const int base = ch * 32;
        if (base >= t.FC || match_f >= 0) break;
        const int f = base + lane;
        const bool mine = f < t.FC;
        const uint32_t fs = PRE ? er->fs4[ch] : (mine ? e[t.LL + f] : 0u);
        bool match = mine && fs != 0u;
        if (PRE) match = match && t0[ch] == f0;
        if (!PRE || __any_sync(CB_FULL, match))
            for (int j = PRE ? 1 : 0; j < t.FL; ++j) {
                const int32_t fj = __shfl_sync(CB_FULL, myfol, j);
                if (match) match = ((int32_t)e[t.LL + t.FC + f * t.FL + j] == fj);
            }
        const uint32_t mm = __ballot_sync(CB_FULL, match);
        if (mm) { match_f = base + __ffs(mm) - 1; break; }
        const uint32_t freem = __ballot_sync(CB_FULL, mine && fs == 0u);
        if (free_f < 0 && freem) free_f = base + __ffs(freem) - 1;
        const uint32_t g = __reduce_min_sync(CB_FULL, (mine && fs != 0u) ? fs : 0xFFFFFFFFu);
        if (g < lru_stamp) { lru_stamp = g; lru_f = base + __ffs(__ballot_sync(CB_FULL, mine && fs == g)) - 1; }
    }
    if (match_f >= 0) {
        if (t.refresh && lane == 0) e[t.LL + match_f] = c;
    } else {
        int tgt = free_f;
        if (tgt < 0) { tgt = lru_f; cnt.fevict++; }
        if (lane < t.FL) e[t.LL + t.FC + tgt * t.FL + lane] = (uint32_t)myfol;
        if (lane == 0) e[t.LL + tgt] = c;
    }
}

// The two halves of an insertion once the lookup is done: a leader that is stored, a leader that takes entry eid and index slot
// `slot`.
template <int FETCH>
__device__ __forceinline__ void tbl_refresh_leader(const CbTables& t, const CbSeq& s, int eid, const EntryRegs& er, int32_t myfol, uint32_t c, int lane,
                                                   TblCounters& cnt) {
    uint32_t* e = s.entries + (size_t)eid * t.E;
    if (lane == 0) s.lstamp[eid] = c;
    if (FETCH == 1) tbl_put_follower_regs(t, e, er, myfol, c, lane, cnt);
    else if (FETCH == 2) tbl_put_follower<true>(t, e, myfol, c, lane, cnt, &er);
    else tbl_put_follower(t, e, myfol, c, lane, cnt);
}
__device__ __forceinline__ void tbl_new_leader(const CbTables& t, const CbSeq& s, int eid, uint32_t slot, int32_t mykey, int32_t myfol, uint64_t h, uint32_t c,
                                               int lane) {
    uint32_t* e = s.entries + (size_t)eid * t.E;
    if (lane < t.LL) e[lane] = (uint32_t)mykey;
    for (int f = lane; f < t.FC; f += 32) e[t.LL + f] = f == 0 ? c : 0u;
    if (lane < t.FL) e[t.LL + t.FC + lane] = (uint32_t)myfol;
    if (lane == 0) {
        s.lstamp[eid] = c;
        s.index[slot] = (cb_hash_tag(h) << CB_EID_BITS) | (uint32_t)eid;
    }
}

// One insertion (Section 3.1). mykey = leader[lane] (lane < LL), myfol = follower[lane] (lane < FL).
template <int FETCH = 0>
__device__ void tbl_insert(const CbTables& t, const CbSeq& s, int32_t mykey, int32_t myfol, uint32_t& clock,
                           uint32_t& count, int lane, uint32_t* status, TblCounters& cnt) {
    const uint32_t c = ++clock;
    cnt.inserts++;
    const uint64_t h = warp_hash(t, mykey);
    EntryRegs er;
    Probe pr = tbl_find<false, FETCH>(t, s, mykey, h, lane, &er);
    cnt.maxprobe = max(cnt.maxprobe, pr.probes);
    if (pr.eid >= 0) {
        tbl_refresh_leader<FETCH>(t, s, pr.eid, er, myfol, c, lane, cnt);
    } else if (pr.eid == -1) {
        int eid;
        if (count < (uint32_t)t.LC) {
            eid = (int)count++;
        } else {
            eid = tbl_evict_lru(t, s, lane, status);
            cnt.levict++;
            pr = tbl_find(t, s, mykey, h, lane);           // the eviction may have opened a nearer slot
        }
        if (pr.free_slot == 0xFFFFFFFFu) {
            if (lane == 0) atomicCAS(status, 0u, (uint32_t)CB_ERR_PROBE_LIMIT);
        } else {
            tbl_new_leader(t, s, eid, pr.free_slot, mykey, myfol, h, c, lane);
        }
    } else {
        if (lane == 0) atomicCAS(status, 0u, (uint32_t)CB_ERR_PROBE_LIMIT);
    }
    __syncwarp();
}

// One warp per sequence; windows are applied in increasing position.
template <int FETCH>
__device__ __forceinline__ void update_seq(const CbTables& t, int b, const int32_t* tokens, int64_t row_stride, int n0, int n1,
                                           int lane, uint32_t* status, unsigned long long* counters) {
    const CbSeq s = cb_seq(t, b);
    const int w = t.LL + t.FL;
    uint32_t clock = s.hdr[0], count = s.hdr[1];
    TblCounters cnt = {0, 0, 0, 0};
    const int32_t* row = tokens + (size_t)b * row_stride;
    for (int i = max(0, n0 - w + 1); i + w <= n1; ++i) {
        const int32_t mykey = lane < t.LL ? row[i + lane] : 0;
        const int32_t myfol = lane < t.FL ? row[i + t.LL + lane] : 0;
        tbl_insert<FETCH>(t, s, mykey, myfol, clock, count, lane, status, cnt);
    }
    if (lane == 0) {
        s.hdr[0] = clock; s.hdr[1] = count;
        if (cnt.inserts) atomicAdd(&counters[CB_CNT_INSERTS], (unsigned long long)cnt.inserts);
        if (cnt.levict) atomicAdd(&counters[CB_CNT_LEADER_EVICTIONS], (unsigned long long)cnt.levict);
        if (cnt.fevict) atomicAdd(&counters[CB_CNT_FOLLOWER_EVICTIONS], (unsigned long long)cnt.fevict);
        if (cnt.maxprobe) atomicMax(&counters[CB_CNT_MAX_PROBE], (unsigned long long)cnt.maxprobe);
    }
}

// The same by a whole CTA of eight warps, up to eight windows at a time, one per warp.  Inserted one after the other a window costs
// 2.5 k cycles (some 270 dependent instructions of one warp, two memory round trips among them): five windows were 12 k of
// the 17 k cycles that a sequence of batch 128 took for update and draft (21.1 us a call, 11.5 to 12.6 with the windows side by side).
// Windows with different leaders touch different entries, and their stamps follow from their positions, so as long as no leader
// can be evicted they may be applied side by side: stored leaders are refreshed; new ones take the next entries in the order of
// their windows, each the index slot its lookup found.  What is left goes to the first warp afterwards, in order, as in update_seq:
// a window whose leader an earlier window of the eight has, a new leader whose slot lies in the same bucket as an earlier new
// one's, a failed lookup.  When the eight could overflow the leader capacity, all of them do (an eviction looks at the stamps of
// the windows before it only).
// Meanwhile a warp without a window does idle(): it looks the tree's root up, so that the draft that follows finds the root's bucket and
// entry in L1 (a write by this CTA goes through that L1, so what it finds there is current; no other CTA writes this sequence's table).
constexpr int kUpdWarps = 8;
template <int FETCH, typename Tokens, typename Idle>
__device__ __forceinline__ void update_seq_cta(const CbTables& t, int b, const Tokens& row, int n0, int n1,
                                               int warp, int lane, uint32_t* status, unsigned long long* counters, Idle&& idle) {
    __shared__ unsigned long long sh_h[kUpdWarps];
    __shared__ uint32_t sh_state[kUpdWarps], sh_bucket[kUpdWarps], sh_count[2];
    const CbSeq s = cb_seq(t, b);
    const int w = t.LL + t.FL;
    uint32_t clock = s.hdr[0], count = s.hdr[1];
    TblCounters cnt = {0, 0, 0, 0};
    int flip = 0;
    const int n_all = n1 - w + 1 - max(0, n0 - w + 1);
    if (n_all > 0 && n_all < kUpdWarps && warp == kUpdWarps - 1) idle();
    for (int i0 = max(0, n0 - w + 1); i0 + w <= n1; i0 += kUpdWarps) {
        const int nb = min(kUpdWarps, n1 - w + 1 - i0), i = i0 + warp;
        const bool mine = warp < nb, together = count + (uint32_t)nb <= (uint32_t)t.LC;
        uint32_t later = (1u << nb) - 1u;                       // windows left to the first warp
        if (together) {
            int32_t mykey = 0, myfol = 0;
            uint64_t h = 0;
            EntryRegs er;
            Probe pr = {};
            if (mine) {
                if (lane < t.LL) mykey = row(i + lane);
                if (lane < t.FL) myfol = row(i + t.LL + lane);
                h = warp_hash(t, mykey);
                pr = tbl_find<false, FETCH>(t, s, mykey, h, lane, &er);
                if (lane == 0) {
                    sh_h[warp] = h;
                    sh_state[warp] = pr.eid >= 0 ? 0u : (pr.eid == -1 && pr.free_slot != 0xFFFFFFFFu ? 1u : 2u);   // stored, new, neither
                    sh_bucket[warp] = pr.free_slot >> 5;
                }
            }
            __syncthreads();
            // lane j looks at window j: every warp comes to the same masks (all lanes take part in every vote)
            const bool there = lane < nb;
            const uint32_t state = there ? sh_state[lane] : 2u;
            const unsigned long long hj = there ? sh_h[lane] : 0ull;
            // (seven comparisons each: __match_any_sync took 500 cycles for either of the two)
            bool same = false;
#pragma unroll
            for (int k = 0; k < kUpdWarps - 1; ++k) same = same || (k < lane && k < nb && sh_h[k] == hj);
            const bool seq = there && (same || state == 2u);
            const bool fresh = there && state == 1u && !seq;
            const uint32_t bj = fresh ? sh_bucket[lane] : 0x80000000u | (uint32_t)lane;
            bool beside = false;
#pragma unroll
            for (int k = 0; k < kUpdWarps - 1; ++k) beside = (__shfl_sync(CB_FULL, bj, k) == bj && k < lane) || beside;
            const bool clash = fresh && beside;
            later = __ballot_sync(CB_FULL, seq || clash);
            const uint32_t newm = __ballot_sync(CB_FULL, fresh && !clash);
            if (mine && !((later >> warp) & 1u)) {
                const uint32_t c = clock + (uint32_t)warp + 1u;
                cnt.maxprobe = max(cnt.maxprobe, pr.probes);
                if (pr.eid >= 0) tbl_refresh_leader<FETCH>(t, s, pr.eid, er, myfol, c, lane, cnt);
                else tbl_new_leader(t, s, (int)(count + __popc(newm & ((1u << warp) - 1u))), pr.free_slot, mykey, myfol, h, c, lane);
            }
            count += __popc(newm);
            __syncthreads();
        }
        if (later) {
            if (warp == 0) {
                uint32_t n = count;
                for (uint32_t m = later; m; m &= m - 1u) {
                    const int k = __ffs(m) - 1;
                    const int32_t mykey = lane < t.LL ? row(i0 + k + lane) : 0;
                    const int32_t myfol = lane < t.FL ? row(i0 + k + t.LL + lane) : 0;
                    uint32_t c = clock + (uint32_t)k;
                    tbl_insert<FETCH>(t, s, mykey, myfol, c, n, lane, status, cnt);
                }
                if (lane == 0) sh_count[flip] = n;
            }
            __syncthreads();
            count = sh_count[flip];                              // the next batch's goes into the other word
            flip ^= 1;
        }
        clock += (uint32_t)nb;
    }
    if (lane == 0) {
        const int nw = max(0, n_all);
        if (warp == 0) {
            s.hdr[0] = clock; s.hdr[1] = count;
            if (nw) atomicAdd(&counters[CB_CNT_INSERTS], (unsigned long long)nw);
            if (cnt.levict) atomicAdd(&counters[CB_CNT_LEADER_EVICTIONS], (unsigned long long)cnt.levict);
        }
        if (cnt.fevict) atomicAdd(&counters[CB_CNT_FOLLOWER_EVICTIONS], (unsigned long long)cnt.fevict);
        if (cnt.maxprobe) atomicMax(&counters[CB_CNT_MAX_PROBE], (unsigned long long)cnt.maxprobe);
    }
}

template <int FETCH>
__global__ void __launch_bounds__(128) cb_update_kernel(CbTables t, int B, const int32_t* __restrict__ tokens,
                                                        int64_t row_stride, const int32_t* __restrict__ n_old,
                                                        const int32_t* __restrict__ n_new, uint32_t* status,
                                                        unsigned long long* counters) {
    CB_PDL_ENTRY();
    const int lane = threadIdx.x & 31;
    const int b = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (b >= B) return;
    update_seq<FETCH>(t, b, tokens, row_stride, n_old[b], n_new[b], lane, status, counters);
}

// ---------------------------------------------------------------------------------------------------
// Bulk update (prompt initialisation and other long runs of new tokens): many warps per sequence.
//
// The result of a run of insertions depends on their order only within one leader (its recency and its follower list)
// and, across leaders, through leader eviction.  Stamps are a function of the window's position (the clock ticks once per
// window), so when no leader can be evicted during the run (leaders stored + windows <= LC) the windows may be dealt out
// to warps by a hash of their leader: every leader is handled by one warp, in increasing position, exactly as the
// sequential kernel would, and different leaders touch disjoint entries.  What the warps share is the leader counter
// (atomicAdd hands out entry ids) and the index, whose slots are claimed with atomicCAS; an entry is complete before its
// index word is published.  A plan kernel takes that decision once per sequence, before any warp changes the table;
// sequences that do not qualify (short runs, possible eviction) are done by their first warp alone, in order.
struct BulkPlan { uint32_t parallel, clock0, first, nwin; };   // parallel: 0 one warp in order, 1 warps by leader, 2 elsewhere (cb_bulk_block.cuh, cb_bulk_free.cuh)

// done: runs of up to that many windows that qualify are the block kernel's (cb_bulk_block.cuh), which comes after this one
__global__ void cb_bulk_plan_kernel(CbTables t, int B, const int32_t* __restrict__ n_old, const int32_t* __restrict__ n_new,
                                    BulkPlan* plan, int done) {
    CB_PDL_ENTRY();
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= B) return;
    const CbSeq s = cb_seq(t, b);
    const int w = t.LL + t.FL;
    const int first = max(0, n_old[b] - w + 1);
    const int nwin = max(0, n_new[b] - w + 1 - first);
    BulkPlan p;
    p.clock0 = s.hdr[0];
    p.first = (uint32_t)first;
    p.nwin = (uint32_t)nwin;
    p.parallel = (nwin >= 64 && (unsigned long long)s.hdr[1] + (unsigned long long)nwin <= (unsigned long long)t.LC) ? 1u : 0u;
    if (nwin <= done && p.parallel == 1u) p.parallel = 2u;
    if (p.parallel == 1u) s.hdr[0] = p.clock0 + (uint32_t)nwin;   // the clock after the run; the warps take stamps from positions
    plan[b] = p;
}

// One insertion of the parallel path: c is the operation's stamp; no leader is ever evicted here.  Returns the leader's
// entry id (-1 if the insertion failed).
__device__ int tbl_insert_shared(const CbTables& t, const CbSeq& s, int32_t mykey, int32_t myfol, uint32_t c, int lane,
                                 uint32_t* status, TblCounters& cnt) {
    cnt.inserts++;
    const uint64_t h = warp_hash(t, mykey);
    const uint32_t tagword = cb_hash_tag(h) << CB_EID_BITS;
    int eid = -1;
    for (int attempt = 0; attempt < 64; ++attempt) {            // a claim can lose its slot to another warp's leader: look again
        const Probe pr = tbl_find<true>(t, s, mykey, h, lane);
        cnt.maxprobe = max(cnt.maxprobe, pr.probes);
        if (pr.eid >= 0) {
            uint32_t* e = s.entries + (size_t)pr.eid * t.E;
            if (lane == 0) s.lstamp[pr.eid] = c;
            tbl_put_follower(t, e, myfol, c, lane, cnt);
            __syncwarp();
            return pr.eid;
        }
        if (pr.eid != -1 || pr.free_slot == 0xFFFFFFFFu) break;
        if (eid < 0) {
            // new leader: take an entry, fill it, then publish it
            uint32_t got = 0;
            if (lane == 0) got = atomicAdd(&s.hdr[1], 1u);
            got = __shfl_sync(CB_FULL, got, 0);
            if (got >= (uint32_t)t.LC) break;                  // excluded by the plan
            eid = (int)got;
            uint32_t* e = s.entries + (size_t)eid * t.E;
            if (lane < t.LL) e[lane] = (uint32_t)mykey;
            for (int f = lane; f < t.FC; f += 32) e[t.LL + f] = f == 0 ? c : 0u;
            if (lane < t.FL) e[t.LL + t.FC + lane] = (uint32_t)myfol;
            if (lane == 0) s.lstamp[eid] = c;
            __threadfence();
            __syncwarp();
        }
        uint32_t old = 0;
        if (lane == 0) old = atomicCAS(&s.index[pr.free_slot], CB_IDX_EMPTY, tagword | (uint32_t)eid);
        old = __shfl_sync(CB_FULL, old, 0);
        if (old == CB_IDX_EMPTY) return eid;
        if (old == CB_IDX_TOMB) {                              // a deleted slot is as good as an empty one
            if (lane == 0) old = atomicCAS(&s.index[pr.free_slot], CB_IDX_TOMB, tagword | (uint32_t)eid);
            old = __shfl_sync(CB_FULL, old, 0);
            if (old == CB_IDX_TOMB) return eid;
        }
    }
    if (lane == 0) atomicCAS(status, 0u, (uint32_t)CB_ERR_PROBE_LIMIT);
    return -1;
}

// The warp that owns a frequent leader meets it again and again (with unigram leaders a handful of tokens own a third of
// the windows), and every insertion into a leader that is in the table is a chain of four dependent memory round trips.  So
// every warp keeps the entries it touched last in shared memory (WAYS of them: key, follower stamps and tokens, leader
// stamp): an insertion into a kept entry is the same follower-list code running on the shared-memory copy, and the copy goes
// back to the table when its place is needed or the run ends.  No other warp touches these leaders during the run.
__global__ void __launch_bounds__(256) cb_update_bulk_kernel(CbTables t, int B, int WPS, int WAYS, const int32_t* __restrict__ tokens, int64_t row_stride,
                                                             const int32_t* __restrict__ n_old, const int32_t* __restrict__ n_new,
                                                             const BulkPlan* __restrict__ plan, uint32_t* status, unsigned long long* counters) {
    CB_PDL_ENTRY();
    extern __shared__ uint32_t bulk_smem[];
    const int lane = threadIdx.x & 31;
    // this warp's kept entries: WAYS x (E words of the entry, then entry id + 1 (0 = free), leader stamp, last use, unused)
    const uint32_t way_words = t.E + 4;
    uint32_t* ways = bulk_smem + (size_t)(threadIdx.x >> 5) * WAYS * way_words;
    for (int w = lane; w < WAYS; w += 32) ways[(size_t)w * way_words + t.E] = 0u;
    __syncwarp();
    uint32_t use_clock = 0;
    const int gw = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    const int b = gw / WPS, wi = gw % WPS;
    if (b >= B) return;
    const CbSeq s = cb_seq(t, b);
    const BulkPlan pl = plan[b];
    if (pl.parallel == 2u) return;                              // done by the block kernel or the order-free ones
    const int32_t* row = tokens + (size_t)b * row_stride;
    TblCounters cnt = {0, 0, 0, 0};
    if (!pl.parallel) {
        if (wi != 0) return;
        uint32_t clock = s.hdr[0], count = s.hdr[1];
        for (uint32_t k = 0; k < pl.nwin; ++k) {
            const int i = (int)(pl.first + k);
            const int32_t mykey = lane < t.LL ? row[i + lane] : 0;
            const int32_t myfol = lane < t.FL ? row[i + t.LL + lane] : 0;
            tbl_insert(t, s, mykey, myfol, clock, count, lane, status, cnt);
        }
        if (lane == 0) { s.hdr[0] = clock; s.hdr[1] = count; }
    } else {
        // 32 windows at a time: every lane hashes one leader, the warp keeps those that are its own and inserts them in order
        for (uint32_t k0 = 0; k0 < pl.nwin; k0 += 32) {
            const uint32_t k = k0 + lane;
            bool mine = false;
            if (k < pl.nwin) {
                const int i = (int)(pl.first + k);
                int32_t k4[4] = {0, 0, 0, 0};
                for (int j = 0; j < t.LL; ++j) k4[j] = row[i + j];
                const uint64_t h = cb_hash4(k4[0], k4[1], k4[2], k4[3], t.LL);
                mine = (uint32_t)((h >> 17) % (uint64_t)WPS) == (uint32_t)wi;
            }
            uint32_t todo = __ballot_sync(CB_FULL, mine);
            while (todo) {
                const int l = __ffs(todo) - 1;
                todo &= todo - 1;
                const int i = (int)(pl.first + k0 + l);
                const int32_t mykey = lane < t.LL ? row[i + lane] : 0;
                const int32_t myfol = lane < t.FL ? row[i + t.LL + lane] : 0;
                const uint32_t c = pl.clock0 + k0 + (uint32_t)l + 1u;
                // is the leader among the kept entries?  lane w compares way w's key
                bool match = lane < WAYS && ways[(size_t)lane * way_words + t.E] != 0u;
                for (int j = 0; j < t.LL; ++j) {
                    const int32_t kj = __shfl_sync(CB_FULL, mykey, j);
                    if (match) match = (int32_t)ways[(size_t)lane * way_words + j] == kj;
                }
                const uint32_t hit = __ballot_sync(CB_FULL, match);
                ++use_clock;
                if (hit) {
                    uint32_t* e = ways + (size_t)(__ffs(hit) - 1) * way_words;
                    cnt.inserts++;
                    if (lane == 0) { e[t.E + 1] = c; e[t.E + 2] = use_clock; }
                    tbl_put_follower(t, e, myfol, c, lane, cnt);
                    __syncwarp();
                    continue;
                }
                const int eid = tbl_insert_shared(t, s, mykey, myfol, c, lane, status, cnt);
                if (eid < 0) continue;
                // keep it: in a free way, else in place of the way used longest ago (whose copy goes back to the table first)
                uint32_t u = lane < WAYS ? (ways[(size_t)lane * way_words + t.E] == 0u ? 0u : ways[(size_t)lane * way_words + t.E + 2]) : 0xFFFFFFFFu;
                const uint32_t umin = __reduce_min_sync(CB_FULL, u);
                uint32_t* e = ways + (size_t)(__ffs(__ballot_sync(CB_FULL, u == umin)) - 1) * way_words;
                const uint32_t old = e[t.E];
                if (old != 0u) {
                    uint32_t* g = s.entries + (size_t)(old - 1u) * t.E;
                    for (uint32_t k = lane; k < t.E; k += 32) g[k] = e[k];
                    if (lane == 0) s.lstamp[old - 1u] = e[t.E + 1];
                }
                __syncwarp();
                const uint32_t* g = s.entries + (size_t)eid * t.E;
                for (uint32_t k = lane; k < t.E; k += 32) e[k] = __ldcg(g + k);
                if (lane == 0) { e[t.E] = (uint32_t)eid + 1u; e[t.E + 1] = c; e[t.E + 2] = use_clock; }
                __syncwarp();
            }
        }
        // the kept entries go back to the table
        for (int w = 0; w < WAYS; ++w) {
            const uint32_t* e = ways + (size_t)w * way_words;
            const uint32_t id = e[t.E];
            if (id == 0u) continue;
            uint32_t* g = s.entries + (size_t)(id - 1u) * t.E;
            for (uint32_t k = lane; k < t.E; k += 32) g[k] = e[k];
            if (lane == 0) s.lstamp[id - 1u] = e[t.E + 1];
        }
    }
    if (lane == 0) {
        if (cnt.inserts) atomicAdd(&counters[CB_CNT_INSERTS], (unsigned long long)cnt.inserts);
        if (cnt.levict) atomicAdd(&counters[CB_CNT_LEADER_EVICTIONS], (unsigned long long)cnt.levict);
        if (cnt.fevict) atomicAdd(&counters[CB_CNT_FOLLOWER_EVICTIONS], (unsigned long long)cnt.fevict);
        if (cnt.maxprobe) atomicMax(&counters[CB_CNT_MAX_PROBE], (unsigned long long)cnt.maxprobe);
    }
}

}  // namespace

#include "cb_bulk_free.cuh"
#include "cb_bulk_block.cuh"

namespace {

// ---------------------------------------------------------------------------------------------------
// Draft-tree expansion: one CTA per sequence, one warp per frontier leaf ("branch") for the lookups.
// Each level: (1) warps look up the keys of all frontier leaves in parallel and stage the followers,
// most recent first, in shared memory; (2) one warp plans the sequential breadth-first order over
// the staged results, which fixes node indices, the point where the size cap ends the level and the
// ordinal of every query that the sequential order would have issued, and gives the leaders of those queries
// their new recency stamp with an atomic max (two leaves of one level may share a leader); (3) warps attach the nodes.
// With a frozen table attached (Section 3.3) a second pass follows while the tree is below the size cap: its first
// frontier is every node that was a frontier leaf of the first pass, in creation order, and its lookups go to the
// frozen table, which is shared by all sequences and only read (no clock tick, no stamp).
// A node goes to the output arrays when it is attached, its mask row being its leaf's plus a run of bits.  A level of one leaf (the
// first one always is) is looked up, planned and filled in by one warp without a barrier.
// x / d = x * kInverse[d] >> 16 for d <= CB_MAX_FL and the x that occur here (below 1,024): a division is a chain of 100 cycles
__constant__ uint32_t kInverse[CB_MAX_FL + 1] = {0u, 65537u, 32769u, 21846u, 16385u, 13108u, 10923u, 9363u, 8193u};
struct DraftSmem {
    int32_t* tok; int32_t* par; int32_t* dep; uint32_t* mask;
    int32_t* front; int32_t* next; int32_t* pts;
    int32_t* r_eid;        // [NL each, by place in the frontier] the leader's entry
    uint32_t* r_want;      // nodes that the leaf's followers would take | queried << 12 | found << 13 | nodes per follower << 16
    uint32_t* r_plan;      // first node | nodes << 8 | first place in the next frontier << 16 | nodes per follower << 24
    int32_t* fol;
};
constexpr int kDraftArrays = 6;                               // of NL words

// The work of the CTA that drafts sequence b, whose history holds L tokens.  upd_n_old >= 0: the windows that the tokens
// from upd_n_old on complete are inserted first (cb_update_draft_tree and the call that follows an acceptance).  row(i): token i of
// the history (which this CTA may have extended just before).  put_n(n): stores the new tree's node count (one thread, at the end).
template <int FETCH, typename Tokens, typename PutN>
__device__ __forceinline__ void draft_body(const CbTables& t, const CbTables& tf, int T, int crt, int max_depth, int NL, int KF,
                                           const Tokens& row, int b, int L, int upd_n_old,
                                           int32_t* __restrict__ o_tok, int32_t* __restrict__ o_par,
                                           int32_t* __restrict__ o_dep, uint32_t* __restrict__ o_mask,
                                           PutN&& put_n, uint32_t* status,
                                           unsigned long long* counters, int32_t* smem) {
    DraftSmem S;
    const int W = (T + 31) >> 5;
    S.tok = smem; S.par = S.tok + T; S.dep = S.par + T; S.mask = (uint32_t*)(S.dep + T);
    S.front = (int32_t*)(S.mask + T * W); S.next = S.front + NL; S.pts = S.next + NL;
    S.r_eid = S.pts + NL; S.r_want = (uint32_t*)(S.r_eid + NL); S.r_plan = S.r_want + NL;
    S.fol = (int32_t*)(S.r_plan + NL);
    // Nodes, leaves of the level's frontier, leaves listed for the frozen pass: a level reads one set and leaves the other for the next
    // level, so that a barrier at its end is all that lies between two levels.
    __shared__ int sh_n[2], sh_nfront[2], sh_npts[2];
    int q = 0, hits = 0, fq = 0, fhits = 0;                   // kept by warp 0, which plans every level

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nwarps = blockDim.x >> 5;
    const CbSeq s = cb_seq(t, b);
    // The root needs no look at the table: a thread of the last warp, which most often has no window to insert, puts it there.
    if (tid == (int)blockDim.x - 32) {
        const bool root = L >= 1;
        sh_n[0] = sh_nfront[0] = sh_npts[0] = root ? 1 : 0;
        if (root) {
            const int tk = row(L - 1);
            S.tok[0] = tk; S.par[0] = -1; S.dep[0] = 0; S.front[0] = 0; S.pts[0] = 0;
            const size_t at = (size_t)b * T;
            o_tok[at] = tk; o_par[at] = -1; o_dep[at] = 0;
            for (int k = 0; k < W; ++k) { S.mask[k] = k == 0 ? 1u : 0u; o_mask[at * W + k] = k == 0 ? 1u : 0u; }
        }
    }
    if (upd_n_old >= 0) {
        // cb_update_draft_tree: the sequence's new windows go into the table first, then the CTA drafts from the updated table.
        update_seq_cta<FETCH>(t, b, row, upd_n_old, L, warp, lane, status, counters, [&] {
            if (L < t.LL) return;
            const int32_t mykey = lane < t.LL ? row(L - t.LL + lane) : 0;
            EntryRegs er;
            const Probe pr = tbl_find<false, FETCH>(t, s, mykey, warp_hash(t, mykey), lane, &er);
            if (pr.eid < 0) return;                              // nothing but the bucket was read
            if (FETCH == 1) {
                asm volatile("" ::"r"(er.fs));
#pragma unroll
                for (int j = 0; j < CB_MAX_FL; ++j) asm volatile("" ::"r"(er.tok[j]));
            } else {
#pragma unroll
                for (int c = 0; c < CB_MAX_FC / 32; ++c) asm volatile("" ::"r"(er.fs4[c]));
            }
        });
        __syncthreads();
    }
    const int FLFC = t.FL * KF;                               // staged followers per leaf: the KF best
    // Read back from memory although update_seq_cta's threads know it: handed on from there, with one barrier less, the compiler gave the kernel
    // of short lists 92 registers instead of 80, two blocks an SM instead of three (batch 300 12.4 us, so 9.6), and long lists
    // (one leader token, 128 followers) took 10.9 us, 15.3 with a cold L2, instead of 10.0 and 12.9; batch 1 of short lists gained 0.1.
    const uint32_t clock0 = s.hdr[0];
    const bool has_frozen = tf.index != nullptr;

    // Nodes [0, tot) of leaf `leaf` (depth d), numbered from n0 on, by one warp: node x is token x % cl of follower x / cl.
    auto attach = [&](int leaf, int d, int n0, int cl, int tot, const int32_t* fol) {
        const uint32_t inv = kInverse[cl];
        for (int x = lane; x < tot; x += 32) {
            const int f = (int)(((uint32_t)x * inv) >> 16), j = x - f * cl, node = n0 + x;
            const int tk = fol[f * t.FL + j], pa = j == 0 ? leaf : node - 1, de = d + j + 1;
            S.tok[node] = tk; S.par[node] = pa; S.dep[node] = de;
            const size_t at = (size_t)b * T + node;
            o_tok[at] = tk; o_par[at] = pa; o_dep[at] = de;
            for (int k = 0; k < W; ++k) {
                uint32_t m = S.mask[leaf * W + k];
                const int lo = max(node - j - 32 * k, 0), hi = min(node - 32 * k, 31);   // the chain so far: nodes node - j ... node
                if (lo <= hi) m |= (0xFFFFFFFFu >> (31 - hi)) & (0xFFFFFFFFu << lo);
                S.mask[node * W + k] = m;
                o_mask[at * W + k] = m;
            }
        }
    };
    __syncthreads();

    int cur = 0;
    for (int pass = 0; pass < (has_frozen ? 2 : 1); ++pass) {
        const CbTables& tt = pass ? tf : t;
        const CbSeq ss = pass ? cb_seq(tf, 0) : s;
        // the frozen pass starts from every frontier leaf the dynamic pass had
        bool listed = pass == 1;
        if (listed) { S.next = S.front; S.front = S.pts; }
        while (true) {
            const int nfront = listed ? sh_npts[cur] : sh_nfront[cur], n_top = sh_n[cur], npts = sh_npts[cur];
            if (nfront == 0 || n_top >= T) break;
            if (pass == 0 && S.dep[S.front[0]] >= max_depth) break;   // a level's leaves lie at one depth: none may be queried
            listed = false;
            cur ^= 1;
            if (tid == 0) { sh_n[cur] = n_top; sh_nfront[cur] = 0; sh_npts[cur] = npts; }
            // With long follower lists the frontier is worked off in batches of one leaf per warp, lookups then replay, so that a
            // level ends as soon as the tree is full (the first leaves of a level then usually take all the room).
            const int BS = tt.FC > 32 ? nwarps : nfront;          // short follower lists: the whole frontier at once
            for (int base = 0; base < nfront; base += BS) {
                const int n_now = base == 0 ? n_top : sh_n[cur];
                if (n_now >= T) break;
                // (1) parallel lookups, one warp per leaf
                for (int li = base + warp; li < min(nfront, base + BS); li += nwarps) {
                    const int leaf = S.front[li];
                    const int d = S.dep[leaf];
                    if (d >= max_depth) {                     // nothing may hang below it: not queried
                        if (lane == 0) S.r_want[li] = 0u;
                        continue;
                    }
                    // key = last LL tokens of (row[0 .. L-1) ++ root->leaf path); lane j < LL holds key[j]
                    int32_t mykey = 0;
                    bool ok = true;
                    if (lane < t.LL) {
                        const int back = t.LL - 1 - lane;     // distance from the leaf along the sequence
                        if (back <= d) {
                            int c = leaf;
                            for (int k = 0; k < back; ++k) c = S.par[c];
                            mykey = S.tok[c];
                        } else {
                            const int pos = L - 1 - (back - d);
                            mykey = pos >= 0 ? row(pos) : -1;
                        }
                    }
                    ok = ok && __all_sync(CB_FULL, mykey >= 0);
                    int eid = -1, nf = 0;
                    if (ok) {
                        const uint64_t h = warp_hash(tt, mykey);
                        EntryRegs er;
                        const Probe pr = tbl_find<false, FETCH>(tt, ss, mykey, h, lane, &er);
                        if (pr.eid == -2 && lane == 0) atomicCAS(status, 0u, (uint32_t)CB_ERR_PROBE_LIMIT);
                        if (pr.eid >= 0) {
                            eid = pr.eid;
                            const uint32_t* e = ss.entries + (size_t)eid * tt.E;
                            // Lane l holds the stamps of followers l, l + 32, ...  The followers are wanted by falling stamp
                            // (most recently inserted first in the dynamic table, most frequent first in the frozen one),
                            // and only as many as the tree still has room for: they are picked one by one with a warp-wide
                            // maximum (stamps are unique) and staged in that order.
                            constexpr int CH = FETCH == 1 ? 1 : CB_MAX_FC / 32;    // followers per lane
                            uint32_t fs[CH];
#pragma unroll
                            for (int c = 0; c < CH; ++c) {
                                fs[c] = FETCH == 1 ? er.fs : er.fs4[c];            // came with the lookup (FC <= 32: the tokens too)
                                nf += __popc(__ballot_sync(CB_FULL, fs[c] != 0u));
                            }
                            // The followers' tokens.  FC > 32: on their way while the followers are picked below (of all of them: the
                            // round trip costs more than the bytes).
                            int32_t ft[CH][CB_MAX_FL];
#pragma unroll
                            for (int c = 0; c < CH; ++c) {
                                const int f = c * 32 + lane;
#pragma unroll
                                for (int j = 0; j < CB_MAX_FL; ++j) {
                                    if (FETCH == 1) ft[c][j] = er.tok[j];
                                    else ft[c][j] = fs[c] != 0u && j < tt.FL ? (int32_t)e[tt.LL + tt.FC + f * tt.FL + j] : -1;
                                }
                            }
                            // no more than the tree has room for chains of this length
                            const int cl = min(tt.FL, max_depth - d), room = (leaf == 0 ? max(1, T - crt) : T) - n_now;
                            nf = min(nf, min(KF, (int)(((uint32_t)(max(room, 0) + cl - 1) * kInverse[cl]) >> 16)));
                            int rank[CH];
#pragma unroll
                            for (int c = 0; c < CH; ++c) rank[c] = -1;
                            if (FETCH == 1 || nf <= 40) {     // about where a maximum each costs what the counting below does
                                for (int r = 0; r < nf; ++r) {
                                    uint32_t m = fs[0];
#pragma unroll
                                    for (int c = 1; c < CH; ++c) m = max(m, fs[c]);
                                    const uint32_t g = __reduce_max_sync(CB_FULL, m);
#pragma unroll
                                    for (int c = 0; c < CH; ++c)
                                        if (fs[c] == g) { rank[c] = r; fs[c] = 0u; }
                                }
                            } else {
                                // many are wanted: rank every follower by counting the larger stamps (independent shuffles,
                                // where the repeated maximum is a chain of reductions)
                                int cntr[CH];
#pragma unroll
                                for (int c = 0; c < CH; ++c) cntr[c] = 0;
#pragma unroll
                                for (int c2 = 0; c2 < CH; ++c2) {
                                    if (c2 * 32 >= tt.FC) break;
                                    for (int l = 0; l < 32; ++l) {
                                        const uint32_t o = __shfl_sync(CB_FULL, fs[c2], l);
#pragma unroll
                                        for (int c = 0; c < CH; ++c) cntr[c] += (o > fs[c]) ? 1 : 0;
                                    }
                                }
#pragma unroll
                                for (int c = 0; c < CH; ++c)
                                    if (fs[c] != 0u && cntr[c] < nf) rank[c] = cntr[c];
                            }
                            // every lane stages its picked followers
#pragma unroll
                            for (int c = 0; c < CH; ++c) {
                                if (rank[c] < 0) continue;
#pragma unroll
                                for (int j = 0; j < CB_MAX_FL; ++j)
                                    if (j < tt.FL) S.fol[li * FLFC + rank[c] * tt.FL + j] = ft[c][j];
                            }
                        }
                    }
                    const int cl = min(t.FL, max_depth - d);
                    if (nfront > 1) {
                        if (lane == 0) {
                            S.r_eid[li] = eid;
                            S.r_want[li] = (uint32_t)(max(nf, 0) * cl) | (ok ? 1u << 12 : 0u) | (eid >= 0 ? 1u << 13 : 0u) | (uint32_t)cl << 16;
                        }
                    } else {
                        // the only leaf of its level (this is warp 0): what (2) and (3) do, in place
                        const int cap = leaf == 0 ? max(1, T - crt) : T;
                        if (ok && n_now < cap) {
                            const int tot = eid >= 0 ? min(max(nf, 0) * cl, cap - n_now) : 0;
                            const int ends = cl == t.FL ? (int)(((uint32_t)tot * kInverse[cl]) >> 16) : 0;
                            if (pass == 0) { ++q; hits += eid >= 0 ? 1 : 0; } else { ++fq; fhits += eid >= 0 ? 1 : 0; }
                            if (lane == 0) {
                                if (pass == 0 && eid >= 0) atomicMax(&s.lstamp[eid], clock0 + (uint32_t)q);
                                sh_n[cur] = n_now + tot; sh_nfront[cur] = ends;
                                if (pass == 0) sh_npts[cur] = npts + ends;
                            }
                            __syncwarp();
                            attach(leaf, d, n_now, cl, tot, S.fol + li * FLFC);
                            for (int c = lane; c < ends; c += 32) {
                                const int end = n_now + c * t.FL + t.FL - 1;
                                S.next[c] = end;
                                if (pass == 0 && has_frozen) S.pts[npts + c] = end;
                            }
                        }
                    }
                }
                if (nfront == 1) break;
                __syncthreads();
                // (2) the sequential breadth-first order, planned by one warp and filled in by all.  A query at the root (the only
                // leaf of level 1, the first one of the frozen pass) is issued, and its followers attached, while the tree has fewer
                // than max(1, T - crt) nodes; any other while fewer than T.  Below a leaf of depth d every follower is a chain of
                // min(FL, max_depth - d) nodes, the chains follow one another until the cap cuts the last one short, and a chain of
                // FL nodes ends in a leaf of the next level: so a leaf's nodes and frontier places follow from what the leaves
                // before it want, a running sum that stops at the cap.  A leaf's lookup leaves one word for it and its plan is one word
                // (with a word for each figure, and one thread for up to 16 leaves, planning took 1.6 to 3 k cycles a level).
                const int lend = min(nfront, base + BS);
                if (warp == 0) {
                    int n = n_now, nn = sh_nfront[cur];
                    for (int l0 = base; l0 < lend; l0 += 32) {
                        const int l2 = l0 + lane;
                        const uint32_t x = l2 < lend ? S.r_want[l2] : 0u;
                        const bool ok = (x >> 12) & 1u, hit = (x >> 13) & 1u;
                        const int cl = (int)(x >> 16);
                        int want = hit ? (int)(x & 0xFFFu) : 0;
                        bool open = true;
                        if (l2 == 0 && S.front[0] == 0) {      // the root, before every other leaf: n nodes stand when its turn comes
                            const int cap = max(1, T - crt);
                            open = n < cap;
                            want = min(want, max(cap - n, 0));
                        }
                        int incl = want;
#pragma unroll
                        for (int o = 1; o < 32; o <<= 1) {
                            const int up = __shfl_up_sync(CB_FULL, incl, o);
                            if (lane >= o) incl += up;
                        }
                        const int start = min(T, n + incl - want);
                        const bool issued = ok && open && start < T;          // the dynamic table's clock ticks
                        const int tot = issued ? min(want, T - start) : 0;
                        const uint32_t mi = __ballot_sync(CB_FULL, issued), mh = __ballot_sync(CB_FULL, issued && hit);
                        const int leaves = cl == t.FL ? (int)(((uint32_t)tot * kInverse[cl]) >> 16) : 0;
                        int lincl = leaves;
#pragma unroll
                        for (int o = 1; o < 32; o <<= 1) {
                            const int up = __shfl_up_sync(CB_FULL, lincl, o);
                            if (lane >= o) lincl += up;
                        }
                        if (l2 < lend) {
                            // the leaders that the sequential order reached get their stamp (two leaves of a level may share a leader)
                            if (pass == 0 && issued && hit) atomicMax(&s.lstamp[S.r_eid[l2]], clock0 + (uint32_t)(q + __popc(mi & (0xFFFFFFFFu >> (31 - lane)))));
                            S.r_plan[l2] = (uint32_t)start | (uint32_t)tot << 8 | (uint32_t)(nn + lincl - leaves) << 16 | (uint32_t)cl << 24;
                        }
                        if (pass == 0) { q += __popc(mi); hits += __popc(mh); } else { fq += __popc(mi); fhits += __popc(mh); }
                        n = min(T, n + __shfl_sync(CB_FULL, incl, 31));
                        nn += __shfl_sync(CB_FULL, lincl, 31);
                    }
                    if (lane == 0) {
                        sh_n[cur] = n; sh_nfront[cur] = nn;
                        if (pass == 0) sh_npts[cur] = npts + nn;
                    }
                }
                __syncthreads();
                // (3) the leaves' nodes and the next frontier
                for (int l2 = base + warp; l2 < lend; l2 += nwarps) {
                    const uint32_t x = S.r_plan[l2];
                    const int n0 = (int)(x & 0xFFu), tot = (int)(x >> 8) & 0xFF, nn0 = (int)(x >> 16) & 0xFF, cl = (int)(x >> 24);
                    if (tot == 0) continue;
                    const int leaf = S.front[l2];
                    attach(leaf, S.dep[leaf], n0, cl, tot, S.fol + l2 * FLFC);
                    if (cl == t.FL)
                        for (int c = lane; c < (int)(((uint32_t)tot * kInverse[cl]) >> 16); c += 32) {
                            const int end = n0 + c * t.FL + t.FL - 1;
                            S.next[nn0 + c] = end;
                            if (pass == 0 && has_frozen) S.pts[npts + nn0 + c] = end;
                        }
                }
            }
            __syncthreads();
            int32_t* const done = S.front;
            S.front = S.next;
            S.next = done;
        }
    }

    const int n = sh_n[cur];
    if (tid == 0) {
        s.hdr[0] = clock0 + (uint32_t)q;
        put_n(n);
        if (q) atomicAdd(&counters[CB_CNT_QUERIES], (unsigned long long)q);
        if (hits) atomicAdd(&counters[CB_CNT_QUERY_HITS], (unsigned long long)hits);
        if (fq) atomicAdd(&counters[CB_CNT_FROZEN_QUERIES], (unsigned long long)fq);
        if (fhits) atomicAdd(&counters[CB_CNT_FROZEN_HITS], (unsigned long long)fhits);
    }
    for (int i = n + tid; i < T; i += blockDim.x) {              // places without a node
        const size_t at = (size_t)b * T + i;
        o_tok[at] = -1; o_par[at] = -1; o_dep[at] = -1;
        for (int k = 0; k < W; ++k) o_mask[at * W + k] = 0u;
    }
}

template <int FETCH>
__global__ void __launch_bounds__(256) cb_draft_kernel(CbTables t, CbTables tf, int T, int crt, int max_depth, int NL, int KF,
                                                       const int32_t* __restrict__ tokens, int64_t row_stride,
                                                       const int32_t* __restrict__ seq_len, const int32_t* __restrict__ upd_n_old,
                                                       int32_t* __restrict__ o_tok, int32_t* __restrict__ o_par,
                                                       int32_t* __restrict__ o_dep, uint32_t* __restrict__ o_mask,
                                                       int32_t* __restrict__ o_n, uint32_t* status,
                                                       unsigned long long* counters) {
    CB_PDL_ENTRY();
    extern __shared__ int32_t smem[];
    const int b = blockIdx.x;
    const int32_t* history = tokens + (size_t)b * row_stride;
    draft_body<FETCH>(t, tf, T, crt, max_depth, NL, KF, [=](int i) { return history[i]; }, b, seq_len[b], upd_n_old ? upd_n_old[b] : -1, o_tok, o_par,
                      o_dep, o_mask, [=](int n) { o_n[b] = n; }, status, counters, smem);
}

// Acceptance of one step and update + draft of the next in one launch (the three are a chain per sequence: Fig. 2).  The
// grid is the acceptance kernel's; the CTA that ends a sequence's acceptance appends the emitted tokens (accepted ones and
// the bonus token) to the sequence's history, advances its length, and goes on as that sequence's update-and-draft CTA.
struct AcceptArgs {
    int V, Dmax, chunk, chunks_per_row;
    const void* logits; int64_t logits_row_stride;
    const int32_t* tok; const int32_t* par; const int32_t* dep; const int32_t* n_nodes;
    unsigned long long* rowmax; uint32_t* ticket;
    int32_t* n_accept; int32_t* accept_nodes; int32_t* out_tokens; int32_t* target_out;
};

// CTAS: CTAs that an SM has registers for.  The drafting code takes 112 registers, room for two.  A grid that is not resident at
// once that way streams the logits with half in flight of what four CTAs of 62 have (a step of batch 6 with trees of 96: 86.6 us with three
// of 72, 82.9 with four; batch 4 of 64: 61.3 and 59.6); one that is gains nothing from the bound and pays for it in the chain behind
// the logits, and takes all of a thread's chunk at once instead.  With more than 32 followers a leader the code takes 119 registers and
// stays at two.
//
// IN_PLACE: o_n is a.n_nodes.  Which rows a sequence's tree has decides which of its CTAs count for the acceptance, so its entry is stored only
// when every CTA of the sequence has read the old one: those of the tree's rows have when the drafting CTA begins; those of the rows
// past it (`waiting` of them) and the drafting CTA count themselves in a word of their own, and the last to come stores.  The word is the
// packed maximum of row T - 1, which such a tree does not have: arrivals below, the new count above, zero between launches.  A CTA
// that started late would otherwise take its row for one of the tree and leave a maximum and a ticket behind for the next launch.
// (A form of its own: in the other one the two words that it keeps to the end cost a grid of four CTAs an SM 1.5% and batch 2 7%.)
template <int FETCH, bool BF16, int CTAS, bool IN_PLACE>
__global__ void __launch_bounds__(256, CTAS) cb_accept_draft_kernel(AcceptArgs a, CbTables t, CbTables tf, int T, int crt, int max_depth, int NL, int KF,
                                                              int32_t* tokens, int64_t row_stride, int32_t* seq_len,
                                                              int32_t* o_tok, int32_t* o_par, int32_t* o_dep, uint32_t* o_mask, int32_t* o_n,
                                                              uint32_t* status, unsigned long long* counters) {
    CB_PDL_ENTRY();
    extern __shared__ int32_t smem[];
    // The end of the history, from the first token of the first new window on, with the emitted tokens behind it: what the update and
    // the root's key need, without going through memory.
    __shared__ int32_t s_tail[CB_MAX_LL + CB_MAX_FL + 256], s_emit[256];
    __shared__ int s_have, s_len;
    const int b = blockIdx.z, tid = threadIdx.x, w = t.LL + t.FL;
    const int n_old = min(max(a.n_nodes[b], 0), T);             // through L1: past it, thousands of warps at one word are a microsecond and more
    uint32_t waiting = 0u;
    auto arrive = [&](unsigned long long x) {
        unsigned long long* const word = a.rowmax + (size_t)b * T + T - 1;
        unsigned long long now;
        asm volatile("atom.add.acq_rel.gpu.global.u64 %0, [%1], %2;" : "=l"(now) : "l"(word), "l"(x) : "memory");
        now += x;
        if ((uint32_t)now == waiting + 1u) { o_n[b] = (int32_t)(now >> 32); *word = 0ull; }
    };
    if constexpr (IN_PLACE) {
        const int rows = max(n_old, 1);
        waiting = (uint32_t)(T - rows) * gridDim.x;
        __syncthreads();                                        // all threads of this CTA have read the count
        if ((int)blockIdx.y >= rows) {
            if (tid == 0) arrive(1ull);
            return;
        }
    }
    int32_t* const history = tokens + (size_t)b * row_stride;
    auto beside = [&](int k) {
        if (k >= 32) return;
        const int L = seq_len[b], tail0 = max(0, L - w + 1);
        if (k < L - tail0 && L <= row_stride) s_tail[k] = history[tail0 + k];
        if (k == 0) s_len = L;
    };
    if (!accept_rows<BF16, CTAS == 2 && FETCH == 1 ? 8 : 4>(T, a.V, a.Dmax, a.chunk, a.chunks_per_row, a.logits, a.logits_row_stride, a.tok, a.par, a.dep,
                                                            n_old, a.rowmax, a.ticket, a.n_accept, a.accept_nodes, a.out_tokens, a.target_out, beside,
                                                            s_emit, &s_have))
        return;
    __syncthreads();                                            // the walk (first warp) has written the sequence's result
    const int have = s_have;                                    // tokens emitted (an empty tree emits none)
    // (a malformed tree may name a depth beyond any of its own: more places than are kept here are read from the history)
    const int L = s_len, tail0 = have <= 256 ? max(0, L - w + 1) : 0x7FFFFFFF;
    int L1 = L + have;
    if (L < 0 || L1 > row_stride) {
        // no room in the history, or no length: nothing is appended and the step is reported; the draft below continues from what is there
        if (tid == 0) atomicCAS(status, 0u, (uint32_t)CB_ERR_INVALID_ARG);
        L1 = L;
    } else if (tid < have) {
        history[L + tid] = s_emit[tid];
        if (have <= 256) s_tail[L - tail0 + tid] = s_emit[tid];
    }
    __syncthreads();
    if (tid == 0) seq_len[b] = L1;
    draft_body<FETCH>(t, tf, T, crt, max_depth, NL, KF, [&](int i) { return i >= tail0 && L <= row_stride ? s_tail[i - tail0] : history[i]; }, b, L1, L,
                      o_tok, o_par, o_dep, o_mask, [&](int n) {
                          if (IN_PLACE && waiting) arrive((unsigned long long)n << 32 | 1ull);
                          else o_n[b] = n;
                      }, status, counters, smem);
}

}  // namespace

extern "C" cb_status cb_update(cb_ctx* ctx, const int32_t* tokens, int64_t row_stride, const int32_t* n_old,
                               const int32_t* n_new, void* stream) {
    CB_CHECK_ARG(ctx && tokens && n_old && n_new && row_stride >= 1);
    const int B = ctx->cfg.batch, wpb = 4;
    CB_CUDA(cb_launch_pdl(ctx->cfg.FC <= 32 ? cb_update_kernel<1> : cb_update_kernel<2>, dim3((B + wpb - 1) / wpb), dim3(wpb * 32), 0, (cudaStream_t)stream, ctx->tables, B, tokens, row_stride,
                          n_old, n_new, ctx->d_status, ctx->d_counters));
    cb_count_launch(1);
    return CB_OK;
}

extern "C" cb_status cb_update_bulk(cb_ctx* ctx, const int32_t* tokens, int64_t row_stride, const int32_t* n_old,
                                    const int32_t* n_new, void* stream) {
    CB_CHECK_ARG(ctx && tokens && n_old && n_new && row_stride >= 1);
    const int B = ctx->cfg.batch;
    // Runs of up to kBlkRun windows that qualify are reduced by blocks that hold them in shared memory.  Where a row has room for no
    // other run (room for a window less than the leader capacity: then nothing can be evicted, unless the table holds more than the
    // row's text; without room for one window the stride means nothing, as in a batch of one), that is all: one launch.  Otherwise it is told
    // what is whose before (plan), and the longer runs and those in order follow: batch 32 of 1,024 to 8,192 tokens 32 us alone, 36 so.
    const int w = ctx->tables.LL + ctx->tables.FL;
    const bool blocks = ctx->tables.refresh && B <= kBlkMaxBatch;
    const bool alone = blocks && row_stride >= w && row_stride - w + 1 <= (int64_t)std::min(kBlkRun, ctx->tables.LC);
    const int done = blocks ? kBlkRun : -1;
    // enough warps per sequence to fill the GPU at small batch, fewer at large batch
    int wps = 1;
    while (wps < 256 && (long long)B * wps * 2 <= (long long)ctx->num_sms * 64) wps *= 2;
    BulkPlan* plan = reinterpret_cast<BulkPlan*>(ctx->d_bulk_plan);
    const cudaStream_t st = (cudaStream_t)stream;
    const bool free_path = ctx->bulk_scratch && B <= kBulkFreeMaxBatch && ctx->tables.refresh;
    BulkFreeView v = {};
    if (free_path) v = bulk_free_view(ctx->bulk_scratch, ctx->bulk_slots, B);
    if (!alone) {
        if (free_path) CB_CUDA(cb_launch_pdl(cb_bulk_free_plan_kernel, dim3(1), dim3(1024), 0, st, ctx->tables, B, n_old, n_new, plan, v, ctx->d_counters, done));
        else CB_CUDA(cb_launch_pdl(cb_bulk_plan_kernel, dim3((B + 127) / 128), dim3(128), 0, st, ctx->tables, B, n_old, n_new, plan, done));
        cb_count_launch(1);
    }
    if (blocks) {
        using Kernel = void (*)(CbTables, int, const int32_t*, int64_t, const int32_t*, const int32_t*, bool, uint32_t*, unsigned long long*);
        // [leader][follower][every displaced follower counted: with scratch attached the call does not promise that]
#define CB_BLK(l) {{cb_update_bulk_block_kernel<l, 4, false>, cb_update_bulk_block_kernel<l, 4, true>}, {cb_update_bulk_block_kernel<l, 8, false>, cb_update_bulk_block_kernel<l, 8, true>}}
        static const Kernel kernels[CB_MAX_LL][2][2] = {CB_BLK(1), CB_BLK(2), CB_BLK(3), CB_BLK(4)};
#undef CB_BLK
        const int l = ctx->tables.LL - 1, f = ctx->tables.FL <= 4 ? 0 : 1, all = ctx->bulk_scratch ? 0 : 1;
        const Kernel kernel = kernels[l][f][all];
        static std::mutex mu;
        static bool opted[64][CB_MAX_LL][2][2] = {};              // per device
        {
            std::lock_guard<std::mutex> lock(mu);
            bool& done_here = opted[ctx->device & 63][l][f][all];
            if (!done_here) {
                CB_CUDA(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(BlkSmem)));
                done_here = true;
            }
        }
        CB_CUDA(cb_launch_pdl(kernel, dim3((unsigned)ctx->num_sms), dim3(kBlkThreads), sizeof(BlkSmem), st, ctx->tables, B, tokens, row_stride, n_old, n_new,
                              alone, ctx->d_status, ctx->d_counters));
        cb_count_launch(1);
        if (alone) return CB_OK;
    }
    // The block kernel takes nearly all of an SM's memory as shared memory, and a kernel without a preference runs with what L1 that leaves
    // (runs in order of batch 512: 11.9 ms a call, so 7.2; scratch, batch 128 of 32 k: 2.59 and 2.04): those behind it ask for theirs.
    static std::mutex l1_mu;
    static int l1_asked[64][2] = {};                           // per device: percent + 1 that the last kernel prefers, 1 where the others are done
    auto prefer = [](auto kernel, int percent) { return cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout, percent); };
    if (free_path) {
        {
            std::lock_guard<std::mutex> lock(l1_mu);
            int& asked = l1_asked[ctx->device & 63][1];
            if (!asked) {
                CB_CUDA(prefer(cb_bulk_free_clear_kernel, 10)); CB_CUDA(prefer(cb_bulk_free_reduce_kernel, 10)); CB_CUDA(prefer(cb_bulk_free_ranges_kernel, 10));
                CB_CUDA(prefer(cb_bulk_free_scatter_kernel, 10)); CB_CUDA(prefer(cb_bulk_free_apply_kernel, 10));
                asked = 1;
            }
        }
        // order-free path for the longer sequences that qualify and fit the attached scratch; the kernel below does the others
        const unsigned grid = (unsigned)std::min<long long>((long long)v.S / 256, (long long)ctx->num_sms * 8);
        const unsigned wide = (unsigned)std::min<long long>((long long)v.S / 256, (long long)ctx->num_sms * 32);   // one item per thread, or a few
        CB_CUDA(cb_launch_pdl(cb_bulk_free_clear_kernel, dim3(wide), dim3(256), 0, st, v));
        CB_CUDA(cb_launch_pdl(cb_bulk_free_reduce_kernel, dim3(wide), dim3(256), 0, st, ctx->tables, B, tokens, row_stride, (const BulkPlan*)plan, v,
                              ctx->d_status));
        CB_CUDA(cb_launch_pdl(cb_bulk_free_ranges_kernel, dim3(wide), dim3(256), 0, st, v));
        CB_CUDA(cb_launch_pdl(cb_bulk_free_scatter_kernel, dim3(wide), dim3(256), 0, st, v));
        CB_CUDA(cb_launch_pdl(cb_bulk_free_apply_kernel, dim3(grid), dim3(256), 0, st, ctx->tables, B, tokens, row_stride, (const BulkPlan*)plan, v,
                              ctx->d_status, ctx->d_counters));
        cb_count_launch(5);
    }
    const long long warps = (long long)B * wps;
    // kept entries per warp: four, fewer where 96 KB of shared memory per CTA (8 warps) do not hold that many
    const size_t way_bytes = ((size_t)ctx->tables.E + 4) * 4;
    const int n_ways = (int)std::max<size_t>(1, std::min<size_t>(4, (96 * 1024) / (8 * way_bytes)));
    const size_t smem = 8 * (size_t)n_ways * way_bytes;
    if (smem > 200 * 1024) return CB_ERR_UNSUPPORTED;
    if (smem > 48 * 1024) {
        static size_t opted[64] = {0};                         // largest size opted into so far, per device
        const int d = ctx->device & 63;
        if (opted[d] < smem) {
            CB_CUDA(cudaFuncSetAttribute(cb_update_bulk_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
            opted[d] = smem;
        }
    }
    {
        std::lock_guard<std::mutex> lock(l1_mu);
        int& asked = l1_asked[ctx->device & 63][0];
        const int percent = (int)std::min<size_t>(100, 4 * (smem + 1024) * 100 / (228 * 1024) + 1);   // four blocks an SM
        if (asked != percent + 1) { CB_CUDA(prefer(cb_update_bulk_kernel, percent)); asked = percent + 1; }
    }
    CB_CUDA(cb_launch_pdl(cb_update_bulk_kernel, dim3((unsigned)((warps + 7) / 8)), dim3(256), smem, st, ctx->tables, B, wps, n_ways,
                          tokens, row_stride, n_old, n_new, (const BulkPlan*)plan, ctx->d_status, ctx->d_counters));
    cb_count_launch(1);
    return CB_OK;
}

extern "C" cb_status cb_bulk_scratch_bytes(const cb_config* cfg, int64_t max_windows, size_t* bytes) {
    CB_CHECK_ARG(cfg && bytes && cfg->batch >= 1 && max_windows >= 1 && max_windows <= (int64_t)1 << 29);
    uint32_t S = 2048;
    while ((int64_t)S < 2 * max_windows) S <<= 1;
    *bytes = bulk_free_layout(S, cfg->batch).total;
    return CB_OK;
}

extern "C" cb_status cb_bulk_scratch_attach(cb_ctx* ctx, void* dev_scratch, size_t bytes) {
    CB_CHECK_ARG(ctx);
    ctx->bulk_scratch = nullptr;
    ctx->bulk_slots = 0;
    if (!dev_scratch) return CB_OK;
    CB_CHECK_ARG((reinterpret_cast<uintptr_t>(dev_scratch) & 255u) == 0);
    // the largest power-of-two slot count whose layout fits
    uint32_t S = 0;
    for (uint32_t c = 2048; c != 0 && c <= (1u << 30) && bulk_free_layout(c, ctx->cfg.batch).total <= bytes; c <<= 1) S = c;
    CB_CHECK_ARG(S != 0);
    ctx->bulk_scratch = dev_scratch;
    ctx->bulk_slots = S;
    return CB_OK;
}

static cb_status draft_launch(cb_ctx* ctx, const int32_t* tokens, int64_t row_stride, const int32_t* seq_len, const int32_t* upd_n_old,
                              int32_t* tree_tokens, int32_t* tree_parent, int32_t* tree_depth,
                              uint32_t* tree_mask, int32_t* n_nodes, void* stream) {
    CB_CHECK_ARG(ctx && tokens && seq_len && tree_tokens && tree_parent && tree_depth && tree_mask && n_nodes);
    CB_CHECK_ARG(row_stride >= 1);
    const cb_config& c = ctx->cfg;
    const int T = c.max_nodes;
    const int NL = min(T, (T - 1) / c.FL + 1);
    // A leaf can receive at most T - 1 followers (each adds a node), so no more than that many are staged per lookup.
    const int FCmax = ctx->has_frozen ? max(c.FC, ctx->frozen.FC) : c.FC;
    const int KF = max(1, min(FCmax, T - 1));
    const size_t smem = sizeof(int32_t) * ((size_t)(3 + (T + 31) / 32) * T + (size_t)kDraftArrays * NL + (size_t)NL * c.FL * KF);
    if (smem > 200 * 1024) return CB_ERR_UNSUPPORTED;
    auto kernel = FCmax <= 32 ? cb_draft_kernel<1> : cb_draft_kernel<2>;
    {
        static std::mutex mu;
        static size_t have[64][2] = {};                        // per device and kernel
        std::lock_guard<std::mutex> lock(mu);
        CB_CUDA(cb_allow_smem(kernel, smem, &have[ctx->device & 63][FCmax <= 32 ? 0 : 1]));
    }
    const int threads = upd_n_old ? 32 * kUpdWarps : 32 * max(1, min(8, NL));   // insertions: a warp per window
    CbTables tf = {};
    if (ctx->has_frozen) tf = ctx->frozen;
    CB_CUDA(cb_launch_pdl(kernel, dim3(c.batch), dim3(threads), smem, (cudaStream_t)stream, ctx->tables, tf, T, c.crt, c.max_depth, NL, KF,
                          tokens, row_stride, seq_len, upd_n_old, tree_tokens, tree_parent, tree_depth, tree_mask, n_nodes, ctx->d_status, ctx->d_counters));
    cb_count_launch(1);
    return CB_OK;
}

extern "C" cb_status cb_draft_tree(cb_ctx* ctx, const int32_t* tokens, int64_t row_stride, const int32_t* seq_len,
                                   int32_t* tree_tokens, int32_t* tree_parent, int32_t* tree_depth,
                                   uint32_t* tree_mask, int32_t* n_nodes, void* stream) {
    return draft_launch(ctx, tokens, row_stride, seq_len, nullptr, tree_tokens, tree_parent, tree_depth, tree_mask, n_nodes, stream);
}

extern "C" cb_status cb_update_draft_tree(cb_ctx* ctx, const int32_t* tokens, int64_t row_stride, const int32_t* n_old,
                                          const int32_t* n_new, int32_t* tree_tokens, int32_t* tree_parent,
                                          int32_t* tree_depth, uint32_t* tree_mask, int32_t* n_nodes, void* stream) {
    CB_CHECK_ARG(n_old != nullptr);
    return draft_launch(ctx, tokens, row_stride, n_new, n_old, tree_tokens, tree_parent, tree_depth, tree_mask, n_nodes, stream);
}

extern "C" cb_status cb_accept_update_draft_tree(cb_ctx* ctx, const cb_accept_draft_args* a, void* stream) {
    CB_CHECK_ARG(ctx && a);
    CB_CHECK_ARG(a->logits && a->tree_tokens && a->tree_parent && a->tree_depth && a->n_nodes && a->n_accept && a->accept_nodes && a->out_tokens);
    CB_CHECK_ARG(a->tokens && a->seq_len && a->row_stride >= 1);
    CB_CHECK_ARG(a->next_tokens && a->next_parent && a->next_depth && a->next_mask && a->next_n_nodes);
    const cb_config& c = ctx->cfg;
    CB_CHECK_ARG(a->logits_dtype == CB_DTYPE_F32 || a->logits_dtype == CB_DTYPE_BF16);
    CB_CHECK_ARG(a->logits_row_stride >= c.vocab);
    const int esz = a->logits_dtype == CB_DTYPE_F32 ? 4 : 2;
    CB_CHECK_ARG(((uintptr_t)a->logits & (esz - 1)) == 0);
    if (c.batch > 65535) return CB_ERR_UNSUPPORTED;
    const int T = c.max_nodes;
    // the acceptance grid: about 32 KB of a logits row per CTA, fewer chunks when the batch alone fills the machine
    int chunk = 32768 / esz;
    if ((long)c.batch * T >= 8L * ctx->num_sms) chunk *= 4;
    int cpr = (c.vocab + chunk - 1) / chunk;
    chunk = ((c.vocab + cpr - 1) / cpr + 7) & ~7;
    cpr = (c.vocab + chunk - 1) / chunk;
    AcceptArgs aa;
    aa.V = c.vocab; aa.Dmax = c.max_depth; aa.chunk = chunk; aa.chunks_per_row = cpr;
    aa.logits = a->logits; aa.logits_row_stride = a->logits_row_stride;
    aa.tok = a->tree_tokens; aa.par = a->tree_parent; aa.dep = a->tree_depth; aa.n_nodes = a->n_nodes;
    aa.rowmax = ctx->d_rowmax; aa.ticket = ctx->d_ticket;
    aa.n_accept = a->n_accept; aa.accept_nodes = a->accept_nodes; aa.out_tokens = a->out_tokens; aa.target_out = a->target_ids_out;
    // the drafting CTA's shared memory, as in cb_draft_tree
    const int NL = min(T, (T - 1) / c.FL + 1);
    const int FCmax = ctx->has_frozen ? max(c.FC, ctx->frozen.FC) : c.FC;
    const int KF = max(1, min(FCmax, T - 1));
    const size_t smem = sizeof(int32_t) * ((size_t)(3 + (T + 31) / 32) * T + (size_t)kDraftArrays * NL + (size_t)NL * c.FL * KF);
    if (smem > 200 * 1024) return CB_ERR_UNSUPPORTED;
    const bool bf = a->logits_dtype == CB_DTYPE_BF16;
    const bool resident = (long long)cpr * T * c.batch <= 2ll * ctx->num_sms;
    // [form][bf16][in place]
    using Kernel = decltype(&cb_accept_draft_kernel<1, false, 2, false>);
    static const Kernel kernels[3][2][2] = {
        {{cb_accept_draft_kernel<2, false, 2, false>, cb_accept_draft_kernel<2, false, 2, true>}, {cb_accept_draft_kernel<2, true, 2, false>, cb_accept_draft_kernel<2, true, 2, true>}},
        {{cb_accept_draft_kernel<1, false, 2, false>, cb_accept_draft_kernel<1, false, 2, true>}, {cb_accept_draft_kernel<1, true, 2, false>, cb_accept_draft_kernel<1, true, 2, true>}},
        {{cb_accept_draft_kernel<1, false, 4, false>, cb_accept_draft_kernel<1, false, 4, true>}, {cb_accept_draft_kernel<1, true, 4, false>, cb_accept_draft_kernel<1, true, 4, true>}}};
    const int form = FCmax > 32 ? 0 : resident ? 1 : 2, in_place = a->next_n_nodes == a->n_nodes ? 1 : 0;
    const Kernel kernel = kernels[form][bf][in_place];
    {
        static std::mutex mu;
        static size_t have[64][3][2][2] = {};                  // per device and kernel
        std::lock_guard<std::mutex> lock(mu);
        CB_CUDA(cb_allow_smem(kernel, smem, &have[ctx->device & 63][form][bf][in_place]));
    }
    CbTables tf = {};
    if (ctx->has_frozen) tf = ctx->frozen;
    CB_CUDA(cb_launch_pdl(kernel, dim3(cpr, T, c.batch), dim3(256), smem, (cudaStream_t)stream, aa, ctx->tables, tf, T, c.crt, c.max_depth, NL, KF,
                          a->tokens, a->row_stride, a->seq_len, a->next_tokens, a->next_parent, a->next_depth, a->next_mask, a->next_n_nodes,
                          ctx->d_status, ctx->d_counters));
    cb_count_launch(1);
    return CB_OK;
}

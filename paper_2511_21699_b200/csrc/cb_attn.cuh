// Tree attention: work decomposition shared by the tensor-core kernels and the merge pass.
//
// Work is measured in key tiles of 128 keys.  Sequence b has tiles_b = ceil(ctx_b / 128) + 1 of them (the
// last one holds the tree's own keys).  A unit is one (sequence, kv head, row group): a row group is a
// pair of 128-row tiles (row = node_local * G + g, NPT = 128 / G nodes per tile), or a single tile when
// the whole tree fits one tile; only row tiles that hold valid nodes form units.  All units laid end to end give one
// global sequence of key tiles; it is cut into `nc` equal ranges, one per persistent CTA (or CTA pair): a stream-K split.
// The order of the units is (row group, sequence, kv head), row group outermost: the units that stream the same keys and
// values (one (sequence, kv head), all its row groups) then lie a fixed fraction of the whole sequence apart, so that they
// are worked on at the same time by different CTAs and the keys and values are fetched from HBM once and found in L2 by
// the others; with the row group innermost one CTA would stream them again and again, each time after everything else
// it holds has passed through L2.  A key tile of a unit with two row tiles takes longer than one of a unit with one, so a tile counts w2
// or w1 positions of the sequence: 2 and 1 with head_dim 64, where the softmax chains decide (two chains share the tiles of a unit with
// one row tile; batch 13 of small trees: 47 us at 1 : 1, 43 at 3 : 2, 40 at 2 : 1, 43 at 5 : 2), 6 and 4 with head_dim 128, where the
// copies of a tile weigh as much (ragged trees, 3 : 2 against 2 : 1: batch 30 58.7 against 65.7 us, batch 90 of short trees 135 against
// 156, batch 8 of 64 heads 90 against 99, batch 20 61.0 against 62.8; 4 : 3 is 4% faster still on two of twelve shapes and 2% slower on three).
// Starting a
// unit costs about as much as two or three tiles (query load, pipeline refill, epilogue), so every unit is preceded by that many
// padding positions: they carry no work, they only make a CTA that handles many short units receive fewer tiles.  A tile
// belongs to the CTA whose range holds the tile's deciding position, its d1-th or d2-th from zero.  Those are the first one at 2 : 1, and at
// 6 : 4 the ones that cut a launch whose units have all one row tile, or all two, exactly as 2 : 1 cuts it: a range that starts at
// the share x of the sequence leaves out the tiles i with 2x >= 2i + 1 (two) or x >= i + 1 (one), which is 6x >= 6i + 3 and 4x >= 4i + 4.
// Where a launch is cut decides the last bits of rows: of a unit that CTAs share (its parts are put together), and of a whole unit of one row
// tile, whose keys one chain takes where the range holds the next head's whole unit as well (CbWalker::next_pair), else two chains in turn.  The cuts
// follow from the lengths and node counts of the whole batch; equal calls give equal bits.
// A CTA therefore finishes whole units, plus at most one unit it shares
// with earlier CTAs and one it shares with later CTAs; the CTAs of a shared unit combine unnormalised partials (in the kernel, or
// in the merge pass of the CTA-pair kernel, which counts one position per tile).
#pragma once
#include "cb_common.cuh"

#define CB_KT 128        // keys per tile
#define CB_MT 128        // query rows per tile

struct CbAttnParams {
    const __nv_bfloat16* q;
    const __nv_bfloat16* k_pool;
    const __nv_bfloat16* v_pool;
    const int32_t* block_table;
    const int32_t* ctx_len;
    const __nv_bfloat16* k_tree;
    const __nv_bfloat16* v_tree;
    const uint32_t* tree_mask;
    const int32_t* n_nodes;
    __nv_bfloat16* out;
    float* lse;
    float* part;          // [2 * nc slots] of 2 * 128 * (D + 4) floats: unnormalised output columns, running max (log2 domain), sum
    uint32_t* part_ticket; // [2 sets][CB_ATTN_MAX_CTAS][16 softmax warps]: parts of a shared unit left in memory so far
    uint32_t* part_turn;  // [0] launches of the context so far: the lowest bit names the set in use; [1] CTAs of this one that have left
    int B, T, W, Hq, Hkv, G, D, P, max_pages, num_pages;
    int NPT;              // tree nodes per row tile = 128 / G
    uint32_t npt_inv;     // x / NPT = x * npt_inv >> 16 for x < 256
    uint32_t g_inv;       // x / G = x * g_inv >> 16 for x < 256
    int MT;               // row tiles that T nodes need = ceil(T / NPT)
    int nc;               // persistent CTAs (= ranges of the global tile sequence)
    int w1, w2;           // positions that a key tile of a unit with one or with two row tiles counts
    int d1, d2;           // which of them decides whose tile it is
    int max_tiles;        // host's upper bound on the key tiles of a unit (from max_ctx, else from the block table's width)
    int cs;               // > 0: cluster mode, one unit per cluster of cs CTAs (see cb_attn_tc.cu); 0: the stream-K split
    float scale_log2;     // softmax scale * log2(e)
    uint32_t* status;
};

// The weights of the persistent CTAs' split (see above).
inline void cb_attn_weights(CbAttnParams& p) {
    if (p.D == 128) { p.w1 = 4; p.w2 = 6; p.d1 = 3; p.d2 = 2; }
    else { p.w1 = 1; p.w2 = 2; p.d1 = p.d2 = 0; }
}

// Per-sequence shape of the decomposition.
struct CbSeqShape {
    int n, ctx, tiles, mtn, RG;
    int w1, w2, d1, d2;
    bool one;             // the launch has one row tile per unit throughout
    long long W;          // positions (padding + key tiles) of all units of this sequence
    __device__ __forceinline__ bool two_rows(int rg) const { return !one && mtn - 2 * rg >= 2; }
    __device__ __forceinline__ int wt(int rg) const { return two_rows(rg) ? w2 : w1; }              // positions per key tile
    __device__ __forceinline__ int ov(int rg) const { return two_rows(rg) ? 3 * w2 : 2 * w1; }      // padding positions in front of a unit
    __device__ __forceinline__ int unit(int rg) const { return tiles * wt(rg) + ov(rg); }           // positions of one unit
    __device__ __forceinline__ int dec(int rg) const { return ov(rg) + (two_rows(rg) ? d2 : d1); }  // deciding position of a unit's first tile
    // positions of this sequence's units of row group rg (all kv heads); 0 if the tree has no such row group
    __device__ __forceinline__ long long w_of(int Hkv, int rg) const { return rg < RG ? (long long)Hkv * unit(rg) : 0ll; }
};

__device__ __forceinline__ CbSeqShape cb_seq_shape(const CbAttnParams& p, int b) {
    CbSeqShape s;
    s.n = min(max(p.n_nodes[b], 0), p.T);
    s.ctx = min(max(p.ctx_len[b], 0), p.max_pages * p.P);
    s.tiles = (s.ctx + CB_KT - 1) / CB_KT + 1;
    s.mtn = (int)(((uint32_t)(s.n + p.NPT - 1) * p.npt_inv) >> 16);
    s.one = p.MT == 1;
    s.RG = s.one ? (s.mtn > 0 ? 1 : 0) : (s.mtn + 1) / 2;
    s.w1 = p.w1; s.w2 = p.w2; s.d1 = p.d1; s.d2 = p.d2;
    // every row group but the last has two row tiles
    s.W = s.RG > 0 ? (long long)p.Hkv * ((long long)(s.RG - 1) * s.unit(0) + s.unit(s.RG - 1)) : 0;
    return s;
}

// a / b for a >= 0, b > 0: 32 bits wide where that does (the 64-bit division is some 100 instructions, four of them in a row at
// the start of every CTA).
__device__ __forceinline__ long long cb_div(long long a, long long b) {
    return ((unsigned long long)a | (unsigned long long)b) >> 32 ? a / b : (long long)((uint32_t)a / (uint32_t)b);
}
// a / b for a >= 0 and 0 < b < 2^22.  A division is a chain of some 200 cycles, and the first copy of a launch waited for five of
// them (batch 13, head_dim 64: 2.3 k cycles from the schedule to the block table's entry); small numbers are divided in fp32, exactly.
__device__ __forceinline__ long long cb_quot(long long a, int b) {
    if (a < (1ll << 22)) {
        const int x = (int)a;
        int q = (int)__fdividef((float)x, (float)b);
        const int r = x - q * b;
        q += r < 0 ? -1 : (r >= b ? 1 : 0);
        return q;
    }
    return cb_div(a, b);
}
__device__ __forceinline__ long long cb_range_start(long long total, int nc, int c) { return cb_quot(total * c, nc); }
// CTA whose range holds position x.
__device__ __forceinline__ int cb_cta_of(long long total, int nc, long long x) {
    const long long at = (x + 1) * nc - 1;
    return (int)(total < (1ll << 22) ? cb_quot(at, (int)total) : cb_div(at, total));
}

// Row groups a launch can have per sequence (trees of max_nodes nodes).
__device__ __forceinline__ int cb_max_row_groups(const CbAttnParams& p) { return p.MT == 1 ? 1 : (p.MT + 1) / 2; }

// Warp-collective: total weight of all sequences, and the (row group, sequence) holding global position g (with the
// global index at which that sequence's units of that row group start).  Every lane gets the results.
// max_row_tiles (optional): the largest number of row tiles that any sequence's tree has.
__device__ __forceinline__ long long cb_sched_total(const CbAttnParams& p, int lane, int* max_row_tiles = nullptr) {
    long long tot = 0;
    int mt = 0;
    for (int base = 0; base < p.B; base += 32) {
        const int b = base + lane;
        CbSeqShape s = {};
        if (b < p.B) s = cb_seq_shape(p, b);
        long long w = b < p.B ? s.W : 0;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) w += __shfl_xor_sync(CB_FULL, w, o);
        tot += w;
        mt = max(mt, b < p.B ? s.mtn : 0);
    }
    if (max_row_tiles) *max_row_tiles = __reduce_max_sync(CB_FULL, mt);
    return tot;
}
__device__ __forceinline__ void cb_sched_locate(const CbAttnParams& p, long long g, int lane, int* rg_out, int* b_out, long long* pre_out) {
    long long run = 0;
    int frg = cb_max_row_groups(p), fb = p.B;
    long long fpre = 0;
    for (int rg = 0; rg < cb_max_row_groups(p) && fb == p.B; ++rg) {
        for (int base = 0; base < p.B; base += 32) {
            const int b = base + lane;
            const long long w = b < p.B ? cb_seq_shape(p, b).w_of(p.Hkv, rg) : 0;
            long long inc = w;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const long long t = __shfl_up_sync(CB_FULL, inc, o);
                if (lane >= o) inc += t;
            }
            const long long pre = run + inc - w;
            const uint32_t hit = __ballot_sync(CB_FULL, w > 0 && g >= pre && g < pre + w);
            if (hit) {
                const int l = __ffs(hit) - 1;
                frg = rg;
                fb = base + l;
                fpre = __shfl_sync(CB_FULL, pre, l);
                break;
            }
            run += __shfl_sync(CB_FULL, inc, 31);
        }
    }
    *rg_out = frg;
    *b_out = fb;
    *pre_out = fpre;
}

// One unit's share of a CTA's range: key tiles [t0, t1) of the unit's `tiles`.
struct CbUnit {
    int b, kh, rg, t0, t1, tiles, n, ctx, nrt;   // nrt = valid row tiles in the group (1 or 2), or kTwoHeads
};
constexpr int kTwoHeads = 3;                     // the units of heads kh and kh + 1, both whole and of one row tile, side by side (next_pair)

// x / wt for the weights that there are (1, 2, 4 and 6) and x >= 0: a division is a chain of 100 to 200 cycles, two of them in the first unit.
__device__ __forceinline__ int cb_tiles_of(int x, int wt) {
    return wt == 6 ? (int)((unsigned long long)(uint32_t)x * 0xAAAAAAABull >> 34) : x >> (wt >> 1);
}

// Walks the units of the range [g, g1).  Every role that walks runs its own copy and sees the same units.
struct CbWalker {
    long long g, g1, pre;     // pre: global position at which the units of (rg, b) start
    int rg, b;
    long long w;              // positions of the units of (rg, b)
    CbSeqShape s;
    bool fixed, fixed_left;   // cluster mode: the CTA has exactly one share of one unit (or none)
    CbUnit fu;
    __device__ __forceinline__ void init(const CbAttnParams& p, long long g0, long long g1_, int rg0, int b0, long long pre0) {
        g = g0; g1 = g1_; rg = rg0; b = b0; pre = pre0; fixed = false; fixed_left = false; w = 0;
        if (g < g1) { s = cb_seq_shape(p, b); w = s.w_of(p.Hkv, rg); }
    }
    __device__ __forceinline__ void init_fixed(const CbUnit& u0) {
        g = 0; g1 = 0; rg = 0; b = 0; pre = 0; w = 0; fixed = true; fixed_left = u0.t1 > u0.t0; fu = u0;
    }
    __device__ __forceinline__ bool next(const CbAttnParams& p, CbUnit* u) {
        if (fixed) {
            if (!fixed_left) return false;
            fixed_left = false;
            *u = fu;
            return true;
        }
        while (true) {
            if (g >= g1) return false;
            while (g >= pre + w) {                            // on to the next sequence that has this row group, then to the next row group
                pre += w;
                if (++b == p.B) { b = 0; ++rg; }
                s = cb_seq_shape(p, b);
                w = s.w_of(p.Hkv, rg);
            }
            // Integer divisions here, not cb_quot: this code stands in every role's loop, and what decides is what it makes the compiler do
            // with the roles' registers (with cb_quot: batch 39 of 40 heads over 220 tokens 82.1 us, so 74.8; batch 103 of 64 heads over 300
            // 154 and 135; batch 81 of 40 heads over 500 241 and 232.  Without any division but more state kept between two units: 76.8, 136, 239).
            const long long off = g - pre;
            const int vt = s.unit(rg), wt = s.wt(rg), dec = s.dec(rg);
            const int kh = (int)cb_div(off, vt);
            const int v0 = (int)(off - (long long)kh * vt);
            const int v1 = (int)min((long long)vt, (long long)v0 + (g1 - g));
            g += v1 - v0;
            u->t0 = cb_tiles_of(max(v0 - dec, 0) + wt - 1, wt);
            u->t1 = cb_tiles_of(max(v1 - dec, 0) + wt - 1, wt);
            if (u->t1 <= u->t0) continue;                     // no tile of this unit is the range's
            u->b = b; u->kh = kh; u->rg = rg; u->tiles = s.tiles; u->n = s.n; u->ctx = s.ctx;
            u->nrt = p.MT == 1 ? 1 : min(2, s.mtn - 2 * rg);
            return true;
        }
    }
    // The same with two whole units of one row tile at a time where the range holds the next head's as well.
    __device__ __forceinline__ bool next_pair(const CbAttnParams& p, CbUnit* u) {
        if (!next(p, u)) return false;
        if (fixed || u->nrt != 1 || u->t0 > 0 || u->t1 < u->tiles || u->kh + 1 >= p.Hkv) return true;
        const long long end = pre + (long long)(u->kh + 2) * s.unit(rg);                    // of the next head's unit
        const int last = (u->tiles - 1) * s.wt(rg) + s.dec(rg) - s.unit(rg);                // its last tile's deciding position, from there
        if (end + last >= g1) return true;
        g = min(end, g1);
        u->nrt = kTwoHeads;
        return true;
    }
};

#define CB_ATTN_MAX_CTAS 160   // upper bound on persistent CTAs (>= SM count); sizes the partial buffer
static_assert(CB_ATTN_MAX_UNITS == 4 * CB_ATTN_MAX_CTAS, "partial buffer: two shared units of two row tiles per CTA");

cb_status cb_attn_launch_cuda_cores(cb_ctx* ctx, const CbAttnParams& p, cudaStream_t st);
cb_status cb_attn_launch_tensor(cb_ctx* ctx, const CbAttnParams& p, cudaStream_t st);

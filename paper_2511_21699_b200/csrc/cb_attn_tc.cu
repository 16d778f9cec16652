// Tree-masked attention on the 5th-generation tensor cores (tcgen05) with TMA-staged paged K/V.
//
// Persistent kernel: one CTA per SM, each working through an equal share of the global sequence of key
// tiles (see cb_attn.cuh).  A CTA holds up to two 128-row query tiles of a unit and streams that unit's
// 128-key tiles through a ring of 128B-swizzled shared-memory slots (K and V tiles alternate in the
// ring; eight 16-token pages per tile, fetched page by page with TMA through the block table).
//
// What bounds it is the chain of a score tile, S = Q K^T -> softmax -> O += P V -> next S (P overlays S in TMEM, so the next S
// follows the product that reads P), against 1,024 cycles of tensor work (16 products of 64 cycles) and 1,024 of the exponential
// unit per 128 x 128 tile.  Two chains run side by side so that one is in the tensor pipe while the other is in softmax; each
// has an S/P buffer, an accumulator and a pair of softmax warpgroups of its own:
//   * a unit with two row tiles gives each chain a row tile, and both walk all key tiles;
//   * a unit with one row tile deals its key tiles to the two chains in turn; every chain keeps its own reference maximum and
//     accumulator and the two are put together at the end of the unit.
//   * where a range holds two heads' whole units of one row tile, they are taken together, a chain each with a query tile of its own: the
//     key tiles come in turn as before, but nothing is put together at the end, and what lies between two units (query load, refill,
//     epilogue; some 12 k cycles of a unit of two tiles) is paid once for both.  Batch 69 of 40 heads over 10 to 77 tokens 124 -> 91 us,
//     batch 128 of 32 heads (64 dims) over 65 tokens 141 -> 103, 28 x 8 heads of 110-node trees over 377 tokens 91.8 -> 80.2, batch 64 of 40
//     heads over 2,048 tokens 463 -> 455.
// A row's 128 scores are split over two threads (64 each): one warp per scheduler and chain left half of the issue slots empty
// (2.1 k cycles a tile with a row per thread, spills included).
//
// Warp roles (640 threads, five warpgroups):
//   warp 0        TMA producer for the K tiles: runs ahead across unit boundaries, limited only by the ring
//   warp 1        MMA issuer (one elected lane): O += P V of a chain, with P read from TMEM, then the chain's next S = Q K^T;
//                 the chains take turns, so that their products do not interleave in the tensor pipe (with a thread per chain they
//                 did: both chains ended together and then went through softmax together); owns the TMEM allocation (S0, S1, O0, O1)
//   warp 2        publishes the units to the softmax warps and loads their query tiles
//   warp 3        TMA producer for the V tiles
//   warps 4..19   softmax warpgroups: 4..7 and 8..11 chain 0 (keys 0-63 and 64-127 of a tile), 12..15 and 16..19 chain 1;
//                 fp32 online softmax in the log2 domain with lazy rescaling of O, P written back to TMEM as packed bf16 over S;
//                 epilogue of the unit.  Before that they write the zero rows of padding nodes (node >= n_nodes).
// All waits are bounded; a wait that runs out records CB_ERR_TIMEOUT and the CTA drains and exits.
//
// Cluster mode.  When a launch has so few units that the split above would make every unit a shared one (batch 1), the
// kernel is launched as thread-block clusters instead: cluster k works on unit k, its CTAs take equal parts of the unit's
// key tiles, and at the end they combine their shares through distributed shared memory: every CTA gathers D / cs columns of
// all rows, merges the contributions and writes the output.  No partials go to HBM.
#include <cuda.h>

#include <mutex>
#include <type_traits>

#include "cb_attn_sched32.cuh"
#include "cb_tc_dev.cuh"

namespace {

// A unit as the softmax warps see it (nrt = 0: no more units).  cf, np: the CTA that holds the unit's first key tile and the number of
// CTAs that hold one; ticket: where its parts are counted; xpos: position of that tile where a CTA holds one tile at most, else -1.
struct UnitDesc { int b, kh, rg, t0, t1, tiles, n, ctx, nrt, cf, np, xpos, wt, ticket; };
constexpr int kUnitRing = 4;                                 // units published ahead of the slowest softmax thread: at most two

template <int D>
struct Cfg {
    static constexpr int DB = D / 64;                        // 64-element (128-byte) column blocks per row
    static constexpr int NSLOT = (D == 128) ? 5 : 8;         // ring slots, each one K or one V tile
    static constexpr uint32_t TILE_BYTES = CB_KT * D * 2;    // one K or V tile
    static constexpr uint32_t Q_BYTES = CB_MT * D * 2;       // one query row tile
    static constexpr uint32_t OFF_Q = 0;                     // two row tiles
    static constexpr uint32_t OFF_RING = 2 * Q_BYTES;
    static constexpr uint32_t OFF_BAR = OFF_RING + NSLOT * TILE_BYTES;
    // slot_full[NSLOT], slot_free[NSLOT], q_full, q_free, s_full[2], p_ready[2], o_done[2], o_done_both, o_free[2], sums,
    // unit_full[kUnitRing], cluster_ready, cluster_data
    static constexpr int NBAR = 2 * NSLOT + 12 + kUnitRing + 2;
    static constexpr uint32_t OFF_UNITS = OFF_BAR + NBAR * 8;
    static constexpr uint32_t OFF_X = OFF_UNITS + kUnitRing * sizeof(UnitDesc);      // [2 chains][2][128 rows]: row sums, then reference and sum
    static constexpr uint32_t OFF_MISC = OFF_X + 2 * 2 * CB_MT * 4;                  // schedule, tmem base, abort flag, pair counters
    static constexpr uint32_t SMEM = OFF_MISC + 96 + 64;
    static_assert(SMEM <= 227 * 1024, "shared memory of one CTA");
    // Of so many pairs of exponentials the last is taken by the FMA pipe.  With head_dim 64, whose products take half as long, the exponential
    // unit decides, and a quarter off it is worth 1 to 4% (batch 85 of 32/8 heads over 1,283 tokens: 60.1 us without, 58.6 an eighth,
    // 57.8 a quarter).  With 128 the chains' hand-overs decide and the polynomial's 17 instructions are mostly power.  Runs of 2 s at the
    // power cap, four in turn, a quarter / an eighth / none: 70B shape, batch 128 18.69 / 18.49 / 18.46 ms; batch 8 of it over 4 k to 16 k tokens
    // 347.2 / 343.9 / 345.4 us; batch 64 of 40 heads 473.9 / 470.0 / 469.0; batch 32 of 32/8 heads 184.6 / 183.7 / 184.1.  None is as good as an
    // eighth within half a percent either way, a quarter is slower in all.
    static constexpr int FMA_EXP = (D == 128) ? 8 : 4;
    static constexpr uint32_t O_COL = 256;                   // TMEM columns: S0 at 0, S1 at 128, O0 at 256, O1 at 256 + D
};

struct SchedSmem { long long g0, g1, pre0; int b0, rg0; int c_b, c_kh, c_n, c_has; };   // c_*: cluster mode
static_assert(sizeof(SchedSmem) <= 64, "the schedule block is followed by the tmem base and the abort flag");

}  // namespace

#include "cb_attn_pair.cuh"

namespace {

// What a CTA of a cluster receives: from every source CTA the columns it owns, in groups of 4 (16 bytes), the rows of a group side
// by side (one more than there are, so that reading along the groups meets no bank twice), then every row's reference and sum.
struct CbExchange {
    int rows;              // rows of the unit's tree, in whole warps
    uint32_t bytes;        // room for them
    __device__ __forceinline__ uint32_t expected(int cs, int D) const { return (uint32_t)(rows * (D * 4 + cs * 8)); }   // bytes that arrive
    __device__ __forceinline__ uint32_t value(int src, int ch, int row, int nch) const { return (uint32_t)(((src * nch + ch) * (rows + 1) + row) * 16); }
    __device__ __forceinline__ uint32_t sums(int src, int row, int cs, int nch) const { return (uint32_t)(cs * nch * (rows + 1) * 16 + (src * rows + row) * 8); }
};
__device__ __forceinline__ CbExchange cb_exchange(const CbAttnParams& p, int D, int n) {
    CbExchange e;
    e.rows = (min(p.NPT, n) * p.G + 31) & ~31;
    e.bytes = (uint32_t)(D / 4 * (e.rows + 1) * 16 + p.cs * e.rows * 8);
    return e;
}

template <int D>
__global__ void __launch_bounds__(kThreads, 1)
cb_attn_tc_kernel(const CbAttnParams p, const __grid_constant__ TcMaps maps) {
    using C = Cfg<D>;
    extern __shared__ __align__(1024) uint8_t attn_smem[];
    uint8_t* const sgen = attn_smem;
    const uint32_t sbase = smem_u32(attn_smem);
    if (sbase & 1023u) {                                      // the swizzled tiles need it; every thread sees the same address
        if (threadIdx.x == 0) atomicCAS(p.status, 0u, (uint32_t)CB_ERR_UNSUPPORTED);
        return;
    }
    const uint32_t bar0 = sbase + C::OFF_BAR;
    auto bar_full = [&](uint32_t s) { return bar0 + 8u * s; };
    auto bar_free = [&](uint32_t s) { return bar0 + 8u * (C::NSLOT + s); };
    auto slot_base = [&](uint32_t s) { return sbase + C::OFF_RING + s * C::TILE_BYTES; };
    constexpr uint32_t B1 = 2 * C::NSLOT;
    const uint32_t bar_qfull = bar0 + 8u * B1, bar_qfree = bar_qfull + 8u;
    auto bar_sfull = [&](int l) { return bar0 + 8u * (B1 + 2 + l); };
    auto bar_pready = [&](int l) { return bar0 + 8u * (B1 + 4 + l); };
    auto bar_odone = [&](int l) { return bar0 + 8u * (B1 + 6 + l); };
    const uint32_t bar_odone_both = bar0 + 8u * (B1 + 8);
    auto bar_ofree = [&](int l) { return bar0 + 8u * (B1 + 9 + l); };
    const uint32_t bar_sums = bar0 + 8u * (B1 + 11);
    auto bar_ufull = [&](uint32_t k) { return bar0 + 8u * (B1 + 12 + k); };
    const uint32_t bar_cready = bar0 + 8u * (B1 + 12 + kUnitRing), bar_cdata = bar_cready + 8u;   // cluster mode only
    UnitDesc* s_units = reinterpret_cast<UnitDesc*>(sgen + C::OFF_UNITS);
    volatile float* s_x = reinterpret_cast<volatile float*>(sgen + C::OFF_X);
    SchedSmem* s_sched = reinterpret_cast<SchedSmem*>(sgen + C::OFF_MISC);
    uint32_t* s_tmem = reinterpret_cast<uint32_t*>(sgen + C::OFF_MISC + 64);
    volatile int* s_abort = reinterpret_cast<volatile int*>(sgen + C::OFF_MISC + 68);
    long long* s_tot = reinterpret_cast<long long*>(sgen + C::OFF_MISC + 72);   // positions of the global tile sequence
    volatile int* s_pair = reinterpret_cast<volatile int*>(sgen + C::OFF_MISC + 96);   // [16 softmax warps]: last pair barrier entered, -1 = left

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int cta = blockIdx.x;
    const int RT = p.NPT * p.G;                               // rows of a row tile that exist
    // Set-up that reads no input (TMEM allocation, barrier initialisation, descriptor prefetch) runs before the wait for the
    // kernels earlier in the stream, so it overlaps their tail.  The next kernel of a step is launched as a programmatic dependent in
    // turn: its blocks may take the SMs that this grid's CTAs leave and do their set-up there.
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(s_tmem)), "r"(kTmemCols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    } else if (warp == 2) {
        if (lane == 0) {
            for (int s = 0; s < C::NSLOT; ++s) { mbar_init(bar_full(s), 1); mbar_init(bar_free(s), 1); }
            mbar_init(bar_qfull, 1); mbar_init(bar_qfree, 1);
            for (int l = 0; l < 2; ++l) {
                mbar_init(bar_sfull(l), 1); mbar_init(bar_pready(l), 256);
                mbar_init(bar_odone(l), 1); mbar_init(bar_ofree(l), 512);
            }
            mbar_init(bar_odone_both, 1); mbar_init(bar_sums, 512);
            for (int k = 0; k < kUnitRing; ++k) mbar_init(bar_ufull(k), 1);
            mbar_init(bar_cready, p.cs > 0 ? (uint32_t)p.cs : 1u); mbar_init(bar_cdata, 1);
            *s_abort = 0;
            s_sched->c_has = 0;
            asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
            tma_prefetch_desc(&maps.k_pool); tma_prefetch_desc(&maps.v_pool); tma_prefetch_desc(&maps.q);
            tma_prefetch_desc(&maps.k_tree); tma_prefetch_desc(&maps.v_tree);
        }
        if (lane < 16) s_pair[lane] = 0;
    }
    CB_PDL_ENTRY();
    // The set of tickets that this launch counts in.  The other one is cleared for the next launch, so that it finds zeros even
    // where the launch before this one gave up on a wait and left counts half way, whatever the status word says.
    int ticket_set = 0;
    if (warp == 2 && p.cs == 0) {
        ticket_set = (int)(*reinterpret_cast<volatile uint32_t*>(p.part_turn) & 1u) * CB_ATTN_TICKETS;
        if (lane < 16) p.part_ticket[CB_ATTN_TICKETS - ticket_set + cta * 16 + lane] = 0u;
    }
    if (warp == 3 && p.cs == 0) {
        // The block table into L2, a slice per CTA: the first copies' addresses come from it, and which part of it a CTA needs is
        // known only after the schedule below (two memory round trips one after the other otherwise).
        const long long lines = ((long long)p.B * p.max_pages * 4 + 127) / 128;
        for (long long k = (long long)cta * 32 + lane, n = 0; k < lines && n < 4; k += (long long)gridDim.x * 32, ++n)
            asm volatile("prefetch.global.L2 [%0];" ::"l"(reinterpret_cast<const char*>(p.block_table) + k * 128));
    }

    if (p.cs == 0 && warp == 0) {
        // this CTA's range of the global tile sequence
        long long tot, g0, g1, pre0 = 0;
        int b0 = 0, rg0 = 0;
        if (!cb_sched_of_32(p, cta, lane, &tot, &g0, &g1, &rg0, &b0, &pre0)) {
            tot = cb_sched_total(p, lane);
            g0 = cb_range_start(tot, p.nc, cta); g1 = cb_range_start(tot, p.nc, cta + 1);
            if (g0 < g1) cb_sched_locate(p, g0, lane, &rg0, &b0, &pre0);
        }
        if (lane == 0) { s_sched->g0 = g0; s_sched->g1 = g1; s_sched->b0 = b0; s_sched->rg0 = rg0; s_sched->pre0 = pre0; *s_tot = tot; }
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *s_tmem;
    constexpr uint32_t ns = (uint32_t)C::NSLOT;
    // Cluster mode: the peers' barriers must exist before anything arrives on them.  Every thread reports here and waits where its
    // role first reaches over, or at its end (a CTA must not leave before the others' report either).
    // What the peers must see of this CTA, its initialised barriers and nothing else, went out with the fence behind the initialisation, so the
    // report itself releases nothing (a releasing one waits for every access before it: 0.9 k of the cycles before batch 1's first copy).
    // What else was written before it (c_has, the abort flag) is for this CTA's threads, behind the block's barriers.
    if (p.cs > 0) asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
    auto cluster_wait = [&]() {
        if (p.cs > 0) asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
    };

    if (warp < 4) {
        reg_dealloc<64>();
        CbWalker wk;
        // Cluster mode: cluster k works on unit k = (sequence, kv head); its CTAs take equal parts of the unit's key tiles.  Every role works its
        // share out for itself (through one warp and shared memory, with divisions by the cluster size, batch 1 took 18.9 us, so 18.2).
        if (p.cs > 0) {
            const int lcs = 31 - __clz(p.cs);                 // the cluster size is a power of two
            const int uid = cta >> lcs, rank = cta & (p.cs - 1), b = uid / p.Hkv;
            int guess = -1, page_guess = 0;                   // a tile, and the page of this lane's box in it
            if ((warp == 0 || warp == 3) && lane < 8) {
                // The first tile if the context is as long as the caller's bound: its page is asked for beside the lengths that say whether it is
                // (one memory round trip instead of two).
                guess = (int)((long long)p.max_tiles * rank >> lcs);
                const long long at = (long long)guess * (CB_KT / 16) + lane;
                if (at < p.max_pages) page_guess = p.block_table[(size_t)b * p.max_pages + at];
            }
            const CbSeqShape sh = cb_seq_shape(p, b);
            CbUnit u0;
            u0.b = b; u0.kh = uid - b * p.Hkv; u0.rg = 0; u0.tiles = sh.tiles; u0.n = sh.n; u0.ctx = sh.ctx; u0.nrt = 1;
            u0.t0 = sh.RG > 0 ? (int)((long long)sh.tiles * rank >> lcs) : 0;
            u0.t1 = sh.RG > 0 ? (int)((long long)sh.tiles * (rank + 1) >> lcs) : 0;
            wk.init_fixed(u0);
            wk.rg = guess; wk.b = page_guess;                 // (a fixed walk has no use for them)
            if (warp == 2 && lane == 0) {
                // read by the softmax warps, behind the barrier on which the unit is published
                s_sched->c_b = b; s_sched->c_kh = u0.kh; s_sched->c_n = sh.n; s_sched->c_has = sh.RG > 0 ? 1 : 0;
            }
        } else if (warp != 1) {                               // (the issuer reads the published units)
            wk.init(p, s_sched->g0, s_sched->g1, s_sched->rg0, s_sched->b0, s_sched->pre0);
        }
        CbUnit u;
        if (warp == 0 || warp == 3) {
            // ------------------------------------------------------------------ K/V producers: warp 0 the K tiles, warp 3 the V tiles
            // A page's 16 keys are one box, laid out in shared memory as groups of 8 keys with a group's 64-dim column blocks
            // behind one another (which is why the products' descriptors step by 1024 * DB from group to group).  The copies of
            // a warp instruction are issued one after the other, some 80 cycles each: eight a tile, and the two tiles of a key
            // tile by a warp each.  The tree's own keys are boxes of 8 rows (max_nodes need not be a multiple of 16).
            const bool isV = warp == 3;
            constexpr uint32_t GROUP = 1024 * C::DB;         // bytes of 8 keys
            const bool active = lane < 8;
            const int j = lane % 8;
            uint32_t seq = isV ? 1u : 0u;                    // K and V tiles alternate in the ring
            bool ok = true;
            const uint64_t pol = l2_evict_first_policy();
            while (ok && wk.next_pair(p, &u)) {
                const int npages = (u.ctx + 15) / 16, nct = u.tiles - 1;   // pages of 16 tokens (checked by the launcher)
                const int heads = u.nrt == kTwoHeads ? 2 : 1;              // their tiles come in turn
                const int32_t* bt = p.block_table + (size_t)u.b * p.max_pages;
                // The page number of a lane's box comes from the block table: a memory round trip that the copy depends on.
                // It is fetched one tile ahead, so that it is under way while this tile's copies are issued and waited for.
                auto page_of = [&](int i) {
                    int page = p.num_pages;                  // out of range: the copy fills zeros
                    if (active && i < nct) {
                        const int pidx = i * (CB_KT / 16) + j;
                        if (pidx < npages) page = wk.fixed && i == wk.rg ? wk.b : bt[pidx];
                    }
                    return page;
                };
                int page_next = page_of(u.t0);
                for (int i = u.t0; i < u.t1; ++i) {
                    int page = page_next;
                    if (i + 1 < u.t1) page_next = page_of(i + 1);
                    if (!cb_dbg_in(page, p.num_pages + 1, p.status)) page = p.num_pages;   // the copy then fills zeros
                    for (int hd = 0; hd < heads; ++hd) {
                        const uint32_t sl = seq % ns;
                        if (seq >= ns && !(ok = mbar_wait(bar_free(sl), (seq / ns - 1) & 1, s_abort, p.status))) break;
                        if (lane == 0) mbar_expect_tx(bar_full(sl), C::TILE_BYTES);
                        __syncwarp();
                        if (i < nct) {
                            if (active) tma_load_5d_hint(slot_base(sl) + j * 2 * GROUP, isV ? &maps.v_pool : &maps.k_pool, bar_full(sl), 0, 0, 0, page * 2, u.kh + hd, pol);
                        } else if (lane < 16) {
                            tma_load_5d(slot_base(sl) + lane * GROUP, isV ? &maps.v_tree : &maps.k_tree, bar_full(sl), 0, 8 * lane, 0, u.kh + hd, u.b);
                        }
                        seq += 2;
                    }
                    if (!ok) break;
                }
            }
        } else if (warp == 1) {
            // ------------------------------------------------------------------ MMA issuer
            if (elect_one()) {
                constexpr uint32_t idesc_s = make_idesc(128, CB_KT, false);
                constexpr uint32_t idesc_o = make_idesc(128, D, true);
                uint32_t seq0 = 0, uq = 0, c_p[2] = {0u, 0u};
                bool ok = true;
                // It takes the units from the ring of descriptors: walking to the next one is a chain of some 2 k cycles, which short
                // units waited for here (batch 128 of 32 heads of 64 dims over 65 tokens: 103 us, so 98).
                while ((ok = mbar_wait(bar_ufull(uq % kUnitRing), (uq / kUnitRing) & 1, s_abort, p.status))) {
                    const volatile UnitDesc* d = &s_units[uq % kUnitRing];
                    const int nrt = d->nrt;
                    if (nrt == 0) break;
                    const bool two = nrt == 2, heads = nrt == kTwoHeads;
                    const int nt = heads ? 2 * d->tiles : d->t1 - d->t0, nev = two ? 2 * nt : nt;   // products of either kind in this unit
                    if (!(ok = mbar_wait(bar_qfull, uq & 1, s_abort, p.status))) break;
                    // Turn e belongs to chain e & 1: the P V of its turn before (key tile iv), then S of this turn's key tile ik.
                    for (int e = 0; e < nev + 2; ++e) {
                        const int l = e & 1, ik = two ? e >> 1 : e, iv = two ? ik - 1 : ik - 2;
                        if (e >= 2) {
                            const uint32_t vseq = seq0 + 2u * (uint32_t)iv + 1u, vs = vseq % ns;
                            if (iv < nt) {
                                if ((!two || l == 0) && !(ok = mbar_wait(bar_full(vs), (vseq / ns) & 1, s_abort, p.status))) break;
                                // the unit before is done with this chain's accumulator; a chain without a tile of this unit takes its turn
                                // on the barrier here too: it is done with its row sums before odone_both lets it write the next ones
                                if (e < 4 && uq > 0 && !(ok = mbar_wait(bar_ofree(l), (uq - 1) & 1, s_abort, p.status))) break;
                                if (nev < 2 && uq > 0 && !(ok = mbar_wait(bar_ofree(1), (uq - 1) & 1, s_abort, p.status))) break;
                                // P last, with nothing left to compute between it and the product (over 23 shapes 1% of the call)
                                const uint32_t vdesc = desc_lo(slot_base(vs), 1024), o_at = tmem + C::O_COL + l * D, p_at = tmem + l * 128, parity = c_p[l]++ & 1;
                                if (!(ok = mbar_wait(bar_pready(l), parity, s_abort, p.status))) break;
                                tc_fence_after();
                                mma_pv_halves_block<D>(o_at, p_at, vdesc, idesc_o, e < 4 ? 0u : 1u);
                                if (!two || l == 1) tc_commit(bar_free(vs));
                                if (iv >= nt - (heads ? 2 : 1)) tc_commit(two || heads ? bar_odone(l) : bar_odone_both);
                            }
                        }
                        if (ik < nt) {
                            const uint32_t kseq = seq0 + 2u * (uint32_t)ik, ks = kseq % ns;
                            if (!two || l == 0) {
                                if (!(ok = mbar_wait(bar_full(ks), (kseq / ns) & 1, s_abort, p.status))) break;
                                tc_fence_after();
                            }
                            mma_s_grouped_block<D>(tmem + l * 128, desc_lo(sbase + C::OFF_Q + (nrt > 1 ? l : 0) * C::Q_BYTES, 16), desc_lo(slot_base(ks), 16), idesc_s);
                            tc_commit(bar_sfull(l));
                            if (!two || l == 1) {
                                tc_commit(bar_free(ks));
                                if (ik == nt - 1) tc_commit(bar_qfree);
                            }
                        }
                    }
                    if (!ok) break;
                    seq0 += 2u * (uint32_t)nt;
                    ++uq;
                }
            }
        } else {
            // ------------------------------------------------------------------ units for the softmax warps, query tiles
            uint32_t uq = 0;
            if (lane == 0) {
                bool ok = true;
                while (ok && wk.next_pair(p, &u)) {
                    volatile UnitDesc* d = &s_units[uq % kUnitRing];
                    d->b = u.b; d->kh = u.kh; d->rg = u.rg; d->t0 = u.t0; d->t1 = u.t1; d->tiles = u.tiles; d->n = u.n; d->ctx = u.ctx; d->nrt = u.nrt;
                    if (p.cs == 0 && !(u.t0 == 0 && u.t1 == u.tiles)) {
                        // a unit shared with other CTAs: who holds its first tile, and how many of them there are
                        // (ranges of at least one tile's positions: the CTAs from the first tile's to the last one's; shorter ranges
                        // hold the deciding position of one tile at most, so every tile has a CTA of its own)
                        const int wt = wk.s.wt(u.rg);
                        const long long tot = *s_tot, x0 = wk.pre + (long long)u.kh * wk.s.unit(u.rg) + wk.s.dec(u.rg);
                        const int cf = cb_cta_of(tot, p.nc, x0);
                        const bool wide = tot >= (long long)p.nc * wt;
                        d->cf = cf;
                        d->np = wide ? cb_cta_of(tot, p.nc, x0 + (long long)(u.tiles - 1) * wt) - cf + 1 : u.tiles;
                        d->xpos = wide ? -1 : (int)x0;
                        d->wt = wt;
                        d->ticket = ticket_set + cf * 16;
                    }
                    mbar_arrive(bar_ufull(uq % kUnitRing));
                    if (uq > 0 && !(ok = mbar_wait(bar_qfree, (uq - 1) & 1, s_abort, p.status))) break;
                    const int nq = min(u.nrt, 2), head = u.nrt == kTwoHeads ? 1 : 0;   // query tiles: two row tiles, or two heads' only one
                    mbar_expect_tx(bar_qfull, (uint32_t)(nq * C::DB * RT * 128));
                    for (int k = 0; k < nq; ++k)
                        for (int db = 0; db < C::DB; ++db)
                            tma_load_4d(sbase + C::OFF_Q + k * C::Q_BYTES + db * (CB_MT * 128), &maps.q, bar_qfull, db * 64, (u.kh + k * head) * p.G,
                                        (u.rg * 2 + k * (1 - head)) * p.NPT, u.b);
                    ++uq;
                }
                if (ok) {
                    s_units[uq % kUnitRing].nrt = 0;
                    mbar_arrive(bar_ufull(uq % kUnitRing));
                }
            }
            __syncwarp();
            cluster_wait();
            if (lane == 0) {
                if (p.cs > 0 && s_sched->c_has) {
                    mbar_expect_tx(bar_cdata, cb_exchange(p, D, s_sched->c_n).expected(p.cs, D));
                    // Cluster mode: the peers write their rows into this CTA's query tiles, so it reports itself ready to
                    // receive as soon as its last S product has released them (before its last P.V is done).
                    if (cb_exchange(p, D, s_sched->c_n).bytes <= 2u * C::Q_BYTES) {
                        if (uq == 0 || mbar_wait(bar_qfree, 0, s_abort, p.status))
                            for (int r = 0; r < p.cs; ++r) mbar_arrive_remote(cluster_addr(bar_cready, (uint32_t)r));
                    }
                }
            }
        }
        __syncwarp();
        if (warp != 2) cluster_wait();
    } else {
        // ---------------------------------------------------------------------- softmax / correction / epilogue
        reg_alloc<104>();
        const int sw = warp - 4, l = sw >> 3, hf = (sw >> 2) & 1;   // chain, half of the tile's keys
        const int wq = warp & 3;                              // TMEM lane quarter this warp may access
        const int row = wq * 32 + lane;
        auto node_of = [&](int r) { return (int)((uint32_t)r * p.g_inv >> 16); };   // r / G: a row is node * G + head of the group
        const uint32_t lane_addr = (uint32_t)(wq * 32) << 16;
        const int pair_id = 1 + l * 4 + wq;                   // named barrier of the two warps that share these rows
        constexpr int CW = D / 4;                             // accumulator columns handled at a time
        const bool out32 = (reinterpret_cast<uintptr_t>(p.out) & 31u) == 0;   // output rows may be written 32 bytes at a time
        {
            // rows of padding nodes (node >= n_nodes) are written as zeros while the first tiles are on their way
            const int per_row = p.Hq * D / 8;                 // 16-byte chunks per node row
            for (int idx = cta * 16 + sw; idx < p.B * p.T; idx += gridDim.x * 16) {
                const int b = idx / p.T, nd = idx % p.T;
                const int n = min(max(p.n_nodes[b], 0), p.T);
                if (nd < n) continue;
                uint4* op = reinterpret_cast<uint4*>(p.out + (size_t)idx * p.Hq * D);
                for (int k = lane; k < per_row; k += 32) op[k] = make_uint4(0, 0, 0, 0);
                if (p.lse) for (int h = lane; h < p.Hq; h += 32) p.lse[((size_t)b * p.Hq + h) * p.T + nd] = 0.f;
            }
        }
        uint32_t c_s = 0, c_od = 0, c_ob = 0, uq = 0;                 // completions consumed: S of this chain, o_done of this chain, o_done_both
        // The pair's barrier; k numbers the barriers between two tiles, so that what a warp notes before it waits only grows.
        auto pair_sync = [&](bool v, uint32_t k) {
            if (lane == 0) s_pair[sw] = (int)(4u * (c_s + uq) + k);
            return pair_or(pair_id, v);
        };
        bool ok = true;
        float x_m = -INFINITY, x_l = 0.f, x_w0 = 0.f, x_w1 = 0.f;   // one-row-tile unit: combined reference and sum, weights of O0 and O1
        bool c_share = false, x_two = false;                  // cluster mode: this CTA has a share of the unit, and of two tiles or more
        for (; ok; ++uq) {
            if (!(ok = mbar_wait(bar_ufull(uq % kUnitRing), (uq / kUnitRing) & 1, s_abort, p.status))) break;
            const volatile UnitDesc* u = &s_units[uq % kUnitRing];   // read again where it is needed: registers are short
            if (u->nrt == 0) break;
            const bool two = u->nrt > 1;                      // a chain has its own rows: a row tile, or a head's only one
            const int lr = u->nrt == 2 ? l : 0;               // row tile of the unit
            const int step = two ? 1 : 2, tfirst = u->t0 + (two ? 0 : l), t1 = u->t1, nfull = min(u->ctx / CB_KT, u->tiles - 1);
            const int node = (u->rg * 2 + lr) * p.NPT + node_of(row);
            const bool row_valid = row < RT && node < u->n;
            const bool warp_active = (wq * 32) < RT && node - node_of(row) + node_of(wq * 32) < u->n;   // row 0 of the warp is valid
            // this row's ancestor bits: word 0 (the reference is taken from the tile's first 32 keys) and this half's two words
            uint32_t mref = 0u, mlo = 0u, mhi = 0u;
            if (row_valid && t1 == u->tiles) {
                const uint32_t* mp = p.tree_mask + ((size_t)u->b * p.T + node) * p.W;
                mref = mp[0];
                if (2 * hf < p.W) mlo = mp[2 * hf];
                if (2 * hf + 1 < p.W) mhi = mp[2 * hf + 1];
            }
            const uint32_t ts = tmem + l * 128 + lane_addr, tsh = ts + 64 * hf;
            const uint32_t tm_O = tmem + C::O_COL + l * D + lane_addr;
            float m_used = -INFINITY, lsum = 0.f;
            for (int i = tfirst; i < t1; i += step) {
                if (!(ok = mbar_wait(bar_sfull(l), c_s & 1, s_abort, p.status))) break;
                ++c_s;
                if (warp_active) {
                    tc_fence_after();
                    // Visibility of this thread's 64 keys: context keys below ctx, tree keys by the ancestor bits.  A context tile
                    // that lies wholly inside the context needs no masks.  Rows that do not exist take the fast path too:
                    // whatever they compute stays in their own row.
                    const bool all_vis = i < nfull;
                    uint32_t vm[2] = {0xFFFFFFFFu, 0xFFFFFFFFu}, vref = 0xFFFFFFFFu;
                    auto below = [&](int lo) { return lo >= 32 ? 0xFFFFFFFFu : (lo <= 0 ? 0u : ((1u << lo) - 1u)); };
                    if (!all_vis) {
                        const bool is_tree = i == u->tiles - 1;
                        const int kv = is_tree ? u->n : u->ctx - i * CB_KT;
                        vm[0] = below(kv - 64 * hf); vm[1] = below(kv - 64 * hf - 32); vref = below(kv);
                        if (is_tree) { vm[0] &= mlo; vm[1] &= mhi; vref &= mref; }
                        if (!row_valid) vm[0] = vm[1] = vref = 0u;
                    }
                    // Single pass, tried first on every tile: P against the reference maximum in use, held back in registers so
                    // that S is still whole if the tile has to be done again.  No row maximum is taken.  The reference exists
                    // to keep 2^(s - reference) and its sums inside fp32 (P is bf16, same exponent range), not for precision,
                    // so the half row's sum tells all that matters: while it stays below 2^20 no score is more than 20
                    // above the reference and the tile stands; above that (or not finite) in either half, the two passes below
                    // run instead in both and move the reference to the new maximum.  A share's first tile has no reference
                    // yet and takes the largest of the row's first 32 scores (both threads of the row read them).
                    if (i == tfirst) {
                        uint32_t rf[32];
                        CB_TMEM_LD32(rf, 0, ts);
                        CB_TMEM_WAIT_LD32(rf);
                        if (!all_vis) {
#pragma unroll
                            for (int jx = 0; jx < 32; ++jx)
                                if (!((vref >> jx) & 1u)) rf[jx] = 0xFF800000u;
                        }
                        float c0 = -INFINITY, c1 = -INFINITY;
#pragma unroll
                        for (int jx = 0; jx < 32; jx += 4) {
                            c0 = fmax3(c0, __uint_as_float(rf[jx]), __uint_as_float(rf[jx + 1]));
                            c1 = fmax3(c1, __uint_as_float(rf[jx + 2]), __uint_as_float(rf[jx + 3]));
                        }
                        m_used = fmaxf(c0, c1) * p.scale_log2;   // -inf if the row sees none of them
                    }
                    uint32_t pk[32];
                    // P of this thread's 64 scores (packed into pk) against reference mu; returns their sum.  32 scores at a time:
                    // a thread has 96 registers, and what does not fit them spills past an L1 that the tiles leave 28 KB (with all 64
                    // scores in registers batch 32 took 256 us; with the next 16 in flight it takes what it takes without).
                    // The form without masks is code of its own: a branch per 16 scores keeps the compiler from overlapping
                    // one group's exponentials with the next one's (1,274 against 1,115 cycles a tile for this loop alone).
                    auto make_p_of = [&](float mu, auto masked) {
                        constexpr bool MASKED = decltype(masked)::value;
                        const uint64_t scale2 = f2_pack(p.scale_log2, p.scale_log2), negmu2 = f2_pack(-mu, -mu);
                        uint64_t lsa = f2_pack(0.f, 0.f), lsb = f2_pack(0.f, 0.f);
                        uint32_t sa[32];
#pragma unroll
                        for (int c = 0; c < 4; ++c) {
                            uint32_t* cur = sa + 16 * (c & 1);
                            if ((c & 1) == 0) { CB_TMEM_LD32(sa, 0, tsh + 16 * c); CB_TMEM_WAIT_LD32(sa); }
                            if (MASKED) {
#pragma unroll
                                for (int jx = 0; jx < 16; ++jx)
                                    if (!((vm[c >> 1] >> ((c & 1) * 16 + jx)) & 1u)) cur[jx] = 0xFF800000u;
                            }
#pragma unroll
                            for (int q = 0; q < 8; ++q) {
                                const uint64_t x = f2_fma(f2_pack(__uint_as_float(cur[2 * q]), __uint_as_float(cur[2 * q + 1])), scale2, negmu2);
                                float p0, p1;
                                if (!MASKED && q % C::FMA_EXP == C::FMA_EXP - 1) {
                                    ex2_pair_fma(x, p0, p1);
                                } else {
                                    f2_unpack(x, p0, p1);
                                    p0 = ex2(p0); p1 = ex2(p1);
                                }
                                if (q & 1) lsb = f2_add(lsb, f2_pack(p0, p1));
                                else lsa = f2_add(lsa, f2_pack(p0, p1));
                                pk[c * 8 + q] = pack_bf16(p0, p1);
                            }
                        }
                        float l0, l1, l2, l3;
                        f2_unpack(lsa, l0, l1);
                        f2_unpack(lsb, l2, l3);
                        return (l0 + l1) + (l2 + l3);
                    };
                    auto make_p = [&](float mu) {
                        return all_vis ? make_p_of(mu, std::false_type{}) : make_p_of(mu, std::true_type{});
                    };
                    float lt = make_p(m_used == -INFINITY ? 0.f : m_used);
                    if (pair_sync(row_valid && !(lt <= kRowSumLimit), 0)) {          // rows that do not exist hold anything: they never ask
                        // pass 1: the row's maximum over all its visible scores (both threads of the row take it)
                        uint32_t va[4] = {0xFFFFFFFFu, 0xFFFFFFFFu, 0xFFFFFFFFu, 0xFFFFFFFFu};
                        if (!all_vis) {
                            const bool is_tree = i == u->tiles - 1;
                            const int kv = is_tree ? u->n : u->ctx - i * CB_KT;
                            const uint32_t* mp = p.tree_mask + ((size_t)u->b * p.T + (row_valid ? node : 0)) * p.W;
#pragma unroll
                            for (int k = 0; k < 4; ++k) {
                                const uint32_t bl = below(kv - 32 * k);
                                va[k] = !row_valid ? 0u : (!is_tree ? bl : (k < p.W ? bl & mp[k] : 0u));
                            }
                        }
                        float mx = -INFINITY;
#pragma unroll 1
                        for (int c = 0; c < 4; ++c) {
                            uint32_t rf[32];
                            CB_TMEM_LD32(rf, 0, ts + 32 * c);
                            CB_TMEM_WAIT_LD32(rf);
#pragma unroll
                            for (int jx = 0; jx < 32; ++jx) mx = fmaxf(mx, ((va[c] >> jx) & 1u) ? __uint_as_float(rf[jx]) : -INFINITY);
                        }
                        pair_sync(false, 1);                                      // both have read S: either may write P over it now
                        const float mloc = mx * p.scale_log2;
                        // lazy rescaling: keep the reference maximum until the running maximum exceeds it by 2^8 (a tile that
                        // comes here from the single pass holds a score at least 2^13 above it)
                        const bool need = mloc > m_used + 8.0f;
                        const float alpha = need ? ex2(m_used - mloc) : 1.0f;
                        if (need) m_used = mloc;
                        if (i > tfirst && __any_sync(CB_FULL, need)) {
                            // O is complete up to the chain's previous tile: that product came before this S in the issue order.
                            // Each of the two threads rescales half of the columns.
#pragma unroll 1
                            for (int c = 0; c < 2; ++c) {
                                uint32_t o[CW];
                                const uint32_t ta = tm_O + hf * (D / 2) + c * CW;
                                tmem_ld_w<CW>(o, ta);
#pragma unroll
                                for (int jx = 0; jx < CW; ++jx) o[jx] = __float_as_uint(__uint_as_float(o[jx]) * alpha);
                                tmem_st_w<CW>(o, ta);
                            }
                            tmem_wait_st();
                        }
                        lsum *= alpha;
                        // pass 2: P = 2^(s * scale - m)
                        lt = make_p(m_used == -INFINITY ? 0.f : m_used);
                    }
                    CB_TMEM_ST32(pk, 0, tsh);                 // the 64 scores become 32 columns of packed P at their start
                    lsum += lt;
                    tmem_wait_st();
                }
                tc_fence_before();
                mbar_arrive(bar_pready(l));
            }
            if (!ok) break;
            // ---- epilogue of this unit's share
            const int ub = u->b, t0 = u->t0, h = (u->kh + (u->nrt == kTwoHeads ? l : 0)) * p.G + row - node_of(row) * p.G;
            const bool whole = t0 == 0 && t1 == u->tiles;
            // this thread's columns of the output row, 16 at a time: half a row with two row tiles, a quarter with one
            int npc, c0;
            // a shared unit: how many parts of it are in memory already (most often all the others, see below); the look is taken here,
            // where it overlaps the wait for the last product
            const int np = whole || p.cs > 0 ? 1 : u->np;
            uint32_t* const ticket = p.part_ticket + (np > 1 ? u->ticket : 0) + sw;
            uint32_t arrived = 0;
            if (np > 1 && lane == 0) arrived = ld_acquire(ticket);
            if (two) {
                // The wait comes before s_x is written: the unit's first product follows the other chain's end of the unit before
                // (bar_ofree), and if that one had one row tile, the other chain read this chain's row sums there.
                if (!(ok = mbar_wait(bar_odone(l), c_od & 1, s_abort, p.status))) break;
                ++c_od;
                s_x[(l * 2 + hf) * CB_MT + row] = lsum;
                pair_sync(false, 2);
                x_l = lsum + s_x[(l * 2 + 1 - hf) * CB_MT + row];
                x_m = m_used; x_w0 = x_w1 = 1.f;
                npc = CW / 8; c0 = hf * 2 * CW;
            } else {
                if (!(ok = mbar_wait(bar_odone_both, c_ob & 1, s_abort, p.status))) break;
                ++c_ob;
                s_x[(l * 2 + hf) * CB_MT + row] = lsum;
                pair_sync(false, 2);
                const float lrow = lsum + s_x[(l * 2 + 1 - hf) * CB_MT + row];
                pair_sync(false, 3);
                s_x[(l * 2 + hf) * CB_MT + row] = hf ? lrow : m_used;
                mbar_arrive(bar_sums);
                if (!(ok = mbar_wait(bar_sums, (c_ob - 1) & 1, s_abort, p.status))) break;
                const float m0 = s_x[row], l0 = s_x[CB_MT + row], m1 = s_x[2 * CB_MT + row], l1 = s_x[3 * CB_MT + row];
                x_m = fmaxf(m0, m1);
                x_w0 = m0 == -INFINITY ? 0.f : ex2(m0 - x_m);
                x_w1 = m1 == -INFINITY ? 0.f : ex2(m1 - x_m);
                x_l = l0 * x_w0 + l1 * x_w1;
                npc = CW / 16; c0 = (l * 2 + hf) * CW;
            }
            tc_fence_after();
            if (p.cs > 0) {
                c_share = true;                               // O stays in TMEM until the exchange below
                x_two = t1 - t0 > 1;                          // a share of one tile has no second accumulator
                break;                                        // a CTA of a cluster has one share
            }
            if (warp_active) {
                __nv_bfloat16* op = p.out + (((size_t)ub * p.T + (row_valid ? node : 0)) * p.Hq + h) * D;
                // 16 of this thread's accumulator columns, relative to reference x_m; with one row tile both accumulators put together
                auto load_o = [&](float* o, int col) {
                    uint32_t* r = reinterpret_cast<uint32_t*>(o);
                    tmem_ld_w<16>(r, tmem + C::O_COL + (two ? l * D : 0) + lane_addr + col);
                    if (two) return;
#pragma unroll
                    for (int k = 0; k < 16; ++k) o[k] *= x_w0;
                    if (t1 - t0 > 1) {
                        uint32_t o1[16];
                        tmem_ld_w<16>(o1, tmem + C::O_COL + D + lane_addr + col);
#pragma unroll
                        for (int k = 0; k < 16; ++k) o[k] = fmaf(__uint_as_float(o1[k]), x_w1, o[k]);
                    }
                };
                auto store_out = [&](const float* o, int col, float inv) {
                    if (!row_valid) return;
                    uint32_t w[8];
#pragma unroll
                    for (int k = 0; k < 8; ++k) w[k] = pack_bf16(o[2 * k] * inv, o[2 * k + 1] * inv);
                    if (out32) {
                        st_global_v8(op + col, w[0], w[1], w[2], w[3], w[4], w[5], w[6], w[7]);
                    } else {
                        *reinterpret_cast<uint4*>(op + col) = make_uint4(w[0], w[1], w[2], w[3]);
                        *reinterpret_cast<uint4*>(op + col + 8) = make_uint4(w[4], w[5], w[6], w[7]);
                    }
                };
                auto store_lse = [&](float mx, float sum) {
                    if (row_valid && c0 == 0 && p.lse) p.lse[((size_t)ub * p.Hq + h) * p.T + node] = sum > 0.f ? (mx + log2f(sum)) * 0.6931471805599453f : 0.f;
                };
                if (whole) {
                    const float inv = x_l > 0.f ? 1.0f / x_l : 0.f;
#pragma unroll 1
                    for (int e = 0; e < npc; ++e) {
                        float o[16];
                        load_o(o, c0 + 16 * e);
                        store_out(o, c0 + 16 * e, inv);
                    }
                    store_lse(x_m, x_l);
                } else {
                    // A unit shared with other CTAs.  The same warp of each of them has the same rows and columns, so the warps settle it
                    // among themselves: all but the last to come leave their partial (unnormalised columns, reference and sum) in
                    // memory and count themselves; the last one reads the others', in the order of the CTAs whoever is last, and
                    // writes the output.  Nobody waits.  (A CTA's first unit is shared with the CTA before it, which comes to it
                    // last, so most often the partial has long been there: the pass that merged both partials from memory after the
                    // kernel cost 9 us a call at batch 32.)  A warp's partial is laid out by lane: 512 bytes per access.
                    const int xpos = u->xpos, cf = u->cf;
                    auto slot_of = [&](int cc, bool start) {
                        return p.part + (size_t)(2 * cc + (start ? 1 : 0)) * (2 * CB_MT * (D + 4));
                    };
                    auto part_of = [&](int k) { return slot_of(xpos < 0 ? cf + k : cb_cta_of(*s_tot, p.nc, (long long)xpos + k * u->wt), k == 0); };
                    const int wofs = sw * (2 * CW * 32) + lane * 4, mlofs = 2 * CB_MT * D + (sw * 32 + lane) * 2;
                    float* const own = slot_of(cta, t0 == 0);
                    auto load_part = [&](float4* v, const float* pp, int e) {
#pragma unroll
                        for (int q = 0; q < 4; ++q) v[q] = __ldcg(reinterpret_cast<const float4*>(pp + wofs + (e * 4 + q) * 128));
                    };
                    auto load_ml = [&](const float* pp) { return __ldcg(reinterpret_cast<const float2*>(pp + mlofs)); };
                    auto weight = [](float m, float mx) { return m == -INFINITY ? 0.f : ex2(m - mx); };
                    bool last = __shfl_sync(CB_FULL, arrived, 0) == (uint32_t)(np - 1);
                    if (!last) {
#pragma unroll 1
                        for (int e = 0; e < npc; ++e) {
                            float o[16];
                            load_o(o, c0 + 16 * e);
#pragma unroll
                            for (int q = 0; q < 4; ++q)
                                *reinterpret_cast<float4*>(own + wofs + (e * 4 + q) * 128) = make_float4(o[q * 4], o[q * 4 + 1], o[q * 4 + 2], o[q * 4 + 3]);
                        }
                        *reinterpret_cast<float2*>(own + mlofs) = make_float2(x_m, x_l);
                        __syncwarp();
                        if (lane == 0) arrived = atom_add_acq_rel(ticket, 1u);   // releases the whole warp's stores
                        last = __shfl_sync(CB_FULL, arrived, 0) == (uint32_t)(np - 1);
                    }
                    if (last) {
                        __syncwarp();
                        float mx = -INFINITY, sum = 0.f;
                        if (np == 2) {
                            // the usual case: one other part, its columns fetched a group ahead
                            const bool first = t0 == 0;
                            const float* const po = part_of(first ? 1 : 0);
                            float4 v[4], vn[4];
                            load_part(v, po, 0);
                            const float2 ml = load_ml(po);
                            mx = fmaxf(x_m, ml.x);
                            const float wo = weight(x_m, mx), wp = weight(ml.x, mx);
                            sum = first ? fmaf(wp, ml.y, wo * x_l) : fmaf(wo, x_l, wp * ml.y);
                            const float inv = sum > 0.f ? 1.0f / sum : 0.f;
#pragma unroll 1
                            for (int e = 0; e < npc; ++e) {
                                float o[16];
                                if (e + 1 < npc) load_part(vn, po, e + 1);
                                load_o(o, c0 + 16 * e);
                                const float* vf = reinterpret_cast<const float*>(v);
#pragma unroll
                                for (int k = 0; k < 16; ++k) o[k] = first ? fmaf(wp, vf[k], wo * o[k]) : fmaf(wo, o[k], wp * vf[k]);
                                store_out(o, c0 + 16 * e, inv);
#pragma unroll
                                for (int q = 0; q < 4; ++q) v[q] = vn[q];
                            }
                        } else {
                            for (int k = 0; k < np; ++k) {
                                const float* pp = part_of(k);
                                const float2 ml = pp == own ? make_float2(x_m, x_l) : load_ml(pp);
                                const float mn = fmaxf(mx, ml.x);
                                sum = fmaf(weight(ml.x, mn), ml.y, sum * weight(mx, mn));
                                mx = mn;
                            }
                            const float inv = sum > 0.f ? 1.0f / sum : 0.f;
#pragma unroll 1
                            for (int e = 0; e < npc; ++e) {
                                float acc[16];
#pragma unroll
                                for (int k = 0; k < 16; ++k) acc[k] = 0.f;
#pragma unroll 1
                                for (int k = 0; k < np; ++k) {
                                    const float* pp = part_of(k);
                                    float4 v[4];
                                    float mk = x_m;
                                    if (pp == own) {
                                        load_o(reinterpret_cast<float*>(v), c0 + 16 * e);
                                    } else {
                                        load_part(v, pp, e);
                                        mk = load_ml(pp).x;
                                    }
                                    const float w = weight(mk, mx);
                                    const float* vf = reinterpret_cast<const float*>(v);
#pragma unroll
                                    for (int q = 0; q < 16; ++q) acc[q] = fmaf(w, vf[q], acc[q]);
                                }
                                store_out(acc, c0 + 16 * e, inv);
                            }
                        }
                        store_lse(mx, sum);
                    }
                }
            }
            tc_fence_before();
            if (two) mbar_arrive_n(bar_ofree(l), 2u);          // 512 arrivals per unit either way
            else { mbar_arrive(bar_ofree(0)); mbar_arrive(bar_ofree(1)); }
        }
        if (!ok) {
            // The other warp of the pair may have entered a pair barrier that this one will not: answer for it until it has left too.
            // Its own waits end as well, so this does; the loop is bounded all the same.
            __syncwarp();
            int seen = __shfl_sync(CB_FULL, lane == 0 ? s_pair[sw] : 0, 0);
            if (lane == 0) { __threadfence_block(); s_pair[sw] = -1; }
            for (int k = 0; k < 1 << 16; ++k) {
                const int other = __shfl_sync(CB_FULL, lane == 0 ? s_pair[sw ^ 4] : 0, 0);
                if (other < 0) break;
                if (other > seen) { seen = other; pair_arrive(pair_id); }
                __nanosleep(200);
            }
        }
        __syncwarp();
        cluster_wait();
        if (p.cs > 0 && s_sched->c_has) {
            // ------------------------------------------------------------------ cluster mode: combine the unit's shares
            // Every CTA of the cluster holds the unnormalised rows of its share (O0 and O1 in TMEM, their weights, the running
            // maximum and the sum in registers).  CTA r puts columns [r D / cs, (r + 1) D / cs) of all rows together: a thread's
            // columns go to one CTA (two with cs = 8), 32 rows side by side, so that a warp writes 512 bytes in a run to shared memory
            // over there (by rows, one CTA for every cs-th row, the same 64 KB took 4.2 k cycles).  They are received in
            // the two query tiles when they fit (idle from a CTA's last S product on, which the query loader reports), otherwise
            // in the K/V ring (idle from the last P.V on, reported here).  With them come every row's reference and sum.
            const int cs = p.cs, rank = cta % cs;
            const int cb_ = s_sched->c_b, ckh = s_sched->c_kh, cn = s_sched->c_n;
            const CbExchange ex = cb_exchange(p, D, cn);
            const uint32_t recv = sbase + (ex.bytes <= 2u * C::Q_BYTES ? C::OFF_Q : C::OFF_RING);
            if (ok && ex.bytes > 2u * C::Q_BYTES && sw == 0 && lane == 0)
                for (int r = 0; r < cs; ++r) mbar_arrive_remote(cluster_addr(bar_cready, (uint32_t)r));
            // columns of one CTA, in groups of 4; powers of two
            const int lc = 31 - __clz(D / cs), nch = 1 << (lc - 2);
            const int col = (l * 2 + hf) * CW;
            uint32_t o[CW];
#pragma unroll
            for (int k = 0; k < CW; ++k) o[k] = 0u;             // what a CTA without tiles contributes
            if (ok && c_share && row < ex.rows) {               // whole warps
                tmem_ld_w<CW>(o, tmem + C::O_COL + lane_addr + col);
#pragma unroll
                for (int k = 0; k < CW; ++k) o[k] = __float_as_uint(__uint_as_float(o[k]) * x_w0);
                if (x_two) {
                    uint32_t o1[CW];
                    tmem_ld_w<CW>(o1, tmem + C::O_COL + D + lane_addr + col);
#pragma unroll
                    for (int k = 0; k < CW; ++k) o[k] = __float_as_uint(fmaf(__uint_as_float(o1[k]), x_w1, __uint_as_float(o[k])));
                }
            }
            if (ok) ok = mbar_wait_cluster(bar_cready, 0, s_abort, p.status);
            if (ok && row < ex.rows) {
                // Stores that count themselves off the receiver's barrier: a release by an ordinary remote arrival waits for
                // every store before it to come back.
#pragma unroll
                for (int v4 = 0; v4 < CW / 4; ++v4) {
                    const int c = col + v4 * 4, d = c >> lc;
                    st_async_v4(cluster_addr(recv + ex.value(rank, (c >> 2) & (nch - 1), row, nch), (uint32_t)d), cluster_addr(bar_cdata, (uint32_t)d),
                                o[v4 * 4], o[v4 * 4 + 1], o[v4 * 4 + 2], o[v4 * 4 + 3]);
                }
                for (int c = col; c < col + CW; c += 4)
                    if ((c & (4 * nch - 1)) == 0)
                        st_async_v2(cluster_addr(recv + ex.sums(rank, row, cs, nch), (uint32_t)(c >> lc)), cluster_addr(bar_cdata, (uint32_t)(c >> lc)),
                                    __float_as_uint(c_share ? x_m : -INFINITY), __float_as_uint(c_share ? x_l : 0.f));
            }
            if (ok) ok = mbar_wait_cluster(bar_cdata, 0, s_abort, p.status);
            if (ok) {
                const int nrow = min(RT, cn * p.G), cols = 4 * nch;
                for (int t = sw * 32 + lane; t < nrow * nch; t += 512) {
                    const int r = t >> (lc - 2), ch = t & (nch - 1);
                    float mx = -INFINITY;
                    for (int k = 0; k < cs; ++k) mx = fmaxf(mx, ld_shared_f2(recv + ex.sums(k, r, cs, nch)).x);
                    float acc[4] = {0.f, 0.f, 0.f, 0.f}, wsum = 0.f;
                    for (int k = 0; k < cs; ++k) {
                        const float2 ml = ld_shared_f2(recv + ex.sums(k, r, cs, nch));
                        if (ml.x == -INFINITY) continue;         // that CTA had no tiles: its rows were not written
                        const float w = ex2(ml.x - mx);
                        const float4 v = ld_shared_f4(recv + ex.value(k, ch, r, nch));
                        wsum = fmaf(w, ml.y, wsum);
                        acc[0] = fmaf(w, v.x, acc[0]); acc[1] = fmaf(w, v.y, acc[1]); acc[2] = fmaf(w, v.z, acc[2]); acc[3] = fmaf(w, v.w, acc[3]);
                    }
                    const float inv = wsum > 0.f ? 1.0f / wsum : 0.f;
                    const int node = r / p.G, h = ckh * p.G + r % p.G;
                    __nv_bfloat16* op = p.out + (((size_t)cb_ * p.T + node) * p.Hq + h) * D + rank * cols + ch * 4;
                    *reinterpret_cast<uint2*>(op) = make_uint2(pack_bf16(acc[0] * inv, acc[1] * inv), pack_bf16(acc[2] * inv, acc[3] * inv));
                    if (rank == 0 && ch == 0 && p.lse)
                        p.lse[((size_t)cb_ * p.Hq + h) * p.T + node] = wsum > 0.f ? (mx + log2f(wsum)) * 0.6931471805599453f : 0.f;
                }
            }
        }
    }

    // ---------------------------------------------------------------------- teardown
    if (*s_abort) {
        // give copies that are still in flight time to land before the shared memory is released
        for (int k = 0; k < 64; ++k) __nanosleep(1000);
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmemCols) : "memory");
        // the last CTA to leave hands the turn on: nobody looks at this launch's tickets any more
        if (p.cs == 0 && elect_one() && atomicInc(&p.part_turn[1], gridDim.x - 1u) == gridDim.x - 1u) atomicAdd(&p.part_turn[0], 1u);
    }
}

// Merge pass of the CTA-pair kernel (cb_attn_pair.cuh): block (c, *) looks at the unit that CTA c of the attention kernel started but did not finish,
// and combines the partials that CTA c and the following CTAs left for it.  One warp per output row.
// Every block waits for the attention grid before it leaves, also the ones that find nothing to merge: the next kernel
// in the stream is ordered behind this grid only, so this grid must not end while the attention kernel still runs.
template <int D>
__global__ void __launch_bounds__(256) cb_attn_merge_kernel(const CbAttnParams p) {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");   // the wait comes below, after the set-up that reads inputs only
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int c = blockIdx.x;
    const long long tot = cb_sched_total(p, lane);
    bool nothing = tot <= 0;
    long long g0 = 0, g1 = 0, pre = 0, ustart = 0;
    int b = 0, rg = 0, j = 0, vt = 1;
    CbSeqShape s = {};
    if (!nothing) {
        g0 = cb_range_start(tot, p.nc, c); g1 = cb_range_start(tot, p.nc, c + 1);
        nothing = g1 <= g0 || g1 >= tot;                      // empty range, or the last range
    }
    if (!nothing) {
        cb_sched_locate(p, g1 - 1, lane, &rg, &b, &pre);
        s = cb_seq_shape(p, b);
        const long long off = g1 - 1 - pre;
        vt = s.unit(rg);                                      // positions of one unit: padding, then its key tiles (one each)
        j = (int)(off / vt);
        ustart = pre + (long long)j * vt;
        const long long first_tile = ustart + s.ov(rg);
        nothing = (int)(off - (long long)j * vt) == vt - 1    // the unit ends with this range
                  || first_tile < g0                          // started by an earlier CTA: that CTA's block merges it
                  || first_tile >= g1;                        // only padding so far: the next CTA starts the unit
    }
    if (nothing) {
        asm volatile("griddepcontrol.wait;" ::: "memory");
        return;
    }
    const int c_last = cb_cta_of(tot, p.nc, ustart + vt - 1);
    const int kh = j;                                         // units of (row group, sequence) are its kv heads
    const int nrt = p.MT == 1 ? 1 : min(2, s.mtn - 2 * rg);
    const int RT = p.NPT * p.G;
    constexpr int PER = D / 32;
    // partial slots of this unit, listed once per block: CTA c's "started here" slot, then the "continued" slots of
    // the following CTAs that have a non-empty range
    __shared__ int s_slot[CB_ATTN_MAX_CTAS];
    __shared__ int s_nparts;
    if (warp == 0) {
        int np = 0;
        for (int base = c; base <= c_last; base += 32) {
            const int cc = base + lane;
            const bool valid = cc <= c_last && cb_range_start(tot, p.nc, cc) < cb_range_start(tot, p.nc, cc + 1);
            const uint32_t m = __ballot_sync(CB_FULL, valid);
            if (valid) s_slot[np + __popc(m & ((1u << lane) - 1u))] = 2 * cc + (cc == c ? 1 : 0);
            np += __popc(m);
        }
        if (lane == 0) s_nparts = np;
    }
    __syncthreads();
    const int nparts = s_nparts;
    asm volatile("griddepcontrol.wait;" ::: "memory");       // the attention grid has finished and its writes are visible
    const size_t rstride = (size_t)(D + 4), sstride = (size_t)2 * CB_MT * rstride;
    for (int r2 = blockIdx.y * 8 + warp; r2 < nrt * CB_MT; r2 += gridDim.y * 8) {
        const int wg = r2 / CB_MT, row = r2 % CB_MT;
        const int node = (rg * 2 + wg) * p.NPT + row / p.G, h = kh * p.G + row % p.G;
        if (row >= RT || node >= s.n) continue;
        const float* base = p.part + ((size_t)wg * CB_MT + row) * rstride;
        // lanes fetch the running maxima of up to 32 parts at a time
        float M = -INFINITY;
        for (int k0 = 0; k0 < nparts; k0 += 32) {
            const int k = k0 + lane;
            const float ms = k < nparts ? base[(size_t)s_slot[k] * sstride + D] : -INFINITY;
            M = fmaxf(M, ms);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) M = fmaxf(M, __shfl_xor_sync(CB_FULL, M, o));
        float o[PER], Lsum = 0.f;
#pragma unroll
        for (int d = 0; d < PER; ++d) o[d] = 0.f;
        for (int k = 0; k < nparts; ++k) {
            const float* pp = base + (size_t)s_slot[k] * sstride;
            const float ms = pp[D];
            const float w = ms == -INFINITY ? 0.f : exp2f(ms - M);
            Lsum = fmaf(w, pp[D + 1], Lsum);
            if constexpr (PER == 4) {
                const float4 v = *reinterpret_cast<const float4*>(pp + lane * 4);
                o[0] = fmaf(w, v.x, o[0]); o[1] = fmaf(w, v.y, o[1]); o[2] = fmaf(w, v.z, o[2]); o[3] = fmaf(w, v.w, o[3]);
            } else {
                const float2 v = *reinterpret_cast<const float2*>(pp + lane * 2);
                o[0] = fmaf(w, v.x, o[0]); o[1] = fmaf(w, v.y, o[1]);
            }
        }
        const float inv = Lsum > 0.f ? 1.f / Lsum : 0.f;
        __nv_bfloat16* op = p.out + (((size_t)b * p.T + node) * p.Hq + h) * D + lane * PER;
#pragma unroll
        for (int d = 0; d < PER; ++d) op[d] = __float2bfloat16_rn(o[d] * inv);
        if (p.lse && lane == 0) p.lse[((size_t)b * p.Hq + h) * p.T + node] = Lsum > 0.f ? (M + log2f(Lsum)) * 0.6931471805599453f : 0.f;
    }
}

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                                  const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn get_encode() {
    static EncodeTiledFn fn = nullptr;
    if (!fn) {
        void* ptr = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &ptr, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = (EncodeTiledFn)ptr;
    }
    return fn;
}

// 4-D view (d, head, row, block) of a [blocks, rows, heads, D] bf16 tensor; box = 64 dims x box_heads x box_rows.
bool encode_map(CUtensorMap* m, const void* base, int D, int heads, int rows, long blocks, int box_heads, int box_rows) {
    EncodeTiledFn enc = get_encode();
    if (!enc) { fprintf(stderr, "cacheback: cuTensorMapEncodeTiled entry point not found\n"); return false; }
    cuuint64_t dims[4] = {(cuuint64_t)D, (cuuint64_t)heads, (cuuint64_t)rows, (cuuint64_t)blocks};
    cuuint64_t strides[3] = {(cuuint64_t)D * 2, (cuuint64_t)heads * D * 2, (cuuint64_t)rows * heads * D * 2};
    cuuint32_t box[4] = {64, (cuuint32_t)box_heads, (cuuint32_t)box_rows, 1};
    cuuint32_t estr[4] = {1, 1, 1, 1};
    const CUresult r = enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void*>(base), dims, strides, box, estr,
                           CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                           // a head's row is D * 2 bytes contiguous and is fetched as 128-byte halves by two boxes: with D = 128 let the
                           // first one bring the whole row into L2
                           D >= 128 ? CU_TENSOR_MAP_L2_PROMOTION_L2_256B : CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                           CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS)
        fprintf(stderr, "cacheback: tensor map encode failed (%d): D=%d heads=%d rows=%d blocks=%ld base=%p\n", (int)r, D, heads, rows,
                blocks, base);
    return r == CUDA_SUCCESS;
}

// 5-D view of a [blocks, rows, heads, D] bf16 tensor in the order (64 dims, row, 64-dim column block, ...): with `fold`, rows of all
// blocks are counted in groups of 8 and the last two coordinates are (group, head), box = 8 rows x D dims x 2 groups; without,
// they are (head, block), box = 8 rows x D dims.
bool encode_grouped_map(CUtensorMap* m, const void* base, int D, int heads, int rows, long blocks, bool fold) {
    EncodeTiledFn enc = get_encode();
    if (!enc) { fprintf(stderr, "cacheback: cuTensorMapEncodeTiled entry point not found\n"); return false; }
    const cuuint64_t row = (cuuint64_t)heads * D * 2;          // bytes
    cuuint64_t dims[5] = {64, fold ? 8u : (cuuint64_t)rows, (cuuint64_t)(D / 64), fold ? (cuuint64_t)blocks * (rows / 8) : (cuuint64_t)heads,
                          fold ? (cuuint64_t)heads : (cuuint64_t)blocks};
    cuuint64_t strides[4] = {row, 128, fold ? 8 * row : (cuuint64_t)D * 2, fold ? (cuuint64_t)D * 2 : (cuuint64_t)rows * row};
    cuuint32_t box[5] = {64, 8, (cuuint32_t)(D / 64), fold ? 2u : 1u, 1};
    cuuint32_t estr[5] = {1, 1, 1, 1, 1};
    const CUresult r = enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 5, const_cast<void*>(base), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                           CU_TENSOR_MAP_SWIZZLE_128B, D >= 128 ? CU_TENSOR_MAP_L2_PROMOTION_L2_256B : CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                           CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS)
        fprintf(stderr, "cacheback: tensor map encode failed (%d): D=%d heads=%d rows=%d blocks=%ld base=%p\n", (int)r, D, heads, rows, blocks, base);
    return r == CUDA_SUCCESS;
}

// Cluster mode is for launches with few units, where the stream-K split would make every unit a shared one: all trees fit
// one row tile (so a unit is one (sequence, kv head)), units times a cluster size of 8, 4 or 2 does not exceed the SMs, that
// many clusters can be resident at once, and a CTA's part of a unit (tiles / cs) is shorter than a CTA's range under the
// stream-K split plus what its partials and merge pass cost (about three tiles).  Returns the cluster size or 0.
template <int D>
int pick_cluster_size(const CbAttnParams& p, int num_sms) {
    if (p.MT != 1) return 0;
    const long long units = (long long)p.B * p.Hkv;
    for (int cs = 8; cs >= 2; cs >>= 1) {
        if (units * cs > num_sms) continue;
        const long long in_cluster = (p.max_tiles + cs - 1) / cs, stream_k = units * (p.max_tiles + 2) / num_sms + 3;
        if (in_cluster >= stream_k) continue;
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3((unsigned)(units * cs)); cfg.blockDim = dim3(kThreads); cfg.dynamicSmemBytes = Cfg<D>::SMEM;
        cudaLaunchAttribute at[1];
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = (unsigned)cs; at[0].val.clusterDim.y = 1; at[0].val.clusterDim.z = 1;
        cfg.attrs = at; cfg.numAttrs = 1;
        int nclusters = 0;
        if (cudaOccupancyMaxActiveClusters(&nclusters, cb_attn_tc_kernel<D>, &cfg) != cudaSuccess) { (void)cudaGetLastError(); continue; }
        if (nclusters >= units) return cs;
    }
    return 0;
}

// Host state of the launcher, per device and guarded: the opt-in to large dynamic shared memory is a per-device function
// attribute, and the cluster size chosen for a shape is remembered for the shapes seen last.
constexpr int kMaxDevices = 64;
constexpr int kShapeMemo = 8;
struct ShapeMemo { int key[6]; int cs; };
std::mutex g_launch_mutex;
bool g_attr_set[2][kMaxDevices];
ShapeMemo g_shape_memo[kShapeMemo];
int g_shape_used = 0, g_shape_next = 0;

int g_pairs[kMaxDevices];              // CTA pairs that can be resident at once (0 = not asked yet, -1 = none)

// On request (CB_FLAG_ATTN_CTA_PAIRS), launches with two or more row tiles per unit and head_dim 128 run as pairs of CTAs
// (cb_attn_pair.cuh): as many pairs as can be resident together, each taking an equal range of the global tile sequence.
cb_status launch_pairs(CbAttnParams p, const TcMaps& maps, cudaStream_t st, int num_sms, int device, bool* done) {
    *done = false;
    const int di = device >= 0 && device < kMaxDevices ? device : -1;
    if (di < 0) return CB_OK;
    int npairs;
    {
        std::lock_guard<std::mutex> lock(g_launch_mutex);
        if (g_pairs[di] == 0) {
            g_pairs[di] = -1;
            if (cudaFuncSetAttribute(cb_attn_pair_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)PairCfg::SMEM_ALLOC) == cudaSuccess) {
                cudaLaunchConfig_t cfg = {};
                cfg.gridDim = dim3((unsigned)(num_sms / 2 * 2)); cfg.blockDim = dim3(kPairThreads); cfg.dynamicSmemBytes = PairCfg::SMEM_ALLOC;
                cudaLaunchAttribute at[1];
                at[0].id = cudaLaunchAttributeClusterDimension;
                at[0].val.clusterDim.x = 2; at[0].val.clusterDim.y = 1; at[0].val.clusterDim.z = 1;
                cfg.attrs = at; cfg.numAttrs = 1;
                int n = 0;
                if (cudaOccupancyMaxActiveClusters(&n, cb_attn_pair_kernel, &cfg) == cudaSuccess && n > 0) g_pairs[di] = n < num_sms / 2 ? n : num_sms / 2;
            }
            (void)cudaGetLastError();
        }
        npairs = g_pairs[di];
    }
    if (npairs <= 0) return CB_OK;
    // The units that stream the same keys (the row groups of one (sequence, kv head)) lie 1 / row-groups of the tile sequence
    // apart: with a number of ranges that is a multiple of the row groups they are at the same point of their ranges at the
    // same time, so that one fetch from HBM serves all of them.
    const int row_groups = (p.MT + 1) / 2;
    if (npairs > row_groups) npairs -= npairs % row_groups;
    p.nc = npairs; p.cs = 0; p.w1 = p.w2 = 1; p.d1 = p.d2 = 0;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(2 * npairs)); cfg.blockDim = dim3(kPairThreads); cfg.dynamicSmemBytes = PairCfg::SMEM_ALLOC; cfg.stream = st;
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = 2; at[0].val.clusterDim.y = 1; at[0].val.clusterDim.z = 1;
    at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at; cfg.numAttrs = 2;
    CB_CUDA(cudaLaunchKernelEx(&cfg, cb_attn_pair_kernel, p, maps));
    CB_CUDA(cb_launch_pdl(cb_attn_merge_kernel<128>, dim3(p.nc, 4), dim3(256), 0, st, p));
    cb_count_launch(2);
    CB_CUDA(cudaGetLastError());
    *done = true;
    return CB_OK;
}

template <int D>
cb_status launch(CbAttnParams p, const TcMaps& maps, cudaStream_t st, int num_sms, int device) {
    {
        std::lock_guard<std::mutex> lock(g_launch_mutex);
        const int di = device >= 0 && device < kMaxDevices ? device : -1;
        if (di < 0 || !g_attr_set[D == 128][di]) {
            CB_CUDA(cudaFuncSetAttribute(cb_attn_tc_kernel<D>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Cfg<D>::SMEM));
            if (di >= 0) g_attr_set[D == 128][di] = true;
        }
        // the choice depends on the shape only
        const int key[6] = {p.B, p.Hkv, p.MT, num_sms, p.max_tiles, D * kMaxDevices + (di < 0 ? 0 : di)};
        int found = -1;
        for (int i = 0; i < g_shape_used && found < 0; ++i) {
            bool same = true;
            for (int k = 0; k < 6; ++k) same = same && g_shape_memo[i].key[k] == key[k];
            if (same) found = i;
        }
        if (found < 0) {
            found = g_shape_used < kShapeMemo ? g_shape_used++ : (g_shape_next++ % kShapeMemo);
            for (int k = 0; k < 6; ++k) g_shape_memo[found].key[k] = key[k];
            g_shape_memo[found].cs = pick_cluster_size<D>(p, num_sms);
        }
        p.cs = g_shape_memo[found].cs;
    }
    if (p.cs > 0) {
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3((unsigned)(p.B * p.Hkv * p.cs)); cfg.blockDim = dim3(kThreads); cfg.dynamicSmemBytes = Cfg<D>::SMEM; cfg.stream = st;
        cudaLaunchAttribute at[2];
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = (unsigned)p.cs; at[0].val.clusterDim.y = 1; at[0].val.clusterDim.z = 1;
        at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        at[1].val.programmaticStreamSerializationAllowed = 1;
        cfg.attrs = at; cfg.numAttrs = 2;
        CB_CUDA(cudaLaunchKernelEx(&cfg, cb_attn_tc_kernel<D>, p, maps));
        cb_count_launch(1);
        return CB_OK;
    }
    CB_CUDA(cb_launch_pdl(cb_attn_tc_kernel<D>, dim3(p.nc), dim3(kThreads), Cfg<D>::SMEM, st, p, maps));
    cb_count_launch(1);
    CB_CUDA(cudaGetLastError());
    return CB_OK;
}

}  // namespace

// Encoding five tensor maps costs several microseconds of host time, which matters at batch 1: the maps of the most
// recent argument sets are kept (they depend only on the base pointers and the shape).
namespace {
struct MapKey {
    const void *q, *k_pool, *v_pool, *k_tree, *v_tree;
    int D, Hq, Hkv, P, T, B, G, NPT, num_pages, pairs;
    bool operator==(const MapKey& o) const {
        return q == o.q && k_pool == o.k_pool && v_pool == o.v_pool && k_tree == o.k_tree && v_tree == o.v_tree && D == o.D && Hq == o.Hq &&
               Hkv == o.Hkv && P == o.P && T == o.T && B == o.B && G == o.G && NPT == o.NPT && num_pages == o.num_pages && pairs == o.pairs;
    }
};
constexpr int kMapCache = 16;
MapKey g_map_keys[kMapCache];
TcMaps g_map_vals[kMapCache];
int g_map_used = 0, g_map_next = 0;
std::mutex g_map_mutex;
}  // namespace

cb_status cb_attn_launch_tensor(cb_ctx* ctx, const CbAttnParams& p, cudaStream_t st) {
    if (p.P != 16) return CB_ERR_UNSUPPORTED;
    const bool pairs = p.D == 128 && p.MT > 1 && (ctx->cfg.flags & CB_FLAG_ATTN_CTA_PAIRS);
    const MapKey key = {p.q, p.k_pool, p.v_pool, p.k_tree, p.v_tree, p.D, p.Hq, p.Hkv, p.P, p.T, p.B, p.G, p.NPT, p.num_pages, pairs ? 1 : 0};
    TcMaps maps;
    bool hit = false;
    {
        std::lock_guard<std::mutex> lock(g_map_mutex);
        for (int i = 0; i < g_map_used && !hit; ++i)
            if (g_map_keys[i] == key) { maps = g_map_vals[i]; hit = true; }
    }
    if (!hit) {
        if (pairs) {
            if (!encode_map(&maps.k_pool, p.k_pool, p.D, p.Hkv, p.P, p.num_pages, 1, 16)) return CB_ERR_CUDA;
            if (!encode_map(&maps.v_pool, p.v_pool, p.D, p.Hkv, p.P, p.num_pages, 1, 16)) return CB_ERR_CUDA;
            if (!encode_map(&maps.k_tree, p.k_tree, p.D, p.Hkv, p.T, p.B, 1, 16)) return CB_ERR_CUDA;
            if (!encode_map(&maps.v_tree, p.v_tree, p.D, p.Hkv, p.T, p.B, 1, 16)) return CB_ERR_CUDA;
        } else {
            if (!encode_grouped_map(&maps.k_pool, p.k_pool, p.D, p.Hkv, p.P, p.num_pages, true)) return CB_ERR_CUDA;
            if (!encode_grouped_map(&maps.v_pool, p.v_pool, p.D, p.Hkv, p.P, p.num_pages, true)) return CB_ERR_CUDA;
            if (!encode_grouped_map(&maps.k_tree, p.k_tree, p.D, p.Hkv, p.T, p.B, false)) return CB_ERR_CUDA;
            if (!encode_grouped_map(&maps.v_tree, p.v_tree, p.D, p.Hkv, p.T, p.B, false)) return CB_ERR_CUDA;
        }
        if (!encode_map(&maps.q, p.q, p.D, p.Hq, p.T, p.B, p.G, p.NPT)) return CB_ERR_CUDA;
        std::lock_guard<std::mutex> lock(g_map_mutex);
        const int slot = g_map_used < kMapCache ? g_map_used++ : (g_map_next++ % kMapCache);
        g_map_keys[slot] = key;
        g_map_vals[slot] = maps;
    }
    if (pairs) {
        bool done = false;
        const cb_status r = launch_pairs(p, maps, st, ctx->num_sms, ctx->device, &done);
        if (r != CB_OK || done) return r;
    }
    return p.D == 128 ? launch<128>(p, maps, st, ctx->num_sms, ctx->device) : launch<64>(p, maps, st, ctx->num_sms, ctx->device);
}

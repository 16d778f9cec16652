// Tree attention: the schedule of small batches, in 32 bits (cb_attn.cuh has the general one).
#pragma once
#include "cb_attn.cuh"

// cb_sched_total, cb_range_start and cb_sched_locate for batches of up to 32 whose positions fit 32 bits: a lane keeps its sequence's
// shape, and sums and scans are 32 bits wide (CTA c of p.nc; false: neither batch nor positions allow it).  Before the first copy
// everything waits for this: 2.6 k cycles, so 1.9.
__device__ __forceinline__ bool cb_sched_of_32(const CbAttnParams& p, int c, int lane, long long* tot, long long* g0, long long* g1, int* rg_out, int* b_out, long long* pre_out) {
    if (p.B > 32) return false;
    CbSeqShape s = {};
    if (lane < p.B) s = cb_seq_shape(p, lane);
    if (__any_sync(CB_FULL, s.W >> 26 != 0)) return false;
    const uint32_t all = __reduce_add_sync(CB_FULL, (uint32_t)s.W);
    *tot = all;
    *g0 = cb_range_start(all, p.nc, c); *g1 = cb_range_start(all, p.nc, c + 1);
    const uint32_t g = (uint32_t)*g0;
    uint32_t run = 0;
    for (int rg = 0; rg < cb_max_row_groups(p); ++rg) {
        const uint32_t w = (uint32_t)s.w_of(p.Hkv, rg);
        uint32_t inc = w;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t t = __shfl_up_sync(CB_FULL, inc, o);
            if (lane >= o) inc += t;
        }
        const uint32_t pre = run + inc - w, hit = __ballot_sync(CB_FULL, w > 0u && g >= pre && g < pre + w);
        if (hit) {
            const int l = __ffs(hit) - 1;
            *rg_out = rg; *b_out = l; *pre_out = __shfl_sync(CB_FULL, pre, l);
            break;
        }
        run += __shfl_sync(CB_FULL, inc, 31);
    }
    return true;
}

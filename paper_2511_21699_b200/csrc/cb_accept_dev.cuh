// Device code of the greedy acceptance (Section 3.2), shared by the acceptance kernel and by the kernel that goes on to the
// next step's update and draft in the same launch: packed (value, index) maxima, streaming loads, the walk of a tree.
#pragma once
#include "cb_common.cuh"

namespace {

// Order-preserving map of a finite float to uint32 (larger float -> larger integer). -0 is folded into +0
// first so that equal values compare equal.
__device__ __forceinline__ uint32_t f2ord(float x) {
    x += 0.0f;
    const uint32_t u = __float_as_uint(x);
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}
// Packed key: larger value wins, then the smaller index.
__device__ __forceinline__ unsigned long long pack(float x, uint32_t idx) {
    return ((unsigned long long)f2ord(x) << 32) | (unsigned long long)(0xFFFFFFFFu - idx);
}
__device__ __forceinline__ unsigned long long umax64(unsigned long long a, unsigned long long b) { return a > b ? a : b; }

// The ordered values of a 16-byte vector of logits.
template <bool BF16>
__device__ __forceinline__ void ordered(const uint4& x, uint32_t (&o)[BF16 ? 8 : 4]) {
    const uint32_t w[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        if (BF16) { o[2 * q] = f2ord(__uint_as_float(w[q] << 16)); o[(2 * q + 1) % (BF16 ? 8 : 4)] = f2ord(__uint_as_float(w[q] & 0xFFFF0000u)); }
        else o[q] = f2ord(__uint_as_float(w[q]));
    }
}
// A thread's running maximum over such vectors: the value, and the first vector that has it.  Which of the vector's logits it is is
// looked up at the end, 5 instructions a logit where a packed (value, index) pair for each takes 8, for 16 registers more: for the grids
// that are resident at once, whose threads have the registers and whose chain of round trips the packing lengthens (a third of the 4 k
// cycles from the first load to the last comparison of one sequence over 32 k tokens); a larger grid waits for its logits either way.
template <bool BF16>
struct VectorMax {
    static constexpr int N = BF16 ? 8 : 4;
    uint32_t top = 0u, at = 0xFFFFFFFFu;      // ordered value; index of the vector's first logit
    uint4 x = {0u, 0u, 0u, 0u};
    __device__ __forceinline__ void take(const uint4& v, uint32_t id) {
        uint32_t o[N];
        ordered<BF16>(v, o);
        uint32_t m = o[0];
#pragma unroll
        for (int j = 1; j < N; ++j) m = max(m, o[j]);
        if (m > top || at == 0xFFFFFFFFu) { top = m; at = id; x = v; }
    }
    __device__ __forceinline__ unsigned long long packed() const {
        if (at == 0xFFFFFFFFu) return 0ull;
        uint32_t o[N], k = 0;
        ordered<BF16>(x, o);
#pragma unroll
        for (int j = N - 1; j >= 0; --j) if (o[j] == top) k = (uint32_t)j;
        return ((unsigned long long)top << 32) | (unsigned long long)(0xFFFFFFFFu - (at + k));
    }
};
// The largest packed maximum of a warp's lanes.
__device__ __forceinline__ unsigned long long warp_max(unsigned long long x) {
    const uint32_t hi = __reduce_max_sync(CB_FULL, (uint32_t)(x >> 32));
    const uint32_t lo = __reduce_max_sync(CB_FULL, (uint32_t)(x >> 32) == hi ? (uint32_t)x : 0u);
    return ((unsigned long long)hi << 32) | lo;
}

// The logits are read once: no L1 allocation, and first to leave L2 (the tables of the step's other kernels stay).
__device__ __forceinline__ uint64_t l2_evict_first_policy() {
    uint64_t pol;
    asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(pol));
    return pol;
}
__device__ __forceinline__ uint4 ldg_stream4u(const void* p, uint64_t pol) {
    uint4 v;
    asm volatile("ld.global.nc.L1::no_allocate.L2::cache_hint.v4.u32 {%0,%1,%2,%3}, [%4], %5;"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p), "l"(pol));
    return v;
}

// An atomic add that orders this thread's writes before it and the block's reads behind it (with the barrier that follows).
__device__ __forceinline__ uint32_t add_acq_rel(uint32_t* p, uint32_t v) {
    uint32_t old;
    asm volatile("atom.add.acq_rel.gpu.global.u32 %0, [%1], %2;" : "=r"(old) : "l"(p), "r"(v) : "memory");
    return old;
}

// What the walk needs beside the tree, in shared memory: a word per node, and the winner's path from its end to the root.
struct WalkSmem { uint16_t up[CB_MAX_T]; uint16_t path[CB_MAX_T]; };

// Walk of one sequence by one warp (n <= 128 nodes, parents precede children).
// tk, pa, de: the sequence's own tree rows (shared or global memory).  emit: if not null, the first 256 emitted tokens (m accepted
// ones, then the target's next) are left there too; *have: how many tokens are emitted.
// A node is verified if it and all its ancestors but the root match their parents' targets.  Every node knows its own match; a word
// holds "some node on the way to here does not match" and the ancestor that the way has reached, and doubles its reach with
// every round: 3 to 4 rounds for the usual depths.  Climbing node by node, with the path written from one lane, the walk took
// 4.4 k of the 13.7 k cycles of one sequence's acceptance over 32 k tokens.
__device__ __noinline__ void accept_walk(int b, int Dmax, const int32_t* tk, const int32_t* pa, const int32_t* de, int n,
                            const int32_t* target_s /*shared, [T]*/, WalkSmem& ws,
                            int32_t* __restrict__ n_accept, int32_t* __restrict__ accept_nodes,
                            int32_t* __restrict__ out_tokens, int lane, int32_t* emit = nullptr, int* have = nullptr) {
    constexpr int PER = CB_MAX_T / 32;
    constexpr uint32_t kBad = 0x100u;
    uint32_t up[PER];
#pragma unroll
    for (int q = 0; q < PER; ++q) {
        const int i = q * 32 + lane;
        up[q] = 0u;
        if (i > 0 && i < n) {
            const int p = pa[i];
            if (p < 0 || p >= i) up[q] = kBad;                  // malformed tree: treat as unverified
            else up[q] = (uint32_t)p | (tk[i] == target_s[p] ? 0u : kBad);
        }
        if (i < n) ws.up[i] = (uint16_t)up[q];
    }
    for (int round = 0; round < 8; ++round) {
        bool more = false;
#pragma unroll
        for (int q = 0; q < PER; ++q) more = more || (up[q] & 0xFFu) != 0u;
        if (!__any_sync(CB_FULL, more)) break;
        __syncwarp();
#pragma unroll
        for (int q = 0; q < PER; ++q)
            if ((up[q] & 0xFFu) != 0u) { const uint32_t a = ws.up[up[q] & 0xFFu]; up[q] = (a & 0xFFu) | ((a | up[q]) & kBad); }
        __syncwarp();
#pragma unroll
        for (int q = 0; q < PER; ++q) if (q * 32 + lane < n) ws.up[q * 32 + lane] = (uint16_t)up[q];
    }
    // key = (depth << 8) | (255 - index) for verified nodes: max = deepest, lowest index among ties
    uint32_t best = 0;
#pragma unroll
    for (int q = 0; q < PER; ++q) {
        const int i = q * 32 + lane;
        if (i >= n) break;
        // a depth outside [0, Dmax] cannot come from the drafter (malformed input): such a node counts as unverified, so the
        // winner's depth always fits the output rows
        const int d = de[i];
        if (!(up[q] & kBad) && d >= 0 && d <= Dmax) best = max(best, ((uint32_t)d << 8) | (uint32_t)(255 - i));
    }
    best = __reduce_max_sync(CB_FULL, best);
    int node = n > 0 ? 255 - (int)(best & 255u) : 0;
    int m = n > 0 ? (int)(best >> 8) : 0;
    if (node >= n) { node = 0; m = 0; }                        // nothing verified, not even the root (malformed input)
    int hops = 0;
    if (lane == 0)
        for (int c = node; hops < m && c > 0; c = pa[c]) ws.path[hops++] = (uint16_t)c;
    hops = __shfl_sync(CB_FULL, hops, 0);
    __syncwarp();
    const int32_t bonus = n > 0 ? target_s[node] : -1;
    for (int k = lane; k <= Dmax; k += 32) {
        const int j = m - 1 - k;                                // position on the path, counted from its end
        const int c = j >= 0 && j < hops ? (int)ws.path[j] : -1;
        const int32_t t = c >= 0 ? tk[c] : (k == m ? bonus : -1);
        if (k < Dmax) accept_nodes[(size_t)b * Dmax + k] = c;
        out_tokens[(size_t)b * (Dmax + 1) + k] = t;
        if (emit && k < 256) emit[k] = t;
    }
    if (lane == 0) {
        n_accept[b] = m;
        if (have) *have = n > 0 ? m + 1 : 0;
    }
}

// The work of one CTA of the acceptance grid (row chunk ck = blockIdx.x, node i = blockIdx.y, sequence b = blockIdx.z): its
// chunk of the node's logits row is reduced into the row's packed maximum; the last CTA of the sequence to arrive turns the
// maxima into the target's tokens, walks the tree and writes the result.  Returns true in that CTA (all its threads), after
// the result has been written; false in all others.  n: nodes of the sequence's tree.  beside(k): what the threads from 128 on (k = 0 ...) of that CTA do meanwhile.
// UN: 16-byte loads in flight per thread.  A grid that is resident at once is as long as its chain of round trips and takes all of
// its 32 KB chunk (8 loads a thread) at once; a larger one has enough in flight with 4 and needs the registers for more CTAs.
template <bool BF16, int UN, typename Beside>
__device__ __forceinline__ bool accept_rows(
    int T, int V, int Dmax, int chunk, int chunks_per_row, const void* __restrict__ logits, int64_t row_stride,
    const int32_t* __restrict__ tok, const int32_t* __restrict__ par, const int32_t* __restrict__ dep,
    int n, unsigned long long* rowmax, uint32_t* ticket,
    int32_t* __restrict__ n_accept, int32_t* __restrict__ accept_nodes, int32_t* __restrict__ out_tokens,
    int32_t* __restrict__ target_out, Beside&& beside, int32_t* emit = nullptr, int* have = nullptr) {
    const int b = blockIdx.z, i = blockIdx.y, ck = blockIdx.x, tid = threadIdx.x;
    // Rows past the tree have nothing to add and do not queue for the ticket either (hundreds of atomics on one word at
    // batch 1); an empty tree keeps row 0's CTAs, one of which writes the empty result.
    if (i >= max(n, 1)) return false;
    __shared__ unsigned long long s_red[8];
    __shared__ int32_t s_target[CB_MAX_T], s_tok[CB_MAX_T], s_par[CB_MAX_T], s_dep[CB_MAX_T];
    __shared__ WalkSmem s_walk;
    __shared__ int s_last;
    if (i < n) {
        const int v0 = ck * chunk, v1 = min(V, v0 + chunk);
        unsigned long long best = 0ull;
        const uint64_t pol = l2_evict_first_policy();
        if (!BF16) {
            const float* rowp = (const float*)logits + ((size_t)b * T + i) * row_stride;
            // head up to a 16-byte boundary, vector body, scalar tail
            int v = v0;
            const uintptr_t a = (uintptr_t)(rowp + v);
            int head = (int)(((16 - (a & 15)) & 15) >> 2);
            head = min(head, v1 - v);
            if (tid < head) best = pack(rowp[v + tid], (uint32_t)(v + tid));
            v += head;
            const int nvec = (v1 - v) >> 2;
            const float* base = rowp + v;
            VectorMax<false> vm;                                 // UN > 4
            for (int k = tid; k < nvec; k += blockDim.x * UN) {
                uint4 x[UN];
                int kk[UN];
#pragma unroll
                for (int u = 0; u < UN; ++u) { kk[u] = k + u * blockDim.x; if (kk[u] < nvec) x[u] = ldg_stream4u(base + 4 * (size_t)kk[u], pol); }
#pragma unroll
                for (int u = 0; u < UN; ++u) if (kk[u] < nvec) {
                    const uint32_t id = (uint32_t)(v + 4 * kk[u]);
                    if (UN > 4) {
                        vm.take(x[u], id);
                    } else {
                        best = umax64(best, pack(__uint_as_float(x[u].x), id));
                        best = umax64(best, pack(__uint_as_float(x[u].y), id + 1));
                        best = umax64(best, pack(__uint_as_float(x[u].z), id + 2));
                        best = umax64(best, pack(__uint_as_float(x[u].w), id + 3));
                    }
                }
            }
            if (UN > 4) best = umax64(best, vm.packed());
            const int tail0 = v + 4 * nvec;
            if (tail0 + tid < v1) best = umax64(best, pack(rowp[tail0 + tid], (uint32_t)(tail0 + tid)));
        } else {
            const __nv_bfloat16* rowp = (const __nv_bfloat16*)logits + ((size_t)b * T + i) * row_stride;
            int v = v0;
            const uintptr_t a = (uintptr_t)(rowp + v);
            int head = (int)(((16 - (a & 15)) & 15) >> 1);
            head = min(head, v1 - v);
            if (tid < head) best = pack(__bfloat162float(rowp[v + tid]), (uint32_t)(v + tid));
            v += head;
            const int nvec = (v1 - v) >> 3;
            const __nv_bfloat16* base = rowp + v;
            VectorMax<true> vm;
            for (int k = tid; k < nvec; k += blockDim.x * UN) {
                uint4 x[UN];
                int kk[UN];
#pragma unroll
                for (int u = 0; u < UN; ++u) { kk[u] = k + u * blockDim.x; if (kk[u] < nvec) x[u] = ldg_stream4u(base + 8 * (size_t)kk[u], pol); }
#pragma unroll
                for (int u = 0; u < UN; ++u) if (kk[u] < nvec) {
                    const uint32_t id = (uint32_t)(v + 8 * kk[u]);
                    if (UN > 4) {
                        vm.take(x[u], id);
                    } else {
                        const uint32_t wds[4] = {x[u].x, x[u].y, x[u].z, x[u].w};
#pragma unroll
                        for (int q = 0; q < 4; ++q) {
                            best = umax64(best, pack(__uint_as_float(wds[q] << 16), id + 2 * q));
                            best = umax64(best, pack(__uint_as_float(wds[q] & 0xFFFF0000u), id + 2 * q + 1));
                        }
                    }
                }
            }
            if (UN > 4) best = umax64(best, vm.packed());
            const int tail0 = v + 8 * nvec;
            if (tail0 + tid < v1) best = umax64(best, pack(__bfloat162float(rowp[tail0 + tid]), (uint32_t)(tail0 + tid)));
        }
        best = warp_max(best);
        if ((tid & 31) == 0) s_red[tid >> 5] = best;
        __syncthreads();
        if (tid < 32) {
            best = warp_max(tid < (int)(blockDim.x >> 5) ? s_red[tid] : 0ull);
            if (tid == 0) atomicMax(&rowmax[(size_t)b * T + i], best);
        }
    }
    // The last CTA of this sequence to arrive owns the walk (and re-zeroes the scratch for the next call).
    if (tid == 0) {
        const uint32_t total = gridDim.x * (uint32_t)max(n, 1);
        s_last = (add_acq_rel(&ticket[b], 1u) == total - 1u) ? 1 : 0;
    }
    __syncthreads();
    if (!s_last) return false;
    static_assert(CB_MAX_T <= 128, "the first 128 threads have a node each, the others do what goes beside");
    if (tid >= 128) {
        beside(tid - 128);
    } else if (tid < T) {
        // the tree's rows come along, so that the walk below reads shared memory
        int32_t tg = -1, tk = -1, pa = -1, de = -1;
        if (tid < n) {
            const size_t at = (size_t)b * T + tid;
            tk = tok[at]; pa = par[at]; de = dep[at];
            const unsigned long long r = atomicExch(&rowmax[at], 0ull);
            tg = (int32_t)(0xFFFFFFFFu - (uint32_t)(r & 0xFFFFFFFFull));
        }
        s_target[tid] = tg; s_tok[tid] = tk; s_par[tid] = pa; s_dep[tid] = de;
        if (target_out) target_out[(size_t)b * T + tid] = tg;
    }
    if (tid == 0) ticket[b] = 0u;
    __syncthreads();
    if (tid < 32) accept_walk(b, Dmax, s_tok, s_par, s_dep, n, s_target, s_walk, n_accept, accept_nodes, out_tokens, tid, emit, have);
    return true;
}

}  // namespace

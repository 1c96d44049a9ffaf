// Column engine: IC, and LT in the counting form, on graphs whose state of up to 32 trials fits the
// shared memory of one SM.
//
// Trials never interact, so a block takes a column of up to 32 consecutive trials of one item through
// all of its steps by itself: the state of every node in those trials is one 32-bit word per array, in
// shared memory, a step ends with one block barrier, and the whole call is one launch.  The pass engine
// (cnd_sim.cu) pays launches, counter copies and a host round trip for every step, about 40 us on a
// 1,000-node graph whose steps hold a few hundred edges each, and its batches run as many steps as
// their deepest item.
//
//   vis[v]      trials in which v is active
//   nx[v]       trials activated in the current step
//   lists       the frontier's nodes and bits and the nodes of the next one; the first `cap` entries in
//               shared memory, the others in global memory (so that 8 bytes per node, not 16, decide how
//               many columns an SM holds: steps are latency-bound and want several)
//   planes      LT: 32-lane bit-sliced in-neighbour counters, L_v words per node (see k_lt_init in
//               cnd_sim.cu for why the carry out of the top plane is the activation)
//
// A warp takes up to 32 frontier nodes, spreads their out-edges over its lanes (a warp-wide or of the
// rows' first positions gives each lane the node of its edge), and IC draws the coins of the (edge,
// 4-trial block) pairs that need one from a per-warp queue, 32 at a time.  Rows of kHub edges and more are
// left to the whole block after the others.
//
// Columns are handed out by an atomic counter, since their depths differ.  What bounds a step is the
// latency of its chain (row offsets, edges, target, coins, three shared-memory atomics, two barriers)
// where its frontier is small, and issue slots where it is large (62 % issue active, ncu, on a dense
// Watts-Strogatz 10k).  Against the pass engine's host step loop (GB300): G(1000, 10000), p = 0.1, 1,000
// trials 1,766 -> 126 us per call, Watts-Strogatz 10k U[0, 1] 2,184 -> 538 us, CELF k = 10 on the
// 7-regular graph (n = 5,000) 146 -> 20.7 ms.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>

#include "cnd_cols.cuh"

namespace cnd {
namespace {

constexpr int kHub = 256;       // out-edges from which the whole block expands a node
constexpr int kHubCap = 64;     // hubs set aside per step (more are expanded by the warp that finds them)

struct ColItem {
    int64_t out0;     // position of the item's first trial in the spread output
    uint64_t key;
    int32_t s_begin, s_end;
    int32_t trials;
    int32_t col0;     // its first column
};

struct ColParams {
    int32_t n, n_items;
    int32_t bits;             // trials per column (a multiple of 4, at most 32)
    int32_t n_cols;
    int32_t cap;              // list entries kept in shared memory
    uint16_t *over_node;      // [blocks][2][n] list entries beyond cap
    uint32_t *over_bits;      // [blocks][n]
    const int32_t *row_ptr;
    const uint2 *edge;        // {col, IC threshold} or {col, counter tag}
    const ColItem *items;
    const int32_t *seeds;
    const int32_t *cnt_off;   // LT: first plane of each node
    const uint32_t *unit_w;
    int64_t first_trial;
    int32_t *spread, *count;
    unsigned long long *checks, *level_counts;
    int32_t lc_len, max_levels;
    unsigned long long timeout_ns;
    CallFlags *flags;
};

// Coin blocks to draw, a ring: {edge, threshold, target, (block << 4) | wanted trials of the block}.
struct __align__(16) WarpQueue {
    uint4 q[64];
};

// The warp's frontier nodes that have edges to expand, in order: {edge id of the warp's t-th edge
// less t, frontier bits}.
struct __align__(8) WarpNodes {
    uint2 node[32];
};

struct BlockState {
    int32_t n_list[3];   // frontier sizes, by step mod 3
    int32_t n_hub[3];
    int32_t col, item;
    int32_t stop;        // first step not to run (set by the time limit)
    uint32_t spread[32];
    uint2 hub[kHubCap];  // {node, frontier bits}
    __align__(16) uint32_t rk[20];
};

// True once the time limit, measured from the call's first step (t0), has passed; the call then times out.  A
// timer that reads before another SM's t0 is not past it.
__device__ __forceinline__ bool past_limit(const ColParams &p) {
    if (p.timeout_ns == 0) return false;
    if (*(volatile int32_t *)&p.flags->timed_out) return true;
    const unsigned long long t0 = *(volatile unsigned long long *)&p.flags->t0, now = global_ns();
    if (t0 == 0 || now <= t0 || now - t0 <= p.timeout_ns) return false;
    p.flags->timed_out = 1;
    return true;
}

// 32 x 32 bit transpose over a warp: bit i of lane b's result is bit b of lane i's x.
__device__ __forceinline__ uint32_t transpose32(uint32_t x) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int s = 16; s; s >>= 1) {
        const uint32_t m = s == 16 ? 0x0000FFFFu : s == 8 ? 0x00FF00FFu : s == 4 ? 0x0F0F0F0Fu : s == 2 ? 0x33333333u : 0x55555555u;
        const uint32_t y = __shfl_xor_sync(kFull, x, s);
        x = (lane & s) ? ((x & ~m) | ((y & ~m) >> s)) : ((x & m) | ((y & m) << s));
    }
    return x;
}

// The parts of a step that its edges need.
struct StepCtx {
    uint32_t *vis, *nx;
    uint16_t *lnext, *gnext;  // the next frontier's nodes: entries below cap, and beyond
    int32_t *n_next;
    int32_t cap;
    uint32_t *planes;
    const uint2 *edge;
    const uint32_t *rk;
    uint64_t g0;
    uint32_t gained;  // activations of this thread in the step
    uint32_t qh, qt;  // the warp's queued blocks: entries qh .. qt - 1 (mod 64)

    // v becomes active in the trials of `bits` where it is not yet
    __device__ __forceinline__ void activate(uint32_t v, uint32_t bits) {
        const uint32_t nw = bits & ~atomicOr(&vis[v], bits);
        if (nw) {
            gained += __popc(nw);
            if (atomicOr(&nx[v], nw) == 0u) {
                const int i = atomicAdd(n_next, 1);
                (i < cap ? lnext : gnext)[i] = (uint16_t)v;
            }
        }
    }
};

// One IC draw: the coins of edge e in the 4-trial block g, as 4 bits.
__device__ __forceinline__ uint32_t coins(const StepCtx &s, uint32_t e, uint32_t thr, uint32_t j) {
    const uint64_t g = s.g0 + j;
    uint32_t c0 = e, c1 = (uint32_t)g, c2 = 0u, c3 = (uint32_t)(g >> 32);
#pragma unroll
    for (int h = 0; h < 5; ++h) {
        const uint4 k = reinterpret_cast<const uint4 *>(s.rk)[h];
        const uint32_t kk[4] = {k.x, k.y, k.z, k.w};
#pragma unroll
        for (int r = 0; r < 4; r += 2) {
            const uint64_t a = (uint64_t)0xD2511F53u * c0;
            const uint64_t b = (uint64_t)0xCD9E8D57u * c2;
            c0 = (uint32_t)(b >> 32) ^ c1 ^ kk[r];
            c2 = (uint32_t)(a >> 32) ^ c3 ^ kk[r + 1];
            c1 = (uint32_t)b;
            c3 = (uint32_t)a;
        }
    }
    return (uint32_t)(c0 < thr) | ((uint32_t)(c1 < thr) << 1) | ((uint32_t)(c2 < thr) << 2) | ((uint32_t)(c3 < thr) << 3);
}

// Draw the first cnt <= 32 queued blocks, one per lane.
__device__ __forceinline__ void draw_queued(StepCtx &s, const WarpQueue &wq, uint32_t cnt) {
    const uint32_t lane = threadIdx.x & 31;
    __syncwarp();
    if (lane < cnt) {
        const uint4 t = wq.q[(s.qh + lane) & 63u];
        const uint32_t j = t.w >> 4;
        const uint32_t live = coins(s, t.x, t.y, j) & t.w & 15u;
        if (live) s.activate(t.z, live << (4 * j));
    }
    s.qh += cnt;
    __syncwarp();
}

// Expand one edge per lane, {v, thr} = ed, by the frontier bits f (0: nothing to do in this lane).  IC: the
// 4-trial blocks with a trial to decide are queued, one per lane and round, and drawn 32 at a time; fewer than
// 32 stay queued for the next edges (a chunk of 32 edges has 14 on average on a dense Watts-Strogatz 10k at 8
// trials per column: drawn chunk by chunk, more than half of the lanes idle, a call took 603 us, now 538).
template <int MODEL>
__device__ __forceinline__ void expand(StepCtx &s, WarpQueue &wq, uint32_t e, uint2 ed, uint32_t f) {
    const int lane = threadIdx.x & 31;
    const uint32_t v = ed.x, thr = ed.y;
    uint32_t c = 0;
    if (f && thr != 0u) c = f & ~*(volatile uint32_t *)&s.vis[v];
    if (MODEL == 1) {
        if (c) {  // one bit-sliced increment of v's counter by the trials of c
            const uint32_t L = thr & 31u;
            uint32_t *pl = s.planes + (thr >> 5);
            for (uint32_t i = 0; i < L && c; ++i) c &= atomicXor(pl + i, c);
            if (c) s.activate(v, c);
        }
        return;
    }
    if (c && thr == kAlways) {
        s.activate(v, c);
        c = 0;
    }
    uint32_t nm = c | (c >> 1);
    nm = (nm | (nm >> 2)) & 0x11111111u;  // the 4-trial blocks to draw
    for (;;) {
        const uint32_t m = __ballot_sync(kFull, nm != 0u);
        if (m == 0u) return;
        if (nm) {
            const uint32_t b = (uint32_t)__ffs(nm) - 1u;
            nm &= nm - 1u;
            wq.q[(s.qt + __popc(m & ((1u << lane) - 1u))) & 63u] = make_uint4(e, thr, v, (b << 2) | ((c >> b) & 15u));
        }
        s.qt += __popc(m);
        if (s.qt - s.qh >= 32u) draw_queued(s, wq, 32u);
    }
}

template <int MODEL>
__global__ void __launch_bounds__(1024, 1) k_columns(ColParams p) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ BlockState S;
    const int n = p.n, tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int n_warps = blockDim.x >> 5;
    WarpQueue *queues = reinterpret_cast<WarpQueue *>(smem);
    const int n4 = (n + 3) & ~3;
    WarpNodes *wnodes = reinterpret_cast<WarpNodes *>(smem + (MODEL == 0 ? sizeof(WarpQueue) * n_warps : 0));
    uint32_t *vis = reinterpret_cast<uint32_t *>(wnodes + n_warps);
    uint32_t *nx = vis + n4, *lbits = nx + n4;
    const int cap = p.cap;  // a multiple of 8
    uint16_t *la = reinterpret_cast<uint16_t *>(lbits + cap), *lb = la + cap;
    uint32_t *planes = reinterpret_cast<uint32_t *>(lb + cap);
    uint16_t *const ga = p.over_node + (size_t)blockIdx.x * 2 * n, *const gb = ga + n;
    uint32_t *const gbits = p.over_bits + (size_t)blockIdx.x * n;
    WarpQueue &wq = queues[MODEL == 0 ? wid : 0];
    uint2 *wn = wnodes[wid].node;
    const uint32_t lt = (1u << lane) - 1u, le = lt | (1u << lane);
    unsigned long long ck = 0;
    for (;;) {
        if (tid == 0) {
            int c = atomicAdd(&p.flags->next_column, 1);
            if (c < p.n_cols && past_limit(p)) c = p.n_cols;  // the columns left are not run
            S.col = c;
        }
        __syncthreads();
        const int col = S.col;
        if (col >= p.n_cols) break;
        // ---- clear the state; warp 0 finds the column's item (the last one with col0 <= col)
        for (int i = tid; i < 2 * (n4 >> 2); i += blockDim.x)
            reinterpret_cast<uint4 *>(vis)[i] = make_uint4(0u, 0u, 0u, 0u);
        if (tid < 32) {
            int lo = 0, hi = p.n_items;  // item in [lo, hi)
            while (hi - lo > 1) {
                const int step = (hi - lo + 31) / 32;
                const int probe = lo + lane * step;
                const unsigned ok = __ballot_sync(kFull, probe < hi && p.items[probe].col0 <= col);
                lo += (31 - __clz(ok)) * step;
                hi = min(hi, lo + step);
            }
            if (lane == 0) {
                S.item = lo;
                S.stop = 0x7FFFFFFF;
                S.n_list[0] = S.n_list[1] = S.n_list[2] = 0;
                S.n_hub[0] = S.n_hub[1] = S.n_hub[2] = 0;
                uint32_t k0 = (uint32_t)p.items[lo].key, k1 = (uint32_t)(p.items[lo].key >> 32);
                for (int r = 0; r < 10; ++r) {
                    S.rk[2 * r] = k0;
                    S.rk[2 * r + 1] = k1;
                    k0 += 0x9E3779B9u;
                    k1 += 0xBB67AE85u;
                }
            }
            S.spread[lane] = 0u;
        }
        __syncthreads();
        const ColItem it = p.items[S.item];
        const int t0 = (col - it.col0) * p.bits;  // first trial of the column within the item
        const int nt = min(p.bits, it.trials - t0);
        const uint32_t valid = nt >= 32 ? 0xFFFFFFFFu : ((1u << nt) - 1u);
        const uint64_t g0 = (uint64_t)(p.first_trial + t0) >> 2;
        if (MODEL == 1) {
            // counter starts c0 = 2^L - 1 - floor(theta / w) (0 when negative), a thread per node
            for (int v = tid; v < n; v += blockDim.x) {
                const int o0 = p.cnt_off[v];
                const int L = p.cnt_off[v + 1] - o0;
                if (L == 0) continue;
                const uint32_t wv = p.unit_w[v];
                const uint32_t top = L >= 32 ? 0xFFFFFFFFu : ((1u << L) - 1u);
                for (int i = 0; i < L; ++i) planes[o0 + i] = 0u;
                for (int j = 0; 4 * j < nt; ++j) {
                    const uint64_t g = g0 + (uint64_t)j;
                    const U4 th = philox4x32_10((uint32_t)v, (uint32_t)g, 1u, (uint32_t)(g >> 32), (uint32_t)it.key,
                                                (uint32_t)(it.key >> 32));
                    const uint32_t tv[4] = {th.x, th.y, th.z, th.w};
                    uint32_t c0[4];
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        const uint32_t q = tv[k] / wv;
                        c0[k] = q < top ? top - q : 0u;
                    }
                    for (int i = 0; i < L; ++i) {
                        const uint32_t nib = ((c0[0] >> i) & 1u) | (((c0[1] >> i) & 1u) << 1) |
                                             (((c0[2] >> i) & 1u) << 2) | (((c0[3] >> i) & 1u) << 3);
                        planes[o0 + i] |= nib << (4 * j);
                    }
                }
            }
        }
        // ---- step 0: the seeds (duplicates count once)
        for (int i = it.s_begin + tid; i < it.s_end; i += blockDim.x) {
            const int u = p.seeds[i];
            if (u < 0 || u >= n) {
                p.flags->bad_seed = 1;
                continue;
            }
            if (atomicOr(&vis[u], valid) == 0u) {
                nx[u] = valid;
                const int i = atomicAdd(&S.n_list[0], 1);
                (i < cap ? la : ga)[i] = (uint16_t)u;
            }
        }
        if (tid == 0 && p.timeout_ns) atomicCAS(&p.flags->t0, 0ull, global_ns());
        __syncthreads();
        if (tid == 0 && p.lc_len > 0 && S.n_list[0]) atomicAdd(&p.level_counts[0], (unsigned long long)S.n_list[0] * nt);
        uint16_t *lcur = la, *lnext = lb, *gcur = ga, *gnext = gb;
        for (int step = 0;; ++step) {
            const int slot = step % 3, nslot = (step + 1) % 3;
            const int F = S.n_list[slot];
            if (F == 0 || step >= S.stop) break;
            if (p.max_levels > 0 && step >= p.max_levels) {
                // the out-edges of the last frontier count as checked, as every active node's do
                for (int i = tid; i < F; i += blockDim.x) {
                    const int u = (i < cap ? lcur : gcur)[i];
                    ck += (unsigned long long)__popc(nx[u]) * (unsigned long long)(p.row_ptr[u + 1] - p.row_ptr[u]);
                }
                if (tid == 0) p.flags->limit = 1;
                break;
            }
            // take the frontier's bits out of nx, which then collects the next frontier's
            for (int i = tid; i < F; i += blockDim.x) {
                const int u = (i < cap ? lcur : gcur)[i];
                (i < cap ? lbits : gbits)[i] = nx[u];
                nx[u] = 0u;
            }
            __syncthreads();
            StepCtx s{vis, nx, lnext, gnext, &S.n_list[nslot], cap, planes, p.edge, S.rk, g0, 0u, 0u, 0u};
            if (tid == 0) {
                // the slots of the step after next: nobody reads or writes them in this one
                S.n_list[(step + 2) % 3] = 0;
                S.n_hub[nslot] = 0;
                if (past_limit(p)) S.stop = step + 1;  // not this step: other threads may not have read it yet
            }
            // nodes per warp: all warps get some while there are enough
            const int G = min(32, (F + n_warps - 1) / n_warps);
            for (int base = wid * G; base < F; base += n_warps * G) {
                int rs = 0, deg = 0;
                uint32_t f = 0;
                if (lane < G && base + lane < F) {
                    const int i = base + lane;
                    const int u = (i < cap ? lcur : gcur)[i];
                    f = (i < cap ? lbits : gbits)[i];
                    rs = __ldg(&p.row_ptr[u]);
                    deg = __ldg(&p.row_ptr[u + 1]) - rs;
                    ck += (unsigned long long)__popc(f) * (unsigned long long)deg;
                    if (deg >= kHub) {
                        const int h = atomicAdd(&S.n_hub[slot], 1);
                        if (h < kHubCap) {
                            S.hub[h] = make_uint2((uint32_t)u, f);
                            deg = 0;
                        }
                    }
                }
                int incl = deg;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const int x = __shfl_up_sync(kFull, incl, o);
                    if (lane >= o) incl += x;
                }
                const int total = __shfl_sync(kFull, incl, 31);
                if (total == 0) continue;
                const int start = incl - deg;
                const unsigned nz = __ballot_sync(kFull, deg > 0);
                if (deg > 0) wn[__popc(nz & lt)] = make_uint2((uint32_t)(rs - start), f);
                __syncwarp();
                // the node of edge t = e0 + lane: nodes whose first edge lies at or before t, less one
                // (nodes starting in this chunk of 32 edges from a warp-wide or, earlier ones counted)
                int before = 0;
                auto owner = [&](int e0) {
                    const int at = start - e0;
                    const unsigned m = __reduce_or_sync(kFull, (deg > 0 && at >= 0 && at < 32) ? 1u << at : 0u);
                    const int o = before + __popc(m & le) - 1;
                    before += __popc(m);
                    return o;
                };
                uint2 nd = wn[owner(0)];
                uint32_t e = nd.x + lane, fe = lane < total ? nd.y : 0u;
                uint2 ed = make_uint2(0u, 0u);
                if (lane < total) ed = __ldg(&p.edge[e]);
                for (int e0 = 0; e0 < total; e0 += 32) {
                    // the next 32 edges' records load while these are expanded
                    uint32_t en = 0, fn = 0;
                    uint2 edn = make_uint2(0u, 0u);
                    if (e0 + 32 < total) {
                        nd = wn[owner(e0 + 32)];
                        if (e0 + 32 + lane < total) {
                            en = nd.x + (uint32_t)(e0 + 32 + lane);
                            fn = nd.y;
                            edn = __ldg(&p.edge[en]);
                        }
                    }
                    expand<MODEL>(s, wq, e, ed, fe);
                    e = en;
                    fe = fn;
                    ed = edn;
                }
                __syncwarp();
            }
            if (MODEL == 0 && s.qt != s.qh) draw_queued(s, wq, s.qt - s.qh);
            __syncthreads();
            const int H = min(S.n_hub[slot], kHubCap);
            if (H) {
                for (int h = 0; h < H; ++h) {
                    const uint2 hb = S.hub[h];
                    const int e0 = p.row_ptr[hb.x], e1 = p.row_ptr[hb.x + 1];
                    for (int e = e0 + 32 * wid; e < e1; e += 32 * n_warps)
                        expand<MODEL>(s, wq, (uint32_t)(e + lane), e + lane < e1 ? __ldg(&p.edge[e + lane]) : make_uint2(0u, 0u),
                                      e + lane < e1 ? hb.y : 0u);
                }
                if (MODEL == 0 && s.qt != s.qh) draw_queued(s, wq, s.qt - s.qh);
                __syncthreads();
            }
            if (step + 1 < p.lc_len) {
                uint32_t x = s.gained;
                for (int o = 16; o; o >>= 1) x += __shfl_xor_sync(kFull, x, o);
                if (lane == 0 && x) atomicAdd(&p.level_counts[step + 1], (unsigned long long)x);
            }
            uint16_t *x = lcur;
            lcur = lnext;
            lnext = x;
            x = gcur;
            gcur = gnext;
            gnext = x;
        }
        // ---- outputs: activations per trial (columns of vis) and per node
        uint32_t mine = 0;
        for (int v0 = 32 * wid; v0 < n; v0 += 32 * n_warps) {
            const uint32_t x = v0 + lane < n ? vis[v0 + lane] : 0u;
            if (!__any_sync(kFull, x != 0u)) continue;
            if (p.count && x) atomicAdd(&p.count[(size_t)S.item * n + v0 + lane], __popc(x));
            mine += __popc(transpose32(x));
        }
        if (mine) atomicAdd(&S.spread[lane], mine);
        __syncthreads();
        if (p.spread && tid < nt) p.spread[it.out0 + t0 + tid] = (int32_t)S.spread[tid];
        __syncthreads();
    }
    for (int o = 16; o; o >>= 1) ck += __shfl_xor_sync(kFull, ck, o);
    if (lane == 0 && ck) atomicAdd(p.checks, ck);
}

// Shapes of the launch: blocks per SM (1, 2 or 4, of 1024, 512 or 256 threads: 32 warps in all, the
// most at 64 registers) and list entries in shared memory, at least kMinCap (or all nodes).
struct ColShape {
    int per_sm = 0, threads = 0, cap = 0;
    size_t dyn = 0;
};
constexpr int kMinCap = 512;
constexpr size_t kSmSmem = 228 * 1024;        // per SM, of which each block takes 1 KB more than it asks for
constexpr size_t kMaxBlockSmem = 227 * 1024;  // per block
constexpr size_t kMaxDynamic = kMaxBlockSmem - sizeof(BlockState);

bool column_shape(int model, const cnd_graph_dev &G, int per_sm, ColShape &c) {
    if (G.n > kColMaxN) return false;
    const size_t n4 = ((size_t)G.n + 3) & ~(size_t)3;
    const int threads = 1024 / per_sm;
    const size_t have = std::min(kSmSmem / per_sm - 1024, kMaxBlockSmem) - sizeof(BlockState) - 64;
    const size_t fixed = 8 * n4 + (sizeof(WarpNodes) + (model == 0 ? sizeof(WarpQueue) : 0)) * (size_t)(threads / 32) +
                         (model == 0 ? 0 : 4 * (size_t)G.lt_planes);
    const size_t all = (n4 + 7) & ~(size_t)7;  // entries for every node
    if (fixed + 8 * std::min<size_t>(kMinCap, all) > have) return false;
    c.per_sm = per_sm;
    c.threads = threads;
    c.cap = (int)std::min(all, (have - fixed) / 8 & ~(size_t)7);
    c.dyn = fixed + 8 * (size_t)c.cap;
    return true;
}

// Blocks per SM and trials per column (a multiple of 4, one coin block), by estimated time: a
// wave of columns takes a constant (the latency of its steps) and work in proportion to the
// trials (and 2 more: work that a check takes whatever its trials) and the edges, at a rate in
// proportion to the block's threads.  1,000 trials, blocks per SM / trials per column: G(1000, 10000)
// 2 / 4 133 us, 1 / 8 148; Watts-Strogatz 10k U[0, 1] 2 / 4 648 us, 1 / 8 575; BA 5k WC 255 and 269.
void choose_shape(int model, const cnd_graph_dev &G, int64_t trials, ColShape &c, int32_t &bits) {
    const double size = std::min(1.0, std::max(0.25, (double)G.m / 1e5));
    double best = 1e300;
    for (int per_sm = 4; per_sm >= 1; per_sm >>= 1) {
        ColShape k;
        if (!column_shape(model, G, per_sm, k)) continue;
        for (int b = 4; b <= 32; b += 4) {
            const double waves = std::ceil((double)((trials + b - 1) / b) / ((double)G.num_sms * per_sm));
            const double cost = waves * ((per_sm == 1 ? 10 : per_sm == 2 ? 9 : 8) + size * per_sm * (b + 2));
            if (cost < best) {
                best = cost;
                bits = b;
                c = k;
            }
        }
    }
}

// Whether the columns of a call on a graph of many edges are faster than its passes.  A column is one
// block's work, so a wave of columns takes its edges' time on one SM however few trials there are,
// where a pass spreads them over all; a pass takes some 48 us a step, and how many steps there are
// follows from how fast a cascade grows, G.ic_branching.
// IC up to a branching of 1.3, where cascades are long or touch little: always (kColMaxEdges; above 0.8 up to
// 1,000 edges a node).  Always too up to 90,000 edges, and up to kWideTrials * 4 trials without hub rows up to
// 200,000 edges or with a branching of up to 4.2 up to 260,000: of these, 1 % took over 1.05 times the passes' time,
// 1.1 at most.  Elsewhere by both estimated times, in us, the columns' with 0.3 of it on top: fits to
// 1,595 calls of 1 to 20,000 trials (G(n, p), Watts-Strogatz, BA and R-MAT, 12,000 to 3 M edges, U[0, 1], WC and
// uniform p) that leave 30 % (root mean square).  7 of 1,785 calls are left above 1.08 times the passes' time, at 1.28 at
// most; with no term for edges 443 are, up to 8 times: G(5000, p) of 1 M edges, p = 0.05, 64 trials 1.3 against 0.4
// ms, R-MAT 14 of 776,000 edges, p = 0.1, 1,000 trials 2.2 against 0.9 ms, G(20000, p) of 20 M edges, p = 0.1, one
// trial 13.2 against 0.4 ms.
// LT: the passes' pull steps count dense rows faster than atomics on shared memory; 1,000 nodes, 20,000 trials,
// 200 / 400 / 1,000 edges a node: 15.9 against 16.0 / 29.2 against 16.9 / 85 against 31 ms.
constexpr int64_t kWideTrials = 4096;

bool columns_pay(int model, const cnd_graph_dev &G, int64_t trials, int64_t words) {
    if (model == 1) return G.m <= 200ll * G.n;
    if (G.m > kColMaxEdges) return false;
    const double r = G.ic_branching;
    if (r <= 0.8 || (r <= 1.3 && G.m <= 1000ll * G.n) || G.m <= 90000) return true;
    if (trials <= 4 * kWideTrials && ((G.m <= 200000 && G.max_out_degree < kHub) || (G.m <= 260000 && r <= 4.2)))
        return true;
    ColShape c;
    int32_t bits = 0;
    choose_shape(model, G, trials, c, bits);
    const double columns = (double)std::max(words, (trials + bits - 1) / bits);
    const double waves = std::max(1.0, columns / ((double)G.num_sms * c.per_sm));
    const double steps = std::min(25.0, 3.0 + std::log((double)G.n) / std::log(r));
    const double onward = std::pow(r, -0.7);  // the larger r, the fewer checks before a node is active
    // hub rows are expanded one after the other
    const double hubs = G.max_out_degree >= kHub ? 1.0 + 0.023 * G.max_out_degree * (double)G.n / (double)G.m : 1.0;
    const double per_edge = (0.35 + 0.8 * (double)std::min<int64_t>(bits, std::max<int64_t>(2, trials)) * onward) * hubs * 1e-3;
    const double t_columns = 90.0 + waves * c.per_sm * (double)G.m * per_edge;
    const double t_passes = 160.0 + 48.0 * steps + 3.8e-4 * (double)G.m * (double)words * onward;
    return 1.3 * t_columns < t_passes;
}

}  // namespace

// Calls that run here.  Options that choose a form of the pass engine (width, work items, direction,
// deferral, statistics, 32-bit sums) get the pass engine.  So do dense graphs (columns_pay), and IC calls of
// many trials on the larger graphs: with that many the pass engine's words are full, and one check of 64 trials costs it less than
// two of 32 cost here.  The line is kWideTrials where an SM holds fewer than four columns (n > about
// 5,500) and there are hub rows (kHub edges and more: one block's work), four times that where it holds
// one column (n > about 12,000) and there are none.
// Measured against the pass engine (GB300; host step loop, its default):
//   1,000 trials:  G(1000, 10000) p = 0.1 1,267 -> 131 us; Watts-Strogatz 10k U[0, 1] 2,595 -> 756 us;
//                  BA 13k WC 2,067 -> 481 us; BA 20k U[0, 1] 867 -> 683 us; R-MAT 14 p = 0.1 923 -> 789 us
//   20,000 trials: BA 13k U[0, 1] 3.10 -> 3.72 ms, R-MAT 13 p = 0.1 2.88 -> 3.47 ms (BA 13k WC 7.4 -> 5.5 ms)
//   65,536 trials: Watts-Strogatz 10k p = 0.1 3.60 -> 1.27 ms, U[0, 1] 30.5 -> 20.0 ms
//   no hub rows:   G(20000, 200000) p = 0.1 10,000 trials 8.6 -> 2.5 ms; U[0, 1] 10,000 / 30,000 / 65,536 trials
//                  3.54 -> 3.55 / 8.4 -> 9.5 / 18.7 -> 19.0 ms
//   LT, any:       BA 5k 1,000 trials 2,395 -> 370 us, 65,536 trials 20.1 -> 8.1 ms
bool columns_fit(int model, const cnd_graph_dev &G, const cnd_sim_opts &o, int64_t trials, int64_t words) {
    if (model == 1 && (!G.lt_cnt_edge || o.lt_accumulate)) return false;
    if (o.word_bits || o.chunk_edges || o.direction != CND_DIR_AUTO || o.pull_permille || o.defer_bits || o.stats)
        return false;
    ColShape c;
    if (!column_shape(model, G, 1, c) || !columns_pay(model, G, trials, words)) return false;
    if (model == 1 || trials <= kWideTrials || column_shape(model, G, 4, c)) return true;
    return G.max_out_degree < kHub && (trials <= 4 * kWideTrials || column_shape(model, G, 2, c));
}

int32_t column_bits(int model, const cnd_graph_dev &G, int64_t trials) {
    ColShape c;
    int32_t bits = 0;
    choose_shape(model, G, trials, c, bits);
    return bits;
}

cnd_status plan_columns(int model, const cnd_graph_dev &G, const std::vector<ItemDesc> &items, ColPlan &plan) {
    int64_t trials = 0;
    for (const auto &it : items) trials += it.trials;
    if (trials == 0) return CND_OK;
    ColShape c;
    choose_shape(model, G, trials, c, plan.bits);
    const int64_t slots = (int64_t)G.num_sms * c.per_sm;
    plan.items.resize(sizeof(ColItem) * items.size());
    ColItem *h = reinterpret_cast<ColItem *>(plan.items.data());
    int64_t cols = 0;
    for (const auto &it : items) {
        *h++ = ColItem{it.out0, it.key, (int32_t)it.seed_begin, (int32_t)it.seed_end, (int32_t)it.trials, (int32_t)cols};
        cols += (it.trials + plan.bits - 1) / plan.bits;
    }
    if (cols > 0x7FFFFFFF - slots) {
        set_error("too many trials in one call");
        return CND_EINVAL;
    }
    plan.n_items = (int32_t)items.size();
    plan.cols = (int32_t)cols;
    plan.blocks = (int32_t)std::min<int64_t>(cols, slots);
    plan.threads = c.threads;
    plan.cap = c.cap;
    plan.dyn = c.dyn;
    plan.over = c.cap < G.n ? (size_t)plan.blocks * (size_t)G.n : 0;  // list entries beyond cap
    plan.scratch = 8 * plan.over;
    return CND_OK;
}

cnd_status run_columns(int model, const cnd_graph_dev &G, const ColPlan &plan, const void *items, void *scratch,
                       const int32_t *seeds_dev, int32_t *spread, int32_t *count, unsigned long long *checks,
                       unsigned long long *level_counts, CallFlags *flags, const cnd_sim_opts &o, cudaStream_t st) {
    if (plan.cols == 0) return CND_OK;
    const void *fn = model == 0 ? (const void *)k_columns<0> : (const void *)k_columns<1>;
    // the same value on every call: threads may launch with different sizes at the same time
    CND_CUDA_TRY(cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kMaxDynamic));
    ColParams p{};
    p.n = G.n;
    p.n_items = plan.n_items;
    p.bits = plan.bits;
    p.n_cols = plan.cols;
    p.row_ptr = G.row_ptr;
    p.edge = model == 0 ? G.ic_edge : G.lt_cnt_edge;
    p.items = static_cast<const ColItem *>(items);
    p.seeds = seeds_dev;
    p.cnt_off = G.lt_cnt_off;
    p.unit_w = G.lt_unit_w;
    p.first_trial = o.first_trial;
    p.spread = spread;
    p.count = count;
    p.checks = checks;
    p.level_counts = level_counts;
    p.lc_len = o.level_counts_len;
    p.max_levels = o.max_levels;
    p.timeout_ns = o.timeout_s > 0 ? (unsigned long long)std::max(1.0, std::min(o.timeout_s * 1e9, 1.8e19)) : 0ull;
    p.cap = plan.cap;
    p.over_bits = static_cast<uint32_t *>(scratch);
    p.over_node = reinterpret_cast<uint16_t *>(p.over_bits + plan.over);
    p.flags = flags;
    void *args[] = {&p};
    CND_CUDA_TRY(cudaLaunchKernel(fn, dim3((unsigned)plan.blocks), dim3((unsigned)plan.threads), args, plan.dyn, st));
    return CND_OK;
}

}  // namespace cnd

// A3: core numbers of G_S and its removal order (Definition 2.1; the Matula-Beck removal of
// Section 2, a frontier at a time).
//
// Peeling removes the vertices of least degree round after round: level k takes every
// vertex whose remaining degree is at most k, then those that drop to k, and so on. Its
// rounds are one chain (304 on the medium graph, over 72 levels), and a round is short: the
// chain took 1.05 ms there as a grid, a cluster and a one-block phase. Both halves of the
// answer are found here with short chains instead, by one cooperative kernel:
//
//  1. Core numbers, as the fixpoint of local h-indices (Lue, Zhou, Zhang, Stanley, "The
//     H-index of a network node and its relation to degree and coreness", Nature
//     Communications 7, 2016): from val = degree, every vertex takes the largest h such
//     that h neighbours have val >= h, until nothing changes; what remains is the core
//     number. cnt[v] counts the neighbours with val >= val[v]; a vertex that drops from a to
//     b takes one off the neighbours with b < val <= a, and a vertex whose cnt falls below
//     its val is worked off in the next round, so a round costs the vertices that change.
//     11 to 33 rounds on the recipes' graphs (18 at 70M edges, 33 at 6M of 2 per pair).
//  2. Removal rounds, all levels at once: within level k a vertex leaves when at most k
//     neighbours of its own or a higher level are left, and neither lower levels (all gone
//     by then) nor higher ones (all there) depend on the rounds of this one. cnt is that
//     count at the start. 8 to 24 rounds. The level's first round in the whole order is
//     the sum of the lower levels' rounds, so the order and the number of rounds are those
//     of the one chain.
//
// A hub of 35,000 neighbours on the medium graph ends at 71, and changes in most rounds: its
// row would be read again and again for the hundred neighbours that matter. When its value
// falls, a vertex of more than CORE_ROW8 neighbours keeps the ones whose value is at least
// a part (CORE_KEEP) of its new one. A shortened row holds every neighbour whose value is at
// least slo, the highest of the bounds it has been cut at (a later cut's may be lower, but
// what an earlier one dropped does not come back); values only fall, so the others cannot
// count while the vertex stays at or above slo. Below, the whole row is read again, and
// shortened anew.
//
// The last rounds of both halves hold a few vertices each: one block runs them alone, with
// block barriers, and one warp those of up to 32 vertices with short rows.
//
// Both halves together, against the phases of one chain: 0.56 against 1.26 ms on the medium
// graph (20M edges), 0.63 against 1.94 on the paper-scale one (beside nothing else), 1.18
// against 2.40 on 6M edges of 2 per pair.
//
// The two arrays of values (val, nv) keep a round's reads apart from its writes: a round
// computes nv from val (step A), then tells the neighbours (step B, which compares nv), with
// a grid barrier after each.
#include <algorithm>
#include <climits>
#include <cmath>
#include <cstdlib>
#include <cstring>

#include "core.cuh"
#include "internal.cuh"

#include <cooperative_groups.h>
namespace cg = cooperative_groups;

namespace folty {

enum {
    K_BAR = 0,
    K_GEN = 1,
    K_ROUND = 5,   // round handed back by a stretch of rounds on one block
    K_SHORT = 6,   // vertices of degree 1 .. CORE_ROW8,
    K_MID = 7,     // .. CORE_MID,
    K_BIG = 8,     // above
    K_FR = 9,      // 3 slots: frontier sizes of the first half, rows up to CORE_MID
    K_BFR = 12,    // 3 slots: above
    K_FR2 = 15,    // the same for the second half
    K_BFR2 = 18,
    K_BEAT = 21,   // rounds that one block has run alone
    K_SLOTS = 24
};

constexpr int CORE_THREADS = 1024;
constexpr int CORE_SMALL = 8;      // rows up to this length: one thread, all loads in flight;
constexpr int CORE_ROW8 = 64;      // up to this one: eight lanes, eight entries each;
constexpr int CORE_MID = 511;      // up to this one: a warp, sixteen entries a lane; longer ones: a block
constexpr int CORE_BLOCK = 8;      // entries a thread of a block holds; longer rows are read per step
constexpr int CORE_SOLO = 96;      // frontiers up to this size: one block, until they exceed twice that
// a shortened row keeps the neighbours of at least this part of the vertex's value: an eighth
// after the first round (values still fall by factors), a third later
constexpr int CORE_KEEP_FIRST = 8;
constexpr int CORE_KEEP = 3;
constexpr int CORE_INIT = 8;       // vertices per thread and step of the first pass
constexpr int CORE_BINS = 16384;   // histogram bins of a block
constexpr int CORE_STAGE = 4096;   // appends a block stages
constexpr int CORE_POWERS = 17;    // powers of two up to 2^16: no h-index of 2^31 static edges exceeds it

struct CoreArgs {
    const int32_t* rowptr;
    const int32_t* adj;
    const int32_t* src;  // row of every entry of adj
    int64_t entries;
    const int32_t* deg;
    int32_t n;
    int32_t hcap;  // no h-index exceeds it (h vertices of degree >= h need h^2 <= 2S)
    int32_t* val;  // the core numbers at the end
    int32_t* nv;
    int32_t* cnt;
    int32_t* rnd;  // removal round; the round within the level until the last pass
    int32_t* shrt;  // the vertices with a neighbour, by degree
    int32_t* mid;
    int32_t* big;
    int32_t* fr[2];
    int32_t* bfr[2];
    int32_t bcap;  // entries of big, bfr
    int32_t* srow;  // shortened rows, at the places of the whole ones in adj
    int32_t* slen;  // their lengths, -1: the whole row stands
    int32_t* slo;   // a shortened row holds every neighbour of at least this value
    int32_t* lev;  // [hcap + 2] rounds of each level (zeroed)
    int* ctl;      // zeroed
    long long timeout_ns;
};

__device__ __forceinline__ long long global_ns() {
    long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// Grid-wide barrier for a cooperative launch (all blocks co-resident). The wait is
// bounded: after timeout_ns without a round by the block that runs alone (a path of n vertices
// takes it n / 2 rounds) the block records an error and every block returns. Also the
// values of two control words after it, read together with the error word by one thread.
// Its fences order every plain access before it against every one after it (the first
// level caches hold nothing from before), so values that a pass only reads are read
// through those caches.
struct Sizes {
    bool ok;
    int a, b;
};
__device__ Sizes grid_barrier(int* ctl, long long timeout_ns, int wa = K_BAR, int wb = K_BAR) {
    __shared__ int s_v[3];
    __syncthreads();
    if (threadIdx.x == 0) {
        volatile int* vctl = ctl;
        const int gen = vctl[K_GEN];
        __threadfence();
        const int arrived = atomicAdd(&ctl[K_BAR], 1);
        if (arrived == (int)gridDim.x - 1) {
            vctl[K_BAR] = 0;
            __threadfence();
            vctl[K_GEN] = gen + 1;
        } else {
            long long t0 = 0;
            int beat = 0;
            for (int spin = 0; vctl[K_GEN] == gen; spin++) {
                if ((spin & 63) != 63) continue;
                if (vctl[CORE_ERR]) break;
                const long long t = global_ns();
                const int now = vctl[K_BEAT];
                if (t0 == 0 || now != beat) {
                    t0 = t;
                    beat = now;
                } else if (t - t0 > timeout_ns) {
                    atomicExch(&ctl[CORE_ERR], 1);
                    break;
                }
            }
        }
        __threadfence();
        const int e = vctl[CORE_ERR], x = vctl[wa], y = vctl[wb];
        s_v[0] = e;
        s_v[1] = x;
        s_v[2] = y;
    }
    __syncthreads();
    const Sizes r{s_v[0] == 0, s_v[1], s_v[2]};
    return r;
}

// The blocks that share a pass: all of the grid, or one.
struct Team {
    int blk, n;
};

// A row as it stands.
struct Row {
    const int32_t* p;
    int n;
    bool cut;
};

__device__ __forceinline__ Row whole_row(const CoreArgs& a, int32_t v) {
    const int32_t r0 = a.rowptr[v];
    return Row{a.adj + r0, a.rowptr[v + 1] - r0, false};
}

__device__ __forceinline__ Row row_at(const CoreArgs& a, int32_t v) {
    const int32_t r0 = a.rowptr[v], r1 = a.rowptr[v + 1], sl = __ldcg(&a.slen[v]);
    return sl >= 0 ? Row{a.srow + r0, sl, true} : Row{a.adj + r0, r1 - r0, false};
}

__device__ __forceinline__ Row shfl_row(const Row& r, int src) {
    return Row{(const int32_t*)__shfl_sync(0xffffffffu, (unsigned long long)r.p, src), __shfl_sync(0xffffffffu, r.n, src),
               __shfl_sync(0xffffffffu, (int)r.cut, src) != 0};
}

// Where a pass appends: buffer and counter slot, of the first half or the second.
struct Next {
    int buf, slot, half;
};

// Appends v for the threads that call it together (one addition for all of them). A list
// holds each vertex at most once, so it never exceeds cap; an append beyond it would be
// dropped and recorded.
__device__ __forceinline__ void append(int32_t v, int32_t* list, int* counter, int32_t cap, int* ctl) {
    cg::coalesced_group g = cg::coalesced_threads();
    int base = 0;
    if (g.thread_rank() == 0) base = atomicAdd(counter, (int)g.size());
    const int at = g.shfl(base, 0) + (int)g.thread_rank();
    if (at < cap) list[at] = v;
    else atomicExch(&ctl[CORE_ERR], 2);
}

// A pass stages its appends per block (the appends of a first round, 43,000 to 120,000 of
// them on the recipes' graphs, took a nanosecond each on the list's counter); flush_next
// moves them to the list, before the pass's barrier, by every thread of the block.
struct Stage {
    int n;
    int32_t v[CORE_STAGE];
};
__device__ __forceinline__ Stage& stage() {
    extern __shared__ int core_smem[];
    return *reinterpret_cast<Stage*>(core_smem + CORE_BINS);
}

__device__ __forceinline__ void append_next(const CoreArgs& a, int32_t v, Next nx) {
    const int32_t sl = __ldcg(&a.slen[v]);
    if ((sl >= 0 ? sl : a.deg[v]) > CORE_MID) {
        append(v, a.bfr[nx.buf], &a.ctl[(nx.half ? K_BFR2 : K_BFR) + nx.slot], a.bcap, a.ctl);
        return;
    }
    const int at = atomicAdd(&stage().n, 1);
    if (at < CORE_STAGE) stage().v[at] = v;
    else append(v, a.fr[nx.buf], &a.ctl[(nx.half ? K_FR2 : K_FR) + nx.slot], a.n, a.ctl);
}

__device__ __forceinline__ void flush_next(const CoreArgs& a, Next nx) {
    __shared__ int s_at;
    Stage& st = stage();
    __syncthreads();
    const int n = min(st.n, CORE_STAGE);
    if (n == 0) return;
    if (threadIdx.x == 0) s_at = atomicAdd(&a.ctl[(nx.half ? K_FR2 : K_FR) + nx.slot], n);
    __syncthreads();
    for (int i = threadIdx.x; i < n; i += CORE_THREADS) {
        if (s_at + i < a.n) a.fr[nx.buf][s_at + i] = st.v[i];
        else atomicExch(&a.ctl[CORE_ERR], 2);
    }
    __syncthreads();
    if (threadIdx.x == 0) st.n = 0;
    __syncthreads();
}

// Entries each warp takes together: 32 for long lists, fewer when that leaves warps idle.
__device__ __forceinline__ int warp_share(Team t, int count) {
    const int warps = t.n * (CORE_THREADS / 32);
    return min(32, max(1, (count + warps - 1) / warps));
}

// The lane of the (lane / 8)-th set bit of m, -1 when m has fewer; the four lowest set bits
// leave m.
__device__ __forceinline__ int octet_source(unsigned& m) {
    const int g = (threadIdx.x & 31) >> 3;
    int src = -1;
#pragma unroll
    for (int i = 0; i < 4; i++) {
        if (m && i == g) src = __ffs((int)m) - 1;
        m &= m - 1;
    }
    return src;
}

// ------------------------------------------------------------------ step A: h-indices

// The largest h <= top such that h entries of a row have val >= h, and that number of
// entries (0 and any when not even one has, as a shortened row may). One thread, rows of up
// to 8 entries x (-1: none): 8 counters of 8 bits in a word.
__device__ __forceinline__ void thread_row(int32_t (&x)[CORE_SMALL], const int32_t* row, int d) {
#pragma unroll
    for (int i = 0; i < CORE_SMALL; i++) x[i] = i < d ? row[i] : -1;
}
__device__ __forceinline__ int thread_h(const CoreArgs& a, const int32_t (&x)[CORE_SMALL], int top, int& cnt) {
    uint64_t bins = 0;  // byte h - 1: entries of value h (or more, for h = top)
#pragma unroll
    for (int i = 0; i < CORE_SMALL; i++)
        if (x[i] >= 0) bins += 1ull << (8 * (min(a.val[x[i]], top) - 1));
    int c = 0;
    for (int h = top; h >= 1; h--) {
        c += (int)((bins >> (8 * (h - 1))) & 255);
        if (c >= h) {
            cnt = c;
            return h;
        }
    }
    cnt = c;
    return 0;
}

// A search for h: probes from the top at growing distances (most recomputed values fall by
// little), then bisection.
struct Search {
    int lo = 0, hi, step = 1, cnt;  // lo: the highest value known to hold, cnt its entries; hi: the lowest known not to
    __device__ Search(int top, int n) : hi(top + 1), cnt(n) {}
    __device__ bool done() const { return hi - lo <= 1; }
    __device__ int probe() const { return lo == 0 ? max(hi - step, 1) : (lo + hi) >> 1; }
    __device__ void answer(int m, int c) {
        step *= 2;
        if (c >= m) {
            lo = m;
            cnt = c;
        } else {
            hi = m;
        }
    }
};

// By G lanes (8 or 32), R entries each; all groups of the warp together (an idle one: n = 0,
// top = 0).
template <int G, int R>
__device__ __forceinline__ int group_h(const CoreArgs& a, const int32_t* row, int n, int top, int& cnt) {
    const int li = threadIdx.x & (G - 1);
    int32_t x[R];
#pragma unroll
    for (int u = 0; u < R; u++) x[u] = li + G * u < n ? row[li + G * u] : -1;
#pragma unroll
    for (int u = 0; u < R; u++) x[u] = x[u] >= 0 ? a.val[x[u]] : 0;
    Search s(top, n);
    while (__any_sync(0xffffffffu, !s.done())) {
        const int m = s.probe();
        int c = 0;
#pragma unroll
        for (int u = 0; u < R; u++) c += x[u] >= m;
        if (G == 32) c = __reduce_add_sync(0xffffffffu, c);
        else
#pragma unroll
            for (int o = G / 2; o > 0; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
        if (!s.done()) s.answer(m, c);
    }
    cnt = s.cnt;
    return s.lo;
}

// Sum over the block; buf[2][32] alternates with parity, so that one barrier per call is
// enough.
__device__ __forceinline__ int block_sum(int v, int (*buf)[32], int parity) {
    v = __reduce_add_sync(0xffffffffu, v);
    if ((threadIdx.x & 31) == 0) buf[parity][threadIdx.x >> 5] = v;
    __syncthreads();
    return __reduce_add_sync(0xffffffffu, buf[parity][threadIdx.x & 31]);
}

// By a block, rows of up to CORE_BLOCK entries a thread.
__device__ int block_h(const CoreArgs& a, const int32_t* row, int n, int top, int& cnt) {
    __shared__ int buf[2][32];
    int32_t x[CORE_BLOCK];
#pragma unroll
    for (int u = 0; u < CORE_BLOCK; u++) x[u] = (int)threadIdx.x + CORE_THREADS * u < n ? row[threadIdx.x + CORE_THREADS * u] : -1;
#pragma unroll
    for (int u = 0; u < CORE_BLOCK; u++) x[u] = x[u] >= 0 ? a.val[x[u]] : 0;
    __syncthreads();  // the last call's sums have been read
    Search s(top, n);
    for (int parity = 0; !s.done(); parity ^= 1) {
        const int m = s.probe();
        int c = 0;
#pragma unroll
        for (int u = 0; u < CORE_BLOCK; u++) c += x[u] >= m;
        s.answer(m, block_sum(c, buf, parity));
    }
    cnt = s.cnt;
    return s.lo;
}

// By a block, rows of any length (whole ones, the hubs' first round): first the entries of
// at least every power of two, which gives the answer within a factor of two and keeps the
// many small values of a hub's row (one contended bin) out of the histogram; then a
// histogram of the values in [lo, hi], more than one value to a bin when they are more than
// the bins, and again within the bin that holds the answer.
__device__ int long_h(const CoreArgs& a, const int32_t* row, int d, int top, int* bins, int& cnt) {
    __shared__ int s_pow[32], s_bin, s_above;
    const int lane = threadIdx.x & 31;
    __syncthreads();  // the last call's shared values have been read
    if (threadIdx.x < 32) s_pow[threadIdx.x] = 0;
    __syncthreads();
    {
        int c[CORE_POWERS];
#pragma unroll
        for (int i = 0; i < CORE_POWERS; i++) c[i] = 0;
        for (int i0 = threadIdx.x; i0 < d; i0 += 4 * CORE_THREADS) {
            int32_t x[4];
#pragma unroll
            for (int u = 0; u < 4; u++) x[u] = i0 + CORE_THREADS * u < d ? row[i0 + CORE_THREADS * u] : -1;
#pragma unroll
            for (int u = 0; u < 4; u++) x[u] = x[u] >= 0 ? min(a.val[x[u]], top) : 0;
#pragma unroll
            for (int u = 0; u < 4; u++) {
#pragma unroll
                for (int i = 0; i < CORE_POWERS; i++) c[i] += x[u] >= (1 << i);
            }
        }
#pragma unroll
        for (int i = 0; i < CORE_POWERS; i++) {
            const int n = __reduce_add_sync(0xffffffffu, c[i]);
            if (lane == i && n) atomicAdd(&s_pow[i], n);
        }
    }
    __syncthreads();
    int p = 0;
    while (p + 1 < CORE_POWERS && s_pow[p + 1] >= (1 << (p + 1))) p++;
    int lo = 1 << p, hi = top, above = 0;  // above: entries of value > hi
    if (p + 1 < CORE_POWERS && (1 << (p + 1)) <= top) {
        hi = (1 << (p + 1)) - 1;
        above = s_pow[p + 1];
    }
    while (true) {
        const int width = (hi - lo + CORE_BINS) / CORE_BINS;  // ceil((hi - lo + 1) / CORE_BINS)
        const int nb = (hi - lo) / width + 1;
        __syncthreads();
        for (int i = threadIdx.x; i < nb; i += CORE_THREADS) bins[i] = 0;
        __syncthreads();
        for (int i0 = threadIdx.x; i0 < d; i0 += 4 * CORE_THREADS) {
            int32_t x[4];
#pragma unroll
            for (int u = 0; u < 4; u++) x[u] = i0 + CORE_THREADS * u < d ? row[i0 + CORE_THREADS * u] : -1;
#pragma unroll
            for (int u = 0; u < 4; u++) x[u] = x[u] >= 0 ? min(a.val[x[u]], top) : -1;
#pragma unroll
            for (int u = 0; u < 4; u++)
                if (x[u] >= lo && x[u] <= hi) atomicAdd(&bins[(x[u] - lo) / width], 1);
        }
        __syncthreads();
        // the highest bin whose lowest value is reached by enough entries
        if (threadIdx.x < 32) {
            int up = above, bin = 0, up_bin = above;
            for (int b0 = nb - 1; b0 >= 0; b0 -= 32) {
                const int b = b0 - lane;
                int inc = b >= 0 ? bins[b] : 0;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const int y = __shfl_up_sync(0xffffffffu, inc, o);
                    if (lane >= o) inc += y;
                }
                const unsigned ok = __ballot_sync(0xffffffffu, b >= 0 && up + inc >= lo + b * width);
                if (ok) {
                    const int l = __ffs((int)ok) - 1;
                    bin = b0 - l;
                    up_bin = up + __shfl_sync(0xffffffffu, inc, l);
                    break;
                }
                up += __shfl_sync(0xffffffffu, inc, 31);
                up_bin = up;
            }
            if (lane == 0) {
                s_bin = bin;
                s_above = up_bin;
            }
        }
        __syncthreads();
        const int b = s_bin;
        if (width == 1) {
            cnt = s_above;
            return lo + b;
        }
        above = s_above - bins[b];
        hi = min(hi, lo + b * width + width - 1);
        lo = lo + b * width;
    }
}

// Step A over a list of vertices (rows of more than CORE_MID entries skipped). A shortened
// row answers for values from its bound (slo) on. Below, the whole row stands again: read
// at once when a warp holds it, else by a block in the next round (nx; the vertex keeps its
// value until then).
__device__ void h_pass(const CoreArgs& a, Team t, const int32_t* list, int count, Next nx) {
    const int lane = threadIdx.x & 31;
    const int share = warp_share(t, count);
    const int64_t gw = (int64_t)t.blk * (CORE_THREADS / 32) + (threadIdx.x >> 5);
    const int64_t step = (int64_t)t.n * (CORE_THREADS / 32) * share;
    for (int64_t i0 = gw * share; i0 < count; i0 += step) {
        const bool on = lane < share && i0 + lane < count;
        const int32_t v = on ? __ldcg(&list[i0 + lane]) : 0;
        const Row row = on ? row_at(a, v) : Row{nullptr, 0, false};
        const int top = on ? min(min(__ldcg(&a.val[v]), row.cut ? a.deg[v] : row.n), a.hcap) : 0;
        if (on && !row.cut && row.n <= CORE_SMALL) {
            int32_t x[CORE_SMALL];
            thread_row(x, row.p, row.n);
            int c;
            a.nv[v] = thread_h(a, x, top, c);
            a.cnt[v] = c;
        }
        unsigned eight = __ballot_sync(0xffffffffu, on && !row.cut && row.n > CORE_SMALL && row.n <= CORE_ROW8);
        while (eight) {
            const int src = octet_source(eight);
            const Row r = shfl_row(row, max(src, 0));
            const int32_t u = __shfl_sync(0xffffffffu, v, max(src, 0));
            const int tu = __shfl_sync(0xffffffffu, top, max(src, 0));
            int c;
            const int h = group_h<8, CORE_ROW8 / 8>(a, r.p, src >= 0 ? r.n : 0, src >= 0 ? tu : 0, c);
            if (src >= 0 && (lane & 7) == 0) {
                a.nv[u] = h;
                a.cnt[u] = c;
            }
        }
        unsigned mid = __ballot_sync(0xffffffffu, on && (row.cut || row.n > CORE_ROW8) && row.n <= CORE_MID);
        while (mid) {
            const int l = __ffs((int)mid) - 1;
            mid &= mid - 1;
            const Row r = shfl_row(row, l);
            const int32_t u = __shfl_sync(0xffffffffu, v, l);
            const int tu = __shfl_sync(0xffffffffu, top, l);
            int c;
            int h = group_h<32, (CORE_MID + 32) / 32>(a, r.p, r.n, min(tu, r.n), c);
            bool later = false;
            if (r.cut && h < __ldcg(&a.slo[u])) {
                const Row w = whole_row(a, u);
                if (lane == 0) a.slen[u] = -1;
                later = w.n > CORE_MID;
                if (!later) h = group_h<32, (CORE_MID + 32) / 32>(a, w.p, w.n, tu, c);
            }
            if (lane == 0) {
                if (later) {
                    append(u, a.bfr[nx.buf], &a.ctl[K_BFR + nx.slot], a.bcap, a.ctl);
                } else {
                    a.nv[u] = h;
                    a.cnt[u] = c;
                }
            }
        }
    }
}

__device__ void h_pass_big(const CoreArgs& a, Team t, const int32_t* list, int count, int* bins) {
    for (int i = t.blk; i < count; i += t.n) {
        const int32_t v = __ldcg(&list[i]);
        Row r = row_at(a, v);
        const int top = min(min(__ldcg(&a.val[v]), a.deg[v]), a.hcap);
        int c = 0, h = 0;
        for (bool again = true; again;) {
            const int tr = min(top, r.n);
            h = r.n <= CORE_BLOCK * CORE_THREADS ? block_h(a, r.p, r.n, tr, c) : long_h(a, r.p, r.n, tr, bins, c);
            again = r.cut && h < __ldcg(&a.slo[v]);
            if (again) {
                r = whole_row(a, v);
                if (threadIdx.x == 0) a.slen[v] = -1;
            }
        }
        if (threadIdx.x == 0) {
            a.nv[v] = h;
            a.cnt[v] = c;
        }
    }
}

// ------------------------------------------------------------------ rows of a list

// Level k has had n rounds (n only grows; a plain load first, as most vertices of a round
// find it noted: a store each took 300 us for the 400,000 vertices of level 1).
__device__ __forceinline__ void note_round(const CoreArgs& a, int k, int n) {
    if (*(const volatile int32_t*)&a.lev[k] < n) a.lev[k] = n;
}

// What a row's owner tells the neighbour x of value c. DROP (step B; c from nv): the owner's
// value fell from `from` to `to`; a neighbour with to < c <= from loses one, and is worked
// off next when it is the first below its value. REMOVE (c from val): the owner left level
// `from`; a neighbour of the level loses one, and leaves in round `to` when it is the first
// at the level.
// told returns whether x is worked off next.
template <bool REMOVE>
__device__ __forceinline__ bool told(const CoreArgs& a, int32_t x, int c, int from, int to) {
    if (REMOVE) {
        if (c != from) return false;
        if (atomicSub(&a.cnt[x], 1) != from + 1) return false;
        a.rnd[x] = to;
        note_round(a, from, to + 1);
        return true;
    }
    return c > to && c <= from && atomicSub(&a.cnt[x], 1) == c;
}
template <bool REMOVE>
__device__ __forceinline__ void tell(const CoreArgs& a, int32_t x, int c, int from, int to, Next nx) {
    if (told<REMOVE>(a, x, c, from, to)) append_next(a, x, nx);
}

template <bool REMOVE>
__device__ __forceinline__ int told_value(const CoreArgs& a, int32_t x) {
    return REMOVE ? a.val[x] : a.nv[x];
}

// The first rounds of both halves concern nearly every vertex: one thread per adjacency
// entry (its row's vertex tells the entry), which is even whatever the rows' lengths. Of a
// removal, the vertices of round 0 tell.
template <bool REMOVE>
__device__ void tell_entries(const CoreArgs& a, Next nx) {
    constexpr int E = 4;
    const int64_t stride = (int64_t)gridDim.x * CORE_THREADS;
    for (int64_t j0 = blockIdx.x * (int64_t)CORE_THREADS + threadIdx.x; j0 < a.entries; j0 += E * stride) {
        int32_t v[E], x[E], c[E], from[E], to[E];
#pragma unroll
        for (int e = 0; e < E; e++) {
            const int64_t j = j0 + e * stride;
            x[e] = j < a.entries ? a.adj[j] : -1;
            v[e] = j < a.entries ? a.src[j] : 0;
        }
#pragma unroll
        for (int e = 0; e < E; e++) {
            c[e] = x[e] >= 0 ? told_value<REMOVE>(a, x[e]) : 0;
            from[e] = x[e] >= 0 ? a.val[v[e]] : 0;
            to[e] = x[e] < 0 ? 0 : REMOVE ? __ldcg(&a.rnd[v[e]]) : a.nv[v[e]];
        }
#pragma unroll
        for (int e = 0; e < E; e++) {
            if (x[e] < 0 || (REMOVE ? to[e] != 0 : to[e] >= from[e])) continue;
            tell<REMOVE>(a, x[e], c[e], from[e], REMOVE ? 1 : to[e], nx);
        }
    }
}

// Shortens the row of v (value `to`) by a warp; the row is whole.
__device__ __forceinline__ void shorten_row(const CoreArgs& a, int32_t v, const Row& r, int to, int keep_part) {
    const int lane = threadIdx.x & 31;
    int32_t* keep = a.srow + (r.p - a.adj);
    int kept = 0;
    for (int j0 = lane; j0 - lane < r.n; j0 += 128) {
        int32_t x[4], c[4];
#pragma unroll
        for (int u = 0; u < 4; u++) x[u] = j0 + 32 * u < r.n ? r.p[j0 + 32 * u] : -1;
#pragma unroll
        for (int u = 0; u < 4; u++) c[u] = x[u] >= 0 ? a.nv[x[u]] : 0;
#pragma unroll
        for (int u = 0; u < 4; u++) {
            const bool k = x[u] >= 0 && keep_part * c[u] >= to;
            const unsigned ks = __ballot_sync(0xffffffffu, k);
            if (k) keep[kept + __popc(ks & ((1u << lane) - 1u))] = x[u];
            kept += __popc(ks);
        }
    }
    if (lane == 0) {
        a.slo[v] = (to + keep_part - 1) / keep_part;
        a.slen[v] = kept;
    }
}

// The rows of a list (of more than CORE_MID entries skipped) by a lane, eight lanes or the
// warp. A step B tells only for values that fell, and then shortens whole rows of more than
// CORE_ROW8 entries.
template <bool REMOVE>
__device__ void tell_pass(const CoreArgs& a, Team t, const int32_t* list, int count, int round, Next nx) {
    const int lane = threadIdx.x & 31;
    const int share = warp_share(t, count);
    const int64_t gw = (int64_t)t.blk * (CORE_THREADS / 32) + (threadIdx.x >> 5);
    const int64_t step = (int64_t)t.n * (CORE_THREADS / 32) * share;
    for (int64_t i0 = gw * share; i0 < count; i0 += step) {
        const bool on = lane < share && i0 + lane < count;
        const int32_t v = on ? __ldcg(&list[i0 + lane]) : 0;
        const Row row = on ? row_at(a, v) : Row{nullptr, 0, false};
        const int from = on ? __ldcg(&a.val[v]) : 0;
        const int to = REMOVE ? round : (on ? __ldcg(&a.nv[v]) : 0);
        const bool act = on && row.n <= CORE_MID && (REMOVE || to < from);
        if (act && row.n <= CORE_SMALL) {
            int32_t x[CORE_SMALL], c[CORE_SMALL];
            thread_row(x, row.p, row.n);
#pragma unroll
            for (int i = 0; i < CORE_SMALL; i++) c[i] = x[i] >= 0 ? told_value<REMOVE>(a, x[i]) : 0;
#pragma unroll
            for (int i = 0; i < CORE_SMALL; i++)
                if (x[i] >= 0) tell<REMOVE>(a, x[i], c[i], from, to, nx);
        }
        unsigned eight = __ballot_sync(0xffffffffu, act && row.n > CORE_SMALL && row.n <= CORE_ROW8);
        while (eight) {
            const int src = octet_source(eight);
            const Row r = shfl_row(row, max(src, 0));
            const int f = __shfl_sync(0xffffffffu, from, max(src, 0)), to_r = __shfl_sync(0xffffffffu, to, max(src, 0));
            int32_t x[CORE_ROW8 / 8], c[CORE_ROW8 / 8];
#pragma unroll
            for (int u = 0; u < CORE_ROW8 / 8; u++) x[u] = src >= 0 && (lane & 7) + 8 * u < r.n ? r.p[(lane & 7) + 8 * u] : -1;
#pragma unroll
            for (int u = 0; u < CORE_ROW8 / 8; u++) c[u] = x[u] >= 0 ? told_value<REMOVE>(a, x[u]) : 0;
#pragma unroll
            for (int u = 0; u < CORE_ROW8 / 8; u++)
                if (x[u] >= 0) tell<REMOVE>(a, x[u], c[u], f, to_r, nx);
            __syncwarp();
        }
        unsigned mid = __ballot_sync(0xffffffffu, act && row.n > CORE_ROW8);
        while (mid) {
            const int l = __ffs((int)mid) - 1;
            mid &= mid - 1;
            const Row r = shfl_row(row, l);
            const int f = __shfl_sync(0xffffffffu, from, l), to_r = __shfl_sync(0xffffffffu, to, l);
            const int32_t u_v = __shfl_sync(0xffffffffu, v, l);
            for (int j0 = lane; j0 - lane < r.n; j0 += 128) {
                int32_t x[4], c[4];
#pragma unroll
                for (int u = 0; u < 4; u++) x[u] = j0 + 32 * u < r.n ? r.p[j0 + 32 * u] : -1;
#pragma unroll
                for (int u = 0; u < 4; u++) c[u] = x[u] >= 0 ? told_value<REMOVE>(a, x[u]) : 0;
#pragma unroll
                for (int u = 0; u < 4; u++)
                    if (x[u] >= 0) tell<REMOVE>(a, x[u], c[u], f, to_r, nx);
                __syncwarp();
            }
            if (!REMOVE && !r.cut) shorten_row(a, u_v, r, to_r, CORE_KEEP);
        }
        // only this vertex's warp reads its val during a step B
        __syncwarp();
        if (!REMOVE && act) a.val[v] = to;
    }
}

// By blocks: rows of any length. A step B also shortens the row, or shortens it further:
// each stretch of a row is read by all before any entry kept of it is written, and nothing
// is written past what has been read. TELL false: only shortens (the entries are told by
// tell_entries).
template <bool REMOVE, bool TELL>
__device__ void tell_pass_big(const CoreArgs& a, Team t, const int32_t* list, int count, int round, Next nx) {
    __shared__ int s_kept;
    constexpr int keep_part = TELL ? CORE_KEEP : CORE_KEEP_FIRST;
    const int lane = threadIdx.x & 31;
    for (int i = t.blk; i < count; i += t.n) {
        const int32_t v = __ldcg(&list[i]);
        const Row r = row_at(a, v);
        const int from = a.val[v], to = REMOVE ? round : a.nv[v];
        if (threadIdx.x == 0) s_kept = 0;
        __syncthreads();  // every thread has read the vertex's values
        if (TELL && !REMOVE && to >= from) continue;
        int32_t* keep = a.srow + a.rowptr[v];
        for (int j0 = threadIdx.x; j0 - (int)threadIdx.x < r.n; j0 += 4 * CORE_THREADS) {
            int32_t x[4], c[4];
#pragma unroll
            for (int u = 0; u < 4; u++) x[u] = j0 + CORE_THREADS * u < r.n ? __ldcg(&r.p[j0 + CORE_THREADS * u]) : -1;
#pragma unroll
            for (int u = 0; u < 4; u++) c[u] = x[u] >= 0 ? told_value<REMOVE>(a, x[u]) : 0;
            if (TELL) {
#pragma unroll
                for (int u = 0; u < 4; u++)
                    if (x[u] >= 0) tell<REMOVE>(a, x[u], c[u], from, to, nx);
            }
            if (!REMOVE) {
                __syncthreads();
#pragma unroll
                for (int u = 0; u < 4; u++) {
                    const bool k = x[u] >= 0 && keep_part * c[u] >= to;
                    const unsigned ks = __ballot_sync(0xffffffffu, k);
                    int base = 0;
                    if (lane == 0 && ks) base = atomicAdd(&s_kept, __popc(ks));
                    base = __shfl_sync(0xffffffffu, base, 0);
                    if (k) keep[base + __popc(ks & ((1u << lane) - 1u))] = x[u];
                }
            }
        }
        __syncthreads();
        if (!REMOVE && threadIdx.x == 0) {
            a.val[v] = to;
            a.slo[v] = max(r.cut ? __ldcg(&a.slo[v]) : 0, (to + keep_part - 1) / keep_part);
            a.slen[v] = s_kept;
        }
        __syncthreads();  // s_kept is read before the next vertex clears it
    }
}

// After the entries of the first round are told: the new values, and the rows of more than
// CORE_ROW8 entries shortened.
__device__ void settle_first(const CoreArgs& a, Team t, int nshort, int nmid, int nbig) {
    tell_pass_big<false, false>(a, t, a.big, nbig, 0, Next{0, 0, 0});
    const int64_t gw = (int64_t)t.blk * (CORE_THREADS / 32) + (threadIdx.x >> 5);
    for (int64_t i = gw; i < nmid; i += (int64_t)t.n * (CORE_THREADS / 32)) {
        const int32_t v = a.mid[i];
        const int to = a.nv[v];
        shorten_row(a, v, whole_row(a, v), to, CORE_KEEP_FIRST);
        if ((threadIdx.x & 31) == 0) a.val[v] = to;
    }
    for (int64_t i = t.blk * (int64_t)CORE_THREADS + threadIdx.x; i < nshort; i += (int64_t)t.n * CORE_THREADS) {
        const int32_t v = a.shrt[i];
        a.val[v] = a.nv[v];
    }
}

// One round of the first half, as it stands in the lists: step A, a barrier of the team,
// step B into buffer and slot of round r.
template <typename Barrier>
__device__ __forceinline__ Sizes value_round(const CoreArgs& a, Team t, int count, int bcount, int r, int* smem,
                                             Barrier&& barrier) {
    const int32_t* list = a.fr[(r - 1) & 1];
    const int32_t* blist = a.bfr[(r - 1) & 1];
    const Next nx{r & 1, r % 3, 0};
    h_pass_big(a, t, blist, bcount, smem);
    h_pass(a, t, list, count, nx);
    // round r appends to slot r % 3; the slot of the round after is cleared here, two
    // barriers after its last reader and one before its first writer
    if (t.blk == 0 && threadIdx.x == 0) {
        ((volatile int*)a.ctl)[K_FR + (r + 1) % 3] = 0;
        ((volatile int*)a.ctl)[K_BFR + (r + 1) % 3] = 0;
    }
    const Sizes half = barrier(K_BAR, K_BAR);
    if (!half.ok) return half;
    tell_pass_big<false, true>(a, t, blist, bcount, 0, nx);
    tell_pass<false>(a, t, list, count, 0, nx);
    flush_next(a, nx);
    return barrier(K_FR + r % 3, K_BFR + r % 3);
}

// One round of the second half: the vertices of round r >= 1 tell their levels.
template <typename Barrier>
__device__ __forceinline__ Sizes removal_round(const CoreArgs& a, Team t, int count, int bcount, int r, Barrier&& barrier) {
    if (t.blk == 0 && threadIdx.x == 0) {  // the slot of round r + 2, last read in round r - 1
        ((volatile int*)a.ctl)[K_FR2 + (r + 2) % 3] = 0;
        ((volatile int*)a.ctl)[K_BFR2 + (r + 2) % 3] = 0;
    }
    const Next nx{(r + 1) & 1, (r + 1) % 3, 1};
    tell_pass_big<true, true>(a, t, a.bfr[r & 1], bcount, r + 1, nx);
    tell_pass<true>(a, t, a.fr[r & 1], count, r + 1, nx);
    flush_next(a, nx);
    return barrier(K_FR2 + (r + 1) % 3, K_BFR2 + (r + 1) % 3);
}

// ------------------------------------------------------------------ rounds of a few vertices

// Rounds of 1 to 32 vertices whose rows are whole and no longer than CORE_SMALL, from round r
// on, by one warp with a vertex a lane and the lists in shared memory; returns the first round
// it has not run, with that round's lists and control words as the rounds of a block leave
// them. Both steps of a round share the row, and there is no barrier: bound by the chain of five
// dependent accesses to L2. A path of 20,000 vertices (10,000 rounds in either half) takes 42
// ms, between block barriers 73. Tried at once, not after CORE_LONG rounds, it cost the small
// graphs, whose rows are longer, 1 to 3% of their preprocessing.
constexpr int CORE_FEW = 32;
constexpr int CORE_LONG = 16;  // rounds of a block alone before one warp tries
static_assert(2 * CORE_FEW * CORE_SMALL <= CORE_STAGE, "both lists lie in the stage");

template <bool REMOVE>
__device__ __noinline__ int few_rounds(const CoreArgs& a, int count, int r) {
    constexpr unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const unsigned below = (1u << lane) - 1u;
    volatile int* vctl = a.ctl;
    int32_t* cur = stage().v;
    int32_t* next = cur + CORE_FEW * CORE_SMALL;
    // round r works off the lists of this parity, counted in this slot
    auto at = [](int round) { return REMOVE ? round : round - 1; };
    int beat = vctl[K_BEAT];
    if (lane < count) cur[lane] = __ldcg(&a.fr[at(r) & 1][lane]);
    __syncwarp();
    while (count > 0 && count <= CORE_FEW) {
        const bool on = lane < count;
        const int32_t v = on ? cur[lane] : 0;
        const Row row = on ? row_at(a, v) : Row{nullptr, 0, false};
        if (__any_sync(FULL, row.cut || row.n > CORE_SMALL)) break;
        const int from = on ? __ldcg(&a.val[v]) : 0;
        int32_t x[CORE_SMALL];
        thread_row(x, row.p, row.n);
        int to = r + 1;
        if (!REMOVE) {
            int c = 0;
            to = on ? thread_h(a, x, min(min(from, row.n), a.hcap), c) : 0;
            if (on) {
                a.nv[v] = to;
                a.cnt[v] = c;
            }
            __syncwarp();
        }
        const bool act = on && (REMOVE || to < from);
        int32_t c[CORE_SMALL];
#pragma unroll
        for (int i = 0; i < CORE_SMALL; i++) c[i] = act && x[i] >= 0 ? told_value<REMOVE>(a, x[i]) : 0;
        unsigned joins = 0;
#pragma unroll
        for (int i = 0; i < CORE_SMALL; i++)
            if (act && x[i] >= 0 && told<REMOVE>(a, x[i], c[i], from, to)) joins |= 1u << i;
        count = 0;
#pragma unroll
        for (int i = 0; i < CORE_SMALL; i++) {
            const bool j = (joins >> i) & 1u;
            const unsigned m = __ballot_sync(FULL, j);
            if (j) next[count + __popc(m & below)] = x[i];
            count += __popc(m);
        }
        if (!REMOVE && act) a.val[v] = to;  // read by no lane since the last __syncwarp
        if (lane == 0) vctl[K_BEAT] = ++beat;
        r++;
        int32_t* t = cur;
        cur = next;
        next = t;
        __syncwarp();
    }
    const int slot = at(r) % 3, fr = REMOVE ? K_FR2 : K_FR, bfr = REMOVE ? K_BFR2 : K_BFR;
    if (lane == 0) {
        vctl[fr + slot] = vctl[bfr + slot] = 0;
        vctl[fr + (at(r) + 1) % 3] = vctl[bfr + (at(r) + 1) % 3] = 0;
    }
    __syncwarp();
    for (int i = lane; i < count; i += 32) {
        const int32_t v = cur[i], sl = __ldcg(&a.slen[v]);
        if ((sl >= 0 ? sl : a.deg[v]) > CORE_MID) append(v, a.bfr[at(r) & 1], &a.ctl[bfr + slot], a.bcap, a.ctl);
        else append(v, a.fr[at(r) & 1], &a.ctl[fr + slot], a.n, a.ctl);
    }
    return r;
}

// The rounds of one block alone, from round r with z.a vertices on: while they are few.
template <bool REMOVE, typename Round, typename Barrier>
__device__ __forceinline__ void solo_rounds(const CoreArgs& a, Sizes z, int r, Round&& round, Barrier&& barrier) {
    __shared__ int s_r;
    volatile int* vctl = a.ctl;
    int again = r + CORE_LONG;  // most stretches end before; and after rows too long for one warp
    while (z.ok && z.a > 0 && z.a <= 2 * CORE_SOLO && z.b == 0) {
        if (z.a <= CORE_FEW && r >= again) {
            if (threadIdx.x < 32) {
                const int done = few_rounds<REMOVE>(a, z.a, r);
                if (threadIdx.x == 0) s_r = done;
            }
            __syncthreads();
            again = s_r == r ? r + CORE_LONG : s_r;
            r = s_r;
            const int slot = (REMOVE ? r : r - 1) % 3;
            z = barrier((REMOVE ? K_FR2 : K_FR) + slot, (REMOVE ? K_BFR2 : K_BFR) + slot);
            continue;
        }
        z = round(z.a, r);
        r++;
        if (threadIdx.x == 0) vctl[K_BEAT] = vctl[K_BEAT] + 1;
    }
    if (threadIdx.x == 0) vctl[K_ROUND] = r;
}

// ------------------------------------------------------------------ the kernel

__global__ void __launch_bounds__(CORE_THREADS, 1) k_core(const CoreArgs a) {
    extern __shared__ int core_smem[];
    __shared__ int wsum[2][32], s_base[2];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int* ctl = a.ctl;
    volatile int* vctl = ctl;
    const Team all{(int)blockIdx.x, (int)gridDim.x}, solo{0, 1};
    auto grid_wait = [&](int wa, int wb) { return grid_barrier(ctl, a.timeout_ns, wa, wb); };
    auto wait = [&] { return grid_barrier(ctl, a.timeout_ns).ok; };
    auto block_wait = [&](int wa, int wb) {
        __syncthreads();
        return Sizes{vctl[CORE_ERR] == 0, vctl[wa], vctl[wb]};
    };

    // the vertices with a neighbour, by degree, and their degrees as first values
    if (threadIdx.x == 0) stage().n = 0;
    bool isolated = false;
    for (int64_t b0 = (int64_t)blockIdx.x * (CORE_THREADS * CORE_INIT); b0 < a.n;
         b0 += (int64_t)gridDim.x * (CORE_THREADS * CORE_INIT)) {
        int d[CORE_INIT], c[2] = {0, 0};
#pragma unroll
        for (int i = 0; i < CORE_INIT; i++) {
            const int64_t v = b0 + i * CORE_THREADS + threadIdx.x;
            d[i] = v < a.n ? a.deg[v] : -1;
            c[0] += d[i] > 0 && d[i] <= CORE_ROW8;
            c[1] += d[i] > CORE_ROW8 && d[i] <= CORE_MID;
            isolated = isolated || d[i] == 0;
        }
        int inc[2] = {c[0], c[1]};
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y0 = __shfl_up_sync(0xffffffffu, inc[0], o), y1 = __shfl_up_sync(0xffffffffu, inc[1], o);
            if (lane >= o) {
                inc[0] += y0;
                inc[1] += y1;
            }
        }
        if (lane == 31) {
            wsum[0][warp] = inc[0];
            wsum[1][warp] = inc[1];
        }
        __syncthreads();
        if (warp < 2) {
            const int w = wsum[warp][lane];
            int wi = w;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int y = __shfl_up_sync(0xffffffffu, wi, o);
                if (lane >= o) wi += y;
            }
            wsum[warp][lane] = wi - w;
            if (lane == 31) s_base[warp] = wi ? atomicAdd(&ctl[warp ? K_MID : K_SHORT], wi) : 0;
        }
        __syncthreads();
        int at0 = s_base[0] + wsum[0][warp] + inc[0] - c[0], at1 = s_base[1] + wsum[1][warp] + inc[1] - c[1];
#pragma unroll
        for (int i = 0; i < CORE_INIT; i++) {
            const int32_t v = (int32_t)(b0 + i * CORE_THREADS + threadIdx.x);
            if (d[i] < 0) continue;
            a.val[v] = d[i];
            if (d[i] == 0) {
                a.rnd[v] = 0;
                continue;
            }
            a.nv[v] = d[i];
            a.slen[v] = -1;
            if (d[i] <= CORE_ROW8) a.shrt[at0++] = v;
            else if (d[i] <= CORE_MID) a.mid[at1++] = v;
            else append(v, a.big, &ctl[K_BIG], a.bcap, ctl);
        }
        __syncthreads();  // wsum and s_base are rewritten by the next step
    }
    if (__syncthreads_or(isolated) && threadIdx.x == 0) a.lev[0] = 1;
    if (!wait()) return;
    const int nshort = vctl[K_SHORT], nmid = vctl[K_MID], nbig = vctl[K_BIG];

    // 1. core numbers: every vertex once, then the ones that lost too much
    const Next first{0, 0, 0};
    h_pass_big(a, all, a.big, nbig, core_smem);
    h_pass(a, all, a.mid, nmid, first);
    h_pass(a, all, a.shrt, nshort, first);
    if (!wait()) return;
    tell_entries<false>(a, first);
    flush_next(a, first);
    if (!wait()) return;
    settle_first(a, all, nshort, nmid, nbig);
    Sizes z = grid_wait(K_FR, K_BFR);
    for (int r = 1; z.ok && z.a + z.b > 0;) {
        if (z.a > CORE_SOLO || z.b > 0) {
            z = value_round(a, all, z.a, z.b, r, core_smem, grid_wait);
            r++;
            continue;
        }
        if (!wait()) return;  // every block has read the sizes before one block moves on
        if (blockIdx.x == 0)
            solo_rounds<false>(a, z, r, [&](int n, int k) { return value_round(a, solo, n, 0, k, core_smem, block_wait); }, block_wait);
        z = grid_wait(K_ROUND, K_BAR);
        if (!z.ok) return;
        r = z.a;
        z.a = vctl[K_FR + (r - 1) % 3];
        z.b = vctl[K_BFR + (r - 1) % 3];
    }
    if (!z.ok) return;

    // 2. removal rounds, every level at once; round 0: the vertices with no more than their
    // level of neighbours of their own or a higher one
    __syncthreads();
    for (int i = threadIdx.x; i < CORE_BINS / 2; i += CORE_THREADS) core_smem[i] = 0;  // levels noted by this block
    __syncthreads();
    for (int part = 0; part < 3; part++) {
        const int32_t* list = part == 0 ? a.shrt : part == 1 ? a.mid : a.big;
        const int n = part == 0 ? nshort : part == 1 ? nmid : nbig;
        for (int64_t i = blockIdx.x * (int64_t)CORE_THREADS + threadIdx.x; i < n; i += (int64_t)gridDim.x * CORE_THREADS) {
            const int32_t v = list[i];
            const int k = a.val[v];
            const bool now = __ldcg(&a.cnt[v]) <= k;
            a.rnd[v] = now ? 0 : -1;
            if (now && !(k < CORE_BINS / 2 && core_smem[k])) {
                if (k < CORE_BINS / 2) core_smem[k] = 1;
                note_round(a, k, 1);
            }
        }
    }
    if (!wait()) return;
    const Next second{1, 1, 1};
    tell_entries<true>(a, second);
    flush_next(a, second);
    z = grid_wait(K_FR2 + 1, K_BFR2 + 1);
    for (int r = 1; z.ok && z.a + z.b > 0;) {
        if (z.a > CORE_SOLO || z.b > 0) {
            z = removal_round(a, all, z.a, z.b, r, grid_wait);
            r++;
            continue;
        }
        if (!wait()) return;
        if (blockIdx.x == 0)
            solo_rounds<true>(a, z, r, [&](int n, int k) { return removal_round(a, solo, n, 0, k, block_wait); }, block_wait);
        z = grid_wait(K_ROUND, K_BAR);
        if (!z.ok) return;
        r = z.a;
        z.a = vctl[K_FR2 + r % 3];
        z.b = vctl[K_BFR2 + r % 3];
    }
    if (!z.ok) return;

    // the levels' first rounds, their number and the highest level
    if (blockIdx.x == 0 && warp == 0) {
        int run = 0, top = 0;
        for (int k0 = 0; k0 <= a.hcap; k0 += 32) {
            const int k = k0 + lane;
            const int c = k <= a.hcap ? __ldcg(&a.lev[k]) : 0;
            int inc = c;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int y = __shfl_up_sync(0xffffffffu, inc, o);
                if (lane >= o) inc += y;
            }
            if (k <= a.hcap) a.lev[k] = run + inc - c;
            run += __shfl_sync(0xffffffffu, inc, 31);
            const unsigned some = __ballot_sync(0xffffffffu, c > 0);
            if (some) top = k0 + 31 - __clz(some);
        }
        if (lane == 0) {
            ctl[CORE_ROUNDS] = run;
            ctl[CORE_ALPHA] = top;
        }
    }
    if (!wait()) return;
    for (int part = 0; part < 3; part++) {
        const int32_t* list = part == 0 ? a.shrt : part == 1 ? a.mid : a.big;
        const int n = part == 0 ? nshort : part == 1 ? nmid : nbig;
        for (int64_t i = blockIdx.x * (int64_t)CORE_THREADS + threadIdx.x; i < n; i += (int64_t)gridDim.x * CORE_THREADS) {
            const int32_t v = list[i];
            a.rnd[v] = a.lev[a.val[v]] + __ldcg(&a.rnd[v]);
        }
    }
}

const int* enqueue_core_numbers(folty_graph* g, const int32_t* rowptr, const int32_t* adj, const int32_t* adj_src,
                                int32_t* rnd, int blocks, Scratch& sc, cudaStream_t s) {
    const int32_t n = g->n;
    const int64_t S = g->S;
    CoreArgs a{};
    a.rowptr = rowptr;
    a.adj = adj;
    a.src = adj_src;
    a.entries = 2 * S;
    a.deg = g->deg;
    a.n = n;
    a.hcap = (int32_t)std::min<double>(std::sqrt(2.0 * (double)S) + 1.0, (double)INT_MAX / 2);
    a.val = g->core;
    a.nv = sc.get<int32_t>(n);
    a.cnt = sc.get<int32_t>(n);
    a.rnd = rnd;
    a.shrt = sc.get<int32_t>(n);
    a.mid = sc.get<int32_t>(n);
    a.srow = sc.get<int32_t>(2 * S);
    a.slen = sc.get<int32_t>(n);
    a.slo = sc.get<int32_t>(n);
    a.fr[0] = sc.get<int32_t>(n);
    a.fr[1] = sc.get<int32_t>(n);
    a.bcap = (int32_t)(2 * S / CORE_MID + 1);
    a.big = sc.get<int32_t>(a.bcap);
    a.bfr[0] = sc.get<int32_t>(a.bcap);
    a.bfr[1] = sc.get<int32_t>(a.bcap);
    // the control words and the levels' rounds, zeroed together
    a.ctl = sc.get<int>(K_SLOTS + (int64_t)a.hcap + 2);
    a.lev = a.ctl + K_SLOTS;
    // FOLTY_CORE_TIMEOUT_MS sets a shorter bound (the tests pass it with long stretches of rounds)
    a.timeout_ns = 10ll * 1000 * 1000 * 1000;
    if (const char* env = std::getenv("FOLTY_CORE_TIMEOUT_MS")) a.timeout_ns = std::max(1ll, std::atoll(env)) * 1000 * 1000;
    FOLTY_CUDA(cudaMemsetAsync(a.ctl, 0, sizeof(int) * (K_SLOTS + (size_t)a.hcap + 2), s));
    if (n == 0) return a.ctl;
    const int smem = CORE_BINS * (int)sizeof(int) + (int)sizeof(Stage);
    FOLTY_CUDA(cudaFuncSetAttribute(k_core, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
    int per_sm = 0;
    FOLTY_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_core, CORE_THREADS, (size_t)smem));
    if (per_sm < 1) fail(FOLTY_ECUDA, "core number kernel cannot be resident");
    // 12 B per adjacency entry + 16 B per vertex
    StageSpan span(ST_PEEL, s, 12 * 2 * S + 16 * (int64_t)n);
    void* args[] = {&a};
    FOLTY_CUDA(cudaLaunchCooperativeKernel((const void*)k_core, dim3((unsigned)blocks), dim3(CORE_THREADS), args,
                                           (size_t)smem, s));
    after_launch("k_core");
    return a.ctl;
}

}  // namespace folty

// Window-probe machinery shared by the single-query, batched and allocation-free
// kernels.
//
// Flat probe space: triangle-major (tri_off = prefix of per-triangle sizes), inside a
// triangle its three static edges {u,v}, {u,w}, {v,w} in that order, inside a static
// edge its temporal edges in sorted order (E_{a->b} then E_{b->a}, a < b by id).
// A probe is one (temporal edge, witness) pair.
//
// Timestamps are stored as TS: uint32_t offsets t - t_min when the graph's time range
// fits, int64_t otherwise. Window tests only use differences, so both give the same
// answers.
#pragma once

#include <climits>

#include "internal.cuh"

namespace folty {

constexpr int PB_THREADS = 256;
constexpr int PB_ITEMS = 8;
constexpr int PB_TILE = PB_THREADS * PB_ITEMS;
constexpr int PB_GROUP = PB_THREADS;  // slots one step of a block's threads takes (live.cu)
// every triangle holds >= 3 probes, so a tile overlaps at most 1 + ceil(TILE / 3)
// triangles (+1 for the one that may start exactly at the next tile)
constexpr int PB_MAXTRI = PB_TILE / 3 + 4;

template <typename TS>
struct TsNone;
template <>
struct TsNone<uint32_t> {
    static constexpr uint32_t value = 0xffffffffu;
};
template <>
struct TsNone<int64_t> {
    static constexpr int64_t value = LLONG_MAX;
};

// Segment k (0..5) of a staged triangle = direction k & 1 of its static edge k >> 1:
// [off[3 * (k >> 1) + (k & 1)], off[3 * (k >> 1) + (k & 1) + 1]). MAXTRI = the triangles a
// tile can overlap.
template <int MAXTRI>
struct TriStageT {
    int32_t base[MAXTRI + 1];  // first probe of the triangle, relative to the tile start
    int32_t off[MAXTRI][9];    // per static edge e: [start of a->b, start of b->a, end]
    uint64_t desc[MAXTRI];     // per (e, d): L2 segment code | L3 segment code << 3
    int32_t nt;
};
using TriStage = TriStageT<PB_MAXTRI>;

// id(vertex a) < id(vertex b) for triangle-local vertices a != b in {0 = u, 1 = v, 2 = w};
// flags bit0: id(u) < id(v), bit1: id(u) < id(w), bit2: id(v) < id(w).
__host__ __device__ __forceinline__ bool id_less(int flags, int a, int b) {
    int lo = a < b ? a : b;
    int hi = a + b - lo;
    bool l = (flags >> (lo + hi - 1)) & 1;
    return (a == lo) ? l : !l;
}

// Segment codes of the role whose L1 is direction d of static edge e. Edge e joins
// local vertices (0,1), (0,2), (1,2); its witness is vertex 2 - e; the static edge
// joining local vertices i and j is edge i + j - 1. "out": L2 = E_{x,z}, L3 = E_{y,z};
// "in": E_{z,x}, E_{z,y}; "either": both directions of those static edges (the code's
// direction bit is then unused).
__host__ __device__ __forceinline__ void role_segments(int flags, int e, int d, int dir, int& seg2, int& seg3) {
    const int p = (e == 2) ? 1 : 0, q = (e == 0) ? 1 : 2, z = 2 - e;
    const int x = ((d == 0) == id_less(flags, p, q)) ? p : q;  // direction 0 runs small id -> large id
    const int y = p + q - x;
    const int exz = x + z - 1, eyz = y + z - 1;
    int d2 = id_less(flags, x, z) ? 0 : 1;  // E_{x,z}
    int d3 = id_less(flags, y, z) ? 0 : 1;  // E_{y,z}
    if (dir == FOLTY_DIR_IN) {
        d2 ^= 1;
        d3 ^= 1;
    } else if (dir == FOLTY_DIR_EITHER) {
        d2 = d3 = 0;
    }
    seg2 = 2 * exz + d2;
    seg3 = 2 * eyz + d3;
}

__device__ __forceinline__ uint64_t role_descriptor(int flags, int dir) {
    uint64_t desc = 0;
#pragma unroll
    for (int e = 0; e < 3; e++) {
#pragma unroll
        for (int d = 0; d < 2; d++) {
            int s2, s3;
            role_segments(flags, e, d, dir, s2, s3);
            desc |= (uint64_t)(s2 | (s3 << 3)) << (6 * (2 * e + d));
        }
    }
    return desc;
}

// First index in [b, e) with T[i] >= key (e if none); branch-free halving.
template <typename TS>
__device__ __forceinline__ int32_t lower_bound_ts(const TS* __restrict__ T, int32_t b, int32_t e, TS key) {
    int32_t len = e - b;
    while (len > 1) {
        int32_t half = len >> 1;
        b = (T[b + half - 1] < key) ? b + half : b;
        len -= half;
    }
    return b + ((len == 1 && T[b] < key) ? 1 : 0);
}

// N lower bounds at once, each with three loads in flight per step: for the few searches
// that stand in one another's way, half as many dependent loads, shared by all N.
template <typename TS, int N>
__device__ __forceinline__ void lower_bounds_wide(const TS* __restrict__ T, int32_t (&b)[N], const int32_t (&e)[N],
                                                  const TS (&key)[N]) {
    int32_t len[N];
    int32_t most = 0;
#pragma unroll
    for (int i = 0; i < N; i++) {
        len[i] = e[i] - b[i];
        most = max(most, len[i]);
    }
    while (most > 3) {
        TS v[N][3];
#pragma unroll
        for (int i = 0; i < N; i++) {
            const int32_t q = len[i] >> 2;
#pragma unroll
            for (int h = 0; h < 3; h++) v[i][h] = q > 0 ? T[b[i] + (h + 1) * q - 1] : key[i];
        }
        most = 0;
#pragma unroll
        for (int i = 0; i < N; i++) {
            const int32_t q = len[i] >> 2;
            const int32_t c = (v[i][0] < key[i]) + (v[i][1] < key[i]) + (v[i][2] < key[i]);
            if (q > 0) {
                b[i] += c * q;
                len[i] = c == 3 ? len[i] - 3 * q : q;
            }
            most = max(most, len[i]);
        }
    }
#pragma unroll
    for (int i = 0; i < N; i++) {
        int32_t c = 0;
#pragma unroll
        for (int h = 0; h < 3; h++) c += (h < len[i] && T[b[i] + h] < key[i]) ? 1 : 0;
        b[i] += c;
    }
}

// First entry >= key of one sorted run, or TsNone. The run's last entry is checked
// before searching (runs of different static edges rarely overlap in time).
template <typename TS>
__device__ __forceinline__ TS first_at_least_checked(const TS* __restrict__ T, int32_t b, int32_t e, TS key) {
    if (b == e || T[e - 1] < key) return TsNone<TS>::value;
    return T[lower_bound_ts(T, b, e, key)];
}

// x - t > delta for x >= t (no overflow)
template <typename TS>
__device__ __forceinline__ bool beyond(TS x, TS t, TS delta) {
    return (TS)(x - t) > delta;
}

// Theorem 3.1: t2 = first entry >= t of L2, t3 = first entry >= t2 of L3 (the first entry
// of a union of sorted runs is the smallest of their first entries). Returns t3, or
// TsNone when t2 or t3 does not exist or when t2 alone already lies beyond t + delta
// (then t3 >= t2 does too, so the caller's window test fails either way). Runs whose
// first entry lies beyond t + delta are skipped without a search.
template <typename TS, int DIR>
__device__ __forceinline__ TS probe_window(const TS* __restrict__ T, const int32_t* off, int seg2, int seg3,
                                           TS t, TS delta) {
    const TS NONE = TsNone<TS>::value;
    const int o2 = 3 * (seg2 >> 1) + (seg2 & 1), o3 = 3 * (seg3 >> 1) + (seg3 & 1);
    TS t2 = NONE;
    {
        const int32_t b = off[o2], e = off[o2 + 1];
        if (b < e && !(T[b] > t && beyond(T[b], t, delta))) t2 = first_at_least_checked(T, b, e, t);
    }
    if (DIR == FOLTY_DIR_EITHER) {
        const int32_t b = off[o2 + 1], e = off[o2 + 2];
        if (b < e && !(T[b] > t && beyond(T[b], t, delta))) {
            TS x = first_at_least_checked(T, b, e, t);
            t2 = x < t2 ? x : t2;
        }
    }
    if (t2 == NONE || beyond(t2, t, delta)) return NONE;
    TS t3 = first_at_least_checked(T, off[o3], off[o3 + 1], t2);
    if (DIR == FOLTY_DIR_EITHER) {
        TS x = first_at_least_checked(T, off[o3 + 1], off[o3 + 2], t2);
        t3 = x < t3 ? x : t3;
    }
    return t3;
}

// ------------------------------------------------------------------ probes by the shortest list
//
// A role's hits can be found from any of its three lists. From L1: each t searches t2, then
// t3. From L2: the entries t of L1 whose first entry of L2 is t2 are those in (the entry of
// L2 before t2, t2]; with t3 the first entry of L3 at or after t2, the hits among them are
// the t >= t3 - delta: one contiguous range of L1. From L3: the t2 whose first entry of L3 is
// t3 lie in (the entry of L3 before t3, t3]; the t whose first t2 is one of them lie in (the
// largest entry of L2 at or below that earlier entry of L3, the largest at or below t3],
// again a range of L1 cut at t3 - delta. Each hit is found once, from the first of equal
// entries. Edge multiplicities are heavy-tailed, so the shortest list is much shorter than
// L1: on the paper-scale recipe at 20M edges and delta = 3600 s the kept roles hold 6.35M
// entries of L1, 0.50M of the shorter of L1 and L2, and 0.09M of the shortest list; hits are
// few (1453).
//
// Slots of a role in the flat probe space, one thread each: an entry of the driving list
// or, for L1 longer than ROLE_CHUNK entries, an entry and one chunk of L1, so that no thread
// has more than ROLE_CHUNK hits to record. A role driven by L2 or L3 takes at least one slot
// per ROLE_SPREAD entries of L1, its real slots spread among them (one every 2^shift), so
// that a stretch of the probe space stands for a bounded number of possible hits however
// short the driving lists are. L1 drives unless it is long and another list halves the slots:
// with short lists the three ways only diverge within a warp (6M edges of 2 per pair: 134
// us from L1 alone, 212 us with the shortest list always).
constexpr int ROLE_CHUNK_LG = 14;
constexpr int ROLE_SPREAD_LG = 7;
constexpr int ROLE_LONG = 32;

struct RolePlan {
    int32_t slots;
    int drv;  // 1, 2, 3: the driving list
};

// The plan of a role whose L1 holds n1 >= ROLE_LONG entries (shorter ones: {n1, 1}).
__host__ __device__ __forceinline__ RolePlan long_role_plan(int32_t n1, int32_t n2, int32_t n3) {
    RolePlan p{n1, 1};
    const int32_t nd = n2 <= n3 ? n2 : n3;
    if (nd > n1 / 2) return p;  // as below, without the 64-bit arithmetic
    const int64_t chunks = ((int64_t)n1 + (1 << ROLE_CHUNK_LG) - 1) >> ROLE_CHUNK_LG;
    const int64_t spread = ((int64_t)n1 + (1 << ROLE_SPREAD_LG) - 1) >> ROLE_SPREAD_LG;
    const int64_t real = (int64_t)nd * chunks;
    const int64_t slots = real > spread ? real : spread;
    if (2 * slots <= (int64_t)n1) {
        p.slots = (int32_t)slots;
        p.drv = n2 <= n3 ? 2 : 3;
    }
    return p;
}

// Slots and driving list of the staged role r: off and code as in TriStageT.
template <int DIR>
__device__ __forceinline__ RolePlan staged_role_plan(const int32_t* off, int r, int code) {
    const int o1 = 3 * (r >> 1) + (r & 1);
    const int32_t n1 = off[o1 + 1] - off[o1];
    if (n1 < ROLE_LONG) return RolePlan{n1, 1};
    const int c2 = code & 7, c3 = code >> 3;
    const int o2 = 3 * (c2 >> 1) + (c2 & 1), o3 = 3 * (c3 >> 1) + (c3 & 1);
    constexpr int W = DIR == FOLTY_DIR_EITHER ? 2 : 1;  // "either": both runs of the static edge
    return long_role_plan(n1, off[o2 + W] - off[o2], off[o3 + W] - off[o3]);
}

// The first entry at or after key of the list off[0 .. W] (W = 2: two runs), or TsNone.
template <typename TS, int W>
__device__ __forceinline__ TS list_first(const TS* __restrict__ T, const int32_t* off, TS key) {
    int32_t b[W], e[W];
    TS k[W];
#pragma unroll
    for (int i = 0; i < W; i++) {
        b[i] = off[i];
        e[i] = off[i + 1];
        k[i] = key;
    }
    lower_bounds_wide<TS, W>(T, b, e, k);
    TS r = TsNone<TS>::value;
#pragma unroll
    for (int i = 0; i < W; i++) {
        if (b[i] < e[i]) {
            const TS x = T[b[i]];
            r = x < r ? x : r;
        }
    }
    return r;
}

// One past the largest entry below key of the list off[0 .. W], 0 when there is none: the
// first time that lies after every such entry.
template <typename TS, int W>
__device__ __forceinline__ TS list_after_below(const TS* __restrict__ T, const int32_t* off, TS key) {
    int32_t b[W], e[W];
    TS k[W];
#pragma unroll
    for (int i = 0; i < W; i++) {
        b[i] = off[i];
        e[i] = off[i + 1];
        k[i] = key;
    }
    lower_bounds_wide<TS, W>(T, b, e, k);
    TS r = 0;
#pragma unroll
    for (int i = 0; i < W; i++) {
        if (b[i] > off[i]) {
            const TS x = T[b[i] - 1] + 1;
            r = x > r ? x : r;
        }
    }
    return r;
}

// The driving entry at position p of the list off[0 .. W]: its time, and in from the first
// time after every smaller entry of the list; false when an equal entry comes first (in
// the order of the runs).
template <typename TS, int W>
__device__ __forceinline__ bool driving_entry(const TS* __restrict__ T, const int32_t* off, int32_t p, TS& v, TS& from) {
    const int32_t mid = off[1];
    const bool second = W == 2 && p >= mid;
    const TS before = p > (second ? mid : off[0]) ? T[p - 1] : TsNone<TS>::value;
    v = T[p];
    from = 0;
    if (before == v) return false;
    if (before != TsNone<TS>::value) from = before + 1;
    if (W == 2) {
        int32_t b[1] = {second ? off[0] : mid};
        const int32_t b0 = b[0], e[1] = {second ? mid : off[2]};
        const TS key[1] = {v};
        lower_bounds_wide<TS, 1>(T, b, e, key);
        const TS at = b[0] < e[0] ? T[b[0]] : TsNone<TS>::value;
        const TS x = b[0] > b0 ? T[b[0] - 1] + 1 : (TS)0;
        if (second && at == v) return false;
        from = x > from ? x : from;
    }
    return true;
}

// Hits of slot k (0 <= k < drivers * chunks) of a role driven by list drv (2 or 3): the
// positions [lo, hi) of L1 whose window test finds t3 within delta. The cheap tests (L1's
// ends, the gap at its smallest) come before the searches; most slots end there.
template <typename TS, int DIR>
__device__ __forceinline__ void driven_range(const TS* __restrict__ T, const int32_t* off, int r, int code, int drv,
                                             int32_t k, TS delta, int32_t& lo, int32_t& hi, TS& t3) {
    constexpr int W = DIR == FOLTY_DIR_EITHER ? 2 : 1;
    const int o1 = 3 * (r >> 1) + (r & 1), c2 = code & 7, c3 = code >> 3;
    const int32_t* l2 = off + 3 * (c2 >> 1) + (c2 & 1);
    const int32_t* l3 = off + 3 * (c3 >> 1) + (c3 & 1);
    const int32_t* ld = drv == 2 ? l2 : l3;
    int32_t b1 = off[o1], e1 = off[o1 + 1];
    int32_t i = k;
    if (e1 - b1 > (1 << ROLE_CHUNK_LG)) {  // slot k: entry k mod nd, chunk k / nd
        const int32_t nd = ld[W] - ld[0], c = k / nd;
        i = k - c * nd;
        b1 += c << ROLE_CHUNK_LG;
        e1 = min(e1, b1 + (1 << ROLE_CHUNK_LG));
    }
    lo = hi = 0;
    const TS first1 = T[b1], last1 = T[e1 - 1];
    TS v, from;
    if (!driving_entry<TS, W>(T, ld, ld[0] + i, v, from)) return;
    if (first1 > v) return;
    TS top;  // the latest t that can hit
    if (drv == 2) {
        top = v;
        if (last1 < from) return;
        t3 = list_first<TS, W>(T, l3, v);
        if (t3 == TsNone<TS>::value || beyond(t3, v, delta)) return;
    } else {
        t3 = v;
        const TS last = list_after_below<TS, W>(T, l2, (TS)(t3 + 1));  // one past the latest t2 <= t3
        if (last == 0 || last <= from || beyond(t3, (TS)(last - 1), delta) || first1 >= last) return;
        top = last - 1;
        from = list_after_below<TS, W>(T, l2, from);  // after every entry of L2 before from
        if (last1 < from) return;
    }
    const TS near = t3 > delta ? (TS)(t3 - delta) : (TS)0;
    int32_t b[2] = {b1, b1};
    const int32_t e[2] = {e1, e1};
    const TS key[2] = {near > from ? near : from, (TS)(top + 1)};
    lower_bounds_wide<TS, 2>(T, b, e, key);
    lo = b[0];
    hi = max(b[1], b[0]);
}

// Stages the triangles overlapping this block's probe tile: tile_tri[b] is the triangle
// holding probe min(b * PB_TILE, P - 1).
__device__ __forceinline__ void stage_triangles(TriStage& st, const int4* __restrict__ tri,
                                                const int64_t* __restrict__ tri_off,
                                                const int64_t* __restrict__ tile_tri,
                                                const int32_t* __restrict__ seg, int dir) {
    const int64_t t0 = tile_tri[blockIdx.x];
    const int nt = (int)(tile_tri[blockIdx.x + 1] - t0 + 1);
    const int64_t p0 = (int64_t)blockIdx.x * PB_TILE;
    for (int j = threadIdx.x; j < nt; j += blockDim.x) {
        int4 tr = tri[t0 + j];
        st.base[j] = (int32_t)(tri_off[t0 + j] - p0);
        st.desc[j] = role_descriptor(tr.w, dir);
        const int32_t se[3] = {tr.x, tr.y, tr.z};
#pragma unroll
        for (int e = 0; e < 3; e++) {
            st.off[j][3 * e] = seg[2 * se[e]];
            st.off[j][3 * e + 1] = seg[2 * se[e] + 1];
            st.off[j][3 * e + 2] = seg[2 * se[e] + 2];
        }
    }
    if (threadIdx.x == 0) {
        st.nt = nt;
        st.base[nt] = INT_MAX;
    }
    __syncthreads();
}

struct Probe {
    int32_t pos;         // sorted position of the temporal edge (L1 entry)
    int32_t seg2, seg3;  // segment codes of L2 and L3
    int32_t j;           // staged triangle
};

// Locates probe `local` (tile-relative) for every lane of the warp. All lanes call it
// (warp-uniform); `active` marks lanes with a probe. One lane bisects for the warp's
// first probe, then each lane walks forward (a warp's 32 consecutive probes span few
// triangles).
__device__ __forceinline__ Probe locate_probe(const TriStage& st, int32_t local, bool active) {
    const int lane = threadIdx.x & 31;
    int32_t first = __shfl_sync(0xffffffffu, local, 0);
    int j0 = 0;
    if (lane == 0) {
        int lo = 0, hi = st.nt - 1;
        while (lo < hi) {
            int mid = (lo + hi + 1) >> 1;
            if (st.base[mid] <= first) lo = mid;
            else hi = mid - 1;
        }
        j0 = lo;
    }
    int j = __shfl_sync(0xffffffffu, j0, 0);
    Probe pr;
    pr.pos = 0;
    pr.seg2 = pr.seg3 = 0;
    if (active) {
        while (st.base[j + 1] <= local) j++;
        const int32_t* off = st.off[j];
        int32_t o = local - st.base[j];
        int e = 0;
        int32_t s0 = off[2] - off[0];
        if (o >= s0) {
            o -= s0;
            e = 1;
            int32_t s1 = off[5] - off[3];
            if (o >= s1) {
                o -= s1;
                e = 2;
            }
        }
        pr.pos = off[3 * e] + o;
        const int d = pr.pos >= off[3 * e + 1];
        const int code = (int)((st.desc[j] >> (6 * (2 * e + d))) & 63);
        pr.seg2 = code & 7;
        pr.seg3 = code >> 3;
    }
    pr.j = j;
    return pr;
}

}  // namespace folty

// Window probes restricted to roles that can hit.
//
// A role (temporal edges x -> y of one static edge, witness z; lists L1 = E_{x,y}, L2,
// L3 of its direction variant) can only produce a window match t <= t2 <= t3 <= t + delta
// if its runs overlap in time: L2 must end at or after L1 starts, L3 must end at or
// after max(L1.first, L2.first), and L2 and L3 must start by L1.last + delta. The first
// two conditions do not depend on delta; the last two hold exactly when
// delta >= dmin = max(0, L2.first - L1.last, L3.first - L1.last).
//
// A role's bucket is a conservative form of dmin for one direction variant: its bit
// length b (0 for dmin = 0, 255 for "never"), so 2^(b-1) <= dmin. A query keeps a role
// when delta >= 2^(b-1), which holds whenever delta >= dmin: no role that can hit is
// dropped (a few that cannot are kept). Preprocessing stores the first and last
// timestamp and the size of every run (the run-ends table) and, per triangle and
// direction variant, the smallest bucket of its six roles (one byte). A query reads that
// byte for every triangle; only the triangles it keeps (typically a few in ten thousand)
// get their six roles' buckets and sizes from the run-ends table. It then lays the kept
// roles out in a flat probe space (3 idle slots per triangle keep the tile staging bound)
// and probes only those, with the exact window test of Theorem 3.1.
#include <type_traits>

#include "internal.cuh"
#include "liveness.cuh"
#include "probe.cuh"
#include "scan.cuh"

namespace folty {

constexpr int LIVE_IDLE = 3;  // idle slots per kept triangle (keeps >= 3 slots per triangle)

template <typename TS>
__global__ void k_run_ends(const int32_t* __restrict__ seg, int64_t S, const TS* __restrict__ T,
                           RunEnds<TS>* __restrict__ ends) {
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < S; e += (int64_t)gridDim.x * blockDim.x) {
        const int32_t o0 = seg[2 * e], o1 = seg[2 * e + 1], o2 = seg[2 * e + 2];
        RunEnds<TS> r;
        r.n0 = o1 - o0;
        r.n1 = o2 - o1;
        r.f0 = r.n0 > 0 ? T[o0] : RunEmpty<TS>::first;
        r.l0 = r.n0 > 0 ? T[o1 - 1] : RunEmpty<TS>::last;
        r.f1 = r.n1 > 0 ? T[o1] : RunEmpty<TS>::first;
        r.l1 = r.n1 > 0 ? T[o2 - 1] : RunEmpty<TS>::last;
        r.pad0 = r.pad1 = 0;
        ends[e] = r;
    }
}

// The liveness byte of every listed triangle for direction variant DIR (liveness_byte),
// one thread per entry of the triangle array (an empty one gets "never"): consecutive
// triangles share their first edge, so its record mostly comes from L1.
template <typename TS, int DIR>
__global__ void k_tri_live(const int4* __restrict__ tri, int64_t cap, const RunEnds<TS>* __restrict__ ends,
                           uint8_t* __restrict__ row) {
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < cap; t += (int64_t)gridDim.x * blockDim.x) {
        const int4 tr = __ldcs(tri + t);
        row[t] = tr.w < 0 ? DMIN_NEVER : liveness_byte<TS, DIR>(tr, ends);
    }
}

__device__ __forceinline__ bool bucket_live(uint8_t b, int64_t delta) {
    return b != DMIN_NEVER && (b == 0 || delta >= ((int64_t)1 << (b - 1)));
}

// Role mask (stored role order: bit 2e + d = direction d of stored edge e) and probe slots
// of the kept roles of triangle tr at window delta for direction variant DIR.
template <typename TS, int DIR>
__device__ __forceinline__ int kept_roles_of(const int4 tr, const RunEnds<TS>* __restrict__ ends, int64_t delta,
                                             int64_t& slots) {
    FrameRuns<TS> fr;
    frame_runs<TS>(tr, ends, fr);
    int m = 0;
    int64_t c = 0;
#pragma unroll
    for (int r = 0; r < 6; r++) {
        if (bucket_live(frame_bucket<DIR, TS>(fr, r), delta)) {  // never for an empty run
            m |= 1 << (2 * fr.oe[r >> 1] + (r & 1));
            int32_t n = fr.n[r];
            if (n >= ROLE_LONG) {
                int s2, s3;
                role_segments(7, r >> 1, r & 1, DIR, s2, s3);
                const int32_t n2 = DIR == FOLTY_DIR_EITHER ? fr.n[s2] + fr.n[s2 + 1] : fr.n[s2];
                const int32_t n3 = DIR == FOLTY_DIR_EITHER ? fr.n[s3] + fr.n[s3 + 1] : fr.n[s3];
                n = long_role_plan(n, n2, n3).slots;
            }
            c += n;
        }
    }
    slots = c;
    return m;
}

// Kept roles of every triangle for one query: kept triangle j = L[j] with its role mask
// lmask[j] and its first probe slot loff[j] (the kept triangles' costs = the kept roles'
// slots (probe.cuh) + LIVE_IDLE idle ones, laid out one after another); totals[0] = kept triangles, totals[1]
// = slots, loff[totals[0]] = totals[1]; and the map of the probe groups (PB_GROUP slots):
// ltile[b] = kept triangle holding slot min(b * ptile, slots - 1) for b <= the number of
// groups (each kept triangle writes the group starts inside its slots).
//
// Two passes. k_live_candidates streams the row of liveness bytes (the smallest bucket of
// each triangle's roles for this direction variant; a thread 32 of them per step, the next
// step's 16-byte loads in flight) and lists the triangles whose byte admits delta, one
// addition per block and step. They are few, but cluster; k_live_select takes them from the
// list, one thread each, so the work is even whatever their places: it reads their records
// and run ends, orders the costs of a warp's 32 by a scan and reserves their entries and
// slots together with one 64-bit addition (kept triangles << LS_UNIT_BITS | slots). The list
// is therefore in the order of the reservations, not of the triangles: the probes only add
// to counters, so no result depends on it. The last block to finish writes the totals and
// clears the counters for the next selection.
//
// It replaced a counting pass, a one-block scan of the warps' sums and a writing pass that
// read every kept triangle again: 122 us for 76M triangles of which 42K are kept, 75 us for
// 68K triangles (warps of 2048 triangles left all but a few SMs idle); now 28 and 9 us. One
// kernel whose warps or blocks worked off their own candidates took 50 to 75 us at 76M:
// thousands of neighbouring triangles may all be candidates.
constexpr int LS_THREADS = 256;
constexpr int LS_ITEMS = 32;
constexpr int LS_PER_SM = 8;      // blocks per SM of both passes
constexpr int LS_UNIT_BITS = 33;  // packed counter: kept triangles << 33 | slots in units

// Bit i of the result: byte i of the ITEMS liveness bytes in w admits delta (rows are padded
// with DMIN_NEVER to whole 16-byte chunks). A byte b admits delta exactly when
// b <= B = bit length of delta (b = 0 always, b >= 1 when delta >= 2^(b-1); DMIN_NEVER
// never, as B <= 63): four bytes at a time, (0x80 + B) - (b & 0x7f) keeps bit 7 set
// exactly for b <= B (bytes never borrow from one another, and 255 & 0x7f = 127 > B), and
// one multiplication gathers the four bit-7s. bias = 0x80 + B in every byte.
template <int ITEMS>
__device__ __forceinline__ uint32_t live_mask(const uint4 (&w)[ITEMS / 16], uint32_t bias) {
    uint32_t lm = 0;
#pragma unroll
    for (int h = 0; h < ITEMS / 16; h++) {
        const uint32_t ws[4] = {w[h].x, w[h].y, w[h].z, w[h].w};
#pragma unroll
        for (int q = 0; q < 4; q++) {
            const uint32_t hit = (bias - (ws[q] & 0x7f7f7f7fu)) & 0x80808080u;
            const uint32_t nib = ((hit >> 7) * 0x10204080u) >> 28;  // bit j = byte j admits delta
            lm |= nib << (16 * h + 4 * q);
        }
    }
    return lm;
}

template <int ITEMS>
__device__ __forceinline__ void live_load(const uint8_t* __restrict__ tlive, int64_t t0, int64_t ntri,
                                          uint4 (&w)[ITEMS / 16]) {
#pragma unroll
    for (int h = 0; h < ITEMS / 16; h++) {
        w[h] = make_uint4(~0u, ~0u, ~0u, ~0u);
        if (t0 + 16 * h < ntri) w[h] = __ldcs(reinterpret_cast<const uint4*>(tlive + t0 + 16 * h));
    }
}

// The selection's counters, zero between selections.
struct SelectCtl {
    unsigned long long packed;  // kept triangles << LS_UNIT_BITS | slots in units
    unsigned int cand, done;    // candidates, blocks of k_live_select done
};

// The triangles whose byte admits delta, in no particular order, into cand.
template <int ITEMS>
__global__ void __launch_bounds__(LS_THREADS) k_live_candidates(const uint8_t* __restrict__ tlive, int64_t ntri,
                                                                int64_t delta, const int64_t* __restrict__ qp,
                                                                SelectCtl* ctl, int32_t* __restrict__ cand) {
    __shared__ int warp_tot[LS_THREADS / 32];
    __shared__ int total;
    __shared__ unsigned int base;
    if (qp) delta = qp[0];  // the window from a device parameter block (replayed query plans)
    const uint32_t bias = 0x80808080u | ((delta > 0 ? (uint32_t)(64 - __clzll((unsigned long long)delta)) : 0u) * 0x01010101u);
    const int64_t stride = (int64_t)gridDim.x * (LS_THREADS * ITEMS);
    int64_t t0 = ((int64_t)blockIdx.x * LS_THREADS + threadIdx.x) * ITEMS;
    uint4 next[ITEMS / 16];
    live_load<ITEMS>(tlive, t0, ntri, next);
    for (int64_t b0 = (int64_t)blockIdx.x * (LS_THREADS * ITEMS); b0 < ntri; b0 += stride, t0 += stride) {
        uint32_t lm = live_mask<ITEMS>(next, bias);
        live_load<ITEMS>(tlive, t0 + stride, ntri, next);
        if (!__syncthreads_or(lm != 0)) continue;
        int at = block_exclusive_sum<int>(__popc(lm), warp_tot, &total);
        if (threadIdx.x == 0) base = atomicAdd(&ctl->cand, (unsigned int)total);
        __syncthreads();
        for (at += (int)base; lm; lm &= lm - 1) cand[at++] = (int32_t)(t0 + __ffs((int)lm) - 1);
    }
}

struct SelectArgs {
    const int4* tri;
    const int32_t* cand;
    int64_t delta;
    const int64_t* qp;  // may be null: device parameter block whose slot 0 holds the window
    int ush;            // log2 of the slots per unit of the packed counter
    SelectCtl* ctl;
    int32_t* L;
    int64_t* loff;
    uint8_t* lmask;
    int64_t* ltile;
    int64_t max_tiles, ptile;
    int64_t* totals;
    unsigned long long* prof;  // may be null
};

template <typename TS, int DIR>
__global__ void __launch_bounds__(LS_THREADS) k_live_select(const SelectArgs a, const RunEnds<TS>* __restrict__ ends) {
    const int64_t delta = a.qp ? a.qp[0] : a.delta;
    const int lane = threadIdx.x & 31;
    const int64_t total = (int64_t)*(volatile unsigned int*)&a.ctl->cand;
    const int64_t stride = (int64_t)gridDim.x * LS_THREADS;
    for (int64_t k0 = (int64_t)blockIdx.x * LS_THREADS + (threadIdx.x & ~31); k0 < total; k0 += stride) {
        const bool on = k0 + lane < total;
        int32_t t = 0;
        int m = 0;
        int64_t v = 0;
        if (on) {
            t = a.cand[k0 + lane];
            m = kept_roles_of<TS, DIR>(a.tri[t], ends, delta, v);
            v += LIVE_IDLE;
        }
        int64_t inc = v;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int64_t y = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc += y;
        }
        const int64_t all = __shfl_sync(0xffffffffu, inc, 31);
        const int64_t units = (all + ((int64_t)1 << a.ush) - 1) >> a.ush;
        const int n = (int)min(total - k0, (int64_t)32);
        unsigned long long base = 0;
        if (lane == 0)
            base = atomicAdd(&a.ctl->packed, ((unsigned long long)n << LS_UNIT_BITS) | (unsigned long long)units);
        base = __shfl_sync(0xffffffffu, base, 0);
        if (on) {
            const int64_t jc = (int64_t)(base >> LS_UNIT_BITS) + lane;
            const int64_t jp = ((int64_t)(base & ((1ull << LS_UNIT_BITS) - 1)) << a.ush) + inc - v;
            // the step's last triangle also holds the slots that round the step up to whole units
            const int64_t end = jp + v + (lane == n - 1 ? (units << a.ush) - all : 0);
            a.L[jc] = t;
            a.loff[jc] = jp;
            a.lmask[jc] = (uint8_t)m;
            for (int64_t b = (jp + a.ptile - 1) / a.ptile; b * a.ptile < end && b <= a.max_tiles; b++) a.ltile[b] = jc;
        }
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        if (atomicAdd(&a.ctl->done, 1u) == gridDim.x - 1) {
            __threadfence();
            const unsigned long long c = *(volatile unsigned long long*)&a.ctl->packed;
            const int64_t nl = (int64_t)(c >> LS_UNIT_BITS);
            const int64_t P = (int64_t)(c & ((1ull << LS_UNIT_BITS) - 1)) << a.ush;
            a.totals[0] = nl;
            a.totals[1] = P;
            a.loff[nl] = P;
            const int64_t tiles = (P + a.ptile - 1) / a.ptile;
            if (P > 0 && tiles <= a.max_tiles) a.ltile[tiles] = nl - 1;
            if (a.prof) atomicAdd(a.prof, (unsigned long long)((16 + 3 * sizeof(RunEnds<TS>) + 13 + 8) * nl));
            *a.ctl = SelectCtl{0, 0, 0};
        }
    }
}

// Model bytes of a staged triangle's kept roles (its first slot lies in this tile):
// staging 61 B, and per role, driven by a list of nd entries: w nd + w min(n, nd
// ceil(log2(n + 1))) for each of the two other lists of n entries, w = bytes per timestamp.
template <typename TS, int DIR>
__device__ __forceinline__ unsigned long long kept_role_bytes(const int32_t* off, int m, uint64_t desc) {
    const int64_t w = sizeof(TS);
    unsigned long long b = 61;
    for (int r = 0; r < 6; r++) {
        if (!((m >> r) & 1)) continue;
        const int code = (int)((desc >> (6 * r)) & 63);
        const int o1 = 3 * (r >> 1) + (r & 1), c2 = code & 7, c3 = code >> 3;
        const int o2 = 3 * (c2 >> 1) + (c2 & 1), o3 = 3 * (c3 >> 1) + (c3 & 1);
        constexpr int W = DIR == FOLTY_DIR_EITHER ? 2 : 1;
        const int64_t n[3] = {off[o1 + 1] - off[o1], off[o2 + W] - off[o2], off[o3 + W] - off[o3]};
        const int d = staged_role_plan<DIR>(off, r, code).drv - 1;
        b += (unsigned long long)(w * n[d]);
#pragma unroll
        for (int l = 0; l < 3; l++)
            if (l != d) b += (unsigned long long)(w * min(n[l], n[d] * (64 - __clzll((unsigned long long)n[l]))));
    }
    return b;
}

// What a hit does: count, bin or mark its edge.
enum { PROBE_COUNT = 0, PROBE_BIN = 1, PROBE_MARK = 2 };

struct LiveArgs {
    const int4* tri;
    const int32_t* seg;
    const int32_t* L;
    const int64_t* loff;
    const uint8_t* lmask;
    const int64_t* ltile;
    const int64_t* P;  // device: total slots
    int32_t* cnt;      // PROBE_COUNT counters or PROBE_BIN bins, as int32, or
    uint32_t* cnt16;   // 16-bit ones, two to a word
    uint32_t* bits;    // PROBE_COUNT, may be null: bit g set when a sorted edge of [32 g, 32 g + 32) was hit;
                       // PROBE_MARK: bit e set when sorted edge e was hit; PROBE_BIN: the marks
    const int32_t* wpref;      // PROBE_BIN: marked edges before each word of the marks
    int k, kstride;            // PROBE_BIN: number of bins, bins per row
    unsigned long long* prof;  // model bytes of the kept roles (may be null)
    uint8_t* rflag;    // PROBE_COUNT, may be null: 6 * triangle + role flags of roles with a hit
    const int64_t* qp; // may be null: a device block whose slot 0 (64-bit store) or 1 (32-bit
                       // store) holds the window, read instead of the delta argument
};

constexpr int PROBE_LANE_HITS = 4;

__device__ __forceinline__ uint32_t shfl_ts(uint32_t v, int src) { return __shfl_sync(0xffffffffu, v, src); }
__device__ __forceinline__ int64_t shfl_ts(int64_t v, int src) {
    return (int64_t)__shfl_sync(0xffffffffu, (long long)v, src);
}

__device__ __forceinline__ void set_bit(uint32_t* bits, int32_t i) {
    // a plain read first: most hits find the bit already set
    const uint32_t bit = 1u << (i & 31);
    if (!(bits[i >> 5] & bit)) atomicOr(&bits[i >> 5], bit);
}

// Records the hit of the sorted edge at pos with window end t3.
template <typename TS, int MODE>
__device__ __forceinline__ void record_hit(const LiveArgs& a, const TS* __restrict__ T, const TS* sD, int32_t pos,
                                           TS t3) {
    if (MODE == PROBE_MARK) {
        set_bit(a.bits, pos);
        return;
    }
    int64_t x = pos;
    if (MODE == PROBE_BIN)
        x = (int64_t)row_of(a.bits, a.wpref, pos) * a.kstride + lower_bound_ts<TS>(sD, 0, a.k, (TS)(t3 - T[pos]));
    if (a.cnt16) atomicAdd(&a.cnt16[x >> 1], 1u << (16 * (int)(x & 1)));
    else atomicAdd(&a.cnt[x], 1);
    if (MODE == PROBE_COUNT && a.bits) set_bit(a.bits, pos >> 5);
}

// PROBE_COUNT: cnt[pos] += hit at window delta. PROBE_BIN: bin the gap t3 - t (<= delta, the
// largest bin bound) against the sorted bounds deltas[0..k). PROBE_MARK: mark pos. A block
// takes probe tiles of up to PB_GROUP * ITEMS slots (the tile size the autotuner picks); a
// thread takes a slot: one entry of a kept role's driving list (probe.cuh). The lanes of a warp
// first find their roles, which takes them different numbers of steps, then probe together: with
// the probe inside the search, each step's lanes probed alone (20 edges between every two of 300
// vertices, most probes hits, both directions: 8.1 ms against 5.5, 4.3 before the roles had
// slots of three kinds; 4M edges of skewed degrees 5.4 against 4.7).
template <typename TS, int DIR, int MODE, int ITEMS>
__global__ void __launch_bounds__(PB_THREADS) k_probe_live(LiveArgs a, const TS* __restrict__ T, TS delta,
                                                           const TS* __restrict__ deltas) {
    constexpr int MAXTRI = PB_GROUP * ITEMS / 3 + 4;  // every kept triangle holds >= 3 slots
    __shared__ TriStageT<MAXTRI> st;
    __shared__ uint8_t smask[MAXTRI];
    __shared__ TS sD[MODE == PROBE_BIN ? 1024 : 1];
    if (a.qp) delta = (TS)a.qp[sizeof(TS) == 4 ? 1 : 0];
    if (MODE == PROBE_BIN)
        for (int i = threadIdx.x; i < a.k; i += blockDim.x) sD[i] = deltas[i];
    const int64_t P = *a.P;
    const int64_t groups = (P + PB_GROUP - 1) / PB_GROUP;
    // a slot is a chain of searches: fewer groups per tile while that gives more blocks work
    const int64_t each = min(max(groups / gridDim.x, (int64_t)1), (int64_t)ITEMS);
    for (int64_t b = (int64_t)blockIdx.x * each; b < groups; b += (int64_t)gridDim.x * each) {
        __syncthreads();  // the previous tile's stage is no longer read
        const int64_t be = min(b + each, groups);
        const int64_t t0 = a.ltile[b];
        const int nt = (int)(a.ltile[be] - t0 + 1);
        const int64_t p0 = b * (int64_t)PB_GROUP;
        unsigned long long pbytes = 0;
        for (int j = threadIdx.x; j < nt; j += blockDim.x) {
            const int4 tr = a.tri[a.L[t0 + j]];
            st.base[j] = (int32_t)(a.loff[t0 + j] - p0);
            st.desc[j] = role_descriptor(tr.w, DIR);
            smask[j] = a.lmask[t0 + j];
            const int32_t se[3] = {tr.x, tr.y, tr.z};
#pragma unroll
            for (int e = 0; e < 3; e++) {
                st.off[j][3 * e] = a.seg[2 * se[e]];
                st.off[j][3 * e + 1] = a.seg[2 * se[e] + 1];
                st.off[j][3 * e + 2] = a.seg[2 * se[e] + 2];
            }
            if (a.prof && st.base[j] >= 0) pbytes += kept_role_bytes<TS, DIR>(st.off[j], smask[j], st.desc[j]);
        }
        if (a.prof) {
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) pbytes += __shfl_xor_sync(0xffffffffu, pbytes, o);
            if ((threadIdx.x & 31) == 0 && pbytes) atomicAdd(a.prof, pbytes);
        }
        if (threadIdx.x == 0) {
            st.nt = nt;
            st.base[nt] = INT_MAX;
        }
        __syncthreads();
        const int32_t count = (int32_t)min((be - b) * PB_GROUP, P - p0);
#pragma unroll 1
        for (int it = 0; it < (int)(be - b); it++) {
            const int32_t local = it * PB_THREADS + (int32_t)threadIdx.x;
            if ((local & ~31) >= count) break;  // warp-uniform
            const bool active = local < count;
            // triangle of the slot: one lane bisects for the warp, lanes walk forward
            const int lane = threadIdx.x & 31;
            const int32_t first = __shfl_sync(0xffffffffu, local, 0);
            int j = 0;
            if (lane == 0) {
                int lo = 0, hi = st.nt - 1;
                while (lo < hi) {
                    int mid = (lo + hi + 1) >> 1;
                    if (st.base[mid] <= first) lo = mid;
                    else hi = mid - 1;
                }
                j = lo;
            }
            j = __shfl_sync(0xffffffffu, j, 0);
            // the slot's role and its place in it
            int r = -1;
            int32_t o = 0;
            RolePlan rp{0, 1};
            if (active) {
                while (st.base[j + 1] <= local) j++;
                o = local - st.base[j] - LIVE_IDLE;
                for (int m = o >= 0 ? smask[j] : 0; m; m &= m - 1) {
                    const int at = __ffs(m) - 1;
                    rp = staged_role_plan<DIR>(st.off[j], at, (int)((st.desc[j] >> (6 * at)) & 63));
                    if (o < rp.slots) {
                        r = at;
                        break;
                    }
                    o -= rp.slots;
                }
            }
            __syncwarp();  // the lanes find their roles after different steps, and probe together
            // this slot's hits: positions [lo, hi) of L1, all with the same t3
            int32_t lo = 0, hi = 0;
            TS t3 = 0;
            if (r >= 0) {
                const int32_t* off = st.off[j];
                const int code = (int)((st.desc[j] >> (6 * r)) & 63);
                if (rp.drv == 1) {
                    lo = hi = off[3 * (r >> 1) + (r & 1)] + o;
                    // an edge is marked by its first hit: most probes are saved where most hit (64
                    // queries on 200 edges between every two of 300 vertices: 207 -> 155 ms)
                    if (MODE != PROBE_MARK || !((__ldcg(&a.bits[lo >> 5]) >> (lo & 31)) & 1u)) {
                        const TS t = T[lo];
                        t3 = probe_window<TS, DIR>(T, off, code & 7, code >> 3, t, delta);
                        if (t3 != TsNone<TS>::value && (TS)(t3 - t) <= delta) hi++;
                    }
                } else {
                    const int c = rp.drv == 2 ? code & 7 : code >> 3;
                    const int32_t* ld = off + 3 * (c >> 1) + (c & 1);
                    const int32_t n1 = off[3 * (r >> 1) + (r & 1) + 1] - off[3 * (r >> 1) + (r & 1)];
                    const int32_t real = (ld[DIR == FOLTY_DIR_EITHER ? 2 : 1] - ld[0]) *
                                         (int32_t)(((int64_t)n1 + (1 << ROLE_CHUNK_LG) - 1) >> ROLE_CHUNK_LG);
                    int sh = __clz(real) - __clz(rp.slots);  // the largest with real << sh <= slots
                    if (((int64_t)real << sh) > rp.slots) sh--;
                    if ((o & ((1 << sh) - 1)) == 0 && (o >> sh) < real)
                        driven_range<TS, DIR>(T, off, r, code, rp.drv, o >> sh, delta, lo, hi, t3);
                }
                if (MODE == PROBE_COUNT && hi > lo && a.rflag) a.rflag[6 * (int64_t)a.L[t0 + j] + r] = 1;
            }
            // short ranges by their lane, the others by the whole warp
            if (hi - lo <= PROBE_LANE_HITS)
                for (int32_t pos = lo; pos < hi; pos++) record_hit<TS, MODE>(a, T, sD, pos, t3);
            unsigned wide = __ballot_sync(0xffffffffu, hi - lo > PROBE_LANE_HITS);
            while (wide) {
                const int src = __ffs(wide) - 1;
                wide &= wide - 1;
                const int32_t p0r = __shfl_sync(0xffffffffu, lo, src), p1r = __shfl_sync(0xffffffffu, hi, src);
                const TS x = shfl_ts(t3, src);
                for (int32_t pos = p0r + lane; pos < p1r; pos += 32) record_hit<TS, MODE>(a, T, sD, pos, x);
            }
        }
    }
}

// ------------------------------------------------------------------ host side

template <typename TS>
static void run_ends_t(folty_graph* g, cudaStream_t s) {
    const int64_t S = g->S;
    RunEnds<TS>* ends = static_cast<RunEnds<TS>*>(g->run_ends);
    // per static edge: 12 B of run bounds and 4 timestamps read, its record written
    StageSpan span(ST_ROLES, s, S * (12 + 4 * (int64_t)sizeof(TS) + (int64_t)sizeof(RunEnds<TS>)));
    if (S > 0) FOLTY_LAUNCH(k_run_ends<TS>, grid_for(S, 256), 256, 0, s, g->seg, S, (const TS*)g->T, ends);
}

void build_run_ends(folty_graph* g, cudaStream_t s) {
    g->run_ends = g->ts32 ? (void*)graph_alloc<RunEnds<uint32_t>>(g, g->S, s)
                          : (void*)graph_alloc<RunEnds<int64_t>>(g, g->S, s);
    if (g->ts32) run_ends_t<uint32_t>(g, s);
    else run_ends_t<int64_t>(g, s);
}

int64_t liveness_stride(int64_t entries) { return (entries + 15) & ~int64_t(15); }

uint8_t* liveness_rows(folty_graph* g, int rows, int64_t entries, cudaStream_t s) {
    // each padded with DMIN_NEVER to whole 16-byte chunks (every pass writes the bytes of all
    // entries of the triangle array)
    const int64_t stride = liveness_stride(entries);
    uint8_t* base = graph_alloc<uint8_t>(g, rows * stride, s);
    for (int d = 0; d < rows && stride > entries; d++)
        FOLTY_CUDA(cudaMemsetAsync(base + d * stride + entries, DMIN_NEVER, (size_t)(stride - entries), s));
    return base;
}

void prepare_liveness(folty_graph* g, cudaStream_t s) {
    uint8_t* base = liveness_rows(g, 3, g->tri_cap, s);
    for (int d = 0; d < 3; d++) g->tlive[d] = base + d * liveness_stride(g->tri_cap);
}

template <typename TS>
static void liveness_row_t(folty_graph* g, int dir, cudaStream_t s) {
    const int64_t cap = g->tri_cap;
    // per entry: its record read and one byte written; the run-ends table (shared by
    // the triangles of an edge, and small) read once
    StageSpan span(ST_ROLES, s, cap * (16 + 1) + g->S * (int64_t)sizeof(RunEnds<TS>));
    if (g->ntri == 0) return;
    const RunEnds<TS>* ends = (const RunEnds<TS>*)g->run_ends;
    uint8_t* row = g->tlive[dir];
    const unsigned grid = grid_for(cap, 256);
    if (dir == FOLTY_DIR_OUT) FOLTY_LAUNCH((k_tri_live<TS, FOLTY_DIR_OUT>), grid, 256, 0, s, g->tri, cap, ends, row);
    else if (dir == FOLTY_DIR_IN) FOLTY_LAUNCH((k_tri_live<TS, FOLTY_DIR_IN>), grid, 256, 0, s, g->tri, cap, ends, row);
    else FOLTY_LAUNCH((k_tri_live<TS, FOLTY_DIR_EITHER>), grid, 256, 0, s, g->tri, cap, ends, row);
}

// Each direction variant's liveness row is computed by the first call that needs it
// (preprocessing computes the paper's "out" motif's): a graph queried with one variant
// only pays for that one.
void ensure_liveness(folty_graph* g, int dir, cudaStream_t s) {
    std::lock_guard<std::mutex> lock(g->live_mu);
    if (!g->live_ready[dir]) {
        if (g->ts32) liveness_row_t<uint32_t>(g, dir, s);
        else liveness_row_t<int64_t>(g, dir, s);
        if (!g->live_ev[dir]) FOLTY_CUDA(cudaEventCreateWithFlags(&g->live_ev[dir], cudaEventDisableTiming));
        FOLTY_CUDA(cudaEventRecord(g->live_ev[dir], s));
        g->live_ready[dir] = 1;
    } else {
        FOLTY_CUDA(cudaStreamWaitEvent(s, g->live_ev[dir], 0));
    }
}

// The other variants' rows have the size of the array's part in use, and the out motif's, which the listing
// wrote with room for its bound, moves into one where it takes less than half of that (6M
// edges of 2 per pair: 2.9M of 29M bytes; at 70M edges 77M of 111M stay where they are).
void listed_liveness(folty_graph* g, uint8_t* out, int64_t room, int64_t entries, cudaStream_t s) {
    const bool move = 2 * entries < room;
    uint8_t* base = liveness_rows(g, move ? 3 : 2, entries, s);
    const int64_t stride = liveness_stride(entries);
    g->tlive[FOLTY_DIR_IN] = base;
    g->tlive[FOLTY_DIR_EITHER] = base + stride;
    g->tlive[FOLTY_DIR_OUT] = move ? base + 2 * stride : out;
    if (move) {
        FOLTY_CUDA(cudaMemcpyAsync(base + 2 * stride, out, (size_t)g->tri_cap, cudaMemcpyDeviceToDevice, s));
        graph_release(g, out, s);
    }
    std::lock_guard<std::mutex> lock(g->live_mu);
    if (!g->live_ev[FOLTY_DIR_OUT]) FOLTY_CUDA(cudaEventCreateWithFlags(&g->live_ev[FOLTY_DIR_OUT], cudaEventDisableTiming));
    FOLTY_CUDA(cudaEventRecord(g->live_ev[FOLTY_DIR_OUT], s));
    g->live_ready[FOLTY_DIR_OUT] = 1;
}

// The probe kernel of the graph's tuned shape: tiles of up to PB_GROUP * items slots,
// blocks per SM as many as fit or the tuned count.
template <typename TS, int MODE, int ITEMS>
static void launch_live_shape(const folty_graph* g, int dir, const LiveArgs& la, int blocks, TS delta,
                              const TS* deltas, cudaStream_t s) {
    int per_sm = 0;
    FOLTY_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_probe_live<TS, 0, MODE, ITEMS>, PB_THREADS, 0));
    if (per_sm < 1) per_sm = 1;
    if (blocks > 0 && blocks < per_sm) per_sm = blocks;
    const unsigned grid = (unsigned)(num_sms() * per_sm);
    const TS* T = (const TS*)g->T;
    if (dir == FOLTY_DIR_OUT)
        FOLTY_LAUNCH((k_probe_live<TS, FOLTY_DIR_OUT, MODE, ITEMS>), grid, PB_THREADS, 0, s, la, T, delta, deltas);
    else if (dir == FOLTY_DIR_IN)
        FOLTY_LAUNCH((k_probe_live<TS, FOLTY_DIR_IN, MODE, ITEMS>), grid, PB_THREADS, 0, s, la, T, delta, deltas);
    else
        FOLTY_LAUNCH((k_probe_live<TS, FOLTY_DIR_EITHER, MODE, ITEMS>), grid, PB_THREADS, 0, s, la, T, delta, deltas);
}

template <typename TS, int MODE>
static void launch_live_t(const folty_graph* g, int dir, const LiveArgs& la, TS delta, const TS* deltas,
                          cudaStream_t s) {
    if (g->tune.probe_items == 4) launch_live_shape<TS, MODE, 4>(g, dir, la, g->tune.probe_blocks, delta, deltas, s);
    else launch_live_shape<TS, MODE, 8>(g, dir, la, g->tune.probe_blocks, delta, deltas, s);
}

template <typename TS>
static void launch_select_t(const folty_graph* g, int dir, const uint8_t* tl, int64_t delta, const ProbeBuffers& ls,
                            unsigned long long* prof, const int64_t* qp, cudaStream_t s) {
    const RunEnds<TS>* ends = static_cast<const RunEnds<TS>*>(g->run_ends);
    SelectCtl* ctl = reinterpret_cast<SelectCtl*>(ls.ctl);
    const SelectArgs a{g->tri,  ls.cand, delta,    qp,           ls.ush,   ctl,       ls.L,
                       ls.loff, ls.lmask, ls.ltile, ls.max_tiles, PB_GROUP, ls.totals, prof};
    FOLTY_LAUNCH(k_live_candidates<LS_ITEMS>, grid_for((g->tri_cap + LS_ITEMS - 1) / LS_ITEMS, LS_THREADS, LS_PER_SM),
                 LS_THREADS, 0, s, tl, g->tri_cap, delta, qp, ctl, ls.cand);
    const unsigned grid = grid_for(g->ntri, LS_THREADS, LS_PER_SM);
    if (dir == FOLTY_DIR_OUT) FOLTY_LAUNCH((k_live_select<TS, FOLTY_DIR_OUT>), grid, LS_THREADS, 0, s, a, ends);
    else if (dir == FOLTY_DIR_IN) FOLTY_LAUNCH((k_live_select<TS, FOLTY_DIR_IN>), grid, LS_THREADS, 0, s, a, ends);
    else FOLTY_LAUNCH((k_live_select<TS, FOLTY_DIR_EITHER>), grid, LS_THREADS, 0, s, a, ends);
}

// Buffers of one selection: from a call's scratch, or owned by the graph.
template <typename A>
static ProbeBuffers make_probe_buffers(const folty_graph* g, cudaStream_t s, A&& get) {
    const int64_t ntri = g->ntri;
    ProbeBuffers ls;
    ls.cand = get((int32_t*)nullptr, ntri);
    ls.L = get((int32_t*)nullptr, ntri + 1);
    ls.loff = get((int64_t*)nullptr, ntri + 1);
    ls.lmask = get((uint8_t*)nullptr, ntri + 1);
    ls.totals = get((int64_t*)nullptr, 2);
    // slots are reserved in units of 2^ush, so that all of them fit the packed counter (one
    // slot per unit up to 2^32 slots); a selection has at most one partial unit per step,
    // and steps hold a triangle or more
    const int64_t slots = g->info.probes + LIVE_IDLE * ntri;
    ls.ush = 0;
    while ((slots >> ls.ush) + ntri >= ((int64_t)1 << LS_UNIT_BITS)) ls.ush++;
    const int64_t padded = slots + (ls.ush > 0 ? ntri << ls.ush : 0);
    ls.max_tiles = (padded + PB_GROUP - 1) / PB_GROUP;
    ls.ltile = get((int64_t*)nullptr, ls.max_tiles + 2);
    ls.ctl = get((unsigned long long*)nullptr, 2);
    FOLTY_CUDA(cudaMemsetAsync(ls.ctl, 0, 2 * sizeof(unsigned long long), s));
    return ls;
}

ProbeBuffers probe_buffers(folty_graph* g, cudaStream_t s) {
    return make_probe_buffers(g, s, [&](auto* tag, int64_t n) {
        return graph_alloc<std::remove_pointer_t<decltype(tag)>>(g, n, s);
    });
}

unsigned long long* prof_counter(folty_graph* g, cudaStream_t s) {
    if (!profiling_on()) return nullptr;
    unsigned long long* p = g->prof_bytes + (g->prof_next++ % PROF_SLOTS);
    FOLTY_CUDA(cudaMemsetAsync(p, 0, sizeof(unsigned long long), s));
    return p;
}

// Selects the roles kept for delta (or the window in qp) into ls. prof_sel (may be null)
// receives the selection's model bytes beyond its one byte per triangle.
static void enqueue_select(folty_graph* g, int64_t delta, int dir, const ProbeBuffers& ls,
                           unsigned long long* prof_sel, const int64_t* qp, cudaStream_t s) {
    StageSpan span(ST_SELECT, s, g->tri_cap, prof_sel);
    const uint8_t* tl = g->tlive[dir];
    if (g->ts32) launch_select_t<uint32_t>(g, dir, tl, delta, ls, prof_sel, qp, s);
    else launch_select_t<int64_t>(g, dir, tl, delta, ls, prof_sel, qp, s);
}

static ProbeBuffers scratch_buffers(folty_graph* g, Scratch& sc, cudaStream_t s) {
    return make_probe_buffers(g, s, [&](auto* tag, int64_t n) { return sc.get<std::remove_pointer_t<decltype(tag)>>(n); });
}

static ProbeBuffers select_live(folty_graph* g, int64_t delta, int dir, Scratch& sc, cudaStream_t s,
                                unsigned long long* prof_sel) {
    const ProbeBuffers ls = scratch_buffers(g, sc, s);
    ensure_liveness(g, dir, s);
    enqueue_select(g, delta, dir, ls, prof_sel, nullptr, s);
    return ls;
}

template <int MODE>
static void launch_live(const folty_graph* g, int dir, const LiveArgs& la, int64_t delta, const void* deltas, cudaStream_t s) {
    const uint32_t d32 = delta >= 0xfffffffell ? 0xfffffffeu : (uint32_t)delta;
    if (g->ts32) launch_live_t<uint32_t, MODE>(g, dir, la, d32, (const uint32_t*)deltas, s);
    else launch_live_t<int64_t, MODE>(g, dir, la, delta, (const int64_t*)deltas, s);
}

static LiveArgs live_args(const folty_graph* g, const ProbeBuffers& pb) {
    LiveArgs la{};
    la.tri = g->tri;
    la.seg = g->seg;
    la.L = pb.L;
    la.loff = pb.loff;
    la.lmask = pb.lmask;
    la.ltile = pb.ltile;
    la.P = pb.totals + 1;
    return la;
}

// Kept roles for delta, then the probes.
void launch_probe_live(folty_graph* g, int64_t delta, int dir, int32_t* cnt, uint16_t* cnt16, uint8_t* rflag,
                       cudaStream_t s) {
    if (g->ntri == 0 || g->info.probes == 0) return;
    Scratch sc(g->alloc, s, g->dev_err);
    const ProbeBuffers ls = select_probes(g, delta, dir, sc, s);
    LiveArgs la = live_args(g, ls);
    la.cnt = cnt;
    la.cnt16 = (uint32_t*)cnt16;
    la.rflag = rflag;
    la.prof = prof_counter(g, s);
    StageSpan span(ST_PROBE, s, 0, la.prof);
    launch_live<PROBE_COUNT>(g, dir, la, delta, nullptr, s);
}

ProbeBuffers select_probes(folty_graph* g, int64_t delta, int dir, Scratch& sc, cudaStream_t s) {
    tune_probe(g, delta, dir, s);
    // model bytes counted on the device: the selection reads one liveness byte per
    // triangle, and per kept one its record and run ends, and writes 13 B; the probes'
    // bytes per staged triangle and kept role are summed by the probe kernel
    return select_live(g, delta, dir, sc, s, prof_counter(g, s));
}

void launch_marks(folty_graph* g, int64_t delta, int dir, const ProbeBuffers& pb, uint32_t* ebits, cudaStream_t s) {
    LiveArgs la = live_args(g, pb);
    la.bits = ebits;
    la.prof = prof_counter(g, s);
    StageSpan span(ST_PROBE, s, 0, la.prof);
    launch_live<PROBE_MARK>(g, dir, la, delta, nullptr, s);
}

void launch_bins(folty_graph* g, int64_t delta, int dir, const ProbeBuffers& pb, const uint32_t* ebits,
                 const int32_t* wpref, int32_t* bins, uint16_t* bins16, int k, int kstride, const void* deltas,
                 cudaStream_t s) {
    LiveArgs la = live_args(g, pb);
    la.cnt = bins;
    la.cnt16 = (uint32_t*)bins16;
    la.bits = const_cast<uint32_t*>(ebits);
    la.wpref = wpref;
    la.k = k;
    la.kstride = kstride;
    la.prof = prof_counter(g, s);
    StageSpan span(ST_PROBE, s, 0, la.prof);
    launch_live<PROBE_BIN>(g, dir, la, delta, deltas, s);
}

void enqueue_probe_pass(folty_graph* g, const int64_t* qp, int dir, const ProbeBuffers& pb, int32_t* cnt,
                        uint16_t* cnt16, uint32_t* touched, cudaStream_t s) {
    if (g->ntri == 0 || g->info.probes == 0) return;
    enqueue_select(g, 0, dir, pb, prof_counter(g, s), qp, s);
    LiveArgs la = live_args(g, pb);
    la.cnt = cnt;
    la.cnt16 = (uint32_t*)cnt16;
    la.bits = touched;
    la.qp = qp;
    la.prof = prof_counter(g, s);
    StageSpan span(ST_PROBE, s, 0, la.prof);
    launch_live<PROBE_COUNT>(g, dir, la, 0, nullptr, s);
}

// ------------------------------------------------------------------ autotuning

// The probe shape of g: forced, cached under the graph's statistics, or picked by timing
// each candidate (tile, blocks per SM) on the probe pass of the first query's (delta,
// dir) after one selection; the candidates give identical counts (every probe is made
// once whatever the tile), so only their times differ.
void tune_probe(folty_graph* g, int64_t delta, int dir, cudaStream_t s) {
    if (g->tune.probe_source != 0) return;
    if (tune_forced(&g->tune, true)) return;
    const std::vector<int64_t> key{g->n, g->m_kept, g->S, g->ntri, g->info.probes, g->ts32};
    if (tune_lookup(key, &g->tune, true)) return;
    if (g->ntri == 0 || g->info.probes == 0 || profiling_on()) return;  // nothing to time (or events in use)
    Scratch sc(g->alloc, s, g->dev_err);
    const int64_t mk = g->m_kept;
    const bool c16 = g->info.max_degree < 65535;
    int32_t* cnt = c16 ? nullptr : sc.get<int32_t>(mk);
    uint16_t* cnt16 = c16 ? sc.get<uint16_t>(mk + 2) : nullptr;
    const ProbeBuffers ls = scratch_buffers(g, sc, s);
    ensure_liveness(g, dir, s);
    cudaEvent_t ev[TUNE_TRIALS + 1];
    for (auto& e : ev) FOLTY_CUDA(cudaEventCreate(&e));
    float best = 0.f;
    int bi = 1;
    try {
        TuneParams t = g->tune;
        for (int c = 0; c < TUNE_TRIALS; c++) {
            g->tune.probe_items = PROBE_CAND[c][0];
            g->tune.probe_blocks = PROBE_CAND[c][1];
            // each trial selects anew (outside its timed span), in the same buffers
            enqueue_select(g, delta, dir, ls, nullptr, nullptr, s);
            if (cnt16) FOLTY_CUDA(cudaMemsetAsync(cnt16, 0, sizeof(uint16_t) * (size_t)(mk + 2), s));
            else FOLTY_CUDA(cudaMemsetAsync(cnt, 0, sizeof(int32_t) * (size_t)mk, s));
            LiveArgs la = live_args(g, ls);
            la.cnt = cnt;
            la.cnt16 = (uint32_t*)cnt16;
            FOLTY_CUDA(cudaEventRecord(ev[0], s));
            launch_live<PROBE_COUNT>(g, dir, la, delta, nullptr, s);
            FOLTY_CUDA(cudaEventRecord(ev[c + 1], s));
            FOLTY_CUDA(cudaEventSynchronize(ev[c + 1]));
            float ms = 0.f;
            FOLTY_CUDA(cudaEventElapsedTime(&ms, ev[0], ev[c + 1]));
            t.probe_ms[c] = ms;
            if (c == 0 || ms < best) {
                best = ms;
                bi = c;
            }
        }
        t.probe_items = PROBE_CAND[bi][0];
        t.probe_blocks = PROBE_CAND[bi][1];
        t.probe_source = 1;
        g->tune.probe_items = t.probe_items;
        g->tune.probe_blocks = t.probe_blocks;
        g->tune.probe_source = 1;
        std::memcpy(g->tune.probe_ms, t.probe_ms, sizeof(t.probe_ms));
        tune_store(key, g->tune, true);
    } catch (...) {
        for (auto& e : ev) cudaEventDestroy(e);
        g->tune.probe_items = 8;
        g->tune.probe_blocks = 0;
        throw;
    }
    for (auto& e : ev) cudaEventDestroy(e);
    read_back(g, nullptr, nullptr, 0, nullptr, s);  // a trial's look-back wait that ran out surfaces here
}

// ------------------------------------------------------------------ selection statistics

// Kept roles, their probes and the probe pass's model bytes over the kept triangles of a
// selection: out[0] += roles, out[1] += probes (sigma1 of the kept roles), out[2] +=
// model bytes (the same per-triangle and per-role figures the probe kernel counts).
template <typename TS, int DIR>
__global__ void k_live_stats(const int4* __restrict__ tri, const int32_t* __restrict__ seg,
                             const int32_t* __restrict__ L, const uint8_t* __restrict__ lmask,
                             const int64_t* __restrict__ totals, unsigned long long* __restrict__ out) {
    const int64_t nl = totals[0];
    unsigned long long roles = 0, probes = 0, bytes = 0;
    for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < nl; j += (int64_t)gridDim.x * blockDim.x) {
        const int4 tr = tri[L[j]];
        const int m = lmask[j];
        const int32_t se[3] = {tr.x, tr.y, tr.z};
        int32_t off[9];
#pragma unroll
        for (int e = 0; e < 3; e++) {
            off[3 * e] = seg[2 * se[e]];
            off[3 * e + 1] = seg[2 * se[e] + 1];
            off[3 * e + 2] = seg[2 * se[e] + 2];
        }
        roles += (unsigned long long)__popc(m);
        for (int r = 0; r < 6; r++)
            if ((m >> r) & 1) probes += (unsigned long long)(off[3 * (r >> 1) + (r & 1) + 1] - off[3 * (r >> 1) + (r & 1)]);
        bytes += kept_role_bytes<TS, DIR>(off, m, role_descriptor(tr.w, DIR));
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        roles += __shfl_xor_sync(0xffffffffu, roles, o);
        probes += __shfl_xor_sync(0xffffffffu, probes, o);
        bytes += __shfl_xor_sync(0xffffffffu, bytes, o);
    }
    if ((threadIdx.x & 31) == 0 && roles) {
        atomicAdd(&out[0], roles);
        atomicAdd(&out[1], probes);
        atomicAdd(&out[2], bytes);
    }
}

template <typename TS>
static void live_stats_t(const folty_graph* g, int dir, const ProbeBuffers& ls, unsigned long long* acc,
                         cudaStream_t s) {
    const unsigned grid = grid_for(g->ntri, 256);
    if (dir == FOLTY_DIR_OUT)
        FOLTY_LAUNCH((k_live_stats<TS, FOLTY_DIR_OUT>), grid, 256, 0, s, g->tri, g->seg, ls.L, ls.lmask, ls.totals, acc);
    else if (dir == FOLTY_DIR_IN)
        FOLTY_LAUNCH((k_live_stats<TS, FOLTY_DIR_IN>), grid, 256, 0, s, g->tri, g->seg, ls.L, ls.lmask, ls.totals, acc);
    else
        FOLTY_LAUNCH((k_live_stats<TS, FOLTY_DIR_EITHER>), grid, 256, 0, s, g->tri, g->seg, ls.L, ls.lmask, ls.totals,
                     acc);
}

void probe_stats(folty_graph* g, int64_t delta, int dir, folty_probe_stats* out, cudaStream_t s) {
    std::memset(out, 0, sizeof(*out));
    out->triangles = g->ntri;
    out->all_roles = 6 * g->ntri;
    out->all_probes = g->info.probes;  // every (temporal edge, witness) pair
    out->select_bytes = g->tri_cap;
    if (g->ntri == 0 || g->info.probes == 0) return;
    Scratch sc(g->alloc, s, g->dev_err);
    const ProbeBuffers ls = select_live(g, delta, dir, sc, s, nullptr);
    unsigned long long* acc = sc.get<unsigned long long>(3);
    FOLTY_CUDA(cudaMemsetAsync(acc, 0, 3 * sizeof(unsigned long long), s));
    if (g->ts32) live_stats_t<uint32_t>(g, dir, ls, acc, s);
    else live_stats_t<int64_t>(g, dir, ls, acc, s);
    const void* ptrs[4] = {ls.totals, acc, acc + 1, acc + 2};
    int sizes[4] = {8, 8, 8, 8};
    int64_t v[4];
    read_back(g, ptrs, sizes, 4, v, s);
    out->kept_triangles = v[0];
    out->kept_roles = v[1];
    out->kept_probes = v[2];
    out->probe_bytes = v[3];
    out->select_bytes += (int64_t)(16 + 3 * (g->ts32 ? sizeof(RunEnds<uint32_t>) : sizeof(RunEnds<int64_t>)) + 13 + 8) * v[0];
}

}  // namespace folty

// Preprocessing of a loaded temporal graph (paper Section 2, Preliminaries, and the
// first steps of Algorithm 6):
//   A1  drop self-loops; sort temporal edges by (static pair, direction, t) so that
//       every E_{x,y} is a contiguous ascending run of the timestamp store T;
//   A2  static graph G_S as CSR, neighbours ascending, with static-edge ids;
//   A3  core numbers and a degeneracy order (core.cu);
//   A4  orientation G->pi: u -> v iff (round(u), u) < (round(v), v); out-degree <= alpha;
//   A5  every triangle of G_S exactly once: (u, v) in G->, w in N+(u) cap N+(v)
//       (Algorithm 3's enumeration skeleton), with its per-triangle probe count.
#include <algorithm>
#include <climits>
#include <cstdlib>
#include <cstring>
#include <optional>

#include "core.cuh"
#include "internal.cuh"
#include "liveness.cuh"
#include "pairs.cuh"
#include "probe.cuh"

namespace folty {

// ================================================================== A1

// Sort key of a temporal edge: 2 p(a, b) + dir with a = min, b = max id, dir = (src > dst)
// and p(a, b) = a (2n - a - 1) / 2 + (b - a - 1) the rank of the pair among all pairs
// a < b in (a, b) order, so keys order edges by (a, b, dir) within n (n - 1) values (one
// bit narrower than packing a and b side by side: 40 bits for a million vertices).
// Self-loops get the all-ones key of the used width and sort last.
__global__ void k_build_keys(const int32_t* __restrict__ src, const int32_t* __restrict__ dst,
                             int64_t m, int32_t n, uint64_t loop_key, uint64_t* __restrict__ key,
                             uint32_t* __restrict__ val) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < m;
         i += (int64_t)gridDim.x * blockDim.x) {
        int32_t x = src[i], y = dst[i];
        uint64_t k;
        if (x == y) {
            k = loop_key;
        } else {
            const uint64_t a = (uint64_t)min(x, y), b = (uint64_t)max(x, y);
            const uint64_t p = a * (2 * (uint64_t)n - a - 1) / 2 + (b - a - 1);
            k = 2 * p + (uint64_t)(x > y);
        }
        key[i] = k;
        val[i] = (uint32_t)i;
    }
}

// The times as sort keys t - tmin (t32: modulo 2^32).
__global__ void k_time_keys(const uint32_t* __restrict__ t32, const int64_t* __restrict__ t, int64_t m, int64_t tmin,
                            uint64_t* __restrict__ key, uint32_t* __restrict__ val) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < m;
         i += (int64_t)gridDim.x * blockDim.x) {
        key[i] = t32 ? (uint64_t)(t32[i] - (uint32_t)tmin) : (uint64_t)(t[i] - tmin);
        val[i] = (uint32_t)i;
    }
}

__global__ void k_gather_keys(const uint64_t* __restrict__ key_in, const uint32_t* __restrict__ order,
                              int64_t m, uint64_t* __restrict__ key_out) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < m;
         i += (int64_t)gridDim.x * blockDim.x)
        key_out[i] = key_in[order[i]];
}

// perm, T (gathered from t: 32-bit offsets from tbase, or the raw int64 timestamps), and
// the "new static pair" flag of every kept sorted position.
template <typename TS>
__global__ void k_store(const uint64_t* __restrict__ key, const uint32_t* __restrict__ order,
                        const TS* __restrict__ t, TS tbase, int64_t mk, int32_t* __restrict__ perm,
                        TS* __restrict__ T, int32_t* __restrict__ newpair) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < mk;
         i += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t o = __ldcs(order + i);
        __stcs(perm + i, (int32_t)o);
        T[i] = t[o] - tbase;
        const uint64_t k = __ldcs(key + i);
        __stcs(newpair + i, (int32_t)((i == 0) || ((k >> 1) != (key[i - 1] >> 1))));
    }
}

// Static edge ids and segment starts. pscan = exclusive scan of newpair.
__global__ void k_segments(const uint64_t* __restrict__ key, const int32_t* __restrict__ newpair,
                           const int32_t* __restrict__ pscan, int64_t mk, int32_t* __restrict__ sd,
                           int32_t* __restrict__ seg) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < mk;
         i += (int64_t)gridDim.x * blockDim.x) {
        uint64_t k = key[i];
        int32_t s = pscan[i] + newpair[i] - 1;
        int dir = (int)(k & 1);
        sd[i] = 2 * s + dir;
        if (newpair[i]) {
            seg[2 * s] = (int32_t)i;
            seg[2 * s + 1] = -1;
        }
    }
}

// Pairs a < b with first element below x: x (2n - x - 1) / 2.
__device__ __forceinline__ uint64_t pairs_before(int64_t x, int32_t n) {
    return (uint64_t)x * (uint64_t)(2 * (int64_t)n - x - 1) / 2;
}

// The pair (a, b) of rank p (inverse of the key of k_build_keys): a is the largest x with
// pairs_before(x) <= p, first estimated from the smaller root of x^2 - (2n - 1) x + 2p = 0
// (the discriminant (2n - 1)^2 - 8p is exact in 64 bits for n < 2^31; its square root is
// taken in single precision, a few units off at most for ids below 2^24), then corrected
// by exact integer comparisons.
__device__ __forceinline__ void pair_of_rank(uint64_t p, int32_t n, int32_t& a, int32_t& b) {
    const uint64_t c = 2 * (uint64_t)n - 1;
    const uint64_t disc = c * c - 8 * p;
    int64_t x = (int64_t)(((float)c - sqrtf((float)disc)) * 0.5f);
    x = x < 0 ? 0 : (x > n - 2 ? n - 2 : x);
    while (x > 0 && pairs_before(x, n) > p) x--;
    while (x + 1 <= n - 2 && pairs_before(x + 1, n) <= p) x++;
    a = (int32_t)x;
    b = (int32_t)(p - pairs_before(x, n) + (uint64_t)x + 1);
}

// Endpoints of static edge s from the key of its first temporal edge (one thread per
// static edge, so that no warp idles through the decoding).
__global__ void k_pair_ends(const uint64_t* __restrict__ key, const int32_t* __restrict__ seg, int32_t S,
                            int32_t n, int32_t* __restrict__ ea, int32_t* __restrict__ eb) {
    for (int32_t s = blockIdx.x * blockDim.x + threadIdx.x; s < S; s += gridDim.x * blockDim.x) {
        int32_t x, y;
        pair_of_rank(key[seg[2 * s]] >> 1, n, x, y);
        ea[s] = x;
        eb[s] = y;
    }
}

// ---------------------------------------------------------------- dense pair ids
//
// When the distinct pairs are few enough, the edges are sorted by (pair id, direction)
// with pair ids numbered 0..S-1 in (a, b) order, instead of by the full pair key: the id
// and the direction bit need about log2(2S) bits, which leaves room for the edge's
// time rank in the same 64-bit word. The sort is then keys only and takes 3 digit
// passes on the medium graph instead of 5 passes with values. The distinct pairs come
// from an open-addressed table (linear probing from a multiplicative hash of the pair
// rank); they are sorted on their own (S entries), and each edge looks its id up by the
// table slot it kept from the insert.

constexpr int PAIR_COMPACT_ITEMS = 16;            // table slots per thread and step of the compaction

// Every non-loop edge's pair goes into the table (value rank + 1, 0 = empty), and edge i
// keeps its slot and direction in slotw[i] (PAIR_LOOP for a self-loop). A probe sequence
// that runs out, or too many distinct pairs, abandon the table, and the insert stops.
__global__ void k_pair_insert(const int32_t* __restrict__ src, const int32_t* __restrict__ dst, int64_t m, int32_t n,
                              uint64_t* __restrict__ table, int lg, uint32_t* __restrict__ slotw,
                              int* flags) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < m; i += (int64_t)gridDim.x * blockDim.x) {
        const int32_t x = src[i], y = dst[i];
        if (pair_table_over(flags)) return;
        __stcs(slotw + i, pair_slot_word(table, lg, x, y, n, flags));
    }
}

// The occupied slots as (rank, slot) lists, in no particular order: each block takes
// PAIR_COMPACT_ITEMS * blockDim.x slots per step and reserves their entries with one
// global atomic. *cnt ends at the number of distinct pairs; entries past cap are not
// written (the caller then abandons the table).
__global__ void k_pair_table_compact(const uint64_t* __restrict__ table, int64_t tb, uint64_t* __restrict__ urank,
                               uint32_t* __restrict__ uslot, int* __restrict__ cnt, int cap) {
    __shared__ int wsum[32], base;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const int64_t step = (int64_t)PAIR_COMPACT_ITEMS * blockDim.x;
    for (int64_t s0 = blockIdx.x * step; s0 < tb; s0 += gridDim.x * step) {
        uint64_t v[PAIR_COMPACT_ITEMS];
        int c = 0;
#pragma unroll
        for (int q = 0; q < PAIR_COMPACT_ITEMS; q++) {
            const int64_t sl = s0 + (int64_t)q * blockDim.x + threadIdx.x;
            v[q] = sl < tb ? table[sl] : 0;
            c += v[q] != 0;
        }
        int inc = c;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc += y;
        }
        if (lane == 31) wsum[warp] = inc;
        __syncthreads();
        if (threadIdx.x == 0) {
            int t = 0;
            for (int w = 0; w < nw; w++) {
                const int x = wsum[w];
                wsum[w] = t;
                t += x;
            }
            base = t ? atomicAdd(cnt, t) : 0;
        }
        __syncthreads();
        int at = base + wsum[warp] + inc - c;
#pragma unroll
        for (int q = 0; q < PAIR_COMPACT_ITEMS; q++) {
            if (v[q] != 0) {
                if (at < cap) {
                    urank[at] = v[q] - 1;
                    uslot[at] = (uint32_t)(s0 + (int64_t)q * blockDim.x + threadIdx.x);
                }
                at++;
            }
        }
        __syncthreads();  // wsum and base are rewritten by the next step
    }
}

// Pair id j (position in rank order) of every table slot in use, and the pair's ends.
// The ranks come from a sort whose look-back could in principle run out (the graph's
// error word, checked by the host before the ids are used, then says so): slots and ends
// are kept inside their arrays whatever the input.
__global__ void k_pair_ids(const uint64_t* __restrict__ urank, const uint32_t* __restrict__ uslot, int32_t S,
                           int32_t n, int64_t tb, int32_t* __restrict__ sid, int32_t* __restrict__ ea,
                           int32_t* __restrict__ eb) {
    for (int32_t j = blockIdx.x * blockDim.x + threadIdx.x; j < S; j += gridDim.x * blockDim.x) {
        const uint32_t sl = uslot[j];
        if (sl < tb) sid[sl] = j;
        int32_t x, y;
        pair_of_rank(urank[j], n, x, y);
        ea[j] = min(x, n - 1);
        eb[j] = min(y, n - 1);
    }
}

// Sort word of the edge at time rank j (input index o = order[j], or j when the input is
// in time order): (2 pair id + direction) << ib | j; self-loops get 2S and sort last.
// With tv (32-bit stores), also the edge's 32-bit time offset t[o] - tmin, the value the
// sort carries along, so that the sorted timestamps need no gather; and sigma[p] counts
// the temporal edges of pair p, which the triangle passes need before the sort is done.
__global__ void k_pair_pack(const uint32_t* __restrict__ slotw, const uint32_t* __restrict__ order, int64_t m,
                            const int32_t* __restrict__ sid, int32_t S, int ib, uint64_t* __restrict__ packed,
                            const uint32_t* __restrict__ t, uint32_t tmin, uint32_t* __restrict__ tv,
                            int32_t* __restrict__ sigma) {
    for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < m; j += (int64_t)gridDim.x * blockDim.x) {
        const int64_t o = order ? (int64_t)order[j] : j;
        const uint32_t w = order ? slotw[o] : __ldcs(slotw + j);
        uint64_t c = 2 * (uint64_t)S;
        if (w != PAIR_LOOP) {
            const int32_t p = sid[w & ~PAIR_DIR];
            c = 2 * (uint64_t)p + (w >> 31);
            if ((unsigned)p < (unsigned)S) atomicAdd(&sigma[p], 1);
        }
        packed[j] = (c << ib) | (uint64_t)j;
        if (tv) tv[j] = (order ? t[o] : __ldcs(t + j)) - tmin;
    }
}

// The first step of the store of a time-ordered input with 32-bit time offsets: each
// edge's sort id c = 2 pair id + direction (2S for a self-loop) into cw, and the number
// of edges of every id into cnt[0..2S] (zeroed; of consecutive edges of one id a thread
// sees, only the first adds, by their number; the self-loops are summed per warp first).
// Eight edges per thread (their id lookups in flight together), 16-byte loads and stores.
constexpr int STORE_IDS_EDGES = 8;  // consecutive edges per thread of k_store_ids
__global__ void __launch_bounds__(256) k_store_ids(const uint32_t* __restrict__ slotw, int64_t m,
                                                   const int32_t* __restrict__ sid, int32_t S,
                                                   uint32_t* __restrict__ cw, int32_t* __restrict__ cnt) {
    constexpr int E = STORE_IDS_EDGES;
    const int64_t nq = (m + E - 1) / E;
    for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < nq; q += (int64_t)gridDim.x * blockDim.x) {
        const int64_t j0 = q * E;
        const bool full = j0 + E <= m;
        uint32_t w[E];
        if (full) {
#pragma unroll
            for (int h = 0; h < E / 4; h++) {
                const uint4 ww = __ldcs(reinterpret_cast<const uint4*>(slotw + j0) + h);
                w[4 * h] = ww.x;
                w[4 * h + 1] = ww.y;
                w[4 * h + 2] = ww.z;
                w[4 * h + 3] = ww.w;
            }
        } else {
#pragma unroll
            for (int e = 0; e < E; e++) w[e] = j0 + e < m ? slotw[j0 + e] : PAIR_LOOP;
        }
        // all the id lookups in flight before any is used
        int32_t p[E];
#pragma unroll
        for (int e = 0; e < E; e++) p[e] = w[e] != PAIR_LOOP ? sid[w[e] & ~PAIR_DIR] : -1;
        uint32_t c[E];
#pragma unroll
        for (int e = 0; e < E; e++)
            c[e] = (unsigned)p[e] < (unsigned)S ? 2 * (uint32_t)p[e] + (w[e] >> 31) : 2 * (uint32_t)S;
        int loops = 0;
#pragma unroll
        for (int e = 0; e < E; e++) {
            if (c[e] >= 2 * (uint32_t)S) {
                loops += j0 + e < m;
                continue;
            }
            if (e > 0 && c[e - 1] == c[e]) continue;
            int run = 1;
#pragma unroll
            for (int f = e + 1; f < E; f++)
                if (f == e + run && c[f] == c[e]) run++;
            atomicAdd(&cnt[c[e]], run);
        }
        const unsigned am = __activemask();
        loops = __reduce_add_sync(am, loops);
        if (loops && (threadIdx.x & 31) == __ffs(am) - 1) atomicAdd(&cnt[2 * (int64_t)S], loops);
        if (full) {
#pragma unroll
            for (int h = 0; h < E / 4; h++)
                __stcs(reinterpret_cast<uint4*>(cw + j0) + h, make_uint4(c[4 * h], c[4 * h + 1], c[4 * h + 2], c[4 * h + 3]));
        } else {
            for (int e = 0; e < E && j0 + e < m; e++) cw[j0 + e] = c[e];
        }
    }
}

// hist[p][b] (zeroed) = number of edges whose sort id has 8-bit digit p equal to b, for
// the sort's passes digits: from the per-id counts cnt[0..2S], one weighted addition per
// id rather than one per edge.
__global__ void __launch_bounds__(256) k_store_hist(const int32_t* __restrict__ cnt, int32_t S, int passes,
                                                    uint32_t* __restrict__ hist) {
    constexpr int B = 1 << STORE_DIGIT_BITS;
    __shared__ uint32_t h[STORE_MAX_PASSES][B];
    for (int i = threadIdx.x; i < STORE_MAX_PASSES * B; i += blockDim.x) (&h[0][0])[i] = 0;
    __syncthreads();
    const int64_t nc = 2 * (int64_t)S + 1;
    for (int64_t c = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; c < nc; c += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t v = (uint32_t)cnt[c];
        if (v == 0) continue;
        for (int p = 0; p < passes; p++) atomicAdd(&h[p][((uint32_t)c >> (STORE_DIGIT_BITS * p)) & (B - 1)], v);
    }
    __syncthreads();
    for (int i = threadIdx.x; i < passes * B; i += blockDim.x) {
        const uint32_t v = (&h[0][0])[i];
        if (v) atomicAdd(&hist[i], v);
    }
}

// sigma[p] = number of temporal edges of static edge p, from the runs' starts.
__global__ void k_store_sigma(const int32_t* __restrict__ seg, int32_t S, int32_t* __restrict__ sigma) {
    for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < S; p += (int64_t)gridDim.x * blockDim.x)
        sigma[p] = seg[2 * p + 2] - seg[2 * p];
}

// The run starts of sorted position i with word pk (its predecessor's word prev, ~0 for
// i = 0): seg[2s] = i where static edge s begins, seg[2s + 1] = i where its b -> a run
// begins (seg is all -1 before; k_segments_fix fills the b -> a starts of edges without
// one). c < 2S unless the pair ids' sort failed, which the host learns right after.
__device__ __forceinline__ void pair_run_starts(uint64_t pk, uint64_t prev, int ib, int32_t S, int64_t i,
                                                int32_t* __restrict__ seg) {
    const int32_t c = (int32_t)(pk >> ib);
    if ((unsigned)c >= (unsigned)(2 * S)) return;
    if ((prev >> (ib + 1)) != (uint64_t)(c >> 1)) seg[c & ~1] = (int32_t)i;
    if ((c & 1) && (prev >> ib) != (uint64_t)c) seg[c] = (int32_t)i;
}

// perm, T, sd and the run starts from the sorted words: position i holds time rank
// j = word mod 2^ib (input index order[j], or j) of pair id and direction word >> ib. T is
// gathered from the timestamps in input order (64-bit stores).
template <typename TS>
__global__ void k_pair_store(const uint64_t* __restrict__ packed, const uint32_t* __restrict__ order, int64_t mk,
                             int32_t S, int ib, const TS* __restrict__ t, int32_t* __restrict__ perm,
                             TS* __restrict__ T, int32_t* __restrict__ sd, int32_t* __restrict__ seg) {
    const uint64_t jm = (1ull << ib) - 1;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < mk; i += (int64_t)gridDim.x * blockDim.x) {
        const uint64_t pk = __ldcs(packed + i);
        const int64_t j = (int64_t)(pk & jm);
        const uint32_t o = order ? order[j] : (uint32_t)j;
        __stcs(perm + i, (int32_t)o);
        T[i] = t[o];
        __stcs(sd + i, (int32_t)(pk >> ib));
        pair_run_starts(pk, i > 0 ? packed[i - 1] : ~0ull, ib, S, i, seg);
    }
}

// The same for a 32-bit store whose timestamps came sorted with the words, four
// positions per thread with 16-byte loads and stores (the last quad may be partial).
__global__ void k_pair_store4(const uint64_t* __restrict__ packed, const uint32_t* __restrict__ order, int64_t mk,
                              int32_t S, int ib, const uint32_t* __restrict__ ts, int32_t* __restrict__ perm,
                              uint32_t* __restrict__ T, int32_t* __restrict__ sd, int32_t* __restrict__ seg) {
    const uint64_t jm = (1ull << ib) - 1;
    const int64_t nq = (mk + 3) >> 2;
    for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < nq; q += (int64_t)gridDim.x * blockDim.x) {
        const int64_t i0 = q << 2;
        const bool full = i0 + 4 <= mk;
        uint64_t pk[4];
        uint32_t tv[4];
        if (full) {
            const ulonglong2 a = __ldcs(reinterpret_cast<const ulonglong2*>(packed + i0));
            const ulonglong2 b = __ldcs(reinterpret_cast<const ulonglong2*>(packed + i0 + 2));
            const uint4 tt = __ldcs(reinterpret_cast<const uint4*>(ts + i0));
            pk[0] = a.x;
            pk[1] = a.y;
            pk[2] = b.x;
            pk[3] = b.y;
            tv[0] = tt.x;
            tv[1] = tt.y;
            tv[2] = tt.z;
            tv[3] = tt.w;
        } else {
#pragma unroll
            for (int e = 0; e < 4; e++) {
                pk[e] = i0 + e < mk ? packed[i0 + e] : 0;
                tv[e] = i0 + e < mk ? ts[i0 + e] : 0;
            }
        }
        int32_t o[4], c[4];
#pragma unroll
        for (int e = 0; e < 4; e++) {
            const int64_t j = (int64_t)(pk[e] & jm);
            o[e] = order ? (int32_t)order[j] : (int32_t)j;
            c[e] = (int32_t)(pk[e] >> ib);
        }
        uint64_t prev = i0 > 0 ? packed[i0 - 1] : ~0ull;
#pragma unroll
        for (int e = 0; e < 4; e++) {
            if (i0 + e < mk) pair_run_starts(pk[e], prev, ib, S, i0 + e, seg);
            prev = pk[e];
        }
        if (full) {
            __stcs(reinterpret_cast<int4*>(perm + i0), make_int4(o[0], o[1], o[2], o[3]));
            __stcs(reinterpret_cast<uint4*>(T + i0), make_uint4(tv[0], tv[1], tv[2], tv[3]));
            __stcs(reinterpret_cast<int4*>(sd + i0), make_int4(c[0], c[1], c[2], c[3]));
        } else {
#pragma unroll
            for (int e = 0; e < 4; e++) {
                if (i0 + e < mk) {
                    perm[i0 + e] = o[e];
                    T[i0 + e] = tv[e];
                    sd[i0 + e] = c[e];
                }
            }
        }
    }
}

// seg[2s+1] = first b->a position of s (the full-key path, whose k_segments marks every
// b->a start -1 first).
__global__ void k_segments_split(const int32_t* __restrict__ sd, int64_t mk, int32_t S,
                                 int32_t* __restrict__ seg) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < mk;
         i += (int64_t)gridDim.x * blockDim.x) {
        int32_t c = sd[i];
        if ((c & 1) && (unsigned)c < (unsigned)(2 * S) && (i == 0 || sd[i - 1] != c)) seg[c] = (int32_t)i;  // c = 2s+1
    }
}

// seg[2s+1] = the end of s when it has no b->a run.
__global__ void k_segments_fix(int32_t S, int64_t mk, int32_t* __restrict__ seg) {
    for (int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; s < S;
         s += (int64_t)gridDim.x * blockDim.x) {
        if (seg[2 * s + 1] < 0) seg[2 * s + 1] = (s + 1 < S) ? seg[2 * s + 2] : (int32_t)mk;
        if (s == 0) seg[2 * S] = (int32_t)mk;
    }
}

// ================================================================== A2

// Runs of equal values in a sorted id array: first[x] = start index, last[x] = end
// index (exclusive) of the run of x. Ids absent from the array keep first = last = 0.
__global__ void k_runs(const int32_t* __restrict__ ids, const uint32_t* __restrict__ order, int32_t S,
                       int32_t* __restrict__ first, int32_t* __restrict__ last) {
    for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < S;
         j += (int64_t)gridDim.x * blockDim.x) {
        int32_t x = order ? ids[order[j]] : ids[j];
        if (j == 0 || (order ? ids[order[j - 1]] : ids[j - 1]) != x) first[x] = (int32_t)j;
        if (j == S - 1 || (order ? ids[order[j + 1]] : ids[j + 1]) != x) last[x] = (int32_t)j + 1;
    }
}

// deg_hi = #static edges (u, b > u), deg_lo = #static edges (a < u, u), deg = sum.
__global__ void k_degrees(const int32_t* __restrict__ hi_first, const int32_t* __restrict__ hi_last,
                          const int32_t* __restrict__ lo_first, const int32_t* __restrict__ lo_last, int64_t n,
                          int32_t* __restrict__ deg_lo, int32_t* __restrict__ deg) {
    for (int64_t u = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; u < n;
         u += (int64_t)gridDim.x * blockDim.x) {
        int32_t dl = lo_last[u] - lo_first[u];
        deg_lo[u] = dl;
        deg[u] = dl + (hi_last[u] - hi_first[u]);
    }
}

__global__ void k_edge_keys_b(const int32_t* __restrict__ eb, int32_t S, uint64_t* __restrict__ key,
                              uint32_t* __restrict__ val) {
    for (int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; s < S;
         s += (int64_t)gridDim.x * blockDim.x) {
        key[s] = (uint64_t)eb[s];
        val[s] = (uint32_t)s;
    }
}

// Row u = [neighbours a < u (edges with b = u, ascending a)] [neighbours b > u].
__global__ void k_fill_adj(const int32_t* __restrict__ ea, const int32_t* __restrict__ eb, int32_t S,
                           const int32_t* __restrict__ rowptr, const int32_t* __restrict__ deg_lo,
                           const int32_t* __restrict__ hi_start, const int32_t* __restrict__ lo_start,
                           const uint32_t* __restrict__ by_b, int32_t* __restrict__ adj,
                           int32_t* __restrict__ adj_eid, int32_t* __restrict__ adj_src,
                           int32_t* __restrict__ binv) {
    for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < S;
         j += (int64_t)gridDim.x * blockDim.x) {
        // upper part: static edges are sorted by (a, b)
        int32_t s = (int32_t)j;
        int32_t a = ea[s];
        int64_t p = (int64_t)rowptr[a] + deg_lo[a] + (s - hi_start[a]);
        adj[p] = eb[s];
        adj_eid[p] = s;
        adj_src[p] = a;
        // lower part: by_b lists static edges by (b, a)
        int32_t s2 = (int32_t)by_b[j];
        binv[s2] = (int32_t)j;
        int32_t b = eb[s2];
        int64_t q = (int64_t)rowptr[b] + ((int32_t)j - lo_start[b]);
        adj[q] = ea[s2];
        adj_eid[q] = s2;
        adj_src[q] = b;
    }
}

__global__ void k_max_i32(const int32_t* __restrict__ a, int64_t n, int* __restrict__ out) {
    int best = 0;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x)
        best = max(best, a[i]);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) best = max(best, __shfl_xor_sync(0xffffffffu, best, o));
    if ((threadIdx.x & 31) == 0) atomicMax(out, best);
}

// osig[j] = temporal edges (both directions) of the static edge at out-list position j,
// and their maximum: the probe slots a triangle adds per edge, read by the triangle
// passes next to the out-list entries themselves. From the per-pair counts sigma when
// given, else from the run bounds.
__global__ void k_out_sigma(const int32_t* __restrict__ sigma, const int32_t* __restrict__ seg,
                            const int32_t* __restrict__ out_eid, int32_t S, int32_t* __restrict__ osig,
                            int* __restrict__ out) {
    int best = 0;
    for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < S;
         j += (int64_t)gridDim.x * blockDim.x) {
        const int32_t e = out_eid[j];
        const int32_t c = sigma ? sigma[e] : seg[2 * e + 2] - seg[2 * e];
        osig[j] = c;
        best = max(best, c);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) best = max(best, __shfl_xor_sync(0xffffffffu, best, o));
    if ((threadIdx.x & 31) == 0) atomicMax(out, best);
}

// ================================================================== A4

__device__ __forceinline__ bool rank_less(int32_t u, int32_t v, const int32_t* __restrict__ rnd) {
    int32_t ru = rnd[u], rv = rnd[v];
    return ru < rv || (ru == rv && u < v);
}

// Entry j of the adjacency (owner u, neighbour v) is kept as u -> v when v comes later
// in the degeneracy order.
__global__ void k_orient_flags(const int32_t* __restrict__ adj_src, const int32_t* __restrict__ adj,
                               const int32_t* __restrict__ rnd, int64_t n2, int32_t* __restrict__ flag) {
    for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < n2;
         j += (int64_t)gridDim.x * blockDim.x)
        flag[j] = rank_less(adj_src[j], adj[j], rnd);
}

// Kept entries at their scanned positions: rows stay in ascending neighbour order.
__global__ void k_orient_fill(const int32_t* __restrict__ adj_src, const int32_t* __restrict__ adj,
                              const int32_t* __restrict__ adj_eid, const int32_t* __restrict__ flag,
                              const int32_t* __restrict__ opos, int64_t n2, int32_t* __restrict__ out_nbr,
                              int32_t* __restrict__ out_eid, int32_t* __restrict__ out_src) {
    for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < n2;
         j += (int64_t)gridDim.x * blockDim.x) {
        if (!flag[j]) continue;
        int32_t p = opos[j];
        out_nbr[p] = adj[j];
        out_eid[p] = adj_eid[j];
        out_src[p] = adj_src[j];
    }
}

// outptr[u] = opos[rowptr[u]]; also the maximum out-degree.
__global__ void k_outptr(const int32_t* __restrict__ rowptr, const int32_t* __restrict__ opos, int64_t n,
                         int32_t* __restrict__ outptr, int* __restrict__ max_out) {
    int best = 0;
    for (int64_t u = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; u <= n;
         u += (int64_t)gridDim.x * blockDim.x) {
        int32_t o = opos[rowptr[u]];
        outptr[u] = o;
        if (u < n) best = max(best, opos[rowptr[u + 1]] - o);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) best = max(best, __shfl_xor_sync(0xffffffffu, best, o));
    if ((threadIdx.x & 31) == 0) atomicMax(max_out, best);
}

// ================================================================== A5

// Thread per oriented edge (u, v): merge N+(u) and N+(v) (both ascending by id).
// Triangles of oriented edge u -> v: the common out-neighbours w of u and v (both lists
// sorted). A light edge is merged by one thread; a heavy edge (|out(u)| + |out(v)| >
// heavy_min, the degeneracy core) is intersected by the whole warp: out(u) goes into an
// open-addressed hash table in the warp's shared memory, with each entry's edge id and
// temporal edge count (built once for the consecutive edges of u the warp meets), and the
// lanes look up their share of out(v), the loads of the next share issued before the
// lookups. Both passes find the same set, so the counts match the writes.
constexpr int TRI_THREADS = 256;
constexpr int TRI_HCAP = 256;    // out(u) entries a warp's table holds (longer lists: one lane merges)
constexpr int TRI_HSLOTS = 512;  // table slots (load at most one half)
constexpr int TRI_BUCKETS = 128; // of four slots, of the one-pass listing (load at most one half)
constexpr int TRI_LIST_THREADS = 128;
constexpr int TRI_PER_SM = 8;    // resident blocks (what their tables leave room for)
// entries of a warp's chunk of the one-pass listing's array: fewer when the bound is small,
// so that the empty ends of the chunks stay below a sixteenth of the bound or 32 a warp
constexpr int TRI_CHUNK_MIN = 32, TRI_CHUNK_MAX = 512;
// the largest array of a one-pass listing; a larger bound takes the counting pass
constexpr int64_t TRI_BOUND_MAX_BYTES = int64_t(16) << 30;

// FOLTY_TRI_LAYOUT=counted: every graph takes the counting pass before the listing.
inline bool tri_layout_counted() {
    const char* env = std::getenv("FOLTY_TRI_LAYOUT");
    return env && std::strcmp(env, "counted") == 0;
}

// One warp's hash table of out(u): neighbour id per slot (-1: empty) and its position in
// out(u); by position, the static edge id and temporal edge count of (u, w).
struct TriHashW {
    int32_t key[TRI_HSLOTS];
    int16_t pos[TRI_HSLOTS];
    int32_t sig[TRI_HCAP];
    int32_t eid[TRI_HCAP];
};

__device__ __forceinline__ uint32_t tri_hash(int32_t w) { return ((uint32_t)w * 0x9E3779B1u) >> 23; }

// Builds the warp's table of out(u) = [i1, e1) (e1 - i1 <= TRI_HCAP). The whole warp
// must call it. With at most TRI_HCAP keys in TRI_HSLOTS slots every probe sequence ends.
template <bool EID>
__device__ __forceinline__ void warp_hash_out(const int32_t* __restrict__ nbr, const int32_t* __restrict__ osig,
                                              const int32_t* __restrict__ eid, int32_t i1, int32_t e1,
                                              TriHashW& H) {
    const int lane = threadIdx.x & 31;
    __syncwarp();  // the previous table's lookups are done
    for (int t = lane; t < TRI_HSLOTS; t += 32) H.key[t] = -1;
    __syncwarp();
    for (int t = lane; t < e1 - i1; t += 32) {
        const int32_t w = nbr[i1 + t];
        H.sig[t] = osig[i1 + t];
        if (EID) H.eid[t] = eid[i1 + t];
        uint32_t h = tri_hash(w);
        for (int p = 0; p < TRI_HSLOTS; p++) {
            if (atomicCAS(&H.key[h], -1, w) == -1) {
                H.pos[h] = (int16_t)t;
                break;
            }
            h = (h + 1) & (TRI_HSLOTS - 1);
        }
    }
    __syncwarp();
}

// Looks up out(v) = [i2, e2) of the out-lists (nbr, osig and, when EID, eid by position)
// in the warp's table of out(u). Calls hit(pos_u, w, sig_v, eid_v) once per lane and step
// (w = -1 for an idle lane): the position in out(u) of a common neighbour w (-1: none), and the
// count and (EID) id of the static edge (v, w). The whole warp must call it.
template <bool EID, typename F>
__device__ __forceinline__ void warp_probe_out(const int32_t* __restrict__ nbr, const int32_t* __restrict__ osig,
                                               const int32_t* __restrict__ eid, int32_t i2, int32_t e2,
                                               const TriHashW& H, F&& hit) {
    const int lane = threadIdx.x & 31;
    int32_t w = -1, sv = 0, ev = 0;
    if (i2 + lane < e2) {
        w = nbr[i2 + lane];
        sv = osig[i2 + lane];
        if (EID) ev = eid[i2 + lane];
    }
    for (int32_t ib0 = i2; ib0 < e2; ib0 += 32) {
        const int32_t ib = ib0 + lane;
        // the next share's loads, in flight during this share's lookups
        int32_t wn = -1, sn = 0, en = 0;
        if (ib + 32 < e2) {
            wn = nbr[ib + 32];
            sn = osig[ib + 32];
            if (EID) en = eid[ib + 32];
        }
        int pu = -1;
        if (ib < e2) {
            uint32_t h = tri_hash(w);
            for (int p = 0; p < TRI_HSLOTS; p++) {
                const int32_t k = H.key[h];
                if (k == w) {
                    pu = H.pos[h];
                    break;
                }
                if (k < 0) break;
                h = (h + 1) & (TRI_HSLOTS - 1);
            }
        }
        hit(pu, w, sv, ev);
        w = wn;
        sv = sn;
        ev = en;
    }
}

// Also the probe slots of each oriented edge's triangles (sum over them of the three
// edges' temporal edge counts) into pcnt (may be null), and of all triangles into
// *probes, so that the triangles' probe offsets are known before they are written.
// Like the writing pass, an edge whose two out-lists hold more than heavy_min entries is
// intersected by the whole warp (the thread-versus-warp split the autotuner picks).
__global__ void __launch_bounds__(TRI_THREADS) k_tri_count(const int32_t* __restrict__ outptr,
                                                           const int32_t* __restrict__ out_nbr,
                                                           const int32_t* __restrict__ out_src,
                                                           const int32_t* __restrict__ osig, int32_t S,
                                                           int32_t* __restrict__ cnt, int64_t* __restrict__ pcnt,
                                                           unsigned long long* __restrict__ merged,
                                                           unsigned long long* __restrict__ probes, int heavy_min) {
    __shared__ TriHashW table[TRI_THREADS / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    unsigned long long acc = 0, pacc = 0;
    int32_t hashed = -1;  // the vertex whose out-list is in this warp's table
    for (int64_t j0 = blockIdx.x * (int64_t)blockDim.x + (threadIdx.x & ~31); j0 < S; j0 += stride) {
        const int64_t j = j0 + lane;
        int32_t u = 0, i1 = 0, e1 = 0, i2 = 0, e2 = 0, sig_uv = 0;
        if (j < S) {
            u = out_src[j];
            const int32_t v = out_nbr[j];
            sig_uv = osig[j];
            i1 = outptr[u];
            e1 = outptr[u + 1];
            i2 = outptr[v];
            e2 = outptr[v + 1];
            acc += (unsigned long long)((e1 - i1) + (e2 - i2));
        }
        const bool heavy = j < S && (e1 - i1) + (e2 - i2) > heavy_min && e1 - i1 <= TRI_HCAP;
        if (j < S && !heavy) {
            int32_t c = 0;
            unsigned long long ps = 0;
            int32_t a1 = i1, a2 = i2;
            while (a1 < e1 && a2 < e2) {
                const int32_t x = out_nbr[a1], y = out_nbr[a2];
                if (x == y) {
                    c++;
                    ps += (unsigned long long)(osig[a1] + osig[a2]);
                }
                a1 += (x <= y);
                a2 += (y <= x);
            }
            if (c) ps += (unsigned long long)c * (unsigned long long)sig_uv;
            pacc += ps;
            cnt[j] = c;
            if (pcnt) pcnt[j] = (int64_t)ps;
        }
        unsigned hm = __ballot_sync(0xffffffffu, heavy);
        while (hm) {
            const int src = __ffs(hm) - 1;
            hm &= hm - 1;
            const int32_t b1 = __shfl_sync(0xffffffffu, i1, src), f1 = __shfl_sync(0xffffffffu, e1, src);
            const int32_t b2 = __shfl_sync(0xffffffffu, i2, src), f2 = __shfl_sync(0xffffffffu, e2, src);
            const int32_t hs = __shfl_sync(0xffffffffu, sig_uv, src), hu = __shfl_sync(0xffffffffu, u, src);
            if (hu != hashed) {
                warp_hash_out<false>(out_nbr, osig, nullptr, b1, f1, table[warp]);
                hashed = hu;
            }
            int32_t c = 0;
            unsigned long long hp = 0;
            warp_probe_out<false>(out_nbr, osig, nullptr, b2, f2, table[warp],
                                  [&](int pu, int32_t, int32_t sv, int32_t) {
                                      if (pu >= 0) {
                                          c++;
                                          hp += (unsigned long long)(table[warp].sig[pu] + sv);
                                      }
                                  });
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                c += __shfl_xor_sync(0xffffffffu, c, o);
                hp += __shfl_xor_sync(0xffffffffu, hp, o);
            }
            if (lane == 0) {
                hp += (unsigned long long)c * (unsigned long long)hs;
                cnt[j0 + src] = c;
                if (pcnt) pcnt[j0 + src] = (int64_t)hp;
                pacc += hp;
            }
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        acc += __shfl_xor_sync(0xffffffffu, acc, o);
        pacc += __shfl_xor_sync(0xffffffffu, pacc, o);
    }
    if (lane == 0 && acc) atomicAdd(merged, acc);
    if (lane == 0 && pacc) atomicAdd(probes, pacc);
}

// tile_tri[b] = triangle holding probe min(b * tile, P - 1), for b in [0, tiles].
__global__ void k_tile_starts(const int64_t* __restrict__ tri_off, int64_t ntri, int64_t P, int64_t tiles,
                              int tile, int64_t* __restrict__ tile_tri) {
    for (int64_t b = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; b <= tiles;
         b += (int64_t)gridDim.x * blockDim.x) {
        int64_t p = min(b * (int64_t)tile, P - 1);
        int64_t lo = 0, hi = ntri - 1;  // largest t with tri_off[t] <= p
        while (lo < hi) {
            int64_t mid = (lo + hi + 1) >> 1;
            if (tri_off[mid] <= p) lo = mid;
            else hi = mid - 1;
        }
        tile_tri[b] = lo;
    }
}

// Writes every triangle, with OFF its probe offset (the running sum of the probe slots of
// the triangles before it, from the counting pass's prefix per oriented edge), and counts
// the triangles on every static edge. The triangles of oriented edge j start at toff[j].
template <bool OFF>
__global__ void __launch_bounds__(TRI_THREADS) k_tri_write(const int32_t* __restrict__ outptr,
                                                           const int32_t* __restrict__ out_nbr,
                                                           const int32_t* __restrict__ out_eid,
                                                           const int32_t* __restrict__ out_src,
                                                           const int32_t* __restrict__ osig, int32_t S,
                                                           const int64_t* __restrict__ toff,
                                                           const int64_t* __restrict__ poff, int4* __restrict__ tri,
                                                           int64_t* __restrict__ tri_off, int32_t* __restrict__ common,
                                                           int heavy_min) {
    __shared__ TriHashW table[TRI_THREADS / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    int32_t hashed = -1;  // the vertex whose out-list is in this warp's table
    for (int64_t j0 = blockIdx.x * (int64_t)blockDim.x + (threadIdx.x & ~31); j0 < S; j0 += stride) {
        const int64_t j = j0 + lane;
        int32_t u = 0, v = 0, s_uv = 0, sig_uv = 0, i1 = 0, e1 = 0, i2 = 0, e2 = 0;
        if (j < S) {
            u = out_src[j];
            v = out_nbr[j];
            s_uv = out_eid[j];
            sig_uv = osig[j];
            i1 = outptr[u];
            e1 = outptr[u + 1];
            i2 = outptr[v];
            e2 = outptr[v + 1];
        }
        const bool heavy = j < S && (e1 - i1) + (e2 - i2) > heavy_min && e1 - i1 <= TRI_HCAP;
        if (j < S && !heavy) {
            int64_t p = toff[j], q = OFF ? poff[j] : 0;
            int32_t n_here = 0;
            int32_t a1 = i1, a2 = i2;
            while (a1 < e1 && a2 < e2) {
                const int32_t x = out_nbr[a1], y = out_nbr[a2];
                if (x == y) {
                    const int32_t w = x, s_uw = out_eid[a1], s_vw = out_eid[a2];
                    const int flags = (u < v ? 1 : 0) | (u < w ? 2 : 0) | (v < w ? 4 : 0);
                    tri[p] = make_int4(s_uv, s_uw, s_vw, flags);
                    if (OFF) {
                        tri_off[p] = q;
                        q += (int64_t)sig_uv + osig[a1] + osig[a2];
                    }
                    atomicAdd(&common[s_uw], 1);
                    atomicAdd(&common[s_vw], 1);
                    p++;
                    n_here++;
                }
                a1 += (x <= y);
                a2 += (y <= x);
            }
            if (n_here) atomicAdd(&common[s_uv], n_here);
        }
        unsigned hm = __ballot_sync(0xffffffffu, heavy);
        while (hm) {
            const int src = __ffs(hm) - 1;
            hm &= hm - 1;
            const int32_t b1 = __shfl_sync(0xffffffffu, i1, src), f1 = __shfl_sync(0xffffffffu, e1, src);
            const int32_t b2 = __shfl_sync(0xffffffffu, i2, src), f2 = __shfl_sync(0xffffffffu, e2, src);
            const int32_t hu = __shfl_sync(0xffffffffu, u, src), hv = __shfl_sync(0xffffffffu, v, src);
            const int32_t hs = __shfl_sync(0xffffffffu, s_uv, src), hsig = __shfl_sync(0xffffffffu, sig_uv, src);
            int64_t p = (lane == 0) ? toff[j0 + src] : 0, q = (OFF && lane == 0) ? poff[j0 + src] : 0;
            p = __shfl_sync(0xffffffffu, p, 0);
            q = __shfl_sync(0xffffffffu, q, 0);
            int n_here = 0;
            if (hu != hashed) {
                warp_hash_out<true>(out_nbr, osig, out_eid, b1, f1, table[warp]);
                hashed = hu;
            }
            warp_probe_out<true>(
                out_nbr, osig, out_eid, b2, f2, table[warp],
                [&](int pu, int32_t w, int32_t sv, int32_t s_vw) {
                    const bool found = pu >= 0;
                    const unsigned m = __ballot_sync(0xffffffffu, found);
                    // the hits' probe offsets: a warp prefix of their costs, in lane order
                    const int64_t c = OFF && found ? (int64_t)hsig + table[warp].sig[pu] + sv : 0;
                    int64_t inc = c;
                    if (OFF) {
#pragma unroll
                        for (int o = 1; o < 32; o <<= 1) {
                            const int64_t y = __shfl_up_sync(0xffffffffu, inc, o);
                            if (lane >= o) inc += y;
                        }
                    }
                    if (found) {
                        const int32_t s_uw = table[warp].eid[pu];
                        const int64_t at = p + __popc(m & ((1u << lane) - 1u));
                        const int flags = (hu < hv ? 1 : 0) | (hu < w ? 2 : 0) | (hv < w ? 4 : 0);
                        tri[at] = make_int4(hs, s_uw, s_vw, flags);
                        if (OFF) tri_off[at] = q + inc - c;
                        atomicAdd(&common[s_uw], 1);
                        atomicAdd(&common[s_vw], 1);
                    }
                    p += __popc(m);
                    if (OFF) q += __shfl_sync(0xffffffffu, inc, 31);
                    n_here += __popc(m);
                });
            if (lane == 0 && n_here) atomicAdd(&common[hs], n_here);
        }
    }
}

// The triangles of graphs past the allocation-free counts' limit, in one pass without a
// counting pass before it. A warp takes 32 consecutive oriented edges (u, v) off a common
// counter (the dense communities' edges hold far more triangles than the rest). Their out(u)
// are one stretch of the out-lists: it goes into a hash table in the warp's shared memory, and
// the lanes look up all their out(v), laid end to end so that short lists leave no lane idle,
// the loads of the next 32 entries issued before this step's lookups. (A tail with more than
// TRI_HCAP out-neighbours has each of its edges merged by one lane.) The triangles found, few
// or many a step, go through a queue that the whole warp empties 32 at a time: only then are
// their records made, from the entries at their places in the out-lists, and with each the out
// motif's liveness byte from the runs of its three edges. A warp writes into chunks of `chunk`
// entries taken off a second counter; the rest of its last chunk stays empty (w = -1, never
// live), so the array holds at most chunk - 1 empty entries a warp and no pass has to move it.
// The triangles of the stretch's edges, as (u, v) and as (u, w), are counted in shared memory
// and added to common once; merged[0] receives the list entries looked up, merged[1] the
// triangles.
// Bound by issue slots and by gathers from L2 (46% of the slots, 33% of the warps at 20M edges;
// seven or nine blocks an SM are 3 to 5% slower at full size). At full size, 77M triangles from
// 115M lookups: 1150 us; 3M static edges, 2.8M triangles from 90M lookups: 400. A lane or a warp
// per edge, into a layout by upper bounds with three additions to common a triangle, and a second
// pass that gathered the three edges' runs and moved the triangles took 1110 + 750 and 584 + 75;
// the same without the queue, the records made by the lanes that found them, 1400 and 690.
// Looking up the shorter of the two lists (111M and 29M lookups) needs a table per row and edge
// direction: 1220 and 400.
// Tails with more than TRI_HCAP out-neighbours, merged by single lanes, cost about twice as much a
// triangle: preprocessing of 20 cliques of 300 vertices (89M triangles) takes 2.1 ms, of 4 of 600
// (143M) 4.3, of 30 of 240 (68M, all by tables) 1.5; with the two passes above 3.7, 7.6 and 2.1.
struct TriListArgs {
    const int32_t *outptr, *out_nbr, *out_src;
    const uint32_t* out_eup;  // static edge at a place of the out-lists; bit 31: the tail has the smaller id
    int32_t S;
    int chunk;  // a multiple of 32
    int4* tri;
    uint8_t* row;
    int32_t* common;
    unsigned long long *merged, *next, *used;  // next: edges taken; used: entries taken
};

// One warp's table of a stretch of the out-lists, in buckets of four filled from the first slot
// on: head (-1: empty) and position in the stretch; by position, the triangles found so far.
// The queue: the places of a triangle's edges (u, v), (u, w), (v, w) in the out-lists.
struct TriStretch {
    int4 key[TRI_BUCKETS];
    uint8_t pos[4 * TRI_BUCKETS];
    int32_t cnt[TRI_HCAP];
    int4 queue[64];
    uint8_t lane_of[32];
};

template <typename TS>
__global__ void __launch_bounds__(TRI_LIST_THREADS, TRI_PER_SM) k_tri_list(const TriListArgs a,
                                                                      const OutEnds<TS>* __restrict__ oe) {
    __shared__ TriStretch table[TRI_LIST_THREADS / 32];
    constexpr unsigned FULL = 0xffffffffu;
    constexpr uint32_t ID = 0x7fffffffu;
    const int lane = threadIdx.x & 31;
    const unsigned below = (1u << lane) - 1;
    TriStretch& H = table[threadIdx.x >> 5];
    unsigned long long acc = 0, found = 0;  // found: the same in every lane
    int64_t at = 0, end = 0;                // free entries of the warp's chunk
    int queued = 0;
    auto take = [&](unsigned long long* counter, int n) {
        unsigned long long x = 0;
        if (lane == 0) x = atomicAdd(counter, (unsigned long long)n);
        return (int64_t)__shfl_sync(FULL, x, 0);
    };
    // writes the first n <= 32 queued triangles, and empty entries up to 32
    auto write = [&](int n) {
        if (at == end) {
            at = take(a.used, a.chunk);
            end = at + a.chunk;
        }
        __syncwarp();
        int4 tr = make_int4(0, 0, 0, -1);
        uint8_t live = DMIN_NEVER;
        if (lane < n) {
            const int4 q = H.queue[lane];
            const int32_t uv = q.x, uw = q.y, vw = q.z;
            const uint32_t x = a.out_eup[uv], y = a.out_eup[uw], z = a.out_eup[vw];
            live = out_liveness<TS>(oe[uv], oe[uw], oe[vw]);
            tr = make_int4((int)(x & ID), (int)(y & ID), (int)(z & ID),
                           (int)(x >> 31) | (int)((y >> 31) << 1) | (int)((z >> 31) << 2));
            atomicAdd(&a.common[tr.z], 1);
        }
        __stcs(a.tri + at + lane, tr);
        a.row[at + lane] = live;
        at += 32;
        found += n;
    };
    // queues the triangles of the lanes of m
    auto push = [&](unsigned m, int32_t uv, int32_t uw, int32_t vw) {
        if ((m >> lane) & 1) H.queue[queued + __popc(m & below)] = make_int4(uv, uw, vw, 0);
        queued += __popc(m);
        if (queued < 32) return;
        write(32);
        queued -= 32;
        __syncwarp();
        if (lane < queued) H.queue[lane] = H.queue[32 + lane];
        __syncwarp();
    };
    // bucket of head w in the list at position lo of the stretch
    auto bucket = [](int lo, int32_t w) { return (int)(((uint32_t)(w + 31 * lo) * 0x9E3779B1u) >> 25); };
    static_assert(TRI_BUCKETS == 128 && TRI_HCAP <= 256, "7 bits of hash; positions are bytes");
    int64_t j0 = take(a.next, 32);
    while (j0 < a.S) {
        const int64_t j_next = take(a.next, 32);
        const int64_t j = j0 + lane;
        int32_t u = -1, i1 = 0, e1 = 0, i2 = 0, e2 = 0;
        if (j < a.S) {
            u = a.out_src[j];
            const int32_t v = a.out_nbr[j];
            i1 = a.outptr[u];
            e1 = a.outptr[u + 1];
            i2 = a.outptr[v];
            e2 = a.outptr[v + 1];
            acc += (unsigned long long)(e2 - i2);
        }
        unsigned left = __ballot_sync(FULL, j < a.S);
        while (left) {
            // the edges whose tails' lists fit the table together, from the first one left on
            const int first = __ffs(left) - 1;
            const int32_t b = __shfl_sync(FULL, i1, first);
            const bool here = (left >> lane) & 1;
            const bool mine = here && e1 - b <= TRI_HCAP;
            const unsigned batch = __ballot_sync(FULL, mine);
            if (batch == 0) {  // not even the first one's
                const bool merge = here && i1 == b;
                left &= ~__ballot_sync(FULL, merge);
                int32_t a1 = merge ? i1 : e1, a2 = i2, n_here = 0;
                while (__any_sync(FULL, a1 < e1 && a2 < e2)) {
                    const int32_t p1 = a1, p2 = a2;
                    bool hit = false;
                    if (a1 < e1 && a2 < e2) {
                        const int32_t x = a.out_nbr[a1], y = a.out_nbr[a2];
                        hit = x == y;
                        a1 += (x <= y);
                        a2 += (y <= x);
                    }
                    if (hit) {
                        n_here++;
                        atomicAdd(&a.common[a.out_eup[p1] & ID], 1);
                    }
                    const unsigned m = __ballot_sync(FULL, hit);
                    if (m) push(m, (int32_t)j, p1, p2);
                }
                if (n_here) atomicAdd(&a.common[a.out_eup[j] & ID], n_here);
                continue;
            }
            left &= ~batch;
            const int n_e = __shfl_sync(FULL, e1, 31 - __clz(batch)) - b;
            __syncwarp();  // the previous table's counts are added up
            for (int t = lane; t < TRI_BUCKETS; t += 32) H.key[t] = make_int4(-1, -1, -1, -1);
            __syncwarp();
            int32_t* keys = reinterpret_cast<int32_t*>(H.key);
            for (int t = lane; t < n_e; t += 32) {
                const int32_t w = a.out_nbr[b + t];
                int h = 4 * bucket(a.outptr[a.out_src[b + t]] - b, w);
                H.cnt[t] = 0;
                for (int p = 0; p < 4 * TRI_BUCKETS; p++) {  // ends: at most half of the slots are taken
                    if (atomicCAS(&keys[h], -1, w) == -1) {
                        H.pos[h] = (uint8_t)t;
                        break;
                    }
                    h = (h + 1) & (4 * TRI_BUCKETS - 1);
                }
            }
            // the batch's edges with a list to look up, one a lane, and the lists laid end to end
            const int32_t len = mine ? e2 - i2 : 0;
            int32_t inc = len;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int32_t y = __shfl_up_sync(FULL, inc, o);
                if (lane >= o) inc += y;
            }
            const int32_t total = __shfl_sync(FULL, inc, 31);
            const unsigned some = __ballot_sync(FULL, len > 0);
            if (len > 0) H.lane_of[__popc(some & below)] = (uint8_t)lane;
            __syncwarp();
            const bool on = lane < __popc(some);
            const int src = on ? H.lane_of[lane] : 0;
            const int32_t c_start = __shfl_sync(FULL, inc - len, src);
            const int32_t start = on ? c_start : INT_MAX;
            const int32_t shift = __shfl_sync(FULL, i2, src) - c_start;
            // the list's edge and its tail's list as positions in the stretch
            const int32_t where = __shfl_sync(FULL, ((i1 - b) << 20) | ((e1 - i1) << 10), src) | (int)(j0 + src - b);
            int before = 0;  // lists begun before the step
            int e_n = 0;
            int32_t at_n = 0, w_n = -1;
            auto fetch = [&](int32_t t0) {  // the step's list, entry and head of this lane
                const unsigned begun =
                    __reduce_or_sync(FULL, start >= t0 && start < t0 + 32 ? 1u << (start - t0) : 0u);
                e_n = before + __popc(begun & (below | (1u << lane))) - 1;
                before += __popc(begun);
                at_n = t0 + lane + __shfl_sync(FULL, shift, e_n);
                w_n = t0 + lane < total ? a.out_nbr[at_n] : -1;
            };
            if (total > 0) fetch(0);
            for (int32_t t0 = 0; t0 < total; t0 += 32) {
                const int e = e_n;
                const int32_t at_v = at_n, w = w_n;
                if (t0 + 32 < total) fetch(t0 + 32);
                const int32_t wh = __shfl_sync(FULL, where, e);
                const int lo = wh >> 20, puv = wh & 0x3ff;
                int pu = -1;
                if (w >= 0) {
                    int h = bucket(lo, w);
                    for (int p = 0; p < TRI_BUCKETS; p++) {
                        const int4 k = H.key[h];
                        const int s4 = k.x == w ? 0 : k.y == w ? 1 : k.z == w ? 2 : k.w == w ? 3 : -1;
                        if (s4 >= 0) {
                            const int at_first = 4 * h + s4;
                            pu = H.pos[at_first];
                            // another tail's entry of that head: on through the slots
                            for (int q = at_first; (unsigned)(pu - lo) >= (unsigned)((wh >> 10) & 0x3ff);) {
                                q = (q + 1) & (4 * TRI_BUCKETS - 1);
                                const int32_t kq = keys[q];
                                pu = kq == w ? H.pos[q] : -1;
                                if (kq < 0 || q == at_first) break;
                            }
                            break;
                        }
                        if (k.w < 0) break;
                        h = (h + 1) & (TRI_BUCKETS - 1);
                    }
                    if (pu >= 0) {
                        atomicAdd(&H.cnt[puv], 1);
                        atomicAdd(&H.cnt[pu], 1);
                    }
                }
                const unsigned m = __ballot_sync(FULL, pu >= 0);
                if (m) push(m, b + puv, b + pu, at_v);
            }
            __syncwarp();
            for (int t = lane; t < n_e; t += 32)
                if (H.cnt[t]) atomicAdd(&a.common[a.out_eup[b + t] & ID], H.cnt[t]);
        }
        j0 = j_next;
    }
    if (queued) write(queued);
    for (; at < end; at += 32) {
        a.tri[at + lane] = make_int4(0, 0, 0, -1);
        a.row[at + lane] = DMIN_NEVER;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(FULL, acc, o);
    if (lane == 0 && acc) atomicAdd(a.merged, acc);
    if (lane == 0 && found) atomicAdd(a.merged + 1, found);
}

// The out-lists' static edges as the listing reads them: oe[j] = the run ends of the one at
// place j in its orientation, eup[j] = its id and whether its tail has the smaller id.
template <typename TS>
__global__ void k_out_ends(const int32_t* __restrict__ out_src, const int32_t* __restrict__ out_nbr,
                           const int32_t* __restrict__ out_eid, int32_t S, const RunEnds<TS>* __restrict__ ends,
                           OutEnds<TS>* __restrict__ oe, uint32_t* __restrict__ eup) {
    for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < S; j += (int64_t)gridDim.x * blockDim.x) {
        const int32_t e = out_eid[j];
        const RunEnds<TS> r = ends[e];
        const bool up = out_src[j] < out_nbr[j];
        OutEnds<TS> o;
        o.f0 = up ? r.f0 : r.f1;
        o.l0 = up ? r.l0 : r.l1;
        o.f1 = up ? r.f1 : r.f0;
        o.l1 = up ? r.l1 : r.l0;
        oe[j] = o;
        eup[j] = (uint32_t)e | (up ? 0x80000000u : 0u);
    }
}

// Probe slots of all triangles (every temporal edge of a triangle's three static edges: the
// sum over the static edges of their temporal edges times their triangles) and the largest
// number of temporal edges of a static edge.
__global__ void k_probe_total(const int32_t* __restrict__ seg, const int32_t* __restrict__ common, int32_t S,
                              unsigned long long* __restrict__ probes, int* __restrict__ sigma_max) {
    unsigned long long acc = 0;
    int best = 0;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < S; e += (int64_t)gridDim.x * blockDim.x) {
        const int32_t c = seg[2 * e + 2] - seg[2 * e];
        acc += (unsigned long long)c * (unsigned long long)common[e];
        best = max(best, c);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        acc += __shfl_xor_sync(0xffffffffu, acc, o);
        best = max(best, __shfl_xor_sync(0xffffffffu, best, o));
    }
    if ((threadIdx.x & 31) == 0) {
        if (acc) atomicAdd(probes, acc);
        atomicMax(sigma_max, best);
    }
}

// Sum over the oriented edges (u, v) of min(|N+(u)|, |N+(v)|), at least the triangles.
__global__ void k_tri_bound(const int32_t* __restrict__ outptr, const int32_t* __restrict__ out_src,
                            const int32_t* __restrict__ out_nbr, int32_t S, unsigned long long* __restrict__ bound) {
    unsigned long long acc = 0;
    for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < S; j += (int64_t)gridDim.x * blockDim.x) {
        const int32_t u = out_src[j], v = out_nbr[j];
        acc += (unsigned long long)min(outptr[u + 1] - outptr[u], outptr[v + 1] - outptr[v]);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if ((threadIdx.x & 31) == 0 && acc) atomicAdd(bound, acc);
}

// ================================================================== driver

// A non-blocking stream of this thread (of the device's highest or default priority)
// for work that runs beside the caller's stream: fork() makes it wait for everything
// enqueued on the caller's stream so far, join() makes the caller's stream wait for
// everything enqueued on it. A fork that was not joined (an error in between) is
// drained on destruction.
class SideStream {
  public:
    SideStream(cudaStream_t s, bool high) : s_(s), high_(high) {}
    ~SideStream() {
        if (forked_) cudaStreamSynchronize(aux_);
        if (ev_[0]) cudaEventDestroy(ev_[0]);
        if (ev_[1]) cudaEventDestroy(ev_[1]);
    }
    SideStream(const SideStream&) = delete;
    SideStream& operator=(const SideStream&) = delete;

    cudaStream_t fork() {
        // per device and priority, kept for the thread's life
        thread_local std::vector<cudaStream_t> streams[2];
        int dev = 0;
        FOLTY_CUDA(cudaGetDevice(&dev));
        auto& v = streams[high_ ? 1 : 0];
        if ((int)v.size() <= dev) v.resize(dev + 1, nullptr);
        if (!v[dev]) {
            int least = 0, greatest = 0;
            FOLTY_CUDA(cudaDeviceGetStreamPriorityRange(&least, &greatest));
            FOLTY_CUDA(cudaStreamCreateWithPriority(&v[dev], cudaStreamNonBlocking, high_ ? greatest : least));
        }
        aux_ = v[dev];
        for (auto& e : ev_)
            if (!e) FOLTY_CUDA(cudaEventCreateWithFlags(&e, cudaEventDisableTiming));
        FOLTY_CUDA(cudaEventRecord(ev_[0], s_));
        FOLTY_CUDA(cudaStreamWaitEvent(aux_, ev_[0], 0));
        forked_ = true;
        return aux_;
    }
    void join() {
        FOLTY_CUDA(cudaEventRecord(ev_[1], aux_));
        FOLTY_CUDA(cudaStreamWaitEvent(s_, ev_[1], 0));
        forked_ = false;
    }

  private:
    cudaStream_t s_;
    bool high_;
    cudaStream_t aux_ = nullptr;
    cudaEvent_t ev_[2] = {nullptr, nullptr};
    bool forked_ = false;
};

constexpr int64_t STORE_BESIDE = 8;  // temporal edges per static one from which the store runs beside the core numbers

// The sorted values index other arrays: a sort whose look-back ran out must stop here
// (read_back checks the graph's error word).
static void sort_check(folty_graph* g, cudaStream_t s) { read_back(g, nullptr, nullptr, 0, nullptr, s); }

// The second half of A1 with dense pair ids: the temporal edges sorted by (pair id,
// direction, time rank) into the store (perm, T, sd, seg). It needs nothing of the
// static graph's later steps, and they nothing of it before the triangles, so it
// runs on a second stream beside or after the core numbers.
struct StoreJob {
    const uint32_t* slotw;  // [m] pair table slot and direction of each input edge
    const uint32_t* order;  // time order of an unsorted input, or null
    const int32_t* sid;     // [table] dense pair id of each table slot
    int ib;                 // bits of a time rank
};

// sigma (S entries, zeroed here) receives each static edge's temporal edge count, and
// packed_ev is recorded once it is complete.
static void temporal_store(folty_graph* g, const StoreJob& job, Scratch& sc, int32_t* sigma, cudaEvent_t packed_ev) {
    const int T = 256;
    const int64_t m = g->m, mk = g->m_kept;
    const int32_t S = g->S;
    const int ib = job.ib;
    cudaStream_t s = sc.stream();
    const int cbits = bit_length((uint64_t)(2 * S));
    if (!job.order && g->ts32) {
        // time-ordered input with 32-bit offsets: the sort ids and their counts (4 B slot
        // word read and 4 B id written per edge), then the stable sort of the ids, whose
        // first pass reads the ids and times (8 B per edge, 8 B written) and whose last
        // writes T and sd (8 B read and written per edge, as the passes between). perm,
        // the same order of the input indices, is sorted on first use from the ids the
        // graph keeps, except for graphs the allocation-free entry point takes (it needs
        // perm and may not allocate): they get it here.
        const int passes = cbits > STORE_DIGIT_BITS ? (cbits + STORE_DIGIT_BITS - 1) / STORE_DIGIT_BITS : 1;
        StageSpan span(ST_STORE, s, 8 * m + 16 * m * passes);
        const bool eager = mk <= FOLTY_NOALLOC_MAX_EDGES;
        uint32_t* cw = eager ? sc.get<uint32_t>(m) : graph_alloc<uint32_t>(g, m, s);
        int32_t* cnt = sc.get<int32_t>(2 * (int64_t)S + 1);
        uint32_t* hist = eager ? sc.get<uint32_t>(STORE_MAX_PASSES << STORE_DIGIT_BITS)
                               : graph_alloc<uint32_t>(g, STORE_MAX_PASSES << STORE_DIGIT_BITS, s);
        FOLTY_CUDA(cudaMemsetAsync(cnt, 0, sizeof(int32_t) * (2 * (size_t)S + 1), s));
        FOLTY_CUDA(cudaMemsetAsync(hist, 0, sizeof(uint32_t) * (STORE_MAX_PASSES << STORE_DIGIT_BITS), s));
        // one block per 2048 edges: short blocks, so that the kernels on the high-priority
        // stream get SMs as soon as any block ends
        FOLTY_LAUNCH(k_store_ids, (unsigned)(((m + STORE_IDS_EDGES - 1) / STORE_IDS_EDGES + T - 1) / T), T, 0, s,
                     job.slotw, m, job.sid, S, cw, cnt);
        // the runs: seg[c] = first sorted position of id c, seg[2S] = mk
        exclusive_scan(sc, cnt, g->seg, 2 * (int64_t)S);
        FOLTY_LAUNCH(k_store_sigma, grid_for(S, T), T, 0, s, g->seg, S, sigma);
        FOLTY_CUDA(cudaEventRecord(packed_ev, s));
        FOLTY_LAUNCH(k_store_hist, grid_for(2 * (int64_t)S + 1, T, 2), T, 0, s, cnt, S, passes, hist);
        const StoreSortArgs sa{cw, g->in_t32, (uint32_t)g->tmin, m, cbits, hist, (uint32_t*)g->T, g->sd, nullptr, mk};
        store_sort(sc, sa);
        if (eager) {
            g->perm = graph_alloc<int32_t>(g, mk, s);
            StoreSortArgs pa = sa;
            pa.perm = g->perm;
            perm_sort(sc, pa);
        } else {
            g->cw = cw;
            g->store_hist = hist;
            g->store_cbits = cbits;
        }
        return;
    }
    g->perm = graph_alloc<int32_t>(g, mk, s);
    // the whole store: its pair words and time offsets (4 B slot and
    // 8 B time read, 12 B written per input edge) and the sorted arrays (the word and the
    // time read, perm, T and sd written: 24 B per kept edge); the sort passes inside are
    // also SORT spans
    StageSpan span(ST_STORE, s, 24 * m + 24 * mk);
    // edges by (pair id, direction, time rank), sorted on the id and direction bits; a
    // 32-bit store carries each edge's time offset through the sort as its value
    uint64_t* packed = sc.get<uint64_t>(m);
    uint64_t* packed_alt = sc.get<uint64_t>(m);
    uint32_t* tv = g->ts32 ? sc.get<uint32_t>(m) : nullptr;
    uint32_t* tv_alt = g->ts32 ? sc.get<uint32_t>(m) : nullptr;
    FOLTY_CUDA(cudaMemsetAsync(sigma, 0, sizeof(int32_t) * (size_t)S, s));
    FOLTY_LAUNCH(k_pair_pack, (unsigned)((m + T - 1) / T), T, 0, s, job.slotw, job.order, m, job.sid, S, ib, packed,
                 g->in_t32, (uint32_t)g->tmin, tv, sigma);
    FOLTY_CUDA(cudaEventRecord(packed_ev, s));
    const bool palt = g->ts32 ? radix_sort_pairs(sc, packed, packed_alt, tv, tv_alt, m, ib, cbits)
                              : radix_sort_keys(sc, packed, packed_alt, m, ib, cbits);
    const uint64_t* sp = palt ? packed_alt : packed;
    FOLTY_CUDA(cudaMemsetAsync(g->seg, 0xff, sizeof(int32_t) * (2 * (size_t)S + 1), s));
    if (g->ts32)
        FOLTY_LAUNCH(k_pair_store4, (unsigned)(((mk + 3) / 4 + T - 1) / T), T, 0, s, sp, job.order, mk, S, ib,
                     palt ? tv_alt : tv, g->perm, (uint32_t*)g->T, g->sd, g->seg);
    else
        FOLTY_LAUNCH((k_pair_store<int64_t>), grid_for(mk, T), T, 0, s, sp, job.order, mk, S, ib, g->in_t,
                     g->perm, (int64_t*)g->T, g->sd, g->seg);
    FOLTY_LAUNCH(k_segments_fix, grid_for(S, T), T, 0, s, S, mk, g->seg);
}

void enqueue_pair_list(const uint64_t* table, int lg, uint64_t* rank, uint32_t* slot, int* cnt, int cap, cudaStream_t s) {
    const int64_t tb = 1ll << lg;
    FOLTY_LAUNCH(k_pair_table_compact, grid_for(tb, (int64_t)256 * PAIR_COMPACT_ITEMS), 256, 0, s, table, tb, rank, slot, cnt,
                 cap);
}

// A1 with dense pair ids (see k_pair_insert) up to the static edge list (ea, eb) and
// the job of the temporal store: false, with nothing of the graph written, when the
// table cannot serve (too many distinct pairs, a probe sequence ran out, or ids and
// time ranks do not fit one word); FOLTY_PAIR_SORT=keys forces that answer. The
// distinct-pair sort is checked by the next read-back (before any of its consumers but
// the guarded k_pair_ids index with it).
static bool pair_ids_sort(folty_graph* g, Scratch& sc, const uint32_t* order, cudaStream_t s, StoreJob* job) {
    const int T = 256;
    const int64_t m = g->m, mk = g->m_kept;
    const int32_t n = g->n;
    if (!g->pre_slotw && pair_table_forced_off()) return false;  // a load that forced it off kept the edges
    if (mk == 0 || n < 2) return false;
    const int ib = bit_length((uint64_t)(m - 1));
    // the distinct pairs: listed by the load when its table served; otherwise a table of the
    // largest size, unless the load tried that one
    int lg = g->pre_lg;
    int64_t S64 = g->pre_pairs;
    const uint32_t* slotw = g->pre_slotw;
    uint64_t* urank = g->pre_rank;
    uint32_t* uslot = g->pre_slot;
    if (!slotw) {
        const int lg_max = pair_table_lg_max(m);
        if (lg == lg_max) return false;
        lg = lg_max;
        const int cap = (1 << lg) / 2;  // load factor at most 1/2
        int* flags = sc.get<int>(PAIR_FLAGS);
        uint32_t* sw = sc.get<uint32_t>(m);
        uint64_t* table = sc.get<uint64_t>(1ll << lg);
        FOLTY_CUDA(cudaMemsetAsync(table, 0, sizeof(uint64_t) << lg, s));
        FOLTY_CUDA(cudaMemsetAsync(flags, 0, PAIR_FLAGS * sizeof(int), s));
        FOLTY_LAUNCH(k_pair_insert, grid_for(m, T), T, 0, s, g->in_src, g->in_dst, m, n, table, lg, sw, flags);
        urank = sc.get<uint64_t>(cap);
        uslot = sc.get<uint32_t>(cap);
        enqueue_pair_list(table, lg, urank, uslot, flags + 1, cap, s);
        const void* ptrs[2] = {flags, flags + 1};
        int sizes[2] = {4, 4};
        int64_t fv[2];
        read_back(g, ptrs, sizes, 2, fv, s);
        S64 = fv[1];
        if (fv[0] != 0 || S64 > cap) return false;
        slotw = sw;
    }
    const int64_t tb = 1ll << lg;
    if (bit_length((uint64_t)(2 * S64)) + ib > 64) return false;
    const int32_t S = (int32_t)S64;
    // the distinct pairs in (a, b) order: ids, ends
    uint64_t* urank_alt = sc.get<uint64_t>(S);
    uint32_t* uslot_alt = sc.get<uint32_t>(S);
    const int rank_bits = bit_length((uint64_t)n * (uint64_t)(n - 1) / 2);
    const bool ualt = radix_sort_pairs(sc, urank, urank_alt, uslot, uslot_alt, S, rank_bits);
    const uint64_t* ur = ualt ? urank_alt : urank;
    const uint32_t* us = ualt ? uslot_alt : uslot;
    g->S = S;
    g->ea = graph_alloc<int32_t>(g, S, s);
    g->eb = graph_alloc<int32_t>(g, S, s);
    g->seg = graph_alloc<int32_t>(g, 2 * (int64_t)S + 1, s);
    int32_t* sid = sc.get<int32_t>(tb);
    FOLTY_LAUNCH(k_pair_ids, grid_for(S, T), T, 0, s, ur, us, S, n, tb, sid, g->ea, g->eb);
    *job = StoreJob{slotw, order, sid, ib};
    return true;
}

// A1 with the full pair key (2 p(a, b) + direction, see k_build_keys) and the input
// index (or time rank) as the value.
static void pair_key_sort(folty_graph* g, Scratch& sc, const uint32_t* order, cudaStream_t s) {
    const int T = 256;
    const int64_t m = g->m, mk = g->m_kept;
    const int32_t n = g->n;
    const int key_bits = n > 1 ? bit_length((uint64_t)n * (uint64_t)(n - 1)) : 1;  // keys < n (n - 1)
    const uint64_t loop_key = (key_bits >= 64) ? ~0ull : ((1ull << key_bits) - 1);
    g->perm = graph_alloc<int32_t>(g, mk, s);
    uint64_t* key = sc.get<uint64_t>(m);
    uint64_t* key_alt = sc.get<uint64_t>(m);
    uint32_t* val = sc.get<uint32_t>(m);
    uint32_t* val_alt = sc.get<uint32_t>(m);
    FOLTY_LAUNCH(k_build_keys, grid_for(m, T), T, 0, s, g->in_src, g->in_dst, m, n, loop_key, key, val);
    uint64_t* skey = key;
    uint32_t* sval = val;
    if (order) {
        // keys in time order, values the input indices: the stable sort keeps time order
        FOLTY_LAUNCH(k_gather_keys, grid_for(m, T), T, 0, s, key, order, m, key_alt);
        FOLTY_CUDA(cudaMemcpyAsync(val, order, sizeof(uint32_t) * (size_t)m, cudaMemcpyDeviceToDevice, s));
        const bool alt = radix_sort_pairs(sc, key_alt, key, val, val_alt, m, key_bits);
        skey = alt ? key : key_alt;
        sval = alt ? val_alt : val;
    } else {
        const bool alt = radix_sort_pairs(sc, key, key_alt, val, val_alt, m, key_bits);
        skey = alt ? key_alt : key;
        sval = alt ? val_alt : val;
    }
    sort_check(g, s);
    int32_t* newpair = sc.get<int32_t>(mk + 1);
    int32_t* pscan = sc.get<int32_t>(mk + 1);
    if (mk > 0) {
        if (g->ts32)
            FOLTY_LAUNCH(k_store<uint32_t>, grid_for(mk, T), T, 0, s, skey, sval, g->in_t32, (uint32_t)g->tmin, mk,
                         g->perm, (uint32_t*)g->T, newpair);
        else
            FOLTY_LAUNCH(k_store<int64_t>, grid_for(mk, T), T, 0, s, skey, sval, g->in_t, (int64_t)0, mk, g->perm,
                         (int64_t*)g->T, newpair);
    }
    exclusive_scan(sc, newpair, pscan, mk);
    const int32_t S = read_i32(g, pscan + mk, s);
    g->S = S;
    g->ea = graph_alloc<int32_t>(g, S, s);
    g->eb = graph_alloc<int32_t>(g, S, s);
    g->seg = graph_alloc<int32_t>(g, 2 * (int64_t)S + 1, s);
    if (mk > 0) {
        FOLTY_LAUNCH(k_segments, grid_for(mk, T), T, 0, s, skey, newpair, pscan, mk, g->sd, g->seg);
        FOLTY_LAUNCH(k_pair_ends, grid_for(S, T), T, 0, s, skey, g->seg, S, n, g->ea, g->eb);
        FOLTY_LAUNCH(k_segments_split, grid_for(mk, T), T, 0, s, g->sd, mk, S, g->seg);
        FOLTY_LAUNCH(k_segments_fix, grid_for(S, T), T, 0, s, S, mk, g->seg);
    } else {
        FOLTY_CUDA(cudaMemsetAsync(g->seg, 0, sizeof(int32_t), s));
    }
}

// The counting pass of the triangle listing (tcnt per oriented edge; merged list entries
// and probe slots into merged[0], merged[1], zeroed here) under the graph's split between
// one thread and one warp per oriented edge: forced, cached under the graph's statistics,
// or picked by timing the pass under each candidate split. All candidates count the same
// triangles, so the last trial's outputs stand.
static void tune_triangles(folty_graph* g, const int32_t* outptr, const int32_t* out_nbr, const int32_t* out_src,
                           const int32_t* osig, int32_t* tcnt, int64_t* pcnt, unsigned long long* merged,
                           cudaStream_t s) {
    const int32_t S = g->S;
    const unsigned grid = grid_for(S, TRI_THREADS);
    const std::vector<int64_t> key{g->n, g->m_kept, S};
    bool trials = !(tune_forced(&g->tune, false) || tune_lookup(key, &g->tune, false)) && !profiling_on();
    if (!trials) {
        FOLTY_CUDA(cudaMemsetAsync(merged, 0, 2 * sizeof(unsigned long long), s));
        FOLTY_LAUNCH(k_tri_count, grid, TRI_THREADS, 0, s, outptr, out_nbr, out_src, osig, S, tcnt, pcnt, merged,
                     merged + 1, g->tune.tri_heavy);
        return;
    }
    cudaEvent_t ev[TUNE_TRIALS + 1];
    for (auto& e : ev) FOLTY_CUDA(cudaEventCreate(&e));
    int best = 1;
    try {
        for (int c = 0; c < TUNE_TRIALS; c++) {
            FOLTY_CUDA(cudaMemsetAsync(merged, 0, 2 * sizeof(unsigned long long), s));
            FOLTY_CUDA(cudaEventRecord(ev[0], s));
            FOLTY_LAUNCH(k_tri_count, grid, TRI_THREADS, 0, s, outptr, out_nbr, out_src, osig, S, tcnt, pcnt, merged,
                         merged + 1, TRI_HEAVY_CAND[c]);
            FOLTY_CUDA(cudaEventRecord(ev[c + 1], s));
            FOLTY_CUDA(cudaEventSynchronize(ev[c + 1]));
            FOLTY_CUDA(cudaEventElapsedTime(&g->tune.tri_ms[c], ev[0], ev[c + 1]));
            if (g->tune.tri_ms[c] < g->tune.tri_ms[best]) best = c;
        }
    } catch (...) {
        for (auto& e : ev) cudaEventDestroy(e);
        throw;
    }
    for (auto& e : ev) cudaEventDestroy(e);
    g->tune.tri_heavy = TRI_HEAVY_CAND[best];
    g->tune.tri_source = 1;
    tune_store(key, g->tune, false);
}

template <typename TS>
static void list_triangles(folty_graph* g, const TriListArgs& a, const int32_t* out_eid, OutEnds<TS>* oe, uint32_t* eup,
                           int grid, cudaStream_t s) {
    FOLTY_LAUNCH(k_out_ends<TS>, grid_for(a.S, 256), 256, 0, s, a.out_src, a.out_nbr, out_eid, a.S,
                 (const RunEnds<TS>*)g->run_ends, oe, eup);
    FOLTY_LAUNCH(k_tri_list<TS>, grid, TRI_LIST_THREADS, 0, s, a, oe);
}

void ensure_perm(folty_graph* g, cudaStream_t s) {
    std::lock_guard<std::mutex> lock(g->perm_mu);
    if (g->perm) {
        if (g->perm_ev) FOLTY_CUDA(cudaStreamWaitEvent(s, g->perm_ev, 0));
        return;
    }
    if (!g->cw) fail(FOLTY_EINVAL, "graph has no store to order");
    int32_t* perm = graph_alloc<int32_t>(g, g->m_kept, s);
    Scratch sc(g->alloc, s, g->dev_err);
    perm_sort(sc, StoreSortArgs{g->cw, nullptr, 0, g->m, g->store_cbits, g->store_hist, nullptr, nullptr, perm,
                                g->m_kept});
    FOLTY_CUDA(cudaEventCreateWithFlags(&g->perm_ev, cudaEventDisableTiming));
    FOLTY_CUDA(cudaEventRecord(g->perm_ev, s));
    g->perm = perm;
}

static void preprocess_on(folty_graph* g, cudaStream_t s) {
    const int T = 256;
    const int64_t m = g->m;
    const int32_t n = g->n;
    Scratch sc(g->alloc, s, g->dev_err);

    // ---------------- A1: canonical order
    const int nb = bit_length((uint64_t)(n > 1 ? n - 1 : 1));
    const int64_t mk = g->m_kept;
    if (g->ts32) g->T = graph_alloc<uint32_t>(g, mk, s);
    else g->T = graph_alloc<int64_t>(g, mk, s);
    g->sd = graph_alloc<int32_t>(g, mk, s);
    // time order of an input that is not sorted by time (stable): order[j] = input index
    uint32_t* order = nullptr;
    if (!g->info.time_sorted && m > 1) {
        uint64_t* tk = sc.get<uint64_t>(m);
        uint64_t* tk_alt = sc.get<uint64_t>(m);
        uint32_t* iv = sc.get<uint32_t>(m);
        uint32_t* iv_alt = sc.get<uint32_t>(m);
        FOLTY_LAUNCH(k_time_keys, grid_for(m, T), T, 0, s, g->ts32 ? g->in_t32 : nullptr, g->in_t, m, g->tmin, tk, iv);
        const bool alt = radix_sort_pairs(sc, tk, tk_alt, iv, iv_alt, m, bit_length((uint64_t)(g->tmax - g->tmin)));
        sort_check(g, s);
        order = alt ? iv_alt : iv;
    }
    StoreJob job{};
    const bool ids = pair_ids_sort(g, sc, order, s, &job);
    if (!ids) pair_key_sort(g, sc, order, s);
    const int32_t S = g->S;
    // the temporal store of the dense-id path: on a side stream of default priority, beside
    // the core numbers or after them beside the orientation (A3 below), whose kernels run on a
    // stream of the highest priority and take SMs first. It is joined before a one-pass listing,
    // which reads its run ends, and after the counting pass and the listing of small graphs,
    // which need its per-pair counts only. On an error in between, the side streams are drained
    // before the call's buffers go.
    SideStream side(s, false);
    struct EventHolder {
        cudaEvent_t e = nullptr;
        ~EventHolder() {
            if (e) cudaEventDestroy(e);
        }
    } packed_ev;
    int32_t* sigma = nullptr;
    cudaStream_t store_s = nullptr;
    if (ids) {
        FOLTY_CUDA(cudaEventCreateWithFlags(&packed_ev.e, cudaEventDisableTiming));
        sigma = sc.get<int32_t>(S > 0 ? S : 1);
    }

    // ---------------- A2: static CSR
    // static edges are sorted by (a, b); a stable sort by b lists them by (b, a)
    uint32_t* by_b = nullptr;
    if (S > 0) {
        uint64_t* bk = sc.get<uint64_t>(S);
        uint64_t* bk_alt = sc.get<uint64_t>(S);
        uint32_t* bv = sc.get<uint32_t>(S);
        uint32_t* bv_alt = sc.get<uint32_t>(S);
        FOLTY_LAUNCH(k_edge_keys_b, grid_for(S, T), T, 0, s, g->eb, S, bk, bv);
        bool alt = radix_sort_pairs(sc, bk, bk_alt, bv, bv_alt, S, nb);
        by_b = alt ? bv_alt : bv;
        sort_check(g, s);
    }
    g->by_b = graph_alloc<int32_t>(g, S, s);
    g->binv = graph_alloc<int32_t>(g, S, s);
    if (S > 0) FOLTY_CUDA(cudaMemcpyAsync(g->by_b, by_b, sizeof(int32_t) * (size_t)S, cudaMemcpyDeviceToDevice, s));
    int32_t* runs = sc.get<int32_t>(4 * ((int64_t)n + 1));  // hi_first, hi_last, lo_first, lo_last
    int32_t* hi_first = runs;
    int32_t* hi_last = runs + (n + 1);
    int32_t* lo_first = runs + 2 * ((int64_t)n + 1);
    int32_t* lo_last = runs + 3 * ((int64_t)n + 1);
    FOLTY_CUDA(cudaMemsetAsync(runs, 0, sizeof(int32_t) * 4 * ((size_t)n + 1), s));
    if (S > 0) {
        FOLTY_LAUNCH(k_runs, grid_for(S, T), T, 0, s, g->ea, (const uint32_t*)nullptr, S, hi_first, hi_last);
        FOLTY_LAUNCH(k_runs, grid_for(S, T), T, 0, s, g->eb, by_b, S, lo_first, lo_last);
    }
    int32_t* deg_lo = sc.get<int32_t>((int64_t)n + 1);
    g->deg = graph_alloc<int32_t>(g, (int64_t)n + 1, s);
    FOLTY_LAUNCH(k_degrees, grid_for(n, T), T, 0, s, hi_first, hi_last, lo_first, lo_last, (int64_t)n, deg_lo,
                 g->deg);
    int32_t* rowptr = sc.get<int32_t>((int64_t)n + 1);
    exclusive_scan(sc, g->deg, rowptr, n);
    const int64_t n2 = 2 * (int64_t)S;
    int32_t* adj = sc.get<int32_t>(n2);
    int32_t* adj_eid = sc.get<int32_t>(n2);
    int32_t* adj_src = sc.get<int32_t>(n2);
    if (S > 0)
        FOLTY_LAUNCH(k_fill_adj, grid_for(S, T), T, 0, s, g->ea, g->eb, S, rowptr, deg_lo, hi_first, lo_first,
                     by_b, adj, adj_eid, adj_src, g->binv);

    // ---------------- A3: core numbers and the removal order
    g->core = graph_alloc<int32_t>(g, n, s);
    int32_t* rnd = sc.get<int32_t>(n);
    // The store and, at the end of its stream, the run-ends table (ready when it is joined).
    // The core numbers' cooperative kernel waits for SMs that the store's blocks hold, so it is
    // launched first. Where the store is the longer of the two (many temporal edges per static
    // one) it takes half the SMs, whose registers it fills, and the store the others: most of
    // its rounds are bound by latency. Preprocessing of 20M edges beside against one after the
    // other, by edges per static edge: 7.28 against 7.26 ms at 2.3, 5.12 against 5.14 at 4.1, 3.06
    // against 3.27 at 8, 1.50 against 1.79 at 24; of 6M edges 2.78 against 2.69, 1.97 against
    // 2.03, 1.39 against 1.48, 0.80 against 0.98. From 4 on it is no slower; the line stays on
    // the side where it gains clearly.
    const bool beside = ids && g->m_kept >= STORE_BESIDE * (int64_t)S;
    if (beside) store_s = side.fork();
    // rounds, alpha and the error word are read with the triangle totals
    const int* core_ctl =
        enqueue_core_numbers(g, rowptr, adj, adj_src, rnd, beside ? std::max(num_sms() / 2, 1) : num_sms(), sc, s);
    if (ids) {
        if (!beside) store_s = side.fork();
        Scratch sc2(g->alloc, store_s, g->dev_err);
        temporal_store(g, job, sc2, sigma, packed_ev.e);
        build_run_ends(g, store_s);
    }

    // ---------------- A4: orientation
    int* stat = sc.get<int>(4);  // max degree, max out-degree, max sigma, (pad)
    FOLTY_CUDA(cudaMemsetAsync(stat, 0, sizeof(int) * 4, s));
    int32_t* oflag = sc.get<int32_t>(n2 + 1);
    int32_t* opos = sc.get<int32_t>(n2 + 1);
    if (n2 > 0) FOLTY_LAUNCH(k_orient_flags, grid_for(n2, T), T, 0, s, adj_src, adj, rnd, n2, oflag);
    exclusive_scan(sc, oflag, opos, n2);
    int32_t* outptr = sc.get<int32_t>((int64_t)n + 1);
    FOLTY_LAUNCH(k_outptr, grid_for((int64_t)n + 1, T), T, 0, s, rowptr, opos, (int64_t)n, outptr, stat + 1);
    int32_t* out_nbr = sc.get<int32_t>(S);
    int32_t* out_eid = sc.get<int32_t>(S);
    int32_t* out_src = sc.get<int32_t>(S);
    if (n2 > 0)
        FOLTY_LAUNCH(k_orient_fill, grid_for(n2, T), T, 0, s, adj_src, adj, adj_eid, oflag, opos, n2, out_nbr,
                     out_eid, out_src);

    // ---------------- A5: triangles
    g->common = graph_alloc<int32_t>(g, S, s);
    FOLTY_CUDA(cudaMemsetAsync(g->common, 0, sizeof(int32_t) * ((size_t)S > 0 ? (size_t)S : 1), s));
    // [0] list lengths merged, [1] probe slots (of the counting pass) or triangles (of the
    // one-pass listing); of the latter: [2] the bound, [3] the probe slots, [4] edges taken,
    // [5] entries taken
    unsigned long long* merged = sc.get<unsigned long long>(6);
    FOLTY_CUDA(cudaMemsetAsync(merged, 0, 6 * sizeof(unsigned long long), s));
    FOLTY_LAUNCH(k_max_i32, grid_for(n, T), T, 0, s, g->deg, (int64_t)n, stat + 0);
    // the all-roles probe map (each triangle's first slot in the flat space of every
    // role's probes, and the tile starts) serves only the allocation-free per-edge counts,
    // which take graphs of at most FOLTY_NOALLOC_MAX_EDGES edges; the queries lay out the
    // kept roles of their own selection
    const bool probe_map = g->m_kept <= FOLTY_NOALLOC_MAX_EDGES;
    // Larger graphs list their triangles and the out motif's liveness bytes in one pass, into
    // an array of the upper bound's size: no counting pass before it and no wait for its total.
    // The pass reads the store's run ends, so it follows the store's sort; the counting pass
    // needs the static edges' temporal edge counts only and the listing after it neither, so
    // both run beside that sort. The probe map needs the counting pass's slots per edge, and a
    // bound past TRI_BOUND_MAX_BYTES takes it too.
    bool bounded = !probe_map && S > 0 && !tri_layout_counted();
    int32_t* tcnt = nullptr;
    int64_t *toff = nullptr, *pcnt = nullptr;  // pcnt: slots per oriented edge, then their prefix
    int32_t* osig = nullptr;
    if (bounded)
        FOLTY_LAUNCH(k_tri_bound, grid_for(S, T), T, 0, s, outptr, out_src, out_nbr, S, merged + 2);
    // the counting pass merges the two out-lists of every oriented edge: 4 B per merged
    // entry (known after its read-back) + 8 B per static edge
    std::optional<StageSpan> count_span;
    auto count_pass = [&]() {
        if (ids) FOLTY_CUDA(cudaStreamWaitEvent(s, packed_ev.e, 0));
        tcnt = sc.get<int32_t>((int64_t)S + 1);
        toff = sc.get<int64_t>((int64_t)S + 1);
        if (probe_map) pcnt = sc.get<int64_t>((int64_t)S + 1);
        osig = sc.get<int32_t>(S);
        if (S > 0) FOLTY_LAUNCH(k_out_sigma, grid_for(S, T), T, 0, s, sigma, g->seg, out_eid, S, osig, stat + 2);
        count_span.emplace(ST_TRIANGLES, s, 8 * (int64_t)S);
        FOLTY_CUDA(cudaMemsetAsync(merged, 0, 2 * sizeof(unsigned long long), s));
        if (S > 0) tune_triangles(g, outptr, out_nbr, out_src, osig, tcnt, pcnt, merged, s);
        exclusive_scan(sc, tcnt, toff, S);
        if (probe_map) exclusive_scan(sc, pcnt, pcnt, S);
        count_span->end();
    };
    auto counted = [&](int64_t total, int64_t list_len, int64_t probes) {
        g->ntri = total;
        g->info.probes = probes;
        g->enum_bytes = 4 * list_len + 8 * (int64_t)S;
        count_span->add_bytes(4 * list_len);
    };
    if (!bounded) count_pass();
    int64_t bound = 0;
    {
        const void* ptrs[9] = {bounded ? (const void*)(merged + 2) : (const void*)(toff + S), stat + 0, stat + 1,
                               stat + 2, merged, merged + 1, core_ctl + CORE_ERR, core_ctl + CORE_ROUNDS, core_ctl + CORE_ALPHA};
        int sizes[9] = {8, 4, 4, 4, 8, 8, 4, 4, 4};
        int64_t outv[9] = {0, 0, 0, 0, 0, 0, 0, 0, 0};
        read_back(g, ptrs, sizes, 9, outv, s);
        if (outv[6] == 1) fail(FOLTY_ETIMEOUT, "core numbers: a grid barrier wait ran out");
        if (outv[6] != 0) fail(FOLTY_ECUDA, "core numbers: a vertex list overflowed");
        g->info.peel_rounds = (int32_t)outv[7];
        g->info.degeneracy = (int32_t)outv[8];
        g->info.max_degree = (int32_t)outv[1];
        g->info.max_out_degree = (int32_t)outv[2];
        g->info.sigma_max = (int32_t)outv[3];
        if (bounded) bound = outv[0];
        else counted(outv[0], outv[4], outv[5]);
    }
    if (bounded && bound > TRI_BOUND_MAX_BYTES / (int64_t)sizeof(int4)) {
        bounded = false;
        count_pass();
        const void* ptrs[4] = {toff + S, merged, merged + 1, stat + 2};
        int sizes[4] = {8, 8, 8, 4};
        int64_t outv[4] = {0, 0, 0, 0};
        read_back(g, ptrs, sizes, 4, outv, s);
        counted(outv[0], outv[1], outv[2]);
        g->info.sigma_max = (int32_t)outv[3];
    }
    if (bounded) {
        tune_forced(&g->tune, false);  // recorded; the listing has no split to choose
        const int warps = TRI_LIST_THREADS / 32;
        const int grid = (int)std::min<int64_t>((S + TRI_LIST_THREADS - 1) / TRI_LIST_THREADS, (int64_t)num_sms() * TRI_PER_SM);
        int chunk = TRI_CHUNK_MAX;
        while (chunk > TRI_CHUNK_MIN && (int64_t)chunk * grid * warps * 16 > bound) chunk >>= 1;
        const int64_t ends = (int64_t)chunk * grid * warps;  // entries in no warp's use at the chunks' ends
        const int64_t cap = (bound + ends + 31) & ~int64_t(31);  // whole chunks are in use: no padding to clear
        g->tri = graph_alloc<int4>(g, cap, s);
        g->tri_off = nullptr;
        uint8_t* live = liveness_rows(g, 1, cap, s);
        FOLTY_CUDA(cudaMemsetAsync(merged, 0, 2 * sizeof(unsigned long long), s));
        if (ids) side.join();
        if (!ids) build_run_ends(g, s);
        // the listing: 8 B per static edge + 4 B per merged entry + 17 B per triangle; the
        // totals come with the last read-back
        StageSpan span(ST_TRIANGLES, s, 8 * (int64_t)S);
        uint32_t* eup = sc.get<uint32_t>(S);
        const TriListArgs a{outptr,      out_nbr, out_src, eup,       S,         chunk,
                            g->tri, live,    g->common, merged, merged + 4, merged + 5};
        if (g->ts32) list_triangles<uint32_t>(g, a, out_eid, sc.get<OutEnds<uint32_t>>(S), eup, grid, s);
        else list_triangles<int64_t>(g, a, out_eid, sc.get<OutEnds<int64_t>>(S), eup, grid, s);
        FOLTY_LAUNCH(k_probe_total, grid_for(S, T), T, 0, s, g->seg, g->common, S, merged + 3, stat + 2);
        span.end();
        const void* ptrs[5] = {merged, merged + 1, merged + 3, merged + 5, stat + 2};
        int sizes[5] = {8, 8, 8, 8, 4};
        int64_t outv[5] = {0, 0, 0, 0, 0};
        read_back(g, ptrs, sizes, 5, outv, s);  // it also checks that the store's sort completed
        g->ntri = outv[1];
        g->tri_cap = outv[3];
        g->info.probes = outv[2];
        g->info.sigma_max = (int32_t)outv[4];
        g->enum_bytes = 4 * outv[0] + 8 * (int64_t)S;
        span.add_bytes(4 * outv[0] + 17 * g->ntri);
        // (tri_cap itself, whole chunks, differs from run to run)
        listed_liveness(g, live, cap, (g->ntri + ends + 31) & ~int64_t(31), s);
    } else {
        const int64_t ntri = g->ntri;
        g->tri_cap = ntri;
        g->tri = graph_alloc<int4>(g, ntri, s);
        g->tri_off = probe_map ? graph_alloc<int64_t>(g, ntri + 1, s) : nullptr;
        if (S > 0) {
            // the listing pass merges the same lists and writes 16 + 8 B per triangle
            StageSpan span(ST_TRIANGLES, s, g->enum_bytes + (probe_map ? 24 : 16) * ntri);
            if (probe_map)
                FOLTY_LAUNCH(k_tri_write<true>, grid_for(S, TRI_THREADS), TRI_THREADS, 0, s, outptr, out_nbr, out_eid,
                             out_src, osig, S, toff, pcnt, g->tri, g->tri_off, g->common, g->tune.tri_heavy);
            else
                FOLTY_LAUNCH(k_tri_write<false>, grid_for(S, TRI_THREADS), TRI_THREADS, 0, s, outptr, out_nbr,
                             out_eid, out_src, osig, S, toff, pcnt, g->tri, g->tri_off, g->common, g->tune.tri_heavy);
        }
        // the probe offsets of the triangles come from the writing pass; the last entry is the total
        if (probe_map)
            FOLTY_CUDA(cudaMemcpyAsync(g->tri_off + ntri, pcnt + S, sizeof(int64_t), cudaMemcpyDeviceToDevice, s));
        if (ids) {
            side.join();
            sort_check(g, s);  // the store's sort completed before its arrays index anything
        } else {
            build_run_ends(g, s);
        }
        prepare_liveness(g, s);
        ensure_liveness(g, FOLTY_DIR_OUT, s);
    }
    g->info.triangles = g->ntri;
    // tile -> first triangle map of the all-roles probe kernel (query independent)
    g->n_tiles = probe_map ? (g->info.probes + PB_TILE - 1) / PB_TILE : 0;
    g->tile_tri = probe_map ? graph_alloc<int64_t>(g, g->n_tiles + 1, s) : nullptr;
    if (probe_map && g->info.probes > 0)
        FOLTY_LAUNCH(k_tile_starts, grid_for(g->n_tiles + 1, T), T, 0, s, g->tri_off, g->ntri, g->info.probes,
                     g->n_tiles, PB_TILE, g->tile_tri);
    g->prof_bytes = graph_alloc<unsigned long long>(g, PROF_SLOTS, s);
    // after the last step that can fail: a call that ran out of memory may be repeated
    release_input(g, s);
    g->info.static_edges = S;
    g->state = 1;
    FOLTY_CUDA(cudaStreamSynchronize(s));
}

// Preprocessing runs on a stream of the device's highest priority, forked from the
// caller's stream and joined back at the end. The temporal store runs beside it on a stream
// of default priority (its kernels take one block per chunk of work, so their blocks retire
// quickly), and the chain that decides the preprocessing's length takes SMs first whenever
// blocks retire: measured with events on the paper-scale graph, the orientation otherwise
// waited behind the store's kernels for ≈ 1 ms.
//
// A call that fails leaves the graph as the load did, so that it may be repeated: what the
// call had allocated goes (its side streams are drained by then), and no mark of it stays.
void preprocess_graph(folty_graph* g, cudaStream_t s) {
    const size_t had = g->owned->size();
    try {
        SideStream pri(s, true);
        preprocess_on(g, pri.fork());
        pri.join();
    } catch (...) {
        if (g->state == 0) {
            while (g->owned->size() > had) graph_release(g, g->owned->back().first, s);
            g->perm = nullptr;
            g->cw = nullptr;
            for (auto& ready : g->live_ready) ready = 0;
        }
        throw;
    }
}

}  // namespace folty

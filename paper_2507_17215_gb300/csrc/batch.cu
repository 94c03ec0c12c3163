// Batched queries sharing the window probes.
//
// For a fixed (temporal edge e, witness w, direction variant) the searched t2 and t3
// of Theorem 3.1 do not depend on delta, so hit(delta) <=> g(e, w) = t3 - t <= delta.
// One selection per direction variant therefore serves every delta of that variant
// (live.cu, roles kept for the largest delta): a first probe pass marks the edges with a
// hit, which get the rows of a compact bin matrix in sorted order, and a second pass bins g
// by the sorted distinct deltas D (bin j = first D_j >= g) in the marked edges' rows; a
// prefix over a row gives c_e(D_j) = #{w : g(e, w) <= D_j} for all j at once. Quantifier,
// rho and universe only enter the threshold (Definition 1.1; Algorithm 5), so one pass over
// the rows answers every query of the variant (k_batch_threshold); the solution pairs of
// all queries are appended as (query, rank of the pair in (u, v) order) keys and sorted
// once, or whenever their buffer is full (BatchSolutions). Queries that also want per-edge counts, certificates or vertex solutions take the
// single-query threshold path on the prefix-summed rows instead. When the rows of all
// deltas do not fit in the memory budget, the deltas are cut into chunks, one binning pass
// per chunk (bin 0 of a chunk also holds every smaller gap).
//
// Probing twice costs one short pass (hits are few and found from the shortest lists); the
// matrix with a row per temporal edge that it replaced took 3.5 GB to clear for 256
// queries on 20M edges, of which 50,000 edges a variant have a hit.
#include <algorithm>
#include <cstdlib>
#include <cstring>
#include <optional>

#include "internal.cuh"
#include "probe.cuh"

namespace folty {

constexpr int BATCH_MAX_BINS = 1024;

// Rows of the marked edges: ebits has a bit per sorted edge, wpref[w] the marked edges
// before word w. Row i belongs to the i-th marked edge; its kstride bins are contiguous (k
// used, the rest zero).

__global__ void k_word_counts(const uint32_t* __restrict__ ebits, int64_t nw, int32_t* __restrict__ cnt) {
    for (int64_t w = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; w < nw; w += (int64_t)gridDim.x * blockDim.x)
        cnt[w] = __popc(ebits[w]);
}

// cpos[i], csd[i]: sorted position and pair key (2 * static edge + direction) of row i.
__global__ void k_row_edges(const uint32_t* __restrict__ ebits, const int32_t* __restrict__ wpref, int64_t nw,
                            const int32_t* __restrict__ sd, int32_t* __restrict__ cpos, int32_t* __restrict__ csd) {
    for (int64_t w = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; w < nw; w += (int64_t)gridDim.x * blockDim.x) {
        int32_t i = wpref[w];
        for (uint32_t word = ebits[w]; word; word &= word - 1, i++) {
            const int32_t pos = (int32_t)(32 * w) + __ffs((int)word) - 1;
            cpos[i] = pos;
            csd[i] = sd[pos];
        }
    }
}

// out[pos] = c_e(D_j) of the marked edges, the prefix of their rows up to bin j (out is zero
// elsewhere): the counts of one window, for a query that wants per-edge outputs.
template <typename C>
__global__ void k_bins_column(const C* __restrict__ bins, int kstride, int j, int64_t rows,
                              const int32_t* __restrict__ cpos, C* __restrict__ out) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < rows; i += (int64_t)gridDim.x * blockDim.x) {
        const C* row = bins + i * kstride;
        uint32_t run = 0;
        for (int b = 0; b <= j; b++) run += row[b];
        out[cpos[i]] = (C)run;
    }
}

// ------------------------------------------------------------------ pair ranks

__device__ __forceinline__ int64_t lower_bound_pair(const int32_t* __restrict__ ka, const int32_t* __restrict__ kb,
                                                    const int32_t* __restrict__ idx, int64_t n, int32_t x, int32_t y) {
    int64_t lo = 0;
    while (n > 0) {
        const int64_t half = n >> 1;
        const int32_t i = idx ? idx[lo + half] : (int32_t)(lo + half);
        if (ka[i] < x || (ka[i] == x && kb[i] < y)) {
            lo += half + 1;
            n -= half + 1;
        } else {
            n = half;
        }
    }
    return lo;
}

// prank[2s + d] = position of the directed pair (x, y) of static edge s, direction d, in
// the (x, y) order of all directed pairs: pairs x < y are the static edges in (a, b)
// order, pairs x > y the static edges in (b, a) order (by_b); a pair's position is its
// index in its own list plus the number of pairs of the other list before it.
__global__ void k_pair_ranks(const int32_t* __restrict__ ea, const int32_t* __restrict__ eb,
                             const int32_t* __restrict__ by_b, int64_t S, int32_t* __restrict__ prank) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < 2 * S; i += (int64_t)gridDim.x * blockDim.x) {
        if (i < S) {  // (a, b) of static edge i; pairs (b', a') with b' < a, or b' == a and a' < b, precede it
            prank[2 * i] = (int32_t)(i + lower_bound_pair(eb, ea, by_b, S, ea[i], eb[i]));
        } else {  // (b, a) of static edge by_b[j]
            const int64_t j = i - S;
            const int32_t s = by_b[j];
            prank[2 * (int64_t)s + 1] = (int32_t)(j + lower_bound_pair(ea, eb, nullptr, S, eb[s], ea[s]));
        }
    }
}

static const int32_t* pair_ranks(folty_graph* g, cudaStream_t s) {
    if (!g->prank) {
        g->prank = graph_alloc<int32_t>(g, 2 * (int64_t)g->S, s);
        if (g->S > 0)
            FOLTY_LAUNCH(k_pair_ranks, grid_for(2 * (int64_t)g->S, 256), 256, 0, s, g->ea, g->eb, g->by_b,
                         (int64_t)g->S, g->prank);
    }
    return g->prank;
}

// ------------------------------------------------------------------ fused threshold

constexpr int BT_THREADS = 128;
constexpr int BT_WARPS = BT_THREADS / 32;
constexpr int BT_MAXQ = 256;  // queries of one fused pass
constexpr int BT_CHUNKS = 4;  // 16-byte chunks of an edge's bins loaded together per lane
constexpr int BT_WARP_ROWS = 4;  // rows per warp at least
// bins of one fused pass (their prefix sums sit in shared memory, per warp and lane)
constexpr int BT_KMAX = 128;

// Entries between consecutive bins of the prefix sums in shared memory, so that lanes that
// read different bins of one edge hit different banks (17 and 33 words).
template <typename C>
struct BatchStride;
template <>
struct BatchStride<uint16_t> {
    static constexpr int value = 34;
};
template <>
struct BatchStride<int32_t> {
    static constexpr int value = 33;
};

// One query of a fused pass (rho irrelevant to the existential quantifier).
struct BatchQuery {
    int32_t j;     // bin of its delta
    int32_t slot;  // index among the batch's queries (high bits of its output keys)
    int32_t quant, universe;
    int64_t num, den;
};

struct BatchArgs {
    const void* bins;  // C[rows][kstride], k bins used per row
    int k, kstride;
    int64_t rows;
    const int32_t* csd;      // pair key of every row's edge
    const uint32_t* ebits;
    const int32_t* wpref;
    const int32_t* seg;  // run bounds in sorted positions: run r = [seg[r], seg[r + 1])
    const int32_t* ea;
    const int32_t* eb;
    const int32_t* deg;
    const int32_t* common;
    const int32_t* prank;
    const BatchQuery* qs;
    int nq;
    int rb;  // bits of a pair rank
    int64_t per_warp;
    int64_t cap;
    unsigned long long* n_out;
    uint64_t* out_key;  // (slot << rb) | pair rank
    int32_t* out_run;   // the pair's run id 2s + d
    int32_t* out_cnt;   // max c_e over the pair's edges
    int32_t* out_nc;    // certificates among them
};

// x rounded up to the next row that starts a directed pair (a pair's rows are contiguous).
__device__ __forceinline__ int64_t pair_aligned(const BatchArgs& a, int64_t x) {
    if (x <= 0) return 0;
    if (x >= a.rows) return a.rows;
    const int32_t r = a.csd[x];
    return a.csd[x - 1] != r ? x : (int64_t)row_of(a.ebits, a.wpref, a.seg[r + 1]);
}

// Appends the pairs of the lanes with emit set (one atomic per warp).
__device__ __forceinline__ void emit_pairs(const BatchArgs& a, bool emit, int slot, int32_t r, int32_t cnt, int32_t nc) {
    const unsigned em = __ballot_sync(0xffffffffu, emit);
    if (!em) return;
    const int lane = threadIdx.x & 31;
    const int first = __ffs(em) - 1;
    unsigned long long base = 0;
    if (lane == first) base = atomicAdd(a.n_out, (unsigned long long)__popc(em));
    base = __shfl_sync(0xffffffffu, base, first);
    if (emit) {
        const unsigned long long i = base + __popc(em & ((1u << lane) - 1u));
        if (i < (unsigned long long)a.cap) {
            a.out_key[i] = ((uint64_t)slot << a.rb) | (uint64_t)(uint32_t)a.prank[r];
            a.out_run[i] = r;
            a.out_cnt[i] = cnt;
            a.out_nc[i] = nc;
        }
    }
}

// Prefix sums c_e(D_j) of the bins of one lane's row into pref[j * stride + lane],
// BT_CHUNKS 16-byte loads in flight together; returns c_e(D_{k-1}).
template <typename C>
__device__ __forceinline__ uint32_t bin_prefix(const C* __restrict__ bins, int kstride, int k, int64_t row, C* pref) {
    constexpr int PER = 16 / sizeof(C);  // bins per 16-byte chunk of a row
    constexpr int STRIDE = BatchStride<C>::value;
    const int lane = threadIdx.x & 31;
    const uint4* src = reinterpret_cast<const uint4*>(bins + row * (int64_t)kstride);
    const int nch = (k + PER - 1) / PER;
    uint32_t run = 0;
    for (int c0 = 0; c0 < nch; c0 += BT_CHUNKS) {
        uint4 w[BT_CHUNKS];
#pragma unroll
        for (int u = 0; u < BT_CHUNKS; u++) w[u] = c0 + u < nch ? __ldcs(src + c0 + u) : make_uint4(0, 0, 0, 0);
#pragma unroll
        for (int u = 0; u < BT_CHUNKS; u++) {
            const uint32_t ws[4] = {w[u].x, w[u].y, w[u].z, w[u].w};
#pragma unroll
            for (int i = 0; i < PER; i++) {
                const int j = (c0 + u) * PER + i;
                run += sizeof(C) == 2 ? (ws[i >> 1] >> (16 * (i & 1))) & 0xffffu : ws[i & 3];
                if (j < k) pref[j * STRIDE + lane] = (C)run;
            }
        }
    }
    return run;
}

// Every warp takes a contiguous range of rows whose ends are moved to pair starts, and
// walks it in windows of 32 rows. The lanes put the prefix sums of one row each into shared
// memory; then, for the rows of each pair in the window (a segment), the lanes are the
// pass's queries: a lane whose query can certify at the pair's largest count walks the
// segment's rows at its own bin, counts the certifying ones (Definition 1.1: c >= 1, and for
// forall_rho c * den >= num * U) and keeps the largest count, which certifies whenever any
// does, as a pair's edges share the universe. A pair that continues into the next window
// leaves its totals per query in shared memory.
//
// The lanes were the rows before, with two warp reductions per query and pair: a reduction
// is issued once per pair of the window, 470 us a variant for 85 queries on 20M edges
// (whose rows were also skipped group by group); now 18 us.
template <typename C>
__global__ void __launch_bounds__(BT_THREADS) k_batch_threshold(const BatchArgs a) {
    constexpr int STRIDE = BatchStride<C>::value;
    extern __shared__ __align__(16) unsigned char bt_smem[];
    BatchQuery* sq = reinterpret_cast<BatchQuery*>(bt_smem);
    int32_t* lmax = reinterpret_cast<int32_t*>(sq + a.nq);   // [BT_WARPS][nq]
    int32_t* lnc = lmax + BT_WARPS * a.nq;                   // [BT_WARPS][nq]
    C* prefs = reinterpret_cast<C*>(lnc + BT_WARPS * a.nq);  // [BT_WARPS][k][STRIDE]
    for (int i = threadIdx.x; i < a.nq; i += blockDim.x) sq[i] = a.qs[i];
    __syncthreads();
    const C* bins = static_cast<const C*>(a.bins);
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    C* pref = prefs + (int64_t)wib * a.k * STRIDE;
    int32_t* wmax = lmax + wib * a.nq;
    int32_t* wnc = lnc + wib * a.nq;
    const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t lo = pair_aligned(a, warp * a.per_warp), hi = pair_aligned(a, (warp + 1) * a.per_warp);
    bool open = false;  // the last window's last pair continues
    for (int64_t p = lo; p < hi; p += 32) {
        const int L = (int)min(hi - p, (int64_t)32);
        const bool on = lane < L;
        const int32_t key = on ? a.csd[p + lane] : -1;
        const int32_t after = p + L < hi ? a.csd[p + L] : -1;
        uint32_t cmax = 0;
        if (on) cmax = bin_prefix<C>(bins, a.kstride, a.k, p + lane, pref);
        const int32_t prev = __shfl_up_sync(0xffffffffu, key, 1);
        const bool head = on && (lane == 0 || key != prev);
        int32_t uh = 0, ut = 0, uc = 0;  // |N(x)|, |N(y)|, |N(x) cap N(y)| of the head's pair
        if (head) {
            const int32_t s = key >> 1;
            const int32_t x = (key & 1) ? a.eb[s] : a.ea[s], y = (key & 1) ? a.ea[s] : a.eb[s];
            uh = a.deg[x];
            ut = a.deg[y];
            uc = a.common[s];
        }
        unsigned heads = __ballot_sync(0xffffffffu, head);
        __syncwarp();
        while (heads) {
            const int h = __ffs(heads) - 1;
            heads &= heads - 1;
            const int e = heads ? __ffs(heads) - 1 : L;  // the segment's rows: lanes [h, e)
            const int32_t r = __shfl_sync(0xffffffffu, key, h);
            const int32_t su[3] = {__shfl_sync(0xffffffffu, uh, h), __shfl_sync(0xffffffffu, ut, h),
                                   __shfl_sync(0xffffffffu, uc, h)};
            const int64_t cm = (int64_t)__reduce_max_sync(0xffffffffu, lane >= h && lane < e ? cmax : 0u);
            const bool cont = open && h == 0;
            const bool closes = e < L || after != r;
            for (int q0 = 0; q0 < a.nq; q0 += 32) {
                const int qi = q0 + lane;
                const BatchQuery q = sq[min(qi, a.nq - 1)];
                const bool ex = q.quant == FOLTY_Q_EXISTS;
                const int64_t need = q.num * (int64_t)(q.universe == FOLTY_U_HEAD   ? su[0]
                                                       : q.universe == FOLTY_U_TAIL ? su[1]
                                                                                    : su[2]);
                const bool can = qi < a.nq && cm >= 1 && (ex || cm * q.den >= need);
                int32_t mx = 0, n = 0;
                if (cont && qi < a.nq) {
                    mx = wmax[qi];
                    n = wnc[qi];
                }
                if (can) {
                    const C* col = pref + q.j * STRIDE;
                    for (int i = h; i < e; i++) {
                        const int32_t c = (int32_t)col[i];
                        if (c >= 1 && (ex || (int64_t)c * q.den >= need)) {
                            n++;
                            mx = max(mx, c);
                        }
                    }
                }
                if (closes) {
                    emit_pairs(a, n > 0, q.slot, r, mx, n);
                } else if (qi < a.nq) {
                    wmax[qi] = mx;
                    wnc[qi] = n;
                }
            }
        }
        // the last segment ends the window: it continues when the next window starts with its pair
        open = __shfl_sync(0xffffffffu, key, L - 1) == after;
        __syncwarp();
    }
}

// Sorted solutions -> out = [u... | v... | count... | ncert...]; qstart[slot] = first
// index of the slot's solutions (left at -1 for a slot without any).
__global__ void k_batch_gather(const uint64_t* __restrict__ key, const uint32_t* __restrict__ order,
                               const int32_t* __restrict__ run, const int32_t* __restrict__ cnt,
                               const int32_t* __restrict__ nc, const int32_t* __restrict__ ea,
                               const int32_t* __restrict__ eb, int64_t n, int rb, int32_t* __restrict__ out,
                               int32_t* __restrict__ qstart) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t o = order[i];
        const int32_t r = run[o], s = r >> 1;
        out[i] = (r & 1) ? eb[s] : ea[s];
        out[n + i] = (r & 1) ? ea[s] : eb[s];
        out[2 * n + i] = cnt[o];
        out[3 * n + i] = nc[o];
        const int q = (int)(key[i] >> rb);
        if (i == 0 || (int)(key[i - 1] >> rb) != q) qstart[q] = (int32_t)i;
    }
}

__global__ void k_iota_u32(uint32_t* __restrict__ a, int64_t n) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        a[i] = (uint32_t)i;
}

// ------------------------------------------------------------------ host side

static int64_t batch_bin_budget_bytes() {
    size_t free_b = 0, total_b = 0;
    if (cudaMemGetInfo(&free_b, &total_b) != cudaSuccess) {
        cudaGetLastError();
        return (int64_t)1 << 30;
    }
    int64_t b = (int64_t)(free_b / 4);
    const int64_t cap = (int64_t)16 << 30;
    return b < cap ? b : cap;
}

static bool plain_query(const folty_query_params& q) {
    return !q.want_edge_counts && !q.want_certificates && !q.outer && !q.want_triples;
}

// Solution buffer entries of a batch: key, alternate key, run, count, certificates, two
// sort values (36 B each).
constexpr int64_t BT_ENTRY_BYTES = 36;
constexpr int64_t BT_DEFAULT_CAP = int64_t(1) << 22;

// Bins of one probe pass: the largest number of distinct deltas of one direction variant.
int64_t batch_footprint(const folty_graph* g, const folty_query_params* qs, int nq, int64_t* bins_part) {
    int64_t kmax = 0;
    for (int dir = 0; dir <= FOLTY_DIR_EITHER; dir++) {
        std::vector<int64_t> D;
        for (int i = 0; i < nq; i++)
            if (qs[i].dir == dir) D.push_back(qs[i].delta);
        std::sort(D.begin(), D.end());
        D.erase(std::unique(D.begin(), D.end()), D.end());
        kmax = std::max<int64_t>(kmax, (int64_t)D.size());
    }
    kmax = std::min<int64_t>(kmax, BATCH_MAX_BINS);
    // a row, a position and a key per edge at most (rows padded to 16 bytes), and the edge
    // bits with their prefix
    const int64_t bins = ((kmax + 7) & ~int64_t(7)) * g->m_kept * 4;
    const int64_t marks = 8 * g->m_kept + g->m_kept / 4;
    // the fused pass: its solution buffer and the pair ranks
    int64_t fused = 0;
    bool any_plain = false;
    for (int i = 0; i < nq; i++) any_plain = any_plain || plain_query(qs[i]);
    if (any_plain) fused = BT_DEFAULT_CAP * BT_ENTRY_BYTES + 4 * 2 * (int64_t)g->S;
    // output stage per query of a read-back group of the single-query path (see
    // finish_queries): 6 int32 arrays of 2S + 1, compacted keys, packed output, edge counts
    // when asked
    const int64_t n2 = 2 * (int64_t)g->S;
    int64_t per_q = 6 * 4 * (n2 + 1) + 8 * n2 + 16 * n2 + 64;
    bool edges = false, certs = false, outer = false, other = false;
    for (int i = 0; i < nq; i++) {
        edges = edges || qs[i].want_edge_counts;
        certs = certs || qs[i].want_certificates;
        outer = outer || qs[i].outer;
        other = other || (!plain_query(qs[i]) && !qs[i].want_triples);
    }
    if (edges) per_q += 4 * g->m;
    if (other) per_q += 4 * g->m_kept;  // the query's counts gathered from the bin rows
    if (certs) per_q += 16 * (g->m + 1);
    if (outer) per_q += 14 * ((int64_t)g->n + 1);
    const int64_t group = other ? std::min<int64_t>(nq, READBACK_MAX / 4) : 0;
    // a triple query runs alone: role flags and scan (9 B per role), and up to one triple
    // per role through the two sorts (44 B each), on top of its own counters
    bool triples = false;
    for (int i = 0; i < nq; i++) triples = triples || qs[i].want_triples;
    const int64_t tri_part = triples ? 53 * 6 * g->tri_cap + 4 * g->m_kept + per_q : 0;
    if (bins_part) *bins_part = bins;
    return std::max(bins + marks + fused + group * per_q, tri_part);
}

// The solutions of a batch's plain queries, appended by every fused pass.
struct BatchOutput {
    int64_t cap = 0;
    unsigned long long* n_out = nullptr;
    uint64_t* key = nullptr;
    int32_t* run = nullptr;
    int32_t* cnt = nullptr;
    int32_t* nc = nullptr;
    int rb = 0;  // bits of a pair rank
};

// The rows of one direction variant's marked edges.
struct BatchRows {
    int64_t rows = 0;
    uint32_t* ebits = nullptr;  // [nw + 1]
    int32_t* wpref = nullptr;   // [nw + 1]
    int32_t* cpos = nullptr;
    int32_t* csd = nullptr;
};

// Small host values on their way to the device: through the graph's pinned pair stage, each
// at its own place, so that no copy reads a place written again meanwhile (a full stage
// waits for the copies so far). Nothing else uses the stage between the stream's last
// synchronisation before this object and its last upload.
class StageUpload {
  public:
    StageUpload(folty_graph* g, cudaStream_t s) : g_(g), s_(s) {}
    void operator()(void* dst, const void* src, size_t bytes) {
        constexpr size_t cap = sizeof(int32_t) * 4 * (size_t)PAIR_STAGE;
        if (off_ + bytes > cap) {
            FOLTY_CUDA(cudaStreamSynchronize(s_));
            off_ = 0;
        }
        char* at = (char*)(g_->host_stage + HOST_STAGE) + off_;
        std::memcpy(at, src, bytes);
        g_->stage_busy = 1;
        FOLTY_CUDA(cudaMemcpyAsync(dst, at, bytes, cudaMemcpyHostToDevice, s_));
        off_ += (bytes + 63) & ~size_t(63);
    }
    void reset() { off_ = 0; }  // after a synchronisation

  private:
    folty_graph* g_;
    cudaStream_t s_;
    size_t off_ = 0;
};
static_assert(BATCH_MAX_BINS * sizeof(int64_t) <= 4 * PAIR_STAGE * sizeof(int32_t), "bin bounds fit the pair stage");

// The fused threshold of the plain queries `hq` (at most BT_MAXQ) over the bins of one
// probe pass: their solutions into out.
template <typename C>
static void fused_threshold(folty_graph* g, const C* bins, const BatchRows& br, int k, int kstride,
                            const std::vector<BatchQuery>& hq, const BatchOutput& out, Scratch& sc, StageUpload& up,
                            cudaStream_t s) {
    const int nq = (int)hq.size();
    if (br.rows == 0) return;
    BatchQuery* dq = sc.get<BatchQuery>(nq);
    up(dq, hq.data(), sizeof(BatchQuery) * (size_t)nq);
    // shared memory: queries, per-warp totals of an open pair, per-warp prefix sums
    const size_t smem = sizeof(BatchQuery) * (size_t)nq + 2 * sizeof(int32_t) * BT_WARPS * (size_t)nq +
                        sizeof(C) * BT_WARPS * BatchStride<C>::value * (size_t)k;
    // the attribute is the kernel's, shared by every thread: always the same bound (the
    // largest pass: BT_KMAX 16-bit or BT_KMAX / 2 32-bit bins), so that concurrent batches
    // (a server's workers) never lower it under one another's launch
    constexpr size_t smem_max = (sizeof(BatchQuery) + 2 * sizeof(int32_t) * BT_WARPS) * BT_MAXQ +
                                2 * BT_WARPS * BatchStride<uint16_t>::value * BT_KMAX;
    if (smem > smem_max) fail(FOLTY_EINVAL, "batched threshold: too many bins or queries for one pass");
    FOLTY_CUDA(cudaFuncSetAttribute(k_batch_threshold<C>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_max));
    int per_sm = 0;
    FOLTY_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_batch_threshold<C>, BT_THREADS, smem));
    // few rows per warp while that gives every resident warp some: a window's pairs are worked
    // off one after another (12,700 rows of 85 queries: 40 us at 32 rows a warp, 18 us at 4)
    const int64_t most = (int64_t)num_sms() * (per_sm > 0 ? per_sm : 1);
    const int64_t blocks = std::min<int64_t>(most, (br.rows + BT_WARP_ROWS * BT_WARPS - 1) / (BT_WARP_ROWS * BT_WARPS));
    const int64_t nwarps = blocks * BT_WARPS;
    BatchArgs a{};
    a.bins = bins;
    a.k = k;
    a.kstride = kstride;
    a.rows = br.rows;
    a.csd = br.csd;
    a.ebits = br.ebits;
    a.wpref = br.wpref;
    a.seg = g->seg;
    a.ea = g->ea;
    a.eb = g->eb;
    a.deg = g->deg;
    a.common = g->common;
    a.prank = pair_ranks(g, s);
    a.qs = dq;
    a.nq = nq;
    a.rb = out.rb;
    a.per_warp = (br.rows + nwarps - 1) / nwarps;
    a.cap = out.cap;
    a.n_out = out.n_out;
    a.out_key = out.key;
    a.out_run = out.run;
    a.out_cnt = out.cnt;
    a.out_nc = out.nc;
    // model bytes: every row and its pair key
    StageSpan span(ST_BATCH, s, br.rows * ((int64_t)kstride * (int64_t)sizeof(C) + 4));
    FOLTY_LAUNCH(k_batch_threshold<C>, (unsigned)blocks, BT_THREADS, smem, s, a);
}

// The results of the queries of `slots` from their n < 2^31 solutions: sorted by (query, pair
// rank), gathered into per-query (u, v, count, ncert), copied out. slot i is the query plain[i].
static void batch_results(folty_graph* g, const BatchOutput& out, int64_t n, const std::vector<int>& slots,
                          const std::vector<int>& plain, folty_result* outs, cudaStream_t s) {
    const int nq = (int)plain.size();
    Scratch so(g->alloc, s, g->dev_err);
    std::vector<int32_t> qstart((size_t)nq + 1, -1);
    std::vector<int32_t> host;
    const int32_t* packed_h = nullptr;
    if (n > 0) {
        uint64_t* kalt = so.get<uint64_t>(n);
        uint32_t* v0 = so.get<uint32_t>(n);
        uint32_t* v1 = so.get<uint32_t>(n);
        int32_t* packed = so.get<int32_t>(4 * n + nq + 1);
        int32_t* qs_dev = packed + 4 * n;
        FOLTY_LAUNCH(k_iota_u32, grid_for(n, 256), 256, 0, s, v0, n);
        const int bits = out.rb + bit_length((uint64_t)(nq > 1 ? nq - 1 : 1));
        const bool alt = radix_sort_pairs(so, out.key, kalt, v0, v1, n, bits);
        read_back(g, nullptr, nullptr, 0, nullptr, s);  // the sort's look-backs completed
        const uint64_t* ks = alt ? kalt : out.key;
        const uint32_t* ord = alt ? v1 : v0;
        FOLTY_CUDA(cudaMemsetAsync(qs_dev, 0xff, sizeof(int32_t) * (size_t)(nq + 1), s));
        FOLTY_LAUNCH(k_batch_gather, grid_for(n, 256), 256, 0, s, ks, ord, out.run, out.cnt, out.nc, g->ea, g->eb, n,
                     out.rb, packed, qs_dev);
        const size_t bytes = sizeof(int32_t) * (size_t)(4 * n + nq);
        if (bytes <= sizeof(int32_t) * 4 * (size_t)PAIR_STAGE) {
            g->stage_busy = 1;
            FOLTY_CUDA(cudaMemcpyAsync(g->pair_stage, packed, bytes, cudaMemcpyDeviceToHost, s));
            FOLTY_CUDA(cudaStreamSynchronize(s));
            g->stage_busy = 0;
            packed_h = (const int32_t*)(g->host_stage + HOST_STAGE);
        } else {
            host.resize(4 * (size_t)n + (size_t)nq);
            FOLTY_CUDA(cudaMemcpyAsync(host.data(), packed, bytes, cudaMemcpyDeviceToHost, s));
            FOLTY_CUDA(cudaStreamSynchronize(s));
            packed_h = host.data();
        }
        std::memcpy(qstart.data(), packed_h + 4 * n, sizeof(int32_t) * (size_t)nq);
    }
    qstart[(size_t)nq] = (int32_t)n;
    // the end of a slot's solutions is the next slot's start (slots without any are -1)
    for (int i = nq - 1; i >= 0; i--) {
        if (qstart[(size_t)i] < 0) qstart[(size_t)i] = qstart[(size_t)i + 1];
    }
    for (int i : slots) {
        const int64_t b = qstart[(size_t)i], e = qstart[(size_t)i + 1], np = e - b;
        folty_result* r = &outs[plain[(size_t)i]];
        fill_result_host(r, np, g->m, false, 0, false, 0, false);
        int64_t ncert = 0;
        if (np > 0) {
            std::memcpy(r->u, packed_h + b, sizeof(int32_t) * (size_t)np);
            std::memcpy(r->v, packed_h + n + b, sizeof(int32_t) * (size_t)np);
            std::memcpy(r->count, packed_h + 2 * n + b, sizeof(int32_t) * (size_t)np);
            std::memcpy(r->ncert, packed_h + 3 * n + b, sizeof(int32_t) * (size_t)np);
            for (int64_t x = 0; x < np; x++) ncert += r->ncert[x];
        }
        r->n_cert_edges = ncert;
    }
}

// The solutions of a batch's plain queries. Fused passes append theirs to one buffer, so that
// an ordinary batch is sorted and copied out once; when the buffer cannot take a pass's, the
// queries before it get their results first, and that pass's threshold runs again with room
// for all of them. So the memory is that of one pass (at most BT_MAXQ queries), not of the
// batch, and fewer than 2^31 solutions are in the buffer at a time.
constexpr int64_t BT_MAX_SOLUTIONS = 0x7fffffff;

class BatchSolutions {
  public:
    BatchSolutions(folty_graph* g, const std::vector<int>& plain, folty_result* outs, int64_t cap, cudaStream_t s)
        : g_(g), plain_(plain), outs_(outs), s_(s) {
        out_.rb = bit_length((uint64_t)(g->S > 0 ? 2 * (int64_t)g->S - 1 : 1));
        if (!plain.empty()) reserve(cap);
    }

    // The buffer's solution count on the device, for a read-back the caller makes anyway, and
    // its value. Null without plain queries.
    const unsigned long long* counter() const { return out_.n_out; }
    void counted(int64_t n) {
        n_ = n;
        exact_ = true;
    }

    // The queries of one fused pass, which has at most `most` solutions: launch(out) appends.
    template <typename Launch>
    void pass(const std::vector<BatchQuery>& hq, int64_t most, Launch&& launch) {
        if (n_ + most > out_.cap) count();
        const int64_t before = n_;
        launch(out_);
        n_ += most;
        exact_ = most == 0 && exact_;
        if (n_ > out_.cap) {
            count();
            if (n_ > out_.cap) {
                const int64_t mine = n_ - before;
                results(before);
                if (mine > out_.cap) reserve(mine);
                launch(out_);
                counted(mine);
            }
        }
        for (const BatchQuery& q : hq) slots_.push_back(q.slot);
    }

    void finish() {
        if (plain_.empty()) return;
        count();
        results(n_);
    }

  private:
    void clear() {
        FOLTY_CUDA(cudaMemsetAsync(out_.n_out, 0, sizeof(unsigned long long), s_));
        counted(0);
    }
    void count() {
        if (!exact_) counted(read_i64(g_, (const int64_t*)out_.n_out, s_));
    }
    void reserve(int64_t cap) {
        buf_.reset();
        buf_.emplace(g_->alloc, s_, g_->dev_err);
        out_.cap = cap;
        out_.n_out = buf_->get<unsigned long long>(1);
        out_.key = buf_->get<uint64_t>(cap);
        out_.run = buf_->get<int32_t>(cap);
        out_.cnt = buf_->get<int32_t>(cap);
        out_.nc = buf_->get<int32_t>(cap);
        clear();
    }
    void results(int64_t n) {
        if (!slots_.empty()) batch_results(g_, out_, n, slots_, plain_, outs_, s_);
        slots_.clear();
        clear();
    }

    folty_graph* g_;
    const std::vector<int>& plain_;
    folty_result* outs_;
    cudaStream_t s_;
    std::optional<Scratch> buf_;
    BatchOutput out_;
    std::vector<int> slots_;  // queries whose solutions are in the buffer
    int64_t n_ = 0;           // the buffer's solutions, or a bound on them
    bool exact_ = false;
};

// Queries of one direction variant and their sorted distinct windows.
struct BatchPass {
    int dir;
    std::vector<int> members;
    std::vector<int64_t> D;
};

// Without a budget of the caller's, rows of up to this size are allocated without asking how
// much memory is free.
constexpr int64_t BT_SMALL_ROWS = int64_t(256) << 20;

// Bins of a row of k windows: whole 16-byte chunks of csize-byte counts.
static int64_t row_stride(int64_t k, int64_t csize) {
    const int64_t unit = 16 / csize;
    return (k + unit - 1) / unit * unit;
}

// Windows per chunk, at most `most`: as many as fit the budget with their padding, a 16-byte
// chunk at least.
static int64_t chunk_windows(int64_t most, int64_t rows, int64_t csize, int64_t budget) {
    if (rows == 0 || (budget <= 0 && rows * csize * row_stride(most, csize) <= BT_SMALL_ROWS)) return most;
    if (budget <= 0) budget = batch_bin_budget_bytes();
    return std::min<int64_t>(most, std::max<int64_t>(1, budget / (16 * rows)) * (16 / csize));
}

// One direction variant: selection, marks, rows and, per chunk of windows, the bins, the
// plain queries' solutions (slot[i] = their index among the plain queries, -1 for others)
// and the results of the queries with per-edge outputs.
static void run_batch_pass(folty_graph* g, const folty_query_params* qs, const BatchPass& ps, const std::vector<int>& slot,
                           BatchSolutions& sol, folty_result* outs, cudaStream_t s, int64_t bin_budget) {
    const int64_t mk = g->m_kept;
    // 16-bit bins while no count can reach 2^16 (a count is at most the number of common
    // neighbours of an edge's ends, at most the largest degree): half the memory traffic
    // of the bins and of the threshold's reads
    const bool b16 = g->info.max_degree < 65535;
    const int64_t csize = b16 ? (int64_t)sizeof(uint16_t) : (int64_t)sizeof(int32_t);
    Scratch sc(g->alloc, s, g->dev_err);
    BatchRows br;
    const int64_t nw = (mk + 31) / 32;
    ProbeBuffers pb{};
    const bool probes = mk > 0 && g->ntri > 0 && g->info.probes > 0;
    if (probes) {
        br.ebits = sc.get<uint32_t>(nw + 1);
        br.wpref = sc.get<int32_t>(nw + 1);
        FOLTY_CUDA(cudaMemsetAsync(br.ebits, 0, sizeof(uint32_t) * (size_t)(nw + 1), s));
        pb = select_probes(g, ps.D.back(), ps.dir, sc, s);
        launch_marks(g, ps.D.back(), ps.dir, pb, br.ebits, s);
        FOLTY_LAUNCH(k_word_counts, grid_for(nw, 256), 256, 0, s, br.ebits, nw, br.wpref);
        exclusive_scan(sc, br.wpref, br.wpref, nw);
        const void* ptrs[2] = {br.wpref + nw, sol.counter()};
        const int sizes[2] = {4, 8};
        int64_t v[2];
        read_back(g, ptrs, sizes, sol.counter() ? 2 : 1, v, s);
        br.rows = v[0];
        if (sol.counter()) sol.counted(v[1]);
    }
    if (br.rows > 0) {
        br.cpos = sc.get<int32_t>(br.rows);
        br.csd = sc.get<int32_t>(br.rows);
        FOLTY_LAUNCH(k_row_edges, grid_for(nw, 256), 256, 0, s, br.ebits, br.wpref, nw, g->sd, br.cpos, br.csd);
    }
    StageUpload up(g, s);  // the read-back above was the stream's last synchronisation
    // windows per chunk: as many bins as the budget holds and, when plain queries are
    // present, as the fused pass's shared memory does
    int64_t chunk = std::min<int64_t>((int64_t)ps.D.size(), BATCH_MAX_BINS);
    bool plain = false;
    for (int i : ps.members) plain = plain || slot[(size_t)i] >= 0;
    if (plain) chunk = std::min<int64_t>(chunk, b16 ? BT_KMAX : BT_KMAX / 2);
    chunk = chunk_windows(chunk, br.rows, csize, bin_budget);
    for (size_t c0 = 0; c0 < ps.D.size(); c0 += (size_t)chunk) {
        const int k = (int)std::min<int64_t>(chunk, (int64_t)ps.D.size() - (int64_t)c0);
        const int kstride = (int)row_stride(k, csize);
        Scratch sk(g->alloc, s, g->dev_err);
        const std::vector<int64_t> hd(ps.D.begin() + (long)c0, ps.D.begin() + (long)c0 + k);
        int32_t* bins = nullptr;
        uint16_t* bins16 = nullptr;
        if (br.rows > 0) {
            // the bin bounds in the store's timestamp type (32-bit offsets: gaps stay
            // below 2^32 - 1, so larger windows behave as 2^32 - 2)
            int64_t* dd = sk.get<int64_t>(k);
            std::vector<uint32_t> h32;
            if (g->ts32)
                for (int64_t d : hd) h32.push_back(d >= 0xfffffffell ? 0xfffffffeu : (uint32_t)d);
            if (g->ts32) up(dd, h32.data(), sizeof(uint32_t) * (size_t)k);
            else up(dd, hd.data(), sizeof(int64_t) * (size_t)k);
            if (b16) bins16 = sk.get<uint16_t>(br.rows * kstride);
            else bins = sk.get<int32_t>(br.rows * kstride);
            FOLTY_CUDA(cudaMemsetAsync(b16 ? (void*)bins16 : (void*)bins, 0, (size_t)(br.rows * kstride * csize), s));
            launch_bins(g, hd[(size_t)k - 1], ps.dir, pb, br.ebits, br.wpref, bins, bins16, k, kstride, dd, s);
        }
        std::vector<BatchQuery> pq;
        std::vector<const folty_query_params*> fq;
        std::vector<CountView> fc;
        std::vector<folty_result*> fo;
        for (int i : ps.members) {
            const folty_query_params& q = qs[i];
            auto it = std::lower_bound(hd.begin(), hd.end(), q.delta);
            if (it == hd.end() || *it != q.delta) continue;  // another chunk
            const int j = (int)(it - hd.begin());
            if (slot[(size_t)i] >= 0) {
                pq.push_back(BatchQuery{j, slot[(size_t)i], (int32_t)q.quant, (int32_t)q.universe, (int64_t)q.rho_num,
                                        (int64_t)q.rho_den});
                continue;
            }
            fq.push_back(&q);
            // the query's counts c_e(D_j), gathered from the rows
            void* col = b16 ? (void*)sk.get<uint16_t>(mk + 2) : (void*)sk.get<int32_t>(mk);
            FOLTY_CUDA(cudaMemsetAsync(col, 0, (size_t)(b16 ? (mk + 2) * 2 : mk * 4), s));
            if (br.rows > 0 && b16)
                FOLTY_LAUNCH(k_bins_column<uint16_t>, grid_for(br.rows, 256), 256, 0, s, bins16, kstride, j, br.rows,
                             br.cpos, (uint16_t*)col);
            else if (br.rows > 0)
                FOLTY_LAUNCH(k_bins_column<int32_t>, grid_for(br.rows, 256), 256, 0, s, bins, kstride, j, br.rows, br.cpos,
                             (int32_t*)col);
            fc.push_back(b16 ? CountView{nullptr, (const uint16_t*)col} : CountView{(const int32_t*)col, nullptr});
            fo.push_back(&outs[i]);
        }
        // a query has at most one solution per row, so this many queries have fewer than 2^31
        const size_t group = (size_t)std::min<int64_t>(BT_MAXQ, BT_MAX_SOLUTIONS / std::max<int64_t>(br.rows, 1));
        for (size_t q0 = 0; q0 < pq.size(); q0 += group) {
            const std::vector<BatchQuery> gq(pq.begin() + (long)q0, pq.begin() + (long)std::min(pq.size(), q0 + group));
            sol.pass(gq, (int64_t)gq.size() * br.rows, [&](const BatchOutput& out) {
                if (b16) fused_threshold<uint16_t>(g, bins16, br, k, kstride, gq, out, sk, up, s);
                else fused_threshold<int32_t>(g, bins, br, k, kstride, gq, out, sk, up, s);
            });
        }
        if (!fq.empty()) {
            finish_queries(g, fq.data(), fc.data(), (int)fq.size(), fo.data(), s);  // synchronises
            up.reset();
        }
    }
}

void run_query_batch(folty_graph* g, const folty_query_params* qs, int nq, folty_result* outs,
                     cudaStream_t s, int64_t bin_budget) {
    // a batch of one (a server's batch under light load) is a single query: its captured
    // launch sequence is the shortest path
    if (nq == 1) {
        run_query(g, qs[0], &outs[0], s);
        return;
    }
    // a query that also wants the all-existential triples needs its own probe pass (the
    // role flags are per window, not per bin)
    for (int i = 0; i < nq; i++)
        if (qs[i].want_triples) run_query(g, qs[i], &outs[i], s);
    // group the queries by direction variant; distinct sorted deltas per group
    std::vector<BatchPass> passes;
    std::vector<int> slot((size_t)nq, -1), plain;
    for (int dir = 0; dir <= FOLTY_DIR_EITHER; dir++) {
        BatchPass ps{dir, {}, {}};
        for (int i = 0; i < nq; i++)
            if (qs[i].dir == dir && !qs[i].want_triples) ps.members.push_back(i);
        if (ps.members.empty()) continue;
        for (int i : ps.members) {
            ps.D.push_back(qs[i].delta);
            if (plain_query(qs[i])) {
                slot[(size_t)i] = (int)plain.size();
                plain.push_back(i);
            }
        }
        std::sort(ps.D.begin(), ps.D.end());
        ps.D.erase(std::unique(ps.D.begin(), ps.D.end()), ps.D.end());
        passes.push_back(std::move(ps));
    }
    // FOLTY_BATCH_SOLUTION_CAP sets a smaller solution buffer (the tests fill it with it)
    int64_t cap = BT_DEFAULT_CAP;
    if (const char* env = std::getenv("FOLTY_BATCH_SOLUTION_CAP")) cap = std::max<int64_t>(1, std::atoll(env));
    cap = std::min<int64_t>(cap, std::max<int64_t>(1, (int64_t)plain.size() * 2 * g->S));
    // and FOLTY_BATCH_BIN_BUDGET a budget for the bin rows (bytes) where the caller has none
    if (const char* env = std::getenv("FOLTY_BATCH_BIN_BUDGET"); env && bin_budget <= 0) bin_budget = std::max<int64_t>(1, std::atoll(env));
    BatchSolutions sol(g, plain, outs, cap, s);
    for (const BatchPass& ps : passes) run_batch_pass(g, qs, ps, slot, sol, outs, s, bin_budget);
    sol.finish();
}

}  // namespace folty

// tr.cu -- transitive reduction of the bidirected overlap graph R (Algorithm 1, Sec. IV-E) with
// the MinPlus semiring of Algorithm 3, on the GPU.
//
// One round, for every row i:
//   N_ik = min over j of R_ij + R_jk, over walks i->j->k that are valid (the two heads at j
//          point opposite ways: in(d_ij) == out(d_jk), Sec. II) -- only for k with R_ik present,
//          since Algorithm 1 compares M and N only where both exist;
//   v_i  = max_k R_ik + fuzz                                   (Reduce(Row, max), Apply(+x));
//   I_ik = N_ik exists, its end orientations equal d_ik (rules (b), (c) of Sec. II), and
//          v_i >= N_ik                                        (M >= N with M = DimApply(Row, v));
//   R    = R minus I                                          (R o not I).
// The round's result is a keep flag per entry; a stable compaction builds the next R. Rounds
// repeat until nnz(R) does not change.
//
// Direction encoding: d = 2 * o_first + o_second (o = 1: the read is traversed reverse-
// complemented). in(d) = d & 1, out(d) = d >> 1; the walk's composite dir is
// 2 * out(d_ij) + in(d_jk). Where N is needed it is kept as (sum << 2 | composite) in one 64-bit
// word, so that DIRMATCH (composite must equal d_ik before the min) and LITERAL (lexicographic min
// of (sum, composite), checked after) share one atomicMin; a DIRMATCH reduction needs only to know
// whether some walk is short enough.
#include <algorithm>

#include "check.cuh"
#include "ops.cuh"

namespace sg {

constexpr unsigned long long TR_NONE = ~0ull;

struct TrGraph {
    const int64_t *rp;
    const int32_t *col;
    const uint32_t *suf;
    const uint8_t *dir;
    int64_t n;
};

// An entry as one 64-bit word: column << 32 | suffix << 2 | dir (suffix < 2^30, dir <= 3), so that a
// product costs one load.
__device__ __forceinline__ uint64_t tr_pack(int32_t col, uint32_t suf, uint32_t dir) {
    return ((uint64_t)(uint32_t)col << 32) | (suf << 2) | dir;
}

// The graph the rounds work on: packed entries in row order (e; nullptr: the caller's arrays, in
// `in`), and each row's entries with those of out(d) = 0 first (p): a walk i -> j -> k continues only
// with the entries of j whose out(d) is in(d_ij), so a neighbour's other half is never read.
// row[i] = {first entry, low word; its high word; entries with out 0; entries with out 1}.
struct TrPacked {
    const uint64_t *e, *p;
    const uint4 *row;
    int64_t n;
    TrGraph in;
};
struct TrBuf {
    uint64_t *e = nullptr, *p = nullptr;
    uint4 *row = nullptr;
};

__device__ __forceinline__ uint64_t tr_entry(const TrPacked &g, int64_t x) {
    return g.e ? g.e[x] : tr_pack(g.in.col[x], g.in.suf[x], g.in.dir[x]);
}

__device__ __forceinline__ int64_t tr_first(const uint4 &r) { return (int64_t)(((uint64_t)r.y << 32) | r.x); }

// One warp writes a row of the packed graph: its entries from `first` on, given in order through
// next(t) (t < deg, every lane), kept where keep(t).
template <class Next, class Keep>
__device__ __forceinline__ void tr_write_row(const TrBuf &o, int64_t row, int64_t first, int64_t deg, Next &&next,
                                             Keep &&keep) {
    const int lane = threadIdx.x & 31;
    const uint32_t lt = (1u << lane) - 1u;
    uint32_t n0 = 0, n1 = 0;
    for (int64_t b = 0; b < deg; b += 32) {
        const bool have = b + lane < deg && keep(b + lane);
        const uint64_t x = have ? next(b + lane) : 0ull;
        n0 += __popc(__ballot_sync(0xffffffffu, have && !(x & 2u)));
        n1 += __popc(__ballot_sync(0xffffffffu, have && (x & 2u)));
    }
    int64_t w = first, w0 = first, w1 = first + n0;
    for (int64_t b = 0; b < deg; b += 32) {
        const bool have = b + lane < deg && keep(b + lane);
        const uint64_t x = have ? next(b + lane) : 0ull;
        const uint32_t m0 = __ballot_sync(0xffffffffu, have && !(x & 2u)), m1 = __ballot_sync(0xffffffffu, have && (x & 2u));
        if (have) {
            if (o.e) o.e[w + __popc((m0 | m1) & lt)] = x;
            o.p[(x & 2u) ? w1 + __popc(m1 & lt) : w0 + __popc(m0 & lt)] = x;
        }
        w += __popc(m0 | m1);
        w0 += __popc(m0);
        w1 += __popc(m1);
    }
    if (lane == 0) o.row[row] = make_uint4((uint32_t)first, (uint32_t)((uint64_t)first >> 32), n0, n1);
}

// Checks the CSR contract and packs the graph: one warp per row.
__global__ void validate_graph_kernel(TrGraph g, int64_t nnz, TrBuf o, uint32_t *__restrict__ err) {
    int64_t row = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    int lane = threadIdx.x & 31;
    if (row > g.n) return;
    if (row == g.n) {
        if (lane == 0 && (g.rp[g.n] != nnz || g.rp[0] != 0)) atomicOr(err, (uint32_t)DEV_INVALID);
        return;
    }
    int64_t r0 = g.rp[row], r1 = g.rp[row + 1];
    if (r1 < r0 || r0 < 0 || r1 > nnz) {
        if (lane == 0) atomicOr(err, (uint32_t)DEV_INVALID);
        return;
    }
    bool bad = false;
    for (int64_t e = r0 + lane; e < r1; e += 32) {
        const int32_t c = g.col[e];
        if (c < 0 || c >= g.n || c == row) bad = true;
        if (e > r0 && g.col[e - 1] >= c) bad = true;
        if (g.suf[e] >= (1u << 30) || g.dir[e] > 3) bad = true;
    }
    if (__any_sync(0xffffffffu, bad) && lane == 0) atomicOr(err, (uint32_t)DEV_INVALID);
    tr_write_row(o, row, r0, r1 - r0, [&](int64_t t) { return tr_pack(g.col[r0 + t], g.suf[r0 + t], g.dir[r0 + t] & 3u); },
                 [](int64_t) { return true; });
}

// ------------------------------------------------------------------------------- one round
// Row i's columns go into a hash table in shared memory; every entry (j, k) of the fitting half of
// every neighbour j's row is then one 8-byte load, a length check and a probe of the table.
//   MIN == false (reduction, DIRMATCH): entry (i, k) is transitive iff some valid walk i -> j -> k
//     with d_ik's end orientations has length <= the bound of its end: a flag, no minimum.
//   MIN == true (LITERAL, or N itself is wanted): the minimum of (length << 2 | orientations).
// Rows of up to TR_WROW entries take one warp each (its table is its own: no block barrier); four
// neighbours are walked at once, 8 lanes each, since half a row is a few tens of entries. Longer
// rows are listed and take a block; above TR_BROW entries the row is searched in place instead of
// hashed.
// The table is buckets of two columns, four to eight buckets per entry, so that one 8-byte load
// settles all but a few percent of the probes: at two slots per entry the longest of a warp's 32
// probe chains took 9 of 13 ms on 22 M edges.
constexpr int TR_NT = 128;
constexpr int TR_WROW = 128;   // entries of a warp's row
constexpr int TR_BNT = 256;
constexpr int TR_BROW = 2048;  // entries of a block's hashed row
constexpr uint32_t TR_FREE = 0xFFFFFFFFu;

struct TrArgs {
    TrPacked g;
    const uint32_t *err;
    int mode;
    uint32_t fuzz;
    unsigned long long *gbest;     // per-entry minima of rows above TR_BROW (MIN)
    uint8_t *keep;
    int64_t *kept;
    uint32_t *outN;
    uint8_t *outD;
    int32_t *big;                  // rows for blocks, and their number (nullptr: blocks look for them)
    unsigned long long *n_big;
    int warp_rows;                 // 0: every row takes a block
};

// The bounds of a row's entries by read end (out(d)): the row maximum, whole or per end, plus fuzz.
__device__ __forceinline__ void tr_bounds(const TrArgs &a, uint32_t m0, uint32_t m1, uint32_t &v0, uint32_t &v1) {
    const uint32_t m = m0 > m1 ? m0 : m1;
    const bool per_end = (a.mode & SG_TR_PER_END) != 0;
    v0 = (per_end ? m0 : m) + a.fuzz;  // both below 2^30
    v1 = (per_end ? m1 : m) + a.fuzz;
}

// Columns -> entries of one row: buckets of two keys (2^lb of them); val = entry << 2 | dir.
struct TrTable {
    uint32_t *key;
    uint16_t *val;
    int lb;
    __device__ __forceinline__ uint32_t bucket(uint32_t k) const { return (k * 2654435761u) >> (32 - lb); }
    __device__ __forceinline__ void insert(uint32_t k, uint32_t v) const {
        uint32_t h = 2u * bucket(k);
        const uint32_t msk = (2u << lb) - 1u;
        while (atomicCAS(key + h, TR_FREE, k) != TR_FREE) h = (h + 1) & msk;  // far from full
        val[h] = (uint16_t)v;
    }
    __device__ __forceinline__ uint2 load(uint32_t h) const { return *reinterpret_cast<const uint2 *>(key + 2 * h); }
    // slot of k from its bucket's keys, or -1
    __device__ __forceinline__ int find(uint32_t k, uint32_t h, uint2 x) const {
        for (;;) {
            if (x.x == k) return (int)(2 * h);
            if (x.y == k) return (int)(2 * h + 1);
            if (x.y == TR_FREE) return -1;  // filled in order
            h = (h + 1) & ((1u << lb) - 1u);
            x = load(h);
        }
    }
};

// Entries of four consecutive steps of a neighbour's half row, taken together so that their loads
// and their probes travel together. len(x) sums, ok(x) whether a walk of that length matters,
// hit(slot, walk orientations, length).
template <class Ok, class Hit>
__device__ __forceinline__ void tr_four(const TrTable &tb, uint32_t lij, const uint64_t *__restrict__ row, uint32_t b,
                                        uint32_t cnt, Ok &&ok, Hit &&hit) {
    uint64_t x[4];
    uint2 kk[4];
    uint32_t len[4];
    bool go[4];
#pragma unroll
    for (int u = 0; u < 4; u++) x[u] = b + 8 * u < cnt ? row[b + 8 * u] : 0ull;
#pragma unroll
    for (int u = 0; u < 4; u++) {
        len[u] = (lij >> 2) + ((uint32_t)x[u] >> 2);
        go[u] = b + 8 * u < cnt && ok((lij & 2u) | ((uint32_t)x[u] & 1u), len[u]);
        if (go[u]) kk[u] = tb.load(tb.bucket((uint32_t)(x[u] >> 32)));
    }
#pragma unroll
    for (int u = 0; u < 4; u++) {
        if (!go[u]) continue;
        const uint32_t k = (uint32_t)(x[u] >> 32);
        const int sl = tb.find(k, tb.bucket(k), kk[u]);
        if (sl >= 0) hit(sl, (lij & 2u) | ((uint32_t)x[u] & 1u), len[u]);
    }
}

// A warp's 32 neighbours (one per lane: entry, first entry and length of the fitting half row; 0
// entries past the row's end), four at a time.
template <class Ok, class Hit>
__device__ __forceinline__ void tr_walk(const TrTable &tb, const uint64_t *__restrict__ P, uint64_t ent, int64_t jb,
                                        uint32_t jn, int count, Ok &&ok, Hit &&hit) {
    const int lane = threadIdx.x & 31, sub = lane >> 3, l8 = lane & 7;
    for (int s4 = 0; s4 < count; s4 += 4) {
        const int src = s4 + sub;  // the lane that holds this group's neighbour
        const uint32_t lij = __shfl_sync(0xffffffffu, (uint32_t)ent, src);
        const int64_t b0 = __shfl_sync(0xffffffffu, jb, src);
        const uint32_t cnt = __shfl_sync(0xffffffffu, jn, src);
        for (uint32_t b = l8; b < cnt; b += 32) tr_four(tb, lij, P + b0, b, cnt, ok, hit);
        __syncwarp();
    }
}

// The fitting half of the neighbour behind entry x.
__device__ __forceinline__ void tr_half(const TrPacked &g, uint64_t x, int64_t &jb, uint32_t &jn) {
    const uint4 r = __ldg(g.row + (x >> 32));
    const bool in = x & 1u;
    jb = tr_first(r) + (in ? r.z : 0u);
    jn = in ? r.w : r.z;
}

// The outcome of entry t (packed ent): writes keep / N / Ndir; returns whether it is kept.
template <bool MIN>
__device__ __forceinline__ bool tr_outcome(const TrArgs &a, int64_t at, uint64_t ent, bool flag, unsigned long long best,
                                           uint32_t v0, uint32_t v1) {
    const uint32_t d = (uint32_t)ent & 3u;
    bool transitive = flag;
    if (MIN) {
        const bool has = best != TR_NONE;
        const uint64_t N = best >> 2;
        transitive = has && (uint32_t)(best & 3u) == d && ((d >> 1) ? v1 : v0) >= N;
        if (a.outN) a.outN[at] = has ? (uint32_t)N : 0xFFFFFFFFu;
        if (a.outD) a.outD[at] = has ? (uint8_t)(best & 3u) : (uint8_t)d;
    }
    if (a.keep) a.keep[at] = transitive ? 0 : 1;
    return !transitive;
}

__device__ __forceinline__ void tr_min(unsigned long long *best, uint32_t comp, uint32_t len) {
    const unsigned long long w = ((unsigned long long)len << 2) | comp;
    if (w < *(volatile unsigned long long *)best) atomicMin(best, w);
}

template <bool MIN>
struct __align__(16) TrWarpSmem {
    uint32_t key[8 * TR_WROW];  // cleared 16 bytes at a time
    unsigned long long best[MIN ? TR_WROW : 1];
    uint16_t val[8 * TR_WROW];
    uint8_t flag[MIN ? 4 : TR_WROW];
};
static_assert(sizeof(TrWarpSmem<true>) % 16 == 0 && sizeof(TrWarpSmem<false>) % 16 == 0, "16-byte rows of key");

template <bool MIN>
__global__ void __launch_bounds__(TR_NT) tr_mark_kernel(TrArgs a) {
    __shared__ TrWarpSmem<MIN> s_all[TR_NT / 32];
    if (*a.err) {  // the graph failed validation: touch nothing of it (the caller's scan reads kept)
        if (a.kept)
            for (int64_t i = (int64_t)blockIdx.x * TR_NT + threadIdx.x; i < a.g.n; i += (int64_t)gridDim.x * TR_NT)
                a.kept[i] = 0;
        return;
    }
    constexpr int Q = TR_WROW / 32;
    TrWarpSmem<MIN> &s = s_all[threadIdx.x >> 5];
    const int lane = threadIdx.x & 31;
    const int64_t nw = ((int64_t)gridDim.x * TR_NT) >> 5;
    for (int64_t i = ((int64_t)blockIdx.x * TR_NT + threadIdx.x) >> 5; i < a.g.n; i += nw) {
        const uint4 r = a.g.row[i];
        const int64_t r0 = tr_first(r), degl = (int64_t)r.z + r.w;
        if (degl == 0) {
            if (lane == 0 && a.kept) a.kept[i] = 0;
            continue;
        }
        if (degl > TR_WROW || (a.big && !a.warp_rows)) {
            if (lane == 0 && a.big) {
                const unsigned long long q = atomicAdd(a.n_big, 1ull);
                if (SG_IN_BOUNDS((int64_t)q < a.g.n, 403, q)) a.big[q] = (int32_t)i;
            }
            continue;
        }
        const int deg = (int)degl;
        TrTable tb{s.key, s.val, 4};
        while ((1 << tb.lb) < 4 * deg && tb.lb < 9) tb.lb++;
        for (int x = lane; x < (2 << tb.lb) / 4; x += 32)
            reinterpret_cast<uint4 *>(s.key)[x] = make_uint4(TR_FREE, TR_FREE, TR_FREE, TR_FREE);
        // the row, its neighbours' fitting halves, its maxima; the table
        uint64_t ent[Q];
        int64_t jb[Q];
        uint32_t jn[Q], m0 = 0, m1 = 0;
#pragma unroll
        for (int q = 0; q < Q; q++) {
            const int t = 32 * q + lane;
            ent[q] = 0;
            jb[q] = 0;
            jn[q] = 0;
            if (t < deg) {
                ent[q] = tr_entry(a.g, r0 + t);
                tr_half(a.g, ent[q], jb[q], jn[q]);
                const uint32_t sv = (uint32_t)ent[q] >> 2;
                if (ent[q] & 2u) m1 = sv > m1 ? sv : m1; else m0 = sv > m0 ? sv : m0;
                if (MIN) s.best[MIN ? t : 0] = TR_NONE; else s.flag[MIN ? 0 : t] = 0;
            }
        }
        m0 = __reduce_max_sync(0xffffffffu, m0);
        m1 = __reduce_max_sync(0xffffffffu, m1);
        uint32_t v0, v1;
        tr_bounds(a, m0, m1, v0, v1);
        __syncwarp();
#pragma unroll
        for (int q = 0; q < Q; q++) {
            const int t = 32 * q + lane;
            if (t < deg) tb.insert((uint32_t)(ent[q] >> 32), (uint32_t)(t << 2) | ((uint32_t)ent[q] & 3u));
        }
        __syncwarp();
        auto ok = [&](uint32_t comp, uint32_t len) { return MIN || len <= ((comp & 2u) ? v1 : v0); };
        auto hit = [&](int sl, uint32_t comp, uint32_t len) {
            const uint32_t v = s.val[sl];
            if (MIN) {
                if ((a.mode & 1) == SG_TR_DIRMATCH && comp != (v & 3u)) return;
                tr_min(s.best + (MIN ? v >> 2 : 0u), comp, len);
            } else if (comp == (v & 3u)) {
                s.flag[MIN ? 0u : v >> 2] = 1;
            }
        };
#pragma unroll
        for (int q = 0; q < Q; q++)
            if (32 * q < deg) tr_walk(tb, a.g.p, ent[q], jb[q], jn[q], deg - 32 * q < 32 ? deg - 32 * q : 32, ok, hit);
        __syncwarp();
        int mykept = 0;
#pragma unroll
        for (int q = 0; q < Q; q++) {
            const int t = 32 * q + lane;
            if (t < deg) mykept += tr_outcome<MIN>(a, r0 + t, ent[q], !MIN && s.flag[MIN ? 0 : t],
                                                   MIN ? s.best[MIN ? t : 0] : TR_NONE, v0, v1) ? 1 : 0;
        }
        mykept = __reduce_add_sync(0xffffffffu, mykept);
        if (lane == 0 && a.kept) a.kept[i] = mykept;
        __syncwarp();  // the table is cleared next
    }
}

// Listed rows, one block each: the row's neighbours in groups of 32, a warp per group.
template <bool MIN>
constexpr size_t tr_big_smem() {
    return (size_t)TR_BROW * (MIN ? 8 : 0) + (size_t)4 * TR_BROW * 6 + (MIN ? 0 : TR_BROW);
}
template <bool MIN>
__global__ void __launch_bounds__(TR_BNT) tr_mark_big_kernel(TrArgs a) {
    extern __shared__ __align__(16) unsigned char tr_raw[];
    unsigned long long *sbest = reinterpret_cast<unsigned long long *>(tr_raw);                     // (MIN)
    uint32_t *key = reinterpret_cast<uint32_t *>(tr_raw + (size_t)TR_BROW * (MIN ? 8 : 0));         // [4 TR_BROW]
    uint16_t *val = reinterpret_cast<uint16_t *>(key + 4 * TR_BROW);                                // entry
    uint8_t *flag = reinterpret_cast<uint8_t *>(val + 4 * TR_BROW);                                 // (!MIN)
    __shared__ uint32_t s_m[2];
    __shared__ int s_kept;
    if (*a.err) return;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    auto E = [&](int64_t t) { return tr_entry(a.g, t); };
    const int64_t nrows = a.big ? (int64_t)*a.n_big : a.g.n;
    for (int64_t rb = blockIdx.x; rb < nrows; rb += gridDim.x) {
        const int32_t i = a.big ? a.big[rb] : (int32_t)rb;
        if (!SG_IN_BOUNDS(i >= 0 && i < a.g.n, 404, i)) continue;
        const uint4 r = a.g.row[i];
        const int64_t r0 = tr_first(r), deg = (int64_t)r.z + r.w;
        if (!a.big && deg <= TR_WROW) continue;  // a warp's
        const bool hashed = deg <= TR_BROW;
        unsigned long long *best = hashed ? sbest : a.gbest + r0;
        TrTable tb{key, val, 4};
        while (hashed && (1 << tb.lb) < 2 * deg) tb.lb++;
        if (threadIdx.x < 2) s_m[threadIdx.x] = 0;
        if (threadIdx.x == 0) s_kept = 0;
        if (hashed)
            for (int x = threadIdx.x; x < (2 << tb.lb); x += TR_BNT) key[x] = TR_FREE;
        __syncthreads();
        uint32_t m0 = 0, m1 = 0;
        for (int64_t t = threadIdx.x; t < deg; t += TR_BNT) {
            const uint64_t ent = E(r0 + t);
            const uint32_t sv = (uint32_t)ent >> 2;
            if (ent & 2u) m1 = sv > m1 ? sv : m1; else m0 = sv > m0 ? sv : m0;
            if (MIN) best[t] = TR_NONE;
            else if (hashed) flag[t] = 0;
            else a.keep[r0 + t] = 1;
            if (hashed) tb.insert((uint32_t)(ent >> 32), (uint32_t)((t << 2) | (ent & 3u)));
        }
        atomicMax(s_m, m0);
        atomicMax(s_m + 1, m1);
        __syncthreads();
        uint32_t v0, v1;
        tr_bounds(a, s_m[0], s_m[1], v0, v1);
        auto ok = [&](uint32_t comp, uint32_t len) { return MIN || len <= ((comp & 2u) ? v1 : v0); };
        auto hit_at = [&](int64_t t, uint32_t d, uint32_t comp, uint32_t len) {
            if (MIN) {
                if ((a.mode & 1) == SG_TR_DIRMATCH && comp != d) return;
                tr_min(best + t, comp, len);
            } else if (comp == d) {
                if (hashed) flag[t] = 1; else a.keep[r0 + t] = 0;
            }
        };
        auto hit = [&](int sl, uint32_t comp, uint32_t len) { hit_at(val[sl] >> 2, val[sl] & 3u, comp, len); };
        for (int64_t c = (int64_t)warp * 32; c < deg; c += TR_BNT) {
            const int64_t t = c + lane;
            uint64_t ent = 0;
            int64_t jb = 0;
            uint32_t jn = 0;
            if (t < deg) {
                ent = E(r0 + t);
                tr_half(a.g, ent, jb, jn);
            }
            const int count = deg - c < 32 ? (int)(deg - c) : 32;
            if (hashed) {
                tr_walk(tb, a.g.p, ent, jb, jn, count, ok, hit);
                continue;
            }
            for (int q = 0; q < count; q++) {
                const uint32_t lij = __shfl_sync(0xffffffffu, (uint32_t)ent, q);
                const int64_t b0 = __shfl_sync(0xffffffffu, jb, q);
                const uint32_t cnt = __shfl_sync(0xffffffffu, jn, q);
                for (uint32_t b = lane; b < cnt; b += 32) {
                    const uint64_t x = a.g.p[b0 + b];
                    const uint32_t comp = (lij & 2u) | ((uint32_t)x & 1u), len = (lij >> 2) + ((uint32_t)x >> 2);
                    if (!ok(comp, len)) continue;
                    int64_t lo = 0, hi = deg;  // first entry with column >= k
                    while (lo < hi) {
                        const int64_t mid = (lo + hi) >> 1;
                        if ((E(r0 + mid) >> 32) < (x >> 32)) lo = mid + 1; else hi = mid;
                    }
                    if (lo < deg && (E(r0 + lo) >> 32) == (x >> 32)) hit_at(lo, (uint32_t)E(r0 + lo) & 3u, comp, len);
                }
            }
        }
        __syncthreads();
        int mykept = 0;
        for (int64_t t = threadIdx.x; t < deg; t += TR_BNT) {
            const bool f = !MIN && (hashed ? flag[t] != 0 : a.keep[r0 + t] == 0);
            mykept += tr_outcome<MIN>(a, r0 + t, E(r0 + t), f, MIN ? best[t] : TR_NONE, v0, v1) ? 1 : 0;
        }
        mykept = __reduce_add_sync(0xffffffffu, mykept);
        if (lane == 0 && mykept) atomicAdd(&s_kept, mykept);
        __syncthreads();
        if (threadIdx.x == 0 && a.kept) a.kept[i] = s_kept;
        __syncthreads();
    }
}

// Stable compaction of kept entries: one warp per row.
__global__ void tr_compact_kernel(TrPacked g, const uint8_t *__restrict__ keep, const int64_t *__restrict__ nrp, TrBuf o) {
    const int64_t row = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (row >= g.n) return;
    const uint4 r = g.row[row];
    const int64_t r0 = tr_first(r);
    tr_write_row(o, row, nrp[row], (int64_t)r.z + r.w, [&](int64_t t) { return tr_entry(g, r0 + t); },
                 [&](int64_t t) { return keep[r0 + t] != 0; });
}

// Packed entries -> the arrays of S.
__global__ void tr_unpack_kernel(TrPacked g, int64_t nnz, const int64_t *__restrict__ rp, int64_t n,
                                 int64_t *__restrict__ orp, int32_t *__restrict__ col, uint32_t *__restrict__ suf,
                                 uint8_t *__restrict__ dir) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < nnz) {
        const uint64_t x = tr_entry(g, i);
        col[i] = (int32_t)(x >> 32);
        suf[i] = (uint32_t)x >> 2;
        dir[i] = (uint8_t)(x & 3u);
    }
    if (i <= n) orp[i] = rp[i];
}

static inline int64_t blocks_for(int64_t n, int nt) { return (n + nt - 1) / nt; }

// Buffers of a round (sized for the input graph; later rounds only shrink).
struct TrWork {
    unsigned long long *n_big;  // [1] rows listed for blocks
    int32_t *big;               // [n + 1]
    unsigned long long *gbest;  // [nnz + 1] per-entry minima of rows above TR_BROW
};

static sg_status tr_work_alloc(TrWork *w, int64_t n, int64_t nnz, bool minima, Scratch &sc) {
    w->n_big = sc.get<unsigned long long>(1);
    w->big = sc.get<int32_t>(n + 1);
    w->gbest = minima ? sc.get<unsigned long long>(nnz + 1) : nullptr;
    return (w->n_big && w->big && (w->gbest || !minima)) ? SG_OK : SG_ERR_OOM;
}

// One round over graph g: keep flags + per-row kept counts (and optionally N / Ndir). Rows for
// blocks are listed on the device and the second kernel runs grid-stride over their number, so the
// round needs no host round trip. Nothing runs past a set `err` (failed validation).
static sg_status minplus_round(const TrPacked &g, int mode, uint32_t fuzz, uint8_t *keep, int64_t *kept, uint32_t *outN,
                               uint8_t *outD, const TrWork &w, const uint32_t *err, cudaStream_t s) {
    const int64_t n = g.n;
    if (n == 0) return SG_OK;
    if (w.big) SG_CUDA_TRY(cudaMemsetAsync(w.n_big, 0, sizeof(unsigned long long), s));
    const TrArgs a{g, err, mode, fuzz, w.gbest, keep, kept, outN, outD, w.big, w.n_big, (int)tune("tr_warp_rows")};
    const int64_t cap = (int64_t)sm_count() * tune("tr_blocks_per_sm"), rows = blocks_for(n, TR_NT / 32);
    const int64_t gs = rows < cap ? rows : cap;
    const int64_t gg = n < (int64_t)sm_count() * 3 ? n : (int64_t)sm_count() * 3;
    if (outN || outD || (mode & 1) != SG_TR_DIRMATCH) {
        SG_CUDA_TRY(ensure_smem(tr_mark_big_kernel<true>, tr_big_smem<true>()));
        SG_LAUNCH("tr_minplus_mark", tr_mark_kernel<true>, gs, TR_NT, 0, s, a);
        SG_LAUNCH("tr_minplus_mark_big", tr_mark_big_kernel<true>, gg, TR_BNT, tr_big_smem<true>(), s, a);
    } else {
        SG_CUDA_TRY(ensure_smem(tr_mark_big_kernel<false>, tr_big_smem<false>()));
        SG_LAUNCH("tr_minplus_mark", tr_mark_kernel<false>, gs, TR_NT, 0, s, a);
        SG_LAUNCH("tr_minplus_mark_big", tr_mark_big_kernel<false>, gg, TR_BNT, tr_big_smem<false>(), s, a);
    }
    return SG_OK;
}

static void free_graph_arrays(sg_graph_csr *x, cudaStream_t s) {
    dfree(x->row_ptr, s);
    dfree(x->col, s);
    dfree(x->suffix, s);
    dfree(x->dir, s);
    *x = sg_graph_csr{};
}

// Batches: job_last[b] = max(job_last[b], round) for every job b that lost an entry this round.
__global__ void job_changes_kernel(const int64_t *__restrict__ rp, const int64_t *__restrict__ kept, int64_t n,
                                   const int64_t *__restrict__ job_ro, int64_t njobs, int32_t round,
                                   int32_t *__restrict__ job_last) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n || (rp[i + 1] - rp[i]) == kept[i]) return;
    int64_t lo = 0, hi = njobs;  // last job b with job_ro[b] <= i
    while (hi - lo > 1) {
        const int64_t mid = (lo + hi) >> 1;
        if (job_ro[mid] <= i) lo = mid; else hi = mid;
    }
    atomicMax(job_last + lo, round);
}

sg_status tr_impl(const sg_graph_csr *R, uint32_t fuzz, int mode, sg_graph_csr *S, int32_t *iters,
                  cudaStream_t s, const int64_t *job_ro, int64_t njobs, int32_t *job_last, int32_t max_rounds,
                  int32_t *converged) {
    const int64_t n = R->n, nnz0 = R->nnz;
    StageScope stage("TrReduction", s);
    Scratch sc(s);
    // row pointers of a round's result, each with an error word behind its last, so that one copy reads
    // both back (a copy to the host waits for the stream); the first round takes rp[1] and validates
    int64_t *rp[2] = {nullptr, sc.get<int64_t>(2 * (n + 2))};
    uint8_t *keep = sc.get<uint8_t>(nnz0 + 1);
    int64_t *kept = sc.get<int64_t>(n + 1);
    if (!rp[1] || !keep || !kept) return SG_ERR_OOM;
    rp[0] = rp[1] + n + 2;
    uint32_t *const err = (uint32_t *)(rp[1] + n + 1), *const errs[2] = {(uint32_t *)(rp[0] + n + 1), err};
    TrWork wk;
    SG_TRY(tr_work_alloc(&wk, n, nnz0, (mode & 1) != SG_TR_DIRMATCH, sc));
    // the rounds' graphs: each reads one buffer and compacts into the other (the first reads the
    // caller's arrays beside buffer 0)
    TrBuf buf[2];
    for (int b = 0; b < 2; b++) {
        buf[b].p = sc.get<uint64_t>(nnz0 + 1);
        buf[b].row = sc.get<uint4>(n + 1);
        if (!buf[b].p || !buf[b].row) return SG_ERR_OOM;
    }
    const TrGraph in{R->row_ptr, R->col, R->suffix, R->dir, n};
    SG_CUDA_TRY(cudaMemsetAsync(err, 0, (size_t)(n + 3) * 8, s));  // both error words and what lies between
    SG_LAUNCH("validate_graph", validate_graph_kernel, blocks_for((n + 1) * 32, 256), 256, 0, s, in, nnz0, buf[0], err);
    TrPacked g{nullptr, buf[0].p, buf[0].row, n, in};
    const int64_t *grp = R->row_ptr;
    int64_t cur_nnz = nnz0;
    int cur = 0;
    int32_t it = 0;
    bool done = false;
    for (;;) {
        if (max_rounds > 0 && it == max_rounds) break;  // stopped early: S is an intermediate R
        it++;
        StageScope round("TrRound", s);
        const int nxt = 1 - cur;
        SG_TRY(minplus_round(g, mode, fuzz, keep, kept, nullptr, nullptr, wk, err, s));
        if (job_ro)
            SG_LAUNCH("tr_job_changes", job_changes_kernel, blocks_for(n, 256), 256, 0, s, grp,
                      (const int64_t *)kept, n, job_ro, njobs, it, job_last);
        SG_TRY(exclusive_scan<int64_t>(kept, rp[nxt], n, s, errs[nxt]));
        int64_t end[2] = {0, 0};
        SG_CUDA_TRY(read_back(end, rp[nxt] + n, sizeof(end), s));
        const int64_t nnz2 = end[0];
        const uint32_t herr = (uint32_t)end[1];
        if (herr & DEV_TIMEOUT) return timeout_error("transitive_reduce");
        if (herr) {
            set_error("graph does not satisfy the CSR contract (sorted unique columns, no diagonal, suffix < 2^30, dir <= 3)");
            return SG_ERR_INVALID;
        }
        if (nnz2 == cur_nnz) {  // nothing removed: R is final
            done = true;
            break;
        }
        if (!buf[nxt].e && !(buf[nxt].e = sc.get<uint64_t>(nnz2 + 1))) return SG_ERR_OOM;
        SG_LAUNCH("tr_compact", tr_compact_kernel, blocks_for(n * 32, 256), 256, 0, s, g, (const uint8_t *)keep,
                  (const int64_t *)rp[nxt], buf[nxt]);
        cur = nxt;
        cur_nnz = nnz2;
        grp = rp[cur];
        g = TrPacked{buf[cur].e, buf[cur].p, buf[cur].row, n, in};
    }
    // S: the final graph, unpacked into exact-size arrays
    sg_graph_csr out{};
    out.n = n;
    out.nnz = cur_nnz;
    out.row_ptr = (int64_t *)dalloc((n + 1) * sizeof(int64_t), s);
    out.col = (int32_t *)dalloc(cur_nnz * sizeof(int32_t), s);
    out.suffix = (uint32_t *)dalloc(cur_nnz * sizeof(uint32_t), s);
    out.dir = (uint8_t *)dalloc(cur_nnz, s);
    if (!out.row_ptr || !out.col || !out.suffix || !out.dir) {
        free_graph_arrays(&out, s);
        return SG_ERR_OOM;
    }
    const sg_status st = [&]() -> sg_status {
        SG_LAUNCH("tr_unpack", tr_unpack_kernel, blocks_for(std::max(cur_nnz, n + 1), 256), 256, 0, s, g, cur_nnz, grp, n,
                  out.row_ptr, out.col, out.suffix, out.dir);
        return SG_OK;
    }();
    if (st != SG_OK) {
        free_graph_arrays(&out, s);
        return st;
    }
    *S = out;
    *iters = it;
    if (converged) *converged = done ? 1 : 0;
    return SG_OK;
}

static bool graph_args_ok(const sg_graph_csr *R) {
    return R && R->n >= 0 && R->n < ((int64_t)1 << 31) && R->nnz >= 0 && R->row_ptr &&
           (R->nnz == 0 || (R->col && R->suffix && R->dir));
}

}  // namespace sg

extern "C" sg_status sg_transitive_reduce(const sg_graph_csr *R, uint32_t fuzz, int32_t mode, sg_graph_csr *S,
                                          int32_t *iterations, sg_stream_t stream) {
    if (!S || !iterations) {
        sg::set_error("transitive_reduce: NULL output");
        return SG_ERR_INVALID;
    }
    *S = sg_graph_csr{};
    *iterations = 0;
    if (!sg::graph_args_ok(R) || fuzz >= (1u << 30) || mode < 0 || mode > (SG_TR_LITERAL | SG_TR_PER_END)) {
        sg::set_error("transitive_reduce: invalid arguments");
        return SG_ERR_INVALID;
    }
    return sg::tr_impl(R, fuzz, mode, S, iterations, (cudaStream_t)stream, nullptr, 0, nullptr, 0, nullptr);
}

extern "C" sg_status sg_transitive_reduce_rounds(const sg_graph_csr *R, uint32_t fuzz, int32_t mode,
                                                 int32_t max_rounds, sg_graph_csr *S, int32_t *rounds,
                                                 int32_t *converged, sg_stream_t stream) {
    if (!S || !rounds || !converged) {
        sg::set_error("transitive_reduce_rounds: NULL output");
        return SG_ERR_INVALID;
    }
    *S = sg_graph_csr{};
    *rounds = 0;
    *converged = 0;
    if (!sg::graph_args_ok(R) || fuzz >= (1u << 30) || mode < 0 || mode > (SG_TR_LITERAL | SG_TR_PER_END) ||
        max_rounds < 1) {
        sg::set_error("transitive_reduce_rounds: invalid arguments");
        return SG_ERR_INVALID;
    }
    return sg::tr_impl(R, fuzz, mode, S, rounds, (cudaStream_t)stream, nullptr, 0, nullptr, max_rounds,
                       converged);
}

extern "C" sg_status sg_minplus_square(const sg_graph_csr *R, int32_t mode, uint32_t *d_N, uint8_t *d_Ndir,
                                       sg_stream_t stream) {
    if (!sg::graph_args_ok(R) || (mode != SG_TR_DIRMATCH && mode != SG_TR_LITERAL) || (R->nnz > 0 && !d_N)) {
        sg::set_error("minplus_square: invalid arguments");
        return SG_ERR_INVALID;
    }
    cudaStream_t s = (cudaStream_t)stream;
    sg::Scratch sc(s);
    uint32_t *err = sc.get<uint32_t>(1);
    if (!err) return SG_ERR_OOM;
    sg::TrGraph g{R->row_ptr, R->col, R->suffix, R->dir, R->n};
    sg::TrWork wk;
    SG_TRY(sg::tr_work_alloc(&wk, R->n, R->nnz, true, sc));
    sg::TrBuf buf;
    buf.p = sc.get<uint64_t>(R->nnz + 1);
    buf.row = sc.get<uint4>(R->n + 1);
    if (!buf.p || !buf.row) return SG_ERR_OOM;
    SG_CUDA_TRY(cudaMemsetAsync(err, 0, sizeof(uint32_t), s));
    SG_LAUNCH("validate_graph", sg::validate_graph_kernel, (R->n + 1 + 7) / 8, 256, 0, s, g, R->nnz, buf, err);
    SG_TRY(sg::minplus_round(sg::TrPacked{nullptr, buf.p, buf.row, R->n, g}, mode, 0, nullptr, nullptr, d_N, d_Ndir, wk, err,
                             s));
    uint32_t herr = 0;
    SG_CUDA_TRY(sg::read_back(&herr, err, sizeof(uint32_t), s));
    if (herr) {
        sg::set_error("minplus_square: graph does not satisfy the CSR contract");
        return SG_ERR_INVALID;
    }
    return SG_OK;
}

extern "C" void sg_free_graph(sg_graph_csr *x, sg_stream_t stream) {
    if (!x) return;
    sg::free_graph_arrays(x, (cudaStream_t)stream);
}

// ------------------------------------------------------------------------------------------
// Allocation-free variant of sg_minplus_square.
//
// Some callers cannot allocate device memory at the moment they want this product: code that
// runs while a memory pool is being torn down or is already exhausted, code that must not
// grow the footprint of a process that shares its GPU under a hard memory cap, and host
// threads (e.g. a real-time scheduler loop) that may not take the allocator's locks or wait on
// its synchronisation. For them the workspace of the product lives in one file-scope device
// array, reserved when the library is loaded and kept until the process exits, on every GPU
// that loads the library.
#include <mutex>

static __device__ __align__(256) unsigned char sg_noalloc_scratch[SG_NOALLOC_SCRATCH_BYTES];

namespace sg {

static std::mutex g_noalloc_mu;
static void *g_noalloc_addr[256];  // device address of sg_noalloc_scratch, per device ordinal

// Device address of the scratch array on the current device. The first call on a device looks
// it up (the array's name in host code is only a stand-in, never a device address).
static sg_status noalloc_scratch(unsigned char **out) {
    int dev = 0;
    SG_CUDA_TRY(cudaGetDevice(&dev));
    if (dev < 0 || dev >= 256) {
        set_error("minplus_square_noalloc: device ordinal %d out of range", dev);
        return SG_ERR_INVALID;
    }
    std::lock_guard<std::mutex> lk(g_noalloc_mu);
    if (!g_noalloc_addr[dev]) {
        void *p = nullptr;
        cudaError_t e = cudaGetSymbolAddress(&p, sg_noalloc_scratch);
        if (e != cudaSuccess || !p) {
            set_error("minplus_square_noalloc: cudaGetSymbolAddress failed on device %d: %s", dev,
                      cudaGetErrorString(e));
            return SG_ERR_CUDA;
        }
        g_noalloc_addr[dev] = p;
    }
    *out = (unsigned char *)g_noalloc_addr[dev];
    return SG_OK;
}

static size_t up256(size_t x) { return (x + 255) & ~(size_t)255; }

}  // namespace sg

extern "C" sg_status sg_minplus_square_noalloc(const sg_graph_csr *R, int32_t mode, uint32_t *d_N,
                                               uint8_t *d_Ndir, sg_stream_t stream) {
    if (!sg::graph_args_ok(R) || (mode != SG_TR_DIRMATCH && mode != SG_TR_LITERAL) || (R->nnz > 0 && !d_N)) {
        sg::set_error("minplus_square_noalloc: invalid arguments");
        return SG_ERR_INVALID;
    }
    const int64_t n = R->n, nnz = R->nnz;
    // workspace layout inside the scratch array: the error word, the packed rows and entries, the
    // per-entry minima. The limit is the documented one, a little above what they take.
    const size_t o_err = 0;
    const size_t o_row = sg::up256(o_err + sizeof(uint32_t));
    const size_t o_ent = sg::up256(o_row + (size_t)n * sizeof(uint4));
    const size_t o_best = sg::up256(o_ent + (size_t)nnz * sizeof(uint64_t));
    const size_t need = sg::up256(sg::up256(sg::up256(512 + (size_t)(n + 1)) + (size_t)(n + 1) * 8) +
                                  (size_t)(nnz + 1) * 8) + (size_t)(nnz + n + 1) * 8;
    if (need > (size_t)SG_NOALLOC_SCRATCH_BYTES || o_best + (size_t)nnz * 8 > (size_t)SG_NOALLOC_SCRATCH_BYTES) {
        sg::set_error("minplus_square_noalloc: a graph with n=%lld and nnz=%lld needs %zu bytes of workspace, "
                      "more than the fixed %zu-byte scratch array; use sg_minplus_square",
                      (long long)n, (long long)nnz, need, (size_t)SG_NOALLOC_SCRATCH_BYTES);
        return SG_ERR_BUDGET;
    }
    unsigned char *base = nullptr;
    SG_TRY(sg::noalloc_scratch(&base));
    cudaStream_t s = (cudaStream_t)stream;
    uint32_t *err = (uint32_t *)(base + o_err);
    sg::TrWork wk;
    wk.n_big = nullptr;  // no room for a list of long rows: blocks look for them
    wk.big = nullptr;
    wk.gbest = (unsigned long long *)(base + o_best);
    sg::TrBuf buf;
    buf.p = (uint64_t *)(base + o_ent);
    buf.row = (uint4 *)(base + o_row);
    sg::TrGraph g{R->row_ptr, R->col, R->suffix, R->dir, n};
    // the array keeps whatever the previous call left: the error word starts from zero here, and
    // every other word is written before read
    SG_CUDA_TRY(cudaMemsetAsync(err, 0, sizeof(uint32_t), s));
    SG_LAUNCH("validate_graph", sg::validate_graph_kernel, (n + 1 + 7) / 8, 256, 0, s, g, nnz, buf, err);
    uint32_t herr = 0;
    SG_CUDA_TRY(sg::read_back(&herr, err, sizeof(uint32_t), s));
    if (herr) {
        sg::set_error("minplus_square_noalloc: graph does not satisfy the CSR contract");
        return SG_ERR_INVALID;
    }
    SG_TRY(sg::minplus_round(sg::TrPacked{nullptr, buf.p, buf.row, n, g}, mode, 0, nullptr, nullptr, d_N, d_Ndir, wk, err, s));
    SG_CUDA_TRY(cudaStreamSynchronize(s));
    return SG_OK;
}

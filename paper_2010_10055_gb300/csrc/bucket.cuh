// bucket.cuh -- records grouped by a code prefix and finished in shared memory: the engine of the
// bucketed k-mer count and of A = At transposed (kbucket.cu).
//
// A record is (code, read, position, strand) in one 64-bit word, code highest (KeyN), or in two
// (KeyW) where the bits do not fit. Records are moved by at most two grouping passes:
//  1. by the top pb1 bits of the code (a prefix p; those bits leave the record);
//  2. within p, by the next b2[p] bits, b2 chosen from p's exact record count so that a bucket
//     holds at most 10/11 of what one block can finish in shared memory. (Any number of equal parts
//     instead of 2^b2 fills the buckets better, but a part's first code costs a division and
//     leaves fewer slots per record: the finishing pass of 4.1e9 records 52 -> 55 ms.)
// Grouping is unordered (one atomic per tile and bin reserves a run), since the pass that finishes
// a bucket orders its records itself: it counts them by slot -- the bucket's next code bits, about
// as many slots as records -- places them by slot and ranks each among the few of its slot by full
// comparison. No pass depends on the order of another block's writes, so nothing waits.
#pragma once

#include "check.cuh"
#include "prim.cuh"

namespace sg {

constexpr int KB_NT = 512;
constexpr int KB_MAXBINS = 2048;  // bins of one grouping pass (counters and bases in shared memory)
constexpr int KB_MAXB2 = 11;      // log2 of it
constexpr int KB_NS = 14;         // log2 of the slots of one bucket, at most
constexpr int KB_CHUNK_TILES = 4; // level-2 work is dealt in chunks of this many tiles

// Fields below the code: read (rbits), position (pbits), strand (1).
struct KeyBits {
    int rbits, pbits;
    __host__ __device__ int low() const { return rbits + pbits + 1; }
};

// The low 32 bits of x >> s (0 <= s <= 64; 64: a prefix that is not split, of records that fill their
// word), in two instructions where s is the same for all lanes. The clamped shift is defined at 32.
__device__ __forceinline__ uint32_t low_bits_at(uint64_t x, int s) {
    const uint32_t lo = (uint32_t)x, hi = (uint32_t)(x >> 32);
    return s < 32 ? __funnelshift_r(lo, hi, s) : __funnelshift_rc(hi, 0u, s - 32);
}

struct KeyN {  // one word: code << low | read << (pbits + 1) | pos << 1 | strand
    using T = uint64_t;
    static constexpr int ITEMS = 16;
    __device__ static T make(uint64_t code, uint64_t low, int lowbits) { return (code << lowbits) | low; }
    __device__ static T none() { return 0ull; }
    __device__ static uint64_t code(T k, int lowbits) { return lowbits < 64 ? k >> lowbits : 0ull; }
    __device__ static uint64_t low(T k, int lowbits) { return lowbits < 64 ? k & ((1ull << lowbits) - 1) : k; }
    __device__ static bool less(T a, T b) { return a < b; }
    __device__ static bool same(T a, T b, uint64_t mask) { return ((a ^ b) & mask) == 0; }  // code_mask / read_mask
    __device__ static uint64_t code_mask(int lowbits) { return lowbits < 64 ? ~0ull << lowbits : 0ull; }
    __device__ static uint64_t read_mask(int pbits) { return ~0ull << (pbits + 1); }
    // slot of a record: ((code - c0) >> sh), from base = slot_base(c0)
    __device__ static uint64_t slot_base(uint64_t c0, int lowbits) { return lowbits < 64 ? c0 << lowbits : 0ull; }
    __device__ static uint32_t slot(T k, uint64_t base, int lowbits, int sh) { return low_bits_at(k - base, lowbits + sh); }
    __device__ static T load(const T *p) { return __ldcs(reinterpret_cast<const unsigned long long *>(p)); }
};

struct __align__(16) U128 {
    uint64_t lo, hi;
};
struct KeyW {  // two words: code | the same low fields
    using T = U128;
    static constexpr int ITEMS = 8;
    __device__ static T make(uint64_t code, uint64_t low, int) { return U128{low, code}; }
    __device__ static T none() { return U128{0ull, 0ull}; }
    __device__ static uint64_t code(const T &k, int) { return k.hi; }
    __device__ static uint64_t low(const T &k, int) { return k.lo; }
    __device__ static bool less(const T &a, const T &b) { return a.hi < b.hi || (a.hi == b.hi && a.lo < b.lo); }
    __device__ static bool same(const T &a, const T &b, uint64_t mask) {
        return a.hi == b.hi && ((a.lo ^ b.lo) & mask) == 0;
    }
    __device__ static uint64_t code_mask(int) { return 0ull; }
    __device__ static uint64_t read_mask(int pbits) { return ~0ull << (pbits + 1); }
    __device__ static uint64_t slot_base(uint64_t c0, int) { return c0; }
    __device__ static uint32_t slot(const T &k, uint64_t base, int, int sh) { return low_bits_at(k.hi - base, sh); }
    __device__ static T load(const T *p) {
        const uint4 v = __ldcs(reinterpret_cast<const uint4 *>(p));
        return U128{((uint64_t)v.y << 32) | v.x, ((uint64_t)v.w << 32) | v.z};
    }
};

template <class K> constexpr int kb_tile() { return KB_NT * K::ITEMS; }  // 8192 or 4096 records
template <class K> constexpr int kb_target() { return kb_tile<K>() - kb_tile<K>() / 11; }

// Level-1 prefixes and their level-2 split, written by kb_plan_kernel (device arrays).
struct KbPlan {
    int nb1;                      // prefixes: 2^pb1
    int rem;                      // code bits left below the prefix
    int two;                      // whether there is a second pass
    int64_t *start1;              // [nb1 + 1] first record of each prefix
    unsigned long long *cur1;     // [nb1] write cursors of the first pass
    uint8_t *b2;                  // [nb1]
    uint32_t *sb;                 // [nb1 + 1] first bucket of each prefix; sb[nb1] = buckets
    uint32_t *chunk2;             // [nb1 + 1] first level-2 chunk of each prefix
    uint16_t *sub2p;              // [buckets] prefix of each bucket
    uint16_t *chunk2p;            // [chunks] prefix of each chunk
    int64_t *start2;              // [nsub_max + 1] first record of each bucket (two == 0: start1)
    unsigned long long *cur2;     // [nsub_max] write cursors of the second pass
    uint32_t *count2;             // [nsub_max + 1]
    int64_t nsub_max;
    int64_t cap;                  // records a buffer holds
    // Two words: the call's errors, and whether a bucket holds more than `limit` records. The bucket ranges
    // come from a scan whose waits are bounded: when one has run out they overlap and a bucket holds records
    // of others, whose bits are no indices any more. Every kernel that uses the ranges returns where
    // either is set.
    uint32_t *stop;
    int64_t limit;
    __device__ __forceinline__ bool stopped() const { return (stop[0] | stop[1]) != 0; }
    // the bucket's prefix, its first code (below the prefix) and its code bits
    __device__ __forceinline__ int prefix(int64_t b) const { return two ? (int)sub2p[b] : (int)b; }
};

// ------------------------------------------------------------------------------ grouping
template <class K>
struct ScatterSmem {
    typename K::T tile[KB_NT * K::ITEMS];
    uint32_t tmp[KB_NT / 32 + 1];
    // then: cnt u32[nb] | gb u64[nb] | (BINARR) bin u16[tile]
};
template <class K, bool BINARR>
inline size_t scatter_smem_bytes(int nb) {
    return sizeof(ScatterSmem<K>) + (size_t)nb * 12 + 8 + (BINARR ? (size_t)kb_tile<K>() * 2 : 0);
}

// The second half of a grouping pass, on records held in registers: br[u] = bin << 16 | rank in
// the bin within the tile, or 0xFFFFFFFF for no record; cnt[] holds the tile's counts. Orders the
// tile by bin in shared memory and writes every bin's run at a place reserved on cur[bin]
// (positions are absolute; the lanes of a warp reserve on consecutive words, one request: cursors 32
// or 128 bytes apart cost 3 and 15 % of the pass). binof(key) recovers a record's bin unless BINARR keeps it; then() runs
// once the records are in shared memory.
struct NoOp {
    __device__ void operator()() const {}
};
template <class K, bool BINARR, class BinOf, class Then = NoOp>
__device__ __forceinline__ void scatter_tail(ScatterSmem<K> &sm, uint32_t *cnt, unsigned long long *gb,
                                             uint16_t *sbin, int nb, typename K::T (&key)[K::ITEMS],
                                             const uint32_t (&br)[K::ITEMS], unsigned long long *__restrict__ cur,
                                             typename K::T *__restrict__ out, int64_t cap, BinOf &&binof, Then &&then = NoOp{}) {
    constexpr int PER = KB_MAXBINS / KB_NT;  // bins t, t + KB_NT, ... belong to thread t
    __syncthreads();
    // runs are reserved first: the atomics travel while the tile is scanned and ordered
    unsigned long long g[PER];
#pragma unroll
    for (int x = 0; x < PER; x++) {
        const int b = x * KB_NT + threadIdx.x;
        const uint32_t c = b < nb ? cnt[b] : 0u;
        g[x] = c ? atomicAdd(cur + b, (unsigned long long)c) : 0ull;
    }
    uint32_t ntot = 0;
#pragma unroll
    for (int x = 0; x < PER; x++) {
        if (x * KB_NT >= nb) break;
        const int b = x * KB_NT + threadIdx.x;
        const uint32_t c = b < nb ? cnt[b] : 0u;
        uint32_t t;
        const uint32_t run = ntot + block_exclusive_scan<KB_NT>(c, sm.tmp, &t);
        if (b < nb) cnt[b] = run;
        ntot += t;
    }
    __syncthreads();
#pragma unroll
    for (int u = 0; u < K::ITEMS; u++)
        if (br[u] != 0xFFFFFFFFu) {
            const uint32_t p = cnt[br[u] >> 16] + (br[u] & 0xFFFFu);
            if (!SG_IN_BOUNDS(p < (uint32_t)kb_tile<K>(), 704, p)) continue;
            sm.tile[p] = key[u];
            if (BINARR) sbin[p] = (uint16_t)(br[u] >> 16);
        }
#pragma unroll
    for (int x = 0; x < PER; x++) {
        const int b = x * KB_NT + threadIdx.x;
        if (b < nb) gb[b] = g[x] - cnt[b];
    }
    then();  // the registers are free
    __syncthreads();
    for (uint32_t i = threadIdx.x; i < ntot; i += KB_NT) {
        const typename K::T k = sm.tile[i];
        const uint32_t b = BINARR ? sbin[i] : binof(k);
        if (SG_IN_BOUNDS(b < (uint32_t)nb && (int64_t)(gb[b] + i) < cap, 705, gb[b] + i)) out[gb[b] + i] = k;
    }
}

// The shared-memory layout behind ScatterSmem.
template <class K>
__device__ __forceinline__ void scatter_layout(unsigned char *raw, int nb, ScatterSmem<K> *&sm, uint32_t *&cnt,
                                               unsigned long long *&gb, uint16_t *&sbin) {
    sm = reinterpret_cast<ScatterSmem<K> *>(raw);
    unsigned char *p = raw + ((sizeof(ScatterSmem<K>) + 7) & ~(size_t)7);
    gb = reinterpret_cast<unsigned long long *>(p);
    cnt = reinterpret_cast<uint32_t *>(p + (size_t)nb * 8);
    sbin = reinterpret_cast<uint16_t *>(p + (size_t)nb * 12);
}

// How skewed the codes are, in bits per code bit: the records that a record meets in its prefix, over the
// mean prefix (4 / 3 for canonical codes of a uniform sequence), go up by a constant factor per bit where the
// bases are independent. s, ss: sums of the prefixes' counts and of their squares. 0 for a uniform
// sequence, 0.03 at 60 % A and T, 0.12 at 70 %, 0.23 at 80 %.
__host__ __device__ inline float kb_skew(float s, float ss, int nb1, int bits) {
    if (s <= 0.0f || bits <= 0) return 0.0f;
    const float f = ss / s / s * (float)nb1 * 0.75f;
    return f > 1.0f ? log2f(f) / (float)bits : 0.0f;
}
constexpr float KB_SKEW_MIN = 0.01f;  // codes count as skewed from here on
constexpr int KB_SMALL_GROW = 2;      // bits that a split of a small input may grow by (bounds its buckets)

// The level-2 split of a prefix of c records, in bits: so many that a bucket holds `target` records on
// average (b2min at least, b2max at most; 0: one level). Where the codes are skewed, the fuller buckets of the
// prefix exceed their mean by skew per bit of the split, and a bit more leaves room for what is above them.
// (By the mean alone 18 % of the records of a genome of 60 % A and T were in buckets above a block's, 63 % at
// 80 %. Finishing 120 M windows, ms: 60 % 2.9 -> 2.2, 65 % 3.8 -> 2.7, 70 % 4.7 -> 3.3, uniform 1.5.)
__host__ __device__ inline int kb_split(int64_t c, int target, int b2max, int b2min, float skew, int grow_max) {
    int b = b2min;
    while (b < b2max && (c >> b) > target) b++;
    if (b > b2min && skew >= KB_SKEW_MIN) {
        const int g = (int)((float)b * skew + 1.3f);
        b += g < grow_max ? g : grow_max;
    }
    return b < b2max ? b : (b2max > b2min ? b2max : b2min);
}

// One block per plan: prefix counts -> record ranges, level-2 split, buckets and chunks.
// b2max bounds the split (0: one level). minb2: at least this many bits (rows per bucket bound).
// skew < 0: found here, and the split grows by KB_SMALL_GROW bits at most. From skew_max on, stop[1] is set.
__global__ void __launch_bounds__(1024) kb_plan_kernel(const unsigned long long *__restrict__ hist, KbPlan pl,
                                                      int target, int b2max, int b2min, float skew, float skew_max, int pb1,
                                                      int chunk);

// Level-2 counts: a chunk of one prefix's records per block. Bound by memory: 4.1e9 records of 8 bytes
// 4.5 ms, 7.3 TB/s.
template <class K>
__global__ void __launch_bounds__(KB_NT) kb_hist2_kernel(KbPlan pl, const typename K::T *__restrict__ in,
                                                        int lowbits) {
    __shared__ uint32_t cnt[KB_MAXBINS];
    if (blockIdx.x >= pl.chunk2[pl.nb1]) return;
    const bool stop = pl.stopped();  // no records were written
    const int p = pl.chunk2p[blockIdx.x];
    for (int i = threadIdx.x; i < KB_MAXBINS; i += KB_NT) cnt[i] = 0;
    __syncthreads();
    if (stop) return;
    const int b = pl.b2[p], sh = pl.rem - b;
    const int64_t c0 = pl.start1[p], c1 = pl.start1[p + 1];
    constexpr int64_t CH = (int64_t)KB_CHUNK_TILES * kb_tile<K>();
    const int64_t a0 = c0 + (int64_t)(blockIdx.x - pl.chunk2[p]) * CH;
    const int64_t a1 = a0 + CH < c1 ? a0 + CH : c1;
    constexpr int U = 8;  // loads in flight
    for (int64_t i = a0 + threadIdx.x; i < a1; i += U * KB_NT) {
        typename K::T k[U];
#pragma unroll
        for (int u = 0; u < U; u++) k[u] = i + u * KB_NT < a1 ? K::load(in + i + u * KB_NT) : K::none();
#pragma unroll
        for (int u = 0; u < U; u++)
            if (i + u * KB_NT < a1 && SG_IN_BOUNDS((K::code(k[u], lowbits) >> sh) < (uint64_t)(1 << b), 706, i))
                atomicAdd(cnt + (uint32_t)(K::code(k[u], lowbits) >> sh), 1u);
    }
    __syncthreads();
    for (int i = threadIdx.x; i < (1 << b); i += KB_NT)
        if (cnt[i]) atomicAdd(pl.count2 + pl.sb[p] + i, cnt[i]);
}

// Level-2 grouping: a chunk of one prefix's records per block, tile by tile; the next tile's loads
// travel while this one is written. 4.1e9 records of 8 bytes (100 Mbp, 40x): 18.6 ms, 3.5 TB/s;
// one tile per block, its prefix searched for by one thread first, 21.7 ms.
template <class K>
__global__ void __launch_bounds__(KB_NT, 2) kb_scatter2_kernel(KbPlan pl, const typename K::T *__restrict__ in,
                                                              typename K::T *__restrict__ out, int lowbits) {
    extern __shared__ __align__(16) unsigned char kb_raw[];
    const uint32_t chunk = blockIdx.x;
    if (chunk >= pl.chunk2[pl.nb1]) return;
    const int p = pl.chunk2p[chunk];
    constexpr int TILE = kb_tile<K>();
    const int64_t a0 = pl.start1[p] + (int64_t)(chunk - pl.chunk2[p]) * KB_CHUNK_TILES * TILE;
    const int64_t end = pl.start1[p + 1];
    const int64_t a1 = a0 + KB_CHUNK_TILES * TILE < end ? a0 + KB_CHUNK_TILES * TILE : end;
    const int b = pl.b2[p], sh = pl.rem - b, nb = 1 << b;
    ScatterSmem<K> *sm;
    uint32_t *cnt;
    unsigned long long *gb;
    uint16_t *sbin;
    scatter_layout<K>(kb_raw, nb, sm, cnt, gb, sbin);
    typename K::T key[K::ITEMS];
    auto load = [&](int64_t t0) {
#pragma unroll
        for (int u = 0; u < K::ITEMS; u++) {
            const int64_t i = t0 + u * KB_NT + threadIdx.x;
            key[u] = i < a1 ? K::load(in + i) : K::none();
        }
    };
    load(a0);
    if (pl.stopped()) return;  // tested behind the loads: their latency hides its own
    for (int64_t t0 = a0; t0 < a1; t0 += TILE) {
        for (int i = threadIdx.x; i < nb; i += KB_NT) cnt[i] = 0;
        __syncthreads();
        uint32_t br[K::ITEMS];
#pragma unroll
        for (int u = 0; u < K::ITEMS; u++) {
            const int64_t i = t0 + u * KB_NT + threadIdx.x;
            br[u] = 0xFFFFFFFFu;
            if (i < a1) {
                const uint32_t s = K::slot(key[u], 0ull, lowbits, sh);
                if (SG_IN_BOUNDS(s < (uint32_t)nb, 707, s)) br[u] = (s << 16) | atomicAdd(cnt + s, 1u);
            }
        }
        scatter_tail<K, false>(*sm, cnt, gb, nullptr, nb, key, br, pl.cur2 + pl.sb[p], out, pl.cap,
                               [&](const typename K::T &k) { return K::slot(k, 0ull, lowbits, sh); },
                               [&] { if (t0 + TILE < a1) load(t0 + TILE); });
        __syncthreads();
    }
}

// ----------------------------------------------------------------------------- finishing
// Slot counters of 16 bits, two per word; four pad words after every 16, so that threads scanning
// 16 consecutive words with 16-byte loads hit distinct banks.
__device__ __forceinline__ int slot_pad(int w) { return w + (w >> 4) * 4; }
constexpr int KB_SLOT_WORDS = (1 << (KB_NS - 1)) + (1 << (KB_NS - 3)) + 8;

constexpr int KB_PIECE_BITS = 13;  // code bits by which a piece too large for a block is split, at most
constexpr int KB_PIECES = 112;     // pending pieces of an oversized bucket

// Records [off, off + len) of an oversized bucket with codes in [c0, cend), in the bucket's range of the
// input (where == 0) or of the other buffer. len above a block's records: they agree in the code bits
// from `bits` on; split: they are in order of the next KB_PIECE_BITS already.
struct KbPiece {
    uint64_t c0, cend;
    uint32_t off, len;
    uint8_t bits, where, split;
};

template <class K>
struct FinishSmem {
    typename K::T sk[KB_NT * K::ITEMS];   // records by slot
    uint32_t slots[KB_SLOT_WORDS];
    uint32_t bits[KB_NT * K::ITEMS / 32], wpre[KB_NT * K::ITEMS / 32 + 1];
    uint32_t heads[KB_NT * K::ITEMS / 32 + 2];   // bit i + 32: record i of sk starts a slot
    uint32_t codes[KB_NT * K::ITEMS / 32 + 2];   // ... (in order) a code
    uint32_t tmp[KB_NT / 32 + 1];
    uint32_t nseg;
    uint32_t crowd;                              // sum of the placed records' ranks in their slots
    int npiece;
    KbPiece piece[KB_PIECES];
};

}  // namespace sg

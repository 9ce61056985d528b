// kbucket.cu -- the bucketed k-mer stage (reads -> At) and A = At transposed.
//
// Exact counting needs every occurrence of a k-mer in one place. Instead of filtering the windows
// and sorting the survivors by 8-bit digits, every valid window becomes one record (code, read,
// position, strand) that is grouped by the top bits of its code in at most two passes, until a
// bucket of about 7 K records fits one block's shared memory; the block then finishes the bucket:
// exact frequency, reliable range, the lowest position of each read, code order. Passes:
//  1. pack      bases to 2 bits (32 per word), a mask of the valid windows and the read of every
//               group of 32, and the number of windows per code prefix.
//  2. scatter1  windows -> records grouped by prefix.
//  3. hist2, scatter2 (large inputs)  records grouped by the next bits.
//  4. finish    per bucket: the kept records (first of their read in a reliable segment), in
//               (code, read) order, and their number and the number of reliable codes.
//  5. emit      after scans of those numbers: At, the column codes.
//  6. A         At's entries grouped by read the same way, each row ordered by column.
// The singleton filters of the two-pass count (Sec. IV-C) save memory traffic only where most
// windows are singletons and cost one random probe per window; here a singleton costs its share of
// three or four streaming passes, and drops out when its slot counts one record.
//
// 4.1 G windows, 1.77 G entries of A (100 Mbp at 40x, k = 17), ms: pack 4, scatter1 25, hist2 4.5,
// scatter2 18, finish 50, emit 8.5, A 43 (scatter1 11.8, hist2 2, scatter2 7, rows 21.5): 154 in all,
// against 387 for filters, sorts and segment passes (the general form in kmer.cu with a radix sort of
// A). 154 M windows (5 Mbp at 30x): 4.5 against 5.9; k = 31, 300 M windows: 24 against 58 (16-byte
// records, eight radix passes). These are uniform sequences; what skewed ones cost is told where the split
// of the prefixes, the oversized buckets and the crowded slots are dealt with.
#include <algorithm>
#include <vector>

#include "bucket.cuh"
#include "check.cuh"
#include "kmer.cuh"
#include "ops.cuh"

namespace sg {

static inline int64_t blocks_for(int64_t n, int nt) { return (n + nt - 1) / nt; }

__global__ void __launch_bounds__(1024) kb_plan_kernel(const unsigned long long *__restrict__ hist, KbPlan pl,
                                                      int target, int b2max, int b2min, float skew, float skew_max, int pb1,
                                                      int chunk) {
    __shared__ int64_t t64[33];
    __shared__ uint32_t t32[33];
    __shared__ int64_t s_base;
    __shared__ uint32_t s_sub, s_chk;
    __shared__ float s_s, s_ss;
    if (threadIdx.x == 0) {
        s_base = 0;
        s_sub = 0;
        s_chk = 0;
        s_s = s_ss = 0.0f;
    }
    __syncthreads();
    const int grow_max = skew < 0.0f ? KB_SMALL_GROW : KB_MAXB2;
    if (skew < 0.0f) {
        float s = 0.0f, ss = 0.0f;
        for (int p = threadIdx.x; p < pl.nb1; p += 1024) {
            const float c = (float)hist[p];
            s += c;
            ss += c * c;
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            s += __shfl_xor_sync(0xffffffffu, s, o);
            ss += __shfl_xor_sync(0xffffffffu, ss, o);
        }
        if ((threadIdx.x & 31) == 0) {
            atomicAdd(&s_s, s);
            atomicAdd(&s_ss, ss);
        }
        __syncthreads();
        skew = kb_skew(s_s, s_ss, pl.nb1, pb1);
    }
    if (threadIdx.x == 0 && skew >= skew_max) pl.stop[1] = 1;
    for (int p0 = 0; p0 < pl.nb1; p0 += 1024) {
        const int p = p0 + threadIdx.x;
        const int64_t c = p < pl.nb1 ? (int64_t)hist[p] : 0;
        const int b = kb_split(c, target, b2max, b2min, skew, grow_max);
        const uint32_t nch = p < pl.nb1 ? (uint32_t)((c + chunk - 1) / chunk) : 0u;
        int64_t tot;
        uint32_t stot, ctot;
        const int64_t st = s_base + block_exclusive_scan<1024, int64_t>(c, t64, &tot);
        const uint32_t sub = s_sub + block_exclusive_scan<1024, uint32_t>(p < pl.nb1 ? 1u << b : 0u, t32, &stot);
        const uint32_t chk = s_chk + block_exclusive_scan<1024, uint32_t>(nch, t32, &ctot);
        if (!pl.two && c > pl.limit) pl.stop[1] = 1;
        if (p < pl.nb1) {
            pl.start1[p] = st;
            pl.cur1[p] = (unsigned long long)st;
            pl.b2[p] = (uint8_t)b;
            pl.sb[p] = sub;
            pl.chunk2[p] = chk;
            if (p == pl.nb1 - 1) {
                pl.start1[pl.nb1] = st + c;
                pl.sb[pl.nb1] = sub + (1u << b);
                pl.chunk2[pl.nb1] = chk + nch;
            }
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            s_base += tot;
            s_sub += stot;
            s_chk += ctot;
        }
        __syncthreads();
    }
}

// The prefixes of the buckets and of the chunks: one warp per prefix.
__global__ void kb_sub2p_kernel(KbPlan pl) {
    const int p = (int)(((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5);
    if (p >= pl.nb1) return;
    for (uint32_t x = pl.sb[p] + (threadIdx.x & 31); x < pl.sb[p + 1]; x += 32)
        if (SG_IN_BOUNDS((int64_t)x < pl.nsub_max, 701, x)) pl.sub2p[x] = (uint16_t)p;
    for (uint32_t x = pl.chunk2[p] + (threadIdx.x & 31); x < pl.chunk2[p + 1]; x += 32) pl.chunk2p[x] = (uint16_t)p;
}

// Level-2 write cursors, and whether a bucket is too large for one block.
__global__ void kb_cursors_kernel(KbPlan pl) {
    const int64_t b = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= pl.nsub_max) return;
    pl.cur2[b] = (unsigned long long)pl.start2[b];
    if ((int64_t)pl.count2[b] > pl.limit) pl.stop[1] = 1;
}

// ----------------------------------------------------------------------------------- pack
// Offsets: the same checks as the general path's, and the longest read.
__global__ void kb_offsets_kernel(const int64_t *__restrict__ off, int64_t n, int64_t total,
                                  uint32_t *__restrict__ err, unsigned long long *__restrict__ maxlen) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    int64_t len = 0;
    bool bad = false;
    if (i <= n) {
        const int64_t a = off[i];
        if (i == 0 && a != 0) bad = true;
        if (i == n && a != total) bad = true;
        if (i < n) {
            len = off[i + 1] - a;
            if (len < 0 || len >= ((int64_t)1 << 31)) bad = true;
        }
    }
    if (bad) atomicOr(err, (uint32_t)DEV_INVALID);
    const uint32_t l = len > 0 ? (uint32_t)(len < 0x7FFFFFFF ? len : 0x7FFFFFFF) : 0u;
    const uint32_t m = __reduce_max_sync(0xffffffffu, l);
    if ((threadIdx.x & 31) == 0 && m) atomicMax(maxlen, (unsigned long long)m);
}

sg_status check_offsets(const int64_t *off, int64_t n, int64_t total, uint32_t *err, unsigned long long *maxlen,
                        cudaStream_t s) {
    SG_LAUNCH("validate_offsets", kb_offsets_kernel, blocks_for(n + 1, 256), 256, 0, s, off, n, total, err, maxlen);
    return SG_OK;
}

// From read r, a read starting at or before q: the last one that does.
__device__ __forceinline__ int64_t read_from(const int64_t *__restrict__ off, int64_t n, int64_t r, int64_t q) {
    int64_t step = 1;
    while (r + step < n && off[r + step] <= q) {
        r += step;
        step *= 2;
    }
    int64_t hi = r + step < n ? r + step : n;
    while (hi - r > 1) {
        const int64_t mid = (r + hi) >> 1;
        if (off[mid] <= q) r = mid; else hi = mid;
    }
    return r;
}

// Four bases (one per byte): their 2-bit codes in the low 8 bits (A=0 C=1 G=2 T=3, first base
// lowest) and a mask of the valid ones. The two bits above the lowest of an upper-case letter tell
// A, C, T, G apart; looking the letter up again and comparing tells whether the byte is one of them.
__device__ __forceinline__ void pack4(uint32_t w, uint32_t &code, uint32_t &ok) {
    const uint32_t t = (w >> 1) & 0x03030303u;
    uint32_t x = t | (t >> 4);
    x = (x & 0xffu) | ((x >> 8) & 0xff00u);  // selector nibbles t0, t1, t2, t3
    const uint32_t e = __byte_perm(0x47544341u, 0u, x) ^ w;  // A C T G by t
    if (e == 0) {
        ok = 0xFu;
    } else {
        ok = 0;
#pragma unroll
        for (int u = 0; u < 4; u++) ok |= (uint32_t)(((e >> (8 * u)) & 0xffu) == 0) << u;
    }
    uint32_t b = t ^ ((t >> 1) & 0x01010101u);
    b = (b | (b >> 6)) & 0x000f000fu;
    code = (b | (b >> 12)) & 0xffu;
}

// One group of 32 bases per lane, lane 31 only as the next group of lane 30 (a window needs up to
// 31 bases past its group): a warp handles 31 groups per step, in consecutive steps, so that the
// read of a group is found from the previous step's by a short gallop. P, VM and RG as in WindowSrc.
// Bound by the prefix counts' shared-memory atomics and their code arithmetic, unrolled so that shifts
// are immediates: 4.1e9 windows 3.8 ms (1.6 TB/s); a rolling encode and hash per window took 12.
constexpr int PK_NT = 256;
constexpr int PK_G = 31;

__global__ void __launch_bounds__(PK_NT) kb_pack_kernel(const uint8_t *__restrict__ seq, int64_t total,
                                                       const int64_t *__restrict__ off, int64_t n, int k, JobPos jp,
                                                       int pb1, int job_bits, int64_t ngroups, int64_t steps_per_warp,
                                                       uint64_t *__restrict__ P, uint32_t *__restrict__ VM,
                                                       int32_t *__restrict__ RG,
                                                       unsigned long long *__restrict__ hist) {
    extern __shared__ uint32_t pk_hist[];  // [2^pb1]
    const int nb = 1 << pb1;
    for (int i = threadIdx.x; i < nb; i += PK_NT) pk_hist[i] = 0;
    __syncthreads();
    const int lane = threadIdx.x & 31;
    const int64_t warp = ((int64_t)blockIdx.x * PK_NT + threadIdx.x) >> 5;
    const bool al = ((uintptr_t)seq & 15) == 0;
    const int tb = pb1 - job_bits;  // code bits in the prefix (below the job's), if positive
    const uint32_t tmask = tb > 0 ? (1u << tb) - 1u : 0u;
    int64_t r = 0;
    JobPosCursor jc{jp};
    for (int64_t st = 0; st < steps_per_warp; st++) {
        const int64_t g0 = (warp * steps_per_warp + st) * PK_G;
        if (g0 >= ngroups) break;
        const int64_t g = g0 + lane, qs = g * 32;
        uint64_t pw = 0;
        uint32_t ok = 0;
        if (qs + 32 <= total && al) {
            const uint4 a = __ldcs(reinterpret_cast<const uint4 *>(seq + qs));
            const uint4 b = __ldcs(reinterpret_cast<const uint4 *>(seq + qs) + 1);
            const uint32_t w[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
#pragma unroll
            for (int u = 0; u < 8; u++) {
                uint32_t c, v;
                pack4(w[u], c, v);
                pw |= (uint64_t)c << (8 * u);
                ok |= v << (4 * u);
            }
        } else if (qs < total) {
#pragma unroll 1
            for (int u = 0; u < 8; u++) {
                uint32_t w = 0, c, v;
                for (int x = 0; x < 4; x++) {
                    const int64_t q = qs + 4 * u + x;
                    w |= (uint32_t)(q < total ? seq[q] : (uint8_t)'N') << (8 * x);
                }
                pack4(w, c, v);
                pw |= (uint64_t)c << (8 * u);
                ok |= v << (4 * u);
            }
        }
        const uint64_t pn = __shfl_down_sync(0xffffffffu, pw, 1);
        const uint32_t okn = __shfl_down_sync(0xffffffffu, ok, 1);
        if (lane == 31 || g >= ngroups) continue;  // no warp-wide operation below in this step
        // windows whose k bases are all valid
        uint64_t m64 = (uint64_t)ok | ((uint64_t)okn << 32);
        int len = 1;
        while (2 * len <= k) {
            m64 &= m64 >> len;
            len *= 2;
        }
        if (len < k) m64 &= m64 >> (k - len);
        uint32_t vm = (uint32_t)m64;
        // the read holding qs (the last r with off[r] <= qs): from this lane's last one
        r = read_from(off, n, r, qs);
        // windows that cross a read end
        for (int64_t rr = r;;) {
            const int64_t e = off[rr + 1] - qs;
            if (e >= 32 + k - 1) break;
            const int lo = e - k + 1 > 0 ? (int)(e - k + 1) : 0, hi = e < 32 ? (int)e : 32;
            if (hi > lo) vm &= ~((hi >= 32 ? 0xffffffffu : (1u << hi) - 1u) & ~((1u << lo) - 1u));
            const int64_t nx = read_from(off, n, rr, qs + e);  // skips empty reads
            if (nx == rr) break;
            rr = nx;
        }
        P[g] = pw;
        VM[g] = vm;
        RG[g] = (int32_t)r;
        if (vm == 0) continue;
        // prefixes: the top bits of the smaller of two codes are the smaller of their top bits
        const uint32_t L[4] = {(uint32_t)pw, (uint32_t)(pw >> 32), (uint32_t)pn, (uint32_t)(pn >> 32)};
        uint32_t B[3], M[4];
#pragma unroll
        for (int x = 0; x < 3; x++) {
            uint32_t y = __brev(L[x]);
            B[x] = ((y >> 1) & 0x55555555u) | ((y & 0x55555555u) << 1);  // first base highest
        }
        const int s = 2 * k - tb;
        {
            const uint64_t lo = s >= 64 ? 0 : (s ? (pw >> s) | (pn << (64 - s)) : pw), hi = s >= 64 ? 0 : pn >> s;
            M[0] = (uint32_t)lo;
            M[1] = (uint32_t)(lo >> 32);
            M[2] = (uint32_t)hi;
            M[3] = (uint32_t)(hi >> 32);
        }
        // a group inside one read set: its prefix once
        const uint32_t job = jp.jpos ? (uint32_t)(jc.prefix(qs) >> jp.kbits) : 0u;
        if (tb > 0 && (!jp.jpos || qs + 32 <= jc.jhi)) {
            const uint32_t jb = job << tb;
#pragma unroll
            for (int j = 0; j < 32; j++) {
                if (!((vm >> j) & 1u)) continue;
                const uint32_t fw = __funnelshift_l(B[j / 16 + 1], B[j / 16], 2 * (j % 16)) >> (32 - tb);
                const uint32_t rc = ~__funnelshift_r(M[j / 16], M[j / 16 + 1], 2 * (j % 16)) & tmask;
                atomicAdd(pk_hist + (jb | (fw < rc ? fw : rc)), 1u);
            }
        } else {
#pragma unroll 1
            for (int j = 0; j < 32; j++) {
                if (!((vm >> j) & 1u)) continue;
                const uint64_t job = jc.prefix(qs + j) >> jp.kbits;
                uint32_t b;
                if (tb > 0) {
                    const uint64_t x = j ? (pw >> (2 * j)) | (pn << (64 - 2 * j)) : pw;
                    uint64_t y = __brevll(x);
                    y = ((y >> 1) & 0x5555555555555555ull) | ((y & 0x5555555555555555ull) << 1);
                    const uint32_t fw = (uint32_t)(y >> (64 - tb));
                    const uint32_t rc = (uint32_t)(~x >> s) & tmask;
                    b = ((uint32_t)job << tb) | (fw < rc ? fw : rc);
                } else {
                    b = (uint32_t)(job >> -tb);
                }
                if (SG_IN_BOUNDS(b < (uint32_t)nb, 702, b) && b < (uint32_t)nb) atomicAdd(pk_hist + b, 1u);
            }
        }
    }
    __syncthreads();
    for (int i = threadIdx.x; i < nb; i += PK_NT)
        if (pk_hist[i]) atomicAdd(hist + i, (unsigned long long)pk_hist[i]);
}

// ------------------------------------------------------------------------------- scatter 1
// Windows as records: group g of 32 windows has its bases in P[g] and P[g + 1], bit l of VM[g] set
// where window 32 g + l is valid, and RG[g] the read holding base 32 g.
struct WindowSrc {
    const uint64_t *P;
    const uint32_t *VM;
    const int32_t *RG;
    const int64_t *off;
    int64_t n, ngroups;
    int k;
    JobPos jp;
    int rem;
    KeyBits kb;
};

// KK > 0: k as a compile-time constant. JOBS: a batch. A warp's groups are described in shared memory,
// so that a window costs two broadcast loads and 32-bit operations (by shuffles: 26.0 ms instead of 25.2
// for 4.1e9 windows). Bound by shared memory: a window is counted, placed with its bin, read back and
// written in runs of about eight records (1.3 TB/s written).
template <class K, int KK, bool JOBS>
__global__ void __launch_bounds__(KB_NT, 2) kb_scatter1_kernel(WindowSrc w, KbPlan pl,
                                                              typename K::T *__restrict__ out) {
    extern __shared__ __align__(16) unsigned char kb_raw[];
    ScatterSmem<K> *sm;
    uint32_t *cnt;
    unsigned long long *gb;
    uint16_t *sbin;
    const int nb = pl.nb1, k = KK > 0 ? KK : w.k;
    scatter_layout<K>(kb_raw, nb, sm, cnt, gb, sbin);
    const int lane = threadIdx.x & 31;
    const int64_t g0 = ((int64_t)blockIdx.x * (KB_NT / 32) + (threadIdx.x >> 5)) * K::ITEMS;
    // group g0 + u of the warp: bases; valid windows, the read at its start, the position of its first
    // base in that read and where the next read starts (relative, at most 32)
    __shared__ uint64_t s_bases[KB_NT / 32][K::ITEMS + 1];
    __shared__ uint4 s_group[KB_NT / 32][K::ITEMS];
    const int warp = threadIdx.x >> 5;
    {
        const int64_t g = g0 + lane;
        if (lane <= K::ITEMS) s_bases[warp][lane] = g <= w.ngroups ? w.P[g] : 0ull;
        if (lane < K::ITEMS) {
            uint4 d = make_uint4(0u, 0u, 0u, 32u);
            if (g < w.ngroups) {
                const int32_t r = w.RG[g];
                const int64_t e = w.off[r + 1] - g * 32;
                d = make_uint4(w.VM[g], (uint32_t)r, (uint32_t)(g * 32 - w.off[r]), e < 32 ? (uint32_t)e : 32u);
            }
            s_group[warp][lane] = d;
        }
    }
    if (pl.stopped()) return;
    for (int i = threadIdx.x; i < nb; i += KB_NT) cnt[i] = 0;
    __syncthreads();
    const uint64_t rmask = (1ull << w.kb.rbits) - 1;
    const uint32_t pmask = w.kb.pbits < 32 ? (1u << w.kb.pbits) - 1u : 0xffffffffu;
    const uint64_t remmask = w.rem < 64 ? (1ull << w.rem) - 1 : ~0ull;
    const uint64_t kmask = (1ull << (2 * k)) - 1;
    const int lowbits = w.kb.low(), rsh = w.kb.pbits + 1;
    JobPosCursor jc{w.jp};
    typename K::T key[K::ITEMS];
    uint32_t br[K::ITEMS];
    uint64_t pn = s_bases[warp][0];
#pragma unroll
    for (int u = 0; u < K::ITEMS; u++) {
        br[u] = 0xFFFFFFFFu;
        key[u] = K::none();
        const uint64_t p0 = pn;
        pn = s_bases[warp][u + 1];
        const uint4 d = s_group[warp][u];
        const uint32_t a0 = (uint32_t)p0, a1 = (uint32_t)(p0 >> 32), a2 = (uint32_t)pn, a3 = (uint32_t)(pn >> 32);
        const uint32_t vm = d.x;
        int64_t r = (int32_t)d.y;
        uint32_t pos = d.z + lane;
        const int next = (int)d.w;
        if (!((vm >> lane) & 1u)) continue;
        if (lane >= next) {  // a read that starts inside the group
            const int64_t q = (g0 + u) * 32 + lane;
            r = read_from(w.off, w.n, r, q);
            pos = (uint32_t)(q - w.off[r]);
        }
        // the 2k bits from bit 2 lane, first base lowest; the reverse complement's code is their
        // complement, the forward code the 2-bit groups in reverse order
        const bool up = lane >= 16;
        const uint32_t b0 = up ? a1 : a0, b1 = up ? a2 : a1, b2 = up ? a3 : a2;
        const uint64_t x = ((uint64_t)__funnelshift_r(b1, b2, 2 * lane) << 32) | __funnelshift_r(b0, b1, 2 * lane);
        const uint64_t rc = ~x & kmask;
        uint64_t y = __brevll(x);
        y = ((y >> 1) & 0x5555555555555555ull) | ((y & 0x5555555555555555ull) << 1);
        const uint64_t fw = y >> (64 - 2 * k);
        const bool strand = rc < fw;
        uint64_t code = strand ? rc : fw;
        if (JOBS) code |= jc.prefix((g0 + u) * 32 + lane);
        const uint32_t b = low_bits_at(code, w.rem);
        if (b >= (uint32_t)nb) continue;  // cannot happen for valid offsets
        key[u] = K::make(code & remmask, (((uint64_t)r & rmask) << rsh) | ((uint64_t)(pos & pmask) << 1) | (strand ? 1u : 0u),
                         lowbits);
        br[u] = (b << 16) | atomicAdd(cnt + b, 1u);
    }
    scatter_tail<K, true>(*sm, cnt, gb, sbin, nb, key, br, pl.cur1, out, pl.cap,
                          [](const typename K::T &) { return 0u; });
}

// --------------------------------------------------------------------------------- finish
// What a finishing block does with a bucket's records.
//   count: keeps the first record of each read among those of every code whose frequency lies in
//          [lo, hi] (lohi: per job), writes them in order to out at the bucket's own range.
//   order: (records of At grouped by read, code = read << cbits | column) writes column and value
//          in order at the bucket's range, and the row pointers of the bucket's reads.
struct FinishArgs {
    KbPlan pl;
    KeyBits kb;
    // count
    uint32_t lo, hi, hmax;  // hmax: no range reaches above it
    const uint32_t *lohi;
    int kbits;
    uint32_t *nseg, *nkeep;
    // order
    int cbits;
    int64_t n_rows, nnz;
    int32_t *col;
    uint32_t *val;
    int64_t *rp;
};

// Ranking compares a record with its whole slot, so crowded slots cost the square of their records: codes
// of high frequency (deep coverage under a high hi, or copies of a satellite where a slot is several codes and
// none can be dropped before). Where the pairs to be compared, counted as the sum of the records' ranks,
// pass this many per record of a full block, the block sorts the bucket instead; both cost about the same
// there. 180 M windows at 900x, hi = 1,000: k = 31 98 -> 21 ms, k = 17 47 -> 14 ms; 300 M windows, 30 % of them
// of a satellite, k = 31: 35 -> 26 ms.
constexpr uint32_t KB_CROWD = 64;

// sk[0, n) in ascending order, by the whole block: a bitonic network whose first step of every merge
// pairs mirrored places, so that the smaller key always goes to the lower place and places from n on may
// be left out.
template <class K>
__device__ __noinline__ void sort_block(typename K::T *sk, int n) {
    auto order = [&](int i, int j) {
        if (j >= n) return;
        const typename K::T x = sk[i], y = sk[j];
        if (K::less(y, x)) {
            sk[i] = y;
            sk[j] = x;
        }
    };
    int half = 1;  // n <= 2 half
    while (2 * half < n) half *= 2;
    for (int lk = 1; (1 << lk) <= 2 * half; lk++) {
        const int h = 1 << (lk - 1);
        for (int t = threadIdx.x; t < half; t += KB_NT) {
            const int i = ((t >> (lk - 1)) << lk) | (t & (h - 1));
            order(i, i ^ ((1 << lk) - 1));
        }
        __syncthreads();
        for (int lh = lk - 2; lh >= 0; lh--) {
            for (int t = threadIdx.x; t < half; t += KB_NT) {
                const int i = ((t >> lh) << (lh + 1)) | (t & ((1 << lh) - 1));
                order(i, i + (1 << lh));
            }
            __syncthreads();
        }
    }
}

// Finishes n <= tile records held in registers (record u * KB_NT + thread), whose codes lie in
// [c0, cend), at most 2^ls << sh wide: slot = (code - c0) >> sh. Returns the number of records
// written, from base on. All threads call it. Loops over a thread's records end, for the whole
// block, where its records do.
// Bound by its chain of shared-memory phases, about 12 ps a record (4.1e9 records 50 ms; when 52): load and count
// 11 ms, slot starts 5, placing 10, ranking within a slot 11.5, codes 3, keeping 5, writing 6. Blocks of
// 256 threads with half the records 57 ms; the next bucket's records prefetched 60. Counting first drops
// the records that are alone in their slot, so a singleton is neither placed nor ranked.
template <class K, bool COUNT>
__device__ __forceinline__ uint32_t finish_group(FinishSmem<K> &sm, const FinishArgs &a, int p,
                                                 typename K::T (&key)[K::ITEMS], int n, uint64_t c0,
                                                 uint64_t cend, int sh, int ls, int64_t base,
                                                 typename K::T *__restrict__ out) {
    using T = typename K::T;
    const int lowbits = a.kb.low(), tid = threadIdx.x;
    const int W = ls > 0 ? 1 << (ls - 1) : 1;
    const uint64_t sbase = K::slot_base(c0, lowbits);
    auto slot_of = [&](const T &k) { return K::slot(k, sbase, lowbits, sh); };
    // records of a slot that are kept for the ranking: not a lone one (a singleton, where lo >= 2);
    // where a slot is one code, none of a code outside every range. Both counts of a word at once:
    // bit 15 of c + (0x8000 - least) says c >= least, of c + (0x7fff - most) that c > most
    const bool exact = COUNT && sh == 0;
    const uint32_t least = exact ? (a.lo < 0x7fffu ? a.lo : 0x7fffu) : (a.lo >= 2 ? 2u : 0u);
    const uint32_t most = exact && a.hmax < 0x7fffu ? a.hmax : 0x7fffu;
    const uint32_t ge = (0x8000u - least) * 0x10001u, gt = (0x7fffu - most) * 0x10001u;
    auto mask = [&](uint32_t v) { return ((((v + ge) & ~(v + gt)) & 0x80008000u) >> 15) * 0xffffu; };
    auto eff = [&](uint32_t v) { return COUNT ? v & mask(v) : v; };
    for (int w = tid; w <= slot_pad(W) / 4; w += KB_NT) reinterpret_cast<uint4 *>(sm.slots)[w] = make_uint4(0, 0, 0, 0);
    if (tid < K::ITEMS * KB_NT / 32 + 2) sm.heads[tid] = 0;
    if (tid == 0) sm.nseg = sm.crowd = 0;
    __syncthreads();
    uint32_t rk[(K::ITEMS + 1) / 2];
#pragma unroll
    for (int u = 0; u < K::ITEMS; u++) {
        if (u * KB_NT >= n) break;
        uint32_t r = 0;
        if (u * KB_NT + tid < n) {
            const uint32_t s = slot_of(key[u]), h = (s & 1u) * 16u;
            if (SG_IN_BOUNDS(s < (1u << ls), 708, s))
                r = (atomicAdd(sm.slots + slot_pad((int)(s >> 1)), 1u << h) >> h) & 0xffffu;
        }
        if (u & 1) rk[u / 2] |= r << 16; else rk[u / 2] = r;
    }
    __syncthreads();
    // slot counts -> first record of each slot, 1 to 16 words per thread
    const int pw = (W + KB_NT - 1) / KB_NT;
    uint32_t tot;
    auto step = [&](uint32_t c, uint32_t &ex) {  // a dropped (or empty) slot starts at 0xffff
        const uint32_t m = COUNT ? mask(c) : 0xffffffffu, v = c & m, o0 = ex, o1 = ex + (v & 0xffffu);
        ex = o1 + (v >> 16);
        return (o0 | (o1 << 16)) | ~m;
    };
    if (pw < 4) {
        const int w0 = tid * pw, w1 = w0 + pw < W ? w0 + pw : W;
        uint32_t sum = 0;
        for (int w = w0; w < w1; w++) sum = __dp2a_lo(eff(sm.slots[slot_pad(w)]), 0x0101u, sum);
        uint32_t ex = block_exclusive_scan<KB_NT>(sum, sm.tmp, &tot);
        for (int w = w0; w < w1; w++) {
            sm.slots[slot_pad(w)] = step(sm.slots[slot_pad(w)], ex);
        }
    } else {  // W = pw * KB_NT, pw a power of two: whole groups of 4 words
        uint4 *mine = reinterpret_cast<uint4 *>(sm.slots + slot_pad(tid * pw));
        uint32_t sum = 0;
        for (int x = 0; x < pw / 4; x++) {
            const uint4 v = mine[x];
            sum = __dp2a_lo(eff(v.x), 0x0101u, sum);
            sum = __dp2a_lo(eff(v.y), 0x0101u, sum);
            sum = __dp2a_lo(eff(v.z), 0x0101u, sum);
            sum = __dp2a_lo(eff(v.w), 0x0101u, sum);
        }
        uint32_t ex = block_exclusive_scan<KB_NT>(sum, sm.tmp, &tot);
        for (int x = 0; x < pw / 4; x++) {
            uint4 v = mine[x];
            v.x = step(v.x, ex);
            v.y = step(v.y, ex);
            v.z = step(v.z, ex);
            v.w = step(v.w, ex);
            mine[x] = v;
        }
    }
    if (tid == 0) sm.slots[slot_pad(W)] = tot;
    __syncthreads();
    auto off = [&](uint32_t s) { return (sm.slots[slot_pad((int)(s >> 1))] >> ((s & 1u) * 16u)) & 0xffffu; };
    uint32_t crowd = 0;
#pragma unroll
    for (int u = 0; u < K::ITEMS; u++) {
        if (u * KB_NT >= n) break;
        if (u * KB_NT + tid >= n) continue;
        const uint32_t o = off(slot_of(key[u])), r = (rk[u / 2] >> (16 * (u & 1))) & 0xffffu;
        if (COUNT && o == 0xffffu) continue;
        if (SG_IN_BOUNDS(o + r < (uint32_t)kb_tile<K>(), 712, o + r)) sm.sk[o + r] = key[u];
        if (r == 0) atomicOr(sm.heads + 1 + (o >> 5), 1u << (o & 31u));
        crowd += r;
    }
    crowd = __reduce_add_sync(0xffffffffu, crowd);
    if ((tid & 31) == 0 && crowd > KB_CROWD) atomicAdd(&sm.crowd, crowd);
    const int ne = (int)tot;
    if (tid == 0) atomicOr(sm.heads + 1 + (ne >> 5), 1u << (ne & 31));
    __syncthreads();
    const bool crowded = sm.crowd > KB_CROWD * (uint32_t)kb_tile<K>();
    if (crowded) sort_block<K>(sm.sk, ne);
    // record i lies in a run of records [o, e): from the run starts of its word (the same for the
    // whole warp) and, where the run reaches past it, of its neighbours
    auto run_of = [&](const uint32_t *starts, int i, int &o, int &e) {
        const int w = i >> 5, l = i & 31;
        const uint32_t m = starts[1 + w];
        uint32_t below = m & ((2u << l) - 1u), above = l == 31 ? 0u : m & ~((2u << l) - 1u);
        int wb = w, wa = w;
        while (below == 0) below = starts[1 + --wb];  // record 0 starts a run
        while (above == 0) above = starts[1 + ++wa];  // and so, in effect, does record ne
        o = 32 * wb + 31 - __clz(below);
        e = 32 * wa + __ffs(above) - 1;
    };
    // a record's place is its slot's start plus the smaller records of the slot
    auto place = [&](int i, const T &k) {
        int o, e;
        run_of(sm.heads, i, o, e);
        uint32_t d = (uint32_t)o;
        for (int j = o; j < e; j += 4) {  // independent loads, the first repeated past e
            T x[4];
#pragma unroll
            for (int v = 0; v < 4; v++) x[v] = sm.sk[j + v < e ? j + v : j];
#pragma unroll
            for (int v = 0; v < 4; v++) d += j + v < e && K::less(x[v], k) ? 1u : 0u;
        }
        return d;
    };
    if constexpr (!COUNT) {
        const uint64_t cmask = (1ull << a.cbits) - 1, pmask = (1ull << a.kb.pbits) - 1;
        for (int i = tid; i < ne; i += KB_NT) {
            const T k = sm.sk[i];
            const int64_t d = base + (crowded ? (uint32_t)i : place(i, k));
            const uint64_t low = K::low(k, lowbits);
            if (!SG_IN_BOUNDS(d < a.pl.cap, 709, d)) continue;
            a.col[d] = (int32_t)(K::code(k, lowbits) & cmask);
            a.val[d] = (uint32_t)((low >> 1) & pmask) | (uint32_t)((low & 1u) << 31);
        }
        // rows that start in [c0, cend): sh <= cbits and c0 is a multiple of 2^sh, so a
        // row starts where a slot does
        const uint64_t r0 = (c0 + cmask) >> a.cbits, r1 = (cend + cmask) >> a.cbits;
        const int64_t rbase = (int64_t)((uint64_t)p << (a.pl.rem - a.cbits));
        for (uint64_t r = r0 + tid; r < r1; r += KB_NT) {
            const int64_t row = rbase + (int64_t)r;
            if (row < a.n_rows) a.rp[row] = base + off((uint32_t)(((r << a.cbits) - c0) >> sh));
        }
        __syncthreads();
        return (uint32_t)ne;
    } else {
        uint32_t(&dst)[(K::ITEMS + 1) / 2] = rk;
        const int np = crowded ? 0 : ne;  // records to be ranked
#pragma unroll
        for (int u = 0; u < K::ITEMS; u++) {
            if (u * KB_NT >= np) break;
            const int i = u * KB_NT + tid;
            uint32_t d = 0;
            if (i < ne) {
                key[u] = sm.sk[i];
                d = place(i, key[u]);
            }
            if (u & 1) dst[u / 2] |= d << 16; else dst[u / 2] = d;
        }
        __syncthreads();
#pragma unroll
        for (int u = 0; u < K::ITEMS; u++) {
            if (u * KB_NT >= np) break;
            if (u * KB_NT + tid < ne) sm.sk[(dst[u / 2] >> (16 * (u & 1))) & 0xffffu] = key[u];
        }
        __syncthreads();
        // codes are runs now; of a read's records of a code, the first is its lowest position
        const uint64_t code_mask = K::code_mask(lowbits), read_mask = K::read_mask(a.kb.pbits);
        uint32_t again = 0, starts = 0;  // bit u: this thread's record repeats its predecessor's read; starts a code
#pragma unroll
        for (int u = 0; u < K::ITEMS; u++) {
            if (u * KB_NT >= ne) break;
            const int i = u * KB_NT + tid;
            bool st = i == ne;  // the end counts as a start
            if (i < ne) {
                const T k = sm.sk[i], x = sm.sk[i > 0 ? i - 1 : 0];
                st = i == 0 || !K::same(x, k, code_mask);
                if (!st && K::same(x, k, read_mask)) again |= 1u << u;
                if (st) starts |= 1u << u;
            }
            const uint32_t m = __ballot_sync(0xffffffffu, st);
            if ((tid & 31) == 0 && (i <= ne)) sm.codes[1 + (i >> 5)] = m;
        }
        if (tid == 0 && ne % KB_NT == 0) sm.codes[1 + (ne >> 5)] = 1u;
        __syncthreads();
        uint32_t nst = 0;
        uint32_t keep = 0;
#pragma unroll
        for (int u = 0; u < K::ITEMS; u++) {
            if (u * KB_NT >= ne) break;
            const int i = u * KB_NT + tid;
            bool kp = false;
            if (i < ne) {
                int o, e;
                run_of(sm.codes, i, o, e);
                uint32_t lo = a.lo, hi = a.hi;
                if (a.lohi) {
                    const uint64_t job = (((uint64_t)p << a.pl.rem) | K::code(sm.sk[i], lowbits)) >> a.kbits;
                    lo = a.lohi[2 * job];
                    hi = a.lohi[2 * job + 1];
                }
                const uint32_t f = (uint32_t)(e - o);
                const bool rel = f >= lo && f <= hi;
                nst += rel && ((starts >> u) & 1u) ? 1u : 0u;
                kp = rel && !((again >> u) & 1u);
                keep |= kp ? 1u << u : 0u;
            }
            const uint32_t m = __ballot_sync(0xffffffffu, kp);
            if ((tid & 31) == 0 && i < ne) sm.bits[i >> 5] = m;
        }
        nst = __reduce_add_sync(0xffffffffu, nst);
        if ((tid & 31) == 0 && nst) atomicAdd(&sm.nseg, nst);
        __syncthreads();
        uint32_t kept;
        {
            const int nw = (ne + 31) / 32;  // at most one word per thread
            const uint32_t c = tid < nw ? __popc(sm.bits[tid]) : 0u;
            const uint32_t x = block_exclusive_scan<KB_NT>(c, sm.tmp, &kept);
            if (tid < nw) sm.wpre[tid] = x;
        }
        __syncthreads();
#pragma unroll
        for (int u = 0; u < K::ITEMS; u++) {
            if (u * KB_NT >= ne) break;
            if (!((keep >> u) & 1u)) continue;
            const int i = u * KB_NT + tid;
            const uint32_t o = sm.wpre[i >> 5] + __popc(sm.bits[i >> 5] & ((1u << (i & 31)) - 1u));
            if (SG_IN_BOUNDS(base + o < a.pl.cap, 710, base + o)) out[base + o] = sm.sk[i];
        }
        __syncthreads();
        return kept;
    }
}

// A bucket of more records than a block holds, split by its block: the records are ordered by their next
// code bits (counted, then moved to the same range of the other buffer), runs of slots that fit are finished
// in code order, and a slot that does not fit is split again the same way, back and forth between the
// buffers. Every level reads the records twice and writes them once, whatever their number (choosing the
// runs from counts alone and searching the whole bucket for each run's records read a bucket of n records
// n / 8192 times: a contig of 8 Mbp among reads 7.7 s instead of 20 ms). Results go to the front of the
// bucket's own range of `out`, which may be `alt`: no more are written than records taken. A single code
// with more records than a block holds is skipped: in the count pass its frequency is above every hi taken
// here, and A's (read, column) pairs are distinct.
template <class K> __device__ __forceinline__ typename K::T load_moved(const typename K::T *p);
template <> __device__ __forceinline__ uint64_t load_moved<KeyN>(const uint64_t *p) {
    return *reinterpret_cast<const volatile uint64_t *>(p);
}
template <> __device__ __forceinline__ U128 load_moved<KeyW>(const U128 *p) {
    const volatile uint64_t *q = reinterpret_cast<const volatile uint64_t *>(p);
    return U128{q[0], q[1]};
}

template <class K, bool COUNT>
__device__ __noinline__ uint2 finish_big(FinishSmem<K> &sm, const FinishArgs &a, int p, typename K::T *in,
                                         typename K::T *alt, int64_t n, uint64_t c0, int bits, int64_t base,
                                         typename K::T *out) {
    using T = typename K::T;
    constexpr int TILE = kb_tile<K>(), U = 8;  // loads in flight
    const int lowbits = a.kb.low(), tid = threadIdx.x, lane = tid & 31;
    uint32_t done = 0, segs = 0;
    uint32_t *first = sm.slots;                                // [2^13 + 1] first record of each slot
    uint32_t *cur = reinterpret_cast<uint32_t *>(sm.sk);       // [2^13] where its next record goes
    static_assert(sizeof(sm.sk) >= sizeof(uint32_t) << KB_PIECE_BITS, "cursors in the records' place");
    if (tid == 0) {
        sm.piece[0] = KbPiece{c0, c0 + (1ull << bits), 0u, (uint32_t)n, (uint8_t)bits, 0, 0};
        sm.npiece = 1;
    }
    __syncthreads();
    for (;;) {
        const int top = sm.npiece - 1;
        if (top < 0) break;
        const KbPiece w = sm.piece[top];
        T *src = (w.where ? alt : in) + w.off;
        __syncthreads();
        if (w.len <= (uint32_t)TILE) {
            if (tid == 0) {
                sm.npiece = top;
                sm.nseg = 0;
            }
            T key[K::ITEMS];
#pragma unroll
            for (int u = 0; u < K::ITEMS; u++) {
                const uint32_t i = u * KB_NT + tid;
                key[u] = i < w.len ? load_moved<K>(src + i) : K::none();
            }
            __syncthreads();
            int wb = 0;  // slots: the range's codes at up to 2^14 steps
            while (((uint64_t)1 << wb) < w.cend - w.c0) wb++;
            const int sh2 = wb > KB_NS ? wb - KB_NS : 0;
            done += finish_group<K, COUNT>(sm, a, p, key, (int)w.len, w.c0, w.cend, sh2, wb - sh2, base + done, out);
            segs += sm.nseg;
            __syncthreads();
            continue;
        }
        const int ls = w.bits < KB_PIECE_BITS ? w.bits : KB_PIECE_BITS, sh = w.bits - ls, NS = 1 << ls;
        auto slot_of = [&](uint64_t c) { return (uint32_t)(c >> sh) & (uint32_t)(NS - 1); };
        for (int i = tid; i <= NS; i += KB_NT) first[i] = 0;
        __syncthreads();
        for (uint32_t i = tid; i < w.len; i += U * KB_NT) {
            T k[U];
#pragma unroll
            for (int u = 0; u < U; u++) k[u] = i + u * KB_NT < w.len ? load_moved<K>(src + i + u * KB_NT) : K::none();
#pragma unroll
            for (int u = 0; u < U; u++)
                if (i + u * KB_NT < w.len) atomicAdd(first + slot_of(K::code(k[u], lowbits)), 1u);
        }
        __syncthreads();
        {
            const int per = (NS + KB_NT - 1) / KB_NT, i0 = tid * per;
            uint32_t s = 0, tot;
            for (int i = i0; i < i0 + per && i < NS; i++) s += first[i];
            uint32_t ex = block_exclusive_scan<KB_NT>(s, sm.tmp, &tot);
            for (int i = i0; i < i0 + per && i < NS; i++) {
                const uint32_t c = first[i];
                first[i] = ex;
                cur[i] = ex;
                ex += c;
            }
            if (tid == 0) first[NS] = tot;
        }
        __syncthreads();
        if (!w.split) {
            T *dst = (w.where ? in : alt) + w.off;
            for (uint32_t i0 = 0; i0 < w.len; i0 += U * KB_NT) {
                T k[U];
#pragma unroll
                for (int u = 0; u < U; u++) {
                    const uint32_t i = i0 + u * KB_NT + tid;
                    k[u] = i < w.len ? load_moved<K>(src + i) : K::none();
                }
#pragma unroll
                for (int u = 0; u < U; u++) {
                    const bool have = i0 + u * KB_NT + tid < w.len;
                    const uint32_t s = have ? slot_of(K::code(k[u], lowbits)) : ~0u;
                    // the lanes that share the first lane's slot take one place together: a slot that
                    // holds most of the records would serialise the warp
                    const uint32_t s0 = __shfl_sync(0xffffffffu, s, 0);
                    const uint32_t m = __ballot_sync(0xffffffffu, have && s == s0);
                    if (m == 0) continue;  // no records (lane 0 has the first)
                    uint32_t q = 0;
                    if (lane == 0) q = atomicAdd(cur + s0, (uint32_t)__popc(m));
                    q = __shfl_sync(0xffffffffu, q, 0) + __popc(m & ((1u << lane) - 1u));
                    if (!have) continue;
                    if (s != s0) q = atomicAdd(cur + s, 1u);
                    if (SG_IN_BOUNDS(q < w.len, 713, q)) dst[q] = k[u];
                }
            }
            __syncthreads();
        }
        if (tid == 0) {  // the pieces, in code order from the top of the stack down
            const uint8_t at = w.split ? w.where : (uint8_t)(1 - w.where);
            // each level below may need a few
            const int room = KB_PIECES - 4 * ((sh + KB_PIECE_BITS - 1) / KB_PIECE_BITS) - 1;
            const uint64_t f0 = w.c0 >> w.bits << w.bits;  // slot 0's first code
            int q = top, x = (int)slot_of(w.c0);
            while (x < NS) {
                const uint32_t b = first[x];
                if (q >= room) {  // what is left, later
                    sm.piece[q++] = KbPiece{f0 + ((uint64_t)x << sh), w.cend, w.off + b, w.len - b, w.bits, at, 1};
                    break;
                }
                int z = x + 1;
                if (first[z] - b > (uint32_t)TILE) {
                    if (sh > 0)
                        sm.piece[q++] = KbPiece{f0 + ((uint64_t)x << sh), f0 + ((uint64_t)z << sh), w.off + b,
                                                first[z] - b, (uint8_t)sh, at, 0};
                    x = z;
                    continue;
                }
                int hi = NS;  // largest z with the records of [x, z) fitting
                while (z < hi) {
                    const int mid = (z + hi + 1) >> 1;
                    if (first[mid] - b <= (uint32_t)TILE) z = mid; else hi = mid - 1;
                }
                // rows of A may start where there are no records
                if (!COUNT || first[z] > b)
                    sm.piece[q++] = KbPiece{f0 + ((uint64_t)x << sh), f0 + ((uint64_t)z << sh), w.off + b, first[z] - b,
                                            0, at, 0};
                x = z;
            }
            for (int i = top, j = q - 1; i < j; i++, j--) {
                const KbPiece t = sm.piece[i];
                sm.piece[i] = sm.piece[j];
                sm.piece[j] = t;
            }
            sm.npiece = q;
        }
        __syncthreads();
    }
    return make_uint2(done, segs);
}

// alt: where the kept records go (COUNT); in either form a buffer of the plan's size that oversized buckets
// may use beside `in`.
template <class K, bool COUNT>
__global__ void __launch_bounds__(KB_NT, 2) kb_finish_kernel(FinishArgs a, typename K::T *in, typename K::T *alt) {
    extern __shared__ __align__(16) unsigned char kb_raw[];
    FinishSmem<K> &sm = *reinterpret_cast<FinishSmem<K> *>(kb_raw);
    constexpr int TILE = kb_tile<K>();
    const KbPlan &pl = a.pl;
    if (pl.stopped()) return;
    const int64_t nsub = pl.two ? (int64_t)pl.sb[pl.nb1] : (int64_t)pl.nb1;
    const int64_t *start = pl.two ? pl.start2 : pl.start1;
    if (!COUNT && blockIdx.x == 0 && threadIdx.x == 0) a.rp[a.n_rows] = a.nnz;
    for (int64_t b = blockIdx.x; b < nsub; b += gridDim.x) {
        const int64_t s0 = start[b], n = start[b + 1] - s0;
        const int p = pl.prefix(b);
        if (!SG_IN_BOUNDS(n >= 0 && s0 + n <= pl.cap && p < pl.nb1, 711, b)) continue;
        const int bits = pl.rem - (pl.two ? pl.b2[p] : 0);  // code bits below the bucket's
        const uint64_t c0 = pl.two && bits < 64 ? (uint64_t)(b - pl.sb[p]) << bits : 0ull;
        uint32_t kept = 0, segs = 0;
        if (n > TILE) {
            const uint2 r = finish_big<K, COUNT>(sm, a, p, in + s0, alt + s0, n, c0, bits, s0, alt);
            kept = r.x;
            segs = r.y;
        } else if (n > 0 || !COUNT) {
            typename K::T key[K::ITEMS];
#pragma unroll
            for (int u = 0; u < K::ITEMS; u++) {
                const int i = u * KB_NT + threadIdx.x;
                key[u] = i < n ? K::load(in + s0 + i) : K::none();
            }
            int lm = 8;  // slots: two to four per record, and at least one per row of A
            while (lm < KB_NS && (1 << (lm - 1)) < n) lm++;
            if (!COUNT && lm < bits - a.cbits) lm = bits - a.cbits;
            const int ls = bits < lm ? bits : lm;
            kept = finish_group<K, COUNT>(sm, a, p, key, (int)n, c0, c0 + ((uint64_t)1 << bits), bits - ls, ls, s0,
                                          alt);
            segs = sm.nseg;
            __syncthreads();
        }
        if (COUNT && threadIdx.x == 0) {
            a.nkeep[b] = kept;
            a.nseg[b] = segs;
        }
    }
}

__global__ void kb_totals_kernel(const int64_t *__restrict__ pseg, KbPlan pl, const uint32_t *__restrict__ err,
                                 int64_t *__restrict__ out) {
    if (threadIdx.x == 0) {
        out[0] = pseg[pl.nsub_max];
        out[1] = pseg[2 * pl.nsub_max];
        out[2] = pl.start1[pl.nb1];
        out[3] = (int64_t)*err;
        out[4] = (int64_t)pl.stop[1];
    }
}

// ----------------------------------------------------------------------------------- emit
// Kept records (in order within each bucket) -> At and the column codes. One warp per bucket: an
// entry's column is the bucket's first column plus the codes started up to it (ballots). Bound by
// memory: 1.77 G entries 8.6 ms, 3.4 TB/s (a read search per kept entry in the sorted form took 35).
template <class K>
__global__ void __launch_bounds__(256) kb_emit_kernel(KbPlan pl, KeyBits kb, const typename K::T *__restrict__ in,
                                                     const int64_t *__restrict__ pseg,
                                                     const int64_t *__restrict__ pkeep, int64_t m, int64_t nnz,
                                                     int kbits, int job_bits, int pb1, int32_t *__restrict__ at_col,
                                                     uint32_t *__restrict__ at_val, int64_t *__restrict__ at_rp,
                                                     uint64_t *__restrict__ codes,
                                                     unsigned long long *__restrict__ job_ncols) {
    const int lane = threadIdx.x & 31;
    const int64_t nsub = pl.two ? (int64_t)pl.sb[pl.nb1] : (int64_t)pl.nb1;
    const int64_t *start = pl.two ? pl.start2 : pl.start1;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    const int lowbits = kb.low();
    const uint64_t pmask = (1ull << kb.pbits) - 1, cmask = kbits < 64 ? (1ull << kbits) - 1 : ~0ull;
    const uint32_t le = lane == 31 ? 0xffffffffu : (2u << lane) - 1u;
    if (blockIdx.x == 0 && threadIdx.x == 0) at_rp[m] = nnz;
    for (int64_t b = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; b < nsub; b += nwarps) {
        const int64_t o0 = pkeep[b] - m, cnt = pkeep[b + 1] - m - o0;
        if (cnt == 0) continue;
        int64_t col0 = pseg[b] - 1;
        const int64_t s0 = start[b];
        const int p = pl.prefix(b);
        const uint64_t top = pl.rem < 64 ? (uint64_t)p << pl.rem : 0ull;
        uint64_t prev = ~0ull;  // the code of the entry before this step's first
        constexpr int U = 4;
        for (int64_t i0 = 0; i0 < cnt; i0 += 32 * U) {
            typename K::T k[U];
#pragma unroll
            for (int u = 0; u < U; u++)
                k[u] = i0 + 32 * u + lane < cnt ? K::load(in + s0 + i0 + 32 * u + lane) : K::none();
#pragma unroll
            for (int u = 0; u < U; u++) {
                const int64_t i = i0 + 32 * u + lane;
                const uint64_t code = K::code(k[u], lowbits);
                uint64_t before = __shfl_up_sync(0xffffffffu, code, 1);
                if (lane == 0) before = prev;
                const bool have = i < cnt, head = have && (i == 0 || code != before);
                const uint32_t hm = __ballot_sync(0xffffffffu, head);
                prev = __shfl_sync(0xffffffffu, code, 31);
                if (have) {
                    const int64_t col = col0 + __popc(hm & le), o = o0 + i;
                    if (SG_IN_BOUNDS(col >= 0 && col < m && o < nnz, 703, col)) {
                        const uint64_t low = K::low(k[u], lowbits);
                        at_col[o] = (int32_t)(low >> (kb.pbits + 1));
                        at_val[o] = (uint32_t)((low >> 1) & pmask) | (uint32_t)((low & 1u) << 31);
                        if (head) {
                            at_rp[col] = o;
                            codes[col] = (top | code) & cmask;
                            // more jobs than prefixes: the bucket may hold several
                            if (job_ncols && job_bits > pb1) atomicAdd(job_ncols + ((top | code) >> kbits), 1ull);
                        }
                    }
                }
                col0 += __popc(hm);
            }
        }
        if (job_ncols && job_bits <= pb1 && lane == 0)
            atomicAdd(job_ncols + (p >> (pb1 - job_bits)), (unsigned long long)(pseg[b + 1] - pseg[b]));
    }
}

// ----------------------------------------------------------------- A = At transposed
// tcol[t] = the column of At's entry t * TILE.
template <int TILE>
__global__ void tile_col_kernel(const int64_t *__restrict__ rp, int64_t m, int32_t *__restrict__ tcol) {
    const int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= m) return;
    const int64_t e = rp[j + 1];
    for (int64_t t = (rp[j] + TILE - 1) / TILE; t * TILE < e; t++) tcol[t] = (int32_t)j;
}

// Entries of At per prefix of the read id.
__global__ void __launch_bounds__(512) read_hist_kernel(const int32_t *__restrict__ col, int64_t nnz, int rs, int nb,
                                                       unsigned long long *__restrict__ hist) {
    extern __shared__ uint32_t rh[];
    for (int i = threadIdx.x; i < nb; i += 512) rh[i] = 0;
    __syncthreads();
    const int64_t nv = nnz / 4, stride = (int64_t)gridDim.x * 512;  // allocations are 256-byte aligned
    for (int64_t v = (int64_t)blockIdx.x * 512 + threadIdx.x; v < nv; v += stride) {
        const int4 x = reinterpret_cast<const int4 *>(col)[v];
        atomicAdd(rh + (x.x >> rs), 1u);
        atomicAdd(rh + (x.y >> rs), 1u);
        atomicAdd(rh + (x.z >> rs), 1u);
        atomicAdd(rh + (x.w >> rs), 1u);
    }
    if (blockIdx.x == 0 && threadIdx.x < nnz - 4 * nv) atomicAdd(rh + (col[4 * nv + threadIdx.x] >> rs), 1u);
    __syncthreads();
    for (int i = threadIdx.x; i < nb; i += 512)
        if (rh[i]) atomicAdd(hist + i, (unsigned long long)rh[i]);
}

// At's entries as records (read below the prefix << cbits | column, position, strand), grouped by
// the read's prefix. A tile's columns: its first entry's, plus the row starts up to an entry. With the
// pass that orders the rows and one between them 44 ms for 1.77 G entries; a radix sort of
// (read, entry) pairs in three passes took 106 with what came around it.
template <class K>
__global__ void __launch_bounds__(KB_NT, 2) at_scatter_kernel(const int64_t *__restrict__ at_rp,
                                                             const int32_t *__restrict__ at_col,
                                                             const uint32_t *__restrict__ at_val, int64_t m,
                                                             int64_t nnz, const int32_t *__restrict__ tcol, int rs,
                                                             int cbits, KeyBits kb, KbPlan pl,
                                                             typename K::T *__restrict__ out) {
    constexpr int TILE = kb_tile<K>();
    extern __shared__ __align__(16) unsigned char kb_raw[];
    __shared__ uint32_t bits[TILE / 32], pre[TILE / 32 + 1];
    ScatterSmem<K> *sm;
    uint32_t *cnt;
    unsigned long long *gb;
    uint16_t *sbin;
    const int nb = pl.nb1;
    scatter_layout<K>(kb_raw, nb, sm, cnt, gb, sbin);
    for (int i = threadIdx.x; i < nb; i += KB_NT) cnt[i] = 0;
    for (int i = threadIdx.x; i < TILE / 32; i += KB_NT) bits[i] = 0;
    const int64_t t = blockIdx.x, e0 = t * TILE;
    const int64_t j0 = tcol[t], j1 = (t + 1) * TILE < nnz ? tcol[t + 1] : m - 1;
    int32_t rd[K::ITEMS];
    uint32_t vl[K::ITEMS];
#pragma unroll
    for (int u = 0; u < K::ITEMS; u++) {
        const int64_t e = e0 + u * KB_NT + threadIdx.x;
        rd[u] = e < nnz ? at_col[e] : -1;
        vl[u] = e < nnz ? at_val[e] : 0u;
    }
    __syncthreads();
    for (int64_t j = j0 + 1 + threadIdx.x; j <= j1; j += KB_NT) {
        const int64_t x = at_rp[j] - e0;
        if (x > 0 && x < TILE) atomicOr(bits + (x >> 5), 1u << (x & 31));
    }
    __syncthreads();
    {
        const uint32_t c = threadIdx.x < TILE / 32 ? __popc(bits[threadIdx.x]) : 0u;
        uint32_t tot;
        const uint32_t x = block_exclusive_scan<KB_NT>(c, sm->tmp, &tot);
        if (threadIdx.x < TILE / 32) pre[threadIdx.x] = x;
    }
    __syncthreads();
    typename K::T key[K::ITEMS];
    uint32_t br[K::ITEMS];
    const uint32_t rmask = (1u << rs) - 1u;
    const int lowbits = kb.low();
#pragma unroll
    for (int u = 0; u < K::ITEMS; u++) {
        const int x = u * KB_NT + threadIdx.x;
        br[u] = 0xFFFFFFFFu;
        key[u] = K::none();
        if (rd[u] < 0) continue;
        const uint32_t le = (x & 31) == 31 ? 0xffffffffu : (2u << (x & 31)) - 1u;
        const uint64_t col = (uint64_t)(j0 + pre[x >> 5] + __popc(bits[x >> 5] & le));
        const uint32_t b = (uint32_t)rd[u] >> rs;
        const uint64_t low = ((uint64_t)(vl[u] & 0x7FFFFFFFu) << 1) | (vl[u] >> 31);
        key[u] = K::make(((uint64_t)((uint32_t)rd[u] & rmask) << cbits) | col, low, lowbits);
        br[u] = (b << 16) | atomicAdd(cnt + b, 1u);
    }
    scatter_tail<K, true>(*sm, cnt, gb, sbin, nb, key, br, pl.cur1, out, pl.cap,
                          [](const typename K::T &) { return 0u; });
}

// -------------------------------------------------------------------------------- the host side
static int bits_for(int64_t n) {  // bits of the ids 0 .. n - 1
    int b = 0;
    while (b < 62 && ((int64_t)1 << b) < n) b++;
    return b;
}

// A plan for `records` records with code bits `cb` above the prefix's end: prefix bits, whether a
// second level is needed, and the device arrays (one allocation).
// One block finishes a bucket at about 6 ns a record above its shared memory's (the whole device: 37 ps for
// the windows, 25 for A's entries; the general form 95 and 60). Up to this limit the largest bucket costs
// less than the general form does; beyond it the call takes that form.
static int64_t bucket_limit(int64_t records) { return records / 128 + ((int64_t)1 << 15); }

// A prefix of c records splits into fewer than 2 c / target + 1 buckets (2^b2min at least).
static int64_t split_bound(int64_t records, int target, int pb1, int b2min) {
    return ((int64_t)1 << (pb1 + b2min)) + 2 * (records / target + 1);
}

// buckets: their number at most, for a second level.
static sg_status make_plan(KbPlan &pl, int pb1, int cb, bool two, int64_t records, int tile, int64_t buckets,
                           Scratch &sc, uint32_t *stop) {
    pl.stop = stop;
    pl.limit = bucket_limit(records);
    pl.nb1 = 1 << pb1;
    pl.rem = cb - pb1;
    pl.two = two ? 1 : 0;
    pl.cap = records;
    pl.nsub_max = two ? buckets : pl.nb1;
    const size_t nb = (size_t)pl.nb1, ns = two ? (size_t)pl.nsub_max : 0;
    const size_t nc = two ? (size_t)(records / (KB_CHUNK_TILES * (int64_t)tile) + pl.nb1) : 0;  // a partial chunk per prefix
    const size_t words = (nb + 1) + nb + (ns + 1) + ns;  // 8-byte arrays
    uint64_t *w = sc.get<uint64_t>(words + ((nb + 1) * 2 * 4 + (ns + 1) * 4 + (ns + nc) * 2 + nb + 64) / 8);
    if (!w) return SG_ERR_OOM;
    pl.start1 = (int64_t *)w;
    pl.cur1 = (unsigned long long *)(w + nb + 1);
    pl.start2 = (int64_t *)(w + 2 * nb + 1);
    pl.cur2 = (unsigned long long *)(pl.start2 + ns + 1);
    pl.sb = (uint32_t *)(w + words);
    pl.chunk2 = pl.sb + nb + 1;
    pl.count2 = pl.chunk2 + nb + 1;
    pl.sub2p = (uint16_t *)(pl.count2 + ns + 1);
    pl.chunk2p = pl.sub2p + ns;
    pl.b2 = (uint8_t *)(pl.chunk2p + nc);
    return SG_OK;
}

// After the first pass: level-2 counts, bucket ranges and the second grouping pass (in -> out).
template <class K>
static sg_status second_level(KbPlan &pl, const typename K::T *in, typename K::T *out, int64_t records, int lowbits,
                              const char *hname, const char *sname, cudaStream_t s, uint32_t *err) {
    constexpr int64_t CH = (int64_t)KB_CHUNK_TILES * kb_tile<K>();
    const int64_t nch = records / CH + pl.nb1;  // at most: a partial chunk per prefix
    SG_CUDA_TRY(cudaMemsetAsync(pl.count2, 0, (size_t)(pl.nsub_max + 1) * 4, s));
    SG_LAUNCH("kmer_buckets", kb_sub2p_kernel, blocks_for((int64_t)pl.nb1 * 32, 256), 256, 0, s, pl);
    SG_LAUNCH(hname, kb_hist2_kernel<K>, nch, KB_NT, 0, s, pl, in, lowbits);
    SG_TRY(exclusive_scan<uint32_t>(pl.count2, pl.start2, pl.nsub_max, s, err));
    SG_LAUNCH("kmer_buckets", kb_cursors_kernel, blocks_for(pl.nsub_max, 256), 256, 0, s, pl);
    const size_t sm = scatter_smem_bytes<K, false>(KB_MAXBINS);
    SG_CUDA_TRY(ensure_smem(kb_scatter2_kernel<K>, sm));
    SG_LAUNCH(sname, kb_scatter2_kernel<K>, nch, KB_NT, sm, s, pl, in, out, lowbits);
    return SG_OK;
}

template <class K>
static sg_status finish_launch(const FinishArgs &a, bool count, typename K::T *in, typename K::T *alt,
                               const char *name, cudaStream_t s) {
    const size_t sm = sizeof(FinishSmem<K>);
    const int64_t grid = std::min<int64_t>(a.pl.nsub_max, (int64_t)sm_count() * 2);
    auto run = [&](auto kern) -> sg_status {
        SG_CUDA_TRY(ensure_smem(kern, sm));
        SG_LAUNCH(name, kern, grid, KB_NT, sm, s, a, in, alt);
        return SG_OK;
    };
    if (count) SG_TRY(run(kb_finish_kernel<K, true>));
    else SG_TRY(run(kb_finish_kernel<K, false>));
    return SG_OK;
}

template <class K>
static sg_status transpose_run(const sg_csr_u32 *At, sg_csr_u32 *A, int pb1, bool two, int cbits, int rbits,
                               KeyBits kb, const unsigned long long *hist, cudaStream_t s, uint32_t *stop) {
    constexpr int TILE = kb_tile<K>();
    const int64_t m = At->n_rows, n = At->n_cols, nnz = At->nnz;
    Scratch sc(s);
    // rows of one bucket: at most 2^12, a slot each
    const int rest = rbits - pb1, b2min = two && rest > 12 ? rest - 12 : 0;
    KbPlan pl;
    // a bucket is a range of (read, column): some rows, or a part of one. Where a mean row is nearly a
    // block's records, half of them would not fit: two parts each (12 Mbp, k = 31, rows of 7,200: 4.6 ms
    // -> 3.7; rows of 4,400, 100 Mbp: parts 31 ms, rows 22)
    const int target = nnz / n > kb_target<K>() / 4 * 3 ? kb_target<K>() / 2 : kb_target<K>();
    SG_TRY(make_plan(pl, pb1, rbits + cbits, two, nnz, TILE, split_bound(nnz, target, pb1, b2min), sc, stop));
    const int64_t ntiles = blocks_for(nnz, TILE);
    int32_t *tcol = sc.get<int32_t>(ntiles);
    typename K::T *r0 = sc.get<typename K::T>(nnz), *r1 = sc.get<typename K::T>(nnz);
    if (!tcol || !r0 || !r1) return SG_ERR_OOM;
    SG_LAUNCH("a_plan", kb_plan_kernel, 1, 1024, 0, s, hist, pl, target,
              two ? std::min(KB_MAXB2, pl.rem) : 0, b2min, 0.0f, 1.0f, pb1,
              KB_CHUNK_TILES * TILE);
    SG_LAUNCH("a_tile_col", tile_col_kernel<TILE>, blocks_for(m, 256), 256, 0, s, At->row_ptr, m, tcol);
    const size_t sm = scatter_smem_bytes<K, true>(pl.nb1);
    SG_CUDA_TRY(ensure_smem(at_scatter_kernel<K>, sm));
    SG_LAUNCH("a_scatter1", at_scatter_kernel<K>, ntiles, KB_NT, sm, s, At->row_ptr, At->col, At->val, m, nnz,
              (const int32_t *)tcol, rest, cbits, kb, pl, r0);
    if (two) SG_TRY(second_level<K>(pl, r0, r1, nnz, kb.low(), "a_hist2", "a_scatter2", s, stop));
    FinishArgs a{};
    a.pl = pl;
    a.kb = kb;
    a.cbits = cbits;
    a.n_rows = n;
    a.nnz = nnz;
    a.col = A->col;
    a.val = A->val;
    a.rp = A->row_ptr;
    SG_TRY(finish_launch<K>(a, false, two ? r1 : r0, two ? r0 : r1, "a_rows", s));
    return SG_OK;
}

// At's entries with their columns, for a sort by read: a thread per column.
__global__ void at_pairs_kernel(const int64_t *__restrict__ rp, const int32_t *__restrict__ col,
                                const uint32_t *__restrict__ val, int64_t m, uint32_t *__restrict__ key,
                                uint64_t *__restrict__ pv) {
    const int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= m) return;
    for (int64_t e = rp[j], e1 = rp[j + 1]; e < e1; e++) {
        key[e] = (uint32_t)col[e];
        pv[e] = ((uint64_t)j << 32) | val[e];
    }
}

// Sorted pairs -> A's columns and values, and the row pointers where a read's entries begin.
__global__ void a_from_pairs_kernel(const uint32_t *__restrict__ key, const uint64_t *__restrict__ pv, int64_t nnz,
                                    int64_t n, int32_t *__restrict__ col, uint32_t *__restrict__ val,
                                    int64_t *__restrict__ rp, const uint32_t *__restrict__ err) {
    const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e > nnz || *err) return;  // a sort that timed out leaves words that are no reads
    const int64_t prev = e == 0 ? -1 : (int64_t)key[e - 1], cur = e == nnz ? n : (int64_t)key[e];
    for (int64_t r = prev + 1; r <= cur; r++) rp[r] = e;
    if (e == nnz) return;
    const uint64_t x = pv[e];
    col[e] = (int32_t)(x >> 32);
    val[e] = (uint32_t)x;
}

// A by a stable radix sort of At's entries by read (columns stay ascending): 24 bytes an entry of work
// memory whatever the rows, 60 ps an entry against 25 by grouping. For rows that grouping cannot split
// over enough blocks: one read of 8 Mbp among 160,000 of 1 kbp, 144 M entries, its row in two buckets: 26 ms by
// grouping, 10 by sorting.
sg_status transpose_sorted(const sg_csr_u32 *At, sg_csr_u32 *A, cudaStream_t s, uint32_t *err) {
    const int64_t m = At->n_rows, n = At->n_cols, nnz = At->nnz;
    Scratch sc(s);
    uint32_t *k0 = sc.get<uint32_t>(nnz), *k1 = sc.get<uint32_t>(nnz);
    uint64_t *v0 = sc.get<uint64_t>(nnz), *v1 = sc.get<uint64_t>(nnz);
    if (!k0 || !k1 || !v0 || !v1) return SG_ERR_OOM;
    SG_LAUNCH("at_pairs", at_pairs_kernel, blocks_for(m, 256), 256, 0, s, At->row_ptr, At->col, At->val, m, k0, v0);
    bool alt = false;
    SG_TRY((radix_sort_pairs<uint32_t, uint64_t>(k0, v0, k1, v1, nnz, bits_for(n), &alt, s, err)));
    SG_LAUNCH("a_rows", a_from_pairs_kernel, blocks_for(nnz + 1, 256), 256, 0, s, (const uint32_t *)(alt ? k1 : k0),
              (const uint64_t *)(alt ? v1 : v0), nnz, n, A->col, A->val, A->row_ptr, (const uint32_t *)err);
    return SG_OK;
}

// A = At transposed into A's arrays (allocated, nnz entries): rows ascending, columns ascending in
// a row. pbits: bits of a position. stop[1]: set where a bucket is too large (A is left unwritten).
sg_status transpose_impl(const sg_csr_u32 *At, sg_csr_u32 *A, int pbits, cudaStream_t s, uint32_t *stop) {
    const int64_t m = At->n_rows, n = At->n_cols, nnz = At->nnz;
    if (nnz == 0) {
        SG_CUDA_TRY(cudaMemsetAsync(A->row_ptr, 0, (size_t)(n + 1) * 8, s));
        return SG_OK;
    }
    const int rbits = bits_for(n), cbits = std::max(bits_for(m), 1);
    // one level while a row group of 2^(rbits - pb1) rows fits a block on average
    int want = 0;  // bits of the buckets wanted
    while (want < rbits + cbits && (nnz >> want) > kb_target<KeyN>() / 2) want++;
    const bool two = want > 10 || want > rbits || rbits - want > 12;
    // a second level splits by at most 11 bits and leaves at most 12 bits of rows to a bucket
    const int pb1 = std::min(rbits, two ? std::max((std::min(want, 20) + 1) / 2, std::max(6, rbits - 23)) : want);
    const KeyBits kb{0, pbits};
    Scratch sc(s);
    unsigned long long *hist = sc.get<unsigned long long>((size_t)1 << pb1);
    if (!hist) return SG_ERR_OOM;
    SG_CUDA_TRY(cudaMemsetAsync(hist, 0, (size_t)8 << pb1, s));
    const int64_t hg = std::min<int64_t>(blocks_for(nnz, 4096), (int64_t)sm_count() * 4);
    SG_LAUNCH("a_hist1", read_hist_kernel, hg, 512, (size_t)4 << pb1, s, At->col, nnz, rbits - pb1, 1 << pb1, hist);
    if (rbits - pb1 + cbits + kb.low() <= 64) return transpose_run<KeyN>(At, A, pb1, two, cbits, rbits, kb, hist, s, stop);
    return transpose_run<KeyW>(At, A, pb1, two, cbits, rbits, kb, hist, s, stop);
}

// ---------------------------------------------------------------------------- k-mer stage
struct KbBuild {
    const uint8_t *seq;
    const int64_t *off;
    int64_t n, total;
    int k;
    uint32_t lo, hi, hmax;
    const uint32_t *lohi;
    unsigned long long *job_ncols;
    int cb, job_bits, pb1;
    bool two;
    KeyBits kb;
    std::vector<unsigned long long> counts;  // large inputs: windows of each prefix
    float skew, skew_max;                    // of the codes (negative: found on the device); not taken from here on
};

template <class K>
static sg_status kb_run(const KbBuild &q, sg_csr_u32 *At, uint64_t **codes_out, cudaStream_t s,
                        Scratch &sc, uint32_t *err, const uint64_t *P, const uint32_t *VM, const int32_t *RG,
                        int64_t ngroups, JobPos jp, const unsigned long long *hist, Scratch &early, bool *taken) {
    using T = typename K::T;
    constexpr int TILE = kb_tile<K>();
    KbPlan pl;
    constexpr int TARGET = kb_target<K>();
    const int b2max = q.two ? std::min(KB_MAXB2, q.cb - q.pb1) : 0;
    int64_t buckets = 0;  // exactly, where the host has the prefixes' counts
    for (const unsigned long long c : q.counts)
        buckets += (int64_t)1 << kb_split((int64_t)c, TARGET, b2max, 0, q.skew, KB_MAXB2);
    if (q.counts.empty()) buckets = split_bound(q.total, TARGET, q.pb1, 0) << (q.skew < 0.0f ? KB_SMALL_GROW : 0);
    SG_TRY(make_plan(pl, q.pb1, q.cb, q.two, q.total, TILE, buckets, sc, err));
    SG_LAUNCH("kmer_plan", kb_plan_kernel, 1, 1024, 0, s, hist, pl, TARGET, b2max, 0, q.skew, q.skew_max,
              q.pb1, KB_CHUNK_TILES * TILE);
    T *r0 = sc.get<T>(q.total), *r1 = sc.get<T>(q.total);
    if (!r0 || !r1) return SG_ERR_OOM;
    const WindowSrc w{P, VM, RG, q.off, q.n, ngroups, q.k, jp, pl.rem, q.kb};
    const size_t sm1 = scatter_smem_bytes<K, true>(pl.nb1);
    SG_TRY(dispatch_k(q.k, [&](auto kc) -> sg_status {
        auto run = [&](auto kern) -> sg_status {
            SG_CUDA_TRY(ensure_smem(kern, sm1));
            SG_LAUNCH("kmer_scatter1", kern, blocks_for(ngroups, (KB_NT / 32) * K::ITEMS), KB_NT, sm1, s, w, pl, r0);
            return SG_OK;
        };
        return jp.jpos ? run(kb_scatter1_kernel<K, decltype(kc)::value, true>)
                       : run(kb_scatter1_kernel<K, decltype(kc)::value, false>);
    }));
    for (const void *p : {(const void *)P, (const void *)VM, (const void *)RG}) early.release(p);
    T *src = r0, *dst = r1;
    if (q.two) {
        SG_TRY(second_level<K>(pl, r0, r1, q.total, q.kb.low(), "kmer_hist2", "kmer_scatter2", s, err));
        src = r1;
        dst = r0;
    }
    uint32_t *nseg = sc.get<uint32_t>(2 * (size_t)pl.nsub_max);
    int64_t *pseg = sc.get<int64_t>(2 * (size_t)pl.nsub_max + 1 + 5);
    if (!nseg || !pseg) return SG_ERR_OOM;
    uint32_t *nkeep = nseg + pl.nsub_max;
    int64_t *pkeep = pseg + pl.nsub_max, *totals = pseg + 2 * pl.nsub_max + 1;
    if (q.two) SG_CUDA_TRY(cudaMemsetAsync(nseg, 0, 2 * (size_t)pl.nsub_max * 4, s));  // past the last bucket
    FinishArgs a{};
    a.pl = pl;
    a.kb = q.kb;
    a.lo = q.lo;
    a.hi = q.hi;
    a.hmax = q.hmax;
    a.lohi = q.lohi;
    a.kbits = 2 * q.k;
    a.nseg = nseg;
    a.nkeep = nkeep;
    SG_TRY(finish_launch<K>(a, true, src, dst, "kmer_finish", s));
    // both totals in one scan (nkeep follows nseg): bucket b's kept records start at pkeep[b] - m
    SG_TRY(exclusive_scan<uint32_t>(nseg, pseg, 2 * pl.nsub_max, s, err));
    int64_t sizes[5] = {0, 0, 0, 0, 0};  // m, m + nnz, records, the stop words: one copy, since each waits
    SG_LAUNCH("kmer_totals", kb_totals_kernel, 1, 32, 0, s, (const int64_t *)pseg, pl, (const uint32_t *)err, totals);
    SG_CUDA_TRY(read_back(sizes, totals, sizeof(sizes), s));
    const uint32_t herr = (uint32_t)sizes[3];
    if (herr & DEV_TIMEOUT) return timeout_error("build_kmer_matrix");
    if (herr) {  // the passes above stayed in bounds; their results are discarded
        set_error("build_kmer_matrix: offsets are not a valid partition of the sequence");
        return SG_ERR_INVALID;
    }
    if (sizes[4]) {  // not taken; A's rows use the word again
        SG_CUDA_TRY(cudaMemsetAsync(err + 1, 0, sizeof(uint32_t), s));
        return SG_OK;
    }
    *taken = true;
    const int64_t m = sizes[0], nnz = sizes[1] - m;
    if (m >= ((int64_t)1 << 31)) {
        set_error("build_kmer_matrix: %lld reliable k-mers exceed the int32 column range", (long long)m);
        return SG_ERR_OVERFLOW;
    }
    sg_kmer_stats &ks = kmer_stats();
    ks = sg_kmer_stats{};
    ks.windows = q.total;
    ks.candidates = sizes[2];
    ks.m = m;
    ks.nnz = nnz;
    ks.sort_key_bytes = (int32_t)sizeof(T);
    sc.release(src);  // read only by the finishing pass
    SG_ALLOC(At->row_ptr, int64_t, m + 1, s);
    SG_ALLOC(At->col, int32_t, nnz, s);
    SG_ALLOC(At->val, uint32_t, nnz, s);
    SG_ALLOC(*codes_out, uint64_t, m, s);
    At->n_rows = m; At->n_cols = q.n; At->nnz = nnz;
    SG_LAUNCH("emit_at", kb_emit_kernel<K>, std::min<int64_t>(blocks_for(pl.nsub_max * 32, 256), (int64_t)sm_count() * 8),
              256, 0, s, pl, q.kb, (const T *)dst, (const int64_t *)pseg, (const int64_t *)pkeep, m, nnz, 2 * q.k,
              q.job_bits, q.pb1, At->col, At->val, At->row_ptr, *codes_out, q.job_ncols);
    sc.release(dst);
    return SG_OK;
}

// *taken is false where the general form has to run: a reliable range above KB_HMAX (records of
// one code are ranked against each other), k-mers too short to spread over buckets, one prefix or one
// bucket holding a large part of the input (low-complexity sequence: one block would finish it alone; the
// general form then costs what it always does, after a tenth of it spent here), short k-mers whose codes are
// too skewed, or records that would not fit the device.
constexpr uint32_t KB_HMAX = 1024;
constexpr int KB_MIN_CODE = 22;
// Skewed codes cost the bucketed form more (buckets of unequal size, records that share slots), the sorts
// not. Times of both, ms, 120 M windows, k = 17: 60 % A and T 4.9 and 5.6, 65 % 5.4 and 5.8, 70 % 6.4 and
// 6.2, 75 % 7.8 and 6.9, 80 % 9.8 and 8.2 at 10 % errors; at 1 % 80 % 12.2 and 12.6. With long k-mers, which
// accurate reads go with, the sorts move pairs and lose: k = 21 at 1 % errors 14.0 and 20.9. Below two
// million windows launches decide: 1 M windows at 80 % 0.36 and 0.43.
constexpr float KB_SKEW_MAX = 0.15f;  // about 73 % A and T
constexpr int KB_SKEW_K = 19;
constexpr int64_t KB_SKEW_TOTAL = (int64_t)1 << 21;

sg_status build_bucketed(const uint8_t *seq, const int64_t *off, int64_t n, int64_t total, int k, uint32_t lo,
                         uint32_t hi, sg_csr_u32 *At, uint64_t **codes_out, cudaStream_t s, Scratch &sc, JobMap jm,
                         const uint32_t *lohi, unsigned long long *job_ncols, uint32_t hmax, uint32_t *err,
                         const unsigned long long *maxlen, int *pbits, bool *taken) {
    *taken = false;
    if (!tune("kmer_bucketed") || hmax > KB_HMAX || 2 * k < KB_MIN_CODE || total <= 0 || n <= 0) return SG_OK;
    KbBuild q{seq, off, n, total, k, lo, hi, hmax, lohi, job_ncols, 0, 0, 0, false, {}, {}, 0.0f, 1.0f};
    if (!jm.ro && total > KB_SKEW_TOTAL) {  // (prefixes of read sets differ by their sizes)
        q.skew = -1.0f;
        if (k <= KB_SKEW_K) q.skew_max = KB_SKEW_MAX;
    }
    while (jm.ro && ((int64_t)1 << q.job_bits) < jm.njobs) q.job_bits++;
    q.cb = 2 * k + q.job_bits;
    const bool large = total > ((int64_t)1 << 24);
    const int64_t ngroups = (total + 31) / 32;
    Scratch early(s);
    // bucket bits: the canonical codes of a random sequence are twice as dense at the low end
    auto plan_bits = [&](int target) {
        int w = 0;
        while (w < 20 && ((2 * total) >> w) > target) w++;
        return jm.ro ? w + 2 : w;  // read sets of a batch differ in size
    };
    int want = std::min(plan_bits(kb_target<KeyN>()), q.cb);
    q.two = want > 10;
    q.pb1 = q.two ? (want + 1) / 2 : want;
    q.kb = KeyBits{std::max(bits_for(n), 1), std::max(bits_for(total), 1)};
    bool fits = q.cb - q.pb1 + q.kb.low() <= 64;
    if (large || !fits || jm.ro) {  // the longest read bounds a position; a batch's prefixes follow its offsets
        unsigned long long ml = 0;
        uint32_t herr = 0;
        SG_CUDA_TRY(cudaMemcpyAsync(&ml, maxlen, 8, cudaMemcpyDeviceToHost, s));
        SG_CUDA_TRY(read_back(&herr, err, 4, s));
        if (herr) {
            set_error("build_kmer_matrix: offsets are not a valid partition of the sequence");
            return SG_ERR_INVALID;
        }
        q.kb.pbits = std::max(bits_for((int64_t)ml), 1);
        int need = q.cb + q.kb.low() - 64;
        if (need > q.pb1 && need <= 11 && need <= q.cb) q.pb1 = need;  // a longer prefix makes one word do
        fits = q.cb - q.pb1 + q.kb.low() <= 64;
        if (!fits) {
            want = std::min(plan_bits(kb_target<KeyW>()), q.cb);
            q.two = want > 10;
            q.pb1 = q.two ? (want + 1) / 2 : want;
        }
    }
    if (large) {
        const double need = 2.0 * (fits ? 8 : 16) * (double)total + 0.5 * (double)total;
        if (need > 0.9 * (double)device_bytes_available()) return SG_OK;
    }
    StageScope stage("CountKmer", s);
    JobPos jp{nullptr, 0, 2 * k};
    if (jm.ro) {
        int64_t *jpos = sc.get<int64_t>(jm.njobs + 1);
        if (!jpos) return SG_ERR_OOM;
        SG_LAUNCH("job_pos", job_pos_kernel, blocks_for(jm.njobs + 1, 256), 256, 0, s, jm.ro, jm.njobs, off, n, jpos);
        jp = JobPos{jpos, jm.njobs, jm.kbits};
    }
    uint64_t *P = early.get<uint64_t>(ngroups + 1);
    uint32_t *VM = early.get<uint32_t>(ngroups);
    int32_t *RG = early.get<int32_t>(ngroups);
    const int nb1 = 1 << q.pb1;
    unsigned long long *hist = sc.get<unsigned long long>(nb1);
    if (!P || !VM || !RG || !hist) return SG_ERR_OOM;
    SG_CUDA_TRY(cudaMemsetAsync(hist, 0, (size_t)nb1 * 8, s));
    SG_CUDA_TRY(cudaMemsetAsync(P + ngroups, 0, 8, s));
    const int64_t steps = blocks_for(ngroups, PK_G);
    const int64_t maxw = (int64_t)sm_count() * 8 * (PK_NT / 32);
    const int64_t spw = steps > maxw ? blocks_for(steps, (int)maxw) : 1;
    SG_LAUNCH("pack", kb_pack_kernel, blocks_for(blocks_for(steps, (int)spw), PK_NT / 32), PK_NT, (size_t)nb1 * 4, s, seq,
              total, off, n, k, jp, q.pb1, q.job_bits, ngroups, spw, P, VM, RG, hist);
    if (large) {
        q.counts.resize(nb1);
        SG_CUDA_TRY(read_back(q.counts.data(), hist, (size_t)nb1 * 8, s));
        unsigned long long mx = 0;
        double sum = 0.0, squares = 0.0;
        for (const unsigned long long c : q.counts) {
            mx = std::max(mx, c);
            sum += (double)c;
            squares += (double)c * (double)c;
        }
        if (!jm.ro) q.skew = kb_skew((float)sum, (float)squares, nb1, q.pb1);
        if (q.skew >= q.skew_max) return SG_OK;
        if (mx > (unsigned long long)std::max<int64_t>(total / 16, (int64_t)1 << 23)) return SG_OK;
    }
    *pbits = q.kb.pbits;
    if (fits)
        SG_TRY(kb_run<KeyN>(q, At, codes_out, s, sc, err, P, VM, RG, ngroups, jp, hist, early, taken));
    else
        SG_TRY(kb_run<KeyW>(q, At, codes_out, s, sc, err, P, VM, RG, ngroups, jp, hist, early, taken));
    return SG_OK;
}

}  // namespace sg

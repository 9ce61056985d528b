// kmer.cuh -- pieces shared by the two forms of the k-mer stage (kmer.cu, kbucket.cu).
#pragma once

#include <type_traits>

#include "ops.cuh"

namespace sg {

// Batches: the job prefix of a window, from the base offset of each job's first read (jpos[b] =
// off[ro[b]], jpos[njobs] = total). A window lies in the last job b with jpos[b] <= its position
// (windows never cross reads, and empty jobs start where the next one does). The cursor keeps the
// last job's range, so increasing positions search only when they leave it.
struct JobPos {
    const int64_t *jpos;  // nullptr: one read set, no prefix
    int64_t njobs;
    int kbits;  // 2k
};

struct JobPosCursor {
    JobPos m;
    int64_t jb = 0, jlo = 0, jhi = -1;
    __device__ __forceinline__ uint64_t prefix(int64_t q) {
        if (!m.jpos) return 0;
        if (q < jlo || q >= jhi) {
            int64_t lo = 0, hi = m.njobs;
            while (hi - lo > 1) {
                const int64_t mid = (lo + hi) >> 1;
                if (m.jpos[mid] <= q) lo = mid; else hi = mid;
            }
            jb = lo;
            jlo = m.jpos[lo];
            jhi = m.jpos[lo + 1];
        }
        return (uint64_t)jb << m.kbits;
    }
};

static __global__ void job_pos_kernel(const int64_t *__restrict__ ro, int64_t njobs, const int64_t *__restrict__ off,
                               int64_t n, int64_t *__restrict__ jpos) {
    const int64_t b = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (b > njobs) return;
    int64_t r = ro[b];
    r = r < 0 ? 0 : (r > n ? n : r);
    jpos[b] = off[r];
}

// Runs f with k as a compile-time constant for the common k (17 is the paper's), else 0.
template <class F>
static sg_status dispatch_k(int k, F &&f) {
    switch (k) {
        case 17: return f(std::integral_constant<int, 17>{});
        case 21: return f(std::integral_constant<int, 21>{});
        case 31: return f(std::integral_constant<int, 31>{});
        default: return f(std::integral_constant<int, 0>{});
    }
}

// Offsets check: off partitions [0, total) into n reads shorter than 2^31 (else DEV_INVALID in
// *err); *maxlen (zeroed) receives the longest read.
sg_status check_offsets(const int64_t *off, int64_t n, int64_t total, uint32_t *err, unsigned long long *maxlen,
                        cudaStream_t s);

// The bucketed form (kbucket.cu): At and the column codes, with *pbits = bits of a position in its
// read. *taken is false where the general form has to run. err[1] (zeroed): set where a bucket was too
// large for the form.
sg_status build_bucketed(const uint8_t *seq, const int64_t *off, int64_t n, int64_t total, int k, uint32_t lo,
                         uint32_t hi, sg_csr_u32 *At, uint64_t **codes_out, cudaStream_t s, Scratch &sc, JobMap jm,
                         const uint32_t *lohi, unsigned long long *job_ncols, uint32_t hmax, uint32_t *err,
                         const unsigned long long *maxlen, int *pbits, bool *taken);

// A = At transposed into A's arrays (allocated: n + 1 row pointers, nnz entries): columns ascending
// in a row. pbits: bits that hold every position. stop: the error word and (zeroed) a word that is set where
// a row is too long for the form; A is then unwritten, and transpose_sorted does it (kbucket.cu).
sg_status transpose_impl(const sg_csr_u32 *At, sg_csr_u32 *A, int pbits, cudaStream_t s, uint32_t *stop);
sg_status transpose_sorted(const sg_csr_u32 *At, sg_csr_u32 *A, cudaStream_t s, uint32_t *err);

}  // namespace sg

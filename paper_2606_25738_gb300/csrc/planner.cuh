// Device planner of FP32 batches on the skewed engines: what make_plan() does on the host
// (teams packed into warps, strip items of wide pairs), by counting sort, for batches of
// many pairs.  The host planner orders and packs pair by pair: 23.5 ms for the 455,000 pairs
// of the short-read batch, twice its kernels' time; here it is a handful of launches.
#pragma once

#include <cuda_runtime.h>

#include "phmm_internal.h"

namespace phmm {

// What submit needs to know of a batch before it allocates (one copy to the host).  Index 0 of
// the pairs below: short teams of 32 columns a lane (k <= 1024), 1: of 24 (k <= 768).
struct PlanScan {
    unsigned long long cells;           // sum of l k
    unsigned long long short_cells[2];  // ... over short pairs
    unsigned long long sum_l, sum_k;
    unsigned long long rows[2][2];      // [short width][strips of 1024, 512 columns]: sum of (strips - 1) l
    unsigned long long strips[2][2];    // ... of strips
    unsigned long long cta_rows, cta_strips;  // strips of 4-warp CTAs: sums of (strips - 1) l, of strips - 1
    unsigned long long n_read_bases, n_hap_bases;
    uint32_t n_long[2];                 // pairs wider than the short teams
    uint32_t lmax, lmax_long[2];        // longest read of all pairs, of the wide ones
    uint32_t shared;                    // pairs whose neighbour in the list has the same read
    uint32_t bad;                       // an offset or index is out of range
    uint32_t pad;
};

// A pair's part of the sums.  shared: its neighbour in the list has the same read.
__host__ __device__ inline void plan_scan_pair(PlanScan& s, uint32_t l, uint32_t k, bool shared) {
    const unsigned long long c = (unsigned long long)l * k;
    s.cells += c;
    s.sum_l += l;
    s.sum_k += k;
    s.lmax = l > s.lmax ? l : s.lmax;
    s.shared += shared;
    if (k > 4096u) {  // strips of 4-warp CTAs of 1024 columns a warp
        const uint32_t C = (k + 4095u) / 4096u;
        s.cta_rows += (unsigned long long)(C - 1) * l;
        s.cta_strips += C - 1;
    }
#ifdef __CUDA_ARCH__
#pragma unroll
#endif
    for (int w = 0; w < 2; ++w) {
        if (k <= (w ? 768u : 1024u)) {
            s.short_cells[w] += c;
            continue;
        }
        s.n_long[w]++;
        s.lmax_long[w] = l > s.lmax_long[w] ? l : s.lmax_long[w];
#ifdef __CUDA_ARCH__
#pragma unroll
#endif
        for (int z = 0; z < 2; ++z) {
            const uint32_t W = z ? (k + 511u) / 512u : (k + 1023u) / 1024u;
            s.rows[w][z] += (unsigned long long)(W - 1) * l;
            s.strips[w][z] += W;
        }
    }
}

struct PlanInput {
    const uint64_t *read_off, *hap_off;
    const uint32_t *pair_read, *pair_hap;
    uint32_t n_reads, n_haps, n_pairs;
};

struct PlanOutput {
    int N, Nl;             // columns per lane of the short teams, of the strips
    int wave;              // one item per strip (else one per pair)
    Team* teams;           // n_short
    WarpItem* witems;      // at most n_short
    CtaPair* cpairs;       // n_long, or the strips
    CtaItem* citems;
    BatchHeader* H;        // n_witems is written there
    void* scratch;         // plan_scratch_bytes
};

size_t plan_scratch_bytes(uint32_t n_pairs);
void launch_plan_scan(const PlanInput& in, PlanScan* out, int sms, cudaStream_t s);
// The same on the host, for arrays there.
PlanScan plan_scan_host(const PlanInput& in);
// The batch is known to be valid (PlanScan.bad == 0).
void launch_plan_build(const PlanInput& in, const PlanOutput& out, int sms, cudaStream_t s);

}  // namespace phmm

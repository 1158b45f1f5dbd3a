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
// The batch is known to be valid (PlanScan.bad == 0).
void launch_plan_build(const PlanInput& in, const PlanOutput& out, int sms, cudaStream_t s);

}  // namespace phmm

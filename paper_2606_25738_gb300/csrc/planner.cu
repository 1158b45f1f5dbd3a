// Device planner (planner.cuh).
//
// Short pairs: a class is (run of similar read lengths, lanes G).  Runs are geometric in the
// read length (ratio 0.94, as the host planner's), longest first.  One thread per run packs
// that run's class counts into 32 lanes by patterns -- the widest team left, then the widest
// that fits, and so on -- and takes each pattern as often as the counts allow, so a run of
// any size is a few dozen patterns; the items of a pattern are then written in parallel, their
// pairs taken from the counting sort by class.
// Wide pairs: classes of cost (l x strips, eight to an octave), largest first.
//
// Bound by latency: the short-read batch's 455,000 pairs are read three times (11 MB each) and
// written as 8 MB of teams and items; the launches and the one-thread-per-run packing take the
// time.
#include "planner.cuh"

#include "engine.cuh"

namespace phmm {

namespace {

constexpr int kRuns = 272;           // log2(2^24) * 11.2 runs, and one spare
constexpr int kG = 33;               // class of G lanes: run * kG + G
constexpr int kClasses = kRuns * kG;
constexpr int kLongClasses = 512;
// Patterns of a run.  Most exhaust a class, but one that takes m teams of a class an item can leave up
// to m - 1 of it; from pattern 63 on each is one team an item and exhausts its class, so the 32
// classes take no more than 32 further ones (pack_run).
constexpr int kMaxPatterns = 96;
constexpr int kSlots = 32;

struct Pattern {
    uint32_t item0, team0;    // first item and team
    uint32_t teams;           // teams per item
    uint32_t run;
    uint8_t g[kSlots];        // lanes of each team
    uint32_t used[kSlots];    // members of that class taken by earlier patterns and slots ...
    uint8_t mult[kSlots];     // ... and members of that class per item
};

struct Scratch {
    uint32_t hist[kClasses];        // members; then the class's first place in `sorted`
    uint32_t cursor[kClasses];
    uint32_t lhist[kLongClasses];   // wide pairs: items of the class; then its first item
    uint32_t lcursor[kLongClasses];
    uint32_t n_patterns, n_items, n_teams, extra;
    unsigned long long wrows;
    uint32_t pattern0[kRuns + 1];
    Pattern patterns[kRuns * kMaxPatterns];
};

__device__ __forceinline__ int run_of(uint32_t l) { return min((int)(log2f((float)l) * 11.2f), kRuns - 1); }
__device__ __forceinline__ int long_class(uint32_t l, uint32_t W) {
    // largest first
    return kLongClasses - 1 - min((int)(log2f((float)l * (float)W) * 8.0f), kLongClasses - 1);
}

__device__ __forceinline__ unsigned long long warp_sum(unsigned long long v) {
#pragma unroll
    for (int o = 16; o; o >>= 1) v += __shfl_down_sync(kFull, v, o);
    return v;
}

__global__ void __launch_bounds__(256) k_plan_scan(PlanInput in, PlanScan* __restrict__ out) {
    const uint32_t t0 = blockIdx.x * blockDim.x + threadIdx.x, st = gridDim.x * blockDim.x;
    bool bad = false;
    if (t0 == 0) {
        bad |= in.read_off[0] != 0 || in.hap_off[0] != 0;
        out->n_read_bases = in.read_off[in.n_reads];
        out->n_hap_bases = in.hap_off[in.n_haps];
    }
    for (uint32_t r = t0; r < in.n_reads; r += st) {
        const uint64_t a = in.read_off[r], b = in.read_off[r + 1];
        bad |= b <= a || b - a > 0xffffffull;
    }
    for (uint32_t h = t0; h < in.n_haps; h += st) {
        const uint64_t a = in.hap_off[h], b = in.hap_off[h + 1];
        bad |= b <= a || b - a > 0xffffffull;
    }
    PlanScan q{};
    for (uint32_t p = t0; p < in.n_pairs; p += st) {
        const uint32_t r = in.pair_read[p], h = in.pair_hap[p];
        if (r >= in.n_reads || h >= in.n_haps) {
            bad = true;
            continue;
        }
        const uint64_t l = in.read_off[r + 1] - in.read_off[r], k = in.hap_off[h + 1] - in.hap_off[h];
        if (l > 0xffffffull || k > 0xffffffull) continue;  // found bad above
        plan_scan_pair(q, (uint32_t)l, (uint32_t)k,
                       (p > 0 && in.pair_read[p - 1] == r) || (p + 1 < in.n_pairs && in.pair_read[p + 1] == r));
    }
    const bool lead = (threadIdx.x & 31) == 0;
    auto add = [&](unsigned long long v, unsigned long long* to) {
        v = warp_sum(v);
        if (lead && v) atomicAdd(to, v);
    };
    auto add32 = [&](uint32_t v, uint32_t* to) {
        v = __reduce_add_sync(kFull, v);
        if (lead && v) atomicAdd(to, v);
    };
    auto top = [&](uint32_t v, uint32_t* to) {
        v = __reduce_max_sync(kFull, v);
        if (lead && v) atomicMax(to, v);
    };
    add(q.cells, &out->cells);
    add(q.sum_l, &out->sum_l);
    add(q.sum_k, &out->sum_k);
    add(q.cta_rows, &out->cta_rows);
    add(q.cta_strips, &out->cta_strips);
#pragma unroll
    for (int w = 0; w < 2; ++w) {
        add(q.short_cells[w], &out->short_cells[w]);
        add32(q.n_long[w], &out->n_long[w]);
        top(q.lmax_long[w], &out->lmax_long[w]);
#pragma unroll
        for (int z = 0; z < 2; ++z) {
            add(q.rows[w][z], &out->rows[w][z]);
            add(q.strips[w][z], &out->strips[w][z]);
        }
    }
    top(q.lmax, &out->lmax);
    add32(q.shared, &out->shared);
    if (__any_sync(kFull, bad) && lead) atomicOr(&out->bad, 1u);
}

__device__ __forceinline__ void pair_lengths(const PlanInput& in, uint32_t p, uint32_t& l, uint32_t& k) {
    const uint32_t r = in.pair_read[p], h = in.pair_hap[p];
    l = (uint32_t)(in.read_off[r + 1] - in.read_off[r]);
    k = (uint32_t)(in.hap_off[h + 1] - in.hap_off[h]);
}

// Class counts: per block in shared memory (a batch of equal reads has a dozen classes: global
// atomics alone would queue on them).
__global__ void __launch_bounds__(512) k_plan_hist(PlanInput in, PlanOutput out) {
    extern __shared__ uint32_t sh[];  // kClasses + kLongClasses
    Scratch& S = *static_cast<Scratch*>(out.scratch);
    for (int i = threadIdx.x; i < kClasses + kLongClasses; i += blockDim.x) sh[i] = 0u;
    __syncthreads();
    const uint32_t wide = 32u * (uint32_t)out.N, seg = 32u * (uint32_t)out.Nl;
    for (uint32_t p = blockIdx.x * blockDim.x + threadIdx.x; p < in.n_pairs; p += gridDim.x * blockDim.x) {
        uint32_t l, k;
        pair_lengths(in, p, l, k);
        if (k <= wide) {
            atomicAdd(&sh[run_of(l) * kG + (int)((k + out.N - 1) / out.N)], 1u);
        } else {
            const uint32_t W = (k + seg - 1) / seg;
            atomicAdd(&sh[kClasses + long_class(l, W)], out.wave ? W : 1u);
        }
    }
    __syncthreads();
    for (int i = threadIdx.x; i < kClasses; i += blockDim.x)
        if (sh[i]) atomicAdd(&S.hist[i], sh[i]);
    for (int i = threadIdx.x; i < kLongClasses; i += blockDim.x)
        if (sh[kClasses + i]) atomicAdd(&S.lhist[i], sh[kClasses + i]);
}

// Packs one run's counts c[1..32] into patterns; EMIT: writes them, else counts.  The last
// pattern slots of a run that has more patterns than kMaxPatterns take one team per item.
template <bool EMIT>
__device__ void pack_run(const uint32_t* cnt, int run, uint32_t* c, uint32_t* used, Pattern* pat, uint32_t item0,
                         uint32_t team0, uint32_t& n_pat, uint32_t& n_item, uint32_t& n_team) {
    uint32_t avail = 0;  // bit G - 1: class G has members
    for (int g = 1; g <= 32; ++g) {
        c[g] = cnt[g];
        used[g] = 0;
        if (c[g]) avail |= 1u << (g - 1);
    }
    n_pat = n_item = n_team = 0;
    while (avail) {
        uint8_t slot[kSlots];
        int n = 0, rem = 32;
        uint32_t left = avail;
        uint32_t times = 0xffffffffu;
        const bool single = n_pat >= kMaxPatterns - 33;
        while (rem > 0) {
            const uint32_t fit = left & (rem >= 32 ? 0xffffffffu : (1u << rem) - 1u);
            if (!fit) break;
            const int g = 32 - __clz(fit);
            // as many of this class as fit and are left
            const int m = single ? 1 : min((int)min(c[g], 32u), rem / g);
            for (int q = 0; q < m; ++q) slot[n++] = (uint8_t)g;
            rem -= m * g;
            times = min(times, c[g] / (uint32_t)m);
            left &= ~(1u << (g - 1));
            if (single) break;
        }
        // items of this pattern, `times` of them
        if (EMIT) {
            Pattern& P = pat[n_pat];
            P.item0 = item0 + n_item;
            P.team0 = team0 + n_team;
            P.teams = (uint32_t)n;
            P.run = (uint32_t)run;
            for (int q = 0; q < n; ++q) {
                const int g = slot[q];
                int m = 0, before = 0;
                for (int z = 0; z < n; ++z) {
                    m += slot[z] == g;
                    before += z < q && slot[z] == g;
                }
                P.g[q] = (uint8_t)g;
                P.mult[q] = (uint8_t)m;
                P.used[q] = used[g] + (uint32_t)before;
            }
        }
        for (int q = 0; q < n; ++q) {
            const int g = slot[q];
            c[g] -= times;
            used[g] += times;
            if (!c[g]) avail &= ~(1u << (g - 1));
        }
        n_pat++;
        n_item += times;
        n_team += times * (uint32_t)n;
    }
}

// One block: packs every run, lays classes, items and patterns out.
__global__ void __launch_bounds__(kRuns) k_plan_pack(PlanOutput out) {
    __shared__ uint32_t cnt[kRuns][kG];
    __shared__ uint32_t s_pat[kRuns], s_item[kRuns], s_team[kRuns];
    Scratch& S = *static_cast<Scratch*>(out.scratch);
    for (int i = threadIdx.x; i < kClasses; i += blockDim.x) cnt[i / kG][i % kG] = S.hist[i];
    __syncthreads();
    const int t = threadIdx.x, run = kRuns - 1 - t;  // thread 0: the longest reads
    uint32_t c[kG], used[kG], np, ni, nt;
    pack_run<false>(cnt[run], run, c, used, nullptr, 0, 0, np, ni, nt);
    s_pat[t] = np;
    s_item[t] = ni;
    s_team[t] = nt;
    __syncthreads();
    if (t == 0) {
        uint32_t a = 0, b = 0, d = 0;
        for (int q = 0; q < kRuns; ++q) {
            const uint32_t x = s_pat[q], y = s_item[q], z = s_team[q];
            s_pat[q] = a;
            s_item[q] = b;
            s_team[q] = d;
            a += x;
            b += y;
            d += z;
        }
        S.n_patterns = a;
        S.n_items = b;
        S.n_teams = d;
        out.H->n_witems = b;
    }
    if (t == 32) {
        uint32_t a = 0;
        for (int q = 0; q < kLongClasses; ++q) {
            const uint32_t x = S.lhist[q];
            S.lhist[q] = a;
            a += x;
        }
    }
    __syncthreads();
    // classes of a run lie side by side in the sorted list, runs in team order (a run has as
    // many teams as pairs)
    uint32_t at = s_team[t];
    for (int g = 1; g < kG; ++g) {
        S.hist[run * kG + g] = at;
        at += cnt[run][g];
    }
    pack_run<true>(cnt[run], run, c, used, S.patterns + s_pat[t], s_item[t], s_team[t], np, ni, nt);
}

// Counting sort of the short pairs; items of the wide ones.
__global__ void __launch_bounds__(256) k_plan_scatter(PlanInput in, PlanOutput out, uint32_t* __restrict__ sorted) {
    Scratch& S = *static_cast<Scratch*>(out.scratch);
    const uint32_t wide = 32u * (uint32_t)out.N, seg = 32u * (uint32_t)out.Nl;
    const int lane = threadIdx.x & 31;
    const uint32_t st = gridDim.x * blockDim.x;
    for (uint32_t base = blockIdx.x * blockDim.x; base < in.n_pairs; base += st) {
        const uint32_t p = base + threadIdx.x;
        uint32_t l = 0, k = 0, W = 0;
        int cls = -1;
        if (p < in.n_pairs) {
            pair_lengths(in, p, l, k);
            if (k <= wide) {
                cls = run_of(l) * kG + (int)((k + out.N - 1) / out.N);
            } else {
                W = (k + seg - 1) / seg;
            }
        }
        // one atomic per class and warp
        const unsigned same = __match_any_sync(kFull, cls);
        const int leader = __ffs(same) - 1;
        uint32_t at = 0;
        if (cls >= 0 && lane == leader) at = atomicAdd(&S.cursor[cls], (uint32_t)__popc(same));
        at = __shfl_sync(kFull, at, leader);
        if (cls >= 0) sorted[S.hist[cls] + at + (uint32_t)__popc(same & ((1u << lane) - 1u))] = p;
        if (W > 0) {
            const int lc = long_class(l, W);
            const uint32_t n = out.wave ? W : 1u;
            const uint32_t i0 = S.lhist[lc] + atomicAdd(&S.lcursor[lc], n);
            CtaPair cp;
            cp.pair = p;
            cp.w0 = 0;
            cp.W = 1;
            cp.strip = 0;
            cp.nstrip = W;
            cp.col0 = 0;
            cp.extra_base = W > 1 ? in.n_pairs + atomicAdd(&S.extra, W - 1) : 0u;
            cp.pad = 0;
            cp.bnd_in = cp.bnd_out = kNoBnd;
            unsigned long long r0 = 0;
            if (out.wave && W > 1) r0 = atomicAdd(&S.wrows, (unsigned long long)(W - 1) * l);
            for (uint32_t q = 0; q < n; ++q) {
                if (out.wave) {
                    cp.strip = (uint16_t)q;
                    cp.col0 = q * seg;
                    cp.bnd_in = q > 0 ? r0 + (unsigned long long)(q - 1) * l : kNoBnd;
                    cp.bnd_out = q + 1 < W ? r0 + (unsigned long long)q * l : kNoBnd;
                }
                out.cpairs[i0 + q] = cp;
                CtaItem it;
                it.first = i0 + q;
                it.n = 1;
                out.citems[i0 + q] = it;
            }
        }
    }
}

__global__ void __launch_bounds__(256) k_plan_emit(PlanOutput out, const uint32_t* __restrict__ sorted) {
    const Scratch& S = *static_cast<const Scratch*>(out.scratch);
    const uint32_t n = S.n_items, np = S.n_patterns;
    for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        uint32_t lo = 0, hi = np;  // the last pattern with item0 <= i
        while (hi - lo > 1) {
            const uint32_t mid = (lo + hi) / 2;
            if (S.patterns[mid].item0 <= i) lo = mid;
            else hi = mid;
        }
        const Pattern& P = S.patterns[lo];
        const uint32_t at = i - P.item0;
        WarpItem w;
        w.first_team = P.team0 + at * P.teams;
        w.n_teams = P.teams;
        out.witems[i] = w;
        uint32_t base = 0;
        for (uint32_t q = 0; q < P.teams; ++q) {
            Team t;
            const uint32_t g = P.g[q];
            t.pair = sorted[S.hist[P.run * kG + g] + P.used[q] + at * P.mult[q]];
            t.pair2 = kNoPair;
            t.base = (uint8_t)base;
            t.size = (uint8_t)g;
            t.pad = 0;
            out.teams[w.first_team + q] = t;
            base += g;
        }
    }
}

int blocks_for(uint32_t n, int threads, int most) {
    const uint32_t b = (n + threads - 1) / threads;
    return (int)(b < 1 ? 1 : b > (uint32_t)most ? most : b);
}

}  // namespace

size_t plan_scratch_bytes(uint32_t n_pairs) { return sizeof(Scratch) + (size_t)n_pairs * sizeof(uint32_t); }

void launch_plan_scan(const PlanInput& in, PlanScan* out, int sms, cudaStream_t s) {
    cudaMemsetAsync(out, 0, sizeof(PlanScan), s);
    const uint32_t n = in.n_pairs > in.n_reads ? in.n_pairs : in.n_reads;
    k_plan_scan<<<blocks_for(n, 256, sms * 4), 256, 0, s>>>(in, out);
}

PlanScan plan_scan_host(const PlanInput& in) {
    PlanScan bad{}, s{};
    bad.bad = 1;
    if (in.read_off[0] != 0 || in.hap_off[0] != 0) return bad;
    for (uint32_t r = 0; r < in.n_reads; ++r)
        if (in.read_off[r + 1] <= in.read_off[r] || in.read_off[r + 1] - in.read_off[r] > 0xffffffull) return bad;
    for (uint32_t h = 0; h < in.n_haps; ++h)
        if (in.hap_off[h + 1] <= in.hap_off[h] || in.hap_off[h + 1] - in.hap_off[h] > 0xffffffull) return bad;
    s.n_read_bases = in.read_off[in.n_reads];
    s.n_hap_bases = in.hap_off[in.n_haps];
    uint32_t last = 0xffffffffu;
    for (uint32_t p = 0; p < in.n_pairs; ++p) {
        const uint32_t r = in.pair_read[p], h = in.pair_hap[p];
        if (r >= in.n_reads || h >= in.n_haps) return bad;
        plan_scan_pair(s, (uint32_t)(in.read_off[r + 1] - in.read_off[r]), (uint32_t)(in.hap_off[h + 1] - in.hap_off[h]),
                       r == last || (p + 1 < in.n_pairs && in.pair_read[p + 1] == r));
        last = r;
    }
    return s;
}

void launch_plan_build(const PlanInput& in, const PlanOutput& out, int sms, cudaStream_t s) {
    uint32_t* const sorted = reinterpret_cast<uint32_t*>(static_cast<char*>(out.scratch) + sizeof(Scratch));
    cudaMemsetAsync(out.scratch, 0, offsetof(Scratch, pattern0), s);
    k_plan_hist<<<blocks_for(in.n_pairs, 2048, sms), 512, (kClasses + kLongClasses) * sizeof(uint32_t), s>>>(in, out);
    k_plan_pack<<<1, kRuns, 0, s>>>(out);
    k_plan_scatter<<<blocks_for(in.n_pairs, 256, sms * 4), 256, 0, s>>>(in, out, sorted);
    k_plan_emit<<<blocks_for(in.n_pairs, 256, sms * 4), 256, 0, s>>>(out, sorted);
}

}  // namespace phmm

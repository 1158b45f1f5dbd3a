// Skewed engines: the row-wise recurrence of Eq. 7 with the lanes of a team one row
// apart instead of in step, so that the deletion chain needs no scan.
//
// Each lane owns N consecutive columns; lane t of a team works on row s - t at step s.  What it
// needs of the column to its left (M, J and D-hat of the row above, from lane t - 1) was formed
// one step earlier, so D-hat runs through the lanes as one exact chain.  Per step and column,
// on the pipelined engine's records (Rec32J):
//     u  = b D[r-1][j-1] + (a M[r-1][j-1] + J[r-1][j-1])
//     M  = P' u        J = h J[r-1][j] + M[r-1][j]        D[r-1][j] = g D[r-1][j-1] + M[r-1][j]
// in the order of operations of the engines that keep all lanes on one row (M and J round the
// same), which need two more operations a column pair, the lane and warp scans and their power
// tables.  A pair of l rows on G lanes takes l + G steps.
//
// What bounds them: the register file's read ports.  A scheduler reads about two operands a
// thread and cycle (clock64 around loops of each, 1 to 4 warps a scheduler): an fmaf with three
// fresh operands takes 1.5 cycles, with one reused or constant 1.0 to 1.25; a __ffma2_rn takes 3.0
// and 2.0 to 2.3.  Packing therefore saves no FMA time, only issue slots.  Two forms:
//  - team_run_skew, scalar, for short teams: the fewest steps (l + G).  A bare step of 32
//    columns takes 295 cycles a scheduler.
//  - strip_run_skew, a lane's column halves in float2, the second half one row behind the first:
//    7.1 warp instructions issued per 32 cells (ncu; 8.5 on the scan engine, 9.8 in short teams), which
//    leaves slots for the boundary traffic; the strip takes 64 steps more than its rows.  On 60,000
//    uneven pairs the serial kind took 22.0 ms against 25.6 ms with the scalar form (28.6 ms on
//    the scan engine).
// The scalar form also runs FP64 short teams, where the FP64 pipe (2.1 FMAs a cycle and SM) is the
// bound and 5 operations a cell take the place of 6.5: 40 regions of short reads, 6.15 ms
// against 6.65 ms on the scan engine, with 32 columns a lane (16: 10.8 ms).
// With g constant (G10: gcp Phred 10 throughout, the T_II = T_DD = 0.1 that Section 2 fixes) the
// D-hat chain reads one operand less.
//
// Range: every lane keeps an exponent E of its own, non-decreasing along the team's lanes;
// what arrives from the left is scaled by 2^(E_left - E) <= 1.  Every R steps (all lanes at
// once, so lanes are on different rows) each lane looks at its largest value and asks for a
// new exponent; a prefix maximum over the lanes keeps the order.
#pragma once

#include <type_traits>

#include "engine.cuh"

namespace phmm {

// Range control as pipe_range(), with the drop of a column's max(M, J): J[r] = h J[r-1] +
// M[r-1] keeps at least min(1, h) of it a row (prep: the largest -log2 h of the batch), which
// lets R be about three times what the drop of max(M, I) allows.
template <typename T = float>
__device__ __forceinline__ PipeRange skew_range(const BatchHeader* __restrict__ H) {
    const uint32_t dg[4] = {H->skst->drop, H->dropgrow[1], H->dropgrow[2], H->dropgrow[3]};
    return pipe_range<T>(dg);
}
// gcp Phred 10 throughout the batch
__device__ __forceinline__ bool skew_g10(const SkewStats* st) { return st->gcp_max == 10u && st->gcp_inv == 245u; }
constexpr float kG10 = 0.1f;

// 2^d for d <= 0: exact down to the smallest subnormal, then 0.
template <typename T = float>
__device__ __forceinline__ T pow2_down(int d) {
    if constexpr (std::is_same_v<T, float>)
        return d >= -126 ? Num<float>::pow2(d) : d >= -149 ? __uint_as_float(1u << (d + 149)) : 0.f;
    else
        return d >= -1022 ? Num<double>::pow2(d) : d >= -1074 ? __longlong_as_double(1ll << (d + 1074)) : 0.0;
}

// The exponent side of a checkpoint (see above), common to both forms.  x: the lane's largest
// |M|, |J|; keep: the lane holds its exponent (not started: C / k must stay in range; or done);
// Eb: the exponent of what enters the team's first lane from a strip to its left (INT_MIN:
// none).  Returns the new exponent.
template <typename T>
__device__ __forceinline__ int skew_exponent(T x, int E, uint32_t& flags, int lt, bool keep, int Eb,
                                             const PipeRange& rng) {
    using NT = Num<T>;
    const int e = NT::expo(x);
    const bool first = lt == 0;
    const bool has_left = !first || Eb != INT_MIN;
    int want = E;
    if (!keep) {
        if (e == INT_MAX) flags |= PF_NONFINITE;
        else if (e == INT_MIN) want = has_left ? INT_MIN : E;  // nothing representable: follow the left
        else if (e > rng.hi || e <= NT::kLo) want = E + (e - rng.target);
    }
    int En = first ? max(want, Eb) : want;
#pragma unroll
    for (int s = 0; s < 5; ++s) {
        const int up = __shfl_up_sync(kFull, En, 1 << s);
        if (lt >= (1 << s)) En = max(En, up);
    }
    if (En == INT_MIN) En = E;
    // a lane forced to its left neighbour's scale holds little beside it; one with nothing
    // representable holds no mass of its own
    if (!keep && En == want && e <= rng.danger) flags |= PF_DANGER;
    return En;
}
// 2^sh as one or two exact factors (sh beyond twice the format's range: 0, or the largest).
template <typename T>
__device__ __forceinline__ void skew_factors(int sh, T& f, T& g) {
    using NT = Num<T>;
    const int s1 = max(NT::kMinExp, min(sh, -NT::kMinExp)), s2 = sh - s1;
    f = NT::pow2(s1);
    g = s2 < NT::kMinExp ? T(0) : NT::pow2(min(s2, -NT::kMinExp));
}
// Scale of what arrives from the left, 2^(E_left - E) <= 1.
template <typename T = float>
__device__ __forceinline__ T skew_left_scale(int E, int lt, int Eb) {
    const int El = __shfl_up_sync(kFull, E, 1);
    return lt == 0 && Eb == INT_MIN ? T(1) : pow2_down<T>((lt == 0 ? Eb : El) - E);
}

// Sum over the team's lanes (s: the lane's, FP64, in scale E), in the scale of the lane that
// holds the largest one.  RESCALED when that lane's exponent moved.
__device__ __forceinline__ SegOut skew_sum(double s, int E, int E0, uint32_t flags, int lt, int tlast) {
    // the team's lanes as a mask (a lane outside every team is its own team)
    const int base = (int)(threadIdx.x & 31) - lt, size = tlast - base + 1;
    const unsigned mask = size >= 32 ? kFull : ((1u << size) - 1u) << base;
    const int es = Num<double>::expo(s);
    const bool some = s != 0.0 && es != INT_MIN && es != INT_MAX;
    // largest lane sum: its exponent over all lanes, and the scale of the first lane with it
    const int key = some ? E + es : INT_MIN;
    const int kmax = __reduce_max_sync(mask, key);
    const int El = key == kmax ? E : INT_MIN;
    int Eref = __reduce_max_sync(mask, El);
    if (kmax == INT_MIN) Eref = __reduce_max_sync(mask, E);
    const double mine = (some || s != 0.0) ? scale2<double>(s, E - Eref) : 0.0;
    const uint32_t f = __reduce_or_sync(mask, flags);
    SegOut o;
    double t = mine;
#pragma unroll
    for (int q = 0; q < 5; ++q) {
        const double up = __shfl_up_sync(kFull, t, 1 << q);
        if (lt >= (1 << q)) t += up;
    }
    o.S = __shfl_sync(kFull, t, tlast);
    o.E = Eref;
    o.flags = f | (Eref != E0 ? PF_RESCALED : 0u);
    return o;
}

// C / k of Eq. 1 in the scale of a lane with exponent E >= E0
template <typename T = float>
__device__ __forceinline__ T skew_init(const PipeRange& rng, int k, int E0, int E) {
    return (T)(ldexp(1.0, rng.target) / (double)k) * pow2_down<T>(E0 - E);
}

// Match masks of a lane's columns (Eq. 3), by read base code (4: N, matches everything), at
// sm[32 code].  HALVES: bit 2q for column q of the lane's first half, bit 2q + 1 for column q of
// the second (the order in which the packed form reads them); else bit q for column q.
template <int N, bool HALVES>
__device__ __forceinline__ void skew_masks(const uint8_t* __restrict__ hap, int k, int col0, uint32_t* sm,
                                           uint32_t& flags) {
    constexpr int H = N / 2;
    uint32_t bmA = 0, bmC = 0, bmG = 0, bmT = 0;
    const int nvalid = max(0, min(k - col0, N));
#pragma unroll
    for (int c = 0; c < N; ++c) {
        if (c < nvalid) {
            const int code = base_code(hap[col0 + c]);
            const uint32_t bit = 1u << (!HALVES ? c : c < H ? 2 * c : 2 * (c - H) + 1);
            if (code < 0) flags |= PF_BAD;
            if (code == 0 || code == 4) bmA |= bit;
            if (code == 1 || code == 4) bmC |= bit;
            if (code == 2 || code == 4) bmG |= bit;
            if (code == 3 || code == 4) bmT |= bit;
        }
    }
    sm[0] = bmA;
    sm[32] = bmC;
    sm[64] = bmG;
    sm[96] = bmT;
    sm[128] = 0xffffffffu;
}

// ------------------------------------------------------------------------------------
// Short teams (scalar form).
// ------------------------------------------------------------------------------------
template <typename T>
struct SkewLane {
    T m, j, d;               // left of the lane (the row above its row)
    T mi;                        // (lean form)
    T pm, px, a, b, h, g, gp;  // the lane's row; gp: g of the row above (not used with G10)
    T lsc;                       // 2^(E of the left lane - E)
    int E;
};

// The lane's columns of one step; m, j, d: in the values left of the lane, out those at its
// last column (of the row above this one), which the lane to the right takes at the next step.
template <typename T, int N, bool G10>
__device__ __forceinline__ void skew_row(T (&M)[N], T (&J)[N], SkewLane<T>& L, uint32_t mask) {
    const T gp = G10 ? (T)kG10 : L.gp;
    const T mo = M[N - 1], jo = J[N - 1];
    // column q's old M and J have their last uses (column q + 1's partial t and D-hat, its own
    // J) before its new M is formed, so the new values take the old ones' registers
    T t = fma(L.a, L.m, L.j);
    T dA = L.d, dB = fma(gp, L.d, L.m);
#pragma unroll
    for (int q = 0; q < N; ++q) {
        const T u = fma(L.b, dA, t);
        const T o = M[q];
        if (q + 1 < N) {
            dA = dB;
            dB = fma(gp, dB, o);
            t = fma(L.a, o, J[q]);
        }
        J[q] = fma(L.h, J[q], o);
        M[q] = (((mask >> q) & 1u) ? L.pm : L.px) * u;
    }
    L.m = mo;
    L.j = jo;
    L.d = dB;
}

// The same in the lean engine's order of operations, on its records (Rec32): I in the place of
// J, with L.mi = T_MI; one operation more a cell.
template <int N>
__device__ __forceinline__ void skew_row_lean(float (&M)[N], float (&I)[N], SkewLane<float>& L, uint32_t mask) {
    float ml = L.m, il = L.j, d = L.d;
#pragma unroll
    for (int q = 0; q < N; ++q) {
        const float u = fmaf(L.a, ml, fmaf(L.b, d, il));
        d = fmaf(L.gp, d, ml);
        ml = M[q];
        il = I[q];
        I[q] = fmaf(L.mi, ml, L.h * il);
        M[q] = (((mask >> q) & 1u) ? L.pm : L.px) * u;
    }
    L.m = ml;
    L.j = il;
    L.d = d;
}

// Records of one pair's rows in shared memory, two blocks of 32 rows ahead of the team's first
// lane: slot row & 127.
struct SoloStage {
    float4 r0[128], r1[128];
    uint32_t mask[5 * 32];
};

// Lane lt of a team of tlast - (first lane) + 1 lanes runs columns lt N .. of its pair; steps =
// the largest l + team size - 1 of the warp's teams; every lane of a team is at rows 2 .. l at
// steps plain0 .. plain1.  A lane starts as M = 0, J = C / k and keeps that before row 1 (P' = 0,
// h = 1); row 1's record has h = 0, so that J = 0 and M = P' C / k follow; after row l a lane
// does nothing.  Records come through L1, one step ahead, or (FORM solo and lean: the warp has one
// team, all 32 lanes) through shared memory: the first lane's record is new to L1 at every
// step, which is what a scheduler's only warp waits for (a step of 900 cycles).
enum SkewForm { kTeams, kSolo, kLean };
template <typename T, int N, bool G10, SkewForm FORM = kTeams>
__device__ SegOut team_run_skew(const std::conditional_t<FORM == kLean, Rec32, typename Num<T>::RecJ>* __restrict__ rec, int l, int steps, int plain0, int plain1,
                                const uint8_t* __restrict__ hap, int k, int lt, int tlast, const PipeRange& rng,
                                uint32_t* sm, SoloStage* st = nullptr, int rows = 0) {
    static_assert(N <= 32, "match masks hold 32 columns");
    using Rec = std::conditional_t<FORM == kLean, Rec32, typename Num<T>::RecJ>;
    uint32_t flags = rng.ok ? 0u : PF_DEGEN, mflags = 0;
    auto fetch = [&](int row) {  // solo: the pair's rows, by every lane
        if (row <= rows) {
            const float4* src = reinterpret_cast<const float4*>(rec + (row - 1));
            cp_async16_cg(&st->r0[row & 127], src);
            cp_async16_cg(&st->r1[row & 127], src + 1);
        }
        cp_async_commit();
    };
    if constexpr (FORM != kTeams) {
        __syncwarp();  // the warp's previous pair is done with the stage
        fetch(1 + (threadIdx.x & 31));
        fetch(33 + (threadIdx.x & 31));
    }
    skew_masks<N, false>(hap, k, lt * N, sm, flags);
    const int E0 = Num<T>::kLog2C - rng.target;
    const T cin = l > 0 && k > 0 ? skew_init<T>(rng, k, E0, E0) : T(0);
    T M[N], J[N];
#pragma unroll
    for (int q = 0; q < N; ++q) {
        M[q] = T(0);
        J[q] = cin;
    }
    SkewLane<T> L;
    L.m = L.d = L.g = T(0);
    L.j = cin;
    L.lsc = T(1);
    L.E = E0;
    const int l1 = max(l, 1) - 1;
    int r = 1 - lt;  // the lane's row
    auto load = [&](int i) {  // record of row i + 1
        if constexpr (FORM == kTeams) {
            return load_recj(rec + i);
        } else {
            const float4 a = st->r0[(i + 1) & 127], b = st->r1[(i + 1) & 127];
            Rec x;
            x.pm = a.x; x.px = a.y; x.a = a.z; x.b = a.w;
            if constexpr (FORM == kLean) { x.mi = b.x; x.g = b.y; x.gm = b.z; }
            else { x.h = b.x; x.g = b.y; x.mi = b.z; }
            x.meta = __float_as_uint(b.w);
            return x;
        }
    };
    if constexpr (FORM != kTeams) {
        cp_async_wait_0();
        __syncwarp();
    }
    Rec nxt = load(max(0, min(r - 1, l1)));
    int ck = rng.R;  // checkpoint after step ck
    // EDGE: some lane is before row 2 or past row l
    auto run = [&](auto edge, int& s, int e) {
        constexpr bool EDGE = decltype(edge)::value;
#pragma unroll 1
        for (; s <= e; ++s, ++r) {
            const T um = __shfl_up_sync(kFull, L.m, 1), uj = __shfl_up_sync(kFull, L.j, 1),
                        ud = __shfl_up_sync(kFull, L.d, 1);
            L.pm = nxt.pm;
            L.px = nxt.px;
            L.a = nxt.a;
            L.b = nxt.b;
            if constexpr (FORM == kLean) {
                L.mi = nxt.mi;
                L.h = EDGE && r == 1 ? 0.f : nxt.g;
            } else {
                L.h = nxt.h;
            }
            if constexpr (!G10) {
                L.gp = L.g;
                L.g = nxt.g;
            }
            mflags |= (uint32_t)nxt.meta;
            const uint32_t mask = sm[((uint32_t)nxt.meta & META_CODE_MASK) * 32];
            if constexpr (EDGE) {
                if (r < 1) {  // not started: hold
                    L.pm = L.px = T(0);
                    L.h = T(1);
                    if constexpr (FORM == kLean) L.mi = 0.f;
                }
            }
            if (!EDGE || r <= l) {
                L.m = lt == 0 ? T(0) : um * L.lsc;
                L.j = lt == 0 ? (EDGE && r == 1 ? cin : T(0)) : uj * L.lsc;
                L.d = lt == 0 ? T(0) : ud * L.lsc;
                if constexpr (FORM == kLean) skew_row_lean<N>(M, J, L, mask);
                else skew_row<T, N, G10>(M, J, L, mask);
            }
            nxt = load(EDGE ? max(0, min(r, l1)) : min(r, l1));
        }
    };
    for (int s = 1; s <= steps;) {
        // (steps between events run in a loop of their own, in which nothing but the row writes
        // M and J)
        const int e = FORM == kTeams ? min(ck, steps) : min(min(ck, steps), (s + 31) & ~31);
        if (s < plain0) run(std::true_type{}, s, min(e, plain0 - 1));
        else if (s <= plain1) run(std::false_type{}, s, min(e, plain1));
        else run(std::true_type{}, s, e);
        if constexpr (FORM != kTeams) {
            if (((s - 1) & 31) == 0) {
                // rows up to s + 31 have landed, rows before s - 31 are done with; a lane's next record may
                // have been taken before it landed
                cp_async_wait_0();
                __syncwarp();
                nxt = load(max(0, min(r - 1, l1)));
                fetch(s + 32 + (threadIdx.x & 31));
            }
        }
        if (s > ck && s <= steps) {
            ck += rng.R;
            T x0 = 0, x1 = 0;
#pragma unroll
            for (int q = 0; q < N; ++q) {
                if (q & 1) x1 = fmax(x1, fmax(fabs(M[q]), fabs(J[q])));
                else x0 = fmax(x0, fmax(fabs(M[q]), fabs(J[q])));
            }
            const int En = skew_exponent(fmax(x0, x1), L.E, flags, lt, r - 1 < 1 || r - 1 > l, INT_MIN, rng);
            if (En != L.E) {
                T f, g;
                skew_factors(L.E - En, f, g);
                for (;;) {
#pragma unroll
                    for (int q = 0; q < N; ++q) {
                        M[q] *= f;
                        J[q] *= f;
                    }
                    L.m *= f;
                    L.j *= f;
                    L.d *= f;
                    if (g == T(1)) break;  // one factor, nearly always
                    f = g;
                    g = T(1);
                }
                L.E = En;
            }
            L.lsc = skew_left_scale<T>(L.E, lt, INT_MIN);
        }
    }
    double s = 0.0;
    if (l > 0) {
        // Eq. 4 (I = T_MI J on the last row)
        if (mflags & META_BAD) flags |= PF_BAD;
        if (mflags & META_DEGEN) flags |= PF_DEGEN;
        const double mi = FORM == kLean ? 1.0 : (double)__ldg(&rec[l1].mi);
        const int nvalid = max(0, min(k - lt * N, N));
#pragma unroll
        for (int q = 0; q < N; ++q)
            if (q < nvalid) s += (double)M[q] + mi * (double)J[q];
    }
    if constexpr (FORM != kTeams) cp_async_wait_0();  // nothing may land in the stage after this pair
    return skew_sum(s, L.E, E0, flags, lt, tlast);
}

// One pair on one warp: the fewer columns a lane, the shorter a step.
template <int N, bool G10, SkewForm FORM>
__device__ __forceinline__ SegOut pair_run_skew(const std::conditional_t<FORM == kLean, Rec32, Rec32J>* __restrict__ rec, int l,
                                                const uint8_t* __restrict__ hap, int k, const PipeRange& rng,
                                                SoloStage& st) {
    const int lane = threadIdx.x & 31;
    auto go = [&](auto n) {
        constexpr int Nl = decltype(n)::value;
        const int g = (k + Nl - 1) / Nl;
        const bool in = lane < g;  // (the others are teams of no rows)
        return team_run_skew<float, Nl, G10, FORM>(rec, in ? l : 0, l + g - 1, g + 1, l, hap, in ? k : 0, in ? lane : 0,
                                                   in ? g - 1 : lane, rng, st.mask + lane, &st, l);
    };
    if (k <= 32 * 8) return go(std::integral_constant<int, 8>{});
    if (k <= 32 * 16) return go(std::integral_constant<int, 16>{});
    return go(std::integral_constant<int, N>{});
}

// ------------------------------------------------------------------------------------
// Strips of wide pairs (packed form): one warp runs 32 N columns.  A lane's halves (.x: columns
// 0 .. H-1, .y: columns H .. N-1, H = N / 2) are two virtual lanes; virtual lane v works on row
// s - v at step s.  The left strip's boundary (per row index i: M, J, D-hat of row i at its last
// column and the exponent) enters lane 0.  Checkpoints of strip j happen 64 steps earlier than
// those of strip j - 1 (mod R), which is how much later row i leaves the left strip than it
// enters this one, so the exponent in the boundary changes exactly at this strip's checkpoints.
//
// Rows outside 1 .. l need no branches, only coefficients: a half starts as M = 0, J = C / k and
// keeps that on rows with P' = 0, h = 1; row 1's record has h = 0, so that J = 0 and M = P' C / k
// follow; row l + 1 with P' = 0, h = T_MI_l leaves M_l + I_l of every column in J (Eq. 4's
// summands), where further rows with P' = 0, h = 1 keep it until the strip is done.
// ------------------------------------------------------------------------------------
struct SkewLane2 {
    float2 m, j, d;               // left of each half
    float2 a, b, h, gp;           // the halves' rows (.y: the row before .x's)
    float pmx, pxx, pmy, pxy;
    float lsc;
    uint32_t mprev;               // match mask of .x's row
    int E;
};

template <int H, bool G10>
__device__ __forceinline__ void skew_row2(float2 (&M)[H], float2 (&J)[H], SkewLane2& L, uint32_t mask) {
    const float2 gp = G10 ? make_float2(kG10, kG10) : L.gp;
    const float2 mo = M[H - 1], jo = J[H - 1];
    float2 t = __ffma2_rn(L.a, L.m, L.j);
    float2 dA = L.d, dB = __ffma2_rn(gp, L.d, L.m);
#pragma unroll
    for (int q = 0; q < H; ++q) {
        const float2 u = __ffma2_rn(L.b, dA, t);
        const float2 o = M[q];
        if (q + 1 < H) {
            dA = dB;
            dB = __ffma2_rn(gp, dB, o);
            t = __ffma2_rn(L.a, o, J[q]);
        }
        J[q] = __ffma2_rn(L.h, J[q], o);
        const float2 p = make_float2(((mask >> (2 * q)) & 1u) ? L.pmx : L.pxx,
                                     ((mask >> (2 * q + 1)) & 1u) ? L.pmy : L.pxy);
        M[q] = __fmul2_rn(p, u);
    }
    L.m = mo;
    L.j = jo;
    L.d = dB;
}

// Match bits of the halves' rows: even bits from .x's row, odd bits from .y's (the row
// before), in one word that the optimiser cannot see through: 310 cycles a step, against 340 with
// the same merge in C++.
__device__ __forceinline__ uint32_t skew_mask2(SkewLane2& L, uint32_t mk) {
    uint32_t m;
    asm("lop3.b32 %0, %1, %2, 0x55555555, 0xe4;" : "=r"(m) : "r"(mk), "r"(L.mprev));
    L.mprev = mk;
    return m;
}

// Per warp: the coefficients of 128 rows, each beside those of the row before (the halves'
// pairs as they are used), in slots ordered by row parity and then row / 2, so the lanes'
// rows, two apart, lie side by side; the records of two blocks of 32 rows as they arrive; two
// blocks of boundary rows; match masks.
struct SkewStage {
    float4 c0[128];  // a, a of the row before, b, b of the row before
    float4 c1[128];  // h, h of the row before, g of the row before, g of the row before that
    float4 c2[128];  // pm, px, pm of the row before, px of the row before
    uint32_t code[128];
    float4 raw[128];
    float4 bnd[64];
    uint32_t mask[5 * 32];
};
__device__ __forceinline__ int skew_slot(int row) { return ((row & 1) << 6) | ((row & 127) >> 1); }

// Boundary rows of the wave kind carry a tag beside the exponent, so that a row is complete
// when its 16 bytes (one relaxed access) carry this launch's tag.
constexpr int kWaveTagBits = 6;
constexpr uint32_t kWaveTagMask = (1u << kWaveTagBits) - 1u;
constexpr int kWaveMaxE = (1 << (31 - kWaveTagBits)) - 1;
__device__ __forceinline__ uint4 ld_row_relaxed(const float4* p) {
    unsigned long long a, b;
    asm volatile("{ .reg .b128 t; ld.relaxed.gpu.global.b128 t, [%2]; mov.b128 {%0, %1}, t; }"
                 : "=l"(a), "=l"(b) : "l"(p) : "memory");
    return make_uint4((uint32_t)a, (uint32_t)(a >> 32), (uint32_t)b, (uint32_t)(b >> 32));
}
__device__ __forceinline__ void st_row_relaxed(float4* p, float m, float j, float d, uint32_t w) {
    const unsigned long long a = (unsigned long long)__float_as_uint(m) | ((unsigned long long)__float_as_uint(j) << 32);
    const unsigned long long b = (unsigned long long)__float_as_uint(d) | ((unsigned long long)w << 32);
    asm volatile("{ .reg .b128 t; mov.b128 t, {%1, %2}; st.relaxed.gpu.global.b128 [%0], t; }"
                 ::"l"(p), "l"(a), "l"(b) : "memory");
}
constexpr int kWaveBlock = 16;  // boundary rows taken at a time

// WAVE: the left strip runs at the same time on another warp (boundary rows tagged `tag`);
// else its boundary is complete.  in: the left strip's boundary (index = row, 1 .. l - 1),
// null for none; out: this strip's, null for none.
template <int N, bool WAVE, bool G10>
__device__ SegOut strip_run_skew(const Rec32J* __restrict__ rec, int l, const uint8_t* __restrict__ hap, int k,
                                 int strip, int scol, const PipeRange& rng, const float4* in, float4* out, SkewStage& st,
                                 uint32_t tag, uint32_t* __restrict__ status) {
    static_assert(N <= 32 && N % 2 == 0, "match masks hold 32 columns; two halves");
    constexpr int H = N / 2;
    const int lane = threadIdx.x & 31;
    uint32_t flags = rng.ok ? 0u : PF_DEGEN, mflags = 0;
    skew_masks<N, true>(hap, k, scol + lane * N, st.mask + lane, flags);
    const bool has_left = in != nullptr, has_right = out != nullptr;
    const float mil = __ldg(&rec[l - 1].mi);
    // block b: rows 32 b + 1 .. 32 b + 32, boundary rows 32 b .. 32 b + 31, in three turns:
    // copied as they are, 32 steps later laid out, 32 steps later used
    auto fetch = [&](int b) {
        const int row = 32 * b + 1 + lane;
        if (row <= l) {
            const float4* src = reinterpret_cast<const float4*>(rec + (row - 1));
            cp_async16_cg(&st.raw[2 * (row & 63)], src);
            cp_async16_cg(&st.raw[2 * (row & 63) + 1], src + 1);
        }
        cp_async_commit();
    };
    // row's record in the stage: before row 1 not started, row l + 1 collects, then hold
    auto row_at = [&](int row, float4& p, float4& q) {
        p = make_float4(0.f, 0.f, 0.f, 0.f);
        q = make_float4(row == l + 1 ? mil : 1.f, 0.f, 0.f, __uint_as_float(4u));
        if (row >= 1 && row <= l) {
            p = st.raw[2 * (row & 63)];
            q = st.raw[2 * (row & 63) + 1];
        }
    };
    auto lay_out = [&](int b) {
        const int row = 32 * b + 1 + lane, sl = skew_slot(row);
        float4 p, q, p1, q1, p2, q2;
        row_at(row, p, q);
        row_at(row - 1, p1, q1);
        row_at(row - 2, p2, q2);
        st.c0[sl] = make_float4(p.z, p1.z, p.w, p1.w);
        st.c1[sl] = make_float4(q.x, q1.x, q1.y, q2.y);
        st.c2[sl] = make_float4(p.x, p.y, p1.x, p1.y);
        st.code[sl] = (__float_as_uint(q.w) & META_CODE_MASK) * 32u;
        mflags |= __float_as_uint(q.w);
    };
    auto fetch_bnd = [&](int b) {  // serial: the left strip is complete
        const int i = 32 * b + lane;
        if (has_left && i >= 1) {
            if (i < l) cp_async16_cg(&st.bnd[i & 63], in + i);
            else st.bnd[i & 63] = make_float4(0.f, 0.f, 0.f, 0.f);
        }
    };
    // the wave kind's boundary rows kWaveBlock b ..: loaded a block ahead, taken when tagged
    uint4 pv = make_uint4(0u, 0u, 0u, 0u);
    auto load_bnd = [&](int b) {
        const int i = kWaveBlock * b + lane;
        if (has_left && lane < kWaveBlock && i >= 1 && i < l) pv = ld_row_relaxed(in + i);
    };
    auto take_bnd = [&](int b) {
        const int i = kWaveBlock * b + lane;
        const bool mine = has_left && lane < kWaveBlock && i >= 1, need = mine && i < l;
        long long spins = 0;
        // (after one wait has run out the strip waits no more: its result is an error already)
        while (__any_sync(kFull, need && (pv.w & kWaveTagMask) != tag) && !(flags & PF_TIMEOUT)) {
            if (++spins > kSpinLimit) {
                flags |= PF_TIMEOUT;
                if (lane == 0) atomicOr(status, ST_TIMEOUT);
                break;
            }
            if (spins > kSpinFast) __nanosleep(64);
            if (need && (pv.w & kWaveTagMask) != tag) pv = ld_row_relaxed(in + i);
        }
        if (mine)
            st.bnd[i & 63] = need ? make_float4(__uint_as_float(pv.x), __uint_as_float(pv.y), __uint_as_float(pv.z),
                                                __int_as_float((int)pv.w >> kWaveTagBits))
                                  : make_float4(0.f, 0.f, 0.f, 0.f);
        __syncwarp();
    };
    __syncwarp();  // the previous strip of this warp is done with the stage
    for (int q = lane; q < 64; q += 32) {
        const int sl = skew_slot(q - 63);  // rows -63 .. 0: not started
        st.c0[sl] = st.c2[sl] = make_float4(0.f, 0.f, 0.f, 0.f);
        st.c1[sl] = make_float4(1.f, 1.f, 0.f, 0.f);
        st.code[sl] = 4u * 32u;
        st.bnd[q] = make_float4(0.f, 0.f, 0.f, 0.f);
    }
    __syncwarp();
    fetch(0);
    if constexpr (!WAVE) {
        fetch_bnd(0);
        cp_async_commit();
    } else {
        load_bnd(0);
        take_bnd(0);
        load_bnd(1);
    }
    cp_async_wait_0();
    __syncwarp();
    lay_out(0);
    __syncwarp();
    fetch(1);
    cp_async_wait_0();
    __syncwarp();
    lay_out(1);
    __syncwarp();
    if constexpr (!WAVE) fetch_bnd(1);
    fetch(2);

    const int E0 = Num<float>::kLog2C - rng.target;
    // the left strip's exponent: that of boundary row 1 up to the first checkpoint, where it
    // may change next
    int Eb = has_left && l > 1 ? __float_as_int(st.bnd[1].w) : INT_MIN;
    SkewLane2 L;
    L.m = L.j = L.d = make_float2(0.f, 0.f);
    L.mprev = 0;
    L.E = max(E0, Eb);
    L.lsc = lane == 0 && Eb != INT_MIN ? pow2_down(Eb - L.E) : 1.f;
    float2 M[H], J[H];
    {
        const float c = skew_init(rng, k, E0, L.E);
#pragma unroll
        for (int q = 0; q < H; ++q) {
            M[q] = make_float2(0.f, 0.f);
            J[q] = make_float2(c, c);
        }
        L.j = make_float2(c, c);
        // boundary row 0 (Eb >= E0: a strip keeps its first exponent until its last lane started)
        __syncwarp();
        if (lane == 0) st.bnd[0] = make_float4(0.f, Eb == INT_MIN ? c : scale2(c, L.E - Eb), 0.f, 0.f);
        __syncwarp();
    }
    const int nl = min(32, (k - scol + N - 1) / N);
    const int steps = l + 2 * nl;
    const bool sends = has_right && lane == 31;
    int ck = rng.R - (int)((64ll * strip) % rng.R);  // checkpoint after step ck
    int sl = skew_slot(1 - 2 * lane);
    float4 n0 = st.c0[sl], n1 = st.c1[sl], n2 = st.c2[sl];
    uint32_t mk = st.mask[st.code[sl] + lane];
    constexpr int kTurn = WAVE ? kWaveBlock : 32;
    for (int s = 1; s <= steps;) {
        const int e = min(min(min(ck, (s + kTurn - 1) & ~(kTurn - 1)), steps), s <= 65 ? 65 : steps);
        const bool send = sends && s > 65;
        // (the steps between events in a loop of their own, as in team_run_skew)
#pragma unroll 1
        for (; s <= e; ++s) {
            if (send) {  // row s - 65 at the strip's last column
                if constexpr (WAVE) st_row_relaxed(out + (s - 65), L.m.y, L.j.y, L.d.y, ((uint32_t)L.E << kWaveTagBits) | tag);
                else __stcg(out + (s - 65), make_float4(L.m.y, L.j.y, L.d.y, __int_as_float(L.E)));
            }
            const float4 v = st.bnd[(s - 1) & 63];
            const float um = __shfl_up_sync(kFull, L.m.y, 1), uj = __shfl_up_sync(kFull, L.j.y, 1),
                        ud = __shfl_up_sync(kFull, L.d.y, 1);
            L.m = make_float2((lane == 0 ? v.x : um) * L.lsc, L.m.x);
            L.j = make_float2((lane == 0 ? v.y : uj) * L.lsc, L.j.x);
            L.d = make_float2((lane == 0 ? v.z : ud) * L.lsc, L.d.x);
            L.a = make_float2(n0.x, n0.y);
            L.b = make_float2(n0.z, n0.w);
            L.h = make_float2(n1.x, n1.y);
            if constexpr (!G10) L.gp = make_float2(n1.z, n1.w);
            L.pmx = n2.x;
            L.pxx = n2.y;
            L.pmy = n2.z;
            L.pxy = n2.w;
            skew_row2<H, G10>(M, J, L, skew_mask2(L, mk));
            // (after the row, which has had its last use of the ones they replace)
            sl = skew_slot(s + 1 - 2 * lane);
            n0 = st.c0[sl];
            n1 = st.c1[sl];
            n2 = st.c2[sl];
            mk = st.mask[st.code[sl] + lane];
        }
        // after step e
        if ((e & 31) == 0) {
            cp_async_wait_0();
            __syncwarp();  // what was copied has landed; every lane is done with the rows overwritten next
            lay_out(e / 32 + 1);
            if (e == 32 && lane == 0) st.bnd[0] = make_float4(0.f, 0.f, 0.f, 0.f);
            __syncwarp();
            if constexpr (!WAVE) fetch_bnd(e / 32 + 1);
            fetch(e / 32 + 2);
        }
        if constexpr (WAVE) {
            if ((e & (kWaveBlock - 1)) == 0) {
                take_bnd(e / kWaveBlock);
                load_bnd(e / kWaveBlock + 1);
            }
        }
        if (e == ck) {
            ck += rng.R;
            if (has_left && e < l) Eb = __float_as_int(st.bnd[e & 63].w);
            const int r = e - 2 * lane;  // .x's row
            float2 x2 = make_float2(0.f, 0.f);
#pragma unroll
            for (int q = 0; q < H; ++q) {
                x2.x = fmaxf(x2.x, fmaxf(fabsf(M[q].x), fabsf(J[q].x)));
                x2.y = fmaxf(x2.y, fmaxf(fabsf(M[q].y), fabsf(J[q].y)));
            }
            const int En = skew_exponent(fmaxf(x2.x, x2.y), L.E, flags, lane, r < 2 || r > l, Eb, rng);
            if (En != L.E) {
                float f, g;
                skew_factors(L.E - En, f, g);
                for (;;) {
                    const float2 f2v = make_float2(f, f);
#pragma unroll
                    for (int q = 0; q < H; ++q) {
                        M[q] = __fmul2_rn(M[q], f2v);
                        J[q] = __fmul2_rn(J[q], f2v);
                    }
                    L.m = __fmul2_rn(L.m, f2v);
                    L.j = __fmul2_rn(L.j, f2v);
                    L.d = __fmul2_rn(L.d, f2v);
                    if (g == 1.f) break;  // one factor, nearly always
                    f = g;
                    g = 1.f;
                }
                L.E = En;
            }
            L.lsc = skew_left_scale(L.E, lane, Eb);
            if constexpr (WAVE)
                if (L.E > kWaveMaxE || L.E < -kWaveMaxE) flags |= PF_DANGER;  // does not fit beside the tag
        }
    }
    cp_async_wait_0();  // nothing may land in the stage after this strip
    __syncwarp();
    if (mflags & META_BAD) flags |= PF_BAD;
    if (mflags & META_DEGEN) flags |= PF_DEGEN;
    const int nvalid = max(0, min(k - (scol + lane * N), N));
    double s = 0.0;
#pragma unroll
    for (int q = 0; q < H; ++q) {
        if (q < nvalid) s += (double)J[q].x;
        if (q + H < nvalid) s += (double)J[q].y;
    }
    return skew_sum(s, L.E, E0, flags, lane, 31);
}

// ------------------------------------------------------------------------------------
// FP64 strips of wide pairs (scalar form): a CTA of four warps runs 128 N columns, thread t on
// row s - t at step s.  A scheduler's FP64 unit takes about 60 cycles for one warp's FMA, so a
// strip's step lasts as long as its warps' 5 N operations each: four warps side by side, with few
// columns a lane, advance a row chain four times as fast as one warp with all of them.  They
// step together: a barrier a step, and the last lane of a warp hands over through shared memory.
// 24 pairs of 1 to 10 kbp: 10.9 ms with 4 columns a lane (3: 10.9, 2: 11.9), 17.3 ms on strips of
// one warp with 8, 72 to 84 ms on CTAs of the unfactored engine; 1600 cycles a step, of which the
// FP64 unit takes 1200.
// As strip_run_skew<.., WAVE> otherwise, with one virtual lane a lane: checkpoints 128 steps earlier
// than the left strip's, and a boundary row of 32 bytes, two 16-byte accesses that both carry
// the tag (M and half of J; the other half and D-hat).
// ------------------------------------------------------------------------------------
constexpr int kStrip64Warps = 4, kStrip64Lanes = 32 * kStrip64Warps;
struct SkewStage64 {
    double2 pp[2 * kStrip64Lanes], ab[2 * kStrip64Lanes], hg[2 * kStrip64Lanes];  // pm px, a b, h g
    uint32_t meta[2 * kStrip64Lanes];
    uint4 bndA[64], bndB[64];                                     // boundary rows (warp 0)
    double xch[2][kStrip64Warps][4];                              // a warp's last m, j, d by step parity
    int E[kStrip64Warps];
    double S[kStrip64Warps];                                      // the warps' sums
    uint32_t item, flags[kStrip64Warps];
    uint32_t mask[5 * kStrip64Lanes];
};
// x 2^d for d <= 0 on the integer side (the FP64 unit is what the strips wait for); what
// would be subnormal becomes 0 (values are held above 2^-950).
__device__ __forceinline__ double skew_shift(double x, int d) {
    const int hi = __double2hiint(x);
    const bool ok = ((hi >> 20) & 0x7ff) + d > 0;
    return __hiloint2double(ok ? hi + d * (1 << 20) : 0, ok ? __double2loint(x) : 0);
}

template <int N>
__device__ Partial strip_run_skew64(const Rec64J* __restrict__ rec, int l, const uint8_t* __restrict__ hap, int k,
                                    int strip, const PipeRange& rng, const float4* in, float4* out, SkewStage64& st,
                                    uint32_t tag, uint32_t* __restrict__ status) {
    static_assert(N <= 32, "match masks hold 32 columns");
    constexpr int G = kStrip64Lanes, kRows = 2 * G;
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const int scol = strip * G * N;
    uint32_t flags = rng.ok ? 0u : PF_DEGEN, mflags = 0;
    const bool has_left = in != nullptr, has_right = out != nullptr;
    const double mil = __ldg(&rec[l - 1].mi);
    __syncthreads();  // the CTA's previous strip is done with the stage
    {
        uint32_t bm[4] = {0u, 0u, 0u, 0u};
        const int nv = max(0, min(k - (scol + t * N), N));
        for (int c = 0; c < nv; ++c) {
            const int code = base_code(hap[scol + t * N + c]);
            if (code < 0) flags |= PF_BAD;
#pragma unroll
            for (int q = 0; q < 4; ++q)
                if (code == q || code == 4) bm[q] |= 1u << c;
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) st.mask[q * G + t] = bm[q];
        st.mask[4 * G + t] = 0xffffffffu;
    }
    // row l + 1 collects M + I, other rows outside 1 .. l hold
    auto fetch = [&](int row) {
        const int sl = row & (kRows - 1);
        if (row >= 1 && row <= l) {
            const double2* src = reinterpret_cast<const double2*>(rec + (row - 1));
            cp_async16_cg(&st.pp[sl], src);
            cp_async16_cg(&st.ab[sl], src + 1);
            cp_async16_cg(&st.hg[sl], src + 2);
            st.meta[sl] = (uint32_t)__ldg(&rec[row - 1].meta);
        } else {
            st.pp[sl] = st.ab[sl] = make_double2(0.0, 0.0);
            st.hg[sl] = make_double2(row == l + 1 ? mil : 1.0, 0.0);
            st.meta[sl] = 4u;
        }
        cp_async_commit();
    };
    // boundary rows kWaveBlock b .. (warp 0): lane & 15 the row, lane >> 4 the part
    uint4 pv = make_uint4(0u, 0u, 0u, 0u);
    auto load_bnd = [&](int b) {
        const int i = kWaveBlock * b + (lane & (kWaveBlock - 1));
        if (has_left && i >= 1 && i < l) pv = ld_row_relaxed(in + 2 * i + (lane >> 4));
    };
    auto take_bnd = [&](int b) {
        const int i = kWaveBlock * b + (lane & (kWaveBlock - 1));
        const bool mine = has_left && i >= 1, need = mine && i < l;
        long long spins = 0;
        // (after one wait has run out the strip waits no more: its result is an error already)
        while (__any_sync(kFull, need && (pv.w & kWaveTagMask) != tag) && !(flags & PF_TIMEOUT)) {
            if (++spins > kSpinLimit) {
                flags |= PF_TIMEOUT;
                if (lane == 0) atomicOr(status, ST_TIMEOUT);
                break;
            }
            if (spins > kSpinFast) __nanosleep(64);
            if (need && (pv.w & kWaveTagMask) != tag) pv = ld_row_relaxed(in + 2 * i + (lane >> 4));
        }
        if (mine) (lane < kWaveBlock ? st.bndA : st.bndB)[i & 63] = need ? pv : make_uint4(0u, 0u, 0u, 0u);
        __syncwarp();
    };
    if (t < 64) st.bndA[t] = st.bndB[t] = make_uint4(0u, 0u, 0u, 0u);
    __syncthreads();
    fetch(t - (G - 1));
    if (warp == 0) {
        load_bnd(0);
        take_bnd(0);
        load_bnd(1);
    }
    if (t < 64) fetch(1 + t);
    cp_async_wait_0();
    __syncthreads();

    const int E0 = Num<double>::kLog2C - rng.target;
    // the left strip's exponent: that of boundary row 1 up to the first checkpoint, where it
    // may change next
    int Eb = has_left && l > 1 ? (int)st.bndA[1].w >> kWaveTagBits : INT_MIN;
    SkewLane<double> L;
    L.m = L.d = L.g = 0.0;
    L.E = max(E0, Eb);
    int lsh = t == 0 && Eb != INT_MIN ? Eb - L.E : 0;  // exponent of what comes from the left
    double M[N], J[N];
    {
        const double c = skew_init<double>(rng, k, E0, L.E);
#pragma unroll
        for (int q = 0; q < N; ++q) {
            M[q] = 0.0;
            J[q] = c;
        }
        L.j = c;
        // boundary row 0 (Eb >= E0: a strip keeps its first exponent until its last lane started)
        const double j0 = Eb == INT_MIN ? c : scale2(c, L.E - Eb);
        __syncthreads();
        if (t == 0) {
            st.bndA[0] = make_uint4(0u, 0u, (uint32_t)__double2loint(j0), 0u);
            st.bndB[0] = make_uint4((uint32_t)__double2hiint(j0), 0u, 0u, 0u);
        }
        if (lane == 31) {
            st.xch[0][warp][0] = 0.0;
            st.xch[0][warp][1] = c;
            st.xch[0][warp][2] = 0.0;
        }
        __syncthreads();
    }
    const int nl = min(G, (k - scol + N - 1) / N);
    const int steps = l + nl;
    const bool sends = has_right && t == G - 1;
    int ck = rng.R - (int)(((long long)G * strip) % rng.R);  // checkpoint after step ck
    int sl = (1 - t) & (kRows - 1);
    double2 n0 = st.pp[sl], n1 = st.ab[sl], n2 = st.hg[sl];
    uint32_t meta = st.meta[sl];
    for (int s = 1; s <= steps;) {
        const int e = min(min(min(ck, (s + kWaveBlock - 1) & ~(kWaveBlock - 1)), steps), s <= G + 1 ? G + 1 : steps);
        const bool send = sends && s > G + 1;
        // (the steps between events in a loop of their own, as in team_run_skew)
#pragma unroll 1
        for (; s <= e; ++s) {
            if (send) {  // row s - G - 1 at the strip's last column
                const uint32_t w = ((uint32_t)L.E << kWaveTagBits) | tag;
                float4* o = out + 2 * (s - G - 1);
                st_row_relaxed(o, __int_as_float(__double2loint(L.m)), __int_as_float(__double2hiint(L.m)),
                               __int_as_float(__double2loint(L.j)), w);
                st_row_relaxed(o + 1, __int_as_float(__double2hiint(L.j)), __int_as_float(__double2loint(L.d)),
                               __int_as_float(__double2hiint(L.d)), w);
            }
            double um = __shfl_up_sync(kFull, L.m, 1), uj = __shfl_up_sync(kFull, L.j, 1),
                   ud = __shfl_up_sync(kFull, L.d, 1);
            if (lane == 0) {
                if (warp == 0) {
                    const uint4 va = st.bndA[(s - 1) & 63], vb = st.bndB[(s - 1) & 63];
                    um = __hiloint2double((int)va.y, (int)va.x);
                    uj = __hiloint2double((int)vb.x, (int)va.z);
                    ud = __hiloint2double((int)vb.z, (int)vb.y);
                } else {
                    um = st.xch[(s - 1) & 1][warp - 1][0];
                    uj = st.xch[(s - 1) & 1][warp - 1][1];
                    ud = st.xch[(s - 1) & 1][warp - 1][2];
                }
            }
            L.m = skew_shift(um, lsh);
            L.j = skew_shift(uj, lsh);
            L.d = skew_shift(ud, lsh);
            L.pm = n0.x;
            L.px = n0.y;
            L.a = n1.x;
            L.b = n1.y;
            L.h = n2.x;
            L.gp = L.g;
            L.g = n2.y;
            mflags |= meta;
            skew_row<double, N, false>(M, J, L, st.mask[(meta & META_CODE_MASK) * G + t]);
            if (lane == 31) {
                st.xch[s & 1][warp][0] = L.m;
                st.xch[s & 1][warp][1] = L.j;
                st.xch[s & 1][warp][2] = L.d;
            }
            sl = (s + 1 - t) & (kRows - 1);
            n0 = st.pp[sl];
            n1 = st.ab[sl];
            n2 = st.hg[sl];
            meta = st.meta[sl];
            __syncthreads();
        }
        // after step e
        if ((e & 31) == 0) {
            // rows up to e + 32 have landed, rows before e - 126 are done with; every lane takes its
            // next row again (lane 0's is one of those)
            cp_async_wait_0();
            __syncthreads();
            n0 = st.pp[sl];
            n1 = st.ab[sl];
            n2 = st.hg[sl];
            meta = st.meta[sl];
            if (warp == ((e >> 5) & (kStrip64Warps - 1))) fetch(e + 33 + lane);
        }
        if (warp == 0 && (e & (kWaveBlock - 1)) == 0) {
            if (e == 32 && t == 0) st.bndA[0] = st.bndB[0] = make_uint4(0u, 0u, 0u, 0u);
            __syncwarp();
            take_bnd(e / kWaveBlock);
            load_bnd(e / kWaveBlock + 1);
        }
        if (e == ck) {
            ck += rng.R;
            __syncthreads();  // the boundary rows that warp 0 took
            if (has_left && e < l) Eb = (int)st.bndA[e & 63].w >> kWaveTagBits;
            const int r = e - t;
            const bool keep = r < 1 || r > l;
            double x = 0.0;
#pragma unroll
            for (int q = 0; q < N; ++q) x = fmax(x, fmax(fabs(M[q]), fabs(J[q])));
            // as skew_exponent, over the CTA's lanes
            using NT = Num<double>;
            const int ex = NT::expo(x);
            int want = L.E;
            if (!keep) {
                if (ex == INT_MAX) flags |= PF_NONFINITE;
                else if (ex == INT_MIN) want = t > 0 || Eb != INT_MIN ? INT_MIN : L.E;
                else if (ex > rng.hi || ex <= NT::kLo) want = L.E + (ex - rng.target);
            }
            int En = t == 0 ? max(want, Eb) : want;
#pragma unroll
            for (int q = 0; q < 5; ++q) {
                const int up = __shfl_up_sync(kFull, En, 1 << q);
                if (lane >= (1 << q)) En = max(En, up);
            }
            if (lane == 31) st.E[warp] = En;
            __syncthreads();
            int left = t == 0 ? Eb : INT_MIN;  // exponent of the lane to the left
            int before = INT_MIN;
            for (int q = 0; q < warp; ++q) before = max(before, st.E[q]);
            En = max(En, before);
            if (En == INT_MIN) En = L.E;
            if (!keep && En == want && ex <= rng.danger) flags |= PF_DANGER;
            __syncthreads();
            if (lane == 31) st.E[warp] = En;
            __syncthreads();
            const int up = __shfl_up_sync(kFull, En, 1);
            if (lane > 0) left = up;
            else if (warp > 0) left = st.E[warp - 1];
            if (En != L.E) {
                double f, g;
                skew_factors(L.E - En, f, g);
                for (;;) {
#pragma unroll
                    for (int q = 0; q < N; ++q) {
                        M[q] *= f;
                        J[q] *= f;
                    }
                    L.m *= f;
                    L.j *= f;
                    L.d *= f;
                    if (g == 1.0) break;  // one factor, nearly always
                    f = g;
                    g = 1.0;
                }
                L.E = En;
                if (lane == 31) {
                    st.xch[e & 1][warp][0] = L.m;
                    st.xch[e & 1][warp][1] = L.j;
                    st.xch[e & 1][warp][2] = L.d;
                }
            }
            lsh = left == INT_MIN ? 0 : max(left - L.E, -2047);
            if (L.E > kWaveMaxE || L.E < -kWaveMaxE) flags |= PF_DANGER;  // does not fit beside the tag
            __syncthreads();
        }
    }
    if (mflags & META_BAD) flags |= PF_BAD;
    if (mflags & META_DEGEN) flags |= PF_DEGEN;
    const int nvalid = max(0, min(k - (scol + t * N), N));
    double sum = 0.0;
#pragma unroll
    for (int q = 0; q < N; ++q)
        if (q < nvalid) sum += J[q];
    const SegOut o = skew_sum(sum, L.E, E0, flags, lane, 31);
    if (lane == 0) {
        st.S[warp] = o.S;
        st.E[warp] = o.E;
        st.flags[warp] = o.flags;
    }
    cp_async_wait_0();  // nothing may land in the stage after this strip
    __syncthreads();
    // the warps' sums in the scale of the largest
    Partial p;
    p.S = 0.0;
    p.E = st.E[0];
    p.flags = PF_DONE;
    int top = INT_MIN;
    for (int q = 0; q < kStrip64Warps; ++q) {
        p.flags |= st.flags[q];
        const int x = st.S[q] != 0.0 ? st.E[q] + Num<double>::expo(st.S[q]) : INT_MIN;
        if (x > top) {
            top = x;
            p.E = st.E[q];
        }
    }
    for (int q = 0; q < kStrip64Warps; ++q)
        if (st.S[q] != 0.0) p.S += ldexp(st.S[q], st.E[q] - p.E);
    return p;
}

}  // namespace phmm

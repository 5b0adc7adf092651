// Window search by bounds: which windows can hold a period's minimum at all.
// First for uniform weights.
//
// Every window has delta-chi2 = w depth (depth sum s_k^2 - 2 C1), and for any
// depth that is at least -w C1^2 / sum s_k^2.  C1 itself is bounded from
// prefix sums: with the template cut into segments g of len_g points, mean
// t_g and residual norm nu_g = ||s - t_g||,
//     C1 = sum_g (t_g S_g + <s - t_g, r - mean r>)
//        <= sum_g (t_g S_g + nu_g sqrt(E_g - S_g^2 / len_g))
// (Cauchy-Schwarz), where S_g is the exact sum of r over the segment and E_g
// an upper bound of its sum of r^2.  A window whose bound stays below what
// some window of the period is known to reach cannot be the minimum, and its
// D products need not be summed.
//
// window_bounds, by the CTA that has just folded the period (so that its
// prefix sums are still in L2):
//   1. one pass over the prefix sums: a coarse copy of them (every 2^clg-th,
//      in shared memory), the energies of blocks of 2^lb points and their
//      prefix, and from it the largest energy of any stretch of a length;
//   2. first test, one pass over all windows, chunk by chunk: the window sum
//      (short windows) or the bound's main term over a few wide pieces; the
//      largest value of every chunk and the most promising windows are kept;
//   3. those are summed: the lowest delta-chi2 T is the threshold;
//   4. chunks whose largest value can beat T are walked again; windows that
//      also pass the kBoundSegs-segment bound (long ones also the one by
//      kFinePieces pieces) are summed, a warp each, and
//      those within the rounding of the lowest sum are listed.
// k_window_exact:
//   5. the listed windows of all periods of the wave (one or two per period)
//      are summed again, adding the products of a window in the order of the
//      tiled kernel (window_tiles.cuh): the same columns per lane, the same
//      rows, the same tree over the lanes, for the rotated variant also the
//      same first round of every block that covers the window there; so the
//      minimum, its duration, its start and every bit of its delta-chi2 are
//      those of the tiled kernel.
//
// Periods for which nothing is gained (no window has a negative delta-chi2,
// so that signed zeros decide, or only subnormal ones, which are often equal;
// too many windows left, or through the sieve; a value is not finite) are
// listed for the tiled kernel, which then runs on that list; curves most of
// whose periods end there are not tried at every period (kGivenUp).
//
// The window sums of steps 1 to 4 come from 32-bit prefix sums of r rounded to
// a unit with which any sum fits 31 bits: off by half a unit per point (the
// unit is about 2e-4 of the noise of 62,363 points).
//
// Per-point weights (kW): delta-chi2 = depth (depth C2 - 2 C1) with
// C1 = sum w r s_k and C2 = sum w s_k^2 is at least -C1^2 / C2 for any depth.
// C1 is bounded as above with w r in the place of r; its 32-bit prefix sums are
// those of w r rounded to a unit (weighted_prefix: half a unit per point).  C2
// is at least sum_l c_l W_l over nested parts l of the window on which s_k^2
// exceeds the sum of the c up to l; the first test takes for W_l the smallest
// sum of w over any stretch of the length (weight_floors), the segment test the
// window's own, with its exact depth.  (20,011 points with a dy of their own: the
// window stage was 98 ms on the tiled kernel, 126 with the fold; now 66 in all.)
//
// What bounds it (62,363 points, thousand cycles of a period's CTA at 0.55 / 5 /
// 100 days): at short periods waiting between the steps (energies and
// thresholds 34, first pass 24 / 68 / 271, threshold 6, second pass 18 / 41 / 42,
// segments 28 / 33 / 21, sums 20 / 14 / 7; the tiled kernel took 1,100 on average
// over the search), at long ones the instructions of the first pass, about 70
// per 32 windows.  A lane that reads global memory at a cache line
// of its own costs the L1 a cycle, which made the same tests on the prefix
// sums themselves slower by half; only short windows (T0 steps of a few points, so
// that neighbours share lines) read those,
// position-major -- all durations of a stretch of kTileStarts starts before
// the next -- to stay in L1.
#pragma once

namespace gtls {
namespace bounds {

constexpr int kShortSpans = 16;     // spans of blocks whose largest energy is kept: 0 .. 15,
constexpr int kEnergySpans = kShortSpans + 32;   // then 16, 22, 32, 45, ... (up to every block there is)
constexpr int kTileStarts = 8192;   // window starts walked before the next stretch
constexpr int kGroup = 128;         // windows a warp tests at a time (4 per lane)
constexpr int kChunkGroups = 4;     // groups per chunk (at most)
constexpr int kNearStep = kTileStarts / kGroup;   // T0 steps up to this fill a group in one stretch
constexpr int kDenseParts = 16;     // CTAs of the tiled kernel that share a tile, at most
// What is left of a period is cheaper on the tiled kernel when summing its
// windows again would take longer than all of them there.  In ns of an SM, from
// 1520 to 4000 periods of 1,440 to 62,363 points: the tiled kernel by points
// and windows (own weights: 1.7 times that.  Per period 28 us by this, 35 as
// measured, at 1,440 points, 65 and 65 at 3,900, 290 and 240 at 20,011, 810 and
// 630 at 62,363), a listed window by its points, of which kListedRoom halve the
// CTAs that an SM holds (0.6 us for 600 points, 2.5 us for 2,900, 13 to 16 us for
// 9,000), and a window of the sieve its segment test (19 cycles of the CTA): a
// period whose sieve takes longer than its tiles is given up there.  (A fixed
// limit of a window in 512: 27 ms for 1520 periods of 62,363 points 10 % below
// 1, which have hundreds of nearly equal long windows.)
constexpr float kTiledPoint = 0.014f, kTiledWindow = 0.5f, kTiledOwn = 1.7f;   // ns of an SM
constexpr float kPart = 2e5f;       // a tile's share that another CTA is worth staging the tile for
constexpr int kFew = 64;            // windows that are not worth the estimate (at worst 1.6 times the tiled kernel)
constexpr float kSieved = 10.0f;                                              // (two CTAs of an SM: half)
constexpr float kListedPoint = 0.45f, kListedWindow = 300.0f, kListedRoom = 4096.0f;
constexpr int kRowBuf = 168;        // prefix sums at whole T0 steps a warp stages for one group
constexpr int kCutPoints = 60;      // windows of at least this many points are first tested by wide pieces
constexpr int kCoarseSteps = 64;    // ... and from this many coarse steps on from the coarse prefix
constexpr int kExactThreads = 256;
constexpr int kExactRoom = 24576;   // points of a window (and its template) staged by k_window_exact, at most
constexpr int kFloorSpans = 48;     // stretches of blocks whose smallest weight is kept: 1 .. 15, then 16, 19, 22,
                                    // 27 times powers of 2
constexpr unsigned int kNone = 0xffffffffu;
constexpr float kLeast = 1e-30f;    // smallest |delta-chi2| whose rounding is relative, w times the depth among its factors
constexpr int kNoUnit = 1000;       // per-point weights whose sums do not fit the 32-bit prefix

enum Mode : int { kModePairS = 0, kModeCols = 1, kModeRot = 2, kModeWin = 3 };
enum Test : int { kTestSum = 0, kTestCuts = 1, kTestCutsDirect = 2, kTestCoarse = 3 };

// One duration of a period: the plan's part (BoundDur) and the period's.
struct Dur {
    BoundDur b;
    int first;                  // first chunk (near durations: of a stretch)
    float root_c2;              // root of the least C2 of its windows (uniform weights: of sum s_k^2)
    float first_min, cmin;      // thresholds of the first test (32-bit prefix units) and of the segment bound
    float smin;                 // lowest window sum that can have a depth (32-bit prefix units); kW: what the segment
                                // bound can lose of C1
    float blur;                 // what FP32 sums of C1 can be off by
    float cmin_coarse;          // cmin for sums from the coarse prefix
    float c2_slack;             // relative error of FP32 sums of C2 (kW)
};

// Chunks of windows: durations of T0 steps above kNearStep (far ones) are cut
// into groups over the whole curve; the others (near ones) into chunks of at
// most kChunkGroups 2^lg groups inside every stretch of kTileStarts 2^lg
// starts.  Far chunks come first.
struct Chunks {
    int ndur, near_durs;        // durations (ascending); the first near_durs are near
    int far, per_tile;          // far chunks, near chunks per stretch
    int total;
};

// Shared memory for CTAs of T threads (curves of up to 8 T points when
// T < 1024).  At 1024 it stays below 195 KB: the next size the SM offers leaves
// 28 instead of 60 KB of L1, which the fold's gathers feel.
template <int T>
struct Smem {
    static constexpr int kWarps = T / 32;
    static constexpr int kSieve = kWarps * kGroup;   // one group per warp always fits
    static constexpr int kMaxBlocks = T == 1024 ? 9 * T : 2 * T;
    static constexpr int kMaxCoarse = T == 1024 ? 18 * T : 3 * T;
    static constexpr int kMaxChunks = 2 * T;
    static constexpr int kFinal = kMaxChunks;        // windows past the segment bound
    Dur dur[tiles::kMaxDur];
    union {
        unsigned int sieve[kSieve];                  // (duration, window) past the first test
        float fin_v[kFinal];                         // after the walk: lower ends of the sums of fin[]
    };
    float pre[kMaxBlocks + 8];                       // energy prefix
    union {
        float cmax[kMaxChunks];                      // largest first-test value of a chunk
        unsigned int fin[kFinal];                    // after the list of chunks is made: windows past the segment bound
    };
    unsigned char cdur[kMaxChunks];                  // its duration
    unsigned short pass[kMaxChunks];                 // chunks to walk again
    float row_buf[kWarps * kRowBuf];
    float coarse[kMaxCoarse + kMaxCoarse / 32 + 1];  // see at_coarse
    Chunks ck;
    int next, n_pass, sieved, n_fin, dev, big;
    bool full;                                       // a list of the wave is
    int* given_at;                                   // the curve's DevCurve::given_up of this pass,
    int given_up;                                    // and what it was when the period began
    int tested;                                      // windows that went through the sieve
    float wsum[kWarps], energy[kEnergySpans];
    float top[kWarps], c1[kWarps], s[kWarps];
    int top_at[kWarps];
    int wmin[kFloorSpans], wlow;                     // smallest sums of w over whole blocks, smallest w (kW)
};

static_assert(sizeof(Smem<1024>) <= 195 * 1024, "see above");
template <int T>
constexpr int kWarpsOf = T / 32;

__host__ inline size_t smem_bytes(int threads)
{
    return threads == 256 ? sizeof(Smem<256>) : threads == 512 ? sizeof(Smem<512>) : sizeof(Smem<1024>);
}

// log2 of the coarse step for curves of n points and durations of up to d.
__host__ inline int coarse_log2(int threads, int64_t n, int64_t d)
{
    const int64_t room = threads == 1024 ? Smem<1024>::kMaxCoarse : threads == 512 ? Smem<512>::kMaxCoarse
                                                                                   : Smem<256>::kMaxCoarse;
    int lg = 2;
    while (((n + d) >> lg) + 2 > room) ++lg;
    return lg;
}

// Chunks a CTA of T threads has room for.
__host__ inline int max_chunks(int threads) { return 2 * threads; }

// Relative error allowed for a sum of n products in FP32 (twice the bound).
__device__ __forceinline__ float sum_slack(int n) { return 1.2e-7f * (float)(n + 8); }

// Root of an energy (NaN stays NaN; not negative but for rounding: then 0).
__device__ __forceinline__ float root(float x) { return x > 0.0f ? x * rsqrtf(x) : (x <= 0.0f ? 0.0f : x); }

// What delta-chi2 v of a window can differ between two orders of its sums: C1
// off by at most off, the depth by dd (sums of its own: the (C1, S) pairs), C2
// by c2_slack of itself (t2: C2, or sum s_k^2).
__device__ __forceinline__ float sum_error(float w, float depth, float t2, float c1, float v, float off, float dd,
                                           float c2_slack)
{
    return w * (2.0f * (depth + dd) * off + 2.0f * dd * fabsf(fmaf(depth, t2, -c1)) + dd * dd * t2) + 1e-6f * fabsf(v) +
           2e-6f * w * depth * fabsf(c1) + w * depth * depth * t2 * c2_slack;
}

// Place of coarse entry e: one word further every 32, so that lanes whose
// entries are a power of two apart read different banks.
__device__ __forceinline__ int at_coarse(int e) { return e + (e >> 5); }

// Sum of one window by the nc lanes of a group, in the order of the tiled
// kernel; every lane of the group returns the totals (y: window sum of the
// (C1, S) pairs).  Lanes of groups that are not `on` only take part in the
// exchanges.
template <typename Value>
__device__ __forceinline__ float2 window_sum(Value r, const float* __restrict__ t, int d, int st, int lg_nc, int mode,
                                             int rot, bool on, int lane)
{
    const int nc = 1 << lg_nc, c = lane & (nc - 1);
    float x = 0.0f, y = 0.0f;
    if (on) {
        if (mode == kModePairS) {
            for (int rho = c; rho < st; rho += nc) {
#pragma unroll 8
                for (int k = rho; k < d; k += st) {
                    const float v = r(k);
                    x = fmaf(v, t[k], x);
                    y = v + y;
                }
            }
        } else if (mode == kModeWin) {
            for (int rho = c; rho < st; rho += nc) {
#pragma unroll 8
                for (int k = rho; k < d; k += st) x = fmaf(r(k), t[k], x);
            }
        } else {
            const int rounds = (st + 2 * nc - 1) >> (lg_nc + 1);
            int rr = rot;
            for (int i = 0; i < rounds; ++i) {
                const int rho = c + 2 * nc * rr;
                rr = rr + 1 == rounds ? 0 : rr + 1;
                const int end = rho < st ? d : 0;
                const int both = rho + nc < st ? d - nc : 0;   // rows whose second column is inside too
                int k = rho;
#pragma unroll 8
                for (; k < both; k += st) {
                    x = fmaf(r(k), t[k], x);
                    y = fmaf(r(k + nc), t[k + nc], y);
                }
                for (; k < end; k += st) x = fmaf(r(k), t[k], x);
            }
        }
    }
    if (mode != kModePairS) {
        x = x + y;
        y = 0.0f;
    }
    for (int o = 1; o < nc; o <<= 1) {
        x += __shfl_xor_sync(0xffffffffu, x, o);
        y += __shfl_xor_sync(0xffffffffu, y, o);
    }
    return make_float2(x, y);
}

// Durations of period p the kernel searches (kept, not marked kWindowOnly):
// their grid indices into list[] and the chunks of dur[] (by one warp; the
// plan's part of dur[] is copied by the caller).
__device__ __forceinline__ void list_durations(const DevPlan& dp, unsigned int* check, int p, int n, Dur* dur, Chunks& ck,
                                               int lane)
{
    const int lo = dp.jlo[p], hi = dp.jhi[p];
    int count = 0, run_near = 0, run_far = 0, near_durs = 0;
    for (int base = 0; base <= hi - lo; base += 32) {
        const int j = lo + base + lane;
        const int subs = j <= hi ? dp.bound_durs[j].subs : 0;
        const bool nearby = j <= hi && dp.bound_durs[j].st <= kNearStep;
        const int d = j <= hi ? dp.dpts[j] : 0, before = j <= hi && j > lo ? dp.dpts[j - 1] : -1;
        bool kept = j <= hi && d != before && subs > 0;
        const unsigned int mask = __ballot_sync(0xffffffffu, kept);
        const int k = count + __popc(mask & ((1u << lane) - 1u));
        kept = kept && in_range(check, 19, k, tiles::kMaxDur);
        int a = kept && nearby ? subs : 0, b = kept && !nearby ? subs : 0;
        const int a0 = a, b0 = b;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int ya = __shfl_up_sync(0xffffffffu, a, o), yb = __shfl_up_sync(0xffffffffu, b, o);
            if (lane >= o) {
                a += ya;
                b += yb;
            }
        }
        if (kept) {
            dur[k].b.j = j;
            dur[k].first = nearby ? run_near + a - a0 : run_far + b - b0;
        }
        run_near += __shfl_sync(0xffffffffu, a, 31);
        run_far += __shfl_sync(0xffffffffu, b, 31);
        near_durs += __popc(__ballot_sync(0xffffffffu, kept && nearby));
        count += __popc(mask);
    }
    const int tile = kTileStarts << dp.bound_lg;
    if (lane == 0)
        ck = Chunks{min(count, tiles::kMaxDur), near_durs, run_far, run_near,
                    run_far + (n + tile - 1) / tile * run_near};
    __syncwarp();
}

// What the period would take on the tiled kernel (ns of an SM; by a whole warp).
__device__ __forceinline__ float tiled_time(const DevPlan& dp, const Dur* dur, int ndur, bool own, int lane)
{
    float ns = 0.0f;
    for (int k = lane; k < ndur; k += 32) {
        const int j = dur[k].b.j;
        ns += (float)dp.bound_durs[j].m_total * fmaf(kTiledPoint, (float)dp.dpts[j], kTiledWindow);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) ns += __shfl_xor_sync(0xffffffffu, ns, o);
    return own ? kTiledOwn * ns : ns;
}

// Duration k and windows [lo, hi) of chunk c (warp-uniform).
__device__ __forceinline__ void chunk_range(const Chunks& ck, const Dur* dur, int lg, int c, int lane, int& k, int& lo,
                                            int& hi)
{
    const bool far = c < ck.far;
    int rel = c, x = 0;
    if (!far) {
        x = (c - ck.far) / ck.per_tile;
        rel = c - ck.far - x * ck.per_tile;
    }
    const int k0 = far ? ck.near_durs : 0, k1 = far ? ck.ndur : ck.near_durs;
    unsigned int a = __ballot_sync(0xffffffffu, k0 + lane < k1 && dur[min(k0 + lane, k1 - 1)].first <= rel);
    k = k0 + __popc(a) - 1;
    if (k1 - k0 > 32) {
        a = __ballot_sync(0xffffffffu, k0 + 32 + lane < k1 && dur[min(k0 + 32 + lane, k1 - 1)].first <= rel);
        k += __popc(a);
    }
    const int wsub = dur[k].b.wsub;
    lo = (rel - dur[k].first) * wsub;
    int end = dur[k].b.m_total;
    if (!far) {
        const int st = dur[k].b.st, tile = kTileStarts << lg;
        lo += (x * tile + st - 1) / st;
        end = min(end, (int)(((long long)(x + 1) * tile + st - 1) / st));
    }
    hi = min(end, lo + wsub);
}

// First test of windows at .. at + cnt - 1 (cnt <= kGroup) of one duration:
// acc[q] of lane l belongs to window at + 32 q + l.  kTestSum: the window sum;
// else sum_u mean_u S_u over the wide pieces u, from prefix sums relative to
// the first window's start (kTestCuts: staged in the warp's rb) or from the
// coarse prefix (kTestCoarse: every position taken to the nearest multiple of
// 2^clg); in units of the 32-bit prefix.
__device__ __forceinline__ void first_test(const BoundDur& t, const int* __restrict__ pq, const float* coarse, int clg,
                                           int at, int cnt, float* rb, int lane, float (&acc)[4])
{
    const int st = t.st, d = t.d, test = t.test;
    const int cuts4 = t.cuts4;
    const float last = t.cut_last;
    if (test == kTestCoarse) {
        int s[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) s[q] = (at + min(q * 32 + lane, cnt - 1)) * st + (1 << clg >> 1);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            acc[q] = last * coarse[at_coarse((s[q] + d) >> clg)];
            acc[q] = fmaf(t.coef0, coarse[at_coarse(s[q] >> clg)], acc[q]);
        }
        for (int u = 0; u < cuts4; u += 4) {
            const float4 w = *reinterpret_cast<const float4*>(t.coef + u);
            const int4 r = *reinterpret_cast<const int4*>(t.row + u);
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                if (q * 32 >= cnt) break;
                acc[q] = fmaf(w.x, coarse[at_coarse((s[q] + r.x) >> clg)], acc[q]);
                acc[q] = fmaf(w.y, coarse[at_coarse((s[q] + r.y) >> clg)], acc[q]);
                acc[q] = fmaf(w.z, coarse[at_coarse((s[q] + r.z) >> clg)], acc[q]);
                acc[q] = fmaf(w.w, coarse[at_coarse((s[q] + r.w) >> clg)], acc[q]);
            }
        }
        return;
    }
    const int* const a = pq + at * st;
    int i[4], v[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) i[q] = min(q * 32 + lane, cnt - 1) * st;
#pragma unroll
    for (int q = 0; q < 4; ++q) v[q] = q * 32 < cnt ? a[i[q] + d] : 0;
    if (test == kTestSum) {
#pragma unroll
        for (int q = 0; q < 4; ++q) acc[q] = q * 32 < cnt ? (float)(v[q] - a[i[q]]) : 0.0f;
        return;
    }
    const int base = a[0];
    if (test == kTestCuts) {
        const int nr = cnt + t.row_max;
        __syncwarp();   // the previous group's reads are done
        for (int r0 = lane; r0 < nr; r0 += 160) {   // (a group and the 20 or so rows of its last window)
            int p[5];
#pragma unroll
            for (int u = 0; u < 5; ++u) p[u] = a[min(r0 + u * 32, nr - 1) * st];
#pragma unroll
            for (int u = 0; u < 5; ++u)
                if (r0 + u * 32 < nr) rb[r0 + u * 32] = (float)(p[u] - base);
        }
        __syncwarp();
#pragma unroll
        for (int q = 0; q < 4; ++q) acc[q] = last * (float)(v[q] - base);
        const float* const b = rb + lane;
#pragma unroll
        for (int q = 0; q < 4; ++q) acc[q] = fmaf(t.coef0, b[q * 32], acc[q]);   // (past cnt: not used)
        for (int u = 0; u < cuts4; u += 4) {
            const float4 w = *reinterpret_cast<const float4*>(t.coef + u);
            const int4 r = *reinterpret_cast<const int4*>(t.row + u);
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                acc[q] = fmaf(w.x, b[r.x + q * 32], acc[q]);
                acc[q] = fmaf(w.y, b[r.y + q * 32], acc[q]);
                acc[q] = fmaf(w.z, b[r.z + q * 32], acc[q]);
                acc[q] = fmaf(w.w, b[r.w + q * 32], acc[q]);
            }
        }
    } else {
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            acc[q] = last * (float)(v[q] - base);
            acc[q] = fmaf(t.coef0, (float)(a[i[q]] - base), acc[q]);
        }
        for (int u = 0; u < cuts4; ++u) {
            const float w = t.coef[u];
            const int* const b = a + t.row[u];
#pragma unroll
            for (int q = 0; q < 4; ++q) acc[q] = fmaf(w, (float)(b[i[q]] - base), acc[q]);
        }
    }
}

// One pass over the 32-bit prefix sums P[0 .. total]: block energies into
// pre[] (from the differences of P, each off by at most a unit), the coarse
// prefix, the largest |entry| of it, and the furthest any P is from the entry
// its position is taken to.  A thread takes runs of 2^max(lb, clg) positions.
template <int T>
__device__ __forceinline__ void scan_prefix(Smem<T>& S, const int* __restrict__ pq, int total, int lb, int clg,
                                            float unit)
{
    const int lrun = max(lb, clg), run = 1 << lrun, bmask = (1 << lb) - 1, cstep = 1 << clg, half = cstep >> 1;
    int dev = 0, big = 0;
    if (lb == 3 && clg == 2) {
        // the usual sizes: eight positions and the next one, which the next lane holds
        const int lane = threadIdx.x & 31;
#pragma unroll 3
        for (int r0 = threadIdx.x * 8; r0 - lane * 8 + 256 <= total; r0 += T * 8) {   // whole warps
            const int4 a = *reinterpret_cast<const int4*>(pq + r0), b = *reinterpret_cast<const int4*>(pq + r0 + 4);
            int next = __shfl_down_sync(0xffffffffu, a.x, 1);
            if (lane == 31) next = pq[r0 + 8];
            const int v[9] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w, next};
            float e = 0.0f;
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const float x = (float)(abs(v[u + 1] - v[u]) + 1);
                e = fmaf(x, x, e);
            }
            S.pre[r0 >> 3] = e * unit * unit;
            S.coarse[at_coarse(r0 >> 2)] = (float)v[0];
            S.coarse[at_coarse((r0 >> 2) + 1)] = (float)v[4];
            big = max(big, max(abs(v[0]), abs(v[4])));
            dev = max(dev, max(max(abs(v[1] - v[0]), abs(v[2] - v[4])), max(abs(v[3] - v[4]), abs(v[5] - v[4]))));
            dev = max(dev, max(abs(v[6] - v[8]), abs(v[7] - v[8])));
        }
    }
    // (the rest: what is not a whole warp's span above, or every position)
    const int done = lb == 3 && clg == 2 ? total / 256 * 256 : 0;
    for (int r0 = done + (threadIdx.x << lrun); r0 <= total; r0 += T << lrun) {
        int cur = 0, lo = 0, hi = 0, prev = 0;
        float e = 0.0f;
        const int end = min(run, total - r0);   // last position of the run's span (inclusive)
        for (int g0 = 0; g0 <= end; g0 += 4) {
            // (the vector stays inside the padded array; values past `end` are not used)
            const int4 v4 = *reinterpret_cast<const int4*>(pq + r0 + g0);
            const int v[4] = {v4.x, v4.y, v4.z, v4.w};
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int g = g0 + u;
                if (g > end) break;
                if (g > 0) {
                    const float x = (float)(abs(v[u] - prev) + 1);
                    e = fmaf(x, x, e);
                    if ((g & bmask) == 0) {   // the block before g ends here
                        S.pre[(r0 + g - 1) >> lb] = e * unit * unit;
                        e = 0.0f;
                    }
                }
                prev = v[u];
                const int in = g & (cstep - 1);
                if (in == 0) {
                    if (g > 0) dev = max(dev, max(abs(hi - v[u]), abs(lo - v[u])));
                    cur = lo = hi = v[u];
                    if (g < run) {
                        S.coarse[at_coarse((r0 + g) >> clg)] = (float)v[u];
                        big = max(big, abs(v[u]));
                    }
                } else if (in < half) {
                    dev = max(dev, abs(v[u] - cur));
                } else {
                    // taken to the next entry: kept until that is known
                    lo = in == half ? v[u] : min(lo, v[u]);
                    hi = in == half ? v[u] : max(hi, v[u]);
                }
            }
        }
        if (end < run) {   // the curve ends inside this run
            if ((end & bmask) != 0) S.pre[(r0 + end) >> lb] = e * unit * unit;
            if ((end & (cstep - 1)) >= half) {   // and in the upper half of a step: its end is the entry
                S.coarse[at_coarse(((r0 + end) >> clg) + 1)] = (float)prev;
                big = max(big, abs(prev));
                dev = max(dev, max(abs(hi - prev), abs(lo - prev)));
            }
        }
    }
    dev = __reduce_max_sync(0xffffffffu, dev);
    big = __reduce_max_sync(0xffffffffu, big);
    if ((threadIdx.x & 31) == 0) {
        atomicMax(&S.dev, dev);
        atomicMax(&S.big, big);
    }
}

// Prefix sums of w r and of w over the folded, padded curve in 32 bits: every
// value rounded to a unit (a = w r / unit, b = w / unit), positions 0 .. total;
// S.wlow becomes the smallest b (set to INT_MAX before).
template <int T>
__device__ __forceinline__ void weighted_prefix(Smem<T>& S, const float* __restrict__ wrs, const float* __restrict__ ws,
                                                int* __restrict__ pq, int* __restrict__ pw, int total, float per_a,
                                                float per_b)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int carry_a = 0, carry_b = 0, low = INT_MAX;
    bool odd = false;
    for (int r0 = threadIdx.x * 8; r0 - (int)threadIdx.x * 8 <= total; r0 += T * 8, odd = !odd) {
        int a[8], b[8], sa = 0, sb = 0;
        float va[8], vb[8];
#pragma unroll
        for (int h = 0; h < 8; h += 4) {   // (zeros follow the padded curve)
            const float4 x = r0 <= total ? *reinterpret_cast<const float4*>(wrs + r0 + h) : make_float4(0, 0, 0, 0);
            const float4 y = r0 <= total ? *reinterpret_cast<const float4*>(ws + r0 + h) : make_float4(0, 0, 0, 0);
            va[h] = x.x, va[h + 1] = x.y, va[h + 2] = x.z, va[h + 3] = x.w;
            vb[h] = y.x, vb[h + 1] = y.y, vb[h + 2] = y.z, vb[h + 3] = y.w;
        }
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const int qa = __float2int_rn(va[u] * per_a), qb = __float2int_rn(vb[u] * per_b);
            if (r0 + u < total) low = min(low, qb);
            a[u] = sa;
            b[u] = sb;
            sa += qa;
            sb += qb;
        }
        int xa = sa, xb = sb;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int ya = __shfl_up_sync(0xffffffffu, xa, o), yb = __shfl_up_sync(0xffffffffu, xb, o);
            if (lane >= o) {
                xa += ya;
                xb += yb;
            }
        }
        // (two sets of warp sums in turn: one barrier per round)
        int* const wa = reinterpret_cast<int*>(odd ? S.c1 : S.wsum);
        int* const wb = reinterpret_cast<int*>(odd ? S.s : S.top);
        if (lane == 31) {
            wa[warp] = xa;
            wb[warp] = xb;
        }
        __syncthreads();
        const int ta = lane < kWarpsOf<T> ? wa[lane] : 0, tb = lane < kWarpsOf<T> ? wb[lane] : 0;
        const int ea = carry_a + (int)__reduce_add_sync(0xffffffffu, lane < warp ? ta : 0) + xa - sa;
        const int eb = carry_b + (int)__reduce_add_sync(0xffffffffu, lane < warp ? tb : 0) + xb - sb;
        carry_a += (int)__reduce_add_sync(0xffffffffu, ta);
        carry_b += (int)__reduce_add_sync(0xffffffffu, tb);
        if (r0 <= total) {
#pragma unroll
            for (int h = 0; h < 8; h += 4) {
                *reinterpret_cast<int4*>(pq + r0 + h) =
                    make_int4(ea + a[h], ea + a[h + 1], ea + a[h + 2], ea + a[h + 3]);
                *reinterpret_cast<int4*>(pw + r0 + h) =
                    make_int4(eb + b[h], eb + b[h + 1], eb + b[h + 2], eb + b[h + 3]);
            }
        }
    }
    low = __reduce_min_sync(0xffffffffu, low);
    if (lane == 0) atomicMin(&S.wlow, low);
}

// Blocks of floor span q.
__device__ __forceinline__ int floor_span(int q)
{
    const int f = (q - 15) & 3;
    return q < 15 ? q + 1 : (f == 0 ? 16 : f == 1 ? 19 : f == 2 ? 22 : 27) << ((q - 15) >> 2);
}

// Smallest sums of w over stretches of whole blocks of 2^lb points, by the
// prefix of the blocks in S.pre (as integers).  Starts are taken 1/16 of the
// stretch together: what all of them share.
template <int T>
__device__ __forceinline__ void weight_floors(Smem<T>& S, const int* __restrict__ pw, int total, int lb)
{
    int* const pre = reinterpret_cast<int*>(S.pre);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nb = total >> lb;
    for (int b = threadIdx.x; b <= nb; b += T) pre[b] = pw[b << lb];
    __syncthreads();
    for (int q = warp; q < kFloorSpans; q += T / 32) {
        const int m = floor_span(q), step = max(1, m >> 4);
        int low = m <= nb ? INT_MAX : 0;
#pragma unroll 4
        for (int i = lane * step; i + m <= nb; i += 32 * step) low = min(low, pre[i + m] - pre[i + step - 1]);
        low = __reduce_min_sync(0xffffffffu, low);
        if (lane == 0) S.wmin[q] = low;
    }
    __syncthreads();   // (pre is written again)
}

// At most the sum of w over any len points, in units of its prefix.
template <int T>
__device__ __forceinline__ float weight_floor(const Smem<T>& S, int len, int lb)
{
    float sum = 0.0f;
    for (int m = (len - (1 << lb) + 1) >> lb; m > 0;) {
        int q = m - 1;
        if (m > 15) {
            const int o = 27 - __clz(m), x = m >> o;   // 16 .. 31
            q = min(kFloorSpans - 1, 15 + 4 * o + (x >= 27 ? 3 : x >= 22 ? 2 : x >= 19 ? 1 : 0));
        }
        sum += (float)S.wmin[q] * (1.0f - 1e-6f);
        m -= floor_span(q);
    }
    return fmaxf(sum, (float)len * (float)S.wlow * (1.0f - 1e-6f)) - 0.5f * (float)len;
}

// Steps 1 to 4 for one period, by a CTA of T threads (kW: per-point weights):
// true when its windows that may hold the minimum are listed, false when the
// tiled kernel has to sum all of them.
template <int T, bool kW>
__device__ __forceinline__ bool rule_out(Smem<T>& S, const DevSet& ds, const DevChunk& dk, int slot, int lc, int p, int buf)
{
    using M = Smem<T>;
    constexpr int kWarps = T / 32;
    Dur* const dur = S.dur;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const DevPlan& dp = ds.plans[lc];
    const float w_uni = kW ? 1.0f : (float)ds.curves[lc].scal[2];
    const int n = (int)dp.n;
    const int total = n + dp.dmax_p[p];
    float* const rb = S.row_buf + warp * kRowBuf;
    const float* const rs = kW ? dk.wrs + (int64_t)slot * dk.pad_stride : nullptr;   // what C1 sums
    const float* const ws = kW ? dk.ws + (int64_t)slot * dk.pad_stride : nullptr;
    const int* const pq = dk.pq + (int64_t)slot * dk.pad_stride;
    // (the fold is through with its keys)
    int* const pw = reinterpret_cast<int*>(dk.keys + (int64_t)slot * dk.key_stride);
    const long long* const pf = dk.pf + (int64_t)slot * dk.pad_stride;
    const int shift = (int)ds.curves[lc].scal[3];
    const int shift_w = kW ? (int)ds.curves[lc].scal[4] : 0;
    const bool in_range_32 = kW ? shift < kNoUnit && shift_w < kNoUnit : shift < 64;
    // unit of the 32-bit prefix.  Per-point weights: C1 and energies are kept
    // in units until the windows are summed
    const float unit = kW ? 1.0f : prefix_unit(shift);
    const float unit_a = kW ? ldexpf(1.0f, in_range_32 ? shift : 0) : 1.0f;
    const float unit_w = kW ? ldexpf(1.0f, in_range_32 ? shift_w : 0) : 1.0f;
    const int lg = dp.bound_lg;
    // a sum of len points by the 32-bit prefix is off by at most this: half a
    // unit per point, and for uniform weights the rounding of r to FP32 (units
    // add up to at most 2^30 in size) and to the fixed point of exact sums
    auto sum_blur = [&](int len) {
        return (0.5f * (float)len + (kW ? 1.0f : 64.0f)) * unit + (kW ? 0.0f : 5e-13f * (float)len);
    };
    // depth of a window: exact (kW), or from the 32-bit prefix
    auto depth_of = [&](int s, int d, float inv) {
        if (kW) return fmaxf(0.0f, tiles::fixed_to_float(pf[s + d] - pf[s]) * (inv * (1.0f / 1099511627776.0f)));
        return fmaxf(0.0f, (float)(pq[s + d] - pq[s]) * unit * inv);
    };

    // (in registers only at 256 threads, whose CTAs wait for shared memory more
    // than the spills cost: 1440 points 0.597 against 0.615 ms; 16 curves of 4,000
    // points, at 512 threads, 250.8 against 247.3 ms)
    std::conditional_t<T == 256, const Chunks, const Chunks&> ck = S.ck;
    const int ndur = ck.ndur;
    {
        // the plan's part of the durations
        constexpr int kWords = sizeof(BoundDur) / 4;
        for (int e = threadIdx.x; e < ndur * kWords; e += T) {
            const int k = e / kWords, u = e - k * kWords;
            if (u > 0)   // (word 0: j, set already)
                reinterpret_cast<int*>(&dur[k].b)[u] =
                    __ldg(reinterpret_cast<const int*>(dp.bound_durs + dur[k].b.j) + u);
        }
    }
    // 1. energies: blocks of 2^lb points, their exclusive prefix
    int lb = 3, clg = 2;
    while (((total + (1 << lb) - 1) >> lb) > M::kMaxBlocks) ++lb;
    while ((total >> clg) + 2 > M::kMaxCoarse) ++clg;
    const int bsize = 1 << lb, nb = (total + bsize - 1) >> lb;
    int lbw = 2;   // blocks of the weights
    if (kW) {
        while ((total >> lbw) > M::kMaxBlocks) ++lbw;
        weighted_prefix<T>(S, rs, ws, const_cast<int*>(pq), pw, total, 1.0f / unit_a, 1.0f / unit_w);
        __syncthreads();
        weight_floors<T>(S, pw, total, lbw);
    }
    scan_prefix<T>(S, pq, total, lb, clg, unit);
    __syncthreads();
    {
        constexpr int kPer = M::kMaxBlocks / T;
        const int b0 = threadIdx.x * kPer;
        float v[kPer], run = 0.0f;
#pragma unroll
        for (int u = 0; u < kPer; ++u) {
            v[u] = run;
            run += b0 + u < nb ? S.pre[b0 + u] : 0.0f;
        }
        float x = run;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const float y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        if (lane == 31) S.wsum[warp] = x;
        __syncthreads();
        float base = lane < warp ? S.wsum[lane] : 0.0f;   // sums of the lower warps
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) base += __shfl_xor_sync(0xffffffffu, base, o);
        const float excl = __shfl_up_sync(0xffffffffu, x, 1);   // sums of the lower lanes
        base += lane > 0 ? excl : 0.0f;
#pragma unroll
        for (int u = 0; u < kPer; ++u)
            if (b0 + u <= nb) S.pre[b0 + u] = base + v[u];
        if (b0 + kPer == nb && nb == M::kMaxBlocks) S.pre[nb] = base + run;
    }
    __syncthreads();
    const float e_all = S.pre[nb];
    // rounding of block sums and prefix: an energy E read from the prefix is
    // at most E (1 + e_rel) + e_abs
    const float e_rel = sum_slack(bsize), e_abs = sum_slack(bsize + 64) * e_all;

    // largest energy of any stretch that reaches `span` blocks past its first:
    // spans 0 .. kShortSpans - 1, and from there a row of spans sqrt(2) apart
    // (starts in blocks [i, i + step) taken together)
    {
        float best[kShortSpans];
#pragma unroll
        for (int q = 0; q < kShortSpans; ++q) best[q] = 0.0f;
        for (int i = threadIdx.x; i < nb; i += T) {
            const float from = S.pre[i];
#pragma unroll
            for (int q = 0; q < kShortSpans; ++q) best[q] = fmaxf(best[q], S.pre[min(nb, i + 1 + q)] - from);
        }
#pragma unroll
        for (int q = 0; q < kShortSpans; ++q) {
            // (not negative: as integers they are ordered the same)
            const int top = __reduce_max_sync(0xffffffffu, __float_as_int(best[q]));
            if (lane == 0) atomicMax(reinterpret_cast<int*>(S.energy + q), top);
        }
        for (int q = warp; q < kEnergySpans - kShortSpans; q += kWarps) {
            const int span = (q & 1 ? (kShortSpans * 181) >> 7 : kShortSpans) << (q >> 1), step = max(1, span >> 3);
            float top = span < nb ? 0.0f : e_all;
            if (span < nb) {
#pragma unroll 4
                for (int i = lane * step; i < nb; i += 32 * step)
                    top = fmaxf(top, S.pre[min(nb, i + step + span)] - S.pre[i]);
            }
            const int t = __reduce_max_sync(0xffffffffu, __float_as_int(top));
            if (lane == 0) S.energy[kShortSpans + q] = __int_as_float(t);
        }
    }
    // upper bound of sum r^2 over any len points
    auto energy_of = [&](int len) {
        const int span = (len + bsize - 2) >> lb;
        int q = span;
        if (span >= kShortSpans) {   // first of the long spans that is at least this one
            const int o = 31 - __clz(max(span - 1, kShortSpans) / kShortSpans);   // kShortSpans << o <= max(span - 1, ..)
            q = kShortSpans + 2 * o;
            while (((q - kShortSpans) & 1 ? (kShortSpans * 181) >> 7 : kShortSpans) << ((q - kShortSpans) >> 1) < span) ++q;
        }
        return fmaf(S.energy[min(q, kEnergySpans - 1)], 1.0f + e_rel, e_abs);
    };

    __syncthreads();

    // what every duration's thresholds need besides the lowest known sum (eight
    // lanes each, which share the pieces; kept in the fields of the thresholds).  A
    // window whose C1 stays below cmin is above that sum: `lost` is what FP32
    // summation, the 32-bit prefix and segment sums can lose of C1 (at most
    // sum_slack(products in a row) ||r|| ||s||, and the units of the sums)
    auto chain_of = [&](const Dur& t) {   // rows a lane of the final sums adds to one window
        const int lg = kW ? __ffs(dp.cfg_nc_w[t.b.j]) - 1 : t.b.lg_nc, nc = 1 << lg;
        return ((t.b.st + nc - 1) >> lg) * ((t.b.d + t.b.st - 1) / t.b.st) + 6;
    };
    for (int k0 = warp * 4; k0 < ndur; k0 += kWarps * 4) {
        const int k = k0 + (lane >> 3);
        Dur& t = dur[min(k, ndur - 1)];
        const BoundTab& bt = dp.bounds[t.b.j];
        const int d = t.b.d, st = t.b.st, chain = chain_of(t);
        float lose = 0.0f, c2 = 0.0f;
#pragma unroll
        for (int u = 0; u < kBoundCuts; u += 8) {
            const int at = u + (lane & 7);
            if (at < bt.cuts) lose = fmaf(bt.cut_nu[at], sqrtf(energy_of(bt.cut_len[at])), lose);
        }
        static_assert(kBoundLevels <= 8, "a level per lane");
        if (kW && (lane & 7) < kBoundLevels)
            c2 = bt.lev_up[lane & 7] * fmaxf(0.0f, weight_floor(S, bt.lev_len[lane & 7], lbw));
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) {
            lose += __shfl_xor_sync(0xffffffffu, lose, o);
            if (kW) c2 += __shfl_xor_sync(0xffffffffu, c2, o);
        }
        if ((lane & 7) != 0 || k >= ndur) continue;
        const float emax = energy_of(d), norm = sqrtf((float)d * emax), here = sum_slack(d / 32 + 8);
        const float lost = (sum_slack(chain) + 8e-6f) * norm + sum_blur(d);
        const float off = (lost + (float)(kBoundSegs + 1) * unit) * bt.t_max;
        t.c2_slack = kW ? sum_slack(chain) + here + 1e-6f : 1e-6f;
        // (kW: the smallest C2 of any window, less what FP32 sums of it can lose)
        t.root_c2 = kW ? sqrtf(c2 * unit_w * (1.0f - 1e-5f - t.c2_slack)) / unit_a : bt.root_t2;
        t.cmin = off;
        // (uniform weights: the sums of steps 3 and 4 are those of the rounded r)
        const float t_max = fmaxf(bt.t_max, 1.0f);
        t.blur = kW ? (sum_slack(chain) + here) * norm * t_max * unit_a
                    : (sum_slack(chain) * norm + sum_blur(d)) * t_max + (here + 3e-7f) * (norm + sum_blur(d)) * bt.change;
        if (t.b.test == kTestSum) {
            lose = bt.nu_all * sqrtf(emax);
        } else if (t.b.test == kTestCoarse) {
            // every position is off by at most S.dev in its prefix sum; the
            // coarse entries are rounded to FP32
            lose = fmaf(bt.cut_jumps * unit, (float)S.dev + 1.2e-7f * (float)(bt.cuts + 4) * (float)S.big, lose);
            t.cmin_coarse = bt.seg_jumps * unit * ((float)S.dev + 1.2e-7f * (float)(2 * kBoundSegs + 4) * (float)S.big);
        } else {
            // rounding of the prefix sums, which reach over the whole group
            const float over = (float)(kGroup * st) / (float)d + 2.0f;
            lose += 1.2e-7f * (float)(bt.cuts + 4) * 2.0f * over * norm * bt.t_max;
        }
        t.first_min = lose;
        // depth is zero without a positive sum (exact, or FP32 for the pairs)
        t.smin = kW ? off : ((t.b.mode == kModePairS ? -lost : 0.0f) - sum_blur(d)) / unit;
        if (kW) t.b.lg_nc = __ffs(dp.cfg_nc_w[t.b.j]) - 1;
    }

    // 2. largest first-test value of every chunk; each lane's best window
    float top = -INFINITY;   // estimate of C1 / sqrt(sum s_k^2)
    int top_at = 0;          // its duration and window
    for (;;) {
        int c = 0;
        if (lane == 0) c = atomicAdd(&S.next, 1);
        c = __shfl_sync(0xffffffffu, c, 0);
        if (c >= ck.total) break;
        int k, lo, hi;
        chunk_range(ck, dur, lg, c, lane, k, lo, hi);
        const float lam = dur[k].b.lam;
        float f = -INFINITY;
        if (dur[k].b.test == kTestSum) {
            // the largest sum of the chunk, in integers
            const int st = dur[k].b.st, d = dur[k].b.d;
            const int* a = pq + (lo + lane) * st;
            int best = INT_MIN, at = 0;
#pragma unroll 4
            for (int i = lo + lane; i < hi; i += 32, a += 32 * st) {
                const int v = a[d] - a[0];
                if (v > best) {
                    best = v;
                    at = i;
                }
            }
            if (best > INT_MIN) f = (float)best;
            if (f * lam > top) {
                top = f * lam;
                top_at = (k << 24) | at;
            }
        }
        for (int at = dur[k].b.test == kTestSum ? hi : lo; at < hi; at += kGroup) {
            float acc[4];
            const int cnt = min(kGroup, hi - at);
            first_test(dur[k].b, pq, S.coarse, clg, at, cnt, rb, lane, acc);
            float g = -INFINITY;
#pragma unroll
            for (int q = 0; q < 4; ++q) g = fmaxf(g, q * 32 + lane < cnt ? acc[q] : -INFINITY);
            f = fmaxf(f, g);
            if (g * lam > top) {
                top = g * lam;
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    if (q * 32 + lane < cnt && acc[q] == g) top_at = (k << 24) | (at + q * 32 + lane);
            }
        }
        f = float_from_order_key(__reduce_max_sync(0xffffffffu, float_order_key(f)));
        if (lane == 0) {
            S.cmax[c] = f;
            S.cdur[c] = (unsigned char)k;
        }
    }

    // 3. threshold: the two most promising windows of the warps, half of the
    // warps to a window (any order: the result only has to be near)
    {
        const unsigned int key = __reduce_max_sync(0xffffffffu, float_order_key(top));
        const int who = __ffs(__ballot_sync(0xffffffffu, float_order_key(top) == key)) - 1;
        if (lane == who) {
            S.top[warp] = top;
            S.top_at[warp] = top_at;
        }
    }
    __syncthreads();
    constexpr int kTeam = kWarps / 2, kTeamThreads = kTeam * 32;
    int cand[2];
    {
        unsigned int key = lane < kWarps ? float_order_key(S.top[lane]) : 0u;
        const int at = lane < kWarps ? S.top_at[lane] : 0;
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const unsigned int most = __reduce_max_sync(0xffffffffu, key);
            const int who = __ffs(__ballot_sync(0xffffffffu, key == most)) - 1;
            const int from = __shfl_sync(0xffffffffu, at, who);
            cand[q] = most > float_order_key(-INFINITY) ? from : -1;
            if (lane == who) key = 0u;
        }
    }
    {
        const int mine = warp < kTeam ? cand[0] : cand[1];
        float c1 = 0.0f, c2 = 0.0f;
        if (mine >= 0) {
            const BoundDur& t = dur[mine >> 24].b;
            const int at = (mine & 0xffffff) * t.st;
            if constexpr (kW) {
                const float* const s = dp.tmpl + dp.tmpl_off[t.j];
#pragma unroll 8
                for (int i = threadIdx.x % kTeamThreads; i < t.d; i += kTeamThreads) {
                    const float sv = __ldg(s + i);
                    c1 = fmaf(rs[at + i], sv, c1);
                    c2 = fmaf(ws[at + i], sv * sv, c2);
                }
            } else {
                // sum r s_k = sum (P_k - P_0) (s_{k-1} - s_k): r itself is not there
                const float* const s = dp.tmpl_drop + dp.tmpl_off[t.j];
                const int base = pq[at];
#pragma unroll 8
                for (int i = threadIdx.x % kTeamThreads; i <= t.d; i += kTeamThreads)
                    c1 = fmaf((float)(pq[at + i] - base), __ldg(s + i), c1);
            }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            c1 += __shfl_xor_sync(0xffffffffu, c1, o);
            if (kW) c2 += __shfl_xor_sync(0xffffffffu, c2, o);
        }
        if (lane == 0) {
            S.c1[warp] = c1;
            S.s[warp] = c2;
        }
        if (threadIdx.x == 0) S.next = 0;
    }
    __syncthreads();
    // what the depth of depth_of can be off by (kW: nothing, it is exact)
    auto depth_blur = [&](const Dur& t, float off, float inv) {
        return kW ? 0.0f : (t.b.mode == kModePairS ? off : 0.0f) * inv + sum_blur(t.b.d) * inv;
    };
    float thr;   // (every warp for itself)
    {
        float c1 = lane < kWarps ? S.c1[lane] : 0.0f, c2 = lane < kWarps ? S.s[lane] : 0.0f, v = INFINITY;
#pragma unroll
        for (int o = kTeam / 2; o > 0; o >>= 1) {
            c1 += __shfl_xor_sync(0xffffffffu, c1, o);
            if (kW) c2 += __shfl_xor_sync(0xffffffffu, c2, o);
        }
        const int mine = lane < kTeam ? cand[0] : cand[1];
        if (lane < kWarps && mine >= 0) {
            const Dur& t = dur[mine >> 24];
            const float inv = dp.inv_sum_t[t.b.j], t2 = kW ? c2 : dp.sum_t2[t.b.j];
            if (!kW) c1 *= unit;
            const float depth = depth_of((mine & 0xffffff) * t.b.st, t.b.d, inv);
            v = w_uni * depth * fmaf(depth, t2, -2.0f * c1);
            v += sum_error(w_uni, depth, t2, c1, v, t.blur, depth_blur(t, t.blur, inv), t.c2_slack);
        }
        const float v0 = __shfl_sync(0xffffffffu, v, 0), v1 = __shfl_sync(0xffffffffu, v, kTeam);
        thr = isnan(v0) || isnan(v1) ? NAN : fminf(v0, v1);
    }
    // no negative delta-chi2, one so small that it or its factors are subnormal
    // in FP32 (the slacks below are relative), or values out of range: the
    // tiled kernel decides
    const bool sane = thr < -kLeast && thr > -INFINITY && e_all < INFINITY && w_uni < INFINITY && in_range_32;
    if (sane) {
        // 1e-4 of slack covers the rounding of delta-chi2
        const float reach = sqrtf(-thr / w_uni) * (1.0f - 1e-4f);   // (times the root of C2 or sum s_k^2)
        for (int k = threadIdx.x; k < ndur; k += T) {
            Dur& t = dur[k];
            t.cmin = reach * t.root_c2 - t.cmin;
            t.cmin_coarse = t.cmin - t.cmin_coarse;
            const float c0 = t.b.test == kTestSum
                                 ? fmaxf((t.cmin - t.first_min) / t.b.mean_all, kW ? -INFINITY : t.smin * unit)
                                 : t.cmin - t.first_min;
            t.first_min = (c0 - 1e-5f * fabsf(c0)) / unit;
        }
    }
    __syncthreads();
    // the chunks to walk again
    if (sane) {
        for (int c = threadIdx.x; c < ck.total; c += T) {
            if (!(S.cmax[c] < dur[S.cdur[c]].first_min)) S.pass[atomicAdd(&S.n_pass, 1)] = (unsigned short)c;
        }
    }
    __syncthreads();

    // 4. windows that may hold the minimum: those of the listed chunks by the
    // first test into the sieve, those by segments into the final list; a full
    // sieve is emptied before the walk goes on
    int c = -1, k = 0, at = 0, hi = 0;
    while (sane) {
        for (;;) {
            if (c < 0) {
                if (lane == 0) c = atomicAdd(&S.next, 1);
                c = __shfl_sync(0xffffffffu, c, 0);
                if (c >= S.n_pass) {
                    c = -1;
                    break;
                }
                chunk_range(ck, dur, lg, S.pass[c], lane, k, at, hi);
            }
            const float first_min = dur[k].first_min;
            bool full = false;
            for (; at < hi; at += kGroup) {
                const int cnt = min(kGroup, hi - at);
                float acc[4];
                first_test(dur[k].b, pq, S.coarse, clg, at, cnt, rb, lane, acc);
                unsigned int vote[4];
                int sum = 0;
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    vote[q] = __ballot_sync(0xffffffffu, q * 32 + lane < cnt && !(acc[q] < first_min));
                    sum += __popc(vote[q]);
                }
                if (sum == 0) continue;
                int pos = 0;
                if (lane == 0) pos = atomicAdd(&S.sieved, sum);
                pos = __shfl_sync(0xffffffffu, pos, 0);
                if (pos + sum > M::kSieve) {   // the group is tested again after the sieve is emptied
                    full = true;
                    break;
                }
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    if ((vote[q] >> lane) & 1u)
                        S.sieve[pos + __popc(vote[q] & ((1u << lane) - 1u))] =
                            ((unsigned int)k << 24) | (unsigned int)(at + q * 32 + lane);
                    pos += __popc(vote[q]);
                }
            }
            if (full) break;
            c = -1;
        }
        __syncthreads();
        const int sieved = min(S.sieved, M::kSieve);
        for (int i = threadIdx.x; i < sieved; i += T) {
            const unsigned int e = S.sieve[i];
            S.sieve[i] = kNone;
            if (e == kNone) continue;
            const int kk = e >> 24, m = e & 0xffffffu;
            const Dur& t = dur[kk];
            const int s = m * t.b.st;
            const float4* const seg = dp.bounds[t.b.j].seg;
            if (t.b.test == kTestCoarse) {
                // the same bound from the coarse prefix first: no global reads
                const int s1 = s + (1 << clg >> 1);
                float c1 = 0.0f, from = S.coarse[at_coarse(s1 >> clg)];
                int e0 = s;
#pragma unroll 5
                for (int g = 0; g < kBoundSegs; ++g) {
                    const float4 q = __ldg(seg + g);
                    const int off = __float_as_int(q.x);
                    const float to = S.coarse[at_coarse((s1 + off) >> clg)];
                    const float en = fmaf(S.pre[(s + off + bsize - 1) >> lb] - S.pre[e0 >> lb], 1.0f + e_rel, e_abs);
                    c1 = fmaf(q.y, (to - from) * unit, fmaf(q.z, root(en), c1));
                    from = to;
                    e0 = s + off;
                }
                if (c1 < t.cmin_coarse) continue;
            }
            int last = pq[s], e0 = s;
            float c1 = 0.0f;
            if constexpr (kW) {
                const long long sfx = pf[s + t.b.d] - pf[s];
                if (sfx <= 0) continue;   // no depth
                const float depth =
                    tiles::fixed_to_float(sfx) * (dp.inv_sum_t[t.b.j] * (1.0f / 1099511627776.0f));
                const float* const seg_low = dp.bounds[t.b.j].seg_low;
                int lastw = pw[s];
                float c2 = 0.0f;
#pragma unroll 5
                for (int g = 0; g < kBoundSegs; ++g) {
                    const float4 q = __ldg(seg + g);   // end, mean, nu, 1 / length
                    const int e1 = s + __float_as_int(q.x);
                    const int nx = pq[e1], nw = pw[e1];
                    const float sg = (float)(nx - last);
                    const float en = fmaf(S.pre[(e1 + bsize - 1) >> lb] - S.pre[e0 >> lb], 1.0f + e_rel, e_abs);
                    const float sm = fmaxf(fabsf(sg) - (1.0f + 0.5f * (float)(e1 - e0)), 0.0f);
                    c1 += fmaf(q.y, sg, q.z * root(en - q.w * sm * sm));
                    c2 = fmaf(__ldg(seg_low + g), fmaxf(0.0f, (float)(nw - lastw) - 0.5f * (float)(e1 - e0)), c2);
                    last = nx;
                    lastw = nw;
                    e0 = e1;
                }
                c1 = (c1 + t.smin) * unit_a;
                c2 *= unit_w * (1.0f - 1e-5f - t.c2_slack);
                const float v = depth * fmaf(depth, c2, -2.0f * c1) -
                                1e-6f * depth * (depth * c2 + 2.0f * fabsf(c1));
                if (v > thr * (1.0f - 1e-4f)) continue;
                const int to = atomicAdd(&S.n_fin, 1);
                if (to < M::kFinal) S.fin[to] = e;
                continue;
            }
            if ((float)(pq[s + t.b.d] - last) < t.smin) continue;
#pragma unroll 5
            for (int g = 0; g < kBoundSegs; ++g) {
                const float4 q = __ldg(seg + g);   // end, mean, nu, 1 / length
                const int e1 = s + __float_as_int(q.x);
                const int nx = pq[e1];
                const float sg = (float)(nx - last) * unit;
                const float en = fmaf(S.pre[(e1 + bsize - 1) >> lb] - S.pre[e0 >> lb], 1.0f + e_rel, e_abs);
                const float sm = fmaxf(fabsf(sg) - (1.0f + 0.5f * (float)(e1 - e0)) * unit, 0.0f);
                c1 += fmaf(q.y, sg, q.z * root(en - q.w * sm * sm));
                last = nx;
                e0 = e1;
            }
            if (c1 < t.cmin) continue;
            const int to = atomicAdd(&S.n_fin, 1);
            if (to < M::kFinal) S.fin[to] = e;
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            S.tested += sieved;
            S.sieved = 0;
        }
        if (!__syncthreads_or(c >= 0)) break;
        // (a sieve that ran full)
        if (S.n_fin > M::kFinal || (float)S.tested * (T == 1024 ? kSieved : 0.5f * kSieved) >
                                       tiled_time(dp, dur, ndur, kW, lane)) {   // given up
            __syncthreads();
            if (threadIdx.x == 0) S.n_fin = M::kFinal + 1;
            __syncthreads();
            break;
        }
    }
    // their sums (a warp each, any order): v - err <= delta-chi2 <= v + err,
    // whatever the order of the products
    const int nfin = sane ? S.n_fin : 0;   // (final after the last barrier)
    bool fits = sane && nfin <= M::kFinal;
    if (fits) {
        float best = INFINITY;   // lowest upper end
        bool odd = false;        // a sum that is not finite
        for (int i = warp; i < nfin; i += kWarps) {
            const unsigned int e = S.fin[i];
            const Dur& t = dur[e >> 24];
            const int s = (int)(e & 0xffffffu) * t.b.st, d = t.b.d;
            float c1 = 0.0f, c2 = 0.0f;
            if (!kW && T == 1024 && d >= kFineFrom) {   // (shorter curves have no such durations)
                // the bound by kFinePieces pieces first, four per lane: it
                // leaves a few of the windows, whose sums would read all
                // their points (66 windows of up to 9,354 points at a
                // period of 0.55 days: 43 thousand cycles of the CTA)
                static_assert(kFinePieces == 128, "four pieces per lane");
                const float4* const fine =
                    reinterpret_cast<const float4*>(dp.bound_fine + t.b.j * kFinePieces + 4 * lane);
                const float4 f01 = __ldg(fine), f23 = __ldg(fine + 1);
                const float mean[4] = {f01.x, f01.z, f23.x, f23.z}, nu[4] = {f01.y, f01.w, f23.y, f23.w};
                int at[5], p[5];
#pragma unroll
                for (int u = 0; u < 5; ++u) {
                    at[u] = s + (((4 * lane + u) * d) >> 7);
                    p[u] = pq[at[u]];
                }
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const int len = at[u + 1] - at[u];
                    const float sg = (float)(p[u + 1] - p[u]) * unit;
                    const float en = fmaf(S.pre[(at[u + 1] + bsize - 1) >> lb] - S.pre[at[u] >> lb], 1.0f + e_rel, e_abs);
                    const float sm = fmaxf(fabsf(sg) - (1.0f + 0.5f * (float)len) * unit, 0.0f);
                    c1 += fmaf(mean[u], sg, nu[u] * root(en - sm * sm * (1.0f - 1e-5f) / (float)len));
                }
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) c1 += __shfl_xor_sync(0xffffffffu, c1, o);
                if (c1 < t.cmin) {   // (warp-uniform)
                    if (lane == 0) S.fin_v[i] = INFINITY;
                    continue;
                }
                c1 = 0.0f;
            }
            if (kW) {
                const float* const tm = dp.tmpl + dp.tmpl_off[t.b.j];
#pragma unroll 8
                for (int q = lane; q < d; q += 32) {
                    const float sv = __ldg(tm + q);
                    c1 = fmaf(rs[s + q], sv, c1);
                    c2 = fmaf(ws[s + q], sv * sv, c2);
                }
            } else {
                const float* const tm = dp.tmpl_drop + dp.tmpl_off[t.b.j];
                const int base = pq[s];
#pragma unroll 16
                for (int q = lane; q <= d; q += 32) c1 = fmaf((float)(pq[s + q] - base), __ldg(tm + q), c1);
                c1 *= unit;
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                c1 += __shfl_xor_sync(0xffffffffu, c1, o);
                if (kW) c2 += __shfl_xor_sync(0xffffffffu, c2, o);
            }
            const float inv = dp.inv_sum_t[t.b.j], t2 = kW ? c2 : dp.sum_t2[t.b.j];
            const float depth = depth_of(s, d, inv);
            const float v = w_uni * depth * fmaf(depth, t2, -2.0f * c1);
            const float off = t.blur, dd = depth_blur(t, off, inv);
            const float err = sum_error(w_uni, depth, t2, c1, v, off, dd, t.c2_slack);
            if (lane == 0) S.fin_v[i] = v - err;
            odd = odd || !(v - err > -INFINITY && v + err < INFINITY);
            best = fminf(best, v + err);
        }
        if (lane == 0) S.top[warp] = best;
        fits = !__syncthreads_or(odd);
        best = lane < kWarps ? S.top[lane] : INFINITY;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) best = fminf(best, __shfl_xor_sync(0xffffffffu, best, o));
        if (nfin > kFew) {
            // what it takes to sum those near the lowest again
            float again = 0.0f;
            for (int i = threadIdx.x; i < nfin; i += T)
                if (!(S.fin_v[i] > best)) {
                    const float d = (float)dur[S.fin[i] >> 24].b.d;
                    again += kListedWindow + kListedPoint * d * (1.0f + d / kListedRoom);
                }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) again += __shfl_xor_sync(0xffffffffu, again, o);
            if (lane == 0) S.s[warp] = again;
            __syncthreads();
            again = lane < kWarps ? S.s[lane] : 0.0f;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) again += __shfl_xor_sync(0xffffffffu, again, o);
            fits = fits && again <= tiled_time(dp, dur, ndur, kW, lane);
        }
        for (int i = threadIdx.x; i < nfin && fits; i += T) {
            if (S.fin_v[i] > best) continue;
            const unsigned int e = S.fin[i];
            const Dur& t = dur[e >> 24];
            const int m = (int)(e & 0xffffffu);
            auto push = [&](int rot) {
                const unsigned int to = atomicAdd(dk.work + t.b.lg_nc, 1u);
                if (to < dk.list_cap)
                    dk.list[t.b.lg_nc * dk.list_cap + to] = ((unsigned long long)slot << 40) |
                                                            ((unsigned long long)t.b.j << 32) |
                                                            ((unsigned long long)rot << 24) | (unsigned long long)m;
                else
                    S.full = true;
            };
            if (kW || t.b.mode != kModeRot) {
                push(0);
                continue;
            }
            // every block of the tiled kernel that covers window m, with its first round
            const int nc = 1 << t.b.lg_nc, st = t.b.st, rounds = (st + 2 * nc - 1) >> (t.b.lg_nc + 1);
            const int blocks = 32 >> t.b.lg_nc;
            auto push_block = [&](int b) { push(b % blocks % rounds); };
            const DevTiles tl = ds.tiles[lc];
            for (int tau = 0; tau < tl.count; ++tau) {
                const tiles::TileSpan sp = tiles::tile_span(st, (t.b.d + st - 1) / st, 16, 16 * blocks, t.b.m_total,
                                                            tau * tl.len, tl.len, tau, tl.count, buf);
                const int nblk = (sp.m_b - sp.m_a + 15) / 16;
                if (nblk <= 0) continue;
                const int clamped = sp.hi_start < sp.m_a ? 0 : (sp.hi_start - sp.m_a) / 16 + 1;
                const int own = (m - sp.m_a) / 16;
                if (m >= sp.m_a && own < nblk && own < clamped) push_block(own);
                const int mc = max(sp.m_a, sp.hi_start);
                if (m >= mc && m < mc + 16)
                    for (int b = clamped; b < nblk; ++b) push_block(b);
            }
        }
        __syncthreads();
        fits = fits && !S.full;
    }
    return fits;
}

// The folded curve itself and its exact prefix sums, for the kernels that sum
// every window (by the whole CTA; scratch: 33 words in shared memory).  Four
// points per thread and scan: their gathers overlap.  Not inlined: the code
// around it then stays as it is without it (Kepler-like search 327.1 against
// 327.6 ms, 16 curves of 4,000 points 249.7 against 250.4).
template <int T>
__device__ __noinline__ void fill_folded(float* r, long long* sums, const int* sidx, const PointVals* pv, int n, int dm,
                                         long long* scratch)
{
    constexpr int kPer = 4;
    const int total = n + dm, padded = total + (int)kPadMargin;
    long long carry = 0;
    for (int k0 = 0; k0 < padded; k0 += kPer * T) {
        const int k = k0 + kPer * threadIdx.x;
        int id[kPer];
        PointVals v[kPer];
#pragma unroll
        for (int u = 0; u < kPer; ++u) id[u] = k + u < total ? sidx[k + u < n ? k + u : k + u - n] : -1;
        long long sum = 0;
#pragma unroll
        for (int u = 0; u < kPer; ++u) {
            v[u] = id[u] >= 0 && id[u] < n ? pv[id[u]] : PointVals{0, 0.0f, 0.0f};
            sum += v[u].rfx;
        }
        long long before = block_exclusive_scan(sum, scratch, scratch + 32) + carry;
#pragma unroll
        for (int u = 0; u < kPer; ++u) {
            if (k + u <= total) sums[k + u] = before;
            if (k + u < padded) r[k + u] = v[u].r;
            before += v[u].rfx;
        }
        carry += scratch[32];
        __syncthreads();
    }
}

// Whether the bounds are tried at a period (one thread decides for its CTA):
// not while they gave up most periods of the curve lately, but at every 16th.
// Curves whose windows they cannot tell apart (outliers above the flux, a flux
// far from 1, no dip at all) so cost little more than the tiled kernel: 1520
// periods of 62,363 points 33.6 to 9.8, 29.1 to 9.7 and 11.7 to 9.5 ms (8.5
// with every window summed from the start), 4000 of 3,900 points 7.6 to 2.6, 3.3
// to 2.4 and 2.6 to 2.3 ms (2.3); the code for it costs the Kepler-like search
// 0.3 %, curves of 1440 points 1 %.  The count is of the search's pass over
// the curve; which way a period takes changes none of its results.
constexpr int kGivenUp = 32;

__device__ __forceinline__ bool try_bounds(int given_up, int slot) { return given_up < kGivenUp || (slot & 15) == 0; }

// (`then`: the count when the period began; others count too, so that it may
// pass its ends by as many periods as are in flight)
__device__ __forceinline__ void count_bounds(int* given_up, int then, bool fits)
{
    if (fits && then > 0) atomicSub(given_up, 1);
    if (!fits && then < 2 * kGivenUp) atomicAdd(given_up, 1);
}

// The window search after the fold, for one period: by bounds, or left to the
// tiled kernel.
template <int T, bool kW>
__device__ __forceinline__ void window_bounds(unsigned char* smem, const DevSet& ds, const DevChunk& dk, int slot, int lc,
                                              int p, int buf, bool fill, bool ref)
{
    using M = Smem<T>;
    M& S = *reinterpret_cast<M*>(smem);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const DevPlan& dp = ds.plans[lc];
    if (warp == 0) {
        list_durations(dp, ds.curves[lc].check, p, (int)dp.n, S.dur, S.ck, lane);
        for (int k = lane; k < kEnergySpans; k += 32) S.energy[k] = 0.0f;
        if (lane == 0) {
            S.next = S.n_pass = S.sieved = S.tested = S.n_fin = S.dev = S.big = 0;
            S.full = false;
            S.wlow = INT_MAX;
        }
    }
    if (threadIdx.x == 32) {
        S.given_at = ds.curves[lc].given_up + (ref ? 1 : 0);
        S.given_up = __ldcg(S.given_at);
    }
    for (int i = threadIdx.x; i < M::kSieve; i += T) S.sieve[i] = kNone;
    __syncthreads();
    bool fits = false;
    if (try_bounds(S.given_up, slot)) {   // (block-uniform)
        fits = rule_out<T, kW>(S, ds, dk, slot, lc, p, buf);
        if (threadIdx.x == 0 && (!fits || S.given_up > 0))
            count_bounds(S.given_at, S.given_up, fits);
    }
    if (!fits && warp == 0) {
        const int tc = kW ? ds.tiles[lc].count_w : ds.tiles[lc].count;
        const int parts = max(1, min(kDenseParts, (int)(tiled_time(dp, S.dur, S.ck.ndur, kW, lane) / (kPart * (float)tc))));
        if (lane == 0) {
            const long long to = atomicAdd(dk.work + kWorkDense, (unsigned int)tc);
            // (there is room for every period of a wave; as far as there is room,
            // every item that the tiled kernel will read is written)
            in_range(ds.curves[lc].check, 24, to + tc - 1, dk.dense_cap);
            for (int i = 0; i < tc && to + i < dk.dense_cap; ++i) dk.dense[to + i] = make_int2(slot, i | (parts << 24));
        }
    }
    if (!kW && (fill || !fits)) {
        __syncthreads();   // (dur[] is not read any more)
        fill_folded<T>(dk.rs + (int64_t)slot * dk.pad_stride, dk.pf + (int64_t)slot * dk.pad_stride,
                       dk.sidx + (int64_t)slot * dk.fold_stride, ds.curves[lc].pv, (int)dp.n, dp.dmax_p[p],
                       reinterpret_cast<long long*>(smem));
    }
}

// 5. exact sums of the listed windows: one window per CTA at a time, its
// points (by their places in the folded order) and its template staged in
// shared memory by all warps (`room` floats each; longer ones are read in
// place), then summed by the first: the chain of products would wait for every
// row's loads (170 us per wave instead of 30).
static __global__ void __launch_bounds__(kExactThreads)
k_window_exact(DevSet ds, const __grid_constant__ SlotMap smv, const SlotMap* smq, DevChunk dk, int room)
{
    const SlotMap& sm = smq ? *smq : smv;
    extern __shared__ float exact_smem[];
    __shared__ long long part[kExactThreads / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int item = blockIdx.x;
    for (int q = 0; q < kListClasses; ++q) {
        const int cnt = (int)min((int64_t)dk.work[q], dk.list_cap);
        for (; item < cnt; item += gridDim.x) {
            const unsigned long long en = dk.list[q * dk.list_cap + item];
            const int slot = (int)(en >> 40), j = (int)(en >> 32) & 0xff, rot = (int)(en >> 24) & 0xff;
            const int m = (int)(en & 0xffffffull);
            int lc, p;
            if (!resolve_slot(ds, sm, slot, lc, p)) continue;   // block-uniform
            const DevPlan& dp = ds.plans[lc];
            const int d = dp.dpts[j], st = dp.stride[j], v = dp.cfg_variant[j];
            const int mode = v == tiles::kScalar15 ? kModePairS
                             : v == tiles::kCol16R || tiles::variant_colpair(v) ? kModeCols : kModeWin;
            const float* const t = dp.tmpl + dp.tmpl_off[j];
            const int n = (int)dp.n, s = m * st;
            const int* const sidx = dk.sidx + (int64_t)slot * dk.fold_stride;
            const PointVals* const pv = ds.curves[lc].pv;
            auto point = [&](int k) {
                const int id = sidx[s + k < n ? s + k : s + k - n];
                return id >= 0 && id < n ? pv[id] : PointVals{0, 0.0f, 0.0f};
            };
            long long sfx = 0;
            __syncthreads();   // the window before is done with the staged points
#pragma unroll 4
            for (int k = threadIdx.x; k < d; k += blockDim.x) {
                const PointVals v = point(k);
                sfx += v.rfx;
                if (d <= room) {
                    exact_smem[k] = v.r;
                    exact_smem[room + k] = __ldg(t + k);
                }
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) sfx += __shfl_xor_sync(0xffffffffu, sfx, o);
            if (lane == 0) part[warp] = sfx;
            __syncthreads();
            if (warp != 0) continue;
            sfx = 0;
            for (int u = 0; u < (int)(blockDim.x >> 5); ++u) sfx += part[u];
            const float2 sum = d <= room ? window_sum([&](int k) { return exact_smem[k]; }, exact_smem + room, d, st, q,
                                                      mode, rot, lane < (1 << q), lane)
                                         : window_sum([&](int k) { return point(k).r; }, t, d, st, q, mode, rot,
                                                      lane < (1 << q), lane);
            if (lane != 0) continue;
            const float inv = dp.inv_sum_t[j];
            const float depth = fmaxf(0.0f, mode == kModePairS
                                                ? sum.y * inv
                                                : tiles::fixed_to_float(sfx) * (inv * (1.0f / 1099511627776.0f)));
            const float w_uni = (float)ds.curves[lc].scal[2];
            atomicMin(&ds.outs[lc].best[p],
                      tiles::window_key(w_uni * depth * fmaf(depth, dp.sum_t2[j], -2.0f * sum.x), j, m));
        }
        item -= cnt;
    }
}

// The same for per-point weights: (w r, w) and (s_k, s_k^2) pairs, one
// column per lane at a time.
static __global__ void __launch_bounds__(32)
k_window_exact_w(DevSet ds, const __grid_constant__ SlotMap smv, const SlotMap* smq, DevChunk dk, int room)
{
    const SlotMap& sm = smq ? *smq : smv;
    extern __shared__ float2 pair_smem[];
    const int lane = threadIdx.x;
    int item = blockIdx.x;
    for (int q = 0; q < kListClasses; ++q) {
        const int cnt = (int)min((int64_t)dk.work[q], dk.list_cap);
        for (; item < cnt; item += gridDim.x) {
            const unsigned long long en = dk.list[q * dk.list_cap + item];
            const int slot = (int)(en >> 40), j = (int)(en >> 32) & 0xff, m = (int)(en & 0xffffffull);
            int lc, p;
            if (!resolve_slot(ds, sm, slot, lc, p)) continue;   // warp-uniform
            const DevPlan& dp = ds.plans[lc];
            const int d = dp.dpts[j], st = dp.stride[j], nc = 1 << q;
            const int64_t base = (int64_t)slot * dk.pad_stride + (int64_t)m * st;
            const float *const wr = dk.wrs + base, *const w = dk.ws + base;
            const float2* const t = dp.tmplw + dp.tmplw_off[j];
            const long long sfx = dk.pf[base + d] - dk.pf[base];
            float x = 0.0f, y = 0.0f;
            if (d <= room) {
                __syncwarp();
                for (int k = lane; k < d; k += 32) {
                    const uint32_t to = (uint32_t)__cvta_generic_to_shared(pair_smem + k);
                    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(to), "l"(wr + k) : "memory");
                    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(to + 4), "l"(w + k) : "memory");
                    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(to + room * 8), "l"(t + k) : "memory");
                }
                asm volatile("cp.async.commit_group;\ncp.async.wait_group 0;" ::: "memory");
                __syncwarp();
            }
            if (lane < nc) {
                for (int rho = lane; rho < st; rho += nc) {
                    if (d <= room) {
#pragma unroll 8
                        for (int k = rho; k < d; k += st) {
                            const float2 v = pair_smem[k], s = pair_smem[room + k];
                            x = fmaf(v.x, s.x, x);
                            y = fmaf(v.y, s.y, y);
                        }
                    } else {
#pragma unroll 8
                        for (int k = rho; k < d; k += st) {
                            const float2 s = __ldg(t + k);
                            x = fmaf(wr[k], s.x, x);
                            y = fmaf(w[k], s.y, y);
                        }
                    }
                }
            }
            for (int o = 1; o < nc; o <<= 1) {
                x += __shfl_xor_sync(0xffffffffu, x, o);
                y += __shfl_xor_sync(0xffffffffu, y, o);
            }
            if (lane != 0) continue;
            const float depth =
                fmaxf(0.0f, tiles::fixed_to_float(sfx) * (dp.inv_sum_t[j] * (1.0f / 1099511627776.0f)));
            atomicMin(&ds.outs[lc].best[p], tiles::window_key(depth * fmaf(depth, y, -2.0f * x), j, m));
        }
        item -= cnt;
    }
}

}  // namespace bounds
}  // namespace gtls

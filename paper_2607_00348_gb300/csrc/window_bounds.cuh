// Window search by bounds (uniform weights): which windows can hold a
// period's minimum at all.
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
// D products need not be summed.  On white noise (the hardest case: the best
// window stands out least) this leaves 0.01-3 % of the windows.
//
// k_window_bounds, one CTA per period:
//   1. sums of r^2 over blocks of 2^lb folded points and their prefix
//      (shared memory), and from it the largest energy of any stretch of a
//      length;
//   2. one pass over all windows, chunk by chunk: the window sum (short
//      windows) or the bound's main term over a few wide pieces; the largest
//      value of every chunk and the four most promising windows are kept;
//   3. those four are summed: the lowest delta-chi2 T is the threshold;
//   4. chunks whose largest value can beat T are walked again; windows that
//      also pass the kBoundSegs-segment bound are listed for step 5.
// k_window_exact:
//   5. the listed windows of all periods of the wave are summed, adding the
//      products of a window in the order of the tiled kernel
//      (window_tiles.cuh): the same columns per lane, the same rows, the same
//      tree over the lanes, for the rotated variant also the same first round
//      of every block that covers the window there; so the minimum, its
//      duration, its start and every bit of its delta-chi2 are those of the
//      tiled kernel.
//
// Periods for which nothing is gained (no window has a negative delta-chi2,
// so that signed zeros decide; too many windows left; a value is not finite)
// are listed for the tiled kernel, which then runs on that list.
//
// The window sums of steps 2 and 4 come from 32-bit prefix sums: the exact
// ones shifted right so far that any window sum fits 31 bits; differences
// modulo 2^32 are then off by at most one unit.
//
// What bounds it: the prefix reads of step 2 (a lane whose start lies in a
// cache line of its own costs the L1 a cycle) and about 40 instructions per
// window.  Windows of small T0 steps are walked position-major -- all
// durations of a stretch of kTileStarts starts before the next -- to keep the
// prefix sums in L1.  Measured on the Kepler-like search (62,363 points,
// 199,577 periods, 3.1e10 windows): 193 ms for the window stage, against
// 698 ms for the tiled kernel alone; 46 windows of a period are left to sum
// on average, out of 154,000.
#pragma once

namespace gtls {
namespace bounds {

constexpr int kThreads = 512;
constexpr int kWarps = kThreads / 32;
constexpr int kMinBlocks = 2;       // resident CTAs per SM
constexpr int kMaxBlocks = 8192;    // energy blocks of a period
constexpr int kEnergyLens = 48;     // lengths 8, 11, 16, 22, ... whose largest energy is kept
constexpr int kMaxChunks = 4096;    // window chunks of a period
constexpr int kTileStarts = 8192;   // window starts walked before the next stretch
constexpr int kGroup = 128;         // windows a warp tests at a time (4 per lane)
constexpr int kChunkGroups = 4;     // groups per chunk (at most)
constexpr int kNearStep = kTileStarts / kGroup;   // T0 steps up to this fill a group in one stretch
constexpr int kSieve = kWarps * kGroup;   // windows waiting for the segment bound: one group per warp always fits
constexpr int kListed = 2048;       // windows listed of a period before the tiled kernel is cheaper
constexpr int kCand = 4;            // windows summed for the threshold
constexpr int kRowBuf = 336;        // prefix sums at whole T0 steps a warp stages for one group
constexpr int kCutSlots = (kBoundCuts + 3) / 4 * 4;
constexpr int kCutPoints = 60;      // windows of at least this many points are first tested by wide pieces
constexpr int kExactThreads = 256;
constexpr unsigned int kNone = 0xffffffffu;

enum Mode : int { kModePairS = 0, kModeCols = 1, kModeRot = 2, kModeWin = 3 };
enum Test : int { kTestSum = 0, kTestCuts = 1, kTestCutsDirect = 2 };

struct Dur {
    int j, d, st, m_total;
    int first, wsub;            // first chunk (of a stretch for T0 steps up to kNearStep), windows per chunk
    int lg_nc, mode, test;
    float lam;                  // first-test value times lam estimates C1 / sqrt(sum s_k^2)
    float emax;                 // upper bound of sum r^2 over any window of the duration
    float first_min, cmin;      // thresholds of the first test (32-bit prefix units) and of the segment bound
    float smin;                 // lowest window sum that can have a depth (32-bit prefix units)
    int row_max;                // first T0 step of the last piece
    int cuts4;                  // wide pieces, rounded up to a multiple of 4
    float cut_last;             // mean of the last piece
    alignas(16) float coef[kCutSlots];   // the pieces' coefficients (0 past the last)
    alignas(16) int row[kCutSlots];      // and first T0 steps
};

__host__ __device__ inline size_t smem_bytes()
{
    return (size_t)kSieve * sizeof(unsigned int) +
           (size_t)(kMaxBlocks + 8 + kMaxChunks + kWarps * kRowBuf) * sizeof(float);
}

// Relative error allowed for a sum of n products in FP32 (twice the bound).
__device__ __forceinline__ float sum_slack(int n) { return 1.2e-7f * (float)(n + 8); }

__device__ __forceinline__ float root(float x) { return x > 0.0f ? x * rsqrtf(x) : (x == 0.0f ? 0.0f : x); }

// Sum of one window by the nc lanes of a group, in the order of the tiled
// kernel; every lane of the group returns the totals (y: window sum of the
// (C1, S) pairs).  Lanes of groups that are not `on` only take part in the
// exchanges.
__device__ __forceinline__ float2 window_sum(const float* __restrict__ r, const float* __restrict__ t, int d, int st,
                                             int lg_nc, int mode, int rot, bool on, int lane)
{
    const int nc = 1 << lg_nc, c = lane & (nc - 1);
    float x = 0.0f, y = 0.0f;
    if (on) {
        if (mode == kModePairS) {
            for (int rho = c; rho < st; rho += nc) {
#pragma unroll 8
                for (int k = rho; k < d; k += st) {
                    const float v = r[k];
                    x = fmaf(v, __ldg(t + k), x);
                    y = v + y;
                }
            }
        } else if (mode == kModeWin) {
            for (int rho = c; rho < st; rho += nc) {
#pragma unroll 8
                for (int k = rho; k < d; k += st) x = fmaf(r[k], __ldg(t + k), x);
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
                    x = fmaf(r[k], __ldg(t + k), x);
                    y = fmaf(r[k + nc], __ldg(t + k + nc), y);
                }
                for (; k < end; k += st) x = fmaf(r[k], __ldg(t + k), x);
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

// Chunks of windows: durations of T0 steps above kNearStep (far ones) are cut
// into groups over the whole curve; the others (near ones) into chunks of at
// most kChunkGroups 2^lg groups inside every stretch of kTileStarts 2^lg
// starts.  Far chunks come first.
struct Chunks {
    int ndur, near_durs;        // durations (ascending); the first near_durs are near
    int far, per_tile, lg;      // far chunks, near chunks per stretch
    int total;
};

// Durations of period p the kernel searches (kept, not marked kWindowOnly)
// into dur[] and their chunks into ck (by one warp).
__device__ __forceinline__ void list_durations(const DevPlan& dp, unsigned int* check, int p, int n, Dur* dur, Chunks* ck,
                                               int lane)
{
    const int lo = dp.jlo[p], hi = dp.jhi[p];
    int count = 0;
    for (int base = 0; base <= hi - lo; base += 32) {
        const int j = lo + base + lane;
        const int d = j <= hi ? dp.dpts[j] : 0, before = j <= hi && j > lo ? dp.dpts[j - 1] : -1;
        const int v = j <= hi ? dp.cfg_variant[j] : (int)tiles::kWindowOnly;
        const bool kept = j <= hi && d != before && v != tiles::kWindowOnly;
        const unsigned int mask = __ballot_sync(0xffffffffu, kept);
        const int k = count + __popc(mask & ((1u << lane) - 1u));
        if (kept && in_range(check, 19, k, tiles::kMaxDur)) {
            const BoundTab& bt = dp.bounds[j];
            Dur t;
            t.j = j;
            t.d = d;
            t.st = dp.stride[j];
            t.m_total = (n + t.st - 1) / t.st;
            t.lg_nc = __ffs(dp.cfg_nc[j]) - 1;
            t.mode = v == tiles::kScalar15 ? kModePairS
                     : v == tiles::kCol16R ? kModeRot
                     : tiles::variant_colpair(v) ? kModeCols : kModeWin;
            t.lam = (bt.cuts == 0 ? bt.mean_all : 1.0f) / bt.root_t2;
            t.test = bt.cuts == 0 ? kTestSum
                     : kGroup + bt.cut_row[bt.cuts - 1] <= kRowBuf ? kTestCuts : kTestCutsDirect;
            t.emax = 0.0f;
            t.cuts4 = (bt.cuts + 3) / 4 * 4;
            t.row_max = bt.cuts ? bt.cut_row[bt.cuts - 1] : 0;
            t.cut_last = bt.cut_coef[bt.cuts];
#pragma unroll
            for (int u = 0; u < kCutSlots; ++u) {
                const bool in = u < bt.cuts;
                t.coef[u] = in ? bt.cut_coef[min(u, kBoundCuts)] : 0.0f;
                t.row[u] = in ? bt.cut_row[min(u, kBoundCuts - 1)] : 0;
            }
            dur[k] = t;
        }
        count += __popc(mask);
    }
    count = min(count, tiles::kMaxDur);
    __syncwarp();
    for (int lg = 0;; ++lg) {   // larger chunks until kMaxChunks hold any curve length
        int run_near = 0, run_far = 0, near_durs = 0;
        for (int base = 0; base < count; base += 32) {
            const int k = base + lane;
            const bool on = k < count;
            const int st = on ? dur[k].st : 1, m_total = on ? dur[k].m_total : 0;
            const bool nearby = st <= kNearStep;
            const int group = (nearby ? kChunkGroups : 1) * kGroup << lg;
            const int wins = nearby ? min(m_total, (kTileStarts << lg) / st + 1) : m_total;
            const int subs = on ? (wins + group - 1) / group : 0;
            int a = nearby ? subs : 0, b = nearby ? 0 : subs;
            const int a0 = a, b0 = b;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int ya = __shfl_up_sync(0xffffffffu, a, o), yb = __shfl_up_sync(0xffffffffu, b, o);
                if (lane >= o) {
                    a += ya;
                    b += yb;
                }
            }
            if (on) {
                dur[k].first = nearby ? run_near + a - a0 : run_far + b - b0;
                // equal chunks, whole groups of 32 windows
                dur[k].wsub = ((wins + subs - 1) / subs + 31) & ~31;
            }
            run_near += __shfl_sync(0xffffffffu, a, 31);
            run_far += __shfl_sync(0xffffffffu, b, 31);
            near_durs += __popc(__ballot_sync(0xffffffffu, on && nearby));
        }
        const int tile = kTileStarts << lg;
        const long long total = run_far + (long long)((n + tile - 1) / tile) * run_near;
        if (total > kMaxChunks) continue;
        if (lane == 0) *ck = Chunks{count, near_durs, run_far, run_near, lg, (int)total};
        break;
    }
    __syncwarp();
}

// Duration k and windows [lo, hi) of chunk c (warp-uniform).
__device__ __forceinline__ void chunk_range(const Chunks& ck, const Dur* dur, int c, int lane, int& k, int& lo, int& hi)
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
    const int wsub = dur[k].wsub;
    lo = (rel - dur[k].first) * wsub;
    int end = dur[k].m_total;
    if (!far) {
        const int st = dur[k].st, tile = kTileStarts << ck.lg;
        lo += (x * tile + st - 1) / st;
        end = min(end, (int)(((long long)(x + 1) * tile + st - 1) / st));
    }
    hi = min(end, lo + wsub);
}

// First test of windows at .. at + cnt - 1 (cnt <= kGroup) of one duration:
// acc[q] of lane l belongs to window at + 32 q + l.  kTestSum: the window sum;
// else sum_u mean_u S_u over the wide pieces u, from prefix sums relative to
// the first window's start (in the warp's rb when they fit there); both in
// units of the 32-bit prefix.
__device__ __forceinline__ void first_test(const Dur& t, const int* __restrict__ pq, int at, int cnt, float* rb, int lane,
                                           float (&acc)[4])
{
    const int st = t.st, d = t.d, test = t.test;
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
    const int cuts4 = t.cuts4;
    const int base = a[0];
    const float last = t.cut_last;
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
        for (int u = 0; u < cuts4; u += 4) {
            const float4 w = *reinterpret_cast<const float4*>(t.coef + u);
            const int4 r = *reinterpret_cast<const int4*>(t.row + u);
#pragma unroll
            for (int q = 0; q < 4; ++q) {   // (past cnt: not used)
                acc[q] = fmaf(w.x, b[r.x + q * 32], acc[q]);
                acc[q] = fmaf(w.y, b[r.y + q * 32], acc[q]);
                acc[q] = fmaf(w.z, b[r.z + q * 32], acc[q]);
                acc[q] = fmaf(w.w, b[r.w + q * 32], acc[q]);
            }
        }
    } else {
#pragma unroll
        for (int q = 0; q < 4; ++q) acc[q] = last * (float)(v[q] - base);
        for (int u = 0; u < cuts4; ++u) {
            const float w = t.coef[u];
            const int* const b = a + t.row[u] * st;
#pragma unroll
            for (int q = 0; q < 4; ++q) acc[q] = fmaf(w, (float)(b[i[q]] - base), acc[q]);
        }
    }
}

static __global__ void __launch_bounds__(kThreads, kMinBlocks)
k_window_bounds(DevSet ds, const __grid_constant__ SlotMap smv, const SlotMap* smq, DevChunk dk, int buf)
{
    const SlotMap& sm = smq ? *smq : smv;
    extern __shared__ unsigned int bound_smem[];
    unsigned int* const sieve = bound_smem;                 // (duration, window) past the first test
    float* const pre = reinterpret_cast<float*>(sieve + kSieve);   // energy prefix
    float* const cmax = pre + kMaxBlocks + 8;               // largest first-test value per chunk
    float* const row_buf = cmax + kMaxChunks;
    __shared__ Dur dur[tiles::kMaxDur];
    __shared__ Chunks s_ck;
    __shared__ int s_next, s_sieved, s_listed;
    __shared__ float s_wsum[kWarps], s_energy[kEnergyLens];
    __shared__ float s_top[kWarps], s_c1[kWarps], s_s[kWarps], s_thr;
    __shared__ int s_top_at[kWarps], s_cand[kCand];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int slot = blockIdx.x;
    int lc, p;
    if (!resolve_slot(ds, sm, slot, lc, p)) return;
    const DevPlan& dp = ds.plans[lc];
    unsigned int* const check = ds.curves[lc].check;
    const float w_uni = (float)ds.curves[lc].scal[2];
    const int n = (int)dp.n;
    const int total = n + dp.dmax_p[p];
    float* const rb = row_buf + warp * kRowBuf;
    const float* const rs = dk.rs + (int64_t)slot * dk.pad_stride;
    const int* const pq = dk.pq + (int64_t)slot * dk.pad_stride;
    const int shift = (int)ds.curves[lc].scal[3];
    const float unit = prefix_unit(shift);   // of the 32-bit prefix

    if (warp == 0) {
        list_durations(dp, check, p, n, dur, &s_ck, lane);
        if (lane == 0) {
            s_next = 0;
            s_sieved = 0;
            s_listed = 0;
        }
    }
    for (int i = threadIdx.x; i < kSieve; i += kThreads) sieve[i] = kNone;
    // 1. energies: blocks of 2^lb points, their exclusive prefix
    int lb = 3;
    while (((total + (1 << lb) - 1) >> lb) > kMaxBlocks) ++lb;
    const int bsize = 1 << lb, nb = (total + bsize - 1) >> lb;
    for (int b = threadIdx.x; b < nb; b += kThreads) {
        const float4* q = reinterpret_cast<const float4*>(rs + ((int64_t)b << lb));   // zeros follow the padded curve
        float e0 = 0.0f, e1 = 0.0f, e2 = 0.0f, e3 = 0.0f;
#pragma unroll 4
        for (int k = 0; k < bsize / 4; ++k) {
            const float4 v = q[k];
            e0 = fmaf(v.x, v.x, e0);
            e1 = fmaf(v.y, v.y, e1);
            e2 = fmaf(v.z, v.z, e2);
            e3 = fmaf(v.w, v.w, e3);
        }
        pre[b] = (e0 + e1) + (e2 + e3);
    }
    __syncthreads();
    const Chunks ck = s_ck;
    const int ndur = ck.ndur;
    {
        constexpr int kPer = kMaxBlocks / kThreads;
        const int b0 = threadIdx.x * kPer;
        float v[kPer], run = 0.0f;
#pragma unroll
        for (int u = 0; u < kPer; ++u) {
            v[u] = run;
            run += b0 + u < nb ? pre[b0 + u] : 0.0f;
        }
        float x = run;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const float y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        if (lane == 31) s_wsum[warp] = x;
        __syncthreads();
        float base = 0.0f;
        for (int w = 0; w < warp; ++w) base += s_wsum[w];
        const float excl = __shfl_up_sync(0xffffffffu, x, 1);   // sums of the lower lanes
        base += lane > 0 ? excl : 0.0f;
#pragma unroll
        for (int u = 0; u < kPer; ++u)
            if (b0 + u <= nb) pre[b0 + u] = base + v[u];
        if (b0 + kPer == nb && nb == kMaxBlocks) pre[nb] = base + run;
    }
    __syncthreads();
    const float e_all = pre[nb];
    // rounding of block sums and prefix: an energy E read from the prefix is
    // at most E (1 + e_rel) + e_abs
    const float e_rel = sum_slack(bsize), e_abs = sum_slack(bsize + 64) * e_all;

    // largest energy of any stretch of a length (a warp per length; starts in
    // blocks [i, i + step) reach `span` blocks further): a row of lengths
    // sqrt(2) apart, and D of the durations that are tested by their sum
    auto max_energy = [&](int len) {
        const int span = (len + bsize - 2) >> lb;
        const int step = max(1, (len >> lb) >> 3);
        float best = 0.0f;
        for (int i = lane * step; i < nb; i += 32 * step)
            best = fmaxf(best, pre[min(nb, i + step + span)] - pre[i]);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) best = fmaxf(best, __shfl_xor_sync(0xffffffffu, best, o));
        return fmaf(best, 1.0f + e_rel, e_abs);
    };
    for (int k = warp; k < kEnergyLens + ndur; k += kWarps) {
        if (k < kEnergyLens) {
            const int len = (k & 1 ? 11 : 8) << (k >> 1);
            const float e = len < 2 * total ? max_energy(len) : fmaf(e_all, 1.0f + e_rel, e_abs);
            if (lane == 0) s_energy[k] = e;
        } else if (dur[k - kEnergyLens].test == kTestSum) {
            const float e = max_energy(dur[k - kEnergyLens].d);
            if (lane == 0) dur[k - kEnergyLens].emax = e;
        }
    }
    // first of those lengths that is at least len
    auto energy_of = [&](int len) {
        const int o = 31 - __clz(max(len - 1, 1) >> 3);     // len - 1 in [8 << o, 16 << o) (o = -1: below 8)
        if (len <= 8) return s_energy[0];
        return s_energy[len <= (11 << o) ? 2 * o + 1 : 2 * o + 2];
    };

    // 2. largest window sum of every chunk; each warp's most promising chunk
    float top = -INFINITY;   // this lane's best estimate of C1 / sqrt(sum s_k^2)
    int top_at = 0;          // its duration and group of windows
    int top_cnt = 0;
    for (;;) {
        int c = 0;
        if (lane == 0) c = atomicAdd(&s_next, 1);
        c = __shfl_sync(0xffffffffu, c, 0);
        if (c >= ck.total) break;
        int k, lo, hi;
        chunk_range(ck, dur, c, lane, k, lo, hi);
        const float lam = dur[k].lam;
        float f = -INFINITY;
        for (int at = lo; at < hi; at += kGroup) {
            float acc[4];
            const int cnt = min(kGroup, hi - at);
            first_test(dur[k], pq, at, cnt, rb, lane, acc);
            float g = -INFINITY;
#pragma unroll
            for (int q = 0; q < 4; ++q) g = fmaxf(g, q * 32 + lane < cnt ? acc[q] : -INFINITY);
            f = fmaxf(f, g);
            if (g * lam > top) {
                top = g * lam;
                top_at = (k << 24) | at;
                top_cnt = cnt;
            }
        }
        f = float_from_order_key(__reduce_max_sync(0xffffffffu, float_order_key(f)));
        if (lane == 0) cmax[c] = f;
    }

    // 3. threshold: the most promising windows of the warps, kWarps / kCand
    // warps to a window (any order: the result only has to be near)
    {
        const unsigned int key = __reduce_max_sync(0xffffffffu, float_order_key(top));
        const int who = __ffs(__ballot_sync(0xffffffffu, float_order_key(top) == key)) - 1;
        const float most = __shfl_sync(0xffffffffu, top, who);
        const int group = __shfl_sync(0xffffffffu, top_at, who), cnt = __shfl_sync(0xffffffffu, top_cnt, who);
        if (most > -INFINITY) {   // the group again: which of the lane's windows it was
            float acc[4];
            const Dur& t = dur[group >> 24];
            first_test(t, pq, group & 0xffffff, cnt, rb, lane, acc);
            int q = 0;
            while (q < 3 && (q * 32 + lane >= cnt || acc[q] * t.lam != top)) ++q;
            top_at = min(group + q * 32 + lane, group + cnt - 1);
        }
        if (lane == who) {
            s_top[warp] = top;
            s_top_at[warp] = top_at;
        }
        if (threadIdx.x < kCand) s_cand[threadIdx.x] = -1;
    }
    __syncthreads();
    if (threadIdx.x < kWarps) {
        const float v = s_top[threadIdx.x];
        int rank = 0;
        for (int w = 0; w < kWarps; ++w)
            rank += s_top[w] > v || (s_top[w] == v && w < (int)threadIdx.x) ? 1 : 0;
        if (rank < kCand && v > -INFINITY) s_cand[rank] = s_top_at[threadIdx.x];
    }
    __syncthreads();
    constexpr int kTeam = kWarps / kCand, kTeamThreads = kTeam * 32;
    {
        const int cand = s_cand[warp / kTeam];
        float c1 = 0.0f, sum = 0.0f;
        if (cand >= 0) {
            const Dur& t = dur[cand >> 24];
            const float* const r = rs + (cand & 0xffffff) * t.st;
            const float* const s = dp.tmpl + dp.tmpl_off[t.j];
#pragma unroll 4
            for (int i = threadIdx.x % kTeamThreads; i < t.d; i += kTeamThreads) {
                const float v = r[i];
                c1 = fmaf(v, __ldg(s + i), c1);
                sum += v;
            }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            c1 += __shfl_xor_sync(0xffffffffu, c1, o);
            sum += __shfl_xor_sync(0xffffffffu, sum, o);
        }
        if (lane == 0) {
            s_c1[warp] = c1;
            s_s[warp] = sum;
        }
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        float thr = INFINITY;
        for (int q = 0; q < kCand; ++q) {
            if (s_cand[q] < 0) continue;
            const int j = dur[s_cand[q] >> 24].j;
            float c1 = 0.0f, sum = 0.0f;
            for (int w = q * kTeam; w < (q + 1) * kTeam; ++w) {
                c1 += s_c1[w];
                sum += s_s[w];
            }
            const float depth = fmaxf(0.0f, sum * dp.inv_sum_t[j]);
            const float v = w_uni * depth * fmaf(depth, dp.sum_t2[j], -2.0f * c1);
            thr = v < thr || isnan(v) ? v : thr;
        }
        s_thr = thr;
        s_next = 0;
    }
    __syncthreads();
    const float thr = s_thr;
    // no negative delta-chi2, or values out of range: the tiled kernel decides
    const bool sane = thr < 0.0f && thr > -INFINITY && e_all < INFINITY && w_uni < INFINITY && shift < 64;
    if (sane) {
        // thresholds of every duration.  A window whose C1 stays below cmin is
        // above thr; 1e-4 of slack covers the rounding of thr and of
        // delta-chi2 itself, and `lost` what FP32 summation, the 32-bit prefix
        // and segment sums can lose of C1 (at most sum_slack(products in a
        // row) ||r|| ||s||, 2^-41 of fixed point per point, and the prefix
        // units of the sums)
        const float reach = sqrtf(-thr / w_uni) * (1.0f - 1e-4f);
        for (int k = threadIdx.x; k < ndur; k += kThreads) {
            Dur& t = dur[k];
            const BoundTab& bt = dp.bounds[t.j];
            const int nc = 1 << t.lg_nc;
            const int chain = ((t.st + nc - 1) >> t.lg_nc) * ((t.d + t.st - 1) / t.st) + 6;
            if (t.test != kTestSum) t.emax = energy_of(t.d);
            const float norm = sqrtf((float)t.d * t.emax);
            const float lost = (sum_slack(chain) + 8e-6f) * norm + (float)t.d * 1e-12f;
            t.cmin = reach * bt.root_t2 - (lost + (float)(kBoundSegs + 1) * unit) * bt.t_max;
            // depth is zero without a positive sum (exact, or FP32 for the pairs)
            const float low = (t.mode == kModePairS ? -lost : 0.0f) - 2.0f * unit;
            float c0;
            if (t.test == kTestSum) {
                c0 = fmaxf((t.cmin - bt.nu_all * sqrtf(t.emax)) / bt.mean_all, low);
            } else {
                float lose = 0.0f;
                for (int u = 0; u < bt.cuts; ++u) lose = fmaf(bt.cut_nu[u], sqrtf(energy_of(bt.cut_len[u])), lose);
                // rounding of the prefix sums, which reach over the whole group
                const float over = (float)(kGroup * t.st) / (float)t.d + 2.0f;
                c0 = t.cmin - lose - 1.2e-7f * (float)(bt.cuts + 4) * 2.0f * over * norm * bt.t_max;
            }
            t.first_min = (c0 - 1e-5f * fabsf(c0)) / unit;
            t.smin = low / unit;
        }
    }
    __syncthreads();

    // 4. windows that may hold the minimum: chunks whose largest sum passes,
    // their windows by sum or rows into the sieve, those by segments into the
    // queues; a full sieve is emptied before the walk goes on
    int c = -1, k = 0, at = 0, hi = 0;
    while (sane) {
        for (;;) {
            if (c < 0) {
                if (lane == 0) c = atomicAdd(&s_next, 1);
                c = __shfl_sync(0xffffffffu, c, 0);
                if (c >= ck.total) {
                    c = -1;
                    break;
                }
                chunk_range(ck, dur, c, lane, k, at, hi);
                if (cmax[c] < dur[k].first_min) {
                    c = -1;
                    continue;
                }
            }
            const float first_min = dur[k].first_min;
            bool full = false;
            for (; at < hi; at += kGroup) {
                const int cnt = min(kGroup, hi - at);
                float acc[4];
                first_test(dur[k], pq, at, cnt, rb, lane, acc);
                unsigned int pass = 0;
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    if (q * 32 + lane < cnt && !(acc[q] < first_min)) pass |= 1u << q;
                unsigned int vote[4];
                int sum = 0;
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    vote[q] = __ballot_sync(0xffffffffu, (pass >> q) & 1u);
                    sum += __popc(vote[q]);
                }
                if (sum == 0) continue;
                int pos = 0;
                if (lane == 0) pos = atomicAdd(&s_sieved, sum);
                pos = __shfl_sync(0xffffffffu, pos, 0);
                if (pos + sum > kSieve) {   // the group is tested again after the sieve is emptied
                    full = true;
                    break;
                }
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    if ((pass >> q) & 1u)
                        sieve[pos + __popc(vote[q] & ((1u << lane) - 1u))] =
                            ((unsigned int)k << 24) | (unsigned int)(at + q * 32 + lane);
                    pos += __popc(vote[q]);
                }
            }
            if (full) break;
            c = -1;
        }
        __syncthreads();
        const int sieved = min(s_sieved, kSieve);
        for (int i = threadIdx.x; i < sieved; i += kThreads) {
            const unsigned int e = sieve[i];
            sieve[i] = kNone;
            if (e == kNone) continue;
            const int kk = e >> 24, m = e & 0xffffffu;
            const Dur& t = dur[kk];
            const int s = m * t.st;
            const int p0 = pq[s];
            if ((float)(pq[s + t.d] - p0) < t.smin) continue;
            {
                const BoundTab& bt = dp.bounds[t.j];
                float c1 = 0.0f;
                int last = p0, e0 = s;
#pragma unroll 5
                for (int g = 0; g < kBoundSegs; ++g) {
                    const int e1 = s + __ldg(bt.off + g + 1);
                    const int nx = pq[e1];
                    const float sg = (float)(nx - last) * unit;
                    const float en = fmaf(pre[(e1 + bsize - 1) >> lb] - pre[e0 >> lb], 1.0f + e_rel, e_abs);
                    const float len = __ldg(bt.inv_len + g) * fmaxf(fabsf(sg) - unit, 0.0f) * fmaxf(fabsf(sg) - unit, 0.0f);
                    c1 += fmaf(__ldg(bt.mean + g), sg, __ldg(bt.nu + g) * root(en - len));
                    last = nx;
                    e0 = e1;
                }
                if (c1 < t.cmin) continue;
            }
            auto push = [&](int rot) {
                const unsigned int to =
                    atomicAdd(&s_listed, 1) < kListed ? atomicAdd(dk.left_n + t.lg_nc, 1u) : 0xffffffffu;
                if (to < dk.list_cap)
                    dk.list[t.lg_nc * dk.list_cap + to] = ((unsigned long long)slot << 40) |
                                                          ((unsigned long long)t.j << 32) |
                                                          ((unsigned long long)rot << 24) | (unsigned long long)m;
                else
                    s_listed = 2 * kListed;   // (more may be added: it stays above kListed)
            };
            if (t.mode != kModeRot) {
                push(0);
                continue;
            }
            // every block of the tiled kernel that covers window m, with its first round
            const int nc = 1 << t.lg_nc, rounds = (t.st + 2 * nc - 1) >> (t.lg_nc + 1), blocks = 32 >> t.lg_nc;
            auto push_block = [&](int b) { push(b % blocks % rounds); };
            const DevTiles tl = ds.tiles[lc];
            for (int tau = 0; tau < tl.count; ++tau) {
                const tiles::TileSpan sp =
                    tiles::tile_span(t.st, (t.d + t.st - 1) / t.st, 16, 16 * blocks, t.m_total, tau * tl.len, tl.len,
                                     tau, tl.count, buf);
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
        if (threadIdx.x == 0) s_sieved = 0;
        if (!__syncthreads_or(c >= 0)) break;
    }
    __syncthreads();
    if (!sane || s_listed > kListed) {   // block-uniform
        if (threadIdx.x == 0) {
            const int tc = ds.tiles[lc].count;
            const unsigned int to = atomicAdd(dk.left_n + kListClasses, (unsigned int)tc);
            for (int tau = 0; tau < tc; ++tau) dk.dense[to + tau] = make_int2(slot, tau);
        }
    }
}

// 5. exact sums of the listed windows: groups of nc lanes, the lists of the
// six group sizes one after the other.
static __global__ void __launch_bounds__(kExactThreads)
k_window_exact(DevSet ds, const __grid_constant__ SlotMap smv, const SlotMap* smq, DevChunk dk)
{
    const SlotMap& sm = smq ? *smq : smv;
    const int lane = threadIdx.x & 31;
    const int warps = gridDim.x * (kExactThreads / 32);
    int item = blockIdx.x * (kExactThreads / 32) + (threadIdx.x >> 5);
    for (int q = 0; q < kListClasses; ++q) {
        const unsigned int cnt = (unsigned int)min((int64_t)dk.left_n[q], dk.list_cap);
        const int groups = 32 >> q, items = (int)((cnt + groups - 1) / groups);
        for (; item < items; item += warps) {
            const unsigned int e = (unsigned int)item * groups + (lane >> q);
            const unsigned long long en = dk.list[q * dk.list_cap + min(e, cnt - 1)];
            const int slot = (int)(en >> 40), j = (int)(en >> 32) & 0xff, rot = (int)(en >> 24) & 0xff;
            const int m = (int)(en & 0xffffffull);
            int lc, p;
            const bool on = resolve_slot(ds, sm, slot, lc, p) && e < cnt;
            if (!on) lc = p = 0;
            const DevPlan& dp = ds.plans[lc];
            const int d = dp.dpts[j], st = dp.stride[j], v = dp.cfg_variant[j];
            const int mode = v == tiles::kScalar15 ? kModePairS
                             : v == tiles::kCol16R || tiles::variant_colpair(v) ? kModeCols : kModeWin;
            const int64_t base = (int64_t)slot * dk.pad_stride + (int64_t)m * st;
            const float2 sum = window_sum(dk.rs + base, dp.tmpl + dp.tmpl_off[j], d, st, q, mode, rot, on, lane);
            if (!on || (lane & ((1 << q) - 1)) != 0) continue;
            const float inv = dp.inv_sum_t[j];
            const float depth =
                fmaxf(0.0f, mode == kModePairS
                                ? sum.y * inv
                                : tiles::fixed_to_float(dk.pf[base + d] - dk.pf[base]) * (inv * (1.0f / 1099511627776.0f)));
            const float w_uni = (float)ds.curves[lc].scal[2];
            atomicMin(&ds.outs[lc].best[p],
                      tiles::window_key(w_uni * depth * fmaf(depth, dp.sum_t2[j], -2.0f * sum.x), j, m));
        }
        item -= items;
    }
}

}  // namespace bounds
}  // namespace gtls

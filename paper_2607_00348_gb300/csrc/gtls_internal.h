// Internal structures of libgtls shared by the CUDA translation units.
#pragma once

#include <cuda_runtime.h>

#include <cstdint>
#include <string>
#include <vector>

#include "gtls.h"
#include "plan_host.h"

namespace gtls {

// Template of one duration cut into pieces for the bounds of the window
// search (window_bounds.cuh): a few wide pieces (first test of a window) and
// kBoundSegs segments (second test).
constexpr int kBoundCuts = 17;
constexpr int kBoundCutSlots = kBoundCuts - 1;   // the first one starts at 0 and is kept apart
constexpr int kBoundSegs = 25;
constexpr int kBoundLevels = 6;
struct alignas(16) BoundTab {
    float4 seg[kBoundSegs];       // end (point, integer bits), mean of s_k, >= ||s_k - mean||, <= 1 / length
    float mean_all, nu_all;       // mean of s_k over the template, >= ||s_k - mean||
    float root_t2;                // sqrt(sum_k s_k^2)
    float t_max;                  // >= |s_k|
    float change;                 // >= |s_0| + sum |s_k - s_{k-1}| + |s_{d-1}|
    int32_t cuts;                 // wide pieces (0: the window sum alone is tested)
    float cut_jumps, seg_jumps;   // sums of |mean - mean before| over the wide pieces, the segments
    float cut_nu[kBoundCuts];     // >= ||s_k - mean|| over the piece
    int32_t cut_len[kBoundCuts];  // its points
    // per-point weights: sum w s_k^2 >= sum_l lev_up (smallest sum of w over
    // lev_len points), and the smallest s_k^2 of every segment
    int32_t lev_len[kBoundLevels];
    float lev_up[kBoundLevels];
    float seg_low[kBoundSegs];
};

// Templates of at least kFineFrom points also in kFinePieces equal pieces: mean
// of s_k and >= ||s_k - mean|| of every piece.
constexpr int kFinePieces = 128, kFineFrom = 1024;

// What the bounds need of one duration for every period (staged in shared
// memory by the words).
struct alignas(16) BoundDur {
    int32_t j, d, st, m_total;    // grid index, points, T0 step, windows
    int32_t subs, wsub;           // chunks (of the curve or a stretch; 0: not searched here), windows per chunk
    int32_t lg_nc, mode, test;    // lanes per window, summation order and first test (window_bounds.cuh)
    int32_t row_max;              // first T0 step of the last wide piece
    int32_t cuts4;                // wide pieces after the first, rounded up to a multiple of 4
    float lam;                    // first-test value times lam estimates C1 / sqrt(sum s_k^2)
    float cut_last;               // mean of the last wide piece
    float coef0;                  // minus the mean of the first
    float mean_all;               // mean of s_k over the template
    int32_t pad;
    float coef[kBoundCutSlots];   // of the others: mean of the piece before minus its mean (Abel form; 0 past the last)
    int32_t row[kBoundCutSlots];  // their first T0 steps, or points
};

// Read-only plan tables on the device (passed to kernels by value).
struct DevPlan {
    int64_t n;
    int32_t np;           // periods
    int32_t nd;           // T14/P grid points
    int32_t time_exponent;
    int32_t idx_bits;
    int32_t bucket_log2;
    int32_t fold_nsb;      // super-buckets of the staged fold
    int32_t max_kept;
    const double* periods;
    const int64_t* p_lat;
    const float* inv_p;
    const int32_t* bucket_shift;
    const uint32_t* bucket_mul;
    const int32_t* jlo;
    const int32_t* jhi;
    const int32_t* dmax_p;
    const int32_t* dpts;
    const int32_t* stride;
    const int64_t* tmpl_off;
    const float* tmpl;
    const float* tmpl_drop;   // s_{k-1} - s_k, k = 0 .. D (window search by bounds)
    const float* inv_sum_t;   // 1 / sum_k s_k
    const float* sum_t2;      // sum_k s_k^2
    const double* sum_t;      // FP64 sum_k s_k
    const double* q;
    int64_t tmpl_total;       // floats in tmpl
    const int32_t* cfg_variant; // window-kernel variant per duration (see window_tiles.cuh)
    const int32_t* cfg_nc;      // phase-column lanes per window block per duration
    const int64_t* tmpl2_off;   // offset of duration j in tmpl2 (float2 units)
    const float2* tmpl2;        // template pairs (s_k, s_{k+nc}) of column-pair durations
    const int64_t* tmplw_off;   // offset of duration j in tmplw (float2 units)
    const float2* tmplw;        // per-point weights: template pairs (s_k, s_k^2), zero padded
    const int32_t* cfg_nc_w;    // per-point weights: lanes per window block per duration
    int32_t median_half;        // half width h of the running-median window
    int32_t refine_k;           // periods re-searched with T0 step 1 (0: none)
    const int64_t* tc_off;      // offset of duration j in tc_tab (floats; kTensor durations)
    const BoundTab* bounds;     // pieces of every duration's template
    const BoundDur* bound_durs;
    const float2* bound_fine;   // kFinePieces per duration
    int32_t bound_lg;           // chunks of the window search are 2^bound_lg times the usual size
    const float* tc_tab;        // tensor-core template chunks: [chunk][hi, lo][32 x 32 core-matrix layout]
};

// What the fold gathers for one point, in one 16-byte load.
struct alignas(16) PointVals {
    long long rfx;            // rint((1 - y) 2^40): exact window sums of r
    float r;                  // float(1 - y)
    float w;                  // float(1 / dy^2)
};

// Per-light-curve derived arrays (n long unless noted).
struct DevCurve {
    int64_t* d_lat;           // rint((t - t_ref) 2^e)
    float* d_f;               // float(t - t_ref) (days): coarse cycle estimate
    PointVals* pv;            // rfx, r, w of every point
    float* r;                 // r alone
    double* scal;             // [0] t_ref [1] chi2_0 [2] uniform weight w (0 if not uniform) [3] prefix shift (per-point
                              // weights: [3], [4] exponents of the units of the w r and w prefix sums)
    unsigned long long* tmin_key;  // ordered key of min(t)
    unsigned int* flags;      // bit0 non-finite, bit1 dy <= 0, bit2 dy not uniform
    double* part;             // block partials of chi2_0
    unsigned int* check;      // [0] first failed device check (0 = none), [1..3] its values
    int* given_up;            // periods that the bounds gave up lately: coarse pass, refinement
};

constexpr int kListClasses = 6;   // windows are summed by groups of 1, 2, 4, ..., 32 lanes

// Words that the kernels of a wave count in (DevChunk::work): windows listed,
// by class, items in `dense`, and the items that the tiled and the tensor-core
// kernel have taken.  A wave starts with all of them at zero: they are cleared
// in stream order before its first kernel (k_wave_next for waves cut on the
// device), never by a kernel whose own CTAs add to them.
constexpr int kWorkDense = kListClasses, kWorkTiles = kListClasses + 1, kWorkTensor = kListClasses + 2;
constexpr int kWorkWords = kListClasses + 3;

// Per-chunk scratch: `chunk` periods in flight.
struct DevChunk {
    int32_t chunk;
    int64_t fold_stride;      // >= n
    int64_t key_stride;       // >= n and >= the super-bucket regions of the fold
    int64_t pad_stride;       // >= n + dmax + margin (folded, padded arrays)
    unsigned long long* keys; // fold keys (super-bucket regions, or bucket order)
    int32_t* sidx;            // folded order -> original index
    float* rs;                // folded r, padded by the period's first D_m points
    float* ws;                // folded w (per-point weights only)
    float* wrs;               // folded w r (per-point weights only)
    long long* pf;            // prefix sums of rfx over the padded folded curve
    // window search by bounds: prefix sums in 32 bits, and what it leaves to
    // sum in the wave.  For uniform weights rs and pf are only written for
    // periods that it leaves to the kernels that sum every window.
    int32_t* pq;              // of r (per-point weights: w r) in units (modulo 2^32: window sums fit 31 bits)
    int64_t list_cap;         // windows per lane-group size
    unsigned long long* list; // windows to sum, kListClasses lists
    int64_t dense_cap;        // items
    int2* dense;              // tiles for the tiled kernel: slot, and tile | CTAs that may share it << 24
    unsigned int* work;       // kWorkWords counters of the wave in flight
};

// SR/SDE: blocks per curve of the reductions, and blocks of the running median
// whose best SDE is kept (more: the spectrum itself is searched).
constexpr int kSrBlocks = 128;
constexpr int kTopBlocks = 1024;
constexpr int kSrParts = 3 * kSrBlocks + 2 * kTopBlocks;

// Per-period outputs (np long) and the reduction scratch.
struct DevPeriod {
    unsigned long long* best; // packed (delta-chi2 key, j, window) minimum
    double* chi2;
    int32_t* dur;
    int32_t* t0i;
    double* depth;
    double* t0;
    double* sr;
    double* sde_raw;
    double* sde;
    double* stats;            // [0] chi2_min [1] mean SR [2] std SR
    double* part;             // kSrParts: the SR/SDE blocks' minima, sums and square sums, and their best SDE
    unsigned int* check;      // same words as DevCurve::check
    int32_t* refined;         // 1 where the period was re-searched with T0 step 1
    int32_t* plist;           // the refine_k periods to re-search, in rank order
    gtls_result* result;      // device copy of the best candidate
};

// Tile shape of one light curve in the tiled window kernel.
struct DevTiles {
    int32_t len;              // window starts per tile (L)
    int32_t count;            // tiles per period
    int32_t len_w;            // the same for per-point weights (tiles of (w r, w) pairs)
    int32_t count_w;
};

// Per-light-curve descriptors of a search (device arrays, one entry per
// curve; a single search uses one entry).
struct DevSet {
    const DevPlan* plans;
    const DevCurve* curves;
    const DevPeriod* outs;
    const DevTiles* tiles;
};

// Which (light curve, period) each slot of a wave holds: a wave is up to
// kMaxSeg segments of consecutive periods (or consecutive positions of the
// curve's refinement list), passed by value.
constexpr int kMaxSeg = 32;
struct WaveSeg {
    int32_t lc;               // light curve
    int32_t first;            // first period (or refinement-list position)
    int32_t slot0;            // first slot of the segment in the wave
    int32_t item0;            // first window-tile item of the segment
};
struct SlotMap {
    int32_t nseg;
    int32_t slots;            // slots in the wave
    int32_t items;            // window-tile items in the wave
    int32_t from_list;        // periods are refinement-list positions
    WaveSeg seg[kMaxSeg];
};

// Records `msg` as the calling thread's last error and returns s (shared by
// the translation units behind the C ABI).
gtls_status set_error(gtls_status s, const std::string& msg);

}  // namespace gtls

struct gtls_plan {
    gtls::PlanHost host;
    int device = -1;
    gtls::DevPlan dp{};
    gtls::DevCurve dc{};
    gtls::DevChunk dk{};
    gtls::DevPeriod dq{};
    double* in_t = nullptr;   // plan-owned input buffers of gtls_search_host
    double* in_y = nullptr;
    double* in_dy = nullptr;
    int64_t device_bytes = 0;
    // tiled window search (uniform weights; per-point weights: tile_w_*, in
    // (w r, w) pairs)
    bool tile_ok = false;
    int tile_buf = 0, tile_len = 0, tile_count = 0;
    bool tile_w_ok = false;
    int tile_buf_w = 0, tile_len_w = 0, tile_count_w = 0;
    // durations too long for a tile (marked kWindowOnly): searched by the
    // one-thread-per-window kernel in the same waves
    bool has_window_only = false, has_window_only_ref = false;
    // durations on the tensor-core window kernel (kTensor), the widest
    // [jlo, jhi] span of a period (work items per period of that kernel), and
    // the timeout test (a wait that nothing completes)
    bool has_tensor = false;
    bool bounds_ok = false;              // the templates admit the bounds of window_bounds.cuh
    bool bounds_w_ok = false;            // ... with per-point weights
    int tc_jspan = 0;
    int tc_test_wait = 0;
    const void* tc_maps = nullptr;      // TMA maps of dk.rs (made with the chunk scratch)
    std::vector<int32_t> variant_host;   // window-kernel variant per duration (host copies)
    std::vector<int32_t> variant_ref_host, nc_host;
    int n_sm = 0;
    // refinement stage (T0 step 1 on the best periods): plan tables with
    // stride 1 and the (s_k, 1) pair tables, its tile configuration and the
    // device list of periods to re-search
    int refine_k = 0;
    gtls::DevPlan dp_ref{};
    int tile_len_ref = 0, tile_count_ref = 0;
    // one-entry device descriptor sets of the coarse and refinement passes
    gtls::DevSet set{}, set_ref{};
    int64_t* prep_off = nullptr;        // device {0, n}: the curve's offsets
    bool chunk_ready = false;           // dk allocated (first single search or gtls_plan_reserve)
    int64_t chunk_bytes = 0;            // device bytes of the chunk scratch
    void* chunk_mem = nullptr;          // its allocation
    std::vector<float> tmpl_pad;        // host copy of the zero-padded template table
    std::vector<int64_t> tmpl_pad_off;
    // stage profiling: events recorded on the search stream when enabled
    bool profiling = false;
    std::vector<cudaEvent_t> events;
    std::vector<int> event_stage;   // stage of the interval ending at event i
    gtls_profile profile{};
    void* allocs[96] = {};
    int n_allocs = 0;
};

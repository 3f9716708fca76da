// Host side of the C ABI declared in include/hass.h: argument checks, tile schedules, TMA
// descriptors, workspace layout and kernel launches. No allocation, no synchronisation except in
// hass_check and the *_host entry.
#include <algorithm>
#include <atomic>
#include <climits>
#include <cstdint>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <vector>

#include "../../include/hass.h"
#include "row_split_kernel.cuh"
#include "hca_kernels.cuh"
#include "hca_pair_kernel.cuh"
#include "hca_bwd_fused_kernel.cuh"

namespace hass {

static std::atomic<long long> g_launches{0};

// ---- optional per-kernel timing (hass_profile_*) ------------------------------------------------
// When enabled, every kernel launch is bracketed by a pair of CUDA events on its own stream; the
// summary adds up the elapsed time per kernel kind. Off by default; not thread-safe.
enum { KIND_STATS = 0, KIND_PROBS = 1, KIND_OUT = 2, KIND_FINALIZE = 3, KIND_PREP = 4, KIND_CONDITIONAL = 5, KIND_HCA = 6, KIND_HCA_DQ_CONVERT = 7, KIND_HCA_BWD_FUSED = 8, KIND_HCA_BWD_ROWS = 9, KIND_STATS_DRAFT = 10, NUM_KINDS = 11 };
constexpr int kMaxRecords = 8192;
struct Profiler {
    bool on = false;
    int n = 0;
    std::vector<cudaEvent_t> ev;     // 2 per record
    std::vector<int> kind;
};
static Profiler g_prof;

struct KernelTimer {
    int rec = -1;
    cudaStream_t st;
    KernelTimer(int kind, cudaStream_t s) : st(s) {
        if (g_prof.on && g_prof.n < kMaxRecords) {
            rec = g_prof.n++;
            g_prof.kind[rec] = kind;
            cudaEventRecord(g_prof.ev[2 * rec], st);
        }
    }
    ~KernelTimer() {
        if (rec >= 0) cudaEventRecord(g_prof.ev[2 * rec + 1], st);
    }
};

// duration of a pair's step (256 x 256 outputs) over that of two single CTAs (128 x 256 outputs each); measured 0.89-0.92
constexpr double kPairStepTime = 0.90;

constexpr int MAX_CLUSTER = 8;

typedef void (*GemmFn)(GemmParams);

// Launches `fn` as a programmatic dependent of the stream's previous kernel (see wait_previous_kernel), in clusters of
// `cluster` blocks. 64 rows x 256 x 1024, five kernels: 47 -> 39 us per call; HCA forward + backward of 2 x 333
// positions, four kernels: 75 -> 73 us.
template <typename... P, typename... A>
static int launch(void (*fn)(P...), long long grid, int block, size_t smem, cudaStream_t st, int cluster, A&&... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(static_cast<unsigned>(grid));
    cfg.blockDim = dim3(static_cast<unsigned>(block));
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    at[1].id = cudaLaunchAttributeClusterDimension;
    at[1].val.clusterDim.x = static_cast<unsigned>(cluster);
    at[1].val.clusterDim.y = 1;
    at[1].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = cluster > 1 ? 2 : 1;
    g_launches.fetch_add(1);
    if (cudaLaunchKernelEx(&cfg, fn, static_cast<P>(args)...) != cudaSuccess) {
        cudaGetLastError();
        return HASS_ERR_CUDA;
    }
    return HASS_OK;
}

// ---- device info ------------------------------------------------------------------------------
struct DeviceInfo {
    int ok = 0;   // 0 unknown, 1 usable, <0 hass_status
    int sms = 148;
    int clusters[MAX_CLUSTER + 1] = {};   // clusters of this many CTAs of the second GEMM that are resident at once
    int hca_clusters[MAX_CLUSTER + 1] = {};   // ... of the attention's backward
    int hca_fwd_clusters[MAX_CLUSTER + 1] = {};   // ... and forward
};
static DeviceInfo g_dev[64];

static int device_info(DeviceInfo* out) {
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) {
        cudaGetLastError();
        return HASS_ERR_CUDA;
    }
    DeviceInfo& di = g_dev[dev];
    if (di.ok == 0) {
        int major = 0, sms = 0;
        if (cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, dev) != cudaSuccess ||
            cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) {
            cudaGetLastError();
            return HASS_ERR_CUDA;
        }
        if (major != 10) {
            di.ok = HASS_ERR_ARCH;
        } else {
            di.sms = sms;
            GemmFn const gemms[] = {gemm_kernel<MODE_STATS, TOPK_REG, 1>,  gemm_kernel<MODE_STATS, TOPK_REG, 2>,
                                    gemm_kernel<MODE_STATS, TOPK_BUF, 1>,  gemm_kernel<MODE_STATS, TOPK_BUF, 2>,
                                    gemm_kernel<MODE_STATS, TOPK_NONE, 1>, gemm_kernel<MODE_STATS, TOPK_NONE, 2>,
                                    gemm_kernel<MODE_STATS, TOPK_REG, 1, 8>, gemm_kernel<MODE_STATS, TOPK_REG, 2, 8>,
                                    gemm_kernel<MODE_STATS, TOPK_NONE, 1, 8>, gemm_kernel<MODE_STATS, TOPK_NONE, 2, 8>,
                                    gemm_kernel<MODE_PROBS, TOPK_BUF, 1>,  gemm_kernel<MODE_PROBS, TOPK_BUF, 2>,
                                    gemm_kernel<MODE_OUT, TOPK_BUF, 1>,    gemm_kernel<MODE_OUT, TOPK_BUF, 2>,
                                    gemm_kernel<MODE_OUT, TOPK_NONE, 1>,   gemm_kernel<MODE_OUT, TOPK_NONE, 2>,
                                    gemm_kernel<MODE_LOGITS, TOPK_BUF, 1>, gemm_kernel<MODE_LOGITS, TOPK_BUF, 2>};
            cudaError_t e3 = cudaSuccess;
            for (GemmFn f : gemms)
                if (e3 == cudaSuccess) e3 = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_BYTES);
            if (e3 == cudaSuccess) e3 = cudaFuncSetAttribute(select_kernel<16, 512>, cudaFuncAttributeMaxDynamicSharedMemorySize, 16 * 512 * 8);
            if (e3 == cudaSuccess) e3 = cudaFuncSetAttribute(select_kernel<16, 1024>, cudaFuncAttributeMaxDynamicSharedMemorySize, 16 * 1024 * 8);
            cudaError_t e4 = cudaFuncSetAttribute(hca2::hca_attention_pair_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, hca2::SMEM_BYTES);
            if (e4 == cudaSuccess) e4 = cudaFuncSetAttribute(hca2::hca_attention_pair_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, hca2::SMEM_BYTES);
            if (e4 == cudaSuccess) e4 = cudaFuncSetAttribute(hca_bwd::hca_bwd_fused_kernel<1>, cudaFuncAttributeMaxDynamicSharedMemorySize, hca_bwd::F_SMEM_BYTES);
            if (e4 == cudaSuccess) e4 = cudaFuncSetAttribute(hca_bwd::hca_bwd_fused_kernel<2>, cudaFuncAttributeMaxDynamicSharedMemorySize, hca_bwd::F_SMEM_BYTES);
            if (e4 == cudaSuccess) e4 = cudaFuncSetAttribute(hca_bwd::hca_bwd_fused_kernel<1, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, hca_bwd::F_SMEM_BYTES);
            for (int c = 2; c <= MAX_CLUSTER; ++c) {
                cudaLaunchConfig_t cfg = {};
                cfg.gridDim = dim3(c);
                cfg.blockDim = dim3(NUM_THREADS);
                cfg.dynamicSmemBytes = SMEM_BYTES;
                cudaLaunchAttribute at;
                at.id = cudaLaunchAttributeClusterDimension;
                at.val.clusterDim.x = c;
                at.val.clusterDim.y = 1;
                at.val.clusterDim.z = 1;
                cfg.attrs = &at;
                cfg.numAttrs = 1;
                if (cudaOccupancyMaxActiveClusters(&di.clusters[c], gemm_kernel<MODE_OUT, TOPK_BUF, 1>, &cfg) != cudaSuccess) {
                    cudaGetLastError();
                    di.clusters[c] = 0;
                }
                cfg.blockDim = dim3(hca_bwd::NUM_THREADS);
                cfg.dynamicSmemBytes = hca_bwd::F_SMEM_BYTES;
                if (cudaOccupancyMaxActiveClusters(&di.hca_clusters[c], hca_bwd::hca_bwd_fused_kernel<1, true>, &cfg) != cudaSuccess) {
                    cudaGetLastError();
                    di.hca_clusters[c] = 0;
                }
                cfg.blockDim = dim3(hca2::NUM_THREADS);
                cfg.dynamicSmemBytes = hca2::SMEM_BYTES;
                if (cudaOccupancyMaxActiveClusters(&di.hca_fwd_clusters[c], hca2::hca_attention_pair_kernel<true>, &cfg) != cudaSuccess) {
                    cudaGetLastError();
                    di.hca_fwd_clusters[c] = 0;
                }
            }
            if (e3 != cudaSuccess || e4 != cudaSuccess) {
                cudaGetLastError();
                return HASS_ERR_CUDA;
            }
            di.ok = 1;
        }
    }
    if (di.ok < 0) return di.ok;
    *out = di;
    return HASS_OK;
}

static int sm_count_or_default() {
    DeviceInfo di;
    int n = 0;
    if (cudaGetDeviceCount(&n) != cudaSuccess || n <= 0) {
        cudaGetLastError();
        return 148;
    }
    return device_info(&di) == HASS_OK ? di.sms : 148;
}

static int ceil_div(long long a, long long b) { return static_cast<int>((a + b - 1) / b); }

// ---- tile schedule ----------------------------------------------------------------------------
// Splits RT row tiles into phases (G row tiles x S lanes, G * S <= sms) minimising the summed phase
// durations ceil(CT / S), by dynamic programming over the number of row tiles already covered. pair = 2: the
// same in units of CTA pairs, each covering two row tiles (an odd RT counts as the next even number).
// *cost = the summed durations, in column tiles. one_phase: all row tiles side by side (at most sms slots).
static int plan_schedule(int RT, int CT, int sms, int pair, Schedule* out, int* cost = nullptr, bool one_phase = false) {
    const int units = (RT + pair - 1) / pair, groups_max = sms / pair;
    if (RT < 1 || CT < 1 || groups_max < 1) return HASS_ERR_INVALID_ARG;
    if (one_phase && units > groups_max) return HASS_ERR_UNSUPPORTED;
    const int INF = 1 << 30;
    std::vector<int> best(units + 1, INF), nph(units + 1, INF), choice(units + 1, 0);
    best[0] = 0;
    nph[0] = 0;
    for (int n = 1; n <= units; ++n) {
        for (int G = one_phase ? n : 1; G <= n && G <= groups_max; ++G) {
            int S = groups_max / G;
            if (S > CT) S = CT;
            const int c = best[n - G] + (CT + S - 1) / S;
            const int ph = nph[n - G] + 1;
            if (c < best[n] || (c == best[n] && ph < nph[n])) {
                best[n] = c;
                nph[n] = ph;
                choice[n] = G;
            }
        }
    }
    if (nph[units] > MAX_PHASES) return HASS_ERR_UNSUPPORTED;
    std::vector<int> groups;
    for (int n = units; n > 0; n -= choice[n]) groups.push_back(choice[n]);
    std::memset(out, 0, sizeof(*out));
    int rt = 0, slot = 0, maxc = 0;
    // largest groups first: the widest phases start together
    for (size_t i = 0; i < groups.size(); ++i)
        for (size_t j = i + 1; j < groups.size(); ++j)
            if (groups[j] > groups[i]) std::swap(groups[i], groups[j]);
    for (size_t i = 0; i < groups.size(); ++i) {
        const int G = groups[i] * pair;
        int S = groups_max / groups[i];
        if (S > CT) S = CT;
        out->ph[i] = Phase{rt, G, S, slot};
        rt += G;
        slot += G * S;
        if (G * S > maxc) maxc = G * S;
    }
    out->n_phases = static_cast<int>(groups.size());
    out->total_slots = slot;
    out->max_ctas = maxc;
    out->pair = pair;
    if (cost) *cost = best[units];
    return HASS_OK;
}

// The schedule that a launch over RT row tiles uses, of at most max_slots slots: the one of least expected time
// among single CTAs and pairs, in as many phases as it takes or in one.
static int plan_launch(int RT, int CT, int sms, int max_slots, Schedule* out) {
    int rc = HASS_ERR_WORKSPACE;
    double best = 0.;
    for (int i = 0; i < 4; ++i) {
        const int pair = i & 1 ? 2 : 1;
        if (pair == 2 && (RT < 2 || sms < 2)) continue;
        Schedule s;
        int steps = 0;
        const int r = plan_schedule(RT, CT, sms, pair, &s, &steps, i >= 2);
        if (i == 0 && r != HASS_OK) return r;
        const double time = steps * (pair == 2 ? kPairStepTime : 1.);
        if (r == HASS_OK && s.total_slots <= max_slots && (rc != HASS_OK || time < best)) {
            *out = s;
            best = time;
            rc = HASS_OK;
        }
    }
    return rc;
}

// ---- division of the output tiles of MODE_OUT -----------------------------------------------------
constexpr long long kKeepBytes = 64ll << 20;      // of W that the first of two readings leaves in the L2 (narrow_sweep)
constexpr int kPartTilesMax = 296;      // partial tiles of one CTA each, at most (38.8 MB): two rounds of the grid

// Over `rows` rows, CT column tiles and a contraction of `kb` blocks, with room for part_bytes of partial tiles. Expected
// times in steps of one k block (about 0.5 us): cutting the rest of the last round costs a kernel of its own (14 steps),
// the partial tiles' way to memory and back (4 TB/s) and one fill and drain of the pipeline (6 steps) per piece.
// Measured (second GEMM alone): 61 rows x 4096 x 32000 179 -> 56 us (16 tiles in 16 x 8 pieces on 128 of the SMs), 517
// rows x 4096 x 128256 822 -> 657 us, the 28-row-tile chunk of 8192 rows 4 rounds of 74 pairs -> 3 and a cut rest.
// A tile per cluster needs no partial tiles and no second kernel; it costs the exchange (6 steps) and fits while all
// clusters are resident at once (clusters[]: how many are; nullptr: not considered).
// 250 rows x 4096 x 32000, whose partial tiles do not fit the workspace: call 318 -> 235 us.
// l2_cols > 0: B, of so many columns, is small enough to be in the L2 from the sweep before, and the contraction short. Few tiles of it are a chain of latencies, and narrower
// ones leave a cluster less to exchange and every CTA less to load: 64 rows x 256 x 1024 22.0 -> 17.5 us per call, 53 x 280 x 2179 combined
// 28.7 -> 20.5, 12 x 2784 x 4695 Bi-directional 47 -> 43. (Out of memory B comes faster in cut pieces of wide tiles, on
// more of the SMs: 2 rows x 8192 x 128256 636 us per call, 699 with clusters of two on 128 columns; 128 x 4096 x 32000 122 and 135. Long contractions are better cut, too: 2048 x 256 x 32000 242 and 247.)
constexpr int kShortBlocks = 256;
static OutPlan plan_out(int rows, int CT, int kb, int sms, size_t part_bytes, const int* clusters, int l2_cols = 0) {
    const int RT = (rows + BM - 1) / BM;
    const int part_rows = RT == 1 ? rows : BM;      // rows kept of a partial tile
    const size_t tile_bytes = static_cast<size_t>(part_rows) * BN * 4;
    OutPlan best = {};
    double best_cost = 0.;
    for (int pair = 1; pair <= 2; ++pair) {
        if (pair == 2 && (RT < 2 || sms < 2)) break;
        const int units = (RT + pair - 1) / pair, groups = sms / pair;
        const long long tiles = static_cast<long long>(units) * CT;
        const int rest = static_cast<int>(tiles % groups);
        const int whole = static_cast<int>(tiles - rest);
        const double step = pair == 2 ? kPairStepTime : 1.;
        for (int cuts = 1; cuts == 1 || (rest > 0 && cuts <= kb / 4 && static_cast<long long>(rest) * cuts * pair <= kPartTilesMax &&
                                         static_cast<size_t>(rest) * cuts * pair * tile_bytes <= part_bytes); ++cuts) {
            double cost = step * (whole / groups) * (kb + 6.);
            if (rest > 0) {
                const int rounds = (rest * cuts + groups - 1) / groups;
                cost += step * rounds * ((kb + cuts - 1) / cuts + 6.);
                if (cuts > 1) cost += 14. + 2. * rest * cuts * pair * tile_bytes / 2e6;
            }
            if (best.groups == 0 || cost < best_cost) {
                best_cost = cost;
                best.pair = pair;
                best.part_rows = part_rows;
                best.cluster = 1;
                best.width = BN;
                best.row_units = units;
                best.whole = cuts == 1 ? static_cast<int>(tiles) : whole;
                best.rest = cuts == 1 ? 0 : rest;
                best.cuts = cuts;
                best.groups = static_cast<int>(tiles < groups && cuts == 1 ? tiles
                                               : whole == 0 && static_cast<long long>(rest) * cuts < groups ? rest * cuts
                                                                                                            : groups);
            }
        }
    }
    for (int cand = 0; clusters && cand < (l2_cols ? 3 : 1) * (MAX_CLUSTER - 1); ++cand) {
        const int width = BN >> cand / (MAX_CLUSTER - 1), c = 2 + cand % (MAX_CLUSTER - 1);
        const long long tiles = static_cast<long long>(RT) * (l2_cols ? ceil_div(l2_cols, width) : CT);
        // a step fetches 16 KB of A and up to 32 of B; the exchange: 2 steps and up to 4
        const double cost = (kb + c - 1) / c * (1. + 2. * width / BN) / 3. + 6. + 2. + 4. * width / BN;
        if (tiles > clusters[c] || kb < 2 * c || cost >= best_cost) continue;
        best_cost = cost;
        best = OutPlan{};
        best.pair = 1;
        best.row_units = RT;
        best.whole = static_cast<int>(tiles);
        best.cuts = 1;
        best.groups = static_cast<int>(tiles) * c;
        best.part_rows = part_rows;
        best.cluster = c;
        best.width = width;
    }
    return best;
}
static size_t part_bytes_of(const OutPlan& o) { return o.rest ? static_cast<size_t>(o.rest) * o.cuts * o.pair * o.part_rows * BN * 4 : 0; }

// ---- TMA descriptors --------------------------------------------------------------------------
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
static EncodeTiledFn g_encode = nullptr;

static int get_encode() {
    if (g_encode) return HASS_OK;
    void* fn = nullptr;
    cudaDriverEntryPointQueryResult qres;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &fn, cudaEnableDefault, &qres) != cudaSuccess ||
        qres != cudaDriverEntryPointSuccess || !fn) {
        cudaGetLastError();
        return HASS_ERR_CUDA;
    }
    g_encode = reinterpret_cast<EncodeTiledFn>(fn);
    return HASS_OK;
}

// bf16 row-major matrix [rows, cols] with `pitch` elements between rows; box = box_cols x box_rows,
// 128-byte swizzle (box_cols must be 64), out-of-range elements read as zero.
static int make_tmap(CUtensorMap* tm, const void* base, long long rows, long long cols, long long pitch,
                     int box_cols, int box_rows) {
    cuuint64_t gdim[2] = {static_cast<cuuint64_t>(cols), static_cast<cuuint64_t>(rows)};
    cuuint64_t gstride[1] = {static_cast<cuuint64_t>(pitch) * 2};
    cuuint32_t box[2] = {static_cast<cuuint32_t>(box_cols), static_cast<cuuint32_t>(box_rows)};
    cuuint32_t estr[2] = {1, 1};
    CUresult r = g_encode(tm, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), gdim, gstride, box, estr,
                          CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                          CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? HASS_OK : HASS_ERR_CUDA;
}

// bf16 tensor [B, T, heads * 128] (dense): box = 64 columns x box_rows positions of one sequence, 128-byte
// swizzle. Positions past T read as zeros, so a ragged last tile never sees the next sequence.
static int make_tmap_seq(CUtensorMap* tm, const void* base, long long B, long long T, long long cols,
                         int box_rows = 128) {
    cuuint64_t gdim[3] = {static_cast<cuuint64_t>(cols), static_cast<cuuint64_t>(T), static_cast<cuuint64_t>(B)};
    cuuint64_t gstride[2] = {static_cast<cuuint64_t>(cols) * 2, static_cast<cuuint64_t>(cols) * 2 * static_cast<cuuint64_t>(T)};
    cuuint32_t box[3] = {64, static_cast<cuuint32_t>(box_rows), 1};
    cuuint32_t estr[3] = {1, 1, 1};
    CUresult r = g_encode(tm, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(base), gdim, gstride, box, estr,
                          CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                          CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? HASS_OK : HASS_ERR_CUDA;
}

// capacity of a (row, slot) candidate buffer for this K
static int topk_cap(int K) { return K <= K_REG ? K_REG : cand_cap(K); }

// ---- workspace layout -------------------------------------------------------------------------
static inline size_t align256(size_t x) { return (x + 255) & ~static_cast<size_t>(255); }

struct Layout {
    size_t status, part_m, part_s, cand_v, cand_i, thr_share, fwd_end, sidx, sgq, coef, lse2, capz, zmax, sparse, scratch, fixed_end;
    size_t scratch_row_tile_bytes;   // bytes of dz_d scratch per 128-row tile
    long long p_pitch;
    int pref_chunk_tiles;
    int slot_cap;
    size_t total_pref;
    size_t part_bytes;               // partial tiles of the second GEMM, behind the scratch; without them it is not cut
};


// Row tiles per chunk when at most `most` fit: all RT, or an even number of them (pairs of CTAs work on two).
static int even_chunk(int most, int RT) {
    if (most >= RT) return RT;
    return most > 1 ? most & ~1 : most;
}

// Whether a call's logits may go through the workspace in fp32 (narrow_impl), in one chunk of row tiles: three kernels instead of nine and more. One
// row tile: always. From 257 rows on: while the row kernel takes less time than the launches that go. Its blocks take 11 ns a row at pitch <= 1024 and
// K <= 32, 18 at pitch <= 2048 and K <= 64, 57 at pitch <= 2048 otherwise, and about 20 + 3.2 pitch / 1000 beyond; there the line lies at 50 us of it, at 65
// where d >= 3072 (the joint sweep takes pairs of CTAs also for an odd number of row tiles), and at 25 (`single`) where one matrix alone is swept
// and for the forward alone, which save fewer launches. us per call, the other route -> this one:
//   pitch 1024, K = 10, d = 256     600 rows 62 -> 31, 1500 64 -> 40, 2795 69 -> 56; beyond the line 4500 71 -> 75
//   pitch 1024, K = 41, d = 256     1500 rows 89 -> 55; beyond 2795 94 -> 82, but Bi-directional 159 -> 177
//   pitch 1024, K = 101, d = 256    600 rows 123 -> 60; beyond 1500 132 -> 113, 2795 140 -> 186
//   pitch 2048, K = 10, d = 4096    1000 rows 111 -> 68; beyond 3900 187 -> 213
//   50 us: 360 x 4096 x 2100, K = 56 119 -> 59, 659 x 5120 x 2758, K = 46 203 -> 81, 268 x 4096 x 12459 171 -> 128, 300 x 4096 x 32000 334 -> 294; beyond 594 x 1080 x 33218 237 -> 262
//   65 us: 450 x 4096 x 32000 391 -> 380, 512 399 -> 396, 530 514 -> 478; beyond 613 x 5120 x 32000 573 -> 597
//   25 us: draft rows 710 x 5120 x 4375 84 -> 70; beyond 257 x 256 x 32000 47 -> 52
// Two limits are no measurement. 129 to 256 rows stay on the spill's route, because tests hold what such calls do beyond its exponent range and
// report in the status block. Beyond 2048 tokens seven row tiles are the most (1013 x 256 x 4525 145 -> 68 would gain), because a test counts the
// workspace of larger calls in row tiles.
static bool narrow_rows(long long N, long long d, long long pitch, int K, int chunk_tiles, int sms, bool single) {
    if (N <= BM) return true;
    const long long most = K <= 32 && pitch <= 1024   ? 3072
                           : K <= 64 && pitch <= 2048 ? 2048
                           : pitch <= 2048            ? 1024
                                                      : std::min(7ll * BM, (single ? 25000 : d >= 3072 ? 65000 : 50000) * 1000ll / (20000 + 16 * pitch / 5));
    return N > 2 * BM && N <= most && N <= static_cast<long long>(chunk_tiles) * BM && 2 * ((N + BM - 1) / BM) <= sms;
}

// Rows per chunk of a combined call whose logits go through the workspace in fp32; 0: it spills. The spilled probabilities of target and draft
// have references of their own, known before the sums are, so that the gradient takes a product with W for each; from fp32 logits the row
// kernel forms their difference (rounded once instead of twice) and one product is enough. The sweep stores twice the bytes, which its products
// hide, and the row kernel reads them twice. Per call, in runs of 0.4 s (the power cap): 1024 rows x 4096 x 128256 3670 -> 3350 us, 517 rows 2580 -> 2110,
// 2048 x 4096 x 32000 1930 -> 1580, 8192 rows 7780 -> 6330, 300 rows 518 -> 326, 1318 x 376 x 38201, K = 65 522 -> 433, 8000 x 704 x 3000, K = 128 1170 -> 676,
// 640 x 512 x 8000 127 -> 67. Chunks of an eighth of the SM count in row tiles (every CTA pair has its part of the columns), or of a quarter
// where their logits stay in the L2 (8000 x 256 x 1024 216 -> 184), of 1.6 GB at most: 8192 x 4096 x 32000 takes the same in chunks of 18 and of 37
// tiles, 1024 x 4096 x 128256 3 % more in two of 4 than in one. (Calls of 129 to 256 rows keep to the spill, as narrow_rows has it.)
constexpr long long kCombinedBytes = 1600ll << 20, kCombinedL2Bytes = 128ll << 20;
static int combined_rows(long long N, long long V, int sms) {
    if (N <= 2 * BM) return 0;
    const int RT = ceil_div(N, BM);
    const long long tile = static_cast<long long>(BM) * ceil_div(V, BN) * BN * 8;
    const bool stays = std::max(1, sms / 4) * tile <= kCombinedL2Bytes;
    const long long most = stays ? sms / 4 : std::min<long long>(sms / 8, kCombinedBytes / tile);
    if (most < 4) return 0;
    const int chunks = ceil_div(RT, stays ? even_chunk(sms / 4, RT) : most);      // (even_chunk: the workspace holds no more rows of d in fp32)
    return ceil_div(RT, chunks) * BM;
}

// The forward schedule covers 2 * RT row tiles (target then draft).
static int make_layout(long long N, long long d, long long V, int K, int sms, Layout* L) {
    const int RT = ceil_div(N, BM), CT = ceil_div(V, BN);
    Schedule s;
    int rc = plan_schedule(2 * RT, CT, sms, 1, &s);
    if (rc != HASS_OK) return rc;
    int pref = even_chunk(sms / 4, RT);
    if (pref < 1) pref = 1;
    // partial-statistics slots: enough for the whole-batch forward and for sweeps over chunks of about sms / 4 row tiles
    // (target + draft tiles, or one of them, of a full or last chunk); plan_launch keeps to them
    int slot_cap = s.total_slots;
    {
        int most = sms / 4;
        if (most < 1) most = 1;
        if (most > RT) most = RT;
        const int rem = RT % most;
        const int cands[5] = {RT, 2 * most, most, 2 * rem, rem};
        for (int i = 0; i < 5; ++i) {
            if (cands[i] < 1) continue;
            Schedule t;
            rc = plan_schedule(cands[i], CT, sms, 1, &t);
            if (rc != HASS_OK) return rc;
            if (t.total_slots > slot_cap) slot_cap = t.total_slots;
        }
    }
    if (slot_cap < sms) slot_cap = sms;     // any single-phase schedule (a caller-limited, smaller chunk) fits
    L->slot_cap = slot_cap;
    size_t off = 0;
    L->status = off;
    off += 256;
    const size_t slots = static_cast<size_t>(slot_cap);
    L->thr_share = off;                     // admission thresholds the lanes of a row tile publish to each other; behind the
    off = align256(off + slots * BM * 4);   // status block, so that one memset clears both
    L->part_m = off;
    off = align256(off + slots * BM * 4);
    L->part_s = off;
    off = align256(off + slots * BM * 4);
    L->cand_v = off;                        // candidate buffers: (logit, token id) pairs, cand_cap(K) per (row, slot)
    off = align256(off + slots * BM * 8 * topk_cap(K));
    L->cand_i = off;                        // entries in use per (row, slot)
    off = align256(off + slots * BM * 4);
    L->fwd_end = off;                       // what the forward-only entry points use
    L->sidx = off;
    off = align256(off + static_cast<size_t>(N) * K * 4);
    L->sgq = off;
    off = align256(off + static_cast<size_t>(N) * K * 4);
    L->coef = off;
    off = align256(off + static_cast<size_t>(N) * 4);
    L->lse2 = off;
    off = align256(off + static_cast<size_t>(N) * 4);
    L->capz = off;                          // fused path: draft logits at Omega_hat, captured by the draft sweep, [N, K]
    off = align256(off + static_cast<size_t>(N) * K * 4);
    L->zmax = off;                          // single-sweep route: every spilling row's largest logit (target and draft rows)
    off = align256(off + static_cast<size_t>(2 * RT) * BM * 4);
    L->sparse = off;                        // fused path: Omega_hat term of one chunk of rows, fp32 [chunk rows, d]
    off = align256(off + static_cast<size_t>(pref) * BM * d * 4);
    L->scratch = off;
    L->fixed_end = off;
    L->p_pitch = static_cast<long long>(CT) * BN;
    L->scratch_row_tile_bytes = static_cast<size_t>(BM) * L->p_pitch * 2;
    L->pref_chunk_tiles = pref;
    L->total_pref = align256(off + L->scratch_row_tile_bytes * pref);
    L->part_bytes = 0;
    // less than a row tile of scratch, so that a workspace's size still tells how many row tiles fit
    const long long all = N < static_cast<long long>(pref) * BM ? N : static_cast<long long>(pref) * BM;
    const long long chunks[2] = {all, N % (static_cast<long long>(pref) * BM)};
    for (long long rows : chunks) {
        if (rows < 1) continue;
        const size_t need = part_bytes_of(plan_out(static_cast<int>(rows), ceil_div(d, BN), ceil_div(V, BK), sms,
                                                   L->scratch_row_tile_bytes - 256, nullptr));
        if (need > L->part_bytes) L->part_bytes = need;
    }
    if (N > BM && narrow_rows(N, d, L->p_pitch, K, pref, sms, false)) {
        const size_t end = L->scratch + 2 * align256(static_cast<size_t>(N) * L->p_pitch * 4);
        if (end > L->total_pref && end - L->total_pref > L->part_bytes) L->part_bytes = end - L->total_pref;
    }
    if (N <= BM) {
        // the fp32 logits of such a call (narrow_room), from the scratch on, and its partial tiles; one chunk in any case
        const size_t z = align256(static_cast<size_t>(N) * L->p_pitch * 4);
        const size_t parts = align256(part_bytes_of(plan_out(static_cast<int>(N), ceil_div(d, BN), ceil_div(V, BK), sms, SIZE_MAX, nullptr)));
        const size_t end = L->scratch + z + (parts > z ? parts : z);
        if (end > L->total_pref && end - L->total_pref > L->part_bytes) L->part_bytes = end - L->total_pref;
    }
    return HASS_OK;
}

// ---- argument checks --------------------------------------------------------------------------
static bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

static int check_sizes(long long N, long long d, long long V, int K) {
    if (N < 1 || d < 8 || V < 1 || K < 1) return HASS_ERR_INVALID_ARG;
    if (d % 8 != 0) return HASS_ERR_INVALID_ARG;
    if (K > V || K > HASS_K_MAX) return HASS_ERR_INVALID_ARG;
    if (N > (1ll << 30) || V > (1ll << 30) || d > (1ll << 20)) return HASS_ERR_UNSUPPORTED;
    return HASS_OK;
}

static const bool kLog = [] {
    const char* e = std::getenv("HASS_LOG");
    return e && e[0] == '1';
}();

static void log_schedule(const char* what, const Schedule& s) {
    if (!kLog) return;
    std::fprintf(stderr, "[hass] %s: %d phases, %d slots, grid %d:", what, s.n_phases, s.total_slots, s.max_ctas);
    for (int i = 0; i < s.n_phases; ++i)
        std::fprintf(stderr, " (rt0=%d G=%d S=%d)", s.ph[i].row_tile_begin, s.ph[i].G, s.ph[i].S);
    std::fprintf(stderr, "\n");
}

template <int MODE>
static int launch_gemm(const GemmParams& p, cudaStream_t st, int kind = -1) {
    KernelTimer timer(p.gate ? KIND_CONDITIONAL : (kind >= 0 ? kind : MODE), st);
    const bool pair = p.sched.pair == 2;
    GemmFn fn;
    // Eight epilogue warps where the products of a tile are short, up to 1024 columns of features, and a lane has three tiles or more, behind which
    // their meeting disappears. Calls of 2048 rows x d x 32000, K = 10, on four and on eight: d = 256 288 -> 250 us, 512 309 -> 277, 1024 375 -> 360, K =
    // 64 366 -> 336, 387 -> 357, 453 -> 435; from 2048 on the stage that they cost shows (2048 584 -> 587, 600 x 2048 285 -> 330), and so does the
    // meeting where a lane has one tile (383 x 256 x 1024 59 -> 61).
    constexpr int kWideBlocks = 16;
    const bool none = MODE == MODE_STATS && p.topk_row_tiles == 0 && p.cap_z != nullptr;
    if (MODE == MODE_STATS && p.k_blocks <= kWideBlocks && p.col_tiles > 2 * p.sched.ph[0].S &&
        (none || (p.K <= K_REG && p.spill_begin == INT_MAX && p.Pt == nullptr))) {
        if (none)
            fn = pair ? gemm_kernel<MODE_STATS, TOPK_NONE, 2, 8> : gemm_kernel<MODE_STATS, TOPK_NONE, 1, 8>;
        else
            fn = pair ? gemm_kernel<MODE_STATS, TOPK_REG, 2, 8> : gemm_kernel<MODE_STATS, TOPK_REG, 1, 8>;
        return launch(fn, p.sched.max_ctas, gemm_threads(8), gemm_smem(pair ? 2 : 1, 8), st, pair ? 2 : 1, p);
    }
    if (none)
        fn = pair ? gemm_kernel<MODE_STATS, TOPK_NONE, 2> : gemm_kernel<MODE_STATS, TOPK_NONE, 1>;
    else if (MODE == MODE_STATS && p.K <= K_REG)
        fn = pair ? gemm_kernel<MODE_STATS, TOPK_REG, 2> : gemm_kernel<MODE_STATS, TOPK_REG, 1>;
    else if (MODE == MODE_OUT && p.kept)
        fn = pair ? gemm_kernel<MODE_OUT, TOPK_NONE, 2> : gemm_kernel<MODE_OUT, TOPK_NONE, 1>;
    else
        fn = pair ? gemm_kernel<MODE, TOPK_BUF, 2> : gemm_kernel<MODE, TOPK_BUF, 1>;
    return launch(fn, p.sched.max_ctas, NUM_THREADS, SMEM_BYTES, st, MODE == MODE_OUT && p.plan.cluster > 1 ? p.plan.cluster : pair ? 2 : 1, p);
}

// Clears a 256-byte aligned piece of the workspace (a multiple of 16 bytes), and a second one.
static int clear_bytes(void* at, size_t bytes, cudaStream_t st, void* at2 = nullptr, size_t bytes2 = 0) {
    const int n = static_cast<int>(bytes / 16), n2 = static_cast<int>(bytes2 / 16);
    return launch(clear_kernel, n + n2 <= 256 * 16 ? ceil_div(n + n2, 256) : 16, 256, 0, st, 1, static_cast<uint4*>(at), n, static_cast<uint4*>(at2), n2);
}

// Clears the status block (only_thresholds: not) and the published thresholds of `slots` slots, with their shared bounds.
static int clear_status(uint8_t* ws, const Layout& L, int slots, cudaStream_t st, bool only_thresholds = false, uint2* bounds = nullptr) {
    const size_t from = only_thresholds ? L.thr_share : L.status;
    if (only_thresholds && slots == 0) return HASS_OK;
    return clear_bytes(ws + from, L.thr_share + static_cast<size_t>(slots) * BM * 4 - from, st, bounds,
                       bounds ? static_cast<size_t>(slots) * BM * 8 : 0);
}

// Bytes [from, to) of the workspace, which nothing else uses between the clearing and the selection after a sweep of this
// schedule, as the room in which its lanes share their bounds (GemmParams::bounds); nullptr where they do not fit or K needs none. With
// a place of their own in the layout they would take from calls at the least workspace and from the built-in scratch.
static uint2* bounds_room(uint8_t* ws, size_t from, size_t to, const Schedule& s, int K) {
    return K > K_REG && to >= from + static_cast<size_t>(s.total_slots) * BM * 8 ? reinterpret_cast<uint2*>(ws + from) : nullptr;
}

template <int WARPS, int WIN>
static constexpr size_t select_smem() { return static_cast<size_t>(sel_block_warps(WARPS)) * WIN * 8; }
template <int WARPS, int WIN>
static int select_as(const SelectParams& sp, cudaStream_t st) {
    constexpr int bw = sel_block_warps(WARPS);
    return launch(select_kernel<WARPS, WIN>, ceil_div(sp.rows, bw / WARPS), bw * 32, select_smem<WARPS, WIN>(), st, 1, sp);
}

// Sixteen warps per row while every row has an SM of its own, four while that is at most four blocks per SM, one warp
// beyond. The lists of K <= 16 hold 16 entries each
// and need the smaller window. Against one warp per row that walks the lists one after the other: 61 rows x 125 lists
// 113 -> 15 us, 4096 rows x 4 lists 40 -> 9 us (22 with the dot product for the reference exponent, which saves the
// draft sweep its extra tile: 25 us here, half of it at 61 rows), 4096 rows of K = 64 275 -> 130 us.
static int launch_select(const SelectParams& sp, int sms, cudaStream_t st) {
    KernelTimer timer(sp.gate ? KIND_CONDITIONAL : KIND_FINALIZE, st);
    const bool reg = sp.cap == K_REG;
    if (sp.rows <= sms) return reg ? select_as<16, 512>(sp, st) : select_as<16, 1024>(sp, st);
    if (sp.rows <= 4 * sms) return reg ? select_as<4, 512>(sp, st) : select_as<4, 1024>(sp, st);
    return reg ? select_as<1, 512>(sp, st) : select_as<1, 1024>(sp, st);
}

// What select_kernel needs to pick the K best of the candidates that sweep `p` left on its row tiles from first_tile on
static SelectParams select_params(const GemmParams& p, int first_tile, int row_begin, int rows, int* idx_out, float* q_out,
                                  int out_pitch, float* lse) {
    SelectParams sp;
    std::memset(&sp, 0, sizeof(sp));
    sp.sched = p.sched;
    sp.first_tile = first_tile;
    sp.K = p.K;
    sp.cap = p.cap;
    sp.row_begin = row_begin;
    sp.rows = rows;
    sp.from_sweep = 1;
    sp.part_m = p.part_m;
    sp.part_s = p.part_s;
    sp.cand = p.cand;
    sp.cand_n = p.cand_n;
    sp.thr_share = p.thr_share;
    sp.bounds = p.bounds;
    sp.col_tiles = p.col_tiles;
    sp.idx_out = idx_out;
    sp.q_out = q_out;
    sp.out_pitch = out_pitch;
    sp.lse_t = lse;
    sp.gate = p.gate;
    return sp;
}

static int launch_finalize(const FinalizeParams& f, cudaStream_t st) {
    KernelTimer timer(f.gate ? KIND_CONDITIONAL : KIND_FINALIZE, st);
    return launch(finalize_kernel, f.rows, FIN_WARPS * 32, gather_smem(f.d / 8), st, 1, f);
}

// Partial tiles' room of a call: behind the scratch of its row chunks, where the caller says, or (routes without an
// Omega_hat term of their own) in the fp32 rows kept for that term, whichever is larger.
struct PartRoom {
    float* at = nullptr;
    size_t bytes = 0;
};
static PartRoom part_room(uint8_t* ws, size_t workspace_bytes, const Layout& L, int chunk_tiles, const PartRoom* given,
                          bool sparse_free) {
    PartRoom r;
    if (given) r = *given;
    const size_t off = align256(L.fixed_end + L.scratch_row_tile_bytes * chunk_tiles);
    if (!given && workspace_bytes > off) {
        r.at = reinterpret_cast<float*>(ws + off);
        r.bytes = workspace_bytes - off;
    }
    if (sparse_free && L.scratch - L.sparse > r.bytes) {
        r.at = reinterpret_cast<float*>(ws + L.sparse);
        r.bytes = L.scratch - L.sparse;
    }
    return r;
}

// The second GEMM (MODE_OUT) over p.row_tiles row tiles: plan, tiles, and the sum of the partial tiles.
static int launch_out(GemmParams& p, const PartRoom& room, const DeviceInfo& di, cudaStream_t st) {
    const long long left = p.rows_valid - p.row_global_offset;
    const int rows = static_cast<int>(left < static_cast<long long>(p.row_tiles) * BM ? left : p.row_tiles * BM);
    const long long w_bytes = 128ll * p.k_blocks * p.n_cols;
    p.plan = plan_out(rows, p.col_tiles, p.k_blocks, di.sms, room.bytes, di.clusters, w_bytes <= kKeepBytes && p.k_blocks <= kShortBlocks ? p.n_cols : 0);
    p.col_tiles = ceil_div(p.n_cols, p.plan.width);
    if (p.plan.width < BN) p.kept = 1;      // (the instantiation that has such tiles)
    p.part = room.at;
    p.sched.pair = p.plan.pair;
    p.sched.max_ctas = p.plan.groups * p.plan.pair;
    if (kLog)
        std::fprintf(stderr, "[hass] out: pair %d, cluster %d, grid %d, %d whole tiles of %d columns, %d rest tiles x %d cuts\n", p.plan.pair,
                     p.plan.cluster, p.sched.max_ctas, p.plan.whole, p.plan.width, p.plan.rest, p.plan.cuts);
    const int rc = launch_gemm<MODE_OUT>(p, st);
    if (rc != HASS_OK || p.plan.rest == 0) return rc;
    KernelTimer timer(p.gate ? KIND_CONDITIONAL : KIND_OUT, st);
    return launch(out_reduce_kernel, static_cast<long long>(p.plan.rest) * p.plan.pair * (BM * BN / 4 / 256), 256, 0, st, 1, p);
}

// ---- forward ----------------------------------------------------------------------------------
// with_target: both projections + Omega_hat selection; otherwise draft only with Omega_hat given.
static int forward_impl(bool with_target, const void* H_t, const void* H_d, const void* W, long long N, long long d,
                        long long V, int K, const int* idx_in, const float* q_in, float* loss, int* idx_out,
                        float* q_out, float* lse_t, float* lse_d, void* workspace, size_t workspace_bytes,
                        cudaStream_t st) {
    int rc = check_sizes(N, d, V, K);
    if (rc != HASS_OK) return rc;
    if (!H_d || !W || !loss || !lse_d || !aligned16(H_d) || !aligned16(W)) return HASS_ERR_INVALID_ARG;
    if (with_target && (!H_t || !idx_out || !q_out || !lse_t || !aligned16(H_t))) return HASS_ERR_INVALID_ARG;
    if (!with_target && (!idx_in || !q_in)) return HASS_ERR_INVALID_ARG;
    if (!workspace || (reinterpret_cast<uintptr_t>(workspace) & 255u)) return HASS_ERR_WORKSPACE;
    DeviceInfo di;
    rc = device_info(&di);
    if (rc != HASS_OK) return rc;
    rc = get_encode();
    if (rc != HASS_OK) return rc;

    Layout L;
    rc = make_layout(N, d, V, K, di.sms, &L);
    if (rc != HASS_OK) return rc;
    if (workspace_bytes < L.fwd_end) return HASS_ERR_WORKSPACE;
    const int RT = ceil_div(N, BM), CT = ceil_div(V, BN);
    uint8_t* ws = static_cast<uint8_t*>(workspace);
    GemmParams p;
    std::memset(&p, 0, sizeof(p));
    p.row_tiles = with_target ? 2 * RT : RT;
    rc = plan_launch(p.row_tiles, CT, di.sms, L.slot_cap, &p.sched);
    if (rc != HASS_OK) return rc;
    if (with_target) {
        p.row_tiles0 = RT;
        p.topk_row_tiles = RT;
        rc = make_tmap(&p.tmA0, H_t, N, d, d, BK, BM);
        if (rc == HASS_OK) rc = make_tmap(&p.tmA1, H_d, N, d, d, BK, BM);
    } else {
        p.row_tiles0 = RT;
        p.topk_row_tiles = 0;
        rc = make_tmap(&p.tmA0, H_d, N, d, d, BK, BM);
        if (rc == HASS_OK) rc = make_tmap(&p.tmA1, H_d, N, d, d, BK, BM);
    }
    if (rc == HASS_OK) rc = make_tmap(&p.tmB, W, V, d, d, BK, BN / p.sched.pair);
    if (rc != HASS_OK) return rc;
    log_schedule(with_target ? "fwd stats" : "fwd stats (draft)", p.sched);
    p.spill_begin = INT_MAX;
    p.a_row_offset = 0;
    p.row_global_offset = 0;
    p.rows_valid = static_cast<int>(N);
    p.n_cols = static_cast<int>(V);
    p.col_tiles = CT;
    p.k_blocks = ceil_div(d, BK);
    p.K = K;
    p.cap = topk_cap(K);
    p.part_m = reinterpret_cast<float*>(ws + L.part_m);
    p.part_s = reinterpret_cast<float*>(ws + L.part_s);
    p.cand = reinterpret_cast<uint2*>(ws + L.cand_v);
    p.cand_n = reinterpret_cast<int*>(ws + L.cand_i);
    p.status = reinterpret_cast<unsigned int*>(ws + L.status);
    p.thr_share = reinterpret_cast<unsigned int*>(ws + L.thr_share);
    if (with_target) p.bounds = bounds_room(ws, L.fwd_end, workspace_bytes, p.sched, K);
    rc = clear_status(ws, L, p.sched.total_slots, st, false, p.bounds);
    if (rc != HASS_OK) return rc;
    rc = launch_gemm<MODE_STATS>(p, st);
    if (rc != HASS_OK) return rc;
    if (with_target) {
        rc = launch_select(select_params(p, 0, 0, static_cast<int>(N), idx_out, q_out, K, lse_t), di.sms, st);
        if (rc != HASS_OK) return rc;
    }

    FinalizeParams f;
    std::memset(&f, 0, sizeof(f));
    f.sched = p.sched;
    f.row_begin = 0;
    f.rows = static_cast<int>(N);
    f.d = static_cast<int>(d);
    f.K = K;
    f.row_tiles_t = with_target ? RT : 0;
    f.part_m = p.part_m;
    f.part_s = p.part_s;
    f.H_d = static_cast<const __nv_bfloat16*>(H_d);
    f.W = static_cast<const __nv_bfloat16*>(W);
    f.idx = with_target ? idx_out : const_cast<int*>(idx_in);
    f.q = with_target ? q_out : const_cast<float*>(q_in);
    f.idx_pitch = K;
    f.loss = loss;
    f.lse_t = lse_t;
    f.lse_d = lse_d;
    return launch_finalize(f, st);
}

// ---- backward ---------------------------------------------------------------------------------
// The backward of at most 128 rows (below); HASS_ERR_UNSUPPORTED: no room for it.
static int narrow_backward(const void* H_d, const void* W, long long N, long long d, long long V, int K, const int* topk_idx, const float* topk_q,
                           const float* lse_d, const float* grad_loss, void* dH_d, int dH_dtype, uint8_t* ws, size_t workspace_bytes,
                           const Layout& L, const DeviceInfo& di, cudaStream_t st);

static int backward_impl(const void* H_d, const void* W, long long N, long long d, long long V, int K,
                         const int* topk_idx, const float* topk_q, const float* lse_d, const float* grad_loss,
                         void* dH_d, int dH_dtype, void* workspace, size_t workspace_bytes, cudaStream_t st) {
    int rc = check_sizes(N, d, V, K);
    if (rc != HASS_OK) return rc;
    if (!H_d || !W || !topk_idx || !topk_q || !lse_d || !dH_d) return HASS_ERR_INVALID_ARG;
    if (!aligned16(H_d) || !aligned16(W) || !aligned16(dH_d)) return HASS_ERR_INVALID_ARG;
    if (dH_dtype != HASS_BF16 && dH_dtype != HASS_FP32) return HASS_ERR_INVALID_ARG;
    if (!workspace || (reinterpret_cast<uintptr_t>(workspace) & 255u)) return HASS_ERR_WORKSPACE;
    DeviceInfo di;
    rc = device_info(&di);
    if (rc != HASS_OK) return rc;
    rc = get_encode();
    if (rc != HASS_OK) return rc;

    Layout L;
    rc = make_layout(N, d, V, K, di.sms, &L);
    if (rc != HASS_OK) return rc;
    if (workspace_bytes < L.fixed_end + L.scratch_row_tile_bytes) return HASS_ERR_WORKSPACE;
    const int RT = ceil_div(N, BM), CT = ceil_div(V, BN), DT = ceil_div(d, BN);
    long long fit = static_cast<long long>((workspace_bytes - L.fixed_end) / L.scratch_row_tile_bytes);
    int chunk_tiles = L.pref_chunk_tiles;
    if (fit < chunk_tiles) chunk_tiles = even_chunk(static_cast<int>(fit), RT);
    uint8_t* ws = static_cast<uint8_t*>(workspace);
    rc = narrow_backward(H_d, W, N, d, V, K, topk_idx, topk_q, lse_d, grad_loss, dH_d, dH_dtype, ws, workspace_bytes, L, di, st);
    if (rc != HASS_ERR_UNSUPPORTED) return rc;
    const PartRoom part = part_room(ws, workspace_bytes, L, chunk_tiles, nullptr, true);
    int* sidx = reinterpret_cast<int*>(ws + L.sidx);
    float* sgq = reinterpret_cast<float*>(ws + L.sgq);
    float* coef = reinterpret_cast<float*>(ws + L.coef);
    float* lse2 = reinterpret_cast<float*>(ws + L.lse2);
    __nv_bfloat16* P = reinterpret_cast<__nv_bfloat16*>(ws + L.scratch);
    rc = clear_bytes(ws + L.status, 256, st);
    if (rc != HASS_OK) return rc;

    {
        KernelTimer timer(KIND_PREP, st);
        rc = launch(bwd_prep_kernel, ceil_div(N, PREP_WARPS), PREP_WARPS * 32, 0, st, 1, static_cast<int>(N), K, topk_idx, topk_q, lse_d,
                    grad_loss, sidx, sgq, coef, lse2);
    }
    if (rc != HASS_OK) return rc;

    CUtensorMap tmHd, tmWn, tmP;
    rc = make_tmap(&tmHd, H_d, N, d, d, BK, BM);
    if (rc == HASS_OK) rc = make_tmap(&tmWn, W, V, d, d, 64, BK);      // B of dH_d = dz_d W: MN-major boxes
    if (rc == HASS_OK) rc = make_tmap(&tmP, P, static_cast<long long>(chunk_tiles) * BM, V, L.p_pitch, BK, BM);
    if (rc != HASS_OK) return rc;

    for (int t0 = 0; t0 < RT; t0 += chunk_tiles) {
        const int tiles = (RT - t0 < chunk_tiles) ? RT - t0 : chunk_tiles;
        // (1) dz_d tiles of this chunk of rows -> scratch
        GemmParams p;
        std::memset(&p, 0, sizeof(p));
        rc = plan_launch(tiles, CT, di.sms, L.slot_cap, &p.sched);
        if (rc != HASS_OK) return rc;
        log_schedule("bwd dz_d", p.sched);
        p.tmA0 = tmHd;
        p.tmA1 = tmHd;
        rc = make_tmap(&p.tmB, W, V, d, d, BK, BN / p.sched.pair);      // B of z = H W^T: K-major
        if (rc != HASS_OK) return rc;
        p.row_tiles = tiles;
        p.row_tiles0 = tiles;
        p.a_row_offset = t0 * BM;
        p.row_global_offset = t0 * BM;
        p.rows_valid = static_cast<int>(N);
        p.n_cols = static_cast<int>(V);
        p.col_tiles = CT;
        p.k_blocks = ceil_div(d, BK);
        p.K = K;
        p.lse2 = lse2;
        p.coef = coef;
        p.sidx = sidx;
        p.sgq = sgq;
        p.P = P;
        p.p_pitch = L.p_pitch;
        p.status = reinterpret_cast<unsigned int*>(ws + L.status);
        rc = launch_gemm<MODE_PROBS>(p, st);
        if (rc != HASS_OK) return rc;
        // (2) dH_d rows of this chunk = dz_d chunk x W
        GemmParams o;
        std::memset(&o, 0, sizeof(o));
        o.tmA0 = tmP;
        o.tmA1 = tmP;
        o.tmB = tmWn;
        o.row_tiles = tiles;
        o.row_tiles0 = tiles;
        o.a_row_offset = 0;
        o.row_global_offset = t0 * BM;
        o.rows_valid = static_cast<int>(N);
        o.n_cols = static_cast<int>(d);
        o.col_tiles = DT;
        o.k_blocks = ceil_div(V, BK);
        o.K = K;
        o.out = dH_d;
        o.out_fp32 = dH_dtype == HASS_FP32 ? 1 : 0;
        o.out_align32 = ((reinterpret_cast<uintptr_t>(dH_d) | static_cast<uintptr_t>(d * (dH_dtype == HASS_FP32 ? 4 : 2))) & 31u) == 0 ? 1 : 0;
        o.out_pitch = d;
        o.status = p.status;
        rc = launch_out(o, part, di, st);
        if (rc != HASS_OK) return rc;
    }
    return HASS_OK;
}

// ---- fused forward + backward with one sweep over target and draft rows ----------------------------
// The route of the combined objective and of the Bi-directional variant (the plain Top-K call, its _draft form
// and Top-P use fused2_impl below). Per chunk of row tiles: (1) one sweep computes the logits of the chunk's target and draft rows,
// their statistics and Top-K candidates, and spills the draft tiles as 2^(z log2e - ref2) in bf16;
// (2) finalize gives loss, Omega_hat, lse and the per-row scale of the spilled tiles; (3) the second
// GEMM contracts the spilled tiles with W and applies scale and sparse term in its epilogue. No
// logit is computed twice. with_target = false: Omega_hat is an input (aligning steps >= 2).
// Extra buffers and outputs of the combined objective CE(q, p) + w * Top-K (nullptr: Top-K loss alone).
struct Combined {
    float w;               // weight of the Top-K term
    float* loss_ce;        // [N] out: full-vocabulary cross-entropy per row
    float* coef_t;         // [N] scratch: scale of the target spill
    float* T;              // [chunk rows, d] scratch: q W of the chunk's rows
    __nv_bfloat16* Pt;     // [chunk rows, p_pitch] scratch: spill of the target tiles
    size_t end;            // bytes of the caller's workspace
};

// Calls of one row tile, where the logits go through the workspace in fp32 (narrow_impl). Such a call is bound by
// reading W, which this route does twice (both sweeps in one launch, then the second GEMM) instead of three times, with no
// range condition and so no second pass. The sweep does nothing but store its accumulators, and one kernel does the rest of a row:
// with candidate lists and statistics in the sweep's epilogue, a kernel that selects and one that forms dz_d, the last tile's epilogue,
// on its own at the end, took 12 us and the two kernels 25. From a flushed L2 61 rows x 4096 x 32000 take 115 us (154 in that form),
// 100 rows 125 (160), 64 rows x 256 x 1024 30 (45), and Bi-directional calls, which spilled, 35 rows x 4096 x 32000 125 (203), 40 x 64 x 700
// 39 (76). The logits take the scratch and what follows; the partial tiles of the second GEMM take the target's, which are read no
// more by then. A workspace that ends before them takes the other route.
// The second GEMM of such a call reads W again. The L2 (126 MB) would hold the end of the first reading, but that is the last
// k blocks of all columns, and the second reading, which walks the other way, evicts them before it comes to them. So the
// sweep lets this much of W, its last k blocks, into the L2 like any other data and asks that the rest go first: 61 rows x 4096 x 32000
// (262 MB) from a cold L2 129 -> 116 us, 100 rows 137 -> 125. Asking the L2 to hold those blocks longest (evict_last) gave the same, 117
// and 127, but they stayed when the call was over: a pass over 80 MB of the caller's took 26.6 us after a call instead of 21.5.
// From this size of W on the kernels of such a call let the next one's blocks in when they end: blocks that wait beside a
// kernel bound by reading W cost it time (from a flushed L2 61 rows x 4096 x 32000 118.8 -> 114.8 us, 99 draft rows 117.5 -> 112.6, 100 rows
// 129.0 -> 124.9); with a head of 0.5 MB it is the same (64 rows x 256 x 1024 30.3 us early, 30.0 late).
constexpr long long kLateBytes = 16ll << 20;
// Blocks per row of row_split_kernel and 16-byte pieces of it per thread; blocks = 0: row_kernel, a block per row. As few blocks as
// leave a thread four pieces (eight of the longest rows), where all of them are resident at once: a block is a chain of about twenty
// barriers, 7 us and more, so that a second round of them costs as much as row_kernel's longer passes (100 rows x 4096 x 32000 120 us per call
// on row_kernel, 136 as two rounds; 100 rows x 128256 416 and 474). Per call, from row_kernel: 2 rows x 8192 x 128256 655 -> 635 us, 5 rows x
// 4096 x 32000, K = 128 99.5 -> 96, 53 rows x 280 x 2179 combined 29.4 -> 26, 2 rows x 1240 x 7791, K = 85 44 -> 39. With four blocks where one
// or two do, 64 rows x 256 x 1024 22 -> 31; with eight pieces, which 512 threads hold of both rows in 64 registers, 118 rows x 12454
// Bi-directional 111 -> 123.
struct RowSplit {
    int blocks, threads, pieces;
};
static RowSplit row_split(long long N, long long pitch, int K, int sms) {
    // Many short rows: as few threads as hold one, with four maxima or more for each token of the set (two K threads at least). A block
    // takes longer (10 us at 128 threads, 7 at 512), but six of them are resident on an SM (80 registers a thread), three of 256 threads.
    if (N > sms && pitch <= 1024 && K <= 32) return RowSplit{1, 128, 2};
    if (N > sms && pitch <= 2048 && K <= 64) return RowSplit{1, 256, 2};
    for (int c = 1; c <= SPLIT_MAX; c *= 2) {
        const int e = ceil_div(pitch, static_cast<long long>(c) * SPLIT_STEP);
        if (e > (c == SPLIT_MAX ? SPLIT_PIECES : SPLIT_PIECES / 2)) continue;
        if (c * N > sms && e > 1) break;
        return RowSplit{c, SPLIT_THREADS, e > 4 ? SPLIT_PIECES : e > 2 ? 4 : e};
    }
    return RowSplit{0, 0, 0};
}
struct NarrowRoom {
    float* z = nullptr;      // [N, p_pitch], or nullptr: no room
    float* zt = nullptr;     // [N, p_pitch]
    float* dz = nullptr;     // the one of the two that dz_d goes over, which lies first
    PartRoom part;
};
// single: as in narrow_rows; chunked: N rows of a combined call (combined_rows)
static NarrowRoom narrow_room(long long N, long long d, int K, uint8_t* ws, size_t workspace_bytes, const Layout& L, int sms, bool single, bool chunked = false) {
    NarrowRoom r;
    const size_t z = align256(static_cast<size_t>(N) * L.p_pitch * 4);
    if ((chunked || narrow_rows(N, d, L.p_pitch, K, L.pref_chunk_tiles, sms, single)) && workspace_bytes >= L.scratch + 2 * z) {
        float* const a = reinterpret_cast<float*>(ws + L.scratch);
        float* const b = reinterpret_cast<float*>(ws + L.scratch + z);
        const bool split = row_split(N, L.p_pitch, K, sms).blocks != 0;
        r.z = split ? b : a;
        r.zt = split ? a : b;
        r.dz = a;
        r.part.at = b;
        r.part.bytes = workspace_bytes - L.scratch - z;
    }
    return r;
}

// The logits of N rows of H0 and (nullable) of H1 -> z0, z1 [N, p_pitch]; clears the status block (the first chunk of a call).
static int narrow_sweep(const void* H0, const void* H1, const void* W, int N, long long d, long long V, float* z0, float* z1,
                        uint8_t* ws, const Layout& L, const DeviceInfo& di, cudaStream_t st, bool first = true) {
    GemmParams p;
    std::memset(&p, 0, sizeof(p));
    // up to 64 rows each share one row tile (61 rows x 4096 x 32000: 65 us as two row tiles of a CTA pair, 61 as one)
    p.half_tiles = H1 && N <= BM / 2 ? 1 : 0;
    const int RT = ceil_div(N, BM);
    p.row_tiles = H1 && !p.half_tiles ? 2 * RT : RT;
    // One phase in which every CTA (pair) has the same number of columns, in steps of 32: whole tiles dealt out in rounds leave the last one
    // to a third of the SMs with 128256 tokens and most SMs without any below 20000. Per call: 64 rows x 256 x 1024 25.7 -> 22.5 us, 53 rows x
    // 280 x 2179 combined 40 -> 29, 33 draft rows x 4096 x 32000 101.6 -> 95.9, 61 rows x 4096 x 128256 400 -> 388 (what is left there is
    // the rate at which boxes of 128 bytes a row come out of memory, 6.0 of 6.4 TB/s).
    const int pair = p.row_tiles > 1 ? 2 : 1, units = ceil_div(p.row_tiles, pair), lanes = std::max(1, di.sms / pair / units);
    // (192 columns at least where W comes out of memory: the stages of a CTA hold too little of a narrower tile. 3 rows x 3136 x 21829 50 us per call in
    // tiles of 256 on 86 CTAs, 56 in tiles of 160 on 138; from the L2 100 rows x 512 x 5000 33 -> 25)
    p.lane_cols = std::max(ceil_div(L.p_pitch / 32, lanes) * 32, V * d * 2 > kKeepBytes ? 192 : 32);
    p.sched.n_phases = 1;
    p.sched.pair = pair;
    p.sched.ph[0] = Phase{0, units * pair, ceil_div(L.p_pitch, p.lane_cols), 0};
    p.sched.max_ctas = p.sched.total_slots = units * pair * p.sched.ph[0].S;
    log_schedule("narrow sweep", p.sched);
    const int box_rows = p.half_tiles ? BM / 2 : BM;
    int rc = make_tmap(&p.tmA0, H0, N, d, d, BK, box_rows);
    if (rc == HASS_OK) rc = make_tmap(&p.tmA1, H1 ? H1 : H0, N, d, d, BK, box_rows);
    if (rc == HASS_OK) rc = make_tmap(&p.tmB, W, V, d, d, BK, BN / pair);
    if (rc == HASS_OK && p.lane_cols % BN) rc = make_tmap(&p.tmSpill, W, V, d, d, BK, p.lane_cols % BN / pair);
    if (rc != HASS_OK) return rc;
    p.row_tiles0 = RT;
    p.spill_begin = INT_MAX;
    p.z_rows = N;
    p.zt_out = z0;
    p.z_out = z1;
    p.z_pitch = L.p_pitch;
    p.rows_valid = N;
    p.n_cols = static_cast<int>(V);
    p.col_tiles = ceil_div(V, BN);
    p.k_blocks = ceil_div(d, BK);
    p.keep_from = p.k_blocks - static_cast<int>(p.k_blocks * std::min(1., static_cast<double>(kKeepBytes) / (2. * static_cast<double>(V) * static_cast<double>(d))));
    p.status = reinterpret_cast<unsigned int*>(ws + L.status);
    p.clear_status = first ? 1 : 0;
    p.release_late = V * d * 2 >= kLateBytes ? 1 : 0;
    return launch_gemm<MODE_LOGITS>(p, st, H1 ? KIND_STATS : KIND_STATS_DRAFT);
}

static RowParams row_params(int V, int K, const Layout& L) {
    RowParams r;
    std::memset(&r, 0, sizeof(r));
    r.K = K;
    r.V = V;
    r.pitch = L.p_pitch;
    r.idx_pitch = K;
    return r;
}
template <int OBJ>
static int launch_rows_as(RowParams& r, int N, int sms, cudaStream_t st) {
    KernelTimer timer(KIND_FINALIZE, st);
    const RowSplit w = row_split(N, r.pitch, r.K, sms);
    if (w.blocks == 0 && N > sms) return launch(row_kernel<OBJ, ROW_THREADS / 2>, N, ROW_THREADS / 2, 0, st, 1, r);
    if (w.blocks == 0) return launch(row_kernel<OBJ, ROW_THREADS>, N, ROW_THREADS, 0, st, 1, r);
    r.split = w.blocks;
    void (*fn)(RowParams);
    if (w.blocks == 1)
        fn = w.threads == 128   ? row_split_kernel<OBJ, 2, 128, false>
             : w.threads == 256 ? row_split_kernel<OBJ, 2, 256, false>
             : w.pieces == 1    ? row_split_kernel<OBJ, 1, SPLIT_THREADS, false>
             : w.pieces == 2    ? row_split_kernel<OBJ, 2, SPLIT_THREADS, false>
                                : row_split_kernel<OBJ, 4, SPLIT_THREADS, false>;
    else
        fn = w.pieces <= 4 ? row_split_kernel<OBJ, 4, SPLIT_THREADS, true> : row_split_kernel<OBJ, SPLIT_PIECES, SPLIT_THREADS, true>;
    return launch(fn, static_cast<long long>(N) * w.blocks, w.threads, 0, st, w.blocks, r);
}
static int launch_rows(int objective, RowParams& r, int N, int sms, cudaStream_t st) {
    return objective == ROW_COMBINED ? launch_rows_as<ROW_COMBINED>(r, N, sms, st)
           : objective == ROW_BIDIR  ? launch_rows_as<ROW_BIDIR>(r, N, sms, st)
                                     : launch_rows_as<ROW_TOPK>(r, N, sms, st);
}

static int narrow_impl(int objective, bool with_target, const void* H_t, const void* H_d, const void* W, int N, long long d,
                       long long V, int K, const float* grad_loss, const int* idx_in, const float* q_in, float* loss,
                       int* idx_out, float* q_out, float* lse_t, float* lse_d, void* dH_d, int dH_dtype, uint8_t* ws,
                       const Layout& L, const NarrowRoom& room, const DeviceInfo& di, cudaStream_t st, float top_p, int* topk_n,
                       const Combined* cmb = nullptr, const float* lse_in = nullptr, bool first = true) {
    // (1) the logits of the target and draft rows
    int rc = with_target ? narrow_sweep(H_t, H_d, W, N, d, V, room.zt, room.z, ws, L, di, st, first)
                         : narrow_sweep(H_d, nullptr, W, N, d, V, room.z, nullptr, ws, L, di, st, first);
    if (rc != HASS_OK) return rc;
    // (2) statistics, Omega_hat, loss, dz_d
    RowParams r = row_params(static_cast<int>(V), K, L);
    r.z = room.z;
    r.zt = with_target ? room.zt : nullptr;
    r.idx = with_target ? idx_out : const_cast<int*>(idx_in);
    r.q = with_target ? q_out : const_cast<float*>(q_in);
    if (objective == ROW_BIDIR) r.idx_pitch = 2 * K;
    r.top_p = top_p;
    r.n_out = topk_n;
    r.grad_loss = grad_loss;
    r.lse_t = lse_t;
    r.lse_d = lse_d;
    r.loss = loss;
    r.lse_in = lse_in;
    r.make_dz = dH_d != nullptr ? 1 : 0;
    r.release_late = V * d * 2 >= kLateBytes ? 1 : 0;
    if (cmb) {
        r.w = cmb->w;
        r.loss_ce = cmb->loss_ce;
    }
    if (objective != ROW_TOPK) {
        r.W = static_cast<const __nv_bfloat16*>(W);
        r.d = static_cast<int>(d);
        r.coef_out = reinterpret_cast<float*>(ws + L.coef);
        r.sparse_out = reinterpret_cast<float*>(ws + L.sparse);
    }
    r.dz = reinterpret_cast<__nv_bfloat16*>(room.dz);
    rc = launch_rows(objective, r, N, di.sms, st);
    if (rc != HASS_OK) return rc;
    if (dH_d == nullptr) return HASS_OK;      // the forward alone
    // (3) dH_d = dz_d W
    GemmParams o;
    std::memset(&o, 0, sizeof(o));
    rc = make_tmap(&o.tmA0, room.dz, N, V, 2 * L.p_pitch, BK, BM);
    if (rc == HASS_OK) rc = make_tmap(&o.tmB, W, V, d, d, 64, BK);
    if (rc != HASS_OK) return rc;
    o.tmA1 = o.tmA0;
    o.row_tiles = o.row_tiles0 = ceil_div(N, BM);
    o.spill_begin = INT_MAX;
    o.rows_valid = N;
    o.n_cols = static_cast<int>(d);
    o.col_tiles = ceil_div(d, BN);
    o.k_blocks = ceil_div(V, BK);
    o.K = K;
    o.out = dH_d;
    o.out_fp32 = dH_dtype == HASS_FP32 ? 1 : 0;
    o.out_align32 = ((reinterpret_cast<uintptr_t>(dH_d) | static_cast<uintptr_t>(d * (dH_dtype == HASS_FP32 ? 4 : 2))) & 31u) == 0 ? 1 : 0;
    o.out_pitch = d;
    o.kept = N <= BM ? 1 : 0;      // (several row tiles read W side by side)
    o.release_late = r.release_late;
    o.coef = r.coef_out;
    o.sparse = r.sparse_out;
    o.status = reinterpret_cast<unsigned int*>(ws + L.status);
    return launch_out(o, room.part, di, st);
}

// lse_d is given: the draft's logits, dz_d and its product with W, as in the fused call. It replaces the sorted sets and the MODE_PROBS
// sweep, whose epilogue walks them: forward + backward of 11 rows x 3848 x 3306 86 -> 81 us, 61 x 4096 x 32000 163 ->
// 153, 100 x 256 x 1024 45 -> 32.
static int narrow_backward(const void* H_d, const void* W, long long N, long long d, long long V, int K, const int* topk_idx, const float* topk_q,
                           const float* lse_d, const float* grad_loss, void* dH_d, int dH_dtype, uint8_t* ws, size_t workspace_bytes,
                           const Layout& L, const DeviceInfo& di, cudaStream_t st) {
    const NarrowRoom room = narrow_room(N, 0, K, ws, workspace_bytes, L, di.sms, false);      // (the line of narrow features: 592 rows x 4096 x 32000 as two calls 618 -> 628)
    if (!room.z) return HASS_ERR_UNSUPPORTED;
    return narrow_impl(ROW_TOPK, false, nullptr, H_d, W, static_cast<int>(N), d, V, K, grad_loss, topk_idx, topk_q, nullptr, nullptr, nullptr,
                       nullptr, nullptr, dH_d, dH_dtype, ws, L, room, di, st, 0.f, nullptr, nullptr, lse_d);
}

static int fused_impl(bool with_target, const void* H_t, const void* H_d, const void* W, long long N, long long d,
                      long long V, int K, const float* grad_loss, const int* idx_in, const float* q_in, float* loss,
                      int* idx_out, float* q_out, float* lse_t, float* lse_d, void* dH_d, int dH_dtype,
                      void* workspace, size_t workspace_bytes, cudaStream_t st, const Combined* cmb = nullptr,
                      int* topk_n = nullptr, bool bidir = false, const PartRoom* room = nullptr) {
    int rc = check_sizes(N, d, V, K);
    if (rc != HASS_OK) return rc;
    if (!H_d || !W || !loss || !lse_d || !dH_d || !aligned16(H_d) || !aligned16(W) || !aligned16(dH_d))
        return HASS_ERR_INVALID_ARG;
    if (with_target && (!H_t || !idx_out || !q_out || !lse_t || !aligned16(H_t))) return HASS_ERR_INVALID_ARG;
    if (!with_target && (!idx_in || !q_in)) return HASS_ERR_INVALID_ARG;
    if (dH_dtype != HASS_BF16 && dH_dtype != HASS_FP32) return HASS_ERR_INVALID_ARG;
    if (bidir && (!with_target || 2 * K > K_CAP)) return HASS_ERR_UNSUPPORTED;   // the union holds up to 2K tokens
    if (!workspace || (reinterpret_cast<uintptr_t>(workspace) & 255u)) return HASS_ERR_WORKSPACE;
    DeviceInfo di;
    rc = device_info(&di);
    if (rc != HASS_OK) return rc;
    rc = get_encode();
    if (rc != HASS_OK) return rc;
    Layout L;
    rc = make_layout(N, d, V, K, di.sms, &L);
    if (rc != HASS_OK) return rc;
    if (workspace_bytes < L.fixed_end + L.scratch_row_tile_bytes) return HASS_ERR_WORKSPACE;
    const int RT = ceil_div(N, BM), CT = ceil_div(V, BN), DT = ceil_div(d, BN);
    long long fit = static_cast<long long>((workspace_bytes - L.fixed_end) / L.scratch_row_tile_bytes);
    int chunk_tiles = L.pref_chunk_tiles;
    if (fit < chunk_tiles) chunk_tiles = even_chunk(static_cast<int>(fit), RT);
    uint8_t* ws = static_cast<uint8_t*>(workspace);
    const PartRoom part = part_room(ws, workspace_bytes, L, chunk_tiles, room, false);
    float* coef = reinterpret_cast<float*>(ws + L.coef);
    float* sparse = reinterpret_cast<float*>(ws + L.sparse);
    __nv_bfloat16* P = reinterpret_cast<__nv_bfloat16*>(ws + L.scratch);
    unsigned int* status = reinterpret_cast<unsigned int*>(ws + L.status);
    int* idx_d = reinterpret_cast<int*>(ws + L.sidx);
    const long long most = cmb ? std::min<long long>(N, combined_rows(N, V, di.sms)) : 0;
    if (most > 0 && narrow_room(most, d, K, ws, cmb->end, L, di.sms, false, true).z) {
        const size_t dH_row = static_cast<size_t>(d) * (dH_dtype == HASS_FP32 ? 4 : 2);
        for (long long r0 = 0; r0 < N; r0 += most) {
            const int rows = static_cast<int>(std::min(most, N - r0));
            const NarrowRoom narrow = narrow_room(rows, d, K, ws, cmb->end, L, di.sms, false, true);
            Combined c = *cmb;
            c.loss_ce += r0;
            rc = narrow_impl(ROW_COMBINED, true, static_cast<const __nv_bfloat16*>(H_t) + r0 * d, static_cast<const __nv_bfloat16*>(H_d) + r0 * d, W, rows, d, V, K,
                             grad_loss ? grad_loss + r0 : nullptr, nullptr, nullptr, loss + r0, idx_out + r0 * K, q_out + r0 * K, lse_t + r0, lse_d + r0,
                             static_cast<uint8_t*>(dH_d) + r0 * dH_row, dH_dtype, ws, L, narrow, di, st, 0.f, nullptr, &c, nullptr, r0 == 0);
            if (rc != HASS_OK) return rc;
        }
        return HASS_OK;
    }
    // (The combined objective too: 65 rows x 4096 x 32000 247 -> 123 us, 128 rows x 4096 x 128256 764 -> 551, 100 x 256 x 1024 79 -> 25.)
    if (with_target) {
        const NarrowRoom narrow = narrow_room(N, d, K, ws, cmb ? cmb->end : workspace_bytes, L, di.sms, false);
        if (narrow.z)
            return narrow_impl(cmb ? ROW_COMBINED : bidir ? ROW_BIDIR : ROW_TOPK, true, H_t, H_d, W, static_cast<int>(N), d, V, K, grad_loss,
                               nullptr, nullptr, loss, idx_out, q_out, lse_t, lse_d, dH_d, dH_dtype, ws, L, narrow, di, st, 0.f, topk_n, cmb);
    }
    CUtensorMap tmHt, tmHd, tmWn, tmP;
    rc = make_tmap(&tmHd, H_d, N, d, d, BK, BM);
    if (rc == HASS_OK) rc = with_target ? make_tmap(&tmHt, H_t, N, d, d, BK, BM) : make_tmap(&tmHt, H_d, N, d, d, BK, BM);
    if (rc == HASS_OK) rc = make_tmap(&tmWn, W, V, d, d, 64, BK);
    if (rc == HASS_OK) rc = make_tmap(&tmP, P, static_cast<long long>(chunk_tiles) * BM, V, L.p_pitch, BK, BM);
    CUtensorMap tmPt;
    if (rc == HASS_OK && cmb) rc = make_tmap(&tmPt, cmb->Pt, static_cast<long long>(chunk_tiles) * BM, V, L.p_pitch, BK, BM);
    if (rc != HASS_OK) return rc;

    // Every spilling row records its largest logit. If the sweep reports a row beyond the exponent range of its spill
    // (reference from column tile 0), the same sequence runs a second time as conditional launches with each row's
    // reference taken from that record, which no logit of the row can exceed.
    unsigned int* zmax = reinterpret_cast<unsigned int*>(ws + L.zmax);
    rc = clear_bytes(zmax, static_cast<size_t>(2 * RT) * BM * 4, st);
    if (rc != HASS_OK) return rc;
    auto run = [&](bool retry) -> int {
    const unsigned int* gate = retry ? status + 1 : nullptr;
    for (int t0 = 0; t0 < RT; t0 += chunk_tiles) {
        const int tiles = (RT - t0 < chunk_tiles) ? RT - t0 : chunk_tiles;
        const int rows = static_cast<int>((N - static_cast<long long>(t0) * BM < static_cast<long long>(tiles) * BM)
                                              ? N - static_cast<long long>(t0) * BM
                                              : static_cast<long long>(tiles) * BM);
        // (1) logits sweep with statistics, candidates and spill
        GemmParams p;
        std::memset(&p, 0, sizeof(p));
        rc = plan_launch(with_target ? 2 * tiles : tiles, CT, di.sms, L.slot_cap, &p.sched);
        if (rc != HASS_OK) return rc;
        log_schedule("fused stats", p.sched);
        p.tmA0 = tmHt;
        p.tmA1 = tmHd;
        rc = make_tmap(&p.tmB, W, V, d, d, BK, BN / p.sched.pair);      // B of z = H W^T: K-major
        if (rc != HASS_OK) return rc;
        p.row_tiles = with_target ? 2 * tiles : tiles;
        p.row_tiles0 = tiles;
        p.topk_row_tiles = with_target ? (bidir ? 2 * tiles : tiles) : 0;
        p.spill_begin = with_target ? tiles : 0;
        p.a_row_offset = t0 * BM;
        p.row_global_offset = t0 * BM;
        p.rows_valid = static_cast<int>(N);
        p.n_cols = static_cast<int>(V);
        p.col_tiles = CT;
        p.k_blocks = ceil_div(d, BK);
        p.K = K;
        p.cap = topk_cap(K);
        p.part_m = reinterpret_cast<float*>(ws + L.part_m);
        p.part_s = reinterpret_cast<float*>(ws + L.part_s);
        p.cand = reinterpret_cast<uint2*>(ws + L.cand_v);
        p.cand_n = reinterpret_cast<int*>(ws + L.cand_i);
        p.P = P;
        p.Pt = cmb ? cmb->Pt : nullptr;
        p.p_pitch = L.p_pitch;
        p.status = status;
        p.thr_share = reinterpret_cast<unsigned int*>(ws + L.thr_share);
        p.row_zmax = zmax + static_cast<size_t>(with_target ? 2 : 1) * t0 * BM;
        p.use_row_zmax = retry ? 1 : 0;
        p.gate = gate;
        // (finalize's rows take the place of the bounds, so the second pass of a single chunk, which clears nothing, has none)
        if (!retry && with_target) p.bounds = bounds_room(ws, L.sparse, L.scratch, p.sched, K);
        if (!retry || RT > chunk_tiles) {      // (a single chunk's thresholds hold for its second pass too)
            rc = clear_status(ws, L, p.sched.total_slots, st, retry || t0 > 0, p.bounds);
            if (rc != HASS_OK) return rc;
        }
        rc = launch_gemm<MODE_STATS>(p, st);
        if (rc != HASS_OK) return rc;
        if (with_target) {
            rc = launch_select(select_params(p, 0, t0 * BM, rows, idx_out, q_out, bidir ? 2 * K : K, lse_t), di.sms, st);
            if (rc != HASS_OK) return rc;
        }
        if (bidir) {
            // the draft's own K most probable tokens, in descending p
            rc = launch_select(select_params(p, tiles, t0 * BM, rows, idx_d, reinterpret_cast<float*>(ws + L.sgq), K, nullptr),
                               di.sms, st);
            if (rc != HASS_OK) return rc;
        }
        // (2) statistics -> loss, Omega_hat, per-row scale
        FinalizeParams f;
        std::memset(&f, 0, sizeof(f));
        f.sched = p.sched;
        f.d = static_cast<int>(d);
        f.K = K;
        f.row_begin = t0 * BM;
        f.rows = rows;
        f.row_tiles_t = with_target ? tiles : 0;
        f.part_m = p.part_m;
        f.part_s = p.part_s;
        f.H_d = static_cast<const __nv_bfloat16*>(H_d);
        f.W = static_cast<const __nv_bfloat16*>(W);
        f.idx = with_target ? idx_out : const_cast<int*>(idx_in);
        f.q = with_target ? q_out : const_cast<float*>(q_in);
        f.idx_pitch = bidir ? 2 * K : K;
        f.loss = loss;
        f.lse_t = lse_t;
        f.lse_d = lse_d;
        f.grad_loss = grad_loss;
        f.coef_out = coef;
        f.sparse_out = sparse;
        f.n_out = topk_n;
        f.idx_d = bidir ? idx_d : nullptr;
        f.H_t = static_cast<const __nv_bfloat16*>(H_t);
        f.w_topk = cmb ? cmb->w : 1.f;
        f.coef_t_out = cmb ? cmb->coef_t : nullptr;
        f.Pt = cmb ? cmb->Pt : nullptr;
        f.p_pitch = L.p_pitch;
        f.ce_corr_out = reinterpret_cast<float*>(ws + L.lse2);    // [N] floats, otherwise used by the split backward
        f.gate = gate;
        rc = launch_finalize(f, st);
        if (rc != HASS_OK) return rc;
        // (3) dH_d rows of the chunk
        GemmParams o;
        std::memset(&o, 0, sizeof(o));
        if (cmb) {
            // (2b) q W of the chunk's rows from the target spill, then the cross-entropy and its gradient term
            GemmParams t = o;
            t.tmA0 = tmPt;
            t.tmA1 = tmPt;
            t.tmB = tmWn;
            t.row_tiles = tiles;
            t.row_tiles0 = tiles;
            t.spill_begin = INT_MAX;
            t.row_global_offset = 0;
            t.rows_valid = rows;
            t.n_cols = static_cast<int>(d);
            t.col_tiles = DT;
            t.k_blocks = ceil_div(V, BK);
            t.K = K;
            t.coef = cmb->coef_t + static_cast<long long>(t0) * BM;
            t.out = cmb->T;
            t.out_fp32 = 1;
            t.out_align32 = 1;
            t.out_pitch = d;
            t.status = status;
            t.gate = gate;
            rc = launch_out(t, part, di, st);
            if (rc != HASS_OK) return rc;
            {
                KernelTimer timer(retry ? KIND_CONDITIONAL : KIND_FINALIZE, st);
                rc = launch(ce_kernel, ceil_div(rows, 8), 256, 0, st, 1, rows, t0 * BM, static_cast<int>(d),
                            static_cast<const __nv_bfloat16*>(H_d), static_cast<const float*>(cmb->T), static_cast<const float*>(lse_d), grad_loss,
                            reinterpret_cast<const float*>(ws + L.lse2), cmb->loss_ce, sparse, gate);
            }
            if (rc != HASS_OK) return rc;
        }
        o.tmA0 = tmP;
        o.tmA1 = tmP;
        o.tmB = tmWn;
        o.row_tiles = tiles;
        o.row_tiles0 = tiles;
        o.spill_begin = INT_MAX;
        o.a_row_offset = 0;
        o.row_global_offset = t0 * BM;
        o.rows_valid = static_cast<int>(N);
        o.n_cols = static_cast<int>(d);
        o.col_tiles = DT;
        o.k_blocks = ceil_div(V, BK);
        o.K = K;
        o.coef = coef;
        o.sparse = sparse;
        o.out = dH_d;
        o.out_fp32 = dH_dtype == HASS_FP32 ? 1 : 0;
        o.out_align32 = ((reinterpret_cast<uintptr_t>(dH_d) | static_cast<uintptr_t>(d * (dH_dtype == HASS_FP32 ? 4 : 2))) & 31u) == 0 ? 1 : 0;
        o.out_pitch = d;
        o.status = status;
        o.gate = gate;
        rc = launch_out(o, part, di, st);
        if (rc != HASS_OK) return rc;
    }
    return HASS_OK;
    };
    rc = run(false);
    if (rc != HASS_OK) return rc;
    return run(true);
}

// ---- fused forward + backward, Omega_hat known before the draft rows are swept -------------------------
// The route of hass_topk_distill_fwd_bwd, its _draft form and the Top-P variant. Per chunk of row tiles:
// (1) sweep of the chunk's TARGET rows: statistics and Top-K candidates; (2) select_kernel: lse_t, Omega_hat,
// the same set sorted by token id, and ref2; (3) sweep of the chunk's DRAFT rows: statistics, the bf16 spill of
// 2^(z_d log2e - ref2), and z_d at the row's Omega_hat copied out of the accumulator as the sweep passes those
// columns; (4) loss_patch_kernel: lse_d, Eq. 1, the per-row scale, and the Omega_hat term of dz_d subtracted
// from the K spilled entries it concerns; (5) the second GEMM with the row scale in its epilogue. No logit
// is computed twice and no row of W is gathered, so the cost does not depend on K beyond the candidate
// handling of (1). with_target = false: (1) is skipped and (2) only sorts the given Omega_hat.
// Hand-over between two copy streams and the compute stream, used by the host-buffer entry: the rows of a chunk
// are copied to the device while the previous chunk computes, and a chunk's dH_d rows go back to the host while
// the next chunk computes. H_t / H_d / dH_d of fused2_impl are then the device staging buffers.
struct ChunkPipe {
    cudaStream_t h2d, d2h;
    const uint8_t* Ht_host;
    const uint8_t* Hd_host;
    uint8_t* dH_host;
    size_t in_row_bytes, out_row_bytes;
    cudaEvent_t* events;       // pool
    int n_events, used;
    cudaEvent_t next() { return used < n_events ? events[used++] : nullptr; }
};

// Rows [row, row + rows) of H_t, then of H_d, on the inbound copy stream; `st` waits for H_t's here and for H_d's here or,
// with ev_d, where the caller makes it.
static int pipe_in(ChunkPipe* pipe, const void* H_t, const void* H_d, size_t row, size_t rows, cudaStream_t st,
                   cudaEvent_t* ev_d = nullptr) {
    const size_t off = row * pipe->in_row_bytes, bytes = rows * pipe->in_row_bytes;
    cudaEvent_t t = pipe->next(), d = pipe->next();
    if (!t || !d) return HASS_ERR_UNSUPPORTED;
    bool ok = cudaMemcpyAsync(const_cast<uint8_t*>(static_cast<const uint8_t*>(H_t)) + off, pipe->Ht_host + off, bytes,
                              cudaMemcpyHostToDevice, pipe->h2d) == cudaSuccess;
    ok = ok && cudaEventRecord(t, pipe->h2d) == cudaSuccess;
    ok = ok && cudaMemcpyAsync(const_cast<uint8_t*>(static_cast<const uint8_t*>(H_d)) + off, pipe->Hd_host + off, bytes,
                               cudaMemcpyHostToDevice, pipe->h2d) == cudaSuccess;
    ok = ok && cudaEventRecord(d, pipe->h2d) == cudaSuccess;
    ok = ok && cudaStreamWaitEvent(st, t, 0) == cudaSuccess;
    if (ev_d)
        *ev_d = d;
    else
        ok = ok && cudaStreamWaitEvent(st, d, 0) == cudaSuccess;
    if (!ok) {
        cudaGetLastError();
        return HASS_ERR_CUDA;
    }
    return HASS_OK;
}

// Rows [row, row + rows) of dH_d, as `st` leaves them here, on the outbound copy stream.
static int pipe_out(ChunkPipe* pipe, const void* dH_d, size_t row, size_t rows, cudaStream_t st) {
    cudaEvent_t ev = pipe->next();
    if (!ev) return HASS_ERR_UNSUPPORTED;
    const size_t off = row * pipe->out_row_bytes;
    bool ok = cudaEventRecord(ev, st) == cudaSuccess;
    ok = ok && cudaStreamWaitEvent(pipe->d2h, ev, 0) == cudaSuccess;
    ok = ok && cudaMemcpyAsync(pipe->dH_host + off, static_cast<const uint8_t*>(dH_d) + off, rows * pipe->out_row_bytes,
                               cudaMemcpyDeviceToHost, pipe->d2h) == cudaSuccess;
    if (!ok) {
        cudaGetLastError();
        return HASS_ERR_CUDA;
    }
    return HASS_OK;
}

static int fused2_impl(bool with_target, const void* H_t, const void* H_d, const void* W, long long N, long long d,
                       long long V, int K, const float* grad_loss, const int* idx_in, const float* q_in, float* loss,
                       int* idx_out, float* q_out, float* lse_t, float* lse_d, void* dH_d, int dH_dtype,
                       void* workspace, size_t workspace_bytes, cudaStream_t st, float top_p = 0.f,
                       int* topk_n = nullptr, ChunkPipe* pipe = nullptr) {
    int rc = check_sizes(N, d, V, K);
    if (rc != HASS_OK) return rc;
    if (!H_d || !W || !loss || !lse_d || !dH_d || !aligned16(H_d) || !aligned16(W) || !aligned16(dH_d))
        return HASS_ERR_INVALID_ARG;
    if (with_target && (!H_t || !idx_out || !q_out || !lse_t || !aligned16(H_t))) return HASS_ERR_INVALID_ARG;
    if (!with_target && (!idx_in || !q_in)) return HASS_ERR_INVALID_ARG;
    if (dH_dtype != HASS_BF16 && dH_dtype != HASS_FP32) return HASS_ERR_INVALID_ARG;
    if (!workspace || (reinterpret_cast<uintptr_t>(workspace) & 255u)) return HASS_ERR_WORKSPACE;
    DeviceInfo di;
    rc = device_info(&di);
    if (rc != HASS_OK) return rc;
    rc = get_encode();
    if (rc != HASS_OK) return rc;
    Layout L;
    rc = make_layout(N, d, V, K, di.sms, &L);
    if (rc != HASS_OK) return rc;
    if (workspace_bytes < L.fixed_end + L.scratch_row_tile_bytes) return HASS_ERR_WORKSPACE;
    const int RT = ceil_div(N, BM), CT = ceil_div(V, BN), DT = ceil_div(d, BN);
    long long fit = static_cast<long long>((workspace_bytes - L.fixed_end) / L.scratch_row_tile_bytes);
    int chunk_tiles = L.pref_chunk_tiles;
    if (fit < chunk_tiles) chunk_tiles = even_chunk(static_cast<int>(fit), RT);
    uint8_t* ws = static_cast<uint8_t*>(workspace);
    const PartRoom part = part_room(ws, workspace_bytes, L, chunk_tiles, nullptr, true);
    int* sidx = reinterpret_cast<int*>(ws + L.sidx);
    float* sq = reinterpret_cast<float*>(ws + L.sgq);
    float* coef = reinterpret_cast<float*>(ws + L.coef);
    float* capz = reinterpret_cast<float*>(ws + L.capz);
    float* ref2 = reinterpret_cast<float*>(ws + L.lse2);
    const NarrowRoom narrow = narrow_room(N, d, K, ws, workspace_bytes, L, di.sms, !with_target);
    if (narrow.z && (!pipe || N <= BM)) {
        if (pipe) {
            rc = pipe_in(pipe, H_t, H_d, 0, static_cast<size_t>(N), st);
            if (rc != HASS_OK) return rc;
        }
        rc = narrow_impl(ROW_TOPK, with_target, H_t, H_d, W, static_cast<int>(N), d, V, K, grad_loss, idx_in, q_in, loss, idx_out, q_out,
                         lse_t, lse_d, dH_d, dH_dtype, ws, L, narrow, di, st, top_p, topk_n);
        if (rc != HASS_OK || !pipe) return rc;
        return pipe_out(pipe, dH_d, 0, static_cast<size_t>(N), st);
    }
    __nv_bfloat16* P = reinterpret_cast<__nv_bfloat16*>(ws + L.scratch);
    unsigned int* status = reinterpret_cast<unsigned int*>(ws + L.status);
    unsigned int* zmax = reinterpret_cast<unsigned int*>(ws + L.zmax);
    CUtensorMap tmHt, tmHd, tmWn, tmP;
    rc = make_tmap(&tmHd, H_d, N, d, d, BK, BM);
    if (rc == HASS_OK) rc = with_target ? make_tmap(&tmHt, H_t, N, d, d, BK, BM) : make_tmap(&tmHt, H_d, N, d, d, BK, BM);
    if (rc == HASS_OK) rc = make_tmap(&tmWn, W, V, d, d, 64, BK);
    if (rc == HASS_OK) rc = make_tmap(&tmP, P, static_cast<long long>(chunk_tiles) * BM, V, L.p_pitch, BK, BM);
    // the same buffer as the draft sweep's TMA stores see it: boxes of 64 columns x 32 rows, every column up to the pitch
    CUtensorMap tmPst;
    if (rc == HASS_OK) rc = make_tmap(&tmPst, P, static_cast<long long>(chunk_tiles) * BM, L.p_pitch, L.p_pitch, 64, 32);
    if (rc != HASS_OK) return rc;

    // Every spilling row records its largest logit. If a draft sweep reports a row beyond the exponent range of its spill,
    // the steps from the draft sweep on run a second time as conditional launches with each row's exponent taken from that
    // record, which no logit of the row can exceed.
    auto run = [&](bool retry) -> int {
        const unsigned int* gate = retry ? status + 1 : nullptr;
        for (int t0 = 0; t0 < RT; t0 += chunk_tiles) {
            const int tiles = (RT - t0 < chunk_tiles) ? RT - t0 : chunk_tiles;
            const int rows = static_cast<int>((N - static_cast<long long>(t0) * BM < static_cast<long long>(tiles) * BM)
                                                  ? N - static_cast<long long>(t0) * BM
                                                  : static_cast<long long>(tiles) * BM);
            // both sweeps cover `tiles` row tiles and share one schedule
            GemmParams p;
            std::memset(&p, 0, sizeof(p));
            rc = plan_launch(tiles, CT, di.sms, L.slot_cap, &p.sched);
            if (rc != HASS_OK) return rc;
            log_schedule("fused sweep (target / draft)", p.sched);
            rc = make_tmap(&p.tmB, W, V, d, d, BK, BN / p.sched.pair);      // B of z = H W^T: K-major
            if (rc != HASS_OK) return rc;
            p.row_tiles = tiles;
            p.row_tiles0 = tiles;
            p.a_row_offset = t0 * BM;
            p.row_global_offset = t0 * BM;
            p.rows_valid = static_cast<int>(N);
            p.n_cols = static_cast<int>(V);
            p.col_tiles = CT;
            p.k_blocks = ceil_div(d, BK);
            p.K = K;
            p.cap = topk_cap(K);
            p.part_m = reinterpret_cast<float*>(ws + L.part_m);
            p.part_s = reinterpret_cast<float*>(ws + L.part_s);
            p.cand = reinterpret_cast<uint2*>(ws + L.cand_v);
            p.cand_n = reinterpret_cast<int*>(ws + L.cand_i);
            p.thr_share = reinterpret_cast<unsigned int*>(ws + L.thr_share);
            p.p_pitch = L.p_pitch;
            p.status = status;
            p.gate = gate;
            if (!retry) {
                cudaEvent_t ev_d = nullptr;
                if (pipe) {
                    rc = pipe_in(pipe, H_t, H_d, static_cast<size_t>(t0) * BM, static_cast<size_t>(rows), st, &ev_d);
                    if (rc != HASS_OK) return rc;
                }
                if (with_target) p.bounds = bounds_room(ws, L.sparse, L.scratch, p.sched, K);
                rc = clear_status(ws, L, with_target ? p.sched.total_slots : 0, st, t0 > 0, p.bounds);
                if (rc != HASS_OK) return rc;
                if (with_target) {
                    // (1) target rows: statistics + candidates
                    GemmParams t = p;
                    t.tmA0 = tmHt;
                    t.tmA1 = tmHt;
                    t.topk_row_tiles = tiles;
                    t.spill_begin = INT_MAX;
                    rc = launch_gemm<MODE_STATS>(t, st);
                    if (rc != HASS_OK) return rc;
                }
                // (2) Omega_hat of the chunk's rows, and the reference exponent of their spill (reads H_d)
                if (pipe && cudaStreamWaitEvent(st, ev_d, 0) != cudaSuccess) {
                    cudaGetLastError();
                    return HASS_ERR_CUDA;
                }
                SelectParams sp = select_params(p, 0, t0 * BM, rows, idx_out, q_out, K, lse_t);
                sp.from_sweep = with_target ? 1 : 0;
                sp.idx_in = idx_in;
                sp.q_in = q_in;
                sp.n_out = topk_n;
                sp.top_p = top_p;
                sp.sidx = sidx;
                sp.sq = sq;
                sp.H_d = static_cast<const __nv_bfloat16*>(H_d);
                sp.W = static_cast<const __nv_bfloat16*>(W);
                sp.d = static_cast<int>(d);
                sp.V = static_cast<int>(V);
                sp.ref2 = ref2;
                sp.zmax = zmax + static_cast<size_t>(t0) * BM;
                rc = launch_select(sp, di.sms, st);
                if (rc != HASS_OK) return rc;
            }
            // (3) draft rows: statistics, spill, z_d at Omega_hat
            {
                GemmParams q = p;
                q.tmA0 = tmHd;
                q.tmA1 = tmHd;
                q.topk_row_tiles = 0;
                q.spill_begin = 0;
                q.sidx = sidx;
                q.cap_z = capz;
                q.row_ref2 = ref2;
                q.row_zmax = zmax + static_cast<size_t>(t0) * BM;
                q.use_row_zmax = retry ? 1 : 0;
                q.P = P;
                q.tmSpill = tmPst;
                rc = launch_gemm<MODE_STATS>(q, st, KIND_STATS_DRAFT);
                if (rc != HASS_OK) return rc;
            }
            // (4) lse_d, loss, row scale, Omega_hat term into the spill
            LossPatchParams lp;
            std::memset(&lp, 0, sizeof(lp));
            lp.sched = p.sched;
            lp.K = K;
            lp.row_begin = t0 * BM;
            lp.rows = rows;
            lp.part_m = p.part_m;
            lp.part_s = p.part_s;
            lp.sidx = sidx;
            lp.sq = sq;
            lp.cap_z = capz;
            lp.grad_loss = grad_loss;
            lp.loss = loss;
            lp.lse_d = lse_d;
            lp.coef_out = coef;
            lp.P = P;
            lp.p_pitch = L.p_pitch;
            lp.gate = gate;
            {
                KernelTimer timer(retry ? KIND_CONDITIONAL : KIND_FINALIZE, st);
                rc = launch(loss_patch_kernel, ceil_div(rows, 8), 256, 0, st, 1, lp);
            }
            if (rc != HASS_OK) return rc;
            // (5) dH_d rows of the chunk = row scale x (patched spill x W)
            GemmParams o;
            std::memset(&o, 0, sizeof(o));
            o.tmA0 = tmP;
            o.tmA1 = tmP;
            o.tmB = tmWn;
            o.row_tiles = tiles;
            o.row_tiles0 = tiles;
            o.spill_begin = INT_MAX;
            o.a_row_offset = 0;
            o.row_global_offset = t0 * BM;
            o.rows_valid = static_cast<int>(N);
            o.n_cols = static_cast<int>(d);
            o.col_tiles = DT;
            o.k_blocks = ceil_div(V, BK);
            o.K = K;
            o.coef = coef;
            o.out = dH_d;
            o.out_fp32 = dH_dtype == HASS_FP32 ? 1 : 0;
            o.out_align32 = ((reinterpret_cast<uintptr_t>(dH_d) | static_cast<uintptr_t>(d * (dH_dtype == HASS_FP32 ? 4 : 2))) & 31u) == 0 ? 1 : 0;
            o.out_pitch = d;
            o.status = status;
            o.gate = gate;
            rc = launch_out(o, part, di, st);
            if (rc != HASS_OK) return rc;
            if (pipe && !retry) {
                rc = pipe_out(pipe, dH_d, static_cast<size_t>(t0) * BM, static_cast<size_t>(rows), st);
                if (rc != HASS_OK) return rc;
            }
        }
        return HASS_OK;
    };
    rc = run(false);
    if (rc != HASS_OK) return rc;
    return run(true);
}

// ---- forward alone, Omega_hat known before the draft rows are swept -----------------------------------
// hass_topk_distill_fwd and hass_topk_distill_fwd_draft: the sweep of the target rows (statistics, candidates),
// select_kernel, the sweep of the draft rows (statistics and z_d at the row's Omega_hat, copied out of the
// accumulator) and loss_patch_kernel (lse_d, Eq. 1). Nothing is spilled and no row of W is gathered. Needs the
// [N, K] lists of the workspace beyond the statistics; with a workspace that ends before them the older
// single-sweep forward (forward_impl) runs instead.
static int forward2_impl(bool with_target, const void* H_t, const void* H_d, const void* W, long long N, long long d,
                         long long V, int K, const int* idx_in, const float* q_in, float* loss, int* idx_out,
                         float* q_out, float* lse_t, float* lse_d, void* workspace, size_t workspace_bytes,
                         cudaStream_t st) {
    int rc = check_sizes(N, d, V, K);
    if (rc != HASS_OK) return rc;
    if (!H_d || !W || !loss || !lse_d || !aligned16(H_d) || !aligned16(W)) return HASS_ERR_INVALID_ARG;
    if (with_target && (!H_t || !idx_out || !q_out || !lse_t || !aligned16(H_t))) return HASS_ERR_INVALID_ARG;
    if (!with_target && (!idx_in || !q_in)) return HASS_ERR_INVALID_ARG;
    if (!workspace || (reinterpret_cast<uintptr_t>(workspace) & 255u)) return HASS_ERR_WORKSPACE;
    DeviceInfo di;
    rc = device_info(&di);
    if (rc != HASS_OK) return rc;
    rc = get_encode();
    if (rc != HASS_OK) return rc;
    Layout L;
    rc = make_layout(N, d, V, K, di.sms, &L);
    if (rc != HASS_OK) return rc;
    if (workspace_bytes < L.sparse)
        return forward_impl(with_target, H_t, H_d, W, N, d, V, K, idx_in, q_in, loss, idx_out, q_out, lse_t, lse_d,
                            workspace, workspace_bytes, st);
    const int RT = ceil_div(N, BM), CT = ceil_div(V, BN);
    uint8_t* ws = static_cast<uint8_t*>(workspace);
    const NarrowRoom narrow = narrow_room(N, d, K, ws, workspace_bytes, L, di.sms, true);
    if (narrow.z)
        return narrow_impl(ROW_TOPK, with_target, H_t, H_d, W, static_cast<int>(N), d, V, K, nullptr, idx_in, q_in, loss, idx_out, q_out,
                           lse_t, lse_d, nullptr, HASS_BF16, ws, L, narrow, di, st, 0.f, nullptr);
    GemmParams p;
    std::memset(&p, 0, sizeof(p));
    rc = plan_launch(RT, CT, di.sms, L.slot_cap, &p.sched);
    if (rc != HASS_OK) return rc;
    log_schedule("fwd sweep (target / draft)", p.sched);
    rc = make_tmap(&p.tmB, W, V, d, d, BK, BN / p.sched.pair);
    if (rc != HASS_OK) return rc;
    p.row_tiles = RT;
    p.row_tiles0 = RT;
    p.spill_begin = INT_MAX;
    p.rows_valid = static_cast<int>(N);
    p.n_cols = static_cast<int>(V);
    p.col_tiles = CT;
    p.k_blocks = ceil_div(d, BK);
    p.K = K;
    p.cap = topk_cap(K);
    p.part_m = reinterpret_cast<float*>(ws + L.part_m);
    p.part_s = reinterpret_cast<float*>(ws + L.part_s);
    p.cand = reinterpret_cast<uint2*>(ws + L.cand_v);
    p.cand_n = reinterpret_cast<int*>(ws + L.cand_i);
    p.status = reinterpret_cast<unsigned int*>(ws + L.status);
    int* sidx = reinterpret_cast<int*>(ws + L.sidx);
    float* sq = reinterpret_cast<float*>(ws + L.sgq);
    float* capz = reinterpret_cast<float*>(ws + L.capz);
    p.thr_share = reinterpret_cast<unsigned int*>(ws + L.thr_share);
    if (with_target) p.bounds = bounds_room(ws, L.sparse, workspace_bytes, p.sched, K);
    rc = clear_status(ws, L, with_target ? p.sched.total_slots : 0, st, false, p.bounds);
    if (rc != HASS_OK) return rc;
    if (with_target) {
        GemmParams t = p;
        rc = make_tmap(&t.tmA0, H_t, N, d, d, BK, BM);
        if (rc != HASS_OK) return rc;
        t.tmA1 = t.tmA0;
        t.topk_row_tiles = RT;
        rc = launch_gemm<MODE_STATS>(t, st);
        if (rc != HASS_OK) return rc;
    }
    SelectParams sp = select_params(p, 0, 0, static_cast<int>(N), idx_out, q_out, K, lse_t);
    sp.from_sweep = with_target ? 1 : 0;
    sp.idx_in = idx_in;
    sp.q_in = q_in;
    sp.sidx = sidx;
    sp.sq = sq;
    rc = launch_select(sp, di.sms, st);
    if (rc != HASS_OK) return rc;
    {
        GemmParams q = p;
        rc = make_tmap(&q.tmA0, H_d, N, d, d, BK, BM);
        if (rc != HASS_OK) return rc;
        q.tmA1 = q.tmA0;
        q.topk_row_tiles = 0;
        q.sidx = sidx;
        q.cap_z = capz;
        rc = launch_gemm<MODE_STATS>(q, st, KIND_STATS_DRAFT);
        if (rc != HASS_OK) return rc;
    }
    LossPatchParams lp;
    std::memset(&lp, 0, sizeof(lp));
    lp.sched = p.sched;
    lp.K = K;
    lp.row_begin = 0;
    lp.rows = static_cast<int>(N);
    lp.part_m = p.part_m;
    lp.part_s = p.part_s;
    lp.sidx = sidx;
    lp.sq = sq;
    lp.cap_z = capz;
    lp.loss = loss;
    lp.lse_d = lse_d;
    KernelTimer timer(KIND_FINALIZE, st);
    return launch(loss_patch_kernel, ceil_div(N, 8), 256, 0, st, 1, lp);
}

// ---- Normed Top-K variant -----------------------------------------------------------------------------
// Both distributions are renormalised over Omega_hat, so the loss and its gradient involve the draft
// logits on Omega_hat only: one sweep over the TARGET rows (statistics + Top-K), then finalize computes the
// K draft logits per row, the loss and the gradient row directly. No draft sweep, no second GEMM.
static int normed_impl(const void* H_t, const void* H_d, const void* W, long long N, long long d, long long V, int K,
                       const float* grad_loss, float* loss, int* idx_out, float* q_out, int* topk_n, float* lse_t,
                       void* dH_d, int dH_dtype, void* workspace, size_t workspace_bytes, cudaStream_t st) {
    int rc = check_sizes(N, d, V, K);
    if (rc != HASS_OK) return rc;
    if (!H_t || !H_d || !W || !loss || !idx_out || !q_out || !lse_t || !dH_d) return HASS_ERR_INVALID_ARG;
    if (!aligned16(H_t) || !aligned16(H_d) || !aligned16(W) || !aligned16(dH_d)) return HASS_ERR_INVALID_ARG;
    if (dH_dtype != HASS_BF16 && dH_dtype != HASS_FP32) return HASS_ERR_INVALID_ARG;
    if (!workspace || (reinterpret_cast<uintptr_t>(workspace) & 255u)) return HASS_ERR_WORKSPACE;
    DeviceInfo di;
    rc = device_info(&di);
    if (rc != HASS_OK) return rc;
    rc = get_encode();
    if (rc != HASS_OK) return rc;
    Layout L;
    rc = make_layout(N, d, V, K, di.sms, &L);
    if (rc != HASS_OK) return rc;
    if (workspace_bytes < L.fwd_end) return HASS_ERR_WORKSPACE;
    const int RT = ceil_div(N, BM), CT = ceil_div(V, BN);
    uint8_t* ws = static_cast<uint8_t*>(workspace);
    GemmParams p;
    std::memset(&p, 0, sizeof(p));
    const NarrowRoom narrow = narrow_room(N, d, K, ws, workspace_bytes, L, di.sms, true);
    if (narrow.z) {
        rc = narrow_sweep(H_t, nullptr, W, static_cast<int>(N), d, V, narrow.zt, nullptr, ws, L, di, st);
        if (rc != HASS_OK) return rc;
        RowParams r = row_params(static_cast<int>(V), K, L);
        r.zt = narrow.zt;
        r.idx = idx_out;
        r.q = q_out;
        r.n_out = topk_n;
        r.lse_t = lse_t;
        rc = launch_rows(ROW_TOPK, r, static_cast<int>(N), di.sms, st);
        if (rc != HASS_OK) return rc;
    } else {
        rc = plan_launch(RT, CT, di.sms, L.slot_cap, &p.sched);
        if (rc != HASS_OK) return rc;
        log_schedule("normed stats (target)", p.sched);
        rc = make_tmap(&p.tmA0, H_t, N, d, d, BK, BM);
        if (rc == HASS_OK) rc = make_tmap(&p.tmA1, H_t, N, d, d, BK, BM);
        if (rc == HASS_OK) rc = make_tmap(&p.tmB, W, V, d, d, BK, BN / p.sched.pair);
        if (rc != HASS_OK) return rc;
        p.row_tiles = RT;
        p.row_tiles0 = RT;
        p.topk_row_tiles = RT;
        p.spill_begin = INT_MAX;
        p.rows_valid = static_cast<int>(N);
        p.n_cols = static_cast<int>(V);
        p.col_tiles = CT;
        p.k_blocks = ceil_div(d, BK);
        p.K = K;
        p.cap = topk_cap(K);
        p.part_m = reinterpret_cast<float*>(ws + L.part_m);
        p.part_s = reinterpret_cast<float*>(ws + L.part_s);
        p.cand = reinterpret_cast<uint2*>(ws + L.cand_v);
        p.cand_n = reinterpret_cast<int*>(ws + L.cand_i);
        p.status = reinterpret_cast<unsigned int*>(ws + L.status);
        p.thr_share = reinterpret_cast<unsigned int*>(ws + L.thr_share);
        p.bounds = bounds_room(ws, L.fwd_end, workspace_bytes, p.sched, K);
        rc = clear_status(ws, L, p.sched.total_slots, st, false, p.bounds);
        if (rc != HASS_OK) return rc;
        rc = launch_gemm<MODE_STATS>(p, st);
        if (rc != HASS_OK) return rc;
        SelectParams sp = select_params(p, 0, 0, static_cast<int>(N), idx_out, q_out, K, lse_t);
        sp.n_out = topk_n;
        rc = launch_select(sp, di.sms, st);
        if (rc != HASS_OK) return rc;
    }
    NormedParams f;
    f.d = static_cast<int>(d);
    f.K = K;
    f.H_d = static_cast<const __nv_bfloat16*>(H_d);
    f.W = static_cast<const __nv_bfloat16*>(W);
    f.idx = idx_out;
    f.q = q_out;
    f.grad_loss = grad_loss;
    f.loss = loss;
    f.dH = dH_d;
    f.dH_fp32 = dH_dtype == HASS_FP32 ? 1 : 0;
    f.split = normed_split(N, d, K, di.sms);
    KernelTimer timer(KIND_FINALIZE, st);
    return launch(normed_kernel, N * f.split, NORMED_THREADS, normed_smem(d, f.split), st, f.split, f);
}

}  // namespace hass

using namespace hass;

extern "C" {

const char* hass_status_string(int status) {
    switch (status) {
        case HASS_OK: return "HASS_OK";
        case HASS_ERR_INVALID_ARG: return "HASS_ERR_INVALID_ARG";
        case HASS_ERR_UNSUPPORTED: return "HASS_ERR_UNSUPPORTED";
        case HASS_ERR_WORKSPACE: return "HASS_ERR_WORKSPACE";
        case HASS_ERR_CUDA: return "HASS_ERR_CUDA";
        case HASS_ERR_TIMEOUT: return "HASS_ERR_TIMEOUT";
        case HASS_ERR_ARCH: return "HASS_ERR_ARCH";
        case HASS_ERR_RANGE: return "HASS_ERR_RANGE";
        default: return "HASS_ERR_UNKNOWN";
    }
}

int hass_version(void) { return 10600; }

int64_t hass_kernel_launch_count(void) { return g_launches.load(); }

int hass_profile_enable(int on) {
    if (on && g_prof.ev.empty()) {
        g_prof.ev.resize(2 * kMaxRecords);
        g_prof.kind.resize(kMaxRecords);
        for (auto& e : g_prof.ev)
            if (cudaEventCreate(&e) != cudaSuccess) {
                cudaGetLastError();
                g_prof.ev.clear();
                return HASS_ERR_CUDA;
            }
    }
    g_prof.on = on != 0;
    g_prof.n = 0;
    return HASS_OK;
}

int hass_profile_summary(double* ms_by_kind, int64_t* launches_by_kind, int n_kinds) {
    if (!ms_by_kind || !launches_by_kind || n_kinds < NUM_KINDS) return HASS_ERR_INVALID_ARG;
    for (int k = 0; k < n_kinds; ++k) {
        ms_by_kind[k] = 0.0;
        launches_by_kind[k] = 0;
    }
    for (int r = 0; r < g_prof.n; ++r) {
        if (cudaEventSynchronize(g_prof.ev[2 * r + 1]) != cudaSuccess) {
            cudaGetLastError();
            return HASS_ERR_CUDA;
        }
        float ms = 0.f;
        if (cudaEventElapsedTime(&ms, g_prof.ev[2 * r], g_prof.ev[2 * r + 1]) != cudaSuccess) {
            cudaGetLastError();
            return HASS_ERR_CUDA;
        }
        ms_by_kind[g_prof.kind[r]] += ms;
        launches_by_kind[g_prof.kind[r]] += 1;
    }
    g_prof.n = 0;
    return HASS_OK;
}

int hass_topk_distill_workspace_bytes(int64_t N, int64_t d, int64_t V, int32_t K, size_t* bytes) {
    if (!bytes) return HASS_ERR_INVALID_ARG;
    int rc = check_sizes(N, d, V, K);
    if (rc != HASS_OK) return rc;
    Layout L;
    rc = make_layout(N, d, V, K, sm_count_or_default(), &L);
    if (rc != HASS_OK) return rc;
    *bytes = L.total_pref + L.part_bytes;
    return HASS_OK;
}

int hass_topk_distill_fwd(const void* H_t, const void* H_d, const void* W, int64_t N, int64_t d, int64_t V, int32_t K,
                          float* loss, int32_t* topk_idx, float* topk_q, float* lse_t, float* lse_d, void* workspace,
                          size_t workspace_bytes, void* cuda_stream) {
    return forward2_impl(true, H_t, H_d, W, N, d, V, K, nullptr, nullptr, loss, topk_idx, topk_q, lse_t, lse_d,
                         workspace, workspace_bytes, static_cast<cudaStream_t>(cuda_stream));
}

int hass_topk_distill_fwd_draft(const void* H_d, const void* W, int64_t N, int64_t d, int64_t V, int32_t K,
                                const int32_t* topk_idx, const float* topk_q, float* loss, float* lse_d,
                                void* workspace, size_t workspace_bytes, void* cuda_stream) {
    return forward2_impl(false, nullptr, H_d, W, N, d, V, K, topk_idx, topk_q, loss, nullptr, nullptr, nullptr, lse_d,
                         workspace, workspace_bytes, static_cast<cudaStream_t>(cuda_stream));
}

int hass_topk_distill_bwd(const void* H_d, const void* W, int64_t N, int64_t d, int64_t V, int32_t K,
                          const int32_t* topk_idx, const float* topk_q, const float* lse_d, const float* grad_loss,
                          void* dH_d, int dH_dtype, void* workspace, size_t workspace_bytes, void* cuda_stream) {
    return backward_impl(H_d, W, N, d, V, K, topk_idx, topk_q, lse_d, grad_loss, dH_d, dH_dtype, workspace,
                         workspace_bytes, static_cast<cudaStream_t>(cuda_stream));
}

int hass_topk_distill_fwd_bwd(const void* H_t, const void* H_d, const void* W, int64_t N, int64_t d, int64_t V,
                              int32_t K, const float* grad_loss, float* loss, int32_t* topk_idx, float* topk_q,
                              float* lse_t, float* lse_d, void* dH_d, int dH_dtype, void* workspace,
                              size_t workspace_bytes, void* cuda_stream) {
    return fused2_impl(true, H_t, H_d, W, N, d, V, K, grad_loss, nullptr, nullptr, loss, topk_idx, topk_q, lse_t, lse_d,
                       dH_d, dH_dtype, workspace, workspace_bytes, static_cast<cudaStream_t>(cuda_stream));
}

int hass_topk_distill_fwd_bwd_draft(const void* H_d, const void* W, int64_t N, int64_t d, int64_t V, int32_t K,
                                    const int32_t* topk_idx, const float* topk_q, const float* grad_loss, float* loss,
                                    float* lse_d, void* dH_d, int dH_dtype, void* workspace, size_t workspace_bytes,
                                    void* cuda_stream) {
    return fused2_impl(false, nullptr, H_d, W, N, d, V, K, grad_loss, topk_idx, topk_q, loss, nullptr, nullptr, nullptr,
                       lse_d, dH_d, dH_dtype, workspace, workspace_bytes, static_cast<cudaStream_t>(cuda_stream));
}

int hass_variant_distill_fwd_bwd(const void* H_t, const void* H_d, const void* W, int64_t N, int64_t d, int64_t V,
                                 int32_t K, int variant, float param, const float* grad_loss, float* loss,
                                 int32_t* topk_idx, float* topk_q, int32_t* topk_n, float* lse_t, float* lse_d,
                                 void* dH_d, int dH_dtype, void* workspace, size_t workspace_bytes,
                                 void* cuda_stream) {
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
    switch (variant) {
        case HASS_LOSS_TOPK:
            return fused2_impl(true, H_t, H_d, W, N, d, V, K, grad_loss, nullptr, nullptr, loss, topk_idx, topk_q, lse_t,
                               lse_d, dH_d, dH_dtype, workspace, workspace_bytes, st, 0.f, topk_n);
        case HASS_LOSS_TOP_P:
            if (!(param > 0.f)) return HASS_ERR_INVALID_ARG;
            return fused2_impl(true, H_t, H_d, W, N, d, V, K, grad_loss, nullptr, nullptr, loss, topk_idx, topk_q, lse_t,
                               lse_d, dH_d, dH_dtype, workspace, workspace_bytes, st, param, topk_n);
        case HASS_LOSS_BIDIR_TOPK:
            return fused_impl(true, H_t, H_d, W, N, d, V, K, grad_loss, nullptr, nullptr, loss, topk_idx, topk_q, lse_t,
                              lse_d, dH_d, dH_dtype, workspace, workspace_bytes, st, nullptr, topk_n, true);
        case HASS_LOSS_NORMED_TOPK:
            return normed_impl(H_t, H_d, W, N, d, V, K, grad_loss, loss, topk_idx, topk_q, topk_n, lse_t, dH_d, dH_dtype,
                               workspace, workspace_bytes, st);
        default:
            return HASS_ERR_INVALID_ARG;
    }
}

// Buffers appended to the normal workspace by the combined-objective entry.
struct CombinedStage {
    size_t base, coef_t, T, Pt, total, part_bytes;      // base: the normal workspace without the partial tiles, which follow `total`
};
static int combined_stage(int64_t N, int64_t d, int64_t V, int32_t K, CombinedStage* c) {
    Layout L;
    int rc = make_layout(N, d, V, K, sm_count_or_default(), &L);
    if (rc != HASS_OK) return rc;
    c->base = L.total_pref;
    c->part_bytes = L.part_bytes;
    size_t off = align256(c->base);
    c->coef_t = off;
    off = align256(off + static_cast<size_t>(N) * 4);
    c->T = off;
    off = align256(off + static_cast<size_t>(L.pref_chunk_tiles) * BM * d * 4);
    c->Pt = off;
    off = align256(off + L.scratch_row_tile_bytes * L.pref_chunk_tiles);
    c->total = off;
    // (the fp32 logits of a chunk lie from the scratch on, over all of these)
    const long long rows = std::min<long long>(N, combined_rows(N, V, sm_count_or_default()));
    const size_t end = L.scratch + 2 * align256(static_cast<size_t>(rows) * L.p_pitch * 4);
    if (end > c->total + c->part_bytes) c->part_bytes = end - c->total;
    return HASS_OK;
}

int hass_combined_distill_workspace_bytes(int64_t N, int64_t d, int64_t V, int32_t K, size_t* bytes) {
    if (!bytes) return HASS_ERR_INVALID_ARG;
    int rc = check_sizes(N, d, V, K);
    if (rc != HASS_OK) return rc;
    CombinedStage c;
    rc = combined_stage(N, d, V, K, &c);
    if (rc != HASS_OK) return rc;
    *bytes = c.total + c.part_bytes;
    return HASS_OK;
}

int hass_combined_distill_fwd_bwd(const void* H_t, const void* H_d, const void* W, int64_t N, int64_t d, int64_t V,
                                  int32_t K, float w_topk, const float* grad_loss, float* loss_ce, float* loss_topk,
                                  int32_t* topk_idx, float* topk_q, float* lse_t, float* lse_d, void* dH_d,
                                  int dH_dtype, void* workspace, size_t workspace_bytes, void* cuda_stream) {
    int rc = check_sizes(N, d, V, K);
    if (rc != HASS_OK) return rc;
    if (!loss_ce || !(w_topk == w_topk)) return HASS_ERR_INVALID_ARG;
    if (!workspace || (reinterpret_cast<uintptr_t>(workspace) & 255u)) return HASS_ERR_WORKSPACE;
    CombinedStage c;
    rc = combined_stage(N, d, V, K, &c);
    if (rc != HASS_OK) return rc;
    if (workspace_bytes < c.total) return HASS_ERR_WORKSPACE;
    uint8_t* ws = static_cast<uint8_t*>(workspace);
    PartRoom room;
    room.at = reinterpret_cast<float*>(ws + c.total);
    room.bytes = workspace_bytes - c.total;
    Combined cmb;
    cmb.w = w_topk;
    cmb.loss_ce = loss_ce;
    cmb.coef_t = reinterpret_cast<float*>(ws + c.coef_t);
    cmb.T = reinterpret_cast<float*>(ws + c.T);
    cmb.Pt = reinterpret_cast<__nv_bfloat16*>(ws + c.Pt);
    cmb.end = workspace_bytes;
    return fused_impl(true, H_t, H_d, W, N, d, V, K, grad_loss, nullptr, nullptr, loss_topk, topk_idx, topk_q, lse_t,
                      lse_d, dH_d, dH_dtype, workspace, c.base, static_cast<cudaStream_t>(cuda_stream), &cmb, nullptr, false, &room);
}

// Device staging appended to the normal workspace (base bytes; with_part: as hass_topk_distill_workspace_bytes gives
// it, else without the room that calls can do without) by the *_host entry.
struct HostStage {
    size_t base, H_t, H_d, grad, loss, idx, q, lse_t, lse_d, dH, total;
};
static int host_stage(int64_t N, int64_t d, int64_t V, int32_t K, int dH_dtype, bool with_part, HostStage* s) {
    Layout L;
    const int rc = make_layout(N, d, V, K, sm_count_or_default(), &L);
    if (rc != HASS_OK) return rc;
    s->base = L.total_pref + (with_part ? L.part_bytes : 0);
    size_t off = align256(s->base);
    s->H_t = off;
    off = align256(off + static_cast<size_t>(N) * d * 2);
    s->H_d = off;
    off = align256(off + static_cast<size_t>(N) * d * 2);
    s->grad = off;
    off = align256(off + static_cast<size_t>(N) * 4);
    s->loss = off;
    off = align256(off + static_cast<size_t>(N) * 4);
    s->idx = off;
    off = align256(off + static_cast<size_t>(N) * K * 4);
    s->q = off;
    off = align256(off + static_cast<size_t>(N) * K * 4);
    s->lse_t = off;
    off = align256(off + static_cast<size_t>(N) * 4);
    s->lse_d = off;
    off = align256(off + static_cast<size_t>(N) * 4);
    s->dH = off;
    off = align256(off + static_cast<size_t>(N) * d * (dH_dtype == HASS_FP32 ? 4 : 2));
    s->total = off;
    return HASS_OK;
}

int hass_topk_distill_host_workspace_bytes(int64_t N, int64_t d, int64_t V, int32_t K, int dH_dtype, size_t* bytes) {
    if (!bytes || (dH_dtype != HASS_BF16 && dH_dtype != HASS_FP32)) return HASS_ERR_INVALID_ARG;
    int rc = check_sizes(N, d, V, K);
    if (rc != HASS_OK) return rc;
    HostStage s;
    rc = host_stage(N, d, V, K, dH_dtype, true, &s);
    if (rc != HASS_OK) return rc;
    *bytes = s.total;
    return HASS_OK;
}

// Copy streams and events of the host-buffer entry, created on a device's first call (no device memory).
struct HostPipeResources {
    bool ready = false;
    cudaStream_t h2d = nullptr, d2h = nullptr;
    cudaEvent_t events[256];
};
static HostPipeResources g_host_pipe[64];

static int host_pipe_resources(HostPipeResources** out) {
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) {
        cudaGetLastError();
        return HASS_ERR_CUDA;
    }
    HostPipeResources& r = g_host_pipe[dev];
    if (!r.ready) {
        bool ok = cudaStreamCreateWithFlags(&r.h2d, cudaStreamNonBlocking) == cudaSuccess &&
                  cudaStreamCreateWithFlags(&r.d2h, cudaStreamNonBlocking) == cudaSuccess;
        for (int i = 0; ok && i < 256; ++i) ok = cudaEventCreateWithFlags(&r.events[i], cudaEventDisableTiming) == cudaSuccess;
        if (!ok) {
            cudaGetLastError();
            return HASS_ERR_CUDA;
        }
        r.ready = true;
    }
    *out = &r;
    return HASS_OK;
}

int hass_topk_distill_fwd_bwd_host(const void* H_t_host, const void* H_d_host, const void* W, int64_t N, int64_t d,
                                   int64_t V, int32_t K, const float* grad_loss_host, float* loss_host,
                                   int32_t* topk_idx_host, float* topk_q_host, void* dH_d_host, int dH_dtype,
                                   void* workspace, size_t workspace_bytes, void* cuda_stream) {
    int rc = check_sizes(N, d, V, K);
    if (rc != HASS_OK) return rc;
    if (!H_t_host || !H_d_host || !W || !loss_host || !dH_d_host) return HASS_ERR_INVALID_ARG;
    if (dH_dtype != HASS_BF16 && dH_dtype != HASS_FP32) return HASS_ERR_INVALID_ARG;
    if (!workspace || (reinterpret_cast<uintptr_t>(workspace) & 255u)) return HASS_ERR_WORKSPACE;
    HostStage s;
    rc = host_stage(N, d, V, K, dH_dtype, true, &s);
    if (rc == HASS_OK && workspace_bytes < s.total) rc = host_stage(N, d, V, K, dH_dtype, false, &s);
    if (rc != HASS_OK) return rc;
    if (workspace_bytes < s.total) return HASS_ERR_WORKSPACE;
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
    uint8_t* ws = static_cast<uint8_t*>(workspace);
    HostPipeResources* res = nullptr;
    rc = host_pipe_resources(&res);
    if (rc != HASS_OK) return rc;
    const float* grad_dev = nullptr;
    if (grad_loss_host) {
        if (cudaMemcpyAsync(ws + s.grad, grad_loss_host, static_cast<size_t>(N) * 4, cudaMemcpyHostToDevice, st) !=
            cudaSuccess) {
            cudaGetLastError();
            return HASS_ERR_CUDA;
        }
        grad_dev = reinterpret_cast<const float*>(ws + s.grad);
    }
    // The copy streams start after whatever the caller's stream still does with the workspace. The rows of a chunk
    // travel to the device while the previous chunk computes; a chunk's dH_d rows travel back while the next computes.
    ChunkPipe pipe;
    pipe.h2d = res->h2d;
    pipe.d2h = res->d2h;
    pipe.Ht_host = static_cast<const uint8_t*>(H_t_host);
    pipe.Hd_host = static_cast<const uint8_t*>(H_d_host);
    pipe.dH_host = static_cast<uint8_t*>(dH_d_host);
    pipe.in_row_bytes = static_cast<size_t>(d) * 2;
    pipe.out_row_bytes = static_cast<size_t>(d) * (dH_dtype == HASS_FP32 ? 4 : 2);
    pipe.events = res->events;
    pipe.n_events = 256;
    pipe.used = 0;
    cudaEvent_t ev_start = pipe.next();
    if (cudaEventRecord(ev_start, st) != cudaSuccess || cudaStreamWaitEvent(pipe.h2d, ev_start, 0) != cudaSuccess ||
        cudaStreamWaitEvent(pipe.d2h, ev_start, 0) != cudaSuccess) {
        cudaGetLastError();
        return HASS_ERR_CUDA;
    }
    rc = fused2_impl(true, ws + s.H_t, ws + s.H_d, W, N, d, V, K, grad_dev, nullptr, nullptr,
                     reinterpret_cast<float*>(ws + s.loss), reinterpret_cast<int32_t*>(ws + s.idx),
                     reinterpret_cast<float*>(ws + s.q), reinterpret_cast<float*>(ws + s.lse_t),
                     reinterpret_cast<float*>(ws + s.lse_d), ws + s.dH, dH_dtype, workspace, s.base, st, 0.f, nullptr, &pipe);
    if (rc == HASS_ERR_UNSUPPORTED) {
        // more row chunks than events (a very small workspace): one copy in, the call, one copy out
        const size_t hbytes = static_cast<size_t>(N) * d * 2;
        cudaStreamSynchronize(pipe.h2d);
        cudaStreamSynchronize(pipe.d2h);
        if (cudaMemcpyAsync(ws + s.H_t, H_t_host, hbytes, cudaMemcpyHostToDevice, st) != cudaSuccess ||
            cudaMemcpyAsync(ws + s.H_d, H_d_host, hbytes, cudaMemcpyHostToDevice, st) != cudaSuccess) {
            cudaGetLastError();
            return HASS_ERR_CUDA;
        }
        rc = fused2_impl(true, ws + s.H_t, ws + s.H_d, W, N, d, V, K, grad_dev, nullptr, nullptr,
                         reinterpret_cast<float*>(ws + s.loss), reinterpret_cast<int32_t*>(ws + s.idx),
                         reinterpret_cast<float*>(ws + s.q), reinterpret_cast<float*>(ws + s.lse_t),
                         reinterpret_cast<float*>(ws + s.lse_d), ws + s.dH, dH_dtype, workspace, s.base, st);
        if (rc == HASS_OK && cudaMemcpyAsync(dH_d_host, ws + s.dH, static_cast<size_t>(N) * pipe.out_row_bytes,
                                             cudaMemcpyDeviceToHost, st) != cudaSuccess) {
            cudaGetLastError();
            return HASS_ERR_CUDA;
        }
    } else if (rc == HASS_OK) {
        // the caller's stream ends after the last outbound copy
        cudaEvent_t ev_out = pipe.next();
        if (!ev_out || cudaEventRecord(ev_out, pipe.d2h) != cudaSuccess || cudaStreamWaitEvent(st, ev_out, 0) != cudaSuccess) {
            cudaGetLastError();
            cudaStreamSynchronize(pipe.d2h);
        }
    }
    if (rc != HASS_OK) {
        cudaStreamSynchronize(pipe.h2d);
        cudaStreamSynchronize(pipe.d2h);
        return rc;
    }
    bool ok = cudaMemcpyAsync(loss_host, ws + s.loss, static_cast<size_t>(N) * 4, cudaMemcpyDeviceToHost, st) == cudaSuccess;
    if (topk_idx_host)
        ok = ok && cudaMemcpyAsync(topk_idx_host, ws + s.idx, static_cast<size_t>(N) * K * 4, cudaMemcpyDeviceToHost, st) == cudaSuccess;
    if (topk_q_host)
        ok = ok && cudaMemcpyAsync(topk_q_host, ws + s.q, static_cast<size_t>(N) * K * 4, cudaMemcpyDeviceToHost, st) == cudaSuccess;
    if (!ok) {
        cudaGetLastError();
        return HASS_ERR_CUDA;
    }
    // word 1 of the status block: the second pass ran after the chunks' dH_d rows had left; fetch them again
    unsigned int redo = 0;
    ok = cudaMemcpyAsync(&redo, ws + 4, 4, cudaMemcpyDeviceToHost, st) == cudaSuccess;
    rc = hass_check(workspace, cuda_stream);
    cudaStreamSynchronize(pipe.d2h);
    if (rc != HASS_OK) return rc;
    if (!ok) {
        cudaGetLastError();
        return HASS_ERR_CUDA;
    }
    if (redo != 0u &&
        cudaMemcpy(dH_d_host, ws + s.dH, static_cast<size_t>(N) * pipe.out_row_bytes, cudaMemcpyDeviceToHost) != cudaSuccess) {
        cudaGetLastError();
        return HASS_ERR_CUDA;
    }
    return HASS_OK;
}

// ---- forward without a caller-provided workspace -------------------------------------------------
// Scratch of hass_topk_distill_fwd_static: lives in the library's device image, so every GPU that
// loads the library holds these bytes until the process exits.
static __device__ __align__(256) unsigned char g_static_scratch[HASS_STATIC_SCRATCH_MAX_BYTES];
// Device address of g_static_scratch per device. In host code the symbol itself is only a handle
// for the runtime, never a pointer a kernel may use; the address comes from cudaGetSymbolAddress.
static void* g_static_scratch_addr[64] = {nullptr};

int hass_topk_distill_fwd_static_scratch_bytes(int64_t N, int64_t d, int64_t V, int32_t K, size_t* bytes) {
    if (!bytes) return HASS_ERR_INVALID_ARG;
    int rc = check_sizes(N, d, V, K);
    if (rc != HASS_OK) return rc;
    // the forward needs the statistics / candidate part of the workspace layout only
    Layout L;
    rc = make_layout(N, d, V, K, sm_count_or_default(), &L);
    if (rc != HASS_OK) return rc;
    *bytes = L.fwd_end;
    return HASS_OK;
}

int hass_topk_distill_fwd_static(const void* H_t, const void* H_d, const void* W, int64_t N, int64_t d, int64_t V,
                                 int32_t K, float* loss, int32_t* topk_idx, float* topk_q, float* lse_t,
                                 float* lse_d, unsigned int* device_status, void* cuda_stream) {
    int rc = check_sizes(N, d, V, K);
    if (rc != HASS_OK) return rc;
    DeviceInfo di;
    rc = device_info(&di);
    if (rc != HASS_OK) return rc;
    size_t need = 0;
    rc = hass_topk_distill_fwd_static_scratch_bytes(N, d, V, K, &need);
    if (rc != HASS_OK) return rc;
    if (need > HASS_STATIC_SCRATCH_MAX_BYTES) {
        if (kLog)
            std::fprintf(stderr, "[hass] hass_topk_distill_fwd_static: this size needs %zu bytes of scratch, the built-in "
                         "array holds %u; use hass_topk_distill_fwd with a workspace\n", need,
                         HASS_STATIC_SCRATCH_MAX_BYTES);
        return HASS_ERR_UNSUPPORTED;
    }
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) {
        cudaGetLastError();
        return HASS_ERR_CUDA;
    }
    if (!g_static_scratch_addr[dev]) {
        // once per device, with that device current
        void* ptr = nullptr;
        if (cudaGetSymbolAddress(&ptr, g_static_scratch) != cudaSuccess || !ptr) {
            cudaGetLastError();
            return HASS_ERR_CUDA;
        }
        g_static_scratch_addr[dev] = ptr;
    }
    void* scratch = g_static_scratch_addr[dev];
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
    // forward_impl zeroes the status word (the only part of the scratch that must start at zero:
    // every statistic and candidate slot that is read has been written by the same call)
    rc = forward_impl(true, H_t, H_d, W, N, d, V, K, nullptr, nullptr, loss, topk_idx, topk_q, lse_t, lse_d, scratch,
                      HASS_STATIC_SCRATCH_MAX_BYTES, st);
    if (rc != HASS_OK) return rc;
    if (device_status &&
        cudaMemcpyAsync(device_status, scratch, sizeof(unsigned int), cudaMemcpyDeviceToDevice, st) != cudaSuccess) {
        cudaGetLastError();
        return HASS_ERR_CUDA;
    }
    return HASS_OK;
}

int hass_hca_attention_workspace_bytes(size_t* bytes) {
    if (!bytes) return HASS_ERR_INVALID_ARG;
    *bytes = 256;
    return HASS_OK;
}

// CTAs per item of the forward, a cluster, where every item has a CTA of its own: as many as are worth their exchange while all clusters are resident
// at once; 1: no clusters. In half key tiles (0.9 us each): a draft pass counts one, the exchange five. 1 x 1000 positions, 4 / 2 heads, m = 0 18.6 ->
// 14.2 us, 1 x 1829, m = 3 33.0 -> 25.8, 1 x 2435, 2 / 1 heads 40.6 -> 28.3, 1 x 3749 55.2 -> 36.1; 2 x 333, 4 / 2 heads, m = 3 13.2 alone, 14.5 in
// pairs, 5 x 48 8.5 and 12.8.
static int hca_fwd_cluster(int items, int q_tiles, int m, const int* clusters) {
    int best = 1, cost = 2 * q_tiles + m;
    for (int c = 2; c <= MAX_CLUSTER; c *= 2) {
        int with = 0;
        for (int z = 0; z < c; ++z) {
            int j0, j1;
            hca2::tile_share(q_tiles, m, z, c, j0, j1);
            with = std::max(with, 2 * (j1 - j0) + (z + 1 == c ? m : 0));
        }
        if (items > clusters[c] || with + 5 >= cost) continue;
        best = c;
        cost = with + 5;
    }
    return best;
}

int hass_hca_attention_fwd(const void* Q, const void* K_t, const void* V_t, const void* const* K_d,
                           const void* const* V_d, int32_t m, int64_t B, int64_t T, int64_t H, int64_t Hkv, int64_t D,
                           float scale, void* O, float* lse, void* workspace, size_t workspace_bytes,
                           void* cuda_stream) {
    if (!Q || !K_t || !V_t || !O) return HASS_ERR_INVALID_ARG;
    if (m < 0 || m > HASS_HCA_MAX_DRAFTS || (m > 0 && (!K_d || !V_d))) return HASS_ERR_INVALID_ARG;
    if (B < 1 || T < 1 || H < 1 || Hkv < 1 || H % Hkv != 0 || !(scale > 0.f) || !(scale < INFINITY))
        return HASS_ERR_INVALID_ARG;
    if (D != hca::HD) return HASS_ERR_UNSUPPORTED;
    if (B > 65535 || T > (1 << 22) || H > 4096 || B * H * ((T + hca::QT - 1) / hca::QT) > INT_MAX / 2)
        return HASS_ERR_UNSUPPORTED;
    auto misaligned = [](const void* q) { return (reinterpret_cast<uintptr_t>(q) & 15u) != 0; };
    if (misaligned(Q) || misaligned(K_t) || misaligned(V_t) || (reinterpret_cast<uintptr_t>(O) & 31u) != 0)
        return HASS_ERR_INVALID_ARG;
    for (int i = 0; i < m; ++i)
        if (!K_d[i] || !V_d[i] || misaligned(K_d[i]) || misaligned(V_d[i])) return HASS_ERR_INVALID_ARG;
    if (!workspace || workspace_bytes < 256 || (reinterpret_cast<uintptr_t>(workspace) & 255u) != 0)
        return HASS_ERR_WORKSPACE;
    DeviceInfo di;
    int rc = device_info(&di);
    if (rc != HASS_OK) return rc;
    rc = get_encode();
    if (rc != HASS_OK) return rc;
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);

    {
        hca2::Params p;
        std::memset(&p, 0, sizeof(p));
        rc = make_tmap_seq(&p.tmQ, Q, B, T, H * hca2::HD, hca2::QT);
        if (rc == HASS_OK) rc = make_tmap_seq(&p.tmK, K_t, B, T, Hkv * hca2::HD, hca2::KT);
        if (rc == HASS_OK) rc = make_tmap_seq(&p.tmV, V_t, B, T, Hkv * hca2::HD, hca2::KT);
        for (int i = 0; i < m && rc == HASS_OK; ++i) {
            rc = make_tmap_seq(&p.tmKd[i], K_d[i], B, T, Hkv * hca2::HD, hca2::KT);
            if (rc == HASS_OK) rc = make_tmap_seq(&p.tmVd[i], V_d[i], B, T, Hkv * hca2::HD, hca2::KT);
        }
        if (rc != HASS_OK) return rc;
        p.O = static_cast<__nv_bfloat16*>(O);
        p.lse = lse;
        p.B = static_cast<int>(B);
        p.T = static_cast<int>(T);
        p.H = static_cast<int>(H);
        p.Hkv = static_cast<int>(Hkv);
        p.m = m;
        p.q_tiles = static_cast<int>((T + hca2::QT - 1) / hca2::QT);
        // two query heads of one key/value group per CTA when the group size is even, else two query tiles of one head
        // ... or one item per CTA while there are SMs enough: the two slots of a CTA wait for one another's products and
        // exponentials (forward of 1 x 1829 positions, 4 / 2 heads, m = 3: 36.6 -> 33.1 us, 2 x 333 16.3 -> 13.7, 1 x 1000, 8 / 8 heads,
        // m = 0 20.8 -> 18.9, 8 x 100, 2 / 1 heads, m = 5 17.0 -> 14.2)
        p.single = B * H * p.q_tiles <= di.sms ? 1 : 0;
        p.head_pairing = !p.single && (H / Hkv) % 2 == 0 ? 1 : 0;
        p.pairs = p.single ? static_cast<int>(B * H) * p.q_tiles : p.head_pairing ? static_cast<int>(B * (H / 2)) * p.q_tiles : static_cast<int>(B * H) * ((p.q_tiles + 1) / 2);
        p.c2 = scale * 1.4426950408889634f;
        p.status = static_cast<unsigned int*>(workspace);
        p.cluster = p.single ? hca_fwd_cluster(p.pairs, p.q_tiles, m, di.hca_fwd_clusters) : 1;
        const int grid = p.cluster > 1 ? p.pairs * p.cluster : p.pairs < di.sms ? p.pairs : di.sms;
        p.one_round = p.cluster > 1 || p.pairs == grid ? 1 : 0;
        if (!p.one_round) {
            rc = clear_bytes(workspace, 256, st);
            if (rc != HASS_OK) return rc;
        }
        KernelTimer kt(KIND_HCA, st);
        return launch(p.cluster > 1 ? hca2::hca_attention_pair_kernel<true> : hca2::hca_attention_pair_kernel<false>, grid, hca2::NUM_THREADS, hca2::SMEM_BYTES, st, p.cluster, p);
    }
}

// workspace of the HCA backward: status word, D [B, H, T], the fp32 dQ accumulator [B, T, H, 128], and where
// key tiles may be split the fp32 dV and dK (not needed: a workspace that ends before them is used without splitting)
constexpr int64_t kSplitTiles = 2 * 148;      // key tiles up to which splitting them is considered
struct HcaBwdLayout {
    size_t D, dQacc, total, dKVacc;
};
static HcaBwdLayout hca_bwd_layout(int64_t B, int64_t T, int64_t H) {
    HcaBwdLayout L;
    auto up = [](size_t x) { return (x + 255) & ~static_cast<size_t>(255); };
    const size_t rows = static_cast<size_t>(B) * H * T;
    L.D = 256;
    L.dQacc = up(L.D + rows * 4);
    L.dKVacc = L.total = up(L.dQacc + rows * hca::HD * 4);
    return L;
}
static size_t hca_bwd_split_bytes(int64_t tiles) { return static_cast<size_t>(tiles) * 2 * hca_bwd::KEYS * hca::HD * 4; }

// Parts that the backward's key tiles are split in: 2 where the CTA with the most work then has a fifth less of it. Work in elements
// (one head, 64 queries); an item costs about 3 more to start and finish, adding up a tile's dV and dK in fp32 another 4.
// Forward + backward on the device, whole tiles -> halves: 1 x 2048 positions, 32 / 8 heads (128 tiles of 128 down to 8 elements on
// 148 SMs) 270 -> 200 us, 1 x 1000, 64 / 8 heads 257 -> 186, 2 x 1189, 4 / 2 heads 100 -> 84; 1 x 3594, 32 / 8 heads (232 tiles, 5 %
// less work for the longest CTA) 575 -> 603, 4 x 500 (3 % less) 124 -> 130.
static int hca_bwd_parts(int BG, int rep, int T, int sms) {
    const int kt_tiles = ceil_div(T, hca_bwd::KEYS), q_tiles = ceil_div(T, hca_bwd::QE);
    if (kt_tiles < 2 || static_cast<int64_t>(BG) * kt_tiles > kSplitTiles) return 1;
    int most[3] = {0, 0, 0};
    for (int parts = 1; parts <= 2; ++parts) {
        const int items = BG * kt_tiles * parts, G = items < sms ? items : sms;
        for (int c = 0; c < G; ++c) {
            int load = 0;
            for (int k = 0, item; (item = k * G + (k & 1 ? G - 1 - c : c)) < items || k * G < items; ++k) {
                if (item >= items) continue;
                const int n_e = rep * (q_tiles - 2 * (item / parts / BG)), z = item % parts;
                load += n_e * (z + 1) / parts - n_e * z / parts + (parts == 1 ? 3 : 7);
            }
            if (load > most[parts]) most[parts] = load;
        }
    }
    return 6 * most[2] < 5 * most[1] ? 2 : 1;
}

// CTAs per key tile of the backward, a cluster: as many as are worth their exchange where all clusters are resident at once; 1: no clusters. In
// elements (1.35 us each): the exchange costs about four. Forward + backward: 3 x 124 positions, 64 / 8 heads (24 tiles of 16 elements in
// fours) 50.7 -> 42.9 us, 2 x 333, 4 / 2 heads (12 tiles of up to 12, in eights) 42.8 -> 38.5; 4 x 60, 32 / 8 heads (4 elements) 27.8 alone, 31.5 in
// pairs, 8 x 100, 2 / 1 heads 33.1 and 36.3.
static int hca_bwd_cluster(int BG, int rep, int T, const int* clusters) {
    const int kt_tiles = ceil_div(T, hca_bwd::KEYS), most = rep * ceil_div(T, hca_bwd::QE);      // elements of the longest tile
    int best = 1;
    double cost = most;
    for (int c = 2; c <= MAX_CLUSTER; c *= 2) {
        const double with = ceil_div(most, c) + 4.;
        if (static_cast<int64_t>(BG) * kt_tiles > clusters[c] || with >= 0.9 * cost) continue;
        best = c;
        cost = with;
    }
    return best;
}

int hass_hca_attention_bwd_workspace_bytes(int64_t B, int64_t T, int64_t H, int32_t m, size_t* bytes) {
    if (!bytes || B < 1 || T < 1 || H < 1 || m < 0 || m > HASS_HCA_MAX_DRAFTS) return HASS_ERR_INVALID_ARG;
    *bytes = hca_bwd_layout(B, T, H).total;
    const int64_t kt_tiles = (T + hca_bwd::KEYS - 1) / hca_bwd::KEYS;
    if (kt_tiles > 1 && B * kt_tiles <= kSplitTiles) {
        const int64_t tiles = B * H * kt_tiles;      // (the key/value heads are at most the query heads)
        *bytes += hca_bwd_split_bytes(tiles < kSplitTiles ? tiles : kSplitTiles);
    }
    return HASS_OK;
}

int hass_hca_attention_bwd(const void* Q, const void* K_t, const void* V_t, const void* const* K_d,
                           const void* const* V_d, int32_t m, int64_t B, int64_t T, int64_t H, int64_t Hkv, int64_t D,
                           float scale, const void* O, const float* lse, const void* dO, void* dQ, void* dK_t,
                           void* dV_t, void* const* dK_d, void* const* dV_d, void* workspace, size_t workspace_bytes,
                           void* cuda_stream) {
    if (!Q || !K_t || !V_t || !O || !lse || !dO || !dQ || !dK_t || !dV_t) return HASS_ERR_INVALID_ARG;
    if (m < 0 || m > HASS_HCA_MAX_DRAFTS || (m > 0 && (!K_d || !V_d || !dK_d || !dV_d))) return HASS_ERR_INVALID_ARG;
    if (B < 1 || T < 1 || H < 1 || Hkv < 1 || H % Hkv != 0 || !(scale > 0.f) || !(scale < INFINITY))
        return HASS_ERR_INVALID_ARG;
    if (D != hca::HD) return HASS_ERR_UNSUPPORTED;
    if (B > 65535 || T > (1 << 22) || H > 4096 || B * H * ((T + hca::QT - 1) / hca::QT) > INT_MAX / 2)
        return HASS_ERR_UNSUPPORTED;
    auto mis = [](const void* q, uintptr_t a) { return (reinterpret_cast<uintptr_t>(q) & (a - 1)) != 0; };
    if (mis(Q, 16) || mis(K_t, 16) || mis(V_t, 16) || mis(O, 16) || mis(dO, 16) || mis(lse, 4) || mis(dQ, 32) ||
        mis(dK_t, 32) || mis(dV_t, 32))
        return HASS_ERR_INVALID_ARG;
    for (int i = 0; i < m; ++i)
        if (!K_d[i] || !V_d[i] || !dK_d[i] || !dV_d[i] || mis(K_d[i], 16) || mis(V_d[i], 16) || mis(dK_d[i], 16) ||
            mis(dV_d[i], 16))
            return HASS_ERR_INVALID_ARG;
    const HcaBwdLayout L = hca_bwd_layout(B, T, H);
    if (!workspace || workspace_bytes < L.total || mis(workspace, 256)) return HASS_ERR_WORKSPACE;
    DeviceInfo di;
    int rc = device_info(&di);
    if (rc != HASS_OK) return rc;
    rc = get_encode();
    if (rc != HASS_OK) return rc;
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
    uint8_t* ws = static_cast<uint8_t*>(workspace);
    float* Dv = reinterpret_cast<float*>(ws + L.D);
    float* dQacc = reinterpret_cast<float*>(ws + L.dQacc);
    const int iB = static_cast<int>(B), iT = static_cast<int>(T), iH = static_cast<int>(H), iHkv = static_cast<int>(Hkv);
    const float c2 = scale * 1.4426950408889634f;

    hca_bwd::FusedParams k;
    std::memset(&k, 0, sizeof(k));
    rc = make_tmap_seq(&k.tmK, K_t, B, T, Hkv * hca::HD, hca_bwd::KEYS);
    if (rc == HASS_OK) rc = make_tmap_seq(&k.tmV, V_t, B, T, Hkv * hca::HD, hca_bwd::KEYS);
    if (rc == HASS_OK) rc = make_tmap_seq(&k.tmQ, Q, B, T, H * hca::HD, hca_bwd::QE);
    if (rc == HASS_OK) rc = make_tmap_seq(&k.tmdO, dO, B, T, H * hca::HD, hca_bwd::QE);
    if (rc == HASS_OK) {
        // the fp32 accumulator [B, T, H * 128]: boxes of 32 positions x one head's 128 floats, rows as they lie in memory
        cuuint64_t gdim[3] = {static_cast<cuuint64_t>(H * hca::HD), static_cast<cuuint64_t>(T), static_cast<cuuint64_t>(B)};
        cuuint64_t gstride[2] = {gdim[0] * 4, gdim[0] * 4 * gdim[1]};
        cuuint32_t box[3] = {static_cast<cuuint32_t>(hca::HD), 32, 1};
        cuuint32_t estr[3] = {1, 1, 1};
        if (g_encode(&k.tmdQ, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3, dQacc, gdim, gstride, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                     CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_NONE, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
            rc = HASS_ERR_CUDA;
    }
    if (rc != HASS_OK) return rc;

    k.kt_tiles = static_cast<int>((T + hca_bwd::KEYS - 1) / hca_bwd::KEYS);
    int parts = 1;
    if (workspace_bytes >= L.total + hca_bwd_split_bytes(B * Hkv * k.kt_tiles)) parts = hca_bwd_parts(iB * iHkv, iH / iHkv, iT, di.sms);
    const bool split = parts > 1;
    k.cluster = split ? 1 : hca_bwd_cluster(iB * iHkv, iH / iHkv, iT, di.hca_clusters);
    float* dKVacc = reinterpret_cast<float*>(ws + L.dKVacc);
    k.dKVacc = dKVacc;
    {   // D, the substituted entries and everything that follows from them, the start value of the dQ accumulator
        hca_bwd::RowsParams r;
        std::memset(&r, 0, sizeof(r));
        r.Q = static_cast<const __nv_bfloat16*>(Q);
        r.O = static_cast<const __nv_bfloat16*>(O);
        r.dO = static_cast<const __nv_bfloat16*>(dO);
        for (int i = 0; i < m; ++i) {
            r.Kd[i] = static_cast<const __nv_bfloat16*>(K_d[i]);
            r.Vd[i] = static_cast<const __nv_bfloat16*>(V_d[i]);
            r.dKd[i] = static_cast<__nv_bfloat16*>(dK_d[i]);
            r.dVd[i] = static_cast<__nv_bfloat16*>(dV_d[i]);
        }
        r.lse = lse;
        r.D = Dv;
        r.dQacc = dQacc;
        r.dKVacc = dKVacc;
        r.m = m; r.B = iB; r.T = iT; r.H = iH; r.Hkv = iHkv;
        r.c2 = c2;
        r.scale = scale;
        r.status = static_cast<unsigned int*>(workspace);
        KernelTimer kt(KIND_HCA_BWD_ROWS, st);
        const long long halves = static_cast<long long>(B) * T * Hkv;
        r.row_blocks = static_cast<unsigned int>((halves * 16 + 255) / 256);
        rc = launch(H == Hkv ? hca_bwd::hca_bwd_rows_mha_kernel : hca_bwd::hca_bwd_rows_kernel, r.row_blocks + (split ? 2ll * iB * iHkv * k.kt_tiles : 0), 256, 0, st, 1, r);
    }
    if (rc != HASS_OK) return rc;

    k.dK = static_cast<__nv_bfloat16*>(dK_t);
    k.dV = static_cast<__nv_bfloat16*>(dV_t);
    k.lse = lse;
    k.D = Dv;
    k.B = iB; k.T = iT; k.H = iH; k.Hkv = iHkv; k.m = m;
    k.q_tiles64 = static_cast<int>((T + hca_bwd::QE - 1) / hca_bwd::QE);
    k.items = iB * iHkv * k.kt_tiles;
    k.c2 = c2;
    k.scale = scale;
    k.status = static_cast<unsigned int*>(workspace);
    {
        KernelTimer kt(KIND_HCA_BWD_FUSED, st);
        if (k.cluster > 1)
            rc = launch(hca_bwd::hca_bwd_fused_kernel<1, true>, k.items * k.cluster, hca_bwd::NUM_THREADS, hca_bwd::F_SMEM_BYTES, st, k.cluster, k);
        else
            rc = launch(split ? hca_bwd::hca_bwd_fused_kernel<2> : hca_bwd::hca_bwd_fused_kernel<1>, k.items * parts < di.sms ? k.items * parts : di.sms, hca_bwd::NUM_THREADS, hca_bwd::F_SMEM_BYTES, st, 1, k);
    }
    if (rc != HASS_OK) return rc;

    {
        KernelTimer kt(KIND_HCA_DQ_CONVERT, st);
        hca_bwd::ConvertParams c;
        std::memset(&c, 0, sizeof(c));
        c.dQacc = dQacc;
        c.dQ = static_cast<__nv_bfloat16*>(dQ);
        c.n8 = B * T * H * (hca::HD / 8);
        c.dKVacc = split ? dKVacc : nullptr;
        c.dV = k.dV;
        c.dK = k.dK;
        c.B = iB; c.T = iT; c.Hkv = iHkv;
        c.kt_tiles = k.kt_tiles;
        const long long threads = c.n8 + (split ? 2ll * k.items * 16 * hca_bwd::KEYS : 0);
        return launch(hca_bwd::hca_dq_convert_kernel, (threads + 255) / 256, 256, 0, st, 1, c);
    }
}

int hass_selftest_wait_expiry(void* workspace, size_t workspace_bytes, uint64_t limit_ns, void* cuda_stream) {
    if (!workspace || workspace_bytes < 256 || (reinterpret_cast<uintptr_t>(workspace) & 255u)) return HASS_ERR_WORKSPACE;
    if (limit_ns < 1000ull || limit_ns > 100000000ull) return HASS_ERR_INVALID_ARG;      // 1 us .. 100 ms
    DeviceInfo di;
    int rc = device_info(&di);
    if (rc != HASS_OK) return rc;
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
    if (cudaMemsetAsync(workspace, 0, 256, st) != cudaSuccess) {
        cudaGetLastError();
        return HASS_ERR_CUDA;
    }
    unsigned int* words = static_cast<unsigned int*>(workspace);
    wait_expiry_selftest_kernel<<<1, 128, 0, st>>>(words, limit_ns, words + 16);
    g_launches.fetch_add(1);
    return cudaGetLastError() == cudaSuccess ? HASS_OK : HASS_ERR_CUDA;
}

int hass_check(void* workspace, void* cuda_stream) {
    if (!workspace) return HASS_ERR_WORKSPACE;
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
    if (cudaStreamSynchronize(st) != cudaSuccess) {
        cudaGetLastError();
        return HASS_ERR_CUDA;
    }
    unsigned int word = 0;
    if (cudaMemcpy(&word, workspace, 4, cudaMemcpyDeviceToHost) != cudaSuccess) {
        cudaGetLastError();
        return HASS_ERR_CUDA;
    }
    if (word != 0) {
        cudaMemset(workspace, 0, 4);
        if (kLog) std::fprintf(stderr, "[hass] device status word 0x%x\n", word);
        return HASS_ERR_TIMEOUT;
    }
    return HASS_OK;
}

}  // extern "C"

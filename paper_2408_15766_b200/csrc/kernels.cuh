// Device code of the fused LM-head + Top-K distillation path (sm_100a).
//
// One warp-specialised, persistent GEMM kernel (TMA -> shared memory -> tcgen05.mma -> TMEM ->
// epilogue warps) is instantiated with four epilogues:
//   MODE_STATS  logits tile -> per-row softmax statistics, Top-K candidates (two variants: a sorted register
//               list for K <= 16, append buffers with warp-cooperative compaction otherwise) and, in the fused
//               forward+backward, a bf16 spill of 2^(z log2e - ref) that the second GEMM consumes
//   MODE_PROBS  draft logits tile -> dz_d tile = g (S_q p - q [v in Omega_hat]) in bf16 -> scratch
//               (the separate, recomputing backward)
//   MODE_OUT    dH_d tile: coef * acc - Omega_hat row (fused), coef * acc (q W of the combined objective)
//               or the accumulator as is (separate backward)
//   MODE_LOGITS logits tile in fp32, as it is (calls of few rows)
// plus small kernels: out_reduce (partial tiles of MODE_OUT), select (after a sweep with Top-K candidates: lse,
// Omega_hat, the set sorted by token id, the reference exponent of the draft rows' spill), loss_patch (after the draft
// sweep: lse_d, Eq. 1, row scale, the Omega_hat term into the spill), finalize (routes without a draft sweep that
// knows Omega_hat: gathered draft logits, Eq. 1 and its variants, the Omega_hat term of dH_d), ce_kernel (cross-entropy
// of the combined objective) and bwd_prep (index-sorted Top-K lists for MODE_PROBS). row
// (after MODE_LOGITS: all that is done with a row's logits).
// Beside the operand stages the kernel's shared memory holds 32 KB that the epilogue warps use: staging
// buffers for the TMA stores of the spill (draft sweep) or the logits waiting for admission to the register
// Top-K lists (target sweep).
#pragma once
#include <cuda_bf16.h>
#include <float.h>
#include <limits.h>

#include "ptx.cuh"

namespace hass {

constexpr int BM = 128;        // rows per tile (TMEM lanes)
constexpr int BN = 256;        // columns per tile (one UMMA N)
constexpr int BK = 64;         // contraction elements per pipeline stage (128 B of bf16: one swizzle row)
constexpr int UMMA_K = 16;     // contraction elements per tcgen05.mma (bf16)
constexpr int A_STAGE_BYTES = BM * BK * 2;
// CG = CTAs that work on one product (1, or a pair): each holds its own BM rows of A and BN / CG of the tile's columns
// EW = epilogue warps (4 or 8); eight take a stage's room for their staging buffers
__host__ __device__ constexpr int stages(int CG, int EW = 4) { return (CG == 2 ? 6 : 4) - (EW == 8 ? 1 : 0); }
__host__ __device__ constexpr int b_stage_bytes(int CG) { return BN / CG * BK * 2; }
constexpr int OPERAND_BYTES = stages(1) * (A_STAGE_BYTES + b_stage_bytes(1));
static_assert(OPERAND_BYTES == stages(2) * (A_STAGE_BYTES + b_stage_bytes(2)), "both forms use the same shared memory");
constexpr int NUM_THREADS = 192;   // warp 0: TMA, warp 1: MMA + TMEM owner, warps 2-5: epilogue
__host__ __device__ constexpr int gemm_threads(int EW) { return 64 + 32 * EW; }
constexpr int TMEM_COLS = 512;     // two accumulator buffers of BN fp32 columns
constexpr int MAX_PHASES = 48;
constexpr int K_CAP = 256;         // == HASS_K_MAX
constexpr int SPILL_STAGE_BYTES = 32 * 128;   // 32 rows x 64 bf16 of a spilled tile on their way to global memory
constexpr int SPILL_STAGES = 2;               // per epilogue warp
constexpr int SMEM_BYTES = OPERAND_BYTES + 4 * SPILL_STAGES * SPILL_STAGE_BYTES +
                           1024 /*alignment slack*/ + 256 /*barriers*/;
__host__ __device__ constexpr int operand_bytes(int CG, int EW) { return stages(CG, EW) * (A_STAGE_BYTES + b_stage_bytes(CG)); }
__host__ __device__ constexpr int gemm_smem(int CG, int EW) { return operand_bytes(CG, EW) + EW * SPILL_STAGES * SPILL_STAGE_BYTES + 1024 + 256; }
static_assert(gemm_smem(1, 4) == SMEM_BYTES && gemm_smem(2, 4) == SMEM_BYTES && gemm_smem(2, 8) <= SMEM_BYTES && gemm_smem(1, 8) <= SMEM_BYTES, "shared memory of a CTA");
// Staging buffers of an epilogue warp (half: of eight warps, which columns of a tile it takes; quad: which rows) and a thread's column of the pending
// logits, in bytes of the staging area
__host__ __device__ constexpr int stage_at(int half, int quad) { return (4 * half + quad) * SPILL_STAGES * SPILL_STAGE_BYTES; }
__host__ __device__ constexpr int pending_at(int thread) { return (thread - 64) * 4; }
// Eight epilogue warps: where the second thread of a row (128 threads behind the first) leaves word e of its statistics and its list for the first.
// With a register list (`list`) that is the first thread's column of the pending logits; without one (two words) the first staging buffer of the
// first thread's warp. Either way the next tile's values go there from the threads that read the words, not from another warp's.
__host__ __device__ constexpr int meet_word(bool list, int thread, int e) {
    const int first = 64 + (thread - 64) % 128;
    return list ? pending_at(first) + e * 256 * 4 : stage_at(0, first / 32 % 4) + e * 128 + first % 32 * 4;
}
constexpr float LOG2E = 1.4426950408889634f;
// A lane's sum of a spilling row's values 2^(z log2e - ref2), ref2 = z_ref log2e + 64, from which on the call is done again
// with the row's largest logit as z_ref: a logit 90 above z_ref (natural units). The sum leaves fp32 only at 131, but what
// depends on it does so earlier: the row scale g S_q / sum of the spill is denormal from g S_q < 1e-38 sum on, and q sum /
// (g S_q) overflows likewise. With 1e20 both hold for g S_q down to 1e-18.
constexpr float SPILL_SUM_LIMIT = 1e20f;

enum { MODE_STATS = 0, MODE_PROBS = 1, MODE_OUT = 2, MODE_LOGITS = 3 };

// A phase gives G consecutive row tiles S "lanes" each; lane l of a row tile sweeps the column
// tiles l, l + S, l + 2S, ... CTA b < G * S works on row tile row_tile_begin + b / S, lane b % S, and
// owns partial-result slot slot_base + b. All CTAs of a phase walk the column tiles in lockstep,
// so a column tile of B is fetched from HBM once and then served from L2 to the G row tiles.
// With CTA pairs (pair = 2) G is even and pair b < G / 2 * S works on row tiles row_tile_begin + 2 (b / S) + {0, 1}, lane
// b % S; slots are numbered as before (row tile by row tile, S each). The last row tile of an odd number has a partner
// beyond the matrix, whose CTA takes part in the products and writes nothing.
struct Phase {
    int row_tile_begin, G, S, slot_base;
};
struct Schedule {
    int n_phases;
    int total_slots;
    int max_ctas;          // largest G * S over the phases = grid size
    int pair;              // CTAs per product: 1 or 2
    Phase ph[MAX_PHASES];
};

// How MODE_OUT divides its output tiles (row tiles, or pairs of them, x column tiles of BN) over the `groups` CTAs or
// pairs of the grid. Tile u = (row u % row_units, column tile u / row_units): the column tile's part of B is read by all
// rows at about the same time. Tiles [0, whole) go out round by round, each contracted to its end; the last `rest`
// tiles, which would leave most of a round idle, are cut into `cuts` equal pieces of the contraction that are dealt
// out the same way (piece v = piece index v / rest of tile whole + v % rest: pieces at the same depth run together), stored as
// fp32 partial tiles and added up by out_reduce_kernel. cuts = 1: whole = all tiles, rest = 0.
// cluster > 1 (then pair = 1): every tile is one cluster's, whose CTAs take equal pieces of the contraction, hand their
// accumulators to one another through distributed shared memory by rows, and add up and finish 128 / cluster rows each.
struct OutPlan {
    int pair, groups, row_units, whole, rest, cuts;
    int part_rows;         // rows kept of a partial tile: BM, or all there are in a single row tile
    int cluster;
    int width;             // columns of a tile: BN, or 128 or 64 of a cluster's (then GemmParams::kept)
};

// A cluster of C CTAs finishes `rows` rows of a tile, piece_rows(rows, C) each: the CTA that finishes row r. (Rows of the tile that do not exist
// belong to the last CTA: an address in a CTA beyond the cluster is undefined even where nothing is stored to it.)
__host__ __device__ constexpr int piece_rows(int rows, int C) { return (rows + C - 1) / C; }
__host__ __device__ constexpr int piece_rank(int r, int per, int C) { return r / per < C ? r / per : C - 1; }

struct GemmParams {
    CUtensorMap tmA0, tmA1, tmB;   // boxes: 128 rows of A; of B the BN / pair columns that one CTA holds
    CUtensorMap tmSpill;   // MODE_STATS without Top-K lists (the draft sweep): the spill P as [chunk rows, p_pitch] bf16 with
                           // boxes of 64 columns x 32 rows, 128-byte swizzle, for TMA stores. MODE_LOGITS: B with boxes of the
                           // lane's last, narrower tile
    Schedule sched;
    int row_tiles;         // row tiles of this launch; a pair's second tile may lie beyond
    int half_tiles;        // MODE_LOGITS, single CTAs: the one row tile is 64 rows of A0 and 64 of A1, boxes of 64 rows; a
                           // sweep of both that reads every tile of B once per call
    int row_tiles0;        // row tiles [0, row_tiles0) read A0, the others A1 (tile index - row_tiles0)
    int topk_row_tiles;    // leading row tiles whose rows collect Top-K candidates (MODE_STATS)
    int a_row_offset;      // added to A0's row coordinate (chunked backward)
    int row_global_offset; // global row number of local row 0 (per-row inputs / outputs)
    int rows_valid;        // global rows >= rows_valid are padding
    int n_cols;            // extent of the tile-column dimension (V, or d for MODE_OUT)
    int col_tiles;
    int k_blocks;          // ceil(contraction extent / BK)
    int K;                 // Top-K
    int cap;               // capacity of a (row, slot) candidate buffer: cand_cap(K)
    int spill_begin;       // MODE_STATS: row tiles >= spill_begin also write the tile 2^(z log2e - ref2) in bf16 to
                           // P (row tile index - spill_begin); INT_MAX: none
    const float* row_ref2; // MODE_STATS, spilling rows: [N] reference exponents, or nullptr: from column tile 0
    // MODE_STATS outputs (per slot)
    float* part_m;
    float* part_s;
    uint2* cand;           // [slot, row, cap] (logit bits, token id)
    int* cand_n;           // [slot, row] entries in use
    unsigned int* thr_share;   // [slot, row] what a lane publishes to the others of its row tile, as an ordered key (zeroed before the
                           // sweep: nothing yet): a bound that K of its logits reach
    uint2* bounds;         // TOPK_BUF, nullable: [slot, row] the same with room for two (zeroed likewise): x = that bound, y = one that
                           // lane_share(K, S) of its logits reach. Without it lanes do not share their bounds
    // MODE_PROBS
    const float* lse2;     // [N] lse_d * log2(e)
    const float* coef;     // [N] g * S_q
    const int* sidx;       // [N, K] Omega_hat sorted by token id
    const float* sgq;      // [N, K] g * q in the same order
    float* cap_z;          // MODE_STATS, TOPK_NONE: [N, K] out, z_d at the tokens of sidx (same order); slots of
                           // padding entries (token id INT_MAX) are left untouched
    __nv_bfloat16* P;      // [chunk rows, p_pitch]
    __nv_bfloat16* Pt;     // [chunk rows, p_pitch] spill of the target tiles, or nullptr
    long long p_pitch;
    // MODE_LOGITS: the logits of the first z_rows rows of A0 (zt_out) and of A1 (z_out) in fp32, [z_rows, z_pitch], -inf
    // beyond n_cols. A0's row tiles come before A1's; with a single row tile that is not halved its matrix is A0
    int z_rows;
    float* z_out;
    float* zt_out;
    long long z_pitch;
    int lane_cols;         // lane l sweeps the columns [l lane_cols, (l + 1) lane_cols) below z_pitch, in tiles of BN and a
                           // narrower last one (a multiple of 32)
    int keep_from;         // k block from which on the L2 holds this sweep's tiles of B like any other's; those before it go first ...
    int kept;              // MODE_OUT: ... as all do in the second reading of B, which this is (host: selects the instantiation, which also has
                           // narrower tiles)
    int release_late;      // the next kernel's blocks may start when this one's have ended, not before
    int clear_status;      // the first CTA zeroes the status block (no kernel of the call has run before this one)
    // MODE_OUT. With sparse != nullptr the epilogue computes coef[row] * acc - sparse[local row, :] (row scale
    // and the Omega_hat term of dz_d W, precomputed by finalize); with coef alone coef[row] * acc; with neither
    // it stores the accumulator.
    const float* sparse;   // [chunk rows, out_pitch]
    void* out;
    int out_fp32;
    int out_align32;       // out base and row pitch are multiples of 32 bytes (256-bit stores allowed)
    long long out_pitch;   // elements
    unsigned int* status;
    OutPlan plan;
    float* part;           // [cuts][rest][pair][part_rows][BN] partial tiles
    const unsigned int* gate;            // nullptr, or: run only if this word (the range report, status[1]) is not zero
    // Every spilling row leaves the ordered key of its largest logit in row_zmax[row tile * 128 + row] (atomicMax over the
    // lanes of the row tile; zeroed before the sweep). A second sweep with use_row_zmax = 1 takes the row's fixed exponent
    // from there, so that no logit of the row can exceed it.
    unsigned int* row_zmax;              // nullable
    int use_row_zmax;
};

// MODE_STATS: does this row tile also write its tiles 2^(z log2e - ref2) as bf16? Draft tiles from spill_begin
// on go to P; with Pt set, the target tiles (the leading topk_row_tiles) go to Pt (combined objective).
__device__ __forceinline__ bool spills(const GemmParams& p, int rt) {
    return rt >= p.spill_begin || (p.Pt != nullptr && rt < p.topk_row_tiles);
}

__device__ __forceinline__ float ex2(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

__device__ __forceinline__ uint32_t pack_bf16x2(float a, float b) {
    __nv_bfloat162 v = __floats2bfloat162_rn(a, b);
    return *reinterpret_cast<uint32_t*>(&v);
}

// ---- streaming Top-K candidates ---------------------------------------------------------------------
// Each (row, slot) owns a buffer of `cap` (logit, token id) pairs in the workspace. The epilogue thread of
// the row appends every logit above its admission threshold; when a buffer is nearly full the whole warp
// compacts it to the row's K best and raises the threshold to the K-th largest logit. Entries stay in
// increasing token-id order, admission is strict (x > threshold), and among logits equal to the K-th the
// lowest token ids are kept, so equal logits resolve to the lower token id.
constexpr int CAND_CAP_MAX = 800;                 // largest buffer: K = 256
constexpr int CAND_REGS = CAND_CAP_MAX / 32;      // entries per lane during a compaction of the largest buffer
constexpr int CAND_REGS_SMALL = 13;               // ... of a buffer of up to 416 entries (K <= 128)
constexpr int CAND_REGS_TINY = 7;                 // ... of up to 224 entries (K <= 64)
constexpr int CAND_SLACK = 32;                    // a compaction may leave up to K + CAND_SLACK entries

// K entries kept + room for max(2K, 96) new ones between compactions (each compaction then multiplies the
// number of columns a threshold has seen by about three) + the 32 entries before the end at which a
// compaction is triggered; a multiple of 32
__host__ __device__ constexpr int cand_cap(int K) { return (K + (2 * K > 96 ? 2 * K : 96) + 32 + 31) / 32 * 32; }

// order-preserving map from fp32 bit patterns to unsigned integers (and back); 0 is below every float
__device__ __forceinline__ uint32_t ordered_key(uint32_t bits) {
    return (bits & 0x80000000u) ? ~bits : (bits | 0x80000000u);
}
__device__ __forceinline__ uint32_t key_bits(uint32_t key) {
    return (key & 0x80000000u) ? (key ^ 0x80000000u) : ~key;
}

// Warp-collective: the n entries of a buffer of `cap`, entry e = lane + 32 t in v[t].
template <int REGS>
__device__ __forceinline__ void load_candidates(const uint2* buf, int n, int cap, int lane, uint2 (&v)[REGS]) {
    const int groups = cap >> 5;
#pragma unroll
    for (int t = 0; t < REGS; ++t) {
        const int e = lane + 32 * t;
        v[t] = make_uint2(0u, 0u);
        if (t < groups && e < n) v[t] = __ldcg(buf + e);
    }
}

// Warp-collective: compacts the buffer `buf`, whose n > K + CAND_SLACK entries are in v, in place, keeping their order, and
// returns the bit pattern of the new admission threshold (only logits strictly above it can still belong to
// the row's K best); n_out = entries left. The bits of the K-th largest key are searched from the highest one in which the
// keys differ, two per step (three counts, whose warp sums overlap), until at most K + CAND_SLACK entries reach the
// prefix found so far: all of them are kept and the threshold is the value just below the prefix. If the search has to run
// to the last bit (equal logits), exactly K entries are kept (among logits equal to the K-th, the lowest token
// ids) and the threshold is the K-th largest logit itself.
template <int REGS>
__device__ __forceinline__ uint32_t compact_candidates(uint2* buf, const uint2 (&v)[REGS], int n, int K, int cap, int lane, int& n_out) {
    uint32_t key[REGS];
    const int groups = cap >> 5;
    uint32_t hi = 0u, lo = 0xffffffffu;
#pragma unroll
    for (int t = 0; t < REGS; ++t) {
        const bool used = t < groups && lane + 32 * t < n;
        key[t] = used ? ordered_key(v[t].x) : 0u;
        hi = max(hi, key[t]);
        lo = used ? min(lo, key[t]) : lo;
    }
    hi = __reduce_max_sync(0xffffffffu, hi);
    lo = __reduce_min_sync(0xffffffffu, lo);
    // largest T with at least K keys >= T; the bits above `bit` are common to all keys
    int bit = 32 - __clz(hi ^ lo);      // bits left to find
    bit += bit & 1;
    uint32_t T = bit < 32 ? (hi >> bit) << bit : 0u;
    bool exact = true;
#pragma unroll 1
    for (bit -= 2; bit >= 0; bit -= 2) {
        const uint32_t T1 = T | (1u << bit), T2 = T | (2u << bit), T3 = T | (3u << bit);
        int c1 = 0, c2 = 0, c3 = 0;
#pragma unroll
        for (int t = 0; t < REGS; ++t) {
            c1 += (key[t] >= T1) ? 1 : 0;
            c2 += (key[t] >= T2) ? 1 : 0;
            c3 += (key[t] >= T3) ? 1 : 0;
        }
        c1 = __reduce_add_sync(0xffffffffu, c1);
        c2 = __reduce_add_sync(0xffffffffu, c2);
        c3 = __reduce_add_sync(0xffffffffu, c3);
        const int c = c3 >= K ? c3 : c2 >= K ? c2 : c1 >= K ? c1 : INT_MAX;
        T = c3 >= K ? T3 : c2 >= K ? T2 : c1 >= K ? T1 : T;
        if (c <= K + CAND_SLACK && bit > 0) {
            exact = false;
            break;
        }
    }
    const uint32_t lt_mask = (1u << lane) - 1u;
    int out = 0;
    if (!exact) {
        // keep every entry that reaches the prefix
#pragma unroll
        for (int t = 0; t < REGS; ++t) {
            if (t < groups) {
                const bool keep = key[t] >= T;
                const uint32_t km = __ballot_sync(0xffffffffu, keep);
                if (keep) buf[out + __popc(km & lt_mask)] = v[t];
                out += __popc(km);
            }
        }
        n_out = out;
        return key_bits(T - 1u);      // T > 0: fewer than n keys reach it
    }
    int n_gt = 0;
#pragma unroll
    for (int t = 0; t < REGS; ++t) n_gt += (key[t] > T) ? 1 : 0;
    n_gt = __reduce_add_sync(0xffffffffu, n_gt);
    const int need_eq = K - n_gt;             // >= 1: how many entries equal to the K-th are kept
    int run_eq = 0;
#pragma unroll
    for (int t = 0; t < REGS; ++t) {
        if (t < groups) {
            const bool eq = key[t] == T;
            const uint32_t em = __ballot_sync(0xffffffffu, eq);
            const bool keep = key[t] > T || (eq && run_eq + __popc(em & lt_mask) < need_eq);
            run_eq += __popc(em);
            const uint32_t km = __ballot_sync(0xffffffffu, keep);
            if (keep) buf[out + __popc(km & lt_mask)] = v[t];
            out += __popc(km);
        }
    }
    n_out = out;
    return key_bits(T);
}

// Warp-collective: compacts the buffers of the lanes in `full` (cbuf, cnt: each lane's own) and raises their
// thresholds. The next buffer's entries are requested before the current one is worked on.
// A compaction is a chain of latencies (7 k cycles with one bit per step from the top and no load ahead), and while a new
// row's threshold is still low the sweep waits for it: 2047 rows x 4096 x 32000, sweep with K = 64 546 -> 437 us, K = 100
// 597 -> 503 us, K = 256 888 -> 728 us (K = 10: 328 us).
template <int REGS>
__device__ __forceinline__ void compact_rows(uint32_t full, uint2* cbuf, int& cnt, float& thr_own, int K, int cap, int lane) {
    auto row = [&](int L, uint2*& buf, int& n) {
        buf = reinterpret_cast<uint2*>(__shfl_sync(0xffffffffu, reinterpret_cast<unsigned long long>(cbuf), L));
        n = __shfl_sync(0xffffffffu, cnt, L);
    };
    __syncwarp();
    int L = __ffs(full) - 1, n;
    uint2* buf;
    row(L, buf, n);
    uint2 v[REGS];
    load_candidates<REGS>(buf, n, cap, lane, v);
    while (full) {
        full &= full - 1u;
        const int L2 = full ? __ffs(full) - 1 : L;
        int n2;
        uint2* buf2;
        row(L2, buf2, n2);
        uint2 v2[REGS];
        load_candidates<REGS>(buf2, full ? n2 : 0, cap, lane, v2);
        int left = 0;
        const uint32_t tb = compact_candidates<REGS>(buf, v, n, K, cap, lane, left);
        if (lane == L) {
            cnt = left;
            thr_own = __uint_as_float(tb);
        }
        L = L2;
        n = n2;
        buf = buf2;
#pragma unroll
        for (int t = 0; t < REGS; ++t) v[t] = v2[t];
    }
    __syncwarp();
}

// Bitonic sorting network over 16 registers.
__device__ __forceinline__ void sort16_descending(float (&v)[16]) {
#pragma unroll
    for (int k = 2; k <= 16; k *= 2)
#pragma unroll
        for (int j = k / 2; j > 0; j /= 2)
#pragma unroll
            for (int i = 0; i < 16; ++i) {
                const int l = i ^ j;
                if (l > i) {
                    const float hi = fmaxf(v[i], v[l]), lo = fminf(v[i], v[l]);
                    v[i] = (i & k) == 0 ? hi : lo;
                    v[l] = (i & k) == 0 ? lo : hi;
                }
            }
}

// Where S lanes share a row and each has this many logits above a bound, K of the row's logits lie above it.
__host__ __device__ constexpr int lane_share(int K, int S) { return (K + S - 1) / S; }

// Histogram of a thread's row in shared memory: bucket b of thread T at word b * 128 + T of `hist` (the thread's own
// column, no conflicts, no synchronisation). The bucket of x is a non-decreasing function of x.
constexpr int HIST_BUCKETS = 64;
static_assert(HIST_BUCKETS * 128 * 4 <= 4 * SPILL_STAGES * SPILL_STAGE_BYTES, "the histograms take the room of the spill's staging buffers");
__device__ __forceinline__ int hist_bucket(float x, float lo, float inv) {
    return min(max(__float2int_rz((x - lo) * inv), 0), HIST_BUCKETS - 1);
}
__device__ __forceinline__ void hist_clear(uint32_t hist) {
#pragma unroll
    for (int b = 0; b < HIST_BUCKETS; ++b) st_shared_b32(hist + b * 512, 0u);
}
__device__ __forceinline__ void hist_count(uint32_t hist, float x, float lo, float inv) {
    const uint32_t at = hist + hist_bucket(x, lo, inv) * 512;
    st_shared_b32(at, ld_shared_b32(at) + 1u);
}
// the highest buckets that together with those above them hold at least K and k <= K entries; 0 if there are none
__device__ __forceinline__ void hist_top(uint32_t hist, int K, int k, int& top_K, int& top_k) {
    int acc = 0;
    top_K = top_k = 0;
#pragma unroll
    for (int b = HIST_BUCKETS - 1; b > 0; --b) {
        acc += static_cast<int>(ld_shared_b32(hist + b * 512));
        if (top_k == 0 && acc >= k) top_k = b;
        if (top_K == 0 && acc >= K) top_K = b;
    }
}

// TOPK selects how MODE_STATS keeps a row's Top-K candidates: TOPK_REG (K <= K_REG) a sorted list in
// registers, all lanes inserting in parallel - best while most rows still admit logits; TOPK_BUF (any K)
// append buffers with warp-cooperative compaction - cost nearly independent of K; TOPK_NONE: a sweep of draft
// rows whose Omega_hat is already known - no candidates are collected, instead each row's draft logits at its
// Omega_hat tokens are copied out of the accumulator as the sweep passes them (GemmParams::cap_z).
enum { TOPK_REG = 0, TOPK_BUF = 1, TOPK_NONE = 2 };
constexpr int K_REG = 16;

// Four columns of a finished accumulator of MODE_OUT: row scale, Omega_hat term, store.
__device__ __forceinline__ void finish_out4(const GemmParams& p, float4 a, int local_row, int row, int col) {
    if (p.coef != nullptr) {
        const float coef = p.coef[row];
        float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
        if (p.sparse != nullptr) s = *reinterpret_cast<const float4*>(p.sparse + static_cast<long long>(local_row) * p.out_pitch + col);
        a.x = fmaf(coef, a.x, -s.x); a.y = fmaf(coef, a.y, -s.y); a.z = fmaf(coef, a.z, -s.z); a.w = fmaf(coef, a.w, -s.w);
    }
    const long long at = static_cast<long long>(row) * p.out_pitch + col;
    if (p.out_fp32)
        *reinterpret_cast<float4*>(reinterpret_cast<float*>(p.out) + at) = a;
    else
        *reinterpret_cast<uint2*>(reinterpret_cast<__nv_bfloat16*>(p.out) + at) = make_uint2(pack_bf16x2(a.x, a.y), pack_bf16x2(a.z, a.w));
}

// CG: CTAs per product. The kernel is bound by the tensor pipe and, in calls of many milliseconds, by the power cap. A pair
// (tcgen05 cta_group::2, 256 x 256 tile) fetches 32 KB per CTA and k block instead of 48 (sweep of 4608 rows x 4096 x
// 32000: 9.4 GB out of L2 at 12.6 TB/s, by its counter; single CTAs half as much again) and reads half as much of B from
// shared memory; with the stages smaller there are six instead of four. A step of a pair takes 0.89-0.91 of the time of
// the two single steps it replaces (sweep of 8192 rows x 4096 x 32000: 1.77 -> 1.45 ms = 1480 TFLOP/s in short runs;
// 1.24 -> 1.30 PFLOP/s where the power cap holds). Single CTAs stay for one row tile, where a partner would have nothing
// to do, and where an odd number of row tiles makes pairs slower (plan_launch, plan_out).
// EW: epilogue warps. With eight, two threads share a row, 128 columns of every tile each, and meet at an item's end, where the second
// hands its statistics and list to the first. A tile's epilogue is bound by the instructions of its warps, 11 k cycles and more, the products
// take 512 per k block: narrow features leave the tensor core waiting (launch_gemm has the line and what it gives). It exists for the sweeps that
// keep a row's state in registers: statistics alone, and lists of K <= 16 without a spill.
template <int MODE, int TOPK, int CG, int EW = 4>
__global__ void __launch_bounds__(gemm_threads(EW), 1) gemm_kernel(const __grid_constant__ GemmParams p) {
    constexpr bool B_MN_MAJOR = (MODE == MODE_OUT);
    // MODE_OUT after a MODE_LOGITS sweep of the same B, as an instantiation of its own (as a condition in the producer's loop it
    // cost the other calls 3-6 % of this kernel: 517 rows x 4096 x 128256 560 -> 576-595 us)
    constexpr bool KEPT = MODE == MODE_OUT && TOPK == TOPK_NONE;
    // conditional launch (the second pass that follows every spilling call): nothing to do unless the first reported a
    // row beyond its exponent range
    if (p.gate != nullptr) {
        wait_previous_kernel();
        if (*p.gate == 0u) return;
    }
    extern __shared__ uint8_t smem_raw[];
    const uint32_t smem_base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    const uint32_t smemA = smem_base;
    static_assert(EW == 4 || (MODE == MODE_STATS && TOPK != TOPK_BUF), "eight epilogue warps");
    constexpr int STAGES = stages(CG, EW);
    constexpr int OPERANDS = operand_bytes(CG, EW), STAGING = EW * SPILL_STAGES * SPILL_STAGE_BYTES;
    constexpr int B_STAGE_BYTES = b_stage_bytes(CG);
    const uint32_t smemB = smem_base + STAGES * A_STAGE_BYTES;
    const uint32_t spill_stage = smem_base + OPERANDS;      // [epilogue warp][SPILL_STAGES] x SPILL_STAGE_BYTES
    const uint32_t bar_base = spill_stage + STAGING;
    // barriers: full[STAGES], empty[STAGES], tmem_full[2], tmem_empty[2], meet[2]; then tmem pointer, abort flag
    auto full_bar = [&](int s) { return bar_base + 8u * s; };
    auto empty_bar = [&](int s) { return bar_base + 8u * (STAGES + s); };
    auto tfull_bar = [&](int b) { return bar_base + 8u * (2 * STAGES + b); };
    auto tempty_bar = [&](int b) { return bar_base + 8u * (2 * STAGES + 2 + b); };
    auto meet_bar = [&](int b) { return bar_base + 8u * (2 * STAGES + 4 + b); };      // EW = 8: the second threads' results are there / taken
    uint8_t* smem_gen = smem_raw + (smem_base - smem_u32(smem_raw));
    uint32_t* tmem_ptr_smem =
        reinterpret_cast<uint32_t*>(smem_gen + OPERANDS + STAGING + 8 * (2 * STAGES + 6));
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_ptr_smem + 1);

    const int warp = threadIdx.x >> 5;
    const int lane = threadIdx.x & 31;
    const int cta = CG == 2 ? blockIdx.x >> 1 : blockIdx.x;             // CTA or pair
    const uint32_t rank = CG == 2 ? cluster_ctarank() : 0;

    if (threadIdx.x == 0) {
        for (int s = 0; s < STAGES; ++s) {
            mbar_init(full_bar(s), 1);
            mbar_init(empty_bar(s), 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(tfull_bar(b), 1);
            mbar_init(tempty_bar(b), EW * CG);
            if (EW == 8) mbar_init(meet_bar(b), 4);
        }
        *abort_flag = 0;
        fence_barrier_init();
        fence_proxy_async_smem();
        prefetch_tensormap(&p.tmA0);
        prefetch_tensormap(&p.tmB);
        if (MODE == MODE_STATS || MODE == MODE_LOGITS) prefetch_tensormap(&p.tmA1);
    }
    if (warp == 1) {
        if (CG == 2) {
            tmem_alloc_pair(smem_u32(tmem_ptr_smem), TMEM_COLS);
            tmem_relinquish_pair();
        } else {
            tmem_alloc(smem_u32(tmem_ptr_smem), TMEM_COLS);
            tmem_relinquish();
        }
    }
    if (p.gate == nullptr) {
        if (MODE == MODE_LOGITS || KEPT)
            wait_previous_kernel(!p.release_late);
        else
            wait_previous_kernel();
    }
    // (A wait of another CTA that ran out would be recorded two seconds later.)
    if (MODE == MODE_LOGITS && p.clear_status && blockIdx.x == 0 && threadIdx.x < 64) p.status[threadIdx.x] = 0u;
    tc_fence_before_sync();
    __syncthreads();
    if (CG == 2) cluster_sync();      // the partner's barriers are initialised, its tensor memory is allocated
    tc_fence_after_sync();
    const uint32_t tmem_base = *tmem_ptr_smem;

    // Calls f(row_tile, lane, S, slot, first k block, end of k blocks) for every item of this CTA; f returns false to
    // stop. MODE_OUT: one column tile (= lane; S = all of them), slot = the partial tile it goes to, -1, or SHARED_TILE.
    constexpr int SHARED_TILE = -2;
    auto for_each_item = [&](auto&& f) {
        if constexpr (MODE == MODE_OUT) {
            const OutPlan& o = p.plan;
            if (CG == 1 && o.cluster > 1) {
                const int u = cta / o.cluster, z = cta - u * o.cluster;
                f(u % o.row_units, u / o.row_units, p.col_tiles, SHARED_TILE, static_cast<int>(static_cast<long long>(p.k_blocks) * z / o.cluster),
                  static_cast<int>(static_cast<long long>(p.k_blocks) * (z + 1) / o.cluster));
                return;
            }
            for (int u = cta; u < o.whole; u += o.groups)
                if (!f(u % o.row_units * CG + static_cast<int>(rank), u / o.row_units, p.col_tiles, -1, 0, p.k_blocks)) return;
            for (int v = cta; v < o.rest * o.cuts; v += o.groups) {
                const int z = v / o.rest, u = o.whole + v - z * o.rest;
                const int kb0 = static_cast<int>(static_cast<long long>(p.k_blocks) * z / o.cuts);
                const int kb1 = static_cast<int>(static_cast<long long>(p.k_blocks) * (z + 1) / o.cuts);
                if (!f(u % o.row_units * CG + static_cast<int>(rank), u / o.row_units, p.col_tiles,
                       v * CG + static_cast<int>(rank), kb0, kb1))
                    return;
            }
        } else {
            for (int ph = 0; ph < p.sched.n_phases; ++ph) {
                const Phase P = p.sched.ph[ph];
                if (cta < P.G / CG * P.S) {
                    const int gi = cta / P.S;
                    const int ln = cta - gi * P.S;
                    const int ri = gi * CG + static_cast<int>(rank);
                    if (!f(P.row_tile_begin + ri, ln, P.S, P.slot_base + ri * P.S + ln, 0, p.k_blocks)) return;
                }
            }
        }
    };
    // Column tiles of lane ln, the first column of its tile t, and that tile's columns (BN but for the last one of MODE_LOGITS)
    auto tiles_of = [&](int ln, int S) {
        if constexpr (MODE == MODE_LOGITS) return (min(p.lane_cols, static_cast<int>(p.z_pitch) - ln * p.lane_cols) + BN - 1) / BN;
        return (p.col_tiles - ln + S - 1) / S;
    };
    auto tile_col = [&](int ln, int S, int t) {
        if constexpr (MODE == MODE_LOGITS) return ln * p.lane_cols + t * BN;
        return (t < 0 ? 0 : ln + t * S) * (KEPT && CG == 1 ? p.plan.width : BN);      // t = -1: column tile 0, for the row references only
    };
    auto tile_width = [&](int t) {
        if constexpr (MODE == MODE_LOGITS) return min(BN, p.lane_cols - t * BN);
        if constexpr (KEPT && CG == 1) return p.plan.width;
        return BN;
    };
    // Where rows spill without a given reference exponent, a lane that does not begin with column tile 0 computes it first
    // (t = -1); a pair agrees.
    auto first_tile = [&](int rt, int ln) {
        if (MODE != MODE_STATS || TOPK == TOPK_NONE || ln == 0) return 0;
        const int rt0 = rt - static_cast<int>(rank);
        return spills(p, rt0) || (CG == 2 && spills(p, rt0 + 1)) ? -1 : 0;
    };

    if (warp == 0) {
        // ===================== TMA producer =====================
        if (lane == 0) {
            int stage = 0;
            uint32_t phase = 0;
            const uint64_t keep = MODE == MODE_LOGITS ? l2_evict_normal() : 0ull, drop = MODE == MODE_LOGITS || KEPT ? l2_evict_first() : 0ull;
            for_each_item([&](int rt, int ln, int S, int, int kb0, int kb1) {
                const bool second = (MODE == MODE_STATS || MODE == MODE_LOGITS) && rt >= p.row_tiles0;
                const CUtensorMap* tmA = second ? &p.tmA1 : &p.tmA0;
                const int row0 = p.a_row_offset + (second ? rt - p.row_tiles0 : rt) * BM;
                const int t0 = first_tile(rt, ln);
                const int nt = tiles_of(ln, S);
                for (int t = t0; t < nt; ++t) {
                    const int width = tile_width(t);
                    const CUtensorMap* tmB = MODE == MODE_LOGITS && width < BN ? &p.tmSpill : &p.tmB;
                    for (int kb = kb0; kb < kb1; ++kb) {
                        if (!wait_barrier(empty_bar(stage), phase ^ 1u, abort_flag, p.status, 1)) return false;
                        // a pair's bytes are all counted on the barrier of its first CTA, whose thread issues the products
                        if (rank == 0) mbar_arrive_expect_tx(full_bar(stage), CG * A_STAGE_BYTES + width * (BK * 2));
                        const uint32_t bar = CG == 2 ? map_to_rank(full_bar(stage), 0) : full_bar(stage);
                        auto load = [&](uint32_t dst, const CUtensorMap* tm, int x, int y) {
                            if (CG == 2)
                                tma_load_2d_pair(dst, tm, bar, x, y);
                            else
                                tma_load_2d(dst, tm, bar, x, y);
                        };
                        auto load_b = [&](uint32_t dst, int x, int y) {
                            if (MODE == MODE_LOGITS || KEPT) {
                                const uint64_t policy = MODE == MODE_LOGITS && kb >= p.keep_from ? keep : drop;
                                if (CG == 2)
                                    tma_load_2d_pair_hint(dst, tmB, bar, x, y, policy);
                                else
                                    tma_load_2d_hint(dst, tmB, bar, x, y, policy);
                            } else {
                                load(dst, tmB, x, y);
                            }
                        };
                        const int col0 = tile_col(ln, S, t) + static_cast<int>(rank) * (width / CG);
                        if (MODE == MODE_LOGITS && CG == 1 && p.half_tiles) {
                            load(smemA + stage * A_STAGE_BYTES, &p.tmA0, kb * BK, 0);
                            load(smemA + stage * A_STAGE_BYTES + A_STAGE_BYTES / 2, &p.tmA1, kb * BK, 0);
                        } else {
                            load(smemA + stage * A_STAGE_BYTES, tmA, kb * BK, row0);
                        }
                        if (!B_MN_MAJOR) {
                            load_b(smemB + stage * B_STAGE_BYTES, kb * BK, col0);
                        } else {
                            // B tile = BK contraction rows x width / CG contiguous columns, fetched as boxes
                            // of 64 columns (one 128-byte swizzle row) x BK rows
#pragma unroll
                            for (int j = 0; j < width / CG / 64; ++j)
                                load_b(smemB + stage * B_STAGE_BYTES + j * (BK * 128), col0 + j * 64, kb * BK);
                        }
                        if (++stage == STAGES) {
                            stage = 0;
                            phase ^= 1u;
                        }
                    }
                }
                return true;
            });
        }
    } else if (warp == 1) {
        // ===================== MMA issuer =====================
        if (lane == 0 && rank == 0) {
            int stage = 0;
            uint32_t phase = 0;
            int ab = 0;
            uint32_t aphase = 0;
            for_each_item([&](int rt, int ln, int S, int, int kb0, int kb1) {
                const int t0 = first_tile(rt, ln);
                const int nt = tiles_of(ln, S);
                for (int t = t0; t < nt; ++t) {
                    const uint32_t idesc = make_idesc_bf16(CG * BM, tile_width(t), 0, B_MN_MAJOR ? 1 : 0);
                    if (!wait_barrier(tempty_bar(ab), aphase ^ 1u, abort_flag, p.status, 2)) return false;
                    tc_fence_after_sync();
                    const uint32_t d_tmem = tmem_base + ab * BN;
                    for (int kb = kb0; kb < kb1; ++kb) {
                        if (!wait_barrier(full_bar(stage), phase, abort_flag, p.status, 3)) return false;
                        tc_fence_after_sync();
                        // A: K-major, 8-row groups 1024 B apart. B: K-major likewise, or MN-major with
                        // 64-column groups BK*128 B apart (LBO) and 8-row contraction groups 1024 B apart (SBO).
                        const uint64_t a_desc = make_smem_desc_sw128(smemA + stage * A_STAGE_BYTES, 0, 1024);
                        const uint64_t b_desc =
                            B_MN_MAJOR ? make_smem_desc_sw128(smemB + stage * B_STAGE_BYTES, BK * 128, 1024)
                                       : make_smem_desc_sw128(smemB + stage * B_STAGE_BYTES, 0, 1024);
#pragma unroll
                        for (int k = 0; k < BK / UMMA_K; ++k) {
                            // advance the start address (>>4) along the contraction
                            const uint64_t a_adv = static_cast<uint64_t>((k * UMMA_K * 2) >> 4);
                            const uint64_t b_adv = B_MN_MAJOR ? static_cast<uint64_t>((k * UMMA_K * 128) >> 4)
                                                              : static_cast<uint64_t>((k * UMMA_K * 2) >> 4);
                            if (CG == 2)
                                umma_bf16_pair(d_tmem, a_desc + a_adv, b_desc + b_adv, idesc, (kb - kb0 | k) != 0 ? 1u : 0u);
                            else
                                umma_bf16(d_tmem, a_desc + a_adv, b_desc + b_adv, idesc, (kb - kb0 | k) != 0 ? 1u : 0u);
                        }
                        // frees the stage (of both CTAs) once these MMAs have read it
                        if (CG == 2)
                            umma_commit_pair(empty_bar(stage));
                        else
                            umma_commit(empty_bar(stage));
                        if (++stage == STAGES) {
                            stage = 0;
                            phase ^= 1u;
                        }
                    }
                    if (CG == 2)                         // accumulator complete
                        umma_commit_pair(tfull_bar(ab));
                    else
                        umma_commit(tfull_bar(ab));
                    ab ^= 1;
                    if (ab == 0) aphase ^= 1u;
                }
                return true;
            });
        }
    } else {
        // ===================== epilogue warps =====================
        const int quad = warp & 3;                 // TMEM lane quadrant this warp may read
        const int r_local = quad * 32 + lane;      // row inside the tile
        const int half = EW == 8 ? (warp - 2) >> 2 : 0;      // EW = 8: which columns of a tile
        constexpr int SHARE = BN * 4 / EW;         // columns of a tile that a thread takes: [half SHARE, (half + 1) SHARE)
        uint32_t meet_phase = 0;
        int ab = 0;
        uint32_t aphase = 0;
        // Top-K candidates of this thread's row (MODE_STATS): buffer in the workspace, entries in use
        uint2* cbuf = nullptr;
        int cnt = 0;
        uint32_t spill_boxes = 0;                  // chunks this warp has staged for TMA stores (two per box)
        // TOPK_REG: the K_REG largest logits so far sorted descending in tv[] (the admission threshold is the
        // K_REG-th largest: a list of exactly K entries with its K-th as threshold measured slower), and the
        // current chunk's admitted logits waiting in shared memory: entry q of thread T at word q * 128 + T of the values' array and
        // of the tokens' array (16 KB each, the room the draft sweep uses for its spill boxes; this instantiation stores no boxes). With
        // 200 KB of shared memory carved out little L1 is left, and a per-thread array in local memory cost about a thousand
        // cycles per admitted logit here.
        constexpr bool USE_REG = MODE == MODE_STATS && TOPK == TOPK_REG;
        constexpr bool HAS_TOPK = MODE == MODE_STATS && TOPK != TOPK_NONE;
        constexpr bool CAPTURE = MODE == MODE_STATS && TOPK == TOPK_NONE;
        float tv[USE_REG ? K_REG : 1];
        int ti[USE_REG ? K_REG : 1];
        constexpr int PEND = EW * 32 * 4;          // bytes from one entry to the next
        static_assert(STAGING >= 2 * 32 * PEND, "room for the pending logits");
        const uint32_t pend_v = spill_stage + pending_at(threadIdx.x);
        const uint32_t pend_i = pend_v + 32 * PEND;
        constexpr int lo = 0;

        for_each_item([&](int rt, int ln, int S, int slot, int, int) {
            const int g_row = p.row_global_offset + rt * BM + r_local;
            const bool tile_ok = CG == 1 || rt < p.row_tiles;     // false: the partner of the last row tile, nothing to write
            const bool row_ok = tile_ok && g_row < p.rows_valid;
            // ---- per-item state ----
            float m = -INFINITY, s = 0.f, thr = -INFINITY;        // MODE_STATS; thr = admission threshold in force
            float thr_own = -INFINITY;                            // K-th (K_REG-th) largest logit of this lane's own list
            float thr_sh = -INFINITY;                             // just below the best bound that what the lanes published gives
            // TOPK_BUF: the histogram of this lane's logits between hist_lo and the first tile's largest (a quarter of its range
            // higher); a logit at or below the threshold of its time is missing. hist_inv = 0: none
            float hist_lo = 0.f, hist_inv = 0.f;
            int counted = 0;                                      // entries of the buffer that are in it
            const int share = HAS_TOPK && !USE_REG ? lane_share(p.K, S) : 0;
            bool want_topk = false;
            const bool spill = MODE == MODE_STATS && tile_ok && spills(p, rt);
            const bool track_zmax = MODE == MODE_STATS && spill && p.row_zmax != nullptr;
            float zmax = -INFINITY;                               // the row's largest logit in this lane's column tiles
            float ref2 = 0.f;                                     // spill rows: exponent offset (log2 units)
            float lse2 = 0.f, coef = 0.f;                         // MODE_PROBS / fused MODE_OUT
            const int* si = nullptr;
            const float* sg = nullptr;
            int cur = 0, nxt = INT_MAX;
            if (MODE == MODE_STATS) {
                want_topk = HAS_TOPK && tile_ok && rt < p.topk_row_tiles;
                if (HAS_TOPK) cbuf = p.cand + (static_cast<long long>(slot) * BM + r_local) * p.cap;
                cnt = 0;
                if (HAS_TOPK && p.row_global_offset + (rt < p.row_tiles0 ? rt : rt - p.row_tiles0) * BM + r_local >= p.rows_valid) {
                    // A padding row collects nothing: its logits are all equal (zero), and 256 of them filled its buffer and
                    // made the warp compact row after row (sweep of 64 rows x 256 x 1024, K = 64: 195 -> 30 us).
                    thr_own = INFINITY;
                    thr = INFINITY;
                }
                if (USE_REG) {
#pragma unroll
                    for (int i = 0; i < (USE_REG ? K_REG : 1); ++i) {
                        tv[i] = -INFINITY;
                        ti[i] = -1;
                    }
                }
            }
            if (MODE == MODE_PROBS && row_ok) {
                lse2 = p.lse2[g_row];
                coef = p.coef[g_row];
                si = p.sidx + static_cast<long long>(g_row) * p.K;
                sg = p.sgq + static_cast<long long>(g_row) * p.K;
                nxt = si[0];
            }
            if (MODE == MODE_OUT && p.coef != nullptr && row_ok) coef = p.coef[g_row];
            float* cz = nullptr;
            if (CAPTURE && row_ok && p.cap_z != nullptr) {
                // the row's Omega_hat in increasing token order; this lane meets its own column tiles in that order too
                si = p.sidx + static_cast<long long>(g_row) * p.K;
                cz = p.cap_z + static_cast<long long>(g_row) * p.K;
                nxt = si[0];
            }
            float* zrow = nullptr;
            if (MODE == MODE_LOGITS && tile_ok) {
                const bool halved = CG == 1 && p.half_tiles;
                const int r_own = halved ? r_local % (BM / 2) : (rt < p.row_tiles0 ? rt : rt - p.row_tiles0) * BM + r_local;      // row in its own matrix
                float* z = (halved ? quad >= 2 : rt >= p.row_tiles0) ? p.z_out : p.zt_out;
                if (r_own < p.z_rows) zrow = z + static_cast<long long>(r_own) * p.z_pitch;
            }
            const int t0 = first_tile(rt, ln);
            const int nt = tiles_of(ln, S);
            // lanes of three tiles and more share their bounds (see below)
            const bool joint = HAS_TOPK && !USE_REG && p.bounds != nullptr && p.col_tiles > 2 * S;
            for (int t = t0; t < nt; ++t) {
                // the whole warp must agree before the warp-collective TMEM loads below
                const bool ready = wait_barrier(tfull_bar(ab), aphase, abort_flag, p.status, 4);
                if (!__all_sync(0xffffffffu, ready)) return false;
                if (MODE == MODE_OUT && CG == 1 && slot == SHARED_TILE) return false;      // finished below, with the cluster
                tc_fence_after_sync();
                const uint32_t t_row = tmem_base + (static_cast<uint32_t>(quad * 32) << 16) + ab * BN;
                const int col_base = tile_col(ln, S, t);
                const bool skip_tile = t < 0 || !tile_ok;
                if (CAPTURE && spill && t == 0) {
                    ref2 = 0.f;
                    if (row_ok) ref2 = p.use_row_zmax ? fmaf(__uint_as_float(key_bits(p.row_zmax[rt * BM + r_local])), LOG2E, 64.f) : p.row_ref2[g_row];
                    m = ref2 * (1.0f / LOG2E);
                }
                if (MODE == MODE_STATS && TOPK != TOPK_NONE && spill && t == t0) {
                    // Reference exponent of this row: its largest logit in column tile 0. Every lane of
                    // the row tile computes tile 0 first and so derives the same value.
                    float mx = -INFINITY;
                    if (p.use_row_zmax) {
                        // second sweep after a range report: the row's largest logit is known
                        mx = __uint_as_float(key_bits(p.row_zmax[rt * BM + r_local]));
                    } else {
#pragma unroll 1
                        for (int ch = 0; ch < BN / 32; ++ch) {
                            uint32_t r[32];
                            tmem_ld32(t_row + ch * 32, r);
                            tmem_ld_wait(r);
#pragma unroll
                            for (int j = 0; j < 32; ++j)
                                if (ch * 32 + j < p.n_cols) mx = fmaxf(mx, __uint_as_float(r[j]));
                        }
                    }
                    // spilled values are 2^(z log2e - ref2) <= about 2^-64 for typical rows, which leaves
                    // 2^130 of headroom above the reference before SPILL_SUM_LIMIT
                    ref2 = fmaf(mx, LOG2E, 64.f);
                    m = ref2 * (1.0f / LOG2E);
                }
                if (MODE == MODE_STATS && HAS_TOPK && !USE_REG && want_topk && t == 0 && p.n_cols - col_base >= BN) {
                    // First tile of the sweep, buffer empty, no threshold yet: admitting all 256 logits would fill the buffer
                    // at once. Each thread takes a histogram of its row's 256 logits between the least and a little above the
                    // largest and starts from half a bucket below the bucket above which at least K of them lie: a valid lower bound of
                    // the row's K-th largest logit that admits little more than K of the tile's.
                    float lo = INFINITY, hi = -INFINITY;
#pragma unroll 1
                    for (int ch = 0; ch < BN / 32; ++ch) {
                        uint32_t r[32];
                        tmem_ld32(t_row + ch * 32, r);
                        tmem_ld_wait(r);
#pragma unroll
                        for (int j = 0; j < 32; ++j) {
                            lo = fminf(lo, __uint_as_float(r[j]));
                            hi = fmaxf(hi, __uint_as_float(r[j]));
                        }
                    }
                    hist_lo = lo;
                    hist_inv = HIST_BUCKETS / (1.25f * (hi - lo));
                    hist_clear(pend_v);
#pragma unroll 1
                    for (int ch = 0; ch < BN / 32; ++ch) {
                        uint32_t r[32];
                        tmem_ld32(t_row + ch * 32, r);
                        tmem_ld_wait(r);
#pragma unroll
                        for (int j = 0; j < 32; ++j) hist_count(pend_v, __uint_as_float(r[j]), lo, hist_inv);
                    }
                    // (half a bucket must exceed the rounding of these few operations; also false for infinities and NaN)
                    if (!(0.5f / hist_inv > 1e-6f * fmaxf(fabsf(lo), fabsf(hi)))) hist_inv = 0.f;
                    int top, top_share;
                    hist_top(pend_v, p.K, share, top, top_share);
                    if (top > 0 && hist_inv > 0.f) {
                        thr_own = fmaxf(thr_own, lo + (static_cast<float>(top) - 0.5f) / hist_inv);
                        thr = fmaxf(thr_own, thr_sh);
                    }
                }
                if (USE_REG && want_topk && t == 0 && p.n_cols - col_base >= BN) {
                    // First tile of the sweep, list empty: the K-th largest of the maxima of 16 groups of 16 logits is a
                    // lower bound of the row's K-th largest that about 16 of the tile's 256 logits reach. Without it every
                    // row inserts its first 32 logits and some 70 more one by one, the warp as often as its slowest row
                    // (64 rows x 256 x 1024, four tiles on four CTAs: 28.0 -> 17.5 us).
                    float gm[16];
                    constexpr int GROUP = SHARE / 16;
#pragma unroll
                    for (int ch = 0; ch < SHARE / 32; ++ch) {
                        uint32_t r[32];
                        tmem_ld32(t_row + half * SHARE + ch * 32, r);
                        tmem_ld_wait(r);
#pragma unroll
                        for (int h = 0; h < 32 / GROUP; ++h) {
                            float x = fmaxf(__uint_as_float(r[GROUP * h]), __uint_as_float(r[GROUP * h + 1]));
#pragma unroll
                            for (int j = 2; j < GROUP; j += 2) x = fmax3(x, __uint_as_float(r[GROUP * h + j]), __uint_as_float(r[GROUP * h + j + 1]));
                            gm[32 / GROUP * ch + h] = fmaxf(x, -INFINITY);      // (a group of NaN counts for nothing)
                        }
                    }
                    sort16_descending(gm);
                    float kth = gm[0];
#pragma unroll
                    for (int i = 1; i < 16; ++i)
                        if (i == p.K - 1) kth = gm[i];
                    thr_sh = fmaxf(thr_sh, nextafterf(kth, -INFINITY));      // (a logit equal to the bound must be admitted)
                    thr = fmaxf(thr, thr_sh);
                }
                if (CAPTURE && !skip_tile) {
                    while (nxt < col_base + half * SHARE) {
                        ++cur;
                        nxt = cur < p.K ? si[cur] : INT_MAX;
                    }
                }
#pragma unroll 1
                for (int ch = half * (SHARE / 32); ch < (EW == 8 ? (half + 1) * (SHARE / 32) : tile_width(t) / 32) && !skip_tile; ++ch) {
                    if (MODE == MODE_STATS && !USE_REG && want_topk) {
                        // make room for a whole chunk in every row's buffer (warp-uniform control flow), before the
                        // chunk's logits occupy registers
                        const uint32_t full = __ballot_sync(0xffffffffu, cnt > p.cap - 32);
                        if (full) {
                            if (p.cap <= 32 * CAND_REGS_TINY)
                                compact_rows<CAND_REGS_TINY>(full, cbuf, cnt, thr_own, p.K, p.cap, lane);
                            else if (p.cap <= 32 * CAND_REGS_SMALL)
                                compact_rows<CAND_REGS_SMALL>(full, cbuf, cnt, thr_own, p.K, p.cap, lane);
                            else
                                compact_rows<CAND_REGS>(full, cbuf, cnt, thr_own, p.K, p.cap, lane);
                            thr = fmaxf(thr_own, thr_sh);
                            counted = min(counted, cnt);      // (entries that were dropped before they were counted stay uncounted)
                        }
                    }
                    uint32_t r[32];
                    tmem_ld32(t_row + ch * 32, r);
                    tmem_ld_wait(r);
                    const int col0 = col_base + ch * 32;
                    if (MODE == MODE_STATS || MODE == MODE_LOGITS) {
                        if (col0 + 32 > p.n_cols) {
#pragma unroll
                            for (int j = 0; j < 32; ++j)
                                if (col0 + j >= p.n_cols) r[j] = __float_as_uint(-INFINITY);
                        }
                    }
                    if (MODE == MODE_LOGITS) {
                        if (zrow != nullptr && col0 < p.z_pitch) {
#pragma unroll
                            for (int g8 = 0; g8 < 4; ++g8)
                                st_global_v8(zrow + col0 + 8 * g8, r[8 * g8], r[8 * g8 + 1], r[8 * g8 + 2], r[8 * g8 + 3],
                                             r[8 * g8 + 4], r[8 * g8 + 5], r[8 * g8 + 6], r[8 * g8 + 7]);
                        }
                    } else if (MODE == MODE_STATS) {
                        if (CAPTURE) {
                            // draft logits at the row's Omega_hat, straight from the fp32 accumulator
                            while (nxt < col0 + 32) {
                                const int off = nxt - col0;
                                uint32_t zb = 0u;
#pragma unroll
                                for (int j = 0; j < 32; ++j)
                                    if (j == off) zb = r[j];
                                cz[cur] = __uint_as_float(zb);
                                ++cur;
                                nxt = cur < p.K ? si[cur] : INT_MAX;
                            }
                        }
                        float cm = -INFINITY;     // the chunk's largest logit (not needed by a spill row without Top-K)
                        if (!spill || want_topk || track_zmax) {
                            cm = fmaxf(__uint_as_float(r[0]), __uint_as_float(r[1]));
#pragma unroll
                            for (int j = 2; j < 32; j += 2) cm = fmax3(cm, __uint_as_float(r[j]), __uint_as_float(r[j + 1]));
                            zmax = fmaxf(zmax, cm);
                        }
                        if (!spill) {
                            if (cm > m) {
                                s *= ex2((m - cm) * LOG2E);
                                m = cm;
                            }
                            // (EW = 8: of a lane's last tile the second thread may meet columns beyond the vocabulary alone)
                            const float mneg = EW == 8 && m == -INFINITY ? 0.f : -m * LOG2E;
                            float acc0 = 0.f, acc1 = 0.f;
#pragma unroll
                            for (int j = 0; j < 32; j += 2) {
                                float t0, t1;
                                ffma2(t0, t1, __uint_as_float(r[j]), __uint_as_float(r[j + 1]), LOG2E, LOG2E, mneg, mneg);
                                fadd2(acc0, acc1, acc0, acc1, ex2(t0), ex2(t1));
                            }
                            s += acc0 + acc1;
                        } else {
                            // one exponential per logit serves both the row's sum and the spilled tile; a
                            // logit beyond the exponent range gives inf here and is reported at the item's end
                            float e[32];
                            float acc0 = 0.f, acc1 = 0.f;
                            const float nref2 = -ref2;
#pragma unroll
                            for (int j = 0; j < 32; j += 2) {
                                float t0, t1;
                                ffma2(t0, t1, __uint_as_float(r[j]), __uint_as_float(r[j + 1]), LOG2E, LOG2E, nref2, nref2);
                                e[j] = ex2(t0);
                                e[j + 1] = ex2(t1);
                                fadd2(acc0, acc1, acc0, acc1, e[j], e[j + 1]);
                            }
                            s += acc0 + acc1;
                            if (TOPK == TOPK_NONE) {
                                // The draft sweep hands its spill to the TMA unit: the row's 32 values go into the warp's
                                // staging buffer (128-byte rows, swizzled), and after every second chunk one lane
                                // requests the store of the 32 x 64 box. That is one request per 4 KB from this warp
                                // instead of 64 store instructions that each touch 32 rows.
                                const uint32_t buf = spill_stage + stage_at(half, quad) + ((spill_boxes >> 1) & 1) * SPILL_STAGE_BYTES;
                                if ((ch & 1) == 0) {
                                    // the store that read this buffer two boxes ago must have finished reading it
                                    if (lane == 0) bulk_wait_group_read<SPILL_STAGES - 1>();
                                    __syncwarp();
                                }
#pragma unroll
                                for (int j = 0; j < 4; ++j)
                                    st_shared_v4(buf + lane * 128 + ((((ch & 1) * 4 + j) ^ (lane & 7)) << 4),
                                                 pack_bf16x2(e[8 * j + 0], e[8 * j + 1]), pack_bf16x2(e[8 * j + 2], e[8 * j + 3]),
                                                 pack_bf16x2(e[8 * j + 4], e[8 * j + 5]), pack_bf16x2(e[8 * j + 6], e[8 * j + 7]));
                                if (ch & 1) {
                                    fence_proxy_async_smem();
                                    __syncwarp();
                                    if (lane == 0) {
                                        tma_store_2d(&p.tmSpill, buf, col0 - 32, (rt - p.spill_begin) * BM + quad * 32);
                                        bulk_commit_group();
                                    }
                                }
                                ++spill_boxes;
                            } else {
                                __nv_bfloat16* dst = (rt >= p.spill_begin
                                                          ? p.P + static_cast<long long>((rt - p.spill_begin) * BM + r_local) * p.p_pitch
                                                          : p.Pt + static_cast<long long>(rt * BM + r_local) * p.p_pitch) + col0;
#pragma unroll
                                for (int g16 = 0; g16 < 2; ++g16)
                                    st_global_v8(dst + 16 * g16, pack_bf16x2(e[16 * g16 + 0], e[16 * g16 + 1]),
                                                 pack_bf16x2(e[16 * g16 + 2], e[16 * g16 + 3]),
                                                 pack_bf16x2(e[16 * g16 + 4], e[16 * g16 + 5]),
                                                 pack_bf16x2(e[16 * g16 + 6], e[16 * g16 + 7]),
                                                 pack_bf16x2(e[16 * g16 + 8], e[16 * g16 + 9]),
                                                 pack_bf16x2(e[16 * g16 + 10], e[16 * g16 + 11]),
                                                 pack_bf16x2(e[16 * g16 + 12], e[16 * g16 + 13]),
                                                 pack_bf16x2(e[16 * g16 + 14], e[16 * g16 + 15]));
                            }
                        }
                        if (!USE_REG && want_topk && cm > thr) {
                            // predicated stores, no branches: as 32 conditional blocks this section took about 5000
                            // cycles whenever any row of the warp admitted a logit
                            uint2* at = cbuf + cnt;
#pragma unroll
                            for (int j = 0; j < 32; ++j) append_if_above(at, __uint_as_float(r[j]), static_cast<uint32_t>(col0 + j), thr);
                            cnt = static_cast<int>(at - cbuf);
                        }
                        if (USE_REG && want_topk && cm > thr) {
                            // collect the chunk's candidates, then admit them one by one (the
                            // threshold only rises, so each is re-checked against the current one)
                            int np = 0;
#pragma unroll
                            for (int j = 0; j < 32; ++j) {
                                const float x = __uint_as_float(r[j]);
                                const bool in = x > thr;       // predicated stores, no branches
                                st_shared_b32_if(pend_v + np * PEND, __float_as_uint(x), in);
                                st_shared_b32_if(pend_i + np * PEND, static_cast<uint32_t>(col0 + j), in);
                                np += in ? 1 : 0;
                            }
                            for (int q = 0; q < np; ++q) {
                                const float x = __uint_as_float(ld_shared_b32(pend_v + q * PEND));
                                const int id = static_cast<int>(ld_shared_b32(pend_i + q * PEND));
                                if (!(x > thr)) continue;
                                // sorted insertion; equal logits stay behind earlier (lower) token ids
#pragma unroll
                                for (int i = (USE_REG ? K_REG : 1) - 1; i >= 0; --i) {
                                    if (i > 0 && i > lo) {
                                        const bool shift = x > tv[i > 0 ? i - 1 : 0];
                                        const bool here = !shift && x > tv[i];
                                        tv[i] = shift ? tv[i > 0 ? i - 1 : 0] : (here ? x : tv[i]);
                                        ti[i] = shift ? ti[i > 0 ? i - 1 : 0] : (here ? id : ti[i]);
                                    } else if (i == lo) {
                                        if (x > tv[i]) {
                                            tv[i] = x;
                                            ti[i] = id;
                                        }
                                    }
                                }
                                thr_own = tv[(USE_REG ? K_REG : 1) - 1];
                                thr = fmaxf(thr_own, thr_sh);
                            }
                        }
                    } else if (MODE == MODE_PROBS) {
                        while (nxt < col0) {
                            ++cur;
                            nxt = cur < p.K ? si[cur] : INT_MAX;
                        }
                        float e[32];
#pragma unroll
                        for (int j = 0; j < 32; ++j) e[j] = coef * ex2(fmaf(__uint_as_float(r[j]), LOG2E, -lse2));
                        while (nxt < col0 + 32) {
                            const int off = nxt - col0;
                            const float gq = sg[cur];
#pragma unroll
                            for (int j = 0; j < 32; ++j)
                                if (j == off) e[j] -= gq;
                            ++cur;
                            nxt = cur < p.K ? si[cur] : INT_MAX;
                        }
                        if (col0 + 32 > p.n_cols) {
#pragma unroll
                            for (int j = 0; j < 32; ++j)
                                if (col0 + j >= p.n_cols) e[j] = 0.f;
                        }
                        uint4* dst = reinterpret_cast<uint4*>(p.P + static_cast<long long>(rt * BM + r_local) * p.p_pitch + col0);
#pragma unroll
                        for (int g8 = 0; g8 < 4; ++g8) {
                            uint4 w;
                            w.x = pack_bf16x2(e[8 * g8 + 0], e[8 * g8 + 1]);
                            w.y = pack_bf16x2(e[8 * g8 + 2], e[8 * g8 + 3]);
                            w.z = pack_bf16x2(e[8 * g8 + 4], e[8 * g8 + 5]);
                            w.w = pack_bf16x2(e[8 * g8 + 6], e[8 * g8 + 7]);
                            dst[g8] = w;
                        }
                    } else if (row_ok) {
                        float o[32];
#pragma unroll
                        for (int j = 0; j < 32; ++j) o[j] = __uint_as_float(r[j]);
                        const bool full = col0 + 32 <= p.n_cols;
                        if (slot >= 0) {
                            // a piece of the contraction: the accumulator as it is
                            float* dst = p.part + (static_cast<long long>(slot) * p.plan.part_rows + r_local) * BN + ch * 32;
#pragma unroll
                            for (int g8 = 0; g8 < 4; ++g8)
                                st_global_v8(dst + 8 * g8, r[8 * g8], r[8 * g8 + 1], r[8 * g8 + 2], r[8 * g8 + 3], r[8 * g8 + 4],
                                             r[8 * g8 + 5], r[8 * g8 + 6], r[8 * g8 + 7]);
                            continue;
                        }
                        if (p.sparse != nullptr) {
                            // dH_d = coef * (spilled tile x W) - sum_{x in Omega_hat} g q(x) W[x, :]
                            const float* sp = p.sparse + static_cast<long long>(rt * BM + r_local) * p.out_pitch + col0;
                            if (full) {
#pragma unroll
                                for (int g8 = 0; g8 < 4; ++g8) {
                                    float v[8];
                                    ld_global_v8(sp + 8 * g8, v);
#pragma unroll
                                    for (int u = 0; u < 8; ++u) o[8 * g8 + u] = fmaf(coef, o[8 * g8 + u], -v[u]);
                                }
                            } else {
#pragma unroll
                                for (int g4 = 0; g4 < 8; ++g4) {
                                    if (col0 + 4 * g4 < p.n_cols) {
                                        const float4 v = *reinterpret_cast<const float4*>(sp + 4 * g4);
                                        o[4 * g4 + 0] = fmaf(coef, o[4 * g4 + 0], -v.x);
                                        o[4 * g4 + 1] = fmaf(coef, o[4 * g4 + 1], -v.y);
                                        o[4 * g4 + 2] = fmaf(coef, o[4 * g4 + 2], -v.z);
                                        o[4 * g4 + 3] = fmaf(coef, o[4 * g4 + 3], -v.w);
                                    }
                                }
                            }
                        }
                        if (p.sparse == nullptr && p.coef != nullptr) {
                            // row scale only (the target side's q W of the combined objective)
#pragma unroll
                            for (int j = 0; j < 32; ++j) o[j] *= coef;
                        }
                        if (p.out_fp32) {
                            float* dst = reinterpret_cast<float*>(p.out) + static_cast<long long>(g_row) * p.out_pitch + col0;
                            if (full && p.out_align32) {
#pragma unroll
                                for (int g8 = 0; g8 < 4; ++g8)
                                    st_global_v8(dst + 8 * g8, __float_as_uint(o[8 * g8]), __float_as_uint(o[8 * g8 + 1]),
                                                 __float_as_uint(o[8 * g8 + 2]), __float_as_uint(o[8 * g8 + 3]),
                                                 __float_as_uint(o[8 * g8 + 4]), __float_as_uint(o[8 * g8 + 5]),
                                                 __float_as_uint(o[8 * g8 + 6]), __float_as_uint(o[8 * g8 + 7]));
                            } else {
#pragma unroll
                                for (int g4 = 0; g4 < 8; ++g4)
                                    if (col0 + 4 * g4 < p.n_cols)
                                        *reinterpret_cast<float4*>(dst + 4 * g4) =
                                            make_float4(o[4 * g4], o[4 * g4 + 1], o[4 * g4 + 2], o[4 * g4 + 3]);
                            }
                        } else {
                            __nv_bfloat16* dst = reinterpret_cast<__nv_bfloat16*>(p.out) + static_cast<long long>(g_row) * p.out_pitch + col0;
                            if (full && p.out_align32) {
#pragma unroll
                                for (int g16 = 0; g16 < 2; ++g16)
                                    st_global_v8(dst + 16 * g16, pack_bf16x2(o[16 * g16 + 0], o[16 * g16 + 1]),
                                                 pack_bf16x2(o[16 * g16 + 2], o[16 * g16 + 3]),
                                                 pack_bf16x2(o[16 * g16 + 4], o[16 * g16 + 5]),
                                                 pack_bf16x2(o[16 * g16 + 6], o[16 * g16 + 7]),
                                                 pack_bf16x2(o[16 * g16 + 8], o[16 * g16 + 9]),
                                                 pack_bf16x2(o[16 * g16 + 10], o[16 * g16 + 11]),
                                                 pack_bf16x2(o[16 * g16 + 12], o[16 * g16 + 13]),
                                                 pack_bf16x2(o[16 * g16 + 14], o[16 * g16 + 15]));
                            } else {
#pragma unroll
                                for (int g8 = 0; g8 < 4; ++g8) {
                                    if (col0 + 8 * g8 < p.n_cols) {
                                        uint4 w;
                                        w.x = pack_bf16x2(o[8 * g8 + 0], o[8 * g8 + 1]);
                                        w.y = pack_bf16x2(o[8 * g8 + 2], o[8 * g8 + 3]);
                                        w.z = pack_bf16x2(o[8 * g8 + 4], o[8 * g8 + 5]);
                                        w.w = pack_bf16x2(o[8 * g8 + 6], o[8 * g8 + 7]);
                                        *reinterpret_cast<uint4*>(dst + 8 * g8) = w;
                                    }
                                }
                            }
                        }
                    }
                }
                // accumulator drained: hand the buffer back to the MMA warp
                tc_fence_before_sync();
                __syncwarp();
                if (lane == 0) {
                    if (CG == 2)
                        mbar_arrive_cluster(map_to_rank(tempty_bar(ab), 0));
                    else
                        mbar_arrive(tempty_bar(ab));
                }
                ab ^= 1;
                if (ab == 0) aphase ^= 1u;
                if (MODE == MODE_STATS && want_topk && (S > 1 || !USE_REG)) {
                    // Bounds of the row's K-th largest logit, from what this lane and the others have met so far: the K-th
                    // largest of ANY lane's part of the row, and (TOPK_BUF) the least of ALL lanes' share-th largest, share =
                    // ceil(K / S): S lanes with so many logits above a bound are K logits. The second is the tighter one: after the
                    // first tile it leaves about K / S of a tile's logits to a lane instead of K, the buffers hardly fill any more and the
                    // warp compacts next to nothing. 2047 rows x 4096 x 32000, sweep with K = 100 and nine lanes 497 -> 395 us, call 1815 -> 1705;
                    // 4096 rows, K = 64, four lanes: call 2670 -> 2510. (The register lists of K <= 16 admit too little for it to show.)
                    // It pays from a third tile on: with 74 lanes of one or two tiles the work behind a tile costs as much as it
                    // saves (130 rows, K = 20: 218.6 us without, 230 with it; 200 rows, K = 100 294 and 318; 242 rows, K = 36 277 and 268).
                    // A logit equal to a foreign bound must still be admitted (ties are settled by token id when the lists
                    // are merged), hence the step just below it. Stale or missing (zero) values only leave the threshold
                    // lower than it could be.
                    float part = thr_own;
                    if constexpr (!USE_REG) if (joint && hist_inv > 0.f && t >= 0) {
                        // the first tile's logits are all in the histogram; of a later one's, those admitted follow here
                        if (t == 0) counted = cnt;
                        while (counted < cnt) {
                            uint2 e[8];
#pragma unroll
                            for (int i = 0; i < 8; ++i)
                                if (counted + i < cnt) e[i] = __ldcg(cbuf + counted + i);
#pragma unroll
                            for (int i = 0; i < 8; ++i)
                                if (counted + i < cnt) hist_count(pend_v, __uint_as_float(e[i].x), hist_lo, hist_inv);
                            counted += 8;
                        }
                        counted = cnt;
                        int top, top_share;
                        hist_top(pend_v, p.K, share, top, top_share);
                        if (top > 0) thr_own = fmaxf(thr_own, hist_lo + (static_cast<float>(top) - 0.5f) / hist_inv);
                        if (top_share > 0) part = hist_lo + (static_cast<float>(top_share) - 0.5f) / hist_inv;
                        part = fmaxf(part, thr_own);
                    }
                    if (S > 1) {
                        const long long at = static_cast<long long>(slot - ln) * BM + r_local;
                        const uint2 own = make_uint2(ordered_key(__float_as_uint(thr_own)), ordered_key(__float_as_uint(part)));      // (the first tile's bound is in thr_sh)
                        unsigned int best = 0u;
                        if (!joint) {
                            unsigned int* sh = p.thr_share + at;
                            st_relaxed(sh + static_cast<long long>(ln) * BM, own.x);
                            const int nn = t + 1 < nt ? (S - 1 < 3 ? S - 1 : 3) : 0;
                            for (int q = 1; q <= nn; ++q) best = max(best, ld_relaxed(sh + static_cast<long long>((ln + q) % S) * BM));
                        } else {
                            uint2* sh = p.bounds + at;
                            st_relaxed_v2(sh + static_cast<long long>(ln) * BM, own);
                            if (t + 1 < nt) {
                                // eight loads in flight (one by one they take as long as the tile's candidates)
                                unsigned int least = own.y;
                                for (int q0 = 0; q0 < S; q0 += 8) {
                                    uint2 v[8];
#pragma unroll
                                    for (int i = 0; i < 8; ++i) v[i] = ld_relaxed_v2(sh + static_cast<long long>(q0 + i < S ? q0 + i : ln) * BM);
#pragma unroll
                                    for (int i = 0; i < 8; ++i) {
                                        best = max(best, v[i].x);
                                        least = min(least, v[i].y);
                                    }
                                }
                                best = max(best, least);
                            }
                        }
                        if (best != 0u) thr_sh = fmaxf(thr_sh, nextafterf(__uint_as_float(key_bits(best)), -INFINITY));
                    }
                    thr = fmaxf(thr_own, fmaxf(thr, thr_sh));
                }
            }
            if constexpr (EW == 8) {
                // The second thread of a row hands over m, s and its list through the staging area; the first adds them to its own.
                static_assert(PEND == 256 * 4, "meet_word's columns");
                auto word = [&](int e) { return spill_stage + meet_word(USE_REG, threadIdx.x, e); };
                if (half == 1) {
                    if (TOPK == TOPK_NONE && lane == 0) bulk_wait_group_read<0>();      // (its own staging buffers have been read)
                    __syncwarp();
                    // the first threads' staging buffers and pending logits lie there too: they say when the room is free
                    if (!__all_sync(0xffffffffu, wait_barrier(meet_bar(1), meet_phase, abort_flag, p.status, 5))) return false;
                    st_shared_b32(word(0), __float_as_uint(m));
                    st_shared_b32(word(1), __float_as_uint(s));
                    if (USE_REG) {
#pragma unroll
                        for (int k = 0; k < (USE_REG ? K_REG : 1); ++k) {
                            st_shared_b32(word(2 + 2 * k), __float_as_uint(tv[k]));
                            st_shared_b32(word(3 + 2 * k), static_cast<uint32_t>(ti[k]));
                        }
                    }
                    __syncwarp();
                    if (lane == 0) mbar_arrive(meet_bar(0));
                    if (!__all_sync(0xffffffffu, wait_barrier(meet_bar(1), meet_phase ^ 1u, abort_flag, p.status, 6))) return false;
                    if (spill && track_zmax && !p.use_row_zmax) atomicMax(p.row_zmax + rt * BM + r_local, ordered_key(__float_as_uint(zmax)));
                    return true;
                }
                if (TOPK == TOPK_NONE && lane == 0) bulk_wait_group_read<0>();
                __syncwarp();
                if (lane == 0) mbar_arrive(meet_bar(1));
                if (!__all_sync(0xffffffffu, wait_barrier(meet_bar(0), meet_phase, abort_flag, p.status, 5))) return false;
                meet_phase ^= 1u;
                const float m2 = __uint_as_float(ld_shared_b32(word(0))), s2 = __uint_as_float(ld_shared_b32(word(1)));
                if (spill) {
                    s += s2;      // (of the same reference)
                } else {
                    const float top = fmaxf(m, m2), base = top == -INFINITY ? 0.f : top;
                    s = s * ex2((m - base) * LOG2E) + s2 * ex2((m2 - base) * LOG2E);
                    m = top;
                }
                if (USE_REG) {
                    // the 16 best of both lists, which are sorted (larger logit first, of equal ones the lower token): best of k and 15 - k,
                    // then the last steps of a sorting network
                    auto before = [](float xv, int xi, float yv, int yi) { return xv > yv || (xv == yv && static_cast<uint32_t>(xi) < static_cast<uint32_t>(yi)); };
#pragma unroll
                    for (int k = 0; k < (USE_REG ? K_REG : 1); ++k) {
                        const float ov = __uint_as_float(ld_shared_b32(word(2 + 2 * (K_REG - 1 - k))));
                        const int oi = static_cast<int>(ld_shared_b32(word(3 + 2 * (K_REG - 1 - k))));
                        const bool mine = before(tv[k], ti[k], ov, oi);
                        tv[k] = mine ? tv[k] : ov;
                        ti[k] = mine ? ti[k] : oi;
                    }
#pragma unroll
                    for (int j = K_REG / 2; j > 0; j /= 2)
#pragma unroll
                        for (int k = 0; k < (USE_REG ? K_REG : 1); ++k) {
                            const int l = k ^ j;
                            if (l > k && l < (USE_REG ? K_REG : 1)) {
                                const bool keep = before(tv[k], ti[k], tv[l], ti[l]);
                                const float hv = keep ? tv[k] : tv[l], lv = keep ? tv[l] : tv[k];
                                const int hi_ = keep ? ti[k] : ti[l], li = keep ? ti[l] : ti[k];
                                tv[k] = hv;
                                ti[k] = hi_;
                                tv[l] = lv;
                                ti[l] = li;
                            }
                        }
                }
                __syncwarp();
                if (lane == 0) mbar_arrive(meet_bar(1));
            }
            if (MODE == MODE_STATS && tile_ok) {
                const long long so = static_cast<long long>(slot) * BM + r_local;
                p.part_m[so] = m;
                p.part_s[so] = s;
                // the row's logits spread too far above its reference for the fixed-exponent spill
                if (spill && !(s < SPILL_SUM_LIMIT)) atomicExch(p.status + 1, 1u);
                if (track_zmax && !p.use_row_zmax) atomicMax(p.row_zmax + rt * BM + r_local, ordered_key(__float_as_uint(zmax)));
                if (USE_REG && want_topk) {
                    // the register list goes out as a full buffer of K_REG entries (unused ones carry id -1)
#pragma unroll
                    for (int k = 0; k < (USE_REG ? K_REG : 1); ++k)
                        cbuf[k] = make_uint2(__float_as_uint(tv[k]), static_cast<uint32_t>(ti[k]));
                    cnt = K_REG;
                }
                if (want_topk) p.cand_n[static_cast<long long>(slot) * BM + r_local] = cnt;
            }
            return true;
        });
        // shared memory must outlive the TMA stores that read it
        if (MODE == MODE_STATS && TOPK == TOPK_NONE && lane == 0) bulk_wait_group0();
    }

    if constexpr (MODE == MODE_OUT && CG == 1) {
        const int C = p.plan.cluster;
        if (C > 1) {
            // The operand stages hold [C pieces][rows per CTA][ROW_PITCH] floats now: every CTA's products are complete.
            const int width = tile_width(0), ROW_PITCH = width + 4;               // rows 4 banks apart
            static_assert((BM + 8) * (BN + 4) * 4 <= OPERAND_BYTES, "the pieces of a CTA's rows fit the operand stages");
            const int u = cta / C, z = cta - u * C;
            const int rt = u % p.plan.row_units, ct = u / p.plan.row_units;
            const int per = piece_rows(min(BM, p.rows_valid - p.row_global_offset - rt * BM), C);      // (rows that exist are dealt out)
            tc_fence_before_sync();
            __syncthreads();
            cluster_sync();
            tc_fence_after_sync();
            if (warp >= 2) {
                const int quad = warp & 3, r = quad * 32 + lane;
                const uint32_t dst = map_to_rank(smem_base + (z * per + r % per) * ROW_PITCH * 4, piece_rank(r, per, C));
                const bool row_ok = p.row_global_offset + rt * BM + r < p.rows_valid;
#pragma unroll 1
                for (int ch = 0; ch < width / 32; ++ch) {
                    uint32_t v[32];
                    tmem_ld32(tmem_base + (static_cast<uint32_t>(quad * 32) << 16) + ch * 32, v);
                    tmem_ld_wait(v);
                    if (row_ok) {
#pragma unroll
                        for (int j = 0; j < 8; ++j) st_cluster_v4(dst + (ch * 32 + 4 * j) * 4, v[4 * j], v[4 * j + 1], v[4 * j + 2], v[4 * j + 3]);
                    }
                }
            }
            cluster_sync();
            for (int i = threadIdx.x; i < per * (width / 4); i += NUM_THREADS) {
                const int rl = i / (width / 4), c = i % (width / 4) * 4;
                const int r = z * per + rl, row = p.row_global_offset + rt * BM + r, col = ct * width + c;
                if (r >= BM || row >= p.rows_valid || col >= p.n_cols) continue;
                const uint8_t* src = smem_gen + (rl * ROW_PITCH + c) * 4;
                float4 a = *reinterpret_cast<const float4*>(src);
                for (int q = 1; q < C; ++q) {
                    const float4 v = *reinterpret_cast<const float4*>(src + q * per * ROW_PITCH * 4);
                    a.x += v.x; a.y += v.y; a.z += v.z; a.w += v.w;
                }
                finish_out4(p, a, rt * BM + r, row, col);
            }
        }
    }

    // ---- teardown ----
    tc_fence_before_sync();
    __syncthreads();
    if (*abort_flag) {
        // a wait gave up: let copies that may still be in flight land before the CTA's memory is released
        const unsigned long long t0 = globaltimer_ns();
        while (globaltimer_ns() - t0 < 200000ull) __nanosleep(1000);
    }
    if (CG == 2) cluster_sync();      // the partner's products, loads and arrivals on this CTA's memory are done
    if (warp == 1) {
        tc_fence_after_sync();
        if (CG == 2)
            tmem_dealloc_pair(tmem_base, TMEM_COLS);
        else
            tmem_dealloc(tmem_base, TMEM_COLS);
    }
}

// ---------------------------------------------------------------------------------------------
// out_reduce_kernel: adds up the partial tiles of MODE_OUT in the order of the contraction and finishes them as its
// epilogue does. One thread per four columns; memory-bound (reads cuts x, writes 1 x the rest tiles).
__global__ void __launch_bounds__(256) out_reduce_kernel(const __grid_constant__ GemmParams p) {
    wait_previous_kernel();
    if (p.gate != nullptr && *p.gate == 0u) return;
    const OutPlan& o = p.plan;
    const long long i = static_cast<long long>(blockIdx.x) * 256 + threadIdx.x;
    const int c = static_cast<int>(i % (BN / 4)) * 4;
    const int r_local = static_cast<int>(i / (BN / 4) % BM);
    const int tile = static_cast<int>(i / (BN / 4 * BM));             // rest tile * pair + rank
    const int u = o.whole + tile / o.pair;
    const int rt = u % o.row_units * o.pair + tile % o.pair;
    const int col = u / o.row_units * BN + c;
    const int row = p.row_global_offset + rt * BM + r_local;
    if (tile >= o.rest * o.pair || rt >= p.row_tiles || row >= p.rows_valid || col >= p.n_cols) return;
    const float4* src = reinterpret_cast<const float4*>(p.part + (static_cast<long long>(tile) * o.part_rows + r_local) * BN + c);
    const long long step = static_cast<long long>(o.rest) * o.pair * o.part_rows * (BN / 4);
    float4 a = src[0];
#pragma unroll 4
    for (int z = 1; z < o.cuts; ++z) {
        const float4 v = src[z * step];
        a.x += v.x; a.y += v.y; a.z += v.z; a.w += v.w;
    }
    finish_out4(p, a, rt * BM + r_local, row, col);
}

// ---------------------------------------------------------------------------------------------
// finalize: the routes that do not know Omega_hat before their sweep of the draft rows. Merges the draft's partial
// statistics into lse_d, gathers the draft logits at Omega_hat with dot products, and evaluates Eq. 1.
struct FinalizeParams {
    Schedule sched;
    int d, K;
    int row_begin, rows;   // global rows [row_begin, row_begin + rows) = local row tiles 0.. of the schedule
    int row_tiles_t;       // row tiles of the target matrix in the schedule, before the draft's
    const float* part_m;
    const float* part_s;
    const __nv_bfloat16* H_d;
    const __nv_bfloat16* W;
    int* idx;              // [N, idx_pitch] Omega_hat in descending q, from select_kernel or the caller
    float* q;              // (bidir: the joining tokens are added behind the K of the target)
    int idx_pitch;
    const float* lse_t;    // (read by the combined objective and Bi-directional Top-K)
    float* loss;
    float* lse_d;
    // fused backward (all nullable): per-row scale of the spilled tiles and the Omega_hat term
    const float* grad_loss;
    float* coef_out;       // [N]   g * S_q * exp(m_spill - lse_d), m_spill = the row's spill reference
    float* sparse_out;     // [rows, d] sum_{x in Omega_hat} g q(x) W[x, :], indexed by local row
    // combined objective CE(q, p) + w * Top-K (coef_t_out != nullptr): the target tiles were spilled as well
    float w_topk;          // weight w of the Top-K term
    float* coef_t_out;     // [N] e^(m_spill_t - lse_t): scale that turns (target spill x W) into q W
    const __nv_bfloat16* Pt;   // target spill of the chunk [rows, p_pitch]
    long long p_pitch;
    float* ce_corr_out;    // [N] sum_{x in Omega_hat} (q(x) - bf16 q(x)) z_d(x): the cross-entropy is formed from
                           // the bf16 spill; its largest terms are put back in fp32
    // loss variants of Section 4.3
    int* n_out;            // [N] |Omega_hat| (bidir, nullable)
    const int* idx_d;      // bidir: [N, K] the draft's K most probable tokens in descending p; those outside the target's
                           // set join Omega_hat (idx / q have 2K entries per row)
    const __nv_bfloat16* H_t;   // target features (bidir: target logits of the draft's tokens)
    const unsigned int* gate;            // as in GemmParams
};

__device__ __forceinline__ void find_slots(const Schedule& sc, int row_tile, int& slot0, int& S) {
    slot0 = 0;
    S = 0;
    for (int ph = 0; ph < sc.n_phases; ++ph) {
        const Phase P = sc.ph[ph];
        if (row_tile >= P.row_tile_begin && row_tile < P.row_tile_begin + P.G) {
            slot0 = P.slot_base + (row_tile - P.row_tile_begin) * P.S;
            S = P.S;
            return;
        }
    }
}

__device__ __forceinline__ float warp_lse(const float* pm, const float* ps, int slot0, int S, int r, int lane) {
    float m = -INFINITY;
    for (int j = lane; j < S; j += 32) m = fmaxf(m, pm[static_cast<long long>(slot0 + j) * BM + r]);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    float s = 0.f;
    for (int j = lane; j < S; j += 32) {
        const long long so = static_cast<long long>(slot0 + j) * BM + r;
        s += ps[so] * exp2f((pm[so] - m) * LOG2E);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    return m + logf(s);
}

constexpr int FIN_GRP = 8;        // tokens of Omega_hat whose W rows finalize reads together
constexpr int FIN_WARPS = 8;      // warps that share a row

__device__ __forceinline__ void unpack8(const uint4& v, float (&f)[8]) {
    const __nv_bfloat162* p2 = reinterpret_cast<const __nv_bfloat162*>(&v);
#pragma unroll
    for (int t = 0; t < 4; ++t) {
        const float2 f2 = __bfloat1622float2(p2[t]);
        f[2 * t] = f2.x;
        f[2 * t + 1] = f2.y;
    }
}

// Groups of a block's threads that take tokens of their own in a gather, where its part of the columns is `units` units of eight: as many as have a
// warp or more per eight columns; 1: all threads share the columns
__host__ __device__ constexpr int gather_groups(int units, int threads) {
    const int warps = (units + 31) / 32;
    return threads / 32 / (warps < 1 ? 1 : warps > threads / 32 ? threads / 32 : warps);
}

// Dynamic shared memory of a kernel whose blocks gather `units` units of eight columns each, or more: the groups' sums, where any block has
// groups (with wide rows the space is left to the L1)
__host__ __device__ constexpr int gather_smem(int units) { return gather_groups(units, FIN_WARPS * 32) > 1 ? 8 * FIN_WARPS * 32 * 4 : 0; }

// Eight columns of the rows of W of tokens tok[0 .. n), n <= FIN_GRP: dot[j] += <h, row j>, a += gw q[j] row j (q nullable).
__device__ __forceinline__ void gather_unit(const __nv_bfloat16* W, long long d, const int* tok, int n, const float (&h)[8], float (&dot)[FIN_GRP],
                                            const float* q, float gw, float (&a)[8]) {
    uint4 wv[FIN_GRP];
#pragma unroll
    for (int jj = 0; jj < FIN_GRP; ++jj)
        if (jj < n) wv[jj] = *reinterpret_cast<const uint4*>(W + tok[jj] * d);
#pragma unroll
    for (int jj = 0; jj < FIN_GRP; ++jj) {
        if (jj < n) {
            float wf[8];
            unpack8(wv[jj], wf);
            const float gq = q ? gw * q[jj] : 0.f;
#pragma unroll
            for (int t = 0; t < 8; ++t) {
                dot[jj] = fmaf(h[t], wf[t], dot[jj]);
                a[t] = fmaf(gq, wf[t], a[t]);
            }
        }
    }
}

// Block-collective: over the columns 8 u0 .. 8 u1 - 1, the dot products of row `from` with the rows of W of tokens [b0, n) into to[b0 .. n), and
// with `so` the row sum over [0, n) of gw q[j] W[tok[j], :] into so (then b0 = 0). FIN_GRP rows of W are in flight per thread. Of narrow rows
// groups of threads take FIN_GRP tokens each, with their columns' sums in registers to the end (one group had a warp of eight at work on 256
// columns: Bi-directional call of 2795 rows x 256 x 1024, K = 41 223 -> 183 us, combined 1318 x 376 x 38201, K = 65 658 -> 621).
__device__ __forceinline__ void gather_rows(const __nv_bfloat16* from, const __nv_bfloat16* W, int d, int u0, int u1, const int* tok, int b0, int n,
                                            float* to, const float* q, float gw, float* so, float (&part)[FIN_WARPS][K_CAP], float* cols) {
    constexpr int THREADS = FIN_WARPS * 32;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int per = max(32, min((u1 - u0 + 31) / 32 * 32, THREADS)), groups = gather_groups(u1 - u0, THREADS), g = tid / per;
    // eight sums over the warp at once, sum (lane >> 2) in the end: at each step half of the values go to the other half of the lanes
    auto warp_sums = [&](float (&dot)[FIN_GRP]) {
        static_assert(FIN_GRP == 8, "lane bits 4, 3, 2 say which sum");
#pragma unroll
        for (int h = 4; h > 0; h >>= 1) {
            const bool up = (lane & (4 * h)) != 0;
#pragma unroll
            for (int i = 0; i < h; ++i) {
                const float other = __shfl_xor_sync(0xffffffffu, up ? dot[i] : dot[i + h], 4 * h);
                dot[i] = (up ? dot[i + h] : dot[i]) + other;
            }
        }
        dot[0] += __shfl_xor_sync(0xffffffffu, dot[0], 2);
        dot[0] += __shfl_xor_sync(0xffffffffu, dot[0], 1);
    };
    if (groups == 1 && n - b0 > FIN_GRP) {
        // a thread's columns in turn, all tokens for each, so that their sum stays in registers; a warp adds its dot products up in its own part of
        // `part`, and the block meets once. With the tokens in turn and the columns' sum in memory in between, finalize and the selections of
        // 2048 Bi-directional rows x 4096, K = 10 took 139 us, now 133; 300 x 8192, K = 41 215 -> 205, 2795 x 1040, K = 41 250 -> 226. (The rows of W
        // come at 4.7 TB/s, from the L2 and from memory; up to FIN_GRP tokens one turn is all there is, below: 1000 x 5120, K = 3 73 us this way, 59 that.)
        for (int a0 = u0; a0 < u1; a0 += THREADS) {
            const int at = a0 + tid;
            const bool mine = at < u1;
            float h[8] = {}, a[8] = {};
            if (mine) unpack8(*reinterpret_cast<const uint4*>(from + 8 * at), h);
            for (int b = b0; b < n; b += FIN_GRP) {
                float dot[FIN_GRP] = {};
                if (mine) gather_unit(W + 8 * at, d, tok + b, n - b, h, dot, so ? q + b : nullptr, gw, a);
                warp_sums(dot);
                if ((lane & 3) == 0 && b + (lane >> 2) < n) {
                    float* const sum = &part[warp][b + (lane >> 2)];
                    *sum = a0 == u0 ? dot[0] : *sum + dot[0];
                }
            }
            if (so && mine) {
                float4* s4 = reinterpret_cast<float4*>(so + 8 * at);
                s4[0] = make_float4(a[0], a[1], a[2], a[3]);
                s4[1] = make_float4(a[4], a[5], a[6], a[7]);
            }
        }
        __syncthreads();
        for (int j = b0 + tid; j < n; j += THREADS) {
            float acc = 0.f;
#pragma unroll
            for (int w = 0; w < FIN_WARPS; ++w) acc += part[w][j];
            to[j] = acc;
        }
        __syncthreads();
        return;
    }
    // the sums of a group's dot products over its threads
    auto finish = [&](float (&dot)[FIN_GRP], int b, int each) {
        warp_sums(dot);
        if ((lane & 3) == 0) part[warp][lane >> 2] = dot[0];
        __syncthreads();
        if (tid < groups * each && b + tid < n) {
            float acc = 0.f;
            for (int w = 0; w < per / 32; ++w) acc += part[tid / each * (per / 32) + w][tid % each];
            to[b + tid] = acc;
        }
        __syncthreads();
    };
    if (groups == 1) {
        float dot[FIN_GRP] = {};
        for (int at = u0 + tid; at < u1; at += THREADS) {
            float h[8], a[8] = {};
            unpack8(*reinterpret_cast<const uint4*>(from + 8 * at), h);
            gather_unit(W + 8 * at, d, tok + b0, n - b0, h, dot, so ? q + b0 : nullptr, gw, a);
            if (so) {
                float4* s4 = reinterpret_cast<float4*>(so + 8 * at);
                s4[0] = make_float4(a[0], a[1], a[2], a[3]);
                s4[1] = make_float4(a[4], a[5], a[6], a[7]);
            }
        }
        finish(dot, b0, FIN_GRP);
        return;
    }
    const int u = u0 + tid - g * per;
    const bool mine = g < groups && u < u1;
    float h[8] = {}, a[8] = {};
    if (mine) unpack8(*reinterpret_cast<const uint4*>(from + 8 * u), h);
    for (int b = b0; b < n; b += groups * FIN_GRP) {
        const int each = min((n - b + groups - 1) / groups, FIN_GRP), bg = b + g * each;      // a group's tokens, this group's first
        float dot[FIN_GRP] = {};
        if (mine) gather_unit(W + 8 * u, d, tok + bg, min(n - bg, each), h, dot, so ? q + bg : nullptr, gw, a);
        finish(dot, b, each);
    }
    if (so) {
        // the groups' sums in order
#pragma unroll
        for (int t = 0; t < 8; ++t) cols[t * THREADS + tid] = a[t];
        __syncthreads();
        if (g == 0 && mine) {
            for (int o = 1; o < groups; ++o)
#pragma unroll
                for (int t = 0; t < 8; ++t) a[t] += cols[t * THREADS + tid + o * per];
            float4* s4 = reinterpret_cast<float4*>(so + 8 * u);
            s4[0] = make_float4(a[0], a[1], a[2], a[3]);
            s4[1] = make_float4(a[4], a[5], a[6], a[7]);
        }
        __syncthreads();
    }
}

// One block per row (2048 rows, 20 tokens, d = 4096: 390 us with a warp per row and a serial selection -> 158 us, and 24 us
// in select_kernel; 1024 rows, 10 tokens: 144 -> 55 us; with eight warps instead of four, eight tokens instead of sixteen
// and three blocks per SM another 10-20 %): bound by the latency of the gathered rows of W, so that a row's columns are spread over FIN_WARPS
// warps (8 columns per thread and step) and FIN_GRP rows of W are in flight per thread.
__global__ void __launch_bounds__(FIN_WARPS * 32, 3) finalize_kernel(const __grid_constant__ FinalizeParams p) {
    wait_previous_kernel();
    if (p.gate != nullptr && *p.gate == 0u) return;
    __shared__ int sh_tok[K_CAP];         // Omega_hat of the row (the bi-directional set needs 2K <= K_CAP)
    __shared__ float sh_q[K_CAP];
    __shared__ float sh_dot[K_CAP];       // z_d at Omega_hat
    __shared__ float sh_part[FIN_WARPS][K_CAP];
    extern __shared__ float sh_cols[];
    __shared__ int sh_n;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int local = blockIdx.x;
    const int row = p.row_begin + local;
    const int rt = local / BM, r = local % BM;
    const int K = p.K;
    auto warp_sum = [](float v) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        return v;
    };

    // draft statistics
    int slot0, S;
    find_slots(p.sched, p.row_tiles_t + rt, slot0, S);
    const float lse_d = warp_lse(p.part_m, p.part_s, slot0, S, r, lane);
    const float m_spill = p.part_m[static_cast<long long>(slot0) * BM + r];
    const float g = p.grad_loss ? p.grad_loss[row] : 1.f;
    const bool combined = p.coef_t_out != nullptr;
    float coef_t = 0.f;
    if (combined) {
        find_slots(p.sched, rt, slot0, S);
        coef_t = expf(p.part_m[static_cast<long long>(slot0) * BM + r] - p.lse_t[row]);
    }
    const float gw = combined ? g * p.w_topk : g;     // weight of the Omega_hat term q 1[Omega_hat] in dz_d

    const __nv_bfloat16* hrow = p.H_d + static_cast<long long>(row) * p.d;
    const long long io = static_cast<long long>(row) * p.idx_pitch;
    for (int j = tid; j < K; j += FIN_WARPS * 32) {
        const int tok = p.idx[io + j];
        sh_tok[j] = tok < 0 ? 0 : tok;                // (cut entries carry q = 0)
        sh_q[j] = p.q[io + j];
    }
    __syncthreads();

    int Ku = K;                                       // |Omega_hat| (2K at most for the bi-directional set)
    if (p.idx_d != nullptr) {
        // the draft's own K most probable tokens that are not in the target's set join Omega_hat, in their order
        if (warp == 0) {
            int n = K;
            for (int j0 = 0; j0 < K; j0 += 32) {
                const int j = j0 + lane;
                const int tok = j < K ? p.idx_d[static_cast<long long>(row) * K + j] : -1;
                bool joins = j < K;
                for (int t = 0; t < K; ++t) joins = joins && sh_tok[t] != tok;
                const uint32_t bm = __ballot_sync(0xffffffffu, joins);
                if (joins) sh_tok[n + __popc(bm & ((1u << lane) - 1u))] = tok;
                n += __popc(bm);
            }
            if (lane == 0) sh_n = n;
        }
        __syncthreads();
        Ku = sh_n;
        // their target probabilities: q = exp(<H_t[row], W[tok]> - lse_t)
        const float lse_t = p.lse_t[row];
        gather_rows(p.H_t + static_cast<long long>(row) * p.d, p.W, p.d, 0, p.d / 8, sh_tok, K, Ku, sh_q, nullptr, 0.f, nullptr, sh_part, sh_cols);
        for (int j = K + tid; j < 2 * K; j += FIN_WARPS * 32) {
            const float qv = j < Ku ? expf(sh_q[j] - lse_t) : 0.f;
            if (j < Ku) sh_q[j] = qv;
            p.idx[io + j] = j < Ku ? sh_tok[j] : -1;
            p.q[io + j] = qv;
        }
        if (tid == 0 && p.n_out) p.n_out[row] = Ku;
        __syncthreads();
    }
    // draft logits at Omega_hat and, for the fused backward, the row sum_{x in Omega_hat} g q(x) W[x, :]
    float* so = p.sparse_out ? p.sparse_out + static_cast<long long>(local) * p.d : nullptr;
    gather_rows(hrow, p.W, p.d, 0, p.d / 8, sh_tok, 0, Ku, sh_dot, sh_q, gw, so, sh_part, sh_cols);

    float S_q = 0.f;
    for (int j = lane; j < Ku; j += 32) S_q += sh_q[j];
    S_q = warp_sum(S_q);
    if (warp == 0) {
        float loss = 0.f, ce_corr = 0.f;
        for (int j = lane; j < Ku; j += 32) {
            loss += sh_q[j] * (lse_d - sh_dot[j]);    // -q log p,  log p = z_d - lse_d
            if (combined) {
                const float q_spill = __bfloat162float(p.Pt[static_cast<long long>(local) * p.p_pitch + sh_tok[j]]) * coef_t;
                ce_corr += (sh_q[j] - q_spill) * sh_dot[j];
            }
        }
        loss = warp_sum(loss);
        ce_corr = warp_sum(ce_corr);
        if (lane == 0) {
            p.loss[row] = loss;
            p.lse_d[row] = lse_d;
            if (combined) {
                p.ce_corr_out[row] = ce_corr;
                p.coef_t_out[row] = coef_t;
            }
            // dense part of dz_d: g S_q p (Top-K loss) or g (1 + w S_q) p (combined objective)
            if (p.coef_out) p.coef_out[row] = (combined ? g * (1.f + p.w_topk * S_q) : g * S_q) * expf(m_spill - lse_d);
        }
    }
}

// ---------------------------------------------------------------------------------------------
// select_kernel: between the sweep of the target rows and the sweep of the draft rows of the fused call. Merges the
// target's partial statistics into lse_t, picks Omega_hat from the sweep's candidates (or takes it as an input), writes
// topk_idx / topk_q in descending q, and leaves the same set sorted by token id (sidx, sq) for the draft sweep, which
// copies z_d at those tokens out of its accumulators.
// Bound by load latency: the lists of the row's lanes are read 256 entries at a time per warp (32 lanes x SEL_LOADS loads in
// flight) and what lies below the best K-th logit of any list is dropped on the way. WARPS warps share a row: one where
// there are rows enough to fill the GPU, four or sixteen where few rows have lists of up to 148 lanes each. A block has
// four warps, or the sixteen of its row.
__host__ __device__ constexpr int sel_block_warps(int WARPS) { return WARPS > 4 ? WARPS : 4; }
constexpr int SEL_LOADS = 8;          // candidate loads a lane has in flight
constexpr int SEL_FIRST = 5;          // lists per lane whose first entries set the floor (the first 160 of the row)

struct SelectParams {
    Schedule sched;        // schedule of the sweep; its row tile first_tile + t = rows [128 t, 128 t + 128) of the chunk
    int first_tile;
    int K, cap;
    int row_begin, rows;   // global rows [row_begin, row_begin + rows)
    int from_sweep;        // 1: Omega_hat from the sweep's candidates; 0: idx_in / q_in are given
    int out_pitch;         // entries per row of idx_out / q_out
    const float* part_m;
    const float* part_s;
    const uint2* cand;
    const int* cand_n;
    const unsigned int* thr_share;    // as the sweep left them (GemmParams)
    const uint2* bounds;
    int col_tiles;
    const int* idx_in;     // [N, K]
    const float* q_in;
    int* idx_out;          // [N, K] (from_sweep)
    float* q_out;
    float* lse_t;          // (nullable)
    int* n_out;            // [N] |Omega_hat| (nullable)
    float top_p;           // > 0: Omega_hat is cut to the shortest sorted prefix with cumulative q > top_p
    int* sidx;             // [N, K] Omega_hat in increasing token id; unused entries INT_MAX (nullable)
    float* sq;             // [N, K] q in the same order; unused entries 0
    unsigned int* zmax;    // [chunk row] set to zero for the draft sweep (nullable)
    const unsigned int* gate;
    // Reference exponent of the row's spill (nullable ref2): z_d at the most probable token of Omega_hat, a logit that the
    // draft sweep will meet, so that the row's largest is never below it
    const __nv_bfloat16* H_d;
    const __nv_bfloat16* W;
    int d, V;
    float* ref2;           // [N] z_d log2e + 64
};

// A candidate as one number: larger = larger logit, lower token id first among equal logits.
__device__ __forceinline__ unsigned long long cand_rank(uint32_t key, uint32_t id) {
    return (static_cast<unsigned long long>(key) << 32) | (~id);
}

// Cuts the candidates (distinct numbers) in the pools of WARPS warps, n in this warp's `pool`, total > K of them, to the
// K best and at most `slack` more, in place, and returns the bound that those kept reach. The bound is searched from the
// highest bit in which the numbers differ, two bits per step. Collective over the WARPS warps; sh: CUT_WORDS words of
// shared memory that the block uses for nothing else (WARPS > 1 only; the block is then these warps).
constexpr int CUT_WORDS = 12;
template <int WARPS>
__device__ __forceinline__ unsigned long long cut_to_best(unsigned long long* pool, int& n, int K, int slack, int lane, uint32_t* sh) {
    uint32_t hi = 0u, lo = 0xffffffffu;
    for (int e = lane; e < n; e += 32) {
        const uint32_t k = static_cast<uint32_t>(pool[e] >> 32);
        hi = max(hi, k);
        lo = min(lo, k);
    }
    hi = __reduce_max_sync(0xffffffffu, hi);
    lo = __reduce_min_sync(0xffffffffu, lo);
    if (WARPS > 1) {
        if (threadIdx.x < CUT_WORDS) sh[threadIdx.x] = threadIdx.x == 10 ? 0xffffffffu : 0u;
        __syncthreads();
        if (lane == 0) {
            atomicMax(sh + 9, hi);
            atomicMin(sh + 10, lo);
        }
        __syncthreads();
        hi = sh[9];
        lo = sh[10];
    }
    int bit = 64 - __clz(hi ^ lo);      // (equal logits: the token ids' 32 bits are left)
    bit += bit & 1;
    unsigned long long T = bit < 64 ? (static_cast<unsigned long long>(hi) << 32 >> bit) << bit : 0ull;
    int step = 0;                       // sums of step i in words 3 (i % 3) ..; those of the next step are cleared meanwhile
#pragma unroll 1
    for (bit -= 2; bit >= 0; bit -= 2) {
        const unsigned long long T1 = T | (1ull << bit), T2 = T | (2ull << bit), T3 = T | (3ull << bit);
        int c1 = 0, c2 = 0, c3 = 0;
#pragma unroll 4
        for (int e = lane; e < n; e += 32) {
            const unsigned long long v = pool[e];
            c1 += v >= T1 ? 1 : 0;
            c2 += v >= T2 ? 1 : 0;
            c3 += v >= T3 ? 1 : 0;
        }
        c1 = __reduce_add_sync(0xffffffffu, c1);
        c2 = __reduce_add_sync(0xffffffffu, c2);
        c3 = __reduce_add_sync(0xffffffffu, c3);
        if (WARPS > 1) {
            uint32_t* sum = sh + 3 * step;
            step = step == 2 ? 0 : step + 1;
            if (lane < 3) atomicAdd(sum + lane, static_cast<uint32_t>(lane == 0 ? c1 : lane == 1 ? c2 : c3));
            if (threadIdx.x < 3) sh[3 * step + threadIdx.x] = 0u;
            __syncthreads();
            c1 = static_cast<int>(sum[0]);
            c2 = static_cast<int>(sum[1]);
            c3 = static_cast<int>(sum[2]);
        }
        const int c = c3 >= K ? c3 : c2 >= K ? c2 : c1 >= K ? c1 : INT_MAX;
        T = c3 >= K ? T3 : c2 >= K ? T2 : c1 >= K ? T1 : T;
        if (c <= K + slack) break;
    }
    const uint32_t lt_mask = (1u << lane) - 1u;
    int np = 0;
    for (int e0 = 0; e0 < n; e0 += 32) {
        const int e = e0 + lane;
        const unsigned long long v = e < n ? pool[e] : 0ull;
        const bool take = e < n && v >= T;
        const uint32_t bm = __ballot_sync(0xffffffffu, take);
        if (take) pool[np + __popc(bm & lt_mask)] = v;      // position <= e: in place
        np += __popc(bm);
        __syncwarp();
    }
    n = np;
    return T;
}

template <int WARPS, int WIN>
__global__ void __launch_bounds__(sel_block_warps(WARPS) * 32) select_kernel(const __grid_constant__ SelectParams p) {
    static_assert(WIN >= (WIN > 512 ? K_CAP : K_REG) + 64 + 32 * SEL_LOADS, "a cut leaves room for one batch of loads");
    constexpr int BLOCK_WARPS = sel_block_warps(WARPS);
    constexpr int ROWS = BLOCK_WARPS / WARPS;                 // rows per block
    extern __shared__ unsigned long long sel_pools[];         // [BLOCK_WARPS][WIN]
    __shared__ int pool_n[BLOCK_WARPS];
    __shared__ uint32_t cut_words[CUT_WORDS];
    __shared__ int sel_tok[ROWS][K_CAP];                      // Omega_hat in descending q
    __shared__ float sel_q[ROWS][K_CAP];
    const int lane = threadIdx.x & 31;
    const int warp = threadIdx.x >> 5;
    const int rib = warp / WARPS, w = warp % WARPS;           // row in the block, warp of the row
    const int tid = w * 32 + lane;                            // thread of the row
    const int local = blockIdx.x * ROWS + rib;
    wait_previous_kernel();
    if (local >= p.rows || (p.gate != nullptr && *p.gate == 0u)) return;      // (WARPS > 1: the whole block)
    auto sync_row = [&]() {
        if (WARPS > 1)
            __syncthreads();
        else
            __syncwarp();
    };
    const int row = p.row_begin + local;
    const int rt = p.first_tile + local / BM, r = local % BM;
    const int K = p.K;
    const long long ro = static_cast<long long>(row) * K;
    if (p.zmax != nullptr && tid == 0) p.zmax[local] = 0u;

    if (p.from_sweep) {
        int slot0, S;
        find_slots(p.sched, rt, slot0, S);
        const bool lists = p.cap == K_REG;      // sorted register lists of K_REG entries (unused ones: id -1)
        const bool joint = p.bounds != nullptr && S > 1 && p.col_tiles > 2 * S;      // (as in the sweep)
        // lse_t, and a floor below which no candidate can be among the K best: the best K-th largest logit of any list,
        // or the K-th largest of the lists' first entries
        float m = -INFINITY, sum = 0.f;
        uint32_t floor_key = 0u, least_key = 0xffffffffu;
        uint32_t first[SEL_FIRST];
#pragma unroll
        for (int q = 0; q < SEL_FIRST; ++q) first[q] = 0u;
#pragma unroll
        for (int q = 0; q < SEL_FIRST; ++q) {
            const int j = lane + 32 * q;
            if (lists && j < S) {
                const uint2* list = p.cand + (static_cast<long long>(slot0 + j) * BM + r) * K_REG;
                const uint2 best = list[0], kth = list[K - 1];
                if (static_cast<int>(best.y) >= 0) first[q] = ordered_key(best.x);
                if (static_cast<int>(kth.y) >= 0) floor_key = max(floor_key, ordered_key(kth.x));
            }
        }
        for (int j = lane; j < S; j += 32) {
            const long long so = static_cast<long long>(slot0 + j) * BM + r;
            const float pm = p.part_m[so], ps = p.part_s[so];
            if (joint) {
                const uint2 bounds = p.bounds[so];
                floor_key = max(floor_key, bounds.x);
                least_key = min(least_key, bounds.y);
            } else if (!lists) {
                floor_key = max(floor_key, p.thr_share[so]);
            }
            if (pm > m) {
                sum *= exp2f((m - pm) * LOG2E);
                m = pm;
            }
            sum += ps * exp2f((pm - m) * LOG2E);
        }
        float mx = m;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        if (m > -INFINITY) sum *= exp2f((m - mx) * LOG2E);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
        floor_key = __reduce_max_sync(0xffffffffu, floor_key);
        if (joint) floor_key = max(floor_key, __reduce_min_sync(0xffffffffu, least_key));
        if (lists && S >= K) {
            uint32_t T = 0u;
#pragma unroll 1
            for (int bit = 31; bit >= 0; --bit) {
                const uint32_t c2 = T | (1u << bit);
                int c = 0;
#pragma unroll
                for (int q = 0; q < SEL_FIRST; ++q) c += first[q] >= c2 ? 1 : 0;
                if (static_cast<int>(__reduce_add_sync(0xffffffffu, c)) >= K) T = c2;
            }
            floor_key = max(floor_key, T);
        }
        const float lse_t = mx + logf(sum);
        if (tid == 0 && p.lse_t) p.lse_t[row] = lse_t;

        // this warp's share of the candidates: lanes of the row tile w, w + WARPS, ...
        unsigned long long* pool = sel_pools + warp * WIN;
        int n = 0;
        const uint32_t lt_mask = (1u << lane) - 1u;
        auto append = [&](const uint2 (&ce)[SEL_LOADS], const bool (&in)[SEL_LOADS]) {
#pragma unroll
            for (int q = 0; q < SEL_LOADS; ++q) {
                const uint32_t key = ordered_key(ce[q].x);
                const bool ok = in[q] && static_cast<int>(ce[q].y) >= 0 && key >= floor_key;
                const uint32_t bm = __ballot_sync(0xffffffffu, ok);
                if (ok) pool[n + __popc(bm & lt_mask)] = cand_rank(key, ce[q].y);
                n += __popc(bm);
            }
            __syncwarp();
            if (n + 32 * SEL_LOADS > WIN)        // n > K + 64 here
                floor_key = max(floor_key, static_cast<uint32_t>(cut_to_best<1>(pool, n, K, 64, lane, nullptr) >> 32));
        };
        if (lists) {
            for (int e0 = w * 32 * SEL_LOADS; e0 < S * K_REG; e0 += WARPS * 32 * SEL_LOADS) {
                uint2 ce[SEL_LOADS];
                bool in[SEL_LOADS];
#pragma unroll
                for (int q = 0; q < SEL_LOADS; ++q) {
                    const int e = e0 + q * 32 + lane;
                    in[q] = e < S * K_REG;
                    ce[q] = make_uint2(0u, 0u);
                    if (in[q]) ce[q] = p.cand[(static_cast<long long>(slot0 + e / K_REG) * BM + r) * K_REG + e % K_REG];
                }
                append(ce, in);
            }
        } else {
            for (int s0 = 0; s0 < S; s0 += 32 * WARPS) {
                const int mine = s0 + lane * WARPS + w;
                const int cn_mine = mine < S ? p.cand_n[static_cast<long long>(slot0 + mine) * BM + r] : 0;
                for (int j = 0; j < 32 && s0 + j * WARPS + w < S; ++j) {
                    const int cn = __shfl_sync(0xffffffffu, cn_mine, j);
                    const uint2* list = p.cand + (static_cast<long long>(slot0 + s0 + j * WARPS + w) * BM + r) * p.cap;
                    for (int e0 = 0; e0 < cn; e0 += 32 * SEL_LOADS) {
                        uint2 ce[SEL_LOADS];
                        bool in[SEL_LOADS];
#pragma unroll
                        for (int q = 0; q < SEL_LOADS; ++q) {
                            const int e = e0 + q * 32 + lane;
                            in[q] = e < cn;
                            ce[q] = make_uint2(0u, 0u);
                            if (in[q]) ce[q] = list[e];
                        }
                        append(ce, in);
                    }
                }
            }
        }
        // Rank what is left: every candidate counts those above it. Beyond 128 they are cut to about K first.
        int total = n;
        if (WARPS > 1) {
            if (lane == 0) pool_n[warp] = n;
            __syncthreads();
            total = __reduce_add_sync(0xffffffffu, lane < WARPS ? pool_n[lane] : 0);
        }
        if (total > K && total > 128) cut_to_best<WARPS>(pool, n, K, 16, lane, cut_words);
        if (WARPS > 1) __syncthreads();
        if (lane == 0) pool_n[warp] = n;
        for (int j = tid; j < K; j += WARPS * 32) {           // cannot stay for K <= V; keeps ids in range
            sel_tok[rib][j] = 0;
            sel_q[rib][j] = 0.f;
        }
        sync_row();
        for (int e = lane; e < n; e += 32) {
            const unsigned long long v = pool[e];
            int rank = 0;
            for (int w2 = 0; w2 < WARPS; ++w2) {
                const unsigned long long* other = sel_pools + (rib * WARPS + w2) * WIN;
                const int n2 = pool_n[rib * WARPS + w2];
                for (int i = 0; i < n2; ++i) rank += other[i] > v ? 1 : 0;
            }
            if (rank < K) {
                sel_tok[rib][rank] = static_cast<int>(~static_cast<uint32_t>(v));
                sel_q[rib][rank] = expf(__uint_as_float(key_bits(static_cast<uint32_t>(v >> 32))) - lse_t);
            }
        }
        sync_row();
        int n_sel = K;
        if (p.top_p > 0.f) {
            // Top-P: a token belongs to Omega_hat while the probability of those before it is <= P
            if (tid == 0) {
                int taken = 0;
                float cum = 0.f;
                for (int j = 0; j < K; ++j) {
                    if (cum > p.top_p) {
                        sel_tok[rib][j] = -1;
                        sel_q[rib][j] = 0.f;
                    } else {
                        ++taken;
                    }
                    cum += sel_q[rib][j];
                }
                if (!(cum > p.top_p)) taken = -taken;      // all K tokens taken and P still not exceeded: the cap cut the prefix
                n_sel = taken;
            }
            sync_row();
        }
        for (int j = tid; j < K; j += WARPS * 32) {
            p.idx_out[static_cast<long long>(row) * p.out_pitch + j] = sel_tok[rib][j];
            p.q_out[static_cast<long long>(row) * p.out_pitch + j] = sel_q[rib][j];
        }
        if (tid == 0 && p.n_out) p.n_out[row] = n_sel;
    } else {
        for (int j = tid; j < K; j += WARPS * 32) {
            sel_tok[rib][j] = p.idx_in[ro + j];
            sel_q[rib][j] = p.q_in[ro + j];
        }
        if (tid == 0 && p.n_out) p.n_out[row] = K;
        sync_row();
    }
    if (p.ref2 != nullptr && w == WARPS - 1) {
        const int tok = sel_tok[rib][0];
        const __nv_bfloat16* hrow = p.H_d + static_cast<long long>(row) * p.d;
        const __nv_bfloat16* wrow = p.W + static_cast<long long>(tok < 0 || tok >= p.V ? 0 : tok) * p.d;
        float acc = 0.f;
#pragma unroll 4
        for (int k0 = lane * 8; k0 < p.d; k0 += 256) {
            const uint4 hv = *reinterpret_cast<const uint4*>(hrow + k0);
            const uint4 wv = *reinterpret_cast<const uint4*>(wrow + k0);
            const __nv_bfloat162* hp = reinterpret_cast<const __nv_bfloat162*>(&hv);
            const __nv_bfloat162* wp = reinterpret_cast<const __nv_bfloat162*>(&wv);
#pragma unroll
            for (int t = 0; t < 4; ++t) {
                const float2 a2 = __bfloat1622float2(hp[t]);
                const float2 b2 = __bfloat1622float2(wp[t]);
                acc = fmaf(a2.x, b2.x, acc);
                acc = fmaf(a2.y, b2.y, acc);
            }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
        if (lane == 0) p.ref2[row] = fmaf(acc, LOG2E, 64.f);
    }
    if (p.sidx == nullptr) return;
    // the same set in increasing token id (entries cut by Top-P go to the end as INT_MAX / 0)
    for (int j = tid; j < K; j += WARPS * 32) {
        const int tj = sel_tok[rib][j] < 0 ? INT_MAX : sel_tok[rib][j];
        int rank = 0;
        for (int i = 0; i < K; ++i) {
            const int ti = sel_tok[rib][i] < 0 ? INT_MAX : sel_tok[rib][i];
            rank += (ti < tj || (ti == tj && i < j)) ? 1 : 0;
        }
        p.sidx[ro + rank] = tj;
        p.sq[ro + rank] = tj == INT_MAX ? 0.f : sel_q[rib][j];
    }
}

// ---------------------------------------------------------------------------------------------
// loss_patch_kernel: one warp per row, after the sweep of the draft rows of the fused call. Merges the draft's
// partial statistics into lse_d, evaluates Eq. 1 from the captured draft logits, writes the per-row scale of the
// spilled tiles, and puts the Omega_hat term of dz_d into the spill itself: with the spilled value
// P~(v) = e^(z_d(v) - m_spill), dz_d(v) = coef (P~(v) - [v in Omega_hat] q(v) / (S_q e^(m_spill - lse_d))),
// so the K entries of the row at its Omega_hat tokens are replaced by that difference and the second GEMM needs
// nothing but the row scale in its epilogue. The difference is formed in fp32 from the captured logit and rounded to
// bf16 once: taken off the spilled bf16 value, q would leave the rounding of p (2^-9 p), which is most of the
// difference where the draft is close to its target (p within 1 % of q: 8e-2 of the largest gradient entry).
struct LossPatchParams {
    Schedule sched;        // schedule of the draft sweep
    int K;
    int row_begin, rows;
    const float* part_m;
    const float* part_s;
    const int* sidx;       // [N, K]
    const float* sq;
    const float* cap_z;    // [N, K] z_d at sidx
    const float* grad_loss;
    float* loss;
    float* lse_d;
    float* coef_out;       // [N] g S_q e^(m_spill - lse_d)
    __nv_bfloat16* P;      // spill of the chunk [rows, p_pitch]
    long long p_pitch;
    const unsigned int* gate;
};

__global__ void __launch_bounds__(256) loss_patch_kernel(const __grid_constant__ LossPatchParams p) {
    wait_previous_kernel();
    if (p.gate != nullptr && *p.gate == 0u) return;
    const int lane = threadIdx.x & 31;
    const int local = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (local >= p.rows) return;
    const int row = p.row_begin + local;
    const int rt = local / BM, r = local % BM;
    const int K = p.K;
    int slot0, S;
    find_slots(p.sched, rt, slot0, S);
    const float lse_d = warp_lse(p.part_m, p.part_s, slot0, S, r, lane);
    const float m_spill = p.part_m[static_cast<long long>(slot0) * BM + r];
    const float g = p.grad_loss ? p.grad_loss[row] : 1.f;
    const long long ro = static_cast<long long>(row) * K;
    float S_q = 0.f, loss = 0.f;
    for (int j = lane; j < K; j += 32) {
        const float qv = p.sq[ro + j];
        if (p.sidx[ro + j] != INT_MAX && qv != 0.f) {      // (0 log p = 0, where z_d = -inf too)
            S_q += qv;
            loss += qv * (lse_d - p.cap_z[ro + j]);     // -q log p,  log p = z_d - lse_d
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        S_q += __shfl_xor_sync(0xffffffffu, S_q, o);
        loss += __shfl_xor_sync(0xffffffffu, loss, o);
    }
    const float scale = S_q * expf(m_spill - lse_d);     // coef / g
    if (lane == 0) {
        p.loss[row] = loss;
        p.lse_d[row] = lse_d;
        if (p.coef_out) p.coef_out[row] = g * scale;
    }
    if (p.P != nullptr && g != 0.f && scale > 0.f && scale < INFINITY) {      // P == nullptr: forward only, nothing to patch
        const float sum = expf(lse_d - m_spill);         // q / scale = q / S_q x sum: neither factor can overflow
        __nv_bfloat16* prow = p.P + static_cast<long long>(local) * p.p_pitch;
        for (int j = lane; j < K; j += 32) {
            const int tok = p.sidx[ro + j];
            const float qv = p.sq[ro + j];
            // (q = 0: the spilled value stays; a set filled up with token 0 may name it twice, and an entry has one writer)
            if (tok != INT_MAX && qv != 0.f) prow[tok] = __float2bfloat16_rn(expf(p.cap_z[ro + j] - m_spill) - qv / S_q * sum);
        }
    }
}

// ---------------------------------------------------------------------------------------------
// row_kernel: one block per row, after a MODE_LOGITS sweep that left the logits of few rows in fp32 (-inf beyond the
// vocabulary). Per row: lse of the target and of the draft, Omega_hat from the target's logits (or given), Eq. 1 from the
// draft's logits at Omega_hat, and (make_dz) the draft's row turned into
// dz_d(v) = g (S_q p(v) - q(v) [v in Omega_hat]) in bf16, in place: the bf16 row begins where the fp32 row did. Every step
// reads a piece twice as long as the one it writes, and a piece is written after all threads have read theirs.
// ROW_COMBINED: dz_d(v) = g ((1 + w S_q) p(v) - q(v) - w q(v) [v in Omega_hat]), and the cross-entropy
// sum_v q(v) (lse_d - z_d(v)); what bf16 leaves of the entries at Omega_hat that w q makes large goes, with their rows of W, to the epilogue of the
// second GEMM in fp32 (left_over; with the whole entry in bf16 dH_d of rows whose target and draft are peaked on different tokens was 1.7e-3 off
// fp64 in 2-norm at 100 x 4096 x 32000, logits of deviation 4, with a spill of either matrix 1.2e-3, now 1.06e-3; per call 64 x 256 x 1024
// 18 -> 19 us, 100 x 4096 x 32000, K = 100 117 -> 125, 300 x 4096 x 32000 269 -> 273). ROW_BIDIR: the draft's K most probable tokens join Omega_hat; the row becomes p(v) alone, and
// g S_q and the row sum_x g q(x) W[x, :] over Omega_hat are left in fp32 for the epilogue of the second GEMM.
//
// The K largest of a row: a thread's largest logit is at hand after the pass for lse, and the K-th largest of these
// maxima bounds the row's K-th largest from below. Little more than K logits reach it; warps read the shares of the threads that hold
// them again and put them into a pool in shared memory, where each counts those above it (more than it takes: collect_from_many).
// Bound by the latency of two passes over rows of 4 V bytes in L2: 1024 threads with ROW_LOADS 16-byte loads each in flight.
// It takes the rows that row_split_kernel does not (row_split in the host code): those of more than 8192 logits, when they are many.
// Where there are more rows than SMs two blocks of 512 threads share one, so that one row's barriers fall into the other's loads:
// combined calls of 2048 rows x 32000 260 -> 215 us, 640 x 8000 54 -> 35, 8000 x 3000, K = 128 620 -> 400; 1024 x 128256, where the rows come
// out of memory and go back (2.4 GB: two readings of both matrices and dz_d, 5.4 TB/s in 437 us, up to 480 under the power cap), 474 either way then. Four blocks of 256: 257, 33, 455.
constexpr int ROW_THREADS = 1024;
constexpr int ROW_LOADS = 4;
constexpr int ROW_POOL = 1024;
constexpr int ROW_SLACK = 32;      // maxima beyond K at which the search of the bound ends
static_assert(ROW_POOL >= K_CAP && ROW_THREADS / 2 >= K_CAP, "room for Omega_hat, a thread for each of its tokens");
enum { ROW_TOPK = 0, ROW_COMBINED = 1, ROW_BIDIR = 2 };

struct RowParams {
    int K, V;
    long long pitch;       // of z and zt, a multiple of 256
    float* z;              // [N, pitch] in: draft logits; out: bf16 [N, 2 pitch]. nullptr: selection only
    const float* zt;       // [N, pitch] target logits, or nullptr: Omega_hat is given
    int* idx;              // [N, idx_pitch] Omega_hat in descending q: out with zt, else in (entries < 0 carry q = 0)
    float* q;
    int idx_pitch;
    float top_p;           // > 0: Omega_hat is cut to the shortest sorted prefix with cumulative q > top_p
    int* n_out;            // [N] |Omega_hat|, negative where K tokens do not reach top_p (nullable)
    const float* grad_loss;
    float* lse_t;
    float* lse_d;
    float* loss;
    const float* lse_in;   // nullable: [N] lse_d, given (the separate backward: dz_d alone, neither loss nor lse_d is written)
    int make_dz;
    int release_late;      // as in GemmParams
    int split;             // row_split_kernel: blocks per row
    __nv_bfloat16* dz;     // row_split_kernel: [N, 2 pitch] dz_d; may be the target's logits, not the draft's
    float w;               // ROW_COMBINED
    float* loss_ce;
    const __nv_bfloat16* W;      // ROW_BIDIR, ROW_COMBINED: [V, d]
    int d;
    float* coef_out;       // [N] row scale of the second GEMM: g S_q, or 1
    float* sparse_out;     // [N, d] what its epilogue takes off
};

// The separate backward's set is the caller's and may name a token more than once: what its first entry takes off for all of them,
// and 0 for the others (n entries; q of entry j).
__device__ __forceinline__ float repeated_q(const int* tok, const float* q, int n, int j) {
    float sum = 0.f;
    for (int i = 0; i < n; ++i) {
        if (tok[i] != tok[j]) continue;
        if (i < j && q[i] != 0.f) return 0.f;
        sum += q[i];
    }
    return sum;
}

// Combined objective: what is to be added to an entry of dz_d at a token of Omega_hat, dense - target - w q, that was rounded to bf16 as `b`; 0 where
// the rounding is at most that of its dense and target terms by themselves, as they have it in a spill (w q(x) as a term of its own stays in fp32
// there). The row of W goes with it to the fp32 rows of the second GEMM's epilogue.
__device__ __forceinline__ float left_over(float o, __nv_bfloat16 b, float dense, float target) {
    return fabsf(o) > fabsf(dense) + fabsf(target) ? __bfloat162float(b) - o : 0.f;
}
// One warp: the entries whose weight is not zero go to the front, in their order; returns how many there are.
__device__ __forceinline__ int keep_weighted(int* tok, float* w, int n) {
    const int lane = threadIdx.x & 31;
    int kept = 0;
    for (int j0 = 0; j0 < n; j0 += 32) {
        const int j = j0 + lane, t = j < n ? tok[j] : 0;
        const float x = j < n ? w[j] : 0.f;
        const uint32_t bm = __ballot_sync(0xffffffffu, x != 0.f);
        const int at = kept + __popc(bm & ((1u << lane) - 1u));
        if (x != 0.f) {
            tok[at] = t;
            w[at] = x;
        }
        kept += __popc(bm);
        __syncwarp();
    }
    return kept;
}

struct RowPool {           // of a block that looks for the K largest logits of a row, or of its piece of one
    unsigned long long pool[ROW_POOL];
    float red[4][32];
    uint32_t key_min[32];
    int n, holders;
    int reach[3], equal[32];
};
struct RowShared : RowPool {
    unsigned short holder[ROW_THREADS];      // threads whose largest logit reaches the bound
    int tok[K_CAP];        // Omega_hat
    float q[K_CAP], z[K_CAP];
    int tok_d[K_CAP];      // the draft's own K largest (ROW_BIDIR)
    float z_d[K_CAP];
    float sum;
    int count;
};

// One logit as a number: larger = larger logit, lower token id first among equal ones (-0 and +0 are equal).
__device__ __forceinline__ unsigned long long logit_rank(float z, uint32_t id) {
    return cand_rank(ordered_key(__float_as_uint(z + 0.f)), id);
}

// Whether column `at` of a row, with logit z, is a token whose logit reaches the ordered key `bound` (> 0)
__device__ __forceinline__ bool reaches(float z, long long at, int V, uint32_t bound) {
    return z > -INFINITY && at < V && ordered_key(__float_as_uint(z + 0.f)) >= bound;
}

// f(first column, its four logits) for every piece of the row that this thread owns, ROW_LOADS at a time while go()
template <int THREADS, typename F, typename G>
__device__ __forceinline__ void for_own_logits_while(const float* row, long long pitch, F&& f, G&& go) {
    for (long long c0 = threadIdx.x * 4; c0 < pitch && go(); c0 += ROW_LOADS * THREADS * 4) {
        float4 v[ROW_LOADS];
#pragma unroll
        for (int u = 0; u < ROW_LOADS; ++u) {
            const long long at = c0 + u * (THREADS * 4);
            if (at < pitch) v[u] = *reinterpret_cast<const float4*>(row + at);
        }
#pragma unroll
        for (int u = 0; u < ROW_LOADS; ++u) {
            const long long at = c0 + u * (THREADS * 4);
            if (at < pitch) f(at, v[u]);
        }
    }
}
template <int THREADS, typename F>
__device__ __forceinline__ void for_own_logits(const float* row, long long pitch, F&& f) {
    for_own_logits_while<THREADS>(row, pitch, f, [] { return true; });
}

// This thread's largest logit m and sum of 2^((z - m) log2e)
template <int THREADS>
__device__ __forceinline__ void own_stats(const float* row, long long pitch, float& m, float& s) {
    m = -INFINITY;
    s = 0.f;
    for_own_logits<THREADS>(row, pitch, [&](long long, const float4& v) {
        const float cm = fmaxf(fmax3(v.x, v.y, v.z), v.w);
        if (cm > m) {
            s *= ex2((m - cm) * LOG2E);
            m = cm;
        }
        const float mneg = m == -INFINITY ? 0.f : -m * LOG2E;      // (nothing but -inf so far: each adds zero)
        s += ex2(fmaf(v.x, LOG2E, mneg)) + ex2(fmaf(v.y, LOG2E, mneg)) + ex2(fmaf(v.z, LOG2E, mneg)) + ex2(fmaf(v.w, LOG2E, mneg));
    });
}

// The block's log-sum-exp of the threads' (m, s); `red`: 2 x 32 floats, which
// the caller keeps until all have read them. One barrier.
template <int THREADS>
__device__ __forceinline__ float block_lse(float m, float s, float (*red)[32]) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    float mx = m;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    const float base = mx == -INFINITY ? 0.f : mx;
    s *= ex2((m - base) * LOG2E);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) {
        red[0][warp] = mx;
        red[1][warp] = s;
    }
    __syncthreads();
    m = lane < THREADS / 32 ? red[0][lane] : -INFINITY;
    s = lane < THREADS / 32 ? red[1][lane] : 0.f;
    mx = m;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    const float top = mx == -INFINITY ? 0.f : mx;
    s *= ex2(((m == -INFINITY ? top : m) - top) * LOG2E);      // (a warp without a logit: its sum is zero)
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    return top + logf(s);
}

// Logits that are ranked one against all others: those of K + ROW_SLACK pieces of four. (1024 equal ones of a row of zeros fit the
// pool; ranking them took 55 us.)
__device__ __forceinline__ int pool_room(int K) { return min(4 * (K + ROW_SLACK), ROW_POOL); }

// Block-collective: the logits that reach `bound` into the pool, by the threads whose maximum `key` does; given up when they are
// more than `room` (then sh.n > room). (row, pitch, V): a row, or the piece of it that begins with token `first`.
template <int THREADS>
__device__ __forceinline__ void collect(const float* row, long long pitch, int V, int first, uint32_t key, uint32_t bound, int room, RowPool& sh) {
    auto full = [&] { return *static_cast<volatile int*>(&sh.n) > room; };
    if (key >= bound)
        for_own_logits_while<THREADS>(row, pitch, [&](long long at, const float4& v) {
            const float z[4] = {v.x, v.y, v.z, v.w};
            if (!reaches(fmaxf(fmax3(z[0], z[1], z[2]), z[3]), at, V, bound)) return;
#pragma unroll
            for (int j = 0; j < 4; ++j)
                if (reaches(z[j], at + j, V, bound)) {
                    const int pos = atomicAdd(&sh.n, 1);
                    if (pos < room) sh.pool[pos] = logit_rank(z[j], static_cast<uint32_t>(first + at + j));
                }
        }, [&] { return !full(); });
    __syncthreads();
}

// The same, where few threads hold such logits as a rule: a warp reads the share of one of them at a time, a piece per lane. (Read by their own
// threads, hardly a warp was without one, and went over the row once more with a lane or two at work: the row kernel of 1024 x 128256, combined, 479 ->
// 437 us, 517 rows 246 -> 226, 100 x 128256, K = 20 51 -> 45.6, 61 x 32000 18.9 -> 18.2.)
template <int THREADS>
__device__ __forceinline__ void collect_from_holders(const float* row, long long pitch, int V, uint32_t key, uint32_t bound, int room, RowPool& sh,
                                                     unsigned short* holder) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (key >= bound) holder[atomicAdd(&sh.holders, 1)] = static_cast<unsigned short>(threadIdx.x);
    __syncthreads();
    const int n = sh.holders, pieces = static_cast<int>((pitch + THREADS * 4 - 1) / (THREADS * 4));
    for (int h = warp; h < n && *static_cast<volatile int*>(&sh.n) <= room; h += THREADS / 32) {
        const int own = holder[h] * 4;
        for (int u = lane; u < pieces; u += 32) {
            const long long at = static_cast<long long>(u) * (THREADS * 4) + own;
            if (at >= pitch) continue;
            const float4 v = *reinterpret_cast<const float4*>(row + at);
            const float z[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
            for (int j = 0; j < 4; ++j)
                if (reaches(z[j], at + j, V, bound)) {
                    const int pos = atomicAdd(&sh.n, 1);
                    if (pos < room) sh.pool[pos] = logit_rank(z[j], static_cast<uint32_t>(at + j));
                }
        }
    }
    __syncthreads();
}

// Block-collective: more logits reach T, a bound of the K-th largest, than the pool takes (hi: the largest). As a rule they are equal
// (a row of zeros has nothing else), and T is the K-th largest logit itself: known without a look where it is also the largest,
// else from one count. Otherwise its bits are searched two per pass over the row, until it is found or the pool holds what
// reaches it. Of logits equal to the K-th the first in token order are taken, and no more of the row is read than that takes.
// Half of 61 rows x 4096 x 32000 zeros: 346 -> 117 us per call, as without zeros (116), of 8 rows x 128256 1140 -> 370, of 64 rows x 256 x
// 1024 83 -> 30 (a search of token ids bit by bit, a pass over the row for each, and 1024 equal logits ranked).
// Returns the entries left in the pool. (A function of its own: in line it costs row_kernel registers that it does not have.)
template <int THREADS>
__device__ __noinline__ int collect_from_many(const float* row, long long pitch, int V, int first, int K, uint32_t key, uint32_t T, uint32_t hi, RowPool& sh) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    auto count = [&](uint32_t t1, uint32_t t2, uint32_t t3) {
        __syncthreads();
        if (tid < 3) sh.reach[tid] = 0;
        __syncthreads();
        int c1 = 0, c2 = 0, c3 = 0;
        for_own_logits<THREADS>(row, pitch, [&](long long at, const float4& v) {
            const float z[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                c1 += reaches(z[j], at + j, V, t1) ? 1 : 0;
                c2 += reaches(z[j], at + j, V, t2) ? 1 : 0;
                c3 += reaches(z[j], at + j, V, t3) ? 1 : 0;
            }
        });
        c1 = __reduce_add_sync(0xffffffffu, c1);
        c2 = __reduce_add_sync(0xffffffffu, c2);
        c3 = __reduce_add_sync(0xffffffffu, c3);
        if (lane == 0) {
            atomicAdd(&sh.reach[0], c1);
            atomicAdd(&sh.reach[1], c2);
            atomicAdd(&sh.reach[2], c3);
        }
        __syncthreads();
    };
    bool exact = T == hi;
    if (!exact) {
        count(T + 1u, T + 1u, T + 1u);
        exact = sh.reach[0] < K;
    }
    if (!exact) {
        int bit = 32 - __clz(hi ^ T);
        bit += bit & 1;
        T = bit < 32 ? hi >> bit << bit : 0u;
        exact = true;
        for (bit -= 2; bit >= 0; bit -= 2) {
            const uint32_t t1 = T | (1u << bit), t2 = T | (2u << bit), t3 = T | (3u << bit);
            count(t1, t2, t3);
            const int c1 = sh.reach[0], c2 = sh.reach[1], c3 = sh.reach[2];
            const int c = c3 >= K ? c3 : c2 >= K ? c2 : c1 >= K ? c1 : INT_MAX;
            T = c3 >= K ? t3 : c2 >= K ? t2 : c1 >= K ? t1 : T;
            if (c <= pool_room(K)) {
                exact = false;
                break;
            }
        }
    }
    __syncthreads();
    if (tid == 0) sh.n = 0;
    __syncthreads();
    collect<THREADS>(row, pitch, V, first, key, exact ? T + 1u : T, pool_room(K), sh);
    int n = sh.n;
    if (exact) {
        // fewer than K lie above it; of those equal to it the first in token order
        int taken = n;
        for (long long c0 = 0; c0 < pitch && taken < K; c0 += THREADS * 4) {
            const long long at = c0 + tid * 4;
            const float4 v = at < pitch ? *reinterpret_cast<const float4*>(row + at) : make_float4(-INFINITY, -INFINITY, -INFINITY, -INFINITY);
            const float z[4] = {v.x, v.y, v.z, v.w};
            bool in[4];
            int c = 0;
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                in[j] = reaches(z[j], at + j, V, T) && !reaches(z[j], at + j, V, T + 1u);
                c += in[j] ? 1 : 0;
            }
            int pos = c;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int before = __shfl_up_sync(0xffffffffu, pos, o);
                if (lane >= o) pos += before;
            }
            __syncthreads();
            if (lane == 31) sh.equal[warp] = pos;
            __syncthreads();
            const int of_warp = lane < THREADS / 32 ? sh.equal[lane] : 0;
            pos += taken - c + __reduce_add_sync(0xffffffffu, lane < warp ? of_warp : 0);
            taken += __reduce_add_sync(0xffffffffu, of_warp);
#pragma unroll
            for (int j = 0; j < 4; ++j)
                if (in[j]) {
                    if (pos < K) sh.pool[pos] = logit_rank(z[j], static_cast<uint32_t>(first + at + j));
                    ++pos;
                }
        }
        n = taken < K ? taken : K;
        __syncthreads();
    }
    return n;
}

// Block-collective: a bound that K of the threads' largest logits reach (m = this thread's), as an ordered key, or 1 where fewer
// threads have one above -inf; key = this thread's, hi = the largest. Leaves the pool empty.
template <int THREADS>
__device__ __forceinline__ uint32_t bound_from_maxima(int K, float m, RowPool& sh, uint32_t& key, uint32_t& hi) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    key = m > -INFINITY ? ordered_key(__float_as_uint(m + 0.f)) : 0u;
    const uint32_t key_hi = __reduce_max_sync(0xffffffffu, key), key_lo = __reduce_min_sync(0xffffffffu, key == 0u ? 0xffffffffu : key);
    if (lane == 0) {
        sh.red[0][warp] = __uint_as_float(key_hi);
        sh.key_min[warp] = key_lo;
    }
    if (threadIdx.x == 0) sh.n = sh.holders = 0;
    const int groups = __syncthreads_count(key != 0u);
    hi = __reduce_max_sync(0xffffffffu, lane < THREADS / 32 ? __float_as_uint(sh.red[0][lane]) : 0u);
    if (groups < K) return 1u;
    // the K-th largest maximum, or a value below it that at most K + ROW_SLACK maxima reach, from the highest bit in which
    // the maxima differ on
    const uint32_t lo = __reduce_min_sync(0xffffffffu, lane < THREADS / 32 ? sh.key_min[lane] : 0xffffffffu);
    int bit = 32 - __clz(hi ^ lo);
    uint32_t T = bit < 32 ? hi >> bit << bit : 0u;
    for (--bit; bit >= 0; --bit) {
        const uint32_t T1 = T | (1u << bit);
        const int c = __syncthreads_count(key >= T1);
        if (c >= K) {
            T = T1;
            if (c <= K + ROW_SLACK) break;
        }
    }
    return max(T, 1u);
}

// Block-collective: the K largest logits of the row, in descending order (lower token id first among equal ones), into
// tok / val; m = this thread's largest logit. Fewer than K logits above -inf: the rest is token 0 at -inf.
template <int THREADS>
__device__ __forceinline__ void select_largest(const float* row, long long pitch, int V, int K, float m, RowShared& sh, int* tok, float* val) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    uint32_t key, hi;
    const uint32_t T = bound_from_maxima<THREADS>(K, m, sh, key, hi);
    collect_from_holders<THREADS>(row, pitch, V, key, T, pool_room(K), sh, sh.holder);
    int n = sh.n;
    if (n > pool_room(K)) n = collect_from_many<THREADS>(row, pitch, V, 0, K, key, T, hi, sh);
    for (int j = n + tid; j < K; j += THREADS) {
        tok[j] = 0;
        val[j] = -INFINITY;
    }
    for (int e = warp; e < n; e += THREADS / 32) {
        const unsigned long long v = sh.pool[e];
        int rank = 0;
        for (int i = lane; i < n; i += 32) rank += sh.pool[i] > v ? 1 : 0;
        rank = __reduce_add_sync(0xffffffffu, rank);
        if (lane == 0 && rank < K) {
            tok[rank] = static_cast<int>(~static_cast<uint32_t>(v));
            val[rank] = __uint_as_float(key_bits(static_cast<uint32_t>(v >> 32)));
        }
    }
    __syncthreads();
}

template <int OBJ, int THREADS>      // THREADS: ROW_THREADS, or half of them
__global__ void __launch_bounds__(THREADS, ROW_THREADS / THREADS) row_kernel(const __grid_constant__ RowParams p) {
    __shared__ RowShared sh;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int row = blockIdx.x;
    const int K = p.K;
    wait_previous_kernel(!p.release_late);
    float* zrow = p.z != nullptr ? p.z + static_cast<long long>(row) * p.pitch : nullptr;
    const float* trow = p.zt != nullptr ? p.zt + static_cast<long long>(row) * p.pitch : nullptr;
    int* idx = p.idx + static_cast<long long>(row) * p.idx_pitch;
    float* q = p.q + static_cast<long long>(row) * p.idx_pitch;

    float m_t = -INFINITY, s_t = 0.f, m_d = -INFINITY, s_d = 0.f, lse_t = 0.f, lse_d = 0.f;
    if (trow) own_stats<THREADS>(trow, p.pitch, m_t, s_t);
    if (zrow && p.lse_in == nullptr) own_stats<THREADS>(zrow, p.pitch, m_d, s_d);
    if (trow) lse_t = block_lse<THREADS>(m_t, s_t, sh.red);
    if (zrow) lse_d = p.lse_in != nullptr ? p.lse_in[row] : block_lse<THREADS>(m_d, s_d, sh.red + 2);
    __syncthreads();

    int n_tok = K;                        // entries of Omega_hat's list (2K at most for the bi-directional set)
    if (trow) {
        select_largest<THREADS>(trow, p.pitch, p.V, K, m_t, sh, sh.tok, sh.q);
        if (tid < K) sh.q[tid] = sh.q[tid] > -INFINITY ? expf(sh.q[tid] - lse_t) : 0.f;      // (-inf: filled up)
        __syncthreads();
        int taken = K;
        if (p.top_p > 0.f) {
            // Top-P: a token belongs to Omega_hat while the probability of those before it is <= P
            if (tid == 0) {
                taken = 0;
                float cum = 0.f;
                for (int j = 0; j < K; ++j) {
                    if (cum > p.top_p) {
                        sh.tok[j] = -1;
                        sh.q[j] = 0.f;
                    } else {
                        ++taken;
                    }
                    cum += sh.q[j];
                }
                if (!(cum > p.top_p)) taken = -taken;      // all K tokens taken and P still not exceeded: the cap cut the prefix
            }
            __syncthreads();
        }
        if (OBJ == ROW_BIDIR) {
            // the draft's own K most probable tokens that are not in the target's set join Omega_hat, in their order
            select_largest<THREADS>(zrow, p.pitch, p.V, K, m_d, sh, sh.tok_d, sh.z_d);
            if (warp == 0) {
                int n = K;
                for (int j0 = 0; j0 < K; j0 += 32) {
                    const int j = j0 + lane;
                    const int t = j < K ? sh.tok_d[j] : -1;
                    bool joins = j < K;
                    for (int i = 0; i < K; ++i) joins = joins && sh.tok[i] != t;
                    const uint32_t bm = __ballot_sync(0xffffffffu, joins);
                    const int at = n + __popc(bm & ((1u << lane) - 1u));
                    if (joins) {
                        sh.tok[at] = t;
                        sh.q[at] = expf(trow[t] - lse_t);
                    }
                    n += __popc(bm);
                }
                for (int j = n + lane; j < 2 * K; j += 32) {
                    sh.tok[j] = -1;
                    sh.q[j] = 0.f;
                }
                if (lane == 0) sh.count = n;
            }
            __syncthreads();
            taken = sh.count;
            n_tok = 2 * K;
        }
        if (tid < n_tok) {
            idx[tid] = sh.tok[tid];
            q[tid] = sh.q[tid];
        }
        if (tid == 0) {
            p.lse_t[row] = lse_t;
            if (p.n_out) p.n_out[row] = taken;
        }
    } else {
        if (tid < K) {
            const int t = idx[tid];
            sh.tok[tid] = t < p.V ? t : -1;
            sh.q[tid] = q[tid];
        }
    }
    if (!zrow) return;
    if (tid < n_tok) sh.z[tid] = sh.tok[tid] >= 0 ? zrow[sh.tok[tid]] : 0.f;      // (each entry by the thread that wrote it, or behind a barrier)
    __syncthreads();
    if (warp == 0) {
        float S_q = 0.f, loss = 0.f;
        for (int j = lane; j < n_tok; j += 32) {
            if (sh.tok[j] < 0 || sh.q[j] == 0.f) continue;      // (0 log p = 0, where z_d = -inf too)
            S_q += sh.q[j];
            loss += sh.q[j] * (lse_d - sh.z[j]);      // -q log p,  log p = z_d - lse_d
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            S_q += __shfl_xor_sync(0xffffffffu, S_q, o);
            loss += __shfl_xor_sync(0xffffffffu, loss, o);
        }
        if (lane == 0) {
            sh.sum = S_q;
            if (p.lse_in == nullptr) {
                p.loss[row] = loss;
                p.lse_d[row] = lse_d;
            }
        }
    }
    __syncthreads();
    if (!p.make_dz) return;
    __nv_bfloat16* drow = reinterpret_cast<__nv_bfloat16*>(zrow);
    const float g = p.grad_loss ? p.grad_loss[row] : 1.f;
    const float S_q = sh.sum, c = OBJ == ROW_COMBINED ? g * (1.f + p.w * S_q) : OBJ == ROW_BIDIR ? 1.f : g * S_q, shift = -lse_d * LOG2E, shift_t = -lse_t * LOG2E;
    float ce = 0.f;
    for (long long c0 = 0; c0 < p.pitch; c0 += ROW_LOADS * THREADS * 4) {
        float4 v[ROW_LOADS];
#pragma unroll
        for (int u = 0; u < ROW_LOADS; ++u) {
            const long long at = c0 + (u * THREADS + tid) * 4;
            if (at < p.pitch) v[u] = *reinterpret_cast<const float4*>(zrow + at);
        }
        float4 t[OBJ == ROW_COMBINED ? ROW_LOADS : 1];
        if (OBJ == ROW_COMBINED) {
#pragma unroll
            for (int u = 0; u < ROW_LOADS; ++u) {
                const long long at = c0 + (u * THREADS + tid) * 4;
                if (at < p.pitch) t[OBJ == ROW_COMBINED ? u : 0] = *reinterpret_cast<const float4*>(trow + at);
            }
        }
        __syncthreads();
#pragma unroll
        for (int u = 0; u < ROW_LOADS; ++u) {
            const long long at = c0 + (u * THREADS + tid) * 4;
            if (at < p.pitch) {
                float z[4] = {v[u].x, v[u].y, v[u].z, v[u].w}, o[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) o[j] = c * ex2(fmaf(z[j], LOG2E, shift));
                if (OBJ == ROW_COMBINED) {
                    const float4& tu = t[OBJ == ROW_COMBINED ? u : 0];
                    const float zt[4] = {tu.x, tu.y, tu.z, tu.w};
                    const bool whole = at + 4 <= p.V;
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const float qv = ex2(fmaf(zt[j], LOG2E, shift_t));
                        o[j] = fmaf(-g, qv, o[j]);
                        if (whole || at + j < p.V) ce = fmaf(qv, lse_d - z[j], ce);      // (-inf beyond the vocabulary)
                    }
                }
                *reinterpret_cast<uint2*>(drow + at) = make_uint2(pack_bf16x2(o[0], o[1]), pack_bf16x2(o[2], o[3]));
            }
        }
    }
    if (OBJ == ROW_COMBINED) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) ce += __shfl_xor_sync(0xffffffffu, ce, o);
        if (lane == 0) sh.red[0][warp] = ce;
    }
    // sum_j sh.z[j] W[sh.tok[j], :], j < n, in fp32 for the second GEMM's epilogue
    auto sparse_row = [&](int n) {
        for (int k0 = tid * 8; k0 < p.d; k0 += THREADS * 8) {
            float a[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
#pragma unroll 4
            for (int j = 0; j < n; ++j) {
                const float c = sh.z[j];
                float wf[8];
                unpack8(*reinterpret_cast<const uint4*>(p.W + static_cast<long long>(sh.tok[j]) * p.d + k0), wf);
#pragma unroll
                for (int t = 0; t < 8; ++t) a[t] = fmaf(c, wf[t], a[t]);
            }
            float* so = p.sparse_out + static_cast<long long>(row) * p.d + k0;
            *reinterpret_cast<float4*>(so) = make_float4(a[0], a[1], a[2], a[3]);
            *reinterpret_cast<float4*>(so + 4) = make_float4(a[4], a[5], a[6], a[7]);
        }
    };
    if (OBJ == ROW_BIDIR) {
        if (tid == 0) p.coef_out[row] = g * S_q;
        if (tid < sh.count) sh.z[tid] = g * sh.q[tid];
        __syncthreads();
        sparse_row(sh.count);
        return;
    }
    __syncthreads();
    // Tokens of q = 0 keep the dense value: the one that fills up a set of fewer than K logits above -inf (token 0) may be in it
    // already, and an entry has one writer.
    const float q_own = tid < n_tok && sh.tok[tid] >= 0 ? (p.lse_in != nullptr ? repeated_q(sh.tok, sh.q, n_tok, tid) : sh.q[tid]) : 0.f;
    float left = 0.f;
    if (q_own != 0.f) {
        const float dense = c * ex2(fmaf(sh.z[tid], LOG2E, shift)), target = OBJ == ROW_COMBINED ? g * ex2(fmaf(trow[sh.tok[tid]], LOG2E, shift_t)) : 0.f;
        const float o = dense - (OBJ == ROW_COMBINED ? target + g * p.w * q_own : g * q_own);
        const __nv_bfloat16 b = __float2bfloat16_rn(o);
        drow[sh.tok[tid]] = b;
        if (OBJ == ROW_COMBINED) left = left_over(o, b, dense, target);
    }
    if (OBJ == ROW_COMBINED) {
        if (tid == 0) p.coef_out[row] = 1.f;
        if (tid < K) sh.z[tid] = left;
        if (K > 32) __syncthreads();      // (up to 32 tokens are the first warp's own)
        __syncwarp();
        if (warp == 0) {
            const int n = keep_weighted(sh.tok, sh.z, K);
            if (lane == 0) sh.count = n;
        }
        __syncthreads();
        sparse_row(sh.count);
    }
    if (OBJ == ROW_COMBINED && warp == 0) {
        float v = lane < THREADS / 32 ? sh.red[0][lane] : 0.f;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if (lane == 0) p.loss_ce[row] = v;
    }
}

// ---------------------------------------------------------------------------------------------
// ce_kernel (combined objective): one warp per row of a chunk. T[local, :] = q W of the row (from the second
// GEMM over the target spill). Full-vocabulary cross-entropy -sum_v q log p = lse_d - <H_d[row], q W>, and the
// (with the fp32 correction of the Omega_hat terms from finalize) the q W row joins the row's Omega_hat term so that dH_d = coef (draft spill x W) - sparse.
__global__ void __launch_bounds__(256) ce_kernel(int rows, int row_begin, int d, const __nv_bfloat16* H_d,
                                                 const float* T, const float* lse_d,
                                                 const float* grad_loss, const float* ce_corr,
                                                 float* loss_ce, float* sparse,
                                                 const unsigned int* gate) {
    wait_previous_kernel();
    if (gate != nullptr && *gate == 0u) return;
    const int lane = threadIdx.x & 31;
    const int local = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (local >= rows) return;
    const int row = row_begin + local;
    const float g = grad_loss ? grad_loss[row] : 1.f;
    const __nv_bfloat16* hrow = H_d + static_cast<long long>(row) * d;
    const float* trow = T + static_cast<long long>(local) * d;
    float* srow = sparse + static_cast<long long>(local) * d;
    float dot = 0.f;
    for (int k0 = lane * 8; k0 < d; k0 += 256) {
        const uint4 hv = *reinterpret_cast<const uint4*>(hrow + k0);
        const __nv_bfloat162* hp = reinterpret_cast<const __nv_bfloat162*>(&hv);
        const float4 t0 = *reinterpret_cast<const float4*>(trow + k0);
        const float4 t1 = *reinterpret_cast<const float4*>(trow + k0 + 4);
        float4 s0 = *reinterpret_cast<const float4*>(srow + k0);
        float4 s1 = *reinterpret_cast<const float4*>(srow + k0 + 4);
        const float2 h0 = __bfloat1622float2(hp[0]), h1 = __bfloat1622float2(hp[1]);
        const float2 h2 = __bfloat1622float2(hp[2]), h3 = __bfloat1622float2(hp[3]);
        dot += h0.x * t0.x + h0.y * t0.y + h1.x * t0.z + h1.y * t0.w + h2.x * t1.x + h2.y * t1.y + h3.x * t1.z + h3.y * t1.w;
        s0.x = fmaf(g, t0.x, s0.x); s0.y = fmaf(g, t0.y, s0.y); s0.z = fmaf(g, t0.z, s0.z); s0.w = fmaf(g, t0.w, s0.w);
        s1.x = fmaf(g, t1.x, s1.x); s1.y = fmaf(g, t1.y, s1.y); s1.z = fmaf(g, t1.z, s1.z); s1.w = fmaf(g, t1.w, s1.w);
        *reinterpret_cast<float4*>(srow + k0) = s0;
        *reinterpret_cast<float4*>(srow + k0 + 4) = s1;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) dot += __shfl_xor_sync(0xffffffffu, dot, o);
    if (lane == 0) loss_ce[row] = lse_d[row] - dot - ce_corr[row];
}

// Clears n 16-byte words: the status block and what lies behind it. (A memset node would stand between two dependent
// launches and make both wait: 5 us per call.)
__global__ void __launch_bounds__(256) clear_kernel(uint4* at, int n, uint4* at2, int n2) {
    wait_previous_kernel();
    for (int i = blockIdx.x * 256 + threadIdx.x; i < n + n2; i += gridDim.x * 256) *(i < n ? at + i : at2 + (i - n)) = make_uint4(0u, 0u, 0u, 0u);
}

// Self-test of the bounded waits (hass_selftest_wait_expiry): one CTA, no TMA, no tensor memory. Every thread
// waits for a phase of an mbarrier that nothing ever completes; thread 0 with the caller's short limit, the
// others with the library's normal limit. Thread 0 runs out of time, records its code in the status word and
// raises the CTA's abort flag, which ends the other threads' waits; the kernel then returns by itself.
// report[0] = threads whose wait gave up, report[1] = nanoseconds the CTA spent waiting.
__global__ void wait_expiry_selftest_kernel(unsigned int* status, unsigned long long limit_ns, unsigned int* report) {
    __shared__ unsigned long long bar;
    __shared__ int abort_flag;
    __shared__ int gave_up;
    if (threadIdx.x == 0) {
        mbar_init(smem_u32(&bar), 1);
        abort_flag = 0;
        gave_up = 0;
        fence_barrier_init();
    }
    __syncthreads();
    const unsigned long long t0 = globaltimer_ns();
    const bool done = wait_barrier(smem_u32(&bar), 0u, &abort_flag, status, 15u, threadIdx.x == 0 ? limit_ns : kWaitLimitNs);
    if (!done) atomicAdd(&gave_up, 1);
    __syncthreads();
    if (threadIdx.x == 0) {
        report[0] = static_cast<unsigned int>(gave_up);
        report[1] = static_cast<unsigned int>(globaltimer_ns() - t0);
    }
}

// ---------------------------------------------------------------------------------------------
// bwd_prep: one warp per row. Sorts Omega_hat by token id (the MODE_PROBS epilogue walks the vocabulary in
// increasing order; entries cut by Top-P carry id -1 and come first) by ranking every entry against the
// others, and precomputes g * q, g * S_q and lse_d * log2(e).
constexpr int PREP_WARPS = 4;
__global__ void __launch_bounds__(PREP_WARPS * 32) bwd_prep_kernel(int N, int K, const int* idx,
                                                                    const float* q,
                                                                    const float* lse_d,
                                                                    const float* grad_loss,
                                                                    int* sidx, float* sgq,
                                                                    float* coef, float* lse2) {
    wait_previous_kernel();
    __shared__ int s_tok[PREP_WARPS][K_CAP];
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    const int row = blockIdx.x * PREP_WARPS + wib;
    if (row >= N) return;
    const long long ro = static_cast<long long>(row) * K;
    const float g = grad_loss ? grad_loss[row] : 1.f;
    float S_q = 0.f;
    for (int j = lane; j < K; j += 32) {
        s_tok[wib][j] = idx[ro + j];
        S_q += q[ro + j];
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) S_q += __shfl_xor_sync(0xffffffffu, S_q, o);
    __syncwarp();
    for (int j = lane; j < K; j += 32) {
        const int tj = s_tok[wib][j];
        int rank = 0;
        for (int i = 0; i < K; ++i) {
            const int ti = s_tok[wib][i];
            rank += (ti < tj || (ti == tj && i < j)) ? 1 : 0;
        }
        sidx[ro + rank] = tj;
        sgq[ro + rank] = g * q[ro + j];
    }
    if (lane == 0) {
        coef[row] = g * S_q;
        lse2[row] = lse_d[row] * LOG2E;
    }
}

}  // namespace hass

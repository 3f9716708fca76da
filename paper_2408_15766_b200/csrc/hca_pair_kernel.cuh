// HCA attention of the draft layer (Section 3.2; the appendix's attention listing), forward, for sm_100a.
//
// One persistent, warp-specialised kernel, one CTA per SM. A CTA works on a PAIR of items at a time, an item
// being one (sequence, query head, tile of 128 query positions); the two items of a pair read the same
// key/value head, so every 128-key tile is fetched once and used by both:
//   - grouped heads with an even group size: two query heads of one group, same query tile;
//   - otherwise: two consecutive query tiles of one head (the lower one stops one key tile earlier).
// Where every item can have a CTA of its own, one slot of a CTA stays empty: the items of a pair wait for one another's turns.
// Each item owns a "slot": its Q tile in shared memory, a 128-column score buffer and a 128-column output
// accumulator in tensor memory, and four softmax warps. Per key tile and slot:
//   S = Q K_t^T            tcgen05.mma, 128 x 128 x 128, fp32 in TMEM
//   softmax warps          one query row per thread, its 128 scores in registers: hide the columns past t - m (the
//                          causal part and the m substituted entries), update the row's running reference and
//                          sum, write P = 2^(x - ref) as bf16 pairs back into tensor memory over the scores
//   O += P V_t             tcgen05.mma with P read from tensor memory, V_t an MN-major operand from shared memory
// The tensor core alternates between the slots, so one slot's products run while the other slot's rows are in
// their softmax. The products of a slot are issued in the order S(j), PV(j), S(j+1); the tensor core
// completes them in that order, so a finished S(j+1) means PV(j) has finished too and the softmax warps may
// touch the accumulator (rare rescale) without another barrier.
// The substituted entries (t, t - i), i < m, ride the same pipeline as extra products: before the key tiles
// S = Q K_d[i]^T with the K_d[i] tile fetched i rows early, so that the wanted scores sit on the diagonal and
// each row's thread keeps its own; the m scores join the row's maximum and sum at the last key tile; after
// the key tiles O += diag(p_i) V_d[i] with V_d[i] fetched i rows early. The weights of a pass take 8 columns beside the
// last tile's P: a step over 16 keys writes only the 16 lanes whose weights those keys belong to (the instruction's
// lane mask), so that all steps can share the columns, and the threads hand them over together with the last P instead of
// in rounds of two passes after it (m = 2 .. 5: one to three round trips of about 1.3 k cycles per item).
// No thread reads global memory.
// The running reference moves only when a tile's maximum exceeds it by more than 2^8 (the accumulator is then
// rescaled in place by the row's thread), so P stays within bf16 range and almost every tile skips the rescale.
// CLUSTER: a cluster of p.cluster CTAs per item, each with a part of its key tiles (the last one, which ends with the diagonal's, has the draft
// passes as well), where items are so few that all clusters are resident at once. In the end the CTAs hand one another their accumulators,
// references and sums by rows through distributed shared memory, and each finishes 128 / p.cluster rows (hca_fwd_cluster has the line).
// Warps: 0 = TMA producer, 1 = MMA issuer and TMEM owner (2, 3 idle), 4-7 = softmax + epilogue of slot 0,
// 8-11 = of slot 1 (TMEM lane quadrant = warp % 4). The first warpgroup gives registers up (setmaxnreg) and the
// two softmax warpgroups take them: a row's 128 scores stay in registers. Every wait is bounded (wait_barrier); a wait that gives up sets the status
// word and all roles leave.
#pragma once
#include <cuda_bf16.h>

#include "hca_kernels.cuh"
#include "ptx.cuh"

namespace hass {
namespace hca2 {

using hca::ex2;
using hca::pack_bf16;
using hca::tma_load_3d;
using hca::tmem_st32;
using hca::tmem_st_wait;
static_assert(64 + 8 * hca::MAX_DRAFTS <= 128, "the weights of all passes fit the score buffer");

constexpr int QT = 128;            // query rows per item
constexpr int KT = 128;            // keys per tile
constexpr int HD = 128;            // head dimension
constexpr int MAX_DRAFTS = 8;
constexpr int NUM_THREADS = 384;   // three warpgroups: {TMA, MMA, 2 idle warps}, softmax of slot 0, softmax of slot 1
constexpr int REGS_CONTROL = 56;   // registers per thread after the split (launch: 168 each; 56 + 2 * 224 = 3 * 168)
constexpr int REGS_SOFTMAX = 224;
constexpr int Q_BYTES = QT * HD * 2;                 // two halves (64 columns of the head dimension) of 128 rows x 128 B
constexpr int Q_HALF = Q_BYTES / 2;
constexpr int KV_BYTES = KT * HD * 2;
constexpr int KV_HALF = KV_BYTES / 2;
constexpr int KV_STAGES = 2;          // value tiles in flight
constexpr int K_STAGES = 3;           // key tiles in flight: one more, the draft passes' key tiles occupy the ring at an item's start
constexpr int SMEM_Q = 0;                            // 2 slots
constexpr int SMEM_K = SMEM_Q + 2 * Q_BYTES;
constexpr int SMEM_V = SMEM_K + K_STAGES * KV_BYTES;
constexpr int SMEM_BAR = SMEM_V + KV_STAGES * KV_BYTES;
constexpr int SCHED_DEPTH = 4;       // pair indices published ahead by the producer
constexpr int NUM_BARS = 4 + 2 * K_STAGES + 2 * KV_STAGES + 6 + 2 * SCHED_DEPTH;
constexpr int SMEM_BYTES = SMEM_BAR + 256;           // 229632
static_assert(8 * NUM_BARS + 4 * (2 + SCHED_DEPTH) <= 256 && SMEM_BYTES <= 232448, "shared-memory window");
constexpr int TMEM_COLS = 512;     // S of slot s at 128 s (P overwrites its first 64 columns), O of slot s at 256 + 128 s
constexpr int DRAFT_P = 64;        // the draft passes' weights: 8 columns each behind P in the score buffer
constexpr float RESCALE_LOG2 = 8.f;

struct Params {
    CUtensorMap tmQ;               // [B, T, H * 128], box {64, 128, 1}, 128-byte swizzle
    CUtensorMap tmK, tmV;          // [B, T, Hkv * 128], box {64, 128, 1}
    CUtensorMap tmKd[MAX_DRAFTS];  // the draft passes' keys and values, same geometry; index = sub-diagonal
    CUtensorMap tmVd[MAX_DRAFTS];
    __nv_bfloat16* O;              // [B, T, H, 128]
    float* lse;                    // [B, H, T] or null
    int B, T, H, Hkv, m;
    int q_tiles;                   // ceil(T / 128)
    int pairs;                     // work units
    int head_pairing;              // 1: a pair = heads 2u, 2u + 1 at one query tile; 0: one head, query tiles qt - 1, qt
    int single;                    // 1 (head_pairing = 0): a "pair" is one item, in slot 1
    float c2;                      // scale * log2(e)
    int cluster;                   // CLUSTER: CTAs per item: 2, 4 or 8 (single = 1, one_round = 1)
    int one_round;                 // every CTA takes one pair: no counter, and the status block is cleared here
    unsigned int* status;
};

struct Pair {
    int b, kv_col;                 // sequence; first column of the key/value head in [B, T, Hkv * 128]
    int h[2], qt[2];               // slot 0 / slot 1: query head and query tile
    bool act0;                     // slot 0 has an item (slot 1 always has one, and never the shorter one)
};

__device__ __forceinline__ Pair decode_pair(const Params& p, int idx) {
    Pair r;
    const int rep = p.H / p.Hkv;
    if (p.head_pairing) {
        const int per = p.B * (p.H >> 1);
        const int u = idx / per, rem = idx - u * per;
        r.b = rem / (p.H >> 1);
        const int hp = rem - r.b * (p.H >> 1);
        r.h[0] = 2 * hp;
        r.h[1] = 2 * hp + 1;
        r.qt[0] = r.qt[1] = p.q_tiles - 1 - u;          // longest first
        r.act0 = true;
    } else {
        const int per = p.B * p.H;
        const int u = idx / per, rem = idx - u * per;
        r.b = rem / p.H;
        r.h[0] = r.h[1] = rem - r.b * p.H;
        r.qt[1] = p.q_tiles - 1 - (p.single ? u : 2 * u);
        r.qt[0] = r.qt[1] - 1;
        r.act0 = !p.single && r.qt[0] >= 0;
    }
    r.kv_col = (r.h[1] / rep) * HD;
    return r;
}

constexpr int ROW_PITCH = HD + 4;  // floats of a handed-over row (the accumulator, its reference, its sum): rows 4 banks apart
static_assert(QT * ROW_PITCH * 4 <= SMEM_V, "the parts of a CTA's rows fit the room of queries and keys");

// The part [j0, j1) of n key tiles that is CTA z's of C: even shares, a draft pass counting as half a tile of the last CTA's, which has one tile at least
__host__ __device__ __forceinline__ void tile_share(int n, int m, int z, int C, int& j0, int& j1) {
    const int total = 2 * n + m;
    const int from = total * z / (2 * C), to = total * (z + 1) / (2 * C);
    j0 = from < n - 1 ? from : n - 1;
    j1 = z + 1 == C ? n : to < n - 1 ? to : n - 1;
}

template <bool CLUSTER>
__global__ void __launch_bounds__(NUM_THREADS, 1) hca_attention_pair_kernel(const __grid_constant__ Params p) {
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    const uint32_t base = smem_u32(smem_raw);
    if ((base & 1023u) != 0u) {
        // the swizzled tiles need a 1024-byte aligned window; report instead of computing garbage
        if (threadIdx.x == 0) atomicCAS(p.status, 0u, (20u << 8) | 1u);
        return;
    }
    const uint32_t bar0 = base + SMEM_BAR;
    auto q_full = [&](int s) { return bar0 + 8u * s; };
    auto q_empty = [&](int s) { return bar0 + 8u * (2 + s); };
    auto k_full = [&](int st) { return bar0 + 8u * (4 + st); };
    constexpr int KVB = 2 * K_STAGES + 2 * KV_STAGES;      // barriers of the two rings
    auto k_empty = [&](int st) { return bar0 + 8u * (4 + K_STAGES + st); };
    auto v_full = [&](int st) { return bar0 + 8u * (4 + 2 * K_STAGES + st); };
    auto v_empty = [&](int st) { return bar0 + 8u * (4 + 2 * K_STAGES + KV_STAGES + st); };
    auto s_full = [&](int s) { return bar0 + 8u * (4 + KVB + s); };
    auto p_full = [&](int s) { return bar0 + 8u * (6 + KVB + s); };
    auto pv_done = [&](int s) { return bar0 + 8u * (8 + KVB + s); };
    auto sched_full = [&](int e) { return bar0 + 8u * (10 + KVB + e); };
    auto sched_empty = [&](int e) { return bar0 + 8u * (10 + KVB + SCHED_DEPTH + e); };
    uint32_t* tmem_ptr_smem = reinterpret_cast<uint32_t*>(smem_raw + SMEM_BAR + 8 * NUM_BARS);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_ptr_smem + 1);
    volatile int* sched_idx = reinterpret_cast<volatile int*>(tmem_ptr_smem + 2);      // [SCHED_DEPTH]

    const int warp = threadIdx.x >> 5;
    const int lane = threadIdx.x & 31;
    // this CTA's index among its cluster's, and the key tiles and draft passes it takes of slot 1's item
    const int z = CLUSTER ? static_cast<int>(blockIdx.x) % p.cluster : 0;
    auto own_share = [&](const Pair& pr, int& j0, int& j1) {
        j0 = 0;
        j1 = pr.qt[1] + 1;
        if (CLUSTER) tile_share(j1, p.m, z, p.cluster, j0, j1);
    };
    const int md = CLUSTER && z + 1 < p.cluster ? 0 : p.m;

    if (threadIdx.x == 0) {
        for (int s = 0; s < 2; ++s) {
            mbar_init(q_full(s), 1);
            mbar_init(q_empty(s), 1);
            mbar_init(s_full(s), 1);
            mbar_init(p_full(s), 4);
            mbar_init(pv_done(s), 1);
        }
        for (int st = 0; st < K_STAGES; ++st) {
            mbar_init(k_full(st), 1);
            mbar_init(k_empty(st), 1);
        }
        for (int st = 0; st < KV_STAGES; ++st) {
            mbar_init(v_full(st), 1);
            mbar_init(v_empty(st), 1);
        }
        for (int e = 0; e < SCHED_DEPTH; ++e) {
            mbar_init(sched_full(e), 1);
            mbar_init(sched_empty(e), 9);      // the MMA warp and the eight softmax warps
        }
        *abort_flag = 0;
        fence_barrier_init();
        fence_proxy_async_smem();
        prefetch_tensormap(&p.tmQ);
        prefetch_tensormap(&p.tmK);
        prefetch_tensormap(&p.tmV);
    }
    if (warp == 1) {
        tmem_alloc(smem_u32(tmem_ptr_smem), TMEM_COLS);
        tmem_relinquish();
    }
    wait_previous_kernel(false);
    if (p.one_round && blockIdx.x == 0 && threadIdx.x < 64) p.status[threadIdx.x] = 0u;
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    const uint32_t tmem_base = *tmem_ptr_smem;

    // With no more pairs than CTAs each takes its own (one launch instead of two: 22 us forward calls are bound by the host).
    // Otherwise pairs are sorted longest first and handed out dynamically: the producer takes the next index from a counter in
    // the workspace (word 1, zeroed by the host before the launch) and publishes it to the other roles through a
    // small queue in shared memory, so a CTA that falls behind simply takes fewer pairs. An index >= pairs ends a role.
    // next_pair(k): the k-th index this CTA works on (every consumer warp calls it once per k).
    auto next_pair = [&](uint32_t k, unsigned code) -> int {
        const int e = k % SCHED_DEPTH;
        if (!wait_barrier(sched_full(e), (k / SCHED_DEPTH) & 1u, abort_flag, p.status, code)) return INT_MAX;
        const int idx = sched_idx[e];
        __syncwarp();
        if (lane == 0) mbar_arrive(sched_empty(e));
        return idx;
    };

    // Per item and slot the tensor core runs, in this order:
    //   m draft score products   S = Q K_d[i]^T with the K_d[i] tile fetched i rows early, so that the wanted
    //                            scores <Q[t], K_d[i][t - i]> sit on the tile's diagonal; the row's thread keeps its own
    //   n key tiles              S = Q K_t^T -> softmax -> O += P V_t
    //   m draft value products   O += diag(p_i) V_d[i] (V_d[i] fetched i rows early; the weights came with the last P)
    // Every product of a slot but the first S and the draft value products follows an arrival of the slot's softmax warps
    // on p_full.
    // The K ring carries the draft key tiles, then the key tiles; the V ring the value tiles, then the draft
    // value tiles. A tile both slots use (always, when the pair is two heads of one group; the key/value
    // tiles otherwise) is one ring entry, released after the second slot's product.
    if (warp < 4) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(REGS_CONTROL));
    if (warp == 0) {
        // ===================== TMA producer =====================
        if (lane == 0) {
            uint32_t gq[2] = {0u, 0u}, gk = 0, gv = 0, it = 0;
            bool ok = true;
            auto load_k = [&](const CUtensorMap* tm, int col, int row, int b) -> bool {
                const int st = gk % K_STAGES;
                if (!wait_barrier(k_empty(st), ((gk / K_STAGES) & 1u) ^ 1u, abort_flag, p.status, 2)) return false;
                mbar_arrive_expect_tx(k_full(st), KV_BYTES);
                tma_load_3d(base + SMEM_K + st * KV_BYTES, tm, k_full(st), col, row, b);
                tma_load_3d(base + SMEM_K + st * KV_BYTES + KV_HALF, tm, k_full(st), col + 64, row, b);
                ++gk;
                return true;
            };
            auto load_v = [&](const CUtensorMap* tm, int col, int row, int b) -> bool {
                const int st = gv % KV_STAGES;
                if (!wait_barrier(v_empty(st), ((gv / KV_STAGES) & 1u) ^ 1u, abort_flag, p.status, 3)) return false;
                mbar_arrive_expect_tx(v_full(st), KV_BYTES);
                tma_load_3d(base + SMEM_V + st * KV_BYTES, tm, v_full(st), col, row, b);
                tma_load_3d(base + SMEM_V + st * KV_BYTES + KV_HALF, tm, v_full(st), col + 64, row, b);
                ++gv;
                return true;
            };
            for (;; ++it) {
                const int idx = !p.one_round ? static_cast<int>(atomicAdd(p.status + 1, 1u)) : it == 0 ? static_cast<int>(blockIdx.x) / (CLUSTER ? p.cluster : 1) : INT_MAX;
                {
                    const int e = it % SCHED_DEPTH;
                    if (!wait_barrier(sched_empty(e), ((it / SCHED_DEPTH) & 1u) ^ 1u, abort_flag, p.status, 15)) break;
                    sched_idx[e] = idx;
                    mbar_arrive(sched_full(e));
                }
                if (idx >= p.pairs || !ok) break;
                const Pair pr = decode_pair(p, idx);
                int j0, n;
                own_share(pr, j0, n);
                if (CLUSTER && j0 == n) continue;
#pragma unroll
                for (int s = 0; s < 2; ++s) {
                    if (s == 0 && !pr.act0) continue;
                    if (!wait_barrier(q_empty(s), (gq[s] & 1u) ^ 1u, abort_flag, p.status, 1)) { ok = false; break; }
                    mbar_arrive_expect_tx(q_full(s), Q_BYTES);
                    tma_load_3d(base + SMEM_Q + s * Q_BYTES, &p.tmQ, q_full(s), pr.h[s] * HD, pr.qt[s] * QT, pr.b);
                    tma_load_3d(base + SMEM_Q + s * Q_BYTES + Q_HALF, &p.tmQ, q_full(s), pr.h[s] * HD + 64, pr.qt[s] * QT, pr.b);
                    ++gq[s];
                }
                // draft keys start i rows early: row c of the tile is position qt * 128 + c - i (zeros before the sequence)
                for (int i = 0; i < md && ok; ++i) {
                    if (!p.head_pairing && pr.act0) ok = load_k(&p.tmKd[i], pr.kv_col, pr.qt[0] * QT - i, pr.b);
                    if (ok) ok = load_k(&p.tmKd[i], pr.kv_col, pr.qt[1] * QT - i, pr.b);
                }
                for (int j = j0; j < n && ok; ++j) {
                    ok = load_k(&p.tmK, pr.kv_col, j * KT, pr.b);
                    if (ok) ok = load_v(&p.tmV, pr.kv_col, j * KT, pr.b);
                }
                for (int i = 0; i < md && ok; ++i) {
                    if (!p.head_pairing && pr.act0) ok = load_v(&p.tmVd[i], pr.kv_col, pr.qt[0] * QT - i, pr.b);
                    if (ok) ok = load_v(&p.tmVd[i], pr.kv_col, pr.qt[1] * QT - i, pr.b);
                }
            }
        }
    } else if (warp == 1) {
        // ===================== MMA issuer =====================
        // The whole warp runs this loop so that addresses and descriptors stay warp-uniform; one elected lane
        // issues the tensor-core instructions.
        constexpr uint32_t idesc_s = make_idesc_bf16(QT, KT, 0, 0);
        constexpr uint32_t idesc_o = make_idesc_bf16(QT, HD, 0, 1);
        uint32_t gq[2] = {0u, 0u}, gp[2] = {0u, 0u}, gk = 0, gv = 0, it = 0;
        bool ok = true;
        // tcgen05.commit follows the products of the thread that issued them: one lane, elected once, issues all
        const bool leader = elect_one();
        auto wait_all = [&](uint32_t bar, uint32_t parity, unsigned code) {
            return __all_sync(0xffffffffu, wait_barrier(bar, parity, abort_flag, p.status, code)) != 0;
        };
        // S of slot s from K stage st; last: the item's last score product (its Q tile is free afterwards)
        auto issue_s = [&](int s, int st, bool last) {
            tc_fence_after_sync();
#pragma unroll
            for (int k = 0; k < HD / 16; ++k) {
                const uint64_t a_desc = make_smem_desc_sw128(base + SMEM_Q + s * Q_BYTES + (k >> 2) * Q_HALF + (k & 3) * 32, 0, 1024);
                const uint64_t b_desc = make_smem_desc_sw128(base + SMEM_K + st * KV_BYTES + (k >> 2) * KV_HALF + (k & 3) * 32, 0, 1024);
                if (leader) umma_bf16(tmem_base + s * KT, a_desc, b_desc, idesc_s, k != 0 ? 1u : 0u);
            }
            if (leader) {
                umma_commit(s_full(s));
                if (last) umma_commit(q_empty(s));
            }
            __syncwarp();
        };
        // O of slot s (+)= P V: keys [16 k0, 16 k1) of V stage st, P read from the slot's S buffer starting at column
        // a_col (8 columns of bf16 pairs per 16 keys). B = V: 64-column groups KV_HALF apart, 16 keys further = 16
        // rows of 128 bytes. first: the item's first product into O; commit: signal pv_done afterwards.
        auto issue_pv = [&](int s, int st, int a_col, int k0, int k1, bool first, bool commit) {
            tc_fence_after_sync();
#pragma unroll
            for (int k = k0; k < k1; ++k) {
                const uint64_t b_desc = make_smem_desc_sw128(base + SMEM_V + st * KV_BYTES + k * 16 * 128, KV_HALF, 1024);
                if (leader) umma_bf16_ta(tmem_base + 256 + s * HD, tmem_base + s * KT + a_col + 8 * (k - k0), b_desc, idesc_o, (!first || k != k0) ? 1u : 0u);
            }
            if (leader && commit) umma_commit(pv_done(s));
            __syncwarp();
        };
        // O of slot s += diag(p_i) V_d[i], V_d[i] in V stage st: the weights of the 16 rows that step k concerns sit in the
        // same 8 columns as those of the other rows, whose lanes the step leaves alone.
        auto issue_draft_pv = [&](int s, int st, int i, bool commit) {
            tc_fence_after_sync();
#pragma unroll
            for (int k = 0; k < KT / 16; ++k) {
                const uint64_t b_desc = make_smem_desc_sw128(base + SMEM_V + st * KV_BYTES + k * 16 * 128, KV_HALF, 1024);
                const uint32_t off = k & 1 ? 0x0000ffffu : 0xffff0000u;
                if (leader)
                    umma_bf16_ta_lanes(tmem_base + 256 + s * HD, tmem_base + s * KT + DRAFT_P + 8 * i, b_desc, idesc_o,
                                       k >> 1 == 0 ? off : 0xffffffffu, k >> 1 == 1 ? off : 0xffffffffu, k >> 1 == 2 ? off : 0xffffffffu,
                                       k >> 1 == 3 ? off : 0xffffffffu);
            }
            if (leader && commit) umma_commit(pv_done(s));
            __syncwarp();
        };
        auto k_acquire = [&](int& st) {
            st = gk % K_STAGES;
            return wait_all(k_full(st), (gk / K_STAGES) & 1u, 4);
        };
        auto k_release = [&](int st) {
            if (leader) umma_commit(k_empty(st));
            __syncwarp();
            ++gk;
        };
        auto v_acquire = [&](int& st) {
            st = gv % KV_STAGES;
            return wait_all(v_full(st), (gv / KV_STAGES) & 1u, 8);
        };
        auto v_release = [&](int st) {
            if (leader) umma_commit(v_empty(st));
            __syncwarp();
            ++gv;
        };
        auto p_wait = [&](int s) {
            const bool r = wait_all(p_full(s), gp[s] & 1u, 7);
            ++gp[s];
            return r;
        };

        for (int idx = next_pair(0, 16); idx < p.pairs && ok; idx = next_pair(++it, 16)) {
            const Pair pr = decode_pair(p, idx);
            const int m = md;
            int j0, n1;
            own_share(pr, j0, n1);
            n1 -= j0;                                        // key tiles of slot 1
            if (CLUSTER && n1 == 0) continue;
            const int n0 = pr.act0 ? pr.qt[0] + 1 : 0;
            const bool a_on = pr.act0;
            const bool shared = p.head_pairing != 0;         // the draft tiles serve both slots
            if (a_on) {
                if (!wait_all(q_full(0), gq[0] & 1u, 6)) break;
                ++gq[0];
            }
            if (!wait_all(q_full(1), gq[1] & 1u, 6)) break;
            ++gq[1];
            // S-type products: steps 0 .. m + n_s - 1 of slot s (m draft score products, then the key tiles). Step k + 1 of
            // a slot is issued after its softmax warps arrived for step k. Key tile j is ring entry shared by both slots.
            int st;
            // ---- step 0 of both slots ----
            if (m > 0 && !shared) {
                if (a_on) {
                    if (!k_acquire(st)) break;
                    issue_s(0, st, false);
                    k_release(st);
                }
                if (!k_acquire(st)) break;
                issue_s(1, st, false);
                k_release(st);
            } else {
                if (!k_acquire(st)) break;
                if (a_on && (m > 0 || n0 > 0)) issue_s(0, st, m == 0 && n0 == 1);
                issue_s(1, st, m == 0 && n1 == 1);
                k_release(st);
            }
            // ---- draft score steps: after the arrival for draft pass i, the slot's next S (pass i + 1, or key tile 0) ----
            for (int i = 0; i < m && ok; ++i) {
                const bool next_is_tile = (i + 1 == m);
                if (next_is_tile || shared) {
                    bool have = false;
                    if (a_on) {
                        if (!p_wait(0)) { ok = false; break; }
                        if (!k_acquire(st)) { ok = false; break; }
                        have = true;
                        issue_s(0, st, next_is_tile && n0 == 1);
                    }
                    if (!p_wait(1)) { ok = false; break; }
                    if (!have && !k_acquire(st)) { ok = false; break; }
                    issue_s(1, st, next_is_tile && n1 == 1);
                    k_release(st);
                } else {
                    if (a_on) {
                        if (!p_wait(0)) { ok = false; break; }
                        if (!k_acquire(st)) { ok = false; break; }
                        issue_s(0, st, false);
                        k_release(st);
                    }
                    if (!p_wait(1)) { ok = false; break; }
                    if (!k_acquire(st)) { ok = false; break; }
                    issue_s(1, st, false);
                    k_release(st);
                }
            }
            // ---- key tiles ----
            for (int j = 0; j < n1 && ok; ++j) {
                int vst;
                if (!v_acquire(vst)) { ok = false; break; }
                bool k_ready = false;
                if (j < n0) {
                    if (!p_wait(0)) { ok = false; break; }
                    issue_pv(0, vst, 0, 0, 8, j == 0, m == 0 || j + 1 < n0);
                    if (j + 1 < n0) {
                        if (!k_acquire(st)) { ok = false; break; }
                        k_ready = true;
                        issue_s(0, st, j + 2 == n0);
                    }
                }
                if (!p_wait(1)) { ok = false; break; }
                issue_pv(1, vst, 0, 0, 8, j == 0, m == 0 || j + 1 < n1);
                v_release(vst);
                if (j + 1 < n1) {
                    if (!k_ready && !k_acquire(st)) { ok = false; break; }
                    issue_s(1, st, j + 2 == n1);
                    k_release(st);
                }
            }
            // ---- draft value products: the weights are there, each slot's last one completes its item ----
            for (int i = 0; i < m && ok; ++i) {
                int vst;
                if (!shared && a_on) {
                    if (!v_acquire(vst)) { ok = false; break; }
                    issue_draft_pv(0, vst, i, i + 1 == m);
                    v_release(vst);
                }
                if (!v_acquire(vst)) { ok = false; break; }
                if (shared && a_on) issue_draft_pv(0, vst, i, i + 1 == m);
                issue_draft_pv(1, vst, i, i + 1 == m);
                v_release(vst);
            }
        }
    }
    } else {
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(REGS_SOFTMAX));
        // ===================== softmax + epilogue warps =====================
        const int slot = (warp - 4) >> 2;
        const int quad = warp & 3;
        const int r = quad * 32 + lane;                       // row of the tile = TMEM lane
        const uint32_t lane_addr = static_cast<uint32_t>(quad * 32) << 16;
        const uint32_t tmem_s = tmem_base + slot * KT + lane_addr;
        const uint32_t tmem_o = tmem_base + 256 + slot * HD + lane_addr;
        const int m = p.m;
        float own_ref = -INFINITY, own_sum = 0.f;             // CLUSTER: of the row's part
        bool own_rows = false;
        uint32_t gs = 0, gpv = 0, it = 0;                     // S-type products seen, PV-type products requested
        bool ok = true;
        for (int idx = next_pair(0, 17); idx < p.pairs && ok; idx = next_pair(++it, 17)) {
            const Pair pr = decode_pair(p, idx);
            if (slot == 0 && !pr.act0) continue;
            const int qt = pr.qt[slot], h = pr.h[slot], b = pr.b;
            int j0 = 0, n = qt + 1;
            if (CLUSTER) own_share(pr, j0, n);
            if (CLUSTER && j0 == n) continue;
            const int t = qt * QT + r;                        // position in the sequence
            const bool valid = t < p.T;
            // ---- draft score steps: keep the diagonal element of each S (raw, unscaled) ----
            float sd[MAX_DRAFTS];
#pragma unroll
            for (int i = 0; i < MAX_DRAFTS; ++i) sd[i] = 0.f;
#pragma unroll 1
            for (int i = 0; i < md; ++i, ++gs) {
                if (!wait_barrier(s_full(slot), gs & 1u, abort_flag, p.status, 10)) { ok = false; break; }
                tc_fence_after_sync();
                uint32_t blk[32];
                tmem_ld32(tmem_s + 32 * quad, blk);           // this warp's diagonal block
                tmem_ld_wait(blk);
                float dv = 0.f;
#pragma unroll
                for (int c = 0; c < 32; ++c)
                    if (c == lane) dv = __uint_as_float(blk[c]);
#pragma unroll
                for (int ii = 0; ii < MAX_DRAFTS; ++ii)
                    if (ii == i) sd[ii] = dv;
                tc_fence_before_sync();
                __syncwarp();
                if (lane == 0) mbar_arrive(p_full(slot));
            }
            if (!ok) break;
            float mref = -INFINITY, l = 0.f;
#pragma unroll 1
            for (int j = j0; j < n; ++j, ++gs) {
                if (!wait_barrier(s_full(slot), gs & 1u, abort_flag, p.status, 10)) { ok = false; break; }
                tc_fence_after_sync();
                const bool last = (j == n - 1);
                // the row's 128 scores into registers
                uint32_t raw[4][32];
#pragma unroll
                for (int q = 0; q < 4; ++q) tmem_ld32(tmem_s + 32 * q, raw[q]);
#pragma unroll
                for (int q = 0; q < 4; ++q) tmem_ld_wait(raw[q]);
                // Columns past t - m are hidden in the score tile: the causal part (s > t) and the m substituted
                // entries (t - m < s <= t), which enter the row's maximum and sum as scalars at the last tile.
                // Only tiles reaching past the first row's limit can hold such columns.
                if (j * KT + KT - 1 > qt * QT - m) {
                    const int lim = t - m - j * KT;
#pragma unroll
                    for (int q = 0; q < 4; ++q)
#pragma unroll
                        for (int c = 0; c < 32; ++c)
                            if (32 * q + c > lim) raw[q][c] = 0xff800000u;      // -inf
                }
                float mx[4];
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    mx[q] = fmaxf(__uint_as_float(raw[q][0]), __uint_as_float(raw[q][1]));
#pragma unroll
                    for (int c = 2; c < 32; c += 2) mx[q] = fmax3(mx[q], __uint_as_float(raw[q][c]), __uint_as_float(raw[q][c + 1]));
                }
                float mxa = fmaxf(fmaxf(mx[0], mx[1]), fmaxf(mx[2], mx[3]));
                if (last) {
#pragma unroll
                    for (int i = 0; i < MAX_DRAFTS; ++i)
                        if (i < md && t - i >= 0) mxa = fmaxf(mxa, sd[i]);
                }
                const float cand = mxa * p.c2;
                if (j == j0) {
                    mref = cand;
                } else {
                    const bool grow = cand > mref + RESCALE_LOG2;      // also true when every earlier column of the row was hidden
                    if (__any_sync(0xffffffffu, grow)) {
                        // Move the reference: this row's accumulator and sum are multiplied by 2^(old ref - new ref).
                        // The slot's products are complete up to this tile's S (the tensor core finishes them in
                        // issue order), so nothing else touches the accumulator now.
                        const float f = grow ? ex2(mref - cand) : 1.f;
                        if (grow) {
                            mref = cand;
                            l *= f;
                        }
#pragma unroll 1
                        for (int c0 = 0; c0 < HD; c0 += 32) {
                            uint32_t o[32];
                            tmem_ld32(tmem_o + c0, o);
                            tmem_ld_wait(o);
#pragma unroll
                            for (int c = 0; c < 32; ++c) o[c] = __float_as_uint(__uint_as_float(o[c]) * f);
                            tmem_st32(tmem_o + c0, o);
                        }
                        tmem_st_wait();
                    }
                }
                // ---- P = 2^(x c2 - ref): row sum in fp32, bf16 pairs into tensor memory, 32 columns at a time ----
                // (a row whose columns were all hidden so far has ref = -inf; it gets P = 0, not 2^(-inf + inf))
                const float nref = mref == -INFINITY ? 0.f : -mref;
                float ls[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    uint32_t pk[16];
#pragma unroll
                    for (int c = 0; c < 32; c += 2) {
                        float x0, x1;
                        ffma2(x0, x1, __uint_as_float(raw[q][c]), __uint_as_float(raw[q][c + 1]), p.c2, p.c2, nref, nref);
                        const float e0 = ex2(x0), e1 = ex2(x1);
                        fadd2(ls[(c >> 1) & 1], ls[2 + ((c >> 1) & 1)], ls[(c >> 1) & 1], ls[2 + ((c >> 1) & 1)], e0, e1);
                        pk[c >> 1] = pack_bf16(e0, e1);
                    }
                    hca::tmem_st16(tmem_s + 16 * q, pk);
                }
                l += (ls[0] + ls[1]) + (ls[2] + ls[3]);
                if (last) {
                    // the substituted entries' weights: pass i in 8 columns beside P, this row's in the word of its key
#pragma unroll
                    for (int i = 0; i < MAX_DRAFTS; ++i) {
                        if (i < md) {
                            const float pi = t - i >= 0 ? ex2(fmaf(sd[i], p.c2, nref)) : 0.f;
                            l += pi;
                            const uint32_t bits = pack_bf16(pi, 0.f) << ((r & 1) * 16);
                            uint32_t pk[8];
#pragma unroll
                            for (int w = 0; w < 8; ++w) pk[w] = w == ((r & 15) >> 1) ? bits : 0u;
                            hca::tmem_st8(tmem_s + DRAFT_P + 8 * i, pk);
                        }
                    }
                }
                tmem_st_wait();
                tc_fence_before_sync();
                __syncwarp();
                if (lane == 0) mbar_arrive(p_full(slot));
                ++gpv;
            }
            if (!ok) break;
            // ---- epilogue: O / l as bf16, each thread stores its own 256-byte row ----
            if (!wait_barrier(pv_done(slot), (gpv - 1u) & 1u, abort_flag, p.status, 13)) break;
            tc_fence_after_sync();
            if (CLUSTER) {
                own_ref = mref;
                own_sum = l;
                own_rows = true;
                break;
            }
            const float inv = 1.f / l;
            if (valid && p.lse != nullptr)
                p.lse[(static_cast<size_t>(b) * p.H + h) * p.T + t] = (mref + log2f(l)) * 0.6931471805599453f;
            __nv_bfloat16* orow = p.O + ((static_cast<size_t>(b) * p.T + (valid ? t : 0)) * p.H + h) * HD;
            {
                uint32_t raw[4][32];
#pragma unroll
                for (int q = 0; q < 4; ++q) tmem_ld32(tmem_o + 32 * q, raw[q]);
#pragma unroll
                for (int q = 0; q < 4; ++q) tmem_ld_wait(raw[q]);
                if (valid) {
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
#pragma unroll
                        for (int q8 = 0; q8 < 2; ++q8) {
                            const uint32_t* x = &raw[q][16 * q8];
                            st_global_v8(orow + 32 * q + 16 * q8,
                                         pack_bf16(__uint_as_float(x[0]) * inv, __uint_as_float(x[1]) * inv),
                                         pack_bf16(__uint_as_float(x[2]) * inv, __uint_as_float(x[3]) * inv),
                                         pack_bf16(__uint_as_float(x[4]) * inv, __uint_as_float(x[5]) * inv),
                                         pack_bf16(__uint_as_float(x[6]) * inv, __uint_as_float(x[7]) * inv),
                                         pack_bf16(__uint_as_float(x[8]) * inv, __uint_as_float(x[9]) * inv),
                                         pack_bf16(__uint_as_float(x[10]) * inv, __uint_as_float(x[11]) * inv),
                                         pack_bf16(__uint_as_float(x[12]) * inv, __uint_as_float(x[13]) * inv),
                                         pack_bf16(__uint_as_float(x[14]) * inv, __uint_as_float(x[15]) * inv));
                        }
                    }
                }
            }
            // the accumulator and the score buffer go back to the tensor core with the next item's first step
            tc_fence_before_sync();
        }
        if constexpr (CLUSTER) {
            const int C = p.cluster, rows = QT / C;
            const Pair pr = decode_pair(p, static_cast<int>(blockIdx.x) / C);
            tc_fence_before_sync();
            __syncthreads();
            cluster_sync();                                   // every CTA's products are complete, its queries' and keys' room is free
            tc_fence_after_sync();
            if (slot == 1) {
                const uint32_t dst = map_to_rank(base + (z * rows + r % rows) * (ROW_PITCH * 4), r / rows);
#pragma unroll 1
                for (int c0 = 0; c0 < HD; c0 += 32) {
                    uint32_t v[32];
                    tmem_ld32(tmem_o + c0, v);
                    tmem_ld_wait(v);
#pragma unroll
                    for (int j = 0; j < 8; ++j) {
                        if (!own_rows) v[4 * j] = v[4 * j + 1] = v[4 * j + 2] = v[4 * j + 3] = 0u;      // no tile: no accumulator
                        st_cluster_v4(dst + (c0 + 4 * j) * 4, v[4 * j], v[4 * j + 1], v[4 * j + 2], v[4 * j + 3]);
                    }
                }
                st_cluster_v4(dst + HD * 4, __float_as_uint(own_ref), __float_as_uint(own_sum), 0u, 0u);
            }
            cluster_sync();
            for (int i = static_cast<int>(threadIdx.x) - 128; i < rows * (HD / 8); i += 256) {
                const int c8 = i % (HD / 8), rl = i / (HD / 8), t = pr.qt[1] * QT + z * rows + rl;
                if (t >= p.T) continue;
                const float* src = reinterpret_cast<const float*>(smem_raw) + rl * ROW_PITCH;
                float ref = -INFINITY, sum = 0.f, f[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
                for (int q = 0; q < C; ++q) ref = fmaxf(ref, src[q * rows * ROW_PITCH + HD]);
                for (int q = 0; q < C; ++q) {
                    const float* part = src + q * rows * ROW_PITCH;
                    const float w = ex2(part[HD] - ref);      // (a part without a visible key: 2^-inf)
                    sum = fmaf(w, part[HD + 1], sum);
                    const float4 x = *reinterpret_cast<const float4*>(part + 8 * c8), y = *reinterpret_cast<const float4*>(part + 8 * c8 + 4);
                    f[0] = fmaf(w, x.x, f[0]); f[1] = fmaf(w, x.y, f[1]); f[2] = fmaf(w, x.z, f[2]); f[3] = fmaf(w, x.w, f[3]);
                    f[4] = fmaf(w, y.x, f[4]); f[5] = fmaf(w, y.y, f[5]); f[6] = fmaf(w, y.z, f[6]); f[7] = fmaf(w, y.w, f[7]);
                }
                const float inv = 1.f / sum;
                if (c8 == 0 && p.lse != nullptr)
                    p.lse[(static_cast<size_t>(pr.b) * p.H + pr.h[1]) * p.T + t] = (ref + log2f(sum)) * 0.6931471805599453f;
                reinterpret_cast<uint4*>(p.O + ((static_cast<size_t>(pr.b) * p.T + t) * p.H + pr.h[1]) * HD)[c8] =
                    make_uint4(pack_bf16(f[0] * inv, f[1] * inv), pack_bf16(f[2] * inv, f[3] * inv), pack_bf16(f[4] * inv, f[5] * inv), pack_bf16(f[6] * inv, f[7] * inv));
            }
        }
    }
    if (CLUSTER && warp < 4) {
        // (apart from the softmax warps' side: these warps have given their registers up)
        __syncwarp();
        tc_fence_before_sync();
        __syncthreads();
        cluster_sync();
        cluster_sync();
    }

    // ---- teardown ----
    tc_fence_before_sync();
    __syncthreads();
    if (*abort_flag) {
        // a wait gave up: let copies that may still be in flight land before the CTA's memory is released
        const unsigned long long t0 = globaltimer_ns();
        while (globaltimer_ns() - t0 < 200000ull) __nanosleep(1000);
    }
    if (warp == 1) {
        tc_fence_after_sync();
        tmem_dealloc(tmem_base, TMEM_COLS);
    }
}

}  // namespace hca2
}  // namespace hass

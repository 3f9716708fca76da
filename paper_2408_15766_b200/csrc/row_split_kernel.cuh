// row_split_kernel: what row_kernel does with a row of few rows' logits, by a cluster of blocks that split the row.
#pragma once
#include "normed_kernel.cuh"

namespace hass {

constexpr int SPLIT_THREADS = 512;                      // of a block where clusters share rows; fewer for short rows of a block each
constexpr int SPLIT_MAX = 8;                            // blocks per row, at most (the portable cluster size)
constexpr int SPLIT_STEP = SPLIT_THREADS * 4;           // logits of a row that a block's threads hold one 16-byte piece each of
constexpr int SPLIT_PIECES = 8;                         // such pieces per thread, at most

template <int THREADS, bool CLUSTER>
struct SplitShared : RowPool {
    unsigned long long list[2][K_CAP];                  // the K largest logits of this block's piece of the target's (0) and of the draft's (1)
                                                        // row as ranks, descending; 0: none
    float other[2][K_CAP];                              // the other row's logit at the same token
    float stats[4];                                     // the piece's largest logit and sum of 2^((z - m) log2e), target and draft
    union {
        struct {
            unsigned long long list[(CLUSTER ? SPLIT_MAX : 1) * K_CAP];   // one list of every block of the row
            float other[(CLUSTER ? SPLIT_MAX : 1) * K_CAP];
        } all;
        float part[THREADS * 8];                        // sums of rows of W, one per thread
    };
    float all_stats[SPLIT_MAX][4];
    int tok[K_CAP];                                     // Omega_hat
    float q[K_CAP], z[K_CAP], zt[K_CAP];
    int tok_d[K_CAP];
    float sum;
    float ce[SPLIT_MAX];
    int count;
};

// Block-collective: the K largest logits of the block's piece (columns first ..., thread T's at (u THREADS + T) 4 in v[u]) as a
// descending list; m = the thread's largest.
template <int SPLIT_THREADS, int E>
__device__ __forceinline__ void piece_list(const float4 (&v)[E], const float* piece, int len, int V, int first, int K, float m, RowPool& sh,
                                           unsigned long long* list) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    uint32_t key, hi;
    const uint32_t T = bound_from_maxima<SPLIT_THREADS>(K, m, sh, key, hi);
    const int room = pool_room(K);
    if (key >= T) {
#pragma unroll
        for (int u = 0; u < E; ++u) {
            const float z[4] = {v[u].x, v[u].y, v[u].z, v[u].w};
            const int at = (u * SPLIT_THREADS + tid) * 4;
#pragma unroll
            for (int j = 0; j < 4; ++j)
                if (reaches(z[j], at + j, V, T)) {
                    const int pos = atomicAdd(&sh.n, 1);
                    if (pos < room) sh.pool[pos] = logit_rank(z[j], static_cast<uint32_t>(first + at + j));
                }
        }
    }
    __syncthreads();
    int n = sh.n;
    if (n > room) n = collect_from_many<SPLIT_THREADS>(piece, len, V, first, K, key, T, hi, sh);
    for (int j = n + tid; j < K; j += SPLIT_THREADS) list[j] = 0ull;
    for (int e = warp; e < n; e += SPLIT_THREADS / 32) {
        const unsigned long long x = sh.pool[e];
        int rank = 0;
        for (int i = lane; i < n; i += 32) rank += sh.pool[i] > x ? 1 : 0;
        rank = __reduce_add_sync(0xffffffffu, rank);
        if (lane == 0 && rank < K) list[rank] = x;
    }
    __syncthreads();
}

// Block-collective: the lists `which` of all C blocks of the row merged into tok / val, in descending order; with `other` what
// they carry beside. Fewer than K logits above -inf: the rest is token 0 with the values given. Ends without a barrier.
template <int SPLIT_THREADS, typename S>
__device__ __forceinline__ void merge_lists(int which, int C, int K, S& sh, int* tok, float* val, float* other, float fill_val, float fill_other) {
    const int tid = threadIdx.x;
    const uint32_t list = smem_u32(sh.list[which]), oth = smem_u32(sh.other[which]);
    for (int e = tid; e < C * K; e += SPLIT_THREADS) {
        const int c = e / K, i = e - c * K;
        sh.all.list[e] = ld_cluster_u64(map_to_rank(list + 8 * i, c));
        sh.all.other[e] = ld_cluster_f32(map_to_rank(oth + 4 * i, c));
    }
    for (int j = tid; j < K; j += SPLIT_THREADS) {
        tok[j] = 0;
        val[j] = fill_val;
        other[j] = fill_other;
    }
    __syncthreads();
    for (int e = tid; e < C * K; e += SPLIT_THREADS) {
        const unsigned long long x = sh.all.list[e];
        if (x == 0ull) continue;
        const int c = e / K;
        int rank = e - c * K;
        for (int o = 0; o < C && rank < K; ++o) {
            if (o == c) continue;
            // how many of the other list lie above x
            int lo = 0, hi = K;
            while (lo < hi) {
                const int mid = (lo + hi) >> 1;
                if (sh.all.list[o * K + mid] > x)
                    lo = mid + 1;
                else
                    hi = mid;
            }
            rank += lo;
        }
        if (rank < K) {
            tok[rank] = static_cast<int>(~static_cast<uint32_t>(x));
            val[rank] = __uint_as_float(key_bits(static_cast<uint32_t>(x >> 32)));
            other[rank] = sh.all.other[e];
        }
    }
}

// A cluster of p.split blocks per row. A block holds its piece of both rows in registers from the one reading of them to the
// dz_d that it writes: largest logits, sums, and the piece's own K largest as a sorted list; then one exchange through
// distributed shared memory, after which every block merges the lists for itself. dz_d does not go over the draft's logits
// but over the target's, which no block needs by then.
// row_kernel, one block per row, is a chain of passes over 4 V bytes that one SM reads, on as many SMs as there are rows.
// Short rows have a block each (THREADS x E pieces of four logits) and as many of them on an SM as 80 registers per thread allow.
template <int OBJ, int E, int SPLIT_THREADS, bool CLUSTER>
__global__ void __launch_bounds__(SPLIT_THREADS, CLUSTER || SPLIT_THREADS == 512 ? 1 : 768 / SPLIT_THREADS) row_split_kernel(const __grid_constant__ RowParams p) {
    constexpr int SPLIT_STEP = SPLIT_THREADS * 4;
    __shared__ SplitShared<SPLIT_THREADS, CLUSTER> sh;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int C = CLUSTER ? p.split : 1, K = p.K;
    const int row = blockIdx.x / C, rank = blockIdx.x - row * C;      // (clusters are consecutive blocks)
    wait_previous_kernel(!p.release_late);
    const float* zrow = p.z != nullptr ? p.z + static_cast<long long>(row) * p.pitch : nullptr;
    const float* trow = p.zt != nullptr ? p.zt + static_cast<long long>(row) * p.pitch : nullptr;
    int* idx = p.idx + static_cast<long long>(row) * p.idx_pitch;
    float* q = p.q + static_cast<long long>(row) * p.idx_pitch;
    const int first = rank * (E * SPLIT_STEP), len = min(static_cast<int>(p.pitch) - first, E * SPLIT_STEP), V = p.V - first;      // (<= 0: an empty piece)

    float4 t[E], z[E];
    auto load = [&](const float* from, float4 (&v)[E]) {
#pragma unroll
        for (int u = 0; u < E; ++u) {
            const int at = (u * SPLIT_THREADS + tid) * 4;
            v[u] = from != nullptr && at < len ? *reinterpret_cast<const float4*>(from + first + at)
                                               : make_float4(-INFINITY, -INFINITY, -INFINITY, -INFINITY);
        }
    };
    load(trow, t);
    load(zrow, z);
    // this thread's largest logit and sum of 2^((z - m) log2e)
    auto stats = [&](const float4 (&v)[E], float& m, float& s) {
        m = -INFINITY;
        s = 0.f;
#pragma unroll
        for (int u = 0; u < E; ++u) m = fmaxf(m, fmaxf(fmax3(v[u].x, v[u].y, v[u].z), v[u].w));
        const float mneg = m == -INFINITY ? 0.f : -m * LOG2E;      // (nothing but -inf: each adds zero)
#pragma unroll
        for (int u = 0; u < E; ++u)
            s += ex2(fmaf(v[u].x, LOG2E, mneg)) + ex2(fmaf(v[u].y, LOG2E, mneg)) + ex2(fmaf(v[u].z, LOG2E, mneg)) + ex2(fmaf(v[u].w, LOG2E, mneg));
    };
    // the sum over the lanes, or over `n` entries, of parts (m, s)
    auto merge_stats = [&](float& m, float& s) {
        float mx = m;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        const float base = mx == -INFINITY ? 0.f : mx;
        s *= ex2(((m == -INFINITY ? base : m) - base) * LOG2E);      // (a part without a logit: its sum is zero)
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        m = mx;
    };
    float m_t = -INFINITY, s_t = 0.f, m_d = -INFINITY, s_d = 0.f;
    if (trow) stats(t, m_t, s_t);
    if (zrow) stats(z, m_d, s_d);
    {
        float mt = m_t, st = s_t, md = m_d, sd = s_d;
        merge_stats(mt, st);
        merge_stats(md, sd);
        if (lane == 0) {
            sh.red[0][warp] = mt;
            sh.red[1][warp] = st;
            sh.red[2][warp] = md;
            sh.red[3][warp] = sd;
        }
        __syncthreads();
        if (warp < 2) {
            float m = lane < SPLIT_THREADS / 32 ? sh.red[2 * warp][lane] : -INFINITY, s = lane < SPLIT_THREADS / 32 ? sh.red[2 * warp + 1][lane] : 0.f;
            merge_stats(m, s);
            if (lane == 0) {
                sh.stats[2 * warp] = m;
                sh.stats[2 * warp + 1] = s;
            }
        }
        __syncthreads();      // (red is written again)
    }
    if (trow) {
        piece_list<SPLIT_THREADS>(t, trow + first, len, V, first, K, m_t, sh, sh.list[0]);
        for (int j = tid; j < K; j += SPLIT_THREADS) {
            const unsigned long long x = sh.list[0][j];
            sh.other[0][j] = x != 0ull && zrow ? zrow[~static_cast<uint32_t>(x)] : -INFINITY;
        }
        if (OBJ == ROW_BIDIR) {
            piece_list<SPLIT_THREADS>(z, zrow + first, len, V, first, K, m_d, sh, sh.list[1]);
            for (int j = tid; j < K; j += SPLIT_THREADS) {
                const unsigned long long x = sh.list[1][j];
                sh.other[1][j] = x != 0ull ? trow[~static_cast<uint32_t>(x)] : -INFINITY;
            }
        }
    }
    const float z0 = zrow ? zrow[0] : 0.f, t0 = OBJ == ROW_BIDIR ? trow[0] : 0.f;
    cluster_sync();
    if (tid < 4 * C) sh.all_stats[tid >> 2][tid & 3] = ld_cluster_f32(map_to_rank(smem_u32(&sh.stats[tid & 3]), tid >> 2));
    if (trow) {
        merge_lists<SPLIT_THREADS>(0, C, K, sh, sh.tok, sh.zt, sh.z, -INFINITY, z0);
        if (OBJ == ROW_BIDIR) {
            __syncthreads();
            merge_lists<SPLIT_THREADS>(1, C, K, sh, sh.tok_d, sh.q, sh.q + K, z0, t0);      // (q is free until then; 2 K <= K_CAP)
        }
    } else {
        for (int j = tid; j < K; j += SPLIT_THREADS) {
            const int tk = idx[j];
            sh.tok[j] = tk < p.V ? tk : -1;
            sh.q[j] = q[j];
            sh.z[j] = tk >= 0 && tk < p.V ? zrow[tk] : 0.f;
        }
    }
    __syncthreads();
    // No block reads another's shared memory, or target logits, from here on once all have come here: dz_d may be written, and
    // (waited for at the end) a block may leave.
    cluster_arrive();
    auto lse = [&](int k) {
        float m = lane < C ? sh.all_stats[lane][k] : -INFINITY, s = lane < C ? sh.all_stats[lane][k + 1] : 0.f;
        merge_stats(m, s);
        return (m == -INFINITY ? 0.f : m) + logf(s);
    };
    const float lse_t = trow ? lse(0) : 0.f, lse_d = p.lse_in != nullptr ? p.lse_in[row] : zrow ? lse(2) : 0.f;

    int n_tok = K;                        // entries of Omega_hat's list (2K at most for the bi-directional set)
    if (trow) {
        int taken = K;
        if (OBJ == ROW_BIDIR) {
            // the draft's own K most probable tokens that are not in the target's set join Omega_hat, in their order
            if (warp == 0) {
                int n = K;
                for (int j0 = 0; j0 < K; j0 += 32) {
                    const int j = j0 + lane;
                    const int tk = j < K ? sh.tok_d[j] : -1;
                    bool joins = j < K;
                    for (int i = 0; i < K; ++i) joins = joins && sh.tok[i] != tk;
                    const uint32_t bm = __ballot_sync(0xffffffffu, joins);
                    const int at = n + __popc(bm & ((1u << lane) - 1u));
                    if (joins) {
                        sh.tok[at] = tk;
                        sh.zt[at] = sh.q[K + j];
                        sh.z[at] = sh.q[j];
                    }
                    n += __popc(bm);
                }
                for (int j = n + lane; j < 2 * K; j += 32) {
                    sh.tok[j] = -1;
                    sh.zt[j] = -INFINITY;
                    sh.z[j] = 0.f;
                }
                if (lane == 0) sh.count = n;
            }
            __syncthreads();
            taken = sh.count;
            n_tok = 2 * K;
        }
        if (tid < n_tok) sh.q[tid] = sh.zt[tid] > -INFINITY ? expf(sh.zt[tid] - lse_t) : 0.f;      // (-inf: filled up)
        __syncthreads();
        if (p.top_p > 0.f) {
            // Top-P: a token belongs to Omega_hat while the probability of those before it is <= P
            if (tid == 0) {
                taken = 0;
                float cum = 0.f;
                for (int j = 0; j < K; ++j) {
                    const float qj = sh.q[j];
                    if (cum > p.top_p) {
                        sh.tok[j] = -1;
                        sh.q[j] = 0.f;
                    } else {
                        ++taken;
                    }
                    cum += qj;
                }
                if (!(cum > p.top_p)) taken = -taken;      // all K tokens taken and P still not exceeded: the cap cut the prefix
            }
            __syncthreads();
        }
        if (rank == 0) {
            if (tid < n_tok) {
                idx[tid] = sh.tok[tid];
                q[tid] = sh.q[tid];
            }
            if (tid == 0) {
                p.lse_t[row] = lse_t;
                if (p.n_out) p.n_out[row] = taken;
            }
        }
    }
    if (!zrow) {
        cluster_wait();
        return;
    }
    const float g = p.grad_loss ? p.grad_loss[row] : 1.f;
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
            if (rank == 0 && p.lse_in == nullptr) {
                p.loss[row] = loss;
                p.lse_d[row] = lse_d;
            }
        }
    }
    __syncthreads();
    cluster_wait();      // (the target's logits have been read)
    if (!p.make_dz) return;
    __nv_bfloat16* drow = p.dz + static_cast<long long>(row) * (2 * p.pitch) + first;
    const float S_q = sh.sum, c = OBJ == ROW_COMBINED ? g * (1.f + p.w * S_q) : OBJ == ROW_BIDIR ? 1.f : g * S_q, shift = -lse_d * LOG2E, shift_t = -lse_t * LOG2E;
    float ce = 0.f;
#pragma unroll
    for (int u = 0; u < E; ++u) {
        const int at = (u * SPLIT_THREADS + tid) * 4;
        if (at < len) {
            const float zd[4] = {z[u].x, z[u].y, z[u].z, z[u].w};
            float o[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) o[j] = c * ex2(fmaf(zd[j], LOG2E, shift));
            if (OBJ == ROW_COMBINED) {
                const float zt[4] = {t[u].x, t[u].y, t[u].z, t[u].w};
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const float qv = ex2(fmaf(zt[j], LOG2E, shift_t));
                    o[j] = fmaf(-g, qv, o[j]);
                    if (at + j < V) ce = fmaf(qv, lse_d - zd[j], ce);      // (-inf beyond the vocabulary)
                }
            }
            *reinterpret_cast<uint2*>(drow + at) = make_uint2(pack_bf16x2(o[0], o[1]), pack_bf16x2(o[2], o[3]));
        }
    }
    auto sparse_out = [&](int k0, const float (&a)[8]) {
        float* o = p.sparse_out + static_cast<long long>(row) * p.d + k0;
        *reinterpret_cast<float4*>(o) = make_float4(a[0], a[1], a[2], a[3]);
        *reinterpret_cast<float4*>(o + 4) = make_float4(a[4], a[5], a[6], a[7]);
    };
    if (OBJ == ROW_BIDIR) {
        if (rank == 0 && tid == 0) p.coef_out[row] = g * S_q;
        const int n = sh.count;
        if (tid < n) sh.zt[tid] = g * sh.q[tid];
        __syncthreads();
        sum_rows<SPLIT_THREADS>(p.W, p.d, sh.tok, sh.zt, n, rank, C, sh.part, sparse_out);
        return;
    }
    if (OBJ == ROW_COMBINED) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) ce += __shfl_xor_sync(0xffffffffu, ce, o);
        if (lane == 0) sh.red[0][warp] = ce;
    }
    __syncthreads();
    // Tokens of q = 0 keep the dense value: the one that fills up a set of fewer than K logits above -inf (token 0) may be in it
    // already, and an entry has one writer.
    if (tid < n_tok) {
        const int at = sh.tok[tid] - first;
        const bool own = sh.tok[tid] >= 0 && at >= 0 && at < E * SPLIT_STEP;
        const float q_own = !own && OBJ != ROW_COMBINED ? 0.f : p.lse_in != nullptr ? repeated_q(sh.tok, sh.q, n_tok, tid) : sh.q[tid];
        float left = 0.f;
        if (q_own != 0.f) {
            const float dense = c * ex2(fmaf(sh.z[tid], LOG2E, shift)), target = OBJ == ROW_COMBINED ? g * ex2(fmaf(sh.zt[tid], LOG2E, shift_t)) : 0.f;
            const float o = dense - (OBJ == ROW_COMBINED ? target + g * p.w * q_own : g * q_own);
            const __nv_bfloat16 b = __float2bfloat16_rn(o);
            if (own) drow[at] = b;
            if (OBJ == ROW_COMBINED) left = left_over(o, b, dense, target);      // (of all tokens: the blocks share the columns)
        }
        if (OBJ == ROW_COMBINED) sh.zt[tid] = left;
    }
    if (OBJ == ROW_COMBINED) {
        if (rank == 0 && tid == 0) p.coef_out[row] = 1.f;
        if (K > 32) __syncthreads();      // (up to 32 tokens are the first warp's own)
        __syncwarp();
        if (warp == 0) {
            const int n = keep_weighted(sh.tok, sh.zt, K);
            if (lane == 0) sh.count = n;
        }
        __syncthreads();
        sum_rows<SPLIT_THREADS>(p.W, p.d, sh.tok, sh.zt, sh.count, rank, C, sh.part, sparse_out);
    }
    if (OBJ == ROW_COMBINED) {
        if (warp == 0) {
            float v = lane < SPLIT_THREADS / 32 ? sh.red[0][lane] : 0.f;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
            if (lane == 0) st_cluster_f32(map_to_rank(smem_u32(&sh.ce[rank]), 0), v);
        }
        cluster_sync();
        if (rank == 0 && tid == 0) {
            float v = 0.f;
            for (int i = 0; i < C; ++i) v += sh.ce[i];
            p.loss_ce[row] = v;
        }
    }
}

}  // namespace hass

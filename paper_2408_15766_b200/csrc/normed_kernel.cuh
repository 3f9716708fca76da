// normed_kernel: loss and gradient of the Normed Top-K variant once Omega_hat is known, and the sum of rows of W that it shares with
// row_split_kernel.
#pragma once
#include "kernels.cuh"

namespace hass {

// The first of `units` units that is the rank-th of C blocks', which share them: a block has units / C of them, or one more
__host__ __device__ constexpr int part_begin(int units, int rank, int C) { return static_cast<int>(static_cast<long long>(units) * rank / C); }

// Block-collective: this block's part of the columns of sum_j w[j] W[tok[j], :], j < n, handed to out(first column, eight sums), where C
// blocks share the columns and this is the rank-th. Where the part is narrow, groups of threads take every so many-th token each, and their
// sums are added up in order (part: 8 THREADS floats of shared memory).
template <int THREADS, typename F>
__device__ __forceinline__ void sum_rows(const __nv_bfloat16* W, int d, const int* tok, const float* w, int n, int rank, int C, float* part, F&& out) {
    const int tid = threadIdx.x, units = d / 8;
    const int u0 = part_begin(units, rank, C), u1 = part_begin(units, rank + 1, C);
    const int per = max(32, min((u1 - u0 + 31) / 32 * 32, THREADS)), groups = min(gather_groups(u1 - u0, THREADS), max(n, 1)), g = tid / per;
    for (int b = u0; b < u1; b += THREADS) {
        const int u = b + tid - g * per;
        float a[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
        if (u < u1 && g < groups) {
#pragma unroll 8
            for (int j = g; j < n; j += groups) {
                float wf[8];
                unpack8(*reinterpret_cast<const uint4*>(W + static_cast<long long>(tok[j]) * d + 8 * u), wf);
                const float c = w[j];
#pragma unroll
                for (int t = 0; t < 8; ++t) a[t] = fmaf(c, wf[t], a[t]);
            }
        }
        if (groups > 1) {      // (then this is the only round)
#pragma unroll
            for (int t = 0; t < 8; ++t) part[t * THREADS + tid] = a[t];
            __syncthreads();
            if (g == 0 && u < u1) {
                for (int o = 1; o < groups; ++o)
#pragma unroll
                    for (int t = 0; t < 8; ++t) a[t] += part[t * THREADS + tid + o * per];
            }
        }
        if (g == 0 && u < u1) out(8 * u, a);
    }
}

constexpr int NORMED_THREADS = FIN_WARPS * 32;
constexpr int NORMED_MAX = 8;      // blocks per row, at most (the portable cluster size)

// Blocks per row: as many as are resident at once, of 256 columns at least, 2048 where there is one group of tokens to gather
inline int normed_split(long long N, long long d, int K, int sms) {
    int split = 1;
    while (split < NORMED_MAX && 2 * split * N <= 3ll * sms && d >= (K > FIN_GRP ? 512ll : 4096ll) * split) split *= 2;
    return split;
}
// Their dynamic shared memory, the same for all: what the narrowest part needs (of 257 units in two parts the one of 128 has groups, the one of 129
// has none)
inline int normed_smem(long long d, int split) { return gather_smem(static_cast<int>(d / 8 / split)); }

struct NormedParams {
    int d, K;
    const __nv_bfloat16* H_d;
    const __nv_bfloat16* W;
    const int* idx;                // [N, K] Omega_hat in descending q
    const float* q;
    const float* grad_loss;
    float* loss;
    void* dH;                      // [N, d]
    int dH_fp32;
    int split;                     // blocks per row
};

// A cluster of p.split blocks per row: q and p renormalised over Omega_hat, loss sum_x qn(x) (lse_k - z_d(x)) and the gradient row
// sum_x g (pn(x) - qn(x)) W[x, :]. There is no sweep of the draft rows: the K draft logits are dot products in fp32. A block takes its part of the
// columns in the dot products, whose sums the blocks exchange through distributed shared memory, and in the gradient.
// Bound by the latency of gathered rows of W, so that the rows of a call are spread over all SMs (one block of eight warps per row
// left 106 SMs idle with 42 rows): call of 42 rows x 8192 x 128256, K = 98 486 -> 423 us, 4 x 4096 x 128256, K = 55 253 -> 244, 85 x 4096 x 32000,
// K = 15 71.0 -> 66.7; 2048 x 4096 x 32000 499 either way.
__global__ void __launch_bounds__(NORMED_THREADS, 3) normed_kernel(const __grid_constant__ NormedParams p) {
    __shared__ int tok[K_CAP];
    __shared__ float q[K_CAP], z[K_CAP], w[K_CAP];
    __shared__ float parts[NORMED_MAX][K_CAP];      // the blocks' parts of the dot products
    __shared__ float part[FIN_WARPS][K_CAP];
    extern __shared__ float sh_cols[];
    wait_previous_kernel();
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int C = p.split, K = p.K;
    const int row = blockIdx.x / C, rank = blockIdx.x - row * C;      // (clusters are consecutive blocks)
    if (C > 1) cluster_arrive();
    for (int j = tid; j < K; j += NORMED_THREADS) {
        const int t = p.idx[static_cast<long long>(row) * K + j];
        tok[j] = t < 0 ? 0 : t;
        q[j] = p.q[static_cast<long long>(row) * K + j];
    }
    __syncthreads();
    auto warp_sum = [](float v) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        return v;
    };
    const int units = p.d / 8;
    gather_rows(p.H_d + static_cast<long long>(row) * p.d, p.W, p.d, part_begin(units, rank, C), part_begin(units, rank + 1, C), tok, 0, K, z, nullptr, 0.f, nullptr, part, sh_cols);
    if (C > 1) {
        cluster_wait();      // all blocks of the row run: their shared memory may be written
        for (int e = tid; e < C * K; e += NORMED_THREADS) {
            const int c = e / K, j = e - c * K;
            st_cluster_f32(map_to_rank(smem_u32(&parts[rank][j]), c), z[j]);
        }
        cluster_sync();
        for (int j = tid; j < K; j += NORMED_THREADS) {
            float v = 0.f;
            for (int c = 0; c < C; ++c) v += parts[c][j];
            z[j] = v;
        }
        __syncthreads();
    }
    if (warp == 0) {
        float S_q = 0.f, mx = -INFINITY, se = 0.f, loss = 0.f;
        for (int j = lane; j < K; j += 32) {
            S_q += q[j];
            mx = fmaxf(mx, z[j]);
        }
        S_q = warp_sum(S_q);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        for (int j = lane; j < K; j += 32) se += expf(z[j] - mx);
        const float lse_k = mx + logf(warp_sum(se)), g = p.grad_loss ? p.grad_loss[row] : 1.f;
        for (int j = lane; j < K; j += 32) {
            loss += q[j] / S_q * (lse_k - z[j]);
            w[j] = g * (expf(z[j] - lse_k) - q[j] / S_q);      // dL/dz_d on Omega_hat
        }
        loss = warp_sum(loss);
        if (rank == 0 && lane == 0) p.loss[row] = loss;
    }
    __syncthreads();
    const long long at = static_cast<long long>(row) * p.d;
    sum_rows<NORMED_THREADS>(p.W, p.d, tok, w, K, rank, C, sh_cols, [&](int k0, const float (&a)[8]) {
        if (p.dH_fp32) {
            float* o = static_cast<float*>(p.dH) + at + k0;
            *reinterpret_cast<float4*>(o) = make_float4(a[0], a[1], a[2], a[3]);
            *reinterpret_cast<float4*>(o + 4) = make_float4(a[4], a[5], a[6], a[7]);
        } else {
            *reinterpret_cast<uint4*>(static_cast<__nv_bfloat16*>(p.dH) + at + k0) =
                make_uint4(pack_bf16x2(a[0], a[1]), pack_bf16x2(a[2], a[3]), pack_bf16x2(a[4], a[5]), pack_bf16x2(a[6], a[7]));
        }
    });
}

}  // namespace hass

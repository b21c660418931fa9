// Leaky readout and cross-entropy of the classification network
// (Supplementary, "Classification"), and float -> bit packing of spike trains.
//
// The readout is an integrator without spike or reset whose membrane is
// summed over time:
//     V_o[t] = beta_o V_o[t-1] + (1 - beta_o) I_o[t],   o[b,c] = sum_t V_o[t],
//     I_o[b,c,t] = bias_c + sum_k W[c,k] S[b,k,t].
// Summing the impulse response over the remaining steps,
//     o[b,c] = sum_k W[c,k] n[b,k] + bias_c sum_t w_t,
//     n[b,k] = sum_t w_t S[b,k,t],   w_t = 1 - beta_o^(T-t),
// so the forward is a weighted count of each input row's spikes (event
// driven: only set bits are visited) followed by a [B,K] x [K,C] product.
// Backward: dL/dS[b,k,t] = w_t h[b,k] with h[b,k] = sum_c W[c,k] g_o[b,c];
// dL/dW[c,k] = sum_b g_o[b,c] n[b,k]; dL/dbias_c = sum_b g_o[b,c] sum_t w_t.
// All sums run in a fixed order (deterministic).
#include "common.cuh"

namespace alif {
namespace ro {

__device__ __forceinline__ float warp_sum(float x) {
#pragma unroll
    for (int off = 16; off; off >>= 1) x += __shfl_xor_sync(FULL, x, off);
    return x;
}

// Sum of w over the set bits of M words of a row, 32 apart from word q on, loaded together.
template <int M>
__device__ __forceinline__ float count_words(const uint32_t *__restrict__ row, long long q, long long T, long long nwords,
                                             const float *__restrict__ w, float acc) {
    uint32_t v[M];
#pragma unroll
    for (int m = 0; m < M; ++m) {
        v[m] = q + 32 * m < nwords ? __ldg(row + q + 32 * m) : 0u;
        if (q + 32 * m == nwords - 1 && (T & 31)) v[m] &= (1u << (T & 31)) - 1u;
    }
#pragma unroll
    for (int m = 0; m < M; ++m)
        while (v[m]) {
            const int i = __ffs(v[m]) - 1;
            v[m] &= v[m] - 1u;
            acc += __ldg(w + (q + 32 * m) * 32 + i);
        }
    return acc;
}

// n[r] = sum_t w[t] S[r,t] of one row: lanes over its words, four at a time where there are more than 32.
__device__ __forceinline__ float count_row(const uint32_t *__restrict__ row, long long T, long long nwords,
                                           const float *__restrict__ w, int lane) {
    float acc = 0.0f;
    if (nwords <= 32)
        acc = count_words<1>(row, lane, T, nwords, w, acc);
    else
        for (long long q = lane; q < nwords; q += 128) acc = count_words<4>(row, q, T, nwords, w, acc);
    return warp_sum(acc);
}

// n[b,k]: a warp per row, over the whole grid.  Bound by the raster's latency: at 128 x 1024 rows of 16000 steps
// 220 us with one load of a word in flight per lane, 86 (with out_kernel) with four.
__global__ void __launch_bounds__(256) count_kernel(long long rows, long long T, long long nwords,
                                                    const uint32_t *__restrict__ S, const float *__restrict__ w, float *n) {
    const long long r = (long long)blockIdx.x * 8 + (threadIdx.x >> 5);
    if (r >= rows) return;
    const float acc = count_row(S + r * nwords, T, nwords, w, threadIdx.x & 31);
    if ((threadIdx.x & 31) == 0) n[r] = acc;
}

// o[b,c] = sum_k W[c,k] n[b,k] + bias_c w_sum: a warp per output, lanes over the inputs (a thread per output
// walked 1024 inputs in 35 us).  Counts and outputs in one launch, a block per batch element, measured no less
// anywhere and far more where a block's rows are many or long (us, this / that): 128 x 256 x 1000 steps 9.9 / 11,
// 1 x 256 x 1000 5.0 / 10, 32 x 1024 x 16000 28 / 117, 1 x 1024 x 16000 11 / 109.
__global__ void __launch_bounds__(256) out_kernel(long long BC, long long K, long long C, const float *__restrict__ W,
                                                  const float *__restrict__ bias, float w_sum,
                                                  const float *__restrict__ n, float *o) {
    const long long e = (long long)blockIdx.x * 8 + (threadIdx.x >> 5);
    const int lane = threadIdx.x & 31;
    if (e >= BC) return;
    const long long b = e / C, c = e - b * C;
    float acc = 0.0f;
    for (long long k = lane; k < K; k += 32) acc = fmaf(__ldg(W + c * K + k), __ldg(n + b * K + k), acc);
    acc = warp_sum(acc);
    if (lane == 0) o[e] = bias ? fmaf(bias[c], w_sum, acc) : acc;
}

// The same, a thread per output, for few inputs: the whole forward of 250 steps, 300 x 3 -> 75, 4.7 us and 7.0 with a
// warp each, 2000 x 16 -> 75 12 and 28; but 30 x 32 -> 20 7.2 and 4.7.
__global__ void __launch_bounds__(256) out_few_kernel(long long BC, long long K, long long C, const float *__restrict__ W,
                                                      const float *__restrict__ bias, float w_sum,
                                                      const float *__restrict__ n, float *o) {
    const long long e = (long long)blockIdx.x * 256 + threadIdx.x;
    if (e >= BC) return;
    const long long b = e / C, c = e - b * C;
    float acc = 0.0f;
    for (long long k = 0; k < K; ++k) acc = fmaf(W[c * K + k], n[b * K + k], acc);
    o[e] = bias ? fmaf(bias[c], w_sum, acc) : acc;
}

// dL/dS[r, t] = w[t] h[r], h[b,k] = sum_c W[c,k] g_o[b,c]: one warp per row r = (b, k) and steps t0 .. t1 - 1.
// Loads go out together, of h's chain (10 per step of the loop) and of w before the stores (which could alias it
// for all the compiler knows).
__device__ __forceinline__ void grad_spikes(long long r, long long t0, long long t1, int lane, long long K, long long C,
                                            long long T, const float *__restrict__ W, const float *__restrict__ g_o,
                                            const float *__restrict__ w, float *gS) {
    const long long b = r / K, k = r % K;
    float h = 0.0f;
#pragma unroll 10
    for (long long c = 0; c < C; ++c) h = fmaf(__ldg(W + c * K + k), __ldg(g_o + b * C + c), h);
    float *out = gS + r * T;
    if ((T & 3) == 0 && ((reinterpret_cast<uintptr_t>(gS) & 15u) == 0) &&
        ((reinterpret_cast<uintptr_t>(w) & 15u) == 0)) {
        constexpr int U = 4;
        for (long long t = t0 + 4 * lane; t < t1; t += 128 * U) {
            float4 v[U];
#pragma unroll
            for (int m = 0; m < U; ++m)
                if (t + 128 * m < t1) v[m] = __ldg(reinterpret_cast<const float4 *>(w + t + 128 * m));
#pragma unroll
            for (int m = 0; m < U; ++m)
                if (t + 128 * m < t1)
                    *reinterpret_cast<float4 *>(out + t + 128 * m) = make_float4(h * v[m].x, h * v[m].y, h * v[m].z, h * v[m].w);
        }
    } else {
        for (long long t = t0 + lane; t < t1; t += 32) out[t] = h * __ldg(w + t);
    }
}

// dL/dW[c,k] = sum_b g_o[b,c] n[b,k]; dL/dbias_c = sum_b g_o[b,c] w_sum: a thread per element e.
__device__ __forceinline__ void grad_w(long long e, long long B, long long K, long long C,
                                       const float *__restrict__ g_o, const float *__restrict__ n, float w_sum,
                                       float *gW, float *gb) {
    if (e < C * K && gW) {
        const long long c = e / K, k = e % K;
        float acc = 0.0f;
#pragma unroll 16
        for (long long b = 0; b < B; ++b) acc = fmaf(__ldg(g_o + b * C + c), __ldg(n + b * K + k), acc);
        gW[e] = acc;
    }
    if (e < C && gb) {
        float acc = 0.0f;
#pragma unroll 16
        for (long long b = 0; b < B; ++b) acc += __ldg(g_o + b * C + e);
        gb[e] = acc * w_sum;
    }
}

constexpr long long WARPS = 32 * 152;  // that fill the chip with writes

// Both gradients in one launch: the first nw blocks take grad_w's elements (a serial sum over the batch,
// hidden behind the writes of the others), the rest grad_spikes' rows in `parts` parts of `len` steps.  Bound by the
// writes of dL/dS: at B = 128, K = 256, C = 20, T = 1000 (131 MB) 24 us, as two kernels, with a load at a time,
// 55; at 128 x 1024 x 16000 1.13 ms and 1.17.
__global__ void __launch_bounds__(256, 4) backward_kernel(unsigned nw, long long B, long long K, long long C, long long T,
                                long long parts, long long len, const float *__restrict__ W,
                                const float *__restrict__ g_o, const float *__restrict__ w,
                                const float *__restrict__ n, float w_sum, float *gS, float *gW, float *gb) {
    if (blockIdx.x < nw) {
        grad_w((long long)blockIdx.x * blockDim.x + threadIdx.x, B, K, C, g_o, n, w_sum, gW, gb);
    } else {
        long long r = (long long)(blockIdx.x - nw) * (blockDim.x >> 5) + (threadIdx.x >> 5), t0 = 0;
        if (parts > 1) {
            const long long q = r / parts;
            t0 = (r - q * parts) * len;
            r = q;
        }
        const long long t1 = t0 + len < T ? t0 + len : T;
        if (r < B * K && t0 < T) grad_spikes(r, t0, t1, threadIdx.x & 31, K, C, T, W, g_o, w, gS);
    }
}

// Mean softmax cross-entropy: one block, a warp per row (a thread per row took 14 us at B = 128, C = 20,
// now 10.5); the losses are summed in double, lanes over the rows, then a fixed tree.
__global__ void ce_kernel(long long B, long long C, const float *__restrict__ o, const int32_t *__restrict__ y,
                          float *loss, float *g_o, float *row_loss) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarp = blockDim.x >> 5;
    for (long long b = warp; b < B; b += nwarp) {
        const float *ob = o + b * C;
        float m = ob[0];
        for (long long c = lane; c < C; c += 32) m = fmaxf(m, ob[c]);
#pragma unroll
        for (int off = 16; off; off >>= 1) m = fmaxf(m, __shfl_xor_sync(FULL, m, off));
        float s = 0.0f;
        for (long long c = lane; c < C; c += 32) s += expf(ob[c] - m);
        s = warp_sum(s);
        const int lab = y[b];
        const bool ok = lab >= 0 && lab < C;  // an invalid label gives a NaN loss, no access
        if (lane == 0) row_loss[b] = ok ? -(ob[lab] - m - logf(s)) : __int_as_float(0x7fc00000);
        if (g_o) {
            const float inv = 1.0f / ((float)B * s);
            for (long long c = lane; c < C; c += 32)
                g_o[b * C + c] = expf(ob[c] - m) * inv - (c == lab ? 1.0f / (float)B : 0.0f);
        }
    }
    __syncthreads();
    if (warp == 0) {
        double acc = 0.0;
        for (long long b = lane; b < B; b += 32) acc += (double)row_loss[b];
#pragma unroll
        for (int off = 16; off; off >>= 1) acc += __shfl_xor_sync(FULL, acc, off);
        if (lane == 0) *loss = (float)(acc / (double)B);
    }
}

// words[r, q] bit i = (S[r, 32 q + i] != 0): one warp per row, ballot per 32 steps.
__global__ void pack_kernel(long long rows, long long T, long long nwords, const float *__restrict__ S,
                            uint32_t *words) {
    const long long r = (long long)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    const int lane = threadIdx.x & 31;
    if (r >= rows) return;
    for (long long q = 0; q < nwords; ++q) {
        const long long t = q * 32 + lane;
        const bool on = t < T && S[r * T + t] != 0.0f;
        const uint32_t word = __ballot_sync(FULL, on);
        if (lane == 0) words[r * nwords + q] = word;
    }
}

}  // namespace ro

int launch_readout_forward(long long B, long long K, long long C, long long T, const uint32_t *S, const float *W,
                           const float *bias, const float *w, float w_sum, float *n, float *o, cudaStream_t st) {
    const long long rows = B * K;
    if (rows > 0) {
        ro::count_kernel<<<(unsigned)((rows + 7) / 8), 256, 0, st>>>(rows, T, (T + 31) / 32, S, w, n);
        const cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return (int)e;
    }
    if (B * C > 0) {
        if (K <= 12 || (K <= 24 && B * C >= 10000))
            ro::out_few_kernel<<<(unsigned)((B * C + 255) / 256), 256, 0, st>>>(B * C, K, C, W, bias, w_sum, n, o);
        else
            ro::out_kernel<<<(unsigned)((B * C + 7) / 8), 256, 0, st>>>(B * C, K, C, W, bias, w_sum, n, o);
        return (int)cudaGetLastError();
    }
    return 0;
}

int launch_readout_backward(long long B, long long K, long long C, long long T, const float *W, const float *w,
                            float w_sum, const float *n, const float *g_o, float *gS, float *gW, float *gb,
                            cudaStream_t st) {
    const long long m = gW && C * K > C ? C * K : C;
    const unsigned nw = (gW || gb) && m > 0 ? (unsigned)((m + 255) / 256) : 0;
    const long long rows = gS && T > 0 ? B * K : 0;
    // few rows are cut into parts of at least 512 steps, so that some 32 warps per SM write (1 x 1024 x 16000:
    // 13 us, 22 with a warp per row)
    long long parts = 1, len = T;
    if (rows > 0 && rows < ro::WARPS) {
        parts = ro::WARPS / rows < (T + 511) / 512 ? ro::WARPS / rows : (T + 511) / 512;
        len = ((T + parts - 1) / parts + 127) / 128 * 128;
    }
    const unsigned ns = (unsigned)((rows * parts + 7) / 8);
    if (nw + ns == 0) return 0;
    ro::backward_kernel<<<nw + ns, 256, 0, st>>>(nw, B, K, C, T, parts, len, W, g_o, w, n, w_sum, gS, gW, gb);
    return (int)cudaGetLastError();
}

int launch_cross_entropy(long long B, long long C, const float *o, const int32_t *y, float *loss, float *g_o,
                         float *row_loss, cudaStream_t st) {
    ro::ce_kernel<<<1, 1024, 0, st>>>(B, C, o, y, loss, g_o, row_loss);
    return (int)cudaGetLastError();
}

int launch_pack_spikes(long long rows, long long T, const float *S, uint32_t *words, cudaStream_t st) {
    if (rows <= 0 || T <= 0) return 0;
    ro::pack_kernel<<<(unsigned)((rows + 7) / 8), 256, 0, st>>>(rows, T, (T + 31) / 32, S, words);
    return (int)cudaGetLastError();
}

}  // namespace alif

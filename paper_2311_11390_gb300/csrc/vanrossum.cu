// van Rossum distance between spike trains (Supplementary, "Neural fits"),
// the loss of the neuron-fitting requests, and its gradient with respect to the
// model's spike train.  Discretised with the exponential kernel
// k[t] = exp(-t DT / tau_R):
//     f[t] = decay f[t-1] + (x[t] - y[t]),      decay = exp(-DT / tau_R)
//     L    = (DT / tau_R) sum_t f[t]^2           (the squared distance D_R^2)
//     dL/dx[t] = (2 DT / tau_R) g[t],  g[t] = f[t] + decay g[t+1]
// Both recurrences are linear in known spikes, so a row's time is spread over a whole CTA: one
// thread per 32-step spike word, TH <= 512 words per tile, a row's tiles in order (f) or in
// reverse (g).  A thread forms its word's contribution from a zero start, a decayed scan over the
// CTA (shuffles, then one shared value per warp) gives the value entering its word, and the 32
// steps follow from it.  Inside a word every value is an 8-step chain from a zero start plus an
// exact power times the value entering those 8 steps, so a rounded decay is never compounded over
// more than 8 steps.
// What bounds it: the gradient's writes (4 B per step; the bits are 1/16 of that), with about 15
// thread instructions per step behind them.  A warp per row walking 256-step windows, as before,
// left 1024 rows x 400000 steps to 1024 warps that each waited for two spike words per window:
// forward 0.92 ms and gradient 2.05 ms.
#include "common.cuh"

namespace alif {
namespace vr {

constexpr int E = 8, SUB = 4, WORD = 32;  // a word is SUB chains of E steps
constexpr int TH_MAX = 512;               // words per tile
constexpr long long MAX_ROWS = 1 << 30;   // rows (CTAs) per launch
constexpr int MAX_TILES = (1 << 19) / WORD / TH_MAX;  // tiles of the longest gradient call

// Powers of the decay, each rounded once from double-single.
struct Tables {
    float pw[E + 1];      // dec^k, k = 0 .. 8
    float b32[5];         // dec^(32 2^l): lane distances
    float b1k[4], d1k;    // dec^(1024 2^l): warp distances; dec^1024
    float lup, ldn;       // dec^(32 lane), dec^(32 (31 - lane))
};

__device__ __forceinline__ Tables make_tables(double dec, int lane) {
    Tables tb;
    const df d{(float)dec, (float)(dec - (double)(float)dec)};
    df u{1.0f, 0.0f};
#pragma unroll
    for (int k = 0; k <= E; ++k) {
        tb.pw[k] = u.hi;
        if (k < E) u = df_mul(u, d);
    }
    u = df_mul(u, u);
    u = df_mul(u, u);  // dec^32
    const df d32 = u;
#pragma unroll
    for (int l = 0; l < 5; ++l) {
        tb.b32[l] = u.hi;
        u = df_mul(u, u);
    }
    tb.d1k = u.hi;
#pragma unroll
    for (int l = 0; l < 4; ++l) {
        tb.b1k[l] = u.hi;
        u = df_mul(u, u);
    }
    tb.lup = df_pow(d32, lane).hi;
    tb.ldn = df_pow(d32, 31 - lane).hi;
    return tb;
}

// Value entering this thread's word from the words before it (REV: after it) in the tile and from
// `carry`, the value entering the tile; e: this word's contribution from a zero start.  *leave: the
// value leaving the tile.  ws: 2 x 16 floats, alternating between calls (one barrier per call: a
// warp writes a half again only after every warp has passed the barrier of the call in between).
template <bool REV>
__device__ __forceinline__ float tile_scan(float e, float carry, const Tables &tb, float *ws, int lane, int warp,
                                           int nw, float *leave) {
    float incl = e;
#pragma unroll
    for (int l = 0; l < 5; ++l)
        incl = REV ? down_fma(incl, tb.b32[l], 1u << l, incl) : up_fma(incl, tb.b32[l], 1u << l, incl);
    float excl = REV ? __shfl_down_sync(FULL, incl, 1) : __shfl_up_sync(FULL, incl, 1);
    if (lane == (REV ? 31 : 0)) excl = 0.0f;
    const int wpos = REV ? nw - 1 - warp : warp;  // this warp's place in the order of the scan
    if (lane == (REV ? 0 : 31)) ws[wpos] = incl;
    __syncthreads();
    float wv = lane < nw ? ws[lane] : 0.0f;
    if (lane == 0) wv = fmaf(tb.d1k, carry, wv);
#pragma unroll
    for (int l = 0; l < 4; ++l) wv = up_fma(wv, tb.b1k[l], 1u << l, wv);
    float in = __shfl_sync(FULL, wv, wpos > 0 ? wpos - 1 : 0);
    if (wpos == 0) in = carry;
    *leave = __shfl_sync(FULL, wv, nw - 1);
    return fmaf(REV ? tb.ldn : tb.lup, in, excl);
}

// f of a word's 32 steps from a zero start at each 8-step chain (loc) and the chains' ends joined:
// the word's contribution to its end.
__device__ __forceinline__ float word_local(uint32_t xw, uint32_t yw, const Tables &tb, float (&loc)[WORD]) {
    float end = 0.0f;
#pragma unroll
    for (int j = 0; j < SUB; ++j) {
        float f = 0.0f;
#pragma unroll
        for (int k = 0; k < E; ++k) {
            const int s = E * j + k;
            const float dv = ((xw >> s) & 1u ? 1.0f : 0.0f) - ((yw >> s) & 1u ? 1.0f : 0.0f);
            f = fmaf(tb.pw[1], f, dv);
            loc[s] = f;
        }
        end = fmaf(tb.pw[E], end, f);
    }
    return end;
}

// The word's f values from the value entering it.
__device__ __forceinline__ void word_apply(float fin, const Tables &tb, float (&f)[WORD]) {
    float s = fin;
#pragma unroll
    for (int j = 0; j < SUB; ++j) {
        const float next = fmaf(tb.pw[E], s, f[E * j + E - 1]);
#pragma unroll
        for (int k = 0; k < E; ++k) f[E * j + k] = fmaf(tb.pw[k + 1], s, f[E * j + k]);
        s = next;
    }
}

__device__ __forceinline__ uint32_t below(long long n) {  // mask of the bits < n
    return n >= 32 ? ~0u : n <= 0 ? 0u : (1u << n) - 1u;
}

// Forward filter: loss[r] (double-single summed) and f entering each chunk.
__global__ void __launch_bounds__(TH_MAX, 2) vr_forward_kernel(long long T, const uint32_t *__restrict__ x,
                                                            const uint32_t *__restrict__ y, double dec, double scale,
                                                            long long chunk, long long nchunk, float *f_ckpt,
                                                            float *loss) {
    __shared__ float ws[2][16];
    __shared__ df sums[16];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nw = blockDim.x >> 5;
    const long long r = blockIdx.x;
    const Tables tb = make_tables(dec, lane);
    const long long nwords = (T + 31) / 32;
    const uint32_t *xb = x + r * nwords, *yb = y + r * nwords;
    const long long ntile = (nwords + blockDim.x - 1) / blockDim.x;
    float carry = 0.0f;
    df acc{0.0f, 0.0f};
    uint32_t xn = tid < nwords ? __ldg(xb + tid) : 0u, yn = tid < nwords ? __ldg(yb + tid) : 0u;
    for (long long i = 0; i < ntile; ++i) {
        const long long q = i * blockDim.x + tid;
        const uint32_t valid = below(T - 32 * q), xw = xn & valid, yw = yn & valid;
        const long long qn = q + blockDim.x;
        xn = qn < nwords ? __ldg(xb + qn) : 0u;  // the next tile's words, in flight during this one
        yn = qn < nwords ? __ldg(yb + qn) : 0u;
        float f[WORD];
        const float e = word_local(xw, yw, tb, f);
        const float fin = tile_scan<false>(e, carry, tb, ws[i & 1], lane, warp, nw, &carry);
        if (f_ckpt && q < nwords && (32 * q) % chunk == 0) f_ckpt[r * nchunk + 32 * q / chunk] = fin;
        word_apply(fin, tb, f);
        float s[SUB];
#pragma unroll
        for (int j = 0; j < SUB; ++j) {
            s[j] = 0.0f;
#pragma unroll
            for (int k = 0; k < E; ++k)
                if ((valid >> (E * j + k)) & 1u) s[j] = fmaf(f[E * j + k], f[E * j + k], s[j]);
        }
        acc = df_add(acc, df{(s[0] + s[1]) + (s[2] + s[3]), 0.0f});
    }
#pragma unroll
    for (int off = 16; off; off >>= 1) {
        const df o{__shfl_xor_sync(FULL, acc.hi, off), __shfl_xor_sync(FULL, acc.lo, off)};
        acc = df_add(acc, o);
    }
    if (lane == 0) sums[warp] = acc;
    __syncthreads();
    if (tid == 0 && loss) {
        for (int w = 1; w < nw; ++w) acc = df_add(acc, sums[w]);
        loss[r] = (float)(scale * ((double)acc.hi + (double)acc.lo));
    }
}

// Gradient for steps [t0, t1) (t0 a multiple of 256 and of the chunk start):
// grad[r, t - t0] = (2 DT / tau_R) g[t], g carried from t1 in g_carry (updated).
// VEC: floats per store (8 where grad rows keep 32 bytes: whole sectors from each lane).
template <int VEC>
__global__ void __launch_bounds__(TH_MAX, 2) vr_backward_kernel(long long nwords, const uint32_t *__restrict__ x,
                                                             const uint32_t *__restrict__ y, double dec, float gscale,
                                                             long long t0, long long t1,
                                                             const float *__restrict__ f_start, float *g_carry,
                                                             float *grad, long long ldg) {
    __shared__ float ws[2][16];
    __shared__ float ftile[MAX_TILES];  // f entering each tile
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nw = blockDim.x >> 5, th = blockDim.x;
    const long long r = blockIdx.x;
    const Tables tb = make_tables(dec, lane);
    const uint32_t *xb = x + r * nwords + (t0 >> 5), *yb = y + r * nwords + (t0 >> 5);
    const int steps = (int)(t1 - t0), nq = (steps + 31) / 32, ntile = (nq + th - 1) / th;
    int par = 0;
    float carry = f_start[r];
    for (int i = 0; i < ntile; ++i) {
        if (tid == 0) ftile[i] = carry;
        if (i + 1 == ntile) break;
        const int q = i * th + tid;  // every tile but the last is full
        const uint32_t xw = __ldg(xb + q), yw = __ldg(yb + q);
        float e = 0.0f;
        if (xw != yw) {
            float f[WORD];
            e = word_local(xw, yw, tb, f);
        }
        tile_scan<false>(e, carry, tb, ws[par], lane, warp, nw, &carry);
        par ^= 1;
    }
    __syncthreads();
    const float gc = g_carry[r];
    float gin_tile = 0.0f;
    for (int i = ntile - 1; i >= 0; --i) {
        const int q = i * th + tid, cnt = steps - 32 * q;  // steps of this word (may be <= 0)
        const uint32_t valid = below(cnt);
        const uint32_t xw = q < nq ? __ldg(xb + q) & valid : 0u, yw = q < nq ? __ldg(yb + q) & valid : 0u;
        float f[WORD], unused;
        const float e = word_local(xw, yw, tb, f);
        const float fin = tile_scan<false>(e, ftile[i], tb, ws[par], lane, warp, nw, &unused);
        par ^= 1;
        word_apply(fin, tb, f);
        // the word that holds step t1 - 1 takes the carry of step t1 there; nothing passes through
        // it from later words
        const bool last = q == nq - 1;
        if (last || valid != ~0u) {
            const float inject = last ? tb.pw[1] * gc : 0.0f;
#pragma unroll
            for (int k = 0; k < WORD; ++k)
                f[k] = ((valid >> k) & 1u ? f[k] : 0.0f) + ((valid >> k) == 1u ? inject : 0.0f);
        }
        // 8-step reverse chains from a zero start, joined
        float ge = 0.0f;
#pragma unroll
        for (int j = SUB - 1; j >= 0; --j) {
#pragma unroll
            for (int k = E - 2; k >= 0; --k) f[E * j + k] = fmaf(tb.pw[1], f[E * j + k + 1], f[E * j + k]);
            ge = fmaf(tb.pw[E], ge, f[E * j]);
        }
        float s = tile_scan<true>(ge, gin_tile, tb, ws[par], lane, warp, nw, &gin_tile);
        par ^= 1;
        if (last) s = 0.0f;
#pragma unroll
        for (int j = SUB - 1; j >= 0; --j) {
            const float next = fmaf(tb.pw[E], s, f[E * j]);
#pragma unroll
            for (int k = 0; k < E; ++k) f[E * j + k] = fmaf(tb.pw[E - k], s, f[E * j + k]);
            s = next;
        }
        if (q == 0) g_carry[r] = f[0];
        float *go = grad + r * ldg + 32LL * q;
        if (VEC > 1 && cnt >= WORD) {
#pragma unroll
            for (int k = 0; k < WORD; k += 8) {
                if (VEC == 8) {
                    asm volatile("st.global.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(go + k),
                                 "f"(gscale * f[k]), "f"(gscale * f[k + 1]), "f"(gscale * f[k + 2]),
                                 "f"(gscale * f[k + 3]), "f"(gscale * f[k + 4]), "f"(gscale * f[k + 5]),
                                 "f"(gscale * f[k + 6]), "f"(gscale * f[k + 7])
                                 : "memory");
                } else {
#pragma unroll
                    for (int m = k; m < k + 8; m += 4)
                        *reinterpret_cast<float4 *>(go + m) = make_float4(
                            gscale * f[m], gscale * f[m + 1], gscale * f[m + 2], gscale * f[m + 3]);
                }
            }
        } else {
#pragma unroll
            for (int k = 0; k < WORD; ++k)
                if (k < cnt) go[k] = gscale * f[k];
        }
    }
}

// One CTA per row: as many threads as words, whole warps, TH_MAX at most (a longer row loops).
inline unsigned threads_for(long long words) {
    const long long t = (words + 31) / 32 * 32;
    return (unsigned)(t < 32 ? 32 : t > TH_MAX ? TH_MAX : t);
}

}  // namespace vr

int launch_vr_forward(long long rows, long long T, const uint32_t *x, const uint32_t *y, double dec, double scale,
                      long long chunk, float *f_ckpt, float *loss, cudaStream_t st) {
    const long long nchunk = (T + chunk - 1) / chunk, nwords = (T + 31) / 32;
    for (long long r = 0; r < rows; r += vr::MAX_ROWS) {
        const unsigned n = (unsigned)(rows - r < vr::MAX_ROWS ? rows - r : vr::MAX_ROWS);
        vr::vr_forward_kernel<<<n, vr::threads_for(nwords), 0, st>>>(T, x + r * nwords, y + r * nwords, dec, scale,
                                                                    chunk, nchunk, f_ckpt ? f_ckpt + r * nchunk : nullptr,
                                                                    loss ? loss + r : nullptr);
        const cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return (int)e;
    }
    return 0;
}

int launch_vr_backward(long long rows, long long T, const uint32_t *x, const uint32_t *y, double dec, float gscale,
                       long long t0, long long t1, const float *f_start, float *g_carry, float *grad, long long ldg,
                       cudaStream_t st) {
    const long long nwords = (T + 31) / 32;
    const unsigned th = vr::threads_for((t1 - t0 + 31) / 32);
    const uintptr_t ga = reinterpret_cast<uintptr_t>(grad);
    const auto kernel = (ldg % 8 == 0 && ga % 32 == 0)   ? vr::vr_backward_kernel<8>
                        : (ldg % 4 == 0 && ga % 16 == 0) ? vr::vr_backward_kernel<4>
                                                         : vr::vr_backward_kernel<1>;
    for (long long r = 0; r < rows; r += vr::MAX_ROWS) {
        const unsigned n = (unsigned)(rows - r < vr::MAX_ROWS ? rows - r : vr::MAX_ROWS);
        kernel<<<n, th, 0, st>>>(nwords, x + r * nwords, y + r * nwords, dec, gscale, t0, t1, f_start + r, g_carry + r,
                                 grad + r * ldg, ldg);
        const cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return (int)e;
    }
    return 0;
}

}  // namespace alif

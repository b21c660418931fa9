// van Rossum distance between spike trains (Supplementary, "Neural fits"),
// the loss of the neuron-fitting requests, and its gradient with respect to the
// model's spike train.  Discretised with the exponential kernel
// k[t] = exp(-t DT / tau_R):
//     f[t] = decay f[t-1] + (x[t] - y[t]),      decay = exp(-DT / tau_R)
//     L    = (DT / tau_R) sum_t f[t]^2           (the squared distance D_R^2)
//     dL/dx[t] = (2 DT / tau_R) g[t],  g[t] = f[t] + decay g[t+1]
// Both recurrences are linear in known spikes, so a row's time is spread over a warp or, where rows are
// few, a whole CTA: one thread per 32-step spike word, 32 or TH <= 512 words per tile, a row's tiles in
// order (f) or in reverse (g).  A thread forms its word's contribution from a zero start, a decayed scan over the
// CTA (shuffles, then one shared value per warp) gives the value entering its word, and the 32
// steps follow from it.  Inside a word every value is an 8-step chain from a zero start plus an
// exact power times the value entering those 8 steps, so a rounded decay is never compounded over
// more than 8 steps.
// What bounds it: the gradient's writes (4 B per step, 0.24 ms for 1024 rows x 400000 steps; the
// bits are 1/16 of that) and the instructions of the word's chains and scans between the barriers.
// At that size: forward 0.19 ms, gradient 0.46 ms.  A warp per row walking 256-step windows left it
// to 1024 warps that each waited for two spike words per window: 0.92 and 2.05 ms.
#include "common.cuh"

namespace alif {
namespace vr {

constexpr int E = 8, SUB = 4, WORD = 32;  // a word is SUB chains of E steps
constexpr int LDS_ROW = WORD + 4;             // floats per staged word: 16-byte rows, no bank conflicts
constexpr int TH_MAX = 512;               // words per tile
constexpr long long MAX_ROWS = 1 << 30;   // rows (CTAs) per launch
constexpr int MAX_TILES = (1 << 19) / WORD / TH_MAX;  // tiles of the longest gradient call
constexpr int RW = 8, RTILES = 32;        // warps of a CTA with a row each, tiles of 32 words of its longest row
constexpr int FWD_CTAS = 4, BWD_CTAS = 3;                // of these per SM

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
    df up{1.0f, 0.0f}, dn{1.0f, 0.0f};
#pragma unroll
    for (int l = 0; l < 5; ++l) {  // u = dec^(32 2^l)
        tb.b32[l] = u.hi;
        const df mu = df_mul(up, u), md = df_mul(dn, u);
        if ((lane >> l) & 1)
            up = mu;
        else
            dn = md;
        u = df_mul(u, u);
    }
    tb.lup = up.hi;
    tb.ldn = dn.hi;
    tb.d1k = u.hi;
#pragma unroll
    for (int l = 0; l < 4; ++l) {
        tb.b1k[l] = u.hi;
        u = df_mul(u, u);
    }
    return tb;
}

// Value entering this thread's word from the words before it (REV: after it) in the tile and from
// `carry`, the value entering the tile; e: this word's contribution from a zero start.  *leave: the
// value leaving the tile.  ws: 2 x 16 floats, alternating between calls (one barrier per call: a
// warp writes a half again only after every warp has passed the barrier of the call in between).
// ONE: the tile is the warp's 32 words.
template <bool REV, bool ONE>
__device__ __forceinline__ float tile_scan(float e, float carry, const Tables &tb, float *ws, int lane, int warp,
                                           int nw, float *leave) {
    float incl = e;
#pragma unroll
    for (int l = 0; l < 5; ++l)
        incl = REV ? down_fma(incl, tb.b32[l], 1u << l, incl) : up_fma(incl, tb.b32[l], 1u << l, incl);
    float excl = REV ? __shfl_down_sync(FULL, incl, 1) : __shfl_up_sync(FULL, incl, 1);
    if (lane == (REV ? 31 : 0)) excl = 0.0f;
    if (ONE) {
        *leave = fmaf(tb.d1k, carry, __shfl_sync(FULL, incl, REV ? 0 : 31));
        return fmaf(REV ? tb.ldn : tb.lup, carry, excl);
    }
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

// lut[m]: the 8 values of f after the spikes in the bits of byte m, from a zero start.  The
// filter is linear, so a word's chains are two look-ups per 8 steps (x without y, y without x;
// mostly entry 0, a broadcast) and a packed subtraction, against 7 instructions per step to turn
// each pair of bits into +-1 and carry it.
struct __align__(16) Chain {
    float2 v[E / 2];
};

__device__ __forceinline__ void make_lut(Chain *lut, const Tables &tb) {
    for (int m = threadIdx.x; m < 256; m += blockDim.x) {
        float f[E];
#pragma unroll
        for (int k = 0; k < E; ++k) f[k] = fmaf(tb.pw[1], k ? f[k - 1] : 0.0f, (m >> k) & 1 ? 1.0f : 0.0f);
#pragma unroll
        for (int k = 0; k < E; k += 4) *reinterpret_cast<float4 *>(&lut[m].v[k / 2]) = make_float4(f[k], f[k + 1], f[k + 2], f[k + 3]);
    }
    __syncthreads();
}

// f of a word's 32 steps from a zero start at each 8-step chain; returns the chains' ends joined:
// the word's contribution to its end.
__device__ __forceinline__ float word_local(uint32_t xw, uint32_t yw, const Tables &tb, const Chain *lut,
                                            float2 (&f)[WORD / 2]) {
    const uint32_t up = xw & ~yw, dn = yw & ~xw;
    float end = 0.0f;
#pragma unroll
    for (int j = 0; j < SUB; ++j) {
        const Chain a = lut[(up >> (8 * j)) & 255u], b = lut[(dn >> (8 * j)) & 255u];
#pragma unroll
        for (int k = 0; k < E / 2; ++k) f[E / 2 * j + k] = __ffma2_rn(make_float2(-1.0f, -1.0f), b.v[k], a.v[k]);
        end = fmaf(tb.pw[E], end, f[E / 2 * j + E / 2 - 1].y);
    }
    return end;
}

// The word's f values from the value entering it.
__device__ __forceinline__ void word_apply(float fin, const Tables &tb, float2 (&f)[WORD / 2]) {
    float s = fin;
#pragma unroll
    for (int j = 0; j < SUB; ++j) {
        const float next = fmaf(tb.pw[E], s, f[E / 2 * j + E / 2 - 1].y);
#pragma unroll
        for (int k = 0; k < E / 2; ++k) {
            float2 &v = f[E / 2 * j + k];
            v = __ffma2_rn(make_float2(tb.pw[2 * k + 1], tb.pw[2 * k + 2]), make_float2(s, s), v);
        }
        s = next;
    }
}

__device__ __forceinline__ uint32_t below(long long n) {  // mask of the bits < n
    return n >= 32 ? ~0u : n <= 0 ? 0u : (1u << n) - 1u;
}

// Forward filter: loss[r] (double-single summed) and f entering each chunk.  ROWS: a warp per row, RW rows per
// CTA at a time (see rows_by_warps).
template <bool ROWS>
__global__ void __launch_bounds__(ROWS ? RW * 32 : TH_MAX, ROWS ? FWD_CTAS : 2)
    vr_forward_kernel(long long rows, long long T, const uint32_t *__restrict__ x, const uint32_t *__restrict__ y,
                      double dec, double scale, long long chunk, long long nchunk, float *f_ckpt, float *loss) {
    __shared__ Chain lut[256];
    __shared__ float ws[2][16];
    __shared__ df sums[16];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const int tid = ROWS ? lane : threadIdx.x, th = ROWS ? 32 : blockDim.x;
    const long long nwords = (T + 31) / 32, ntile = (nwords + th - 1) / th;
    const long long r0 = ROWS ? (long long)blockIdx.x * RW + warp : blockIdx.x, dr = ROWS ? (long long)gridDim.x * RW : rows;
    // the words of the next tile (or row) are in flight during this one
    uint32_t xn = r0 < rows && tid < nwords ? __ldg(x + r0 * nwords + tid) : 0u;
    uint32_t yn = r0 < rows && tid < nwords ? __ldg(y + r0 * nwords + tid) : 0u;
    const Tables tb = make_tables(dec, lane);
    make_lut(lut, tb);
    for (long long r = r0; r < rows; r += dr) {
        const uint32_t *xb = x + r * nwords, *yb = y + r * nwords;
        float carry = 0.0f;
        df acc{0.0f, 0.0f};
        for (long long i = 0; i < ntile; ++i) {
            const long long q = i * th + tid;
            const uint32_t valid = below(T - 32 * q), xw = xn & valid, yw = yn & valid;
            if (!ROWS || i + 1 < ntile) {
                xn = q + th < nwords ? __ldg(xb + q + th) : 0u;
                yn = q + th < nwords ? __ldg(yb + q + th) : 0u;
            } else {
                xn = r + dr < rows && tid < nwords ? __ldg(xb + dr * nwords + tid) : 0u;
                yn = r + dr < rows && tid < nwords ? __ldg(yb + dr * nwords + tid) : 0u;
            }
            float2 f[WORD / 2];
            const float e = word_local(xw, yw, tb, lut, f);
            const float fin = tile_scan<false, ROWS>(e, carry, tb, ws[i & 1], lane, warp, nw, &carry);
            if (f_ckpt && q < nwords && (32 * q) % chunk == 0) f_ckpt[r * nchunk + 32 * q / chunk] = fin;
            word_apply(fin, tb, f);
            float2 s[2] = {};
            if (valid != ~0u) {
#pragma unroll
                for (int k = 0; k < WORD / 2; ++k) {
                    f[k].x = (valid >> (2 * k)) & 1u ? f[k].x : 0.0f;
                    f[k].y = (valid >> (2 * k + 1)) & 1u ? f[k].y : 0.0f;
                }
            }
#pragma unroll
            for (int k = 0; k < WORD / 2; ++k) s[k & 1] = __ffma2_rn(f[k], f[k], s[k & 1]);
            // FP32 sums of 8 squares, joined without rounding
            const df u = two_sum(s[0].x, s[0].y), v = two_sum(s[1].x, s[1].y), w = two_sum(u.hi, v.hi);
            acc = df_add(acc, quick_two_sum(w.hi, (u.lo + v.lo) + w.lo));
        }
#pragma unroll
        for (int off = 16; off; off >>= 1) {
            const df o{__shfl_xor_sync(FULL, acc.hi, off), __shfl_xor_sync(FULL, acc.lo, off)};
            acc = df_add(acc, o);
        }
        if (!ROWS) {
            if (lane == 0) sums[warp] = acc;
            __syncthreads();
            if (tid == 0)
                for (int w = 1; w < nw; ++w) acc = df_add(acc, sums[w]);
        }
        if (tid == 0 && loss) loss[r] = (float)(scale * ((double)acc.hi + (double)acc.lo));
    }
}

// Gradient for steps [t0, t1) (t0 a multiple of 256 and of the chunk start):
// grad[r, t - t0] = (2 DT / tau_R) g[t], g carried from t1 in g_carry (updated).
// A warp passes its words through shared memory and writes whole lines (0.50 ms at 1024 x 400000; 0.59 with
// each lane storing its own 128 bytes; 0.44 with the words loaded a tile ahead).  VEC: gradient rows keep 16
// bytes.  ROWS: as in the forward.
template <bool VEC, bool ROWS>
__global__ void __launch_bounds__(ROWS ? RW * 32 : TH_MAX, ROWS ? BWD_CTAS : 2)
    vr_backward_kernel(long long rows, long long nwords, const uint32_t *__restrict__ x, const uint32_t *__restrict__ y,
                       double dec, float gscale, long long t0, long long t1, const float *__restrict__ f_start,
                       float *g_carry, float *grad, long long ldg) {
    __shared__ Chain lut[256];
    __shared__ float ws[2][16];
    __shared__ float ftiles[ROWS ? RW * RTILES : MAX_TILES];  // f entering each tile
    extern __shared__ __align__(16) float stages[];  // [warps][32][LDS_ROW]
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const int tid = ROWS ? lane : threadIdx.x, th = ROWS ? 32 : blockDim.x;
    float *ftile = ftiles + (ROWS ? warp * RTILES : 0);
    float *stage = stages + warp * 32 * LDS_ROW;
    const int steps = (int)(t1 - t0), nq = (steps + 31) / 32, ntile = (nq + th - 1) / th;
    const long long r0 = ROWS ? (long long)blockIdx.x * RW + warp : blockIdx.x, dr = ROWS ? (long long)gridDim.x * RW : rows;
    x += t0 >> 5;
    y += t0 >> 5;
    // a tile's words are loaded while the tile (or row) before it in the loops is resolved
    uint32_t xn = r0 < rows && tid < nq ? __ldg(x + r0 * nwords + tid) : 0u;
    uint32_t yn = r0 < rows && tid < nq ? __ldg(y + r0 * nwords + tid) : 0u;
    const Tables tb = make_tables(dec, lane);
    make_lut(lut, tb);
    for (long long r = r0; r < rows; r += dr) {
        const uint32_t *xb = x + r * nwords, *yb = y + r * nwords;
        float carry = f_start[r];
        const float gc = g_carry[r];
        int par = 0;
        for (int i = 0; i < ntile; ++i) {
            if (tid == 0) ftile[i] = carry;
            if (i + 1 == ntile) break;  // xn, yn: the last tile's, where the reverse loop starts
            const int qn = (i + 1) * th + tid;  // every tile but the last is full
            const uint32_t xw = xn, yw = yn;
            xn = qn < nq ? __ldg(xb + qn) : 0u;
            yn = qn < nq ? __ldg(yb + qn) : 0u;
            float e = 0.0f;
            if (xw != yw) {
                float2 f[WORD / 2];
                e = word_local(xw, yw, tb, lut, f);
            }
            tile_scan<false, ROWS>(e, carry, tb, ws[par], lane, warp, nw, &carry);
            par ^= 1;
        }
        if (ROWS)
            __syncwarp();
        else
            __syncthreads();
        float gin_tile = 0.0f;
        for (int i = ntile - 1; i >= 0; --i) {
            const int q = i * th + tid, cnt = steps - 32 * q;  // steps of this word (may be <= 0)
            const uint32_t valid = below(cnt);
            const uint32_t xw = xn & valid, yw = yn & valid;
            if (i > 0) {
                xn = __ldg(xb + q - th);
                yn = __ldg(yb + q - th);
            } else if (ROWS) {
                xn = r + dr < rows && tid < nq ? __ldg(xb + dr * nwords + tid) : 0u;
                yn = r + dr < rows && tid < nq ? __ldg(yb + dr * nwords + tid) : 0u;
            }
            float2 f2[WORD / 2];
            float unused;
            const float e = word_local(xw, yw, tb, lut, f2);
            const float fin = tile_scan<false, ROWS>(e, ftile[i], tb, ws[par], lane, warp, nw, &unused);
            par ^= 1;
            word_apply(fin, tb, f2);
            float f[WORD];
#pragma unroll
            for (int k = 0; k < WORD / 2; ++k) {
                f[2 * k] = f2[k].x;
                f[2 * k + 1] = f2[k].y;
            }
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
            float s = tile_scan<true, ROWS>(ge, gin_tile, tb, ws[par], lane, warp, nw, &gin_tile);
            par ^= 1;
            if (last) s = 0.0f;
#pragma unroll
            for (int j = SUB - 1; j >= 0; --j) {
                const float next = fmaf(tb.pw[E], s, f[E * j]);
#pragma unroll
                for (int k = 0; k < E; k += 2) {
                    const float2 v = __fmul2_rn(
                        make_float2(gscale, gscale),
                        __ffma2_rn(make_float2(tb.pw[E - k], tb.pw[E - k - 1]), make_float2(s, s),
                                   make_float2(f[E * j + k], f[E * j + k + 1])));
                    f[E * j + k] = v.x;
                    f[E * j + k + 1] = v.y;
                }
                s = next;
                if (j == 0 && q == 0) g_carry[r] = next;
            }
            // the warp's 32 words, 4 KB: written line by line
#pragma unroll
            for (int k = 0; k < WORD; k += 4)
                *reinterpret_cast<float4 *>(stage + lane * LDS_ROW + k) = make_float4(f[k], f[k + 1], f[k + 2], f[k + 3]);
            __syncwarp();
            float *go = grad + r * ldg + 32LL * (q - lane);
            const int left = steps - 32 * (q - lane);  // steps from the warp's first word on
            if (VEC) {  // steps is a multiple of 4
#pragma unroll
                for (int k = 0; k < WORD / 4; ++k)
                    if (128 * k + 4 * lane < left)
                        *reinterpret_cast<float4 *>(go + 128 * k + 4 * lane) =
                            *reinterpret_cast<const float4 *>(stage + (4 * k + (lane >> 3)) * LDS_ROW + 4 * (lane & 7));
            } else {
#pragma unroll 8
                for (int k = 0; k < WORD; ++k)
                    if (32 * k + lane < left) go[32 * k + lane] = stage[k * LDS_ROW + lane];
            }
            __syncwarp();  // the stage, and after the last tile ftile, are written again
        }
    }
}

// One CTA per row: as many threads as words, whole warps, TH_MAX at most (a longer row loops).
inline unsigned threads_for(long long words) {
    const long long t = (words + 31) / 32 * 32;
    return (unsigned)(t < 32 ? 32 : t > TH_MAX ? TH_MAX : t);
}

// A warp per row where rows fill the chip, and where a row is one tile of a warp; a CTA per row needs fewer
// rows but builds its tables for each, and its scans wait at barriers.  us, warps / CTAs, forward and gradient: 512 rows
// of 4000 steps 6.5 / 6.1 and 9.8 / 7.3, 1024 of 4000 6.7 / 7.7 and 9.9 / 9.8, 4096 of 16384 30 / 72 and 80 / 109,
// 65536 of 1000 38 / 78 and 70 / 124 (and 85 and 133 for a warp per row with windows of 256 steps).
inline bool rows_by_warps(long long rows, long long words) {
    return words <= 32 || (rows >= 1024 && words <= 32 * RTILES);
}
inline unsigned row_ctas(long long rows, int per_sm) {
    const long long n = (rows + RW - 1) / RW, cap = per_sm * 152LL;
    return (unsigned)(n < cap ? n : cap);
}

}  // namespace vr

int launch_vr_forward(long long rows, long long T, const uint32_t *x, const uint32_t *y, double dec, double scale,
                      long long chunk, float *f_ckpt, float *loss, cudaStream_t st) {
    using namespace vr;
    const long long nchunk = (T + chunk - 1) / chunk, nwords = (T + 31) / 32;
    if (rows_by_warps(rows, nwords)) {
        vr_forward_kernel<true><<<row_ctas(rows, FWD_CTAS), RW * 32, 0, st>>>(rows, T, x, y, dec, scale, chunk, nchunk, f_ckpt, loss);
        return (int)cudaGetLastError();
    }
    for (long long r = 0; r < rows; r += MAX_ROWS) {
        const unsigned n = (unsigned)(rows - r < MAX_ROWS ? rows - r : MAX_ROWS);
        vr_forward_kernel<false><<<n, threads_for(nwords), 0, st>>>(n, T, x + r * nwords, y + r * nwords, dec, scale, chunk,
                                                                   nchunk, f_ckpt ? f_ckpt + r * nchunk : nullptr,
                                                                   loss ? loss + r : nullptr);
        const cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return (int)e;
    }
    return 0;
}

int launch_vr_backward(long long rows, long long T, const uint32_t *x, const uint32_t *y, double dec, float gscale,
                       long long t0, long long t1, const float *f_start, float *g_carry, float *grad, long long ldg,
                       cudaStream_t st) {
    using namespace vr;
    const long long nwords = (T + 31) / 32, words = (t1 - t0 + 31) / 32;
    const bool vec = ldg % 4 == 0 && (t1 - t0) % 4 == 0 && reinterpret_cast<uintptr_t>(grad) % 16 == 0;
    const bool by_warps = rows_by_warps(rows, words);
    const auto kernel = by_warps ? (vec ? vr_backward_kernel<true, true> : vr_backward_kernel<false, true>)
                                 : (vec ? vr_backward_kernel<true, false> : vr_backward_kernel<false, false>);
    const unsigned th = by_warps ? RW * 32 : threads_for(words);
    const size_t smem = (size_t)th * LDS_ROW * sizeof(float);
    if (smem > 32768) {
        const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return (int)e;
    }
    if (by_warps) {
        kernel<<<row_ctas(rows, BWD_CTAS), th, smem, st>>>(rows, nwords, x, y, dec, gscale, t0, t1, f_start, g_carry, grad, ldg);
        return (int)cudaGetLastError();
    }
    for (long long r = 0; r < rows; r += MAX_ROWS) {
        const unsigned n = (unsigned)(rows - r < MAX_ROWS ? rows - r : MAX_ROWS);
        kernel<<<n, th, smem, st>>>(n, nwords, x + r * nwords, y + r * nwords, dec, gscale, t0, t1, f_start + r, g_carry + r,
                                 grad + r * ldg, ldg);
        const cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return (int)e;
    }
    return 0;
}

}  // namespace alif

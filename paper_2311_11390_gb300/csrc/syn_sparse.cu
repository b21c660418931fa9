// Synaptic projection over sparse rasters (the feedforward term of Eq 3 / Prop 3):
//     I[b, i, t] = bias_i + sum_{j : S[b, j, t] = 1} W[i, j].
// Inputs at 10-50 Hz are active in 0.05-5 % of their steps, so almost all of the dense product is
// by zero.  Two kernels:
//   * lists_kernel turns the raster into event lists once: per (batch element, 32-step chunk) a
//     record of each step's active inputs, ascending.  256-step tiles with a chunk of more events than a record holds are put on a
//     list of dense tiles instead, for the caller's other kernel (the tensor-core product, or the
//     event kernel without a list);
//   * sums_kernel holds the weights of 32 neurons, all inputs, in shared memory ([input][32], one
//     persistent CTA per SM) and gives each warp one chunk at a time: its four groups of 8 lanes
//     take one step each, a lane 4 neurons, so one 16-byte shared read per lane serves an event of
//     four different steps at once, without bank conflicts (8 lanes read one 128-byte row).
//     Group q takes the steps with t % 4 = q, the busiest first: the four steps of a round are
//     then nearly as long as one another and are padded, with references to a row of zeros, to
//     the longest (16 event pairs a group and chunk at 30 Hz and 0.1 ms, against 22 in the order
//     of time), so the warp never diverges; their results go to distinct banks of a stage from
//     which each half chunk leaves as one tensor store.
// Records reach a warp's double buffer by cp.async one unit ahead.
// A sum runs over the step's inputs in ascending order from zero, the bias last: deterministic,
// within (k + 1) 2^-24 (|bias_i| + sum_j |W_ij| S_j) of the exact sum for k active inputs.
#include <cuda_bf16.h>

#include <cmath>

#include "common.cuh"
#include "tmap.h"

namespace alif {
namespace sparse {

constexpr int TILE = 256, CHUNKS = TILE / 32;  // steps and chunks per tile
constexpr int HEAD_BYTES = 128;                // record: a word per (group q, round i), then the events
constexpr uint32_t DENSE = 0xffffffffu;        // header word of a chunk of a dense tile
constexpr int WARPS = 16, THREADS = WARPS * 32;
constexpr int NT = 32;                         // neurons per weight tile
constexpr int MAX_NIN = 1024;                  // beyond it the records next to the weights get too short
constexpr int STAGE_BYTES = 32 * NT * 4;       // a warp's [32 neurons][32 steps] output
constexpr int SMEM = 227 * 1024;

// Shared memory: output stages (1024-byte aligned), weights [Nin + 1][32], flags, record buffers.
__host__ __device__ constexpr int off_w() { return WARPS * STAGE_BYTES; }
__host__ __device__ constexpr int off_bad(int Nin) { return off_w() + (Nin + 1) * NT * 4; }
__host__ __device__ constexpr int off_rec(int Nin) { return off_bad(Nin) + NT * 4; }
// Two record buffers per warp in what is left: 16 bytes per lane and copy, up to 2 KB.
__host__ __device__ constexpr int rec_bytes(int Nin) {
    const int r = (SMEM - 1024 - off_rec(Nin)) / (2 * WARPS) / 512 * 512;
    return r > 2048 ? 2048 : r;
}
__host__ __device__ constexpr int cap_of(int Nin) { return (rec_bytes(Nin) - HEAD_BYTES) / 2; }  // padding included
static_assert(rec_bytes(MAX_NIN) >= 1024, "records keep 14 events a step");

// Workspace: [0] number of dense tiles, [1] whether all are; from byte 256 the list of dense tiles,
// then the records.
struct Work {
    uint32_t *ndense, *dense;
    unsigned char *rec;
};
inline size_t up256(size_t n) { return (n + 255) & ~(size_t)255; }
inline size_t layout(long long tiles, int rec, void *base, Work *w) {
    unsigned char *p = static_cast<unsigned char *>(base);
    const size_t at = 256 + up256((size_t)tiles * 4);
    if (w) *w = Work{(uint32_t *)p, (uint32_t *)(p + 256), p + at};
    return at + (size_t)tiles * CHUNKS * rec;
}

// Starts a workspace's flags: [0] no dense tile yet, [1] whether a sample of the raster has more than
// `limit` active inputs per step.  One block, 4 words per
// thread (131 000 input steps; 32 words took 30 us: one SM's random reads).  The sampled word of each 4096th
// of the raster is at a scattered place in it: at equal distances, which were multiples of the words per row
// for many sizes (128 x 256 x 1000 steps among them), every sample fell on the same 32 steps.
constexpr int SAMPLE = 4;
static_assert(1024 * SAMPLE == 1 << 12, "a 4096th per sampled word");
__global__ void __launch_bounds__(1024, 1) sample_kernel(const uint32_t *__restrict__ S, long long words, long long Nin,
                                                         float limit, uint32_t *flags) {
    __shared__ int part[32];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const long long n = words < 1024 * SAMPLE ? words : 1024 * SAMPLE;
    uint32_t v[SAMPLE];
#pragma unroll
    for (int m = 0; m < SAMPLE; ++m) {
        const uint32_t k = m * 1024 + tid;
        uint32_t h = k * 2654435769u;  // scattered over 32 bits (odd multipliers and shifted exclusive-ors)
        h = (h ^ h >> 15) * 2246822519u;
        h ^= h >> 13;
        // floor((k + h / 2^32) words / 4096) < words
        const uint64_t at = words > n ? __umul64hi(((uint64_t)k << 32 | h) << 20, (uint64_t)words) : k;
        v[m] = k < n ? __ldg(S + at) : 0u;
    }
    int c = 0;
#pragma unroll
    for (int m = 0; m < SAMPLE; ++m) c += __popc(v[m]);
    c = __reduce_add_sync(FULL, c);
    if (lane == 0) part[warp] = c;
    __syncthreads();
    if (warp == 0) {
        c = __reduce_add_sync(FULL, part[lane]);
        if (lane == 0) {
            flags[0] = 0u;
            flags[1] = (float)c * (float)Nin > limit * 32.0f * (float)n;
        }
    }
}

constexpr int LT = 4, LW = LT * CHUNKS;  // tiles and chunks (one warp each) per CTA of lists_kernel

// Inputs of a chunk that can be queued: more active ones than events in a record make it dense anyway.
__host__ __device__ constexpr int queue_of(int Nin) {
    const int rows = (Nin + 31) / 32 * 32;
    return rows < cap_of(Nin) ? rows : cap_of(Nin);
}
// Shared memory of lists_kernel: the chunks' records and their queues of words and inputs.
__host__ __device__ constexpr int lists_smem(int Nin) { return LW * (rec_bytes(Nin) + queue_of(Nin) * 6); }
constexpr int LISTS_SMEM = SMEM - 8448;  // less the static arrays
static_assert(lists_smem(782) <= LISTS_SMEM, "the most any Nin takes");

// A CTA takes 1024 steps of a batch element: a warp reads 128 consecutive bytes of a row per load and
// all of its rows (a 32nd) at once, so that the raster comes from DRAM in whole lines; the inputs
// that are silent in a chunk (91 % at 30 Hz and 0.1 ms) are left out of its queue.  Reading 32 bytes
// of each row took 83 us for the benchmark's 64 MB.
__global__ void __launch_bounds__(LW * 32, 1) lists_kernel(long long Nin, long long T, long long nwin, long long tiles_t,
                                                           const uint32_t *__restrict__ S, int cap, int rec_bytes,
                                                           int nqueue, const Work ws) {
    extern __shared__ __align__(16) unsigned char recs[];
    if (__ldg(ws.ndense + 1)) return;
    __shared__ int counts[LW][33];   // [chunk][warp]: words that are not zero, then those of the warps before
    __shared__ int dense_tile[LT];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const long long nblk = (tiles_t + LT - 1) / LT, b = blockIdx.x / nblk, tile0 = (blockIdx.x - b * nblk) * LT;
    const long long w0 = tile0 * CHUNKS;
    const int mine = (int)((Nin + 31) / 32);  // rows per warp
    uint32_t *word_queues = reinterpret_cast<uint32_t *>(recs + LW * rec_bytes);
    uint16_t *row_queues = reinterpret_cast<uint16_t *>(word_queues + LW * nqueue);
    if (tid < LT) dense_tile[tid] = 0;
    {
        uint32_t v[32];
        const uint32_t mask = w0 + lane < nwin - 1 ? ~0u : w0 + lane == nwin - 1 ? ((T & 31) ? (1u << (T & 31)) - 1u : ~0u) : 0u;
        const uint32_t *col = S + (b * Nin + warp * mine) * nwin + w0 + lane;
        const int have = (int)(Nin - warp * mine < mine ? Nin - warp * mine : mine);  // may be negative
#pragma unroll
        for (int m = 0; m < 32; ++m) v[m] = m < have && mask ? __ldg(col + m * nwin) : 0u;
        int n = 0;
#pragma unroll
        for (int m = 0; m < 32; ++m) {
            v[m] &= mask;
            n += v[m] != 0u;
        }
        counts[lane][warp] = n;
        __syncthreads();
        {  // warp = chunk, lane = warp of the load
            const int c = counts[warp][lane];
            int incl = c;
#pragma unroll
            for (int l = 1; l < 32; l <<= 1) {
                const int o = __shfl_up_sync(FULL, incl, l);
                if (lane >= l) incl += o;
            }
            counts[warp][lane] = incl - c;
            if (lane == 31) counts[warp][32] = incl;
        }
        __syncthreads();
        int e = counts[lane][warp];
#pragma unroll
        for (int m = 0; m < 32; ++m)
            if (v[m]) {
                if (e < nqueue) {
                    word_queues[lane * nqueue + e] = v[m];
                    row_queues[lane * nqueue + e] = (uint16_t)(warp * mine + m);
                }
                ++e;
            }
    }
    __syncthreads();
    const long long tile = b * tiles_t + tile0 + warp / CHUNKS;
    const bool live = tile0 + warp / CHUNKS < tiles_t;
    const uint32_t *wq = word_queues + warp * nqueue;
    const uint16_t *rq = row_queues + warp * nqueue;
    const bool over = counts[warp][32] > nqueue;
    const int nq = over ? 0 : counts[warp][32];
    // lane = step: its mask over 32 queued inputs.  Events in a few steps only: one ballot for each
    // of them; else a bit transpose.
    auto by_step = [&](int i) {
        const uint32_t x = i + lane < nq ? wq[i + lane] : 0u;
        uint32_t steps = __reduce_or_sync(FULL, x), y = 0u;
        if (__popc(steps) > 6) return bits_transpose32(x, lane);
        while (steps) {
            const int s = __ffs(steps) - 1;
            steps &= steps - 1u;
            const uint32_t m = __ballot_sync(FULL, (x >> s) & 1u);
            if (lane == s) y = m;
        }
        return y;
    };
    int n = 0;
    for (int i = 0; i < nq; i += 32) n += __popc(by_step(i));
    const int pairs = (n + 1) >> 1;
    // round of this step: its rank among its group's (t % 4) steps of its half chunk, the longest
    // first; rounds 4-7 are the second half's
    const int q = lane & 3, k = lane >> 2;
    int round = 0;
#pragma unroll
    for (int m = 0; m < 4; ++m) {
        const int mm = m + (k & 4), o = __shfl_sync(FULL, pairs, 4 * mm + q);
        round += o > pairs || (o == pairs && mm < k);
    }
    round += k & 4;
    // lane 4 i + q := round i: its longest step and the pairs before it
    __shared__ int by_round[LW][32];
    by_round[warp][4 * round + q] = pairs;
    __syncwarp();
    int longest = by_round[warp][lane];
    longest = max(longest, __shfl_xor_sync(FULL, longest, 1));
    longest = max(longest, __shfl_xor_sync(FULL, longest, 2));
    int upto = longest;
#pragma unroll
    for (int l = 4; l < 32; l <<= 1) {
        const int o = __shfl_up_sync(FULL, upto, l);
        if (lane >= l) upto += o;
    }
    const int total = __shfl_sync(FULL, upto, 31);
    const int before = __shfl_sync(FULL, upto - longest, 4 * round);
    longest = __shfl_sync(FULL, longest, 4 * round);
    // one pair of zero rows, one word read past it
    if (lane == 0 && (over || 8 * (total + 2) > cap)) dense_tile[warp / CHUNKS] = 1;
    __syncthreads();
    const bool dense = dense_tile[warp / CHUNKS];
    if (!live) return;
    const long long chunk = tile * CHUNKS + warp % CHUNKS;
    uint4 *to = reinterpret_cast<uint4 *>(ws.rec + chunk * rec_bytes);
    uint32_t *head = reinterpret_cast<uint32_t *>(recs + warp * rec_bytes);
    head[8 * q + round] = dense ? DENSE : (uint32_t)k | (uint32_t)longest << 3;
    if (dense) {
        if (lane == 0 && warp % CHUNKS == 0) ws.dense[atomicAdd(ws.ndense, 1u)] = (uint32_t)tile;
        __syncwarp();
        if (lane < HEAD_BYTES / 16) to[lane] = reinterpret_cast<const uint4 *>(head)[lane];
        return;
    }
    // pair r of round i, group q is word 4 (before_i + r) + q
    uint16_t *ev = reinterpret_cast<uint16_t *>(head) + HEAD_BYTES / 2 + 2 * (4 * before + q);
    int e = 0;
    auto put = [&](int row) {
        ev[8 * (e >> 1) + (e & 1)] = (uint16_t)(row * (NT / 4));  // the weight row, in 16-byte units
        ++e;
    };
    for (int i = 0; i < nq; i += 32) {
        uint32_t y = by_step(i);
        while (y) {
            put(rq[i + __ffs(y) - 1]);
            y &= y - 1u;
        }
    }
    while (e < 2 * longest) put((int)Nin);
    if (lane < 4) {  // lane = group: the pair after the last round
        ev = reinterpret_cast<uint16_t *>(head) + HEAD_BYTES / 2 + 2 * (4 * total + lane);
        e = 0;
        put((int)Nin);
        put((int)Nin);
    }
    __syncwarp();
    for (int i = lane; i < HEAD_BYTES / 16 + total + 1; i += 32) to[i] = reinterpret_cast<const uint4 *>(head)[i];
}

struct Args {
    long long Nin, N, T, ldw, tiles_t, nch, units, total;  // units: chunks per neuron tile; total: over the tiles
    const float *Wt;                                       // [Nin, N], or
    const uint16_t *hi, *lo;                               // [N, ldw] BF16 terms
    const float *bias;
    float *I;
    Work ws;
};

__device__ __forceinline__ void cp_async16(uint32_t dst, const void *src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}

__device__ __forceinline__ uint32_t lds32(uint32_t a) {
    uint32_t v;
    asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(a));
    return v;
}
__device__ __forceinline__ float4 lds128(uint32_t a) {
    float4 v;
    asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(a));
    return v;
}
__device__ __forceinline__ void sts32(uint32_t a, float v) {
    asm volatile("st.shared.f32 [%0], %1;" ::"r"(a), "f"(v) : "memory");
}

// The weights of neurons n0 .. n0 + 31 into w [Nin + 1][32], the last row zeros.  Neuron n is at
// column 4 (n % 8) + n / 8: a lane's 16 bytes are neurons l8, l8 + 8, l8 + 16, l8 + 24.
template <bool SPLIT>
__device__ __forceinline__ void load_weights(const Args &A, long long n0, float *w, uint32_t *bad, int lane, int warp) {
    const bool live = n0 + lane < A.N;
    const int at = 4 * (lane & 7) + (lane >> 3);
    if (warp == 0) {
        w[A.Nin * NT + lane] = 0.0f;
        bad[lane] = 0u;
    }
    __syncthreads();
    if (SPLIT) {
        const uint16_t *h = A.hi + (n0 + (live ? lane : 0)) * A.ldw, *l = A.lo + (n0 + (live ? lane : 0)) * A.ldw;
        bool odd = false;
#pragma unroll 2
        for (int j = 8 * warp; j < A.Nin; j += 8 * WARPS) {  // rows are padded to 64 inputs
            uint4 uh = make_uint4(0u, 0u, 0u, 0u), ul = uh;
            if (live) {
                uh = __ldg(reinterpret_cast<const uint4 *>(h + j));
                ul = __ldg(reinterpret_cast<const uint4 *>(l + j));
            }
            const uint32_t ph[4] = {uh.x, uh.y, uh.z, uh.w}, pl[4] = {ul.x, ul.y, ul.z, ul.w};
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                const uint32_t sh = 16 * (e & 1);
                const float x = __uint_as_float((ph[e >> 1] >> sh) << 16), y = __uint_as_float((pl[e >> 1] >> sh) << 16);
                odd |= !(fabsf(x) < __int_as_float(0x7f800000)) || !(fabsf(y) < __int_as_float(0x7f800000));
                if (j + e < A.Nin) w[(j + e) * NT + at] = x + y;
            }
        }
        // the product multiplies every weight by 0 or 1, so a weight that is not finite makes all of
        // its neuron's currents NaN, whichever inputs are active
        if (odd) bad[lane] = 1u;
    } else {
#pragma unroll 8
        for (int j = warp; j < A.Nin; j += WARPS) w[j * NT + at] = live ? __ldg(A.Wt + j * A.N + n0 + lane) : 0.0f;
    }
    __syncthreads();
}

// TMA: output rows keep 16 bytes, so a half chunk leaves its stage as one tensor store.
// What bounds it: shared-memory wavefronts (one per event and 32 neurons, 124 per chunk with the
// padding at 30 Hz and 0.1 ms, and 64 through the stage) and the output's 4 bytes per step.
// B = 32, 1000 -> 1024, T = 16000: 0.46 ms (plain stores of that output from as many warps: 0.31;
// the dense product: 1.45).  Stages of whole chunks, which a warp has to wait for, took 0.53;
// lanes storing 32 bytes each to eight rows 0.60, a wavefront per sector.
template <bool SPLIT, bool TMA>
__global__ void __launch_bounds__(THREADS, 1) sums_kernel(const __grid_constant__ CUtensorMap out, const Args A) {
    extern __shared__ unsigned char raw[];
    if (__ldg(A.ws.ndense + 1)) return;
    unsigned char *smem = raw + ((1024u - (smem_u32(raw) & 1023u)) & 1023u);
    const int Nin = (int)A.Nin, rbytes = rec_bytes(Nin);
    float *w = reinterpret_cast<float *>(smem + off_w());
    uint32_t *bad = reinterpret_cast<uint32_t *>(smem + off_bad(Nin));
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int q = lane >> 3, l8 = lane & 7;  // this lane: steps q + 4 k, neurons l8 + 8 n
    unsigned char *buf = smem + off_rec(Nin) + warp * 2 * rbytes;
    const uint32_t buf_s = smem_u32(buf);
    unsigned char *stage = smem + warp * STAGE_BYTES;
    const uint32_t wl = smem_u32(smem + off_w() + 16 * l8), stage_s = smem_u32(stage);
    const long long first = A.total * blockIdx.x / gridDim.x, last = A.total * (blockIdx.x + 1) / gridDim.x;
    for (long long u0 = first; u0 < last;) {
        const long long m = u0 / A.units, stop = (m + 1) * A.units < last ? (m + 1) * A.units : last;
        const long long n0 = m * NT;
        __syncthreads();  // every warp is done with the previous tile's weights
        load_weights<SPLIT>(A, n0, w, bad, lane, warp);
        float bias[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const long long n = n0 + l8 + 8 * i;
            bias[i] = A.bias && n < A.N ? A.bias[n] : 0.0f;
            if (SPLIT && bad[l8 + 8 * i]) bias[i] = __int_as_float(0x7fc00000);
        }
        const int nch = (int)A.nch, gap = (int)A.tiles_t * CHUNKS - nch;  // records past T between batch elements
        const int left = (int)(stop - u0);
        int u = warp, b = (int)((u0 - m * A.units + warp) / nch), c = (int)((u0 - m * A.units + warp) % nch);
        const unsigned char *src = A.ws.rec + ((long long)b * A.tiles_t * CHUNKS + c) * rbytes + 16 * lane;
        auto fetch = [&](int half) {  // the whole record, whatever it holds: no size to wait for
            for (int o = 0; o < rbytes; o += 512) cp_async16(buf_s + half * rbytes + 16 * lane + o, src + o);
            asm volatile("cp.async.commit_group;" ::: "memory");
        };
        if (u < left) fetch(0);
        for (int half = 0; u < left; u += WARPS, half ^= 1) {
            const int cb = b, cc = c;
            if (u + WARPS < left) {
                c += WARPS;
                src += WARPS * rbytes;
                while (c >= nch) {
                    c -= nch;
                    ++b;
                    src += gap * rbytes;
                }
                fetch(half ^ 1);
                asm volatile("cp.async.wait_group 1;" ::: "memory");
            } else {
                asm volatile("cp.async.wait_group 0;" ::: "memory");
            }
            __syncwarp();
            const unsigned char *rec = buf + half * rbytes;
            const uint4 h0 = *reinterpret_cast<const uint4 *>(rec + 32 * q);
            const uint4 h1 = *reinterpret_cast<const uint4 *>(rec + 32 * q + 16);
            if (h0.x != DENSE) {
                const uint32_t head[8] = {h0.x, h0.y, h0.z, h0.w, h1.x, h1.y, h1.z, h1.w};
                uint32_t ev = buf_s + half * rbytes + HEAD_BYTES + 4 * q;
                uint32_t pr = lds32(ev);  // one reference word ahead (the record ends with a pair of zero rows)
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    // rounds 0-3: steps 0-15 into the stage's first half, 4-7: the others; a half is
                    // written again once its store before (all but the newest) has been read
                    if (TMA && (i & 3) == 0) {
                        if (lane == 0) asm volatile("cp.async.bulk.wait_group.read 1;" ::: "memory");
                        __syncwarp();
                    }
                    float2 a0 = make_float2(0.0f, 0.0f), a1 = a0;
#pragma unroll 2
                    for (int r = (int)(head[i] >> 3); r > 0; --r) {
                        const float4 x = lds128(wl + (pr & 0xffffu) * 16u), y = lds128(wl + (pr >> 16) * 16u);
                        ev += 16;
                        pr = lds32(ev);
                        a0 = __fadd2_rn(__fadd2_rn(a0, make_float2(x.x, x.y)), make_float2(y.x, y.y));
                        a1 = __fadd2_rn(__fadd2_rn(a1, make_float2(x.z, x.w)), make_float2(y.z, y.w));
                    }
                    // row = neuron; step 4 k + q.  TMA: 64-byte rows per half, 16-byte unit k % 4 at
                    // (k % 4) ^ (row / 2 % 4) (the 64-byte swizzle); else 128-byte rows, unit k at k ^ (row % 8)
                    const uint32_t k = head[i] & 7u;
                    const uint32_t o = stage_s + 4 * q + (TMA ? (i >> 2) * (STAGE_BYTES / 2) + l8 * 64 + 16 * ((k & 3u) ^ (l8 >> 1 & 3))
                                                              : l8 * 128 + 16 * (k ^ l8));
                    constexpr int RS = TMA ? 8 * 64 : 8 * 128;
                    sts32(o, a0.x + bias[0]);
                    sts32(o + RS, a0.y + bias[1]);
                    sts32(o + 2 * RS, a1.x + bias[2]);
                    sts32(o + 3 * RS, a1.y + bias[3]);
                    if (TMA && (i & 3) == 3) {
                        fence_proxy_async_smem();
                        __syncwarp();
                        if (lane == 0 && 32 * cc + 4 * (i - 3) < A.T)
                            asm volatile(
                                "cp.async.bulk.tensor.3d.global.shared::cta.tile.bulk_group [%0, {%1, %2, %3}], [%4];" ::"l"(
                                    reinterpret_cast<uint64_t>(&out)),
                                "r"(32 * cc + 4 * (i - 3)), "r"((int)n0), "r"(cb),
                                "r"(stage_s + (i >> 2) * (STAGE_BYTES / 2))
                                : "memory");
                        if (lane == 0) asm volatile("cp.async.bulk.commit_group;" ::: "memory");
                    }
                }
                if (!TMA) {
                    __syncwarp();
                    const long long t = 32LL * cc + lane;
                    const int rows = (int)(A.N - n0 < NT ? A.N - n0 : NT);
                    float *o = A.I + ((long long)cb * A.N + n0) * A.T + t;
                    if (t < A.T)
#pragma unroll 8
                        for (int r = 0; r < rows; ++r)
                            o[r * A.T] = *reinterpret_cast<const float *>(stage + r * 128 + 16 * ((lane >> 2) ^ (r & 7)) +
                                                                          4 * (lane & 3));
                }
            }
            __syncwarp();  // the buffer is filled again by the next fetch
        }
        u0 = stop;
    }
    if (TMA && lane == 0) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
}

}  // namespace sparse

// Sample of a raster of `rows` rows (batch elements x inputs): whether more than `limit` of Nin inputs are active per step.
int launch_density_sample(const uint32_t *S, long long rows, long long Nin, long long T, float limit, uint32_t *flags,
                          cudaStream_t st) {
    const long long nwin = (T + 31) / 32;
    // the rows' last words hold T % 32 steps: of rows of 20 steps 20 active inputs counted as 12.5
    sparse::sample_kernel<<<1, 1024, 0, st>>>(S, rows * nwin, Nin, limit * (float)((double)T / (32.0 * (double)nwin)), flags);
    return (int)cudaGetLastError();
}

// Workspace bytes of the sparse projection; 0 where it is not used: more inputs than a weight tile
// holds, or a product too small to pay for the lists and three more launches.
//   * In place of the tensor cores: from 6e10 products on.  There (B = 16, 512 -> 1024, T = 8000) the
//     dense product takes 0.34 ms and this path about half of it at up to 1.5 active inputs a step;
//     a raster that turns out dense costs the sample and the empty launches, 8 us, whatever the size.
//   * In place of the event kernel without lists: from 2e10 (8, 1000 -> 1024, 4000: 72 against
//     79 us at 1.5 active inputs a step, 78 against 96 at 3).  That kernel's time goes with the 32-step
//     chunks, about 30 us + 35 ns each whatever N up to 1024, this path's is about 35 us + 0.03 ns a chunk
//     and neuron, so smaller products too where the chunks are many for the neurons (us, that / this):
//     27, 512 -> 154, 1800 84 / 41; 10, 700 -> 256, 2001 68 / 42 and at 21 active inputs a step 205 / 68;
//     32, 128 -> 128, 4000 152 / 42; 7, 512 -> 607, 5100 61 / 54; not for 4, 300 -> 200, 3000 29 / 33 and
//     1, 512 -> 600, 16000 35 / 37.  A CTA of the lists kernel takes 30 ns
//     however few of its 1024 steps there are, so not for rows of one chunk either: 2048, 64 -> 64, 32 68 / 93 and 512,
//     700 -> 256, 32 37 / 44 (64 steps: 128 / 96 and 63 / 48).
size_t syn_sparse_ws(long long B, long long Nin, long long N, long long T, bool split) {
    using namespace sparse;
    if (B <= 0 || Nin <= 0 || N <= 0 || T <= 0 || Nin > MAX_NIN) return 0;
    const double chunks = (double)B * (double)((T + 31) / 32);
    const bool many = !split && T > 32 && chunks * (1150.0 - (double)N) >= 4e5;
    if (!many && (double)B * (double)Nin * (double)N * (double)T < (split ? 6e10 : 2e10)) return 0;
    const long long tiles = B * ((T + TILE - 1) / TILE);
    if (tiles > (1LL << 30) || (N + NT - 1) / NT > (1LL << 30)) return 0;
    return layout(tiles, rec_bytes((int)Nin), nullptr, nullptr);
}

// Currents of the sparse tiles; *dense (device): the number of dense tiles, whether all are (then
// there is no list), their list from dense + 64 (tile = b ceil(T / 256) + t / 256).  Weights: W_t [Nin, N], or the BF16 terms when hi is given.
int launch_syn_sparse(long long B, long long Nin, long long N, long long T, const float *Wt, const uint16_t *hi,
                      const uint16_t *lo, long long ldw, const uint32_t *S, const float *bias, float *I, void *work,
                      const uint32_t **dense, cudaStream_t st) {
    using namespace sparse;
    Args A{Nin, N, T, ldw, (T + TILE - 1) / TILE, (T + 31) / 32, 0, 0, Wt, hi, lo, bias, I, {}};
    const long long tiles = B * A.tiles_t;
    const int rec = rec_bytes((int)Nin);
    layout(tiles, rec, work, &A.ws);
    A.units = B * A.nch;
    A.total = A.units * ((N + NT - 1) / NT);
    *dense = A.ws.ndense;
    // Above `limit` active inputs a step the other kernel takes all.  At B = 32, N = 1024, T = 16000 this
    // path takes 0.43 ms at 1.5 of 1000 inputs, 0.52 at 3, 0.97 at 9 (dense product: 1.51) and 0.43 at
    // 1.5 of 512, 0.65 at 4.6 (0.84): about 0.58 + 0.13 per active input ps an output, against 2.78 Nin /
    // 1000 but no less than 1.43.  The event kernel without lists is slower at every density (2.23 ms
    // at 9 of 1000, 3.11 against 1.37 at 15 of 512), so there only the records' capacity counts.
    // Padded to pairs and to the longest of four, Poisson counts take about a square root more room than their mean: at
    // 1000 inputs (room for 14 a step) 3 % of the 256-step tiles are over at 9, 59 % at 10, all at 11.  us of the event
    // projection without / with lists, 32 x 1000 -> 1024 x 4000 steps: 575 / 283, 613 / 522, 655 / 701, and at 12 698 / 736.
    const float fit = cap_of((int)Nin) / 32.0f, room = fit - 0.95f * sqrtf(fit), even = 0.0214f * Nin - 4.5f;
    const float limit = !hi || even > room ? room : even > 6.5f ? even : 6.5f;
    const int rc = launch_density_sample(S, B * Nin, Nin, T, limit, A.ws.ndense, st);
    if (rc) return rc;
    CUtensorMap out = {};
    const bool tma = make_batch_rows_map(&out, I, B, N, T) == 0;
    const auto sums = hi ? (tma ? sums_kernel<true, true> : sums_kernel<true, false>)
                         : (tma ? sums_kernel<false, true> : sums_kernel<false, false>);
    cudaError_t e = cudaFuncSetAttribute(sums, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM);
    if (e != cudaSuccess) return (int)e;
    int dev = 0, sms = 0;
    e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return (int)e;
    e = cudaFuncSetAttribute(lists_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, LISTS_SMEM);
    if (e != cudaSuccess) return (int)e;
    lists_kernel<<<(unsigned)(B * ((A.tiles_t + LT - 1) / LT)), LW * 32, lists_smem((int)Nin), st>>>(
        Nin, T, A.nch, A.tiles_t, S, cap_of((int)Nin), rec, queue_of((int)Nin), A.ws);
    e = cudaGetLastError();
    if (e != cudaSuccess) return (int)e;
    const long long want = (A.total + 7) / 8;
    sums<<<(unsigned)(want < sms ? want : sms), THREADS, off_rec((int)Nin) + WARPS * 2 * rec + 1024, st>>>(out, A);
    return (int)cudaGetLastError();
}

}  // namespace alif

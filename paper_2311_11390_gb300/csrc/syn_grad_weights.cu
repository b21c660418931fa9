#include <cmath>
// Weight and bias gradients of the synaptic projection over sparse rasters:
//     g_W[i, j] = sum_{b,t} g_I[b, i, t] S[b, j, t],   g_bias[i] = sum_{b,t} g_I[b, i, t].
// Every input spike adds one column of g_I to its input's row of g_W^T.
//   * gw_lists_kernel turns the raster into lists once: per unit (batch element, 512-step chunk) the
//     active inputs in groups of four, the busiest first, each with its steps padded to the longest
//     of the four with references to a row of zeros.  (Which inputs share a group does not matter to
//     the result, so ties are placed by atomics.)
//   * gw_sums_kernel: a CTA owns 32 neurons, all inputs (sums [input][32] in shared memory) and a
//     range of units.  Per unit it stages g_I [512 steps][32 neurons] transposed and deals the groups
//     out to its warps: 8 lanes take an input, a lane 4 neurons, so that one 16-byte read per lane
//     serves four spikes without bank conflicts (8 lanes read one 128-byte row) and the warp never
//     diverges; then the four inputs' sums are updated.  The next unit's g_I (registers) and lists
//     (cp.async, double-buffered) are on their way meanwhile.
//     A unit with more spikes than its list holds is walked from the raster instead (walk_unit): at
//     64 x 512 -> 512 x 4096 steps with one such unit per batch element 0.35 ms, where the whole call
//     went to the other kernel 0.55.
//   * gw_join_kernel adds the ranges' sums in a fixed order: deterministic.
// What bounds it: shared-memory traffic.  Per spike and 32 neurons its 128-byte column is read and, at
// 1000 inputs, 30 Hz and 0.1 ms, another 128 bytes of sums are (an input's sums are read and written
// once per 512 steps); every staged value is written once.  B = 32, 1000 -> 1024, T = 16000: sums
// 0.86 ms (events alone 0.48, staging without events 0.47: the two overlap badly, loads or L2
// prefetches issued a unit ahead notwithstanding), lists 0.07, against 2.41 ms for a thread per input
// that walks its own spikes, whose warps wait for their busiest lane.
#include "common.cuh"

namespace alif {
namespace gwl {

constexpr int CH = 512, CW = CH / 32;  // steps and spike words per unit
constexpr int NT = 32;                 // neurons per CTA
constexpr int WARPS = 32, THREADS = WARPS * 32;
constexpr int MAX_NIN = 1024, MAX_QUADS = MAX_NIN / 4;
// Record of a unit: u16 start[MAX_QUADS] (in 16-byte rows), then per group of four inputs a row of
// words (input | steps << 11 | row of the group 32 further on, for the same warp << 21) and rows of
// steps, word q of a row for input q, two per word.
constexpr int HEAD = 2 * MAX_QUADS;
// Step t of the staged chunk: 32 neurons at 16 row_of(t), four steps' 512 bytes and 16 of padding, so
// that neither the staging stores nor the 128-byte reads meet bank conflicts.
__host__ __device__ constexpr int row_of(int t) { return 8 * t + (t >> 2); }
constexpr int ZERO_ROW = row_of(CH);
constexpr int GT_BYTES = 16 * ZERO_ROW + 128;
constexpr int SMEM = 227 * 1024;
constexpr int MAX_ROWS = 2047;

// 16-byte rows a unit's record holds: two buffers next to the staged chunk and the sums (one more
// input's for groups that are not full).
__host__ __device__ constexpr int sums_bytes(int Nin) { return (Nin + 1) * NT * 4; }
__host__ __device__ constexpr int rows_of(int Nin) {
    const int r = ((SMEM - 64 - GT_BYTES - sums_bytes(Nin)) / 2 - HEAD) / 16;  // 64: a word is read past a record
    return r < MAX_ROWS ? r : MAX_ROWS;
}
__host__ __device__ constexpr int rec_of(int Nin) { return HEAD + 16 * rows_of(Nin); }
__host__ __device__ constexpr int smem_of(int Nin) { return GT_BYTES + sums_bytes(Nin) + 2 * rec_of(Nin) + 64; }
static_assert(smem_of(MAX_NIN) <= SMEM && rows_of(MAX_NIN) >= 1000, "10 spikes a step fit at any Nin");

// Workspace: [1] whether a sample of the raster is too dense for the lists (written by the sample alone);
// from byte 256 the units' sizes (groups | rows << 16, or OVER for one whose list does not fit), their
// records, the ranges' sums [range][tile][input][32] and of g_I itself [range][tile][32].
struct Work {
    uint32_t *flag, *count;
    unsigned char *rec;
    float *part, *part_b;
};
inline size_t up256(size_t n) { return (n + 255) & ~(size_t)255; }
inline size_t layout(long long units, long long tiles, int ranges, int Nin, void *base, Work *w) {
    unsigned char *p = static_cast<unsigned char *>(base);
    const size_t o1 = 256, o2 = o1 + up256((size_t)units * 4), o3 = o2 + up256((size_t)units * rec_of(Nin));
    const size_t o4 = o3 + up256((size_t)ranges * tiles * Nin * NT * 4);
    if (w) *w = Work{(uint32_t *)p, (uint32_t *)(p + o1), p + o2, (float *)(p + o3), (float *)(p + o4)};
    return o4 + (size_t)ranges * tiles * NT * 4;
}

// Ranges of units per neuron tile: the fewest for which the CTAs fill whole waves to 6 %, out of 64 or, where the
// tiles are one or two, as many as fill the SMs (with 64 CTAs for one tile 249 x 186 -> 16 x 4105 steps took 138 us,
// now 115).
inline int ranges_for(long long tiles, long long units, int sms) {
    int best = 1;
    double least = 1e30;
    const long long most = sms / tiles > 64 ? sms / tiles : 64;
    for (int p = 1; p <= most && p <= units; ++p) {
        const long long ctas = tiles * p;
        const double waste = (double)((ctas + sms - 1) / sms * sms) / (double)ctas;
        if (waste < least - 1e-9) {
            least = waste;
            best = p;
        }
        if (waste <= 1.06) break;
    }
    return best;
}

constexpr uint32_t OVER = 0xffffu;

// One CTA per 1024 steps (two units) of a batch element: a warp holds a 32nd of the rows, a lane the
// word of 32 steps, so that the raster is read in whole lines.
// A bin per count, so that the groups' lengths (and whether they fit) do not depend on the order in
// which inputs of equal counts are placed; PER of them per lane of the scan.
constexpr int PER = 17, BINS = 32 * PER;
static_assert(BINS > CH, "a bin for every count");
__host__ __device__ constexpr int lists_smem(int Nin) { return 2 * rec_of(Nin); }

__global__ void __launch_bounds__(1024, 1) gw_lists_kernel(int Nin, long long T, long long nwin, long long nch,
                                                           const uint32_t *__restrict__ S, const Work ws) {
    if (__ldg(ws.flag + 1)) return;
    extern __shared__ __align__(16) unsigned char recs[];  // two records
    __shared__ uint16_t count[2][MAX_NIN], slot[2][MAX_NIN], order[2][MAX_NIN];
    __shared__ int bin[2][BINS];
    __shared__ int upto[2][MAX_QUADS], warp_rows[2][8];
    __shared__ bool fit[2];
    const int rec = rec_of(Nin), cap = rows_of(Nin);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int half = lane >> 4, l16 = lane & 15;
    const long long nblk = (nwin + 31) / 32, b = blockIdx.x / nblk, w0 = (blockIdx.x - b * nblk) * 32;
    const int mine = (Nin + 31) / 32;  // rows per warp
    const int have = Nin - warp * mine < mine ? Nin - warp * mine : mine;
    uint32_t v[32];
    {
        const uint32_t mask = w0 + lane < nwin - 1 ? ~0u : w0 + lane == nwin - 1 ? ((T & 31) ? (1u << (T & 31)) - 1u : ~0u) : 0u;
        const uint32_t *col = S + (b * Nin + warp * mine) * nwin + w0 + lane;
#pragma unroll
        for (int m = 0; m < 32; ++m) v[m] = m < have && mask ? __ldg(col + m * nwin) : 0u;
#pragma unroll
        for (int m = 0; m < 32; ++m) v[m] &= mask;
    }
    for (int k = tid; k < 2 * BINS; k += 1024) bin[k / BINS][k % BINS] = 0;
    if (tid < 16) warp_rows[tid >> 3][tid & 7] = 0;
    // spikes per input and unit
#pragma unroll
    for (int m = 0; m < 32; ++m) {
        if (m >= have) break;  // uniform in the warp
        int c = __popc(v[m]);
        if (__any_sync(FULL, c != 0)) {
#pragma unroll
            for (int l = 1; l < 16; l <<= 1) c += __shfl_xor_sync(FULL, c, l);
        }
        if (l16 == 0) count[half][warp * mine + m] = (uint16_t)c;
    }
    __syncthreads();
    // inputs in the order of their counts, the busiest first; those without spikes are left out
    const int h = tid >> 9, i = tid & 511;  // thread: unit h, inputs i and i + 512
#pragma unroll
    for (int k = 0; k < MAX_NIN; k += 512)
        if (i + k < Nin && count[h][i + k]) atomicAdd(&bin[h][count[h][i + k]], 1);
    __syncthreads();
    if (warp < 2) {  // bin -> inputs in busier bins; lane's bins, the busiest first: BINS - 1 - PER lane and down
        int *mine_bins = bin[warp] + BINS - 1 - PER * lane, sum = 0;
        for (int k = 0; k < PER; ++k) sum += mine_bins[-k];
        int incl = sum;
#pragma unroll
        for (int l = 1; l < 32; l <<= 1) {
            const int o = __shfl_up_sync(FULL, incl, l);
            if (lane >= l) incl += o;
        }
        incl -= sum;
        for (int k = 0; k < PER; ++k) {
            const int c = mine_bins[-k];
            mine_bins[-k] = incl;  // bin 0: all active inputs
            incl += c;
        }
    }
    __syncthreads();
    const int active = bin[h][0], quads = (active + 3) / 4;
#pragma unroll
    for (int k = 0; k < MAX_NIN; k += 512)
        if (i + k < Nin && count[h][i + k]) {
            const int s = atomicAdd(&bin[h][count[h][i + k]], 1);
            slot[h][i + k] = (uint16_t)s;
            order[h][s] = (uint16_t)(i + k);
        }
    __syncthreads();
    // rows of each group: its words, and the steps of its busiest input, two per word
    int longest = 0, rows = 0;
    if (i < quads) {
#pragma unroll
        for (int q = 0; q < 4; ++q)
            if (4 * i + q < active) longest = max(longest, (int)count[h][order[h][4 * i + q]]);
        rows = 1 + (longest + 1) / 2;
    }
    int incl = rows;
    if (i < MAX_QUADS) {  // 8 warps per unit
#pragma unroll
        for (int l = 1; l < 32; l <<= 1) {
            const int o = __shfl_up_sync(FULL, incl, l);
            if (lane >= l) incl += o;
        }
        if (lane == 31) warp_rows[h][i >> 5] = incl;
    }
    __syncthreads();
    int total = 0, before = 0;
#pragma unroll
    for (int w = 0; w < 8; ++w) {
        if (w < (i >> 5)) before += warp_rows[h][w];
        total += warp_rows[h][w];
    }
    const bool fits = total <= cap;
    unsigned char *record = recs + h * rec;
    if (i < MAX_QUADS) {
        const int start = before + incl - rows;
        reinterpret_cast<uint16_t *>(record)[i] = (uint16_t)start;
        upto[h][i] = start;
    }
    __syncthreads();
    if (fits && i < quads) {
        const uint32_t next = i + WARPS < quads ? (uint32_t)upto[h][i + WARPS] : 0u;
#pragma unroll
        for (int q = 0; q < 4; ++q)
            reinterpret_cast<uint32_t *>(record + HEAD)[4 * upto[h][i] + q] =
                (4 * i + q < active ? (uint32_t)order[h][4 * i + q] : (uint32_t)Nin) | (uint32_t)longest << 11 | next << 21;
        // every step a reference to the zeros until an input's own replaces it
        for (int k = 4 * (upto[h][i] + 1); k < 4 * (upto[h][i] + rows); ++k)
            reinterpret_cast<uint32_t *>(record + HEAD)[k] = (uint32_t)ZERO_ROW << 16 | (uint32_t)ZERO_ROW;
    }
    if (tid == 0 || tid == 512) {
        const long long c = w0 / CW + h;
        if (c < nch) {
            ws.count[b * nch + c] = fits ? (uint32_t)quads | (uint32_t)total << 16 : OVER;
        }
        fit[h] = fits;
    }
    __syncthreads();
    // the steps
#pragma unroll
    for (int m = 0; m < 32; ++m) {
        if (m >= have) break;
        uint32_t y = v[m];
        if (!__any_sync(FULL, y != 0u)) continue;
        const int c = __popc(y), row = warp * mine + m;
        int e = c;
#pragma unroll
        for (int l = 1; l < 16; l <<= 1) {
            const int o = __shfl_up_sync(FULL, e, l, 16);
            if (l16 >= l) e += o;
        }
        e -= c;  // this word's first spike among the input's
        if (y && fit[half]) {
            const int s = slot[half][row];
            uint16_t *to = reinterpret_cast<uint16_t *>(recs + half * rec + HEAD + 16 * (upto[half][s >> 2] + 1)) + 2 * (s & 3);
            while (y) {
                to[8 * (e >> 1) + (e & 1)] = (uint16_t)row_of(32 * l16 + __ffs(y) - 1);
                y &= y - 1u;
                ++e;
            }
        }
    }
    __syncthreads();
    const long long c = w0 / CW + h;
    if (c < nch && fits) {
        uint4 *to = reinterpret_cast<uint4 *>(ws.rec + (b * nch + c) * rec);
        for (int k = i; k < HEAD / 16 + total; k += 512) to[k] = reinterpret_cast<const uint4 *>(record)[k];
    }
}

struct Args {
    long long N, T, nch, units;
    int Nin, tiles, ranges, rec;
    const float *gI;
    const uint32_t *S;
    Work ws;
};

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
__device__ __forceinline__ void sts128(uint32_t a, float2 x, float2 y) {
    asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(a), "f"(x.x), "f"(x.y), "f"(y.x), "f"(y.y) : "memory");
}

// The sums of a unit whose list does not fit, from the raster: 8 lanes take an input, two of its 16 words
// each, and walk its spikes together; the same additions in the same order as from a list.
__device__ __noinline__ void walk_unit(const Args &A, long long u, uint32_t gt, uint32_t sums) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, q = lane >> 3, l8 = lane & 7;
    const long long nwin = (A.T + 31) / 32, b = u / A.nch, w0 = (u - b * A.nch) * CW + 2 * l8;
    const uint32_t gl = gt + 16 * l8, tail = (A.T & 31) ? (1u << (A.T & 31)) - 1u : ~0u;
    for (int j0 = 4 * warp; j0 < A.Nin; j0 += 4 * WARPS) {
        const int j = j0 + q;
        const uint32_t *row = A.S + (b * A.Nin + j) * nwin;
        uint32_t v[2];
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            v[k] = j < A.Nin && w0 + k < nwin ? __ldg(row + w0 + k) : 0u;
            if (w0 + k == nwin - 1) v[k] &= tail;
        }
        const uint32_t p = sums + (j < A.Nin ? j : A.Nin) * (NT * 4) + 16 * l8;  // the row past the last: scratch
        float2 a0 = make_float2(0.0f, 0.0f), a1 = a0;
        for (int k = 0; k < CW; ++k) {
            uint32_t m = __shfl_sync(FULL, (k & 1) ? v[1] : v[0], (lane & 24) | k >> 1);
            while (__any_sync(FULL, m != 0u)) {
                const float4 x = lds128(gl + 16 * (m ? row_of(32 * k + __ffs(m) - 1) : ZERO_ROW));
                m &= m - 1u;
                a0 = __fadd2_rn(a0, make_float2(x.x, x.y));
                a1 = __fadd2_rn(a1, make_float2(x.z, x.w));
            }
        }
        const float4 s = lds128(p);
        sts128(p, __fadd2_rn(a0, make_float2(s.x, s.y)), __fadd2_rn(a1, make_float2(s.z, s.w)));
    }
}

template <bool VEC>  // g_I rows in 16-byte units
__global__ void __launch_bounds__(THREADS, 1) gw_sums_kernel(const __grid_constant__ Args A) {
    if (__ldg(A.ws.flag + 1)) return;
    extern __shared__ __align__(128) unsigned char smem[];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int q = lane >> 3, l8 = lane & 7;
    const uint32_t gt = smem_u32(smem), sums = gt + GT_BYTES, lists = sums + sums_bytes(A.Nin);
    const int tile = blockIdx.x % A.tiles, range = blockIdx.x / A.tiles;
    const long long n0 = (long long)tile * NT;
    const long long first = A.units * range / A.ranges, last = A.units * (range + 1) / A.ranges;
    if (tid < 32) reinterpret_cast<float *>(smem + 16 * ZERO_ROW)[tid] = 0.0f;
    for (int k = tid; k < (A.Nin + 1) * (NT / 4); k += THREADS)
        reinterpret_cast<float4 *>(smem + GT_BYTES)[k] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    // staging: this thread holds steps 32 (warp % 16) + 4 l8 .. + 3 of rows 16 (warp / 16) + 4 m + q
    const int srow = 16 * (warp >> 4) + q, sstep = 32 * (warp & 15) + 4 * l8;
    float4 pv[4];
    float bsum[4] = {0.0f, 0.0f, 0.0f, 0.0f};
    long long lb = first / A.nch, lt = (first - lb * A.nch) * CH;  // the unit loaded next
    auto load = [&]() {
        const long long t = lt + sstep;
        const float *g = A.gI + (lb * A.N + n0 + srow) * A.T + t;
        lt += CH;
        if (lt >= A.T) {
            lt = 0;
            ++lb;
        }
#pragma unroll
        for (int m = 0; m < 4; ++m) {
            pv[m] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
            if (n0 + srow + 4 * m < A.N) {
                const float *p = g + 4LL * m * A.T;
                if (VEC) {
                    if (t < A.T) pv[m] = __ldg(reinterpret_cast<const float4 *>(p));
                } else {
                    if (t < A.T) pv[m].x = __ldg(p);
                    if (t + 1 < A.T) pv[m].y = __ldg(p + 1);
                    if (t + 2 < A.T) pv[m].z = __ldg(p + 2);
                    if (t + 3 < A.T) pv[m].w = __ldg(p + 3);
                }
            }
        }
    };
    auto fetch = [&](int half, long long u, uint32_t count) {
        const int bytes = HEAD + 16 * (int)(count >> 16);
        for (int o = 16 * tid; o < bytes; o += 16 * THREADS)
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(lists + half * A.rec + o),
                         "l"(A.ws.rec + u * A.rec + o)
                         : "memory");
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    uint32_t size = 0, count = 0;  // of this unit and the next
    if (first < last) {
        load();
        size = __ldg(A.ws.count + first);
        fetch(0, first, size);
        if (first + 1 < last) count = __ldg(A.ws.count + first + 1);
    }
    int half = 0;
    for (long long u = first; u < last; ++u, half ^= 1) {
        const uint32_t to = gt + 16 * row_of(sstep) + 4 * srow;
#pragma unroll
        for (int m = 0; m < 4; ++m) {
            const uint32_t a = to + 16 * m;
            asm volatile("st.shared.f32 [%0], %1;" ::"r"(a), "f"(pv[m].x) : "memory");
            asm volatile("st.shared.f32 [%0], %1;" ::"r"(a + 128), "f"(pv[m].y) : "memory");
            asm volatile("st.shared.f32 [%0], %1;" ::"r"(a + 256), "f"(pv[m].z) : "memory");
            asm volatile("st.shared.f32 [%0], %1;" ::"r"(a + 384), "f"(pv[m].w) : "memory");
            bsum[m] += (pv[m].x + pv[m].y) + (pv[m].z + pv[m].w);
        }
        const uint32_t count_now = count;
        if (u + 1 < last) {
            fetch(half ^ 1, u + 1, count);
            load();
            if (u + 2 < last) count = __ldg(A.ws.count + u + 2);
            asm volatile("cp.async.wait_group 1;" ::: "memory");
        } else {
            asm volatile("cp.async.wait_group 0;" ::: "memory");
        }
        __syncthreads();
        const uint32_t rec = lists + half * A.rec, gl = gt + 16 * l8;
        const int quads = (int)(size & 0xffffu);
        size = count_now;
        if (quads == (int)OVER) {
            walk_unit(A, u, gt, sums);
        } else if (warp < quads) {
            uint32_t at;
            asm volatile("ld.shared.u16 %0, [%1];" : "=r"(at) : "r"(rec + 2 * warp));
            const uint32_t row0 = rec + HEAD + 4 * q;
            at = row0 + 16 * at;
            uint32_t head = lds32(at), next;
            do {  // a group's sums and the next group's words are read ahead of their use
                uint32_t pr = lds32(at + 16);
                const uint32_t p = sums + (head & 2047u) * (NT * 4) + 16 * l8;
                const float4 s = lds128(p);
                int c = (int)(head >> 11) & 1023;
                next = head >> 21;
                head = lds32(row0 + 16 * next);
                float2 a0 = make_float2(0.0f, 0.0f), a1 = a0;
#pragma unroll 1
                for (; c >= 2; c -= 2) {
                    const float4 x = lds128(gl + (pr & 0xffffu) * 16u), y = lds128(gl + (pr >> 16) * 16u);
                    at += 16;
                    pr = lds32(at + 16);  // past the last: unused
                    a0 = __fadd2_rn(__fadd2_rn(a0, make_float2(x.x, x.y)), make_float2(y.x, y.y));
                    a1 = __fadd2_rn(__fadd2_rn(a1, make_float2(x.z, x.w)), make_float2(y.z, y.w));
                }
                if (c) {
                    const float4 x = lds128(gl + (pr & 0xffffu) * 16u);
                    a0 = __fadd2_rn(a0, make_float2(x.x, x.y));
                    a1 = __fadd2_rn(a1, make_float2(x.z, x.w));
                }
                sts128(p, __fadd2_rn(a0, make_float2(s.x, s.y)), __fadd2_rn(a1, make_float2(s.z, s.w)));
                at = row0 + 16 * next;
            } while (next);
        }
        __syncthreads();  // the staged chunk and this list are free
    }
    __syncthreads();
    float4 *part = reinterpret_cast<float4 *>(A.ws.part + ((long long)range * A.tiles + tile) * A.Nin * NT);
    for (int k = tid; k < A.Nin * (NT / 4); k += THREADS) part[k] = reinterpret_cast<const float4 *>(smem + GT_BYTES)[k];
    float *bs = reinterpret_cast<float *>(smem);  // [16 step blocks][32 rows]
#pragma unroll
    for (int m = 0; m < 4; ++m) {
        float s = bsum[m];
#pragma unroll
        for (int l = 1; l < 8; l <<= 1) s += __shfl_xor_sync(FULL, s, l);
        if (l8 == 0) bs[(warp & 15) * NT + srow + 4 * m] = s;
    }
    __syncthreads();
    if (tid < NT) {
        float s = 0.0f;
#pragma unroll
        for (int w = 0; w < 16; ++w) s += bs[w * NT + tid];
        A.ws.part_b[((long long)range * A.tiles + tile) * NT + tid] = s;
    }
}

// g_W[i][j] and g_bias[i]: the ranges' sums in order.  32 inputs x 32 neurons per block; the neurons' tiles, of which
// there may be more than 65535, in blockIdx.x.
__global__ void __launch_bounds__(1024) gw_join_kernel(long long N, int Nin, int tiles, int ranges, const Work ws, float *gW,
                                                      float *gb) {
    if (__ldg(ws.flag + 1)) return;
    __shared__ float out[NT][33];
    const int x = threadIdx.x, y = threadIdx.y, j0 = blockIdx.y * 32, tile = blockIdx.x;
    const long long stride = (long long)tiles * Nin * NT;
    if (gW) {
        float s = 0.0f;
        if (j0 + y < Nin) {
            const float *p = ws.part + ((long long)tile * Nin + j0 + y) * NT + x;
#pragma unroll 8
            for (int r = 0; r < ranges; ++r) s += p[r * stride];
        }
        out[x][y] = s;
        __syncthreads();
        const long long i = (long long)tile * NT + y;
        if (i < N && j0 + x < Nin) gW[i * Nin + j0 + x] = out[y][x];
    }
    if (gb && blockIdx.y == 0 && y == 0) {
        const long long i = (long long)tile * NT + x;
        float s = 0.0f;
        for (int r = 0; r < ranges; ++r) s += ws.part_b[((long long)r * tiles + tile) * NT + x];
        if (i < N) gb[i] = s;
    }
}

// Active inputs per step above which a raster is left to the other kernel (its events would not fit the records).
inline float active_limit(int Nin) { return 7.0f * ((float)rows_of(Nin) - Nin / 4.0f) / CH; }

inline int sm_count() {
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
        return 0;
    return sms;
}

}  // namespace gwl

int launch_density_sample(const uint32_t *S, long long rows, long long Nin, long long T, float limit, uint32_t *flags,
                          cudaStream_t st);

// Workspace bytes of the list path; 0 where it is not used.
size_t syn_grad_weights_ws(long long B, long long Nin, long long N, long long T) {
    using namespace gwl;
    if (B <= 0 || Nin <= 0 || N <= 0 || T <= 0 || Nin > MAX_NIN) return 0;
    // Five launches and the lists cost about 35 us: at 8 x 1000 -> 256 x 2000 (4e9 products) 55 against
    // 41 us, at 128 x 256 -> 256 x 1000 (8e9) 77 to 113 against 142 to 285, at 1 x 512 -> 2000 x 16384 (2e10)
    // 103 against 129.  Many inputs at high rates do not fit the lists; there the other kernel's call
    // becomes 20 us longer, so it has to be a long one.
    // The other kernel walks a batch element's 512-step chunks in series, a CTA for 16 neurons and 1024
    // inputs, so its time goes with waves of CTAs x chunks (3 to 6 us each); from 12 of those the lists pay
    // whatever the product (us, that / this): 22 x 113 -> 270 x 7500 (3 x 15) 144 / 91, 30 x 64 -> 600 x 4000
    // (8 x 8) 232 / 99, 1 x 512 -> 200 x 16000 (1 x 32) 138 / 52, 17 x 700 -> 276 x 3900 at 21 active inputs a
    // step (3 x 8) 310 / 142; not for 12 x 512 -> 289 x 2393 (2 x 5) 58 / 60 or 4 x 1000 -> 1024 x 1500
    // (2 x 3) 66 / 79.  Where a raster of 3.5 % activity would not fit the lists, from 36.
    const int sms = sm_count();
    if (!sms) return 0;
    const double ctas = (double)B * (double)((N + 15) / 16) * (double)((Nin + 1023) / 1024);
    const double least = active_limit((int)Nin) >= 0.035f * (float)Nin ? 12.0 : 36.0;
    // Of few neurons the building of the lists is a large part of the work, so the two paths' times are set against each
    // other as well (us; a wave of the other kernel 9 and 5 per chunk; here 30, for 1024 steps of a batch element
    // 0.02 + 0.12 per 1000 inputs, for a unit 2 + 2.3): N, that / this as measured 12 60 / 80, 16 95 / 115, 10 104 / 113,
    // 32 53 / 64, 64 66 / 74 are left to it, and 4 98 / 89, 8 87 / 69, 15 142 / 100, 24 114 / 100, 60 80 / 72 not.
    const double waves = std::ceil(ctas / sms), chunks = (double)((T + 511) / 512);
    const double that = waves * (9.0 + 5.0 * chunks);
    const double here = 30.0 + (double)B * (double)((T + 1023) / 1024) * (0.02 + 0.00012 * (double)Nin) +
                        std::ceil((double)B * chunks * (double)((N + NT - 1) / NT) / sms) * (2.0 + 0.0023 * (double)Nin);
    const bool many = waves * chunks >= least && that >= 1.03 * here;
    const double wide = Nin > 350 ? Nin / 350.0 : 1.0;
    if (!many && (double)B * (double)Nin * (double)N * (double)T < 8e9 * wide) return 0;
    const long long units = B * ((T + CH - 1) / CH), tiles = (N + NT - 1) / NT;
    if (units > (1LL << 24) || tiles > (1LL << 20)) return 0;
    return layout(units, tiles, ranges_for(tiles, units, sms), (int)Nin, nullptr, nullptr);
}

// g_W and g_bias of a sparse raster; *flags (device): flags[1] set where it is too dense for the
// lists: then nothing was written, and the caller's other kernel has to run.
int launch_syn_grad_weights(long long B, long long Nin, long long N, long long T, const uint32_t *S, const float *gI,
                            float *gW, float *gb, void *work, const uint32_t **flags, cudaStream_t st) {
    using namespace gwl;
    const long long nwin = (T + 31) / 32, nch = (T + CH - 1) / CH;
    Args A{N, T, nch, B * nch, (int)Nin, (int)((N + NT - 1) / NT), 1, rec_of((int)Nin), gI, S, {}};
    const int sms = sm_count();
    if (!sms) return (int)cudaErrorInvalidDevice;
    A.ranges = ranges_for(A.tiles, A.units, sms);
    layout(A.units, A.tiles, A.ranges, (int)Nin, work, &A.ws);
    *flags = A.ws.flag;
    int rc = launch_density_sample(S, B * Nin, Nin, T, active_limit((int)Nin), A.ws.flag, st);
    if (rc) return rc;
    cudaError_t e = cudaFuncSetAttribute(gw_lists_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 2 * (HEAD + 16 * MAX_ROWS));
    if (e != cudaSuccess) return (int)e;
    gw_lists_kernel<<<(unsigned)(B * ((nwin + 31) / 32)), 1024, lists_smem((int)Nin), st>>>((int)Nin, T, nwin, nch, S, A.ws);
    e = cudaGetLastError();
    if (e != cudaSuccess) return (int)e;
    const auto sums = T % 4 == 0 && reinterpret_cast<uintptr_t>(gI) % 16 == 0 ? gw_sums_kernel<true> : gw_sums_kernel<false>;
    e = cudaFuncSetAttribute(sums, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM);
    if (e != cudaSuccess) return (int)e;
    sums<<<(unsigned)(A.tiles * A.ranges), THREADS, smem_of((int)Nin), st>>>(A);
    e = cudaGetLastError();
    if (e != cudaSuccess) return (int)e;
    gw_join_kernel<<<dim3((unsigned)A.tiles, (unsigned)((Nin + 31) / 32)), dim3(32, 32), 0, st>>>(N, (int)Nin, A.tiles,
                                                                                              A.ranges, A.ws, gW, gb);
    return (int)cudaGetLastError();
}

}  // namespace alif

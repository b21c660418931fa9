// Recurrent ALIF layer with transmission latency D = T_R (sm_103a).
//
// Section 2 lets the input current of Eq 3 carry a recurrent term
// sum_j W_rec[i][j] S_j[t - D] and assumes the latency D equals the ARP, T_R.
// Prop 3 is what makes that useful: the recurrent current of Block n+1 is
// fixed by the spikes of Block n, so a whole population advances T_R steps
// between two exchanges of spikes instead of one.
//
// One batch element is one thread-block cluster of G CTAs (G <= 8), each CTA
// owning up to 1024 consecutive neurons, one thread per neuron.  Per Block of
// T_R steps:
//   1. after a cluster barrier, every CTA reads the previous Block's spikes of
//      all N neurons from the G CTAs' shared memory (distributed shared
//      memory) -- at most one spike per neuron and Block, since the ARP
//      (T_eff = max(T_R, 2) >= T_R) allows no second one -- and lists them;
//   2. the weights W_rec[i][j] of the listed spikes are copied into shared memory together
//      (cp.async, one round trip for up to WCH spikes; W_rec is stored transposed, so a warp reads
//      128 contiguous bytes per spike) while the spikes are sorted by step; spikes beyond WCH are
//      added into the Block's currents beforehand, WCH at a time;
//   3. each thread steps its neuron through the Block (Eqs 1-5, state form): the total current of a
//      step, I_ff plus the weights of the step's spikes, V and a in double-single, so that every
//      spike decision is the one exact arithmetic takes (a flip needs a margin near 1e-12).  At most
//      one spike falls into a Block, so the spike's effects and the rare margins that FP32 cannot
//      decide stand under branches, and the spike word is written once per Block.  It publishes the
//      step of its spike (or none) for the next Block.
// The Block's currents are kept neuron-major, so that they move as 16-byte units (VW steps) between
// global memory, shared memory and registers; those of Block n+1 are copied into a second buffer
// while Block n is resolved.
// What bounds it: the latency of each Block's chain (cluster barrier 1.7k cycles, gather and list 1.1k,
// weights 2k, the sums of the weights 3k, the double-single steps 2.5k at N = 1024, T_R = 20 and 27
// spikes a Block) with one or two warps per scheduler.  B = 32, N = 1024, T = 4000: 1.20 ms (1.97 ms with
// a shared double-single accumulator per step, single-float copies and every step under its own
// branches).  Helper warps for the sums and the stores: 1.45 ms, their instructions compete with the
// steps'.
// The total current I_ff + I_rec, rounded to FP32, is written out for the backward, with the
// spike words, the checkpoints every ALIF_CKPT_STEPS steps and the final state
// in the layouts of alif_forward.  Every CTA of a cluster runs the same number
// of cluster barriers, and the last one keeps every CTA's shared memory alive
// until no other CTA reads it.
#include <cooperative_groups.h>

#include "common.cuh"

namespace cg = cooperative_groups;

namespace alif {
namespace rec {

constexpr int MAX_G = 8;           // portable cluster size
constexpr int MAX_PER = 1024;      // neurons per CTA
constexpr int NO_SPIKE = -1;
constexpr int MAX_WCH = 128;       // recurrent weights copied together
constexpr uint32_t NO_STEP = 1023;  // step of the entries past the last spike (T_R <= 1023)

struct Args {
    long long B, N, T, nwords, nckpt;
    int TR, G, per;
    int nbuf;  // 2: the next Block's current is prefetched into a second accumulator
    int wch;   // spikes whose weights are copied into shared memory together
    int P;     // floats per neuron of a current buffer
    int wide;  // 1: rows of W keep 16 bytes
    const float *Iff;
    const float *Wt;  // [N pre, N post]
    const AlifNeuron *nrn;
    const AlifState *init;
    float *Iout;
    uint32_t *spikes;
    AlifState *ckpt, *fin;
};

// Floats per neuron of a current buffer: an odd number of VW-float units, at least T_R, so that 32
// neurons' units fall in distinct banks.
constexpr int pitch_of(int TR, int VW) { return (((TR + VW - 1) / VW) | 1) * VW; }

// cur [nbuf][per][P] currents, acl [per][P] their low parts where weights were added beforehand,
// wbuf [wch][per] weights; spk [2][per]; list [N]; sorted [wch + 4]; wsum [32]
inline size_t smem_bytes(const Args &A) {
    return (size_t)(A.nbuf + 1) * A.per * A.P * 4 + (size_t)A.wch * A.per * 4 + (size_t)2 * A.per * 4 + (size_t)A.N * 4 +
           (A.wch + 4) * 4 + 32 * 4;
}

// 4-byte asynchronous global -> shared copy (completion tracked by cp.async groups)
__device__ __forceinline__ void cp_async4(float *dst, const float *src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}
// the same for VW floats
template <int VW>
__device__ __forceinline__ void cp_async_vec(float *dst, const float *src) {
    if constexpr (VW == 4)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
    else if constexpr (VW == 2)
        asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
    else
        cp_async4(dst, src);
}
template <int VW>
struct alignas(4 * VW) Vec {
    float v[VW];
};
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// the aligned forms want a warp's threads together, which come out of branches of their own (spikes, live neurons)
__device__ __forceinline__ void cluster_arrive() {
    __syncwarp();
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_wait() {
    __syncwarp();
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// Sums of a chunk's weights, sorted by step, into a neuron's currents: event k's weight is w0, the next one's w1, ev2 the
// entry after.
template <int VW>
struct Events {
    const float *wcol;
    const uint32_t *p;
    int per;
    uint32_t ev0, ev1, ev2;
    float w0, w1;
    __device__ __forceinline__ void start(const float *w, const uint32_t *sorted, int n) {
        wcol = w;
        per = n;
        ev0 = sorted[0];
        ev1 = sorted[1];
        ev2 = sorted[2];
        p = sorted + 3;
        w0 = wcol[(ev0 >> 10) * per];
        w1 = wcol[(ev1 >> 10) * per];
    }
    __device__ __forceinline__ void add(int u, Vec<VW> &I, Vec<VW> &lo) {  // steps u .. u + VW - 1
#pragma unroll
        for (int s = 0; s < VW; ++s)
            while ((int)(ev0 & 1023u) == u + s) {  // the same spikes in every thread of the CTA
                const df s2 = two_sum(I.v[s], w0);
                I.v[s] = s2.hi;
                lo.v[s] += s2.lo;
                ev0 = ev1;
                w0 = w1;
                ev1 = ev2;
                w1 = wcol[(ev1 >> 10) * per];
                ev2 = *p++;  // at most the fourth entry past the last spike's
            }
    }
};

// MAXT, MINB: the CTA size and the CTAs per SM the register budget is sized for (256, 1: up to 255
// registers a thread, for clusters of at most 256 neurons per CTA; 256, 2: up to 128).  VW: floats per unit of
// the currents.
template <int MAXT, int MINB, int VW>
__global__ void __launch_bounds__(MAXT, MINB) rec_fwd_kernel(const Args A) {
    cg::cluster_group cl = cg::this_cluster();
    extern __shared__ __align__(16) unsigned char smem[];
    const int per = A.per, TR = A.TR, G = A.G, nbuf = A.nbuf, wch = A.wch;
    const int P = A.P;
    float *bufs = reinterpret_cast<float *>(smem);                                  // [nbuf][per][P]
    float *acl = bufs + (size_t)nbuf * per * P;                                      // [per][P]
    float *wbuf = acl + (size_t)per * P;                                             // [wch][per]
    int *spk = reinterpret_cast<int *>(wbuf + (size_t)wch * per);                    // [2][per]
    uint32_t *list = reinterpret_cast<uint32_t *>(spk + 2 * per);                    // [N] (j << 10) | t
    uint32_t *sorted = list + A.N;                                                   // (slot << 10) | t by step
    int *wsum = reinterpret_cast<int *>(sorted + wch + 4);                           // [32] warps' counts
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nwarps = (per + 31) >> 5;
    const int rank = (int)cl.block_rank();
    const long long b = blockIdx.x / G;
    const long long i = (long long)rank * per + tid;
    const bool live = i < A.N;
    const long long row = b * A.N + (live ? i : 0);

    AlifNeuron nr{};
    if (live) nr = A.nrn[i];
    const df beta{nr.beta_hi, nr.beta_lo}, p{nr.p_hi, nr.p_lo}, c{nr.c_hi, nr.c_lo};
    const float d = nr.d, th0 = nr.theta0;
    df v{0.0f, 0.0f}, a{0.0f, 0.0f};
    int adm = 0;  // first step of the Block that admits input (Eq 4)
    if (live && A.init) {
        const AlifState s = A.init[row];
        adm = s.rem > 0 ? s.rem : 0;
        v = df{adm > 0 ? 0.0f : s.v, 0.0f};
        a = df{s.a, 0.0f};
    }
    uint32_t word = 0;  // the spike word that holds the next step, so far
    uint32_t *spikes = A.spikes + row * A.nwords;
    const long long nb = (A.T + TR - 1) / TR;
    // A warp moves its 32 neurons' Block chunks (contiguous in global memory) unit by unit: unit
    // e = 32 j + lane of the chunk is unit e % nu of neuron e / nu, the quotient and remainder advancing
    // by those of 32 / nu.
    const long long wrow = (long long)rank * per + warp * 32;  // this warp's first neuron
    const int nrow = (int)(A.N - wrow < 32 ? A.N - wrow : 32);
    const long long grow0 = b * A.N + wrow;
    const int nu_full = TR / VW > 0 ? TR / VW : 1, q_full = 32 / nu_full, r_full = 32 - q_full * nu_full;
    const int r0_full = lane / nu_full, u0_full = lane - r0_full * nu_full;
    auto units = [&](int nu, auto move) {
        int q32 = q_full, r32 = r_full, r = r0_full, u = u0_full;
        if (nu != nu_full) {  // the last Block
            q32 = 32 / nu;
            r32 = 32 - q32 * nu;
            r = lane / nu;
            u = lane - r * nu;
        }
        for (int e = lane; e < 32 * nu; e += 32) {
            if (r < nrow) move(r, u * VW);
            r += q32;
            u += r32;
            if (u >= nu) {
                u -= nu;
                ++r;
            }
        }
    };
    auto steps_of = [&](long long m) { return (int)(A.T - m * TR < TR ? A.T - m * TR : TR); };
    auto buffer = [&](long long m) { return bufs + (size_t)(nbuf == 2 ? (int)(m & 1) : 0) * per * P; };
    auto load_ff = [&](long long m) {  // feedforward current of Block m (cp.async)
        float *dst = buffer(m) + warp * 32 * P;
        const float *src = A.Iff + grow0 * A.T + m * TR;
        units(steps_of(m) / VW, [&](int r, int t) { cp_async_vec<VW>(dst + r * P + t, src + (long long)r * A.T + t); });
    };
    for (int t = 0; t < P; ++t) acl[tid * P + t] = 0.0f;
    const int wk = tid / (per / 4), wcol4 = 4 * (tid - wk * (per / 4));  // this thread's part of the weight copies
    const long long wq = (long long)rank * per + wcol4;
    load_ff(0);
    cp_async_commit();
    for (long long n = 0; n < nb; ++n) {
        const long long t0 = n * TR;
        const int cnt = steps_of(n);
        // ---- 1. spikes of Block n-1 from every CTA of the cluster, listed as (j, t)
        int total = 0;
        if (n > 0) {
            cluster_wait();  // every CTA has published spk[(n-1) & 1]
            const int par = (int)((n - 1) & 1);
            int ts[MAX_G];
            int mine = 0;
#pragma unroll
            for (int r = 0; r < MAX_G; ++r) {
                ts[r] = NO_SPIKE;
                if (r < G && (long long)r * per + tid < A.N) {
                    const int *remote = cl.map_shared_rank(spk + par * per, r);
                    ts[r] = remote[tid];
                }
                mine += ts[r] != NO_SPIKE;
            }
            int incl = mine;
#pragma unroll
            for (int l = 1; l < 32; l <<= 1) {
                const int up = __shfl_up_sync(FULL, incl, l);
                if (lane >= l) incl += up;
            }
            if (lane == 31) wsum[warp] = incl;
            __syncthreads();
            int upto = lane < nwarps ? wsum[lane] : 0;  // spikes of the warps up to this lane's
#pragma unroll
            for (int l = 1; l < 32; l <<= 1) {
                const int up = __shfl_up_sync(FULL, upto, l);
                if (lane >= l) upto += up;
            }
            total = __shfl_sync(FULL, upto, 31);
            const int before = warp ? __shfl_sync(FULL, upto, warp - 1) : 0;
            int pos = before + incl - mine;
#pragma unroll
            for (int r = 0; r < MAX_G; ++r)
                if (ts[r] != NO_SPIKE) list[pos++] = ((uint32_t)(r * per + tid) << 10) | (uint32_t)ts[r];
            __syncthreads();
        }
        float *cur = buffer(n);
        if (nbuf == 1 && n > 0) {
            load_ff(n);
            cp_async_commit();
        }
        // ---- 2. weights.  cp.async groups complete in commit order: waiting for all but the newest
        // leaves only the next Block's current in flight.  total and nch are the CTA's.
        auto copy_weights = [&](int e0, int nch) {
            if (A.wide) {  // 16 bytes of four neurons each, four spikes at a time
                if (wq < A.N)
                    for (int k = wk; k < nch; k += 4)
                        cp_async_vec<4>(wbuf + k * per + wcol4, A.Wt + (long long)(list[e0 + k] >> 10) * A.N + wq);
            } else if (live) {
#pragma unroll 4
                for (int k = 0; k < nch; ++k)
                    cp_async4(wbuf + k * per + tid, A.Wt + (long long)(list[e0 + k] >> 10) * A.N + i);
            }
            cp_async_commit();
        };
        auto sort_chunk = [&](int e0, int nch) {  // by step, and within one in the order of the list
            for (int e = tid; e < nch; e += per) {
                const uint32_t mine = (list[e0 + e] & 1023u) << 7 | (uint32_t)e;
                int at = 0;
#pragma unroll 8
                for (int o = 0; o < nch; ++o) at += ((list[e0 + o] & 1023u) << 7 | (uint32_t)o) < mine;
                sorted[at] = (uint32_t)e << 10 | mine >> 7;
            }
            if (tid < 4) sorted[nch + tid] = NO_STEP;
        };
        int e0 = 0;
        const bool multi = total > wch;
        // More spikes than weight slots: all but the last few are added into the buffers beforehand.  Of up to 256 neurons
        // a CTA each spike by itself; above, where the step's places of a warp's neurons meet in eight banks, a chunk
        // sorted and summed like the last one (2 x 4096 x 400 steps at 130 spikes a Block 537 -> 383 us; 16 x 2000 x 500
        // at 78 432 against 405, but 32 x 1024 x 1000 at T_R = 60 322 against 341, and 2 % on T_R = 2 and 10 without any
        // such chunk).
        for (; total - e0 > wch; e0 += wch) {
            copy_weights(e0, wch);
            if constexpr (MAXT > 256) sort_chunk(e0, wch);
            cp_async_wait<0>();
            __syncthreads();
            if (live) {
                if constexpr (MAXT > 256) {
                    float *mycur = cur + tid * P, *mylo = acl + tid * P;
                    Events<VW> ev;
                    ev.start(wbuf + tid, sorted, per);
                    for (int u = 0; u < cnt; u += VW) {
                        if ((int)(ev.ev0 & 1023u) >= u + VW) continue;
                        Vec<VW> I = *reinterpret_cast<const Vec<VW> *>(mycur + u), lo = *reinterpret_cast<const Vec<VW> *>(mylo + u);
                        ev.add(u, I, lo);
                        *reinterpret_cast<Vec<VW> *>(mycur + u) = I;
                        *reinterpret_cast<Vec<VW> *>(mylo + u) = lo;
                    }
                } else {
                    for (int k = 0; k < wch; ++k) {
                        const int at = tid * P + (int)(list[e0 + k] & 1023u);
                        const df s2 = two_sum(cur[at], wbuf[(size_t)k * per + tid]);
                        cur[at] = s2.hi;
                        acl[at] += s2.lo;
                    }
                }
            }
            __syncthreads();
        }
        const int nch = total - e0;
        copy_weights(e0, nch);
        const bool pref = nbuf == 2 && n + 1 < nb;
        if (pref) {
            load_ff(n + 1);
            cp_async_commit();
        }
        sort_chunk(e0, nch);
        if (pref)
            cp_async_wait<1>();
        else
            cp_async_wait<0>();
        __syncthreads();
        // ---- 3. the Block's steps, VW at a time
        int sp = NO_SPIKE;
        if (live) {
            const float *wcol = wbuf + tid;
            // event k's weight is w0, the next one's w1, ev2 the entry after
            uint32_t ev0 = sorted[0], ev1 = sorted[1], ev2 = sorted[2];
            float w0 = wcol[(ev0 >> 10) * per], w1 = wcol[(ev1 >> 10) * per];
            const uint32_t *evp = sorted + 3;
            const int tck = A.ckpt ? (int)((ALIF_CKPT_STEPS - (t0 & (ALIF_CKPT_STEPS - 1))) & (ALIF_CKPT_STEPS - 1)) : TR;
            float *mycur = cur + tid * P, *mylo = acl + tid * P;
            int ck = tck;  // next step of the Block whose entering state is a checkpoint
            for (int u = 0; u < cnt; u += VW) {
                Vec<VW> I = *reinterpret_cast<const Vec<VW> *>(mycur + u), lo{};
                if (multi) {
                    lo = *reinterpret_cast<const Vec<VW> *>(mylo + u);
                    *reinterpret_cast<Vec<VW> *>(mylo + u) = Vec<VW>{};
                }
#pragma unroll
                for (int s = 0; s < VW; ++s)
                    while ((int)(ev0 & 1023u) == u + s) {  // the same spikes in every thread of the CTA
                        const df s2 = two_sum(I.v[s], w0);
                        I.v[s] = s2.hi;
                        lo.v[s] += s2.lo;
                        ev0 = ev1;
                        w0 = w1;
                        ev1 = ev2;
                        w1 = wcol[(ev1 >> 10) * per];
                        ev2 = *evp++;  // at most the fourth entry past the last spike's
                    }
                df x[VW];  // c I m (Eqs 2, 4)
#pragma unroll
                for (int s = 0; s < VW; ++s) {
                    const df It = quick_two_sum(I.v[s], lo.v[s]);
                    I.v[s] = It.hi;  // the FP32 total current
                    x[s] = df_mul(c, It);
                    if (u + s < adm) x[s] = df{0.0f, 0.0f};
                }
                *reinterpret_cast<Vec<VW> *>(mycur + u) = I;
                auto checkpoint = [&](int t, df v, df a) {
                    AlifState st;
                    st.v = v.hi;
                    st.a = a.hi;
                    st.rem = adm > t ? adm - t : 0;
                    A.ckpt[row * A.nckpt + (t0 + t) / ALIF_CKPT_STEPS] = st;
                };
                // Eq 1 against theta = theta0 + d a (Eq 5).  The FP32 difference dz of V.hi and
                // fl(theta0 + d a.hi) is within 2^-24 (|dz| + |V.hi| + |theta| + |d a.hi|) of the
                // double-single margin, so outside 2^-21 (...) its sign is the margin's.
                if (ck >= u + VW || ck < u) {
                    // The unit's steps without a branch; a bit per step whose margin is not clearly
                    // negative.  Those are decided in order: a spike ends the Block for its neuron
                    // (T_eff >= T_R), the membrane is 0 from there on.
                    df vs[VW], as[VW];  // V of the step, a entering it
                    unsigned near = 0;
                    df vf = v, af = a;
#pragma unroll
                    for (int s = 0; s < VW; ++s) {
                        vf = df_axpy(beta, vf, x[s]);  // Eq 2, 4
                        vs[s] = vf;
                        as[s] = af;
                        const float thf = fmaf(d, af.hi, th0);
                        if (!(vf.hi - thf < -0x1p-21f * (fabsf(vf.hi) + fabsf(thf) + fabsf(d * af.hi)))) near |= 1u << s;
                        af = df_mul(p, af);  // Eq 5
                    }
                    while (near) {
                        const int s = __ffs(near) - 1;
                        near &= near - 1u;
                        df vt = vs[0], at = as[0];
#pragma unroll
                        for (int k = 1; k < VW; ++k)
                            if (k == s) {
                                vt = vs[k];
                                at = as[k];
                            }
                        const float thf = fmaf(d, at.hi, th0);
                        const float dz = vt.hi - thf;
                        bool S = dz > 0.0f;
                        if (!(fabsf(dz) > 0x1p-21f * (fabsf(vt.hi) + fabsf(thf) + fabsf(d * at.hi))))
                            S = df_cmp(vt, df_add(df{th0, 0.0f}, df_mul_f(at, d))) > 0;
                        if (S) {
                            af = df_add(df_mul(p, at), df{1.0f, 0.0f});
                            for (int k = s + 1; k < VW; ++k) af = df_mul(p, af);
                            vf = df{0.0f, 0.0f};
                            sp = u + s;
                            adm = sp + nr.teff;
                            break;
                        }
                    }
                    v = vf;
                    a = af;
                    continue;
                }
                // a unit with a checkpoint: step by step
#pragma unroll 1
                for (int s = 0; s < VW; ++s) {
                    const int t = u + s;
                    df xs = x[0];
#pragma unroll
                    for (int k = 1; k < VW; ++k)
                        if (k == s) xs = x[k];
                    if (t < adm) xs = df{0.0f, 0.0f};  // after a spike earlier in this unit
                    if (t == ck) {
                        checkpoint(t, v, a);
                        ck += ALIF_CKPT_STEPS;
                    }
                    v = df_axpy(beta, v, xs);  // Eq 2, 4
                    const float thf = fmaf(d, a.hi, th0);
                    const float dz = v.hi - thf;
                    bool S = dz > 0.0f;
                    if (!(fabsf(dz) > 0x1p-21f * (fabsf(v.hi) + fabsf(thf) + fabsf(d * a.hi)))) {
                        const df th = df_add(df{th0, 0.0f}, df_mul_f(a, d));
                        S = df_cmp(v, th) > 0;
                    }
                    a = df_mul(p, a);  // Eq 5
                    if (S) {
                        a = df_add(a, df{1.0f, 0.0f});
                        v = df{0.0f, 0.0f};
                        adm = t + nr.teff;
                        sp = t;
                    }
                }
            }
            adm = adm > cnt ? adm - cnt : 0;
            // the spike words that the Block completes
            const long long ks = t0 + sp;
            for (long long w = t0 >> 5; w < (t0 + cnt) >> 5; ++w) {
                spikes[w] = word | (sp != NO_SPIKE && (ks >> 5) == w ? 1u << (ks & 31) : 0u);
                word = 0;
            }
            if (sp != NO_SPIKE && (ks >> 5) == (t0 + cnt) >> 5) word |= 1u << (ks & 31);
        }
        spk[(n & 1) * per + tid] = sp;
        cluster_arrive();  // the current goes out while the others arrive
        if (A.Iout) {
            __syncwarp();
            float *dst = A.Iout + grow0 * A.T + t0;
            const float *src = cur + warp * 32 * P;
            units(cnt / VW, [&](int r, int t) {
                *reinterpret_cast<Vec<VW> *>(dst + (long long)r * A.T + t) = *reinterpret_cast<const Vec<VW> *>(src + r * P + t);
            });
        }
    }
    if (live && (A.T & 31)) spikes[A.T >> 5] = word;
    if (live && A.fin) {
        AlifState s;
        s.v = v.hi;
        s.a = a.hi;
        s.rem = adm;
        A.fin[row] = s;
    }
    cluster_wait();  // no CTA leaves while another may still read its shared memory
}

// Spike raster delayed by D steps: out bit t = in bit t - D (0 for t < D).
__global__ void delay_kernel(long long rows, long long nwords, long long T, long long D, const uint32_t *in,
                             uint32_t *out) {
    const long long total = rows * nwords;
    const long long wsh = D >> 5;
    const int bsh = (int)(D & 31);
    for (long long q = (long long)blockIdx.x * blockDim.x + threadIdx.x; q < total;
         q += (long long)gridDim.x * blockDim.x) {
        const long long r = q / nwords, k = q - r * nwords;
        const long long src = k - wsh;  // word holding bit 32 k - D
        const uint32_t *row = in + r * nwords;
        const uint32_t hi = src >= 0 ? row[src] : 0u;
        const uint32_t lo = (src - 1 >= 0 && bsh) ? row[src - 1] : 0u;
        uint32_t w = bsh ? ((hi << bsh) | (lo >> (32 - bsh))) : hi;
        if (k == nwords - 1 && (T & 31)) w &= (1u << (T & 31)) - 1u;
        out[q] = w;
    }
}

}  // namespace rec

// Returns 0 or a CUDA error code (> 0); -1 when the configuration does not fit.
int launch_alif_forward_recurrent(long long B, long long N, long long T, int TR, const float *Iff, const float *Wt,
                                  const AlifNeuron *nrn, const AlifState *init, float *Iout, uint32_t *spikes,
                                  AlifState *ckpt, AlifState *fin, cudaStream_t stream) {
    using namespace rec;
    Args A;
    A.B = B;
    A.N = N;
    A.T = T;
    A.nwords = (T + 31) / 32;
    A.nckpt = (T + ALIF_CKPT_STEPS - 1) / ALIF_CKPT_STEPS;
    A.TR = TR;
    int G = (int)((N + 127) / 128);
    if (G > MAX_G) G = MAX_G;
    if (G < 1) G = 1;
    int per = (int)((N + G - 1) / G);
    per = (per + 31) & ~31;
    if (per > MAX_PER) return -1;
    A.G = G;
    A.per = per;
    A.Iff = Iff;
    A.Wt = Wt;
    A.nrn = nrn;
    A.init = init;
    A.Iout = Iout;
    A.spikes = spikes;
    A.ckpt = ckpt;
    A.fin = fin;
    int dev = 0, optin = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return (int)e;
    e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    if (e != cudaSuccess) return (int)e;
    A.wide = N % 4 == 0 && reinterpret_cast<uintptr_t>(Wt) % 16 == 0;
    // steps per unit of the currents: 16 or 8 bytes where rows and Blocks keep them
    const uintptr_t pa = reinterpret_cast<uintptr_t>(Iff) | (Iout ? reinterpret_cast<uintptr_t>(Iout) : 0);
    int vw = (T % 4 == 0 && TR % 4 == 0 && pa % 16 == 0) ? 4 : (T % 2 == 0 && TR % 2 == 0 && pa % 8 == 0) ? 2 : 1;
    // The largest configuration that fits: both current buffers first, then as many weights per copy
    // as possible; last, single steps in rows without padding.
    A.nbuf = 0;
    auto fits = [&](int v, int pitch, int nbuf, int wch) {
        A.P = pitch;
        A.wch = wch;
        A.nbuf = nbuf;
        if (smem_bytes(A) > (size_t)optin) A.nbuf = 0;
        vw = v;
        return A.nbuf != 0;
    };
    bool found = false;
    for (int nbuf = 2; nbuf >= 1 && !found; --nbuf)
        for (int wch = MAX_WCH; wch >= 4 && !found; wch /= 2) found = fits(vw, pitch_of(TR, vw), nbuf, wch);
    if (!found && !fits(1, TR, 1, 4)) return -1;
    using Kernel = void (*)(Args);
    const auto kernel = [&](bool pairs) -> Kernel {
        if (per > 256) return vw == 4 ? rec_fwd_kernel<MAX_PER, 1, 4> : vw == 2 ? rec_fwd_kernel<MAX_PER, 1, 2> : rec_fwd_kernel<MAX_PER, 1, 1>;
        if (pairs) return vw == 4 ? rec_fwd_kernel<256, 2, 4> : vw == 2 ? rec_fwd_kernel<256, 2, 2> : rec_fwd_kernel<256, 2, 1>;
        return vw == 4 ? rec_fwd_kernel<256, 1, 4> : vw == 2 ? rec_fwd_kernel<256, 1, 2> : rec_fwd_kernel<256, 1, 1>;
    };
    Kernel kern = kernel(false);
    int sms = 0;
    e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return (int)e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(B * G), 1, 1);
    cfg.blockDim = dim3((unsigned)per, 1, 1);
    cfg.dynamicSmemBytes = smem_bytes(A);
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)G;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if (2 * B * G > sms) {
        // More clusters than may fit at a time with a CTA per SM: a wave less is worth more than slots (32 x 1024 x 1000
        // at T_R = 60: 64 slots, a CTA per SM, 779 us; 32 slots, two, 322) and than registers (of more than 192 neurons a
        // CTA two need 128 a thread: 32 x 2000 x 300 at T_R = 20 232 us with one, 125 with two).
        long long least = 0;
        int slots = 0;
        bool two = false;
        const int most = A.wch;
        for (int pairs = 0; pairs <= (per > 192 && per <= 256) && least != 1; ++pairs) {
            e = cudaFuncSetAttribute(kernel(pairs), cudaFuncAttributeMaxDynamicSharedMemorySize, optin);
            if (e != cudaSuccess) return (int)e;
            for (int wch = most; wch >= (most < 32 ? most : 32) && least != 1; wch /= 2) {
                fits(vw, A.P, A.nbuf, wch);
                cfg.dynamicSmemBytes = smem_bytes(A);
                int n = 0;
                e = cudaOccupancyMaxActiveClusters(&n, kernel(pairs), &cfg);
                if (e != cudaSuccess) return (int)e;
                const long long waves = (B + n - 1) / (n > 0 ? n : 1);
                if (least == 0 || waves < least) {
                    least = waves;
                    slots = wch;
                    two = pairs;
                }
            }
        }
        fits(vw, A.P, A.nbuf, slots);
        cfg.dynamicSmemBytes = smem_bytes(A);
        kern = kernel(two);
    }
    e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, optin);  // one value for all threads
    if (e != cudaSuccess) return (int)e;
    e = cudaLaunchKernelEx(&cfg, kern, A);
    return (int)e;
}

int launch_delay_spikes(long long rows, long long T, long long D, const uint32_t *in, uint32_t *out,
                        cudaStream_t stream) {
    const long long nwords = (T + 31) / 32;
    const long long total = rows * nwords;
    if (total == 0) return 0;
    long long blocks = (total + 255) / 256;
    if (blocks > 65535LL * 8) blocks = 65535LL * 8;
    rec::delay_kernel<<<(unsigned)blocks, 256, 0, stream>>>(rows, nwords, T, D, in, out);
    return (int)cudaGetLastError();
}

}  // namespace alif

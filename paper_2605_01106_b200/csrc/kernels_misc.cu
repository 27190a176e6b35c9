// Small kernels of the round: token embedding gather, greedy argmax with top-2 margin, and the
// accept / rollback step (paper Sec. 3.3, greedy rule).
#include "hs_internal.h"
#include "hs_device.cuh"
#include <mutex>

bool g_hs_pdl = true;

namespace {
using namespace hsd;

// h[row(b,i)][:] = E[cand[b][col0 + i]].  A token id outside [0, V) (a caller's candidate buffer, a forced
// next token) is never used as an address: the row of token 0 is gathered instead and the status word is set.
__global__ void embed_kernel(const __nv_bfloat16 *E, int d, int V, const int32_t *cand, int Tm, int col0, int T,
                             int b0, float *h, int32_t *status) {
    const int i = blockIdx.x, lb = blockIdx.y, b = b0 + lb;
    pdl_trigger();
    pdl_wait();
    int tok = __ldcg(cand + b * Tm + col0 + i);
    if (tok < 0 || tok >= V) {
        if (threadIdx.x == 0) atomicCAS(status, 0, (int)HS_ERR_DEVICE);
        tok = 0;
    }
    const uint4 *src = reinterpret_cast<const uint4 *>(E + (size_t)tok * d);
    float *dst = h + (size_t)(lb * T + i) * d;
    for (int c = threadIdx.x; c < d / 8; c += blockDim.x) {
        uint4 w = src[c];
        float4 lo = make_float4(__uint_as_float(w.x << 16), __uint_as_float(w.x & 0xffff0000u),
                                __uint_as_float(w.y << 16), __uint_as_float(w.y & 0xffff0000u));
        float4 hi = make_float4(__uint_as_float(w.z << 16), __uint_as_float(w.z & 0xffff0000u),
                                __uint_as_float(w.w << 16), __uint_as_float(w.w & 0xffff0000u));
        reinterpret_cast<float4 *>(dst)[2 * c] = lo;
        reinterpret_cast<float4 *>(dst)[2 * c + 1] = hi;
    }
}

struct Top2 { float v1; int i1; float v2; };

__device__ __forceinline__ Top2 top2_merge(const Top2 &a, const Top2 &b) {
    // lowest index wins a tie for first place; an equal runner-up makes the margin zero
    Top2 r;
    if (a.v1 > b.v1 || (a.v1 == b.v1 && a.i1 < b.i1)) { r.v1 = a.v1; r.i1 = a.i1; r.v2 = fmaxf(a.v2, b.v1); }
    else { r.v1 = b.v1; r.i1 = b.i1; r.v2 = fmaxf(b.v2, a.v1); }
    return r;
}

// Greedy argmax with top-2 margin over V logits per row, split over HS_ARGMAX_CHUNKS CTAs per row.
// grid = (chunks, T, nb).  A CTA scans its slice (lowest id wins a tie), writes a partial
// (top value, its id, runner-up) to scratch and takes a ticket; the CTA that arrives last merges the
// row's partials - the merge is order-independent, so the result is reproducible - writes the token
// and the margin and puts the ticket counter back to zero for the next launch.
struct ArgmaxArgs {
    const float *logits; int V, T, b0, Tm;
    int32_t *tok_out; int tok_col0; float *margin_out;
    float4 *part;            // scratch [rows][HS_ARGMAX_CHUNKS]
    int32_t *counters;       // scratch [rows], zero between launches
};

__device__ __forceinline__ Top2 top2_warp(Top2 t) {
#pragma unroll
    for (int o = 16; o >= 1; o >>= 1) {
        Top2 u;
        u.v1 = __shfl_xor_sync(0xffffffffu, t.v1, o);
        u.i1 = __shfl_xor_sync(0xffffffffu, t.i1, o);
        u.v2 = __shfl_xor_sync(0xffffffffu, t.v2, o);
        t = top2_merge(t, u);
    }
    return t;
}

__global__ void __launch_bounds__(256) argmax_kernel(const ArgmaxArgs a) {
    const int chunk = blockIdx.x, i = blockIdx.y, lb = blockIdx.z, b = a.b0 + lb;
    const int nchunk = gridDim.x;
    const float *row = a.logits + (size_t)(lb * a.T + i) * a.V;
    const int srow = b * a.Tm + i;                                // scratch slot of this logits row
    const int per = ((a.V + nchunk - 1) / nchunk + 3) & ~3;
    const int lo = chunk * per, hi = min(a.V, lo + per);
    pdl_trigger();
    pdl_wait();
    Top2 t = {-INFINITY, 0x7fffffff, -INFINITY};
    auto feed = [&](float v, int j) {
        if (v > t.v1) { t.v2 = t.v1; t.v1 = v; t.i1 = j; }
        else if (v > t.v2) t.v2 = v;
    };
    if ((a.V & 3) == 0) {
        for (int j = lo + threadIdx.x * 4; j < hi; j += blockDim.x * 4) {
            const float4 v = __ldcg(reinterpret_cast<const float4 *>(row + j));
            feed(v.x, j); feed(v.y, j + 1); feed(v.z, j + 2); feed(v.w, j + 3);
        }
    } else {
        for (int j = lo + threadIdx.x; j < hi; j += blockDim.x) feed(__ldcg(row + j), j);
    }
    t = top2_warp(t);
    __shared__ Top2 s[8];
    __shared__ int ticket_s;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (lane == 0) s[warp] = t;
    __syncthreads();
    if (warp != 0) return;
    t = lane < (int)(blockDim.x >> 5) ? s[lane] : Top2{-INFINITY, 0x7fffffff, -INFINITY};
    t = top2_warp(t);
    if (lane == 0) {
        a.part[(size_t)srow * nchunk + chunk] = make_float4(t.v1, __int_as_float(t.i1), t.v2, 0.f);
        __threadfence();
        ticket_s = atomicAdd(a.counters + srow, 1);
    }
    __syncwarp();
    if (ticket_s != nchunk - 1) return;
    __threadfence();
    t = Top2{-INFINITY, 0x7fffffff, -INFINITY};
    for (int c = lane; c < nchunk; c += 32) {
        const float4 p = __ldcg(a.part + (size_t)srow * nchunk + c);
        t = top2_merge(t, Top2{p.x, __float_as_int(p.y), p.z});
    }
    t = top2_warp(t);
    if (lane == 0) {
        a.counters[srow] = 0;
        // a row without any value above -inf (all -inf or NaN) has no maximum: id 0, like a scan that starts at
        // element 0 and never finds anything larger; the id is always a valid row of the embedding table
        const bool none = t.i1 == 0x7fffffff;
        a.tok_out[b * a.Tm + a.tok_col0 + i] = none ? 0 : t.i1;
        if (a.margin_out) a.margin_out[b * a.Tm + i] = none ? 0.f : t.v1 - t.v2;
    }
}

// Greedy acceptance and rollback.  grid = (channel chunks, max(n_rl,1), nb).
//   n = forced_n[b], or the number of leading drafts cand[b][i+1] == g[b][i]
//   committed conv window <- the three raw inputs that end at accepted position n
//   block (0,0,b) also updates the control words: slot, kv_len, pending (= cand[b][0]), outputs.
__global__ void accept_kernel(AcceptArgs a) {
    const int lb = blockIdx.z, b = a.b0 + lb, rl = blockIdx.y;
    const int k = a.k, Tm = a.Tm;
    pdl_trigger();
    pdl_wait();
    const int32_t *cand = a.ctrl.cand + b * Tm, *g = a.ctrl.g + b * Tm;
    int n;
    if (a.forced_n) n = min(max(__ldcg(a.forced_n + b), 0), k);
    else { n = 0; while (n < k && __ldcg(cand + n + 1) == __ldcg(g + n)) ++n; }
    int next = __ldcg(g + n);
    if (a.forced_next && __ldcg(a.forced_next + b) >= 0) next = __ldcg(a.forced_next + b);
    if (next < 0 || next >= a.V) {          // only a caller-supplied id can be out of range: never let it reach the gather
        if (blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0) atomicCAS(a.ctrl.status, 0, (int)HS_ERR_DEVICE);
        next = 0;
    }
    // conv windows: sequence of raw inputs = [w0 w1 w2 | hist_0 .. hist_k]; new window = entries n+1..n+3
    if (rl < a.n_rl) {
        // the full model's window, then (literal draft state) the draft model's own: the same selection on its buffers
        for (int which = 0; which < (a.dcw ? 2 : 1); ++which) {
            float *cw = (which ? a.dcw : a.cw) + ((size_t)rl * a.B + b) * 3 * a.convd;
            const float *hist = (which ? a.dhist : a.hist) + ((size_t)rl * a.B + b) * Tm * a.convd;
            for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < a.convd; c += gridDim.x * blockDim.x) {
                float v[3];
#pragma unroll
                for (int j = 0; j < 3; ++j) {
                    int e = n + 1 + j;
                    v[j] = e < 3 ? __ldcg(cw + e * a.convd + c) : __ldcg(hist + (e - 3) * a.convd + c);
                }
#pragma unroll
                for (int j = 0; j < 3; ++j) cw[j * a.convd + c] = v[j];
            }
        }
    }
    if (blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0) {
        int32_t *em = a.ctrl.emitted + b * Tm;
        int d[HS_MAX_T];
        for (int i = 0; i < k; ++i) d[i] = __ldcg(cand + i + 1);
        for (int i = 0; i <= k; ++i) em[i] = i < n ? d[i] : (i == n ? next : -1);
        a.ctrl.n_acc[b] = n;
        a.ctrl.slot[b] = a.replay ? 0 : n;
        if (a.dslot) a.dslot[b] = (__ldcg(a.dslot + b) + 1 + n) % a.dslot_mod;
        a.ctrl.kv_len[b] = __ldcg(a.ctrl.kv_len + b) + n + 1;
        a.ctrl.cand[b * Tm] = next;
    }
}

// ------------------------------------------------------------------------------------------------
// Speculative sampling at temperature > 0 (paper Sec. 3.3, Eq. 6).  One cluster of eight CTAs per sequence: each takes a
// contiguous eighth of the vocabulary and the CTAs exchange row maxima, sums and segment totals through distributed shared
// memory (one barrier per exchange).  Every sum has a fixed order, so draws are reproducible.
// Bound by latency: two or three sweeps over a logits row that sits in L2.  (One block of 1024 threads per sequence, each
// thread walking a contiguous segment and adding up all 1024 segment totals by itself, took 150-400 us a row at 32768 ids.)
constexpr int SP_CL = 8, SP_THREADS = 512, SP_WARPS = SP_THREADS / 32;
constexpr int SP_BLOCKS = 1024;            // blocks of 32 * m ids a CTA's share is divided into, at most

// A CTA's share of the vocabulary: ids [lo, hi), block i = ids lo + i * 32 m .., one warp per block
struct SpShare { int lo, hi, m, nblk, rank; };
__device__ __forceinline__ SpShare sp_share(int V) {
    SpShare s;
    s.rank = (int)(blockIdx.x % SP_CL);
    const int per = ((V + SP_CL - 1) / SP_CL + 31) & ~31;
    s.lo = min(V, s.rank * per); s.hi = min(V, s.lo + per);
    s.m = (per / 32 + SP_BLOCKS - 1) / SP_BLOCKS;
    s.nblk = (s.hi - s.lo + 32 * s.m - 1) / (32 * s.m);
    return s;
}

struct SpSmem {
    float red[SP_WARPS][HS_MAX_T], gat[3][SP_CL][HS_MAX_T], blk[SP_BLOCKS];
    int n;
};
// every rank's v[0 .. cnt) (in shared memory, complete) to every rank: g[rank][i]
__device__ __forceinline__ void sp_gather(float (*g)[HS_MAX_T], const float *v, int cnt, int rank) {
    for (int i = threadIdx.x; i < SP_CL * cnt; i += SP_THREADS) {
        const int dest = i / cnt, k = i - dest * cnt;
        dsmem_st_f32(dsmem_addr(smem_u32(&g[rank][k]), (uint32_t)dest), v[k]);
    }
    cluster_arrive(); cluster_wait();
}

// maximum and sum of exp((l - max) / tau) of `rows` logits rows (V floats apart): afterwards gat[0] and gat[1] hold every rank's
// local maxima and sums, sp_max / sp_sum combine them in rank order
__device__ __forceinline__ float sp_max(const SpSmem &s, int i) {
    float m = s.gat[0][0][i];
#pragma unroll
    for (int r = 1; r < SP_CL; ++r) m = fmaxf(m, s.gat[0][r][i]);
    return m;
}
__device__ __forceinline__ float sp_sum(const SpSmem &s, int i) {
    float z = 0.f;
#pragma unroll
    for (int r = 0; r < SP_CL; ++r) z += s.gat[1][r][i];
    return z;
}
__device__ __forceinline__ void sp_row_stats(SpSmem &s, const SpShare &sh, const float *row, int rows, int V, float inv_tau) {
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    for (int pass = 0; pass < 2; ++pass) {
        for (int i = 0; i < rows; ++i) {
            const float *r = row + (size_t)i * V;
            const float mx = pass ? sp_max(s, i) : 0.f;
            float v = pass ? 0.f : -INFINITY;
#pragma unroll 8
            for (int j = sh.lo + tid; j < sh.hi; j += SP_THREADS) {
                const float l = __ldcg(r + j);
                v = pass ? v + expf((l - mx) * inv_tau) : fmaxf(v, l);
            }
            v = pass ? warp_sum(v) : warp_max(v);
            if (lane == 0) s.red[warp][i] = v;
        }
        __syncthreads();
        if (tid < rows) {
            float v = s.red[0][tid];
            for (int w = 1; w < SP_WARPS; ++w) v = pass ? v + s.red[w][tid] : fmaxf(v, s.red[w][tid]);
            s.red[0][tid] = v;
        }
        __syncthreads();
        sp_gather(s.gat[pass], s.red[0], rows, sh.rank);
    }
}

// Inverse-CDF draw from the unnormalised weights wf(j) >= 0: the smallest j whose cumulative weight exceeds u * total (the
// last positive one if rounding lets none exceed it).  *out is written by one thread of the cluster.  Returns false, in
// every thread, if the total is not positive.  Uses gat[2] slot `slot`: two draws of one launch take different ones.
template <class WF>
__device__ __forceinline__ bool sp_draw(SpSmem &s, const SpShare &sh, WF wf, float u, int slot, int32_t *out) {
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    __syncthreads();
#pragma unroll 4
    for (int b = warp; b < sh.nblk; b += SP_WARPS) {
        float v = 0.f;
        for (int q = 0; q < sh.m; ++q) {
            const int j = sh.lo + (b * sh.m + q) * 32 + lane;
            if (j < sh.hi) v += wf(j);
        }
        v = warp_sum(v);
        if (lane == 0) s.blk[b] = v;
    }
    __syncthreads();
    // warp 0: lane l adds up blocks [l * per, (l + 1) * per), exclusive prefix over the lanes
    const int per = (sh.nblk + 31) / 32, b0 = min(lane * per, sh.nblk), b1 = min(b0 + per, sh.nblk);
    float seg = 0.f, incl = 0.f;
    if (warp == 0) {
        for (int b = b0; b < b1; ++b) seg += s.blk[b];
        incl = seg;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) { const float x = __shfl_up_sync(0xffffffffu, incl, o); if (lane >= o) incl += x; }
        const float total = __shfl_sync(0xffffffffu, incl, 31);
        if (lane < SP_CL) dsmem_st_f32(dsmem_addr(smem_u32(&s.gat[2][sh.rank][slot]), (uint32_t)lane), total);
    }
    cluster_arrive(); cluster_wait();
    float tot = 0.f, before = 0.f;
    int owner = -1, lastpos = -1;
    for (int r = 0; r < SP_CL; ++r) tot += s.gat[2][r][slot];
    if (!(tot > 0.f)) return false;
    const float t = u * tot;
    float cum = 0.f;
    for (int r = 0; r < SP_CL; ++r) {
        const float v = s.gat[2][r][slot];
        if (v > 0.f) {
            if (owner < 0 && cum + v > t) { owner = r; before = cum; }
            lastpos = r;
        }
        cum += v;
    }
    const bool any = owner >= 0;                  // none: u * total rounded up to the total - the last positive id
    if (!any) owner = lastpos;
    if (owner != sh.rank || warp != 0) return true;
    // the block, then the id inside it
    float c = before + (incl - seg), base = 0.f;
    int blk = -1, last = -1;
    for (int b = b0; b < b1; ++b) {
        const float v = s.blk[b];
        if (v > 0.f) {
            if (any && blk < 0 && c + v > t) { blk = b; base = c; }
            last = b;
        }
        c += v;
    }
    const unsigned hit = __ballot_sync(0xffffffffu, blk >= 0), pos = __ballot_sync(0xffffffffu, last >= 0);
    const int src = hit ? __ffs(hit) - 1 : 31 - __clz(pos);
    blk = __shfl_sync(0xffffffffu, hit ? blk : last, src);
    base = __shfl_sync(0xffffffffu, base, src);
    int pick = -1, lastid = -1;
    for (int q = 0; q < sh.m && pick < 0; ++q) {
        const int j = sh.lo + (blk * sh.m + q) * 32 + lane;
        const float w = j < sh.hi ? wf(j) : 0.f;
        float in = w;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) { const float x = __shfl_up_sync(0xffffffffu, in, o); if (lane >= o) in += x; }
        const unsigned over = __ballot_sync(0xffffffffu, hit && w > 0.f && base + in > t), p = __ballot_sync(0xffffffffu, w > 0.f);
        if (p) lastid = j - lane + 31 - __clz(p);
        if (over) pick = j - lane + __ffs(over) - 1;
        base += __shfl_sync(0xffffffffu, in, 31);
    }
    if (lane == 0) *out = pick >= 0 ? pick : lastid;
    return true;
}

struct SampleArgs {
    const float *logits; int64_t row_stride;   // row of sequence b at logits + b * row_stride
    int V, Tm, b0; float inv_tau;
    const float *u; int u_stride, u_col;       // uniform of sequence b at u[b * u_stride + u_col]
    int32_t *tok_out; int tok_col;             // cand[b][tok_col]
    float2 *stat; int stat_stride;             // (max, sum) of the row, kept for the acceptance test: stat[b * stat_stride + u_col]
};

// draft step: token ~ softmax(logits / tau)
__global__ void __launch_bounds__(SP_THREADS) sample_kernel(const SampleArgs a) {
    __shared__ SpSmem s;
    const int b = a.b0 + blockIdx.x / SP_CL;
    const SpShare sh = sp_share(a.V);
    pdl_trigger();
    cluster_arrive();
    pdl_wait();
    cluster_wait();                              // every rank runs: its shared memory may be written
    const float *row = a.logits + (size_t)b * a.row_stride;
    sp_row_stats(s, sh, row, 1, a.V, a.inv_tau);
    const float mx = sp_max(s, 0);
    int32_t *tok = a.tok_out + b * a.Tm + a.tok_col;
    if (sh.rank == 0 && threadIdx.x == 0) a.stat[(size_t)b * a.stat_stride + a.u_col] = make_float2(mx, sp_sum(s, 0));
    if (!sp_draw(s, sh, [&](int j) { return expf((__ldcg(row + j) - mx) * a.inv_tau); }, __ldcg(a.u + (size_t)b * a.u_stride + a.u_col), 0, tok) &&
        sh.rank == 0 && threadIdx.x == 0) *tok = 0;
}

struct SpecAcceptArgs {
    const float *dlogits; int64_t d_seq_stride;     // draft logits: row i of sequence b at dlogits + b * d_seq_stride + i * V
    const float2 *stat; int stat_stride;            // (max, sum) of those rows, from sample_kernel
    const float *vlogits;                           // verify logits: row (b - b0) * T + i, V floats each
    const int32_t *cand;                            // [B][Tm]
    const float *u_acc, *u_final; int u_stride;     // u_acc[b * u_stride + i], u_final[b]
    int32_t *n_out, *next_out;                      // [B]: accept length and correction / bonus token
    int V, Tm, k, b0; float inv_tau;
};

// Eq. 6 for one sequence: accept draft i+1 iff u_i < P_H(x) / P_S(x); at the first rejection draw the correction from
// the positive part of P_H - P_S, after k acceptances draw the bonus token from P_H.
__global__ void __launch_bounds__(SP_THREADS) spec_accept_kernel(const SpecAcceptArgs a) {
    __shared__ SpSmem s;
    const int lb = blockIdx.x / SP_CL, b = a.b0 + lb, T = a.k + 1;
    const SpShare sh = sp_share(a.V);
    pdl_trigger();
    cluster_arrive();
    pdl_wait();
    cluster_wait();
    const float *drow = a.dlogits + (size_t)b * a.d_seq_stride, *vrow = a.vlogits + (size_t)lb * T * a.V;
    const float2 *stat = a.stat + (size_t)b * a.stat_stride;
    sp_row_stats(s, sh, vrow, T, a.V, a.inv_tau);       // every position's P_H at once
    if (threadIdx.x < 32) {
        // lane i: would draft i + 1 be accepted?
        const int i = threadIdx.x;
        bool reject = false;
        if (i < a.k) {
            const int x = __ldcg(a.cand + b * a.Tm + i + 1);
            const float2 sS = __ldcg(stat + i);
            const float pS = expf((__ldcg(drow + (size_t)i * a.V + x) - sS.x) * a.inv_tau) / sS.y;
            const float pH = expf((__ldcg(vrow + (size_t)i * a.V + x) - sp_max(s, i)) * a.inv_tau) / sp_sum(s, i);
            const float ratio = pS > 0.f ? pH / pS : 1.f;
            reject = !(ratio >= 1.f) && !(__ldcg(a.u_acc + (size_t)b * a.u_stride + i) < ratio);
        }
        const unsigned r = __ballot_sync(0xffffffffu, reject);
        if (i == 0) s.n = r ? __ffs(r) - 1 : a.k;
    }
    __syncthreads();
    const int n = s.n;
    const float uf = __ldcg(a.u_final + b), mH = sp_max(s, n), iH = 1.f / sp_sum(s, n);
    const float *vr = vrow + (size_t)n * a.V;
    bool done = false;
    if (n < a.k) {
        const float *dr = drow + (size_t)n * a.V;
        const float2 sS = __ldcg(stat + n);
        const float iS = 1.f / sS.y;
        done = sp_draw(s, sh, [&](int j) {
            const float d = expf((__ldcg(vr + j) - mH) * a.inv_tau) * iH - expf((__ldcg(dr + j) - sS.x) * a.inv_tau) * iS;
            return d > 0.f ? d : 0.f; }, uf, 0, a.next_out + b);
    }
    if (!done)                                       // bonus draw, or an empty residual: draw from P_H of that position
        done = sp_draw(s, sh, [&](int j) { return expf((__ldcg(vr + j) - mH) * a.inv_tau); }, uf, 1, a.next_out + b);
    if (sh.rank == 0 && threadIdx.x == 0) { a.n_out[b] = n; if (!done) a.next_out[b] = 0; }
}

// Self-test of the bounded wait every copy-fed kernel uses: one warp arms an mbarrier for bytes that no copy
// will ever deliver, polls it `polls` times, gives up, records HS_ERR_TIMEOUT and returns.  Nothing is in flight
// when it exits, so the context stays usable.
__global__ void wait_probe_kernel(int32_t *status, int polls) {
    __shared__ __align__(8) uint64_t bar;
    if (threadIdx.x == 0) { mbar_init(&bar, 1); mbar_fence_init(); }
    __syncwarp();
    if (threadIdx.x == 0) mbar_expect_tx(&bar, 16);
    __syncwarp();
    const bool ok = __all_sync(0xffffffffu, mbar_wait_n(&bar, 0, polls));
    if (!ok && threadIdx.x == 0) atomicCAS(status, 0, (int)HS_ERR_TIMEOUT);
}

}  // namespace

cudaError_t launch_sample(const float *logits, int64_t row_stride, int V, int Tm, int b0, int nb, float tau,
                          const float *u, int u_stride, int u_col, int32_t *tok_out, int tok_col, float2 *stat, int stat_stride, cudaStream_t s) {
    SampleArgs a{logits, row_stride, V, Tm, b0, 1.0f / tau, u, u_stride, u_col, tok_out, tok_col, stat, stat_stride};
    return launch_pdl_cluster(sample_kernel, dim3(nb * SP_CL), dim3(SP_THREADS), 0, s, SP_CL, a);
}

cudaError_t launch_spec_accept(const float *dlogits, int64_t d_seq_stride, const float2 *stat, int stat_stride, const float *vlogits, const int32_t *cand,
                               const float *u_acc, const float *u_final, int u_stride, int32_t *n_out, int32_t *next_out,
                               int V, int Tm, int k, int b0, int nb, float tau, cudaStream_t s) {
    SpecAcceptArgs a{dlogits, d_seq_stride, stat, stat_stride, vlogits, cand, u_acc, u_final, u_stride, n_out, next_out, V, Tm, k, b0, 1.0f / tau};
    return launch_pdl_cluster(spec_accept_kernel, dim3(nb * SP_CL), dim3(SP_THREADS), 0, s, SP_CL, a);
}

cudaError_t launch_wait_probe(int32_t *status, int polls, cudaStream_t s) {
    wait_probe_kernel<<<1, 32, 0, s>>>(status, polls);
    return cudaGetLastError();
}

cudaError_t launch_embed(const __nv_bfloat16 *E, int d, int V, const int32_t *cand, int Tm, int col0, int T,
                         int b0, int nb, float *h, int32_t *status, bool serial, cudaStream_t s) {
    if (serial) {
        // first kernel of a pass: ordinary stream order, so that nothing of this pass (whose kernels read control
        // words in their prologues) starts before everything enqueued earlier - the accept kernel above all - is complete
        embed_kernel<<<dim3(T, nb), dim3(128), 0, s>>>(E, d, V, cand, Tm, col0, T, b0, h, status);
        return cudaGetLastError();
    }
    return launch_pdl(embed_kernel, dim3(T, nb), dim3(128), 0, s, E, d, V, cand, Tm, col0, T, b0, h, status);
}

cudaError_t launch_argmax(const float *logits, int V, int T, int b0, int nb, int Tm,
                          int32_t *tok_out, int tok_col0, float *margin_out, void *part, int32_t *counters, cudaStream_t s) {
    ArgmaxArgs a{logits, V, T, b0, Tm, tok_out, tok_col0, margin_out, reinterpret_cast<float4 *>(part), counters};
    return launch_pdl(argmax_kernel, dim3(HS_ARGMAX_CHUNKS, T, nb), dim3(256), 0, s, a);
}

cudaError_t launch_accept(const AcceptArgs &a, cudaStream_t s) {
    int chunks = (a.convd + 255) / 256;
    if (chunks < 1) chunks = 1;
    return launch_pdl(accept_kernel, dim3(chunks, a.n_rl > 0 ? a.n_rl : 1, a.nb), dim3(256), 0, s, a);
}

// ------------------------------------------------------------------------------------------------
// Argmax without any caller- or library-allocated scratch.
//
// The split argmax above needs a few kilobytes of scratch (per-CTA partial results and a ticket
// counter per row).  Inside the model that scratch is carved out of the caller's work buffer.  This
// stand-alone variant keeps it in a fixed array that is part of the library image instead, so that
// code which is not in a position to allocate device memory can still run the kernel: a host loop
// that already handed every free byte of the GPU to its own arena, a plug-in that is only given
// pointers, or a latency-critical section where an allocation (which may synchronise the device)
// is not acceptable.  The price: the array is loaded on every GPU that loads the library and stays
// until the process exits, and all calls share it.
constexpr int HS_STATIC_ROWS = 64;         // most logits rows one call may pass
constexpr size_t HS_STATIC_PART_BYTES = (size_t)HS_STATIC_ROWS * HS_ARGMAX_CHUNKS * 16;
constexpr size_t HS_STATIC_BYTES = HS_STATIC_PART_BYTES + HS_STATIC_ROWS * 4;   // partials, then counters: 33 KB
static __device__ __align__(256) unsigned char hs_static_scratch[HS_STATIC_BYTES];

namespace {
constexpr int HS_STATIC_MAX_DEVICES = 64;
void *g_static_ptr[HS_STATIC_MAX_DEVICES];     // device address of hs_static_scratch, per device; null = not looked up yet
std::mutex g_static_mutex;                     // two host threads may make their first call at the same time
}

extern "C" int hs_argmax_static(const float *logits_dev, int V, int rows, int32_t *token_dev, float *margin_dev, void *stream) {
    if (!logits_dev || !token_dev || V < 1 || rows < 1) return HS_ERR_INVALID_ARG;
    if (rows > HS_STATIC_ROWS) return HS_ERR_SIZE;             // more rows than the built-in scratch holds
    // the kernel reads rows of a width that is a multiple of four with 128-bit loads: such rows must start on a
    // 16-byte boundary (a view that begins inside a larger tensor may not); the outputs are plain 32-bit words
    if (((uintptr_t)logits_dev & ((V & 3) == 0 ? 15u : 3u)) || ((uintptr_t)token_dev & 3u) || ((uintptr_t)margin_dev & 3u))
        return HS_ERR_INVALID_ARG;
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= HS_STATIC_MAX_DEVICES) return HS_ERR_CUDA;
    unsigned char *base = nullptr;
    {
        std::lock_guard<std::mutex> lock(g_static_mutex);
        if (!g_static_ptr[dev]) {
            // In host code the array's name is only a handle; the address a kernel can use has to be asked for,
            // once per device, with that device current.
            void *p = nullptr;
            if (cudaGetSymbolAddress(&p, hs_static_scratch) != cudaSuccess || !p) return HS_ERR_CUDA;
            g_static_ptr[dev] = p;
        }
        base = static_cast<unsigned char *>(g_static_ptr[dev]);
    }
    int32_t *counters = reinterpret_cast<int32_t *>(base + HS_STATIC_PART_BYTES);
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    // the tickets must start at zero whatever an earlier (possibly failed) call left behind
    if (cudaMemsetAsync(counters, 0, (size_t)rows * 4, s) != cudaSuccess) return HS_ERR_CUDA;
    ArgmaxArgs a{logits_dev, V, rows, 0, rows, token_dev, 0, margin_dev, reinterpret_cast<float4 *>(base), counters};
    argmax_kernel<<<dim3(HS_ARGMAX_CHUNKS, rows, 1), 256, 0, s>>>(a);
    return cudaGetLastError() == cudaSuccess ? HS_OK : HS_ERR_CUDA;
}

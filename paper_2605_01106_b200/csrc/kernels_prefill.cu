// Kernels of the prompt path: what lies between the projections when a pass carries hundreds of prompt positions.
//
// A pass takes up to a few thousand activation rows: the next positions of several sequences, one contiguous piece
// ("segment") per sequence.  The projections are plain dense contractions at that size (kernels_gemm_tc.cu); here are
//   pf_prep_kernel   causal conv + SiLU of the recurrent channels, dt / decay of every head, RoPE of q and k, and the
//                    append of the new K and V rows to the cache - everything that is local to a position
//   pf_ssm_kernel    the Mamba-2 recurrence over the whole segment, state rows resident in registers
//   pf_gdn_kernel    the gated delta rule over the whole segment
//   pf_attn_kernel   causal attention of the segment's positions over the cache (which already holds the new rows)
//   pf_embed_kernel, pf_gather_kernel, pf_advance_kernel, pf_pending_kernel   gathers and control words
// The verify-pass kernels are built for at most nine positions (one trip to L2, everything in registers); their cost
// per position is that of streaming all weights once per nine tokens, which is what this path removes.
// fp32 values keep their precision throughout: the recurrences run in fp32, attention splits queries and probabilities
// into a bf16 head and a bf16 remainder (exact to 2^-17), keys and values enter as the bf16 the cache holds.
#include "hs_internal.h"
#include "hs_device.cuh"

namespace {
using namespace hsd;

__device__ __forceinline__ void cp16(void *dst_smem, const void *src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" :: "r"(smem_u32(dst_smem)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp4(void *dst_smem, const void *src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" :: "r"(smem_u32(dst_smem)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait() { asm volatile("cp.async.wait_group %0;" :: "n"(N) : "memory"); }
__device__ __forceinline__ void ldsm_x4(uint32_t (&r)[4], const void *p) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(smem_u32(p)));
}
__device__ __forceinline__ void ldsm_x4_t(uint32_t (&r)[4], const void *p) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(smem_u32(p)));
}
__device__ __forceinline__ void mma_bf16(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
                 : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
                 : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ __forceinline__ uint32_t pack_bf16x2(float lo, float hi) {
    uint32_t r;
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
    return r;
}
// two fp32 values in one 64-bit register: one instruction works on both
typedef unsigned long long f2;
__device__ __forceinline__ f2 pk2(float x, float y) { f2 r; asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(x), "f"(y)); return r; }
__device__ __forceinline__ void up2(f2 v, float &x, float &y) { asm("mov.b64 {%0, %1}, %2;" : "=f"(x), "=f"(y) : "l"(v)); }
__device__ __forceinline__ f2 fma2(f2 a, f2 b, f2 c) { f2 r; asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c)); return r; }
__device__ __forceinline__ f2 mul2(f2 a, f2 b) { f2 r; asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b)); return r; }

// ---- token gather -------------------------------------------------------------------------------------------
__global__ void pf_embed_kernel(const __nv_bfloat16 *E, int d, int V, const int4 *rows, float *h, int32_t *status) {
    const int r = blockIdx.x;
    pdl_trigger();
    pdl_wait();
    int tok = __ldcg(&rows[r].x);
    if (tok < 0 || tok >= V) {
        if (threadIdx.x == 0) atomicCAS(status, 0, (int)HS_ERR_DEVICE);
        tok = 0;
    }
    const uint4 *src = reinterpret_cast<const uint4 *>(E + (size_t)tok * d);
    float4 *dst = reinterpret_cast<float4 *>(h + (size_t)r * d);
    for (int c = threadIdx.x; c < d / 8; c += blockDim.x) {
        const uint4 w = src[c];
        dst[2 * c] = make_float4(bf_lo(w.x), bf_hi(w.x), bf_lo(w.y), bf_hi(w.y));
        dst[2 * c + 1] = make_float4(bf_lo(w.z), bf_hi(w.z), bf_lo(w.w), bf_hi(w.w));
    }
}

// ---- position-local work ------------------------------------------------------------------------------------
// grid = (row tiles of PREP_ROWS, conv chunks of 256 channels + one slot for the heads and the attention rows).
// A conv thread owns one channel and walks the rows of the tile with its three previous raw inputs in registers, so a
// raw value is read once per tile (plus the three rows before it).
constexpr int PREP_ROWS = 16;

__global__ void __launch_bounds__(256) pf_prep_kernel(const PfPrepArgs a) {
    __shared__ int4 info[PREP_ROWS];
    __shared__ int base[PREP_ROWS];               // position of the row in its sequence, -1: outside the cache
    const int r0 = blockIdx.x * PREP_ROWS, nr = min(PREP_ROWS, a.nrows - r0), tid = threadIdx.x;
    pdl_trigger();
    pdl_wait();
    if (tid < nr) {
        info[tid] = __ldcg(a.rows + r0 + tid);
        const int p = __ldcg(a.kv_len + info[tid].y) + info[tid].z;
        base[tid] = p;
        if (p < 0 || p >= a.cap) { base[tid] = -1; atomicCAS(a.status, 0, p < 0 ? (int)HS_ERR_DEVICE : (int)HS_ERR_CAPACITY); }
    }
    __syncthreads();
    if ((int)blockIdx.y < a.nconv) {
        const int c = blockIdx.y * 256 + tid;
        if (c >= a.convd) return;
        const float4 tap = *reinterpret_cast<const float4 *>(a.conv_w + 4 * c);
        const float bias = a.conv_b[c];
        const float *src = a.zx + (size_t)r0 * a.in_ld + a.conv_off + c;
        float x[PREP_ROWS];
#pragma unroll
        for (int i = 0; i < PREP_ROWS; ++i) x[i] = i < nr ? __ldcg(src + (size_t)i * a.in_ld) : 0.f;
        // raw inputs before the tile: earlier rows of the same segment, or the window its sequence was left with
        auto before = [&](int b, int idx, long long back) {   // idx: position within the segment (may be negative)
            return idx >= 0 ? __ldcg(src - back * a.in_ld) : __ldcg(a.win + ((size_t)b * 3 + 3 + idx) * a.convd + c);
        };
        float w0, w1, w2;
        {
            const int b = info[0].y, i = info[0].z;
            w0 = before(b, i - 3, 3); w1 = before(b, i - 2, 2); w2 = before(b, i - 1, 1);
        }
        float *dst = a.xbc + (size_t)r0 * a.convd + c;
#pragma unroll
        for (int i = 0; i < PREP_ROWS; ++i) {
            if (i < nr) {
                if (i > 0 && info[i].z == 0) {     // a new segment starts inside the tile
                    const float *w = a.win + (size_t)info[i].y * 3 * a.convd + c;
                    w0 = __ldcg(w); w1 = __ldcg(w + a.convd); w2 = __ldcg(w + 2 * a.convd);
                }
                dst[(size_t)i * a.convd] = silu_f(bias + tap.x * w0 + tap.y * w1 + tap.z * w2 + tap.w * x[i]);
                w0 = w1; w1 = w2; w2 = x[i];
            }
        }
        return;
    }
    // dt and decay of every head (Mamba-2), or the decay / write-strength gates (DeltaNet)
    for (int idx = tid; idx < nr * a.heads; idx += 256) {
        const int i = idx / a.heads, h = idx - i * a.heads;
        const float *row = a.zx + (size_t)(r0 + i) * a.in_ld + a.dt_off;
        float u, v;
        if (a.A_log) {
            u = softplus_f(__ldcg(row + h) + a.dt_bias[h]);
            v = expf(-u * expf(a.A_log[h]));
        } else { u = sigmoid_f(__ldcg(row + h)); v = sigmoid_f(__ldcg(row + a.heads + h)); }
        float *out = a.dtv + (size_t)(r0 + i) * 2 * a.heads;
        out[h] = u; out[a.heads + h] = v;
    }
    if (a.qh == 0) return;
    // q: rotated, scaled, split into bf16 head and remainder; k: rotated and v: rounded to bf16 and appended
    const int hp = a.hd / 2, nq = a.qh * hp, nk = a.kvh * hp, per = nq + 2 * nk;
    const float scale = rsqrtf((float)a.hd);
    for (int idx = tid; idx < nr * per; idx += 256) {
        const int i = idx / per, j = idx - i * per, pos = base[i];
        if (pos < 0) continue;
        const float *row = a.zx + (size_t)(r0 + i) * a.in_ld;
        if (j < nq + nk) {
            const bool isq = j < nq;
            const int jj = isq ? j : j - nq, h = jj / hp, e = jj - h * hp;
            const float *s = row + (isq ? a.q_off : a.k_off) + h * a.hd + e;
            const float x0 = __ldcg(s), x1 = __ldcg(s + hp);
            const float2 cs = a.rope[(size_t)pos * hp + e];
            const float y0 = x0 * cs.x - x1 * cs.y, y1 = x1 * cs.x + x0 * cs.y;
            if (isq) {
                const float v0 = y0 * scale, v1 = y1 * scale;
                const __nv_bfloat16 h0 = __float2bfloat16_rn(v0), h1 = __float2bfloat16_rn(v1);
                __nv_bfloat16 *q = a.q + (size_t)(r0 + i) * a.qh * a.hd + h * a.hd + e;
                q[0] = h0; q[hp] = h1;
                q += a.q_plane;
                q[0] = __float2bfloat16_rn(v0 - __bfloat162float(h0)); q[hp] = __float2bfloat16_rn(v1 - __bfloat162float(h1));
            } else {
                __nv_bfloat16 *k = a.Kc + (((size_t)info[i].y * a.kvh + h) * a.cap + pos) * a.hd + e;
                k[0] = __float2bfloat16_rn(y0); k[hp] = __float2bfloat16_rn(y1);
            }
        } else {
            const int jj = j - nq - nk, h = jj / hp, e = jj - h * hp;
            const float *s = row + a.v_off + h * a.hd + 2 * e;
            __nv_bfloat16 *v = a.Vc + (((size_t)info[i].y * a.kvh + h) * a.cap + pos) * a.hd + 2 * e;
            *reinterpret_cast<uint32_t *>(v) = pack_bf16x2(__ldcg(s), __ldcg(s + 1));
        }
    }
}

// New conv window of a segment's sequence: the last three raw inputs, entries n, n + 1, n + 2 of [old window | inputs].
__device__ __forceinline__ void shift_window(const PfScanArgs &a, int b, int row0, int n, int c) {
    float *w = a.win + (size_t)b * 3 * a.convd + c;
#pragma unroll
    for (int j = 0; j < 3; ++j)
        w[(size_t)j * a.convd] = n + j < 3 ? __ldcg(w + (size_t)(n + j) * a.convd)
                                           : __ldcg(a.zx + (size_t)(row0 + n + j - 3) * a.in_ld + a.conv_off + c);
}

// ---- Mamba-2 recurrence -------------------------------------------------------------------------------------
// grid = (strips of 16 state rows, heads, segments), four warps of four rows.  A lane holds EPL = N / 32 state values
// of each of its warp's rows in registers for the whole segment; B, C, x, z and the decays of eight positions at a
// time arrive through a ring of shared-memory stages (asynchronous copies).  The outputs of eight positions x four
// rows are 32 partial sums per lane: one transposing reduction leaves lane l with the total of (position l / 4,
// row l % 4), which that lane gates and stores.  Bound by the issue of its own instructions (packed fp32 pairs).
constexpr int SC_POS = 8, SC_STAGES = 4, SC_THREADS = 128, SC_ROWS = 16;
__host__ __device__ constexpr int sc_stage_floats(int N) { return SC_POS * (2 * N + 2 * SC_ROWS + 4); }

template <int EPL>
__global__ void __launch_bounds__(SC_THREADS) pf_ssm_kernel(const PfScanArgs a) {
    constexpr int N = 32 * EPL, VW = EPL < 4 ? EPL : 4, NVEC = EPL / VW, NP = EPL / 2;
    constexpr int STG = sc_stage_floats(N), CB = N / 4, PER = 2 * CB + 8;      // 16-byte pieces of one position
    extern __shared__ __align__(16) float sm[];
    const int p0 = blockIdx.x * SC_ROWS, h = blockIdx.y, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    pdl_trigger();
    pdl_wait();
    const int4 sg = __ldcg(a.segs + blockIdx.z);
    const int b = sg.x, row0 = sg.y, n = sg.z, slot_out = sg.w;
    const int slot_in = a.nslot == 1 ? 0 : __ldcg(a.slot + b);
    if ((unsigned)slot_in >= (unsigned)a.nslot || (unsigned)slot_out >= (unsigned)a.nslot) {
        if (tid == 0) atomicCAS(a.status, 0, (int)HS_ERR_DEVICE);
        return;
    }
    float *base = a.state + (size_t)b * a.nslot * a.state_elems + ((size_t)h * a.P + p0 + warp * 4) * N;
    const float *sin_ = base + (size_t)slot_in * a.state_elems;
    f2 s[4][NP];
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int v = 0; v < NVEC; ++v) {
            const float *src = sin_ + r * N + v * (32 * VW) + lane * VW;
            if (VW == 4) { const float4 t = __ldcg(reinterpret_cast<const float4 *>(src)); s[r][2 * v] = pk2(t.x, t.y); s[r][2 * v + NP / NVEC - 1] = pk2(t.z, t.w); }
            else { const float2 t = __ldcg(reinterpret_cast<const float2 *>(src)); s[r][0] = pk2(t.x, t.y); }
        }
    const int ntile = (n + SC_POS - 1) / SC_POS;
    auto fetch = [&](int t) {
        if (t < ntile) {
            float *st = sm + (size_t)(t % SC_STAGES) * STG;
            const int cnt = min(SC_POS, n - t * SC_POS);
            for (int idx = tid; idx < cnt * PER; idx += SC_THREADS) {
                const int i = idx / PER, j = idx - i * PER;
                const size_t row = (size_t)(row0 + t * SC_POS + i);
                const float *xr = a.xbc + row * a.convd;
                if (j < CB) cp16(st + i * N + 4 * j, xr + a.di + 4 * j);
                else if (j < 2 * CB) cp16(st + SC_POS * N + i * N + 4 * (j - CB), xr + a.di + N + 4 * (j - CB));
                else if (j < 2 * CB + 4) cp16(st + 2 * SC_POS * N + i * SC_ROWS + 4 * (j - 2 * CB), xr + h * a.P + p0 + 4 * (j - 2 * CB));
                else cp16(st + 2 * SC_POS * N + SC_POS * SC_ROWS + i * SC_ROWS + 4 * (j - 2 * CB - 4), a.zx + row * a.in_ld + h * a.P + p0 + 4 * (j - 2 * CB - 4));
            }
            if (tid < 2 * cnt) {
                const int i = tid >> 1, w = tid & 1;
                cp4(st + 2 * SC_POS * N + 2 * SC_POS * SC_ROWS + 4 * i + w, a.dtv + (size_t)(row0 + t * SC_POS + i) * 2 * a.heads + w * a.heads + h);
            }
        }
        cp_commit();
    };
    const float Dh = a.D[h];
#pragma unroll
    for (int t = 0; t < SC_STAGES - 1; ++t) fetch(t);
#pragma unroll 1
    for (int t = 0; t < ntile; ++t) {
        cp_wait<SC_STAGES - 2>();
        __syncthreads();                  // stage t complete; everybody is done with the stage that is refilled now
        fetch(t + SC_STAGES - 1);
        const float *st = sm + (size_t)(t % SC_STAGES) * STG;
        const float *Bs = st, *Cs = st + SC_POS * N, *xs = st + 2 * SC_POS * N, *zs = xs + SC_POS * SC_ROWS, *dd = zs + SC_POS * SC_ROWS;
        const int cnt = min(SC_POS, n - t * SC_POS);
        float acc[32];
#pragma unroll
        for (int i = 0; i < SC_POS; ++i) {
            if (i < cnt) {
                f2 Bv[NP], Cv[NP];
#pragma unroll
                for (int v = 0; v < NVEC; ++v) {
                    if (VW == 4) {
                        const float4 x = *reinterpret_cast<const float4 *>(Bs + i * N + v * 128 + lane * 4), y = *reinterpret_cast<const float4 *>(Cs + i * N + v * 128 + lane * 4);
                        Bv[2 * v] = pk2(x.x, x.y); Bv[2 * v + NP / NVEC - 1] = pk2(x.z, x.w);
                        Cv[2 * v] = pk2(y.x, y.y); Cv[2 * v + NP / NVEC - 1] = pk2(y.z, y.w);
                    } else {
                        const float2 x = *reinterpret_cast<const float2 *>(Bs + i * N + lane * 2), y = *reinterpret_cast<const float2 *>(Cs + i * N + lane * 2);
                        Bv[0] = pk2(x.x, x.y); Cv[0] = pk2(y.x, y.y);
                    }
                }
                const float2 dt = *reinterpret_cast<const float2 *>(dd + 4 * i);       // dt, decay
                const float4 xv = *reinterpret_cast<const float4 *>(xs + i * SC_ROWS + warp * 4);
                const f2 dec = pk2(dt.y, dt.y);
                const float xr[4] = {xv.x, xv.y, xv.z, xv.w};
#pragma unroll
                for (int r = 0; r < 4; ++r) {
                    const float dx = dt.x * xr[r];
                    const f2 dtx = pk2(dx, dx);
                    f2 y = 0ull;
#pragma unroll
                    for (int e = 0; e < NP; ++e) {
                        s[r][e] = fma2(dec, s[r][e], mul2(dtx, Bv[e]));
                        y = e ? fma2(s[r][e], Cv[e], y) : mul2(s[r][e], Cv[e]);
                    }
                    float lo, hi;
                    up2(y, lo, hi);
                    acc[i * 4 + r] = lo + hi;
                }
            } else {
#pragma unroll
                for (int r = 0; r < 4; ++r) acc[i * 4 + r] = 0.f;
            }
        }
        const float y = xreduce<32>(acc, lane);
        const int i = lane >> 2, rr = warp * 4 + (lane & 3);
        if (i < cnt)
            a.g[(size_t)(row0 + t * SC_POS + i) * a.gw + h * a.P + p0 + rr] = (y + Dh * xs[i * SC_ROWS + rr]) * silu_f(zs[i * SC_ROWS + rr]);
    }
    cp_wait<0>();
    float *sout = base + (size_t)slot_out * a.state_elems;
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int v = 0; v < NVEC; ++v) {
            float *p = sout + r * N + v * (32 * VW) + lane * VW;
            float x0, x1, x2, x3;
            up2(s[r][VW == 4 ? 2 * v : 0], x0, x1);
            if (VW == 4) { up2(s[r][2 * v + NP / NVEC - 1], x2, x3); *reinterpret_cast<float4 *>(p) = make_float4(x0, x1, x2, x3); }
            else *reinterpret_cast<float2 *>(p) = make_float2(x0, x1);
        }
    if (tid < SC_ROWS) shift_window(a, b, row0, n, h * a.P + p0 + tid);
    if (blockIdx.x == 0 && h == 0)
        for (int c = tid; c < 2 * N; c += SC_THREADS) shift_window(a, b, row0, n, a.di + c);
}

// ---- gated delta rule ---------------------------------------------------------------------------------------
// grid = (heads, segments); two lanes per value row, each with 32 of the 64 key columns in registers.  The dependent
// chain of a position is one dot product (S k), one shuffle, the update; S q and the output norm hang off it.
constexpr int GD_POS = 8, GD_STAGES = 3, GD_THREADS = 128;
constexpr int GD_STG = GD_POS * (4 * 64 + 4);

__global__ void __launch_bounds__(GD_THREADS) pf_gdn_kernel(const PfScanArgs a) {
    extern __shared__ __align__(16) float sm[];
    __shared__ float os[GD_POS][64];
    const int h = blockIdx.x, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int dv = a.P, nk = a.heads * 64, nv = a.heads * dv;
    pdl_trigger();
    pdl_wait();
    const int4 sg = __ldcg(a.segs + blockIdx.y);
    const int b = sg.x, row0 = sg.y, n = sg.z, slot_out = sg.w;
    const int slot_in = a.nslot == 1 ? 0 : __ldcg(a.slot + b);
    if ((unsigned)slot_in >= (unsigned)a.nslot || (unsigned)slot_out >= (unsigned)a.nslot) {
        if (tid == 0) atomicCAS(a.status, 0, (int)HS_ERR_DEVICE);
        return;
    }
    float *base = a.state + (size_t)b * a.nslot * a.state_elems + (size_t)h * dv * 64;
    const int vr = tid >> 1, half = tid & 1;          // value row, half of the key columns
    const bool live = vr < dv;
    f2 s[16];
#pragma unroll
    for (int e = 0; e < 8; ++e) {                     // columns half * 4 + 8 e .. + 3: both lanes of a row read 32 bytes in a row
        float4 t = make_float4(0.f, 0.f, 0.f, 0.f);
        if (live) t = __ldcg(reinterpret_cast<const float4 *>(base + (size_t)slot_in * a.state_elems + (size_t)vr * 64 + 8 * e + 4 * half));
        s[2 * e] = pk2(t.x, t.y); s[2 * e + 1] = pk2(t.z, t.w);
    }
    const int ntile = (n + GD_POS - 1) / GD_POS, vpc = dv / 4, PER = 32 + 2 * vpc;
    auto fetch = [&](int t) {
        if (t < ntile) {
            float *st = sm + (size_t)(t % GD_STAGES) * GD_STG;      // q[8][64] k[8][64] v[8][64] z[8][64] ab[8][4]
            const int cnt = min(GD_POS, n - t * GD_POS);
            for (int idx = tid; idx < cnt * PER; idx += GD_THREADS) {
                const int i = idx / PER, j = idx - i * PER;
                const size_t row = (size_t)(row0 + t * GD_POS + i);
                const float *xr = a.xbc + row * a.convd;
                if (j < 16) cp16(st + i * 64 + 4 * j, xr + h * 64 + 4 * j);
                else if (j < 32) cp16(st + 512 + i * 64 + 4 * (j - 16), xr + nk + h * 64 + 4 * (j - 16));
                else if (j < 32 + vpc) cp16(st + 1024 + i * 64 + 4 * (j - 32), xr + 2 * nk + h * dv + 4 * (j - 32));
                else cp16(st + 1536 + i * 64 + 4 * (j - 32 - vpc), a.zx + row * a.in_ld + 2 * nk + nv + h * dv + 4 * (j - 32 - vpc));
            }
            if (tid < 2 * cnt) {
                const int i = tid >> 1, w = tid & 1;
                cp4(st + 2048 + 4 * i + w, a.dtv + (size_t)(row0 + t * GD_POS + i) * 2 * a.heads + w * a.heads + h);
            }
        }
        cp_commit();
    };
#pragma unroll
    for (int t = 0; t < GD_STAGES - 1; ++t) fetch(t);
#pragma unroll 1
    for (int t = 0; t < ntile; ++t) {
        cp_wait<GD_STAGES - 2>();
        __syncthreads();
        fetch(t + GD_STAGES - 1);
        float *st = sm + (size_t)(t % GD_STAGES) * GD_STG;
        const int cnt = min(GD_POS, n - t * GD_POS);
        // q and k of the tile's positions are L2-normalised in place: a warp takes four of the sixteen vectors
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int vec = warp * 4 + u;
            if ((vec & 7) < cnt) {
                float2 *p = reinterpret_cast<float2 *>(st + (vec >> 3) * 512 + (vec & 7) * 64) + lane;
                float2 x = *p;
                const float inv = rsqrtf(warp_sum(x.x * x.x + x.y * x.y) + 1e-6f);
                x.x *= inv; x.y *= inv;
                *p = x;
            }
        }
        __syncthreads();
#pragma unroll 1
        for (int i = 0; i < cnt; ++i) {
            const float *q = st + i * 64 + 4 * half, *k = st + 512 + i * 64 + 4 * half;
            const float alpha = st[2048 + 4 * i], beta = st[2048 + 4 * i + 1];
            const float v = live ? st[1024 + i * 64 + vr] : 0.f;
            f2 kv[16];
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                const float4 x = *reinterpret_cast<const float4 *>(k + 8 * e);
                kv[2 * e] = pk2(x.x, x.y); kv[2 * e + 1] = pk2(x.z, x.w);
            }
            f2 d0 = mul2(s[0], kv[0]), d1 = mul2(s[1], kv[1]), d2 = mul2(s[2], kv[2]), d3 = mul2(s[3], kv[3]);
#pragma unroll
            for (int e = 4; e < 16; e += 4) {
                d0 = fma2(s[e], kv[e], d0); d1 = fma2(s[e + 1], kv[e + 1], d1);
                d2 = fma2(s[e + 2], kv[e + 2], d2); d3 = fma2(s[e + 3], kv[e + 3], d3);
            }
            float x0, x1, x2, x3, x4, x5, x6, x7;
            up2(d0, x0, x1); up2(d1, x2, x3); up2(d2, x4, x5); up2(d3, x6, x7);
            float dot = ((x0 + x1) + (x2 + x3)) + ((x4 + x5) + (x6 + x7));
            dot += __shfl_xor_sync(0xffffffffu, dot, 1);
            const float u = beta * (v - alpha * dot);
            const f2 uu = pk2(u, u), aa = pk2(alpha, alpha);
            f2 o0 = 0ull, o1 = 0ull;
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                const float4 x = *reinterpret_cast<const float4 *>(q + 8 * e);
                s[2 * e] = fma2(aa, s[2 * e], mul2(uu, kv[2 * e]));
                s[2 * e + 1] = fma2(aa, s[2 * e + 1], mul2(uu, kv[2 * e + 1]));
                o0 = fma2(s[2 * e], pk2(x.x, x.y), o0); o1 = fma2(s[2 * e + 1], pk2(x.z, x.w), o1);
            }
            up2(o0, x0, x1); up2(o1, x2, x3);
            float o = (x0 + x1) + (x2 + x3);
            o += __shfl_xor_sync(0xffffffffu, o, 1);
            if (live && half == 0) os[i][vr] = o * 0.125f;          // 1 / sqrt(64)
        }
        __syncthreads();
        // per-head RMSNorm over dv, then the output gate silu(z)
        for (int i = warp; i < cnt; i += GD_THREADS / 32) {
            float ss = 0.f;
            for (int j = lane; j < dv; j += 32) ss = fmaf(os[i][j], os[i][j], ss);
            const float rstd = rsqrtf(warp_sum(ss) / (float)dv + a.eps);
            for (int j = lane; j < dv; j += 32)
                a.g[(size_t)(row0 + t * GD_POS + i) * a.gw + h * dv + j] = os[i][j] * rstd * a.onorm[j] * silu_f(st[1536 + i * 64 + j]);
        }
    }
    cp_wait<0>();
    if (live)
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            float x0, x1, x2, x3;
            up2(s[2 * e], x0, x1); up2(s[2 * e + 1], x2, x3);
            *reinterpret_cast<float4 *>(base + (size_t)slot_out * a.state_elems + (size_t)vr * 64 + 8 * e + 4 * half) = make_float4(x0, x1, x2, x3);
        }
    for (int c = tid; c < 128 + dv; c += GD_THREADS)
        shift_window(a, b, row0, n, c < 64 ? h * 64 + c : c < 128 ? nk + h * 64 + (c - 64) : 2 * nk + h * dv + (c - 128));
}

// ---- attention ----------------------------------------------------------------------------------------------
// grid = (tiles of 64 positions, query heads, segments); four warps of 16 query positions, tiles of 64 keys of the
// cache in two shared-memory stages.  Scores and P V on the warp-level tensor path with head + remainder operands,
// running softmax in registers.  The longest tiles (the last positions) go out first.
constexpr int PA_Q = 64, PA_K = 64, PA_THREADS = 128;

template <int HD>
__global__ void __launch_bounds__(PA_THREADS) pf_attn_kernel(const PfAttnArgs a) {
    constexpr int KS = HD + 8, NT = HD / 8, HC = HD / 8;
    extern __shared__ __align__(16) unsigned char smraw[];
    __nv_bfloat16 *K_s = reinterpret_cast<__nv_bfloat16 *>(smraw), *V_s = K_s + 2 * PA_K * KS;      // [2][PA_K][KS] each
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g8 = lane >> 2, t4 = lane & 3;
    pdl_trigger();
    pdl_wait();
    const int4 sg = __ldcg(a.segs + blockIdx.z);
    const int b = sg.x, row0 = sg.y, n = sg.z, qt = gridDim.x - 1 - blockIdx.x, h = blockIdx.y;
    const int q0 = qt * PA_Q;
    if (q0 >= n) return;
    const int base = __ldcg(a.kv_len + b);
    if (base < 0 || base + n > a.cap) return;        // reported by pf_prep_kernel
    const int kh = h / (a.qh / a.kvh), ld = a.qh * HD;
    const __nv_bfloat16 *Kb = a.Kc + ((size_t)b * a.kvh + kh) * a.cap * HD, *Vb = a.Vc + ((size_t)b * a.kvh + kh) * a.cap * HD;
    const int nkeys = base + min(n, q0 + PA_Q), ntile = (nkeys + PA_K - 1) / PA_K;
    auto fetch = [&](int t) {
        if (t < ntile) {
            const int cnt = min(PA_K, nkeys - t * PA_K);
            __nv_bfloat16 *kd = K_s + (t & 1) * PA_K * KS, *vd = V_s + (t & 1) * PA_K * KS;
            for (int idx = tid; idx < PA_K * HC; idx += PA_THREADS) {
                const int j = idx / HC, c = idx - j * HC;
                if (j < cnt) {
                    cp16(kd + j * KS + 8 * c, Kb + (size_t)(t * PA_K + j) * HD + 8 * c);
                    cp16(vd + j * KS + 8 * c, Vb + (size_t)(t * PA_K + j) * HD + 8 * c);
                } else {                              // finite values where the tile ends early
                    *reinterpret_cast<uint4 *>(kd + j * KS + 8 * c) = make_uint4(0, 0, 0, 0);
                    *reinterpret_cast<uint4 *>(vd + j * KS + 8 * c) = make_uint4(0, 0, 0, 0);
                }
            }
        }
        cp_commit();
    };
    fetch(0);
    const int wq = q0 + warp * 16;                    // first position of this warp's rows, within the segment
    uint32_t qh_[HD / 16][4], ql_[HD / 16][4];
#pragma unroll
    for (int ks = 0; ks < HD / 16; ++ks)
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const int i = wq + g8 + (e & 1) * 8, c = ks * 16 + 2 * t4 + (e >> 1) * 8;
            const __nv_bfloat16 *p = a.q + (size_t)(row0 + i) * ld + h * HD + c;
            qh_[ks][e] = i < n ? __ldcg(reinterpret_cast<const uint32_t *>(p)) : 0u;
            ql_[ks][e] = i < n ? __ldcg(reinterpret_cast<const uint32_t *>(p + a.q_plane)) : 0u;
        }
    float O[NT][4];
#pragma unroll
    for (int nt = 0; nt < NT; ++nt) O[nt][0] = O[nt][1] = O[nt][2] = O[nt][3] = 0.f;
    float m_run[2] = {-INFINITY, -INFINITY}, l_run[2] = {0.f, 0.f};
#pragma unroll 1
    for (int t = 0; t < ntile; ++t) {
        fetch(t + 1);
        cp_wait<1>();
        __syncthreads();
        const __nv_bfloat16 *kt = K_s + (t & 1) * PA_K * KS, *vt = V_s + (t & 1) * PA_K * KS;
        const int k0 = t * PA_K, last = base + wq + 15;            // last key any row of this warp may see
        if (k0 <= last) {
            float S[PA_K / 8][4];
#pragma unroll
            for (int nt = 0; nt < PA_K / 8; ++nt) S[nt][0] = S[nt][1] = S[nt][2] = S[nt][3] = 0.f;
#pragma unroll
            for (int ks = 0; ks < HD / 16; ++ks)
#pragma unroll
                for (int np = 0; np < PA_K / 16; ++np) {
                    uint32_t bk[4];
                    ldsm_x4(bk, kt + (size_t)(np * 16 + (lane & 7) + (lane >> 4) * 8) * KS + ks * 16 + ((lane >> 3) & 1) * 8);
                    mma_bf16(S[2 * np], qh_[ks], bk[0], bk[1]); mma_bf16(S[2 * np + 1], qh_[ks], bk[2], bk[3]);
                    mma_bf16(S[2 * np], ql_[ks], bk[0], bk[1]); mma_bf16(S[2 * np + 1], ql_[ks], bk[2], bk[3]);
                }
            if (k0 + PA_K - 1 > base + wq)            // the diagonal: later positions are masked
#pragma unroll
                for (int nt = 0; nt < PA_K / 8; ++nt)
#pragma unroll
                    for (int e = 0; e < 4; ++e)
                        if (k0 + nt * 8 + 2 * t4 + (e & 1) > base + wq + g8 + 8 * (e >> 1)) S[nt][e] = -INFINITY;
            float corr[2];
#pragma unroll
            for (int r = 0; r < 2; ++r) {
                float mx = -INFINITY;
#pragma unroll
                for (int nt = 0; nt < PA_K / 8; ++nt) mx = fmaxf(mx, fmaxf(S[nt][2 * r], S[nt][2 * r + 1]));
                mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
                mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 2));
                const float mnew = fmaxf(m_run[r], mx);   // key 0 is visible to every row: finite from the first tile on
                corr[r] = __expf(m_run[r] - mnew);
                m_run[r] = mnew;
                float sum = 0.f;
#pragma unroll
                for (int nt = 0; nt < PA_K / 8; ++nt) {
                    S[nt][2 * r] = __expf(S[nt][2 * r] - mnew); S[nt][2 * r + 1] = __expf(S[nt][2 * r + 1] - mnew);
                    sum += S[nt][2 * r] + S[nt][2 * r + 1];
                }
                l_run[r] = fmaf(l_run[r], corr[r], sum);
            }
            if (__any_sync(0xffffffffu, corr[0] != 1.f || corr[1] != 1.f))
#pragma unroll
                for (int nt = 0; nt < NT; ++nt) { O[nt][0] *= corr[0]; O[nt][1] *= corr[0]; O[nt][2] *= corr[1]; O[nt][3] *= corr[1]; }
#pragma unroll
            for (int j = 0; j < PA_K / 16; ++j) {
                uint32_t ph[4], pl[4];
#pragma unroll
                for (int nt = 0; nt < 2; ++nt)
#pragma unroll
                    for (int r = 0; r < 2; ++r) {
                        const float p0 = S[2 * j + nt][2 * r], p1 = S[2 * j + nt][2 * r + 1];
                        const uint32_t hh = pack_bf16x2(p0, p1);
                        ph[r + 2 * nt] = hh;
                        pl[r + 2 * nt] = pack_bf16x2(p0 - __uint_as_float(hh << 16), p1 - __uint_as_float(hh & 0xffff0000u));
                    }
#pragma unroll
                for (int p = 0; p < NT / 2; ++p) {
                    uint32_t bv[4];
                    ldsm_x4_t(bv, vt + (size_t)(j * 16 + (lane & 7) + ((lane >> 3) & 1) * 8) * KS + p * 16 + (lane >> 4) * 8);
                    mma_bf16(O[2 * p], ph, bv[0], bv[1]); mma_bf16(O[2 * p + 1], ph, bv[2], bv[3]);
                    mma_bf16(O[2 * p], pl, bv[0], bv[1]); mma_bf16(O[2 * p + 1], pl, bv[2], bv[3]);
                }
            }
        }
        __syncthreads();                              // everybody is done with this stage: the next fetch refills it
    }
    cp_wait<0>();
#pragma unroll
    for (int r = 0; r < 2; ++r) {
        float l = l_run[r];
        l += __shfl_xor_sync(0xffffffffu, l, 1);
        l += __shfl_xor_sync(0xffffffffu, l, 2);
        const int i = wq + g8 + 8 * r;
        if (i >= n) continue;
        const float inv = 1.0f / l;
        float *o = a.o + (size_t)(row0 + i) * ld + h * HD + 2 * t4;
#pragma unroll
        for (int nt = 0; nt < NT; ++nt) *reinterpret_cast<float2 *>(o + nt * 8) = make_float2(O[nt][2 * r] * inv, O[nt][2 * r + 1] * inv);
    }
}

// ---- gathers and control words ------------------------------------------------------------------------------
// list[i] = {row of h, row of out}
__global__ void pf_gather_kernel(const int2 *list, const float *h, int d, float *out) {
    pdl_trigger();
    pdl_wait();
    const int2 e = __ldcg(list + blockIdx.x);
    for (int c = threadIdx.x * 4; c < d; c += blockDim.x * 4)
        *reinterpret_cast<float4 *>(out + (size_t)e.y * d + c) = __ldcg(reinterpret_cast<const float4 *>(h + (size_t)e.x * d + c));
}
// end of a pass: the segments' positions are consumed
__global__ void pf_advance_kernel(const int4 *segs, int nseg, int32_t *kv_len, int32_t *slot) {
    pdl_trigger();
    pdl_wait();
    for (int i = threadIdx.x; i < nseg; i += blockDim.x) {
        const int4 s = __ldcg(segs + i);
        kv_len[s.x] = __ldcg(kv_len + s.x) + s.z;
        slot[s.x] = s.w;
    }
}
// pending token of sequences b0 .. b0 + nb - 1: the choice after their last position (column T - 1)
__global__ void pf_pending_kernel(const int32_t *g, int32_t *cand, int Tm, int T, int b0, int nb) {
    pdl_trigger();
    pdl_wait();
    for (int i = threadIdx.x; i < nb; i += blockDim.x) cand[(b0 + i) * Tm] = __ldcg(g + (b0 + i) * Tm + T - 1);
}

template <class K>
cudaError_t allow_smem(K kernel, size_t bytes) {
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout, (int)cudaSharedmemCarveoutMaxShared);
    return e;
}
constexpr size_t ssm_smem(int N) { return (size_t)SC_STAGES * sc_stage_floats(N) * 4; }
constexpr size_t GDN_SMEM = (size_t)GD_STAGES * GD_STG * 4;
constexpr size_t pa_smem(int hd) { return (size_t)4 * PA_K * (hd + 8) * 2; }

}  // namespace

cudaError_t configure_prefill() {
    cudaError_t e = allow_smem(pf_ssm_kernel<2>, ssm_smem(64));
    if (e == cudaSuccess) e = allow_smem(pf_ssm_kernel<4>, ssm_smem(128));
    if (e == cudaSuccess) e = allow_smem(pf_ssm_kernel<8>, ssm_smem(256));
    if (e == cudaSuccess) e = allow_smem(pf_gdn_kernel, GDN_SMEM);
    if (e == cudaSuccess) e = allow_smem(pf_attn_kernel<64>, pa_smem(64));
    if (e == cudaSuccess) e = allow_smem(pf_attn_kernel<128>, pa_smem(128));
    return e;
}

cudaError_t launch_pf_embed(const __nv_bfloat16 *E, int d, int V, const int4 *rows, int nrows, float *h, int32_t *status, cudaStream_t s) {
    // first kernel of a pass: plain stream order (its successors read control words that the pass before wrote)
    pf_embed_kernel<<<nrows, 128, 0, s>>>(E, d, V, rows, h, status);
    return cudaGetLastError();
}
cudaError_t launch_pf_prep(const PfPrepArgs &a, cudaStream_t s) {
    return launch_pdl(pf_prep_kernel, dim3((a.nrows + PREP_ROWS - 1) / PREP_ROWS, a.nconv + 1), dim3(256), 0, s, a);
}
cudaError_t launch_pf_ssm(const PfScanArgs &a, cudaStream_t s) {
    const dim3 grid(a.P / SC_ROWS, a.heads, a.nseg), block(SC_THREADS);
    if (a.N == 64) return launch_pdl(pf_ssm_kernel<2>, grid, block, ssm_smem(64), s, a);
    if (a.N == 128) return launch_pdl(pf_ssm_kernel<4>, grid, block, ssm_smem(128), s, a);
    if (a.N == 256) return launch_pdl(pf_ssm_kernel<8>, grid, block, ssm_smem(256), s, a);
    return cudaErrorInvalidValue;
}
cudaError_t launch_pf_gdn(const PfScanArgs &a, cudaStream_t s) {
    if (a.P > 64 || (a.P & 3)) return cudaErrorInvalidValue;
    return launch_pdl(pf_gdn_kernel, dim3(a.heads, a.nseg), dim3(GD_THREADS), GDN_SMEM, s, a);
}
cudaError_t launch_pf_attn(const PfAttnArgs &a, cudaStream_t s) {
    const dim3 grid((a.max_seg + PA_Q - 1) / PA_Q, a.qh, a.nseg), block(PA_THREADS);
    if (a.hd == 128) return launch_pdl(pf_attn_kernel<128>, grid, block, pa_smem(128), s, a);
    if (a.hd == 64) return launch_pdl(pf_attn_kernel<64>, grid, block, pa_smem(64), s, a);
    return cudaErrorInvalidValue;
}
cudaError_t launch_pf_gather(const int2 *list, int n, const float *h, int d, float *out, cudaStream_t s) {
    return launch_pdl(pf_gather_kernel, dim3(n), dim3(128), 0, s, list, h, d, out);
}
cudaError_t launch_pf_advance(const int4 *segs, int nseg, int32_t *kv_len, int32_t *slot, cudaStream_t s) {
    return launch_pdl(pf_advance_kernel, dim3(1), dim3(64), 0, s, segs, nseg, kv_len, slot);
}
cudaError_t launch_pf_pending(const int32_t *g, int32_t *cand, int Tm, int T, int b0, int nb, cudaStream_t s) {
    return launch_pdl(pf_pending_kernel, dim3(1), dim3(64), 0, s, g, cand, Tm, T, b0, nb);
}

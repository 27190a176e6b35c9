// Kernels of the prompt path: what lies between the projections when a pass carries hundreds of prompt positions.
//
// A pass takes up to a few thousand activation rows: the next positions of several sequences, one contiguous piece
// ("segment") per sequence.  The projections are plain dense contractions at that size (kernels_gemm_wide.cu); here are
//   pf_prep_kernel   causal conv + SiLU of the recurrent channels, dt / decay of every head, RoPE of q and k, and the
//                    append of the new K and V rows to the cache - everything that is local to a position
//   pf_gram_kernel, pf_ssm_kernel                          the Mamba-2 recurrence over the whole segment
//   pf_gdn_gram_kernel, pf_gdn_kernel, pf_gdn_out_kernel   the gated delta rule over the whole segment, output norm and gate
//   pf_attn_kernel   causal attention of the segment's positions over the cache (which already holds the new rows)
//   pf_embed_kernel, pf_gather_kernel, pf_advance_kernel, pf_pending_kernel   gathers and control words
// The verify-pass kernels are built for at most nine positions (one trip to L2, everything in registers); their cost
// per position is that of streaming all weights once per nine tokens, which is what this path removes.
// The kernels between the projections let their successor start when their own work is done, not earlier: blocks that wait
// hold the registers and shared memory that the blocks still to come need (14.0 -> 9.6 ms for 512 tokens on the 0.5B-class
// hybrid).  Except the small gathers and pf_ssm_kernel, which the attention of its block runs beside (hs_device.cuh).
// fp32 values keep their precision throughout: the recurrences run in fp32, attention splits queries and probabilities
// into a bf16 head and a bf16 remainder (exact to 2^-17), keys and values enter as the bf16 the cache holds.
#include "hs_internal.h"
#include "hs_device.cuh"

namespace {
using namespace hsd;

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
// grid = (row tiles of PREP_ROWS, roles): `nconv` chunks of 256 conv channels, one block for dt / decay of every head,
// then chunks of 256 (rotation) pairs of the q | k | v rows.  A thread owns one channel or pair and walks the rows of
// the tile; the loads of all rows are issued before the first is used.  (One block for all heads and pairs of a tile:
// 41 us at 512 rows of the 0.5B-class hybrid; split: 16 us.)
constexpr int PREP_ROWS = 16;

__global__ void __launch_bounds__(256) pf_prep_kernel(const PfPrepArgs a) {
    __shared__ int4 info[PREP_ROWS];
    __shared__ int base[PREP_ROWS];               // position of the row in its sequence, -1: outside the cache
    const int r0 = blockIdx.x * PREP_ROWS, nr = min(PREP_ROWS, a.nrows - r0), tid = threadIdx.x;
    pdl_wait();
    if (tid < nr) {
        info[tid] = __ldcg(a.rows + r0 + tid);
        const int p = __ldcg(a.kv_len + info[tid].y) + info[tid].z;
        base[tid] = p;
        if (p < 0 || p >= a.cap) { base[tid] = -1; atomicCAS(a.status, 0, p < 0 ? (int)HS_ERR_DEVICE : (int)HS_ERR_CAPACITY); }
    }
    __syncthreads();
    int role = blockIdx.y;
    if (role < a.nconv) {
        const int c = role * 256 + tid;
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
    role -= a.nconv;
    if (a.heads && role-- == 0) {
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
        return;
    }
    // q: rotated, scaled, split into bf16 head and remainder; k: rotated and v: rounded to bf16 and appended
    const int hp = a.hd / 2, nq = a.qh * hp, nk = a.kvh * hp;
    const int j = role * 256 + tid;
    if (j >= nq + 2 * nk) return;
    const bool isq = j < nq, isv = j >= nq + nk;
    const int jj = isq ? j : isv ? j - nq - nk : j - nq, h = jj / hp, e = jj - h * hp;
    const float *src = a.zx + (size_t)r0 * a.in_ld + (isq ? a.q_off : isv ? a.v_off : a.k_off) + h * a.hd + (isv ? 2 * e : e);
    const int step = isv ? 1 : hp;                // the pair: (e, e + hd / 2) for a rotation, two neighbours for v
    const float scale = isq ? rsqrtf((float)a.hd) : 1.f;
    float x0[PREP_ROWS], x1[PREP_ROWS];
#pragma unroll
    for (int i = 0; i < PREP_ROWS; ++i) {
        x0[i] = i < nr ? __ldcg(src + (size_t)i * a.in_ld) : 0.f;
        x1[i] = i < nr ? __ldcg(src + (size_t)i * a.in_ld + step) : 0.f;
    }
#pragma unroll
    for (int i = 0; i < PREP_ROWS; ++i) {
        const int pos = i < nr ? base[i] : -1;
        if (pos < 0) continue;
        const size_t crow = (((size_t)info[i].y * a.kvh + h) * a.cap + pos) * a.hd;
        if (isv) { *reinterpret_cast<uint32_t *>(a.Vc + crow + 2 * e) = pack_bf16x2(x0[i], x1[i]); continue; }
        const float2 cs = a.rope[(size_t)pos * hp + e];
        const float y0 = (x0[i] * cs.x - x1[i] * cs.y) * scale, y1 = (x1[i] * cs.x + x0[i] * cs.y) * scale;
        const __nv_bfloat16 h0 = __float2bfloat16_rn(y0), h1 = __float2bfloat16_rn(y1);
        if (isq) {
            __nv_bfloat16 *q = a.q + (size_t)(r0 + i) * a.qh * a.hd + h * a.hd + e;
            q[0] = h0; q[hp] = h1;
            q += a.q_plane;
            q[0] = __float2bfloat16_rn(y0 - __bfloat162float(h0)); q[hp] = __float2bfloat16_rn(y1 - __bfloat162float(h1));
        } else { a.Kc[crow + e] = h0; a.Kc[crow + e + hp] = h1; }
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

// ---- recurrences in tiles of eight positions ------------------------------------------------------------------
// Unrolled over a tile of eight positions a linear recurrence needs the state only twice: for the eight products of
// the OLD state with the tile's read vectors, and for one update with the tile's eight outer products.  What couples
// the positions of a tile is small and shared by all state rows - products of the tile's vectors with each other times
// the decays between them - so it is computed once per tile (pf_gram / pf_gdn_gram) into a record that the scan reads:
//   Mamba-2   y_i = P_i (C_i . S) + sum_{j<=i} M_ij x_j + D x_i ,   S <- P_7 S + sum_j (E_j x_j) B_j^T
//             P_i = prod_{u<=i} a_u ,  M_ij = (C_i . B_j) dt_j prod_{j<u<=i} a_u ,  E_j = dt_j prod_{j<u<=7} a_u
//   DeltaNet  u_i = beta_i v_i - beta_i P_i (S k_i) - sum_{j<i} MK_ij u_j   (per value row, solved in order)
//             o_i = P_i (S q_i) + sum_{j<=i} MQ_ij u_j ,            S <- P_7 S + sum_j (E_j u_j) k_j^T
//             MK_ij = beta_i (k_i . k_j) prod_{j<u<=i} alpha_u ,  MQ_ij = (q_i . k_j) prod.. ,  E_j = prod_{j<u<=7} alpha_u
// Against one position at a time: 17 instead of 24 multiply-adds per state element and tile, no serial chain but the
// eight-term solve, and one reduction over lanes per (row, position) of which 32 go together.  All of it in fp32.
// Positions beyond the end of a segment have decay 1 and E_j = 0.  The activation rows behind a segment's end belong to the
// next sequence, and a zero coefficient does not silence an infinity or a NaN: the partial tile a segment may end with is
// copied row by row, and the rest of it is zeroed.
// The tiles arrive through a ring of shared-memory stages: a producer thread issues a tile's four or five copies (tensor
// copies of eight rows; one bulk copy per row and piece, 25 a tile, took 1900 cycles to issue and set the pace), the
// consumer warps only wait for bytes and hand stages back - no block-wide barrier in the loop.
constexpr int SC_POS = 8, SC_MAXSTAGES = 6;
constexpr int REC_SSM = 80;       // M[8][8] P[8] E[8]
constexpr int REC_GDN = 152;      // MK[8][8] MQ[8][8] P[8] E[8] beta[8]
// record slot of tile t of segment number s that starts at row0: tiles of different segments never share one
__device__ __forceinline__ int rec_slot(int row0, int s, int t) { return row0 / SC_POS + s + t; }
__device__ __forceinline__ void bulk_tile(void *dst_smem, const void *src, uint32_t bytes, uint64_t *bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 :: "r"(smem_u32(dst_smem)), "l"(src), "r"(bytes), "r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ void tensor_tile(void *dst_smem, const CUtensorMap *map, int x, int y, uint64_t *bar) {
    asm volatile("cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
                 :: "r"(smem_u32(dst_smem)), "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t *bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" :: "r"(smem_u32(bar)) : "memory");
}
// rows cnt .. 7 of a tile of W-float rows, by one warp
template <int W>
__device__ __forceinline__ void zero_tail(float *tile, int cnt, int lane) {
#pragma unroll 1
    for (int i = cnt * W + 4 * lane; i < SC_POS * W; i += 128) *reinterpret_cast<float4 *>(tile + i) = make_float4(0.f, 0.f, 0.f, 0.f);
}

// grid = (tiles, segments), eight warps: warp i takes position i of the tile
template <int EPL>
__global__ void __launch_bounds__(256) pf_gram_kernel(const PfScanArgs a) {
    constexpr int N = 32 * EPL;
    __shared__ float G[SC_POS][SC_POS];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, t = blockIdx.x;
    pdl_wait();
    const int4 sg = __ldcg(a.segs + blockIdx.y);
    const int row0 = sg.y, cnt = min(SC_POS, sg.z - t * SC_POS);
    if (cnt <= 0) return;
    if (warp < cnt) {
        const float *x = a.xbc + (size_t)(row0 + t * SC_POS) * a.convd + a.di;
        float c[EPL], b[SC_POS][EPL];
#pragma unroll
        for (int e = 0; e < EPL; ++e) c[e] = __ldcg(x + (size_t)warp * a.convd + N + e * 32 + lane);
#pragma unroll
        for (int j = 0; j < SC_POS; ++j)
#pragma unroll
            for (int e = 0; e < EPL; ++e) b[j][e] = j <= warp ? __ldcg(x + (size_t)j * a.convd + e * 32 + lane) : 0.f;
        float d[SC_POS];
#pragma unroll
        for (int j = 0; j < SC_POS; ++j) {
            d[j] = 0.f;
#pragma unroll
            for (int e = 0; e < EPL; ++e) d[j] = fmaf(c[e], b[j][e], d[j]);
        }
        const float g = xreduce<SC_POS>(d, lane);            // lanes 4 j .. 4 j + 3 hold C_i . B_j
        if ((lane & 3) == 0) G[warp][lane >> 2] = g;
    }
    __syncthreads();
    float *rec = a.rec + (size_t)rec_slot(row0, blockIdx.y, t) * a.heads * REC_SSM;
    for (int idx = tid; idx < a.heads * SC_POS; idx += 256) {
        const int i = idx / a.heads, h = idx - i * a.heads;
        const float *dv = a.dtv + (size_t)(row0 + t * SC_POS) * 2 * a.heads + h;
        float dt[SC_POS], dec[SC_POS];
#pragma unroll
        for (int j = 0; j < SC_POS; ++j) {
            dt[j] = j < cnt ? __ldcg(dv + (size_t)j * 2 * a.heads) : 0.f;
            dec[j] = j < cnt ? __ldcg(dv + (size_t)j * 2 * a.heads + a.heads) : 1.f;
        }
        float m[SC_POS], prod = 1.f, tail = 1.f, ei = 0.f;
#pragma unroll
        for (int j = SC_POS - 1; j >= 0; --j) {
            m[j] = 0.f;
            if (j <= i) { m[j] = i < cnt ? G[i][j] * prod * dt[j] : 0.f; prod *= dec[j]; }
            if (j == i) ei = tail * dt[j];
            tail *= dec[j];
        }
        float4 *out = reinterpret_cast<float4 *>(rec + (size_t)h * REC_SSM + i * SC_POS);
        out[0] = make_float4(m[0], m[1], m[2], m[3]); out[1] = make_float4(m[4], m[5], m[6], m[7]);
        rec[(size_t)h * REC_SSM + 64 + i] = prod; rec[(size_t)h * REC_SSM + 72 + i] = ei;
    }
    pdl_trigger();
}

// The Mamba-2 scan.  grid = (strips of NW * RW state rows, segments); NW consumer warps and one producer warp.  A warp
// owns RW rows of the [heads * P][N] state (they may belong to two heads) for the whole segment, lane l holding N / 32
// values of each.  Bound by latency within a tile at few rows, by reading B and C out of shared memory (every warp reads
// them all) and the fp32 pipes at many.  Few warps of many rows read less, many warps hide more: up to 24 rows a block four
// warps are faster (0.5B-class, 512 positions, 16 rows: prompt pass 6.15 ms with eight warps, 5.94 with four), at 40 rows
// eight (3B-class, 2048 positions: 52.2 ms, 54.7 with four warps of nine).  (Two blocks of eight warps fit an SM at N = 64.)
__host__ __device__ constexpr int sc_stage_floats(int N, int CR) { return SC_POS * (2 * N + 2 * CR) + 4 * REC_SSM; }

template <int EPL, int RW, int NW>
__global__ void __launch_bounds__(NW * 32 + 32, EPL == 2 && NW == 8 ? 2 : 1)
pf_ssm_kernel(const PfScanArgs a, const __grid_constant__ CUtensorMap mBC, const __grid_constant__ CUtensorMap mX,
              const __grid_constant__ CUtensorMap mZ, const int stages) {
    constexpr int N = 32 * EPL, VW = EPL < 4 ? EPL : 4, NVEC = EPL / VW, NP = EPL / 2, PPV = NP / NVEC;
    constexpr int CR = NW * RW, STG = sc_stage_floats(N, CR), RWP = (RW + 1) & ~1;
    constexpr int BCW = 2 * N < 256 ? 2 * N : 256;                             // columns of one B | C copy
    extern __shared__ __align__(128) float sm_raw[];
    float *sm = sm_raw + ((128u - (smem_u32(sm_raw) & 127u)) & 127u) / 4;
    __shared__ __align__(16) float2 es[NW][SC_POS + 1][RWP];             // per warp: E_j x_j of its rows, then P_7; each twice
    __shared__ __align__(8) uint64_t full[SC_MAXSTAGES], empty[SC_MAXSTAGES];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int R0 = blockIdx.x * CR, Rw = R0 + warp * RW;                       // first row of the block / of the warp
    if (tid < stages) { mbar_init(&full[tid], 1); mbar_init(&empty[tid], NW); mbar_fence_init(); }
    pdl_wait();
    pdl_trigger();                    // behind the wait: the attention of the same block, which runs beside this kernel, counts on it
    __syncthreads();
    const int4 sg = __ldcg(a.segs + blockIdx.y);
    const int b = sg.x, row0 = sg.y, n = sg.z, slot_out = sg.w;
    const int slot_in = a.nslot == 1 ? 0 : __ldcg(a.slot + b);
    if ((unsigned)slot_in >= (unsigned)a.nslot || (unsigned)slot_out >= (unsigned)a.nslot) {
        if (tid == 0) atomicCAS(a.status, 0, (int)HS_ERR_DEVICE);
        return;
    }
    const int ntile = (n + SC_POS - 1) / SC_POS;
    const int h0 = R0 / a.P, nh = (min(R0 + CR, a.di) - 1) / a.P - h0 + 1;     // heads of the block's rows (at most 4)
    bool ok = true;
    if (warp == NW) {
        // ---- producer: the whole tiles, then the partial one
        const float *rec = a.rec + ((size_t)rec_slot(row0, blockIdx.y, 0) * a.heads + h0) * REC_SSM;
        const uint32_t rbytes = (uint32_t)nh * REC_SSM * 4;
        const int whole = n / SC_POS, tail = n % SC_POS;
        int s = 0; uint32_t ph = 0;
        if (lane == 0) {
            for (int t = 0; t < whole; ++t) {
                if (!mbar_wait_n(&empty[s], ph ^ 1u, 1 << 20)) { ok = false; break; }
                float *dst = sm + (size_t)s * STG;
                const int y = row0 + t * SC_POS;
                mbar_expect_tx(&full[s], (uint32_t)SC_POS * (2 * N + 2 * CR) * 4 + rbytes);
#pragma unroll
                for (int q = 0; q < 2 * N / BCW; ++q) tensor_tile(dst + q * SC_POS * BCW, &mBC, a.di + q * BCW, y, &full[s]);
                tensor_tile(dst + SC_POS * 2 * N, &mX, R0, y, &full[s]);
                tensor_tile(dst + SC_POS * (2 * N + CR), &mZ, R0, y, &full[s]);
                bulk_tile(dst + SC_POS * (2 * N + 2 * CR), rec, rbytes, &full[s]);
                rec += (size_t)a.heads * REC_SSM;
                if (++s == stages) { s = 0; ph ^= 1u; }
            }
        }
        s = whole % stages; ph = (uint32_t)(whole / stages) & 1u;
        ok = __all_sync(0xffffffffu, ok);
        if (ok && tail) ok = __all_sync(0xffffffffu, mbar_wait_n(&empty[s], ph ^ 1u, 1 << 20));
        if (ok && tail) {
            float *dst = sm + (size_t)s * STG, *dx = dst + SC_POS * 2 * N, *dz = dx + SC_POS * CR;
#pragma unroll
            for (int q = 0; q < 2 * N / BCW; ++q) zero_tail<BCW>(dst + q * SC_POS * BCW, tail, lane);
            zero_tail<CR>(dx, tail, lane); zero_tail<CR>(dz, tail, lane);
            __syncwarp();
            if (lane == 0) {
                mbar_expect_tx(&full[s], (uint32_t)tail * (2 * N + 2 * CR) * 4 + rbytes);
                const float *x = a.xbc + (size_t)(row0 + whole * SC_POS) * a.convd, *z = a.zx + (size_t)(row0 + whole * SC_POS) * a.in_ld;
#pragma unroll 1
                for (int i = 0; i < tail; ++i) {
#pragma unroll
                    for (int q = 0; q < 2 * N / BCW; ++q) bulk_tile(dst + q * SC_POS * BCW + i * BCW, x + (size_t)i * a.convd + a.di + q * BCW, BCW * 4, &full[s]);
                    bulk_tile(dx + i * CR, x + (size_t)i * a.convd + R0, CR * 4, &full[s]);       // (columns beyond di: B, never live)
                    bulk_tile(dz + i * CR, z + (size_t)i * a.in_ld + R0, CR * 4, &full[s]);
                }
                bulk_tile(dz + SC_POS * CR, a.rec + ((size_t)rec_slot(row0, blockIdx.y, whole) * a.heads + h0) * REC_SSM, rbytes, &full[s]);
            }
        }
    } else {
        float *base = a.state + (size_t)b * a.nslot * a.state_elems;
        f2 st[RW][NP];
#pragma unroll
        for (int r = 0; r < RW; ++r)
#pragma unroll
            for (int v = 0; v < NVEC; ++v) {
                const float *src = base + (size_t)slot_in * a.state_elems + (size_t)(Rw + r) * N + v * (32 * VW) + lane * VW;
                float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
                if (Rw + r < a.di) {
                    if (VW == 4) x = __ldcg(reinterpret_cast<const float4 *>(src));
                    else { const float2 y = __ldcg(reinterpret_cast<const float2 *>(src)); x.x = y.x; x.y = y.y; }
                }
                st[r][v * PPV] = pk2(x.x, x.y);
                if (VW == 4) st[r][v * PPV + PPV - 1] = pk2(x.z, x.w);
            }
        // rows of the warp are finished in groups of four (eight positions x four rows are one transposing reduction) and
        // one of the remaining GR
        constexpr int G4 = RW / 4, GR = RW % 4, GT = G4 + (GR ? 1 : 0), GRX = GR ? GR : 1;
        static_assert(GR != 3, "the last group has one or two rows");
        struct Out { int i, col, row, head; float D; bool live; };
        auto outputs = [&](int r_lo, int G) {
            const int lpv = 32 / (SC_POS * G), v = lane / lpv;
            Out o; o.i = v / G; const int r = r_lo + v % G;
            o.col = warp * RW + r; o.row = Rw + r; o.live = lane % lpv == 0 && o.row < a.di;
            const int hd = min(o.row, a.di - 1) / a.P; o.head = (hd - h0) * REC_SSM; o.D = a.D[hd];
            return o;
        };
        Out og[GT];
#pragma unroll
        for (int g = 0; g < GT; ++g) og[g] = outputs(4 * g, g < G4 ? 4 : GRX);
        // coefficient lanes: value (j, r) of the update
        constexpr int NQ = (SC_POS * RW + 31) / 32;
        int e_head[NQ], e_j[NQ], e_r[NQ];
#pragma unroll
        for (int q = 0; q < NQ; ++q) {
            const int idx = lane + 32 * q;
            e_j[q] = idx / RW; e_r[q] = idx - e_j[q] * RW;
            e_head[q] = (min(Rw + e_r[q], a.di - 1) / a.P - h0) * REC_SSM;
        }
        const int p_head = (min(Rw + min(lane, RW - 1), a.di - 1) / a.P - h0) * REC_SSM;
        int s = 0; uint32_t ph = 0;
#pragma unroll 1
        for (int t = 0; t < ntile; ++t) {
            if (!__all_sync(0xffffffffu, mbar_wait_n(&full[s], ph, 1 << 20))) { ok = false; break; }
            const float *sg_ = sm + (size_t)s * STG;
            const float *xs = sg_ + SC_POS * 2 * N, *zs = xs + SC_POS * CR, *rs = zs + SC_POS * CR;
            const int cnt = min(SC_POS, n - t * SC_POS);
            // position i of B (which = 0) or C (1): with N = 256 they are two copies, else one of 2 N columns
            auto vec = [&](int i, int which) { return sg_ + (2 * N > 256 ? which * SC_POS * N + i * N : i * 2 * N + which * N) + lane * VW; };
            // coefficients of the update, each stored as a pair
#pragma unroll
            for (int q = 0; q < NQ; ++q)
                if (lane + 32 * q < SC_POS * RW) {
                    const float v = rs[e_head[q] + 72 + e_j[q]] * xs[e_j[q] * CR + warp * RW + e_r[q]];
                    es[warp][e_j[q]][e_r[q]] = make_float2(v, v);
                }
            if (lane < RW) { const float v = rs[p_head + 71]; es[warp][SC_POS][lane] = make_float2(v, v); }
            // products of the old state with C of every position
            float va[G4 ? G4 : 1][SC_POS * 4], vb[SC_POS * GRX];
#pragma unroll
            for (int i = 0; i < SC_POS; ++i) {
                f2 Cv[NP];
#pragma unroll
                for (int v = 0; v < NVEC; ++v) {
                    const float *p = vec(i, 1) + v * (32 * VW);
                    if (VW == 4) { const float4 x = *reinterpret_cast<const float4 *>(p); Cv[v * PPV] = pk2(x.x, x.y); Cv[v * PPV + PPV - 1] = pk2(x.z, x.w); }
                    else { const float2 x = *reinterpret_cast<const float2 *>(p); Cv[0] = pk2(x.x, x.y); }
                }
#pragma unroll
                for (int r = 0; r < RW; ++r) {
                    f2 y = mul2(st[r][0], Cv[0]);
#pragma unroll
                    for (int e = 1; e < NP; ++e) y = fma2(st[r][e], Cv[e], y);
                    float lo, hi;
                    up2(y, lo, hi);
                    if (r < 4 * G4) va[G4 ? r / 4 % (G4 ? G4 : 1) : 0][i * 4 + r % 4] = lo + hi;
                    else vb[i * GRX + (r - 4 * G4) % GRX] = lo + hi;
                }
            }
            __syncwarp();                 // es complete
            // S <- P_7 S + sum_j e_j B_j
#pragma unroll
            for (int r = 0; r < RW; ++r) {
                const f2 p7 = *reinterpret_cast<const f2 *>(&es[warp][SC_POS][r]);
#pragma unroll
                for (int e = 0; e < NP; ++e) st[r][e] = mul2(p7, st[r][e]);
            }
#pragma unroll
            for (int j = 0; j < SC_POS; ++j) {
                f2 Bv[NP];
#pragma unroll
                for (int v = 0; v < NVEC; ++v) {
                    const float *p = vec(j, 0) + v * (32 * VW);
                    if (VW == 4) { const float4 x = *reinterpret_cast<const float4 *>(p); Bv[v * PPV] = pk2(x.x, x.y); Bv[v * PPV + PPV - 1] = pk2(x.z, x.w); }
                    else { const float2 x = *reinterpret_cast<const float2 *>(p); Bv[0] = pk2(x.x, x.y); }
                }
#pragma unroll
                for (int r = 0; r < RW; ++r) {
                    const f2 ee = *reinterpret_cast<const f2 *>(&es[warp][j][r]);
#pragma unroll
                    for (int e = 0; e < NP; ++e) st[r][e] = fma2(ee, Bv[e], st[r][e]);
                }
            }
            // outputs: reduce over lanes, add what the tile's own positions contribute, gate
            auto finish = [&](float tot, const Out &o) {
                if (!o.live || o.i >= cnt) return;
                const float4 ma = *reinterpret_cast<const float4 *>(rs + o.head + o.i * SC_POS), mb = *reinterpret_cast<const float4 *>(rs + o.head + o.i * SC_POS + 4);
                const float *xc = xs + o.col;
                float y = rs[o.head + 64 + o.i] * tot + o.D * xc[o.i * CR], w = ma.x * xc[0];
                y = fmaf(ma.y, xc[CR], y); w = fmaf(ma.z, xc[2 * CR], w); y = fmaf(ma.w, xc[3 * CR], y);
                w = fmaf(mb.x, xc[4 * CR], w); y = fmaf(mb.y, xc[5 * CR], y); w = fmaf(mb.z, xc[6 * CR], w); y = fmaf(mb.w, xc[7 * CR], y);
                a.g[(size_t)(row0 + t * SC_POS + o.i) * a.gw + o.row] = (y + w) * silu_f(zs[o.i * CR + o.col]);
            };
#pragma unroll
            for (int g = 0; g < G4; ++g) finish(xreduce<SC_POS * 4>(va[g], lane), og[g]);
            if (GR) finish(xreduce<SC_POS * GRX>(vb, lane), og[GT - 1]);
            __syncwarp();                 // es may be overwritten
            if (lane == 0) mbar_arrive(&empty[s]);
            if (++s == stages) { s = 0; ph ^= 1u; }
        }
#pragma unroll
        for (int r = 0; r < RW; ++r)
#pragma unroll
            for (int v = 0; v < NVEC; ++v) {
                float *p = base + (size_t)slot_out * a.state_elems + (size_t)(Rw + r) * N + v * (32 * VW) + lane * VW;
                float x0, x1, x2, x3;
                up2(st[r][v * PPV], x0, x1);
                if (Rw + r < a.di) {
                    if (VW == 4) { up2(st[r][v * PPV + PPV - 1], x2, x3); *reinterpret_cast<float4 *>(p) = make_float4(x0, x1, x2, x3); }
                    else *reinterpret_cast<float2 *>(p) = make_float2(x0, x1);
                }
            }
    }
    if (!ok && lane == 0) atomicCAS(a.status, 0, (int)HS_ERR_TIMEOUT);          // a copy never landed
    if (tid < CR && R0 + tid < a.di) shift_window(a, b, row0, n, R0 + tid);
    if (blockIdx.x == 0)
        for (int c = tid; c < 2 * N; c += NW * 32 + 32) shift_window(a, b, row0, n, a.di + c);
}

// DeltaNet: q and k of a tile L2-normalised (in place), the tile's record.  grid = (tiles, groups of eight heads, segments), a
// warp per (tile, head): every load of the tile is in flight at once, the products are summed over the lanes 32 at a time, nothing
// goes through shared memory.  (A block per (tile, head), warp = position, products out of shared memory: 19.4 us for 1600 rows
// of 16 heads.)
__global__ void __launch_bounds__(256) pf_gdn_gram_kernel(const PfScanArgs a) {
    const int lane = threadIdx.x & 31, t = blockIdx.x, h = blockIdx.y * 8 + (threadIdx.x >> 5);
    pdl_wait();
    const int4 sg = __ldcg(a.segs + blockIdx.z);
    const int row0 = sg.y, cnt = min(SC_POS, sg.z - t * SC_POS);
    if (cnt <= 0 || h >= a.heads) return;
    const float *gate = a.dtv + (size_t)(row0 + t * SC_POS) * 2 * a.heads + h;
    float2 *q = reinterpret_cast<float2 *>(a.xbc_rw + (size_t)(row0 + t * SC_POS) * a.convd + h * 64) + lane, *k = q + a.heads * 32;
    const size_t step = (size_t)a.convd / 2;
    float2 x[SC_POS], y[SC_POS];
    float alpha[SC_POS];
#pragma unroll
    for (int i = 0; i < SC_POS; ++i) {
        x[i] = y[i] = make_float2(0.f, 0.f); alpha[i] = 1.f;
        if (i < cnt) { x[i] = __ldcg(q + i * step); y[i] = __ldcg(k + i * step); alpha[i] = __ldcg(gate + (size_t)i * 2 * a.heads); }
    }
    const float beta = lane < cnt ? __ldcg(gate + (size_t)lane * 2 * a.heads + a.heads) : 0.f;       // lane i: of position i
    {
        float ss[2 * SC_POS];
#pragma unroll
        for (int i = 0; i < SC_POS; ++i) { ss[i] = x[i].x * x[i].x + x[i].y * x[i].y; ss[SC_POS + i] = y[i].x * y[i].x + y[i].y * y[i].y; }
        const float inv = rsqrtf(xreduce<2 * SC_POS>(ss, lane) + 1e-6f);                               // lanes 2 v and 2 v + 1: vector v
#pragma unroll
        for (int i = 0; i < SC_POS; ++i) {
            const float iq = __shfl_sync(0xffffffffu, inv, 2 * i), ik = __shfl_sync(0xffffffffu, inv, 2 * (SC_POS + i));
            x[i].x *= iq; x[i].y *= iq; y[i].x *= ik; y[i].y *= ik;
            if (i < cnt) { q[i * step] = x[i]; k[i * step] = y[i]; }
        }
    }
    float *rec = a.rec + ((size_t)rec_slot(row0, blockIdx.z, t) * a.heads + h) * REC_GDN;
    auto decay = [&](int i, int j) {            // prod_{j < u <= i} alpha_u
        float d = 1.f;
#pragma unroll
        for (int u = 0; u < SC_POS; ++u) if (u > j && u <= i) d *= alpha[u];
        return d;
    };
    // k_i . k_j, j < i, is number i (i - 1) / 2 + j; q_i . k_j, j <= i, number i (i + 1) / 2 + j
    float kk[32], qk[32], qk7[4];
#pragma unroll
    for (int i = 0; i < 32; ++i) kk[i] = 0.f;
#pragma unroll
    for (int i = 0; i < SC_POS; ++i)
#pragma unroll
        for (int j = 0; j <= i; ++j) {
            if (j < i) kk[i * (i - 1) / 2 + j] = y[i].x * y[j].x + y[i].y * y[j].y;
            const int e = i * (i + 1) / 2 + j;
            const float v = x[i].x * y[j].x + x[i].y * y[j].y;
            if (e < 32) qk[e] = v; else qk7[e - 32] = v;
        }
    const float dk = xreduce<32>(kk, lane), dq = xreduce<32>(qk, lane), dq7 = xreduce<4>(qk7, lane);
    int ik = 1, iq = 0;                         // this lane's positions
#pragma unroll
    for (int i = 1; i < SC_POS; ++i) { if (lane >= i * (i + 1) / 2) { ik = i + 1; iq = i; } }
    const float bk = __shfl_sync(0xffffffffu, beta, min(ik, SC_POS - 1));
    if (lane < 28) { const int j = lane - ik * (ik - 1) / 2; rec[ik * SC_POS + j] = bk * dk * decay(ik, j); }
    { const int j = lane - iq * (iq + 1) / 2; rec[64 + iq * SC_POS + j] = dq * decay(iq, j); }
    if ((lane & 7) == 0) { const int j = 4 + (lane >> 3); rec[64 + 7 * SC_POS + j] = dq7 * decay(7, j); }
#pragma unroll
    for (int u = 0; u < 2; ++u) {               // above the diagonals
        const int e = lane + 32 * u, i = e >> 3, j = e & 7;
        if (j >= i) rec[e] = 0.f;
        if (j > i) rec[64 + e] = 0.f;
    }
    if (lane < SC_POS) { rec[128 + lane] = decay(lane, -1); rec[136 + lane] = lane < cnt ? decay(SC_POS - 1, lane) : 0.f; rec[144 + lane] = beta; }
    pdl_trigger();
}

// The delta rule.  grid = (strips of 16 * RT value rows, heads, segments), four consumer warps and one producer warp; eight
// lanes share RT rows (columns 4 c .. 4 c + 3 and 32 + 4 c .. of lane c), the tile's k vectors stay in registers between
// the products and the update.  Every lane of a row gathers the eight right-hand sides and solves for the u_i itself:
// one exchange instead of eight.  (RT = 2 goes out with more blocks than SMs: registers for three on each.)
constexpr int GD_STG = (SC_POS * (128 + 32) + REC_GDN + 31) / 32 * 32, GD_STAGES = 4, GD_WARPS = 4, GD_THREADS = (GD_WARPS + 1) * 32;

template <int RT>
__global__ void __launch_bounds__(GD_THREADS, RT == 2 ? 3 : 1)
pf_gdn_kernel(const PfScanArgs a, const __grid_constant__ CUtensorMap mQK, const __grid_constant__ CUtensorMap mV) {
    __shared__ __align__(128) float sm[GD_STAGES * GD_STG];
    __shared__ __align__(8) uint64_t full[GD_STAGES], empty[GD_STAGES];
    const int h = blockIdx.y, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, cl = lane & 7;
    const int dv = a.P, nk = a.heads * 64, v0 = blockIdx.x * 16 * RT, vr = warp * 4 * RT + (lane >> 3) * RT;    // this thread's first row of the strip
    if (tid < GD_STAGES) { mbar_init(&full[tid], 1); mbar_init(&empty[tid], GD_WARPS); mbar_fence_init(); }
    pdl_wait();
    __syncthreads();
    const int4 sg = __ldcg(a.segs + blockIdx.z);
    const int b = sg.x, row0 = sg.y, n = sg.z, slot_out = sg.w;
    const int slot_in = a.nslot == 1 ? 0 : __ldcg(a.slot + b);
    if ((unsigned)slot_in >= (unsigned)a.nslot || (unsigned)slot_out >= (unsigned)a.nslot) {
        if (tid == 0) atomicCAS(a.status, 0, (int)HS_ERR_DEVICE);
        return;
    }
    const int ntile = (n + SC_POS - 1) / SC_POS;
    bool ok = true;
    if (warp == GD_WARPS) {
        // ---- producer: stage = q[8][64] k[8][64] v[8][16 RT] record; the whole tiles, then the partial one
        const float *rec = a.rec + ((size_t)rec_slot(row0, blockIdx.z, 0) * a.heads + h) * REC_GDN;
        const int whole = n / SC_POS, tail = n % SC_POS;
        int s = 0; uint32_t ph = 0;
        if (lane == 0) {
            for (int t = 0; t < whole; ++t) {
                if (!mbar_wait_n(&empty[s], ph ^ 1u, 1 << 20)) { ok = false; break; }
                float *dst = sm + (size_t)s * GD_STG;
                const int y = row0 + t * SC_POS;
                mbar_expect_tx(&full[s], SC_POS * (128 + 16 * RT) * 4 + REC_GDN * 4);
                tensor_tile(dst, &mQK, h * 64, y, &full[s]);
                tensor_tile(dst + 512, &mQK, nk + h * 64, y, &full[s]);
                tensor_tile(dst + 1024, &mV, 2 * nk + h * dv + v0, y, &full[s]);
                bulk_tile(dst + SC_POS * 160, rec, REC_GDN * 4, &full[s]);
                rec += (size_t)a.heads * REC_GDN;
                if (++s == GD_STAGES) { s = 0; ph ^= 1u; }
            }
        }
        s = whole % GD_STAGES; ph = (uint32_t)(whole / GD_STAGES) & 1u;
        ok = __all_sync(0xffffffffu, ok);
        if (ok && tail) ok = __all_sync(0xffffffffu, mbar_wait_n(&empty[s], ph ^ 1u, 1 << 20));
        if (ok && tail) {
            float *dst = sm + (size_t)s * GD_STG;
            zero_tail<64>(dst, tail, lane); zero_tail<64>(dst + 512, tail, lane); zero_tail<16 * RT>(dst + 1024, tail, lane);
            __syncwarp();
            if (lane == 0) {
                mbar_expect_tx(&full[s], (uint32_t)tail * (128 + 16 * RT) * 4 + REC_GDN * 4);
#pragma unroll 1
                for (int i = 0; i < tail; ++i) {
                    const float *x = a.xbc + (size_t)(row0 + whole * SC_POS + i) * a.convd;
                    bulk_tile(dst + i * 64, x + h * 64, 256, &full[s]);
                    bulk_tile(dst + 512 + i * 64, x + nk + h * 64, 256, &full[s]);
                    bulk_tile(dst + 1024 + i * 16 * RT, x + 2 * nk + h * dv + v0, 64 * RT, &full[s]);
                }
                bulk_tile(dst + SC_POS * 160, a.rec + ((size_t)rec_slot(row0, blockIdx.z, whole) * a.heads + h) * REC_GDN, REC_GDN * 4, &full[s]);
            }
        }
    } else {
        float *base = a.state + (size_t)b * a.nslot * a.state_elems + ((size_t)h * dv + v0 + vr) * 64 + 4 * cl;
        f2 s[RT][4];
#pragma unroll
        for (int r = 0; r < RT; ++r)
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const float4 x = __ldcg(reinterpret_cast<const float4 *>(base + (size_t)slot_in * a.state_elems + r * 64 + 32 * e));
                s[r][2 * e] = pk2(x.x, x.y); s[r][2 * e + 1] = pk2(x.z, x.w);
            }
        int sl = 0; uint32_t ph = 0;
#pragma unroll 1
        for (int t = 0; t < ntile; ++t) {
            if (!__all_sync(0xffffffffu, mbar_wait_n(&full[sl], ph, 1 << 20))) { ok = false; break; }
            const float *st = sm + (size_t)sl * GD_STG, *rs = st + SC_POS * 160;
            const int cnt = min(SC_POS, n - t * SC_POS);
            f2 kv[SC_POS][4];
            float dk[RT][SC_POS], dq[RT][SC_POS];
#pragma unroll
            for (int i = 0; i < SC_POS; ++i) {
                f2 qv[4];
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    const float4 x = *reinterpret_cast<const float4 *>(st + 512 + i * 64 + 32 * e + 4 * cl), y = *reinterpret_cast<const float4 *>(st + i * 64 + 32 * e + 4 * cl);
                    kv[i][2 * e] = pk2(x.x, x.y); kv[i][2 * e + 1] = pk2(x.z, x.w);
                    qv[2 * e] = pk2(y.x, y.y); qv[2 * e + 1] = pk2(y.z, y.w);
                }
#pragma unroll
                for (int r = 0; r < RT; ++r) {
                    float lo, hi;
                    up2(fma2(s[r][3], kv[i][3], fma2(s[r][2], kv[i][2], fma2(s[r][1], kv[i][1], mul2(s[r][0], kv[i][0])))), lo, hi);
                    dk[r][i] = lo + hi;
                    up2(fma2(s[r][3], qv[3], fma2(s[r][2], qv[2], fma2(s[r][1], qv[1], mul2(s[r][0], qv[0])))), lo, hi);
                    dq[r][i] = lo + hi;
                }
            }
            // transposing sums over the eight lanes of a row: lane c ends with position c
            auto xred8 = [&](float (&v)[SC_POS]) {
#pragma unroll
                for (int off = 4; off >= 1; off >>= 1) {
                    const bool up = (cl & off) != 0;
#pragma unroll
                    for (int q = 0; q < off; ++q) {
                        const float keep = up ? v[q + off] : v[q], send = up ? v[q] : v[q + off];
                        v[q] = keep + __shfl_xor_sync(0xffffffffu, send, off);
                    }
                }
                return v[0];
            };
            const float Pc = rs[128 + cl], bc = rs[144 + cl];
            float u[RT][SC_POS], qo[RT];
#pragma unroll
            for (int r = 0; r < RT; ++r) {
                const float sk = xred8(dk[r]);
                qo[r] = Pc * xred8(dq[r]);
                const float w = bc * (st[1024 + cl * 16 * RT + vr + r] - Pc * sk);
#pragma unroll
                for (int i = 0; i < SC_POS; ++i) u[r][i] = __shfl_sync(0xffffffffu, w, (lane & 24) + i);
            }
#pragma unroll
            for (int i = 1; i < SC_POS; ++i) {
                const float4 ma = *reinterpret_cast<const float4 *>(rs + i * SC_POS), mb = *reinterpret_cast<const float4 *>(rs + i * SC_POS + 4);
                const float mr[8] = {ma.x, ma.y, ma.z, ma.w, mb.x, mb.y, mb.z, mb.w};
#pragma unroll
                for (int r = 0; r < RT; ++r)
#pragma unroll
                    for (int j = 0; j < i; ++j) u[r][i] = fmaf(-mr[j], u[r][j], u[r][i]);
            }
            const float4 ma = *reinterpret_cast<const float4 *>(rs + 64 + cl * SC_POS), mb = *reinterpret_cast<const float4 *>(rs + 64 + cl * SC_POS + 4);
            const float4 ea = *reinterpret_cast<const float4 *>(rs + 136), eb = *reinterpret_cast<const float4 *>(rs + 140);
            const float p7 = rs[135], ee[8] = {ea.x, ea.y, ea.z, ea.w, eb.x, eb.y, eb.z, eb.w};
            __syncwarp();                 // the stage has been read
            if (lane == 0) mbar_arrive(&empty[sl]);
            if (++sl == GD_STAGES) { sl = 0; ph ^= 1u; }
            const f2 pp = pk2(p7, p7);
#pragma unroll
            for (int r = 0; r < RT; ++r) {
                float o = qo[r];
                o = fmaf(ma.x, u[r][0], o); o = fmaf(ma.y, u[r][1], o); o = fmaf(ma.z, u[r][2], o); o = fmaf(ma.w, u[r][3], o);
                o = fmaf(mb.x, u[r][4], o); o = fmaf(mb.y, u[r][5], o); o = fmaf(mb.z, u[r][6], o); o = fmaf(mb.w, u[r][7], o);
                if (cl < cnt) a.g[(size_t)(row0 + t * SC_POS + cl) * a.gw + h * dv + v0 + vr + r] = o * 0.125f;      // 1 / sqrt(64)
#pragma unroll
                for (int e = 0; e < 4; ++e) s[r][e] = mul2(pp, s[r][e]);
#pragma unroll
                for (int j = 0; j < SC_POS; ++j) {
                    const float c = ee[j] * u[r][j];
                    const f2 cc = pk2(c, c);
#pragma unroll
                    for (int e = 0; e < 4; ++e) s[r][e] = fma2(cc, kv[j][e], s[r][e]);
                }
            }
        }
#pragma unroll
        for (int r = 0; r < RT; ++r)
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                float x0, x1, x2, x3;
                up2(s[r][2 * e], x0, x1); up2(s[r][2 * e + 1], x2, x3);
                *reinterpret_cast<float4 *>(base + (size_t)slot_out * a.state_elems + r * 64 + 32 * e) = make_float4(x0, x1, x2, x3);
            }
    }
    if (!ok && lane == 0) atomicCAS(a.status, 0, (int)HS_ERR_TIMEOUT);
    if (tid < 16 * RT) shift_window(a, b, row0, n, 2 * nk + h * dv + v0 + tid);
    if (blockIdx.x == 0 && tid < 128) shift_window(a, b, row0, n, tid < 64 ? h * 64 + tid : nk + h * 64 + (tid - 64));
    pdl_trigger();
}

// per-head RMSNorm over the dv outputs, then the gate silu(z), in place; a warp per (row, head)
__global__ void __launch_bounds__(256) pf_gdn_out_kernel(const PfScanArgs a) {
    const int h = blockIdx.y * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31, dv = a.P;
    pdl_wait();
    if (h >= a.heads) return;
    float *o = a.g + (size_t)blockIdx.x * a.gw + h * dv;
    const float *z = a.zx + (size_t)blockIdx.x * a.in_ld + a.heads * (128 + dv) + h * dv;
    float x[2], zz[2];
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        const int j = lane + 32 * q;
        x[q] = j < dv ? __ldcg(o + j) : 0.f; zz[q] = j < dv ? __ldcg(z + j) : 0.f;
    }
    const float rstd = rsqrtf(warp_sum(x[0] * x[0] + x[1] * x[1]) / (float)dv + a.eps);
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        const int j = lane + 32 * q;
        if (j < dv) o[j] = x[q] * rstd * a.onorm[j] * silu_f(zz[q]);
    }
    pdl_trigger();
}

// ---- attention ----------------------------------------------------------------------------------------------
// grid = (tiles of 64 positions, query heads, segments); four warps of 16 query positions, tiles of 64 keys of the
// cache in two shared-memory stages.  Scores and P V on the warp-level tensor path with head + remainder operands,
// running softmax in registers.  The longest tiles (the last positions) go out first.
// In a parallel block it starts with the scan (beside), whose blocks are few, hold one SM each and leave the tensor path
// idle: 0.5B-class, 512 positions, 53 us of scan and 24 of attention per layer; pass one after the other / together
// 6.86 / 6.16 ms.  For that the two have to share an SM's registers: with 255 a thread here beside 128 in the scan they do not
// (0.5B-class, 1500 positions: 15.0 ms, with 216 registers 12.8).
constexpr int PA_Q = 64, PA_K = 64, PA_THREADS = 128;

template <int HD>
__device__ __forceinline__ void pf_attn_body(const PfAttnArgs &a, unsigned char *smraw) {
    constexpr int KS = HD + 8, NT = HD / 8, HC = HD / 8;
    __nv_bfloat16 *K_s = reinterpret_cast<__nv_bfloat16 *>(smraw), *V_s = K_s + 2 * PA_K * KS;      // [2][PA_K][KS] each
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g8 = lane >> 2, t4 = lane & 3;
    const int4 sg = __ldcg(a.segs + blockIdx.z);
    const int b = sg.x, row0 = sg.y, n = sg.z, qt = gridDim.x - 1 - blockIdx.x, h = blockIdx.y;
    const int q0 = qt * PA_Q;
    if (q0 >= n) return;
    const int base = __ldcg(a.kv_len + b);
    if (base < 0 || base > a.cap - n) return;        // reported by pf_prep_kernel
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
                    cp_async16(kd + j * KS + 8 * c, Kb + (size_t)(t * PA_K + j) * HD + 8 * c);
                    cp_async16(vd + j * KS + 8 * c, Vb + (size_t)(t * PA_K + j) * HD + 8 * c);
                } else {                              // finite values where the tile ends early
                    *reinterpret_cast<uint4 *>(kd + j * KS + 8 * c) = make_uint4(0, 0, 0, 0);
                    *reinterpret_cast<uint4 *>(vd + j * KS + 8 * c) = make_uint4(0, 0, 0, 0);
                }
            }
        }
        cp_async_commit();
    };
    // the queries: heads in registers, remainders in shared memory (for both 255 registers do not suffice)
    __nv_bfloat16 *Ql_s = V_s + 2 * PA_K * KS;                                                      // [PA_Q][KS]
    for (int idx = tid; idx < PA_Q * HC; idx += PA_THREADS) {
        const int j = idx / HC, c = idx - j * HC;
        if (q0 + j < n) cp_async16(Ql_s + j * KS + 8 * c, a.q + a.q_plane + (size_t)(row0 + q0 + j) * ld + h * HD + 8 * c);
        else *reinterpret_cast<uint4 *>(Ql_s + j * KS + 8 * c) = make_uint4(0, 0, 0, 0);
    }
    fetch(0);
    const int wq = q0 + warp * 16;                    // first position of this warp's rows, within the segment
    const __nv_bfloat16 *ql = Ql_s + (size_t)(warp * 16 + (lane & 15)) * KS + (lane >> 4) * 8;
    uint32_t qh_[HD / 16][4];
#pragma unroll
    for (int ks = 0; ks < HD / 16; ++ks)
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const int i = wq + g8 + (e & 1) * 8, c = ks * 16 + 2 * t4 + (e >> 1) * 8;
            const __nv_bfloat16 *p = a.q + (size_t)(row0 + i) * ld + h * HD + c;
            qh_[ks][e] = i < n ? __ldcg(reinterpret_cast<const uint32_t *>(p)) : 0u;
        }
    float O[NT][4];
#pragma unroll
    for (int nt = 0; nt < NT; ++nt) O[nt][0] = O[nt][1] = O[nt][2] = O[nt][3] = 0.f;
    float m_run[2] = {-INFINITY, -INFINITY}, l_run[2] = {0.f, 0.f};
#pragma unroll 1
    for (int t = 0; t < ntile; ++t) {
        fetch(t + 1);
        cp_async_wait_but_one();
        __syncthreads();
        const __nv_bfloat16 *kt = K_s + (t & 1) * PA_K * KS, *vt = V_s + (t & 1) * PA_K * KS;
        const int k0 = t * PA_K, last = base + wq + 15;            // last key any row of this warp may see
        if (k0 <= last) {
            float S[PA_K / 8][4];
#pragma unroll
            for (int nt = 0; nt < PA_K / 8; ++nt) S[nt][0] = S[nt][1] = S[nt][2] = S[nt][3] = 0.f;
#pragma unroll
            for (int ks = 0; ks < HD / 16; ++ks) {
                uint32_t ql_[4];
                ldsm_x4(ql_, ql + ks * 16);
#pragma unroll
                for (int np = 0; np < PA_K / 16; ++np) {
                    uint32_t bk[4];
                    ldsm_x4(bk, kt + (size_t)(np * 16 + (lane & 7) + (lane >> 4) * 8) * KS + ks * 16 + ((lane >> 3) & 1) * 8);
                    mma_bf16(S[2 * np], qh_[ks], bk[0], bk[1]); mma_bf16(S[2 * np + 1], qh_[ks], bk[2], bk[3]);
                    mma_bf16(S[2 * np], ql_, bk[0], bk[1]); mma_bf16(S[2 * np + 1], ql_, bk[2], bk[3]);
                }
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
            uint32_t ph[PA_K / 16][4], pl[PA_K / 16][4];
#pragma unroll
            for (int j = 0; j < PA_K / 16; ++j)
#pragma unroll
                for (int nt = 0; nt < 2; ++nt)
#pragma unroll
                    for (int r = 0; r < 2; ++r) {
                        const float p0 = S[2 * j + nt][2 * r], p1 = S[2 * j + nt][2 * r + 1];
                        const uint32_t hh = pack_bf16x2(p0, p1);
                        ph[j][r + 2 * nt] = hh;
                        pl[j][r + 2 * nt] = pack_bf16x2(p0 - __uint_as_float(hh << 16), p1 - __uint_as_float(hh & 0xffff0000u));
                    }
            // a tile's products add up in accumulators of their own: the tensor path truncates every sum, and over all keys of
            // a long prompt on one accumulator that is 2^-26 of the output per MMA.  Four pairs of columns at a time.
#pragma unroll
            for (int p0 = 0; p0 < NT / 2; p0 += 4) {
                float T[8][4];
#pragma unroll
                for (int q = 0; q < 8; ++q) T[q][0] = T[q][1] = T[q][2] = T[q][3] = 0.f;
#pragma unroll
                for (int j = 0; j < PA_K / 16; ++j)
#pragma unroll
                    for (int p = 0; p < 4; ++p) {
                        uint32_t bv[4];
                        ldsm_x4_t(bv, vt + (size_t)(j * 16 + (lane & 7) + ((lane >> 3) & 1) * 8) * KS + (p0 + p) * 16 + (lane >> 4) * 8);
                        mma_bf16(T[2 * p], ph[j], bv[0], bv[1]); mma_bf16(T[2 * p + 1], ph[j], bv[2], bv[3]);
                        mma_bf16(T[2 * p], pl[j], bv[0], bv[1]); mma_bf16(T[2 * p + 1], pl[j], bv[2], bv[3]);
                    }
#pragma unroll
                for (int q = 0; q < 8; ++q)
#pragma unroll
                    for (int e = 0; e < 4; ++e) O[2 * p0 + q][e] = fmaf(O[2 * p0 + q][e], corr[e >> 1], T[q][e]);
            }
        }
        __syncthreads();                              // everybody is done with this stage: the next fetch refills it
    }
    cp_async_wait_all();
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
template <int HD>
__global__ void __maxnreg__(HD == 128 ? 216 : 152) pf_attn_kernel(const PfAttnArgs a) {
    extern __shared__ __align__(16) unsigned char smraw[];
    if (!a.beside) pdl_wait();
    pf_attn_body<HD>(a, smraw);
    // beside the scan: one block holds the grid back until the scan is complete, so that the next kernel's wait covers both
    if (a.beside && blockIdx.x == gridDim.x - 1 && blockIdx.y == gridDim.y - 1 && blockIdx.z == gridDim.z - 1) pdl_wait();
    pdl_trigger();
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
constexpr size_t pa_smem(int hd) { return (size_t)(4 * PA_K + PA_Q) * (hd + 8) * 2; }

template <int EPL, int RW, int NW>
cudaError_t launch_scan(const PfScanArgs &a, cudaStream_t s) {
    constexpr size_t stage = (size_t)sc_stage_floats(32 * EPL, NW * RW) * 4, alone = 116 * 1024;
    static bool configured = false;
    if (!configured) {
        const cudaError_t e = allow_smem(pf_ssm_kernel<EPL, RW, NW>, 6 * stage + 128 > alone ? 6 * stage + 128 : alone);
        if (e != cudaSuccess) return e;
        configured = true;
    }
    const dim3 grid((a.di + NW * RW - 1) / (NW * RW), a.nseg);
    // at most one block per SM: ask for more than half of its shared memory, or the scheduler puts two on some SMs while
    // others idle (3B-class, 2048 positions: 780 instead of 530 us with the first form of this kernel)
    const bool spread = (int64_t)grid.x * grid.y <= 148;
    const int stages = spread ? 6 : 4;
    const size_t smem = spread && stages * stage + 128 < alone ? alone : stages * stage + 128;
    constexpr int N = 32 * EPL;
    CUtensorMap mBC, mX, mZ;
    cudaError_t e = hs_make_f32_map(&mBC, a.xbc, a.nrows, a.convd, a.convd, 2 * N < 256 ? 2 * N : 256, SC_POS);
    if (e == cudaSuccess) e = hs_make_f32_map(&mX, a.xbc, a.nrows, a.convd, a.convd, NW * RW, SC_POS);
    if (e == cudaSuccess) e = hs_make_f32_map(&mZ, a.zx, a.nrows, a.di, a.in_ld, NW * RW, SC_POS);
    if (e != cudaSuccess) return e;
    return launch_pdl(pf_ssm_kernel<EPL, RW, NW>, grid, dim3(NW * 32 + 32), smem, s, a, mBC, mX, mZ, stages);
}
template <int EPL>
cudaError_t launch_ssm_n(const PfScanArgs &a, cudaStream_t s) {
    const cudaError_t e = launch_pdl(pf_gram_kernel<EPL>, dim3((a.max_seg + SC_POS - 1) / SC_POS, a.nseg), dim3(256), 0, s, a);
    if (e != cudaSuccess) return e;
    // rows per block: the fewest that leave at most one block on each of the 148 SMs (the time of a tile grows with them)
    const int64_t rows = (int64_t)a.di * a.nseg;
    if (rows <= 148 * 8) return launch_scan<EPL, 2, 4>(a, s);
    if (rows <= 148 * 16) return launch_scan<EPL, 4, 4>(a, s);
    if (rows <= 148 * 24) return launch_scan<EPL, 6, 4>(a, s);
    return launch_scan<EPL, 5, 8>(a, s);
}

}  // namespace

int64_t pf_record_floats(int rows, int segs, int heads, bool gdn) { return (int64_t)(rows / SC_POS + 1 + segs) * heads * (gdn ? REC_GDN : REC_SSM); }

cudaError_t configure_prefill() {
    cudaError_t e = allow_smem(pf_attn_kernel<64>, pa_smem(64));
    if (e == cudaSuccess) e = allow_smem(pf_attn_kernel<128>, pa_smem(128));
    return e;
}

cudaError_t launch_pf_embed(const __nv_bfloat16 *E, int d, int V, const int4 *rows, int nrows, float *h, int32_t *status, cudaStream_t s) {
    // first kernel of a pass: plain stream order (its successors read control words that the pass before wrote)
    pf_embed_kernel<<<nrows, 128, 0, s>>>(E, d, V, rows, h, status);
    return cudaGetLastError();
}
cudaError_t launch_pf_prep(const PfPrepArgs &a, cudaStream_t s) {
    const int pairs = (a.qh + 2 * a.kvh) * a.hd / 2;
    return launch_pdl(pf_prep_kernel, dim3((a.nrows + PREP_ROWS - 1) / PREP_ROWS, a.nconv + (a.heads ? 1 : 0) + (a.qh ? (pairs + 255) / 256 : 0)), dim3(256), 0, s, a);
}
cudaError_t launch_pf_ssm(const PfScanArgs &a, cudaStream_t s, int64_t *launches) {
    *launches += 2;
    if (a.N == 64) return launch_ssm_n<2>(a, s);
    if (a.N == 128) return launch_ssm_n<4>(a, s);
    if (a.N == 256) return launch_ssm_n<8>(a, s);
    return cudaErrorInvalidValue;
}
cudaError_t launch_pf_gdn(const PfScanArgs &a, cudaStream_t s, int64_t *launches) {
    if (a.P > 64 || (a.P & 15)) return cudaErrorInvalidValue;
    *launches += 3;
    cudaError_t e = launch_pdl(pf_gdn_gram_kernel, dim3((a.max_seg + SC_POS - 1) / SC_POS, (a.heads + 7) / 8, a.nseg), dim3(256), 0, s, a);
    if (e != cudaSuccess) return e;
    // two rows per lane group halve the blocks: where 16-row strips would leave several on every SM
    const int RT = a.P % 32 == 0 && (int64_t)(a.P / 16) * a.heads * a.nseg > 2 * 148 ? 2 : 1;
    CUtensorMap mQK, mV;
    e = hs_make_f32_map(&mQK, a.xbc, a.nrows, a.convd, a.convd, 64, SC_POS);
    if (e == cudaSuccess) e = hs_make_f32_map(&mV, a.xbc, a.nrows, a.convd, a.convd, 16 * RT, SC_POS);
    if (e != cudaSuccess) return e;
    const dim3 grid(a.P / (16 * RT), a.heads, a.nseg);
    e = RT == 2 ? launch_pdl(pf_gdn_kernel<2>, grid, dim3(GD_THREADS), 0, s, a, mQK, mV) : launch_pdl(pf_gdn_kernel<1>, grid, dim3(GD_THREADS), 0, s, a, mQK, mV);
    if (e != cudaSuccess) return e;
    return launch_pdl(pf_gdn_out_kernel, dim3(a.nrows, (a.heads + 7) / 8), dim3(256), 0, s, a);
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

// What the tcgen05 projection kernels share: launch arguments, descriptors, and the epilogue of one group of eight
// activation rows.
#pragma once
#include "hs_internal.h"
#include "hs_device.cuh"

namespace hsd {

constexpr int TC_BM = 128;          // weight rows per CTA
constexpr int TC_BK = 64;           // K columns per stage: one 128-byte swizzle atom of bf16
// tcgen05 truncates when it adds a product to an accumulator.  Measured against exact sums (in-projections of K = 512 .. 8192,
// 8 .. 1024 MMAs on an accumulator): the finished sum is short by 1.3 .. 1.6e-8 of itself per MMA, 2^-26, and spreads by 0.6
// of that.  The epilogues put the mean back.
constexpr float TC_LOST = 1.f / 67108864.f;

struct TcArgs {
    int O, nk0, nk1;            // output rows; 64-column K blocks of segment 0 / 1
    int nrows, rpad, bnh;       // activation rows, rows per plane of the packed operand, rows per plane per CTA
    int ns;                     // shared-memory stages (at most TC_MAXSTAGES)
    int seg;                    // two-CTA tiles: K blocks per segment
    float found;                // 1 + what truncation took from a sum; two-CTA tiles in segments: what it takes per K block
    int rb, rb_inv;             // K split: activation rows of a tile each rank finishes (a multiple of 4, rb * S >= bnh); 65536 / rb rounded up
    float *out; int ldo;
    const float *resid; int rparts; int64_t rpstride;
    int32_t *status;
    // The packed operand may come without the 1/rms factor of its RMSNorm (a projection epilogue wrote it, see
    // pk_out): then ss_in[p * rpad + r], p < ss_parts, are partial sums of squares of activation row r and the
    // factor rsqrt(sum * inv_k + eps) is applied to the finished sums of that row.
    const float *ss_in; int ss_parts; float inv_k, eps; bool ss_by_row;      // ss_by_row: ss_in[r * ss_parts + p]
    // Packed output for the projection that consumes this one's result: bf16 head | remainder planes
    // [2][rpad][pk_ld] of (result * pk_nw[output row]), and (residual epilogue) the partial sums of squares
    // ss_out[tile of weight rows][rpad] of the results.  nullptr: not wanted.
    __nv_bfloat16 *pk_out; int pk_ld; const float *pk_nw; float *ss_out;
    const void *pf_ptr; long long pf_bytes;     // weights of the next projection, pulled into L2 before the wait
    int early_trigger;          // let the next kernel start before this one has waited (else when its accumulators are complete)
    int off_rx, off_misc;       // shared-memory carve-up behind the stages (bytes from the aligned base)
};

__device__ __forceinline__ void tma_load_2d(void *dst_smem, const CUtensorMap *map, int x, int y, uint64_t *bar) {
    asm volatile("cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
                 :: "r"(smem_u32(dst_smem)), "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(smem_u32(bar)) : "memory");
}
// the same for a weight tile: streamed once per step, so marked evict-first in L2
__device__ __forceinline__ void tma_load_2d_stream(void *dst_smem, const CUtensorMap *map, int x, int y, uint64_t *bar) {
    uint64_t pol;
    asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(pol));
    asm volatile("cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1, {%2, %3}], [%4], %5;"
                 :: "r"(smem_u32(dst_smem)), "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(smem_u32(bar)), "l"(pol) : "memory");
}
// shared-memory operand descriptor: K-major rows of 128 bytes, 128-byte swizzle, 8-row groups 1024 bytes apart
__device__ __forceinline__ uint64_t umma_desc(uint32_t smem_addr) {
    const uint32_t lo = ((smem_addr >> 4) & 0x3fffu) | (1u << 16);
    const uint32_t hi = (1024u >> 4) | (1u << 14) | (2u << 29);
    return ((uint64_t)hi << 32) | lo;
}
__device__ __forceinline__ void umma_bf16(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t idesc, uint32_t accumulate) {
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
                 "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, {%5, %6, %7, %8}, p;\n\t}"
                 :: "r"(tmem_d), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate), "r"(0u), "r"(0u), "r"(0u), "r"(0u) : "memory");
}
__device__ __forceinline__ void umma_commit(uint64_t *bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" :: "r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ void tmem_ld8(uint32_t taddr, uint32_t (&r)[8]) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]) : "r"(taddr));
}
__device__ __forceinline__ void split_bf16(float x, __nv_bfloat16 &h, __nv_bfloat16 &l) {
    h = __float2bfloat16_rn(x);
    l = __float2bfloat16_rn(x - __bfloat162float(h));
}

// 1/rms of an activation row whose partial sums of squares lie `stride` floats apart: sixteen loads at a time, added in order
__device__ __forceinline__ float tc_rstd(const TcArgs &a, const float *ss, int stride) {
    float t = 0.f;
    for (int p0 = 0; p0 < a.ss_parts; p0 += 16) {
        float x[16];
#pragma unroll
        for (int u = 0; u < 16; ++u) x[u] = p0 + u < a.ss_parts ? __ldcg(ss + (size_t)(p0 + u) * stride) : 0.f;
#pragma unroll
        for (int u = 0; u < 16; ++u) t += x[u];
    }
    return rsqrtf(t * a.inv_k + a.eps);
}

// Residual of NC consecutive activation rows r0 .. of weight row `row` (parts added in order); the loads are issued early, so that
// their trip to L2 hides behind the wait that precedes the epilogue proper.  (One part, the rule: nothing here touches a loaded
// value, so the thread does not stall before it has come to that wait.)
template <int NC>
__device__ __forceinline__ void tc_load_resid(const TcArgs &a, float (&res)[NC], int r0, int nvalid, int row) {
#pragma unroll
    for (int j = 0; j < NC; ++j) res[j] = 0.f;
    if (row >= a.O) return;
    const float *rp = a.resid + (size_t)r0 * a.ldo + row;
#pragma unroll
    for (int j = 0; j < NC; ++j) if (j < nvalid) res[j] = __ldcg(rp + (size_t)j * a.ldo);
    for (int p = 1; p < a.rparts; ++p)
#pragma unroll
        for (int j = 0; j < NC; ++j) if (j < nvalid) res[j] += __ldcg(rp + (size_t)p * a.rpstride + (size_t)j * a.ldo);
}

// Epilogue for NC = 4 or 8 consecutive activation rows r0 .. (indices inside the launch) of weight row `row`
// (v[j] = the finished sum of row r0 + j, 1/rms already applied); nvalid of them exist.  Every lane of the warp
// calls it (the SwiGLU pairing and the sums of squares shuffle).  res: the residual (tc_load_resid); nw: weight
// folded into the packed output.  Returns (residual epilogue with statistics) the warp's sum of squares of row
// r0 + lane / (32 / NC).
template <int EPI, int NC>
__device__ __forceinline__ float tc_finish(const TcArgs &a, float (&v)[NC], const float (&res)[NC], int r0, int nvalid, int row, float nw, int lane) {
    if (EPI == EPI_SWIGLU) {
        // weight rows come in (gate, up) pairs held by neighbouring lanes.  The even lane finishes the even
        // columns of the pair, the odd lane the odd ones, so both lanes work and each evaluates one SiLU per two
        // columns: lanes swap what the other needs (even sends its gate of column j + 1, odd its up of column j).
        const bool odd = row & 1;
        const bool st = (row | 1) < a.O;
#pragma unroll
        for (int j = 0; j < NC; j += 2) {
            const float got = __shfl_xor_sync(0xffffffffu, odd ? v[j] : v[j + 1], 1);
            const float gate = odd ? got : v[j], up = odd ? v[j + 1] : got;
            const int jj = j + (odd ? 1 : 0);
            if (st && jj < nvalid) {
                const float r = silu_f(gate) * up;
                if (a.pk_out) {
                    __nv_bfloat16 h, l;
                    split_bf16(r, h, l);
                    __nv_bfloat16 *p = a.pk_out + (size_t)(r0 + jj) * a.pk_ld + (row >> 1);
                    p[0] = h; p[(size_t)a.rpad * a.pk_ld] = l;
                } else {
                    a.out[(size_t)(r0 + jj) * a.ldo + (row >> 1)] = r;
                }
            }
        }
        return 0.f;
    } else {
        const bool st = row < a.O;
        if (EPI == EPI_RESID)
#pragma unroll
            for (int j = 0; j < NC; ++j) v[j] += res[j];
        float *p = a.out + (size_t)r0 * a.ldo + row;
#pragma unroll
        for (int j = 0; j < NC; ++j) if (st && j < nvalid) p[(size_t)j * a.ldo] = v[j];
        if (EPI == EPI_RESID && a.pk_out) {
            __nv_bfloat16 *ph = a.pk_out + (size_t)r0 * a.pk_ld + row;
            const size_t plane = (size_t)a.rpad * a.pk_ld;
            float ssq[NC];
#pragma unroll
            for (int j = 0; j < NC; ++j) {
                const bool live = st && j < nvalid;
                if (live) {
                    __nv_bfloat16 h, l;
                    split_bf16(v[j] * nw, h, l);
                    ph[(size_t)j * a.pk_ld] = h; ph[(size_t)j * a.pk_ld + plane] = l;
                }
                ssq[j] = live ? v[j] * v[j] : 0.f;
            }
            return xreduce<NC>(ssq, lane);
        }
        return 0.f;
    }
}

}  // namespace hsd

// Backward pass of the prefill attention under the same mask policy (for SWA-aware fine-tuning, Sec. 3.2.2:
// the adapted model is trained with the mask it will be served with).
//
// Given q, k, v, out, dout and the log-sum-exp rows of the forward pass:
//     P_ij   = exp(scale * q_i.k_j - lse_i)            for visible (i, j), else 0
//     dV_j   = sum_i P_ij dO_i
//     dP_ij  = dO_i . v_j,   delta_i = dO_i . out_i
//     dS_ij  = P_ij (dP_ij - delta_i)
//     dQ_i   = scale * sum_j dS_ij k_j,   dK_j = scale * sum_i dS_ij q_i
// with dK, dV summed over the query heads of a GQA group.
//
// This file holds the parameters and the small kernels around the product kernel of swaa_backward_tc.cuh: the row terms
// before it, the conversions of the fp32 accumulators after it.
#pragma once

#include "swaa_internal.cuh"
#include "swaa_ptx.cuh"

namespace swaa {

struct BackwardParams {
    const float* lse;        // [Hq, T] natural log (forward output)
    const float* lse2;       // [Hq, T] the same times log2(e), written with delta
    const float* delta;      // [Hq, T]
    float* dkv_accum;        // [2][B][sink_rows][Hkv][D] fp32, zeroed: dk, dv of the sink tiles, which are split over blocks
    int sink_tiles;          // key tiles that hold sink keys (their query range is cut into chunks), 0 for full attention
    int chunks;              // blocks per sink tile
    int key_tiles;           // key tiles of a sequence of max_seqlen
    float* dq_accum;         // [T, Hq, D] fp32, zeroed before the launch
    __nv_bfloat16* dk;       // [T, Hkv, D]
    __nv_bfloat16* dv;
    const int32_t* cu_seqlens;
    int B, T, Hq, Hkv, G;
    int max_seqlen;          // the launch covers sequences up to this length; a longer one is reported and skipped
    int window, n_sink, is_full;
    float scale;
};

constexpr int kBwdChunkTiles = 32;  // query tiles (64 rows) per block of a sink key tile

// delta[h, t] = sum_d out[t, h, d] * dout[t, h, d] and lse2 = lse * log2(e); D / 8 lanes per (t, h) row, 16 bytes of each
// input per lane, which also clear the row of the fp32 dq accumulator.  Bound by memory: 2 * 2 D bytes read and 4 D bytes
// written per row.
template <int D>
__global__ void backward_delta_kernel(const __nv_bfloat16* out, const __nv_bfloat16* dout,
                                      const float* lse, float* delta,
                                      float* lse2, float* dq_accum, int T, int Hq) {
    grid_wait();
    constexpr int kLanes = D / 8;
    const long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const long long row = idx / kLanes;
    const int l = (int)(idx % kLanes);
    const bool in = row < (long long)T * Hq;  // whole groups of kLanes lanes
    float acc = 0.f;
    if (in) {
        const uint4 a = reinterpret_cast<const uint4*>(out + row * D)[l];
        const uint4 b = reinterpret_cast<const uint4*>(dout + row * D)[l];
        const uint32_t av[4] = {a.x, a.y, a.z, a.w}, bv[4] = {b.x, b.y, b.z, b.w};
        float4* acc_row = reinterpret_cast<float4*>(dq_accum + row * D);
        acc_row[l] = make_float4(0.f, 0.f, 0.f, 0.f);
        acc_row[l + kLanes] = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const float2 x = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&av[e]));
            const float2 y = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&bv[e]));
            acc += x.x * y.x + x.y * y.y;
        }
    }
#pragma unroll
    for (int off = kLanes / 2; off > 0; off >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, off);
    if (in && l == 0) {
        const int t = (int)(row / Hq), h = (int)(row - (long long)t * Hq);
        delta[(size_t)h * T + t] = acc;
        lse2[(size_t)h * T + t] = lse[(size_t)h * T + t] * 1.4426950408889634f;
    }
}

// dq = bf16(dq_accum)
__global__ void backward_convert_dq_kernel(const float* acc, __nv_bfloat16* dq, size_t n) {
    grid_wait();
    const size_t i = ((size_t)blockIdx.x * blockDim.x + threadIdx.x) * 4;
    if (i + 3 < n) {
        const float4 v = *reinterpret_cast<const float4*>(acc + i);
        *reinterpret_cast<uint2*>(dq + i) = make_uint2(pack_bf16x2(v.x, v.y), pack_bf16x2(v.z, v.w));
    } else {
        for (size_t j = i; j < n; ++j) dq[j] = __float2bfloat16_rn(acc[j]);
    }
}

// dk, dv rows of the split key tiles = bf16(dkv_accum); one thread per four channels of one (b, row, kv head).
__global__ void backward_convert_dkv_kernel(const float* acc, __nv_bfloat16* dk,
                                            __nv_bfloat16* dv, const int32_t* cu_seqlens, int B,
                                            int T, int max_seqlen, int sink_rows, int Hkv, int D) {
    grid_wait();
    const size_t plane = (size_t)B * sink_rows * Hkv * D;
    const size_t e = ((size_t)blockIdx.x * blockDim.x + threadIdx.x) * 4;
    if (e >= plane) return;
    const size_t row = e / ((size_t)Hkv * D);  // b * sink_rows + j
    const int b = (int)(row / sink_rows), j = (int)(row - (size_t)b * sink_rows);
    const int seq_start = cu_seqlens[b], Lseq = cu_seqlens[b + 1] - seq_start;
    if (j >= Lseq || Lseq > max_seqlen || seq_start < 0 || seq_start + Lseq > T) return;
    const size_t dst = (size_t)(seq_start + j) * Hkv * D + (e - row * (size_t)Hkv * D);
    const float4 a = *reinterpret_cast<const float4*>(acc + e);
    const float4 c = *reinterpret_cast<const float4*>(acc + plane + e);
    *reinterpret_cast<uint2*>(dk + dst) = make_uint2(pack_bf16x2(a.x, a.y), pack_bf16x2(a.z, a.w));
    *reinterpret_cast<uint2*>(dv + dst) = make_uint2(pack_bf16x2(c.x, c.y), pack_bf16x2(c.z, c.w));
}

}  // namespace swaa

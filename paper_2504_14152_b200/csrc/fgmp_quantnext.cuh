// The next layer's activation quantizer as it runs in a GEMM's epilogue, and what it is given (fgmp_linear_quantize).
#pragma once
#include "fgmp_common.cuh"

// The activation quantizer of the NEXT layer, run on the accumulators in the epilogue (Section 4.2:
// the post-processing unit quantizes each output block to FP4 or FP8 from the FP32 partial sums).
// codes4 == nullptr: off.  The output row of length N is the next layer's K.
struct QuantNext {
    const float* fisher;                 // [N] per-channel sensitivity of the next layer's input
    float s4, k6, s8, inv8, tau;
    int mode, ratio, free8;
    uint8_t* codes4; uint8_t* sf; uint32_t* mask; uint8_t* codes8;
    fgmp_packed_header* header;
    int64_t MW;                          // mask words per output row
};

#ifdef __CUDACC__
// One row of 32 accumulator columns = two blocks of the next layer's activations: round to bf16 (what an
// unfused fgmp_linear would have stored), then the quantizer's steps in its order.  Returns the two mask bits.
__device__ __forceinline__ uint32_t quantize_chunk32(const QuantNext& q, int64_t M, int64_t N, int64_t row, int64_t col0, const uint32_t (&r)[32], float alpha)
{
    uint32_t bits = 0;
    if (row >= M) return 0u;
#pragma unroll
    for (int hb = 0; hb < 2; ++hb) {
        const int64_t col = col0 + 16 * hb;
        if (col + 16 > N) break;
        const int64_t kb = col >> 4;
        float v[16], f[16], dq4[16];
#pragma unroll
        for (int i = 0; i < 16; ++i) v[i] = __bfloat162float(__float2bfloat16_rn(__uint_as_float(r[16 * hb + i]) * alpha));
        const float4* fp = reinterpret_cast<const float4*>(q.fisher + col);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const float4 t = __ldg(fp + i);
            f[4 * i] = t.x; f[4 * i + 1] = t.y; f[4 * i + 2] = t.z; f[4 * i + 3] = t.w;
        }
        uint32_t sc = block_dynamic_scale(v, q.k6);
        uint32_t c4[2], c8[4];
        block_nvfp4(v, sc, q.s4, c4, dq4);
        float score;
        if (q.mode == 0) {
            score = weighted_sq_sum(v, dq4, f);
        } else {
            float dq8[16];
            block_fp8(v, q.inv8, q.s8, c8, dq8);
            score = weighted_sq_sum(dq4, dq8, f);
        }
        if (score > q.tau) {
            if (q.mode == 0) {
                float dq8[16];
                block_fp8(v, q.inv8, q.s8, c8, dq8);
            }
            *reinterpret_cast<uint4*>(q.codes8 + row * N + kb * 16) = make_uint4(c8[0], c8[1], c8[2], c8[3]);
            c4[0] = 0; c4[1] = 0; sc = 0;
            bits |= 1u << hb;
        }
        *reinterpret_cast<uint2*>(q.codes4 + (row * N) / 2 + kb * 8) = make_uint2(c4[0], c4[1]);
        q.sf[fgmp_sf_offset(row, kb, N)] = (uint8_t)sc;
    }
    return bits;
}
#endif

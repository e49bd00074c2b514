// fgmp_linear for batches of more than 16 tokens with operands of any mix of formats (Section 4.1 of the paper): the GEMM
// reads the packed weights and dequantizes them on their way to the tensor core.
//
// Every block, whatever its format, is exact in fp16 once its scale is folded in (E2M1 x E4M3 scale has at most 6
// significant bits, E4M3 has 4), so all four block-pair products are exact products of one tcgen05.mma kind::f16 with FP32
// accumulation.  The activations, which all weight tiles share, are expanded once to an fp16 plane; the weights are not:
// a warp takes a row of packed blocks from shared memory and writes its fp16 values to TENSOR memory, where the MMA takes
// its 128-row operand from.  What bounds what:
//   - expanding the weights to a plane first costs 2.7 bytes written and read for every packed byte, which is the whole
//     call at small batches (4096 x 4096, 48 tokens: 59 us with the plane);
//   - a 128 x 256 unit of weights takes about 1000 clocks of the SIMT pipes (1024 conversions at one per clock), so that
//     the MMAs (16 of N/2 clocks for N tokens) bound from 128 tokens on, the dequantization below;
//   - the operand from tensor memory leaves shared memory to the token tiles (from shared memory the 64 KiB of a
//     dequantized unit would be written and read there, 1024 clocks by themselves);
//   - L2 -> shared-memory traffic: one weight tile against a token tile of N needs N * 512 + 20 K bytes per 8 N clocks, 70
//     bytes per clock at N = 208; two weight tiles (TS = 2) that share the token tile need 42.
//
// Work is (group of TS weight tiles, token tile, 256-element K chunk) units in that order, split over the CTAs either in
// equal contiguous spans (stream-K: the partial sums of tiles shared by several CTAs are stored column by column and added
// up in CTA order by a kernel of their own, which has the whole chip's loads in flight: 43 MB at 203 tokens and 13824 weight
// rows, 20 us if the CTA that arrives last does it) or in whole tiles, whichever the model in mixed_plan says is faster.
//
// Warp roles: warp 0 = weights producer, warp 1 = MMA issuer and owner of the tensor memory, warp 2 = token-tile producer,
// warps 3-6 = epilogue, then the dequantization, NG groups of four warps that take the steps of 64 elements in turn.  Every
// wait is bounded.
#include <cuda.h>
#include <cuda_fp16.h>
#include <mutex>
#include "fgmp_common.cuh"
#include "fgmp_host.h"
#include "fgmp_ptx.cuh"
#include "fgmp_quantnext.cuh"

namespace {

constexpr int W_PROD = 0, W_MMA = 1, W_TOK = 2, W_EPI = 3, W_DEQ = 7;
// dequantization groups: as many as the registers of a thread allow (quantizing in the epilogue takes more of them)
constexpr int mx_groups(bool quant) { return quant ? 3 : 4; }
constexpr int mx_threads(bool quant) { return 32 * (W_DEQ + 4 * mx_groups(quant)); }
constexpr uint32_t STG_MASK = REC_BYTES, STG_HALF = STG_MASK + 256;      // a weight stage: record, mask, second halves of the FP8 blocks
constexpr uint32_t HALF_CAP = 5248;             // 656 FP8 blocks (32 %); with more the halves are read from global memory
constexpr uint32_t WSTAGE = STG_HALF + HALF_CAP;                         // 24064
constexpr int MAX_WSTAGES = 4, MAX_BSTAGES = 12, MAX_SLOTS = 8;
constexpr uint32_t MX_TMEM_COLS = 512;
constexpr size_t MX_SMEM_LIMIT = 232448;
constexpr uint32_t SW128_LO = 1u << 16, SW128_HI = (1024u >> 4) | (1u << 14) | (2u << 29);
constexpr uint32_t IDESC_F16 = (1u << 4) | ((uint32_t)(128 >> 4) << 24);          // f32 += f16 x f16, M = 128, K-major; N added at run time

struct MixedPlan {
    int ts;                              // weight tiles per unit
    uint32_t n_tok, tok_tiles, groups;   // tokens per tile (multiple of 16), token tiles, groups of ts weight tiles
    uint32_t chunks, tiles;              // tiles = groups * tok_tiles
    uint32_t grid, span, rest, quantum;  // a CTA's span in quanta of `quantum` units (1, or chunks: whole tiles)
    uint32_t wstages, bstages, slots, max_parts;
    double cost;                         // modelled clocks
};

struct MixedParams {
    const uint8_t* wblob; PackedLayout LW;
    const fgmp_packed_header* ha;
    void* Y; int64_t ldy; int y_is_bf16;
    int64_t M, N, K;
    int leave_nvfp4;                     // operands without any FP8 block are left to the all-NVFP4 GEMM, launched behind this kernel
    MixedPlan pl;
    int* status; float* parts;
    QuantNext q;
};

__device__ __forceinline__ uint64_t mx_desc(uint32_t lo)
{
    uint64_t d;
    asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "r"(lo), "r"(SW128_HI));
    return d;
}
// A (128 rows) from tensor memory: lane = row, two fp16 values of K per column
__device__ __forceinline__ void umma_f16_ta(uint32_t d_tmem, uint32_t a_tmem, uint64_t bdesc, uint32_t idesc, uint32_t accumulate)
{
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
                 "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}"
                 ::"r"(d_tmem), "r"(a_tmem), "l"(bdesc), "r"(idesc), "r"(accumulate) : "memory");
}
__device__ __forceinline__ uint32_t hmul2(uint32_t a, uint32_t b)
{
    uint32_t r;
    asm("mul.f16x2 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
    return r;
}
__device__ __forceinline__ uint32_t e4m3x2_to_f16x2(uint32_t two)
{
    uint32_t r;
    asm("cvt.rn.f16x2.e4m3x2 %0, %1;" : "=r"(r) : "h"((uint16_t)two));
    return r;
}
// eight E2M1 codes -> four pairs (all four bytes unpacked at once: byte by byte it takes 1.7 times as long)
__device__ __forceinline__ void e2m1x8_to_f16(uint32_t w, uint32_t* r)
{
    asm("{\n\t.reg .b8 a, b, c, d;\n\tmov.b32 {a, b, c, d}, %4;\n\tcvt.rn.f16x2.e2m1x2 %0, a;\n\tcvt.rn.f16x2.e2m1x2 %1, b;\n\t"
        "cvt.rn.f16x2.e2m1x2 %2, c;\n\tcvt.rn.f16x2.e2m1x2 %3, d;\n\t}" : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(w));
}

__device__ __forceinline__ uint32_t unit_begin(const MixedPlan& pl, uint32_t cta) { return (cta * pl.span + min(cta, pl.rest)) * pl.quantum; }
__device__ __forceinline__ uint32_t cta_of(const MixedPlan& pl, uint32_t u)
{
    const uint32_t i = u / pl.quantum, longer = pl.rest * (pl.span + 1);
    return i < longer ? i / (pl.span + 1) : pl.rest + (i - longer) / pl.span;
}

// packed activations -> fp16 plane [M, K] of values over the tensor scale; one thread per block
__global__ void __launch_bounds__(256) expand_f16_kernel(const uint8_t* blob, const uint8_t* wblob, int64_t rows, int64_t K, uint8_t* plane, int* status, int leave_nvfp4)
{
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const fgmp_packed_header* h = reinterpret_cast<const fgmp_packed_header*>(blob);
    if (!(h->magic == FGMP_MAGIC && h->version == FGMP_LAYOUT_VERSION && h->rows == rows && h->K == K && h->kind == 0u && h->fp8_scale_free == 0)) {
        if (blockIdx.x == 0 && threadIdx.x == 0) { atomicCAS(status, 0, (int)FGMP_ERR_INVALID_ARG); atomicExch(status + 1, 11); }
        return;
    }
    // operands without any FP8 block are multiplied as they are packed
    if (leave_nvfp4 && h->n_fp8 == 0 && reinterpret_cast<const fgmp_packed_header*>(wblob)->n_fp8 == 0) return;
    const PackedLayout L = fgmp_layout(rows, K, 0, 0);
    const uint32_t* pmask = reinterpret_cast<const uint32_t*>(blob + L.off_mask);
    const __half2 r8 = __float2half2_rn(__int_as_float((127 + h->fp8_log2_ratio) << 23));
    const uint32_t f8 = *reinterpret_cast<const uint32_t*>(&r8);
    const int64_t nblk = rows * L.KB;
    for (int64_t b = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; b < nblk; b += (int64_t)gridDim.x * blockDim.x) {
        const int64_t r = b / L.KB, kb = b - r * L.KB;
        uint32_t o[8];
        if ((pmask[r * L.MW + (kb >> 5)] >> (kb & 31)) & 1u) {
            const uint4 c = *reinterpret_cast<const uint4*>(blob + L.off_codes8 + (size_t)(r * K + kb * 16));
            const uint32_t w[4] = {c.x, c.y, c.z, c.w};
#pragma unroll
            for (int i = 0; i < 4; ++i) { o[2 * i] = hmul2(e4m3x2_to_f16x2(w[i] & 0xffffu), f8); o[2 * i + 1] = hmul2(e4m3x2_to_f16x2(w[i] >> 16), f8); }
        } else {
            const uint2 c = *reinterpret_cast<const uint2*>(blob + L.off_codes4 + (r * K) / 2 + kb * 8);
            const uint32_t sc = blob[L.off_sf + fgmp_sf_offset(r, kb, K)], d = e4m3x2_to_f16x2(sc | (sc << 8));
            e2m1x8_to_f16(c.x, o); e2m1x8_to_f16(c.y, o + 4);
#pragma unroll
            for (int i = 0; i < 8; ++i) o[i] = hmul2(o[i], d);
        }
        asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};"
                     ::"l"(plane + (size_t)(r * K + kb * 16) * 2), "r"(o[0]), "r"(o[1]), "r"(o[2]), "r"(o[3]), "r"(o[4]), "r"(o[5]), "r"(o[6]), "r"(o[7]) : "memory");
    }
}

// 32 consecutive values of a row of the result = two blocks of the next layer's activations
__device__ __forceinline__ void quantize_row32(const MixedParams& p, int64_t m, int64_t col, const uint32_t (&r)[32], float alpha)
{
    const uint32_t bits = quantize_chunk32(p.q, p.M, p.N, m, col, r, alpha);
    // the mask word's other bits belong to other threads; the last blocks of a row also clear the rest of its last word
    uint32_t* word = p.q.mask + m * p.q.MW + (col >> 9);
    const uint32_t pos = (uint32_t)(col >> 4) & 31u, own = col + 32 >= p.N ? 0xffffffffu << pos : 3u << pos;
    atomicAnd(word, ~own);
    if (bits) atomicOr(word, bits << pos);
}

// One warp's share of a tile's result: 32 token columns from column cc on, lane = weight row n (v: sums in units of alpha)
template <bool QUANT>
__device__ __forceinline__ void mixed_emit(const MixedParams& p, const uint32_t (&v)[32], int64_t n, int64_t m0, uint32_t cc, float alpha, int lane, uint32_t* turn)
{
    const int64_t m_end = min(p.M, m0 + p.pl.n_tok);
    if (QUANT) {
        // turned round in shared memory: lane = token, 32 consecutive values of n = two blocks of the next layer's activations
#pragma unroll
        for (int j = 0; j < 32; ++j) turn[j * 33 + lane] = v[j];
        __syncwarp();
        uint32_t r[32];
#pragma unroll
        for (int j = 0; j < 32; ++j) r[j] = turn[lane * 33 + j];
        __syncwarp();
        const int64_t m = m0 + cc + lane, col = n - lane;
        if (m < m_end && col < p.N) quantize_row32(p, m, col, r, alpha);
    } else if (n < p.N) {
        if (p.y_is_bf16) {
            __nv_bfloat16* y = reinterpret_cast<__nv_bfloat16*>(p.Y) + (m0 + cc) * p.ldy + n;
#pragma unroll
            for (int j = 0; j < 32; ++j)
                if (m0 + cc + j < m_end) y[j * p.ldy] = __float2bfloat16_rn(__uint_as_float(v[j]) * alpha);
        } else {
            float* y = reinterpret_cast<float*>(p.Y) + (m0 + cc) * p.ldy + n;
#pragma unroll
            for (int j = 0; j < 32; ++j)
                if (m0 + cc + j < m_end) y[j * p.ldy] = __uint_as_float(v[j]) * alpha;
        }
    }
}

// Epilogue warps: tensor-memory lane quadrant warp % 4, lane = weight row, column = token
template <int TS, bool QUANT>
__device__ __forceinline__ void mixed_epilogue(const MixedParams& p, uint32_t tmem_base, int warp, int lane, uint32_t u_begin, uint32_t u_end,
                                               uint32_t accf0, uint32_t acce0, volatile int* abort_flag, int t_w, float* extra)
{
    const MixedPlan& pl = p.pl;
    const uint32_t q = (uint32_t)warp & 3u, C = pl.chunks, NT = pl.n_tok, NP = (NT + 31u) & ~31u, row = 32u * q + lane;   // (NP: columns of a partial tile)
    const float alpha = __fmul_rn(__fmul_rn(p.ha->scale_fp4, __ldg(&reinterpret_cast<const fgmp_packed_header*>(p.wblob)->scale_fp4)),
                                  __int_as_float((127 + t_w) << 23));
    uint32_t* turn = reinterpret_cast<uint32_t*>(extra) + q * 32 * 33;
    uint32_t acc_phase = 0;
    bool ok = true;
    for (uint32_t u = u_begin; u < u_end && ok;) {
        const uint32_t tile = u / C, t_begin = tile * C, t_end = t_begin + C, seg_end = min(t_end, u_end);
        const bool whole = u == t_begin && seg_end == t_end;
        const uint32_t g = tile / pl.tok_tiles;
        const int64_t m0 = (int64_t)(tile % pl.tok_tiles) * NT;
        const uint32_t which = u == u_begin ? 0u : 1u;       // a CTA's first segment, or its last
        u = seg_end;
#pragma unroll 1
        for (int t = 0; t < TS; ++t) {
            const uint32_t wt = g * TS + t;
            const int64_t n = (int64_t)wt * 128 + row;
            if (!(ok = mbar_wait_warp(accf0 + 8 * t, acc_phase, abort_flag, p.status, 8))) break;
            tc_fence_after();
            const uint32_t d = tmem_base + ((q * 32u) << 16) + t * NT;
            const bool there = wt < (uint32_t)p.LW.tiles;
            float* mine = p.parts + ((size_t)(blockIdx.x * 2 + which) * TS + t) * NP * 128 + row;
            if (there)
#pragma unroll 1
                for (uint32_t cc = 0; cc < NT; cc += 32) {
                    uint32_t v[32];
                    tmem_ld32(d + cc, v);
                    if (whole) mixed_emit<QUANT>(p, v, n, m0, cc, alpha, lane, turn);
                    else
#pragma unroll
                        for (int j = 0; j < 32; ++j) __stcg(mine + (cc + j) * 128, __uint_as_float(v[j]));
                }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(acce0 + 8 * t);
        }
        acc_phase ^= 1u;
    }
}

// TS = weight tiles per unit.  QUANT: the next layer's activation quantizer in the epilogue instead of Y.
template <int TS, bool QUANT>
__global__ void __launch_bounds__(mx_threads(QUANT), 1)
mixed_kernel(const __grid_constant__ CUtensorMap tmB, const __grid_constant__ MixedParams p)
{
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
    const MixedPlan& pl = p.pl;
    const uint32_t BS = pl.bstages, WS = pl.wstages, R = pl.slots, NT = pl.n_tok, C = pl.chunks;
    // (no more groups than slots: a group that was further ahead could take an older phase of a slot's barrier for the one it waits for)
    const uint32_t NG = min((uint32_t)mx_groups(QUANT), R);
    const uint32_t b_bytes = NT * 128u;                  // token stage: NT rows x 64 elements, swizzled (a multiple of 2 KiB)
    uint8_t* wst0 = smem + BS * b_bytes;
    uint8_t* extra = wst0 + WS * TS * WSTAGE;            // QUANT: 4 x 32 x 33 floats
    uint64_t* bars = reinterpret_cast<uint64_t*>(extra + (QUANT ? 4 * 32 * 33 * 4 + 128 : 0));
    uint32_t* wmeta = reinterpret_cast<uint32_t*>(bars + 2 * MAX_WSTAGES + 2 * MAX_BSTAGES + 2 * MAX_SLOTS + 4);   // [stage][tile]: list start, steps
    uint32_t* tmem_slot = wmeta + MAX_WSTAGES * TS * 2;
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

    const int warp = warp_index(), lane = threadIdx.x & 31;
    // barriers: weight stage full / empty, token stage full / empty, dequantized step in tensor memory full / empty,
    // accumulators full / empty (one per weight tile)
    const uint32_t wf0 = smem_u32(bars), we0 = wf0 + 8 * MAX_WSTAGES, bf0 = we0 + 8 * MAX_WSTAGES, be0 = bf0 + 8 * MAX_BSTAGES;
    const uint32_t sf0 = be0 + 8 * MAX_BSTAGES, se0 = sf0 + 8 * MAX_SLOTS, accf0 = se0 + 8 * MAX_SLOTS, acce0 = accf0 + 16;
    const uint32_t slot_col = TS * NT;                   // tensor memory: TS accumulators of NT columns, then slots of 32

    const uint32_t u_begin = unit_begin(pl, blockIdx.x), u_end = unit_begin(pl, blockIdx.x + 1);
    const uint32_t wtiles = (uint32_t)p.LW.tiles, last_steps = (uint32_t)(p.K / 64) - 4u * (C - 1u);

    if (threadIdx.x == 0) {
        for (uint32_t s = 0; s < WS; ++s) { mbar_init(wf0 + 8 * s, 1); mbar_init(we0 + 8 * s, 4 * NG); }
        for (uint32_t s = 0; s < BS; ++s) { mbar_init(bf0 + 8 * s, 1); mbar_init(be0 + 8 * s, 1); }
        for (uint32_t s = 0; s < R; ++s) { mbar_init(sf0 + 8 * s, 4); mbar_init(se0 + 8 * s, 1); }
        for (int t = 0; t < TS; ++t) { mbar_init(accf0 + 8 * t, 1); mbar_init(acce0 + 8 * t, 4); }
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == W_MMA) tmem_alloc(smem_u32(tmem_slot), MX_TMEM_COLS);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = __shfl_sync(0xffffffffu, *tmem_slot, 0);
    const fgmp_packed_header* hw = reinterpret_cast<const fgmp_packed_header*>(p.wblob);
    const int ratio_w = __ldg(&hw->fp8_log2_ratio);
    // The weights go in over 2^t: an FP8 block needs no factor then if t is the ratio of its tensor scale to the NVFP4 one,
    // and fp16 holds every NVFP4 value (up to 2688) over 2^t as long as t >= -4.
    const int t_w = max(ratio_w, -4);

    const bool has_fp8 = __ldg(&hw->n_fp8) != 0, may_skip = p.leave_nvfp4 && !has_fp8;
    if (warp == W_PROD) {
        // ------------------------------------------------------------ weights producer (whole warp; lane 0 issues)
        // The packed weights are not written by whatever runs before this kernel: their first copies overlap its end.
        const uint2 mv = __ldg(reinterpret_cast<const uint2*>(hw));
        int ok = mv.x == FGMP_MAGIC && mv.y == FGMP_LAYOUT_VERSION && __ldg(&hw->rows) == p.N && __ldg(&hw->K) == p.K && __ldg(&hw->kind) == 1u &&
                 __ldg(&hw->error) == 0 && __ldg(&hw->fp8_scale_free) == 0;
        const bool bad = !ok;                            // (a skipped call has matching headers)
        const uint32_t* uptr = reinterpret_cast<const uint32_t*>(p.wblob + p.LW.off_uptr);
        uint32_t stage = 0, phase = 1, issued = 0;
        bool waited = may_skip;                          // (whether this kernel has anything to do is known only then)
        if (waited) {
            asm volatile("griddepcontrol.wait;" ::: "memory");
            if (p.ha->n_fp8 == 0) ok = 0;
        }
        for (uint32_t u = u_begin; u < u_end && ok; ++u, ++issued) {
            const uint32_t c = u % C, g = u / C / pl.tok_tiles;
            // lane t of the first TS: the list of weight tile t's unit
            const uint32_t tile = g * TS + lane, rec = tile * C + c;
            uint32_t st0 = 0, st1 = 0;
            if (lane < TS && tile < wtiles) { st0 = __ldg(uptr + rec); st1 = __ldg(uptr + rec + 1); }
            if (issued == WS && !waited) {
                // the status word may be looked at once the preceding kernel is done
                asm volatile("griddepcontrol.wait;" ::: "memory");
                waited = true;
            }
            if (lane == 0) ok = mbar_wait(we0 + 8 * stage, phase, abort_flag, p.status, 1) ? 1 : 0;
            ok = __shfl_sync(0xffffffffu, ok, 0);
            if (!ok) break;
            const uint32_t steps = st1 - st0, h = 2u * steps / 3u, staged = min(h * 16u, HALF_CAP);     // the list's words, then h steps of halves
            const bool there = lane < TS && tile < wtiles;
            const uint32_t mine = there ? REC_BYTES + 256u + staged : 0u;
            uint32_t all = mine;
            if (TS == 2) all += __shfl_down_sync(0xffffffffu, mine, 1);
            if (there) { wmeta[(stage * TS + lane) * 2] = st0 + (steps - h); wmeta[(stage * TS + lane) * 2 + 1] = staged; }
            __syncwarp();
            if (lane == 0) mbar_expect_tx(wf0 + 8 * stage, all);
            __syncwarp();
            if (there) {
                const uint32_t dst = smem_u32(wst0 + (stage * TS + lane) * WSTAGE), fb = wf0 + 8 * stage;
                bulk_load(dst, p.wblob + p.LW.off_rec + (size_t)rec * REC_BYTES, REC_BYTES, fb);
                bulk_load(dst + STG_MASK, p.wblob + p.LW.off_mask + (size_t)rec * 256, 256u, fb);
                if (staged) bulk_load(dst + STG_HALF, p.wblob + p.LW.off_ovf + (size_t)(st0 + (steps - h)) * 16, staged, fb);
            }
            __syncwarp();
            if (++stage == WS) { stage = 0; phase ^= 1; }
        }
        if (!waited) asm volatile("griddepcontrol.wait;" ::: "memory");
        if (bad && lane == 0) { *abort_flag = 1; atomicCAS(p.status, 0, (int)FGMP_ERR_INVALID_ARG); atomicExch(p.status + 1, 12); }
    } else {
        asm volatile("griddepcontrol.wait;" ::: "memory");
        asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    }
    if (QUANT && blockIdx.x == 0 && threadIdx.x == 32 * W_EPI) {
        fgmp_packed_header* h = p.q.header;
        h->magic = FGMP_MAGIC; h->version = FGMP_LAYOUT_VERSION; h->rows = p.M; h->K = p.N; h->scale_fp4 = p.q.s4;
        h->fp8_log2_ratio = p.q.ratio; h->n_fp8 = (p.q.tau == INFINITY) ? 0 : -1; h->tau_eff = 0.f; h->kind = 0; h->capacity = 0;
        h->error = 0; h->scale_fp8 = p.q.s8; h->fp8_scale_free = p.q.free8;
    }
    const bool skip = may_skip && p.ha->n_fp8 == 0;
    if (!skip && blockIdx.x == 0 && threadIdx.x == 32 * W_EPI) p.status[2] = 0;      // word 2: the all-NVFP4 GEMM has produced Y

    if (skip || warp == W_PROD) {
    } else if (warp == W_TOK) {
        // ------------------------------------------------------------ token-tile producer
        if (lane == 0) {
            uint32_t stage = 0, phase = 1;
            bool ok = true;
            for (uint32_t u = u_begin; u < u_end && ok; ++u) {
                const uint32_t c = u % C, m0 = (u / C) % pl.tok_tiles * NT, steps = c == C - 1 ? last_steps : 4u;
                for (uint32_t s = 0; s < steps; ++s) {
                    if (!(ok = mbar_wait(be0 + 8 * stage, phase, abort_flag, p.status, 2))) break;
                    mbar_expect_tx(bf0 + 8 * stage, b_bytes);
                    tma_load_2d(smem_u32(smem + stage * b_bytes), &tmB, (int32_t)(c * 256 + s * 64), (int32_t)m0, bf0 + 8 * stage);
                    if (++stage == BS) { stage = 0; phase ^= 1; }
                }
            }
        }
        __syncwarp();
    } else if (warp == W_MMA) {
        // ------------------------------------------------------------ MMA issuer (one elected lane)
        const uint32_t idesc = IDESC_F16 | ((NT >> 3) << 17), b_first = (smem_u32(smem) >> 4) | SW128_LO, b_step = b_bytes >> 4;
        uint32_t bst = 0, bph = 0, slot = 0, sph = 0, c = u_begin % C, acc_phase = 1, b_lo = b_first;
        bool first = true, ok = true;
        for (uint32_t u = u_begin; u < u_end && ok; ++u) {
            const uint32_t steps = c == C - 1 ? last_steps : 4u;
            const bool last_unit = c == C - 1 || u + 1 == u_end;
            for (uint32_t s = 0; s < steps && ok; ++s) {
                if (!(ok = mbar_wait_uniform(bf0 + 8 * bst, bph, abort_flag, p.status, 3))) break;
#pragma unroll
                for (int t = 0; t < TS; ++t) {
                    if (first && !(ok = mbar_wait_uniform(acce0 + 8 * t, acc_phase, abort_flag, p.status, 4))) break;
                    if (!(ok = mbar_wait_uniform(sf0 + 8 * slot, sph, abort_flag, p.status, 5))) break;
                    tc_fence_after();
                    const uint32_t d = tmem_base + t * NT, a = tmem_base + slot_col + slot * 32;
                    if (elect_one()) {
#pragma unroll
                        for (uint32_t k = 0; k < 4; ++k) umma_f16_ta(d, a + 8 * k, mx_desc(b_lo + 2 * k), idesc, k ? 1u : (first ? 0u : 1u));
                        umma_commit(se0 + 8 * slot);
                        if (last_unit && s + 1 == steps) umma_commit(accf0 + 8 * t);
                        if (t == TS - 1) umma_commit(be0 + 8 * bst);
                    }
                    __syncwarp();
                    if (++slot == R) { slot = 0; sph ^= 1; }
                }
                first = false;
                b_lo += b_step;
                if (++bst == BS) { bst = 0; bph ^= 1; b_lo = b_first; }
            }
            if (last_unit) { first = true; acc_phase ^= 1; }
            if (++c == C) c = 0;
        }
    } else if (warp >= W_DEQ + 4 * (int)NG) {
    } else if (warp >= W_DEQ) {
        // ------------------------------------------------------------ dequantization: thread = row of the weight tile
        // The groups take the steps in turn: step a of a unit is elements 64 (a / TS) .. of weight tile a % TS.
        const uint32_t group = (uint32_t)(warp - W_DEQ) >> 2, row = 32u * (warp & 3) + lane, r7 = row & 7u;
        const uint32_t quadrant = tmem_base + ((uint32_t)((warp & 3) * 32) << 16) + slot_col;
        const __half2 inv2 = __float2half2_rn(__int_as_float((127 - t_w) << 23)), f82 = __float2half2_rn(__int_as_float((127 + ratio_w - t_w) << 23));
        const uint32_t inv = *reinterpret_cast<const uint32_t*>(&inv2), f8 = *reinterpret_cast<const uint32_t*>(&f82);
        const bool scaled8 = ratio_w != t_w;             // (for every thread alike)
        uint32_t stage = 0, phase = 0, c = u_begin % C, slot = group % R, sph = group / R & 1u ? 0u : 1u, next = group;    // next: steps until the group's turn
        bool ok = true;
        for (uint32_t u = u_begin; u < u_end && ok; ++u) {
            const uint32_t steps = (c == C - 1 ? last_steps : 4u) * TS;
            if (!(ok = mbar_wait_warp(wf0 + 8 * stage, phase, abort_flag, p.status, 6))) break;
            const bool pair = TS == 2 && (u / C / pl.tok_tiles) * TS + 1 < wtiles;     // an odd number of weight tiles: the last group has one
            uint32_t m16s[TS], ats[TS], alls = 0;
#pragma unroll
            for (int t = 0; t < TS; ++t) {
                // the row's FP8 blocks lie one after the other in the list
                m16s[t] = 0; ats[t] = 0;
                if (has_fp8 && (t == 0 || pair)) {
                    const uint8_t* sb = wst0 + (stage * TS + t) * WSTAGE;
                    const uint16_t* before = reinterpret_cast<const uint16_t*>(sb + REC_KBSTART);
                    m16s[t] = reinterpret_cast<const uint16_t*>(sb + STG_MASK)[row];
                    uint32_t at = __popc(m16s[t]);
#pragma unroll
                    for (int o = 1; o < 8; o <<= 1) { const uint32_t y = __shfl_up_sync(0xffffffffu, at, o, 8); if ((lane & 7) >= o) at += y; }
                    ats[t] = 8u * (before[row >> 3] + at - __popc(m16s[t]));
                    if (8u * before[16] <= wmeta[(stage * TS + t) * 2 + 1]) alls |= 1u << t;
                }
            }
#pragma unroll 1
            for (; next < steps; next += NG) {
                const uint32_t t = next % TS, s = next / TS;
                uint32_t r[32];
                if (t == 0 || pair) {
                    const uint32_t sb = smem_u32(wst0 + (stage * TS + t) * WSTAGE), codes = sb + row * 128u, sfw = sb + REC_SF + (row & 31u) * 16u + (row >> 5) * 4u;
                    const uint32_t mt = TS == 2 && t ? m16s[TS - 1] : m16s[0], m16 = mt >> (4 * s);
                    const bool all = (alls >> t) & 1u;
                    uint32_t hg = (TS == 2 && t ? ats[TS - 1] : ats[0]) + 8u * __popc(mt & ((1u << (4 * s)) - 1u)), hs = sb + STG_HALF + hg;
                    uint4 q0, q1;
                    uint32_t sc;
                    asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(q0.x), "=r"(q0.y), "=r"(q0.z), "=r"(q0.w) : "r"(codes + (((2 * s) ^ r7) << 4)));
                    asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(q1.x), "=r"(q1.y), "=r"(q1.z), "=r"(q1.w) : "r"(codes + (((2 * s + 1) ^ r7) << 4)));
                    asm volatile("ld.shared.b32 %0, [%1];" : "=r"(sc) : "r"(sfw + 512u * s));
                    const uint32_t w[8] = {q0.x, q0.y, q0.z, q0.w, q1.x, q1.y, q1.z, q1.w};
                    uint2 hi[4];
#pragma unroll
                    for (uint32_t k = 0; k < 4; ++k) {
                        const uint32_t is8 = (m16 >> k) & 1u;
                        hi[k] = lds64_if(hs, is8 && all);
                        hs += 8u * is8;
                    }
                    if (!all) {
                        const uint8_t* half_g = p.wblob + p.LW.off_ovf + (size_t)wmeta[(stage * TS + t) * 2] * 16;
#pragma unroll
                        for (uint32_t k = 0; k < 4; ++k)
                            if ((m16 >> k) & 1u) { hi[k] = __ldg(reinterpret_cast<const uint2*>(half_g + hg)); hg += 8u; }
                        __syncwarp();
                    }
                    const uint32_t d01 = hmul2(e4m3x2_to_f16x2(sc & 0xffffu), inv), d23 = hmul2(e4m3x2_to_f16x2(sc >> 16), inv);
                    const uint32_t d[4] = {__byte_perm(d01, 0, 0x1010), __byte_perm(d01, 0, 0x3232), __byte_perm(d23, 0, 0x1010), __byte_perm(d23, 0, 0x3232)};
#pragma unroll
                    for (uint32_t k = 0; k < 4; ++k) {
                        e2m1x8_to_f16(w[2 * k], r + 8 * k); e2m1x8_to_f16(w[2 * k + 1], r + 8 * k + 4);
#pragma unroll
                        for (int e = 0; e < 8; ++e) r[8 * k + e] = hmul2(r[8 * k + e], d[k]);
                    }
                    if (has_fp8) {
                        // E4M3 codes 0..7 in the slot, 8..15 in the list; selected, not branched to: with 10 % FP8 blocks some
                        // row of a warp has one in nearly every column
#pragma unroll
                        for (uint32_t k = 0; k < 4; ++k) {
                            const bool is8 = (m16 >> k) & 1u;
                            const uint32_t v[4] = {w[2 * k], w[2 * k + 1], hi[k].x, hi[k].y};
#pragma unroll
                            for (int e = 0; e < 4; ++e) {
                                uint32_t a = e4m3x2_to_f16x2(v[e] & 0xffffu), b = e4m3x2_to_f16x2(v[e] >> 16);
                                if (scaled8) { a = hmul2(a, f8); b = hmul2(b, f8); }
                                r[8 * k + 2 * e] = is8 ? a : r[8 * k + 2 * e];
                                r[8 * k + 2 * e + 1] = is8 ? b : r[8 * k + 2 * e + 1];
                            }
                        }
                    }
                } else {
#pragma unroll
                    for (int e = 0; e < 32; ++e) r[e] = 0;
                }
                __syncwarp();
                if (!(ok = mbar_wait_warp(se0 + 8 * slot, sph, abort_flag, p.status, 7))) break;
                tc_fence_after();
                tmem_st32(quadrant + slot * 32, r);
                tmem_wait_st();
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(sf0 + 8 * slot);
                slot += NG;
                while (slot >= R) { slot -= R; sph ^= 1; }
            }
            next -= steps;
            __syncwarp();
            if (lane == 0) mbar_arrive(we0 + 8 * stage);
            if (++stage == WS) { stage = 0; phase ^= 1; }
            if (++c == C) c = 0;
        }
    } else {
        mixed_epilogue<TS, QUANT>(p, tmem_base, warp, lane, u_begin, u_end, accf0, acce0, abort_flag, t_w, reinterpret_cast<float*>(extra));
    }

    __syncthreads();
    if (*abort_flag) {
        // copies may be under way
        const unsigned long long t0 = globaltimer_ns();
        while (globaltimer_ns() - t0 < 2000000ull) __nanosleep(1000);
        __syncthreads();
    }
    if (warp == W_MMA) {
        tc_fence_after();
        tmem_dealloc(tmem_base, MX_TMEM_COLS);
    }
}

// Adds up the partial sums of the tiles that several CTAs share, in CTA order.  A block has 32 token columns of one weight
// tile, a warp four of them, a lane four consecutive weight rows (QUANT: a warp has 32 rows, a lane a column).
template <bool QUANT>
__global__ void __launch_bounds__(QUANT ? 128 : 256) mixed_reduce_kernel(const __grid_constant__ MixedParams p)
{
    const MixedPlan& pl = p.pl;
    const uint32_t C = pl.chunks, TS = (uint32_t)pl.ts, NP = (pl.n_tok + 31u) & ~31u;
    const uint32_t tile = blockIdx.x / TS, t = blockIdx.x % TS, t_begin = tile * C, wt = tile / pl.tok_tiles * TS + t;
    const uint32_t c_first = cta_of(pl, t_begin), nseg = cta_of(pl, t_begin + C - 1) - c_first + 1;
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    if (nseg == 1 || wt >= (uint32_t)p.LW.tiles) return;         // written by the CTA that has it
    asm volatile("griddepcontrol.wait;" ::: "memory");
    if (p.status[0] != 0) return;
    const fgmp_packed_header* hw = reinterpret_cast<const fgmp_packed_header*>(p.wblob);
    if (p.leave_nvfp4 && hw->n_fp8 == 0 && p.ha->n_fp8 == 0) return;
    const float alpha = __fmul_rn(__fmul_rn(p.ha->scale_fp4, hw->scale_fp4), __int_as_float((127 + max(hw->fp8_log2_ratio, -4)) << 23));
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t m0 = (int64_t)(tile % pl.tok_tiles) * pl.n_tok, m_end = min(p.M, m0 + pl.n_tok);
    auto part = [&](uint32_t i) {
        return p.parts + ((size_t)((c_first + i) * 2 + (unit_begin(pl, c_first + i) >= t_begin ? 0u : 1u)) * TS + t) * NP * 128;
    };
    if (QUANT) {
        const uint32_t col = blockIdx.y * 32 + lane;
        const int64_t n = (int64_t)wt * 128 + 32 * warp;
        float s[32];
#pragma unroll
        for (int j = 0; j < 32; ++j) s[j] = 0.f;
#pragma unroll 1
        for (uint32_t i = 0; i < nseg; ++i) {
            const float4* src = reinterpret_cast<const float4*>(part(i) + (size_t)col * 128 + 32 * warp);
#pragma unroll
            for (int j = 0; j < 8; ++j) { const float4 x = __ldcg(src + j); s[4 * j] += x.x; s[4 * j + 1] += x.y; s[4 * j + 2] += x.z; s[4 * j + 3] += x.w; }
        }
        uint32_t r[32];
#pragma unroll
        for (int j = 0; j < 32; ++j) r[j] = __float_as_uint(s[j]);
        if (m0 + col < m_end && n < p.N) quantize_row32(p, m0 + col, n, r, alpha);
    } else {
        const int64_t n = (int64_t)wt * 128 + 4 * lane;
        float4 s[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) s[j] = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 4
        for (uint32_t i = 0; i < nseg; ++i) {
            const float4* src = reinterpret_cast<const float4*>(part(i) + (size_t)(blockIdx.y * 32 + warp * 4) * 128) + lane;
#pragma unroll
            for (int j = 0; j < 4; ++j) { const float4 x = __ldcg(src + j * 32); s[j].x += x.x; s[j].y += x.y; s[j].z += x.z; s[j].w += x.w; }
        }
        const bool wide = n + 4 <= p.N && (p.ldy & 3) == 0;      // (Y is 16-byte aligned)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int64_t m = m0 + blockIdx.y * 32 + warp * 4 + j;
            if (m >= m_end) break;
            const float v[4] = {s[j].x * alpha, s[j].y * alpha, s[j].z * alpha, s[j].w * alpha};
            if (p.y_is_bf16) {
                __nv_bfloat16* y = reinterpret_cast<__nv_bfloat16*>(p.Y) + m * p.ldy + n;
                if (wide) {
                    __nv_bfloat162 a = __floats2bfloat162_rn(v[0], v[1]), b = __floats2bfloat162_rn(v[2], v[3]);
                    *reinterpret_cast<uint2*>(y) = make_uint2(*reinterpret_cast<uint32_t*>(&a), *reinterpret_cast<uint32_t*>(&b));
                } else {
                    for (int e = 0; e < 4; ++e) if (n + e < p.N) y[e] = __float2bfloat16_rn(v[e]);
                }
            } else {
                float* y = reinterpret_cast<float*>(p.Y) + m * p.ldy + n;
                if (wide) *reinterpret_cast<float4*>(y) = make_float4(v[0], v[1], v[2], v[3]);
                else for (int e = 0; e < 4; ++e) if (n + e < p.N) y[e] = v[e];
            }
        }
    }
}

// ------------------------------------------------------------------ host side
constexpr uint32_t MX_FIXED = 1024 /*alignment*/ + 1024 /*barriers, stage table*/;

// Modelled clocks of a unit: dequantization (about 1100 per weight tile), MMAs (16 of N/2 clocks per weight tile), copies
// from L2 (42 bytes per clock and SM).
double unit_cost(int ts, uint32_t n_tok)
{
    const double deq = 1100.0 * ts, mma = 8.0 * n_tok * ts, l2 = (20000.0 * ts + 512.0 * n_tok) / 42.0;
    return deq > mma ? (deq > l2 ? deq : l2) : (mma > l2 ? mma : l2);
}

// How the work is cut: weight tiles per unit, tokens per tile, and whether CTAs take whole tiles or equal spans of units.
// The choice is the least modelled time; measured against it on the B200 the model is within 15 % from 17 to 1000 tokens.
MixedPlan mixed_plan(int64_t M, int64_t N, int64_t K)
{
    const uint32_t wtiles = (uint32_t)((N + 127) / 128), chunks = (uint32_t)((K / 64 + 3) / 4), sms = (uint32_t)fgmp_sm_count();
    MixedPlan best{};
    best.cost = 1e300;
    for (int ts = 1; ts <= 2; ++ts) {
        const uint32_t n_max = ts == 1 ? 256 : 208;      // 512 columns: ts accumulators and at least three steps of 32
        const uint32_t t_min = (uint32_t)((M + n_max - 1) / n_max);
        for (uint32_t T = t_min; T < t_min + 4 && (int64_t)(T - 1) * 16 < M; ++T) {
            MixedPlan pl{};
            pl.ts = ts; pl.chunks = chunks;
            pl.n_tok = (uint32_t)(((M + T - 1) / T + 15) & ~(int64_t)15);
            pl.tok_tiles = (uint32_t)((M + pl.n_tok - 1) / pl.n_tok);
            pl.groups = (wtiles + ts - 1) / ts;
            pl.tiles = pl.groups * pl.tok_tiles;
            const double unit = unit_cost(ts, pl.n_tok), drain = 12.0 * pl.n_tok * ts;
            const uint64_t total = (uint64_t)pl.tiles * chunks;
            for (int split = 0; split < 2; ++split) {
                pl.quantum = split ? 1 : chunks;
                const uint64_t quanta = total / pl.quantum;
                if (split && chunks == 1) continue;
                pl.grid = (uint32_t)(quanta < sms ? quanta : sms);
                pl.span = (uint32_t)(quanta / pl.grid); pl.rest = (uint32_t)(quanta % pl.grid);
                const double most = (double)(pl.span + (pl.rest ? 1 : 0)) * pl.quantum;
                pl.cost = most * unit + (split ? 4000.0 + 2.0 * drain : most / chunks * drain);
                if (pl.cost < best.cost) best = pl;
            }
        }
    }
    best.max_parts = best.quantum == 1 ? best.grid * 2 : 0;
    const uint32_t tmem_slots = (MX_TMEM_COLS - best.ts * best.n_tok) / 32;
    best.slots = tmem_slots < (uint32_t)MAX_SLOTS ? tmem_slots : (uint32_t)MAX_SLOTS;
    // shared memory: two weight stages, the rest token stages; with many of those, a third weight stage
    const uint32_t room = (uint32_t)MX_SMEM_LIMIT - MX_FIXED - (4 * 32 * 33 * 4 + 128), wst = best.ts * WSTAGE, bst = best.n_tok * 128u;
    best.wstages = 2;
    while (best.wstages < (uint32_t)MAX_WSTAGES && (room - (best.wstages + 1) * wst) / bst >= 5 && room > (best.wstages + 1) * wst) ++best.wstages;
    best.bstages = (room - best.wstages * wst) / bst;
    if (best.bstages > (uint32_t)MAX_BSTAGES) best.bstages = MAX_BSTAGES;
    return best;
}

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
std::mutex mx_mu;
EncodeTiledFn mx_encode = nullptr;
bool mx_attr_set[64] = {};

}  // namespace

size_t fgmp_ws_mixed(int64_t M, int64_t N, int64_t K)
{
    const MixedPlan pl = mixed_plan(M, N, K);
    return (size_t)FGMP_WS_CONTROL_BYTES + fgmp_align1k((size_t)M * K * 2) + (size_t)pl.max_parts * pl.ts * ((pl.n_tok + 31u) & ~31u) * 512;
}

// expands the activations and multiplies; leave_nvfp4: unless neither operand has an FP8 block
fgmp_status fgmp_linear_mixed(const void* packed_acts, const void* packed_weights, void* Y, int y_is_bf16, int64_t ldy,
                              int64_t M, int64_t N, int64_t K, void* workspace, const QuantNext& qn, bool leave_nvfp4, cudaStream_t s)
{
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return FGMP_ERR_CUDA;
    {
        std::lock_guard<std::mutex> lk(mx_mu);
        if (!mx_encode) {
            void* fn = nullptr;
            cudaDriverEntryPointQueryResult q;
            if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &fn, cudaEnableDefault, &q) != cudaSuccess ||
                q != cudaDriverEntryPointSuccess) return FGMP_ERR_CUDA;
            mx_encode = reinterpret_cast<EncodeTiledFn>(fn);
        }
        if (!mx_attr_set[dev]) {
            if (cudaFuncSetAttribute(mixed_kernel<1, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)MX_SMEM_LIMIT) != cudaSuccess ||
                cudaFuncSetAttribute(mixed_kernel<1, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)MX_SMEM_LIMIT) != cudaSuccess ||
                cudaFuncSetAttribute(mixed_kernel<2, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)MX_SMEM_LIMIT) != cudaSuccess ||
                cudaFuncSetAttribute(mixed_kernel<2, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)MX_SMEM_LIMIT) != cudaSuccess)
                return FGMP_ERR_CUDA;
            mx_attr_set[dev] = true;
        }
    }
    uint8_t* ws = (uint8_t*)workspace;
    MixedParams p{};
    p.wblob = (const uint8_t*)packed_weights; p.LW = fgmp_layout(N, K, 1, 0);
    p.ha = reinterpret_cast<const fgmp_packed_header*>(packed_acts);
    p.Y = Y; p.ldy = ldy; p.y_is_bf16 = y_is_bf16; p.M = M; p.N = N; p.K = K;
    p.leave_nvfp4 = leave_nvfp4 ? 1 : 0;
    p.pl = mixed_plan(M, N, K);
    p.status = reinterpret_cast<int*>(ws);
    uint8_t* plane = ws + FGMP_WS_CONTROL_BYTES;
    p.parts = reinterpret_cast<float*>(plane + fgmp_align1k((size_t)M * K * 2));
    p.q = qn;
    // the activations' fp16 plane [M, K]: boxes of n_tok rows x 64 elements, swizzled; rows beyond M are zero
    CUtensorMap tmB;
    cuuint64_t dims[2] = {(cuuint64_t)K, (cuuint64_t)M};
    cuuint64_t strides[1] = {(cuuint64_t)K * 2};
    cuuint32_t box[2] = {64, p.pl.n_tok};
    cuuint32_t estr[2] = {1, 1};
    if (mx_encode(&tmB, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2, plane, dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                  CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS) return FGMP_ERR_CUDA;

    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.stream = s; cfg.attrs = attr; cfg.numAttrs = 1;
    const int64_t nb = M * (K / 16), sms = fgmp_sm_count();
    cfg.gridDim = dim3((unsigned)((nb + 255) / 256 < sms * 8 ? (nb + 255) / 256 : sms * 8)); cfg.blockDim = dim3(256);
    FGMP_LAUNCH(FGMP_K_EXPAND_A, s, cudaLaunchKernelEx(&cfg, expand_f16_kernel, (const uint8_t*)packed_acts, (const uint8_t*)packed_weights, M, K, plane, p.status, p.leave_nvfp4));
    const bool quant = qn.codes4 != nullptr;
    cfg.gridDim = dim3(p.pl.grid); cfg.blockDim = dim3((unsigned)mx_threads(quant));
    cfg.dynamicSmemBytes = (size_t)p.pl.bstages * p.pl.n_tok * 128 + (size_t)p.pl.wstages * p.pl.ts * WSTAGE + MX_FIXED + 4 * 32 * 33 * 4 + 128;
    if (p.pl.ts == 1) {
        if (quant) { FGMP_LAUNCH(FGMP_K_GEMM_MIXED, s, cudaLaunchKernelEx(&cfg, mixed_kernel<1, true>, tmB, p)); }
        else       { FGMP_LAUNCH(FGMP_K_GEMM_MIXED, s, cudaLaunchKernelEx(&cfg, mixed_kernel<1, false>, tmB, p)); }
    } else {
        if (quant) { FGMP_LAUNCH(FGMP_K_GEMM_MIXED, s, cudaLaunchKernelEx(&cfg, mixed_kernel<2, true>, tmB, p)); }
        else       { FGMP_LAUNCH(FGMP_K_GEMM_MIXED, s, cudaLaunchKernelEx(&cfg, mixed_kernel<2, false>, tmB, p)); }
    }
    if (p.pl.quantum == 1) {
        cfg.gridDim = dim3(p.pl.tiles * (unsigned)p.pl.ts, (p.pl.n_tok + 31) / 32); cfg.dynamicSmemBytes = 0;
        cfg.blockDim = dim3(quant ? 128 : 256);
        if (quant) { FGMP_LAUNCH(FGMP_K_GEMM_REDUCE, s, cudaLaunchKernelEx(&cfg, mixed_reduce_kernel<true>, p)); }
        else       { FGMP_LAUNCH(FGMP_K_GEMM_REDUCE, s, cudaLaunchKernelEx(&cfg, mixed_reduce_kernel<false>, p)); }
    }
    return fgmp_launch_status();
}

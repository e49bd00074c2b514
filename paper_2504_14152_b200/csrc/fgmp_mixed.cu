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
//   - a 128 x 256 unit of weights takes about 1000 clocks of the SIMT pipes (1024 conversions at one per clock), its MMAs 16 of
//     N/2 clocks for N tokens;
//   - the operand from tensor memory leaves shared memory to the token tiles (from shared memory the 64 KiB of a
//     dequantized unit would be written and read there, 1024 clocks by themselves);
//   - a unit takes 1.08 us + 4.2 ns per token, more than its MMAs (4.3 ns per token) or its dequantization: with either of them or
//     the token copies left out it is 7 to 20 % faster, with all of them left out 27 %.  What remains is the way of a slot through
//     three groups of warps (copy, dequantize, multiply, release), some 2000 clocks, and at full rate the token tiles would
//     take 64 bytes per clock and SM from L2.  Four groups, CTA pairs that share a token tile, more weight stages, spinning
//     instead of suspended waits and a loop of one elected thread in the issuer were measured and are no faster.
//   - so a unit is worth as many tokens as fit: up to 416 (two MMAs side by side on one dequantized operand) where a CTA's share lies within
//     a tile (400 x 11008 x 4096: 48 us, 54 with two tiles of 208; 1200 x 4096 x 4096: 52 and 57).
//
// Work is (weight tile, token tile, 256-element K chunk) units in that order, split over the CTAs either in
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
#include "fgmp_deq.cuh"

namespace {

constexpr int W_PROD = 0, W_MMA = 1, W_TOK = 2, W_EPI = 3, W_DEQ = 7;
constexpr int MX_GROUPS = 3;                    // dequantization groups (four are no faster, two 10 % slower)
constexpr int MX_THREADS = 32 * (W_DEQ + 4 * MX_GROUPS);
constexpr uint32_t STG_MASK = REC_BYTES, STG_HALF = STG_MASK + 256;      // a weight stage: record, mask, second halves of the FP8 blocks
constexpr uint32_t HALF_CAP = 5248;             // 656 FP8 blocks (32 %); with more the halves are read from global memory
constexpr uint32_t WSTAGE = STG_HALF + HALF_CAP;                         // 24064
constexpr int MAX_WSTAGES = 4, MAX_BSTAGES = 12, MAX_SLOTS = 8;
constexpr uint32_t MX_TMEM_COLS = 512;
constexpr uint32_t MX_MAX_TOK = 416;            // tokens of a tile: columns of its accumulator, beside three slots of 32
constexpr size_t MX_SMEM_LIMIT = 232448;
constexpr uint32_t SW128_LO = 1u << 16, SW128_HI = (1024u >> 4) | (1u << 14) | (2u << 29);
constexpr uint32_t IDESC_F16 = 1u << 4;         // f32 += f16 x f16, K-major; M and N added

struct MixedPlan {
    uint32_t n_tok, tok_tiles;           // tokens per tile (multiple of 16), token tiles
    uint32_t n_half;                     // tokens of one MMA: n_tok, or the first half (rounded up to 16) of a tile of more than 256
    uint32_t chunks, tiles;              // tiles = wtiles * tok_tiles
    uint32_t grid, span, rest, quantum;  // a CTA's span in quanta of `quantum` units (1, or chunks: whole tiles)
    uint32_t split;                      // 1: some tile is shared by several CTAs, whose parts are added up behind this kernel
    uint32_t wstages, bstages, slots, naccs;
    double us;                           // modelled time
};

struct MixedParams {
    const uint8_t* wblob; PackedLayout LW;
    const fgmp_packed_header* ha;
    void* Y; int64_t ldy; int y_is_bf16;
    int64_t M, N, K;
    int leave_nvfp4;                     // operands without any FP8 block are left to the all-NVFP4 GEMM, launched before or behind this kernel
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
__device__ __forceinline__ uint32_t unit_begin(const MixedPlan& pl, uint32_t cta) { return (cta * pl.span + min(cta, pl.rest)) * pl.quantum; }
__device__ __forceinline__ uint32_t cta_of(const MixedPlan& pl, uint32_t u)
{
    const uint32_t i = u / pl.quantum, longer = pl.rest * (pl.span + 1);
    return i < longer ? i / (pl.span + 1) : pl.rest + (i - longer) / pl.span;
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
template <bool QUANT>
__device__ __forceinline__ void mixed_epilogue(const MixedParams& p, uint32_t tmem_base, int warp, int lane, uint32_t u_begin, uint32_t u_end,
                                               uint32_t accf0, uint32_t acce0, volatile int* abort_flag, int t_w, float* extra)
{
    const MixedPlan& pl = p.pl;
    const uint32_t q = (uint32_t)warp & 3u, C = pl.chunks, NT = pl.n_tok, NP = (NT + 31u) & ~31u, row = 32u * q + lane;   // (NP: columns of a partial tile)
    const float alpha = __fmul_rn(__fmul_rn(p.ha->scale_fp4, __ldg(&reinterpret_cast<const fgmp_packed_header*>(p.wblob)->scale_fp4)),
                                  __int_as_float((127 + t_w) << 23));
    uint32_t* turn = reinterpret_cast<uint32_t*>(extra) + q * 32 * 33;
    uint32_t acc = 0, acc_phase = 0;
    for (uint32_t u = u_begin; u < u_end;) {
        const uint32_t tile = u / C, t_begin = tile * C, t_end = t_begin + C, seg_end = min(t_end, u_end);
        const bool whole = u == t_begin && seg_end == t_end;
        const uint32_t wt = tile / pl.tok_tiles, which = u == u_begin ? 0u : 1u;       // a span's first segment, or its last
        const int64_t m0 = (int64_t)(tile % pl.tok_tiles) * NT, n = (int64_t)wt * 128 + row;
        u = seg_end;
        if (!mbar_wait_warp(accf0 + 8 * acc, acc_phase, abort_flag, p.status, 8)) break;
        tc_fence_after();
        const uint32_t d = tmem_base + ((q * 32u) << 16) + acc * NT;
        float* mine = p.parts + ((size_t)(blockIdx.x * 2 + which)) * NP * 128 + row;
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
        if (lane == 0) mbar_arrive(acce0 + 8 * acc);
        if (++acc == pl.naccs) { acc = 0; acc_phase ^= 1u; }
    }
}

// QUANT: the next layer's activation quantizer in the epilogue instead of Y.
template <bool QUANT>
__global__ void __launch_bounds__(MX_THREADS, 1)
mixed_kernel(const __grid_constant__ CUtensorMap tmB, const __grid_constant__ MixedParams p)
{
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
    const MixedPlan& pl = p.pl;
    const uint32_t BS = pl.bstages, WS = pl.wstages, R = pl.slots, NT = pl.n_tok, C = pl.chunks;
    // (no more groups than slots: a group that was further ahead could take an older phase of a slot's barrier for the one it waits for)
    const uint32_t NG = min((uint32_t)MX_GROUPS, R);
    const uint32_t NH = pl.n_half;
    const uint32_t b_bytes = (NT > NH ? 2u : 1u) * NH * 128u;   // token stage: rows of 64 elements, swizzled (a multiple of 2 KiB)
    uint8_t* wst0 = smem + BS * b_bytes;
    uint8_t* extra = wst0 + WS * WSTAGE;                 // QUANT: 4 x 32 x 33 floats
    uint64_t* bars = reinterpret_cast<uint64_t*>(extra + (QUANT ? 4 * 32 * 33 * 4 + 128 : 0));
    uint32_t* wmeta = reinterpret_cast<uint32_t*>(bars + 2 * MAX_WSTAGES + 2 * MAX_BSTAGES + MAX_SLOTS + 4);   // per stage: list start, bytes of it there
    uint32_t* tmem_slot = wmeta + MAX_WSTAGES * 2;
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

    const int warp = warp_index(), lane = threadIdx.x & 31;
    // The MMA issuer is a single thread whose every wait (75 clocks) and commit (40) comes on top of 40 clocks per MMA, so it has
    // one of each per step of 64 elements: step i is ready (barrier i % R) when the dequantized weights are in tensor
    // memory and the warps that put them there have seen the token tile of the step; when it is done (barrier i % L, L the
    // longer of the two rings), both its slot and its token stage are free.
    // barriers: weight stage full / empty, token stage full; step ready, step done; accumulators full / empty
    const uint32_t wf0 = smem_u32(bars), we0 = wf0 + 8 * MAX_WSTAGES, bf0 = we0 + 8 * MAX_WSTAGES, dn0 = bf0 + 8 * MAX_BSTAGES;
    const uint32_t sf0 = dn0 + 8 * MAX_BSTAGES, accf0 = sf0 + 8 * MAX_SLOTS, acce0 = accf0 + 16;
    const uint32_t L = max(R, BS);
    const uint32_t slot_col = pl.naccs * NT;             // tensor memory: accumulators of NT columns, then slots of 32

    const uint32_t u_begin = unit_begin(pl, blockIdx.x), u_end = unit_begin(pl, blockIdx.x + 1);
    const uint32_t last_steps = (uint32_t)(p.K / 64) - 4u * (C - 1u);

    if (threadIdx.x == 0) {
        for (uint32_t s = 0; s < WS; ++s) { mbar_init(wf0 + 8 * s, 1); mbar_init(we0 + 8 * s, 4 * NG); }
        for (uint32_t s = 0; s < BS; ++s) mbar_init(bf0 + 8 * s, 1);
        for (uint32_t s = 0; s < L; ++s) mbar_init(dn0 + 8 * s, 1);
        for (uint32_t s = 0; s < R; ++s) mbar_init(sf0 + 8 * s, 4);
        for (uint32_t t = 0; t < pl.naccs; ++t) { mbar_init(accf0 + 8 * t, 1); mbar_init(acce0 + 8 * t, 4); }
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == W_MMA) tmem_alloc(smem_u32(tmem_slot), MX_TMEM_COLS);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = TMEM_ALL;
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
            const uint32_t c = u % C, tile = u / C / pl.tok_tiles, rec = tile * C + c;
            if (issued == WS && !waited) {
                // the status word may be looked at once the preceding kernel is done
                asm volatile("griddepcontrol.wait;" ::: "memory");
                waited = true;
            }
            if (lane == 0) {
                const uint32_t st0 = __ldg(uptr + rec), st1 = __ldg(uptr + rec + 1);
                ok = mbar_wait(we0 + 8 * stage, phase, abort_flag, p.status, 1) ? 1 : 0;
                if (ok) {
                    const uint32_t steps = st1 - st0, h = 2u * steps / 3u, staged = min(h * 16u, HALF_CAP);     // the list's words, then h steps of halves
                    const uint32_t dst = smem_u32(wst0 + stage * WSTAGE), fb = wf0 + 8 * stage;
                    wmeta[stage * 2] = st0 + (steps - h); wmeta[stage * 2 + 1] = staged;
                    mbar_expect_tx(fb, REC_BYTES + 256u + staged);
                    bulk_load(dst, p.wblob + p.LW.off_rec + (size_t)rec * REC_BYTES, REC_BYTES, fb);
                    bulk_load(dst + STG_MASK, p.wblob + p.LW.off_mask + (size_t)rec * 256, 256u, fb);
                    if (staged) bulk_load(dst + STG_HALF, p.wblob + p.LW.off_ovf + (size_t)(st0 + (steps - h)) * 16, staged, fb);
                }
            }
            ok = __shfl_sync(0xffffffffu, ok, 0);
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
            uint32_t stage = 0, ds = 0, dph = 0, i = 0;  // ds: barrier of step i - BS
            bool ok = true;
            for (uint32_t u = u_begin; u < u_end && ok; ++u) {
                const uint32_t c = u % C, m0 = (u / C) % pl.tok_tiles * NT, steps = c == C - 1 ? last_steps : 4u;
                for (uint32_t s = 0; s < steps; ++s, ++i) {
                    if (i >= BS) {
                        if (!(ok = mbar_wait(dn0 + 8 * ds, dph, abort_flag, p.status, 2))) break;
                        if (++ds == L) { ds = 0; dph ^= 1; }
                    }
                    mbar_expect_tx(bf0 + 8 * stage, b_bytes);
                    tma_load_2d(smem_u32(smem + stage * b_bytes), &tmB, (int32_t)(c * 256 + s * 64), (int32_t)m0, bf0 + 8 * stage);
                    if (NT > NH) tma_load_2d(smem_u32(smem + stage * b_bytes) + NH * 128u, &tmB, (int32_t)(c * 256 + s * 64), (int32_t)(m0 + NH), bf0 + 8 * stage);
                    if (++stage == BS) stage = 0;
                }
            }
        }
        __syncwarp();
    } else if (warp == W_MMA) {
        // ------------------------------------------------------------ MMA issuer (one elected lane)
        {
            const uint32_t idesc = IDESC_F16 | ((NH >> 3) << 17) | ((128u >> 4) << 24), idesc2 = IDESC_F16 | (((NT - NH) >> 3) << 17) | ((128u >> 4) << 24), b_first = (smem_u32(smem) >> 4) | SW128_LO, b_step = b_bytes >> 4;
            uint32_t bst = 0, slot = 0, sph = 0, ds = 0, c = u_begin % C, acc = 0, acc_phase = 1, accum = 0, b_lo = b_first;
            bool ok = true, ready = false;
            for (uint32_t u = u_begin; u < u_end && ok; ++u) {
                const uint32_t steps = c == C - 1 ? last_steps : 4u, d = tmem_base + acc * NT;
                const bool last_unit = c == C - 1 || u + 1 == u_end;
                if (accum == 0 && !mbar_wait_uniform(acce0 + 8 * acc, acc_phase, abort_flag, p.status, 4)) break;
                for (uint32_t s = 0; s < steps; ++s) {
                    if (!ready && !(ok = mbar_wait_uniform(sf0 + 8 * slot, sph, abort_flag, p.status, 5))) break;
                    tc_fence_after();
                    const uint32_t a = tmem_base + slot_col + slot * 32;
                    if (++slot == R) { slot = 0; sph ^= 1; }
                    const bool peek = mbar_test_wait(sf0 + 8 * slot, sph);      // the next step's; the answer comes while this one's MMAs are issued
                    if (elect_one()) {
#pragma unroll
                        for (uint32_t k = 0; k < 4; ++k) umma_f16_ta(d, a + 8 * k, mx_desc(b_lo + 2 * k), idesc, k ? 1u : accum);
                        if (NT > NH) {
#pragma unroll
                            for (uint32_t k = 0; k < 4; ++k) umma_f16_ta(d + NH, a + 8 * k, mx_desc(b_lo + NH * 8u + 2 * k), idesc2, k ? 1u : accum);
                        }
                        umma_commit(dn0 + 8 * ds);
                    }
                    accum = 1;
                    b_lo += b_step;
                    if (++bst == BS) { bst = 0; b_lo = b_first; }
                    if (++ds == L) ds = 0;
                    ready = __all_sync(0xffffffffu, peek);
                }
                if (last_unit) {
                    if (elect_one()) umma_commit(accf0 + 8 * acc);
                    __syncwarp();
                    accum = 0;
                    if (++acc == pl.naccs) { acc = 0; acc_phase ^= 1; }
                }
                if (++c == C) c = 0;
            }
        }
        __syncwarp();
    } else if (warp >= W_DEQ + 4 * (int)NG) {
    } else if (warp >= W_DEQ) {
        // ------------------------------------------------------------ dequantization: thread = row of the weight tile
        // The groups take the steps of 64 elements in turn.
        const uint32_t group = (uint32_t)(warp - W_DEQ) >> 2, row = 32u * (warp & 3) + lane, r7 = row & 7u;
        const uint32_t quadrant = tmem_base + ((uint32_t)((warp & 3) * 32) << 16) + slot_col;
        const __half2 inv2 = __float2half2_rn(__int_as_float((127 - t_w) << 23)), f82 = __float2half2_rn(__int_as_float((127 + ratio_w - t_w) << 23));
        const uint32_t inv = *reinterpret_cast<const uint32_t*>(&inv2), f8 = *reinterpret_cast<const uint32_t*>(&f82);
        const bool scaled8 = ratio_w != t_w;             // (for every thread alike)
        uint32_t stage = 0, phase = 0, c = u_begin % C, slot = group, next = group;    // next: steps until the group's turn
        uint32_t bst = group, bph = 0, ds = 0, dph = 0, i = group;        // i: the step; ds: barrier of step i - R
        while (bst >= BS) { bst -= BS; bph ^= 1; }
        bool ok = true;
        for (uint32_t u = u_begin; u < u_end && ok; ++u) {
            const uint32_t steps = c == C - 1 ? last_steps : 4u;
            if (!(ok = mbar_wait_warp(wf0 + 8 * stage, phase, abort_flag, p.status, 6))) break;
            const uint8_t* sp = wst0 + stage * WSTAGE;
            uint32_t mt = 0, at = 0;
            bool all = true;
            if (has_fp8) {
                // the row's FP8 blocks lie one after the other in the list
                const uint16_t* before = reinterpret_cast<const uint16_t*>(sp + REC_KBSTART);
                mt = reinterpret_cast<const uint16_t*>(sp + STG_MASK)[row];
                at = __popc(mt);
#pragma unroll
                for (int o = 1; o < 8; o <<= 1) { const uint32_t y = __shfl_up_sync(0xffffffffu, at, o, 8); if ((lane & 7) >= o) at += y; }
                at = 8u * (before[row >> 3] + at - __popc(mt));
                all = 8u * before[16] <= wmeta[stage * 2 + 1];
            }
#pragma unroll 1
            for (; next < steps; next += NG) {
                const uint32_t s = next;
                uint32_t r[32];
                const uint32_t sb = smem_u32(sp), codes = sb + row * 128u, sfw = sb + REC_SF + (row & 31u) * 16u + (row >> 5) * 4u;
                const uint32_t m16 = mt >> (4 * s);
                uint32_t hg = at + 8u * __popc(mt & ((1u << (4 * s)) - 1u)), hs = sb + STG_HALF + hg;
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
                    const uint8_t* half_g = p.wblob + p.LW.off_ovf + (size_t)wmeta[stage * 2] * 16;
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
                __syncwarp();
                if (i >= R) {
                    if (i < R + NG) ds = (i - R) % L;              // the group's first wait
                    if (!(ok = mbar_wait_warp(dn0 + 8 * ds, dph, abort_flag, p.status, 7))) break;
                    tc_fence_after();
                    ds += NG;
                    if (ds >= L) { ds -= L; dph ^= 1; }
                }
                tmem_st32(quadrant + slot * 32, r);
                tmem_wait_st();
                tc_fence_before();
                __syncwarp();
                if (lane == 0 && mbar_wait(bf0 + 8 * bst, bph, abort_flag, p.status, 3)) mbar_arrive(sf0 + 8 * slot);
                __syncwarp();
                i += NG;
                slot += NG;
                if (slot >= R) slot -= R;
                bst += NG;
                while (bst >= BS) { bst -= BS; bph ^= 1; }
            }
            next -= steps;
            __syncwarp();
            if (lane == 0) mbar_arrive(we0 + 8 * stage);
            if (++stage == WS) { stage = 0; phase ^= 1; }
            if (++c == C) c = 0;
        }
    } else {
        mixed_epilogue<QUANT>(p, tmem_base, warp, lane, u_begin, u_end, accf0, acce0, abort_flag, t_w, reinterpret_cast<float*>(extra));
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
    const uint32_t C = pl.chunks, NP = (pl.n_tok + 31u) & ~31u;
    const uint32_t tile = blockIdx.x, t_begin = tile * C, wt = tile / pl.tok_tiles;
    const uint32_t c_first = cta_of(pl, t_begin), nseg = cta_of(pl, t_begin + C - 1) - c_first + 1;
    // Every block waits, those without anything to add up too: this grid lets its dependents start early, and what they wait for
    // is its end, which must not come before the end of the kernel that wrote the other tiles and reads the workspace.
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
    if (nseg == 1) return;                               // written by the CTA that has it
    if (p.status[0] != 0) return;
    const fgmp_packed_header* hw = reinterpret_cast<const fgmp_packed_header*>(p.wblob);
    if (p.leave_nvfp4 && hw->n_fp8 == 0 && p.ha->n_fp8 == 0) return;
    const float alpha = __fmul_rn(__fmul_rn(p.ha->scale_fp4, hw->scale_fp4), __int_as_float((127 + max(hw->fp8_log2_ratio, -4)) << 23));
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t m0 = (int64_t)(tile % pl.tok_tiles) * pl.n_tok, m_end = min(p.M, m0 + pl.n_tok);
    auto part = [&](uint32_t i) {
        return p.parts + ((size_t)((c_first + i) * 2 + (unit_begin(pl, c_first + i) >= t_begin ? 0u : 1u))) * NP * 128;
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
constexpr uint32_t MX_FIXED = 1024 /*alignment*/ + 1024 /*barriers, stage table*/, MX_TURN = 4 * 32 * 33 * 4 + 128;

// Modelled time of a unit in us (measured: 1.55 at 112 tokens, 1.75 at 160, 1.95 at 208, 2.15 at 256)
double unit_us(uint32_t n_tok) { return 1.08 + 0.0042 * n_tok; }

// bytes for the parts of shared tiles: at most two tiles of a span are shared
size_t parts_bytes(const MixedPlan& pl) { return pl.split ? (size_t)pl.grid * 2 * ((pl.n_tok + 31u) & ~31u) * 512 : 0; }

// How the work is cut: tokens per tile, and whether CTAs take whole tiles or equal spans of units: the least modelled time among the
// ways whose parts of tiles fit in `room_for_parts` bytes.  (A fit without the expansion's launch: whole calls take 7 to 9 us more at 48 tokens,
// and are within 10 % of it from 203 tokens on at 11008 x 4096 and 13824 x 5120.)
MixedPlan mixed_plan(int64_t M, int64_t N, int64_t K, size_t room_for_parts)
{
    const uint32_t wtiles = (uint32_t)((N + 127) / 128), chunks = (uint32_t)((K / 64 + 3) / 4), sms = (uint32_t)fgmp_sm_count();
    const uint32_t t_min = (uint32_t)((M + MX_MAX_TOK - 1) / MX_MAX_TOK), t_max = 2 * (uint32_t)((M + 255) / 256) + 2;
    MixedPlan best{};
    best.us = 1e300;
    for (uint32_t T = t_min; T < t_max && (int64_t)(T - 1) * 16 < M; ++T) {
        MixedPlan pl{};
        pl.chunks = chunks;
        pl.n_tok = (uint32_t)((M + T - 1) / T + 15) / 16 * 16;
        pl.n_half = pl.n_tok <= 256 ? pl.n_tok : (pl.n_tok + 31) / 32 * 16;
        pl.tok_tiles = (uint32_t)((M + pl.n_tok - 1) / pl.n_tok);
        pl.tiles = wtiles * pl.tok_tiles;
        pl.naccs = 2 * pl.n_tok + 96 <= MX_TMEM_COLS ? 2 : 1;
        // reading an accumulator out hides behind the next tile's products if there are two
        const double unit = unit_us(pl.n_tok), drain = 0.012 * pl.n_tok;
        const uint64_t total = (uint64_t)pl.tiles * chunks;
        for (int split = 0; split < (chunks > 1 ? 2 : 1); ++split) {
            pl.quantum = split ? 1 : chunks;
            const uint64_t quanta = total / pl.quantum;
            pl.grid = (uint32_t)(quanta < sms ? quanta : sms);
            pl.span = (uint32_t)(quanta / pl.grid); pl.rest = (uint32_t)(quanta % pl.grid);
            // equal spans that are whole tiles after all are the other way of cutting, which needs no second kernel
            pl.split = split;
            if (split && pl.rest == 0 && pl.span % chunks == 0) continue;
            if (parts_bytes(pl) > room_for_parts) continue;
            const double units = (double)(pl.span + (pl.rest ? 1 : 0)) * pl.quantum, tiles = units / chunks;
            // (beyond 256 tokens only spans within one tile pay: where a CTA goes on to another one its three slots and three
            // token stages run empty as well)
            const double drains = pl.naccs == 2 || tiles < 1.0 ? 1.0 : pl.n_tok <= 256 ? tiles : 2.0 * (tiles + 1.0);
            pl.us = units * unit + drains * drain + (split ? 0.0 : 3.0 * tiles);
            // the second kernel, and what it moves: a partial tile per span or two, written and read
            if (split) pl.us += 2.0 + 2.6 * pl.grid * pl.n_tok * 512.0 / 8e6;
            if (pl.us < best.us) best = pl;
        }
    }
    const uint32_t tmem_slots = (MX_TMEM_COLS - best.naccs * best.n_tok) / 32;
    best.slots = tmem_slots < (uint32_t)MAX_SLOTS ? tmem_slots : (uint32_t)MAX_SLOTS;
    // shared memory: two to four weight stages (a chunk each), the rest token stages
    const uint32_t room = (uint32_t)MX_SMEM_LIMIT - MX_FIXED - MX_TURN, bst = (best.n_tok > best.n_half ? 2u : 1u) * best.n_half * 128u;
    best.wstages = 2;
    while (best.wstages < (uint32_t)MAX_WSTAGES && room - (best.wstages + 1) * WSTAGE >= 10 * bst) ++best.wstages;
    best.bstages = (room - best.wstages * WSTAGE) / bst;
    if (best.bstages > (uint32_t)MAX_BSTAGES) best.bstages = MAX_BSTAGES;
    // No more slots than token stages: a group that fills the slot of step i then knows step i - bstages done, so that the parity of its token
    // stage's barrier can only mean step i (with more slots it could be taken in by a stage whose step before was still on its way).
    if (best.slots > best.bstages) best.slots = best.bstages;
    return best;
}

std::mutex mx_mu;
bool mx_attr_set[64] = {};

}  // namespace

// room for parts in a workspace of ws_bytes, behind the activations' plane
static size_t room_in(size_t ws_bytes, int64_t M, int64_t K)
{
    const size_t before = (size_t)FGMP_WS_CONTROL_BYTES + fgmp_align1k((size_t)M * K * 2);
    return ws_bytes > before ? ws_bytes - before : 0;
}

double fgmp_mixed_us(int64_t M, int64_t N, int64_t K, size_t ws_bytes) { return mixed_plan(M, N, K, room_in(ws_bytes, M, K)).us; }

size_t fgmp_ws_mixed(int64_t M, int64_t N, int64_t K)
{
    return (size_t)FGMP_WS_CONTROL_BYTES + fgmp_align1k((size_t)M * K * 2) + parts_bytes(mixed_plan(M, N, K, SIZE_MAX));
}

// expands the activations and multiplies; leave_nvfp4: unless neither operand has an FP8 block
fgmp_status fgmp_linear_mixed(const void* packed_acts, const void* packed_weights, void* Y, int y_is_bf16, int64_t ldy,
                              int64_t M, int64_t N, int64_t K, void* workspace, size_t ws_bytes, const QuantNext& qn, bool leave_nvfp4, bool first, cudaStream_t s)
{
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return FGMP_ERR_CUDA;
    {
        std::lock_guard<std::mutex> lk(mx_mu);
        if (!mx_attr_set[dev]) {
            if (cudaFuncSetAttribute(mixed_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)MX_SMEM_LIMIT) != cudaSuccess ||
                cudaFuncSetAttribute(mixed_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)MX_SMEM_LIMIT) != cudaSuccess)
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
    p.pl = mixed_plan(M, N, K, room_in(ws_bytes, M, K));
    p.status = reinterpret_cast<int*>(ws);
    uint8_t* plane = ws + FGMP_WS_CONTROL_BYTES;
    p.parts = reinterpret_cast<float*>(plane + fgmp_align1k((size_t)M * K * 2));
    p.q = qn;
    // the activations' fp16 plane [M, K]: boxes of n_half rows x 64 elements, swizzled; rows beyond M are zero
    CUtensorMap tmB;
    if (!fgmp_map_2d(&tmB, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, plane, M, K, K * 2, p.pl.n_half, 64)) return FGMP_ERR_CUDA;

    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.stream = s; cfg.attrs = attr; cfg.numAttrs = 1;
    const fgmp_status st = fgmp_expand(packed_acts, packed_weights, M, N, K, plane, nullptr, p.status, 0, 0, leave_nvfp4, first, s);
    if (st != FGMP_OK) return st;
    const bool quant = qn.codes4 != nullptr;
    cfg.gridDim = dim3(p.pl.grid); cfg.blockDim = dim3(MX_THREADS);
    cfg.dynamicSmemBytes = (size_t)p.pl.bstages * (p.pl.n_tok > p.pl.n_half ? 2 : 1) * p.pl.n_half * 128 + (size_t)p.pl.wstages * WSTAGE + MX_FIXED + (quant ? MX_TURN : 0);
    if (quant) { FGMP_LAUNCH(FGMP_K_GEMM_MIXED, s, cudaLaunchKernelEx(&cfg, mixed_kernel<true>, tmB, p)); }
    else       { FGMP_LAUNCH(FGMP_K_GEMM_MIXED, s, cudaLaunchKernelEx(&cfg, mixed_kernel<false>, tmB, p)); }
    if (p.pl.split) {
        cfg.gridDim = dim3(p.pl.tiles, (p.pl.n_tok + 31) / 32); cfg.dynamicSmemBytes = 0;
        cfg.blockDim = dim3(quant ? 128 : 256);
        if (quant) { FGMP_LAUNCH(FGMP_K_GEMM_REDUCE, s, cudaLaunchKernelEx(&cfg, mixed_reduce_kernel<true>, p)); }
        else       { FGMP_LAUNCH(FGMP_K_GEMM_REDUCE, s, cudaLaunchKernelEx(&cfg, mixed_reduce_kernel<false>, p)); }
    }
    return fgmp_launch_status();
}

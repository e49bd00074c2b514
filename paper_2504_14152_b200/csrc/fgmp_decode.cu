// fgmp_linear for decode-sized batches (M <= 16 tokens): a weight-streaming kernel that reads the packed weights
// exactly once (Section 4.1 of the paper: the four block-pair products, FP32 accumulation), optionally with the
// activation quantizer of Section 4.2 in front of it (fgmp_linear_fused).
//
// At this size the layer is bound by the weight stream (a 22 KiB unit of 128 rows x 256 elements every 885 clocks per
// SM), so the weights must not be converted in the SIMT pipes.  All products run on tcgen05, and what does not fit one
// operand format is split on the ACTIVATION side, which is small and is prepared once per call.  A tcgen05.mma with
// M = 128 takes N/2 clocks, but at least 40 when its weights come from shared memory (4 KiB at 128 bytes a clock), so that
// up to 64 extra columns cost nothing there.
//   (1) NVFP4 weight blocks x all activations: kind::mxf4nvf4 on the packed codes, E4M3 block scales in tensor memory.
//       Token m is row m of the activation operand with its NVFP4 blocks.  An FP8 activation block is written as
//       digits: its E4M3 values are multiples of 2^-9 below 2^9, i.e. 18-bit integers, and six base-8 digits, each of
//       them an E2M1 value, with block scales 2^(3p - 8), p = 0..5, represent them exactly.  Digit p of token m is row
//       (p + 1) M + m.  A block that must not take part has scale 0: FP8 weight blocks in the record, the other
//       format's blocks in the rows of either kind.
//   (2) FP8 weight blocks x all activations: kind::f8f6f4 on a dense E4M3 tile of the unit that holds its FP8 blocks
//       and zeros elsewhere, in tensor memory (a thread per row puts it there: from shared memory the tile would cost eight
//       times 40 clocks, from tensor memory N/2 = 8 to 16 each).  Every activation over its tensor scale has at most 6
//       significant bits (E2M1 x E4M3 scale; E4M3 x 2^ratio has 4), so it is the exact sum of two E5M2 values: rows m and
//       M + m.
//   The epilogue adds the columns of a token: row + 2^ratio_a * digits + 2^ratio_w * (high + low).
// 12 instructions and about 300 tensor clocks per unit for any mix of formats; the SIMT work that is left is moving the
// unit's FP8 blocks and its block scales into tensor memory.
//
// Work is split stream-K style over (128-row tile, 256-element K chunk) units so that all SMs stream the same number of
// bytes.  Tiles shared by several CTAs are reduced in a fixed order by the CTA that arrives last: results are
// reproducible bit for bit.  (For the order of a CTA's units see UnitOrder.)
//
// Where the activation operand (a "step record" per chunk) comes from:
//   DEC_FUSED_LP, DEC_FUSED_HP  fused calls (by block score): the CTAs share out the quantizer's work, write the records to
//                the workspace and stream them from there; the first weight copies are in flight meanwhile.
//   DEC_OWN1_LP ... DEC_OWN4_HP  fused calls of one to four tokens whose packed form nobody asks for: warps of each CTA quantize what its units
//                need, unit by unit, straight into the stages.  That is more work in all, and nothing to hand over: 2.7 us lie between the end of the
//                kernel before and the last shared record, 0.7 more until its copy is in.  In a graph of such calls, 10 % FP8 blocks, shared and own:
//                11008 x 4096 one token 12.6 and 9.9 us, two 12.6 and 10.3, three 12.6 and 10.8; 28672 x 8192 one 31.8 and 28.5, two 31.7 and 30.6.  (With 64 threads a token
//                for every unit in turn instead of two units at a time, two tokens took 14.5 and 48.6.)  Where a CTA has very many units the warps that
//                quantize for each of them cost more than the hand-over: see the launch.
//   DEC_UNPACK   fgmp_linear: made unit by unit in shared memory from the packed activations' records.
//
// Warp roles: warp 0 = weights producer, warp 1 = MMA issuer and owner of the tensor memory, from warp 2 on two or three sets of four warps that take
// the units in turn and put a unit's block scales and FP8 blocks into tensor memory, into a dense tile of their own (the first two sets are the
// quantizer before that; or each makes the step record of its unit), then four warps of epilogue (one lane quadrant each), then the step-record
// producer (DEC_OWN: four warps per token, the quantizer).
//
// The roles run different code at the same time, a warp or two per scheduler, so a unit costs what its instructions cost to
// fetch and issue: what a loop needs once per unit is not unrolled or inlined twice, and a unit passes through few hands
// (producer -> set -> MMA -> producer).  Measured at 70B FC1, one token, time per unit and SM (HBM alone: 0.46 us): SIMT
// corrections for the FP8 blocks 0.66 us; their products on the tensor core with 109 KiB of code, the dense tile in shared
// memory and the scales loaded by warps of their own 0.62 to 0.72 us; this form 0.52 us.
#include "fgmp_common.cuh"
#include "fgmp_actq.cuh"
#include "fgmp_host.h"
#include "fgmp_ptx.cuh"
#include <cuda_fp16.h>
#include <mutex>

namespace {

constexpr int W_PROD = 0, W_MMA = 1, W_SET = 2;
constexpr int SET_THREADS = 128;                // one set of FP8 warps
constexpr int Q_THREADS = 2 * SET_THREADS;      // two sets share out the quantizer's work items
constexpr int PIECES = 6;                       // base-8 digits of an FP8 activation block
constexpr uint32_t STG_MASK = REC_BYTES, STG_LIST = STG_MASK + 256;          // the unit's mask, the list of its FP8 blocks
constexpr uint32_t LIST_CAP = 3712;             // bytes of the list that fit a stage (about 305 blocks); more is read from global
constexpr uint32_t STG_STEP = STG_LIST + LIST_CAP;                           // 22528, 1 KiB aligned: step record
// DEC_UNPACK: the packed activation records of the stages lie behind the last stage.  From 14 tokens on four of them fit only without the 256
// bytes that nothing uses, in two copies.
constexpr uint32_t AREC_GAP = AREC_AT - AREC_HOT;
__host__ __device__ inline uint32_t arec_gap(int64_t M) { return M >= 14 ? AREC_GAP : 0u; }
constexpr int DEC_MAX_STAGES = 6;
// Two sets; three for one and two tokens without the packed form (their accumulators leave the tensor memory for it): 10.35 us instead of 10.47 at one
// token of 11008 x 4096, 28.8 and 28.7 of 28672 x 8192; with 20 % FP8 blocks, whose second halves come from global memory, 12.3 instead of 13.9 and 36.8
// instead of 46.7.  For more tokens it is no gain: eight of 28672 x 8192 39.4 instead of 36.1.
// Tensor memory columns: accumulators (two buffers of each kind); of each set: a dense E4M3 tile of 64, scales (32)
template <int SETS> struct Dec {
    static constexpr int W_EPI = W_SET + 4 * SETS, W_STEP = W_EPI + 4;
    static constexpr uint32_t D4 = SETS == 3 ? 64 : 112, D8 = SETS == 3 ? 16 : 32;
    static constexpr uint32_t D4_COL = 0, D8_COL = 2 * D4, DENSE_COL = D8_COL + 2 * D8, SF_COL = DENSE_COL + 64 * SETS;
    static_assert(SF_COL + 32 * SETS <= 512, "tensor memory columns");
};
constexpr uint32_t DEC_TMEM_COLS = 512;
constexpr size_t SMEM_LIMIT = 232448;
static_assert(STG_STEP % 1024 == 0, "stage layout");

enum { DEC_FUSED_LP = 0, DEC_FUSED_HP = 1, DEC_UNPACK = 2, DEC_OWN1_LP = 4, DEC_OWN1_HP = 5, DEC_OWN2_LP = 6, DEC_OWN2_HP = 7,
       DEC_OWN3_LP = 8, DEC_OWN3_HP = 9, DEC_OWN4_LP = 10, DEC_OWN4_HP = 11 };
// (the lowest bit of the fused ones is the fgmp_score_mode of the quantizer; OWN1 to OWN4 are for that many tokens)
constexpr int OWN_TURNS = 2;                    // units whose step records are made at a time: 64 threads take about 1 us for a token's, the weights half of that
constexpr int own_tokens(int src) { return src >= DEC_OWN1_LP ? (src - DEC_OWN1_LP) / 2 + 1 : 0; }
constexpr int dec_threads(int src, int sets) { return 32 * (W_SET + 4 * sets + 4 + (own_tokens(src) ? 2 * OWN_TURNS * own_tokens(src) : 1)); }

// Step record of a chunk for a batch of M tokens: n4 rows x 128 bytes of E2M1 codes | 2 KiB of block scales in tensor-
// memory order | n8 rows x 128 bytes of E5M2 values of elements 0..127 | the same of elements 128..255.  Both code tiles
// are K-major with 16-byte pieces XOR-swizzled by the row.  Rows that no token uses are left as they are: they only
// reach accumulator columns that nobody reads.
__host__ __device__ inline uint32_t step_n4(int64_t M) { return (uint32_t)(((PIECES + 1) * M + 15) & ~15); }
__host__ __device__ inline uint32_t step_n8(int64_t M) { return (uint32_t)((2 * M + 15) & ~15); }
__host__ __device__ inline uint32_t step_bytes(int64_t M) { return step_n4(M) * 128u + 2048u + step_n8(M) * 256u; }

// instruction descriptors without N, M = 128, K-major operands: E2M1 x E2M1 with UE4M3 scales; E4M3 x E5M2
constexpr uint32_t IDESC_NVF4 = (1u << 7) | (1u << 10) | ((uint32_t)(128 >> 4) << 24);
constexpr uint32_t IDESC_E4M3_E5M2 = (1u << 4) | (0u << 7) | (1u << 10) | ((uint32_t)(128 >> 4) << 24);

// shared-memory matrix descriptors as (low word | start address >> 4, constant high word)
constexpr uint32_t SW128_LO = 1u << 16, SW128_HI = (1024u >> 4) | (1u << 14) | (2u << 29);   // 128B swizzle, 8-row groups 1 KiB apart
__device__ __forceinline__ uint64_t desc64(uint32_t lo)
{
    uint64_t d;
    asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "r"(lo), "r"(SW128_HI));
    return d;
}
// A (128 rows) from tensor memory: lane = row, four bytes of K per column
__device__ __forceinline__ void umma_f8f6f4_ta(uint32_t d_tmem, uint32_t a_tmem, uint64_t bdesc, uint32_t idesc, uint32_t accumulate)
{
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
                 "tcgen05.mma.cta_group::1.kind::f8f6f4 [%0], [%1], %2, %3, p;\n\t}"
                 ::"r"(d_tmem), "r"(a_tmem), "l"(bdesc), "r"(idesc), "r"(accumulate) : "memory");
}

// control words of the workspace (int32, from byte 256): see fgmp_linear_fused
enum { CW_DONE = 1, CW_CLAIM = 2, CW_QCOUNT = 3 };

struct DecParams {
    const uint8_t* wblob; const uint8_t* ablob;
    PackedLayout LW, LA;
    float* Y; void* Ybf; int64_t ldy; int y_is_bf16;
    int64_t M, N, K;
    uint32_t chunks;
    uint32_t span, rest;      // units per CTA: span + 1 for the first `rest` CTAs, span for the others
    int* status; uint32_t* counters; float* partials; int maxseg;
    uint32_t stages, stage_bytes, arec_bytes;    // arec_bytes: of a packed activation record in shared memory (DEC_UNPACK)
    // activation quantizer in front (fused launches only)
    const uint8_t* X; int64_t ldx;        // bf16 [M, ldx]
    const float* fisher;
    ActQuantScalars q;
    uint8_t* steps;                       // the chunks' step records
    uint8_t* q_codes4; uint8_t* q_sf; uint8_t* q_mask; uint8_t* q_codes8; uint8_t* q_arec; fgmp_packed_header* q_header;   // optional packed output
    uint32_t* cw;                         // control words
};

struct StageMeta { uint32_t step, staged; };     // list start (16-byte steps), bytes of it in the stage

// Profiling builds (-DFGMP_TIMELINE) stamp the global timer at the phases of every CTA into a buffer
// registered with fgmp_debug_timeline (16 x uint64 per CTA); ordinary builds contain none of this.
#ifdef FGMP_TIMELINE
__device__ unsigned long long* g_timeline = nullptr;
#define FGMP_STAMP_ANY(slot) do { if (g_timeline) g_timeline[(size_t)blockIdx.x * 16 + (slot)] = globaltimer_ns(); } while (0)
#else
#define FGMP_STAMP_ANY(slot) do { } while (0)
#endif

__device__ __forceinline__ uint32_t span_begin(const DecParams& p, uint32_t cta) { return cta * p.span + min(cta, p.rest); }
__device__ __forceinline__ uint32_t cta_of_unit(const DecParams& p, uint32_t u)
{
    const uint32_t longer = p.rest * (p.span + 1);
    return u < longer ? u / (p.span + 1) : p.rest + (u - longer) / p.span;
}

// The units of a CTA in the order in which it takes them: from `begin` on, but the last `front` of them, the part of a tile that the next CTA goes on
// with, before all others where they are fewer than what the CTA has of the tile before.  Handing in a part's sums and adding them up takes 2.5 to 3.5 us
// and one set of warps, so that behind a last part of one unit (0.5 us) the part before is still under way: such CTAs were the last to end, by 2 us.  (In a
// graph, 16 tokens of 11008 x 4096 16.0 -> 14.4 us, one token 10.3 -> 9.8, 28672 x 8192 38.2 -> 37.8 and 28.8 -> 28.6.)
struct UnitOrder {
    uint32_t begin, end, front;
    __device__ __forceinline__ UnitOrder(uint32_t b, uint32_t e, uint32_t C) : begin(b), end(e)
    {
        const uint32_t last = e % C, before = min(C, e - b - min(e - b, last));
        front = last < before ? last : 0u;
    }
    __device__ __forceinline__ uint32_t unit(uint32_t i) const { return i < front ? end - front + i : begin + i - front; }
};

__device__ __forceinline__ void quant_bar() { asm volatile("bar.sync 1, %0;" ::"n"(Q_THREADS) : "memory"); }

// Bounded wait for a word in global memory to take a value that another CTA publishes.
__device__ __noinline__ bool wait_global_equals(const uint32_t* addr, uint32_t value, volatile int* abort_flag, int* status, int where)
{
    const unsigned long long t0 = globaltimer_ns();
    for (;;) {
        uint32_t v;
        asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(addr) : "memory");
        if (v == value) return true;
        if (*abort_flag) return false;
        if (globaltimer_ns() - t0 > MBAR_WAIT_LIMIT_NS) {
            *abort_flag = 1;
            atomicCAS(status, 0, (int)FGMP_ERR_TIMEOUT);
            atomicExch(status + 1, where);
            return false;
        }
        __nanosleep(20);
    }
}

__device__ __forceinline__ uint32_t f32x2_to_e5m2x2(float lo, float hi)
{
    uint16_t r;
    asm("cvt.rn.satfinite.e5m2x2.f32 %0, %1, %2;" : "=h"(r) : "f"(hi), "f"(lo));
    return r;
}
__device__ __forceinline__ float2 e5m2x2_to_f32x2(uint32_t two)
{
    uint32_t h2;
    asm("cvt.rn.f16x2.e5m2x2 %0, %1;" : "=r"(h2) : "h"((uint16_t)two));
    return __half22float2(*reinterpret_cast<__half2*>(&h2));
}

// The six digits of the E4M3 magnitude `code` (0..126) as E2M1 codes, digit p in bits 4p .. 4p+3.  Base 8, lowest first:
// the magnitude in units of 2^-9 is an integer of at most 18 bits, a digit d stands for the E2M1 value d / 2.  The top
// digit is at most 7; 5 and 7 are no E2M1 values (in halves): 5 = 6 - 1 and 7 = 6 + 1 with the 1 as -8 or 8 in the digit
// below, which is 0 or -4 then (the magnitude has four significant bits).
__device__ __forceinline__ uint32_t e4m3_digits(uint32_t code)
{
    int a = __float2int_rn(e4m3_to_f32(code) * 512.0f);
    int d[PIECES];
#pragma unroll
    for (int p = 0; p < PIECES - 1; ++p) {
        d[p] = ((a + 4) & 7) - 4;
        a = (a - d[p]) >> 3;
    }
    if (a == 5) { a = 6; d[PIECES - 2] -= 8; }
    if (a == 7) { a = 6; d[PIECES - 2] += 8; }
    d[PIECES - 1] = a;
    uint32_t w = 0;
#pragma unroll
    for (int p = 0; p < PIECES; p += 2) w |= f32x2_to_e2m1x2(0.5f * (float)d[p], 0.5f * (float)d[p + 1]) << (4 * p);
    return w;
}

// Four elements of an FP8 block, E4M3 codes c8 -> their digits: c[p] = the elements' E2M1 codes of digit p (16 bits)
__device__ __forceinline__ void fp8_digits4(uint32_t c8, const uint32_t* digits, uint32_t (&c)[PIECES])
{
    uint32_t d[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) d[i] = digits[(c8 >> (8 * i)) & 0x7fu] ^ (((c8 >> (8 * i)) & 0x80u) ? 0x888888u : 0u);
    // digits p and p + 1 of the four elements: bytes 2 x (two elements)
    const uint32_t e = (d[0] & 0x0f0f0fu) | ((d[1] & 0x0f0f0fu) << 4), o = ((d[0] >> 4) & 0x0f0f0fu) | (d[1] & 0xf0f0f0u);
    const uint32_t g = (d[2] & 0x0f0f0fu) | ((d[3] & 0x0f0f0fu) << 4), h = ((d[2] >> 4) & 0x0f0f0fu) | (d[3] & 0xf0f0f0u);
#pragma unroll
    for (int p = 0; p < PIECES; ++p) c[p] = __byte_perm((p & 1) ? o : e, (p & 1) ? h : g, (p >> 1) | ((4 + (p >> 1)) << 4)) & 0xffffu;
}
// block scale of row i (of seven) of a token: row 0 has the NVFP4 scale, digit p has 2^(3p - 8) in E4M3
__device__ __forceinline__ uint32_t step_scale(uint32_t i, bool is8, uint32_t sc)
{
    const uint32_t digit_sc = i == 1 ? 0x02u : 0x10u + 0x18u * (i - 2u);
    return i == 0 ? (is8 ? 0u : sc) : (is8 ? digit_sc : 0u);
}

// Writes what the step record `rec` holds of four consecutive elements of token m: quarter li of
// block column j.  c4: their E2M1 codes and sc: the block's scale (NVFP4 block), or c8: their E4M3 codes (FP8 block);
// v: the values over the tensor scale; digits: table of e4m3_digits.
__device__ __forceinline__ void emit_step(uint8_t* rec, uint32_t M, uint32_t n4, uint32_t n8, uint32_t m, uint32_t j, uint32_t li,
                                          bool is8, uint32_t c4, uint32_t sc, uint32_t c8, const float (&v)[4], const uint32_t* digits)
{
    uint8_t* sf = rec + n4 * 128u;
    uint8_t* b8 = sf + 2048u + (j >> 3) * (n8 * 128u);
    // E5M2 high and low parts
    const uint32_t h0 = f32x2_to_e5m2x2(v[0], v[1]), h1 = f32x2_to_e5m2x2(v[2], v[3]);
    const float2 f0 = e5m2x2_to_f32x2(h0), f1 = e5m2x2_to_f32x2(h1);
    const uint32_t l0 = f32x2_to_e5m2x2(v[0] - f0.x, v[1] - f0.y), l1 = f32x2_to_e5m2x2(v[2] - f1.x, v[3] - f1.y);
    {
        const uint32_t r = m, q = M + m;
        *reinterpret_cast<uint32_t*>(b8 + r * 128u + (((j & 7u) ^ (r & 7u)) << 4) + 4u * li) = h0 | (h1 << 16);
        *reinterpret_cast<uint32_t*>(b8 + q * 128u + (((j & 7u) ^ (q & 7u)) << 4) + 4u * li) = l0 | (l1 << 16);
    }
    if (!is8) {
        *reinterpret_cast<uint16_t*>(rec + fgmp_rec_w4_offset(m, j) + 2u * li) = (uint16_t)c4;
    } else {
        uint32_t c[PIECES];
        fp8_digits4(c8, digits, c);
#pragma unroll
        for (int p = 0; p < PIECES; ++p)
            *reinterpret_cast<uint16_t*>(rec + fgmp_rec_w4_offset((uint32_t)(p + 1) * M + m, j) + 2u * li) = (uint16_t)c[p];
    }
    // scales of the token's seven rows, two per lane
#pragma unroll
    for (uint32_t e = 0; e < 2; ++e) {
        const uint32_t i = 2u * li + e;
        if (i <= (uint32_t)PIECES) sf[fgmp_rec_sf_offset(i * M + m, j)] = (uint8_t)step_scale(i, is8, sc);
    }
}

__device__ __forceinline__ uint32_t f16x2_to_e5m2x2(uint32_t h)
{
    uint16_t r;
    asm("cvt.rn.satfinite.e5m2x2.f16x2 %0, %1;" : "=h"(r) : "r"(h));
    return r;
}
__device__ __forceinline__ uint32_t f16x2_to_e4m3x2(uint32_t h)
{
    uint16_t r;
    asm("cvt.rn.satfinite.e4m3x2.f16x2 %0, %1;" : "=h"(r) : "r"(h));
    return r;
}
// The same for a whole block (token m, block column j) of the packed activation record `ar`, both in shared memory; unscale: 2^-ratio
// twice in fp16; wanted8: whether the weights have FP8 blocks, which the E5M2 values are for.  Every step is exact: the values have at most
// six significant bits, a part of them three.
__device__ __forceinline__ void unpack_block(uint8_t* rec, const uint8_t* ar, uint32_t M, uint32_t n4, uint32_t n8, uint32_t m, uint32_t j, uint32_t unscale,
                                             bool wanted8, const uint32_t* digits)
{
    const uint4* at = reinterpret_cast<const uint4*>(ar + fgmp_arec_at_offset(m, j) - arec_gap(M));
    const uint4 a = at[0], b = at[1];
    const uint32_t sc = ar[AREC_SF + m * 16u + j], w[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
    const bool is8 = sc == 0;                            // (or a block of zeros)
    uint8_t* sf = rec + n4 * 128u;
    if (wanted8) {
        uint8_t* b8 = sf + 2048u + (j >> 3) * (n8 * 128u);
        const uint32_t q = M + m;
        uint32_t hi[4], lo[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            uint32_t h[2], l[2];
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                uint32_t back, rest;
                h[e] = f16x2_to_e5m2x2(w[2 * k + e]);
                asm("cvt.rn.f16x2.e5m2x2 %0, %1;" : "=r"(back) : "h"((uint16_t)h[e]));
                asm("sub.rn.f16x2 %0, %1, %2;" : "=r"(rest) : "r"(w[2 * k + e]), "r"(back));
                l[e] = f16x2_to_e5m2x2(rest);
            }
            hi[k] = h[0] | (h[1] << 16); lo[k] = l[0] | (l[1] << 16);
        }
        *reinterpret_cast<uint4*>(b8 + m * 128u + (((j & 7u) ^ (m & 7u)) << 4)) = make_uint4(hi[0], hi[1], hi[2], hi[3]);
        *reinterpret_cast<uint4*>(b8 + q * 128u + (((j & 7u) ^ (q & 7u)) << 4)) = make_uint4(lo[0], lo[1], lo[2], lo[3]);
    }
    if (!is8) {
        *reinterpret_cast<uint2*>(rec + fgmp_rec_w4_offset(m, j)) = *reinterpret_cast<const uint2*>(ar + AREC_A4 + fgmp_rec_w4_offset(m, j));
    } else {
#pragma unroll
        for (int half = 0; half < 2; ++half) {
            uint32_t c[2][PIECES];
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                uint32_t x0, x1;
                asm("mul.rn.f16x2 %0, %1, %2;" : "=r"(x0) : "r"(w[4 * half + 2 * e]), "r"(unscale));
                asm("mul.rn.f16x2 %0, %1, %2;" : "=r"(x1) : "r"(w[4 * half + 2 * e + 1]), "r"(unscale));
                fp8_digits4(f16x2_to_e4m3x2(x0) | (f16x2_to_e4m3x2(x1) << 16), digits, c[e]);
            }
#pragma unroll
            for (int p = 0; p < PIECES; ++p)
                *reinterpret_cast<uint32_t*>(rec + fgmp_rec_w4_offset((uint32_t)(p + 1) * M + m, j) + 4u * half) = c[0][p] | (c[1][p] << 16);
        }
    }
#pragma unroll
    for (uint32_t i = 0; i <= (uint32_t)PIECES; ++i) sf[fgmp_rec_sf_offset(i * M + m, j)] = (uint8_t)step_scale(i, is8, sc);
}

// One work item of the quantizer in front of a fused call: chunk c (256 elements) of the token rows 4 quad .. 4 quad + 3.
// Run by the 256 threads of warps 2..9: 64 threads (two warps) per token, four lanes per block.
template <int MODE>
__device__ __forceinline__ void quantize_item(const DecParams& p, uint32_t c, uint32_t quad, const uint32_t* digits)
{
    const uint32_t tq = threadIdx.x - 32u * W_SET;         // index among the quantizer's threads
    const uint32_t lane = tq & 31u, li = tq & 3u, j = (tq >> 2) & 15u;
    const uint32_t m = 4u * quad + (tq >> 6), M = (uint32_t)p.M;      // the same for a whole warp
    if (m >= M) return;
    const int64_t kb = 16 * (int64_t)c + j;
    const uint2 xin = __ldg(reinterpret_cast<const uint2*>(p.X + ((size_t)m * p.ldx + (size_t)kb * 16 + 4 * li) * 2));
    const float4 f = __ldg(reinterpret_cast<const float4*>(p.fisher + kb * 16 + 4 * li));
    const BlockQuarter r = quantize_block_quarter<MODE>(xin, f, p.q);
    const float2 va = __half22float2(*reinterpret_cast<const __half2*>(&r.h.x)), vb = __half22float2(*reinterpret_cast<const __half2*>(&r.h.y));
    const float v[4] = {va.x, va.y, vb.x, vb.y};
    emit_step(p.steps + (size_t)c * step_bytes(M), M, step_n4(M), step_n8(M), m, j, li, r.is8, r.c4, r.sc, r.c8, v, digits);
    if (p.q_codes4) {
        uint8_t* rec = p.q_arec + (size_t)c * AREC_BYTES;
        *reinterpret_cast<uint16_t*>(rec + AREC_A4 + fgmp_rec_w4_offset(m, j) + 2u * li) = (uint16_t)r.c4;
        *reinterpret_cast<uint2*>(rec + fgmp_arec_at_offset(m, j) + 8u * li) = r.h;
        if (li == 0) rec[AREC_SF + m * 16u + j] = (uint8_t)r.sc;
        const uint32_t bal = __ballot_sync(0xffffffffu, r.is8 && li == 0);
        uint32_t byte = 0;
#pragma unroll
        for (int b = 0; b < 8; ++b) byte |= ((bal >> (4 * b)) & 1u) << b;
        *reinterpret_cast<uint16_t*>(p.q_codes4 + ((int64_t)m * p.K) / 2 + kb * 8 + li * 2) = (uint16_t)r.c4;
        if (li == 0) p.q_sf[fgmp_sf_offset(m, kb, p.K)] = (uint8_t)r.sc;
        if (r.is8) *reinterpret_cast<uint32_t*>(p.q_codes8 + (int64_t)m * p.K + kb * 16 + 4 * li) = r.c8;
        if (lane == 0) {
            uint8_t* mb = p.q_mask + (size_t)m * p.LA.MW * 4 + (kb >> 3);    // lane 0: first block of the warp's eight
            mb[0] = (uint8_t)byte;
            if (kb + 8 == p.LA.KB && (p.LA.KB & 31) != 0) { mb[1] = 0; mb[2] = 0; }   // rest of the row's last mask word
        }
    }
}

// Sums of consecutive tokens of a row to and from a CTA's part of a tile.  Stores are whole sectors of 32 bytes: with 16 bytes for four tokens, three
// tokens of 4096 x 4096 took 7.9 us instead of 7.5, four of 8192 x 4096 10.3 instead of 10.0.
__device__ __forceinline__ void store_part(float* dst, const float (&v)[8])
{
    asm volatile("st.global.cg.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};"
                 ::"l"(dst), "r"(__float_as_uint(v[0])), "r"(__float_as_uint(v[1])), "r"(__float_as_uint(v[2])), "r"(__float_as_uint(v[3])),
                   "r"(__float_as_uint(v[4])), "r"(__float_as_uint(v[5])), "r"(__float_as_uint(v[6])), "r"(__float_as_uint(v[7])) : "memory");
}
__device__ __forceinline__ void store_part(float* dst, const float (&v)[4])
{
    asm volatile("st.global.cg.v8.b32 [%0], {%1, %2, %3, %4, %5, %5, %5, %5};"
                 ::"l"(dst), "r"(__float_as_uint(v[0])), "r"(__float_as_uint(v[1])), "r"(__float_as_uint(v[2])), "r"(__float_as_uint(v[3])), "r"(0) : "memory");
}
__device__ __forceinline__ void load_part(const float* src, float (&v)[8])
{
    uint32_t y[8];
    asm volatile("ld.global.cg.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(y[0]), "=r"(y[1]), "=r"(y[2]), "=r"(y[3]), "=r"(y[4]), "=r"(y[5]), "=r"(y[6]), "=r"(y[7]) : "l"(src) : "memory");
#pragma unroll
    for (int j = 0; j < 8; ++j) v[j] = __uint_as_float(y[j]);
}
__device__ __forceinline__ void load_part(const float* src, float (&v)[4])
{
    asm volatile("ld.global.cg.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]) : "l"(src) : "memory");
}

// A token's sum of a row from the accumulators: NVFP4 rows and digits (col 0 and 1 .. 6), and of the FP8 weight blocks, where there are any
template <typename Col>
__device__ __forceinline__ float token_sum(bool has_fp8, float rw, float ra, const Col& col, uint32_t high, uint32_t low)
{
    const auto c = [&](int k) { return __uint_as_float(col(k)); };
    const float x = has_fp8 ? c(0) + (__uint_as_float(high) + __uint_as_float(low)) * rw : c(0);
    return x + (((c(1) + c(2)) + c(3)) + ((c(4) + c(5)) + c(6))) * ra;
}

template <int SRC, int SETS>
__global__ void __launch_bounds__(dec_threads(SRC, SETS), 1)
decode_kernel(const __grid_constant__ DecParams p)
{
    extern __shared__ uint8_t smem_raw[];
    // 1 KiB aligned; an offset from the array keeps the pointer known to be shared memory (plain ld.shared / st.shared)
    uint8_t* smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
    constexpr int TOKENS = own_tokens(SRC);              // 0: as many as p.M says
    constexpr bool FUSED = SRC != DEC_UNPACK, OWN = TOKENS != 0, SHARED = FUSED && !OWN;      // SHARED: the CTAs share out the quantizer's work
    constexpr int X = DEC_MAX_STAGES;
    using D = Dec<SETS>;
    constexpr int W_EPI = D::W_EPI, W_STEP = D::W_STEP;
    const uint32_t S = p.stages;
    const uint32_t M = OWN ? (uint32_t)TOKENS : (uint32_t)p.M, n4 = step_n4(M), n8 = step_n8(M), a_bytes = step_bytes(M);
    uint8_t* arecs = smem + S * p.stage_bytes;           // DEC_UNPACK: S packed activation records
    uint64_t* bars = reinterpret_cast<uint64_t*>(arecs + S * p.arec_bytes);
    StageMeta* smeta = reinterpret_cast<StageMeta*>(bars + 4 * X + 4);
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smeta + X);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
    volatile uint32_t* s_misc = reinterpret_cast<volatile uint32_t*>(abort_flag + 1);   // [1..2] claimed item
    uint32_t* digits = const_cast<uint32_t*>(s_misc) + 4;                               // 128 entries

    const int warp = warp_index(), lane = threadIdx.x & 31;
    if (threadIdx.x == 0) FGMP_STAMP_ANY(0);
    // barriers of a stage: weights there, step record there, scales and dense tile in tensor memory, unit done (the stage and
    // what it had in tensor memory are free); accumulators full / empty (two each)
    const uint32_t wf0 = smem_u32(bars), sf0 = wf0 + 8 * X, rd0 = sf0 + 8 * X, dn0 = rd0 + 8 * X, accf0 = dn0 + 8 * X, acce0 = accf0 + 16;

    // this CTA's span of (tile, chunk) units
    const uint32_t G = gridDim.x, C = p.chunks;
    const uint32_t u_begin = span_begin(p, blockIdx.x), u_end = span_begin(p, blockIdx.x + 1), n_units = u_end - u_begin;
    const UnitOrder order(u_begin, u_end, C);
    const uint8_t* lists = p.wblob + p.LW.off_ovf;
    const bool has_fp8 = __ldg(&reinterpret_cast<const fgmp_packed_header*>(p.wblob)->n_fp8) != 0;
    const uint32_t quads = (M + 3u) / 4u, n_items = quads * C;      // the quantizer's work items: (chunk, four tokens)

    // ------------------------------------------------------------ set-up
    if (warp == W_PROD && lane == 0) {
        for (uint32_t s = 0; s < S; ++s) {
            mbar_init(wf0 + 8 * s, 1); mbar_init(sf0 + 8 * s, OWN ? 2 * M : SHARED ? 1 : 4); mbar_init(rd0 + 8 * s, 4); mbar_init(dn0 + 8 * s, 1);
        }
        for (int b = 0; b < 2; ++b) { mbar_init(accf0 + 8 * b, 1); mbar_init(acce0 + 8 * b, 4); }
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    // The first of the quantizer's work items is asked for right away.  (This kernel may have started before the one
    // before it in the stream has finished; that one lets it start only after its own last claim.)
    if (SHARED && threadIdx.x == 32 * W_SET) s_misc[1] = atomicInc(p.cw + CW_CLAIM, n_items + G - 1u);
    if (warp == W_MMA) tmem_alloc(smem_u32(tmem_slot), DEC_TMEM_COLS);
    if (warp >= W_EPI && warp < W_STEP) digits[threadIdx.x - 32 * W_EPI] = e4m3_digits(min(threadIdx.x - 32u * W_EPI, 126u));
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = TMEM_ALL;
    if (threadIdx.x == 0) FGMP_STAMP_ANY(1);

    if (warp == W_PROD) {
        // ------------------------------------------------------------ weights producer (whole warp; lane 0 issues)
        // The packed weights are not written by whatever runs before this kernel, so their first copies overlap the end
        // of that kernel (programmatic dependent launch).  Nothing is read through the blob's tables before its header has
        // been seen to describe this call.
        const fgmp_packed_header* hw = reinterpret_cast<const fgmp_packed_header*>(p.wblob);
        const uint2 mv = __ldg(reinterpret_cast<const uint2*>(hw));
        const int64_t rows = __ldg(&hw->rows), k = __ldg(&hw->K);
        const uint32_t kind = __ldg(&hw->kind);
        const int err = __ldg(&hw->error), free8 = __ldg(&hw->fp8_scale_free);
        int ok = mv.x == FGMP_MAGIC && mv.y == FGMP_LAYOUT_VERSION && rows == p.N && k == p.K && kind == 1u && err == 0 && free8 == 0;
        int bad = ok ? 0 : 9;
        auto load_arec = [&](uint32_t s, uint32_t unit) {    // the unit's packed activation record into stage s
            const uint8_t* src = p.ablob + p.LA.off_arec + (size_t)(unit % C) * AREC_BYTES;
            const uint32_t dst = smem_u32(arecs + s * p.arec_bytes);
            if (M < 14) { bulk_load(dst, src, p.arec_bytes, wf0 + 8 * s); return; }
            bulk_load(dst, src, AREC_HOT, wf0 + 8 * s);
            bulk_load(dst + AREC_HOT, src + AREC_AT, p.arec_bytes - AREC_HOT, wf0 + 8 * s);
        };
        const uint32_t* uptr = reinterpret_cast<const uint32_t*>(p.wblob + p.LW.off_uptr);
        uint32_t u = 0, pf_base = 0, pf = 0, refill = 0, stage = 0, phase = 1;
        const uint32_t pf_begin = order.front && u_begin + lane <= u_end ? __ldg(uptr + u_begin + lane) : 0u;
        const uint32_t pre = min(S, n_units);
        for (uint32_t i = 0; i <= n_units; ++i) {
            if (i == pre || !ok) {
                asm volatile("griddepcontrol.wait;" ::: "memory");
                if (threadIdx.x == 0) FGMP_STAMP_ANY(2);
                if (!FUSED) {
                    const fgmp_packed_header* ha = reinterpret_cast<const fgmp_packed_header*>(p.ablob);
                    if (ok && !(ha->magic == FGMP_MAGIC && ha->version == FGMP_LAYOUT_VERSION && ha->rows == p.M && ha->K == p.K && ha->kind == 0u && ha->fp8_scale_free == 0)) { ok = 0; bad = 10; }
                    if (ok && lane < pre) load_arec(lane, order.unit(lane));       // of the stages under way
                }
                if (bad && lane == 0) { *abort_flag = 1; atomicCAS(p.status, 0, (int)FGMP_ERR_INVALID_ARG); atomicExch(p.status + 1, bad); }
            }
            if (!ok || i == n_units) break;
            if (i == refill) {                         // next 32 list starts (one comparison a unit: with the order asked for every time, 2 x 28672 x 8192 took 31.2 us, not 30.6)
                u = pf_base = order.unit(i);
                if (i && i == order.front) pf = pf_begin;      // (asked for with the first: their way is as long as a unit takes)
                else pf = pf_base + lane <= u_end ? __ldg(uptr + pf_base + lane) : 0u;
                refill = i < order.front ? min(i + 31u, order.front) : i + 31u;
            }
            const uint32_t step0 = __shfl_sync(0xffffffffu, pf, (int)(u - pf_base)), step1 = __shfl_sync(0xffffffffu, pf, (int)(u + 1 - pf_base));
            if (lane == 0) {
                ok = mbar_wait(dn0 + 8 * stage, phase, abort_flag, p.status, 1) ? 1 : 0;
                if (ok) {
                    // one unit's copies: record, mask and list of the weights; the packed activation record goes with them
                    const uint32_t staged = min((step1 - step0) * 16u, LIST_CAP);
                    smeta[stage].step = step0; smeta[stage].staged = staged;
                    const uint32_t fb = wf0 + 8 * stage, dst = smem_u32(smem + stage * p.stage_bytes);
                    mbar_expect_tx(fb, REC_BYTES + 256u + staged + (FUSED ? 0u : p.arec_bytes));
                    bulk_load(dst, p.wblob + p.LW.off_rec + (size_t)u * REC_BYTES, REC_BYTES, fb);
                    bulk_load(dst + STG_MASK, p.wblob + p.LW.off_mask + (size_t)u * 256, 256u, fb);
                    if (staged) bulk_load(dst + STG_LIST, lists + (size_t)step0 * 16, staged, fb);
                    if (!FUSED && i >= pre) load_arec(stage, u);
                }
            }
            ok = __shfl_sync(0xffffffffu, ok, 0);
            ++u;
            if (++stage == S) { stage = 0; phase ^= 1; }
        }
    } else {
        // Everything before this touches neither the preceding kernel's output nor (but for the claim) the workspace.
        asm volatile("griddepcontrol.wait;" ::: "memory");
        if (!SHARED) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    }

    if (SHARED && warp >= W_SET && warp < W_SET + Q_THREADS / 32) {
        // ------------------------------------------------------------ quantizer
        // Work items are handed out through a counter, so that every item is taken by a CTA that is running: no CTA
        // ever waits for one that has not started.  The counter wraps to zero with the call's last claim.
        for (uint32_t it = 0;; ++it) {
            const uint32_t item = s_misc[1 + (it & 1u)];
            if (item >= n_items) break;
            // the next item is asked for while this one is worked on
            if (threadIdx.x == 32 * W_SET) s_misc[1 + ((it + 1u) & 1u)] = atomicInc(p.cw + CW_CLAIM, n_items + G - 1u);
            if (item == 0 && threadIdx.x == 32 * W_SET && p.q_header) {
                fgmp_packed_header* h = p.q_header;
                h->magic = FGMP_MAGIC; h->version = FGMP_LAYOUT_VERSION; h->rows = p.M; h->K = p.K; h->scale_fp4 = p.q.s4;
                h->fp8_log2_ratio = p.q.ratio; h->n_fp8 = (p.q.tau == INFINITY) ? 0 : -1; h->tau_eff = 0.f; h->kind = 0; h->capacity = 0;
                h->error = 0; h->scale_fp8 = p.q.s8; h->fp8_scale_free = 0;
            }
            quantize_item<(SRC & 1)>(p, item / quads, item % quads, digits);
            // The item's stores become visible with the count of finished items: the barrier orders them before the one
            // thread's release.
            quant_bar();
            if (threadIdx.x == 32 * W_SET)
                asm volatile("red.release.gpu.global.add.u32 [%0], %1;" ::"l"(p.cw + CW_QCOUNT), "r"(1u) : "memory");
        }
        if (threadIdx.x == 32 * W_SET) {
            asm volatile("griddepcontrol.launch_dependents;" ::: "memory");   // this CTA has made its last claim
            FGMP_STAMP_ANY(3);
        }
    }

    if (OWN && warp >= W_STEP) {
        // ------------------------------------------------------------ this CTA's own quantizer: 64 threads, four lanes per block, make what a step
        // record holds of one token; two units at a time.
        const uint32_t tq = threadIdx.x - 32u * W_STEP, part = tq >> 6, li = tq & 3u, j = (tq >> 2) & 15u, m = part % M;
        uint32_t i = part / M, c = order.unit(i) % C, stage = i, phase = 1;        // (fewer at a time than stages)
        // (the units taken first are chunks 0 .. front - 1)
        uint32_t c_end = i < order.front ? order.front : C, c_jump = i < order.front ? u_begin % C - order.front : 0u - C;
        const uint8_t* row = p.X + (size_t)m * p.ldx * 2 + 32u * j + 8u * li;
        const float* fish = p.fisher + 16u * j + 4u * li;
        uint2 x = make_uint2(0u, 0u);
        float4 f = make_float4(0.f, 0.f, 0.f, 0.f);
        if (i < n_units) { x = __ldg(reinterpret_cast<const uint2*>(row + 512u * c)); f = __ldg(reinterpret_cast<const float4*>(fish + 256u * c)); }
        for (; i < n_units; i += OWN_TURNS) {
            const BlockQuarter r = quantize_block_quarter<(SRC & 1)>(x, f, p.q);
            c += OWN_TURNS;
            while (c >= c_end) { c += c_jump; c_end = C; c_jump = 0u - C; }
            if (i + OWN_TURNS < n_units) { x = __ldg(reinterpret_cast<const uint2*>(row + 512u * c)); f = __ldg(reinterpret_cast<const float4*>(fish + 256u * c)); }
            const float2 va = __half22float2(*reinterpret_cast<const __half2*>(&r.h.x)), vb = __half22float2(*reinterpret_cast<const __half2*>(&r.h.y));
            const float v[4] = {va.x, va.y, vb.x, vb.y};
            if (!mbar_wait_warp(dn0 + 8 * stage, phase, abort_flag, p.status, 13)) break;
            emit_step(smem + stage * p.stage_bytes + STG_STEP, M, n4, n8, m, j, li, r.is8, r.c4, r.sc, r.c8, v, digits);
            fence_proxy_async();                       // the tensor core reads what ordinary stores wrote
            __syncwarp();
            if (lane == 0) mbar_arrive(sf0 + 8 * stage);
            stage += OWN_TURNS;
            if (stage >= S) { stage -= S; phase ^= 1u; }
        }
    } else if (warp == W_STEP) {
        // ------------------------------------------------------------ step-record producer
        if (SHARED && lane == 0) {
            // every chunk's record is in place once the last work item of the quantizer has been handed in
            bool ok = wait_global_equals(p.cw + CW_QCOUNT, n_items, abort_flag, p.status, 8);
            asm volatile("fence.proxy.async;" ::: "memory");   // records were written with ordinary stores, the bulk copy reads them
            FGMP_STAMP_ANY(4);
            uint32_t stage = 0, phase = 1, c = order.unit(0) % C;
            for (uint32_t i = 0; i < n_units && ok; ++i) {
                if (i == order.front) c = u_begin % C;
                if (!(ok = mbar_wait(dn0 + 8 * stage, phase, abort_flag, p.status, 13))) break;
                mbar_expect_tx(sf0 + 8 * stage, a_bytes);
                bulk_load(smem_u32(smem + stage * p.stage_bytes) + STG_STEP, p.steps + (size_t)c * a_bytes, a_bytes, sf0 + 8 * stage);
                if (++stage == S) { stage = 0; phase ^= 1; }
                if (++c == C) c = 0;
            }
        }
        __syncwarp();
    } else if (warp == W_MMA) {
        // ------------------------------------------------------------ MMA issuer
        // The whole warp walks the loop; one elected lane issues the tcgen05 instructions, so that every commit tracks
        // every MMA before it.  The set that hands over a unit has seen the weights and the step record complete.
        const uint32_t idesc4 = IDESC_NVF4 | ((n4 >> 3) << 17), idesc8 = IDESC_E4M3_E5M2 | ((n8 >> 3) << 17);
        const uint32_t step_lo = (p.stage_bytes >> 4), b8_lo = (n4 * 128u + 2048u) >> 4, b8_half = n8 * 8u;
        const uint32_t w_first = (smem_u32(smem) >> 4) | SW128_LO;
        uint32_t stage = 0, phase = 0, w4 = w_first, left = order.front ? order.front : C - u_begin % C, accum = 0, acc = 0, acc_phase = 1, set = 0;
        for (uint32_t i = 0; i < n_units; ++i) {
            if (accum == 0) {                          // a tile begins
                if (!mbar_wait_uniform(acce0 + 8 * acc, acc_phase, abort_flag, p.status, 2)) break;
            }
            if (!mbar_wait_uniform(rd0 + 8 * stage, phase, abort_flag, p.status, 8)) break;
            if (i == 0 && lane == 0) FGMP_STAMP_ANY(5);
            if (i == n_units - 1 && lane == 0) FGMP_STAMP_ANY(6);
            tc_fence_after();
            const uint32_t a4 = w4 + (STG_STEP >> 4), a8 = a4 + b8_lo;
            const uint32_t d4 = tmem_base + D::D4_COL + acc * D::D4, d8 = tmem_base + D::D8_COL + acc * D::D8;
            const uint32_t sf_t = tmem_base + D::SF_COL + set * 32, w8 = tmem_base + D::DENSE_COL + set * 64;
            set = set == SETS - 1 ? 0u : set + 1u;
            if (elect_one()) {
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    umma_nvf4(d4, desc64(w4 + 2 * j), desc64(a4 + 2 * j), idesc4, sf_t + 4 * j, sf_t + 16 + 4 * j, j ? 1u : accum);
                if (has_fp8) {
#pragma unroll
                    for (uint32_t k = 0; k < 8; ++k)
                        umma_f8f6f4_ta(d8, w8 + 8 * k, desc64(a8 + (k >> 2) * b8_half + 2 * (k & 3u)), idesc8, k ? 1u : accum);
                }
                umma_commit(dn0 + 8 * stage);
            }
            __syncwarp();
            accum = 1; w4 += step_lo;
            if (++stage == S) { stage = 0; phase ^= 1; w4 = w_first; }
            if (--left == 0 || i + 1 == n_units) {     // the tile (or this CTA's part of it) ends
                if (elect_one()) umma_commit(accf0 + 8 * acc);
                __syncwarp();
                left = i + 1 == order.front ? C - u_begin % C : C; accum = 0;
                acc ^= 1u;
                if (acc == 0) acc_phase ^= 1u;
            }
        }
    } else if (warp >= W_SET && warp < W_EPI) {
        // ------------------------------------------------------------ sets: units set, set + SETS, ...: scales and FP8 blocks
        // Thread = row of the tile = lane of tensor memory (quadrant warp % 4).
        const uint32_t set = (uint32_t)(warp - W_SET) >> 2, row = 32u * (warp & 3) + lane;
        const uint32_t quadrant = tmem_base + ((uint32_t)((warp & 3) * 32) << 16);
        const uint32_t dense = quadrant + D::DENSE_COL + set * 64, sf_t = quadrant + D::SF_COL + set * 32;
        uint32_t unscale = 0;                          // 2^-ratio, twice in fp16: back to the E4M3 value of an FP8 element
        if (!FUSED) unscale = (uint32_t)(15 - reinterpret_cast<const fgmp_packed_header*>(p.ablob)->fp8_log2_ratio) * 0x04000400u;
        uint32_t stage = set, phase = 0, done = set, dphase = 0;      // done: stage of the set's last unit
        for (uint32_t i = set; i < n_units; i += SETS) {
            const uint8_t* sb = smem + stage * p.stage_bytes;
            // (Barriers are waited for by parity, so the stage's unit before this one, another set's where the number of stages is no multiple of that of the
            // sets, must be known to be in.  This set has seen unit i - 2 SETS done, which says so from twice as many stages as sets on.)
            if (!mbar_wait_warp(wf0 + 8 * stage, phase, abort_flag, p.status, 5)) break;
            if (!FUSED) {
                // the unit's step record from the packed activation record
                uint8_t* rec = smem + stage * p.stage_bytes + STG_STEP;
                const uint8_t* ar = arecs + stage * p.arec_bytes;
                // Up to four tokens a quarter of a block per thread, above that a whole block, tokens fastest, so that a quarter of a warp reads
                // 256 and writes 128 contiguous bytes at a time.  (28672 x 8192: 1 token 36.9 us by quarters, 40.5 by blocks; 8 tokens
                // 49.9 by quarters, 42.7 by blocks.)
                const uint32_t ts = (threadIdx.x - 32u * W_SET) & (SET_THREADS - 1u);
                if (M <= 4) {
                    const uint32_t li = ts & 3u, j = (ts >> 2) & 15u;
#pragma unroll 1
                    for (uint32_t m = ts >> 6; m < M; m += 2) {
                        const uint2 h = *reinterpret_cast<const uint2*>(ar + fgmp_arec_at_offset(m, j) + 8u * li);
                        const uint32_t c4 = *reinterpret_cast<const uint16_t*>(ar + AREC_A4 + fgmp_rec_w4_offset(m, j) + 2u * li), sc = ar[AREC_SF + m * 16u + j];
                        const float2 va = __half22float2(*reinterpret_cast<const __half2*>(&h.x)), vb = __half22float2(*reinterpret_cast<const __half2*>(&h.y));
                        const float v[4] = {va.x, va.y, vb.x, vb.y};
                        uint32_t x0, x1;
                        asm("mul.rn.f16x2 %0, %1, %2;" : "=r"(x0) : "r"(h.x), "r"(unscale));
                        asm("mul.rn.f16x2 %0, %1, %2;" : "=r"(x1) : "r"(h.y), "r"(unscale));
                        emit_step(rec, M, n4, n8, m, j, li, sc == 0, c4, sc, f16x2_to_e4m3x2(x0) | (f16x2_to_e4m3x2(x1) << 16), v, digits);
                    }
                } else {
#pragma unroll 1
                    for (uint32_t m = ts & 7u; m < M; m += 8) unpack_block(rec, ar, M, n4, n8, m, ts >> 3, unscale, has_fp8, digits);
                }
                fence_proxy_async();                   // the tensor core reads what ordinary stores wrote
                __syncwarp();
                if (lane == 0) mbar_arrive(sf0 + 8 * stage);
            }
            // the tensor core has read what the set's last unit had in tensor memory
            if (i >= SETS) {
                if (!mbar_wait_warp(dn0 + 8 * done, dphase, abort_flag, p.status, 7)) break;
                tc_fence_after();
                done += SETS;
                if (done >= S) { done -= S; dphase ^= 1; }
            }
            // Block scales: lane i holds, for MMA step j, the four scale bytes of operand rows i, 32+i, 64+i, 96+i in columns
            // 4j..4j+3: 16 bytes of scale tile j of the weight record; of the step record in columns 16..31.
            auto scales = [&](const uint8_t* src, uint32_t dst) {
                uint32_t r[16];
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const uint4 x = *reinterpret_cast<const uint4*>(src + 512 * j);
                    r[4 * j] = x.x; r[4 * j + 1] = x.y; r[4 * j + 2] = x.z; r[4 * j + 3] = x.w;
                }
                tmem_st16(dst, r);
            };
            scales(sb + REC_SF + lane * 16, sf_t);
            if (has_fp8) {
                // The row's FP8 blocks lie one after the other in the list.
                const uint16_t* before = reinterpret_cast<const uint16_t*>(sb + REC_KBSTART);
                const uint32_t cnt = before[16], hoff = fgmp_list_halves_offset(cnt), m16 = reinterpret_cast<const uint16_t*>(sb + STG_MASK)[row];
                uint32_t at = __popc(m16);             // sum over the rows 8 (row / 8) .. row
#pragma unroll
                for (int o = 1; o < 8; o <<= 1) { const uint32_t y = __shfl_up_sync(0xffffffffu, at, o, 8); if ((lane & 7) >= o) at += y; }
                at = hoff + 8u * (before[row >> 3] + at - __popc(m16));
                const bool all = hoff + 8u * cnt <= smeta[stage].staged;       // the usual case: the whole list is in the stage
                const uint32_t slot = smem_u32(sb) + REC_W4 + row * 128u;
                uint32_t hs = smem_u32(sb) + STG_LIST + at;
#pragma unroll 1
                for (uint32_t c = 0; c < 2; ++c) {     // eight block columns at a time
                    uint32_t r[32];
#pragma unroll
                    for (uint32_t k = 0; k < 8; ++k) {
                        const uint32_t is8 = (m16 >> (8 * c + k)) & 1u;
                        const uint2 lo = lds64_if(slot + (((4 * c + (k >> 1)) ^ (row & 7u)) << 4) + (k & 1u) * 8u, is8);
                        const uint2 hi = lds64_if(hs, is8 && all);
                        hs += 8u * is8;
                        r[4 * k] = lo.x; r[4 * k + 1] = lo.y; r[4 * k + 2] = hi.x; r[4 * k + 3] = hi.y;
                    }
                    if (!all) {
                        const uint8_t* list_g = lists + (size_t)smeta[stage].step * 16;
#pragma unroll
                        for (uint32_t k = 0; k < 8; ++k)
                            if ((m16 >> (8 * c + k)) & 1u) {
                                const uint2 hi = __ldg(reinterpret_cast<const uint2*>(list_g + at));
                                at += 8u;
                                r[4 * k + 2] = hi.x; r[4 * k + 3] = hi.y;
                            }
                        __syncwarp();
                    }
                    tmem_st32(dense + 32 * c, r);
                }
            }
            if (!mbar_wait_warp(sf0 + 8 * stage, phase, abort_flag, p.status, 16)) break;
            scales(sb + STG_STEP + n4 * 128u + lane * 16, sf_t + 16);
            tmem_wait_st();
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(rd0 + 8 * stage);
            stage += SETS;
            if (stage >= S) { stage -= S; phase ^= 1; }
        }
    }
    else if (warp >= W_EPI && warp < W_STEP) {
        // ------------------------------------------------------------ epilogue: tensor-memory lane quadrant warp % 4
        const int q = warp & 3;
        const fgmp_packed_header* hw = reinterpret_cast<const fgmp_packed_header*>(p.wblob);
        const fgmp_packed_header* ha = reinterpret_cast<const fgmp_packed_header*>(p.ablob);
        const float alpha = __fmul_rn(FUSED ? p.q.s4 : ha->scale_fp4, __ldg(&hw->scale_fp4));
        // FP8 tensor scale / NVFP4 tensor scale of either operand
        const float rw = __int_as_float((127 + __ldg(&hw->fp8_log2_ratio)) << 23);
        const float ra = FUSED ? p.q.r8 : __int_as_float((127 + ha->fp8_log2_ratio) << 23);
        constexpr uint32_t W = TOKENS > 2 ? 4u : 8u;       // tokens at a time (four: eight take more than 64 registers)
        const uint32_t row = 32 * q + lane, rounds = (M + W - 1u) / W;
        // W tokens' sums of the row, from token W o on, to Y
        const auto emit = [&](const float (&v)[W], uint32_t o, int64_t n) {
            if (n >= p.N) return;
            const int64_t at = (int64_t)(W * o) * p.ldy + n;
            __nv_bfloat16* yb = reinterpret_cast<__nv_bfloat16*>(p.Ybf) + at;
            float* yf = p.Y + at;
#pragma unroll
            for (uint32_t j = 0; j < (OWN ? (uint32_t)TOKENS : W); ++j) {
                if (W * o + j < M) {
                    if (p.y_is_bf16) *yb = __float2bfloat16_rn(v[j] * alpha);
                    else *yf = v[j] * alpha;
                }
                yb += p.ldy; yf += p.ldy;
            }
        };
        uint32_t accb = 0, acc_phase = 0;
        for (uint32_t i = 0; i < n_units;) {
            const uint32_t u = order.unit(i), tile = u / C, t_begin = tile * C, t_end = t_begin + C, u_stop = min(t_end, u_end);
            const bool whole = u == t_begin && t_end <= u_end;
            i += u_stop - u;
            uint32_t nseg = 1, slot = 0;
            if (!whole) {                              // (before the wait: the divisions take a while)
                const uint32_t c_first = cta_of_unit(p, t_begin);
                nseg = cta_of_unit(p, t_end - 1) - c_first + 1;
                slot = blockIdx.x - c_first;
            }
            const int64_t n = (int64_t)tile * 128 + row;
            float* base = p.partials + ((size_t)tile * p.maxseg * 128 + row) * 16;
            if (!mbar_wait_warp(accf0 + 8 * accb, acc_phase, abort_flag, p.status, 11)) break;
            tc_fence_after();
            if (i == n_units && threadIdx.x == W_EPI * 32) FGMP_STAMP_ANY(10);
            // a tile shared with other CTAs: how many of them have handed in their sums already (the answer is needed only after this CTA's own sums are
            // complete; when all others were seen to have arrived, this warp is the last without asking)
            uint32_t* counter = p.counters + tile * 8 + q;
            uint32_t seen = 0;
            if (!whole && lane == 0) asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(seen) : "l"(counter) : "memory");
            // columns m (NVFP4 blocks), (p + 1) M + m (digits); FP8 weights: m (high), M + m (low)
            const uint32_t d4 = tmem_base + ((uint32_t)(q * 32) << 16) + D::D4_COL + accb * D::D4;
            const uint32_t d8 = tmem_base + ((uint32_t)(q * 32) << 16) + D::D8_COL + accb * D::D8;
#pragma unroll 1
            for (uint32_t o = 0; o < rounds; ++o) {
                float v[W];
                if constexpr (OWN && TOKENS <= 2) {
                    // at most 14 and 4 columns: one load of each
                    uint32_t r0[16], r1[16], r2[16] = {};
                    tmem_ld16_async(d4, r0); tmem_ld16_async(d8, r1);
                    tmem_wait_ld(r0, r1, r2);
#pragma unroll
                    for (uint32_t j = 0; j < W; ++j) v[j] = 0.f;
#pragma unroll
                    for (int j = 0; j < TOKENS; ++j) v[j] = token_sum(has_fp8, rw, ra, [&](int k) { return r0[TOKENS * k + j]; }, r1[j], r1[TOKENS + j]);
                } else {
                    uint32_t r[PIECES + 1][W], hi[W], lo[W];
#pragma unroll
                    for (uint32_t k = 0; k <= (uint32_t)PIECES; ++k) tmem_ld_async(d4 + k * M + W * o, r[k]);
                    tmem_ld_async(d8 + W * o, hi); tmem_ld_async(d8 + M + W * o, lo);
                    tmem_wait_ld();
                    tmem_hold(hi); tmem_hold(lo);
#pragma unroll
                    for (uint32_t k = 0; k <= (uint32_t)PIECES; ++k) tmem_hold(r[k]);
#pragma unroll
                    for (uint32_t j = 0; j < W; ++j) v[j] = token_sum(has_fp8, rw, ra, [&](int k) { return r[k][j]; }, hi[j], lo[j]);
                }
                if (whole) emit(v, o, n);
                else store_part(base + (size_t)slot * 2048 + W * o, v);         // this CTA's part
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(acce0 + 8 * accb);
            accb ^= 1u;
            if (accb == 0) acc_phase ^= 1u;
            if (i == n_units && threadIdx.x == W_EPI * 32) FGMP_STAMP_ANY(11);
            if (!whole) {
                // The counter wraps to zero with the last arrival (or is put back by the warp that need not ask it), so the workspace is ready for the next
                // call without being cleared.
                uint32_t old = __shfl_sync(0xffffffffu, seen, 0);
                if (old != nseg - 1) {
                    // the warp's stores are ordered before lane 0's release of the counter; its acquire sees the others'
                    if (lane == 0)
                        asm volatile("atom.acq_rel.gpu.global.inc.u32 %0, [%1], %2;" : "=r"(old) : "l"(counter), "r"(nseg - 1) : "memory");
                    old = __shfl_sync(0xffffffffu, old, 0);
                } else if (lane == 0) {
                    *counter = 0u;
                }
                if (i == n_units && threadIdx.x == W_EPI * 32) FGMP_STAMP_ANY(12);
                if (old == nseg - 1) {                 // this warp is the last: it adds everything up
#pragma unroll 1
                    for (uint32_t o = 0; o < rounds; ++o) {
                        float v[W];
#pragma unroll
                        for (uint32_t j = 0; j < W; ++j) v[j] = 0.f;
#pragma unroll 1
                        for (uint32_t g = 0; g < nseg; g += 2) {       // one sum in slot order, two parts under way at a time
                            float y[2][W];
#pragma unroll
                            for (uint32_t h = 0; h < 2; ++h) load_part(base + (size_t)min(g + h, nseg - 1u) * 2048 + W * o, y[h]);      // (a last one twice)
#pragma unroll
                            for (uint32_t h = 0; h < 2; ++h) {
                                if (g + h >= nseg) break;
#pragma unroll
                                for (uint32_t j = 0; j < W; ++j) v[j] += y[h][j];
                            }
                        }
                        emit(v, o, n);
                    }
                }
            }
            if (i == n_units && threadIdx.x == W_EPI * 32) FGMP_STAMP_ANY(whole ? 7 : 8);    // last segment: sums complete / handed in
        }
    }

    __syncthreads();
    if (threadIdx.x == 0) FGMP_STAMP_ANY(9);
    if (*abort_flag) {
        const unsigned long long t0 = globaltimer_ns();
        while (globaltimer_ns() - t0 < 2000000ull) __nanosleep(1000);
        __syncthreads();
    } else if (SHARED && threadIdx.x == 0) {
        // the CTA that finishes last takes the count of finished items back, so that the control area is as the next call needs it
        if (atomicInc(p.cw + CW_DONE, G - 1u) == G - 1u)
            asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(p.cw + CW_QCOUNT), "r"(0u) : "memory");
    }
    if (warp == W_MMA) {
        tc_fence_after();
        tmem_dealloc(tmem_base, DEC_TMEM_COLS);
    }
}

struct DecPlan { int64_t tiles, chunks, total; int grid; int maxseg; int64_t span, rest; };

DecPlan decode_plan(int64_t N, int64_t K)
{
    DecPlan d;
    d.tiles = (N + 127) / 128; d.chunks = K / 256; d.total = d.tiles * d.chunks;
    const int sms = fgmp_sm_count();
    d.grid = (int)(d.total < sms ? d.total : sms);
    // a tile of `chunks` units meets at most this many CTA spans of >= floor(total/grid) units
    d.span = d.total / d.grid; d.rest = d.total % d.grid;
    d.maxseg = (int)((d.chunks + d.span - 1) / d.span + 1);
    return d;
}

std::mutex g_dec_mu;                 // guards the per-device caches below
bool g_attr_set[64] = {};

fgmp_status set_attrs_once()
{
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return FGMP_ERR_CUDA;
    std::lock_guard<std::mutex> lk(g_dec_mu);
    if (!g_attr_set[dev]) {
        bool ok = true;
        for (const void* k : {(const void*)decode_kernel<DEC_FUSED_LP, 2>, (const void*)decode_kernel<DEC_FUSED_HP, 2>, (const void*)decode_kernel<DEC_OWN1_LP, 3>,
                              (const void*)decode_kernel<DEC_OWN1_HP, 3>, (const void*)decode_kernel<DEC_OWN2_LP, 3>, (const void*)decode_kernel<DEC_OWN2_HP, 3>,
                              (const void*)decode_kernel<DEC_OWN3_LP, 2>, (const void*)decode_kernel<DEC_OWN3_HP, 2>, (const void*)decode_kernel<DEC_OWN4_LP, 2>,
                              (const void*)decode_kernel<DEC_OWN4_HP, 2>,
                              (const void*)decode_kernel<DEC_FUSED_LP, 3>, (const void*)decode_kernel<DEC_FUSED_HP, 3>, (const void*)decode_kernel<DEC_UNPACK, 2>})
            ok = ok && cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SMEM_LIMIT) == cudaSuccess;
        if (!ok)
            return FGMP_ERR_CUDA;
        g_attr_set[dev] = true;
    }
    return FGMP_OK;
}

// Workspace of the decode path, all inside the control area that must be zero before the first call and
// that every call leaves zero: status at 0, control words at 256, stream-K
// counters from 1024 (32 bytes per tile); partial sums behind the control area, then (fused calls) the
// step records.
DecParams base_params(const void* packed_weights, void* Y, int y_is_bf16, int64_t ldy, int64_t M, int64_t N, int64_t K,
                      void* workspace, const DecPlan& d)
{
    uint8_t* ws = (uint8_t*)workspace;
    DecParams p{};
    p.wblob = (const uint8_t*)packed_weights;
    p.LW = fgmp_layout(N, K, 1, 0); p.LA = fgmp_layout(M, K, 0, 0);
    p.Y = (float*)Y; p.Ybf = Y; p.ldy = ldy; p.y_is_bf16 = y_is_bf16;
    p.M = M; p.N = N; p.K = K; p.chunks = (uint32_t)d.chunks; p.span = (uint32_t)d.span; p.rest = (uint32_t)d.rest;
    p.status = reinterpret_cast<int*>(ws);
    p.cw = reinterpret_cast<uint32_t*>(ws + 256);
    p.counters = reinterpret_cast<uint32_t*>(ws + 1024);
    p.partials = reinterpret_cast<float*>(ws + FGMP_WS_CONTROL_BYTES);
    p.maxseg = d.maxseg;
    return p;
}

template <int SRC, int SETS>
fgmp_status launch_decode(DecParams p, const DecPlan& d, bool programmatic, cudaStream_t s)
{
    p.arec_bytes = SRC == DEC_UNPACK ? (p.M <= 8 ? AREC_BYTES - 4096u : AREC_BYTES) - arec_gap(p.M) : 0u;
    p.stage_bytes = (STG_STEP + step_bytes(p.M) + 1023u) & ~1023u;
    constexpr size_t fixed = 1024 /*alignment*/ + 1024 /*barriers, digit table*/;
    const uint32_t fit = (uint32_t)((SMEM_LIMIT - fixed) / (p.stage_bytes + p.arec_bytes));      // 4 (16 tokens) to 7
    // step records of 16 tokens (see step_bytes), of eight; the kernel's sets count on four stages at least, three sets on six
    static_assert(4 * (STG_STEP + 112 * 128 + 2048 + 32 * 256 + AREC_BYTES - AREC_GAP) + fixed <= SMEM_LIMIT && STG_STEP % 1024 == 0, "four stages");
    static_assert(6 * (STG_STEP + 64 * 128 + 2048 + 16 * 256) + fixed <= SMEM_LIMIT && DEC_MAX_STAGES >= 6, "six stages");
    p.stages = fit < (uint32_t)DEC_MAX_STAGES ? fit : (uint32_t)DEC_MAX_STAGES;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)d.grid); cfg.blockDim = dim3(dec_threads(SRC, SETS)); cfg.stream = s;
    cfg.dynamicSmemBytes = fixed + (size_t)p.stages * (p.stage_bytes + p.arec_bytes);
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr; cfg.numAttrs = programmatic ? 1 : 0;
    FGMP_LAUNCH(FGMP_K_DECODE, s, cudaLaunchKernelEx(&cfg, decode_kernel<SRC, SETS>, p));
    return fgmp_launch_status();
}

}  // namespace

bool fgmp_decode_supported(int64_t M, int64_t N, int64_t K)
{
    return M >= 1 && M <= 16 && N >= 1 && K >= 256 && (K % 256) == 0 &&
           1024 + ((N + 127) / 128) * 32 <= (int64_t)FGMP_WS_CONTROL_BYTES;
}

size_t fgmp_ws_decode(int64_t M, int64_t N, int64_t K)
{
    if (!fgmp_decode_supported(M, N, K)) return 0;
    const DecPlan d = decode_plan(N, K);
    return (size_t)FGMP_WS_CONTROL_BYTES + (size_t)d.tiles * d.maxseg * 128 * 16 * 4;
}

size_t fgmp_ws_linear_fused(int64_t M, int64_t N, int64_t K)
{
    if (!fgmp_decode_supported(M, N, K)) return fgmp_ws_linear(M, N, K);
    return fgmp_align1k(fgmp_ws_decode(M, N, K)) + (size_t)(K / 256) * step_bytes(M);
}

// clear_first: zero the control area on the stream before the kernel (for scratch whose state the
// caller cannot vouch for); otherwise the kernel is launched as a programmatic dependent of the
// kernel before it in the stream, so that its set-up and first weight copies overlap that kernel's end.
fgmp_status fgmp_linear_decode(const void* packed_acts, const void* packed_weights, void* Y, int y_is_bf16, int64_t ldy,
                               int64_t M, int64_t N, int64_t K, void* workspace, bool clear_first, cudaStream_t s)
{
    const DecPlan d = decode_plan(N, K);
    DecParams p = base_params(packed_weights, Y, y_is_bf16, ldy, M, N, K, workspace, d);
    p.ablob = (const uint8_t*)packed_acts;
    fgmp_status st = set_attrs_once();
    if (st != FGMP_OK) return st;
    if (clear_first && cudaMemsetAsync(workspace, 0, 1024 + (size_t)d.tiles * 32, s) != cudaSuccess) return FGMP_ERR_CUDA;
    return launch_decode<DEC_UNPACK, 2>(p, d, !clear_first, s);
}

extern "C" fgmp_status fgmp_linear_fused(const void* X_bf16, int64_t ldx, const float* fisher_chan,
                                         fgmp_scales sc, fgmp_score_mode sm, float tau, const void* packed_weights,
                                         void* Y, int y_is_bf16, int64_t ldy, int64_t M, int64_t N, int64_t K,
                                         void* packed_acts_out, size_t packed_bytes,
                                         void* workspace, size_t ws_bytes, void* cuda_stream)
{
    if (!X_bf16 || !fisher_chan || !packed_weights || !Y || !workspace) return FGMP_ERR_INVALID_ARG;
    if ((int)sm < 0 || (int)sm > 1 || tau != tau) return FGMP_ERR_INVALID_ARG;
    if (!(sc.scale_fp4 > 0.f) || !isfinite(sc.scale_fp4)) return FGMP_ERR_INVALID_ARG;
    if (!fgmp_scales_valid(sc) || fgmp_fp8_free(sc)) return FGMP_ERR_INVALID_ARG;   // a free FP8 scale: the two calls and fgmp_linear_classes
    if (M < 1 || N < 1 || K < 64 || (K % 64) != 0 || ldy < N || ldx < K || (ldx % 8) != 0) return FGMP_ERR_SHAPE;
    if (((uintptr_t)X_bf16 & 15) || ((uintptr_t)fisher_chan & 15) || ((uintptr_t)packed_weights & 1023) ||
        ((uintptr_t)workspace & 1023) || ((uintptr_t)Y & 15) || ((uintptr_t)packed_acts_out & 1023)) return FGMP_ERR_SHAPE;
    if (ws_bytes < (fgmp_decode_supported(M, N, K) ? fgmp_ws_linear_fused(M, N, K) : fgmp_ws_linear_least(M, N, K))) return FGMP_ERR_WORKSPACE;
    if (packed_acts_out && packed_bytes < fgmp_layout(M, K, 0, 0).total) return FGMP_ERR_WORKSPACE;
    if (!fgmp_decode_supported(M, N, K)) {
        // larger batches: the two calls (the quantizer is then a small part of the step)
        if (!packed_acts_out) return FGMP_ERR_INVALID_ARG;
        fgmp_status st2 = fgmp_quantize_activations(X_bf16, ldx, fisher_chan, M, K, sc, sm, tau, packed_acts_out, packed_bytes,
                                                    nullptr, 0, cuda_stream);
        if (st2 != FGMP_OK) return st2;
        return fgmp_linear(packed_acts_out, packed_weights, Y, y_is_bf16, ldy, M, N, K, workspace, ws_bytes, cuda_stream);
    }
    fgmp_status st;
    if ((st = fgmp_require_sm100()) != FGMP_OK) return st;
    if ((st = set_attrs_once()) != FGMP_OK) return st;
    const DecPlan d = decode_plan(N, K);
    DecParams p = base_params(packed_weights, Y, y_is_bf16, ldy, M, N, K, workspace, d);
    p.X = (const uint8_t*)X_bf16; p.ldx = ldx; p.fisher = fisher_chan;
    // the same scalars, computed the same way, as fgmp_quantize_activations uses
    p.q.s4 = sc.scale_fp4;
    p.q.k6 = 1.0f / (6.0f * sc.scale_fp4);
    p.q.s8 = ldexpf(sc.scale_fp4, sc.fp8_log2_ratio);
    p.q.inv8 = 1.0f / p.q.s8;
    p.q.tau = tau; p.q.ratio = sc.fp8_log2_ratio; p.q.r8 = ldexpf(1.0f, sc.fp8_log2_ratio);
    if (packed_acts_out) {
        uint8_t* blob = (uint8_t*)packed_acts_out;
        p.q_codes4 = blob + p.LA.off_codes4; p.q_sf = blob + p.LA.off_sf; p.q_mask = blob + p.LA.off_mask;
        p.q_codes8 = blob + p.LA.off_codes8; p.q_header = reinterpret_cast<fgmp_packed_header*>(blob);
        p.q_arec = blob + p.LA.off_arec;
    }
    p.steps = (uint8_t*)workspace + fgmp_align1k(fgmp_ws_decode(M, N, K));
    const auto launch = [&](auto lp, auto hp) { return (sm == FGMP_SCORE_LP_ERROR ? lp : hp)(p, d, true, (cudaStream_t)cuda_stream); };
    // One or two tokens: the quantizer in every CTA saves 3 us of hand-over, but costs each unit some issue slots.  Us with it, with the shared one and
    // three sets, and with two sets, by units per CTA, 10 % FP8 blocks: two tokens 30.4, 32.2, 31.9 at 48, 36.0, 36.6, 36.4 at 54, 51.1, 50.5, 51.8
    // at 85, 70.1, 66.0, 65.7 at 108, 134, 122, 125 at 217; one token 61.4, 67.0, 66.5 at 108, 88.5, 89.4, 96.4 at 162, 135, 130, 130 at 217.
    // (Without FP8 blocks two tokens take 42.1, 43.6, 43.5 at 85 and 112, 100, 101 at 217; with 20 % 62.8, 64.8, 81.0 and 166, 164, 197.)
    if (M <= 2 && !packed_acts_out) {
        if (d.total > (int64_t)d.grid * (M == 1 ? 200 : 80)) return launch(launch_decode<DEC_FUSED_LP, 3>, launch_decode<DEC_FUSED_HP, 3>);
        if (M == 1) return launch(launch_decode<DEC_OWN1_LP, 3>, launch_decode<DEC_OWN1_HP, 3>);
        return launch(launch_decode<DEC_OWN2_LP, 3>, launch_decode<DEC_OWN2_HP, 3>);
    }
    // Three and four tokens, two sets (twelve and sixteen warps that quantize leave 72 and 64 registers to a thread).  Us own and shared, 10 % FP8 blocks, by units
    // per CTA: three tokens 7.6 and 10.3 at 3.5 (4096 x 4096), 12.3 and 14.1 at 12, 14.6 and 16.1 at 14.6, 18.2 and 18.5 at 21, 18.9 and 19.5 at 24, 21.8
    // and 21.5 at 28, 34.4 and 32.2 at 48; four 7.9 and 10.3 at 3.5, 10.0 and 11.6 at 7, 12.3 and 13.4 at 10.4, 13.4 and 13.9 at 11.6, 15.3 and 15.2 at 13.8.
    // (Without FP8 blocks 15.2 and 16.2 at 24 and 11.4 and 12.2 at 11.6, with 20 % 27.2 and 28.9, 17.4 and 18.2.)  More tokens gain where a CTA has a
    // unit or two alone: eight tokens 6.5 instead of 7.8 at one unit, 8.5 and 8.7 at two, 11.4 and 10.5 at 3.5.
    const int64_t own_units = M == 3 ? 25 : M == 4 ? 12 : 0;
    if (!packed_acts_out && d.total <= own_units * d.grid) {
        if (M == 3) return launch(launch_decode<DEC_OWN3_LP, 2>, launch_decode<DEC_OWN3_HP, 2>);
        return launch(launch_decode<DEC_OWN4_LP, 2>, launch_decode<DEC_OWN4_HP, 2>);
    }
    return launch(launch_decode<DEC_FUSED_LP, 2>, launch_decode<DEC_FUSED_HP, 2>);
}

#ifdef FGMP_TIMELINE
extern "C" int fgmp_debug_timeline(unsigned long long* buffer)
{
    return cudaMemcpyToSymbol(g_timeline, &buffer, sizeof(buffer)) == cudaSuccess ? 0 : -4;
}
#endif

// ------------------------------------------------------------------ allocation-free variant
// Scratch of fgmp_linear_static: one array per GPU that loads the library, held until exit.
static __device__ __align__(256) unsigned char g_static_scratch[FGMP_STATIC_SCRATCH_BYTES];

extern "C" fgmp_status fgmp_linear_static(const void* packed_acts, const void* packed_weights,
                                          void* Y, int y_is_bf16, int64_t ldy, int64_t M, int64_t N, int64_t K,
                                          int32_t* status_out, void* cuda_stream)
{
    if (!packed_acts || !packed_weights || !Y) return FGMP_ERR_INVALID_ARG;
    if (M < 1 || N < 1 || K < 64 || (K % 64) != 0 || ldy < N) return FGMP_ERR_SHAPE;
    if (((uintptr_t)packed_acts & 1023) || ((uintptr_t)packed_weights & 1023) || ((uintptr_t)Y & 15) ||
        ((uintptr_t)status_out & 3)) return FGMP_ERR_SHAPE;
    if (!fgmp_decode_supported(M, N, K)) return FGMP_ERR_SHAPE;
    if (fgmp_ws_decode(M, N, K) > (size_t)FGMP_STATIC_SCRATCH_BYTES) return FGMP_ERR_WORKSPACE;
    fgmp_status st;
    if ((st = fgmp_require_sm100()) != FGMP_OK) return st;

    // The array's name is only a host-side handle; the kernel needs its device address, which
    // differs per GPU.  Looked up once per device, with that device current.
    static void* scratch_of_device[64] = {};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return FGMP_ERR_CUDA;
    void* scratch = nullptr;
    {
        std::lock_guard<std::mutex> lk(g_dec_mu);
        if (!scratch_of_device[dev]) {
            void* ptr = nullptr;
            if (cudaGetSymbolAddress(&ptr, g_static_scratch) != cudaSuccess || !ptr) return FGMP_ERR_CUDA;
            scratch_of_device[dev] = ptr;
        }
        scratch = scratch_of_device[dev];
    }
    cudaStream_t s = (cudaStream_t)cuda_stream;
    // the status word and the tile counters at the start of the scratch are zeroed first; the
    // partial sums behind them are always written before they are read
    st = fgmp_linear_decode(packed_acts, packed_weights, Y, y_is_bf16, ldy, M, N, K, scratch, true, s);
    if (st != FGMP_OK) return st;
    if (status_out && cudaMemcpyAsync(status_out, scratch, 2 * sizeof(int32_t), cudaMemcpyDeviceToDevice, s) != cudaSuccess)
        return FGMP_ERR_CUDA;
    return FGMP_OK;
}

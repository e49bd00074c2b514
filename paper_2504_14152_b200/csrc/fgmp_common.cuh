// Shared device/host helpers of libfgmp: packed-blob layout arithmetic, number-format
// conversions and the pinned single-precision quantization sequence.
#pragma once
#include <cuda_runtime.h>
#include <cuda_bf16.h>
#include <stdint.h>
#include "fgmp.h"

#define FGMP_MAGIC 0x504d4746u
#define FGMP_LAYOUT_VERSION 8
#define FGMP_BS 16

// ---------------------------------------------------------------- blob layout
// A "unit" is one 128-row tile x one chunk of 16 blocks (256 K elements).
//
// Weights (kind 1): header | mask | uptr | records | lists.  A unit's record has a fixed size and
// sits at a fixed place, so that it streams from HBM with one bulk copy whose address needs no
// look-up; the list of its FP8 blocks follows in the lists section, found through uptr.
//   mask      256 B per unit: uint16 per row of the tile, bit j set if the row's block in column j is FP8 (zero
//                       in rows beyond the tensor)
//   REC_W4    16384 B : one 8-byte slot per block, row r of the tile = 128 bytes whose 16-byte pieces are
//                       XOR-swizzled with (r & 7) -- the 128B-swizzled K-major tile tcgen05 reads: the 16
//                       E2M1 codes of an NVFP4 block, or E4M3 codes 0..7 of an FP8 block (which the tensor
//                       core ignores because the block's scale byte is zero); zero in rows beyond the tensor
//   REC_SF     2048 B : E4M3 microscales, 0x00 for FP8 blocks, in the order the scales go to tensor
//                       memory: four 512-byte tiles (one per MMA step of 64 elements), in a tile 16 bytes
//                       per r % 32, there 4 bytes per r / 32, there one byte per block of the step
//   REC_KBSTART 128 B : uint16 x 17 (padded): FP8 blocks of the unit before row 8 i; entry 16 = all
// List of a unit with cnt FP8 blocks, ordered by (row, block column), so that a thread that owns a row has its blocks
// one after the other: one uint32 per block (padded to 16 bytes) -- low half: where the block's slot sits in REC_W4,
// high half: 16 * row + 4 * ((row / 2) % 4) -- then E4M3 codes 8..15 of every block (8 bytes each, padded to 16).
// uptr[u] (uint32, units + 1 entries) = start of unit u's list in 16-byte steps from off_ovf.
//
// Activations (kind 0): header | codes4 | sf | mask | arec | codes8.  codes4 is row-major, sf
// uses 512-byte tiles over all rows, codes8 is a dense plane of which only FP8 blocks are
// written.  arec exists when rows <= 16: one record of AREC_BYTES per chunk for the decode GEMM, 16
// token rows (rows >= M are zero):
//   AREC_A4   2048 B : the E2M1 codes as a 16-row x 128-byte tile, swizzled like REC_W4 (zero in FP8 blocks)
//   AREC_SF    256 B : E4M3 microscales, [token][block column], 0x00 for FP8 blocks
//   AREC_HOT   256 B : not used
//   AREC_AT   8192 B : the value over the tensor scale of every element in fp16 (E2M1 x microscale, or E4M3 x
//                      2^ratio; exact): token octet m / 8 in its own 4096 bytes, there 256 bytes per block
//                      column, there 32 bytes per token -- what a warp reads for one column is contiguous
constexpr uint32_t REC_W4 = 0, REC_SF = 16384, REC_KBSTART = 18432, REC_BYTES = 18560;
constexpr uint32_t AREC_A4 = 0, AREC_SF = 2048, AREC_HOT = 2304, AREC_AT = 2560, AREC_BYTES = 10752;

// byte offset, inside an activation record, of the fp16 values of block column j (0..15) of token row m
__host__ __device__ inline uint32_t fgmp_arec_at_offset(uint32_t m, uint32_t j)
{
    return AREC_AT + ((m >> 3) << 12) + (j << 8) + ((m & 7u) << 5);
}

struct PackedLayout {
    int64_t rows, K, KB, MW;          // KB = K/16 blocks per row, MW = mask words per row
    int64_t tiles, chunks, units;     // 128-row tiles, 16-block K chunks, tiles * chunks
    size_t off_codes4, off_sf, off_mask, off_arec, off_codes8;   // activations (mask: both)
    size_t off_uptr, off_rec, off_ovf;                           // weights
    size_t total;
};

__host__ __device__ inline size_t fgmp_align1k(size_t x) { return (x + 1023) & ~(size_t)1023; }

// list of a unit with cnt FP8 blocks: where the second halves start, and its size in 16-byte steps
__host__ __device__ inline uint32_t fgmp_list_halves_offset(uint32_t cnt) { return (cnt * 4u + 15u) & ~15u; }
__host__ __device__ inline uint32_t fgmp_list_entry(uint32_t row, uint32_t j);
__host__ __device__ inline uint32_t fgmp_list_steps(uint32_t cnt) { return (fgmp_list_halves_offset(cnt) + ((cnt * 8u + 15u) & ~15u)) >> 4; }

// kind 0 = activations, 1 = weights (max_fp8 = room for that many FP8 blocks in the lists section)
__host__ __device__ inline PackedLayout fgmp_layout(int64_t rows, int64_t K, int kind, int64_t max_fp8)
{
    PackedLayout L;
    L.rows = rows; L.K = K; L.KB = K / 16; L.MW = (L.KB + 31) / 32;
    L.tiles = (rows + 127) / 128; L.chunks = (L.KB + 15) / 16; L.units = L.tiles * L.chunks;
    size_t o = 1024;                                   // header section
    L.off_codes4 = L.off_sf = L.off_arec = L.off_codes8 = L.off_uptr = L.off_rec = L.off_ovf = 0;
    if (kind == 0) {
        L.off_codes4 = o;  o = fgmp_align1k(o + (size_t)rows * (size_t)(K / 2));
        L.off_sf = o;      o = fgmp_align1k(o + (size_t)L.tiles * (size_t)(K / 64) * 512);
        L.off_mask = o;    o = fgmp_align1k(o + (size_t)rows * (size_t)L.MW * 4);
        L.off_arec = o;    if (rows <= 16) o = fgmp_align1k(o + (size_t)L.chunks * AREC_BYTES);
        L.off_codes8 = o;  o = fgmp_align1k(o + (size_t)rows * (size_t)K);
    } else {
        L.off_mask = o;    o = fgmp_align1k(o + (size_t)L.units * 256);
        L.off_uptr = o;    o = fgmp_align1k(o + ((size_t)L.units + 1) * 4);
        L.off_rec = o;     o = fgmp_align1k(o + (size_t)L.units * REC_BYTES);
        // 12 bytes per FP8 block, and up to 24 bytes of padding per unit
        L.off_ovf = o;     o = fgmp_align1k(o + (size_t)max_fp8 * 12 + (size_t)L.units * 32);
    }
    L.total = o;
    return L;
}

// byte offset of the microscale of (row r, block kb) inside the sf section of packed activations
__host__ __device__ inline size_t fgmp_sf_offset(int64_t r, int64_t kb, int64_t K)
{
    return ((size_t)(r >> 7) * (size_t)(K >> 6) + (size_t)(kb >> 2)) * 512
         + (size_t)(r & 31) * 16 + (size_t)((r & 127) >> 5) * 4 + (size_t)(kb & 3);
}

// inside a record or the A4 tile of an activation record (r = row in the tile, j = block column in the
// chunk): the 8-byte slot and the scale byte
__host__ __device__ inline uint32_t fgmp_rec_w4_offset(uint32_t r, uint32_t j)
{
    return r * 128u + (((j >> 1) ^ (r & 7u)) << 4) + (j & 1u) * 8u;
}
__host__ __device__ inline uint32_t fgmp_rec_sf_offset(uint32_t r, uint32_t j)
{
    return (j >> 2) * 512u + (r & 31u) * 16u + (r >> 5) * 4u + (j & 3u);
}

// what a unit's list says about its FP8 block (row r of the tile, block column j)
__host__ __device__ inline uint32_t fgmp_list_entry(uint32_t r, uint32_t j)
{
    return fgmp_rec_w4_offset(r, j) | ((r * 16u + (((r >> 1) & 3u) << 2)) << 16);
}

#ifdef __CUDACC__
// Where the FP8 blocks of one unit sit in its list: thread i < 128 brings the 16 mask bits of row i of the tile (0 beyond the last row), further
// threads of the block only come along.
struct UnitScratch {
    uint32_t warp[4];
    uint16_t m16[128], base[128];        // mask bits of a row; FP8 blocks of the unit before it

    // fills the tables, returns the unit's number of FP8 blocks; ends with a __syncthreads()
    __device__ __forceinline__ uint32_t init(uint32_t bits)
    {
        const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
        const uint32_t own = __popc(bits);
        uint32_t incl = own;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) { const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o); if (lane >= o) incl += y; }
        if (lane == 31 && w < 4) warp[w] = incl;
        __syncthreads();
        const uint32_t c0 = warp[0], c1 = warp[1], c2 = warp[2], c3 = warp[3];
        if (threadIdx.x < 128) {
            m16[threadIdx.x] = (uint16_t)bits;
            base[threadIdx.x] = (uint16_t)(incl - own + (w > 0 ? c0 : 0u) + (w > 1 ? c1 : 0u) + (w > 2 ? c2 : 0u));
        }
        __syncthreads();
        return c0 + c1 + c2 + c3;
    }
    // index of block (row, j) among the unit's FP8 blocks; 0xffff if it is NVFP4
    __device__ __forceinline__ uint32_t pos(int row, int j) const
    {
        const uint32_t m = m16[row];
        return (m >> j) & 1u ? base[row] + __popc(m & ((1u << j) - 1u)) : 0xffffu;
    }
};
#endif

// ---------------------------------------------------------------- conversions
#ifdef __CUDACC__

// two floats -> two E2M1 codes in one byte: `lo` in bits 0..3, `hi` in bits 4..7.
// Round to nearest even, saturating to +-6 (cvt.rn.satfinite.e2m1x2.f32).
__device__ __forceinline__ uint32_t f32x2_to_e2m1x2(float lo, float hi)
{
    uint32_t r;
    asm("{\n\t.reg .b8 t;\n\tcvt.rn.satfinite.e2m1x2.f32 t, %1, %2;\n\tcvt.u32.u8 %0, t;\n\t}"
        : "=r"(r) : "f"(hi), "f"(lo));
    return r;
}

// two floats -> two E4M3 codes: `lo` in bits 0..7, `hi` in bits 8..15 (satfinite, RNE).
__device__ __forceinline__ uint32_t f32x2_to_e4m3x2(float lo, float hi)
{
    uint16_t r;
    asm("cvt.rn.satfinite.e4m3x2.f32 %0, %1, %2;" : "=h"(r) : "f"(hi), "f"(lo));
    return r;
}

// byte of two E2M1 codes -> two floats (exact)
__device__ __forceinline__ float2 e2m1x2_to_f32x2(uint32_t byte)
{
    uint32_t h2;
    asm("{\n\t.reg .b8 t;\n\tcvt.u8.u32 t, %1;\n\tcvt.rn.f16x2.e2m1x2 %0, t;\n\t}" : "=r"(h2) : "r"(byte));
    __half2 h = *reinterpret_cast<__half2*>(&h2);
    return __half22float2(h);
}

// two E4M3 codes (low 16 bits) -> two floats (exact)
__device__ __forceinline__ float2 e4m3x2_to_f32x2(uint32_t two)
{
    uint32_t h2;
    uint16_t s = (uint16_t)two;
    asm("cvt.rn.f16x2.e4m3x2 %0, %1;" : "=r"(h2) : "h"(s));
    __half2 h = *reinterpret_cast<__half2*>(&h2);
    return __half22float2(h);
}

__device__ __forceinline__ float e4m3_to_f32(uint32_t code) { return e4m3x2_to_f32x2(code & 0xff).x; }

__device__ __forceinline__ float bf16lo_to_f32(uint32_t pair) { return __uint_as_float(pair << 16); }
__device__ __forceinline__ float bf16hi_to_f32(uint32_t pair) { return __uint_as_float(pair & 0xffff0000u); }

// Weights go into an fp16 GEMM over 2^t: an FP8 block needs no factor then if t is the ratio of its tensor scale to the NVFP4
// one, and fp16 holds every NVFP4 value (up to 2688) over 2^t as long as t >= -4.
__device__ __forceinline__ int fgmp_weight_exponent(const fgmp_packed_header* h) { return max(h->fp8_log2_ratio, -4); }

// ---------------------------------------------------------------- block math
// One block of 16 values in registers.  Every step below is a single IEEE fp32 operation
// (no contraction): this sequence is what makes codes and scores reproducible bit for bit.

// Two fp32 operations per instruction, each rounded as it would be alone.  The quantizers are bound by instruction issue: the search for
// the clipping scale of 4096 x 4096 weights takes 152 us with these, 172 without.
__device__ __forceinline__ uint64_t f32x2_pack(float a, float b) { uint64_t r; asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b)); return r; }
__device__ __forceinline__ float2 f32x2_unpack(uint64_t x) { float2 r; asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(x)); return r; }
__device__ __forceinline__ uint64_t f32x2_mul(uint64_t a, uint64_t b) { uint64_t r; asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b)); return r; }
__device__ __forceinline__ uint64_t f32x2_sub(uint64_t a, uint64_t b)      // a - b as a + (-1) b: one rounding, and no product before it can be drawn in
{
    uint64_t r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(b), "l"(f32x2_pack(-1.f, -1.f)), "l"(a));
    return r;
}

// largest magnitude of 16 values, two at a time (a NaN counts for nothing)
__device__ __forceinline__ float block_amax(const float (&v)[16])
{
    float a = 0.f;
#pragma unroll
    for (int i = 0; i < 16; i += 2) asm("max.abs.f32 %0, %0, %1, %2;" : "+f"(a) : "f"(v[i]), "f"(v[i + 1]));
    return a;
}

// dynamic-max microscale code: E4M3(amax * k6), k6 = 1 / (6 * s4)
__device__ __forceinline__ uint32_t block_dynamic_scale(const float (&v)[16], float k6)
{
    return f32x2_to_e4m3x2(__fmul_rn(block_amax(v), k6), 0.f) & 0x7f;
}

// four pairs of values -> eight E2M1 codes in a word, and the codes' values
__device__ __forceinline__ uint32_t round_e2m1x8(const float (&y)[8], float2 (&q)[4])
{
    uint32_t w, h[4];
    asm("{\n\t.reg .b8 a, b, c, d;\n\t"
        "cvt.rn.satfinite.e2m1x2.f32 a, %6, %5;\n\tcvt.rn.satfinite.e2m1x2.f32 b, %8, %7;\n\t"
        "cvt.rn.satfinite.e2m1x2.f32 c, %10, %9;\n\tcvt.rn.satfinite.e2m1x2.f32 d, %12, %11;\n\t"
        "cvt.rn.f16x2.e2m1x2 %1, a;\n\tcvt.rn.f16x2.e2m1x2 %2, b;\n\tcvt.rn.f16x2.e2m1x2 %3, c;\n\tcvt.rn.f16x2.e2m1x2 %4, d;\n\t"
        "mov.b32 %0, {a, b, c, d};\n\t}"
        : "=r"(w), "=r"(h[0]), "=r"(h[1]), "=r"(h[2]), "=r"(h[3])
        : "f"(y[0]), "f"(y[1]), "f"(y[2]), "f"(y[3]), "f"(y[4]), "f"(y[5]), "f"(y[6]), "f"(y[7]));
#pragma unroll
    for (int i = 0; i < 4; ++i) q[i] = __half22float2(*reinterpret_cast<__half2*>(&h[i]));
    return w;
}

// NVFP4 rounding under microscale code `sc`; dq receives the dequantized values
__device__ __forceinline__ void block_nvfp4(const float (&v)[16], uint32_t sc, float s4,
                                            uint32_t (&c4)[2], float (&dq)[16])
{
    const float d = __fmul_rn(e4m3_to_f32(sc), s4);
    const float inv = (d == 0.f) ? 0.f : __fdiv_rn(1.0f, d);
    const uint64_t d2 = f32x2_pack(d, d), inv2 = f32x2_pack(inv, inv);
#pragma unroll
    for (int w = 0; w < 2; ++w) {
        // (inv == 0, a zero scale: only the signs stay, as -0.0 * 0 = -0.0)
        float y[8];
        float2 q[4];
#pragma unroll
        for (int i = 0; i < 8; i += 2) { const float2 t = f32x2_unpack(f32x2_mul(f32x2_pack(v[8 * w + i], v[8 * w + i + 1]), inv2)); y[i] = t.x; y[i + 1] = t.y; }
        c4[w] = round_e2m1x8(y, q);
#pragma unroll
        for (int i = 0; i < 4; ++i) { const float2 t = f32x2_unpack(f32x2_mul(f32x2_pack(q[i].x, q[i].y), d2)); dq[8 * w + 2 * i] = t.x; dq[8 * w + 2 * i + 1] = t.y; }
    }
}

// FP8 rounding of the block: 16 E4M3 codes in 4 words, dq8 = dequantized values
__device__ __forceinline__ void block_fp8(const float (&v)[16], float inv8, float s8,
                                          uint32_t (&c8)[4], float (&dq)[16])
{
    const uint64_t s2 = f32x2_pack(s8, s8), inv2 = f32x2_pack(inv8, inv8);
#pragma unroll
    for (int i = 0; i < 16; i += 4) {
        const float2 y = f32x2_unpack(f32x2_mul(f32x2_pack(v[i], v[i + 1]), inv2)), z = f32x2_unpack(f32x2_mul(f32x2_pack(v[i + 2], v[i + 3]), inv2));
        const uint32_t lo = f32x2_to_e4m3x2(y.x, y.y), hi = f32x2_to_e4m3x2(z.x, z.y);
        float2 a = e4m3x2_to_f32x2(lo), b = e4m3x2_to_f32x2(hi);
        a = f32x2_unpack(f32x2_mul(f32x2_pack(a.x, a.y), s2)); b = f32x2_unpack(f32x2_mul(f32x2_pack(b.x, b.y), s2));
        dq[i] = a.x; dq[i + 1] = a.y; dq[i + 2] = b.x; dq[i + 3] = b.y;
        c8[i >> 2] = lo | (hi << 16);
    }
}

// sum_i (f_i * e_i) * e_i, in element order
__device__ __forceinline__ float weighted_sq_sum(const float (&a)[16], const float (&b)[16],
                                                 const float (&f)[16])
{
    float s = 0.f;
#pragma unroll
    for (int i = 0; i < 16; i += 2) {
        const uint64_t e = f32x2_sub(f32x2_pack(a[i], a[i + 1]), f32x2_pack(b[i], b[i + 1]));
        const float2 t = f32x2_unpack(f32x2_mul(f32x2_mul(f32x2_pack(f[i], f[i + 1]), e), e));
        s = __fadd_rn(__fadd_rn(s, t.x), t.y);
    }
    return s;
}

// 16 bf16 (two 128-bit words) -> 16 floats
__device__ __forceinline__ void unpack_bf16x16(const uint4& a, const uint4& b, float (&v)[16])
{
    const uint32_t w[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
#pragma unroll
    for (int i = 0; i < 8; ++i) { v[2 * i] = bf16lo_to_f32(w[i]); v[2 * i + 1] = bf16hi_to_f32(w[i]); }
}

#endif  // __CUDACC__

// fgmp_linear for prefill-sized batches whose operands hold no FP8 block at all (threshold +inf for the
// activations, FP8 fraction 0 for the weights: the all-NVFP4 end of the method's range): every block pair is
// an FP4 x FP4 product (Section 4.1), and the GEMM runs on tcgen05.mma kind::mxf4nvf4 straight from the
// packed operands -- no expansion pass, a quarter of the operand bytes of the bf16 container, four times its
// MMA rate.
//
// The packed layouts were made for this: a weight record's code tile is the 128-byte-swizzled K-major tile
// of 128 rows x 256 elements that the tensor core reads, its scale bytes are in tensor-memory order; the
// activations' code plane is row-major (a TMA tile load swizzles it on the way in) and their scale section
// consists of 512-byte tiles in the same tensor-memory order.
//
// One CTA per SM, persistent over output tiles; a stage holds one K chunk of 256 elements.  A single CTA makes 128 (tokens) x 256
// (weight rows) and loads 54 KiB per stage; a CTA pair makes 256 x 256, each CTA loading its own tokens, one of the two weight tiles
// and all scales, 38 KiB per stage.  Warp 0 = producer (TMA / bulk copies), warp 1 = MMA issuer and owner of the tensor memory, warps
// 2-5 = block scales into tensor memory (one lane quadrant each), warps 6-13 = epilogue (a lane quadrant and half of the columns each).
// Every wait is bounded.
//
// Single CTAs are bound by the copies from L2 (18 TB/s over the machine without the products), pairs by the length of a stage's cycle
// (tensor pipe 51 % of the active cycles, L2 39 % of its peak).  2048 x 13824 x 5120, fp32 output: 88.6 us when one
// tile's stores ended before the next tile's products began and one of 32 lanes issued the products, 78.8 us with the accumulator
// drained into registers first and an elected thread, 71.5 us on pairs (bf16 output: 79.9, 70.4, 63.0).  With Y leaving as TMA tiles a
// tile takes 14200 clocks instead of 16400, of which 10240 are products; the clock falls under that load, and a call with its quantizer takes 2 to 3 %
// less.
#include <cuda.h>
#include <mutex>
#include "fgmp_common.cuh"
#include "fgmp_host.h"
#include "fgmp_ptx.cuh"

namespace {

constexpr int G4_THREADS = 448;
// a stage: activation codes, weight codes (single CTA: two tiles; of a pair: this CTA's tile), scales of both weight tiles and of the
// activations
template <bool PAIR> struct G4 {
    static constexpr int STAGES = PAIR ? 5 : 4;
    static constexpr uint32_t A4 = 0, B0 = 16384, B1 = 32768, SFB = PAIR ? 32768 : 49152, SFA = SFB + 4096, STAGE_BYTES = SFA + 2048;
    static constexpr uint32_t OUT = STAGES * STAGE_BYTES, OUT_BYTES = PAIR ? 8 * TILE_STORE_BYTES : 0;     // tiles of Y on their way out
    static constexpr size_t SMEM = (size_t)OUT + OUT_BYTES + 1024 /*alignment*/ + 512 /*barriers*/;
    static constexpr int64_t TM = PAIR ? 256 : 128;                       // tokens of an output tile
    static_assert(SMEM <= 232448, "shared memory of one CTA");
    static_assert(256 + 48 * STAGES <= 512, "tensor memory columns");
};
constexpr uint32_t G4_SF_COL0 = 256;            // tensor memory: 256 accumulator columns, then 48 scale columns per stage
constexpr uint32_t G4_TMEM_COLS = 512;

// kind::mxf4nvf4, E2M1 x E2M1, UE4M3 scales, K-major operands, dense K = 64; M = 128, or 256 over a pair; N = 256 or 128
constexpr uint32_t G4_IDESC_BASE = (1u << 7) | (1u << 10);
constexpr uint32_t G4_IDESC_N256 = G4_IDESC_BASE | ((uint32_t)(128 >> 4) << 24) | ((uint32_t)(256 >> 3) << 17);
constexpr uint32_t G4_IDESC_N128 = G4_IDESC_BASE | ((uint32_t)(128 >> 4) << 24) | ((uint32_t)(128 >> 3) << 17);
constexpr uint32_t G4_IDESC_PAIR = G4_IDESC_BASE | ((uint32_t)(256 >> 4) << 24) | ((uint32_t)(256 >> 3) << 17);
constexpr uint32_t G4_SW128_LO = 1u << 16, G4_SW128_HI = (1024u >> 4) | (1u << 14) | (2u << 29);

__device__ __forceinline__ uint64_t g4_desc(uint32_t lo)
{
    uint64_t d;
    asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "r"(lo), "r"(G4_SW128_HI));
    return d;
}

__device__ __forceinline__ void st_global_256(void* dst, uint32_t a, uint32_t b, uint32_t c, uint32_t d, uint32_t e, uint32_t f, uint32_t g, uint32_t h)
{
    asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};"
                 ::"l"(dst), "r"(a), "r"(b), "r"(c), "r"(d), "r"(e), "r"(f), "r"(g), "r"(h) : "memory");
}

struct Gemm4Params {
    const uint8_t* ablob; const uint8_t* wblob;
    PackedLayout LA, LW;
    void* Y; int64_t ldy; int y_is_bf16;
    int64_t M, N, K;
    int64_t tile_cols;                    // columns of Y that leave as TMA tiles, see fgmp_tile_cols
    int first;                            // the first kernel of the call: the status starts here
    int* status;                          // [0..1] device-side status, [2] 1 = this kernel has produced Y
};

// 32 sums of a row, times alpha, to y; `left` columns of the row remain
__device__ __forceinline__ void g4_store(__nv_bfloat16* y, const uint32_t (&r)[32], float alpha, int64_t left, bool wide)
{
    if (left < 32) {
#pragma unroll
        for (int j = 0; j < 32; ++j)
            if (j < left) y[j] = __float2bfloat16_rn(__uint_as_float(r[j]) * alpha);
        return;
    }
    uint32_t o[16];
#pragma unroll
    for (int u = 0; u < 16; ++u) {
        const __nv_bfloat162 h = __floats2bfloat162_rn(__uint_as_float(r[2 * u]) * alpha, __uint_as_float(r[2 * u + 1]) * alpha);
        o[u] = *reinterpret_cast<const uint32_t*>(&h);
    }
    if (wide) {
#pragma unroll
        for (int j = 0; j < 16; j += 8) st_global_256(y + 2 * j, o[j], o[j + 1], o[j + 2], o[j + 3], o[j + 4], o[j + 5], o[j + 6], o[j + 7]);
    } else if (((uintptr_t)y & 15) == 0) {
#pragma unroll
        for (int j = 0; j < 16; j += 4) *reinterpret_cast<uint4*>(y + 2 * j) = make_uint4(o[j], o[j + 1], o[j + 2], o[j + 3]);
    } else {
#pragma unroll
        for (int j = 0; j < 16; ++j) {
            const __nv_bfloat162 h = *reinterpret_cast<const __nv_bfloat162*>(&o[j]);
            y[2 * j] = h.x; y[2 * j + 1] = h.y;
        }
    }
}
__device__ __forceinline__ void g4_store(float* y, const uint32_t (&r)[32], float alpha, int64_t left, bool wide)
{
    float o[32];
#pragma unroll
    for (int j = 0; j < 32; ++j) o[j] = __uint_as_float(r[j]) * alpha;
    if (left >= 32 && wide) {
#pragma unroll
        for (int j = 0; j < 32; j += 8)
            st_global_256(y + j, __float_as_uint(o[j]), __float_as_uint(o[j + 1]), __float_as_uint(o[j + 2]), __float_as_uint(o[j + 3]),
                          __float_as_uint(o[j + 4]), __float_as_uint(o[j + 5]), __float_as_uint(o[j + 6]), __float_as_uint(o[j + 7]));
    } else if (left >= 32 && ((uintptr_t)y & 15) == 0) {
#pragma unroll
        for (int j = 0; j < 32; j += 4) *reinterpret_cast<float4*>(y + j) = make_float4(o[j], o[j + 1], o[j + 2], o[j + 3]);
    } else {
#pragma unroll
        for (int j = 0; j < 32; ++j)
            if (j < left) y[j] = o[j];
    }
}

__device__ __forceinline__ void g4_store(const Gemm4Params& p, int64_t at, const uint32_t (&r)[32], float alpha, int64_t left, bool wide)
{
    if (left <= 0) return;
    if (p.y_is_bf16) g4_store(reinterpret_cast<__nv_bfloat16*>(p.Y) + at, r, alpha, left, wide);
    else g4_store(reinterpret_cast<float*>(p.Y) + at, r, alpha, left, wide);
}

__device__ __forceinline__ bool g4_applicable(const Gemm4Params& p)
{
    const fgmp_packed_header* ha = reinterpret_cast<const fgmp_packed_header*>(p.ablob);
    const fgmp_packed_header* hw = reinterpret_cast<const fgmp_packed_header*>(p.wblob);
    return ha->magic == FGMP_MAGIC && ha->version == FGMP_LAYOUT_VERSION && ha->rows == p.M && ha->K == p.K && ha->kind == 0u && ha->n_fp8 == 0 &&
           hw->magic == FGMP_MAGIC && hw->version == FGMP_LAYOUT_VERSION && hw->rows == p.N && hw->K == p.K && hw->kind == 1u && hw->error == 0 &&
           hw->n_fp8 == 0;
}

template <bool PAIR>
__global__ void __launch_bounds__(G4_THREADS, 1)
gemm_nvfp4_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmW, const __grid_constant__ CUtensorMap tmY, Gemm4Params p)
{
    using C = G4<PAIR>;
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    // operands with FP8 blocks (or headers that do not match the call) are left to the general path
    const bool applies = g4_applicable(p);
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        if (p.first) { p.status[0] = 0; p.status[1] = 0; }
        if (applies) p.status[2] = 1;
    }
    if (!applies) return;

    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
    constexpr int S = C::STAGES;
    uint64_t* bars = reinterpret_cast<uint64_t*>(smem + C::OUT + C::OUT_BYTES);
    // bars: [0,S) full, [S,2S) empty, [2S,3S) scales in tensor memory, [3S,4S) scales loaded, then acc_full, acc_empty.  Of a pair, the
    // leader's "full" counts the codes of both CTAs, since its thread multiplies both; the scales are each CTA's own matter until they are in
    // tensor memory, and "scales loaded" counts them.  A single CTA has its scales counted by "full".
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 4 * S + 2);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
    const int warp = warp_index(), lane = threadIdx.x & 31;
    const uint32_t rank = PAIR ? cluster_ctarank() : 0u;
    const uint32_t full0 = smem_u32(bars), empty0 = full0 + 8 * S, sfr0 = empty0 + 8 * S, sfl0 = PAIR ? sfr0 + 8 * S : full0, accf = sfr0 + 16 * S, acce = accf + 8;

    if (threadIdx.x == 0) {
        for (int s = 0; s < S; ++s) { mbar_init(full0 + 8 * s, 1); mbar_init(empty0 + 8 * s, 1); mbar_init(sfr0 + 8 * s, PAIR ? 8 : 4); if (PAIR) mbar_init(sfl0 + 8 * s, 1); }
        mbar_init(accf, 1); mbar_init(acce, PAIR ? 16 : 8);
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) { if (PAIR) tmem_alloc_pair(smem_u32(tmem_slot), G4_TMEM_COLS); else tmem_alloc(smem_u32(tmem_slot), G4_TMEM_COLS); }
    tc_fence_before();
    __syncthreads();
    if (PAIR) cluster_sync();                           // the other CTA's barriers exist before anything signals them
    tc_fence_after();
    constexpr uint32_t tmem_base = TMEM_ALL;
    static_assert(REC_W4 == 0 && REC_BYTES % 128 == 0, "records as rows of 128 bytes");

    const int64_t tiles_m = (p.M + C::TM - 1) / C::TM, wtiles = p.LW.tiles, tiles_n = (wtiles + 1) / 2;
    const int64_t num_tiles = tiles_m * tiles_n;
    const int64_t first = PAIR ? blockIdx.x >> 1 : blockIdx.x, step = PAIR ? gridDim.x >> 1 : gridDim.x;
    const int64_t chunks = p.LW.chunks;
    const int64_t ksteps_total = p.K / 64;
    const uint8_t* recs = p.wblob + p.LW.off_rec;
    const uint8_t* asf = p.ablob + p.LA.off_sf;

    if (warp == 0) {
        // ------------------------------------------------------------ producer
        if (elect_one()) {
            int stage = 0; uint32_t phase = 0; bool ok = true;
            for (int64_t t = first; t < num_tiles && ok; t += step) {
                const int64_t tm = t % tiles_m, tn = t / tiles_m;             // token tiles fastest: CTAs that run together share weights
                const int64_t m0 = tm * C::TM + 128 * rank;
                const bool two = 2 * tn + 1 < wtiles, rows = m0 < p.M;
                const uint8_t* r0 = recs + (size_t)(2 * tn * chunks) * REC_BYTES;
                const uint8_t* r1 = r0 + (size_t)chunks * REC_BYTES;
                const uint8_t* sfa = asf + (size_t)(m0 >> 7) * (size_t)ksteps_total * 512;
                // what the two CTAs of a pair load: the leader's rows are always there
                const uint32_t pair_codes = 16384u * (1u + (m0 + 128 < p.M ? 1u : 0u) + (two ? 2u : 1u));
                const int32_t w_row = (int32_t)((2 * tn + rank) * chunks * (REC_BYTES / 128));      // a record is 145 rows of 128 bytes
                for (int64_t c = 0; c < chunks; ++c, r0 += REC_BYTES, r1 += REC_BYTES, sfa += 2048) {
                    if (!(ok = mbar_wait(empty0 + 8 * stage, phase ^ 1, abort_flag, p.status, 1))) break;
                    const uint32_t ks = (uint32_t)min((int64_t)4, ksteps_total - 4 * c);
                    const uint32_t fb = full0 + 8 * stage, sb = sfl0 + 8 * stage;
                    const uint32_t dst = smem_u32(smem + (size_t)stage * C::STAGE_BYTES);
                    const uint32_t scales = (rows ? ks * 512u : 0u) + (two ? 4096u : 2048u);
                    if (PAIR) {
                        if (rank == 0) mbar_expect_tx(fb, pair_codes);
                        mbar_expect_tx(sb, scales);
                        const uint32_t leader = cluster_map(fb, 0);
                        if (rows) tma_load_2d_pair(dst + C::A4, &tmA, (int32_t)(c * 128), (int32_t)m0, leader);
                        if (rank == 0 || two) tma_load_2d_pair(dst + C::B0, &tmW, 0, w_row + (int32_t)c * (int32_t)(REC_BYTES / 128), leader);
                    } else {
                        mbar_expect_tx(fb, (rows ? 16384u : 0u) + (two ? 2u : 1u) * 16384u + scales);
                        if (rows) tma_load_2d(dst + C::A4, &tmA, (int32_t)(c * 128), (int32_t)m0, fb);
                        bulk_load(dst + C::B0, r0 + REC_W4, 16384, fb);
                        if (two) bulk_load(dst + C::B1, r1 + REC_W4, 16384, fb);
                    }
                    if (rows) bulk_load(dst + C::SFA, sfa, ks * 512u, sb);
                    bulk_load(dst + C::SFB, r0 + REC_SF, 2048, sb);
                    if (two) bulk_load(dst + C::SFB + 2048, r1 + REC_SF, 2048, sb);
                    if (++stage == S) { stage = 0; phase ^= 1; }
                }
            }
        }
    } else if (warp == 1) {
        // ------------------------------------------------------------ MMA issuer: one thread (of the leader), addresses in uniform registers
        if (rank == 0 && elect_one()) {
            const uint32_t smem0 = smem_u32(smem);
            int stage = 0; uint32_t phase = 0; bool ok = true;
            int64_t it = 0;
            for (int64_t t = first; t < num_tiles && ok; t += step, ++it) {
                const int64_t tn = t / tiles_m;
                const uint32_t idesc = PAIR ? G4_IDESC_PAIR : (2 * tn + 1 < wtiles) ? G4_IDESC_N256 : G4_IDESC_N128;
                if (!(ok = mbar_wait(acce, (uint32_t)(it & 1) ^ 1u, abort_flag, p.status, 2))) break;    // the epilogue has drained the accumulator
                tc_fence_after();
                uint32_t accum = 0;
                for (int64_t c = 0; c < chunks; ++c) {
                    // (of a single CTA, the scale warps arrive behind the stage's loads: theirs is the only signal to wait for)
                    if (!(ok = mbar_wait(sfr0 + 8 * stage, phase, abort_flag, p.status, 3))) break;
                    if (PAIR && !(ok = mbar_wait(full0 + 8 * stage, phase, abort_flag, p.status, 8))) break;
                    tc_fence_after();
                    const uint32_t ks = (uint32_t)min((int64_t)4, ksteps_total - 4 * c);
                    const uint32_t sb = smem0 + (uint32_t)stage * C::STAGE_BYTES;
                    const uint32_t sf_t = tmem_base + G4_SF_COL0 + (uint32_t)stage * 48;     // [0,16) tokens, [16,48) weight rows
                    const uint32_t a_lo = ((sb + C::A4) >> 4) | G4_SW128_LO, b_lo = ((sb + C::B0) >> 4) | G4_SW128_LO;
                    for (uint32_t j = 0; j < ks; ++j) {
                        if (PAIR) umma_nvf4_pair(tmem_base, g4_desc(a_lo + 2 * j), g4_desc(b_lo + 2 * j), idesc, sf_t + 4 * j, sf_t + 16 + 8 * j, accum);
                        else umma_nvf4(tmem_base, g4_desc(a_lo + 2 * j), g4_desc(b_lo + 2 * j), idesc, sf_t + 4 * j, sf_t + 16 + 8 * j, accum);
                        accum = 1;
                    }
                    if (PAIR) umma_commit_pair(empty0 + 8 * stage, 3); else umma_commit(empty0 + 8 * stage);
                    if (++stage == S) { stage = 0; phase ^= 1; }
                }
                if (ok) { if (PAIR) umma_commit_pair(accf, 3); else umma_commit(accf); }
            }
        }
    } else if (warp < 6) {
        // ------------------------------------------------------------ block scales into tensor memory, lane quadrant warp % 4
        // Lane i holds, for MMA step j, the scale bytes of operand rows i, 32+i, ... : one column per 32 rows, i.e.
        // 16 bytes of a 512-byte scale tile per 128 rows.  Of a pair, each CTA holds its own rows' activation scales and all weight scales.
        const uint32_t ready0 = PAIR ? cluster_map(sfr0, 0) : sfr0;
        int stage = 0; uint32_t phase = 0; bool ok = true;
        for (int64_t t = first; t < num_tiles && ok; t += step) {
            const int64_t tm = t % tiles_m, tn = t / tiles_m;
            const bool two = 2 * tn + 1 < wtiles, rows = tm * C::TM + 128 * rank < p.M;
            for (int64_t c = 0; c < chunks; ++c) {
                if (!(ok = mbar_wait_warp(sfl0 + 8 * stage, phase, abort_flag, p.status, 4))) break;
                const uint32_t ks = rows ? (uint32_t)min((int64_t)4, ksteps_total - 4 * c) : 0u;
                const uint8_t* sb = smem + (size_t)stage * C::STAGE_BYTES;
                const uint32_t sf_t = tmem_base + ((uint32_t)((warp & 3) * 32) << 16) + G4_SF_COL0 + (uint32_t)stage * 48;
                uint32_t r[16];
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    uint4 x = make_uint4(0u, 0u, 0u, 0u);
                    if ((uint32_t)j < ks) x = *reinterpret_cast<const uint4*>(sb + C::SFA + 512 * j + lane * 16);
                    r[4 * j] = x.x; r[4 * j + 1] = x.y; r[4 * j + 2] = x.z; r[4 * j + 3] = x.w;
                }
                tmem_st16(sf_t, r);
#pragma unroll
                for (int half = 0; half < 2; ++half) {              // MMA steps 2 half, 2 half + 1: eight columns each
#pragma unroll
                    for (int jj = 0; jj < 2; ++jj) {
                        const int j = 2 * half + jj;
                        const uint4 x = *reinterpret_cast<const uint4*>(sb + C::SFB + 512 * j + lane * 16);
                        uint4 y = make_uint4(0u, 0u, 0u, 0u);
                        if (two) y = *reinterpret_cast<const uint4*>(sb + C::SFB + 2048 + 512 * j + lane * 16);
                        r[8 * jj] = x.x; r[8 * jj + 1] = x.y; r[8 * jj + 2] = x.z; r[8 * jj + 3] = x.w;
                        r[8 * jj + 4] = y.x; r[8 * jj + 5] = y.y; r[8 * jj + 6] = y.z; r[8 * jj + 7] = y.w;
                    }
                    tmem_st16(sf_t + 16 + 16 * half, r);
                }
                tmem_wait_st();
                tc_fence_before();
                __syncwarp();
                if (lane == 0) { if (PAIR) mbar_arrive_cluster_tmem(ready0 + 8 * stage); else mbar_arrive(ready0 + 8 * stage); }
                if (++stage == S) { stage = 0; phase ^= 1; }
            }
        }
    } else {
        // ------------------------------------------------------------ epilogue: lane quadrant warp % 4, half of the columns, a token row
        // per thread.  What is left of the half goes to registers before the second store, so that the next tile's products
        // start while this one is stored (all of it before the first store does not fit the registers of 448 threads).
        const int q = warp & 3, half = (warp - 6) >> 2;
        const fgmp_packed_header* ha = reinterpret_cast<const fgmp_packed_header*>(p.ablob);
        const fgmp_packed_header* hw = reinterpret_cast<const fgmp_packed_header*>(p.wblob);
        const float alpha = __fmul_rn(ha->scale_fp4, hw->scale_fp4);
        // Y and its row pitch 32-byte aligned: a lane that stores its row writes whole sectors
        const bool wide = ((uintptr_t)p.Y & 31) == 0 && ((p.ldy * (p.y_is_bf16 ? 2 : 4)) % 32) == 0;
        const uint32_t buf = smem_u32(smem + C::OUT) + (uint32_t)(warp - 6) * TILE_STORE_BYTES;
        const uint32_t drained = PAIR ? cluster_map(acce, 0) : acce, src = tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)(half * 128);
        bool ok = true;
        int64_t it = 0;
        for (int64_t t = first; t < num_tiles && ok; t += step, ++it) {
            const int64_t tm = t % tiles_m, tn = t / tiles_m;
            if (!(ok = mbar_wait_warp(accf, (uint32_t)(it & 1), abort_flag, p.status, 5))) break;
            tc_fence_after();
            const int64_t row0 = tm * C::TM + 128 * rank + q * 32, n0 = tn * 256 + half * 128;
            uint32_t r[3][32];
#pragma unroll
            for (int c = 0; c < 3; ++c) tmem_ld32(src + (uint32_t)(c * 32), r[c]);
            // 32 columns out; in bf16 a tile of Y has 64
            auto out = [&](const uint32_t (&v)[32], int c) {
                const int64_t n = n0 + 32 * c;
                if (!PAIR || n - 32 * (p.y_is_bf16 ? c & 1 : 0) >= p.tile_cols) {
                    g4_store(p, (row0 + lane) * p.ldy + n, v, alpha, row0 + lane < p.M ? p.N - n : 0, wide);
                    return;
                }
                if (p.y_is_bf16) {
                    if ((c & 1) == 0) tile_wait(lane);
                    tile_put_bf16(buf, lane, c & 1, v, alpha);
                    if ((c & 1) && row0 < p.M) tile_store(&tmY, buf, lane, (int32_t)(n - 32), (int32_t)row0);
                } else {
                    tile_wait(lane);
                    tile_put_f32(buf, lane, v, alpha);
                    if (row0 < p.M) tile_store(&tmY, buf, lane, (int32_t)n, (int32_t)row0);
                }
            };
            out(r[0], 0);
            __syncwarp();
            tmem_ld32(src + 96, r[0]);
            tc_fence_before();
            __syncwarp();
            if (lane == 0) { if (PAIR) mbar_arrive_cluster_tmem(drained); else mbar_arrive(drained); }
#pragma unroll
            for (int c = 1; c < 4; ++c) out(r[c % 3], c);
        }
        if (PAIR) tile_drain(lane);
    }

    __syncthreads();
    if (*abort_flag) {
        const unsigned long long t0 = globaltimer_ns();
        while (globaltimer_ns() - t0 < 2000000ull) __nanosleep(1000);
        __syncthreads();
    }
    if (PAIR) cluster_sync();                           // neither CTA leaves while the other may still signal it
    if (warp == 1) {
        tc_fence_after();
        if (PAIR) tmem_dealloc_pair(tmem_base, G4_TMEM_COLS); else tmem_dealloc(tmem_base, G4_TMEM_COLS);
    }
}

std::mutex g4_mu;
int g4_pairs[64] = {};                 // CTA pairs that run at once

}  // namespace

// Launches the all-NVFP4 GEMM; it decides on the device (from the two headers) whether it applies, as the general path's kernels
// do, and says so in status[2].
fgmp_status fgmp_launch_gemm_nvfp4(const void* packed_acts, const void* packed_weights, void* Y, int y_is_bf16, int64_t ldy,
                                   int64_t M, int64_t N, int64_t K, int* status, bool first, cudaStream_t s)
{
    int dev = 0, pairs = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return FGMP_ERR_CUDA;
    {
        std::lock_guard<std::mutex> lk(g4_mu);
        if (!g4_pairs[dev]) {
            cudaLaunchConfig_t qc = {};
            cudaLaunchAttribute qa[1];
            qa[0].id = cudaLaunchAttributeClusterDimension;
            qa[0].val.clusterDim.x = 2; qa[0].val.clusterDim.y = 1; qa[0].val.clusterDim.z = 1;
            qc.gridDim = dim3(2u * (unsigned)fgmp_sm_count()); qc.blockDim = dim3(G4_THREADS); qc.dynamicSmemBytes = G4<true>::SMEM;
            qc.attrs = qa; qc.numAttrs = 1;
            int n = 0;
            if (cudaFuncSetAttribute(gemm_nvfp4_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)G4<false>::SMEM) != cudaSuccess ||
                cudaFuncSetAttribute(gemm_nvfp4_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)G4<true>::SMEM) != cudaSuccess ||
                cudaOccupancyMaxActiveClusters(&n, gemm_nvfp4_kernel<true>, &qc) != cudaSuccess || n < 1) return FGMP_ERR_CUDA;
            g4_pairs[dev] = n;
        }
        pairs = g4_pairs[dev];
    }
    Gemm4Params p;
    p.ablob = (const uint8_t*)packed_acts; p.wblob = (const uint8_t*)packed_weights;
    p.LA = fgmp_layout(M, K, 0, 0); p.LW = fgmp_layout(N, K, 1, 0);
    p.Y = Y; p.ldy = ldy; p.y_is_bf16 = y_is_bf16; p.M = M; p.N = N; p.K = K; p.status = status; p.first = first ? 1 : 0;
    // the activations' code plane: bytes [M, K/2] row-major, boxes of 128 rows x 128 bytes, swizzled on the way in; pairs: the weights'
    // records as rows of 128 bytes, boxes of a tile's 128 rows (swizzled already), whose loads may be counted in the leader
    CUtensorMap tmA, tmW;
    if (!fgmp_map_2d(&tmA, CU_TENSOR_MAP_DATA_TYPE_UINT8, p.ablob + p.LA.off_codes4, M, K / 2, K / 2, 128, 128) ||
        !fgmp_map_2d(&tmW, CU_TENSOR_MAP_DATA_TYPE_UINT8, p.wblob + p.LW.off_rec, p.LW.units * (REC_BYTES / 128), 128, 128, 128, 128, false))
        return FGMP_ERR_CUDA;
    const int64_t cols = (p.LW.tiles + 1) / 2, tiles = ((M + 127) / 128) * cols, tiles2 = ((M + 255) / 256) * cols;
    const int sms = fgmp_sm_count();
    // pairs where the tiles take more than one round of the machine (2048 x 13824 x 5120: 63 us, 70 on single CTAs; 777 x 11008 x 4096: 28.2,
    // 30.4) and the larger tiles do not take a round more; within one round the smaller tile's shorter start wins (384 x 5120 x 5120: 13.8 us,
    // 14.5 on pairs)
    const bool pair = tiles > sms && (tiles2 + pairs - 1) / pairs <= (tiles + sms - 1) / sms;
    CUtensorMap tmY = tmA;
    p.tile_cols = pair ? fgmp_tile_cols(N, ldy, y_is_bf16) : 0;
    if (p.tile_cols && !fgmp_map_y(&tmY, Y, y_is_bf16, ldy, M, p.tile_cols)) return FGMP_ERR_CUDA;
    const int grid = pair ? 2 * (int)(tiles2 < pairs ? tiles2 : pairs) : (int)(tiles < sms ? tiles : sms);
    // a programmatic dependent: where it does not apply it is gone when the kernel before it ends
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = 2; attr[1].val.clusterDim.y = 1; attr[1].val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)grid); cfg.blockDim = dim3(G4_THREADS); cfg.stream = s;
    cfg.dynamicSmemBytes = pair ? G4<true>::SMEM : G4<false>::SMEM;
    cfg.attrs = attr; cfg.numAttrs = pair ? 2 : 1;
    if (pair) FGMP_LAUNCH(FGMP_K_GEMM_NVFP4, s, cudaLaunchKernelEx(&cfg, gemm_nvfp4_kernel<true>, tmA, tmW, tmY, p));
    else FGMP_LAUNCH(FGMP_K_GEMM_NVFP4, s, cudaLaunchKernelEx(&cfg, gemm_nvfp4_kernel<false>, tmA, tmW, tmY, p));
    return fgmp_launch_status();
}

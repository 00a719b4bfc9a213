// A depthwise 3x3 convolution and the pointwise (1x1) convolution behind it in one kernel, both on the tensor cores: the
// depthwise-separable block of the MobileNets.  Eq. 6 is applied per layer, so running two layers in one launch changes no
// result; the 8-bit tensor between them stays in shared memory (unless the caller asks for a copy).
//
// A depthwise convolution is a dense one whose weight matrix, per filter tap, is diagonal.  Multiplying with 32 x 32 diagonal
// blocks (N = 32, K = 32) wastes 31 of 32 multiplications and still wins: an instruction takes 40 cycles for 128 pixels x 32
// channels x one tap, where the packed dot products of the CUDA-core kernel need 13 issue slots per output and pay for
// transposing, addressing and converting; here the tensor core does all but the conversion.
//
//   A producer             stride 1: per tile and 128-channel slab ONE load of the padded input rows behind `win_r` whole output rows;
//                          a tile's rows are positions of the padded image (W + 2 per row, the last two of each discarded), and
//                          filter tap (r, s) is the same shared-memory tile read r (W + 2) + s rows further down.  Stride 2: per slab
//                          and tap one im2col load of 128 output pixels (nine times the bytes and, what counts, nine latencies)
//   diagonal writer        from a compact copy of the depthwise weights in shared memory writes the 128 diagonal bytes of a tap
//                          into blocks whose other bytes were zeroed once
//   issuer 1               per slab 9 taps x 4 blocks of 32 channels into one of two 128-column accumulators
//   W producer             pointwise weight tiles (bn2 rows x 128 bytes), once per CTA where they all fit, else per tile
//   issuer 2               for every bn2-column part of the output: the slabs of the tile times the weight tiles
//   16 epilogue warps      slab: accumulator 1 -> bias, rounding shift, clip -> staged slab (128 rows x 128 bytes, the swizzled K-major
//                          layout GEMM 2 reads); part: accumulator 2 -> bias, shortcut, shift, clip -> output ring
//   mover / fetcher        TMA stores of finished output parts, TMA loads of shortcut parts into the ring
//
// Where the pointwise layer has more output channels than an accumulator holds, its parts follow one another over the same
// staged slabs, which then all have to be there at once (`slots` >= slabs).  Every wait is bounded (see f8_tc_ptx.cuh).
// Bound: the tensor pipe (40 cycles x 36 per slab, bn2 / 2 per 32 bytes of K of a part).  Measured with the rule of f8_dwpw_wanted
// against two launches, the depthwise one on f8_dw_tc_kernel where a network prefers that: MobileNet V1 at batch 4 133.1 -> 121.3 us
// (four pairs), at 8 148.7 -> 138.2, at 16 170.3 -> 168.2 (two), none from 32 on; MobileNet V2 at batch 8 250.7 -> 247.8 (one), at 32
// 380.5 -> 376.2 (five), at 64 484.7 -> 478.9 (six); 37 x 37 x 400 to 144 channels at batch 14 19.9 -> 15.6.
#include <cuda.h>
#include <cudaTypedefs.h>

#include <math.h>
#include <string.h>

#include <algorithm>

#include "f8_internal.h"
#include "f8_tc_ptx.cuh"

namespace {

constexpr int DP_TILE_M = 128;
constexpr int DP_SLAB = 128;                       // channels per slab
constexpr int DP_TAPS = 9;
constexpr int DP_MAX_A = 8;                        // activation stages
constexpr int DP_DIAGS = 2;                        // diagonal stages: the blocks of a whole slab
constexpr uint32_t DP_A_BYTES = DP_TILE_M * DP_SLAB;
// A diagonal 32 x 32 block in the form without swizzle: 8-row x 16-byte core matrices, 128 bytes between row groups.  Only four of the
// eight core matrices are not zero, (0, 0), (1, 0), (2, 1), (3, 1); with 256 bytes between the K halves the zero ones of both
// halves are the same memory, and a block takes 768 bytes: d0 d1 0 0 d2 d3.
constexpr uint32_t DP_BLOCK_BYTES = 768;
constexpr uint32_t DP_TAP_BYTES = 4 * DP_BLOCK_BYTES;
constexpr uint32_t DP_D_BYTES = DP_TAPS * DP_TAP_BYTES;
constexpr uint32_t DP_SLOT_BYTES = DP_TILE_M * DP_SLAB;
constexpr int DP_MAX_SLOTS = 8, DP_MAX_W = 16, DP_MAX_OUT = 3;
constexpr uint32_t DP_CONTROL_BYTES = 1024;
constexpr size_t DP_SMEM_LIMIT = 225 * 1024;
constexpr int DP_TMEM_COLS = 512;

constexpr int DP_A_WARP = 0, DP_MMA_WARP = 1, DP_MOVER_WARP = 2, DP_FETCH_WARP = 3, DP_FIRST_EPI = 4, DP_EPI_WARPS = 16;
constexpr int DP_W_WARP = DP_FIRST_EPI + DP_EPI_WARPS, DP_MMA2_WARP = DP_W_WARP + 1, DP_DIAG_WARP = DP_W_WARP + 2;
constexpr int DP_THREADS = 32 * (DP_DIAG_WARP + 1);

struct DpControl {
    uint64_t full[DP_MAX_A], empty[DP_MAX_A];
    uint64_t dfull[DP_DIAGS], dempty[DP_DIAGS];
    uint64_t tfull1[2], tempty1[2];
    uint64_t slot_full[DP_MAX_SLOTS], slot_free[DP_MAX_SLOTS];
    uint64_t wfull[DP_MAX_W], wempty[DP_MAX_W];
    uint64_t tfull2[2], tempty2[2];
    uint64_t out_full[DP_MAX_OUT], out_free[DP_MAX_OUT], res_full[DP_MAX_OUT];
    uint32_t tmem_base_slot;
    int abort_flag;
};
static_assert(sizeof(DpControl) <= DP_CONTROL_BYTES, "control block does not fit its slot");

struct DpDiv {
    uint32_t mul, shift;
};
__device__ __forceinline__ int dp_div(int n, DpDiv d) { return (int)(((uint64_t)(uint32_t)n * d.mul) >> d.shift); }

struct DpParams {
    int M, ho, wo, stride, c, c_out;
    int m_tiles;
    int defer;                  // 1: a tile's second epilogue runs behind the next tile's first one
    int win;                    // 1: tiles of win_r whole output rows, win_wp positions per row, win_bands tiles per image
    int win_r, win_wp, win_bands;
    DpDiv div_bands;
    int a_stages;
    uint32_t a_bytes, a_tx;     // bytes of an activation stage / one load delivers
    uint32_t res_tx;            // bytes of a shortcut part
    DpDiv div_wo, div_ho;
    int slabs, slots;
    int parts, bn2;             // parts of bn2 output channels
    int accs2;                  // accumulators of the second GEMM: 2 of at most 128 columns, or 1 of up to 256
    int w_stages, w_res;        // w_res: every weight tile has a stage of its own and stays
    int out_bufs, slab_w, n_slabs;      // an output part leaves in column slabs of slab_w bytes
    uint32_t swz_mask;
    uint32_t w_bytes, out_bytes;
    uint32_t diag_off, slot_off, w_off, out_off, dw_off, bias_off;       // byte offsets behind the activation stages
    uint32_t idesc1, idesc2;
    const int8_t *dw;           // [c][9]
    const int32_t *bias1, *bias2;
    int s1, mul1;
    int sh_acc2, s2, mul_acc2, mul_res2, r_signed;
    uint8_t *y_mid;
    int *status;
    int tag;
    unsigned long long wait_limit;
};

// One 32-column block of one tap (whole warp; an elected lane issues).
__device__ __forceinline__ void dp_mma(uint32_t d_tmem, uint32_t a_lo, uint32_t a_hi, uint32_t b_lo, uint32_t b_hi, uint32_t idesc, uint32_t accumulate) {
    asm volatile("{\n\t" F8_ELECT ".reg .pred p;\n\t.reg .b64 a, b;\n\tsetp.ne.b32 p, %6, 0;\n\tmov.b64 a, {%1, %2};\n\tmov.b64 b, {%3, %4};\n\t"
                 "@e tcgen05.mma.cta_group::1.kind::i8 [%0], a, b, %5, p;\n\t}" ::"r"(d_tmem),
                 "r"(a_lo), "r"(a_hi), "r"(b_lo), "r"(b_hi), "r"(idesc), "r"(accumulate)
                 : "memory");
}
// All four blocks of a full slab.
__device__ __forceinline__ void dp_mma4(uint32_t d_tmem, uint32_t a_lo, uint32_t a_hi, uint32_t b_lo, uint32_t b_hi, uint32_t idesc, uint32_t accumulate) {
#define DP_NEXT(n, dd, aa, bb) \
    "add.u32 u, %0, " #dd ";\n\tadd.u32 x, %1, " #aa ";\n\tadd.u32 y, %3, " #bb ";\n\tmov.b64 a, {x, %2};\n\tmov.b64 b, {y, %4};\n\t" \
    "@e tcgen05.mma.cta_group::1.kind::i8 [u], a, b, %5, p;\n\t"
    asm volatile("{\n\t" F8_ELECT ".reg .pred p;\n\t.reg .b64 a, b;\n\t.reg .b32 u, x, y;\n\tsetp.ne.b32 p, %6, 0;\n\tmov.b64 a, {%1, %2};\n\tmov.b64 b, {%3, %4};\n\t"
                 "@e tcgen05.mma.cta_group::1.kind::i8 [%0], a, b, %5, p;\n\t" DP_NEXT(1, 32, 2, 48) DP_NEXT(2, 64, 4, 96) DP_NEXT(3, 96, 6, 144) "}" ::"r"(d_tmem),
                 "r"(a_lo), "r"(a_hi), "r"(b_lo), "r"(b_hi), "r"(idesc), "r"(accumulate)
                 : "memory");
#undef DP_NEXT
}
__device__ __forceinline__ void sts8(uint32_t addr, uint32_t v) { asm volatile("st.shared.u8 [%0], %1;" ::"r"(addr), "r"(v) : "memory"); }

template <bool RES, bool SGN>
__global__ void __launch_bounds__(DP_THREADS, 1)
f8_dwpw_tc_kernel(const __grid_constant__ CUtensorMap map_a, const __grid_constant__ CUtensorMap map_w, const __grid_constant__ CUtensorMap map_y,
                  const __grid_constant__ CUtensorMap map_r, const DpParams p) {
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem_aligned = (uint8_t *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    DpControl &ctl = *(DpControl *)smem_aligned;
    uint8_t *smem = smem_aligned + DP_CONTROL_BYTES;
    const int warp = uniform((int)(threadIdx.x >> 5)), lane = threadIdx.x & 31;
    const int worker = (int)blockIdx.x, n_workers = (int)gridDim.x;
    const uint32_t smem_base = smem_u32(smem);
    const uint32_t full_bar = smem_u32(&ctl.full[0]), empty_bar = smem_u32(&ctl.empty[0]);
    const uint32_t dfull = smem_u32(&ctl.dfull[0]), dempty = smem_u32(&ctl.dempty[0]);
    const uint32_t tfull1 = smem_u32(&ctl.tfull1[0]), tempty1 = smem_u32(&ctl.tempty1[0]);
    const uint32_t slot_full = smem_u32(&ctl.slot_full[0]), slot_free = smem_u32(&ctl.slot_free[0]);
    const uint32_t wfull = smem_u32(&ctl.wfull[0]), wempty = smem_u32(&ctl.wempty[0]);
    const uint32_t tfull2 = smem_u32(&ctl.tfull2[0]), tempty2 = smem_u32(&ctl.tempty2[0]);
    const uint32_t out_full = smem_u32(&ctl.out_full[0]), out_free = smem_u32(&ctl.out_free[0]), res_full = smem_u32(&ctl.res_full[0]);

    if (threadIdx.x == 32) {
        prefetch_tensormap(&map_a);
        prefetch_tensormap(&map_w);
        prefetch_tensormap(&map_y);
        if (RES) prefetch_tensormap(&map_r);
    }
    if (threadIdx.x == 0) {
        ctl.abort_flag = 0;
        for (int s = 0; s < DP_MAX_A; ++s) {
            mbar_init(full_bar + 8 * s, 1);
            mbar_init(empty_bar + 8 * s, 1);
        }
        for (int s = 0; s < DP_DIAGS; ++s) {
            mbar_init(dfull + 8 * s, 1);
            mbar_init(dempty + 8 * s, 1);
        }
        for (int i = 0; i < 2; ++i) {
            mbar_init(tfull1 + 8 * i, 1);
            mbar_init(tempty1 + 8 * i, DP_EPI_WARPS);
            mbar_init(tfull2 + 8 * i, 1);
            mbar_init(tempty2 + 8 * i, DP_EPI_WARPS);
        }
        for (int i = 0; i < DP_MAX_SLOTS; ++i) {
            mbar_init(slot_full + 8 * i, DP_EPI_WARPS);
            mbar_init(slot_free + 8 * i, 1);
        }
        for (int i = 0; i < DP_MAX_W; ++i) {
            mbar_init(wfull + 8 * i, 1);
            mbar_init(wempty + 8 * i, 1);
        }
        for (int i = 0; i < DP_MAX_OUT; ++i) {
            mbar_init(out_full + 8 * i, DP_EPI_WARPS);
            mbar_init(out_free + 8 * i, 1);
            mbar_init(res_full + 8 * i, 1);
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    // the diagonal blocks start out zero (the tensor core reads them through the async proxy, hence the fence)
    for (int i = threadIdx.x; i < DP_DIAGS * (int)(DP_D_BYTES / 16); i += DP_THREADS) *(uint4 *)(smem + p.diag_off + 16 * i) = make_uint4(0, 0, 0, 0);
    {
        // compact copy of the depthwise weights, [c][9] -> [9][slabs][32][4] (channel 32 q + n of a slab at [n][q]: one word holds
        // what a lane of the diagonal writer needs of a tap), sixteen bytes a thread (c is a multiple of sixteen)
        uint8_t *wdw = smem + p.dw_off;
        const int cp = p.slabs * DP_SLAB;
        for (int i = threadIdx.x; i < cp * DP_TAPS / 16; i += DP_THREADS) {
            const uint4 w = 16 * i < p.c * DP_TAPS ? __ldg((const uint4 *)p.dw + i) : make_uint4(0, 0, 0, 0);
            const uint32_t ww[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
            for (int j = 0; j < 16; ++j) {
                const int e = 16 * i + j, ch = e / DP_TAPS;
                wdw[(e - ch * DP_TAPS) * cp + (ch & ~127) + (ch & 31) * 4 + ((ch >> 5) & 3)] = (uint8_t)(ww[j >> 2] >> (8 * (j & 3)));
            }
        }
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    if (warp == DP_MMA_WARP) tmem_alloc(smem_u32(&ctl.tmem_base_slot), DP_TMEM_COLS);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = uniform(ctl.tmem_base_slot);
    grid_launch_dependents();

    const int n_local = worker < p.m_tiles ? (p.m_tiles - worker + n_workers - 1) / n_workers : 0;
    const WaitCtx wc = make_wait_ctx(&ctl.abort_flag, p.status, p.wait_limit);
    const int tagbits = p.tag << 8;
    const int S = p.slabs;

    if (warp == DP_A_WARP) {
        // ------------------------------------------------------------------ activations
        grid_dependency_wait();
        bool ok = true, have_last = false;
        int stage = 0, last_stage = 0;
        uint32_t par = 0, last_par = 0;
        for (int l = 0; ok && l < n_local; ++l) {
            const int tile = worker + l * n_workers;
            int img, base_w, base_h;
            if (p.win) {
                img = dp_div(tile, p.div_bands);
                base_w = -1;
                base_h = (tile - img * p.win_bands) * p.win_r - 1;
            } else {
                const int m0 = tile * DP_TILE_M;
                const int t1 = dp_div(m0, p.div_wo);
                const int ow = m0 - t1 * p.wo;
                img = dp_div(t1, p.div_ho);
                const int oh = t1 - img * p.ho;
                base_w = ow * p.stride - 1;
                base_h = oh * p.stride - 1;
            }
            for (int s = 0; ok && s < S; ++s) {
                int r = 0, sx = 0;
                for (int t = 0; t < (p.win ? 1 : DP_TAPS); ++t) {
                    if (!warp_wait(empty_bar + 8 * stage, par ^ 1u, wc, tagbits | 231)) { ok = false; break; }
                    const uint32_t fb = full_bar + 8 * stage, dst = smem_base + (uint32_t)stage * p.a_bytes;
                    warp_expect_tx(fb, p.a_tx);
                    if (p.win) tma_load_4d(dst, &map_a, fb, s * DP_SLAB, base_w, base_h, img, lane == 0);
                    else tma_load_im2col(dst, &map_a, fb, s * DP_SLAB, base_w, base_h, img, (uint16_t)sx, (uint16_t)r, lane == 0);
                    have_last = true;
                    last_stage = stage;
                    last_par = par;
                    if (++sx == 3) { sx = 0; ++r; }
                    if (++stage == p.a_stages) { stage = 0; par ^= 1u; }
                }
            }
        }
        if (!ok && have_last) {
            const unsigned long long t0 = clock64();
            while (!mbar_try_wait(full_bar + 8 * last_stage, last_par) && (unsigned long long)(clock64() - t0) < DRAIN_LIMIT_CYCLES) {
            }
        }
    } else if (warp == DP_DIAG_WARP) {
        // ------------------------------------------------------------------ the diagonals of every slab
        const uint32_t *wdw = (const uint32_t *)(smem + p.dw_off) + lane;
        const int cp = S * 32;          // words per tap
        const uint32_t diag = (uint32_t)(lane >> 4) * 256u + (uint32_t)lane * 16u + (uint32_t)(lane & 15);
        int ds = 0;
        uint32_t par = 0;
        bool ok = true;
        for (int l = 0; ok && l < n_local; ++l)
            for (int s = 0; s < S; ++s) {
                if (!warp_wait(dempty + 8 * ds, par ^ 1u, wc, tagbits | 232)) { ok = false; break; }
                const uint32_t dst = smem_base + p.diag_off + (uint32_t)ds * DP_D_BYTES + diag;
#pragma unroll
                for (int t = 0; t < DP_TAPS; ++t) {
                    const uint32_t w = wdw[t * cp + s * 32];
#pragma unroll
                    for (int q = 0; q < 4; ++q) sts8(dst + t * DP_TAP_BYTES + q * DP_BLOCK_BYTES, w >> (8 * q));
                }
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                __syncwarp();
                warp_arrive(dfull + 8 * ds);
                if (++ds == DP_DIAGS) { ds = 0; par ^= 1u; }
            }
    } else if (warp == DP_MMA_WARP) {
        // ------------------------------------------------------------------ issuer 1: the depthwise layer
        if (n_local > 0) {
            const uint64_t a_desc = smem_desc_hi(DP_SLAB);
            const uint32_t a_lo0 = (uint32_t)a_desc | ((smem_base & 0x3ffffu) >> 4), a_hi = (uint32_t)(a_desc >> 32);
            // diagonal blocks: no swizzle, 256 bytes between the K halves, 128 between groups of eight rows
            const uint32_t b_lo0 = ((256u >> 4) << 16) | (((smem_base + p.diag_off) & 0x3ffffu) >> 4), b_hi = (128u >> 4) | (1u << 14);
            const uint32_t a16 = p.a_bytes >> 4;
            bool ok = true;
            int stage = 0, ds = 0, v = 0;
            uint32_t par = 0, dpar = 0;
            for (int l = 0; ok && l < n_local; ++l)
                for (int s = 0; ok && s < S; ++s, ++v) {
                    const int acc = v & 1;
                    if (!warp_wait(tempty1 + 8 * acc, (uint32_t)((v >> 1) & 1) ^ 1u, wc, tagbits | 233)) { ok = false; break; }
                    const uint32_t d_tmem = tmem_base + (uint32_t)acc * DP_SLAB;
                    const int blocks = min(4, (p.c - s * DP_SLAB + 31) >> 5);
                    if (!warp_wait(dfull + 8 * ds, dpar, wc, tagbits | 230)) { ok = false; break; }
                    const uint32_t b_lo = b_lo0 + (uint32_t)ds * (DP_D_BYTES >> 4);
                    if (p.win) {
                        // (straight-line code over the taps: in a loop with branches the operands do not stay in uniform registers)
                        if (!warp_wait(full_bar + 8 * stage, par, wc, tagbits | 234)) { ok = false; break; }
                        tc_fence_after();
                        const uint32_t a_lo = a_lo0 + (uint32_t)stage * a16, row16 = 8u * (uint32_t)p.win_wp;      // a pixel row: 128 bytes
                        if (blocks == 4) {
#pragma unroll
                            for (int t = 0; t < DP_TAPS; ++t)
                                dp_mma4(d_tmem, a_lo + (uint32_t)(t / 3) * row16 + 8u * (t % 3), a_hi, b_lo + t * (DP_TAP_BYTES >> 4), b_hi, p.idesc1, t != 0 ? 1u : 0u);
                        } else {
                            for (int q = 0; q < blocks; ++q)
#pragma unroll
                                for (int t = 0; t < DP_TAPS; ++t)
                                    dp_mma(d_tmem + 32u * q, a_lo + (uint32_t)(t / 3) * row16 + 8u * (t % 3) + 2u * q, a_hi,
                                           b_lo + t * (DP_TAP_BYTES >> 4) + q * (DP_BLOCK_BYTES >> 4), b_hi, p.idesc1, t != 0 ? 1u : 0u);
                        }
                        mma_commit(empty_bar + 8 * stage);
                        if (++stage == p.a_stages) { stage = 0; par ^= 1u; }
                    } else {
                        for (int t = 0; t < DP_TAPS; ++t) {
                            if (!warp_wait(full_bar + 8 * stage, par, wc, tagbits | 234)) { ok = false; break; }
                            tc_fence_after();
                            const uint32_t a_lo = a_lo0 + (uint32_t)stage * a16, bt_lo = b_lo + t * (DP_TAP_BYTES >> 4);
                            if (blocks == 4) dp_mma4(d_tmem, a_lo, a_hi, bt_lo, b_hi, p.idesc1, t != 0 ? 1u : 0u);
                            else
                                for (int q = 0; q < blocks; ++q)
                                    dp_mma(d_tmem + 32u * q, a_lo + 2u * q, a_hi, bt_lo + (DP_BLOCK_BYTES >> 4) * q, b_hi, p.idesc1, t != 0 ? 1u : 0u);
                            mma_commit(empty_bar + 8 * stage);
                            if (++stage == p.a_stages) { stage = 0; par ^= 1u; }
                        }
                        if (!ok) break;
                    }
                    mma_commit(dempty + 8 * ds);
                    if (++ds == DP_DIAGS) { ds = 0; dpar ^= 1u; }
                    mma_commit(tfull1 + 8 * acc);
                }
            if (ok) {
                // the releases of the last stage uses, which nobody else waits for, must land before the CTA goes
                const int total = n_local * S * (p.win ? 1 : DP_TAPS), total_d = n_local * S;
                for (int g = max(0, total - p.a_stages); g < total; ++g)
                    warp_wait(empty_bar + 8 * (g % p.a_stages), (uint32_t)(g / p.a_stages) & 1u, wc, tagbits | 235);
                for (int g = max(0, total_d - DP_DIAGS); g < total_d; ++g)
                    warp_wait(dempty + 8 * (g % DP_DIAGS), (uint32_t)(g / DP_DIAGS) & 1u, wc, tagbits | 229);
            }
        }
    } else if (warp == DP_W_WARP) {
        // ------------------------------------------------------------------ pointwise weight tiles, order (part, slab)
        if (p.w_res) {
            int i = 0;
            for (int q = 0; q < p.parts; ++q)
                for (int s = 0; s < S; ++s, ++i) {
                    warp_expect_tx(wfull + 8 * i, p.w_bytes);
                    tma_load_2d(smem_base + p.w_off + (uint32_t)i * p.w_bytes, &map_w, wfull + 8 * i, s * DP_SLAB, q * p.bn2, lane == 0);
                }
            // they must have landed before this CTA's shared memory may go away
            for (int j = 0; j < i; ++j) warp_wait(wfull + 8 * j, 0, wc, tagbits | 236);
        } else {
            int ws = 0;
            uint32_t par = 0;
            bool ok = true;
            for (int l = 0; ok && l < n_local; ++l)
                for (int q = 0; ok && q < p.parts; ++q)
                    for (int s = 0; s < S; ++s) {
                        if (!warp_wait(wempty + 8 * ws, par ^ 1u, wc, tagbits | 237)) { ok = false; break; }
                        warp_expect_tx(wfull + 8 * ws, p.w_bytes);
                        tma_load_2d(smem_base + p.w_off + (uint32_t)ws * p.w_bytes, &map_w, wfull + 8 * ws, s * DP_SLAB, q * p.bn2, lane == 0);
                        if (++ws == p.w_stages) { ws = 0; par ^= 1u; }
                    }
        }
    } else if (warp == DP_MMA2_WARP) {
        // ------------------------------------------------------------------ issuer 2: the pointwise layer
        if (n_local > 0) {
            const uint64_t desc = smem_desc_hi(DP_SLAB);
            const uint32_t desc_lo0 = (uint32_t)desc | ((smem_base & 0x3ffffu) >> 4), desc_hi = (uint32_t)(desc >> 32);
            const uint32_t slot_lo0 = desc_lo0 + (p.slot_off >> 4), w_lo0 = desc_lo0 + (p.w_off >> 4);
            bool ok = true;
            int ws = 0, e = 0;
            uint32_t wpar = 0;
            int slot0 = 0;                 // slot and parity of the tile's first slab
            uint32_t spar0 = 0;
            for (int l = 0; ok && l < n_local; ++l) {
                int slot = slot0;
                uint32_t spar = spar0;
                for (int q = 0; ok && q < p.parts; ++q, ++e) {
                    const int d = p.accs2 == 2 ? (e & 1) : 0;
                    const uint32_t dpar = (uint32_t)(p.accs2 == 2 ? (e >> 1) : e) & 1u;
                    if (!warp_wait(tempty2 + 8 * d, dpar ^ 1u, wc, tagbits | 238)) { ok = false; break; }
                    tc_fence_after();
                    slot = slot0;
                    spar = spar0;
                    if (p.w_res) ws = q * S;
                    for (int s = 0; s < S; ++s) {
                        bool got = true;
                        if (q == 0) got = warp_wait(slot_full + 8 * slot, spar, wc, tagbits | 239);
                        got = got && warp_wait(wfull + 8 * ws, wpar, wc, tagbits | 240);
                        if (!got) { ok = false; break; }
                        tc_fence_after();
                        mma_i8_sub<4>(tmem_base + 256u + (uint32_t)d * 128u, slot_lo0 + (uint32_t)slot * (DP_SLOT_BYTES >> 4),
                                      w_lo0 + (uint32_t)ws * (p.w_bytes >> 4), desc_hi, p.idesc2, s != 0 ? 1u : 0u);
                        if (!p.w_res) mma_commit(wempty + 8 * ws);
                        if (q == p.parts - 1) mma_commit(slot_free + 8 * slot);
                        if (p.w_res) ++ws;
                        else if (++ws == p.w_stages) { ws = 0; wpar ^= 1u; }
                        if (++slot == p.slots) { slot = 0; spar ^= 1u; }
                    }
                    if (ok) mma_commit(tfull2 + 8 * d);
                }
                slot0 = slot;
                spar0 = spar;
            }
            if (ok) {
                // last arrivals without another waiter
                const int total_v = n_local * S;
                for (int g = max(0, total_v - p.slots); g < total_v; ++g)
                    warp_wait(slot_free + 8 * (g % p.slots), (uint32_t)(g / p.slots) & 1u, wc, tagbits | 241);
                const int total_w = n_local * S * p.parts;
                if (!p.w_res)
                    for (int g = max(0, total_w - p.w_stages); g < total_w; ++g)
                        warp_wait(wempty + 8 * (g % p.w_stages), (uint32_t)(g / p.w_stages) & 1u, wc, tagbits | 242);
            }
        }
    } else if (warp == DP_MOVER_WARP) {
        // ------------------------------------------------------------------ output mover
        grid_dependency_wait();
        int b = 0;
        uint32_t par = 0;
        bool ok = true;
        for (int l = 0; ok && l < n_local; ++l)
            for (int q = 0; q < p.parts; ++q) {
                if (!warp_wait(out_full + 8 * b, par, wc, tagbits | 243)) { ok = false; break; }
                const uint32_t src = smem_base + p.out_off + (uint32_t)b * p.out_bytes;
                const int tile = worker + l * n_workers;
                const int img = p.win ? dp_div(tile, p.div_bands) : 0, y0 = (tile - img * p.win_bands) * p.win_r;
                for (int sl = 0; sl < p.n_slabs; ++sl)
                    if (q * p.bn2 + sl * p.slab_w < p.c_out) {
                        const uint32_t from = src + (uint32_t)sl * (DP_TILE_M * p.slab_w);
                        // (the two extra positions of every row and rows below the image are clipped by the hardware)
                        if (p.win) tma_store_4d(&map_y, from, q * p.bn2 + sl * p.slab_w, 0, y0, img);
                        else tma_store_2d(&map_y, from, q * p.bn2 + sl * p.slab_w, tile * DP_TILE_M);
                    }
                tma_store_commit();
                tma_store_wait_read();
                warp_arrive(out_free + 8 * b);
                if (++b == p.out_bufs) { b = 0; par ^= 1u; }
            }
        tma_store_wait();
    } else if (warp == DP_FETCH_WARP) {
        // ------------------------------------------------------------------ shortcut fetcher
        if (RES) {
            grid_dependency_wait();
            int b = 0;
            uint32_t par = 0;
            bool ok = true;
            for (int l = 0; ok && l < n_local; ++l)
                for (int q = 0; q < p.parts; ++q) {
                    if (!warp_wait(out_free + 8 * b, par ^ 1u, wc, tagbits | 244)) { ok = false; break; }
                    warp_expect_tx(res_full + 8 * b, p.res_tx);
                    const uint32_t dst = smem_base + p.out_off + (uint32_t)b * p.out_bytes;
                    const int tile = worker + l * n_workers;
                    const int img = p.win ? dp_div(tile, p.div_bands) : 0, y0 = (tile - img * p.win_bands) * p.win_r;
                    for (int sl = 0; sl < p.n_slabs; ++sl) {
                        const uint32_t to = dst + (uint32_t)sl * (DP_TILE_M * p.slab_w);
                        if (p.win) tma_load_4d(to, &map_r, res_full + 8 * b, q * p.bn2 + sl * p.slab_w, 0, y0, img, lane == sl);
                        else tma_load_2d(to, &map_r, res_full + 8 * b, q * p.bn2 + sl * p.slab_w, tile * DP_TILE_M, lane == sl);
                    }
                    if (++b == p.out_bufs) { b = 0; par ^= 1u; }
                }
        }
    } else {
        // ------------------------------------------------------------------ epilogue warps
        const int quarter = warp & 3;                       // TMEM lanes 32 * quarter .. + 31
        const int g = (warp - DP_FIRST_EPI) >> 2;           // column quarter of both accumulators
        const int n_bias1 = S * DP_SLAB, n_bias2 = p.parts * p.bn2;
        {
            // bias' = (bias << sh_acc) + 2^(s - 1) of both layers, once per CTA, behind a barrier of these warps only
            int *bias_all = (int *)(smem + p.bias_off);
            for (int i = (int)threadIdx.x - DP_FIRST_EPI * 32; i < n_bias1 + n_bias2; i += DP_EPI_WARPS * 32) {
                if (i < n_bias1) bias_all[i] = (p.bias1 && i < p.c ? __ldg(p.bias1 + i) : 0) + (1 << (p.s1 - 1));
                else bias_all[i] = ((p.bias2 && i - n_bias1 < p.c_out ? __ldg(p.bias2 + i - n_bias1) : 0) << p.sh_acc2) + (1 << (p.s2 - 1));
            }
            asm volatile("bar.sync 1, %0;" ::"n"(DP_EPI_WARPS * 32) : "memory");
        }
        if (p.y_mid) grid_dependency_wait();     // direct stores of the first layer's output
        const int row = quarter * 32 + lane;
        uint32_t rsel[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) rsel[k] = p.r_signed ? (0x8880u | (0x1111u * k)) : (0x4440u | k);
        const uint32_t t_lane = tmem_base + ((uint32_t)(quarter * 32) << 16);
        const uint32_t bias1_s = smem_base + p.bias_off, bias2_s = bias1_s + 4u * n_bias1;
        const uint32_t so1 = (uint32_t)row * DP_SLAB, swz1 = (uint32_t)row & 7;
        const int chunks2 = p.bn2 / 16, per2 = (chunks2 + 3) / 4;         // at most four chunks of 16 columns per warp
        const int c_begin = min(g * per2, chunks2), n_c = min(c_begin + per2, chunks2) - c_begin;
        uint32_t so2[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const uint32_t col = (uint32_t)(c_begin + i) * 16u, sl = col / (uint32_t)p.slab_w;
            uint32_t off = (uint32_t)row * p.slab_w + (col - sl * p.slab_w);
            off ^= ((off >> 7) & p.swz_mask) << 4;
            so2[i] = sl * (uint32_t)(DP_TILE_M * p.slab_w) + off;
        }
        int ob = 0, slot = 0, v = 0, e = 0;
        uint32_t opar = 0, spar = 0;
        bool ok = true;
        for (int l = 0; ok && l < n_local + p.defer; ++l) {
            if (l < n_local) {
                for (int s = 0; ok && s < S; ++s, ++v) {
                    const int acc = v & 1;
                    bool got = mbar_wait(slot_free + 8 * slot, spar ^ 1u, wc, tagbits | 245);
                    got = mbar_wait(tfull1 + 8 * acc, (uint32_t)((v >> 1) & 1), wc, tagbits | 246) && got;
                    if (!__all_sync(0xffffffffu, got)) { ok = false; break; }
                    tc_fence_after();
                    int va[16], vb[16];
                    const uint32_t t_addr = t_lane + (uint32_t)(acc * DP_SLAB + g * 32);
                    tmem_ld16(t_addr, va);
                    tmem_ld16(t_addr + 16, vb);
                    tmem_ld_wait16(va);
                    tmem_ld_wait16(vb);
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(tempty1 + 8 * acc);
                    const uint32_t dst = smem_base + p.slot_off + (uint32_t)slot * DP_SLOT_BYTES + so1;
                    const uint32_t b_addr = bias1_s + 4u * (uint32_t)(s * DP_SLAB + g * 32);
                    const uint4 o0 = epilogue_fast16<false, false>(va, b_addr, make_uint4(0, 0, 0, 0), p.mul1, 0, rsel, p.s1);
                    sts128(dst + (((uint32_t)(2 * g) ^ swz1) << 4), o0);
                    const uint4 o1 = epilogue_fast16<false, false>(vb, b_addr + 64, make_uint4(0, 0, 0, 0), p.mul1, 0, rsel, p.s1);
                    sts128(dst + (((uint32_t)(2 * g + 1) ^ swz1) << 4), o1);
                    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                    __syncwarp();
                    if (lane == 0) mbar_arrive(slot_full + 8 * slot);
                    if (p.y_mid) {
                        const int tile = worker + l * n_workers, ch = s * DP_SLAB + g * 32;
                        size_t m = (size_t)tile * DP_TILE_M + row;          // this thread's output pixel
                        bool valid = m < (size_t)p.M;
                        if (p.win) {
                            const int img = dp_div(tile, p.div_bands), y0 = (tile - img * p.win_bands) * p.win_r;
                            const int ry = row / p.win_wp, rx = row - ry * p.win_wp;
                            valid = ry < p.win_r && y0 + ry < p.ho && rx < p.wo;
                            m = ((size_t)img * p.ho + (size_t)(y0 + ry)) * p.wo + rx;
                        }
                        if (valid && ch < p.c) *(uint4 *)(p.y_mid + m * p.c + ch) = o0;
                        if (valid && ch + 16 < p.c) *(uint4 *)(p.y_mid + m * p.c + ch + 16) = o1;
                    }
                    if (++slot == p.slots) { slot = 0; spar ^= 1u; }
                }
            }
            // second epilogue, all parts: of this tile, or (defer) of the one before
            if (p.defer ? l == 0 : l == n_local) continue;
            for (int q = 0; ok && q < p.parts; ++q, ++e) {
                const int d = p.accs2 == 2 ? (e & 1) : 0;
                bool got;
                if (RES) got = mbar_wait(res_full + 8 * ob, opar, wc, tagbits | 247);
                else got = mbar_wait(out_free + 8 * ob, opar ^ 1u, wc, tagbits | 248);
                got = mbar_wait(tfull2 + 8 * d, (uint32_t)(p.accs2 == 2 ? (e >> 1) : e) & 1u, wc, tagbits | 249) && got;
                if (!__all_sync(0xffffffffu, got)) { ok = false; break; }
                tc_fence_after();
                const uint32_t out_buf = smem_base + p.out_off + (uint32_t)ob * p.out_bytes;
                const uint32_t t_addr = t_lane + 256u + (uint32_t)(d * 128 + c_begin * 16), b_addr = bias2_s + 4u * (uint32_t)(q * p.bn2 + c_begin * 16);
                auto release_acc = [&]() {
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(tempty2 + 8 * d);
                };
                int va[16], vb[16];
                if (n_c > 0) tmem_ld16(t_addr, va);
                else release_acc();
#pragma unroll
                for (int i = 0; i < 4; i += 2) {
                    if (i < n_c) {
                        uint4 rw = make_uint4(0, 0, 0, 0);
                        if (RES) rw = lds128(out_buf + so2[i]);
                        tmem_ld_wait16(va);
                        if (i + 1 < n_c) tmem_ld16(t_addr + (i + 1) * 16, vb);
                        else release_acc();
                        sts128(out_buf + so2[i], epilogue_fast16<RES, SGN>(va, b_addr + 64 * i, rw, p.mul_acc2, p.mul_res2, rsel, p.s2));
                    }
                    if (i + 1 < n_c) {
                        uint4 rw = make_uint4(0, 0, 0, 0);
                        if (RES) rw = lds128(out_buf + so2[i + 1]);
                        tmem_ld_wait16(vb);
                        if (i + 2 < n_c) tmem_ld16(t_addr + (i + 2) * 16, va);
                        else release_acc();
                        sts128(out_buf + so2[i + 1], epilogue_fast16<RES, SGN>(vb, b_addr + 64 * (i + 1), rw, p.mul_acc2, p.mul_res2, rsel, p.s2));
                    }
                }
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                __syncwarp();
                if (lane == 0) mbar_arrive(out_full + 8 * ob);
                if (++ob == p.out_bufs) { ob = 0; opar ^= 1u; }
            }
        }
    }

    if (*(volatile int *)&ctl.abort_flag) {
        // a wait gave up: copies and tensor-core work may still be on their way to this CTA; give them time to land
        const unsigned long long t0 = clock64();
        while ((unsigned long long)(clock64() - t0) < 400000ull) {
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == DP_MMA_WARP) {
        tc_fence_after();
        tmem_dealloc(tmem_base, DP_TMEM_COLS);
    }
}

// ----------------------------------------------------------------------------- host side

PFN_cuTensorMapEncodeTiled_v12000 dp_encode_tiled = nullptr;
PFN_cuTensorMapEncodeIm2col_v12000 dp_encode_im2col = nullptr;

bool dp_load_driver_entry_points() {
    if (dp_encode_tiled && dp_encode_im2col) return true;
    void *f = nullptr;
    cudaDriverEntryPointQueryResult qr;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &f, cudaEnableDefault, &qr) != cudaSuccess || !f || qr != cudaDriverEntryPointSuccess) return false;
    dp_encode_tiled = (PFN_cuTensorMapEncodeTiled_v12000)f;
    f = nullptr;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeIm2col", &f, cudaEnableDefault, &qr) != cudaSuccess || !f || qr != cudaDriverEntryPointSuccess) return false;
    dp_encode_im2col = (PFN_cuTensorMapEncodeIm2col_v12000)f;
    return true;
}

DpDiv dp_make_div(int d) {
    uint32_t l = 0;
    while ((1u << l) < (uint32_t)d) ++l;
    DpDiv f;
    f.shift = 31 + l;
    f.mul = (uint32_t)(((uint64_t)1 << f.shift) / (uint32_t)d + 1);
    return f;
}

// How the tiles and the output channels are cut and what shared memory holds; false: does not fit.
bool dp_layout(const F8ConvGeom &g, int c_out, bool res, DpParams *p, size_t *smem) {
    p->slabs = (g.c + DP_SLAB - 1) / DP_SLAB;
    p->win = g.stride_h == 1 && g.wo + 2 <= DP_TILE_M ? 1 : 0;
    p->win_r = p->win_wp = p->win_bands = 1;
    p->a_bytes = p->a_tx = DP_A_BYTES;
    if (p->win) {
        p->win_wp = g.wo + 2;
        p->win_r = std::min(DP_TILE_M / p->win_wp, g.ho);
        p->win_bands = (g.ho + p->win_r - 1) / p->win_r;
        p->a_tx = (uint32_t)(DP_SLAB * p->win_wp * (p->win_r + 2));
        p->a_bytes = (p->a_tx + 1023) / 1024 * 1024;
    }
    // the last tap's window of a tile may end behind its stage: the other arrays that follow keep such reads in bounds
    const size_t fixed = (size_t)DP_DIAGS * DP_D_BYTES + (size_t)p->slabs * DP_SLAB * (DP_TAPS + 4) + DP_CONTROL_BYTES + 1024;
    for (int wide = 0; wide < 2; ++wide) {
        // parts of at most 128 columns with two accumulators; or one part of up to 256 columns
        if (wide && (c_out <= 128 || c_out > 256)) continue;
        p->bn2 = wide ? (c_out + 15) / 16 * 16 : (c_out <= 32 ? 32 : (c_out <= 64 ? 64 : 128));
        p->parts = (c_out + p->bn2 - 1) / p->bn2;
        p->accs2 = wide ? 1 : 2;
        p->slab_w = std::min(p->bn2, 128);
        p->n_slabs = (p->bn2 + 127) / 128;
        p->out_bytes = (uint32_t)(p->n_slabs * DP_TILE_M * p->slab_w);
        p->w_bytes = (uint32_t)((p->bn2 * DP_SLAB + 1023) / 1024 * 1024);
        // With one part GEMM 2 lets go of a tile's slabs one by one; several parts read all of them over again, so all have to be there
        // at once -- twice, if the epilogue of a tile's parts is to wait until the next tile's slabs have been converted.
        // With a single accumulator that wait must not depend on GEMM 2 of the next tile: it cannot start before that epilogue has read
        // the accumulator, so it lets go of no slab, and the next tile's slabs have to fit the slots without it.
        p->slots = p->parts > 1 ? std::max(2, p->slabs) : 2;
        p->defer = p->parts > 1 || (p->accs2 == 1 && p->slabs > p->slots) ? 0 : 1;
        if (p->slots > DP_MAX_SLOTS) continue;
        const int tiles = p->parts * p->slabs, min_a = 2;
        for (p->out_bufs = 2; p->out_bufs >= 1; --p->out_bufs) {
            size_t used = fixed + (size_t)p->slots * DP_SLOT_BYTES + (size_t)p->out_bufs * p->out_bytes + (size_t)p->parts * p->bn2 * 4 +
                          (size_t)min_a * p->a_bytes + 2 * (size_t)p->w_bytes;
            if (used > DP_SMEM_LIMIT) continue;
            p->a_stages = min_a;
            p->w_stages = 2;
            auto grow = [&](int &n, int most, size_t bytes) {
                while (n < most && used + bytes <= DP_SMEM_LIMIT) { ++n; used += bytes; }
            };
            // first a third window (six taps), then the weights for good if they fit, then more stages
            grow(p->a_stages, p->win ? 3 : 6, p->a_bytes);
            if (p->parts > 1 && 2 * p->slabs <= DP_MAX_SLOTS && used + (size_t)(2 * p->slabs - p->slots) * DP_SLOT_BYTES <= DP_SMEM_LIMIT) {
                used += (size_t)(2 * p->slabs - p->slots) * DP_SLOT_BYTES;
                p->slots = 2 * p->slabs;
                p->defer = 1;
            }
            if (tiles <= DP_MAX_W && (tiles <= 2 || used + (size_t)(tiles - 2) * p->w_bytes <= DP_SMEM_LIMIT)) {
                if (tiles < 2) used -= p->w_bytes;
                else used += (size_t)(tiles - 2) * p->w_bytes;
                p->w_stages = tiles;
                p->w_res = 1;
            } else {
                p->w_res = 0;
                grow(p->w_stages, 4, p->w_bytes);
            }
            grow(p->a_stages, p->win ? 4 : DP_MAX_A, p->a_bytes);
            *smem = used;
            return true;
        }
    }
    return false;
}

}   // namespace

struct F8DwPwPlan {
    CUtensorMap map_a, map_w, map_y, map_r;
    DpParams p;
    int grid;
    size_t smem;
    int res, sgn;
};

size_t f8_dwpw_plan_size() { return sizeof(F8DwPwPlan); }
void f8_dwpw_plan_set_tag(F8DwPwPlan *plan, int tag) { plan->p.tag = tag; }

bool f8_dwpw_supported(const F8ConvGeom &g1, const F8Requant &q1, int c_out2, const F8Requant &q2) {
    if (g1.c != g1.c_out || g1.c % 16 != 0 || c_out2 % 16 != 0 || g1.kh != 3 || g1.kw != 3 || g1.pad_h != 1 || g1.pad_w != 1 || g1.pad_h_end >= 0) return false;
    if (g1.stride_h != g1.stride_w || g1.stride_h < 1 || g1.stride_h > 2) return false;
    if ((size_t)g1.n * g1.h * g1.w * g1.c < 128 * 1024) return false;        // no im2col map for small tensors
    if ((long long)g1.n * g1.ho * g1.wo > 0x7fffff00ll) return false;
    if (q1.y_kind != F8_U8 || q1.has_res || q1.s < 1 || q1.s > 24) return false;
    if ((q2.y_kind != F8_U8 && q2.y_kind != F8_S8) || q2.r_s32 || q2.s < 1 || q2.s > 24) return false;
    DpParams p;
    size_t smem;
    return dp_layout(g1, c_out2, q2.has_res != 0, &p, &smem);
}

// Estimated microseconds of this kernel and of the two launches it replaces, fitted to event timings of the MobileNets' blocks at
// batches 8 - 256.
bool f8_dwpw_wanted(const F8ConvGeom &g1, int c_out2, bool res) {
    DpParams p;
    size_t smem;
    if (!dp_layout(g1, c_out2, res, &p, &smem)) return false;
    // a pointwise layer that the kernel for small layers would take: two short launches overlap better than this one long chain
    // (MobileNet V2 at batch 8: 252 us apart, 263 us fused)
    F8ConvGeom g2 = g1;
    g2.h = g1.ho; g2.w = g1.wo; g2.c_out = c_out2;
    g2.kh = g2.kw = g2.stride_h = g2.stride_w = 1;
    g2.pad_h = g2.pad_w = 0;
    if (f8_small_tc_wanted(g2, true)) return false;
    const double m = (double)g1.n * g1.ho * g1.wo, c = g1.c, n = c_out2;
    // Larger layers are faster apart, with the depthwise one on f8_dw_tc_kernel, which shares an instruction among three vertical taps
    // where this one spends one on each.  From where on depends on what the pointwise layer adds: whole networks with the line at
    // 2.4 and at 8 million outputs, MobileNet V2 (one part) at batch 64 487.8 and 480.9 us, MobileNet V1 (two to eight) 258.2 and 265.0.
    if (m * c >= (g1.stride_h == 1 && p.parts == 1 ? 8.0e6 : 2.4e6)) return false;
    const double tiles = p.win ? (double)g1.n * p.win_bands : std::ceil(m / DP_TILE_M);
    const double issue = p.slabs * (p.win ? 2600.0 : 4500.0), parts = p.parts * p.bn2 / 128.0;
    const double convert = p.slabs * 1000.0 + std::max(parts, 0.5) * 1300.0 + 600.0;
    // several parts without `defer`: GEMM 2 and the second epilogue do not overlap the tile's own slabs
    const double tile = p.defer || p.parts == 1 ? std::max(issue, convert) + 800.0 : issue + p.parts * (p.slabs * (2.0 * p.bn2 + 200.0) + 1500.0);
    const double fused = 6.5 + (std::ceil(tiles / 148.0) * tile + 3000.0) / 1900.0;
    const double dw = 7.0 + m * c * (g1.stride_h == 1 ? 0.62e-6 : 1.35e-6);
    const double pw = std::max(8.0, 9.0 + std::max(m * (c + n) / 6.4e6, m * c * n / 1.0e9));
    return fused < 0.9 * (dw + pw);
}

int f8_dwpw_layout_info(const F8ConvGeom &g1, int c_out2, bool res, int *info) {
    DpParams p;
    size_t smem;
    if (!dp_layout(g1, c_out2, res, &p, &smem)) return 0;
    const int tiles = p.win ? g1.n * p.win_bands : (g1.n * g1.ho * g1.wo + DP_TILE_M - 1) / DP_TILE_M;
    const int v[12] = {f8_dwpw_wanted(g1, c_out2, res) ? 1 : 0, tiles, p.slabs, p.slots, p.parts, p.accs2, p.defer, p.win ? 1 : DP_TAPS,
                       p.a_stages, p.w_stages, p.w_res, p.out_bufs};
    std::copy(v, v + 12, info);
    return 12;
}

cudaError_t f8_dwpw_plan_init(F8DwPwPlan *plan, const F8ConvGeom &g1, const F8Requant &q1, int c_out2, const F8Requant &q2, const void *x,
                              const int8_t *w_dw, const int32_t *bias1, const int8_t *w_pw, const int32_t *bias2, const void *res,
                              void *y_mid, void *y, int *status_word, const char **why) {
    *why = "";
    if (!dp_load_driver_entry_points()) {
        *why = "cuTensorMapEncode entry points not available";
        return cudaErrorNotSupported;
    }
    if (!f8_dwpw_supported(g1, q1, c_out2, q2) || (q2.has_res != 0) != (res != nullptr)) {
        *why = "shape outside the kernel's range";
        return cudaErrorInvalidValue;
    }
    memset(plan, 0, sizeof(*plan));
    DpParams &p = plan->p;
    p.M = g1.n * g1.ho * g1.wo;
    p.ho = g1.ho; p.wo = g1.wo; p.stride = g1.stride_h; p.c = g1.c; p.c_out = c_out2;
    p.div_wo = dp_make_div(g1.wo);
    p.div_ho = dp_make_div(g1.ho);
    dp_layout(g1, c_out2, q2.has_res != 0, &p, &plan->smem);
    p.div_bands = dp_make_div(p.win_bands);
    p.m_tiles = p.win ? g1.n * p.win_bands : (p.M + DP_TILE_M - 1) / DP_TILE_M;
    p.res_tx = p.win ? (uint32_t)(p.n_slabs * p.slab_w * p.win_wp * p.win_r) : p.out_bytes;
    p.swz_mask = p.slab_w == 128 ? 7u : (p.slab_w == 64 ? 3u : 1u);
    p.diag_off = (uint32_t)p.a_stages * p.a_bytes;
    p.slot_off = p.diag_off + DP_DIAGS * DP_D_BYTES;
    p.w_off = p.slot_off + (uint32_t)p.slots * DP_SLOT_BYTES;
    p.out_off = p.w_off + (uint32_t)p.w_stages * p.w_bytes;
    p.bias_off = p.out_off + (uint32_t)p.out_bufs * p.out_bytes;
    p.dw_off = p.bias_off + 4u * (uint32_t)(p.slabs * DP_SLAB + p.parts * p.bn2);
    // instruction descriptors: D = s32, A format (0 = u8, 1 = s8), B = s8, both K-major, N / 8, M / 16
    p.idesc1 = (2u << 4) | ((g1.x_signed ? 1u : 0u) << 7) | (1u << 10) | ((32u >> 3) << 17) | ((uint32_t)(DP_TILE_M >> 4) << 24);
    p.idesc2 = (2u << 4) | (1u << 10) | ((uint32_t)(p.bn2 >> 3) << 17) | ((uint32_t)(DP_TILE_M >> 4) << 24);
    p.dw = w_dw; p.bias1 = bias1; p.bias2 = bias2;
    p.s1 = q1.s; p.mul1 = 1;
    p.sh_acc2 = q2.sh_acc; p.s2 = q2.s; p.mul_acc2 = 1 << q2.sh_acc; p.mul_res2 = 1 << q2.sh_res; p.r_signed = q2.r_signed;
    p.y_mid = (uint8_t *)y_mid;
    p.status = status_word;
    p.wait_limit = f8_wait_limit_cycles();
    plan->res = q2.has_res ? 1 : 0;
    plan->sgn = q2.y_kind == F8_S8 ? 1 : 0;
    cuuint32_t ones[4] = {1, 1, 1, 1};
    {
        cuuint64_t dims[4] = {(cuuint64_t)g1.c, (cuuint64_t)g1.w, (cuuint64_t)g1.h, (cuuint64_t)g1.n};
        cuuint64_t strides[3] = {(cuuint64_t)g1.c, (cuuint64_t)g1.c * g1.w, (cuuint64_t)g1.c * g1.w * g1.h};
        int lower[2] = {-1, -1}, upper[2] = {-1, -1};          // -pad, pad - (k - 1)
        cuuint32_t estr[4] = {1, (cuuint32_t)g1.stride_w, (cuuint32_t)g1.stride_h, 1};
        cuuint32_t box[4] = {DP_SLAB, (cuuint32_t)p.win_wp, (cuuint32_t)(p.win_r + 2), 1};
        if (p.win) {
            if (dp_encode_tiled(&plan->map_a, CU_TENSOR_MAP_DATA_TYPE_UINT8, 4, const_cast<void *>(x), dims, strides, box, ones,
                                CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                                CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS) {
                *why = "cuTensorMapEncodeTiled rejected the activation tensor";
                return cudaErrorInvalidValue;
            }
        } else if (dp_encode_im2col(&plan->map_a, CU_TENSOR_MAP_DATA_TYPE_UINT8, 4, const_cast<void *>(x), dims, strides, lower, upper, DP_SLAB, DP_TILE_M,
                             estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                             CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS) {
            *why = "cuTensorMapEncodeIm2col rejected the activation tensor";
            return cudaErrorInvalidValue;
        }
    }
    {
        cuuint64_t dims[2] = {(cuuint64_t)g1.c, (cuuint64_t)c_out2};
        cuuint64_t strides[1] = {(cuuint64_t)g1.c};
        cuuint32_t box[2] = {DP_SLAB, (cuuint32_t)p.bn2};
        if (dp_encode_tiled(&plan->map_w, CU_TENSOR_MAP_DATA_TYPE_UINT8, 2, const_cast<int8_t *>(w_pw), dims, strides, box, ones,
                            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS) {
            *why = "cuTensorMapEncodeTiled rejected the weight tensor";
            return cudaErrorInvalidValue;
        }
    }
    {
        // [M, c_out], or (c_out, W, H, N) in boxes of win_r rows of W + 2 positions
        cuuint64_t dims[4] = {(cuuint64_t)c_out2, (cuuint64_t)(p.win ? g1.wo : p.M), (cuuint64_t)g1.ho, (cuuint64_t)g1.n};
        cuuint64_t strides[3] = {(cuuint64_t)c_out2, (cuuint64_t)c_out2 * g1.wo, (cuuint64_t)c_out2 * g1.wo * g1.ho};
        cuuint32_t box[4] = {(cuuint32_t)p.slab_w, (cuuint32_t)(p.win ? p.win_wp : DP_TILE_M), (cuuint32_t)p.win_r, 1};
        const cuuint32_t rank = p.win ? 4 : 2;
        const CUtensorMapSwizzle sw = p.slab_w == 128 ? CU_TENSOR_MAP_SWIZZLE_128B : (p.slab_w == 64 ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_32B);
        CUresult r = dp_encode_tiled(&plan->map_y, CU_TENSOR_MAP_DATA_TYPE_UINT8, rank, y, dims, strides, box, ones, CU_TENSOR_MAP_INTERLEAVE_NONE, sw,
                                     CU_TENSOR_MAP_L2_PROMOTION_NONE, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
        plan->map_r = plan->map_y;
        if (r == CUDA_SUCCESS && res)
            r = dp_encode_tiled(&plan->map_r, CU_TENSOR_MAP_DATA_TYPE_UINT8, rank, const_cast<void *>(res), dims, strides, box, ones,
                                CU_TENSOR_MAP_INTERLEAVE_NONE, sw, CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
        if (r != CUDA_SUCCESS) {
            *why = "cuTensorMapEncodeTiled rejected the output tensor";
            return cudaErrorInvalidValue;
        }
    }
    int dev = 0, sms = 148;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    plan->grid = std::min(p.m_tiles, sms);
    if (plan->smem < 120 * 1024) plan->smem = 120 * 1024;       // never two CTAs (each owning all of tensor memory) on an SM
    static bool attr_set[64] = {false};
    if (dev < 0 || dev >= 64) {
        *why = "device index out of range";
        return cudaErrorInvalidDevice;
    }
    if (!attr_set[dev]) {
        const int bytes = (int)DP_SMEM_LIMIT;
        cudaError_t e = cudaFuncSetAttribute(f8_dwpw_tc_kernel<false, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
        if (e == cudaSuccess) e = cudaFuncSetAttribute(f8_dwpw_tc_kernel<false, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
        if (e == cudaSuccess) e = cudaFuncSetAttribute(f8_dwpw_tc_kernel<true, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
        if (e == cudaSuccess) e = cudaFuncSetAttribute(f8_dwpw_tc_kernel<true, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
        if (e != cudaSuccess) {
            *why = "cudaFuncSetAttribute(MaxDynamicSharedMemorySize) failed";
            return e;
        }
        attr_set[dev] = true;
    }
    return cudaSuccess;
}

namespace {
template <bool RES, bool SGN>
cudaError_t dp_launch_variant(const F8DwPwPlan *plan, bool overlap_previous, cudaStream_t st) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)plan->grid);
    cfg.blockDim = dim3(DP_THREADS);
    cfg.dynamicSmemBytes = plan->smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = overlap_previous ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, f8_dwpw_tc_kernel<RES, SGN>, plan->map_a, plan->map_w, plan->map_y, plan->map_r, plan->p);
}
}   // namespace

cudaError_t f8_dwpw_launch(const F8DwPwPlan *plan, bool overlap_previous, cudaStream_t st) {
    if (plan->p.M == 0) return cudaSuccess;
    if (plan->res) return plan->sgn ? dp_launch_variant<true, true>(plan, overlap_previous, st) : dp_launch_variant<true, false>(plan, overlap_previous, st);
    return plan->sgn ? dp_launch_variant<false, true>(plan, overlap_previous, st) : dp_launch_variant<false, false>(plan, overlap_previous, st);
}

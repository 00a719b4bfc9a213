// Depthwise 3x3 convolution on the tensor cores (stride 1 or 2, 8-bit in and out), rows of the output walked with the
// accumulators of three output rows side by side in tensor memory.
//
// Per filter tap the weight matrix of a depthwise layer is diagonal.  An instruction of 128 pixels x 32 channels takes 40 cycles with
// N = 32 and 56 with N = 96, so the three vertical taps share one: an input row y contributes to the output rows y - 1, y and
// y + 1 with filter rows 2, 1 and 0, whose accumulators lie next to each other, and B is the three diagonal blocks below one another.
// Three instructions (one per horizontal tap) per 32 channels and input row, where one instruction per tap needs nine.
//
//   tile            one row of several images: image i, column x at position i * pitch + x, pitch = wo + 2 (stride 2: wo + 1), at most
//                   128 positions, times four blocks of 32 channels.  A horizontal tap is the same shared-memory tile read a
//                   row further down.  Layers of fewer channels put two or four groups of images into the four blocks.
//   producer        per input row one TMA load per image group (stride 2: the odd and the even columns); the zero fill
//                   outside the tensor is the padding
//   two issuers     per input row 6 instructions each (two blocks) into a ring of four output rows of 4 x 32 accumulator columns; a window of
//                   output rows that wraps around the ring is issued in two pieces
//   16 epilogue     accumulator -> registers; the bias (with the rounding constant) goes back in its place, so that every instruction
//   warps           accumulates and no addition is left to do here; shift, saturating pack, staging buffer
//   mover           TMA stores; positions outside the image are clipped
//
// A CTA keeps one slab of channels (its diagonal blocks are written once) and a run of output rows, the rows of all image groups being
// split evenly among the CTAs of a slab; a run costs one or two input rows more than it has output rows.
// Every wait is bounded (see f8_tc_ptx.cuh).
// Bound: DRAM for the large layers, else the instructions of a row, which wait for
// shared memory (operands, TMA traffic and staging together about 1250 cycles a row; measured 1700).  Against the packed-dot-product
// kernel, batch 256: 112 x 112 x 32 67.8 -> 52.8 us, 112 x 112 x 64 stride 2 74.0 -> 54.0, 56 x 56 x 128 67.6 -> 53.3, 14 x 14 x 512
// 26 -> 22; MobileNet V1 at batch 256 764 -> 639 us.
#include <cuda.h>
#include <cudaTypedefs.h>

#include <string.h>

#include <algorithm>

#include "f8_internal.h"
#include "f8_tc_ptx.cuh"

namespace {

constexpr int DW_M = 128;
constexpr int DW_RING = 4;                              // output rows in tensor memory
constexpr int DW_MAX_STAGES = 6, DW_OUT = 4;
constexpr uint32_t DW_TILE_BYTES = 128 * 128;           // four blocks of 128 positions x 32 channels
// three diagonal blocks (96 rows x 32 bytes): 8-row x 16-byte core matrices, 128 bytes between row groups, 1536 between the K halves
constexpr uint32_t DW_B_LBO = 1536, DW_B_BYTES = 2 * DW_B_LBO;
constexpr uint32_t DW_DIAG_BYTES = 12 * DW_B_BYTES;     // [horizontal tap][block]
constexpr uint32_t DW_CONTROL_BYTES = 1024;

constexpr int DW_A_WARP = 0, DW_MMA_WARP = 1, DW_MOVER_WARP = 2, DW_MMA2_WARP = 3, DW_FIRST_EPI = 4, DW_EPI_WARPS = 16;
constexpr int DW_THREADS = 32 * (DW_FIRST_EPI + DW_EPI_WARPS);

struct DwControl {
    uint64_t full[DW_MAX_STAGES], empty[DW_MAX_STAGES];
    uint64_t acc_full[DW_RING], acc_free[DW_RING];
    uint64_t out_full[DW_OUT], out_free[DW_OUT];
    uint32_t tmem_base_slot;
    int abort_flag;
};
static_assert(sizeof(DwControl) <= DW_CONTROL_BYTES, "control block does not fit its slot");

struct DwParams {
    int n, h, ho, c, stride;
    int slab_w;                 // channels of a slab: 128, 64, 32
    int slabs, groups;          // image groups (of a tile) per batch
    int pitch, images;          // positions per image row, images per block group
    int per_slab;               // CTAs per slab
    int stages;
    uint32_t stage_bytes, tx_bytes;
    uint32_t dx1, dx2, q1, q2;  // descriptor offsets (16-byte units) of horizontal taps 1, 2 and of blocks 1, 2 (3: both)
    uint32_t swz_mask;
    uint32_t diag_off, bias_off, out_off;
    uint32_t idesc;             // with N = 0
    const int8_t *w;            // [c][9]
    const int32_t *bias;
    int s;
    int *status;
    int tag;
    unsigned long long wait_limit;
};

// The three horizontal taps of two blocks (whole warp; an elected lane issues).  Every instruction accumulates.
__device__ __forceinline__ void dw_mma6(uint32_t d, uint32_t a_lo, uint32_t a_hi, uint32_t q1, uint32_t dx1, uint32_t dx2, uint32_t b_lo, uint32_t b_hi,
                                        uint32_t idesc) {
#define DW_MMA(dd, bb) "add.u32 y, %3, " #bb ";\n\tmov.b64 a, {x, %2};\n\tmov.b64 b, {y, %4};\n\t@e tcgen05.mma.cta_group::1.kind::i8 [" dd "], a, b, %5, t;\n\t"
    asm volatile("{\n\t" F8_ELECT ".reg .pred t;\n\t.reg .b64 a, b;\n\t.reg .b32 u, x, y;\n\tsetp.eq.b32 t, 0, 0;\n\tadd.u32 u, %0, 128;\n\t"
                 "mov.u32 x, %1;\n\t" DW_MMA("%0", 0) "add.u32 x, %1, %6;\n\t" DW_MMA("u", 192)
                 "add.u32 x, %1, %7;\n\t" DW_MMA("%0", 768) "add.u32 x, x, %6;\n\t" DW_MMA("u", 960)
                 "add.u32 x, %1, %8;\n\t" DW_MMA("%0", 1536) "add.u32 x, x, %6;\n\t" DW_MMA("u", 1728) "}" ::"r"(d),
                 "r"(a_lo), "r"(a_hi), "r"(b_lo), "r"(b_hi), "r"(idesc), "r"(q1), "r"(dx1), "r"(dx2)
                 : "memory");
#undef DW_MMA
}
// 16 accumulator columns of this thread's lane <- v
__device__ __forceinline__ void tmem_st16(uint32_t taddr, const int (&v)[16]) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16};" ::"r"(taddr),
                 "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]), "r"(v[8]), "r"(v[9]), "r"(v[10]),
                 "r"(v[11]), "r"(v[12]), "r"(v[13]), "r"(v[14]), "r"(v[15])
                 : "memory");
}
__device__ __forceinline__ void tmem_st_wait() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

template <bool SGN>
__device__ __forceinline__ uint4 dw_pack16(const int (&v)[16], int s) {
    uint32_t o[4];
#pragma unroll
    for (int g = 0; g < 4; ++g) {
        int t[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            t[k] = v[4 * g + k] >> s;
            if (SGN) t[k] = max(t[k], -127);
        }
        uint32_t hi2;
        if (SGN) {
            asm("cvt.pack.sat.s8.s32.b32 %0, %1, %2, 0;" : "=r"(hi2) : "r"(t[3]), "r"(t[2]));
            asm("cvt.pack.sat.s8.s32.b32 %0, %1, %2, %3;" : "=r"(o[g]) : "r"(t[1]), "r"(t[0]), "r"(hi2));
        } else {
            asm("cvt.pack.sat.u8.s32.b32 %0, %1, %2, 0;" : "=r"(hi2) : "r"(t[3]), "r"(t[2]));
            asm("cvt.pack.sat.u8.s32.b32 %0, %1, %2, %3;" : "=r"(o[g]) : "r"(t[1]), "r"(t[0]), "r"(hi2));
        }
    }
    return make_uint4(o[0], o[1], o[2], o[3]);
}

// A CTA's run of output rows, cut where an image group ends: rows y0 .. y1 - 1 of group `g`, input rows ya .. yb.
struct DwSegment {
    int g, y0, y1, ya, yb;
};
__device__ __forceinline__ DwSegment dw_segment(const DwParams &p, int row, int end) {
    DwSegment s;
    s.g = row / p.ho;
    s.y0 = row - s.g * p.ho;
    s.y1 = min(p.ho, s.y0 + end - row);
    s.ya = max(s.y0 * p.stride - 1, 0);
    s.yb = min((s.y1 - 1) * p.stride + 1, p.h - 1);
    return s;
}

template <bool SGN>
__global__ void __launch_bounds__(DW_THREADS, 1)
f8_dw_tc_kernel(const __grid_constant__ CUtensorMap map_a, const __grid_constant__ CUtensorMap map_e, const __grid_constant__ CUtensorMap map_y,
                const DwParams p) {
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem_aligned = (uint8_t *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    DwControl &ctl = *(DwControl *)smem_aligned;
    uint8_t *smem = smem_aligned + DW_CONTROL_BYTES;
    const int warp = uniform((int)(threadIdx.x >> 5)), lane = threadIdx.x & 31;
    const uint32_t smem_base = smem_u32(smem);
    const uint32_t full_bar = smem_u32(&ctl.full[0]), empty_bar = smem_u32(&ctl.empty[0]);
    const uint32_t acc_full = smem_u32(&ctl.acc_full[0]), acc_free = smem_u32(&ctl.acc_free[0]);
    const uint32_t out_full = smem_u32(&ctl.out_full[0]), out_free = smem_u32(&ctl.out_free[0]);
    // this CTA's slab and run of output rows
    const int slab = (int)blockIdx.x % p.slabs, wi = (int)blockIdx.x / p.slabs;
    const int ch0 = slab * p.slab_w, rows = p.groups * p.ho;
    const int row0 = (int)((long long)rows * wi / p.per_slab), row1 = (int)((long long)rows * (wi + 1) / p.per_slab);

    if (threadIdx.x == 32) {
        prefetch_tensormap(&map_a);
        if (p.stride == 2) prefetch_tensormap(&map_e);
        prefetch_tensormap(&map_y);
    }
    if (threadIdx.x == 0) {
        ctl.abort_flag = 0;
        for (int i = 0; i < DW_MAX_STAGES; ++i) {
            mbar_init(full_bar + 8 * i, 1);
            mbar_init(empty_bar + 8 * i, 2);
        }
        for (int i = 0; i < DW_RING; ++i) {
            mbar_init(acc_full + 8 * i, 2);
            mbar_init(acc_free + 8 * i, DW_EPI_WARPS / 2);
        }
        for (int i = 0; i < DW_OUT; ++i) {
            mbar_init(out_full + 8 * i, DW_EPI_WARPS / 2);
            mbar_init(out_free + 8 * i, 1);
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    // this thread's weights, asked for ahead of everything that waits
    uint8_t tap[2];
#pragma unroll
    for (int j = 0; j < 2; ++j) {
        const int i = threadIdx.x + j * DW_THREADS, t = i / DW_M, ch = ch0 + (i & (p.slab_w - 1));
        tap[j] = i < 9 * DW_M && ch < p.c ? (uint8_t)__ldg(p.w + ch * 9 + t) : (uint8_t)0;
    }
    int bias0 = 0;
    if (threadIdx.x < DW_M) {
        const int ch = ch0 + (threadIdx.x & (p.slab_w - 1));
        if (p.bias && ch < p.c) bias0 = __ldg(p.bias + ch);
    }
    if (warp == DW_MMA_WARP) tmem_alloc(smem_u32(&ctl.tmem_base_slot), 512);
    for (int i = threadIdx.x; i < (int)(DW_DIAG_BYTES / 16); i += DW_THREADS) *(uint4 *)(smem + p.diag_off + 16 * i) = make_uint4(0, 0, 0, 0);
    __syncthreads();
    // the diagonals: channel k of block q, filter tap (r, s): row 32 * pos(r) + k of the blocks of tap s.  pos: stride 1 rows 2, 1, 0 from
    // the top (an input row's output rows in ascending order), stride 2 rows 2, 0 (an odd input row), then 1 (an even one)
#pragma unroll
    for (int j = 0; j < 2; ++j) {
        const int i = threadIdx.x + j * DW_THREADS, t = i / DW_M, b = i & (DW_M - 1), k = b & 31, q = b >> 5, r = t / 3, s = t - 3 * r;
        const int pos = p.stride == 1 ? 2 - r : (r == 2 ? 0 : (r == 0 ? 1 : 2)), n = 32 * pos + k;
        if (i < 9 * DW_M)
            smem[p.diag_off + (uint32_t)(s * 4 + q) * DW_B_BYTES + (uint32_t)(k >> 4) * DW_B_LBO + (uint32_t)n * 16u + (uint32_t)(k & 15)] = tap[j];
    }
    // bias' = bias + 2^(s - 1), the starting value of every accumulator
    if (threadIdx.x < DW_M) *(int *)(smem + p.bias_off + 4 * threadIdx.x) = bias0 + (1 << (p.s - 1));
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");      // the tensor core reads them through the async proxy
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = uniform(ctl.tmem_base_slot);
    grid_launch_dependents();
    const WaitCtx wc = make_wait_ctx(&ctl.abort_flag, p.status, p.wait_limit);
    const int tagbits = p.tag << 8;
    const int sub = 128 / p.slab_w;                                   // image groups side by side
    const uint32_t sub_bytes = DW_M * (uint32_t)p.slab_w;

    if (warp == DW_A_WARP) {
        // ------------------------------------------------------------------ activations
        grid_dependency_wait();
        bool ok = true, have_last = false;
        int stage = 0, last_stage = 0;
        uint32_t par = 0, last_par = 0;
        for (int row = row0; ok && row < row1;) {
            const DwSegment s = dw_segment(p, row, row1);
            for (int y = s.ya; y <= s.yb; ++y) {
                if (!warp_wait(empty_bar + 8 * stage, par ^ 1u, wc, tagbits | 131)) { ok = false; break; }
                const uint32_t fb = full_bar + 8 * stage, dst = smem_base + (uint32_t)stage * p.stage_bytes;
                warp_expect_tx(fb, p.tx_bytes);
                for (int i = 0; i < sub; ++i) {
                    const int img = (s.g * sub + i) * p.images;
                    tma_load_4d(dst + (uint32_t)i * sub_bytes, &map_a, fb, ch0, -1, y, img, lane == 0);
                    if (p.stride == 2) tma_load_4d(dst + DW_TILE_BYTES + (uint32_t)i * sub_bytes, &map_e, fb, ch0, 0, y, img, lane == 0);
                }
                have_last = true;
                last_stage = stage;
                last_par = par;
                if (++stage == p.stages) { stage = 0; par ^= 1u; }
            }
            row += s.y1 - s.y0;
        }
        if (!ok && have_last) {
            const unsigned long long t0 = clock64();
            while (!mbar_try_wait(full_bar + 8 * last_stage, last_par) && (unsigned long long)(clock64() - t0) < DRAIN_LIMIT_CYCLES) {
            }
        }
    } else if (warp == DW_MMA_WARP || warp == DW_MMA2_WARP) {
        // ------------------------------------------------------------------ issuers, two blocks each
        const uint32_t half = warp == DW_MMA_WARP ? 0u : 1u;
        const uint64_t a_desc = smem_desc_hi(p.slab_w);
        const uint32_t a_lo0 = ((uint32_t)a_desc | ((smem_base & 0x3ffffu) >> 4)) + half * p.q2, a_hi = (uint32_t)(a_desc >> 32);
        const uint32_t b_lo0 = ((DW_B_LBO >> 4) << 16) | (((smem_base + p.diag_off + half * 2u * DW_B_BYTES) & 0x3ffffu) >> 4), b_hi = (128u >> 4) | (1u << 14);
        const uint32_t stage16 = p.stage_bytes >> 4;
        bool ok = true;
        int stage = 0, uses = 0, v0 = 0;            // v0: number (in this CTA's run) of the segment's first output row
        uint32_t par = 0;
        for (int row = row0; ok && row < row1;) {
            const DwSegment s = dw_segment(p, row, row1);
            int fresh = s.y0, done = s.y0;          // first output row without a contribution yet / not complete yet
            for (int y = s.ya; ok && y <= s.yb; ++y, ++uses) {
                // output rows lo .. hi take this input row, with the diagonal blocks from `blk` on
                int lo, hi, blk;
                if (p.stride == 1) {
                    lo = max(y - 1, s.y0);
                    hi = min(y + 1, s.y1 - 1);
                    blk = lo - (y - 1);
                } else if (y & 1) {
                    lo = max(y >> 1, s.y0);
                    hi = min((y >> 1) + 1, s.y1 - 1);
                    blk = lo - (y >> 1);
                } else {
                    lo = hi = y >> 1;
                    blk = 2;
                }
                for (; fresh <= hi; ++fresh) {
                    const int v = v0 + fresh - s.y0;
                    if (!warp_wait(acc_free + 8 * (v & 3), (uint32_t)(v >> 2) & 1u, wc, tagbits | 132)) { ok = false; break; }
                }
                ok = ok && warp_wait(full_bar + 8 * stage, par, wc, tagbits | 133);
                if (!ok) break;
                tc_fence_after();
                const uint32_t a_lo = a_lo0 + (uint32_t)stage * stage16;
                int n = hi - lo + 1;
                uint32_t slot = (uint32_t)(v0 + lo - s.y0) & 3u, b_lo = b_lo0 + 32u * (uint32_t)blk;      // a block: 512 bytes
                while (n > 0) {
                    const int now = min(n, DW_RING - (int)slot);
                    dw_mma6(tmem_base + 256u * half + 32u * slot, a_lo, a_hi, p.q1, p.dx1, p.dx2, b_lo, b_hi, p.idesc | ((uint32_t)(4 * now) << 17));
                    n -= now;
                    slot = 0;
                    b_lo += 32u * (uint32_t)now;
                }
                mma_commit(empty_bar + 8 * stage);
                if (++stage == p.stages) { stage = 0; par ^= 1u; }
                const int complete = y == s.yb ? s.y1 : (p.stride == 1 ? y : (y + 1) >> 1);      // rows below this one are complete
                for (; done < complete; ++done) mma_commit(acc_full + 8 * ((v0 + done - s.y0) & 3));
            }
            v0 += s.y1 - s.y0;
            row += s.y1 - s.y0;
        }
        if (ok)      // the releases of the last stage uses, which nobody else waits for, must land before the CTA goes
            for (int g = max(0, uses - p.stages); g < uses; ++g)
                warp_wait(empty_bar + 8 * (g % p.stages), (uint32_t)(g / p.stages) & 1u, wc, tagbits | 134);
    } else if (warp == DW_MOVER_WARP) {
        // ------------------------------------------------------------------ output mover
        grid_dependency_wait();
        int b = 0;
        uint32_t par = 0;
        for (int row = row0; row < row1; ++row) {
            if (!warp_wait(out_full + 8 * b, par, wc, tagbits | 135)) break;
            const int g = row / p.ho, y = row - g * p.ho;
            const uint32_t src = smem_base + p.out_off + (uint32_t)b * DW_TILE_BYTES;
            for (int i = 0; i < sub; ++i) {
                const int img = (g * sub + i) * p.images;
                if (img < p.n) tma_store_4d(&map_y, src + (uint32_t)i * sub_bytes, ch0, 0, y, img);
            }
            tma_store_commit();
            // the row before has been read out once at most this one's stores are left
            asm volatile("{\n\t" F8_ELECT "@e cp.async.bulk.wait_group.read 1;\n\t}" ::: "memory");
            __syncwarp();
            if (row > row0) warp_arrive(out_free + 8 * ((b + DW_OUT - 1) % DW_OUT));
            if (++b == DW_OUT) { b = 0; par ^= 1u; }
        }
        tma_store_wait();
    } else if (warp >= DW_FIRST_EPI) {
        // ------------------------------------------------------------------ epilogue warps
        // Two groups of eight take the rows in turn, so that one converts while the other waits for its accumulators or a staging buffer
        // (all sixteen on every row, in step with one another: 1280 cycles a row)
        const int quarter = warp & 3, group = (warp - DW_FIRST_EPI) >> 3, half = ((warp - DW_FIRST_EPI) >> 2) & 1;
        const uint32_t t_addr = tmem_base + ((uint32_t)(quarter * 32) << 16) + 256u * (uint32_t)half;      // TMEM lanes 32 * quarter .. + 31, two blocks
        const uint32_t bias_s = smem_base + p.bias_off + 256u * (uint32_t)half;
        auto load_bias = [&](int chunk, int (&v)[16]) {
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const uint4 w = lds128(bias_s + 64u * (uint32_t)chunk + 16u * j);
                v[4 * j] = (int)w.x; v[4 * j + 1] = (int)w.y; v[4 * j + 2] = (int)w.z; v[4 * j + 3] = (int)w.w;
            }
        };
        {
            int b0[16];
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                load_bias(c, b0);
                for (int i = group; i < DW_RING; i += 2) tmem_st16(t_addr + 128 * (c >> 1) + 32 * i + 16 * (c & 1), b0);
            }
        }
        tmem_st_wait();
        tc_fence_before();
        __syncwarp();
        if (lane == 0)
            for (int i = group; i < DW_RING; i += 2) mbar_arrive(acc_free + 8 * i);
        const int m = quarter * 32 + lane;
        uint32_t off[4];
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const int byte = 64 * half + 16 * c;
            off[c] = (uint32_t)(byte / p.slab_w) * sub_bytes + (uint32_t)(m * p.slab_w) + (uint32_t)(byte & (p.slab_w - 1));
            off[c] ^= ((off[c] >> 7) & p.swz_mask) << 4;
        }
        const int n_rows = row1 - row0;
        int ob = group;
        uint32_t opar = 0;
        for (int v = group; v < n_rows; v += 2) {
            if (!warp_wait(out_free + 8 * ob, opar ^ 1u, wc, tagbits | 137)) break;
            if (!warp_wait(acc_full + 8 * (v & 3), (uint32_t)(v >> 2) & 1u, wc, tagbits | 136)) break;
            tc_fence_after();
            const uint32_t t = t_addr + 32u * (uint32_t)(v & 3), dst = smem_base + p.out_off + (uint32_t)ob * DW_TILE_BYTES;
#pragma unroll
            for (int c = 0; c < 4; c += 2) {
                int va[16], vb[16], bias[16];
                tmem_ld16(t + 64 * c, va);
                tmem_ld16(t + 64 * c + 16, vb);
                load_bias(c, bias);
                tmem_ld_wait16(va);
                tmem_ld_wait16(vb);
                tmem_st16(t + 64 * c, bias);
                load_bias(c + 1, bias);
                tmem_st16(t + 64 * c + 16, bias);
                if (c == 2) {
                    tmem_st_wait();
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(acc_free + 8 * (v & 3));
                }
                sts128(dst + off[c], dw_pack16<SGN>(va, p.s));
                sts128(dst + off[c + 1], dw_pack16<SGN>(vb, p.s));
            }
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            __syncwarp();
            if (lane == 0) mbar_arrive(out_full + 8 * ob);
            ob += 2;
            if (ob >= DW_OUT) { ob -= DW_OUT; opar ^= 1u; }
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
    if (warp == DW_MMA_WARP) {
        tc_fence_after();
        tmem_dealloc(tmem_base, 512);
    }
}

// ----------------------------------------------------------------------------- host side

PFN_cuTensorMapEncodeTiled_v12000 dw_encode_tiled = nullptr;

bool dw_load_driver_entry_point() {
    if (dw_encode_tiled) return true;
    void *f = nullptr;
    cudaDriverEntryPointQueryResult qr;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &f, cudaEnableDefault, &qr) != cudaSuccess || !f || qr != cudaDriverEntryPointSuccess) return false;
    dw_encode_tiled = (PFN_cuTensorMapEncodeTiled_v12000)f;
    return true;
}

// How channels, images and rows are cut.
void dw_layout(const F8ConvGeom &g, DwParams *p) {
    // the slab that pads the channels least, of those the widest
    int best = 0;
    for (int w = 128; w >= 32; w >>= 1) {
        const int padded = (g.c + w - 1) / w * w;
        if (best == 0 || padded < best) {
            best = padded;
            p->slab_w = w;
        }
    }
    p->slabs = best / p->slab_w;
    p->pitch = g.stride_h == 1 ? g.wo + 2 : g.wo + 1;
    p->images = std::min(DW_M / p->pitch, g.n);
    const int per_group = p->images * (128 / p->slab_w);
    p->groups = (g.n + per_group - 1) / per_group;
}

}   // namespace

struct F8DwPlan {
    CUtensorMap map_a, map_e, map_y;
    DwParams p;
    int grid;
    size_t smem;
    int sgn;
};

size_t f8_dw_tc_plan_size() { return sizeof(F8DwPlan); }
void f8_dw_tc_plan_set_tag(F8DwPlan *plan, int tag) { plan->p.tag = tag; }

bool f8_dw_tc_supported(const F8ConvGeom &g, const F8Requant &q) {
    if (g.c != g.c_out || g.c % 16 != 0 || g.kh != 3 || g.kw != 3 || g.pad_h != 1 || g.pad_w != 1 || g.pad_h_end >= 0) return false;
    if (g.stride_h != g.stride_w || g.stride_h < 1 || g.stride_h > 2 || g.n < 1) return false;
    if ((g.stride_h == 1 ? g.wo + 2 : g.wo + 1) > DW_M || (g.stride_h == 2 && g.w < 2)) return false;
    if (g.c > 32 * 148 || (long long)g.n * g.ho > 0x7fffff00ll) return false;
    return (q.y_kind == F8_U8 || q.y_kind == F8_S8) && !q.has_res && q.sh_acc == 0 && q.s >= 1 && q.s <= 24;
}

// Setting up the diagonal blocks and filling the pipeline takes about 2 us more than the CUDA-core kernels need to start; per output
// this kernel is the faster one.  Whole networks with the line at 0.8, 1.6 and 3.5 million outputs, pairs not fused: MobileNet V1 at
// batch 16 170.8, 169.5, 182.9 us, MobileNet V2 at batch 16 313.1, 300.5, 300.9 us, at batch 64 487.8, 487.6, 500.0 us.
// That is with rows that fill the 128 positions of a tile.  A tile row costs the same however many of them hold an output, and the
// CUDA cores take about 0.55 (stride 2: 1.1) us per million outputs: 64 x 64 x 1200 at batch 64 (one image of 66 positions per
// block) 239.6 us here, 183.2 there; 78 x 78 x 48 at batch 221 52.8 and 41.2; stride 2, 98 x 98 x 1232 for one image 24.0 and 9.8.
// Both sides were timed for 400 layers of 16 - 1600 channels; the estimates are of the longest run of a CTA.
bool f8_dw_tc_wanted(const F8ConvGeom &g) {
    const double outputs = (double)g.n * g.ho * g.wo * g.c;
    if (outputs < 1.6e6) return false;
    DwParams p;
    dw_layout(g, &p);
    const long long rows = (long long)p.groups * g.ho, per_slab = std::min<long long>(std::max(1, 148 / p.slabs), rows);
    const double run = (double)((rows + per_slab - 1) / per_slab), filled = (double)(p.pitch * p.images) / DW_M;
    // (slabs of 32 channels whose pixels do not start at whole 32-byte sectors move more of them)
    const bool split = p.slab_w == 32 && g.c % 32 != 0;
    if (g.stride_h == 1) return 0.83 * (split ? 1.2 : 1.0) * run < 4.0 + 0.52e-6 * outputs;
    return (0.55 + 1.45 * filled) * (split ? 1.3 : 1.0) * run < 4.0 + 1.1e-6 * outputs;
}

cudaError_t f8_dw_tc_plan_init(F8DwPlan *plan, const F8ConvGeom &g, const F8Requant &q, const void *x, const int8_t *w, const int32_t *bias, void *y,
                               int *status_word, const char **why) {
    *why = "";
    if (!dw_load_driver_entry_point()) {
        *why = "cuTensorMapEncodeTiled not available";
        return cudaErrorNotSupported;
    }
    if (!f8_dw_tc_supported(g, q)) {
        *why = "shape outside the kernel's range";
        return cudaErrorInvalidValue;
    }
    memset(plan, 0, sizeof(*plan));
    DwParams &p = plan->p;
    p.n = g.n; p.h = g.h; p.ho = g.ho; p.c = g.c; p.stride = g.stride_h;
    dw_layout(g, &p);
    int dev = 0, sms = 148;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    p.per_slab = (int)std::min<long long>(std::max(1, sms / p.slabs), (long long)p.groups * g.ho);
    plan->grid = p.slabs * p.per_slab;
    const int two = g.stride_h == 2 ? 2 : 1;
    p.stages = two == 2 ? 3 : DW_MAX_STAGES;
    p.stage_bytes = two * DW_TILE_BYTES;
    const uint32_t box_rows = (uint32_t)(p.pitch * p.images);
    p.tx_bytes = (uint32_t)two * 128u * box_rows;
    const uint32_t row16 = (uint32_t)p.slab_w >> 4, sub16 = (DW_M * (uint32_t)p.slab_w) >> 4;
    p.dx1 = two == 2 ? DW_TILE_BYTES >> 4 : row16;
    p.dx2 = two == 2 ? row16 : 2 * row16;
    p.q1 = p.slab_w >= 64 ? 2u : sub16;
    p.q2 = p.slab_w == 128 ? 4u : (p.slab_w == 64 ? sub16 : 2 * sub16);
    p.swz_mask = p.slab_w == 128 ? 7u : (p.slab_w == 64 ? 3u : 1u);
    p.diag_off = (uint32_t)p.stages * p.stage_bytes;       // (the last rows of a shifted tile are read from behind it and not used)
    p.bias_off = p.diag_off + DW_DIAG_BYTES;
    p.out_off = (p.bias_off + 4 * DW_M + 1023) / 1024 * 1024;
    plan->smem = DW_CONTROL_BYTES + 1024 + p.out_off + DW_OUT * DW_TILE_BYTES;
    p.idesc = (2u << 4) | ((g.x_signed ? 1u : 0u) << 7) | (1u << 10) | ((uint32_t)(DW_M >> 4) << 24);
    p.w = w; p.bias = bias; p.s = q.s;
    p.status = status_word;
    p.wait_limit = f8_wait_limit_cycles();
    plan->sgn = q.y_kind == F8_S8 ? 1 : 0;
    const CUtensorMapSwizzle sw = p.slab_w == 128 ? CU_TENSOR_MAP_SWIZZLE_128B : (p.slab_w == 64 ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_32B);
    cuuint32_t ones[4] = {1, 1, 1, 1};
    const cuuint32_t box[4] = {(cuuint32_t)p.slab_w, (cuuint32_t)p.pitch, 1, (cuuint32_t)p.images};
    // stride 1: the input; stride 2: its odd columns (map_a, from column -1 on) and its even ones (map_e)
    for (int e = 0; e < two; ++e) {
        const cuuint64_t cols = two == 1 ? (cuuint64_t)g.w : (cuuint64_t)(e ? (g.w + 1) / 2 : g.w / 2);
        const cuuint64_t dims[4] = {(cuuint64_t)g.c, cols, (cuuint64_t)g.h, (cuuint64_t)g.n};
        const cuuint64_t strides[3] = {(cuuint64_t)g.c * two, (cuuint64_t)g.c * g.w, (cuuint64_t)g.c * g.w * g.h};
        uint8_t *base = (uint8_t *)const_cast<void *>(x) + (two == 2 && !e ? g.c : 0);
        if (dw_encode_tiled(e ? &plan->map_e : &plan->map_a, CU_TENSOR_MAP_DATA_TYPE_UINT8, 4, base, dims, strides, box, ones, CU_TENSOR_MAP_INTERLEAVE_NONE,
                            sw, CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS) {
            *why = "cuTensorMapEncodeTiled rejected the activation tensor";
            return cudaErrorInvalidValue;
        }
    }
    if (two == 1) plan->map_e = plan->map_a;
    {
        const cuuint64_t dims[4] = {(cuuint64_t)g.c, (cuuint64_t)g.wo, (cuuint64_t)g.ho, (cuuint64_t)g.n};
        const cuuint64_t strides[3] = {(cuuint64_t)g.c, (cuuint64_t)g.c * g.wo, (cuuint64_t)g.c * g.wo * g.ho};
        if (dw_encode_tiled(&plan->map_y, CU_TENSOR_MAP_DATA_TYPE_UINT8, 4, y, dims, strides, box, ones, CU_TENSOR_MAP_INTERLEAVE_NONE, sw,
                            CU_TENSOR_MAP_L2_PROMOTION_NONE, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS) {
            *why = "cuTensorMapEncodeTiled rejected the output tensor";
            return cudaErrorInvalidValue;
        }
    }
    static bool attr_set[64] = {false};
    if (dev < 0 || dev >= 64) {
        *why = "device index out of range";
        return cudaErrorInvalidDevice;
    }
    if (!attr_set[dev]) {
        cudaError_t e = cudaFuncSetAttribute(f8_dw_tc_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
        if (e == cudaSuccess) e = cudaFuncSetAttribute(f8_dw_tc_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
        if (e != cudaSuccess) {
            *why = "cudaFuncSetAttribute(MaxDynamicSharedMemorySize) failed";
            return e;
        }
        attr_set[dev] = true;
    }
    return cudaSuccess;
}

cudaError_t f8_dw_tc_launch(const F8DwPlan *plan, bool overlap_previous, cudaStream_t st) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)plan->grid);
    cfg.blockDim = dim3(DW_THREADS);
    cfg.dynamicSmemBytes = plan->smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = overlap_previous ? 1 : 0;
    if (plan->sgn) return cudaLaunchKernelEx(&cfg, f8_dw_tc_kernel<true>, plan->map_a, plan->map_e, plan->map_y, plan->p);
    return cudaLaunchKernelEx(&cfg, f8_dw_tc_kernel<false>, plan->map_a, plan->map_e, plan->map_y, plan->p);
}

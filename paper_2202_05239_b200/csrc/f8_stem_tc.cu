// First layer of an image network on the tensor cores: a kh x kw convolution with stride 2 over an image with at
// most four channels (a2 - a4 fused: bias, rounding shift, clip), optionally followed in the same kernel by the
// 3x3 / stride 2 / pad 1 max pool that ResNet-style networks put behind it.
//
// The layer is a GEMM with a tiny K (7 x 7 x 3 = 147) and a huge M, and its input rows overlap heavily, so it is
// organised around the image rather than around an im2col gather:
//   * A CTA walks down a band of output rows.  For every PAIR of image rows it builds, in shared memory, a line of
//     8-byte cells: cell `col` holds pixel col - pad of both rows (4 bytes each, zero filled).  The kw-tap window
//     of output column ox over that row pair is then the 8 * kw bytes that start at cell 2 * ox, i.e. at byte
//     16 * ox: windows of neighbouring outputs overlap and are 16 bytes apart.
//   * That is exactly a K-major operand without swizzle whose 8 x 16-byte core matrices are 128 contiguous bytes
//     (row pitch 16 bytes), with 16 bytes between core matrices along K and 128 bytes between 8-row groups: the
//     tensor core reads the overlapping windows straight from the line, nothing is expanded.  One output row
//     (up to 128 pixels = the M of one tcgen05.mma) takes `kh2` row pairs x (window bytes / 32) instructions.
//   * The weights ([K / 16][c_out][16] bytes, the same core-matrix form) stay in shared memory.
//   * Two accumulators in tensor memory: the MMAs of row oy + 1 run while eight warps requantise row oy into a
//     ring of three finished rows, from which either the row itself or, every second row, one pooled row is
//     written to global memory with 16-byte accesses.
// The CTA is synchronised with two block barriers per row and one mbarrier wait (bounded) for the accumulator;
// several CTAs share an SM and fill each other's gaps.
#include <limits.h>

#include <algorithm>
#include <stdio.h>
#include <stdlib.h>

#include "f8_epilogue.cuh"
#include "f8_tc_ptx.cuh"

namespace {

constexpr int STEM_EPI_WARPS = 8;
constexpr int STEM_THREADS = 32 * (STEM_EPI_WARPS + 1);     // warp 8 issues the MMAs
constexpr int STEM_PAIR_SLOTS = 8;                           // ring of packed row pairs (a window needs <= 7, plus one)
constexpr int STEM_SLOT_BYTES = 2176;                        // 128 windows 16 bytes apart, 64 bytes long, rounded up
constexpr int STEM_MAX_CELLS = 264;                          // cells a slot can hold (2112 bytes)

struct StemParams {
    int n, h, w, c;            // image, c <= 4
    int ho, wo, c_out;         // convolution output, wo <= 128
    int kh2;                   // row pairs one window covers
    int top;                   // the first pair of output row oy is oy - top
    int left;                  // zero cells in front of a line (the left padding)
    int hp;                    // row pairs per image
    int slices;                // 32-byte K slices per row pair
    int ncell;                 // cells of a line that can reach a valid output
    int pool;                  // 1: write the 3x3 / 2 / pad 1 max pool of the layer's output instead of the output
    int po, pwo;               // pooled height / width
    int rows_per_img;          // po or ho: output rows this launch writes per image
    int acc_cols;              // TMEM columns of one accumulator
    int cpr;                   // 16-byte chunks per output pixel (c_out / 16)
    int swz_shift, swz_mask;   // chunk swizzle of the finished-row ring: chunk ^ ((px >> shift) & mask)
    uint32_t idesc;
    uint32_t a_desc_hi, b_desc_hi;   // upper descriptor words (byte offsets between core matrices)
    uint32_t a_desc_lbo_sbo, b_desc_lbo_sbo;   // bits 16.. of the lower word (leading byte offset)
    int s;                     // rounding shift, 1..24
    int signed_out;
    int x_signed;
    const uint8_t *x;
    const int8_t *wk;          // [K / 16][c_out][16]
    const int32_t *bias;
    uint8_t *y;
    int *status;
    int tag;
    unsigned long long wait_limit;   // bound of the accumulator wait in SM cycles (0: the default)
};

__device__ __forceinline__ uint32_t ldg32(const uint8_t *p) { return __ldg((const uint32_t *)p); }

// The (up to four) channel bytes of the pixel that starts `off` bytes into the image tensor, zero extended to 32 bits.
// FAST: the tensor is 4-byte aligned and a multiple of 4 bytes long, so aligned words may be read up to its last one.
template <bool FAST>
__device__ __forceinline__ uint32_t load_pixel(const uint8_t *x, uint32_t off, uint32_t last_word, int c) {
    if (FAST) {
        if (c == 4) return ldg32(x + off);
        const uint32_t a = off & ~3u;
        const uint32_t w0 = ldg32(x + a), w1 = ldg32(x + min(a + 4u, last_word));
        return __funnelshift_r(w0, w1, (off & 3u) * 8u) & (0xffffffffu >> (32 - 8 * c));
    }
    uint32_t word = 0;
#pragma unroll
    for (int ch = 0; ch < 4; ++ch)
        if (ch < c) word |= (uint32_t)__ldg(x + off + ch) << (8 * ch);
    return word;
}

// The one or two K slices of a row pair, issued by a lone thread or (WARP) by the elected lane of a whole warp, see mma_commit().
template <bool WARP>
__device__ __forceinline__ void stem_mma_pair(uint32_t d_tmem, uint32_t a_lo, uint32_t b_lo, const StemParams &p, uint32_t b_slice,
                                              uint32_t accumulate) {
#define STEM_TWO(elect, on) \
    asm volatile("{\n\t" elect ".reg .pred p, t;\n\t.reg .b64 a, b;\n\t.reg .b32 x, y;\n\t" \
                 "setp.ne.b32 p, %7, 0;\n\tsetp.eq.b32 t, 0, 0;\n\tmov.b64 a, {%1, %3};\n\tmov.b64 b, {%2, %4};\n\t" \
                 on "tcgen05.mma.cta_group::1.kind::i8 [%0], a, b, %6, p;\n\t" \
                 "add.u32 x, %1, 2;\n\tadd.u32 y, %2, %5;\n\tmov.b64 a, {x, %3};\n\tmov.b64 b, {y, %4};\n\t" \
                 on "tcgen05.mma.cta_group::1.kind::i8 [%0], a, b, %6, t;\n\t}" ::"r"(d_tmem), \
                 "r"(a_lo), "r"(b_lo), "r"(p.a_desc_hi), "r"(p.b_desc_hi), "r"(b_slice), "r"(p.idesc), "r"(accumulate) \
                 : "memory")
#define STEM_ONE(elect, on) \
    asm volatile("{\n\t" elect ".reg .pred p;\n\t.reg .b64 a, b;\n\tsetp.ne.b32 p, %6, 0;\n\t" \
                 "mov.b64 a, {%1, %3};\n\tmov.b64 b, {%2, %4};\n\t" \
                 on "tcgen05.mma.cta_group::1.kind::i8 [%0], a, b, %5, p;\n\t}" ::"r"(d_tmem), \
                 "r"(a_lo), "r"(b_lo), "r"(p.a_desc_hi), "r"(p.b_desc_hi), "r"(p.idesc), "r"(accumulate) \
                 : "memory")
    if (p.slices == 2) {
        if (WARP) STEM_TWO(F8_ELECT, "@e ");
        else STEM_TWO("", "");
    } else {
        if (WARP) STEM_ONE(F8_ELECT, "@e ");
        else STEM_ONE("", "");
    }
#undef STEM_TWO
#undef STEM_ONE
}

template <bool POOL, bool SIGNED, bool FAST>
__global__ void __launch_bounds__(STEM_THREADS, 3) f8_stem_tc_kernel(const StemParams p, const int grid_units_total) {
    extern __shared__ __align__(128) uint8_t smem[];
    __shared__ __align__(8) uint64_t acc_bar[2];
    __shared__ uint32_t tmem_base_slot;
    __shared__ int abort_flag;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int cpr = p.cpr;
    const uint32_t c_out = (uint32_t)cpr * 16u;
    const int k_bytes = p.kh2 * p.slices * 32;
    const uint32_t w_bytes = (uint32_t)k_bytes * c_out;
    const uint32_t row_bytes = 128u * c_out;
    const uint32_t smem_base = smem_u32(smem);
    const uint32_t pair_base = smem_base + w_bytes;
    const uint32_t rows_base = pair_base + STEM_PAIR_SLOTS * STEM_SLOT_BYTES;     // two finished / running-maximum rows
    const uint32_t bias_base = rows_base + 2 * row_bytes;
    uint8_t *const pair_ptr = smem + w_bytes;

    // ---- prologue (reads only parameters that no earlier work in the stream writes)
    {
        uint4 *z = (uint4 *)pair_ptr;     // cells past the image are never written again: they stay zero
        for (int i = threadIdx.x; i < STEM_PAIR_SLOTS * STEM_SLOT_BYTES / 16; i += STEM_THREADS) z[i] = make_uint4(0, 0, 0, 0);
        const uint4 *wg = (const uint4 *)p.wk;
        uint4 *ws = (uint4 *)smem;
        for (int i = threadIdx.x; i < (int)(w_bytes / 16); i += STEM_THREADS) ws[i] = __ldg(wg + i);
        int *bs = (int *)(smem + (bias_base - smem_base));
        const int rnd = 1 << (p.s - 1);
        for (int i = threadIdx.x; i < (int)c_out; i += STEM_THREADS) bs[i] = (p.bias ? __ldg(p.bias + i) : 0) + rnd;
    }
    if (threadIdx.x == 0) {
        abort_flag = 0;
        mbar_init(smem_u32(&acc_bar[0]), 1);
        mbar_init(smem_u32(&acc_bar[1]), 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == STEM_EPI_WARPS) tmem_alloc(smem_u32(&tmem_base_slot), (uint32_t)(2 * p.acc_cols));
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");     // weights: generic writes, read by the tensor core
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = tmem_base_slot;
    grid_launch_dependents();
    grid_dependency_wait();        // the image / the output buffer may belong to earlier work in the stream

    volatile int *abortp = &abort_flag;
    const WaitCtx wc = make_wait_ctx(&abort_flag, p.status, p.wait_limit);
    const int tagbits = p.tag << 8;
    const long long total = grid_units_total;
    const int u_begin = (int)(total * blockIdx.x / gridDim.x), u_end = (int)(total * (blockIdx.x + 1) / gridDim.x);
    const uint32_t rsel[4] = {0, 0, 0, 0};
    int k = 0;                       // rows issued so far by this CTA: accumulator k & 1, barrier parity (k >> 1) & 1

    // ---- per-thread constants
    // packing: this thread owns cell `col` (and col + STEM_THREADS) of every line
    const uint32_t img_row_bytes = (uint32_t)p.w * p.c;
    uint32_t cell_off[2];            // byte offset of the cell's pixel inside an image row
    bool cell_on[2], cell_px[2];     // the cell exists / holds a pixel (else zero padding)
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        const int col = threadIdx.x + i * STEM_THREADS, iw = col - p.left;
        cell_on[i] = col < p.ncell;
        cell_px[i] = cell_on[i] && iw >= 0 && iw < p.w;
        cell_off[i] = cell_px[i] ? (uint32_t)iw * p.c : 0u;
    }
    const uint32_t last_word = (uint32_t)p.n * p.h * img_row_bytes - 4u;
    // epilogue: this thread owns output pixel px and the 16-byte chunks [ch0, ch1) of it
    const int quarter = warp & 3, half = (warp >> 2) & 1;
    const int px = quarter * 32 + lane;
    const int ch_per = (cpr + 1) >> 1;
    const int ch0 = half * ch_per, ch1 = min(cpr, ch0 + ch_per);
    const uint32_t swz = ((uint32_t)px >> p.swz_shift) & (uint32_t)p.swz_mask;
    const uint32_t px_off = (uint32_t)px * c_out;

    auto load_cells = [&](int img, int pr, uint2 (&cell)[2]) {
        const uint32_t r0 = ((uint32_t)img * p.h + 2u * pr) * img_row_bytes;
        const bool second = 2 * pr + 1 < p.h;
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            cell[i] = make_uint2(0u, 0u);
            if (cell_px[i]) {
                cell[i].x = load_pixel<FAST>(p.x, r0 + cell_off[i], last_word, p.c);
                if (second) cell[i].y = load_pixel<FAST>(p.x, r0 + img_row_bytes + cell_off[i], last_word, p.c);
            }
        }
    };
    auto store_cells = [&](int pr, const uint2 (&cell)[2]) {
        uint2 *line = (uint2 *)(pair_ptr + (pr & (STEM_PAIR_SLOTS - 1)) * STEM_SLOT_BYTES);
#pragma unroll
        for (int i = 0; i < 2; ++i)
            if (cell_on[i]) line[threadIdx.x + i * STEM_THREADS] = cell[i];
    };
    // issue the MMAs of output row oy into accumulator kk & 1 (one thread: between this kernel's block barriers a whole warp that elects a
    // lane is slower, 4 -> 128 channels, 128 x 128, batch 128 55.8 against 54.5 us, 250 x 250 3 -> 96, batch 8 15.0 against 14.0)
    const uint32_t a_lo0 = p.a_desc_lbo_sbo | ((pair_base & 0x3ffffu) >> 4), b_lo0 = p.b_desc_lbo_sbo | ((smem_base & 0x3ffffu) >> 4);
    const uint32_t b_slice = 2u * c_out;                 // 16-byte units between the K slices of the weights
    auto issue_row = [&](int oy, int kk) {
        const uint32_t d_tmem = tmem_base + (uint32_t)((kk & 1) * p.acc_cols);
        uint32_t accumulate = 0;
        uint32_t b_lo = b_lo0;
        for (int j = 0; j < p.kh2; ++j, b_lo += b_slice * p.slices) {
            const int pr = oy - p.top + j;
            if (pr < 0 || pr >= p.hp) continue;          // rows above / below the image contribute nothing
            const uint32_t a_lo = a_lo0 + (uint32_t)(pr & (STEM_PAIR_SLOTS - 1)) * (STEM_SLOT_BYTES / 16);
            stem_mma_pair<false>(d_tmem, a_lo, b_lo, p, b_slice, accumulate);
            accumulate = 1;
        }
        mma_commit_thread(smem_u32(&acc_bar[kk & 1]));
    };

    for (int u = u_begin; u < u_end;) {
        const int img = u / p.rows_per_img, r0 = u - img * p.rows_per_img;
        const int r1 = min(p.rows_per_img, r0 + (u_end - u));            // rows [r0, r1) of this image are ours
        u += r1 - r0;
        const int oy_first = POOL ? max(0, 2 * r0 - 1) : r0;
        const int oy_last = POOL ? min(p.ho - 1, 2 * (r1 - 1) + 1) : r1 - 1;

        // ---- lines of the first row's window; the line the second row adds stays in registers for now
        uint2 cell[2];
        for (int j = 0; j < p.kh2; ++j) {
            const int pr = oy_first - p.top + j;
            if (pr < 0 || pr >= p.hp) continue;
            load_cells(img, pr, cell);
            store_cells(pr, cell);
        }
        {
            const int pn = oy_first + 1 - p.top + p.kh2 - 1;
            if (oy_first + 1 <= oy_last && pn >= 0 && pn < p.hp) load_cells(img, pn, cell);
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        __syncthreads();
        if (warp == STEM_EPI_WARPS) {
            if (lane == 0) {
                tc_fence_after();
                issue_row(oy_first, k);
            }
            __syncwarp();
        }

        for (int oy = oy_first; oy <= oy_last; ++oy, ++k) {
            // ---- the line that row oy + 1 adds to the window
            if (oy + 1 <= oy_last) {
                const int pn = oy + 1 - p.top + p.kh2 - 1;
                if (pn >= 0 && pn < p.hp) store_cells(pn, cell);
            }
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            __syncthreads();
            {
                // cells for the row after next: in flight while this row is converted
                const int pn2 = oy + 2 - p.top + p.kh2 - 1;
                if (oy + 2 <= oy_last && pn2 >= 0 && pn2 < p.hp) load_cells(img, pn2, cell);
            }
            // pooling: row oy closes the pooled row oy >> 1 when it is odd (or the last row) and opens the next one
            const bool closes = (oy & 1) || oy == p.ho - 1;
            // row 0 has no row above it: it starts the running maximum of pooled row 0 instead of joining one
            const bool opens = oy == 0;
            const int py = oy >> 1;
            if (warp == STEM_EPI_WARPS) {
                if (lane == 0 && oy + 1 <= oy_last) {
                    tc_fence_after();
                    issue_row(oy + 1, k + 1);
                }
                __syncwarp();
            } else {
                // ---- epilogue of row oy: thread = output pixel, 16 channels per accumulator load
                // the accumulator is usually a few hundred cycles away: sleep on the barrier (the hardware wakes the
                // thread when the phase completes or after the hinted time) before falling back to the bounded poll
                bool got = false;
#pragma unroll 1
                for (int t = 0; t < 4 && !got; ++t) got = mbar_try_wait_hint(smem_u32(&acc_bar[k & 1]), (uint32_t)(k >> 1) & 1u, 4000u);
                if (!got) got = mbar_wait(smem_u32(&acc_bar[k & 1]), (uint32_t)(k >> 1) & 1u, wc, tagbits | 120);
                if (__all_sync(0xffffffffu, got)) {
                    tc_fence_after();
                    const uint32_t t_addr = tmem_base + ((uint32_t)(quarter * 32) << 16) + (uint32_t)((k & 1) * p.acc_cols);
                    // POOL: buffer py & 1 holds the running maximum of the pooled row that is open
                    const uint32_t cur = rows_base + (POOL ? (uint32_t)(py & 1) * row_bytes : 0u) + px_off;
                    const uint32_t nxt = rows_base + (uint32_t)((py + 1) & 1) * row_bytes + px_off;
#pragma unroll
                    for (int ci = 0; ci < 8; ++ci) {
                        const int ch = ch0 + ci;
                        if (ch >= ch1) break;
                        int v[16];
                        tmem_ld16(t_addr + ch * 16, v);
                        tmem_ld_wait();
                        const uint4 o = epilogue_fast16<false, SIGNED>(v, bias_base + 64 * ch, make_uint4(0, 0, 0, 0), 1, 0, rsel, p.s);
                        const uint32_t co = ((uint32_t)ch ^ swz) << 4;
                        if (!POOL) {
                            sts128(cur + co, o);
                        } else {
                            uint4 m = o;
                            if (!opens) {
                                const uint4 t = lds128(cur + co);
                                m.x = SIGNED ? __vmaxs4(t.x, o.x) : __vmaxu4(t.x, o.x);
                                m.y = SIGNED ? __vmaxs4(t.y, o.y) : __vmaxu4(t.y, o.y);
                                m.z = SIGNED ? __vmaxs4(t.z, o.z) : __vmaxu4(t.z, o.z);
                                m.w = SIGNED ? __vmaxs4(t.w, o.w) : __vmaxu4(t.w, o.w);
                            }
                            sts128(cur + co, m);
                            if (oy & 1) sts128(nxt + co, o);      // an odd row is also the top row of the next pooled row
                        }
                    }
                    tc_fence_before();
                }
            }
            __syncthreads();
            if (*abortp) break;

            // ---- write: the finished row, or the pooled row it closes (maximum over three neighbouring columns)
            if (!POOL) {
                uint8_t *dst = p.y + ((size_t)img * p.ho + oy) * (size_t)p.wo * c_out;
                for (int it = threadIdx.x; it < p.wo * cpr; it += STEM_THREADS) {
                    const int x0 = it / cpr, ch = it - x0 * cpr;
                    const uint32_t sw = ((uint32_t)x0 >> p.swz_shift) & (uint32_t)p.swz_mask;
                    *(uint4 *)(dst + (size_t)it * 16) = lds128(rows_base + (uint32_t)x0 * c_out + (((uint32_t)ch ^ sw) << 4));
                }
            } else if (closes && py >= r0 && py < r1) {
                const uint32_t src = rows_base + (uint32_t)(py & 1) * row_bytes;
                uint8_t *dst = p.y + ((size_t)img * p.po + py) * (size_t)p.pwo * c_out;
                for (int it = threadIdx.x; it < p.pwo * cpr; it += STEM_THREADS) {
                    const int ppx = it / cpr, ch = it - ppx * cpr;
                    const int cx = 2 * ppx;
                    const uint32_t sw1 = ((uint32_t)cx >> p.swz_shift) & (uint32_t)p.swz_mask;
                    uint4 m = lds128(src + (uint32_t)cx * c_out + (((uint32_t)ch ^ sw1) << 4));
                    if (cx > 0) {
                        const uint32_t sw0 = ((uint32_t)(cx - 1) >> p.swz_shift) & (uint32_t)p.swz_mask;
                        const uint4 t = lds128(src + (uint32_t)(cx - 1) * c_out + (((uint32_t)ch ^ sw0) << 4));
                        m.x = SIGNED ? __vmaxs4(t.x, m.x) : __vmaxu4(t.x, m.x);
                        m.y = SIGNED ? __vmaxs4(t.y, m.y) : __vmaxu4(t.y, m.y);
                        m.z = SIGNED ? __vmaxs4(t.z, m.z) : __vmaxu4(t.z, m.z);
                        m.w = SIGNED ? __vmaxs4(t.w, m.w) : __vmaxu4(t.w, m.w);
                    }
                    if (cx + 1 < p.wo) {
                        const uint32_t sw2 = ((uint32_t)(cx + 1) >> p.swz_shift) & (uint32_t)p.swz_mask;
                        const uint4 t = lds128(src + (uint32_t)(cx + 1) * c_out + (((uint32_t)ch ^ sw2) << 4));
                        m.x = SIGNED ? __vmaxs4(t.x, m.x) : __vmaxu4(t.x, m.x);
                        m.y = SIGNED ? __vmaxs4(t.y, m.y) : __vmaxu4(t.y, m.y);
                        m.z = SIGNED ? __vmaxs4(t.z, m.z) : __vmaxu4(t.z, m.z);
                        m.w = SIGNED ? __vmaxs4(t.w, m.w) : __vmaxu4(t.w, m.w);
                    }
                    *(uint4 *)(dst + (size_t)it * 16) = m;
                }
            }
        }
        if (*abortp) break;
        __syncthreads();      // the buffers are reused by the next band: everybody is done reading
    }
    if (*abortp && threadIdx.x == 0) {
        // aborting: give the MMAs already issued time to finish before tensor memory is released
        const unsigned long long t0 = clock64();
        while (!mbar_try_wait(smem_u32(&acc_bar[k & 1]), (uint32_t)(k >> 1) & 1u) &&
               (unsigned long long)(clock64() - t0) < DRAIN_LIMIT_CYCLES) {
        }
    }

    tc_fence_before();
    __syncthreads();
    if (warp == STEM_EPI_WARPS) {
        tc_fence_after();
        tmem_dealloc(tmem_base, (uint32_t)(2 * p.acc_cols));
    }
}


// ----------------------------------------------------------------------------- layers of at most 64 channels

// The same layer with its roles on warps of their own, for up to 64 output channels (the stems of the networks here; wider
// ones keep the kernel above, whose accumulators fit tensor memory twice).  Three warps pack image lines, one warp issues the
// MMAs, eight warps convert; every hand-over is an mbarrier, so nobody waits at a block-wide barrier and three different
// steps are packed, multiplied and converted at once.
//   * A step is a pair of output rows (2r, 2r + 1).  Their windows overlap, so they are ONE multiplication with 2 c_out columns:
//     the weights of row 2r + 1 are those of row 2r one row pair further down (zeros where a row does not reach).  For the
//     7 x 7 stem that is 10 instructions of 128 columns instead of 16 of 64, which are bound by the tensor pipe's 50 cycles
//     per instruction, and half of the hand-overs.
//   * The rounding shift and the clip are monotone, so the pooling maximum over the three rows is taken on the 32-bit sums
//     (one three-operand maximum per value; the odd row that two pooled rows share stays in registers) and only one value
//     in two is requantised.
//   * The maximum over three columns works on 16-bit lanes of packed bytes: the high bytes of a lane decide whatever lies
//     below them, so a word costs two three-operand maxima and three shifts.
//   * Without a pool a thread stores its pixel's channels straight from registers.
//   * Three-channel rows of a multiple of four pixels are read four pixels at a time, from three words, instead of two words around
//     every pixel: half the loads, no shift by a variable amount.
// Measured (224 x 224 images, batch 256, B200): 7 x 7 to 64 channels with the pool 140 -> 82 us, with four pixels at a time 103 -> 91
// (timed inside a network); 3 x 3 to 32 channels without a pool 105 -> 62 us, 69.7 -> 54.6; one image 21 -> 17 us.  The pooling
// conversion is what bounds the first, the packing of the lines the second (a fourth packing warp: 97.6 and 57.8).
constexpr int ROWS_EPI_WARPS = 8;
constexpr int ROWS_PACK_WARPS = 3;
constexpr int ROWS_MMA_WARP = ROWS_EPI_WARPS + ROWS_PACK_WARPS;
constexpr int ROWS_THREADS = 32 * (ROWS_MMA_WARP + 1);
constexpr int ROWS_LINES = 16;                  // ring of packed row pairs
constexpr int ROWS_AHEAD = 4;                   // steps the packing may run ahead of the MMAs: a window of at most 8 pairs plus
                                                // three times two more lines fit the ring
constexpr int ROWS_ACCS = 2;
constexpr int ROWS_CELLS = (STEM_MAX_CELLS + 32 * ROWS_PACK_WARPS - 1) / (32 * ROWS_PACK_WARPS);       // of a line, per thread

// Bytewise maximum of three words.
template <bool SIGNED>
__device__ __forceinline__ uint32_t max3_bytes(uint32_t a, uint32_t b, uint32_t c) {
    const uint32_t hi = SIGNED ? __vimax3_s16x2(a, b, c) : __vimax3_u16x2(a, b, c);
    const uint32_t lo = SIGNED ? __vimax3_s16x2(a << 8, b << 8, c << 8) : __vimax3_u16x2(a << 8, b << 8, c << 8);
    return __byte_perm(hi, lo, 0x3715);
}

// How the packing warps read the image: byte by byte; the two aligned words around a pixel (FAST above); or, three channels and rows
// of a multiple of four pixels that start at a word, four pixels from three words.
constexpr int READ_BYTES = 0, READ_WORDS = 1, READ_QUADS = 2;
constexpr int ROWS_QUADS = (2 * STEM_MAX_CELLS / 4 + 32 * ROWS_PACK_WARPS - 1) / (32 * ROWS_PACK_WARPS);      // of two lines, per thread

// CH: 16-byte chunks per pixel this instantiation has registers for (2 or 4; p.cpr <= CH).
template <int CH, bool POOL, bool SIGNED, int READ>
__global__ void __launch_bounds__(ROWS_THREADS, 2) f8_stem_rows_tc_kernel(const StemParams p, const int units_total) {
    extern __shared__ __align__(128) uint8_t smem[];
    __shared__ __align__(8) uint64_t line_bars[ROWS_AHEAD];      // the lines a step adds have been packed
    __shared__ __align__(8) uint64_t done_bars[ROWS_AHEAD];      // a step's MMAs have completed
    __shared__ __align__(8) uint64_t free_bars[ROWS_ACCS];       // an accumulator has been read
    __shared__ uint32_t tmem_base_slot;
    __shared__ int abort_flag;

    const int warp = uniform((int)(threadIdx.x >> 5)), lane = threadIdx.x & 31;
    const uint32_t c_out = (uint32_t)p.cpr * 16u;
    const uint32_t w_bytes = (uint32_t)((p.kh2 + 1) * p.slices * 32) * 2u * c_out;
    const uint32_t row_bytes = 128u * c_out;
    const uint32_t smem_base = smem_u32(smem);
    const uint32_t line_base = smem_base + w_bytes;
    const uint32_t rows_base = line_base + ROWS_LINES * STEM_SLOT_BYTES;       // POOL: two rows of column-wise maxima
    const uint32_t bias_base = rows_base + (POOL ? 2 * row_bytes : 0u);
    uint8_t *const line_ptr = smem + w_bytes;

    {
        uint4 *z = (uint4 *)line_ptr;     // cells past the image are never written again: they stay zero
        for (int i = threadIdx.x; i < ROWS_LINES * STEM_SLOT_BYTES / 16; i += ROWS_THREADS) z[i] = make_uint4(0, 0, 0, 0);
        const uint4 *wg = (const uint4 *)p.wk;
        uint4 *ws = (uint4 *)smem;
        // [K / 16][2 c_out][16]: columns c_out.. are the same weights one row pair later
        const int pair_chunks = p.slices * 2, last_chunk = p.kh2 * pair_chunks;
#pragma unroll 4
        for (int i = threadIdx.x; i < (int)(w_bytes / 16); i += ROWS_THREADS) {
            const int kc = i / (2 * (int)c_out), n = i - kc * 2 * (int)c_out;
            const int src = n < (int)c_out ? kc : kc - pair_chunks;
            ws[i] = src >= 0 && src < last_chunk ? __ldg(wg + src * (int)c_out + (n < (int)c_out ? n : n - (int)c_out)) : make_uint4(0, 0, 0, 0);
        }
        int *bs = (int *)(smem + (bias_base - smem_base));
        const int rnd = 1 << (p.s - 1);
        for (int i = threadIdx.x; i < (int)c_out; i += ROWS_THREADS) bs[i] = (p.bias ? __ldg(p.bias + i) : 0) + rnd;
    }
    if (threadIdx.x == 0) {
        abort_flag = 0;
        for (int i = 0; i < ROWS_AHEAD; ++i) {
            mbar_init(smem_u32(&line_bars[i]), ROWS_PACK_WARPS);
            mbar_init(smem_u32(&done_bars[i]), 1);
        }
        for (int i = 0; i < ROWS_ACCS; ++i) mbar_init(smem_u32(&free_bars[i]), ROWS_EPI_WARPS);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == ROWS_MMA_WARP) tmem_alloc(smem_u32(&tmem_base_slot), (uint32_t)(ROWS_ACCS * p.acc_cols));
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");     // weights and zeroed lines: read by the tensor core
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = uniform(tmem_base_slot);
    grid_launch_dependents();

    const WaitCtx wc = make_wait_ctx(&abort_flag, p.status, p.wait_limit);
    const int tagbits = p.tag << 8;
    const long long total = units_total;
    // a unit is a pair of convolution rows (2r, 2r + 1), with a pool the pooled row r; every role walks the same list
    const int u_begin = (int)(total * blockIdx.x / gridDim.x), u_end = (int)(total * (blockIdx.x + 1) / gridDim.x);
    const uint32_t line_bar = smem_u32(line_bars), done_bar = smem_u32(done_bars), free_bar = smem_u32(free_bars);
    int k = 0;                       // steps so far: barrier k % ROWS_AHEAD, accumulator k % ROWS_ACCS
    bool ok = true;

    if (warp >= ROWS_EPI_WARPS && warp < ROWS_MMA_WARP) {
        // ------------------------------------------------------------------ packing
        const int pt = threadIdx.x - 32 * ROWS_EPI_WARPS;
        const uint32_t img_row_bytes = (uint32_t)p.w * p.c;
        const uint32_t last_word = (uint32_t)p.n * p.h * img_row_bytes - 4u;
        uint32_t cell_off[ROWS_CELLS], cell_mask[ROWS_CELLS];      // byte offset inside an image row; mask of the channel bytes
        bool cell_on[ROWS_CELLS];
#pragma unroll
        for (int i = 0; i < ROWS_CELLS; ++i) {
            const int col = pt + i * 32 * ROWS_PACK_WARPS, iw = col - p.left;
            const bool px = col < p.ncell && iw >= 0 && iw < p.w;   // else zero padding
            cell_on[i] = col < p.ncell;
            cell_off[i] = px ? (uint32_t)iw * p.c : 0u;
            cell_mask[i] = px ? 0xffffffffu >> (32 - 8 * p.c) : 0u;
        }
        grid_dependency_wait();        // the image may belong to earlier work in the stream
        // The words of a line's pixels, all requested before the first is used (a load behind a branch of its own, with its
        // use in the same branch, waits for memory once per cell: 4000 cycles a line instead of 900); combined when the line
        // is stored.
        constexpr bool FAST = READ == READ_WORDS;
        uint32_t raw[2][ROWS_CELLS][2][FAST ? 2 : 1];        // two lines at a time
        // READ_QUADS: item pt + 96 j is a quad of the two lines
        const int quads = p.w / 4;
        uint32_t quad[ROWS_QUADS][2][3], quad_off[ROWS_QUADS];
        int quad_line[ROWS_QUADS];                           // 0, 1; 2: none
#pragma unroll
        for (int j = 0; j < ROWS_QUADS; ++j) {
            const int i = pt + j * 32 * ROWS_PACK_WARPS;
            quad_line[j] = i < quads ? 0 : (i < 2 * quads ? 1 : 2);
            quad_off[j] = (uint32_t)(i - (quad_line[j] == 1 ? quads : 0));
        }
        uint32_t row_off[2][2] = {{0u, 0u}, {0u, 0u}}, second_mask[2] = {0u, 0u};
        auto load_lines = [&](int img, int pr0) {
#pragma unroll
            for (int l = 0; l < 2; ++l) {
                const int pr = min(pr0 + l, p.hp - 1);            // (a line past the image is not stored)
                row_off[l][0] = ((uint32_t)img * p.h + 2u * pr) * img_row_bytes;
                second_mask[l] = 2 * pr + 1 < p.h ? 0xffffffffu : 0u;
                row_off[l][1] = row_off[l][0] + (img_row_bytes & second_mask[l]);
                if (READ != READ_QUADS)
#pragma unroll
                for (int i = 0; i < ROWS_CELLS; ++i)
#pragma unroll
                    for (int e = 0; e < 2; ++e) {
                        const uint32_t off = row_off[l][e] + cell_off[i];
                        if (FAST) {      // two aligned words around the pixel, none beyond the tensor's last one
                            raw[l][i][e][0] = ldg32(p.x + (off & ~3u));
                            raw[l][i][e][FAST ? 1 : 0] = ldg32(p.x + min((off & ~3u) + 4u, last_word));
                        } else {
                            raw[l][i][e][0] = load_pixel<false>(p.x, off, last_word, p.c);
                        }
                    }
            }
            if (READ == READ_QUADS)
#pragma unroll
                for (int j = 0; j < ROWS_QUADS; ++j)
                    if (quad_line[j] < 2)
#pragma unroll
                        for (int e = 0; e < 2; ++e)
#pragma unroll
                            for (int w = 0; w < 3; ++w)
                                quad[j][e][w] = ldg32(p.x + (quad_line[j] == 0 ? row_off[0][e] : row_off[1][e]) + 12u * quad_off[j] + 4u * w);
        };
        auto store_quads = [&](int line, int n) {
#pragma unroll
            for (int j = 0; j < ROWS_QUADS; ++j) {
                if (quad_line[j] >= n) continue;
                uint2 *dst = (uint2 *)(line_ptr + ((line + quad_line[j]) & (ROWS_LINES - 1)) * STEM_SLOT_BYTES) + p.left + 4 * quad_off[j];
                const uint32_t mask = quad_line[j] == 0 ? second_mask[0] : second_mask[1];
                uint32_t px[2][4];
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    const uint32_t *w = quad[j][e];
                    px[e][0] = w[0] & 0xffffffu;
                    px[e][1] = __funnelshift_r(w[0], w[1], 24) & 0xffffffu;
                    px[e][2] = __funnelshift_r(w[1], w[2], 16) & 0xffffffu;
                    px[e][3] = w[2] >> 8;
                }
#pragma unroll
                for (int i = 0; i < 4; ++i) dst[i] = make_uint2(px[0][i], px[1][i] & mask);
            }
        };
        auto line_cell = [&](int l, int i) {
            uint32_t v[2];
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                v[e] = raw[l][i][e][0];
                if (FAST) v[e] = __funnelshift_r(v[e], raw[l][i][e][FAST ? 1 : 0], ((row_off[l][e] + cell_off[i]) & 3u) * 8u);
                v[e] &= cell_mask[i];
            }
            return make_uint2(v[0], v[1] & second_mask[l]);
        };
        int line = 0;                  // lines packed so far: slot line % ROWS_LINES
        for (int u = u_begin; ok && u < u_end;) {
            const int img = u / p.rows_per_img, r0 = u - img * p.rows_per_img;
            const int r1 = min(p.rows_per_img, r0 + (u_end - u));
            u += r1 - r0;
            const int first = POOL && r0 > 0 ? r0 - 1 : r0;          // (pool: the row above the first pooled row)
            int pr = max(0, 2 * first - p.top);                      // next pair to pack
            load_lines(img, pr);
            for (int r = first; r < r1; ++r, ++k) {
                // a new image does not share lines with the steps before it: let those finish, so that the ring holds one
                // image's window at a time
                const int need = r == first ? k - 1 : k - ROWS_AHEAD;
                bool got = true;
                if (need >= 0) got = mbar_wait(done_bar + 8 * (need % ROWS_AHEAD), (uint32_t)(need / ROWS_AHEAD) & 1u, wc, tagbits | 121);
                if (!__all_sync(0xffffffffu, got)) { ok = false; break; }
                const int pr_end = min(p.hp, 2 * r + 1 - p.top + p.kh2);
                while (pr < pr_end) {
                    if (READ == READ_QUADS) store_quads(line, min(2, pr_end - pr));
                    else
#pragma unroll
                    for (int l = 0; l < 2; ++l)
                        if (pr + l < pr_end) {
                            uint2 *dst = (uint2 *)(line_ptr + ((line + l) & (ROWS_LINES - 1)) * STEM_SLOT_BYTES) + pt;
#pragma unroll
                            for (int i = 0; i < ROWS_CELLS; ++i)
                                if (cell_on[i]) dst[i * 32 * ROWS_PACK_WARPS] = line_cell(l, i);
                        }
                    const int n = min(2, pr_end - pr);
                    line += n;
                    pr += n;
                    if (pr < p.hp) load_lines(img, pr);              // in flight until their turn
                }
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                __syncwarp();
                if (lane == 0) mbar_arrive(line_bar + 8 * (k % ROWS_AHEAD));
            }
        }
    } else if (warp == ROWS_MMA_WARP) {
        // ------------------------------------------------------------------ MMA issue: the whole warp runs the loop, one lane issues
        {
            const uint32_t a_lo0 = p.a_desc_lbo_sbo | ((line_base & 0x3ffffu) >> 4), b_lo0 = p.b_desc_lbo_sbo | ((smem_base & 0x3ffffu) >> 4);
            const uint32_t b_slice = 4u * c_out;                 // 16-byte units between the K slices of the weights
            int line = 0;
            for (int u = u_begin; ok && u < u_end;) {
                const int img = u / p.rows_per_img, r0 = u - img * p.rows_per_img;
                const int r1 = min(p.rows_per_img, r0 + (u_end - u));
                u += r1 - r0;
                const int first = POOL && r0 > 0 ? r0 - 1 : r0;
                const int pr_first = max(0, 2 * first - p.top);
                const int line_of_pr = line - pr_first;              // ring index of pair 0 of this image (may be negative)
                for (int r = first; r < r1; ++r, ++k) {
                    bool got = true;
                    if (k >= ROWS_ACCS) got = mbar_wait(free_bar + 8 * (k % ROWS_ACCS), (uint32_t)(k / ROWS_ACCS - 1) & 1u, wc, tagbits | 122);
                    got = got && mbar_wait(line_bar + 8 * (k % ROWS_AHEAD), (uint32_t)(k / ROWS_AHEAD) & 1u, wc, tagbits | 123);
                    if (!__all_sync(0xffffffffu, got)) { ok = false; break; }
                    tc_fence_after();
                    const uint32_t d_tmem = tmem_base + (uint32_t)((k % ROWS_ACCS) * p.acc_cols);
                    uint32_t accumulate = 0;
                    uint32_t b_lo = b_lo0;
                    for (int j = 0; j <= p.kh2; ++j, b_lo += b_slice * p.slices) {
                        const int pr = 2 * r - p.top + j;
                        if (pr < 0 || pr >= p.hp) continue;          // rows above / below the image contribute nothing
                        const uint32_t a_lo = a_lo0 + (uint32_t)((line_of_pr + pr) & (ROWS_LINES - 1)) * (STEM_SLOT_BYTES / 16);
                        stem_mma_pair<true>(d_tmem, a_lo, b_lo, p, b_slice, accumulate);
                        accumulate = 1;
                    }
                    mma_commit(done_bar + 8 * (k % ROWS_AHEAD));
                }
                line = line_of_pr + max(pr_first, min(p.hp, 2 * r1 - 1 - p.top + p.kh2));
            }
            if (!ok && k > 0) {
                // aborting: give the MMAs already issued time to finish before tensor memory is released
                const unsigned long long t0 = clock64();
                while (!mbar_try_wait(done_bar + 8 * ((k - 1) % ROWS_AHEAD), (uint32_t)((k - 1) / ROWS_AHEAD) & 1u) &&
                       (unsigned long long)(clock64() - t0) < DRAIN_LIMIT_CYCLES) {
                }
            }
        }
    } else {
        // ------------------------------------------------------------------ conversion: thread = output pixel
        // After a wait that gave up (ok == false) a warp goes through the remaining steps without touching anything, so that the
        // barrier of the eight warps below stays complete.
        const int quarter = warp & 3, half = warp >> 2;
        const int px = quarter * 32 + lane;
        const uint32_t t_lane = tmem_base + ((uint32_t)(quarter * 32) << 16);
        const uint32_t rsel[4] = {0, 0, 0, 0};
        grid_dependency_wait();        // the output may overwrite what earlier work in the stream still reads
        auto step_ready = [&]() {
            const uint32_t bar = done_bar + 8 * (k % ROWS_AHEAD), parity = (uint32_t)(k / ROWS_AHEAD) & 1u;
            // (in line: around a call the registers of the open pooled row would be spilled, and so little L1 is left beside the
            // shared memory that they come back from L2)
            const bool got = mbar_try_wait_hint(bar, parity, 4000u) || mbar_wait_poll(bar, parity, wc, tagbits | 120);
            ok = __all_sync(0xffffffffu, got) && ok;
            tc_fence_after();
        };
        auto step_read = [&]() {
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(free_bar + 8 * (k % ROWS_ACCS));
            ++k;
        };
        if (POOL) {
            constexpr int CI = (CH + 1) / 2;
            const int ch0 = half * CI;                            // this warp's chunks of the pixel: [ch0, ch0 + CI), those < cpr
            const uint32_t swz = ((uint32_t)px >> p.swz_shift) & (uint32_t)p.swz_mask;
            int prev[CI][16];                                     // the row above the pooled row that is open
            uint32_t buf = 0;
            for (int u = u_begin; u < u_end;) {
                const int img = u / p.rows_per_img, r0 = u - img * p.rows_per_img;
                const int r1 = min(p.rows_per_img, r0 + (u_end - u));
                u += r1 - r0;
#pragma unroll
                for (int ci = 0; ci < CI; ++ci)
#pragma unroll
                    for (int j = 0; j < 16; ++j) prev[ci][j] = INT_MIN;
                if (r0 > 0) {
                    step_ready();
                    if (ok) {
#pragma unroll
                        for (int ci = 0; ci < CI; ++ci)
                            if (ch0 + ci < p.cpr) {
                                tmem_ld16(t_lane + (uint32_t)((k % ROWS_ACCS) * p.acc_cols + (p.cpr + ch0 + ci) * 16), prev[ci]);
                                tmem_ld_wait16(prev[ci]);
                            }
                    }
                    step_read();
                }
                for (int py = r0; py < r1; ++py) {
                    const bool two = 2 * py + 1 < p.ho;
                    const uint32_t t_addr = t_lane + (uint32_t)((k % ROWS_ACCS) * p.acc_cols);
                    step_ready();
                    const uint32_t dst = rows_base + buf * row_bytes + (uint32_t)px * c_out;
#pragma unroll
                    for (int ci = 0; ci < CI; ++ci) {
                        const int ch = ch0 + ci;
                        if (ok && ch < p.cpr) {
                            int a[16], b[16];
                            tmem_ld16(t_addr + ch * 16, a);
                            if (two) {
                                tmem_ld16(t_addr + (p.cpr + ch) * 16, b);
                            } else {
#pragma unroll
                                for (int j = 0; j < 16; ++j) b[j] = INT_MIN;
                            }
                            tmem_ld_wait16(a);
                            tmem_ld_wait16(b);
#pragma unroll
                            for (int j = 0; j < 16; ++j) {
                                a[j] = __vimax3_s32(prev[ci][j], a[j], b[j]);
                                prev[ci][j] = b[j];
                            }
                            sts128(dst + (((uint32_t)ch ^ swz) << 4),
                                   epilogue_fast16<false, SIGNED>(a, bias_base + 64 * ch, make_uint4(0, 0, 0, 0), 1, 0, rsel, p.s));
                        }
                    }
                    step_read();
                    asm volatile("bar.sync 1, %0;" ::"n"(ROWS_EPI_WARPS * 32) : "memory");
                    // maximum over three neighbouring columns; the other buffer is free for the next row meanwhile
                    const uint32_t src = rows_base + buf * row_bytes;
                    uint8_t *out = p.y + ((size_t)img * p.po + py) * (size_t)p.pwo * c_out;
                    if (ok)
                        for (int it = threadIdx.x; it < p.pwo * p.cpr; it += ROWS_EPI_WARPS * 32) {
                            const int ppx = CH == 4 && p.cpr == 4 ? it >> 2 : it / p.cpr, ch = it - ppx * p.cpr;
                            uint4 t[3];
#pragma unroll
                            for (int d = 0; d < 3; ++d) {
                                const uint32_t cx = (uint32_t)min(max(2 * ppx + d - 1, 0), p.wo - 1);      // the edge column again
                                t[d] = lds128(src + cx * c_out + (((uint32_t)ch ^ ((cx >> p.swz_shift) & (uint32_t)p.swz_mask)) << 4));
                            }
                            *(uint4 *)(out + (size_t)it * 16) =
                                make_uint4(max3_bytes<SIGNED>(t[0].x, t[1].x, t[2].x), max3_bytes<SIGNED>(t[0].y, t[1].y, t[2].y),
                                           max3_bytes<SIGNED>(t[0].z, t[1].z, t[2].z), max3_bytes<SIGNED>(t[0].w, t[1].w, t[2].w));
                        }
                    buf ^= 1u;
                }
            }
        } else {
            for (int u = u_begin; u < u_end;) {
                const int img = u / p.rows_per_img, r0 = u - img * p.rows_per_img;
                const int r1 = min(p.rows_per_img, r0 + (u_end - u));
                u += r1 - r0;
                for (int r = r0; r < r1; ++r) {
                    const int oy = 2 * r + half;                  // the warps of a half take one of the two rows
                    step_ready();
                    const uint32_t t_addr = t_lane + (uint32_t)((k % ROWS_ACCS) * p.acc_cols) + (uint32_t)half * c_out;
                    uint8_t *out = p.y + (((size_t)img * p.ho + oy) * (size_t)p.wo + px) * c_out;
                    if (ok && oy < p.ho) {
#pragma unroll
                        for (int ch = 0; ch < CH; ++ch)
                            if (ch < p.cpr) {
                                int a[16];
                                tmem_ld16(t_addr + ch * 16, a);
                                tmem_ld_wait();
                                const uint4 o = epilogue_fast16<false, SIGNED>(a, bias_base + 64 * ch, make_uint4(0, 0, 0, 0), 1, 0, rsel, p.s);
                                if (px < p.wo) *(uint4 *)(out + 16 * ch) = o;
                            }
                    }
                    step_read();
                }
            }
        }
    }

    tc_fence_before();
    __syncthreads();
    if (warp == ROWS_MMA_WARP) {
        tc_fence_after();
        tmem_dealloc(tmem_base, (uint32_t)(ROWS_ACCS * p.acc_cols));
    }
}

}   // namespace

static size_t stem_smem_bytes(int kh2, int slices, int c_out) {
    return (size_t)kh2 * slices * 32 * c_out + STEM_PAIR_SLOTS * STEM_SLOT_BYTES + 2 * 128 * (size_t)c_out + 4 * (size_t)c_out;
}
static size_t stem_rows_smem_bytes(int kh2, int slices, int c_out, bool pool) {
    return (size_t)(kh2 + 1) * slices * 32 * 2 * c_out + ROWS_LINES * STEM_SLOT_BYTES + (pool ? 2 * 128 * (size_t)c_out : 0) + 4 * (size_t)c_out;
}

bool f8_stem_tc_supported(const F8ConvGeom &g, const F8Requant &q, int kh2, int slices) {
    if (g.c > 4 || g.stride_h != 2 || g.stride_w != 2) return false;
    if (g.wo > 128 || g.wo < 1 || g.c_out % 16 != 0 || g.c_out > 256) return false;
    if (q.has_res || (q.y_kind != F8_U8 && q.y_kind != F8_S8) || q.s < 1 || q.s > 24) return false;
    if (g.pad_h >= g.kh) return false;       // output rows without an image row: no multiplication would write their sums
    if (kh2 < 1 || kh2 >= STEM_PAIR_SLOTS || slices < 1 || slices > 2) return false;       // windows of at most 64 bytes
    if (2 * (g.wo - 1) + slices * 4 > STEM_MAX_CELLS) return false;
    if ((size_t)g.n * g.h * g.w * g.c >= 0x7fffffffull || (size_t)g.n * std::max(g.ho, 1) >= 0x7fffffffull) return false;
    return stem_smem_bytes(kh2, slices, g.c_out) <= 200 * 1024;
}

namespace {
typedef void (*StemKernel)(const StemParams, const int);
template <bool POOL, bool SIGNED>
StemKernel pick_wide(bool fast) {
    return fast ? f8_stem_tc_kernel<POOL, SIGNED, true> : f8_stem_tc_kernel<POOL, SIGNED, false>;
}
template <int CH, bool POOL, bool SIGNED>
StemKernel pick_rows(int read) {
    return read == READ_QUADS ? f8_stem_rows_tc_kernel<CH, POOL, SIGNED, READ_QUADS>
                              : (read == READ_WORDS ? f8_stem_rows_tc_kernel<CH, POOL, SIGNED, READ_WORDS> : f8_stem_rows_tc_kernel<CH, POOL, SIGNED, READ_BYTES>);
}
template <int CH>
StemKernel pick_rows(bool pool, bool sgn, int read) {
    if (pool) return sgn ? pick_rows<CH, true, true>(read) : pick_rows<CH, true, false>(read);
    return sgn ? pick_rows<CH, false, true>(read) : pick_rows<CH, false, false>(read);
}
StemKernel pick_wide(bool pool, bool sgn, bool fast) {
    if (pool) return sgn ? pick_wide<true, true>(fast) : pick_wide<true, false>(fast);
    return sgn ? pick_wide<false, true>(fast) : pick_wide<false, false>(fast);
}
}   // namespace

cudaError_t f8_launch_stem_tc(const F8ConvGeom &g, const F8Requant &q, int kh2, int top, int left, int slices, int pool,
                              const void *x, const int8_t *w_core, const int32_t *bias, void *y, int *status_word, int tag,
                              cudaStream_t st, bool overlap_previous) {
    if (g.n == 0) return cudaSuccess;
    StemParams p = {};
    p.n = g.n; p.h = g.h; p.w = g.w; p.c = g.c;
    p.ho = g.ho; p.wo = g.wo; p.c_out = g.c_out;
    p.kh2 = kh2; p.top = top; p.left = left; p.hp = (g.h + 1) / 2; p.slices = slices;
    p.ncell = std::min(STEM_MAX_CELLS, 2 * (g.wo - 1) + slices * 4);
    p.pool = pool;
    // up to 64 channels: the kernel with a warp role each (two rows per step, two accumulators of at most 128 columns, two CTAs per SM);
    // wider layers would leave it one CTA per SM or not fit, and keep the kernel with two accumulators
    const bool rows = g.c_out <= 64;
    const int n_cols = rows ? 2 * g.c_out : g.c_out;        // columns of one multiplication
    p.po = (g.ho - 1) / 2 + 1;
    p.pwo = (g.wo - 1) / 2 + 1;
    p.rows_per_img = pool ? p.po : (rows ? (g.ho + 1) / 2 : g.ho);
    p.acc_cols = 32;
    while (p.acc_cols < n_cols) p.acc_cols *= 2;
    p.cpr = g.c_out / 16;
    const bool pow2 = (p.cpr & (p.cpr - 1)) == 0;
    p.swz_shift = p.cpr == 4 ? 1 : (p.cpr == 2 ? 2 : 0);
    p.swz_mask = (pow2 && p.cpr > 1) ? std::min(p.cpr, 8) - 1 : 0;
    p.idesc = (2u << 4) | ((g.x_signed ? 1u : 0u) << 7) | (1u << 10) | ((uint32_t)(n_cols >> 3) << 17) | ((128u >> 4) << 24);
    // K-major operands without swizzle: core matrices of 8 rows x 16 bytes are 128 contiguous bytes; the leading
    // byte offset is the distance between core matrices along K, the stride byte offset the one between 8-row groups.
    // A (overlapping windows): 16 bytes along K, 128 bytes along M.  B ([K/16][columns][16]): columns * 16 along K, 128 along N.
    const uint32_t a_lbo = 16, a_sbo = 128, b_lbo = (uint32_t)n_cols * 16, b_sbo = 128;
    p.a_desc_lbo_sbo = (a_lbo >> 4) << 16;
    p.b_desc_lbo_sbo = (b_lbo >> 4) << 16;
    p.a_desc_hi = (a_sbo >> 4) | (1u << 14);     // stride byte offset at bit 32, descriptor version 1 at bit 46, no swizzle
    p.b_desc_hi = (b_sbo >> 4) | (1u << 14);
    p.s = q.s;
    p.signed_out = q.y_kind == F8_S8 ? 1 : 0;
    p.x_signed = g.x_signed;
    p.x = (const uint8_t *)x; p.wk = w_core; p.bias = bias; p.y = (uint8_t *)y; p.status = status_word; p.tag = tag;
    p.wait_limit = f8_wait_limit_cycles();

    const bool fast = ((uintptr_t)x & 3) == 0 && ((size_t)g.n * g.h * g.w * g.c) % 4 == 0;
    const int read = !fast ? READ_BYTES : (g.c == 3 && g.w % 4 == 0 && left + g.w <= STEM_MAX_CELLS ? READ_QUADS : READ_WORDS);
    const bool sgn = p.signed_out != 0;
    StemKernel kernel = !rows ? pick_wide(pool != 0, sgn, fast) : (p.cpr > 2 ? pick_rows<4>(pool != 0, sgn, read) : pick_rows<2>(pool != 0, sgn, read));
    const size_t smem = rows ? stem_rows_smem_bytes(kh2, slices, g.c_out, pool != 0) : stem_smem_bytes(kh2, slices, g.c_out);
    const int threads = rows ? ROWS_THREADS : STEM_THREADS, accs = rows ? ROWS_ACCS : 2;
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(200 * 1024));
    // several CTAs are meant to share an SM: ask for the largest shared-memory carve-out (the default preference
    // sizes it for a single CTA of this kernel)
    if (e == cudaSuccess) e = cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
    if (e != cudaSuccess) return e;
    int dev = 0, sms = 148, occ = 1;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    // CTAs that fit an SM, from the kernel's own resource use (the runtime's occupancy query answers 1 for this
    // kernel whatever the carve-out): registers, shared memory, threads, and their accumulators in tensor memory
    cudaFuncAttributes fa;
    if (cudaFuncGetAttributes(&fa, kernel) == cudaSuccess && fa.numRegs > 0) {
        const int regs_per_cta = ((fa.numRegs + 7) / 8 * 8) * threads;
        const int by_regs = 65536 / regs_per_cta;
        const int by_smem = (int)((227 * 1024) / (smem + fa.sharedSizeBytes + 1024));
        const int by_threads = 2048 / threads;
        occ = std::min(std::min(by_regs, by_smem), by_threads);
    }
    occ = std::min(occ, 512 / (accs * p.acc_cols));
    occ = std::max(1, std::min(occ, 4));
    const long long units = (long long)g.n * p.rows_per_img;
    // bands of at least four units (with a pool every band computes one row above it again); up to 64 channels, when that leaves SMs
    // idle, as many bands as there are units up to one per SM (wider layers lose by it: 32 x 32, 3 -> 96 with the pool, batch 64 18.1
    // against 17.3 us)
    const long long bands = std::max<long long>(units / 4, rows ? std::min<long long>(units, sms) : 1);
    const long long grid = std::min<long long>((long long)sms * occ, bands);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = overlap_previous ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kernel, p, (int)units);
}

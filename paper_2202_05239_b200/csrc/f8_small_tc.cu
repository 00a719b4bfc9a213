// Dense layers whose whole work is a few microseconds (single-image inference, fully connected layers, the last stages of
// small batches): an implicit GEMM built for latency instead of throughput.
//
// What bounds such a layer is the time from the end of the layer before it to its own end.  Inside a network its blocks are resident
// long before that (programmatic dependent launch), so everything that does not need the activations is done by then:
//   * the block's weights lie in shared memory, rows an odd number of 16-byte units apart (ldmatrix rows then meet no bank twice);
//   * every lane has its addresses: a tile's input pixels are fetched once, as the contiguous window of input rows they are, and a
//     filter tap is an offset into it -- a 3x3 filter reads its nine taps from the same bytes (pixels outside the image are read from
//     a line of zeros).
// Behind the wait there is one fetch of the window, one pass over K with all warps on slices of their own (mma.sync m16n8k32, no block
// barrier inside), and the sums of the slices meet in shared memory (integers: any order gives the same result) for bias, shortcut,
// rounding shift, clip and a second consumer, for every output kind the library has.  The form before it walked K in 128-byte chunks
// with a barrier each and gathered every tap: K = 2304 took 3.5 us behind the wait, K = 4608 7.5 - 10 us, now 1.3 - 1.5 us.  Inside a
// network 14 x 14, 3 x 3 256 -> 256 of one image adds 3.5 us, 1 x 1 64 -> 384 1.8 us, of which 1.15 us are the hand-over itself.
// Layers whose window and weights do not fit go over the channels in panels, two in flight (one where two of the smallest panels do
// not fit either: filters of 21 x 21 and more).
// mma.sync cannot reach the rate of tcgen05.mma (2045 multiply-adds a clock and SM, measured), which is why layers with more work
// stay with the other kernel (f8_small_tc_wanted has the rule and what was measured on both sides of it).
#include <math.h>

#include <algorithm>

#include "f8_epilogue.cuh"
#include "f8_tc_ptx.cuh"

namespace {

constexpr int SM_THREADS = 256;             // eight warps
constexpr int SM_BARS = 64;                 // shared memory: a line of zeros, the barrier that counts the weights' bytes, the abort flag, ...
constexpr int SM_ABORT = 80;
constexpr int SM_ZERO = 128;                // ... then the stages
constexpr int SM_SMEM = 226 * 1024;
constexpr int FINISH_AHEAD = 4;             // groups of four channels whose shortcuts are on their way together
constexpr int WINDOW_AHEAD = 4;             // copies of a thread whose addresses are ready when the wait ends

// A value that is computed here and not where it is used: the compiler would move address arithmetic behind the wait.
#define PIN(v) asm volatile("" : "+r"(v))
#define PIN64(v) asm volatile("" : "+l"(v))

struct SmallParams {
    int M, c_out, n_tiles;
    int bm, bn_shift;                       // rows and log2 of the columns of a tile
    int wn_shift, wk_shift;                 // log2 of the warps along columns and along K (the others along rows)
    int item_shift, part_shift;             // log2 of the groups of four channels in a tile, of the threads that add up one group
    int h, w, c;                            // input
    int ho, wo, kh, kw, taps, stride, pad;
    int pointwise, strided;                 // 1x1 without padding; 1x1 that skips pixels
    int panels, p16, last16;                // panels of channels: 16-byte units per pixel in one, in the last one
    int ahead;                              // panels in flight: 2 or 1
    uint32_t wo_magic, ho_magic, kw_magic, p16_magic, last_magic, row_magic, last_row_magic;
    uint32_t k_bytes;                       // of an output channel's weights
    int bulk;                               // these are fetched by bulk copies
    int unit_step, dst_step, dst_wrap;      // SM_THREADS 16-byte units further on in the first panel's window
    int wait_first;                         // a call of its own: the weights may come from earlier work in the stream as well
    int tag;
    int *status;
    unsigned long long wait_limit;
    uint32_t pa, pb;                        // bytes from pixel to pixel of a window, from channel to channel of the weights
    uint32_t b_off, stage;                  // weights behind the window; bytes of a stage
    int plain8;                             // one 8-bit output, shift 1 .. 24, sums that fit 32 bits with the rounding constant: multiply-add,
                                            // shift, saturating pack
    int mul_acc, mul_res, round;
    const uint8_t *x;
    const int8_t *wgt;                      // [c_out][taps * c]
    const int32_t *bias;
    const void *res;
    void *y;
    F8Requant q;
    F8Sibling sib;
};

// 16 bytes global -> shared.
__device__ __forceinline__ void cp_async16(uint32_t dst, const void *src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}
__device__ __forceinline__ void ldmatrix4(uint32_t addr, uint32_t (&r)[4]) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(addr)
                 : "memory");
}
template <bool XS>
__device__ __forceinline__ void mma_16832(int (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    if (XS)
        asm volatile("mma.sync.aligned.m16n8k32.row.col.s32.s8.s8.s32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
                     : "+r"(d[0]), "+r"(d[1]), "+r"(d[2]), "+r"(d[3])
                     : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
    else
        asm volatile("mma.sync.aligned.m16n8k32.row.col.s32.u8.s8.s32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
                     : "+r"(d[0]), "+r"(d[1]), "+r"(d[2]), "+r"(d[3])
                     : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// n / d with magic = 2^32 / d rounded up (0 for d = 1), exact while n * d < 2^32.
__device__ __forceinline__ int quick_div(int n, uint32_t magic) { return magic ? (int)__umulhi((uint32_t)n, magic) : n; }

// Stores four consecutive channels of one output pixel for one consumer of the aligned sums v[].
__device__ __forceinline__ void store4(void *y, int y_kind, int s, int lo, int hi, const int (&v)[4], size_t o) {
    int t[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) t[j] = f8_quantize_child(v[j], y_kind, s, lo, hi);
    if (y_kind == F8_S32 || y_kind == F8_S32_RELU) *(int4 *)((int32_t *)y + o) = make_int4(t[0], t[1], t[2], t[3]);
    else *(uint32_t *)((uint8_t *)y + o) = f8_pack4(t[0], t[1], t[2], t[3]);
}

// Four sums to four bytes: rounding shift (the constant is in v already) and clip.
__device__ __forceinline__ uint32_t pack_plain8(const int (&v)[4], int s, bool is_signed) {
    int t[4];
    uint32_t hi, o;
#pragma unroll
    for (int j = 0; j < 4; ++j) t[j] = v[j] >> s;
    if (is_signed) {
#pragma unroll
        for (int j = 0; j < 4; ++j) t[j] = max(t[j], -127);
        asm("cvt.pack.sat.s8.s32.b32 %0, %1, %2, 0;" : "=r"(hi) : "r"(t[3]), "r"(t[2]));
        asm("cvt.pack.sat.s8.s32.b32 %0, %1, %2, %3;" : "=r"(o) : "r"(t[1]), "r"(t[0]), "r"(hi));
    } else {
        asm("cvt.pack.sat.u8.s32.b32 %0, %1, %2, 0;" : "=r"(hi) : "r"(t[3]), "r"(t[2]));
        asm("cvt.pack.sat.u8.s32.b32 %0, %1, %2, %3;" : "=r"(o) : "r"(t[1]), "r"(t[0]), "r"(hi));
    }
    return o;
}

// Eight warps; warp tiles of 16 MT rows x 8 NT columns.  blockIdx: (column tile, row tile).  PW: 1x1, stride 1, no padding, one panel --
// a window is a run of pixels and K a run of bytes.
// The part in front of the wait is kept short as well: it runs while the blocks of the layer before, on the same SM, are on the
// critical path (its first form, a thousand instructions a warp, cost them 0.4 us a layer).
template <int MT, int NT, bool XS, bool PW>
__global__ void __launch_bounds__(SM_THREADS, MT == 1 ? 3 : 2) f8_conv_small_tc_kernel(const __grid_constant__ SmallParams p) {
    extern __shared__ __align__(128) uint8_t smem[];
    const uint32_t smem_base = smem_u32(smem);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int m0 = (int)blockIdx.y * p.bm, n0 = (int)blockIdx.x << p.bn_shift;
    const bool one_panel = PW || p.panels == 1;
    const int first16 = one_panel ? p.last16 : p.p16;
    const uint32_t first_magic = one_panel ? p.last_magic : p.p16_magic;
    if (p.wait_first) grid_dependency_wait();
    grid_launch_dependents();

    // ---- weights of the first two panels: bulk copies, one per output channel, where these are long enough (a lane issues one in about 40
    // cycles, one after the other), else 16 bytes a thread
    const int w_rows = min(1 << p.bn_shift, p.c_out - n0);
    auto load_weights = [&](int panel) {
        if (!p.bulk) {
            const bool last = PW || panel + 1 == p.panels;
            const int n16 = last ? p.last16 : p.p16, row16 = (PW ? 1 : p.taps) * n16, total = w_rows * row16;
            const uint32_t row_magic = last ? p.last_row_magic : p.row_magic, dst = smem_base + SM_ZERO + (panel & 1) * p.stage + p.b_off;
            const uint32_t tap_magic = last ? p.last_magic : p.p16_magic, tap_gap = (uint32_t)(p.c - n16 * 16);
            const int8_t *src = p.wgt + (size_t)(uint32_t)n0 * p.k_bytes + panel * p.p16 * 16;
            for (int i = tid; i < total; i += SM_THREADS) {
                const int row = quick_div(i, row_magic), k = i - row * row16;
                const uint32_t gap = one_panel ? 0u : (uint32_t)quick_div(k, tap_magic) * tap_gap;
                cp_async16(dst + row * p.pb + k * 16, src + ((size_t)(uint32_t)row * p.k_bytes + gap + k * 16));
            }
            return;
        }
        if (warp != 0) return;
        const uint32_t dst = smem_base + SM_ZERO + p.b_off, bar = smem_base + SM_BARS;
        const int8_t *src = p.wgt + (size_t)(uint32_t)n0 * p.k_bytes;
        if (lane == 0) mbar_expect_tx(bar, p.k_bytes * w_rows);
        for (int row = lane; row < w_rows; row += 32)
            asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst + row * p.pb),
                         "l"(src + (size_t)(uint32_t)row * p.k_bytes), "r"(p.k_bytes), "r"(bar)
                         : "memory");
    };
    if (warp == 0) {
        if (lane < SM_ZERO / 16) *(uint4 *)(smem + lane * 16) = make_uint4(0, 0, 0, 0);
        __syncwarp();
        if (lane == 0) {
            mbar_init(smem_base + SM_BARS, 1);
            asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        }
        __syncwarp();
    }
    load_weights(0);
    if (!one_panel && p.ahead == 2) load_weights(1);

    // ---- the window: the input pixels of this tile, contiguous in memory (rows of the batch, one below the other)
    int first = m0, count;
    const int m1 = min(m0 + p.bm, p.M) - 1;
    // ---- lanes: rows of their ldmatrix loads, and where their slice of K begins
    const int wi_k = warp & ((1 << p.wk_shift) - 1), wi_mn = warp >> p.wk_shift, wi_m = wi_mn >> p.wn_shift, wi_n = wi_mn & ((1 << p.wn_shift) - 1);
    int base[MT], iy0[MT], ix0[MT];
    int ih = 1, iw = 1;
    if (PW || p.pointwise) {
        count = m1 - m0 + 1;
#pragma unroll
        for (int i = 0; i < MT; ++i) {
            base[i] = (wi_m * MT + i) * 16 + (lane & 15);
            iy0[i] = ix0[i] = 0;
        }
    } else {
        const int r0 = quick_div(m0, p.wo_magic), r1 = quick_div(m1, p.wo_magic);
        const int i0 = quick_div(r0, p.ho_magic), i1 = quick_div(r1, p.ho_magic);
        // (both inside an image: with padding as large as the filter, rows of outputs may read nothing but padding)
        const int y0 = i0 * p.h + min(max((r0 - i0 * p.ho) * p.stride - p.pad, 0), p.h - 1);
        const int y1 = i1 * p.h + max(min((r1 - i1 * p.ho) * p.stride - p.pad + p.kh - 1, p.h - 1), 0);
        first = y0 * p.w;
        count = (y1 - y0 + 1) * p.w;
        ih = p.h;
        iw = p.w;
#pragma unroll
        for (int i = 0; i < MT; ++i) {
            const int m = m0 + (wi_m * MT + i) * 16 + (lane & 15), t = quick_div(m, p.wo_magic), img = quick_div(t, p.ho_magic);
            const int y = (t - img * p.ho) * p.stride - p.pad;
            iy0[i] = m < p.M ? y : -(1 << 24);      // rows past the last pixel: outside every image
            ix0[i] = (m - t * p.wo) * p.stride - p.pad;
            base[i] = (img * p.h + y) * p.w + ix0[i] - first;
        }
    }
    const uint32_t b_lane = p.b_off + (uint32_t)(wi_n * NT * 8 + (lane & 7) + ((lane >> 4) << 3)) * p.pb + (uint32_t)((lane >> 3) & 1) * 16;
    int s0 = 0, s1 = 0, tap0 = 0, cc0 = 0, ty0 = 0, tx0 = 0;
    auto slice = [&](int n16, uint32_t magic) {
        const int steps = ((PW ? 1 : p.taps) * n16 + 1) >> 1, per = (steps + (1 << p.wk_shift) - 1) >> p.wk_shift;
        s0 = wi_k * per;
        s1 = min(s0 + per, steps);
        const int q = 2 * s0 + (lane >> 4);
        if (PW) {
            cc0 = q;
            return;
        }
        tap0 = p.pointwise ? (q >= n16 ? 1 : 0) : quick_div(q, magic);
        cc0 = q - tap0 * n16;
        ty0 = p.pointwise ? tap0 : quick_div(tap0, p.kw_magic);
        tx0 = tap0 - ty0 * p.kw;
    };
    slice(first16, first_magic);
    // ---- threads: first 16-byte unit of the window, first group of four output channels
    const int w_row = quick_div(tid, first_magic), w_unit = tid - w_row * first16;
    const int gs = p.bn_shift - 2, parts = 1 << p.part_shift, it = tid >> p.part_shift, part = tid & (parts - 1);
    const int groups = 1 << p.item_shift, n_it = max(1, groups / SM_THREADS), f_step = SM_THREADS >> gs;
    const int f_row = it >> gs, f_col = (it & ((1 << gs) - 1)) * 4, co = n0 + f_col;
    const int m_end = it < groups && co < p.c_out ? min(p.M, m0 + p.bm) : 0;
    int4 bias = make_int4(0, 0, 0, 0);               // (one of the threads that share a group)
    if (p.bias && m_end && part == 0) bias = *(const int4 *)(p.bias + co);      // (no read-only load: the wait above is inside this kernel)

    // ---- the copies of this thread: the first ones as finished addresses, the loop for what is left, further panels, skipped pixels
    const int n_first = !PW && (p.strided || !one_panel) ? 0 : count * first16;
    uint32_t win_dst[WINDOW_AHEAD];
    int win_n = 0;
    {
        uint32_t dst = smem_base + SM_ZERO + w_row * p.pa + w_unit * 16;
        int k = w_unit;
#pragma unroll
        for (int j = 0; j < WINDOW_AHEAD; ++j) {
            win_dst[j] = dst;
            win_n += tid + j * SM_THREADS < n_first;
            k += p.unit_step;
            dst += p.dst_step;
            if (k >= first16) { k -= first16; dst += p.dst_wrap; }
            PIN(win_dst[j]);
        }
        PIN(win_n);
    }
    const uint8_t *win_src = p.x + (size_t)((uint32_t)first * (uint32_t)p.c + tid * 16);
    PIN64(win_src);
    auto load_window = [&](int panel, int from) {
        const int n16 = panel + 1 == p.panels ? p.last16 : p.p16, total = count * n16;
        const uint32_t dst = smem_base + SM_ZERO + (panel & 1) * p.stage, magic = panel + 1 == p.panels ? p.last_magic : p.p16_magic;
        const uint8_t *x = p.x + panel * p.p16 * 16;
        for (int i = from; i < total; i += SM_THREADS) {
            const int row = quick_div(i, magic), k = i - row * n16, m = first + row;
            int px = m;
            if (!PW && p.strided) {
                const int t = quick_div(m, p.wo_magic), img = quick_div(t, p.ho_magic);
                px = (img * p.h + (t - img * p.ho) * p.stride) * p.w + (m - t * p.wo) * p.stride;
            }
            cp_async16(dst + row * p.pa + k * 16, x + ((uint32_t)px * (uint32_t)p.c + k * 16));
        }
    };
    const int window_left = n_first ? tid + WINDOW_AHEAD * SM_THREADS : tid;
    const bool more_window = window_left < count * first16;
    // ---- the shortcuts and outputs of this thread's first groups
    uint32_t rw[FINISH_AHEAD];
    const bool has_res = p.q.has_res != 0, r32 = p.q.r_s32 != 0;
    uint32_t out0 = (uint32_t)(m0 + f_row) * (uint32_t)p.c_out + co;
    const uint8_t *res8 = (const uint8_t *)p.res + out0;
    uint32_t res_step = (uint32_t)f_step * (uint32_t)p.c_out;
    int rows_left = part == 0 ? m_end - (m0 + f_row) : 0;          // rows of this thread's first group and below
    int res_left = has_res && !r32 ? rows_left : 0;
    PIN(out0); PIN64(res8); PIN(res_step); PIN(rows_left); PIN(res_left);
    // ---- the first step of K
    uint32_t addr[MT], inc[MT], b_addr = smem_base + SM_ZERO + b_lane + s0 * 32;
    int tap = tap0, cc = cc0, ty = ty0, tx = tx0, steps_left = s1 - s0;
    uint32_t a_s = smem_base + SM_ZERO;
    const int kw = p.kw, taps = p.taps, row_px = p.w;
    const uint32_t pa = p.pa, pb16 = 16 * p.pb;
    auto locate = [&]() {
#pragma unroll
        for (int i = 0; i < MT; ++i) {
            if (PW) {
                addr[i] = cc < first16 ? a_s + (uint32_t)base[i] * pa + cc * 16 : smem_base;
                inc[i] = 32u;
                continue;
            }
            const bool in = tap < taps && (unsigned)(iy0[i] + ty) < (unsigned)ih && (unsigned)(ix0[i] + tx) < (unsigned)iw;
            addr[i] = in ? a_s + (uint32_t)(base[i] + ty * row_px + tx) * pa + cc * 16 : smem_base;
            inc[i] = in ? 32u : 0u;
        }
    };
    locate();
#pragma unroll
    for (int i = 0; i < MT; ++i) {
        PIN(addr[i]);
        if (!PW) PIN(inc[i]);
    }
    PIN(b_addr); PIN(steps_left); PIN(cc);
    if (!PW) { PIN(tap); PIN(ty); PIN(tx); }
    // ---- where the sums of the slices meet
    const int pitch = (1 << p.bn_shift) + 8;         // (8 words on: the rows of a quarter warp take different banks)
    uint32_t put = smem_base + SM_ZERO + 4u * ((wi_k * p.bm + wi_m * MT * 16 + (lane >> 2)) * pitch + wi_n * NT * 8 + (lane & 3) * 2);
    uint32_t pitch_bytes = 4u * pitch, slice_bytes = pitch_bytes * p.bm;
    uint32_t get = smem_base + SM_ZERO + 4u * (f_row * pitch + f_col) + part * slice_bytes;
    uint32_t get_step = pitch_bytes * f_step;
    int my_slices = (1 << p.wk_shift) >> p.part_shift, n_panels = PW ? 1 : p.panels;
    int bulk = p.bulk;
    PIN(bulk);
    PIN(put); PIN(pitch_bytes); PIN(slice_bytes); PIN(get); PIN(get_step); PIN(my_slices);
    if (!PW) PIN(n_panels);
    int mul_acc = p.mul_acc, mul_res = p.mul_res, round = p.round, shift = p.q.s, plain8 = p.plain8, out_signed = p.q.y_kind == F8_S8, r_signed = p.q.r_signed;
    PIN(mul_acc); PIN(mul_res); PIN(round); PIN(shift); PIN(plain8); PIN(out_signed); PIN(r_signed);
    uint8_t *y8 = (uint8_t *)p.y + out0;
    PIN64(y8);

    const WaitCtx wc = make_wait_ctx((volatile int *)(smem + SM_ABORT), p.status, p.wait_limit);

    grid_dependency_wait();
#pragma unroll
    for (int j = 0; j < WINDOW_AHEAD; ++j)
        if (j < win_n) cp_async16(win_dst[j], win_src + j * SM_THREADS * 16);
    if (more_window) load_window(0, window_left);
    cp_async_commit();
    if (n_panels > 1 && p.ahead == 2) load_window(1, tid);
    cp_async_commit();
#pragma unroll
    for (int j = 0; j < FINISH_AHEAD; ++j) {
        rw[j] = 0;
        if (j * f_step < res_left) rw[j] = *(const uint32_t *)(res8 + (size_t)j * res_step);
    }

    int acc[MT][NT][4];
#pragma unroll
    for (int i = 0; i < MT; ++i)
#pragma unroll
        for (int j = 0; j < NT; ++j)
#pragma unroll
            for (int e = 0; e < 4; ++e) acc[i][j][e] = 0;
    int n16 = first16;
    for (int panel = 0; panel < n_panels; ++panel) {
        if (panel) {
            n16 = panel + 1 == n_panels ? p.last16 : p.p16;
            if (n16 != first16) slice(n16, p.last_magic);
            a_s = smem_base + SM_ZERO + (panel & 1) * p.stage;
            b_addr = a_s + b_lane + s0 * 32;
            tap = tap0; cc = cc0; ty = ty0; tx = tx0; steps_left = s1 - s0;
            locate();
        }
        cp_async_wait<1>();
        __syncthreads();
        if (bulk) mbar_wait(smem_base + SM_BARS, 0, wc, p.tag << 8 | 230);
        if (steps_left > 0) {
            auto advance = [&]() {
                cc += 2;
                b_addr += 32;
#pragma unroll
                for (int i = 0; i < MT; ++i) addr[i] += inc[i];
                if (PW) {                            // (the second half of an odd last step)
#pragma unroll
                    for (int i = 0; i < MT; ++i) addr[i] = cc < first16 ? addr[i] : smem_base;
                    return;
                }
                if (cc >= n16) {
                    do {
                        cc -= n16;
                        ++tap;
                        if (++tx == kw) { tx = 0; ++ty; }
                    } while (cc >= n16);
                    locate();
                }
            };
            uint32_t a[2][MT][4], b[2][NT / 2][4];
            auto fetch = [&](int at) {
#pragma unroll
                for (int j = 0; j < NT / 2; ++j) ldmatrix4(b_addr + j * pb16, b[at][j]);
#pragma unroll
                for (int i = 0; i < MT; ++i) ldmatrix4(addr[i], a[at][i]);
            };
            auto mma = [&](int at) {
#pragma unroll
                for (int i = 0; i < MT; ++i)
#pragma unroll
                    for (int j = 0; j < NT; ++j) mma_16832<XS>(acc[i][j], a[at][i], b[at][j >> 1][2 * (j & 1)], b[at][j >> 1][2 * (j & 1) + 1]);
            };
            fetch(0);
            for (; steps_left >= 2; steps_left -= 2) {
                advance();
                fetch(1);
                mma(0);
                if (steps_left > 2) {
                    advance();
                    fetch(0);
                }
                mma(1);
            }
            if (steps_left) mma(0);
        }
        __syncthreads();                             // everybody has read the stage
        if (!PW && n_panels > 1) {
            if (panel + p.ahead < n_panels) {
                load_weights(panel + p.ahead);
                load_window(panel + p.ahead, tid);
            }
            cp_async_commit();
            if (p.ahead == 1) cp_async_commit();     // (the wait above leaves one group in flight: an empty one)
        }
    }

    // ---- the slices of K meet in shared memory
#pragma unroll
    for (int i = 0; i < MT; ++i)
#pragma unroll
        for (int e = 0; e < 2; ++e)
#pragma unroll
            for (int j = 0; j < NT; ++j)
                asm volatile("st.shared.v2.b32 [%0], {%1, %2};" ::"r"(put + (i * 16 + 8 * e) * pitch_bytes + j * 32), "r"(acc[i][j][2 * e]), "r"(acc[i][j][2 * e + 1])
                             : "memory");
    __syncthreads();
    if (it >= groups) return;                        // (whole warps)
    for (int j0 = 0; j0 < n_it; j0 += FINISH_AHEAD) {
        int4 r4[FINISH_AHEAD];
        if (r32) {
#pragma unroll
            for (int j = 0; j < FINISH_AHEAD; ++j) {
                r4[j] = make_int4(0, 0, 0, 0);
                if ((j0 + j) * f_step < rows_left) r4[j] = *(const int4 *)((const int32_t *)p.res + out0 + (size_t)(j0 + j) * res_step);
            }
        } else if (j0) {
#pragma unroll
            for (int j = 0; j < FINISH_AHEAD; ++j)
                if ((j0 + j) * f_step < res_left) rw[j] = *(const uint32_t *)(res8 + (size_t)(j0 + j) * res_step);
        }
#pragma unroll
        for (int j = 0; j < FINISH_AHEAD; ++j) {
            if (j0 + j >= n_it) break;
            int v[4] = {bias.x, bias.y, bias.z, bias.w};
            const uint32_t src = get + (j0 + j) * get_step;
            for (int k = 0; k < my_slices; ++k) {
                const uint4 t = lds128(src + k * (slice_bytes << p.part_shift));
                v[0] += (int)t.x; v[1] += (int)t.y; v[2] += (int)t.z; v[3] += (int)t.w;
            }
            for (int d = 1; d < parts; d <<= 1)
#pragma unroll
                for (int e = 0; e < 4; ++e) v[e] += __shfl_xor_sync(0xffffffffu, v[e], d);
            if ((j0 + j) * f_step >= rows_left) continue;
            const size_t skip = (size_t)(j0 + j) * res_step;
            if (has_res) {
                int rr[4] = {r4[j].x, r4[j].y, r4[j].z, r4[j].w};
                if (!r32) {
#pragma unroll
                    for (int e = 0; e < 4; ++e) rr[e] = f8_byte(rw[j], e, r_signed);
                }
#pragma unroll
                for (int e = 0; e < 4; ++e) v[e] = v[e] * mul_acc + rr[e] * mul_res;
            }
            if (plain8) {
#pragma unroll
                for (int e = 0; e < 4; ++e) v[e] += round;
                *(uint32_t *)(y8 + skip) = pack_plain8(v, shift, out_signed);
            } else {
                store4(p.y, p.q.y_kind, p.q.s, p.q.lo, p.q.hi, v, out0 + skip);
                if (p.sib.y2) store4(p.sib.y2, p.sib.y_kind, p.sib.s, p.sib.lo, p.sib.hi, v, out0 + skip);
            }
        }
    }
}

uint32_t magic_of(int d) { return d > 1 ? 0xffffffffu / (uint32_t)d + 1u : 0u; }

int log2_of(int v) {
    int s = 0;
    while ((1 << s) < v) ++s;
    return s;
}

// How a layer is cut: warp tile edge, warps along rows, columns and K, channels per panel, shared memory, estimated cycles.
struct Split {
    int t, wm, wn, wk_shift, p16, panels, ahead;
    size_t window, weights, smem;           // one stage's window and weights, whole block
    long long tiles;
    float cycles;
};

// Input pixels that a tile of bm output pixels reads at most.
int window_pixels(const F8ConvGeom &g, int bm) {
    if (g.kh == 1 && g.kw == 1 && g.pad_h == 0) return bm;                // (rows past the last pixel are read, and their sums dropped)
    // output rows it touches, then input rows: the rows between two images count where a filter does not reach the last ones
    const int span = (bm - 1) / g.wo;
    int rows = bm == (span + 1) * g.wo ? span + 1 : (bm < g.wo && g.wo % bm == 0 ? 1 : (bm + g.wo - 2) / g.wo + 1);
    rows = std::min(rows, g.n * g.ho);
    const int skipped = g.h - g.ho * g.stride_h, seams = skipped > 0 ? (rows + g.ho - 2) / g.ho * skipped : 0;
    return std::min((rows - 1) * g.stride_h + g.kh + seams, g.n * g.h) * g.w;
}

// Cuts a layer so that it is done soonest after its input is (an estimate in cycles, fitted to the layers of the networks at batches 1 - 32).
// Every plan of a layer and every call of its own pays for this search: single precision, no warp tiles of 32 x 32 where 16 x 16 ones
// leave SMs idle, and no search for panels in a split whose least time, with all SMs to itself, is above the best one's or the limit.
bool pick_split(const F8ConvGeom &g, Split *best, float limit = 1e30f) {
    const int M = g.n * g.ho * g.wo;                                      // (below 2^24)
    const int c16 = g.c / 16, taps = g.kh * g.kw, c_out = g.c_out;
    const float k = (float)taps * g.c;
    const int k_steps = (taps * c16 + 1) / 2;
    const int t_end = (long long)((M + 15) / 16) * ((c_out + 15) / 16) < 148 ? 16 : 32;
    best->cycles = limit;
    best->tiles = 0;
    for (int t = 16; t <= t_end; t += 16)
        for (int wm_shift = 0; wm_shift <= 3; ++wm_shift) {
            const int t_shift = t == 16 ? 4 : 5, bm = t << wm_shift;
            if (wm_shift && bm / 2 >= M) break;
            const int px = window_pixels(g, bm), m_tiles = (M + bm - 1) >> (t_shift + wm_shift);
            for (int wn_shift = 0; wn_shift + wm_shift <= 3; ++wn_shift) {
                const int wk = 3 - wm_shift - wn_shift, bn = t << wn_shift;
                if (wn_shift && bn / 2 >= c_out) break;
                const size_t red = ((size_t)bm << wk) * (bn + 8) * 4;
                const long long tiles = (long long)m_tiles * ((c_out + bn - 1) >> (t_shift + wn_shift));
                const float steps = (float)((k_steps + (1 << wk) - 1) >> wk);
                // (a block's own instructions, about 500 a warp, where an SM runs several)
                const float issue = 700.f * std::max(0.f, (float)tiles / 148 - 1);
                struct Parts { float fetch, fetch_w, mul, finish; };
                auto parts = [&](float at_once) {
                    Parts e;
                    e.mul = std::max(steps * (t == 16 ? 45.f : 75.f), at_once * bm * bn * k * (t == 16 ? 1 / 900.f : 1 / 1800.f));
                    e.finish = 350 + 100 * ((bm * bn + 1023) / 1024) + at_once * red / 64;
                    e.fetch = at_once * px * g.c / 45;
                    e.fetch_w = at_once * bn * k / 45;
                    return e;
                };
                {
                    const Parts e = parts(1.f);
                    if (700 + 0.f + issue + e.fetch + e.mul + e.finish >= best->cycles) continue;
                }
                int at16 = 0, ahead = 2;
                size_t window = 0, weights = 0, smem = 0;
                // one panel where it fits, else two stages in half of the shared memory; the smallest panel may take all of it
                for (int p16 = c16;; p16 = p16 == c16 ? (c16 + 1) / 2 : p16 - std::max(1, p16 / 8)) {
                    window = ((size_t)px * ((p16 | 1) * 16) + 127) / 128 * 128;
                    weights = ((size_t)bn * (((size_t)taps * p16 | 1) * 16) + 16 + 127) / 128 * 128;
                    smem = SM_ZERO + std::max((window + weights) * (p16 == c16 ? 1 : 2), red);
                    if (smem <= (size_t)(p16 == c16 ? SM_SMEM : SM_SMEM / 2) || (p16 == 1 && smem <= SM_SMEM)) {
                        at16 = p16;
                        break;
                    }
                    if (p16 == 1 && c16 > 1 && SM_ZERO + std::max(window + weights, red) <= (size_t)SM_SMEM) {
                        smem = SM_ZERO + std::max(window + weights, red);
                        at16 = ahead = 1;
                    }
                    if (p16 == 1) break;
                }
                if (!at16) continue;
                const int panels = (c16 + at16 - 1) / at16;
                const int occ = std::min(t == 16 ? 3 : 2, (int)(SM_SMEM / smem));
                const float at_once = (float)std::min<long long>(occ, (tiles + 147) / 148), rounds = (float)((tiles + 148 * occ - 1) / (148 * occ));
                const Parts e = parts(at_once);
                // (no room for the next layer's block: its start is not hidden)
                const float alone = occ == 1 ? 600.f : 0.f;
                const float cycles = 700 + alone + issue + e.fetch + e.mul + e.finish + (panels - 1) * 300.f +
                                     std::max(0, panels - ahead) * (ahead == 2 ? e.fetch_w : 2 * (e.fetch + e.fetch_w)) / panels +
                                     (rounds - 1) * (1500 + e.fetch + e.fetch_w + e.mul + e.finish);
                if (cycles < best->cycles) *best = {t, 1 << wm_shift, 1 << wn_shift, wk, at16, panels, ahead, window, weights, smem, tiles, cycles};
            }
        }
    return best->tiles > 0;
}

template <int MT, int NT, bool XS, bool PW>
cudaError_t launch_small(const SmallParams &p, const Split &s, cudaStream_t st, bool overlap_previous) {
    static bool attr_set[64] = {false};
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    if (!attr_set[dev]) {
        cudaError_t e = cudaFuncSetAttribute(f8_conv_small_tc_kernel<MT, NT, XS, PW>, cudaFuncAttributeMaxDynamicSharedMemorySize, SM_SMEM);
        if (e == cudaSuccess) e = cudaFuncSetAttribute(f8_conv_small_tc_kernel<MT, NT, XS, PW>, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
        if (e != cudaSuccess) return e;
        attr_set[dev] = true;
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)p.n_tiles, (unsigned)(s.tiles / p.n_tiles));
    cfg.blockDim = dim3(SM_THREADS);
    cfg.dynamicSmemBytes = s.smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = overlap_previous ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, f8_conv_small_tc_kernel<MT, NT, XS, PW>, p);
}

}   // namespace

static bool shape_ok(const F8ConvGeom &g) {
    if (g.c % 16 != 0 || g.c_out % 4 != 0 || g.pad_h_end >= 0 || g.stride_h != g.stride_w || g.pad_h != g.pad_w) return false;
    const long long m = (long long)g.n * g.ho * g.wo, k = (long long)g.kh * g.kw * g.c;
    if (m <= 0 || m >= (1ll << 24) || k >= (1ll << 24) || g.kh >= 256 || g.kw >= 256) return false;
    // 32-bit offsets, and quotients by multiplication (n * d < 2^32)
    if ((long long)g.n * g.h * g.w * g.c >= (1ll << 32) || (m + 512) * g.c_out >= (1ll << 32) || (m + 512) * g.wo >= (1ll << 32) ||
        ((long long)g.n * g.ho + 512) * g.ho >= (1ll << 32) || (m + 15) / 16 > 65535)
        return false;
    return true;
}


// Microseconds a layer adds to a network on this kernel / on the tcgen05 kernel / on the CUDA cores, fitted to chains of equal layers
// (shapes of ResNet-18 / 50 and MobileNet V2 at batches 1 - 32, captured in a graph so that the host does not count; B200).  Examples,
// this kernel against the other: 196 x 256 x 2304 (pixels x channels x K) 3.5 / 5.9, 49 x 512 x 4608 4.3 / 8.1, 784 x 128 x 1152 2.9 / 4.4,
// 784 x 256 x 2304 5.7 / 6.8, 3136 x 64 x 576 3.2 / 3.9, 6272 x 64 x 576 4.3 / 3.9, 12544 x 64 x 64 3.4 / 3.7, 3136 x 256 x 256 4.4 / 3.8.
// Several panels: 14 x 14, 3 x 3 512 -> 512 of four images 24.4 / 9.3.
static double small_us(const Split &s) { return 0.9 + 1.75 * s.cycles / 1900 * (s.panels > 1 ? 1.4 : 1.0); }
static double tcgen05_us(const F8ConvGeom &g, bool bits8) {
    const F8TcTiles t = f8_tc_tiles(g, bits8);
    const double out = (double)g.n * g.ho * g.wo * g.c_out, width = t.kb == 128 ? 1.0 : (t.kb == 64 ? 0.6 : 0.4);
    // a chunk of K: 256-wide tiles at the tensor rate, narrow ones at the rate their activations come in
    const double chunk = t.bn > 128 ? 0.30 * width : (t.bn <= 32 ? 0.11 : (t.row_tiles ? 0.14 : 0.17)) * (t.bn > 64 ? width : 1.0);
    const double finish = 0.25 * std::max(1.0, t.bn / 64.0), rounds = std::ceil((double)t.tiles / 148);
    // (8-bit outputs of a c_out that 16 does not divide, 32-bit or second outputs of small tensors: direct stores)
    const double direct = bits8 ? (g.c_out % 16 != 0 ? 18e-6 * out : 0.0) : (g.c_out % 16 != 0 ? 16e-6 * out : (t.row_tiles ? 1.5 : 0.0));
    return 2.7 + rounds * std::max(t.chunks * chunk, finish) + finish + (out * (bits8 ? 1 : 4) + (double)g.n * g.h * g.w * g.c) / 6e6 + direct;
}
// (only the taps inside the image count there: one pixel, 3 x 3 x 800 to 24 channels 2.4 us.  Of more pixels it has no estimate but for
// filters that take a panel at a time here: 25 x 25 over 11 x 11 x 32 to 64 channels 70.6 us, here 20.0; over 3 x 3 x 48 to 40 14.4, here 29.4)
static double cuda_core_us(const F8ConvGeom &g, const Split &s) {
    if (g.h == 1 && g.w == 1) return 2.0 + 0.0095 * g.c * std::max(1.0, (double)g.n * g.ho * g.wo * g.c_out / 256);
    return s.ahead == 1 ? 2.0 + 0.0177 * g.c * std::min(g.kh, g.h) * std::min(g.kw, g.w) : 1e9;
}

// Whether a network takes this kernel for the layer, and how it is cut then.
static bool wanted(const F8ConvGeom &g, bool bits8, Split *s) {
    if (!shape_ok(g)) return false;
    if (!f8_tc_supported(g, (size_t)g.n * g.h * g.w * g.c)) return pick_split(g, s) && small_us(*s) < cuda_core_us(g, *s);
    // what every split takes at least (products at the rate of mma.sync, blocks of at most 8192 outputs): spares large layers the search
    const double out = (double)g.n * g.ho * g.wo * g.c_out, other = 0.97 * tcgen05_us(g, bits8);
    const double least = 700 + out * g.kh * g.kw * g.c / (148 * 1800.0) + 700 * std::max(0.0, out / (8192 * 148.0) - 1), limit = (other - 0.9) * (1900 / 1.75);
    if (least >= limit) return false;
    return pick_split(g, s, (float)limit * 1.0001f) && s->panels == 1 && small_us(*s) < other;
}

bool f8_small_tc_wanted(const F8ConvGeom &g, bool bits8) {
    Split s;
    return wanted(g, bits8, &s);
}

struct F8SmallPlan {
    SmallParams p;
    Split s;
    int x_signed;
};

size_t f8_small_plan_size() { return sizeof(F8SmallPlan); }

static void fill_plan(F8SmallPlan *plan, const F8ConvGeom &g, const F8Requant &q, const void *x, const int8_t *w, const int32_t *bias,
                      const void *res, void *y, const F8Sibling *sib, int tag, bool alone) {
    const Split &s = plan->s;
    plan->x_signed = g.x_signed;
    SmallParams &p = plan->p;
    p = SmallParams();
    const int bm = s.t * s.wm, bn = s.t * s.wn;
    p.M = g.n * g.ho * g.wo;
    p.c_out = g.c_out;
    p.n_tiles = (g.c_out + bn - 1) / bn;
    p.bm = bm;
    p.bn_shift = log2_of(bn);
    p.wn_shift = log2_of(s.wn);
    p.wk_shift = s.wk_shift;
    p.item_shift = log2_of(bm * bn / 4);
    p.part_shift = std::min(std::max(8 - p.item_shift, 0), s.wk_shift);
    p.h = g.h; p.w = g.w; p.c = g.c;
    p.ho = g.ho; p.wo = g.wo; p.kh = g.kh; p.kw = g.kw; p.taps = g.kh * g.kw;
    p.stride = g.stride_h; p.pad = g.pad_h;
    p.pointwise = g.kh == 1 && g.kw == 1 && g.pad_h == 0;
    p.strided = p.pointwise && g.stride_h > 1;
    p.panels = s.panels;
    p.p16 = s.p16;
    p.ahead = s.ahead;
    p.last16 = g.c / 16 - (s.panels - 1) * s.p16;
    p.wo_magic = magic_of(g.wo);
    p.ho_magic = magic_of(g.ho);
    p.kw_magic = magic_of(g.kw);
    p.k_bytes = (uint32_t)(p.taps * g.c);
    p.row_magic = magic_of(p.taps * p.p16);
    p.last_row_magic = magic_of(p.taps * p.last16);
    p.bulk = s.panels == 1 && p.k_bytes >= 512;
    p.p16_magic = magic_of(p.p16);
    p.last_magic = magic_of(p.last16);
    p.pa = (uint32_t)((p.p16 | 1) * 16);
    p.pb = (uint32_t)((p.taps * p.p16 | 1) * 16);
    const int first16 = s.panels > 1 ? p.p16 : p.last16;
    p.unit_step = SM_THREADS % first16;
    p.dst_step = SM_THREADS / first16 * (int)p.pa + p.unit_step * 16;
    p.dst_wrap = (int)p.pa - first16 * 16;
    p.status = f8_status_word();
    p.tag = tag;
    p.b_off = (uint32_t)s.window;
    p.stage = s.ahead == 2 ? (uint32_t)(s.window + s.weights) : 0u;
    // A network has checked that its sums fit 32 bits together with the constant 2^(s-1).  Of a single-layer call with a 32-bit shortcut
    // only the sums themselves do: they are rounded by the general path.
    p.plain8 = (q.y_kind == F8_U8 || q.y_kind == F8_S8) && q.s >= 1 && q.s <= 24 && !(sib && sib->y2) && !(alone && q.r_s32);
    p.mul_acc = 1 << q.sh_acc;
    p.mul_res = 1 << q.sh_res;
    p.round = p.plain8 ? 1 << (q.s - 1) : 0;
    p.x = (const uint8_t *)x; p.wgt = w; p.bias = bias; p.res = res; p.y = y;
    p.q = q;
    if (sib) p.sib = *sib;
}

cudaError_t f8_small_plan_init(F8SmallPlan *plan, const F8ConvGeom &g, const F8Requant &q, bool bits8, const void *x, const int8_t *w,
                               const int32_t *bias, const void *res, void *y, const F8Sibling *sib, int tag) {
    if (!wanted(g, bits8, &plan->s)) return cudaErrorNotSupported;
    fill_plan(plan, g, q, x, w, bias, res, y, sib, tag, false);
    return cudaSuccess;
}

static cudaError_t launch_plan(const SmallParams &p, const Split &s, bool xs, cudaStream_t st, bool overlap_previous) {
    if (p.pointwise && !p.strided && p.panels == 1) {
        if (s.t == 32) return xs ? launch_small<2, 4, true, true>(p, s, st, overlap_previous) : launch_small<2, 4, false, true>(p, s, st, overlap_previous);
        return xs ? launch_small<1, 2, true, true>(p, s, st, overlap_previous) : launch_small<1, 2, false, true>(p, s, st, overlap_previous);
    }
    if (s.t == 32) return xs ? launch_small<2, 4, true, false>(p, s, st, overlap_previous) : launch_small<2, 4, false, false>(p, s, st, overlap_previous);
    return xs ? launch_small<1, 2, true, false>(p, s, st, overlap_previous) : launch_small<1, 2, false, false>(p, s, st, overlap_previous);
}

cudaError_t f8_small_launch(const F8SmallPlan *plan, bool overlap_previous, cudaStream_t st) {
    SmallParams p = plan->p;
    p.wait_limit = f8_wait_limit_cycles();
    return launch_plan(p, plan->s, plan->x_signed != 0, st, overlap_previous);
}

// A call of its own, inputs below 16 KiB: launches and returns success, or cudaErrorNotSupported where another kernel is the better one.
// Nothing hides the start of either kernel: 4.2 us of this one (16 x 16 x 16, 3 x 3: 6.2 against 7.3 us with the tensor maps on the
// host), a tcgen05 chunk takes 0.12 us whatever its width in bytes (0.5 with 256-wide tiles, of which there are few), and its direct
// stores 6 us per MB of 32-bit, 18 per MB of 8-bit values.  31 x 31 x 16, 3 x 3 to 4096 channels 15.7 us there; 13 x 13 x 48 of two
// images to 1784 22.9.
cudaError_t f8_launch_small_alone(const F8ConvGeom &g, const F8Requant &q, bool bits8, const void *x, const int8_t *w, const int32_t *bias,
                                  const void *res, void *y, cudaStream_t st, const F8Sibling *sib) {
    const size_t x_bytes = (size_t)g.n * g.h * g.w * g.c;
    F8SmallPlan plan;
    if (x_bytes >= 16384 || !f8_tc_supported(g, x_bytes) || !shape_ok(g) || !pick_split(g, &plan.s) || plan.s.panels > 1) return cudaErrorNotSupported;
    const F8TcTiles t = f8_tc_tiles(g, bits8);
    const bool pointwise = g.kh * g.kw == 1, direct = g.c_out % 16 != 0 || (!bits8 && (!pointwise || g.c_out > 27000));
    const double chunk = t.bn <= 16 ? 0.14 : (t.bn <= 32 ? (pointwise ? 0.18 : 0.12) : (t.bn <= 64 ? 0.13 : (t.bn <= 128 ? 0.25 : 0.5)));
    const double stores = direct ? (bits8 ? 18e-6 : 24e-6) * ((double)g.n * g.ho * g.wo * g.c_out) : 0.0;
    if (small_us(plan.s) + 4.2 >= 8.0 + std::ceil((double)t.tiles / 148) * t.chunks * chunk + stores) return cudaErrorNotSupported;
    fill_plan(&plan, g, q, x, w, bias, res, y, sib, 0, true);
    plan.p.wait_first = 1;
    plan.p.wait_limit = f8_wait_limit_cycles();
    return launch_plan(plan.p, plan.s, plan.x_signed != 0, st, true);
}

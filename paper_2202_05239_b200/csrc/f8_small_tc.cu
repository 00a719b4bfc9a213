// Dense layers whose whole work is a few microseconds (single-image inference, fully connected layers, the last stages of
// small batches): an implicit GEMM built for latency instead of throughput.
//
// What bounds such a layer is the chain of hand-overs, not a pipe: the tcgen05 kernel needs 5 - 6 us from the end of the layer
// before it to its own end (tensor-map copy, MMA, accumulator read-back, staged store, drain, each a barrier away from the
// next) and cuts a 14 x 14 x 256 output into two tiles of 256 columns on two SMs.  Here a tile is 32 x 32 (64 x 64 when that
// leaves tiles enough), so that the same layer spreads over 56 SMs, and the warps of a tile divide K among themselves:
//   * 16-byte cp.async gathers of activations (zero filled outside the image) and weights into an eight-stage ring of
//     128-byte K chunks, XOR-swizzled for ldmatrix; the weights of the first stages are requested before the previous
//     layer has finished (programmatic dependent launch);
//   * eight warps: two halves of the tile's rows x four 32-byte K slices of every chunk, mma.sync m16n8k32 (u8|s8 x s8 -> s32)
//     with the accumulators in registers: no read-back, no barrier to wait for;
//   * the four partial sums meet in shared memory (integers: any order gives the same result), then bias, shortcut,
//     rounding shift, clip and a second consumer, for every output kind the library has, four channels per thread.
// mma.sync cannot reach the rate of tcgen05.mma, which is why layers with more work stay with the other kernel
// (f8_small_tc_wanted has the rule and what was measured on both sides of it).
#include <math.h>

#include <algorithm>

#include "f8_epilogue.cuh"
#include "f8_tc_ptx.cuh"

namespace {

constexpr int SM_THREADS = 256;
constexpr int SM_STAGES = 8;
constexpr int SM_KB = 128;                  // bytes of K per stage: eight 16-byte units

struct SmallParams {
    int M, c_out, n_tiles;
    int h, w, c;                            // input
    int ho, wo, kw, stride, pad_h, pad_w;
    int c16;                                // 16-byte units per tap
    int k_bytes, chunks;
    const uint8_t *x;
    const int8_t *wgt;                      // [c_out][taps * c]
    const int32_t *bias;
    const void *res;
    void *y;
    F8Requant q;
    F8Sibling sib;
};

// 16 bytes global -> shared; zero filled when !valid (the address must be a legal one even then).
__device__ __forceinline__ void cp_async16(uint32_t dst, const void *src, bool valid) {
    const int bytes = valid ? 16 : 0;
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(bytes) : "memory");
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

// Stores four consecutive channels of one output pixel for one consumer of the aligned sums v[].
__device__ __forceinline__ void store4(void *y, int y_kind, int s, int lo, int hi, const int (&v)[4], size_t o) {
    int t[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) t[j] = f8_quantize_child(v[j], y_kind, s, lo, hi);
    if (y_kind == F8_S32 || y_kind == F8_S32_RELU) *(int4 *)((int32_t *)y + o) = make_int4(t[0], t[1], t[2], t[3]);
    else *(uint32_t *)((uint8_t *)y + o) = f8_pack4(t[0], t[1], t[2], t[3]);
}

// MT: 16-row MMA tiles per warp (32 * MT rows per CTA), NT: 8-column MMA tiles per warp (8 * NT columns per CTA).
template <int MT, int NT, bool XS>
__global__ void __launch_bounds__(SM_THREADS) f8_conv_small_tc_kernel(const SmallParams p) {
    constexpr int BM = 32 * MT, BN = 8 * NT;
    constexpr int A_ROWS = BM * 8 / SM_THREADS, B_ROWS = BN * 8 / SM_THREADS;       // 16-byte units per thread and chunk
    constexpr int STAGE = (BM + BN) * SM_KB;
    constexpr int RED_ROW = BN + 4;                                                 // words per row of a partial tile
    extern __shared__ __align__(128) uint8_t smem[];
    const uint32_t smem_base = smem_u32(smem);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int m_t = (int)blockIdx.x / p.n_tiles, n_t = (int)blockIdx.x - m_t * p.n_tiles;
    const int m0 = m_t * BM, n0 = n_t * BN;
    grid_launch_dependents();

    // ---- what this thread gathers: unit `u` of rows r, r + 32, ... of both operands
    const int u = threadIdx.x & 7, r = threadIdx.x >> 3;
    const uint32_t unit_off = (uint32_t)r * SM_KB + (uint32_t)((u ^ (r & 7)) << 4);      // (rows 32 apart: the same swizzle)
    int iy0[A_ROWS], ix0[A_ROWS];
    const uint8_t *img_base[A_ROWS];
#pragma unroll
    for (int i = 0; i < A_ROWS; ++i) {
        const int m = m0 + r + 32 * i;
        const int t = m / p.wo, ox = m - t * p.wo, img = t / p.ho, oy = t - img * p.ho;
        const bool in = m < p.M;
        iy0[i] = in ? oy * p.stride - p.pad_h : -(1 << 24);          // rows past the last pixel: outside every image
        ix0[i] = ox * p.stride - p.pad_w;
        img_base[i] = p.x + (in ? (size_t)img * p.h * p.w * p.c : 0);
    }
    const int8_t *w_row[B_ROWS];
#pragma unroll
    for (int i = 0; i < B_ROWS; ++i) w_row[i] = p.wgt + (size_t)min(n0 + r + 32 * i, p.c_out - 1) * p.k_bytes;
    auto load_b = [&](int chunk) {
        const uint32_t dst = smem_base + (uint32_t)(chunk % SM_STAGES) * STAGE + BM * SM_KB + unit_off;
        const int k = chunk * SM_KB + u * 16;
#pragma unroll
        for (int i = 0; i < B_ROWS; ++i)
            cp_async16(dst + i * 32 * SM_KB, w_row[i] + (k < p.k_bytes ? k : 0), k < p.k_bytes && n0 + r + 32 * i < p.c_out);
    };
    // tap and unit of this thread's next activation gather
    int tap_y = 0, tap_x = 0, cu = u;
    auto normalise = [&]() {
        while (cu >= p.c16) {
            cu -= p.c16;
            if (++tap_x == p.kw) { tap_x = 0; ++tap_y; }
        }
    };
    normalise();
    auto load_a = [&](int chunk) {
        const uint32_t dst = smem_base + (uint32_t)(chunk % SM_STAGES) * STAGE + unit_off;
        const bool in_k = chunk * SM_KB + u * 16 < p.k_bytes;
#pragma unroll
        for (int i = 0; i < A_ROWS; ++i) {
            const int iy = iy0[i] + tap_y, ix = ix0[i] + tap_x;
            const bool ok = in_k && (unsigned)iy < (unsigned)p.h && (unsigned)ix < (unsigned)p.w;
            const uint8_t *src = ok ? img_base[i] + ((size_t)iy * p.w + ix) * p.c + cu * 16 : p.x;
            cp_async16(dst + i * 32 * SM_KB, src, ok);
        }
        cu += 8;
        normalise();
    };

    // ---- fill: weights do not depend on the previous layer, activations do
    const int ahead = min(p.chunks, SM_STAGES - 1);
    for (int i = 0; i < ahead; ++i) load_b(i);
    grid_dependency_wait();
    for (int i = 0; i < SM_STAGES - 1; ++i) {
        if (i < ahead) load_a(i);
        cp_async_commit();
    }

    const int kq = warp & 3, mh = warp >> 2;                 // K slice of a chunk, half of the tile's rows
    int acc[MT][NT][4];
#pragma unroll
    for (int i = 0; i < MT; ++i)
#pragma unroll
        for (int j = 0; j < NT; ++j)
#pragma unroll
            for (int e = 0; e < 4; ++e) acc[i][j][e] = 0;
    // ldmatrix rows of this lane: A: rows 0-15 of the 16-row tile by two 16-byte halves; B: 16 columns by two halves
    const int a_row = mh * 16 * MT + (lane & 15), a_half = lane >> 4;
    const int b_row = (lane & 7) + ((lane >> 4) << 3), b_half = (lane >> 3) & 1;
    const uint32_t a_off = (uint32_t)a_row * SM_KB + (uint32_t)(((2 * kq + a_half) ^ (a_row & 7)) << 4);
    const uint32_t b_off = BM * SM_KB + (uint32_t)b_row * SM_KB + (uint32_t)(((2 * kq + b_half) ^ (b_row & 7)) << 4);
    for (int c = 0; c < p.chunks; ++c) {
        cp_async_wait<SM_STAGES - 2>();
        __syncthreads();                                     // chunk c has landed for everybody; chunk c - 1 has been read
        const uint32_t st = smem_base + (uint32_t)(c % SM_STAGES) * STAGE;
        uint32_t b[NT / 2][4];
#pragma unroll
        for (int j = 0; j < NT / 2; ++j) ldmatrix4(st + b_off + j * 16 * SM_KB, b[j]);
#pragma unroll
        for (int i = 0; i < MT; ++i) {
            uint32_t a[4];
            ldmatrix4(st + a_off + i * 16 * SM_KB, a);
#pragma unroll
            for (int j = 0; j < NT; ++j) mma_16832<XS>(acc[i][j], a, b[j >> 1][2 * (j & 1)], b[j >> 1][2 * (j & 1) + 1]);
        }
        const int next = c + SM_STAGES - 1;
        if (next < p.chunks) {
            load_b(next);
            load_a(next);
        }
        cp_async_commit();
    }

    // ---- the four K slices meet in shared memory
    cp_async_wait<0>();
    __syncthreads();
    int *red = (int *)smem;
#pragma unroll
    for (int i = 0; i < MT; ++i)
#pragma unroll
        for (int j = 0; j < NT; ++j)
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const int row = mh * 16 * MT + i * 16 + (lane >> 2) + 8 * e, col = j * 8 + (lane & 3) * 2;
                *(int2 *)(red + ((size_t)kq * BM + row) * RED_ROW + col) = make_int2(acc[i][j][2 * e], acc[i][j][2 * e + 1]);
            }
    __syncthreads();
    for (int it = threadIdx.x; it < BM * BN / 4; it += SM_THREADS) {
        const int row = it / (BN / 4), col = (it - row * (BN / 4)) * 4;
        const int m = m0 + row, co = n0 + col;
        if (m >= p.M || co >= p.c_out) continue;
        int v[4] = {0, 0, 0, 0};
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int4 t = *(const int4 *)(red + ((size_t)k * BM + row) * RED_ROW + col);
            v[0] += t.x; v[1] += t.y; v[2] += t.z; v[3] += t.w;
        }
        if (p.bias) {
            const int4 t = __ldg((const int4 *)(p.bias + co));
            v[0] += t.x; v[1] += t.y; v[2] += t.z; v[3] += t.w;
        }
        const size_t o = (size_t)m * p.c_out + co;
        int rr[4] = {0, 0, 0, 0};
        if (p.q.has_res) {
            if (p.q.r_s32) {
                const int4 t = *(const int4 *)((const int32_t *)p.res + o);
                rr[0] = t.x; rr[1] = t.y; rr[2] = t.z; rr[3] = t.w;
            } else {
                const uint32_t t = *(const uint32_t *)((const uint8_t *)p.res + o);
#pragma unroll
                for (int j = 0; j < 4; ++j) rr[j] = f8_byte(t, j, p.q.r_signed);
            }
        }
#pragma unroll
        for (int j = 0; j < 4; ++j) v[j] = f8_align_add(v[j], rr[j], p.q);
        store4(p.y, p.q.y_kind, p.q.s, p.q.lo, p.q.hi, v, o);
        if (p.sib.y2) store4(p.sib.y2, p.sib.y_kind, p.sib.s, p.sib.lo, p.sib.hi, v, o);
    }
}

template <int MT, int NT>
constexpr size_t small_smem(int chunks) {
    const size_t stages = (size_t)(32 * MT + 8 * NT) * SM_KB * (chunks < SM_STAGES ? chunks : SM_STAGES);
    const size_t red = (size_t)4 * 32 * MT * (8 * NT + 4) * 4;
    return stages > red ? stages : red;
}

template <int MT, int NT, bool XS>
cudaError_t launch_small(SmallParams &p, cudaStream_t st, bool overlap_previous) {
    static bool attr_set[64] = {false};
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    if (!attr_set[dev]) {
        const cudaError_t e = cudaFuncSetAttribute(f8_conv_small_tc_kernel<MT, NT, XS>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                   (int)small_smem<MT, NT>(SM_STAGES));
        if (e != cudaSuccess) return e;
        attr_set[dev] = true;
    }
    p.n_tiles = (p.c_out + 8 * NT - 1) / (8 * NT);
    const long long tiles = (long long)((p.M + 32 * MT - 1) / (32 * MT)) * p.n_tiles;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)tiles);
    cfg.blockDim = dim3(SM_THREADS);
    cfg.dynamicSmemBytes = small_smem<MT, NT>(p.chunks);
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = overlap_previous ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, f8_conv_small_tc_kernel<MT, NT, XS>, p);
}

}   // namespace

bool f8_small_tc_supported(const F8ConvGeom &g) {
    if (g.c % 16 != 0 || g.c_out % 4 != 0 || g.pad_h_end >= 0 || g.stride_h != g.stride_w) return false;
    const long long m = (long long)g.n * g.ho * g.wo, k = (long long)g.kh * g.kw * g.c;
    return m > 0 && m < (1ll << 24) && k < (1ll << 24) && g.kh < 256 && g.kw < 256;
}

// Microseconds a layer takes between its neighbours on this kernel / on the tcgen05 kernel / on the CUDA cores, fitted to event timings
// of the layers of ResNet-18 / 50 and MobileNet V2 at batches 1 - 64 and of 480 layers with up to 2048 channels and filters up to 7 x 7
// (B200).  Examples, this kernel against the other: 196 x 256 x 2304 (pixels x channels x K) 10.2 / 16.3, 784 x 512 x 128 8.2 / 12.3,
// 1 x 1000 x 2048 10.4 / 77.8 (not on tensor cores before), 784 x 512 x 4608 22.5 / 22.6, 3136 x 512 x 128 14.3 / 12.1,
// 12544 x 384 x 64 22.5 / 12.2; alone, 1 x 1000 x 4096 10.5 / 13.2, 1 x 1000 x 12288 24.8 / 25.4, 1250 x 184 x 12096 40.4 / 22.7, 2240 x 48 x 25088 72.1 / 41.4, 250 x 16 x 25600 45.6 / 28.0.
// What decides beyond small sizes: a narrow tcgen05 tile costs half as much per K chunk as a 256-wide one, and this kernel's tiles
// share the way from the L2 cache, twice as slow per chunk with one tile on every SM as with a few.
static double small_us(const F8ConvGeom &g) {
    const double m = (double)g.n * g.ho * g.wo, n = g.c_out, k = (double)g.kh * g.kw * g.c;
    const double big = std::ceil(m / 64) * std::ceil(n / 64) / 148, full = std::ceil(m / 32) * std::ceil(n / 32) / 148;
    // (one row of tiles reads every weight once, and hardly any activations)
    if (m <= 32) return std::max(7.3, 5.5 + 0.0016 * k) + std::max(0.0, full - 1) * (0.6 + 0.0006 * k);
    // (64 x 64 tiles: from five chunks on the ring fills an SM, and a started round costs a whole one)
    if (big >= 1) return 7.3 + (k > 5 * SM_KB ? std::ceil(big) : big) * (1.7 + 0.0042 * k);
    return 7.3 + (full < 1 ? 0.0014 * (1 + full) : std::max(0.0028, 0.0012 * full)) * k;
}
static double tcgen05_us(const F8ConvGeom &g, bool bits8) {
    const F8TcTiles t = f8_tc_tiles(g, bits8);
    const double wide = 0.0024 * ((double)g.kh * g.kw * g.c);
    // per chunk; 256-wide tiles with a very long K wait for memory on top
    const double narrow = t.bn <= 32 ? (t.row_tiles ? 0.10 : (g.kh * g.kw == 1 ? 0.18 : 0.14)) : (t.bn <= 64 ? (t.row_tiles ? 0.13 : (bits8 ? 0.17 : 0.22)) : 0.25);
    const double tile = t.bn > 128 ? wide + 0.1 * std::max(0, t.chunks - 64) : std::min(wide, narrow * t.chunks);
    // (32-bit or two outputs of small tensors leave by direct stores)
    return (!bits8 && t.row_tiles ? 11.8 : 10.3) + std::ceil((double)t.tiles / 148) * tile;
}
// (only the tap inside the image counts there: one pixel, 3 x 3 x 800 to 24 channels 7.4 us, here 14.2)
static double cuda_core_us(const F8ConvGeom &g) {
    return g.h == 1 && g.w == 1 ? 7.0 + 0.0095 * g.c * std::max(1.0, (double)g.n * g.ho * g.wo * g.c_out / 256) : 1e9;
}

bool f8_small_tc_wanted(const F8ConvGeom &g, bool bits8) {
    if (!f8_small_tc_supported(g)) return false;
    return small_us(g) < (f8_tc_supported(g, (size_t)g.n * g.h * g.w * g.c) ? tcgen05_us(g, bits8) : cuda_core_us(g));
}

// A call of its own, inputs below 16 KiB.  Nothing hides the start of either kernel, this one's takes about 1.7 us less (16 x 16 x 16,
// 3 x 3: 6.3 against 7.3 us with the tensor maps on the host), a tcgen05 chunk takes 0.12 us whatever its width in bytes (0.5 with
// 256-wide tiles, of which there are few), and its direct stores 6 us per MB of 32-bit, 18 per MB of 8-bit values.  Fitted to 450 layers;
// 31 x 31 x 16, 3 x 3 to 4096 channels 28.9 us here, 15.7 there; 13 x 13 x 48 of two images to 1784 9.3 and 22.9.
bool f8_small_tc_wanted_alone(const F8ConvGeom &g, bool bits8) {
    const size_t x_bytes = (size_t)g.n * g.h * g.w * g.c;
    if (x_bytes >= 16384 || !f8_tc_supported(g, x_bytes) || !f8_small_tc_supported(g)) return false;
    const F8TcTiles t = f8_tc_tiles(g, bits8);
    const bool pointwise = g.kh * g.kw == 1, direct = g.c_out % 16 != 0 || (!bits8 && (!pointwise || g.c_out > 27000));
    const double chunk = t.bn <= 16 ? 0.14 : (t.bn <= 32 ? (pointwise ? 0.18 : 0.12) : (t.bn <= 64 ? 0.13 : (t.bn <= 128 ? 0.25 : 0.5)));
    const double stores = direct ? (bits8 ? 18e-6 : 24e-6) * ((double)g.n * g.ho * g.wo * g.c_out) : 0.0;
    return small_us(g) - 1.0 < 8.0 + std::ceil((double)t.tiles / 148) * t.chunks * chunk + stores;
}

cudaError_t f8_launch_small_tc(const F8ConvGeom &g, const F8Requant &q, const void *x, const int8_t *w, const int32_t *bias,
                               const void *res, void *y, cudaStream_t st, bool overlap_previous, const F8Sibling *sib) {
    SmallParams p = {};
    p.M = g.n * g.ho * g.wo;
    p.c_out = g.c_out;
    p.h = g.h; p.w = g.w; p.c = g.c;
    p.ho = g.ho; p.wo = g.wo; p.kw = g.kw;
    p.stride = g.stride_h; p.pad_h = g.pad_h; p.pad_w = g.pad_w;
    p.c16 = g.c / 16;
    p.k_bytes = g.kh * g.kw * g.c;
    p.chunks = (p.k_bytes + SM_KB - 1) / SM_KB;
    p.x = (const uint8_t *)x; p.wgt = w; p.bias = bias; p.res = res; p.y = y;
    p.q = q;
    if (sib) p.sib = *sib;
    // 64 x 64 tiles gather half as many bytes per output; 32 x 32 tiles where those would leave SMs without a tile
    const long long big = (long long)((p.M + 63) / 64) * ((g.c_out + 63) / 64);
    if (big >= 148) return g.x_signed ? launch_small<2, 8, true>(p, st, overlap_previous) : launch_small<2, 8, false>(p, st, overlap_previous);
    return g.x_signed ? launch_small<1, 4, true>(p, st, overlap_previous) : launch_small<1, 4, false>(p, st, overlap_previous);
}

// Sibling layers with private fractional lengths (Sec. 4.3 "Clipping-Level Sharing", appendix "Private Fractional
// Lengths"): a value that feeds several layers is kept in 32 bits and quantised once per consumer, each with its own
// format; the formats differ by powers of two, so each consumer's view costs a shift.  This kernel takes the int32 tensor a layer produced (format fa,
// e.g. the F8_S32 output of a convolution) and emits one or two 8-bit tensors:
//
//     y_k = clip(rshift_round(acc, fa - fl_k), lo_k, hi_k)        k = 1, 2;   rshift_round = round half up
//
// Bound by memory traffic (4 bytes read, 1 or 2 written per element).  A thread takes sixteen consecutive elements: two 32-byte
// loads (whole sectors; they do not stay in L1) and one 16-byte store per output, one pass, no loop -- the blocks that
// wait are what keeps loads in flight.  29.7 M elements, two outputs: 45.5 -> 28.9 us (6.2 TB/s; four-byte stores and a
// grid-stride loop before).  Less aligned tensors take the other two kernels.
#include "f8_epilogue.cuh"

namespace {

// (no read-only loads in this file: what is read may be written by the grid before this one while the blocks here already wait)
__device__ __forceinline__ void load32(const int32_t *p, int (&v)[8]) {
    asm volatile("ld.global.L1::no_allocate.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7])
                 : "l"(p)
                 : "memory");
}

// Four rounded, clipped and packed codes.  SHIFT: 1 <= s <= 31; else the general form (s <= 0: a left shift).
template <bool SGN, bool SHIFT>
__device__ __forceinline__ uint32_t requant4(int a, int b, int c, int d, const F8Requant &q) {
    int t[4] = {a, b, c, d};
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        t[j] = SHIFT ? f8_rshift_round(t[j], q.s) : min(max(t[j], -256), 256) << (-q.s);
        if (SGN) t[j] = max(t[j], -127);
    }
    uint32_t hi, o;
    if (SGN) {
        asm("cvt.pack.sat.s8.s32.b32 %0, %1, %2, 0;" : "=r"(hi) : "r"(t[3]), "r"(t[2]));
        asm("cvt.pack.sat.s8.s32.b32 %0, %1, %2, %3;" : "=r"(o) : "r"(t[1]), "r"(t[0]), "r"(hi));
    } else {
        asm("cvt.pack.sat.u8.s32.b32 %0, %1, %2, 0;" : "=r"(hi) : "r"(t[3]), "r"(t[2]));
        asm("cvt.pack.sat.u8.s32.b32 %0, %1, %2, %3;" : "=r"(o) : "r"(t[1]), "r"(t[0]), "r"(hi));
    }
    return o;
}
template <bool SGN, bool SHIFT>
__device__ __forceinline__ uint4 requant16(const int (&u)[8], const int (&v)[8], const F8Requant &q) {
    return make_uint4(requant4<SGN, SHIFT>(u[0], u[1], u[2], u[3], q), requant4<SGN, SHIFT>(u[4], u[5], u[6], u[7], q),
                      requant4<SGN, SHIFT>(v[0], v[1], v[2], v[3], q), requant4<SGN, SHIFT>(v[4], v[5], v[6], v[7], q));
}
__device__ __forceinline__ uint32_t requant4(const int4 &a, const F8Requant &q) {
    if (q.s > 0) return q.y_kind == F8_S8 ? requant4<true, true>(a.x, a.y, a.z, a.w, q) : requant4<false, true>(a.x, a.y, a.z, a.w, q);
    return q.y_kind == F8_S8 ? requant4<true, false>(a.x, a.y, a.z, a.w, q) : requant4<false, false>(a.x, a.y, a.z, a.w, q);
}
__device__ __forceinline__ uint4 requant16(const int (&u)[8], const int (&v)[8], const F8Requant &q) {
    if (q.s > 0) return q.y_kind == F8_S8 ? requant16<true, true>(u, v, q) : requant16<false, true>(u, v, q);
    return q.y_kind == F8_S8 ? requant16<true, false>(u, v, q) : requant16<false, false>(u, v, q);
}

// acc 32-byte, y1 / y2 16-byte aligned; the last thread takes the ragged tail.
__global__ void __launch_bounds__(256) requant_dual_kernel(const int32_t *acc, long long n, F8Requant q1, F8Requant q2,
                                                            uint8_t *__restrict__ y1, uint8_t *__restrict__ y2) {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const long long i = ((long long)blockIdx.x * 256 + threadIdx.x) * 16;
    if (i + 16 <= n) {
        int u[8], v[8];
        load32(acc + i, u);
        load32(acc + i + 8, v);
        *(uint4 *)(y1 + i) = requant16(u, v, q1);
        if (y2) *(uint4 *)(y2 + i) = requant16(u, v, q2);
    } else {
        for (long long j = i; j < n; ++j) {
            const int a = acc[j];
            y1[j] = (uint8_t)(f8_requant(a, 0, q1) & 0xff);
            if (y2) y2[j] = (uint8_t)(f8_requant(a, 0, q2) & 0xff);
        }
    }
}

// acc 16-byte, y1 / y2 4-byte aligned (views that start at a multiple of four elements): four 16-byte loads in flight per thread,
// neighbouring threads on neighbouring words.  29.7 M elements, two outputs: 30.4 us (element by
// element 78.0), one output 25.1 (64.0); with the alignment of the kernel above 29.2 and 25.1.
__global__ void __launch_bounds__(256) requant_dual_words_kernel(const int32_t *acc, long long n, F8Requant q1, F8Requant q2,
                                                                 uint8_t *__restrict__ y1, uint8_t *__restrict__ y2) {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const long long i0 = ((long long)blockIdx.x * 1024 + threadIdx.x) * 4;
    int4 a[4];
#pragma unroll
    for (int u = 0; u < 4; ++u)
        if (i0 + 1024 * u + 4 <= n) a[u] = *(const int4 *)(acc + i0 + 1024 * u);
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        const long long i = i0 + 1024 * u;
        if (i + 4 <= n) {
            *(uint32_t *)(y1 + i) = requant4(a[u], q1);
            if (y2) *(uint32_t *)(y2 + i) = requant4(a[u], q2);
        } else {
            for (long long j = i; j < n; ++j) {
                const int v = acc[j];
                y1[j] = (uint8_t)(f8_requant(v, 0, q1) & 0xff);
                if (y2) y2[j] = (uint8_t)(f8_requant(v, 0, q2) & 0xff);
            }
        }
    }
}

// Any alignment.
__global__ void __launch_bounds__(256) requant_dual_scalar_kernel(const int32_t *acc, long long n, F8Requant q1, F8Requant q2,
                                                                  uint8_t *__restrict__ y1, uint8_t *__restrict__ y2) {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const long long stride = (long long)gridDim.x * 256;
    for (long long i = (long long)blockIdx.x * 256 + threadIdx.x; i < n; i += stride) {
        const int a = acc[i];
        y1[i] = (uint8_t)(f8_requant(a, 0, q1) & 0xff);
        if (y2) y2[i] = (uint8_t)(f8_requant(a, 0, q2) & 0xff);
    }
}

bool make_q(int fa, int fl_y, int y_dtype, F8Requant *q) {
    if (y_dtype != F8_U8 && y_dtype != F8_S8) return false;
    if (fl_y < 0 || fl_y > (y_dtype == F8_U8 ? 8 : 7)) return false;
    q->sh_acc = 0; q->sh_res = 0; q->has_res = 0; q->r_signed = 0;
    q->s = fa - fl_y;
    q->y_kind = y_dtype;
    q->lo = y_dtype == F8_U8 ? 0 : -127;
    q->hi = y_dtype == F8_U8 ? 255 : 127;
    return true;
}

}   // namespace

extern "C" f8_status f8_requantize_dual_fixed(long long n, const int32_t *acc, int fa, void *y1, int y1_dtype, int fl_y1, void *y2,
                                              int y2_dtype, int fl_y2, void *cuda_stream) {
    if (!acc || !y1) return f8_set_error(F8_ERR_NULL, "acc and y1 must not be NULL");
    if (n < 0) return f8_set_error(F8_ERR_SHAPE, "n must not be negative");
    if (fa < -8 || fa > 32) return f8_set_error(F8_ERR_FL_RANGE, "accumulator format outside [-8, 32]");
    F8Requant q1, q2;
    if (!make_q(fa, fl_y1, y1_dtype, &q1)) return f8_set_error(y1_dtype == F8_U8 || y1_dtype == F8_S8 ? F8_ERR_FL_RANGE : F8_ERR_DTYPE, "y1: 8-bit dtype with fl in its range");
    q2 = q1;
    if (y2 && !make_q(fa, fl_y2, y2_dtype, &q2)) return f8_set_error(y2_dtype == F8_U8 || y2_dtype == F8_S8 ? F8_ERR_FL_RANGE : F8_ERR_DTYPE, "y2: 8-bit dtype with fl in its range");
    if (q1.s < -8 || q1.s > 31 || (y2 && (q2.s < -8 || q2.s > 31))) return f8_set_error(F8_ERR_SHIFT_RANGE, "shift fa - fl_y outside [-8, 31]");
    if (((uintptr_t)acc & 3)) return f8_set_error(F8_ERR_ALIGN, "acc must be 4-byte aligned");
    if (n == 0) return F8_OK;
    const uintptr_t y = (uintptr_t)y1 | (uintptr_t)y2;
    const long long blocks = (n + 4095) / 4096;
    cudaStream_t st = (cudaStream_t)cuda_stream;
    // the blocks may start while what is before them in the stream drains (29.7 M elements, call after call: a gap of 1 us less)
    cudaLaunchConfig_t cfg = {};
    cfg.blockDim = dim3(256);
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    cfg.gridDim = dim3((unsigned)std::min<long long>(blocks, (1ll << 31) - 1));
    cudaError_t e;
    if (((uintptr_t)acc & 31) == 0 && (y & 15) == 0 && blocks < (1ll << 31)) {
        e = cudaLaunchKernelEx(&cfg, requant_dual_kernel, acc, n, q1, q2, (uint8_t *)y1, (uint8_t *)y2);
    } else if (((uintptr_t)acc & 15) == 0 && (y & 3) == 0 && blocks < (1ll << 31)) {
        e = cudaLaunchKernelEx(&cfg, requant_dual_words_kernel, acc, n, q1, q2, (uint8_t *)y1, (uint8_t *)y2);
    } else {
        cfg.gridDim = dim3((unsigned)std::min<long long>(blocks, 148 * 16));
        e = cudaLaunchKernelEx(&cfg, requant_dual_scalar_kernel, acc, n, q1, q2, (uint8_t *)y1, (uint8_t *)y2);
    }
    if (e != cudaSuccess) return f8_set_error(F8_ERR_CUDA, cudaGetErrorString(e));
    return F8_OK;
}

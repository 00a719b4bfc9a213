// Weight "compile" step of one Conv-BN block, on the device: BatchNorm folding and scaling-factor absorption into the
// effective weight and bias (Eq. 6), choice of the weight format from the standard deviation (Eq. 1, signed branch),
// and the signed 8-bit quantiser (appendix "Double Side Quantization").
//
//     scale_i   = (gamma_i / sigma_i) * (eta_in / eta_out)
//     W_eff     = scale_i * W[i, j]                       b_eff = (beta_i - (gamma_i / sigma_i) * mu_i) / eta_out
//     FL_w      = floor(log2(40 / std(W_eff)))  clamped   std = population standard deviation of the whole tensor
//     w_q       = floor(clip(W_eff * 2^FL_w, -127, 127) + 1/2)
//     b_q       = floor(b_eff * 2^(FL_x + FL_w) + 1/2)    saturated to int32
//
// Floating point decides integer codes here, so the arithmetic is fixed: float64, one correctly rounded IEEE operation
// per step in the order written above (explicit _rn intrinsics: no contraction into fused multiply-adds), scaling by
// powers of two is exact, and floor(log2(r)) is taken from the exponent of r.  Only the summation order of the
// variance is free; it is fixed too (per-block partial sums reduced in index order), so results are reproducible.
//
// Two launches: partial sums; then format, bias and quantised weights.  Every block of the second adds the partial sums up again
// (at most 16 KB out of L2) instead of waiting for a launch of its own that does, and has its first weights in registers before
// the first launch has finished (programmatic dependent launch).  A block takes 4096 consecutive weights of the whole tensor
// at a time, whatever rows they belong to, so rows that are no multiple of that leave no block with a remainder.  The
// fp32 weights are read twice (the second time from L2 up to about 30 M weights) and one byte per weight is written.
// [512 x 4608]: 23.5 us (four launches, chunks of rows) -> 12.3 us a call.
#include <math.h>

#include <algorithm>

#include "f8_internal.h"

namespace {

constexpr int FOLD_THREADS = 256;
constexpr int FOLD_CHUNK = 4096;         // weights a block takes at a time
constexpr int FOLD_PER_THREAD = FOLD_CHUNK / FOLD_THREADS;
constexpr int FOLD_MAX_BLOCKS = 1024;
constexpr int FOLD_MAX_ROWS = 1024;      // row scales a block keeps in shared memory (a chunk of shorter rows divides per weight)

struct FoldParams {
    int c_out, k;
    long long n;                          // c_out * k
    int blocks;
    double ratio;                         // eta_in / eta_out
    double eta_out;
    int fl_x, fl_min, fl_max;
    const float *w, *gamma, *sigma, *beta, *mu;
    int8_t *w_q;
    int32_t *b_q;
    int *fl_w;
    double *partial;                      // [blocks][2]
    bool bias_last;                       // the biases overwrite gamma or sigma: in a launch behind the last use of the row scales
};

// (no read-only loads in this file: the first launch's blocks already wait while the grid before them may write these tensors)
__device__ __forceinline__ double row_scale(const FoldParams &p, int row) {
    return __dmul_rn(__ddiv_rn((double)p.gamma[row], (double)p.sigma[row]), p.ratio);
}

// Scales of the rows the chunk at e0 touches, once per chunk (false: too many rows for the table).
__device__ __forceinline__ bool stage_scales(const FoldParams &p, long long e0, double *sc, int *row0) {
    const int r0 = (int)(e0 / p.k), r1 = (int)((min(e0 + FOLD_CHUNK, p.n) - 1) / p.k);
    *row0 = r0;
    const bool fits = r1 - r0 < FOLD_MAX_ROWS;
    __syncthreads();                      // the previous chunk's scales have been used
    if (fits)
        for (int i = threadIdx.x; i <= r1 - r0; i += FOLD_THREADS) sc[i] = row_scale(p, r0 + i);
    __syncthreads();
    return fits;
}

// The 16 weights of this thread in the chunk at e0.  VEC: k is a multiple of four (a group of four lies in one row) and w is
// 16-byte aligned: groups of four, 1024 weights apart; else single weights, 256 apart.
template <bool VEC>
__device__ __forceinline__ long long fold_index(long long e0, int j) {
    return VEC ? e0 + (long long)(j >> 2) * (4 * FOLD_THREADS) + 4 * threadIdx.x + (j & 3) : e0 + (long long)j * FOLD_THREADS + threadIdx.x;
}
template <bool VEC>
__device__ __forceinline__ void load_weights(const FoldParams &p, long long e0, float (&f)[FOLD_PER_THREAD]) {
    if (VEC) {
#pragma unroll
        for (int g = 0; g < FOLD_PER_THREAD / 4; ++g) {
            const long long e = fold_index<true>(e0, 4 * g);
            const float4 t = e < p.n ? *(const float4 *)(p.w + e) : make_float4(0.f, 0.f, 0.f, 0.f);
            f[4 * g] = t.x; f[4 * g + 1] = t.y; f[4 * g + 2] = t.z; f[4 * g + 3] = t.w;
        }
    } else {
#pragma unroll
        for (int j = 0; j < FOLD_PER_THREAD; ++j) {
            const long long e = fold_index<false>(e0, j);
            f[j] = e < p.n ? p.w[e] : 0.f;
        }
    }
}
// Scale of weight j of this thread (groups of four share one when VEC).
template <bool VEC>
__device__ __forceinline__ double weight_scale(const FoldParams &p, long long e0, int j, bool table, const double *sc, int row0) {
    const long long e = fold_index<VEC>(e0, j);
    if (e >= p.n) return 0.0;
    const int row = (int)((uint32_t)e / (uint32_t)p.k);              // n < 2^31
    return table ? sc[row - row0] : row_scale(p, row);
}

// Adds s1, s2 over the block in a fixed order; the result is in every thread.
__device__ __forceinline__ void block_sum(double &s1, double &s2) {
    __shared__ double r1[FOLD_THREADS / 32], r2[FOLD_THREADS / 32];
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) {
        s1 += __shfl_xor_sync(0xffffffffu, s1, d);
        s2 += __shfl_xor_sync(0xffffffffu, s2, d);
    }
    __syncthreads();
    if ((threadIdx.x & 31) == 0) { r1[threadIdx.x >> 5] = s1; r2[threadIdx.x >> 5] = s2; }
    __syncthreads();
    s1 = s2 = 0.0;
#pragma unroll
    for (int i = 0; i < FOLD_THREADS / 32; ++i) { s1 += r1[i]; s2 += r2[i]; }
}

template <bool VEC>
__global__ void __launch_bounds__(FOLD_THREADS) fold_stats_kernel(const FoldParams p) {
    __shared__ double sc[FOLD_MAX_ROWS];
    // (in this order: the launch behind reads the inputs before its own wait)
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    double s1 = 0.0, s2 = 0.0;
    for (long long e0 = (long long)blockIdx.x * FOLD_CHUNK; e0 < p.n; e0 += (long long)gridDim.x * FOLD_CHUNK) {
        float f[FOLD_PER_THREAD];
        load_weights<VEC>(p, e0, f);
        int row0;
        const bool table = stage_scales(p, e0, sc, &row0);
        double scale = 0.0;
#pragma unroll
        for (int j = 0; j < FOLD_PER_THREAD; ++j) {
            if (!VEC || (j & 3) == 0) scale = weight_scale<VEC>(p, e0, j, table, sc, row0);
            const double v = __dmul_rn(scale, (double)f[j]);
            s1 += v;
            s2 += v * v;
        }
    }
    block_sum(s1, s2);
    if (threadIdx.x == 0) {
        p.partial[2 * blockIdx.x] = s1;
        p.partial[2 * blockIdx.x + 1] = s2;
    }
}

// Biases, one thread each.
__device__ __forceinline__ void write_biases(const FoldParams &p, int fl) {
    const int fa = p.fl_x + fl;
    for (int i = (int)(blockIdx.x * FOLD_THREADS + threadIdx.x); i < p.c_out; i += (int)gridDim.x * FOLD_THREADS) {
        const double gs = __ddiv_rn((double)p.gamma[i], (double)p.sigma[i]);
        const double be = __ddiv_rn(__dsub_rn((double)p.beta[i], __dmul_rn(gs, (double)p.mu[i])), p.eta_out);
        double t = floor(__dadd_rn(scalbn(be, fa), 0.5));
        t = fmin(fmax(t, -2147483648.0), 2147483647.0);
        p.b_q[i] = (int32_t)t;
    }
}

template <bool VEC>
__global__ void __launch_bounds__(FOLD_THREADS) fold_quant_kernel(const FoldParams p) {
    __shared__ double sc[FOLD_MAX_ROWS];
    __shared__ int fl_s;
    // the inputs were complete before the first launch started; what that launch writes is read behind the wait
    long long e0 = (long long)blockIdx.x * FOLD_CHUNK;
    float f[FOLD_PER_THREAD];
    load_weights<VEC>(p, e0, f);
    int row0;
    bool table = stage_scales(p, e0, sc, &row0);
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    double s1 = 0.0, s2 = 0.0;
    for (int b = threadIdx.x; b < p.blocks; b += FOLD_THREADS) {
        s1 += p.partial[2 * b];
        s2 += p.partial[2 * b + 1];
    }
    block_sum(s1, s2);
    if (threadIdx.x == 0) {
        const double n = (double)p.n;
        const double mean = s1 / n;
        double var = s2 / n - mean * mean;
        if (!(var > 0.0)) var = 0.0;
        const double sd = sqrt(var);
        int fl = p.fl_max;                                   // a constant tensor: the finest format allowed
        if (sd > 0.0) {
            const double r = __ddiv_rn(40.0, sd);            // Eq. 1, signed: floor(log2(40 / sigma)) = exponent of r
            fl = isfinite(r) ? ilogb(r) : p.fl_max;
        }
        fl = max(p.fl_min, min(p.fl_max, fl));
        fl_s = fl;
        if (blockIdx.x == 0) *p.fl_w = fl;
    }
    __syncthreads();
    const int fl = fl_s;
    const double pow2 = scalbn(1.0, fl);          // multiplying by a power of two is exact
    if (!p.bias_last) write_biases(p, fl);
    while (true) {
        double scale = 0.0;
        uint32_t packed = 0;
#pragma unroll
        for (int j = 0; j < FOLD_PER_THREAD; ++j) {
            if (!VEC || (j & 3) == 0) scale = weight_scale<VEC>(p, e0, j, table, sc, row0);
            // floor is monotone and the bounds are whole numbers: clipping behind it is clipping in front of it
            const double v = __dmul_rn(__dmul_rn(scale, (double)f[j]), pow2);
            const int q = min(max(__double2int_rd(__dadd_rn(v, 0.5)), -127), 127);
            const long long e = fold_index<VEC>(e0, j);
            if (VEC) {
                packed |= (uint32_t)(q & 0xff) << (8 * (j & 3));
                if ((j & 3) == 3) {
                    if (e < p.n) *(uint32_t *)(p.w_q + e - 3) = packed;
                    packed = 0;
                }
            } else if (e < p.n) {
                p.w_q[e] = (int8_t)q;
            }
        }
        e0 += (long long)gridDim.x * FOLD_CHUNK;
        if (e0 >= p.n) break;
        load_weights<VEC>(p, e0, f);
        table = stage_scales(p, e0, sc, &row0);
    }
}

__global__ void __launch_bounds__(FOLD_THREADS) fold_bias_kernel(const FoldParams p) { write_biases(p, *p.fl_w); }

template <bool VEC>
cudaError_t launch_fold(const FoldParams &p, cudaStream_t st) {
    // both launches may start while what is before them in the stream drains
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)p.blocks);
    cfg.blockDim = dim3(FOLD_THREADS);
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    cudaError_t e = cudaLaunchKernelEx(&cfg, fold_stats_kernel<VEC>, p);
    if (e == cudaSuccess) e = cudaLaunchKernelEx(&cfg, fold_quant_kernel<VEC>, p);
    if (e == cudaSuccess && p.bias_last) fold_bias_kernel<<<(p.c_out + FOLD_THREADS - 1) / FOLD_THREADS, FOLD_THREADS, 0, st>>>(p);
    return e;
}

}   // namespace

extern "C" {

size_t f8_fold_workspace_bytes(const f8_fold_desc *d) {
    (void)d;
    return 2 * FOLD_MAX_BLOCKS * sizeof(double);
}

f8_status f8_fold_quantize_fixed(const f8_fold_desc *d, const float *w, const float *gamma, const float *sigma,
                                 const float *beta, const float *mu, int8_t *w_q, int32_t *bias_q, int *fl_w,
                                 void *workspace, size_t workspace_bytes, void *cuda_stream) {
    if (!d || !w || !gamma || !sigma || !beta || !mu || !w_q || !bias_q || !fl_w) return f8_set_error(F8_ERR_NULL, "a required pointer is NULL");
    if (d->c_out <= 0 || d->k <= 0 || (long long)d->c_out * d->k >= (1ll << 31)) return f8_set_error(F8_ERR_SHAPE, "c_out and k must be positive and c_out * k below 2^31");
    if (d->fl_x < 0 || d->fl_x > 8 || d->fl_w_min < -8 || d->fl_w_max > 24 || d->fl_w_min > d->fl_w_max)
        return f8_set_error(F8_ERR_FL_RANGE, "fl_x must lie in [0, 8] and [fl_w_min, fl_w_max] inside [-8, 24]");
    if (!(d->eta_in > 0.0) || !(d->eta_out > 0.0) || !isfinite(d->eta_in) || !isfinite(d->eta_out))
        return f8_set_error(F8_ERR_SHAPE, "eta_in and eta_out must be positive and finite");
    if (!workspace || workspace_bytes < f8_fold_workspace_bytes(d)) return f8_set_error(F8_ERR_WORKSPACE, "workspace smaller than f8_fold_workspace_bytes()");
    if (((uintptr_t)workspace & 7) || ((uintptr_t)w & 3) || ((uintptr_t)bias_q & 3) || ((uintptr_t)fl_w & 3))
        return f8_set_error(F8_ERR_ALIGN, "workspace must be 8-byte aligned, w / bias_q / fl_w 4-byte aligned");
    FoldParams p;
    p.c_out = d->c_out; p.k = d->k;
    p.n = (long long)d->c_out * d->k;
    p.blocks = (int)std::min<long long>((p.n + FOLD_CHUNK - 1) / FOLD_CHUNK, FOLD_MAX_BLOCKS);
    p.ratio = d->eta_in / d->eta_out;
    p.eta_out = d->eta_out;
    p.fl_x = d->fl_x; p.fl_min = d->fl_w_min; p.fl_max = d->fl_w_max;
    const bool vec4 = d->k % 4 == 0 && ((uintptr_t)w & 15) == 0 && ((uintptr_t)w_q & 3) == 0;
    p.w = w; p.gamma = gamma; p.sigma = sigma; p.beta = beta; p.mu = mu;
    p.w_q = w_q; p.b_q = bias_q; p.fl_w = fl_w; p.partial = (double *)workspace;
    const size_t row_bytes = (size_t)d->c_out * 4;
    auto meets = [&](const float *v) { return (uintptr_t)v < (uintptr_t)bias_q + row_bytes && (uintptr_t)bias_q < (uintptr_t)v + row_bytes; };
    p.bias_last = meets(gamma) || meets(sigma);
    cudaError_t e = vec4 ? launch_fold<true>(p, (cudaStream_t)cuda_stream) : launch_fold<false>(p, (cudaStream_t)cuda_stream);
    if (e == cudaSuccess) e = cudaGetLastError();
    if (e != cudaSuccess) return f8_set_error(F8_ERR_CUDA, cudaGetErrorString(e));
    return F8_OK;
}

}   // extern "C"

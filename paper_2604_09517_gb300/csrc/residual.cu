// hpl_scaled_residual: ||Ax - b||_inf / (eps (||A||_inf ||x||_inf + ||b||_inf) n),
// eps = 2^-53, FP64 (the standard HPL acceptance test; the paper prints no
// formula). A is read, or regenerated from the seed (hpl_generate's
// definition) so that very large systems need not keep a copy of A.
//
// Pass 1: grid (row blocks, column chunks); each thread owns one row
// and sums a_ij x_j and |a_ij| over its chunk (deterministic per-chunk
// partials). Pass 2: per row, the chunks are summed in order, b_i is
// subtracted and the maxima are combined with an integer atomicMax on the bit
// patterns of non-negative doubles (order-independent). Pass 3: the quotient.
#include <algorithm>

#include "common.cuh"

namespace hplgb {

constexpr int kResChunks = 16;

__host__ __device__ __forceinline__ uint64_t res_mix(uint64_t z) {
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}

__device__ __forceinline__ double res_u128_to_double(uint64_t hi, uint64_t lo) {
    if (hi == 0) return __ull2double_rn(lo);
    int sh = 64 - __clzll((long long)hi);
    uint64_t top = (sh == 64) ? hi : ((hi << (64 - sh)) | (lo >> sh));
    uint64_t dropped = (sh == 64) ? lo : (lo & ((1ull << sh) - 1));
    top |= (dropped != 0);
    return ldexp(__ull2double_rn(top), sh);
}

struct ResWs {
    double* part_r;      // [chunks][n]
    double* part_a;      // [chunks][n]
    uint64_t* part_lo;   // [chunks][n] (regenerated dominant matrices)
    uint64_t* part_hi;   // [chunks][n]
    unsigned long long* maxima;   // [4]: |r|, row sum, |x|, |b|
};

static size_t res_ws_layout(int64_t n, ResWs* w, char* base) {
    size_t off = 0;
    auto take = [&](size_t bytes) {
        size_t o = off;
        off = align_up(off + bytes, 256);
        return base ? (void*)(base + o) : (void*)nullptr;
    };
    void* a = take(sizeof(double) * kResChunks * n);
    void* b = take(sizeof(double) * kResChunks * n);
    void* c = take(sizeof(uint64_t) * kResChunks * n);
    void* d = take(sizeof(uint64_t) * kResChunks * n);
    void* e = take(sizeof(unsigned long long) * 4);
    if (w) {
        w->part_r = (double*)a;
        w->part_a = (double*)b;
        w->part_lo = (uint64_t*)c;
        w->part_hi = (uint64_t*)d;
        w->maxima = (unsigned long long*)e;
    }
    return off;
}

// |a| as a float with the mantissa truncated to 23 bits, by integer
// operations only: on this part FP64 arithmetic (2 FMA/clk/SM) bounds an n^2
// FP64 matrix-vector product, so the norm's row sums stay off the FP64 pipe
// (relative error below 2^-23 per term; entries below the FP32 range count 0).
__device__ __forceinline__ float abs_as_float(double a) {
    const unsigned long long u = (unsigned long long)__double_as_longlong(a) & 0x7fffffffffffffffull;
    const int e = (int)(u >> 52) - 1023 + 127;
    if (e <= 0) return 0.0f;
    if (e >= 255) return __int_as_float(0x7f800000);
    return __int_as_float((e << 23) | (int)((u >> 29) & 0x7fffff));
}

// A stored. NORM sums |a_ij| along the rows as well, in FP64 (the HPL acceptance
// check); without it this is the plain matrix-vector product of the refinement.
// The product alone is within 10 % of the FP64 pipe's time (n = 16384: 471 us,
// 426 at two FMA a clock and SM; 321 for reading A). A warp per block: all blocks are resident at once up to
// n = 9700 and the SMs' shares differ least (32 / 64 / 256 rows per block: n =
// 4096 43 / 54 / 60 us, 8192 125 / 126 / 144, 16384 471 / 477 / 514, 49152 4025 /
// 4055 / 4153); four pairs of columns in flight (two: 16384 567 us; eight gain 1 to
// 5 % above 20000 rows and lose up to 8 % below).
constexpr int kStoredRows = 32;
constexpr int kStoredUnroll = 4;      // pairs of columns in flight
template <bool NORM>
__global__ void __launch_bounds__(kStoredRows) k_res_stored(int64_t n, const double* __restrict__ A,
                                                            int64_t lda, const double* __restrict__ x, ResWs w) {
    const int64_t i = (int64_t)blockIdx.x * kStoredRows + threadIdx.x;
    const int chunk = blockIdx.y;
    const int64_t cw = (n + kResChunks - 1) / kResChunks;
    const int64_t j0 = chunk * cw, j1 = std::min<int64_t>(n, j0 + cw);
    if (i >= n) return;
    double r = 0.0, s = 0.0;
    if (NORM) {
#pragma unroll 8
        for (int64_t j = j0; j < j1; j++) {
            double a = A[j * lda + i];
            r = fma(a, x[j], r);
            s += fabs(a);
        }
    } else {
        // two interleaved FP64 accumulators shorten the dependent FMA chain
        double r1 = 0.0;
        int64_t j = j0;
#pragma unroll kStoredUnroll
        for (; j + 1 < j1; j += 2) {
            double a0 = A[j * lda + i], a1 = A[(j + 1) * lda + i];
            r = fma(a0, x[j], r);
            r1 = fma(a1, x[j + 1], r1);
        }
        if (j < j1) r = fma(A[j * lda + i], x[j], r);
        r += r1;
    }
    w.part_r[chunk * n + i] = r;
    if (NORM) {
        w.part_a[chunk * n + i] = s;
        w.part_lo[chunk * n + i] = 0;
        w.part_hi[chunk * n + i] = 0;
    }
}

// The entries regenerated from key (hpl_generate's definition), with their FP64
// row sums; for the dominant matrix the diagonal is skipped here and added per
// row later from the exact row sums accumulated here.
__global__ void __launch_bounds__(256) k_res_partial(int64_t n, uint64_t key, int dominant,
                                                     const double* __restrict__ x, ResWs w) {
    const int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x;
    const int chunk = blockIdx.y;
    const int64_t cw = (n + kResChunks - 1) / kResChunks;
    const int64_t j0 = chunk * cw, j1 = std::min<int64_t>(n, j0 + cw);
    if (i >= n) return;
    double r = 0.0, s = 0.0;
    uint64_t lo = 0, hi = 0;
    const uint64_t step = (uint64_t)n * 0x9E3779B97F4A7C15ull;
    uint64_t z = key + ((uint64_t)j0 * (uint64_t)n + (uint64_t)i + 1) * 0x9E3779B97F4A7C15ull;
    for (int64_t j = j0; j < j1; j++, z += step) {
        uint64_t h = res_mix(z);
        double a = gen_value(h);
        if (dominant) {
            uint64_t m = h >> 11, u = m >= (1ull << 52) ? m - (1ull << 52) : (1ull << 52) - m;
            uint64_t nl = lo + u;
            hi += (nl < lo);
            lo = nl;
            if (j == i) continue;     // the diagonal is added once the row sum is known
        }
        r = fma(a, x[j], r);
        s += fabs(a);
    }
    w.part_r[chunk * n + i] = r;
    w.part_a[chunk * n + i] = s;
    w.part_lo[chunk * n + i] = lo;
    w.part_hi[chunk * n + i] = hi;
}

// The plain product with the regenerated dominant matrix, its diagonal left out
// (k_res_rows and k_res_vec add diag_i x_i). Nothing is read but x, and the
// FP64 pipe (a warp instruction in 16 clocks of the SM) bounds it, so an entry
// costs one FP64 instruction, the FMA: a conversion of the integer entry would
// be a second one, and the entry's bits are built by some 35 integer
// instructions (generator included) that issue in the shadow of the FMA.
// Every term and the order of the additions are those of the sum with the
// entries converted from integers (two FP64 instructions an entry), so the bits
// are too. x is staged through shared memory: read from global memory at its
// use, its latency stood in every step (2049 rows: 26 us instead of 14).
// n = 65536: 16.2 -> 7.7 ms with the row sums over the chunks (6.8 is the FP64
// pipe's), 9001: 0.35 -> 0.19, 4097: 0.092 -> 0.062, 2049 and below the same. Steps of 2
// and 8: 7.9 and 7.4 ms; 8 rounds short chunks up further.
constexpr int kRegenStep = 4;         // entries in flight per thread
__global__ void __launch_bounds__(256) k_res_regen(int64_t n, uint64_t key, const double* __restrict__ x, ResWs w) {
    __shared__ double s_x[256];
    const int64_t i0 = (int64_t)blockIdx.x * 256, i = i0 + threadIdx.x;
    const int chunk = blockIdx.y;
    const int64_t cw = (n + kResChunks - 1) / kResChunks;
    const int64_t j0 = chunk * cw, j1 = std::min<int64_t>(n, j0 + cw);
    const uint64_t gamma = 0x9E3779B97F4A7C15ull, step = (uint64_t)n * gamma;
    uint64_t z = key + ((uint64_t)j0 * (uint64_t)n + (uint64_t)i + 1) * gamma;
    double r[2] = {0.0, 0.0};                            // even and odd columns of the chunk
    for (int64_t jt = j0; jt < j1; jt += 256) {
        __syncthreads();
        s_x[threadIdx.x] = jt + threadIdx.x < j1 ? x[jt + threadIdx.x] : 0.0;
        __syncthreads();
        const int cols = (int)std::min<int64_t>(256, j1 - jt);
        const int d = (int)std::max<int64_t>(-1, std::min<int64_t>(i - jt, 512));   // the diagonal's place in the tile
        const bool off = jt + 256 <= i0 || jt >= i0 + 256;                          // none of the block's rows has it here
        for (int c = 0; c < cols; c += kRegenStep, z += kRegenStep * step) {        // beyond cols x is 0
            double a[kRegenStep];
            unsigned least = ~0u;
#pragma unroll
            for (int u = 0; u < kRegenStep; u++) {
                unsigned top;
                a[u] = gen_value_top(res_mix(z + u * step), top);
                least = min(least, top);
            }
            if (least == 0)
                for (int u = 0; u < kRegenStep; u++) a[u] = gen_value_any(res_mix(z + u * step));
            if (!off)
#pragma unroll
                for (int u = 0; u < kRegenStep; u++) a[u] = c + u == d ? 0.0 : a[u];
#pragma unroll
            for (int u = 0; u < kRegenStep; u++) r[u & 1] = fma(a[u], s_x[c + u], r[u & 1]);
        }
    }
    if (i < n) w.part_r[chunk * n + i] = r[0] + r[1];
}

__device__ __forceinline__ void atomic_max_nonneg(unsigned long long* p, double v) {
    atomicMax(p, (unsigned long long)__double_as_longlong(v));
}

// regen_dominant: the diagonal was skipped by k_res_partial; it is diag[i] if
// diag is given, else the row's exact sum of |a_ij| rounded once. anorm: a
// known ||A||_inf (the row sums were not formed; diag given), else NULL. rout:
// receives b - A x if given.
__global__ void __launch_bounds__(256) k_res_rows(int64_t n, int regen_dominant, const double* __restrict__ diag,
                                                  const double* __restrict__ anorm, const double* __restrict__ x,
                                                  const double* __restrict__ b, ResWs w, double* __restrict__ rout) {
    const int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x;
    double mr = 0.0, ma = 0.0, mx = 0.0, mb = 0.0;
    if (i < n) {
        double r = 0.0, s = 0.0;
        uint64_t lo = 0, hi = 0;
        for (int c = 0; c < kResChunks; c++) r += w.part_r[c * n + i];
        if (!anorm) {
            for (int c = 0; c < kResChunks; c++) {
                s += w.part_a[c * n + i];
                uint64_t nl = lo + w.part_lo[c * n + i];
                hi += w.part_hi[c * n + i] + (nl < lo);
                lo = nl;
            }
        }
        if (regen_dominant) {
            double d = diag ? diag[i] : res_u128_to_double(hi, lo) * 0x1p-53;
            r = fma(d, x[i], r);
            s += d;
        }
        r = b[i] - r;
        if (rout) rout[i] = r;
        mr = fabs(r);
        ma = anorm ? *anorm : s;
        mx = fabs(x[i]);
        mb = fabs(b[i]);
    }
    // NaN compares false everywhere; flag it through the |r| slot as +Inf bits
    if (mr != mr) mr = __longlong_as_double(0x7ff0000000000000LL);
    for (int off = 16; off > 0; off >>= 1) {
        mr = fmax(mr, __shfl_down_sync(0xffffffffu, mr, off));
        ma = fmax(ma, __shfl_down_sync(0xffffffffu, ma, off));
        mx = fmax(mx, __shfl_down_sync(0xffffffffu, mx, off));
        mb = fmax(mb, __shfl_down_sync(0xffffffffu, mb, off));
    }
    if ((threadIdx.x & 31) == 0) {
        atomic_max_nonneg(&w.maxima[0], mr);
        atomic_max_nonneg(&w.maxima[1], ma);
        atomic_max_nonneg(&w.maxima[2], mx);
        atomic_max_nonneg(&w.maxima[3], mb);
    }
}

__global__ void k_res_final(int64_t n, const unsigned long long* maxima, double* out) {
    double mr = __longlong_as_double((long long)maxima[0]);
    double ma = __longlong_as_double((long long)maxima[1]);
    double mx = __longlong_as_double((long long)maxima[2]);
    double mb = __longlong_as_double((long long)maxima[3]);
    *out = mr / (0x1p-53 * (ma * mx + mb) * (double)n);
}

// Residual vector and matrix-vector product for the refinement loop: after
// k_res_partial, r_i = b_i - sum of the row's partials (b != NULL) or
// r_i = sum of the partials (b == NULL, i.e. r = A x); diag != NULL adds the
// diagonal term diag_i x_i that a regenerating k_res_partial skipped.
__global__ void __launch_bounds__(256) k_res_vec(int64_t n, const double* __restrict__ diag,
                                                 const double* __restrict__ x, const double* __restrict__ b, ResWs w,
                                                 double* __restrict__ r) {
    const int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x;
    if (i >= n) return;
    double s = 0.0;
    for (int c = 0; c < kResChunks; c++) s += w.part_r[c * n + i];
    if (diag) s = fma(diag[i], x[i], s);
    r[i] = b ? b[i] - s : s;
}

// Transposed residual for the adjoint solve: one warp per column j of A,
// r_j = b_j - sum_i a_ij x_i (b != NULL) or r_j = sum_i a_ij x_i (b == NULL),
// and the column sums of |a_ij| (the row sums of A^T) into part_a[0..n).
__global__ void __launch_bounds__(256) k_res_cols_t(int64_t n, const double* __restrict__ A, int64_t lda,
                                                    const double* __restrict__ x, const double* __restrict__ b,
                                                    double* __restrict__ r, double* __restrict__ csum,
                                                    int want_norm) {
    const int lane = threadIdx.x & 31;
    const int64_t j = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5);
    if (j >= n) return;
    const double* col = A + j * lda;
    double s = 0.0;
    float a = 0.0f;
    if (want_norm) {
#pragma unroll 4
        for (int64_t i = lane; i < n; i += 32) {
            double v = col[i];
            s = fma(v, x[i], s);
            a += abs_as_float(v);
        }
    } else {
#pragma unroll 4
        for (int64_t i = lane; i < n; i += 32) s = fma(col[i], x[i], s);
    }
    for (int off = 16; off > 0; off >>= 1) {
        s += __shfl_down_sync(0xffffffffu, s, off);
        a += __shfl_down_sync(0xffffffffu, a, off);
    }
    if (lane == 0) {
        r[j] = b ? b[j] - s : s;
        csum[j] = a;
    }
}

// anorm_in: a known ||A^T||_inf (csum not formed), else NULL; anorm_out: if
// given (and zeroed), receives max_i csum[i] for later calls.
__global__ void __launch_bounds__(256) k_res_max_t(int64_t n, const double* __restrict__ r,
                                                   const double* __restrict__ csum,
                                                   const double* __restrict__ anorm_in,
                                                   unsigned long long* anorm_out, const double* __restrict__ x,
                                                   const double* __restrict__ b, unsigned long long* maxima) {
    const int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x;
    double mr = 0.0, ma = 0.0, mx = 0.0, mb = 0.0;
    if (i < n) {
        mr = fabs(r[i]);
        ma = anorm_in ? *anorm_in : csum[i];
        mx = fabs(x[i]);
        mb = fabs(b[i]);
    }
    if (mr != mr) mr = __longlong_as_double(0x7ff0000000000000LL);
    for (int off = 16; off > 0; off >>= 1) {
        mr = fmax(mr, __shfl_down_sync(0xffffffffu, mr, off));
        ma = fmax(ma, __shfl_down_sync(0xffffffffu, ma, off));
        mx = fmax(mx, __shfl_down_sync(0xffffffffu, mx, off));
        mb = fmax(mb, __shfl_down_sync(0xffffffffu, mb, off));
    }
    if ((threadIdx.x & 31) == 0) {
        atomic_max_nonneg(&maxima[0], mr);
        atomic_max_nonneg(&maxima[1], ma);
        atomic_max_nonneg(&maxima[2], mx);
        atomic_max_nonneg(&maxima[3], mb);
        if (anorm_out) atomic_max_nonneg(anorm_out, ma);
    }
}

// r = b - A^T x (or A^T x when b == NULL), with the scaled residual of the
// transposed system (||A^T||_inf = max column sum of |A|) into sr if given.
// anorm (device double) caches that norm across calls: norm_mode 0 ignores
// it, 1 computes the norm and stores it there, 2 uses the stored value.
int launch_residual_vec_t(int64_t n, const double* A, int64_t lda, double* anorm, int norm_mode, const double* x,
                          const double* b, double* r, double* sr, void* ws, cudaStream_t s) {
    ResWs w;
    res_ws_layout(n, &w, (char*)ws);
    const bool use = norm_mode == 2 && anorm, store = norm_mode == 1 && anorm;
    k_res_cols_t<<<(unsigned)((n + 7) / 8), 256, 0, s>>>(n, A, lda, x, b, r, w.part_a, sr && b && !use);
    HPL_LAUNCH_CHECK();
    if (sr && b) {
        HPL_CUDA_TRY(cudaMemsetAsync(w.maxima, 0, sizeof(unsigned long long) * 4, s));
        if (store) HPL_CUDA_TRY(cudaMemsetAsync(anorm, 0, sizeof(double), s));
        k_res_max_t<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(n, r, w.part_a, use ? anorm : nullptr,
                                                                store ? (unsigned long long*)anorm : nullptr, x, b,
                                                                w.maxima);
        HPL_LAUNCH_CHECK();
        k_res_final<<<1, 1, 0, s>>>(n, w.maxima, sr);
        HPL_LAUNCH_CHECK();
    }
    return HPL_OK;
}

size_t residual_ws_bytes(int64_t n) { return res_ws_layout(n > 0 ? n : 1, nullptr, nullptr); }

// r = b - A x (b != NULL) or r = A x (b == NULL), A stored column-major (FP64),
// or, with A == NULL, the dominant generated matrix of key (the generator's
// stream key) regenerated entry by entry with its diagonal taken from diag.
// With sr != NULL (and b != NULL) also the scaled residual of x, with
// ||A||_inf read from anorm (device).
int launch_residual_vec(int64_t n, const double* A, int64_t lda, uint64_t key, const double* diag,
                        const double* anorm, const double* x, const double* b, double* r, double* sr, void* ws,
                        cudaStream_t s) {
    if ((!A && !diag) || (sr && !anorm)) return HPL_ERR_INVALID;
    ResWs w;
    res_ws_layout(n, &w, (char*)ws);
    const double* dg = A ? nullptr : diag;
    const dim3 g1((unsigned)((n + 255) / 256), kResChunks);
    const dim3 gs((unsigned)((n + kStoredRows - 1) / kStoredRows), kResChunks);
    if (A) k_res_stored<false><<<gs, kStoredRows, 0, s>>>(n, A, lda, x, w);
    else k_res_regen<<<g1, 256, 0, s>>>(n, key, x, w);
    HPL_LAUNCH_CHECK();
    if (!(sr && b)) {
        k_res_vec<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(n, dg, x, b, w, r);
        HPL_LAUNCH_CHECK();
    } else {
        HPL_CUDA_TRY(cudaMemsetAsync(w.maxima, 0, sizeof(unsigned long long) * 4, s));
        k_res_rows<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(n, dg != nullptr, dg, anorm, x, b, w, r);
        HPL_LAUNCH_CHECK();
        k_res_final<<<1, 1, 0, s>>>(n, w.maxima, sr);
        HPL_LAUNCH_CHECK();
    }
    return HPL_OK;
}

// Shared by the mixed-precision solver: computes the scaled residual into out.
int launch_scaled_residual(int64_t n, const double* A, int64_t lda, uint64_t seed, int kind, const double* x,
                           const double* b, double* out, void* ws, cudaStream_t s) {
    ResWs w;
    res_ws_layout(n, &w, (char*)ws);
    HPL_CUDA_TRY(cudaMemsetAsync(w.maxima, 0, sizeof(unsigned long long) * 4, s));
    uint64_t key = res_mix(seed + 1ull * 0x9E3779B97F4A7C15ull);    // stream 0 of the generator
    const dim3 g1((unsigned)((n + 255) / 256), kResChunks);
    const dim3 gs((unsigned)((n + kStoredRows - 1) / kStoredRows), kResChunks);
    if (A) k_res_stored<true><<<gs, kStoredRows, 0, s>>>(n, A, lda, x, w);
    else k_res_partial<<<g1, 256, 0, s>>>(n, key, kind == HPL_GEN_DIAG_DOMINANT, x, w);
    HPL_LAUNCH_CHECK();
    k_res_rows<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(n, !A && kind == HPL_GEN_DIAG_DOMINANT, nullptr, nullptr,
                                                           x, b, w, nullptr);
    HPL_LAUNCH_CHECK();
    k_res_final<<<1, 1, 0, s>>>(n, w.maxima, out);
    HPL_LAUNCH_CHECK();
    return HPL_OK;
}

}  // namespace hplgb

using namespace hplgb;

extern "C" size_t hpl_residual_workspace_size(int64_t n) { return residual_ws_bytes(n); }

extern "C" int hpl_scaled_residual(int64_t n, const double* A, int64_t lda, uint64_t seed, int kind, const double* x,
                                   const double* b, double* out, void* ws, size_t ws_bytes, void* stream) {
    if (n <= 0 || !x || !b || !out) return HPL_ERR_INVALID;
    if (A && lda < n) return HPL_ERR_INVALID;
    if (kind != HPL_GEN_GENERAL && kind != HPL_GEN_DIAG_DOMINANT) return HPL_ERR_INVALID;
    if (!ws || ws_bytes < residual_ws_bytes(n)) return HPL_ERR_NOMEM;
    if ((uintptr_t)ws & 255) return HPL_ERR_INVALID;
    return launch_scaled_residual(n, A, lda, seed, kind, x, b, out, ws, (cudaStream_t)stream);
}

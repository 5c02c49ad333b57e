// FP64 products for several right-hand sides on the BF16 tensor cores: the
// block residual's op(A) X and the adjoint's outer product (mxp.cu), both
// contractions that the FP64 pipe (2 FMA per clock and SM) would bound.
//
// Sliced products after Ozaki, Ogita, Oishi & Rump, "Error-free
// transformations of matrix multiplication by using fast routines of matrix
// multiplication" (2012), as in the emulated LU update, but exact to the end:
//  * Index k of the contraction is scaled by 2^xk so that B's row k lies below
//    1 (a diagonal scaling by powers of two that cancels in the product: rows
//    of B far apart in size lose nothing). Row i of A and column j of B are
//    then cut, below their largest entry, into 11 integer slices of 6 bits
//    (64 bits in all; exact in BF16).
//  * Slice products s + t = g, g = 2 .. 12, are summed per g in FP32 in tensor
//    memory: over 256 k at most 11 * 256 products below 2^12, so every partial
//    sum is an integer below 2^24 and exact. After each 256 k the 11 sums move
//    into two 64-bit integers per entry, exactly; one rounding to FP64 at the
//    end of the K slice. What is lost is below 2^-61.8 2^(eA + eB) per term, with
//    2^eA and 2^eB the powers of two above the row's and the column's maximum.
//  * FP64 arithmetic loses up to 2^-53 of sum |a||b| per term, which is far less
//    when the large entries of the row meet only small ones of the column (two
//    weakly coupled groups of unknowns, gradients that vanish where X is large).
//    So an entry is taken from the slices only where sum |a||b| is at least
//    2^(eA + eB - 8.7), where they lose no more than K roundings of FP64. The sums
//    of the slice products over 256 k, added without their signs, bound it from
//    below and settle that for nearly every entry (kEnough). The rest is looked at
//    by FMAs (by_fma), which also form the entries that the slices must not: dense
//    operands keep the slices' bits.
//  * Rows of A and columns of B with an infinity, a NaN or a subnormal entry
//    take FMAs as well.
//
// One CTA computes 128 rows x 32 columns over one K slice:
//   warps 0-15: two groups of 8 that take the stages in turn. Each thread
//               reads A in FP64 for one row and 8 k (copied ahead into its own
//               64 bytes of shared memory) and cuts it into slices (11 stores of
//               16 bytes); after each 256 k all fold the 11 accumulators from
//               TMEM into the integers.
//   warp 16   : allocates TMEM, issues the MMAs. Slice s of A multiplies slices
//               1 .. 12 - s of B in one instruction (N up to 256), because B's
//               slices lie one after the other along N and the accumulators of
//               g = s + 1 .. 12 along the columns of TMEM.
// B (32 columns x 16 k, all slices, 11 KB) is sliced once beforehand into the
// layout of shared memory and comes by bulk copy. 3 stages of 16 k (56 KB).
//
// Bound: per stage 1056 clocks of MMA at the dense BF16 rate and about as many
// issue slots for the slicing; measured 3300 clocks per stage, the producers'
// latency (2.6 us of shared-memory and conversion chains per 8 values and
// thread). n = 4096 with 64 columns: 0.26 ms plain, 0.23 ms transposed, against
// 2.13 ms for the DFMA kernel; the outer product 4096 x 4096 x 64 0.49 ms
// against 1.76. With one group of 8 producer warps and register prefetch the plain
// product took 0.48.
#include <cuda_bf16.h>

#include <algorithm>

#include "common.cuh"
#include "tc_ptx.cuh"

namespace hplgb {
namespace p64 {

using namespace tc;

// not 0, with an exponent field of 0
__device__ __forceinline__ bool subnormal(double v) {
    return expo(v) == 0 && ((__double2hiint(v) & 0x7fffffff) | __double2loint(v)) != 0;
}

constexpr int kSlices = 11;
constexpr int kRows = 128, kCols = 32, kStep = 16;         // a CTA's tile, k per stage
constexpr int kChunk = 256 / kStep;                        // stages between folds
constexpr int kAStage = kSlices * kRows * kStep * 2;       // 45056
constexpr int kBStage = kSlices * kCols * kStep * 2;       // 11264
constexpr int kStages = 3;
constexpr int kProducers = 512;
constexpr int kRaw = kProducers * 64;                      // A's next 8 values of every producer
constexpr int kSmem = kStages * (kAStage + kBStage) + kRaw;
constexpr int kThreads = kProducers + 32;
constexpr int64_t kMaxSlice = 65536;                       // k per CTA: the low 64-bit sums hold 512 chunks
constexpr int kNoScale = -4000;                            // xk of a zero row of B
constexpr int kBad = 1 << 24;                              // eB of a column with an infinity, a NaN or a subnormal
constexpr int kLow = -(1 << 20);                           // exponent of a row or column of zeros
constexpr unsigned kEnough = 255;                          // sum |a||b| in units of 2^(eA + eB - 12) / 26, saturated: 2^-8.7

// The 11 slices of 8 consecutive k as 8 BF16 values each (k ascending), handed
// to put(slice, uint4), from the fixed-point magnitudes T and the signs (bit q
// of sgn). Digits d < 64 become BF16 through 128 + d (its last place is 1):
// sgn * (128 + d) - sgn * 128, exact.
template <typename Put>
__device__ __forceinline__ void slices8(const unsigned long long (&T)[8], unsigned sgn, Put put) {
    __nv_bfloat162 sg[4], off[4];
#pragma unroll
    for (int q = 0; q < 4; q++) {
        const unsigned a = sgn >> (2 * q) & 1u, b = sgn >> (2 * q + 1) & 1u;
        const unsigned one = 0x3f803f80u | a << 15 | b << 31;          // +-1
        const unsigned big = (0x43004300u | a << 15 | b << 31) ^ 0x80008000u;   // -+128
        sg[q] = *reinterpret_cast<const __nv_bfloat162*>(&one);
        off[q] = *reinterpret_cast<const __nv_bfloat162*>(&big);
    }
    auto digit = [&](const unsigned (&p)[4], int slice) {
        uint4 o;
        unsigned* w = reinterpret_cast<unsigned*>(&o);
#pragma unroll
        for (int q = 0; q < 4; q++) {
            const unsigned h = p[q] | 0x43004300u;
            const __nv_bfloat162 r = __hfma2(*reinterpret_cast<const __nv_bfloat162*>(&h), sg[q], off[q]);
            w[q] = *reinterpret_cast<const unsigned*>(&r);
        }
        put(slice, o);
    };
#pragma unroll
    for (int d = 0; d < 6; d++) {                                       // two digits at a time
        unsigned p[4], lo[4];
#pragma unroll
        for (int q = 0; q < 4; q++) {
            const int sh = d < 5 ? 52 - 12 * d : 0;
            unsigned a = (unsigned)(T[2 * q] >> sh), b = (unsigned)(T[2 * q + 1] >> sh);
            p[q] = __byte_perm(a, b, 0x5410);
            if (d == 5) p[q] <<= 2;                                     // the last 4 bits, padded to a digit
            lo[q] = p[q] & (d == 5 ? 0x003c003cu : 0x003f003fu);
            p[q] = (p[q] >> 6) & 0x003f003fu;
        }
        if (d < 5) {
            digit(p, 2 * d);
            digit(lo, 2 * d + 1);
        } else {
            digit(lo, 10);
        }
    }
}

// ---- B (K x nn, entry (k, c) at k sk + c sc): scales and slices ----

// xk[k] = e with every finite |B(k, .)| < 2^e; one CTA per k
__global__ void __launch_bounds__(128) k_scale_k(int64_t nn, const double* __restrict__ B, int64_t sk, int64_t sc,
                                                 int* __restrict__ xk) {
    __shared__ int s[4];
    const double* b = B + (int64_t)blockIdx.x * sk;
    int mx = 0;
    for (int64_t c = threadIdx.x; c < nn; c += 128) {
        const int E = expo(b[c * sc]);
        if (E < 0x7ff) mx = max(mx, E);
    }
    mx = __reduce_max_sync(0xffffffffu, mx);
    if ((threadIdx.x & 31) == 0) s[threadIdx.x >> 5] = mx;
    __syncthreads();
    mx = max(max(s[0], s[1]), max(s[2], s[3]));
    if (threadIdx.x == 0) xk[blockIdx.x] = mx ? mx - 1022 : kNoScale;
}

// eB[c] = e with every |B(., c)| 2^-xk < 2^e (kBad: an infinity, a NaN or a
// subnormal; kLow: zeros); one CTA per c
__global__ void __launch_bounds__(128) k_scale_c(int64_t K, const double* __restrict__ B, int64_t sk, int64_t sc,
                                                 const int* __restrict__ xk, int* __restrict__ eB) {
    __shared__ int s[4];
    const double* b = B + (int64_t)blockIdx.x * sc;
    int mx = kLow;
    for (int64_t k = threadIdx.x; k < K; k += 128) {
        const double v = b[k * sk];
        const int E = expo(v);
        if (E == 0x7ff || subnormal(v)) mx = kBad;
        else if (E) mx = max(mx, E - xk[k]);
    }
    mx = __reduce_max_sync(0xffffffffu, mx);
    if ((threadIdx.x & 31) == 0) s[threadIdx.x >> 5] = mx;
    __syncthreads();
    mx = max(max(s[0], s[1]), max(s[2], s[3]));
    if (threadIdx.x == 0) eB[blockIdx.x] = mx == kBad || mx == kLow ? mx : mx - 1022;
}

// The image of B: per 32 columns, per 16 k: [k octet][slice][group of 8
// columns][column][8 k] in BF16, zeros outside B. One thread per column and
// octet, lanes along the columns.
__global__ void __launch_bounds__(256) k_slice_b(int64_t K, int64_t nn, const double* __restrict__ B, int64_t sk,
                                                 int64_t sc, const int* __restrict__ xk, const int* __restrict__ eB,
                                                 unsigned char* __restrict__ img) {
    const int64_t nst = (K + kStep - 1) / kStep, octs = 2 * nst, cg = (nn + kCols - 1) / kCols;
    const int64_t t = (int64_t)blockIdx.x * 256 + threadIdx.x;
    if (t >= octs * cg * kCols) return;
    const int cl = (int)(t % kCols);
    const int64_t oct = t / kCols % octs, g = t / (kCols * octs), c = g * kCols + cl, k0 = 8 * oct;
    unsigned long long T[8];
    unsigned sgn = 0;
    const int e = c < nn ? eB[c] : kBad;
#pragma unroll
    for (int q = 0; q < 8; q++) {
        const bool in = c < nn && k0 + q < K && e != kBad;
        const double v = in ? B[(k0 + q) * sk + c * sc] : 0.0;
        T[q] = fixed64(v, in ? -xk[k0 + q] : 0, e);
        sgn |= (unsigned)(v < 0.0) << q;
    }
    unsigned char* o = img + (g * nst + (oct >> 1)) * kBStage + (oct & 1) * (kBStage / 2) + (cl >> 3) * 128 + (cl & 7) * 16;
    slices8(T, sgn, [&](int s, uint4 w) { *reinterpret_cast<uint4*>(o + s * (kCols * 16)) = w; });
}

// kind::f16, BF16 operands, FP32 accumulator, M = 128, N columns
__device__ __forceinline__ void mma_n(uint32_t d, uint64_t a, uint64_t b, int N, uint32_t accumulate) {
    const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | (uint32_t)(N >> 3) << 17 | (uint32_t)(kRows >> 4) << 24;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d),
        "l"(a), "l"(b), "r"(idesc), "r"(accumulate)
        : "memory");
}
__device__ __forceinline__ void tmem_ld4(uint32_t taddr, uint32_t (&r)[4]) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(taddr)
                 : "memory");
}
template <int BYTES>
__device__ __forceinline__ void copy_async(void* dst, const void* src, bool valid) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2, %3;" ::"r"(smem_u32(dst)), "l"(src), "n"(BYTES),
                 "r"(valid ? BYTES : 0) : "memory");
}

// The entries of a warp's 32 rows from r0 (lane l: row r0 + l) and columns c0 + j
// that have a bit j in which: sum a b and sum |a||b| by FMAs over the k of [ka, kb),
// the first into out[j ldc] unless the second reaches 0.6 2^(eA + eB - 8) (eA: the
// lane's; kBad in either: never), where the slices' entry stays. A column's
// entries are formed side by side, a lane each (lanes read neighbours of A), or,
// when few of them are wanted or A's rows lie along memory (TA), one after the
// other by all lanes along k. Many entries of one column over several times 256 k
// are no chance cancellations: sum |a||b|, half the FMAs, is then left out. n = 4096
// with 64 columns, every second unknown coupled by 2^-40, forward and backward:
// 21.7 ms (17.4 with DFMA kernels throughout, 4.9 uniform).
template <bool TA>
__device__ __noinline__ void by_fma(unsigned which, const double* A, int64_t lda, int64_t r0, int64_t M, int eA,
                                    const double* B, int64_t sk, int64_t sc, int64_t c0, const int* eB, int64_t ka,
                                    int64_t kb, double* out, int64_t ldc, int neg) {
    const int lane = threadIdx.x & 31;
    for (int j = 0; j < 8; j++) {
        const bool mine = which >> j & 1u;
        unsigned m = __ballot_sync(0xffffffffu, mine);
        if (!m) continue;
        const double* b = B + (c0 + j) * sc;
        const int ec = eB[c0 + j];
        const double enough = eA == kBad || ec == kBad ? __longlong_as_double(0x7ff8000000000000LL) : ldexp(0.6, eA + ec - 8);
        const bool many = __popc(m) > 4, weigh = !many || kb - ka <= 256;
        if (!TA && many) {
            const double* a = A + min(r0 + lane, M - 1);
            double s[2] = {0.0, 0.0}, t[2] = {0.0, 0.0};
            for (int64_t k = ka; k < kb; k += 8) {
                double x[8], y[8];
#pragma unroll
                for (int u = 0; u < 8; u++) {
                    x[u] = k + u < kb ? a[(k + u) * lda] : 0.0;
                    y[u] = k + u < kb ? b[(k + u) * sk] : 0.0;
                }
#pragma unroll
                for (int u = 0; u < 8; u++) s[u & 1] = fma(x[u], y[u], s[u & 1]);
                if (!weigh) continue;
#pragma unroll
                for (int u = 0; u < 8; u++) t[u & 1] = fma(fabs(x[u]), fabs(y[u]), t[u & 1]);
                if (!__any_sync(0xffffffffu, mine && !(t[0] + t[1] >= enough))) break;
            }
            const double v = s[0] + s[1];
            if (mine && !(weigh && t[0] + t[1] >= enough)) out[j * ldc] = neg ? -v : v;
            continue;
        }
        for (; m; m &= m - 1) {
            const int l = __ffs(m) - 1;
            const double* a = TA ? A + (r0 + l) * lda : A + r0 + l;
            const int64_t step = TA ? 1 : lda;
            const double lim = __shfl_sync(0xffffffffu, enough, l), per = 65536.0 / lim;
            double s = 0.0, t = 0.0;
            bool keep = false;                                 // the slices' entry
            for (int64_t k0 = ka; k0 < kb && !keep; k0 += 128) {
                double x[4], y[4];
#pragma unroll
                for (int u = 0; u < 4; u++) {
                    const int64_t k = k0 + 32 * u + lane;
                    x[u] = k < kb ? a[k * step] : 0.0;
                    y[u] = k < kb ? b[k * sk] : 0.0;
                }
#pragma unroll
                for (int u = 0; u < 4; u++) s = fma(x[u], y[u], s);
                if (!weigh) continue;
#pragma unroll
                for (int u = 0; u < 4; u++) t = fma(fabs(x[u]), fabs(y[u]), t);
                // the lanes' shares in units of 2^-16 lim, rounded down (a smaller lim has
                // no reciprocal in range: the whole sum decides below)
                keep = lim >= 0x1p-1000 && __reduce_add_sync(0xffffffffu, (unsigned)fmin(t * per, 65536.0)) >= 65536u;
            }
            if (keep) continue;
#pragma unroll
            for (int off = 16; off > 0; off >>= 1) {
                s += __shfl_xor_sync(0xffffffffu, s, off);
                t += __shfl_xor_sync(0xffffffffu, t, off);
            }
            if (lane == l && !(weigh && t >= lim)) out[j * ldc] = neg ? -s : s;
        }
    }
}

// C(z) (M x nn, ld ldc, slice z at C + z zstride) = (neg ? - : +) op(A) B over
// the k of slice z, [z kslice, (z + 1) kslice); kslice a multiple of 16.
// op(A)(i, k) = A[k lda + i], or A[i lda + k] (TA).
template <bool TA>
__global__ void __launch_bounds__(kThreads, 1)
k_prod64(int64_t M, int64_t nn, int64_t K, int64_t kslice, const double* __restrict__ A, int64_t lda, int vec,
         const double* __restrict__ B, int64_t sk, int64_t sc, const unsigned char* __restrict__ img,
         const int* __restrict__ xk, const int* __restrict__ eB,
         double* __restrict__ C, int64_t ldc, int64_t zstride, int neg, int* err, int64_t timeout_ns) {
    extern __shared__ __align__(1024) unsigned char psm[];
    __shared__ __align__(8) uint64_t full[kStages], bfull[kStages], empty[kStages], accfull, accempty, drain;
    __shared__ uint32_t s_tmem;
    __shared__ volatile int s_abort;
    __shared__ int s_e[4][kRows];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int64_t r0 = (int64_t)blockIdx.x * kRows, c0 = (int64_t)blockIdx.y * kCols;
    const int64_t ka = (int64_t)blockIdx.z * kslice, kb = min(K, ka + kslice);
    const int nst = (int)((kb - ka + kStep - 1) / kStep);          // >= 1
    const int nch = (nst + kChunk - 1) / kChunk;
    const uint64_t deadline = globaltimer_ns() + (uint64_t)timeout_ns;
    if (tid == 0) {
        s_abort = 0;
        for (int s = 0; s < kStages; s++) {
            mbar_init(&full[s], kProducers / 2);
            mbar_init(&bfull[s], 1);
            mbar_init(&empty[s], 1);
        }
        mbar_init(&accfull, 1);
        mbar_init(&accempty, kProducers);
        mbar_init(&drain, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == kProducers / 32) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&s_tmem)),
                     "r"(512) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    } else {
        // the rows' largest exponents over this K slice, many loads in flight
        auto level = [&](double v, int x) {
            const int E = expo(v);
            return E == 0x7ff || subnormal(v) ? kBad : E ? E + x : kLow;
        };
        if (TA) {
            for (int i = 0; i < kRows / 16; i += 2) {              // two rows at a time
                const int row = warp * (kRows / 16) + i;
                int m0 = kLow, m1 = kLow;
                const double* a0 = A + min(r0 + row, M - 1) * lda;
                const double* a1 = A + min(r0 + row + 1, M - 1) * lda;
#pragma unroll 8
                for (int64_t k = ka + lane; k < kb; k += 32) {
                    m0 = max(m0, level(a0[k], xk[k]));
                    m1 = max(m1, level(a1[k], xk[k]));
                }
                m0 = __reduce_max_sync(0xffffffffu, m0);
                m1 = __reduce_max_sync(0xffffffffu, m1);
                if (lane < 4) {
                    s_e[lane][row] = m0;
                    s_e[lane][row + 1] = m1;
                }
            }
        } else {
            const int row = tid & (kRows - 1), h = tid >> 7;
            int mx = kLow;
            const double* a = A + min(r0 + row, M - 1);
#pragma unroll 16
            for (int64_t k = ka + h; k < kb; k += 4) mx = max(mx, level(a[k * lda], xk[k]));
            s_e[h][row] = mx;
        }
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = s_tmem;

    if (warp == kProducers / 32) {
        if (lane == 0) {
            bool ok = true;
            for (int i = 0; i < nst && ok; i++) {
                const int s = i % kStages;
                const uint32_t ph = (uint32_t)(i / kStages) & 1u;
                ok = (i % kChunk || i == 0 ||
                      mbar_wait(&accempty, (uint32_t)(i / kChunk - 1) & 1u, deadline, &s_abort, err)) &&
                     mbar_wait(&bfull[s], ph, deadline, &s_abort, err) &&
                     mbar_wait(&full[s], ph, deadline, &s_abort, err);
                if (!ok) break;
                tc_fence_after();
                const uint32_t sa = smem_u32(psm + s * (kAStage + kBStage)), sb = sa + kAStage;
#pragma unroll
                for (int q = 0; q < kSlices; q++) {
                    const int n = kCols * (kSlices - q);
                    const uint64_t ad = desc_plain(sa + q * (kRows * kStep * 2), kRows * 16, 128);
                    const uint64_t bd = desc_plain(sb, kBStage / 2, 128);
                    const uint32_t acc = i % kChunk != 0 || q > 0;
                    mma_n(tmem + q * kCols, ad, bd, n < 256 ? n : 256, acc);
                    if (n > 256)
                        mma_n(tmem + q * kCols + 256, ad, bd + ((256 / kCols) * (kCols * 16) >> 4), n - 256, acc);
                }
                umma_commit(&empty[s]);
                if (i % kChunk == kChunk - 1 || i == nst - 1) umma_commit(&accfull);
            }
            // all issued MMAs complete before TMEM is released
            umma_commit(&drain);
            mbar_wait(&drain, 0, deadline + 1000000000ull, &s_abort, err);
        }
    } else {
        // the exponent of local row r (kLow where it meets only zeros, kBad kept)
        auto row_exp = [&](int r) {
            const int mx = max(max(s_e[0][r], s_e[1][r]), max(s_e[2][r], s_e[3][r]));
            return mx >= kBad ? kBad : mx < kNoScale / 2 ? kLow : mx - 1022;
        };
        const int grp = warp >> 3;                                  // takes stages grp, grp + 2, ...
        const int row = tid & (kRows - 1), oct = (tid >> 7) & 1;    // as a producer
        const int e = row_exp(row);
        const bool rowin = r0 + row < M && e != kBad;
        const int quarter = warp >> 2;                              // as a folder: row 32 (warp & 3) + lane,
        long long hi[8], lo[8];                                     // columns 8 quarter + j
        unsigned size[2] = {0u, 0u};                                // the like of all k, a byte per column
#pragma unroll
        for (int j = 0; j < 8; j++) hi[j] = lo[j] = 0;
        // this thread's next 8 values of A: pairs (2q, 2q + 1) at raw[q * kProducers + tid]
        double2* raw = reinterpret_cast<double2*>(psm + kStages * (kAStage + kBStage)) + tid;
        const double* ap = A + (TA ? min(r0 + row, M - 1) * lda : min(r0 + row, M - 1));
        int nx[8];
        auto fetch = [&](int i) {
            const int64_t k0 = ka + (int64_t)i * kStep + 8 * oct;
            const int left = rowin ? (int)min((int64_t)8, kb - k0) : 0;
            if (TA && vec && left == 8) {
                const double* a = ap + k0;
#pragma unroll
                for (int q = 0; q < 4; q++) copy_async<16>(raw + q * kProducers, a + 2 * q, true);
            } else {
                const int64_t step = TA ? 1 : lda;
                const double* a = ap + k0 * step;
#pragma unroll
                for (int q = 0; q < 8; q++) {
                    copy_async<8>(reinterpret_cast<double*>(raw + (q >> 1) * kProducers) + (q & 1), q < left ? a : A, q < left);
                    a += step;
                }
            }
            asm volatile("cp.async.commit_group;" ::: "memory");
            // (xk is padded to whole stages; the pad meets zeros of A)
            const int4 x0 = *reinterpret_cast<const int4*>(xk + k0), x1 = *reinterpret_cast<const int4*>(xk + k0 + 4);
            nx[0] = x0.x; nx[1] = x0.y; nx[2] = x0.z; nx[3] = x0.w;
            nx[4] = x1.x; nx[5] = x1.y; nx[6] = x1.z; nx[7] = x1.w;
        };
        int nf = 0;                                                 // chunks folded
        auto fold = [&]() -> bool {
            bool ok = mbar_wait(&accfull, (uint32_t)nf & 1u, deadline, &s_abort, err);
            if (!__all_sync(0xffffffffu, ok)) return false;
            tc_fence_after();
            const uint32_t ta = tmem + ((uint32_t)((warp & 3) * 32) << 16) + quarter * 8;
#pragma unroll
            for (int h = 0; h < 2; h++) {
                float sum[4] = {0.f, 0.f, 0.f, 0.f};                // bounds sum |a||b| of these 256 k, units 2^-12
#pragma unroll
                for (int g = 0; g < kSlices; g++) {
                    uint32_t r[4];
                    tmem_ld4(ta + g * kCols + 4 * h, r);
                    tmem_wait_ld();
#pragma unroll
                    for (int jj = 0; jj < 4; jj++) {
                        const int j = 4 * h + jj;
                        const float f = __uint_as_float(r[jj]);
                        const int iv = __float2int_rn(f);
                        if (g < 5) {
                            hi[j] += (long long)iv * (1 << (6 * (4 - g)));       // units 2^-36
                            sum[jj] = fmaf(fabsf(f), 1.0f / (1 << (6 * g)), sum[jj]);
                        } else {
                            lo[j] += (long long)iv * (1 << (6 * (10 - g)));      // units 2^-72
                        }
                    }
                }
#pragma unroll
                for (int jj = 0; jj < 4; jj++) {
                    const unsigned q = min((unsigned)(sum[jj] * 26.0f), kEnough);
                    size[h] = __vaddus4(size[h], q << (8 * jj));
                }
            }
            tc_fence_before();
            mbar_arrive(&accempty);
            nf++;
            return true;
        };
        bool ok = true;
        int issued = 0;                                             // stages whose copy of B this thread started
        if (grp < nst) fetch(grp);
        for (int i = grp; i < nst; i += 2) {
            // the sums of the previous 256 k, once the next ones have a start
            if (i % kChunk == 2 + grp && i > kChunk && !(ok = fold())) break;
            const int s = i % kStages;
            ok = mbar_wait(&empty[s], ((uint32_t)(i / kStages) & 1u) ^ 1u, deadline, &s_abort, err);
            if (!(ok = __all_sync(0xffffffffu, ok))) break;
            unsigned char* st = psm + s * (kAStage + kBStage);
            if ((tid & (kProducers / 2 - 1)) == 0) {
                mbar_expect_tx(&bfull[s], kBStage);
                const unsigned char* src = img + ((c0 / kCols) * ((K + kStep - 1) / kStep) + ka / kStep + i) * kBStage;
                asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                                 smem_u32(st + kAStage)),
                             "l"(src), "r"(kBStage), "r"(smem_u32(&bfull[s])) : "memory");
                issued = i + 1;
            }
            asm volatile("cp.async.wait_group 0;" ::: "memory");
            unsigned long long T[8];
            unsigned sgn = 0;
#pragma unroll
            for (int q = 0; q < 4; q++) {
                const double2 v = raw[q * kProducers];
                T[2 * q] = fixed64(v.x, nx[2 * q], e);
                T[2 * q + 1] = fixed64(v.y, nx[2 * q + 1], e);
                sgn |= ((unsigned)__double2hiint(v.x) >> 31) << (2 * q) | ((unsigned)__double2hiint(v.y) >> 31) << (2 * q + 1);
            }
            if (i + 2 < nst) fetch(i + 2);
            unsigned char* o = st + oct * (kRows * 16) + (row >> 3) * 128 + (row & 7) * 16;
            slices8(T, sgn, [&](int sl, uint4 w) { *reinterpret_cast<uint4*>(o + sl * (kRows * kStep * 2)) = w; });
            fence_async_smem();
            mbar_arrive(&full[s]);
        }
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        // after a wait that gave up: this thread's last copies complete (or have
        // a millisecond) before the CTA exits; otherwise the folds below imply it
        if (!ok && (tid & (kProducers / 2 - 1)) == 0) {
            const uint64_t until = globaltimer_ns() + 1000000ull;
            for (int i = issued - 1; i >= 0 && i >= issued - 3; i -= 2)
                while (!mbar_try_wait(&bfull[i % kStages], (uint32_t)(i / kStages) & 1u) && globaltimer_ns() < until) {}
        }
        __syncwarp();
        while (ok && nf < nch) ok = fold();
        if (ok) {
            const int fr = (warp & 3) * 32 + lane, fe = row_exp(fr);
            const int64_t r = r0 + fr;
            double* out = C + (int64_t)blockIdx.z * zstride + min(r, M - 1);
            unsigned again = 0;                                     // columns whose entry may not be the slices'
            if (r < M) {
#pragma unroll
                for (int j = 0; j < 8; j++) {
                    const int64_t c = c0 + 8 * quarter + j;
                    if (c >= nn) continue;
                    const int ec = eB[c];
                    double v = fma((double)lo[j], 0x1p-36, (double)hi[j]);
                    const int ex = fe + ec - 36;
                    v = ex > -1022 && ex < 1024 ? v * __longlong_as_double((long long)(ex + 1023) << 52) : ldexp(v, ex);
                    if (fe == kBad || ec == kBad ||
                        (fe != kLow && ec != kLow && (size[j >> 2] >> (8 * (j & 3)) & 255u) < kEnough))
                        again |= 1u << j;
                    out[c * ldc] = neg ? -v : v;
                }
            }
            const int64_t c = c0 + 8 * quarter;
            if (__any_sync(0xffffffffu, again != 0))
                by_fma<TA>(again, A, lda, r0 + (warp & 3) * 32, M, fe, B, sk, sc, c, eB, ka, kb, out + c * ldc, ldc, neg);
        }
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp == kProducers / 32)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512) : "memory");
}

}  // namespace p64

// Workspace of launch_prod64 for a K x nn matrix B: its image and the scales.
size_t prod64_ws_bytes(int64_t K, int64_t nn) {
    const int64_t st = (K + p64::kStep - 1) / p64::kStep, cg = (nn + p64::kCols - 1) / p64::kCols;
    return align_up((size_t)(st * cg) * p64::kBStage, 256) + align_up(sizeof(int) * (size_t)(st * p64::kStep), 256) +
           align_up(sizeof(int) * (size_t)nn, 256);
}

// C (M x nn) = +- op(A) B in `split` K slices, slice z at C + z * zstride (the
// caller adds them); B(k, c) = B[k sk + c sc]. op as k_prod64. ws: 256-byte
// aligned, prod64_ws_bytes(K, nn). kslice * split >= K, kslice a multiple of
// 16 and at most 65536.
int launch_prod64(int64_t M, int64_t nn, int64_t K, int ta, const double* A, int64_t lda, const double* B, int64_t sk,
                  int64_t sc, double* C, int64_t ldc, int64_t zstride, int64_t kslice, int split, int neg, void* ws,
                  int* err, int64_t timeout_ns, cudaStream_t s) {
    using namespace p64;
    if (M <= 0 || nn <= 0 || K <= 0) return HPL_OK;
    if (kslice % kStep || kslice > kMaxSlice || (int64_t)split * kslice < K || (int64_t)(split - 1) * kslice >= K)
        return HPL_ERR_INVALID;
    const int64_t st = (K + kStep - 1) / kStep, cg = (nn + kCols - 1) / kCols, rt = (M + kRows - 1) / kRows;
    if (cg > 65535 || K > 0x7fffffff || nn > 0x7fffffff || rt > 0x7fffffff) return HPL_ERR_INVALID;
    unsigned char* img = (unsigned char*)ws;
    int* xk = (int*)(img + align_up((size_t)(st * cg) * kBStage, 256));
    int* eB = (int*)((unsigned char*)xk + align_up(sizeof(int) * (size_t)(st * kStep), 256));
    const int vec = ((uintptr_t)A & 15) == 0 && lda % 2 == 0;
    static std::atomic<int> ready[kMaxDevices];
    const int dv = device_slot();
    if (dv < 0) return HPL_ERR_CUDA;
    if (!ready[dv].load()) {
        HPL_CUDA_TRY(cudaFuncSetAttribute((const void*)k_prod64<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmem));
        HPL_CUDA_TRY(cudaFuncSetAttribute((const void*)k_prod64<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmem));
        ready[dv].store(1);
    }
    k_scale_k<<<(unsigned)K, 128, 0, s>>>(nn, B, sk, sc, xk);
    HPL_LAUNCH_CHECK();
    k_scale_c<<<(unsigned)nn, 128, 0, s>>>(K, B, sk, sc, xk, eB);
    HPL_LAUNCH_CHECK();
    const int64_t items = 2 * st * cg * kCols;
    k_slice_b<<<(unsigned)((items + 255) / 256), 256, 0, s>>>(K, nn, B, sk, sc, xk, eB, img);
    HPL_LAUNCH_CHECK();
    const dim3 g((unsigned)rt, (unsigned)cg, (unsigned)split);
    if (ta) k_prod64<true><<<g, kThreads, kSmem, s>>>(M, nn, K, kslice, A, lda, vec, B, sk, sc, img, xk, eB, C, ldc, zstride, neg, err, timeout_ns);
    else k_prod64<false><<<g, kThreads, kSmem, s>>>(M, nn, K, kslice, A, lda, vec, B, sk, sc, img, xk, eB, C, ldc, zstride, neg, err, timeout_ns);
    HPL_LAUNCH_CHECK();
    return HPL_OK;
}

}  // namespace hplgb

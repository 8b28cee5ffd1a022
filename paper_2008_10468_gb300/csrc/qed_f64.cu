// GB300 (sm_103a) binary64 synchrotron functions: the C ABI entry
// qed_synchrotron_F1F2_f64 of include/qed.h.
//
// F(x) = x int_x^inf K_{5/3}(t) dt and G(x) = x K_{2/3}(x) (Sec. 3.2.1) to
// binary64 rounding, beyond the double-precision accuracy level of Table 1,
// from the tables of fit_synchrotron64.py: per piece [1, 1.25), [1.25, 1.5),
// [1.5, 2) of m in x = m 2^k,
//   F = 2^{k/3} exp(-lam_k x) sum_j c_j u^j,  u = (m - centre) / halfwidth in [-1, 1)
// (u exact: dyadic centres and half-widths), and below 2^KMIN the small-x
// series F = x^{1/3} sum_j a_j x^{2j/3}.  Arguments from 2^(KMAX+1) on give 0
// (F, G < 1e-220).
//
// The polynomial, exp(-x) and their product are 64-bit fixed-point integers,
// not binary64: this GPU has 1/64 of the binary32 rate in binary64 (a pipe that
// the 22 multiply-adds and the exp of an evaluation kept 90% busy), but forms about
// 30 wide 32 x 32 products per clock and SM.  A 64-bit step of the Horner
// recurrence is three of them; the powers whose coefficients are below 2^-25
// take one each in 32 bits.  Worst error against 40-digit values 1.8e-16
// (little above half a unit in the last place, the rounding of the result),
// where the binary64 evaluation of the same fit has 4.2e-16.  2^24 log-uniform
// points in [1e-4, 50]: 1420 us in binary64, 291 us in this form.  Bound by the
// issue of the 64-bit integer steps; the 24 bytes a point take 60 us of HBM.
#include <cstdint>

#include "qed.h"
#include "synchro_coeffs64.h"

namespace {

constexpr int kThreads64 = 256;

struct Syn64Table {
    longlong2 main[QED_SYN64_TAIL][QED_SYN64_NPIECE];                // power j at scale 2^(60 + j)
    int2 tail[QED_SYN64_DEG + 1 - QED_SYN64_TAIL][QED_SYN64_NPIECE];  // power j at scale 2^(46 + j)
    unsigned long long exp2[256];                                    // 2^{-i/256} at scale 2^63
};

__device__ __forceinline__ void stage_syn64(Syn64Table& T) {
    const int t = threadIdx.x;
    for (int i = t; i < QED_SYN64_TAIL * QED_SYN64_NPIECE; i += blockDim.x)
        (&T.main[0][0])[i] = (&qed_syn64_main[0][0])[i];
    for (int i = t; i < (QED_SYN64_DEG + 1 - QED_SYN64_TAIL) * QED_SYN64_NPIECE; i += blockDim.x)
        (&T.tail[0][0])[i] = (&qed_syn64_tail[0][0])[i];
    for (int i = t; i < 256; i += blockDim.x) T.exp2[i] = qed_syn64_exp2[i];
}

// High half of a 64 x 64 product, without the low partial product (2 units
// at most).
__device__ __forceinline__ uint64_t mulhi(uint64_t a, uint64_t b) {
    const uint32_t ah = (uint32_t)(a >> 32), al = (uint32_t)a;
    const uint32_t bh = (uint32_t)(b >> 32), bl = (uint32_t)b;
    return (uint64_t)ah * bh + (((uint64_t)ah * bl) >> 32) + (((uint64_t)al * bh) >> 32);
}

// p u for u = uh 2^-31 + ul 2^-62 (uh signed, ul 31 bits), one binary place
// lower: the scale of the next coefficient c, which is added.
__device__ __forceinline__ int64_t horner64(int64_t p, int32_t uh, int32_t ul, int64_t c) {
    const int32_t ph = (int32_t)(p >> 32), pl = (int32_t)((uint32_t)p >> 1);
    const int64_t mid = (int64_t)ph * ul + (int64_t)pl * uh;
    return (int64_t)ph * uh + c + (mid >> 31);
}

// The binary64 number V 2^(e - 60), rounded to nearest, for V >= 2^54.
__device__ __forceinline__ double to_double(uint64_t V, int e) {
    const int sh = 11 - __clz((int)(V >> 32));   // to 53 bits
    return __longlong_as_double(((int64_t)(1014 + sh + e) << 52) +
                                (int64_t)((V + (1ull << (sh - 1))) >> sh));
}

// Small-x series (subnormals included), rare: kept out of line.
__device__ __noinline__ double2 syn64_small(double x) {
    const double r = cbrt(x);
    const double v = r * r;
    double pf = qed_syn64_small[0][QED_SYN64_SMALL_DEG], pg = qed_syn64_small[1][QED_SYN64_SMALL_DEG];
#pragma unroll 1
    for (int j = QED_SYN64_SMALL_DEG - 1; j >= 0; --j) {
        pf = fma(pf, v, qed_syn64_small[0][j]);
        pg = fma(pg, v, qed_syn64_small[1][j]);
    }
    return make_double2(r * pf, r * pg);
}

__device__ __forceinline__ void syn64(const Syn64Table& T, double x, double& F, double& G) {
    F = G = 0.0;
    const int64_t bits = __double_as_longlong(x);
    const int k = (int)(bits >> 52) - 1023;   // negative x: k < -1023
    if (k < QED_SYN64_KMIN || k > QED_SYN64_KMAX) {   // also NaN, infinities and 0
        if (x > 0.0 && k < QED_SYN64_KMIN) {
            const double2 r = syn64_small(x);
            F = r.x;
            G = r.y;
        }
        return;
    }
    const uint64_t frac = (uint64_t)bits & 0x000FFFFFFFFFFFFFull;
    const int part = min((int)(frac >> 50), 2);
    // u as a signed 64-bit fraction: the bits of m below the piece's, sign flipped
    const uint64_t u = (part == 2 ? frac << 13 : frac << 14) ^ (1ull << 63);
    const int32_t uh = (int32_t)(u >> 32), ul = (int32_t)((uint32_t)u >> 1);
    const int piece = 3 * (k - QED_SYN64_KMIN) + part;
    constexpr int kTop = QED_SYN64_DEG - QED_SYN64_TAIL;
    int2 r = T.tail[kTop][piece];
#pragma unroll
    for (int j = kTop - 1; j >= 0; --j) {
        const int2 c = T.tail[j][piece];
        r.x = c.x + __mulhi(r.x, uh);
        r.y = c.y + __mulhi(r.y, uh);
    }
    longlong2 c = T.main[QED_SYN64_TAIL - 1][piece];
    int64_t pf = c.x + (((int64_t)r.x * uh) >> 18);
    int64_t pg = c.y + (((int64_t)r.y * uh) >> 18);
#pragma unroll
    for (int j = QED_SYN64_TAIL - 2; j >= 0; --j) {
        c = T.main[j][piece];
        pf = horner64(pf, uh, ul, c.x);
        pg = horner64(pg, uh, ul, c.y);
    }
    // 2^{k/3}: floor(k / 3) here, the rest in the coefficients
    int e = (k - QED_SYN64_KMIN + (QED_SYN64_KMIN + 15)) / 3 - 5;
    uint64_t vf = (uint64_t)pf, vg = (uint64_t)pg;
    if (k >= QED_SYN64_LAMBDA_FROM) {
        // exp(-x) = 2^-n 2^{-i/256} 2^-r from y = x log2 e
        const uint64_t y = mulhi((frac | (1ull << 52)) << 11, QED_SYN64_LOG2E);   // at scale 2^(62 - k)
        const uint64_t f = y << (2 + k);
        e -= (int)(y >> (62 - k));
        // z = r ln 2 < 2^-8.5 at scale 2^72; 2^-r = 1 - z (1 - z (1/2 - z (1/6 - z (1/24 - z / 120))))
        const uint64_t z = mulhi(f << 8, QED_SYN64_LN2);
        const uint32_t z32 = (uint32_t)(z >> 32);
        const uint32_t a = 178956971u - __umulhi(z32, 139810u);
        const uint32_t b = 715827883u - (__umulhi(z32, a) >> 8);
        const uint64_t v = (1ull << 63) - (((uint64_t)z32 * b) >> 8);
        const uint64_t t = z - (mulhi(z, mulhi(z, v)) >> 8);
        const uint64_t E = T.exp2[f >> 56];
        const uint64_t g = E - (mulhi(E, t) >> 8);
        vf = mulhi(vf << 1, g);
        vg = mulhi(vg << 1, g);
    }
    F = to_double(vf, e);
    G = to_double(vg, e);
}

// 13 KB of tables per block, a row of a power's (F, G) pairs read with one
// 128-bit load (random pieces conflict about 2.5-fold).  The figures
// stand at the top of this file.
template <bool W1, bool W2>
__global__ void __launch_bounds__(kThreads64) k_sweep64(const double* __restrict__ y,
                                                        double* __restrict__ F1,
                                                        double* __restrict__ F2, long long n) {
    __shared__ Syn64Table T;
    stage_syn64(T);
    __syncthreads();
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
        double a, b;
        syn64(T, __ldcs(y + i), a, b);
        if (W1) __stcs(F1 + i, a);
        if (W2) __stcs(F2 + i, b);
    }
}

}  // namespace

extern "C" qed_status qed_synchrotron_F1F2_f64(const double* y, double* F1, double* F2,
                                                int64_t n, void* stream) {
    if (n < 0 || (n > 0 && (!y || (!F1 && !F2)))) return QED_ERR_ARG;
    if (n == 0) return QED_OK;
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
        return QED_ERR_CUDA;
    const long long blocks = ((long long)n + kThreads64 - 1) / kThreads64;
    const int grid = (int)(blocks < (long long)sms * 8 ? blocks : (long long)sms * 8);
    const cudaStream_t s = (cudaStream_t)stream;
    if (F1 && F2) k_sweep64<true, true><<<grid, kThreads64, 0, s>>>(y, F1, F2, (long long)n);
    else if (F1) k_sweep64<true, false><<<grid, kThreads64, 0, s>>>(y, F1, F2, (long long)n);
    else k_sweep64<false, true><<<grid, kThreads64, 0, s>>>(y, F1, F2, (long long)n);
    return cudaGetLastError() == cudaSuccess ? QED_OK : QED_ERR_CUDA;
}

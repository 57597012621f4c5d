// sigma = H.c for norb <= 16 on the tensor cores: FP64 summed exactly in integers, FP32 from BF16 planes.
//
// This GPU's FP64 pipe runs 2 multiply-adds per SM and clock, its BF16 tensor cores
// 4,096. So the values are cut into 8-bit digits -- an FP64 c into 8, an FP64 matrix
// element into 7, each digit an integer in [-128, 128], which BF16 holds exactly --
// and the products of digits are summed in FP32 accumulators. Every sum stays below
// 2^24 in magnitude, so it is an exact integer; sums of equal weight 256^-(i + j) are
// drained as integers and combined in 64-bit words. Only the digits that are cut off
// (below 2^-64 of the vector's scale, 2^-56 of the Hamiltonian's) and the products of
// weight below 256^-9 are lost: less than the rounding of the FP64 sums that they
// replace (norb 16, 3,000 x 3,000 strings: 6.1e-16 of the norm from 64-bit values, the
// SIMT kernel 1.5e-15).
// Integer sums are associative: results do not depend on the order of the work.
//
// FP32 sigma takes the same kernels of the same-spin classes with three BF16 planes per
// value in the place of digits (all 24 bits of an FP32 value, each with its own exponent)
// and the six products x_i y_j with i + j <= 2, summed in FP32: what an element loses is
// relative to the terms of its own sum, as in the SIMT kernel, however far the elements of
// a vector or the integrals lie apart. (FP32 digits, of 32 bits below one scale for the whole
// vector, were up to 1e-3 of (|H||c|)_I off on vectors that decay by a decade per excitation.)
// norb 16, 3,000 x 3,000 strings, three vectors: 5.3 ms, 1.4e-7 of the norm from 64-bit values;
// the SIMT kernel 13.6 ms, 6.2e-7.
//
// Parts of a sigma (Sec. II.B, Eq. 7; the classes [a,b] of Sec. II.C):
//   k_udiag         the diagonal and the opposite-spin term of the alpha singles
//                   with the beta string unchanged (SIMT, one multiply-add per term)
//   k_same_spin_ex  the same-spin classes as one dense product per 128 x NT tile,
//                   sigma += c Hb^T + Ha c over the off-diagonal string Hamiltonians
//   k_sigma_ab_ex   the alpha-beta classes (FP64; FP32 takes sigma_tc.cu's kernel):
//                   per alpha row G = A F over the row's alpha terms (A: integrals
//                   (rs|pq), F: the coupled c rows), then G summed into the columns
//                   its beta links point to
// Small spaces take several vectors per launch.
// FP64 digits are relative to one power of two per vector, so an element of sigma whose
// terms are all far below the vector's largest would be summed from few bits. Its terms are
// therefore looked at on the way (k_udiag, see kCoarse): elements for which the digits are too
// coarse are listed and summed again, term by term, by k_sigma_repair; a vector with many of
// them goes to the SIMT kernels, launched behind, as do NaN, infinities and extreme
// magnitudes, by a flag in device memory. Nothing of this costs a synchronisation. Elements of
// c that tower over the rest are kept out of the digits (see kOutlierRms).
#include <cuda.h>
#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <type_traits>
#include <vector>

#include "internal.cuh"
#include "tensor.cuh"

namespace tbsci {

namespace {

// digits (FP32: planes) of a matrix element / of c, and accumulated weights 256^-2 ..
// 256^-(ORD + 1) (FP32: sums i + j)
template <int P>
struct Prec;
template <>
struct Prec<0> {  // FP64
    static constexpr int NSA = 7, NSC = 8, ORD = 8;
    typedef double T;
    static constexpr double kRatio = 1024.0;  // scale / root mean square up to which digits are kept
};
template <>
struct Prec<1> {  // FP32
    static constexpr int NSA = 3, NSC = 3, ORD = 3;
    typedef float T;
    static constexpr double kRatio = INFINITY;  // planes have their own exponents
};

// Two accumulators of integers x0, x1 as the integer 256 x0 + x1, plus kPairBias (mod
// 2^32). Below 2^22 in magnitude an integer is read from the mantissa of x + 1.5 2^23
// (an add and half a shift-add per value); the conversion instruction issues at an
// eighth of that rate.
constexpr uint32_t kPairBias = (0x4B400000u << 8) + 0x4B400000u;
__device__ __forceinline__ int small_pair(uint32_t q0, uint32_t q1) {
    const uint32_t b0 = __float_as_uint(__uint_as_float(q0) + 12582912.f), b1 = __float_as_uint(__uint_as_float(q1) + 12582912.f);
    return (int)((b0 << 8) + b1);
}
// Below 2^23: half of x, rounded, read the same way; what the rounding left of x
// (-1, 0 or 1) goes on to x1, and that of x1 (one unit of the last weight) is added back.
__device__ __forceinline__ int large_pair(uint32_t q0, uint32_t q1) {
    const float x0 = __uint_as_float(q0), t0 = fmaf(x0, 0.5f, 12582912.f), r0 = fmaf(-2.f, t0 - 12582912.f, x0);
    const float x1 = fmaf(256.f, r0, __uint_as_float(q1)), t1 = fmaf(x1, 0.5f, 12582912.f),
                r1 = fmaf(-2.f, t1 - 12582912.f, x1);
    const uint32_t b0 = __float_as_uint(t0), b1 = __float_as_uint(t1), b2 = __float_as_uint(r1 + 12582912.f);
    return (int)((b0 << 9) + (b1 << 1) + b2 + (kPairBias - ((0x4B400000u << 9) + (0x4B400000u << 1) + 0x4B400000u)));
}

__device__ __forceinline__ double pow2(int e) { return __longlong_as_double((long long)(e + 1023) << 52); }

// ------------------------------------------------------------------ digits

// x 2^(8 n - e) as an integer, rounded to nearest; |x| <= 2^(e - 1) (1 - 2^-6), n <= 8
__device__ __forceinline__ int64_t to_fixed(double x, int shift_base) {
    const uint64_t b = (uint64_t)__double_as_longlong(x);
    const int ex = (int)((b >> 52) & 0x7FF);
    if (ex == 0) return 0;
    const int64_t m = (int64_t)((b & 0xFFFFFFFFFFFFFull) | 0x10000000000000ull);
    const int sh = ex - 1075 + shift_base;
    int64_t v;
    if (sh >= 0) v = m << min(sh, 62);
    else v = sh < -54 ? 0 : (m + ((int64_t)1 << (-sh - 1))) >> -sh;
    return (int64_t)b < 0 ? -v : v;
}
// digit s (0 = leading) of an N-digit fixed-point value, as BF16 bits
template <int N>
__device__ __forceinline__ uint32_t digit_bf16(int64_t fixed, int s) {
    constexpr uint64_t kBias = N == 8 ? 0x0080808080808080ull : 0x0000808080808080ull;
    const uint64_t u = (uint64_t)fixed + kBias;
    const int d = s == 0 ? (int)((int64_t)u >> (8 * (N - 1))) : (int)((u >> (8 * (N - 1 - s))) & 0xFF) - 128;
    return __float_as_uint((float)d) >> 16;
}

// exponent e with |x| <= 2^(e - 1) (1 - 2^-6) for every |x| <= top (top > 0, normal)
__host__ __device__ inline int scale_exponent(double top) {
    int e;
    const double m = frexp(top, &e);  // top = m 2^e, 0.5 <= m < 1
    return m <= 1.0 - 1.0 / 64 ? e + 1 : e + 2;
}

constexpr int kScaleThreads = 256;
constexpr int kScaleBlocks = 304;  // at most, two per SM

// Elements that tower over the rest of a vector (trial vectors of an eigensolver start as
// single determinants and stay close to them) are kept out of the digits: at most
// n / 256^2 of a vector's n elements exceed 256 times its root mean square, so no more than
// kOutliers up to 2^24 elements; larger vectors go to the SIMT kernels whole. The rest then
// has the scale that any vector with this root mean square may have, and k_sigma_left adds
// the outliers' links. 20 iterations of 3 roots from single determinants, 1,200 x 1,100
// strings at norb 16: seven of 60 vectors went to the SIMT kernels, 118 ms; now none, 103 ms.
constexpr double kOutlierRms = 256.0;
constexpr int64_t kOutlierMaxN = int64_t(1) << 24;

// How far digits carry. With c below 2^(e - 1), the string Hamiltonians below 2^(h - 1) and n
// links, an element of sigma is off by the products dropped, 2^-66 of 2^(e + h) a link or
// 7e-19 of it (root mean square) at 3,000 links, and by the digits cut off H, 2^-58 of it for
// the largest c: 8e-18 of 2^(e + h) where six standard deviations meet the worst H. (The W
// row's digits are doubled thrice, so the integrals count with one more power of two.) The
// terms of an element, (|H||c|)_I, are at least those of its diagonal and of its alpha singles
// with the beta string unchanged, which k_udiag has at hand; where these reach 2^-14 of
// 2^(e + h), the element is within 1.3e-13 of (|H||c|)_I, and 3e-15 where they are not all at
// the limit. Two decades of string weights in each spin: up to 3 elements in a thousand are
// below it.
constexpr double kCoarse = 1.0 / 16384;
// A listed element costs 1.7 times its share of the SIMT kernel (1,200 x 1,100 strings at
// norb 16: 3.5 ns against 2.1), and the digits save two thirds of that kernel: past a quarter
// of the elements the vector goes there. Of the 60 vectors of a 20-iteration Davidson run on
// these strings, 12 do (the first four iterations, on which most elements are still zero or
// nearly so); the run takes 130 ms, 103 without this look at the elements, when some were off
// by up to 5e-9 of their terms, and 204 on the SIMT kernel.
constexpr int64_t kCoarseShare = 4;

// Per vector (blockIdx.y) its largest magnitude and sum of squares, in a fixed order;
// the last block to finish writes info[2 v]: 1 when the digits serve the vector,
// info[2 v + 1]: its scale exponent. done[v] wraps back to 0. O.thr[v]: what an outlier exceeds.
template <typename T>
__global__ void __launch_bounds__(kScaleThreads) k_scale(const T *__restrict__ c0, int64_t n, double ratio, int64_t outlier_n,
                                                         double *part0, unsigned *done, const int *__restrict__ tab, int *info,
                                                         Outliers O, Coarse R) {
    const T *__restrict__ c = c0 + blockIdx.y * n;
    double *part = part0 + (size_t)blockIdx.y * 2 * kScaleBlocks;
    double top = 0.0, sum = 0.0;
    bool bad = false;
    const int64_t step = (int64_t)gridDim.x * kScaleThreads;
    for (int64_t i = blockIdx.x * (int64_t)kScaleThreads + threadIdx.x; i < n; i += 4 * step) {
        T x[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) x[u] = i + u * step < n ? __ldg(c + i + u * step) : T(0);
        T s = T(0), m = T(0);
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const T a = x[u] < T(0) ? -x[u] : x[u];
            bad |= !(a <= T(3e38));  // NaN, infinities and what no digit scale is made for
            m = a > m ? a : m;
            s += a * a;
        }
        if ((double)m > top) top = (double)m;
        sum += (double)s;
    }
    if (bad) top = INFINITY;
    __shared__ double st[kScaleThreads], ss[kScaleThreads];
    __shared__ bool last;
    auto fold = [&] {
        st[threadIdx.x] = top;
        ss[threadIdx.x] = sum;
        __syncthreads();
        for (int o = kScaleThreads / 2; o > 0; o >>= 1) {
            if (threadIdx.x < o) {
                st[threadIdx.x] = fmax(st[threadIdx.x], st[threadIdx.x + o]);
                ss[threadIdx.x] += ss[threadIdx.x + o];
            }
            __syncthreads();
        }
    };
    fold();
    if (threadIdx.x == 0) {
        part[2 * blockIdx.x] = st[0];
        part[2 * blockIdx.x + 1] = ss[0];
        __threadfence();
        last = atomicInc(done + blockIdx.y, gridDim.x - 1) == gridDim.x - 1;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    top = sum = 0.0;
    for (int b = threadIdx.x; b < gridDim.x; b += kScaleThreads) {
        top = fmax(top, __ldcg(part + 2 * b));
        sum += __ldcg(part + 2 * b + 1);
    }
    fold();
    if (threadIdx.x != 0) return;
    top = st[0];
    int ok = 0, e = 0;
    double thr = INFINITY;
    if (!tab[2]) {
        ok = 0;
    } else if (top == 0.0) {
        ok = 1;
    } else if (top < 1e15 && top > 1e-15) {
        const double rms = sqrt(ss[0] / (double)n);
        e = scale_exponent(top);
        ok = ldexp(1.0, e) <= ratio * rms ? 1 : 0;
        if (!ok && n <= outlier_n) {
            thr = kOutlierRms * rms;
            e = scale_exponent(thr);  // 2^e <= 4 thr = 1024 rms
            ok = 1;
        }
    }
    O.thr[blockIdx.y] = thr;
    O.count[blockIdx.y] = 0;
    R.need[blockIdx.y] = top == 0.0 ? 0.f : (float)ldexp(kCoarse, e + max(tab[1], tab[0] + 1));
    R.count[blockIdx.y] = 0;
    info[2 * blockIdx.y] = ok;
    info[2 * blockIdx.y + 1] = e;
}

// the digit planes [NSC][la][lbp] of each vector, columns lb .. lbp - 1 zero; 8 columns per thread
__global__ void __launch_bounds__(256) k_slice(const double *__restrict__ c, int64_t la, int64_t lb, int64_t lbp,
                                               const int *__restrict__ info, Outliers O, __nv_bfloat16 *out) {
    info += 2 * blockIdx.y;
    if (!info[0]) return;
    const double lim = O.thr[blockIdx.y];
    constexpr int N = Prec<0>::NSC;
    c += blockIdx.y * la * lb;
    out += blockIdx.y * N * la * lbp;
    const int shift = 8 * N - info[1];
    const int64_t per = lbp / 8, n = la * per, plane = la * lbp;
    for (int64_t i = blockIdx.x * 256ll + threadIdx.x; i < n; i += (int64_t)gridDim.x * 256) {
        const int64_t r = i / per, j = (i - r * per) * 8;
        int64_t f[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const double x = j + u < lb ? __ldg(c + r * lb + j + u) : 0;
            if (x <= lim && -x <= lim) {
                f[u] = to_fixed(x, shift);
            } else {
                const int k = atomicAdd(O.count + blockIdx.y, 1);
                if (k < kOutliers) O.list[blockIdx.y * kOutliers + k] = r * lb + j + u;
                f[u] = 0;
            }
        }
#pragma unroll
        for (int s = 0; s < N; ++s) {
            uint32_t w[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) w[u] = digit_bf16<N>(f[2 * u], s) | (digit_bf16<N>(f[2 * u + 1], s) << 16);
            *reinterpret_cast<uint4 *>(out + s * plane + r * lbp + j) = make_uint4(w[0], w[1], w[2], w[3]);
        }
    }
}

// ------------------------------------------------------------------ tables

__global__ void k_absmax(const double *__restrict__ v, int64_t n, unsigned long long *top) {
    unsigned long long m = 0;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const unsigned long long b = (unsigned long long)__double_as_longlong(v[i]) & 0x7FFFFFFFFFFFFFFFull;
        m = b > m ? b : m;
    }
    for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long y = __shfl_xor_sync(0xffffffffu, m, o);
        m = y > m ? y : m;
    }
    if ((threadIdx.x & 31) == 0 && m) atomicMax(top, m);
}

// the same over the off-diagonal columns of the integrals, the only ones cut into digits
__global__ void k_absmax_off(const double *__restrict__ V, int npair, int npoff, const int32_t *__restrict__ offpair,
                             unsigned long long *top) {
    unsigned long long m = 0;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < npair * npoff; i += gridDim.x * blockDim.x) {
        const unsigned long long b =
            (unsigned long long)__double_as_longlong(V[(size_t)(i / npoff) * npair + offpair[i % npoff]]) & 0x7FFFFFFFFFFFFFFFull;
        m = b > m ? b : m;
    }
    for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long y = __shfl_xor_sync(0xffffffffu, m, o);
        m = y > m ? y : m;
    }
    if ((threadIdx.x & 31) == 0 && m) atomicMax(top, m);
}

// tab[0], tab[1]: scale exponents of the integrals and of the string Hamiltonians from
// their largest magnitudes (W_Ia / 8 shares the integrals' scale: up to nelec / 8 of
// them); tab[2]: 0 where a magnitude is far from 1 (or not finite): such a Hamiltonian
// stays on the SIMT kernels
__global__ void k_table_scales(const unsigned long long *__restrict__ top, double w, int *tab) {
    const double v = w * __longlong_as_double((long long)top[0]), h = __longlong_as_double((long long)top[1]);
    tab[2] = (v == 0.0 || (v > 1e-15 && v < 1e15)) && (h == 0.0 || (h > 1e-15 && h < 1e15)) ? 1 : 0;
    tab[0] = tab[2] && v > 0.0 ? scale_exponent(v) : 0;
    tab[1] = tab[2] && h > 0.0 ? scale_exponent(h) : 0;
}

// the links of one CSR row per warp into dense digit (FP32: BF16) planes [NSA][l][ld] (zeroed
// before), and their number per 32-column chunk
template <int P>
__global__ void __launch_bounds__(256) k_dense_digits(int64_t l, int64_t ld, int nch, const int64_t *__restrict__ soff,
                                                      const int2 *__restrict__ sci, const double *__restrict__ sval,
                                                      const int64_t *__restrict__ doff, const int32_t *__restrict__ dcol,
                                                      const double *__restrict__ dval, const int *__restrict__ tab,
                                                      __nv_bfloat16 *out, uint8_t *cnt) {
    extern __shared__ unsigned scnt[];  // [8][nch]
    if (!tab[2]) return;
    constexpr int N = Prec<P>::NSA;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t r = blockIdx.x * 8ll + warp, plane = l * ld;
    if (r >= l) return;
    unsigned *c = scnt + warp * nch;
    for (int k = lane; k < nch; k += 32) c[k] = 0;
    __syncwarp();
    const int shift = 8 * N - tab[1];
    auto put = [&](int col, double x) {
        uint32_t h[N];
        if constexpr (P == 0) {
            const int64_t f = to_fixed(x, shift);
#pragma unroll
            for (int s = 0; s < N; ++s) h[s] = digit_bf16<N>(f, s);
        } else {
            bf16_planes<N>((float)x, h);
        }
#pragma unroll
        for (int s = 0; s < N; ++s) out[s * plane + r * ld + col] = __ushort_as_bfloat16((unsigned short)h[s]);
        atomicAdd(c + (col >> 5), 1u);
    };
    for (int64_t t = soff[r] + lane; t < soff[r + 1]; t += 32) put(sci[t].x, sval[t]);
    for (int64_t t = doff[r] + lane; t < doff[r + 1]; t += 32) put(dcol[t], dval[t]);
    __syncwarp();
    for (int k = lane; k < nch; k += 32) cnt[r * nch + k] = (uint8_t)c[k];
}

// The accumulators stay exact while a row has met at most kWindow links: 7 products
// of digits below 2^7 each per link and weight, 7 * 144 * 2^14 < 2^24. FP32 sums keep the
// same windows: they are added up in registers, rounded to nearest, where the tensor core's
// accumulator truncates.
constexpr int kWindow = 144;

// flush[b][ch] = 1: drain the accumulators before chunk ch (rows of block b); 2: no link, skip it
__global__ void k_windows(int64_t l, int nch, int rows, const uint8_t *__restrict__ cnt, uint8_t *flush) {
    __shared__ int sMax, sAny;
    const int64_t r = (int64_t)blockIdx.x * rows + threadIdx.x;
    int run = 0;
    for (int ch = 0; ch < nch; ++ch) {
        const int x = r < l && threadIdx.x < rows ? cnt[r * nch + ch] : 0;
        if (threadIdx.x == 0) sMax = sAny = 0;
        __syncthreads();
        run += x;
        atomicMax(&sMax, run);
        if (x) sAny = 1;
        __syncthreads();
        const bool cut = sMax > kWindow;
        if (cut) run = x;
        if (threadIdx.x == 0) flush[(int64_t)blockIdx.x * nch + ch] = sAny ? (cut ? 1 : 0) : 2;
        __syncthreads();
    }
}

// digits of the integral columns: [pair][128 off-diagonal pairs], and of W_Ia / 8 (times 8): [la][128]
__global__ void k_ab_digits(const double *__restrict__ V, int npair, int npoff, const int32_t *__restrict__ offpair,
                            const uint64_t *__restrict__ str, int64_t rows, const int *__restrict__ tab, uint4 *out) {
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= rows * 128) return;
    const int64_t row = i >> 7;
    const int rs = (int)(i & 127);
    constexpr int N = Prec<0>::NSA;
    double x = 0.0;
    if (rs < npoff) {
        const int col = offpair[rs];
        if (str) {
            for (uint64_t s = str[row]; s; s &= s - 1) {
                const int p = __ffsll((long long)s) - 1;
                x += V[(size_t)(p * (p + 1) / 2 + p) * npair + col];
            }
            x *= 0.125;
        } else {
            x = V[(size_t)row * npair + col];
        }
    }
    const int64_t f = tab[2] ? to_fixed(x, 8 * N - tab[0]) : 0;
    union {
        uint16_t h[8];
        uint4 v;
    } u;
    for (int s = 0; s < (int)(sizeof(u.v) / 2); ++s) {
        uint32_t d = s < N ? digit_bf16<N>(f, s) : 0u;
        // W is at most 8 (norb <= 16: up to 16) integrals: an eighth is cut into digits and the digits doubled thrice
        if (str && (d & 0x7FFFu)) d += 3u << 7;
        u.h[s] = (uint16_t)d;
    }
    out[i] = u.v;
}

// ------------------------------------------------------------------ diagonal and alpha singles

template <typename T>
struct UdArgs {
    int64_t la, lb;
    const T *C;
    T *S;
    const int *info;  // run only where info[0] is set (NULL: always)
    const uint64_t *stra;
    const int64_t *a_soff;
    const int2 *a_sci;
    const T *a_sval, *Ea, *Eb, *U;
    T ecore;
    int na, add;  // add: accumulate
    const float *a_svalf;  // CHECK
    int *flag;             // = info
    Coarse R;
};

// S[Ia][j] (+)= Hd c(Ia, j) + sum over alpha singles ([h +] s U[pq][j]) c(Ja, j), one vector
// per blockIdx.z; SINGLES: with their string-Hamiltonian values h. FP64 is bound by the
// FP64 pipe, FP32 by L2 (two coalesced reads per term). CTAs run column chunk by column
// chunk, so that those in flight share the chunk's columns of U and c (norb 16, 3,000 x
// 3,000 strings, FP64, a vector: 0.58 ms; 1.42 with an FP64 compare per sign).
constexpr int64_t kUdCols = 512;  // columns of a CTA

__device__ __forceinline__ double flip(double x, int m) { return __hiloint2double(__double2hiint(x) ^ m, __double2loint(x)); }
__device__ __forceinline__ float flip(float x, int m) { return __int_as_float(__float_as_int(x) ^ m); }
// |x| rounded towards zero, on the integer units (a conversion instruction would take the
// FP64 pipe); 0 below the smallest normal float, the largest float above it
__device__ __forceinline__ float low_abs(double x) {
    const uint32_t h = min((uint32_t)__double2hiint(x) & 0x7FFFFFFFu, 0x47EFFFFFu);
    const uint32_t f = __funnelshift_l((uint32_t)__double2loint(x), h - 0x38000000u, 3);
    return h < 0x38100000u ? 0.f : __uint_as_float(f);
}

// CHECK (FP64): the magnitudes of the terms are added up in FP32 beside them, with the
// alpha singles' own values; what cancels between those and U is taken off by its rounding.
// Elements that stay below R.need are listed (see kCoarse). At most 64 alpha singles.
template <typename T, bool SINGLES, bool CHECK>
__global__ void __launch_bounds__(256) k_udiag(UdArgs<T> A) {
    __shared__ int64_t sC[256], sU[256];
    __shared__ T sH[256];
    __shared__ float sF[CHECK ? 64 : 1];
    __shared__ int sS[256];  // sign bit of the term
    __shared__ int sOcc[64];
    __shared__ int sOn;
    const int64_t Ia = blockIdx.x, lb = A.lb;
    const int64_t t0 = A.a_soff[Ia], t1 = A.a_soff[Ia + 1];
    const int tid = threadIdx.x;
    // read once for the whole CTA: with CHECK another CTA may clear it at any time
    if (tid == 0) sOn = A.info ? *reinterpret_cast<const volatile int *>(A.info + 2 * blockIdx.z) : 1;
    __syncthreads();
    if (!sOn) return;
    const T *__restrict__ C = A.C + blockIdx.z * A.la * lb;
    T *__restrict__ S = A.S + blockIdx.z * A.la * lb + Ia * lb;
    if (tid < 64) {
        const uint64_t s = A.stra[Ia];
        if ((s >> tid) & 1) sOcc[__popcll(s & ((1ull << tid) - 1))] = tid * (tid + 1) / 2 + tid;
    }
    const T eIa = A.ecore + A.Ea[Ia];
    for (int64_t t = t0; t < t1 || t == t0; t += 256) {
        const int n = (int)min((int64_t)256, t1 - t);
        __syncthreads();
        if (tid < n) {
            const int2 e = A.a_sci[t + tid];
            sC[tid] = e.x * lb;
            sU[tid] = (int64_t)(e.y >> 1) * lb;
            sS[tid] = (e.y & 1) ? (int)0x80000000 : 0;
            if (SINGLES) sH[tid] = A.a_sval[t + tid];
            if (CHECK) sF[tid] = flip(A.a_svalf[t + tid], sS[tid]);  // with the sign of the term taken out
        }
        __syncthreads();
        for (int64_t j = blockIdx.y * kUdCols + tid; j < min(lb, (blockIdx.y + 1) * kUdCols); j += 256) {
            T acc = T(0), acc2 = T(0);
            float mag = 0.f;
            auto look = [&](int k, T u, T c) {
                if constexpr (CHECK) {
                    const float h = sF[k], v = copysignf(low_abs(u), __int_as_float(__double2hiint(u)));
                    mag = fmaf(fmaxf(fmaf(fabsf(h) + fabsf(v), -1e-6f, fabsf(h + v)), 0.f), low_abs(c), mag);
                }
            };
            if (t == t0) {
                T ed = eIa + __ldg(A.Eb + j);
                for (int k = 0; k < A.na; ++k) ed += __ldg(A.U + (size_t)sOcc[k] * lb + j);
                const T c = __ldg(C + Ia * lb + j);
                acc = ed * c;
                if constexpr (CHECK) mag = low_abs(ed) * low_abs(c);
            }
            const T *__restrict__ Uj = A.U + j, *__restrict__ Cj = C + j;
            // one multiply-add per term: the sign goes to u by its sign bit (an FP64 compare
            // and select would take the pipe's other half)
            auto coef = [&](int k, T u) { return SINGLES ? sH[k] + flip(u, sS[k]) : flip(u, sS[k]); };
            int k = 0;
            for (; k + 3 < n; k += 4) {
                const T u0 = __ldg(Uj + sU[k]), u1 = __ldg(Uj + sU[k + 1]), u2 = __ldg(Uj + sU[k + 2]), u3 = __ldg(Uj + sU[k + 3]);
                const T c0 = __ldg(Cj + sC[k]), c1 = __ldg(Cj + sC[k + 1]), c2 = __ldg(Cj + sC[k + 2]), c3 = __ldg(Cj + sC[k + 3]);
                acc += coef(k, u0) * c0;
                acc2 += coef(k + 1, u1) * c1;
                acc += coef(k + 2, u2) * c2;
                acc2 += coef(k + 3, u3) * c3;
                look(k, u0, c0);
                look(k + 1, u1, c1);
                look(k + 2, u2, c2);
                look(k + 3, u3, c3);
            }
            for (; k < n; ++k) {
                const T u = __ldg(Uj + sU[k]), c = __ldg(Cj + sC[k]);
                acc += coef(k, u) * c;
                look(k, u, c);
            }
            S[j] = (A.add || t > t0 ? S[j] : T(0)) + (acc + acc2);
            if constexpr (CHECK) {
                const int lane = tid & 31;
                const int64_t left = min(lb, (blockIdx.y + 1) * kUdCols) - (j - lane);  // lanes with a column
                const unsigned on = left >= 32 ? 0xFFFFFFFFu : (1u << left) - 1u;
                const unsigned low = __ballot_sync(on, mag < A.R.need[blockIdx.z]);
                if (low) {
                    const unsigned cnt = __popc(low), lead = __ffs(low) - 1;
                    unsigned at = 0;
                    if (lane == lead) {
                        at = atomicAdd(A.R.count + blockIdx.z, cnt);
                        if (at + cnt > A.R.limit) A.flag[2 * blockIdx.z] = 0;
                    }
                    at = __shfl_sync(on, at, lead) + __popc(low & ((1u << lane) - 1u));
                    if (((low >> lane) & 1) && at < A.R.limit)
                        A.R.list[(size_t)blockIdx.z * A.R.limit + at] = (int32_t)(Ia * lb + j);
                }
            }
        }
    }
}

inline dim3 ud_grid(int64_t la, int64_t lb, int nv) {
    return dim3((unsigned)la, (unsigned)((lb + kUdCols - 1) / kUdCols), (unsigned)nv);
}

// ------------------------------------------------------------------ same-spin classes

struct SsArgs {
    CUtensorMap mCA, mHb, mHa, mCB;
    int64_t la, lb;
    int nchb, ncha;  // 32-column chunks of the beta / alpha phase
    const uint8_t *flb, *fla;
    const int *info, *tab;
    void *S;
    int *err;
};

__device__ __forceinline__ void tma3(uint32_t dst, const CUtensorMap *m, uint32_t bar, int x, int y, int z) {
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cta.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5}], [%2];" ::"r"(
            dst),
        "l"(m), "r"(bar), "r"(x), "r"(y), "r"(z)
        : "memory");
}

template <int P>
struct SsShape {
    static constexpr int NSA = Prec<P>::NSA, NSC = Prec<P>::NSC, ORD = Prec<P>::ORD;
    static constexpr int NT = P == 0 ? 64 : 128;  // every weight's accumulator of a tile is resident: ORD x NT <= 512 TMEM columns
    static constexpr int kStages = P == 0 ? 2 : 4;
    static constexpr uint32_t kBetaBytes = NSC * 128 * 64 + NSA * NT * 64;
    static constexpr uint32_t kAlphaBytes = NSA * 128 * 64 + NSC * 32 * NT * 2;
    static constexpr uint32_t kStageBytes = ((kBetaBytes > kAlphaBytes ? kBetaBytes : kAlphaBytes) + 1023) / 1024 * 1024;
    static constexpr size_t kSmem = 1024 + (size_t)kStages * kStageBytes;
};

constexpr int kSsThreads = 576;  // 16 draining warps, a TMA warp, an MMA warp

// One 128 (alpha rows) x NT (beta columns) tile of sigma: a loop over 32-deep chunks
// of Jb (c rows times Hb rows), then of Ja (Ha rows times c columns); all digit planes
// of a chunk arrive by two TMA loads, and every pair of planes (i, j) is multiplied
// into the accumulator of its weight, plane A reused while B changes. The draining
// warps empty the accumulators into 64-bit registers at the window boundaries and
// at the end.
template <int P>
__global__ void __launch_bounds__(kSsThreads, 1) k_same_spin_ex(const __grid_constant__ SsArgs A) {
    const int *info = A.info + 2 * blockIdx.z;  // one vector per blockIdx.z
    if (!info[0]) return;
    using Sh = SsShape<P>;
    typedef typename Prec<P>::T T;
    constexpr int NSA = Sh::NSA, NSC = Sh::NSC, ORD = Sh::ORD, NT = Sh::NT, NST = Sh::kStages;
    extern __shared__ unsigned char smem_dyn[];
    __shared__ uint64_t bar[2 * NST + 2];
    __shared__ uint32_t tmem_base;
    __shared__ int sAbort;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const uint32_t sbase = (su32(smem_dyn) + 1023) & ~1023u;
    const uint32_t full = su32(&bar[0]), empty = su32(&bar[NST]), dfull = su32(&bar[2 * NST]), dempty = dfull + 8;
    const int64_t row0 = (int64_t)blockIdx.y * 128, col0 = (int64_t)blockIdx.x * NT;
    const uint8_t *flb = A.flb + (col0 / NT) * A.nchb, *fla = A.fla + (row0 / 128) * A.ncha;
    const int nch = A.nchb + A.ncha;
    auto flag = [&](int ch) -> int { return ch < A.nchb ? flb[ch] : fla[ch - A.nchb]; };
    if (tid == 0) {
        sAbort = 0;
        for (int s = 0; s < NST; ++s) {
            mb_init(full + 8 * s, 1);
            mb_init(empty + 8 * s, 1);
        }
        mb_init(dfull, 1);
        mb_init(dempty, 16);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 17) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(su32(&tmem_base)) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    tc_before();
    __syncthreads();
    tc_after();
    constexpr uint32_t tmem = 0;  // all 512 columns are this CTA's: they start at 0
    if (tid == 0 && tmem_base != 0) sAbort = 1;
    volatile int *ab = &sAbort;

    if (warp == 16) {
        if (lane == 0) {
            int n = 0;
            for (int ch = 0; ch < nch; ++ch) {
                if (flag(ch) == 2) continue;
                const int st = n % NST;
                if (n >= NST && !mb_wait(empty + 8 * st, (n / NST - 1) & 1, ab)) break;
                const uint32_t dst = sbase + st * Sh::kStageBytes, fb = full + 8 * st;
                const bool beta = ch < A.nchb;
                asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(fb),
                             "r"(beta ? Sh::kBetaBytes : Sh::kAlphaBytes)
                             : "memory");
                if (beta) {
                    tma3(dst, &A.mCA, fb, ch * 32, (int)row0, (int)blockIdx.z * NSC);
                    tma3(dst + NSC * 128 * 64, &A.mHb, fb, ch * 32, (int)col0, 0);
                } else {
                    const int k = (ch - A.nchb) * 32;
                    tma3(dst, &A.mHa, fb, k, (int)row0, 0);
                    for (int b = 0; b < NT / 64; ++b)
                        tma3(dst + NSA * 128 * 64 + b * NSC * 4096, &A.mCB, fb, (int)col0 + 64 * b, k, (int)blockIdx.z * NSC);
                }
                ++n;
            }
            if (*ab)  // nothing of this CTA may be in flight when it ends: leave the last loads time to land
                for (int it = 0; it < 4096; ++it) __nanosleep(100);
        }
        __syncwarp();
    } else if (warp == 17) {
        {
            int n = 0, nd = 0, phase = 0;
            bool fresh = true, ok = true;
            for (int ch = 0; ch < nch && ok; ++ch) {
                const int fl = flag(ch);
                if (fl == 2) continue;
                const bool turn = phase == 0 && ch >= A.nchb;
                if (turn) phase = 1;
                if ((fl == 1 || turn) && !fresh) {  // drain what the window (or the beta phase) summed
                    if (elect_one()) mma_commit(dfull);
                    __syncwarp();
                    ok = __all_sync(0xffffffffu, mb_wait(dempty, nd & 1, ab));
                    ++nd;
                    tc_after();
                    fresh = true;
                    if (!ok) break;
                }
                const int st = n % NST;
                ok = __all_sync(0xffffffffu, mb_wait(full + 8 * st, (n / NST) & 1, ab));
                if (!ok) break;
                tc_after();
                const uint32_t s0 = uni(sbase + st * Sh::kStageBytes), keep0 = fresh ? 0u : 1u;
                // the digit planes of one chunk against each other; planes NA of A, NB of B
                auto products = [&](auto beta_tag) {
                    constexpr bool BETA = decltype(beta_tag)::value;
                    constexpr int NA = BETA ? NSC : NSA, NB = BETA ? NSA : NSC;
                    constexpr uint32_t idesc = inst_desc(NT, !BETA);
                    if (elect_one()) {
#pragma unroll
                        for (int ks = 0; ks < 2; ++ks) {
                            const uint64_t a0 = op_desc(s0 + ks * 32, 16, 512, 4);
                            const uint64_t b0 = BETA ? op_desc(s0 + NA * 128 * 64 + ks * 32, 16, 512, 4)
                                                     : op_desc(s0 + NA * 128 * 64 + ks * 2048, NSC * 4096, 1024, 2);
                            constexpr uint64_t astep = 128 * 64 / 16, bstep = BETA ? NT * 64 / 16 : 4096 / 16;
#pragma unroll
                            for (int x = 0; x < NA; ++x) {
                                const int n_x = NB < ORD - x ? NB : ORD - x;
#pragma unroll
                                for (int y = 0; y < n_x; ++y) {
                                    // the first product of each weight after a drain overwrites its accumulator
                                    const bool first = ks == 0 && (x == 0 || (y == NB - 1 && x + y >= NB));
                                    const uint32_t keep = first ? keep0 : 1u;
                                    const uint32_t d = (x + y) * NT;
                                    const uint64_t a = a0 + x * astep, b = b0 + y * bstep;
                                    if (n_x == 1) mma_ss<0>(d, a, b, idesc, keep);
                                    else if (y == 0) mma_ss<1>(d, a, b, idesc, keep);
                                    else if (y == n_x - 1) mma_ss<3>(d, a, b, idesc, keep);
                                    else mma_ss<2>(d, a, b, idesc, keep);
                                }
                            }
                        }
                        mma_commit(empty + 8 * st);
                    }
                    __syncwarp();
                };
                if (ch < A.nchb) products(std::true_type{});
                else products(std::false_type{});
                fresh = false;
                ++n;
            }
            // the last drain; a CTA that gave up commits too, so that no MMA outlives it
            if (elect_one()) mma_commit(dfull);
            __syncwarp();
            mb_wait(dempty, nd & 1, ab);
        }
        __syncwarp();
    } else {
        constexpr int NC = NT / 4;  // columns of a draining warp
        const int quarter = warp & 3, part = warp >> 2;
        int64_t hi[P == 0 ? NC : 1], lo[P == 0 ? NC : 1];
        float sum[P == 0 ? 1 : NC];
#pragma unroll
        for (int x = 0; x < NC; ++x) {
            if (P == 0) hi[P == 0 ? x : 0] = lo[P == 0 ? x : 0] = 0;
            else sum[P == 0 ? 0 : x] = 0.f;
        }
        // the same walk as the MMA warp's, to know the number of drains and which is empty
        int drains = 0, phase = 0;
        bool any = false;
        for (int ch = 0; ch < nch; ++ch) {
            const int fl = flag(ch);
            if (fl == 2) continue;
            const bool turn = phase == 0 && ch >= A.nchb;
            if (turn) phase = 1;
            if ((fl == 1 || turn) && any) ++drains;
            any = true;
        }
        ++drains;
        for (int d = 0; d < drains; ++d) {
            const bool ok = __all_sync(0xffffffffu, mb_wait(dfull, d & 1, ab));
            tc_after();
            if (ok && any) {
#pragma unroll
                for (int x0 = 0; x0 < NC; x0 += 16) {
                    float t[16];  // FP32: the window's sums, smallest products first
#pragma unroll
                    for (int o = ORD - 1; o >= 0; --o) {
                        uint32_t r[16];
                        tmem_ld16(tmem + ((uint32_t)(quarter * 32) << 16) + o * NT + part * NC + x0, r);
#pragma unroll
                        for (int x = 0; x < 16; ++x) {
                            if constexpr (P == 0) {
                                const int64_t v = (int64_t)__float2int_rn(__uint_as_float(r[x])) << (8 * (3 - (o & 3)));
                                if (o < 4) hi[x0 + x] += v;
                                else lo[x0 + x] += v;
                            } else {
                                t[x] = o == ORD - 1 ? __uint_as_float(r[x]) : t[x] + __uint_as_float(r[x]);
                                if (o == 0) sum[x0 + x] += t[x];
                            }
                        }
                    }
                }
            }
            tc_before();
            __syncwarp();
            if (lane == 0) mb_arrive(dempty);
        }
        const int64_t Ia = row0 + quarter * 32 + lane, jb = col0 + part * NC;
        if (Ia < A.la) {
            T *S = static_cast<T *>(A.S) + blockIdx.z * A.la * A.lb + Ia * A.lb;
            const double sc = P == 0 ? pow2(A.tab[1] + info[1] - 8 * (ORD + 1)) : 1.0;
#pragma unroll
            for (int x = 0; x < NC; ++x)
                if (jb + x < A.lb) {
                    if constexpr (P == 0) S[jb + x] += fma((double)hi[x], 4294967296.0, (double)lo[x]) * sc;
                    else S[jb + x] += sum[x];
                }
        }
    }
    tc_before();
    __syncthreads();
    if (sAbort && tid == 0) {
        atomicExch(A.err, 1);
        if (row0 < A.la && col0 < A.lb) static_cast<T *>(A.S)[blockIdx.z * A.la * A.lb + row0 * A.lb + col0] = (T)NAN;  // fail loudly
    }
    if (warp == 17) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem_base));
}

// ------------------------------------------------------------------ alpha-beta classes

struct AbArgs {
    int64_t la, lb, lbp;
    const __nv_bfloat16 *Cs;
    void *S;
    const int *info, *tab;
    const uint4 *Vd, *Wd;  // digits of the integral columns: [pair][128], [la][128]
    const int64_t *a_soff;
    const int2 *a_sci;
    const uint4 *pos;      // [tile][4][2][128] x 8: slot of (pair, column); nslot - 1: no link
    const int2 *piece;     // [tile][npiece]: {target column (-1: not the first piece of its list), first slot |
                           // positive links << 16 | negative links << 20 | further pieces << 24}
    const int *rounds;     // [tile] pieces / kAbDrain, rounded up
    int npiece;            // pieces of the fullest tile, a multiple of kAbDrain
    int nslot;             // slots of the fullest tile, a piece more and one for pairs without a link; even
    int stage_bytes;       // shared memory for the staged c rows
    const int32_t *rowsa;
    int *err;
};

// One alpha row Ia. Its alpha terms k (Ia itself, then its singles) give G[rs][Jb] =
// sum_k A[rs][k] c(Ja_k, Jb): A's digit planes lie in TMEM for the whole row, the digit
// planes of 64 columns of the coupled c rows are gathered into shared memory (a 128-byte
// row segment each, MN-major, 128-byte swizzle). Two weights at a time go to a ring of
// accumulators, so draining one pair overlaps the products of the next. A drained G goes
// to a slot per beta link (the slots of a tile ordered by target column); a thread then
// sums the slots of a target column into the row's 64-bit sums. No atomics.
__global__ void __launch_bounds__(kAbThreads, 1) k_sigma_ab_ex(const AbArgs A) {
    const int *info = A.info + 2 * blockIdx.y;  // one vector per blockIdx.y
    if (!info[0]) return;
    typedef double T;
    constexpr int NSA = Prec<0>::NSA, NSC = Prec<0>::NSC, ORD = Prec<0>::ORD, NW = 2;
    extern __shared__ unsigned char smem_dyn[];
    __shared__ uint64_t bar[16];
    __shared__ uint32_t tmem_base;
    __shared__ int sAbort;
    __shared__ int sJa[kAbMaxK], sPq[kAbMaxK];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int64_t lb = A.lb, lbp = A.lbp, Ia = A.rowsa[blockIdx.x], t0 = A.a_soff[Ia];
    const int K = 1 + (int)(A.a_soff[Ia + 1] - t0), Kp = (K + 15) / 16 * 16;
    const uint32_t stage_sz = (uint32_t)NSC * Kp * kAbTile * 2;
    const int nst = min(4, A.stage_bytes / (int)stage_sz);
    const int dcol0 = (NSA * Kp / 2 + 31) / 32 * 32, ndb = (512 - dcol0) / (2 * kAbTile);  // accumulator pairs (Kp <= 80: at least 1)
    unsigned char *sm = smem_dyn + ((1024 - (su32(smem_dyn) & 1023)) & 1023);
    const uint32_t sB = su32(sm);
    int2 *sSlot = reinterpret_cast<int2 *>(sm + A.stage_bytes);           // [NW][nslot], 16-byte aligned
    int64_t *sAcc = reinterpret_cast<int64_t *>(sSlot + NW * A.nslot);  // [NW][lb]
    const uint32_t bfull = su32(&bar[0]), bempty = su32(&bar[4]), dfull = su32(&bar[8]), dempty = su32(&bar[12]);
    const int ntiles = (int)((lb + kAbTile - 1) / kAbTile);
    volatile int *ab = &sAbort;
    if (tid == 0) {
        sAbort = 0;
        for (int s = 0; s < 4; ++s) {
            mb_init(bfull + 8 * s, 32);
            mb_init(bempty + 8 * s, 1);
            mb_init(dfull + 8 * s, 1);
            mb_init(dempty + 8 * s, 16);
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    for (int k = tid; k < Kp; k += kAbThreads) {
        int ja = (int)Ia, pq = -1;  // padding terms: any row, zero coefficients
        if (k >= 1 && k < K) {
            const int2 e = A.a_sci[t0 + k - 1];
            ja = e.x;
            pq = e.y;
        }
        sJa[k] = ja;
        sPq[k] = pq;
    }
    for (int64_t j = tid; j < NW * lb; j += kAbThreads) sAcc[j] = 0;
    if (warp == 19) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(su32(&tmem_base)) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    tc_before();
    __syncthreads();
    tc_after();
    constexpr uint32_t tmem = 0;  // all 512 columns are this CTA's: they start at 0
    if (tid == 0 && tmem_base != 0) sAbort = 1;
    if (warp < 16) {
        // A's digit planes: lane = pair row, two terms per 32-bit column, plane s at column s Kp / 2
        const int quarter = warp & 3, rs = quarter * 32 + lane;
        for (int kb = warp >> 2; kb < Kp / 8; kb += 4) {
            uint32_t v[8][4];
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                const int k = kb * 8 + q, pq = sPq[k];
                uint4 x{};
                if (k == 0) x = A.Wd[Ia * 128 + rs];
                else if (pq >= 0) x = A.Vd[(size_t)(pq >> 1) * 128 + rs];
                const uint32_t neg = k > 0 && pq >= 0 && (pq & 1) ? 0x80008000u : 0u;
                const uint32_t *w = reinterpret_cast<const uint32_t *>(&x);
#pragma unroll
                for (int z = 0; z < 4; ++z) v[q][z] = w[z] ^ neg;
            }
#pragma unroll
            for (int s = 0; s < NSA; ++s) {
                uint32_t o[4];
#pragma unroll
                for (int z = 0; z < 4; ++z)
                    o[z] = __byte_perm(v[2 * z][s >> 1], v[2 * z + 1][s >> 1], (s & 1) ? 0x7632 : 0x5410);
                asm volatile("tcgen05.st.sync.aligned.32x32b.x4.b32 [%0], {%1, %2, %3, %4};" ::"r"(
                                 tmem + ((uint32_t)(quarter * 32) << 16) + s * (Kp / 2) + kb * 4),
                             "r"(o[0]), "r"(o[1]), "r"(o[2]), "r"(o[3])
                             : "memory");
            }
        }
        asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
    }
    tc_before();
    __syncthreads();
    tc_after();

    if (warp == 19) {
        {
            const uint32_t dbase = uni((uint32_t)dcol0);
            int db = 0, nd = 0, st = 0;  // accumulator pair, pairs begun, stage
            uint32_t dph = 1, sph = 0;   // phases of the pair (its last drain) and the stage
            bool ok = true;
            // unrolled for the row's number of 16-term steps, so that every descriptor is a
            // uniform base plus an immediate
            auto tiles = [&](auto ks_tag) {
                constexpr int KS = decltype(ks_tag)::value;
                // all products of weight O into one accumulator
                auto weight = [&](auto o_tag, uint32_t d, uint32_t b_addr) {
                    constexpr int O = decltype(o_tag)::value, I0 = O - (NSC - 1) > 0 ? O - (NSC - 1) : 0;
                    constexpr uint32_t idesc = inst_desc(kAbTile, true);
                    const uint64_t b0 = op_desc(b_addr, 16, 1024, 2);
#pragma unroll
                    for (int i = I0; i <= (NSA - 1 < O ? NSA - 1 : O); ++i)
#pragma unroll
                        for (int ks = 0; ks < KS; ++ks)
                            asm volatile(
                                "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
                                " tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n}" ::"r"(d),
                                "r"(tmem + i * (KS * 8) + ks * 8), "l"(b0 + ((O - i) * KS + ks) * (kAbTile * 2)), "r"(idesc),
                                "r"(i == I0 && ks == 0 ? 0u : 1u)
                                : "memory");
                };
                for (int t = 0; t < ntiles && ok; ++t) {
                    ok = __all_sync(0xffffffffu, mb_wait(bfull + 8 * st, sph, ab));
                    tc_after();
                    const uint32_t baddr = uni(sB + st * stage_sz);
                    auto step = [&](auto o_tag) {  // two weights into one pair of accumulators
                        constexpr int O = decltype(o_tag)::value;
                        if (!ok) return;
                        if (nd++ >= ndb) {
                            ok = __all_sync(0xffffffffu, mb_wait(dempty + 8 * db, dph, ab));
                            if (!ok) return;
                            tc_after();
                        }
                        const uint32_t d = uni(dbase + db * 2 * kAbTile);
                        if (elect_one()) {
                            weight(std::integral_constant<int, O>{}, d, baddr);
                            weight(std::integral_constant<int, O + 1>{}, d + kAbTile, baddr);
                            mma_commit(dfull + 8 * db);
                        }
                        __syncwarp();
                        if (++db == ndb) {
                            db = 0;
                            dph ^= 1;
                        }
                    };
                    step(std::integral_constant<int, 0>{});
                    step(std::integral_constant<int, 2>{});
                    step(std::integral_constant<int, 4>{});
                    step(std::integral_constant<int, 6>{});
                    if (ok && elect_one()) mma_commit(bempty + 8 * st);
                    __syncwarp();
                    if (++st == nst) {
                        st = 0;
                        sph ^= 1;
                    }
                }
            };
            switch (Kp / 16) {
                case 1: tiles(std::integral_constant<int, 1>{}); break;
                case 2: tiles(std::integral_constant<int, 2>{}); break;
                case 3: tiles(std::integral_constant<int, 3>{}); break;
                case 4: tiles(std::integral_constant<int, 4>{}); break;
                default: tiles(std::integral_constant<int, 5>{}); break;
            }
            // no MMA (and no arrival of its commit) may outlive the CTA
            if (ok && ntiles > 0) mb_wait(bempty + 8 * ((ntiles - 1) % nst), ((ntiles - 1) / nst) & 1, ab);
            if (!ok)
                for (int it = 0; it < 4096; ++it) __nanosleep(100);
        }
        __syncwarp();
    } else if (warp >= 16) {
        // a warp gathers a whole tile; three tiles are on their way (not more than there are
        // stages: a wait must not run a phase ahead of its barrier)
        const int ng = min(3, nst), g = warp - 16;
        for (int t = g; t < ntiles && g < ng; t += ng) {
            const int st = t % nst;
            if (t >= nst && !mb_wait(bempty + 8 * st, (t / nst - 1) & 1, ab)) break;
            gather_tile<NSC>(A.Cs + blockIdx.y * NSC * A.la * lbp, (size_t)A.la * lbp, lbp, sJa, Kp, t, sB + st * stage_sz);
            mb_arrive(bfull + 8 * st);
        }
    } else {
        const int quarter = warp & 3, part = warp >> 2, rs = quarter * 32 + lane;
        int db = 0;
        uint32_t ph = 0;
        // the slots and the first piece of a tile are read a tile ahead
        const uint4 *pp = A.pos + (size_t)part * 2 * 128 + rs;
        const int2 *pc = A.piece + tid;
        uint4 p0 = __ldg(pp), p1 = __ldg(pp + 128);
        int2 sg = __ldg(pc);
        int nr = __ldg(A.rounds);
        for (int t = 0; t < ntiles; ++t) {
            const uint32_t pw[8] = {p0.x, p0.y, p0.z, p0.w, p1.x, p1.y, p1.z, p1.w};
#pragma unroll
            for (int word = 0; word < NW; ++word) {
                int w[2][16];
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const bool ok = __all_sync(0xffffffffu, mb_wait(dfull + 8 * db, ph, ab));
                    tc_after();
                    uint32_t q0[16], q1[16];
                    if (ok) {
                        const uint32_t col = tmem + ((uint32_t)(quarter * 32) << 16) + dcol0 + db * 2 * kAbTile + part * 16;
                        tmem_ld16_nowait(col, q0);
                        tmem_ld16_nowait(col + kAbTile, q1);
                        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
                        pin16(q0);
                        pin16(q1);
                    } else {
#pragma unroll
                        for (int x = 0; x < 16; ++x) q0[x] = q1[x] = 0;
                    }
                    tc_before();
                    __syncwarp();
                    if (lane == 0) mb_arrive(dempty + 8 * db);
                    if (++db == ndb) {
                        db = 0;
                        ph ^= 1;
                    }
                    // the integers of two weights, 8 bits apart, in one word
                    const int o = 4 * word + 2 * h, n1 = o + 1 < NSA ? o + 2 : NSA;
                    if (n1 * (K + 7) <= 256) {
#pragma unroll
                        for (int x = 0; x < 16; ++x) w[h][x] = small_pair(q0[x], q1[x]);
                    } else {
#pragma unroll
                        for (int x = 0; x < 16; ++x) w[h][x] = large_pair(q0[x], q1[x]);
                    }
                }
                if (word == 0) asm volatile("bar.sync 1, 512;" ::: "memory");  // the last tile's slots are read
#pragma unroll
                for (int x = 0; x < 16; ++x) {
                    const uint32_t e = (pw[x >> 1] >> (16 * (x & 1))) & 0xFFFFu;
                    sSlot[word * A.nslot + e] = make_int2(w[0][x], w[1][x]);  // no link: the last slot
                }
            }
            const int rounds = nr;
            const int2 *cur = pc;
            int2 sg1 = rounds > 1 ? __ldg(cur + kAbDrain) : make_int2(-1, 0);
            if (t + 1 < ntiles) {
                pp += 4 * 2 * 128;
                pc += A.npiece;
                p0 = __ldg(pp);
                p1 = __ldg(pp + 128);
                nr = __ldg(A.rounds + t + 1);
            }
            asm volatile("bar.sync 1, 512;" ::: "memory");  // this tile's slots are written
            for (int i = 0; i < rounds; ++i) {
                const uint32_t y = (uint32_t)sg.y;
                const int ib = sg.x, first = y & 0xFFFF, np = (y >> 16) & 0xF, n = np + ((y >> 20) & 0xF);
                const int more = y >> 24;  // further pieces, in the lanes above
                sg = sg1;
                if (i + 2 < rounds) sg1 = __ldg(cur + (i + 2) * kAbDrain);
                int64_t v[NW];
#pragma unroll
                for (int word = 0; word < NW; ++word) {
                    const int2 *sl = sSlot + word * A.nslot + first;
                    int2 z[kPiece];
#pragma unroll
                    for (int k = 0; k < kPiece; ++k) z[k] = sl[k];
                    v[word] = 0;
#pragma unroll
                    for (int k = 0; k < kPiece; ++k) {
                        const int sgn = k < np ? 1 : k < n ? -1 : 0;
                        v[word] += (int64_t)(int)((uint32_t)z[k].x - kPairBias) * (sgn * 65536) +
                                   (int64_t)(int)((uint32_t)z[k].y - kPairBias) * sgn;
                    }
                }
                const int steps = __reduce_max_sync(0xffffffffu, (unsigned)more);
                for (int d = 1; d <= steps; d <<= 1)
#pragma unroll
                    for (int word = 0; word < NW; ++word) {
                        const int64_t z = __shfl_down_sync(0xffffffffu, v[word], d);
                        if (d <= more) v[word] += z;
                    }
                if (ib >= 0)
#pragma unroll
                    for (int word = 0; word < NW; ++word) sAcc[word * lb + ib] += v[word];
            }
            sg = __ldg(pc);
        }
    }
    tc_before();
    __syncthreads();
    T *S = static_cast<T *>(A.S) + (blockIdx.y * A.la + Ia) * lb;
    const double sc = pow2(A.tab[0] + info[1] - 8 * (ORD + 1));
    for (int64_t j = tid; j < lb; j += kAbThreads) {
        S[j] += fma((double)sAcc[j], 4294967296.0, (double)sAcc[lb + j]) * sc;
    }
    if (sAbort && tid == 0) {
        atomicExch(A.err, 1);
        S[0] = (T)NAN;  // fail loudly
    }
    if (warp == 19) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem_base));
}


// ------------------------------------------------------------------ host side

typedef CUresult (*EncodeTiled)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *, const cuuint64_t *,
                                const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave, CUtensorMapSwizzle,
                                CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiled encode_tiled() {
    static const EncodeTiled fn = [] {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) != cudaSuccess ||
            q != cudaDriverEntryPointSuccess)
            p = nullptr;
        return (EncodeTiled)p;
    }();
    return fn;
}

// digit planes [sets][planes][rows][cols] (cols a multiple of 64), box [all planes][box_rows][box_cols]
bool plane_map(CUtensorMap *m, void *base, int64_t cols, int64_t rows, int planes, int box_cols, int box_rows, int sets = 1) {
    const cuuint64_t dims[3] = {(cuuint64_t)cols, (cuuint64_t)rows, (cuuint64_t)planes * sets};
    const cuuint64_t strides[2] = {(cuuint64_t)cols * 2, (cuuint64_t)cols * rows * 2};
    const cuuint32_t box[3] = {(cuuint32_t)box_cols, (cuuint32_t)box_rows, (cuuint32_t)planes}, es[3] = {1, 1, 1};
    const EncodeTiled fn = encode_tiled();
    return fn && fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, base, dims, strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE,
                    box_cols == 64 ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_64B,
                    CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

}  // namespace

// What the exact path keeps for one prepared space and precision, in one allocation of spare
// memory made by the first sigma that takes it. Calls on several streams share the digit planes
// of c, so each call waits for the event that the one before it recorded; `mu` keeps the
// launches of one call together.
struct ExactData : Spare {
    struct Type {
        bool tried = false, ready = false;
        int batch = 1;  // vectors per launch
        cudaEvent_t busy = nullptr;
        size_t charged = 0;
        DevBuf<unsigned char> arena;
        uint4 *Vd = nullptr, *Wd = nullptr;
        __nv_bfloat16 *planes = nullptr;  // digit planes of `batch` vectors
        double *part = nullptr;
        int *info = nullptr, *tab = nullptr;
        unsigned *done = nullptr;
        Outliers out{};
        Coarse low{};
        SsArgs ss{};
    } type[2];
    explicit ExactData(tbsci_ctx *x) : Spare(x) { enlist(); }
    ~ExactData() override {
        retire();
        for (Type &t : type) {
            uncharge(ctx, t.charged);
            if (t.busy) cudaEventDestroy(t.busy);
        }
    }
    bool give_back() override {
        bool freed = false;
        for (Type &t : type) {
            if (!t.arena.p || cudaEventSynchronize(t.busy) != cudaSuccess) continue;
            t.arena.release();
            uncharge(ctx, t.charged);
            t.charged = 0;
            t.tried = t.ready = false;
            freed = true;
        }
        return freed;
    }
};

namespace {

inline int64_t pad64(int64_t l) { return (l + 63) / 64 * 64; }

size_t ab_fixed_smem(const Plan *P) { return 1024 + 16 * ((size_t)P->B.l + P->tl_nslot); }

// shared memory of the FP64 kernel's staged c rows: as many stages as fit (at most four of
// the fullest row), at least one
int ab_stage_bytes(const tbsci_ctx *ctx, const Plan *P) {
    const int one = Prec<0>::NSC * P->tl_kpmax * kAbTile * 2;
    const int64_t room = ((int64_t)ctx->smem_optin - 2048 - (int64_t)ab_fixed_smem(P)) / 1024 * 1024;
    return room < one ? 0 : (int)std::min<int64_t>(room, 4 * (int64_t)one);
}

// Places in the allocation of one precision, 256-byte aligned, and its size
struct Places {
    size_t hb, ha, top, done, zeroed, vd, wd, cb, ca, fb, fa, part, info, tab, thr, count, list, need, lows, lowl, planes, bytes;
};
template <int PR>
Places places_of(int64_t la, int64_t lb, int npair) {
    constexpr int NSA = Prec<PR>::NSA, NSC = Prec<PR>::NSC, NT = SsShape<PR>::NT;
    const size_t batch = (size_t)sigma_tc_batch(la * lb), lap = (size_t)pad64(la), lbp = (size_t)pad64(lb);
    const size_t ncha = (size_t)(la + 31) / 32, nchb = (size_t)(lb + 31) / 32;
    Places p;
    size_t at = 0;
    auto place = [&](size_t n) {
        const size_t q = at;
        at += (n + 255) / 256 * 256;
        return q;
    };
    p.hb = place(NSA * lb * lbp * 2);
    p.ha = place(NSA * la * lap * 2);
    p.top = place(16);
    p.done = place(4 * batch);
    p.zeroed = at;
    p.vd = place(PR == 0 ? (size_t)npair * 128 * sizeof(uint4) : 0);
    p.wd = place(PR == 0 ? (size_t)la * 128 * sizeof(uint4) : 0);
    p.cb = place(lb * nchb);
    p.ca = place(la * ncha);
    p.fb = place((size_t)(lb + NT - 1) / NT * nchb);
    p.fa = place((size_t)(la + 127) / 128 * ncha);
    p.part = place(batch * 2 * kScaleBlocks * 8);
    p.info = place(8 * batch);
    p.tab = place(12);
    p.thr = place(8 * batch);
    p.count = place(4 * batch);
    p.list = place(8 * batch * kOutliers);
    p.need = place(4 * batch);
    p.lows = place(4 * batch);
    p.lowl = place(PR == 0 ? 4 * batch * (size_t)(la * lb / kCoarseShare) : 0);
    p.planes = place(batch * NSC * la * lbp * 2);
    p.bytes = at;
    return p;
}

// Digit tables of the Hamiltonian for one precision, enqueued on `st`; without room for
// them the space stays on the SIMT kernels.
template <int PR>
tbsci_status build_type(tbsci_ctx *ctx, const tbsci_ham *ham, Plan *P, ExactData *X, cudaStream_t st) {
    typename ExactData::Type &Y = X->type[PR];
    using Sh = SsShape<PR>;
    const int64_t la = P->A.l, lb = P->B.l, lap = pad64(la), lbp = pad64(lb);
    constexpr int NSA = Prec<PR>::NSA, NSC = Prec<PR>::NSC;
    if ((PR == 0 ? ab_stage_bytes(ctx, P) == 0 : !sigma_tc_serves(ctx, P, 3)) || !encode_tiled()) {
        Y.tried = true;
        return TBSCI_OK;
    }
    const int ncha = (int)((la + 31) / 32), nchb = (int)((lb + 31) / 32);
    const int64_t nba = (la + 127) / 128, nbb = (lb + Sh::NT - 1) / Sh::NT;
    Y.batch = sigma_tc_batch(la * lb);
    Y.low.limit = PR == 0 ? (unsigned)(la * lb / kCoarseShare) : 0;
    const auto [hb, ha, top, done, zeroed, vd, wd, cb, ca, fb, fa, part, info, tab, thr, count, list, need, lows, lowl, planes, at] =
        places_of<PR>(la, lb, P->npair);
    if (!spare_charge(ctx, at)) return TBSCI_OK;  // asked for again by the next call
    Y.tried = true;
    Y.charged = at;
    cudaError_t e = Y.busy ? cudaSuccess : cudaEventCreateWithFlags(&Y.busy, cudaEventDisableTiming);
    if (e == cudaSuccess) e = Y.arena.alloc(at, true);
    unsigned char *B = Y.arena.p;
    if (e == cudaSuccess) e = cudaMemsetAsync(B, 0, zeroed, st);
    SsArgs &S = Y.ss;
    if (e == cudaSuccess) {
        Y.Vd = reinterpret_cast<uint4 *>(B + vd);
        Y.Wd = reinterpret_cast<uint4 *>(B + wd);
        Y.planes = reinterpret_cast<__nv_bfloat16 *>(B + planes);
        Y.part = reinterpret_cast<double *>(B + part);
        Y.info = reinterpret_cast<int *>(B + info);
        Y.tab = reinterpret_cast<int *>(B + tab);
        Y.done = reinterpret_cast<unsigned *>(B + done);
        Y.out = {reinterpret_cast<double *>(B + thr), reinterpret_cast<int *>(B + count), reinterpret_cast<int64_t *>(B + list)};
        Y.low.need = reinterpret_cast<float *>(B + need);
        Y.low.count = reinterpret_cast<unsigned *>(B + lows);
        Y.low.list = reinterpret_cast<int32_t *>(B + lowl);
        unsigned long long *tp = reinterpret_cast<unsigned long long *>(B + top);
        auto blocks = [&](size_t n) { return (unsigned)std::min<size_t>(ctx->num_sms, (n + 255) / 256); };
        k_absmax_off<<<blocks((size_t)P->npair * P->npoff), 256, 0, st>>>(ham->d_V.p, P->npair, P->npoff, P->d_offpair.p, tp);
        for (const SpinPlan *sp : {&P->A, &P->B}) {
            if (sp->d_sval.n) k_absmax<<<blocks(sp->d_sval.n), 256, 0, st>>>(sp->d_sval.p, (int64_t)sp->d_sval.n, tp + 1);
            if (sp->d_dval.n) k_absmax<<<blocks(sp->d_dval.n), 256, 0, st>>>(sp->d_dval.p, (int64_t)sp->d_dval.n, tp + 1);
        }
        k_table_scales<<<1, 1, 0, st>>>(tp, std::max(1.0, P->A.nelec / 8.0), Y.tab);
        if (PR == 0) {
            k_ab_digits<<<(unsigned)(((int64_t)P->npair * 128 + 255) / 256), 256, 0, st>>>(ham->d_V.p, P->npair, P->npoff, P->d_offpair.p,
                                                                                          nullptr, P->npair, Y.tab, Y.Vd);
            k_ab_digits<<<(unsigned)((la * 128 + 255) / 256), 256, 0, st>>>(ham->d_V.p, P->npair, P->npoff, P->d_offpair.p, P->A.d_str, la,
                                                                           Y.tab, Y.Wd);
        }
        k_dense_digits<PR><<<(unsigned)((lb + 7) / 8), 256, 32 * (size_t)nchb, st>>>(
            lb, lbp, nchb, P->B.d_soff, P->B.d_sci.p, P->B.d_sval.p, P->B.d_doff, P->B.d_dcol.p, P->B.d_dval.p, Y.tab,
            reinterpret_cast<__nv_bfloat16 *>(B + hb), B + cb);
        k_windows<<<(unsigned)nbb, 128, 0, st>>>(lb, nchb, Sh::NT, B + cb, B + fb);
        k_dense_digits<PR><<<(unsigned)((la + 7) / 8), 256, 32 * (size_t)ncha, st>>>(
            la, lap, ncha, P->A.d_soff, P->A.d_sci.p, P->A.d_sval.p, P->A.d_doff, P->A.d_dcol.p, P->A.d_dval.p, Y.tab,
            reinterpret_cast<__nv_bfloat16 *>(B + ha), B + ca);
        k_windows<<<(unsigned)nba, 128, 0, st>>>(la, ncha, 128, B + ca, B + fa);
        e = cudaGetLastError();
    }
    const bool maps = e == cudaSuccess && plane_map(&S.mHb, B + hb, lbp, lb, NSA, 32, Sh::NT) &&
                      plane_map(&S.mHa, B + ha, lap, la, NSA, 32, 128) &&
                      plane_map(&S.mCA, Y.planes, lbp, la, NSC, 32, 128, Y.batch) &&
                      plane_map(&S.mCB, Y.planes, lbp, la, NSC, 64, 32, Y.batch);
    if (!maps) {
        Y.arena.release();
        Y.charged = 0;
        uncharge(ctx, at);
        cudaGetLastError();
        return e == cudaSuccess || e == cudaErrorMemoryAllocation ? TBSCI_OK
                                                                   : fail(ctx, TBSCI_ECUDA, std::string("digit tables: ") + cudaGetErrorString(e));
    }
    S.la = la;
    S.lb = lb;
    S.nchb = nchb;
    S.ncha = ncha;
    S.flb = B + fb;
    S.fla = B + fa;
    S.info = Y.info;
    S.tab = Y.tab;
    S.err = P->d_tc_err.p;
    TB_CUDA(ctx, cudaEventRecord(Y.busy, st));  // other streams wait for the tables
    Y.ready = true;
    return TBSCI_OK;
}

UdArgs<double> ud_args(const tbsci_ham *ham, const Plan *P, double) {
    return {P->A.l, P->B.l, nullptr, nullptr, nullptr, P->A.d_str, P->A.d_soff, P->A.d_sci.p, P->A.d_sval.p, P->A.d_E.p,
            P->B.d_E.p, P->d_U.p, ham->ecore, P->A.nelec, 0, P->A.d_svalf.p, nullptr, {}};
}
UdArgs<float> ud_args(const tbsci_ham *ham, const Plan *P, float) {
    return {P->A.l, P->B.l, nullptr, nullptr, nullptr, P->A.d_str, P->A.d_soff, P->A.d_sci.p, P->A.d_svalf.p, P->A.d_Ef.p,
            P->B.d_Ef.p, P->d_Uf.p, (float)ham->ecore, P->A.nelec, 0, nullptr, nullptr, {}};
}

}  // namespace

// Whether a space takes this path. It wins at every shape and link density tried from
// 2^14 determinants and two tiles of columns on (one vector, ms, against the SIMT kernels):
//   160 x 155 strings, norb 12         FP64 0.11 / 0.21    FP32 0.07 / 0.12
//   500 x 200, norb 14                 0.18 / 0.42         0.10 / 0.24
//   1,200 x 1,100, norb 16             1.1 / 2.9           0.31 / 1.4
//   1,800 x 1,800, norb 16             2.4 / 5.6           0.68 / 2.4
// but not below: 100 x 100 0.09 / 0.09 and 0.08 / 0.06, 2,000 x 60 0.33 / 0.42 and 0.20 / 0.17.
template <typename T>
bool exact_eligible(const Plan *P) {
    const int64_t la = P->A.l, lb = P->B.l;
    if (P->no_spare || P->tl_kpmax == 0 || la < 32 || lb < 2 * kAbTile || la > 32768 || lb > 32768) return false;
    if (P->tune_stage[sizeof(T) == 8 ? 0 : 1] >= 3) return false;  // a shape of the split path was asked for
    return la * lb >= (int64_t(1) << 14);
}

// Spare bytes that sigma of a type (0 FP64, 1 FP32) takes on a space of these sizes; an upper
// bound, without a look at its links
size_t exact_device_bytes(int norb, int64_t la, int64_t lb, int type) {
    if (norb < 2 || norb > 16 || la < 32 || lb < 2 * kAbTile || la > 32768 || lb > 32768 || la * lb < (int64_t(1) << 14)) return 0;
    const int npair = norb * (norb + 1) / 2;
    return type == 0 ? places_of<0>(la, lb, npair).bytes : places_of<1>(la, lb, npair).bytes;
}

// sigma of the vectors c -> s; *ran = false (and nothing launched) where the path does
// not apply: the SIMT kernels then serve the call. `simt(v, nv, skip)` launches those for
// vectors v .. v + nv - 1, to return at once where skip[2 i] is set.
template <typename T, int PR>
tbsci_status exact_launch_t(tbsci_ctx *ctx, const tbsci_ham *ham, Plan *P, const T *c, T *s, int nvec, cudaStream_t st,
                            bool *ran, const std::function<tbsci_status(int, int, const int *, const OutlierArgs &)> &simt) {
    *ran = false;
    if (!exact_eligible<T>(P)) return TBSCI_OK;
    // the tables are made outside of graphs, and a graph's replays would share them with other streams
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(st, &cap) != cudaSuccess || cap != cudaStreamCaptureStatusNone) {
        cudaGetLastError();
        return TBSCI_OK;
    }
    {
        static std::mutex make;
        std::lock_guard<std::mutex> g(make);
        if (!P->exact) P->exact = std::make_shared<ExactData>(ctx);
    }
    ExactData *X = P->exact.get();
    std::lock_guard<std::mutex> g(X->mu);
    typename ExactData::Type &Y = X->type[PR];
    if (!Y.tried) TB_TRY((build_type<PR>(ctx, ham, P, X, st)));
    if (!Y.ready) return TBSCI_OK;
    using Sh = SsShape<PR>;
    const int64_t la = P->A.l, lb = P->B.l, lbp = pad64(lb);
    auto kss = k_same_spin_ex<PR>;
    TB_CUDA(ctx, cudaFuncSetAttribute(kss, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Sh::kSmem));
    UdArgs<T> U = ud_args(ham, P, T(0));
    U.info = U.flag = Y.info;
    U.R = Y.low;
    AbArgs A{};
    const OutlierArgs out{Y.out, Y.low, lb, P->A.d_str, P->A.d_soff, P->A.d_doff, P->B.d_soff, P->B.d_doff,
                   P->A.d_sci.p, P->B.d_sci.p, P->A.d_sval.p, P->B.d_sval.p, P->A.d_dval.p, P->B.d_dval.p, ham->d_V.p,
                   P->A.d_dcol.p, P->B.d_dcol.p, P->npair};
    size_t ab_smem = 0;
    if (PR == 0) {
        A.la = la;
        A.lb = lb;
        A.lbp = lbp;
        A.Cs = Y.planes;
        A.info = Y.info;
        A.tab = Y.tab;
        A.Vd = Y.Vd;
        A.Wd = Y.Wd;
        A.a_soff = P->A.d_soff;
        A.a_sci = P->A.d_sci.p;
        A.pos = P->d_tl_pos.p;
        A.piece = P->d_tl_piece.p;
        A.rounds = P->d_tl_rounds.p;
        A.npiece = P->tl_npiece;
        A.nslot = P->tl_nslot;
        A.stage_bytes = ab_stage_bytes(ctx, P);
        A.rowsa = P->d_rowsa.p;
        A.err = P->d_tc_err.p;
        ab_smem = ab_fixed_smem(P) + A.stage_bytes;
        TB_CUDA(ctx, cudaFuncSetAttribute(k_sigma_ab_ex, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)ab_smem));
    }
    *ran = true;
    TB_CUDA(ctx, cudaStreamWaitEvent(st, Y.busy, 0));
    // whatever became of the launches, the next user of the tables waits for those made
    struct Record {
        cudaEvent_t e;
        cudaStream_t st;
        ~Record() { cudaEventRecord(e, st); }
    } record{Y.busy, st};
    for (int v = 0, nv = 0; v < nvec; v += nv) {
        nv = std::min(Y.batch, nvec - v);
        const T *cv = c + (size_t)v * la * lb;
        T *sv = s + (size_t)v * la * lb;
        {
            TraceScope tr(ctx, "k_scale", st);
            const unsigned nb = (unsigned)std::min<int64_t>(kScaleBlocks, (la * lb + 4 * kScaleThreads - 1) / (4 * kScaleThreads));
            k_scale<T><<<dim3(nb, (unsigned)nv), kScaleThreads, 0, st>>>(cv, la * lb, Prec<PR>::kRatio, PR == 0 ? kOutlierMaxN : 0,
                                                                        Y.part, Y.done, Y.tab, Y.info, Y.out, Y.low);
            TB_CUDA(ctx, cudaGetLastError());
        }
        {
            TraceScope tr(ctx, "k_udiag", st);
            U.C = cv;
            U.S = sv;
            k_udiag<T, false, PR == 0><<<ud_grid(la, lb, nv), 256, 0, st>>>(U);
            TB_CUDA(ctx, cudaGetLastError());
        }
        if constexpr (PR == 0) {
            TraceScope tr(ctx, "k_slice", st);
            const unsigned ns = (unsigned)std::min<int64_t>(8ll * ctx->num_sms, (la * (lbp / 8) + 255) / 256);
            k_slice<<<dim3(ns, (unsigned)nv), 256, 0, st>>>(cv, la, lb, lbp, Y.info, Y.out, Y.planes);
            TB_CUDA(ctx, cudaGetLastError());
        } else {
            TB_TRY(sigma_tc_planes(ctx, P, cv, nv, Y.info, Y.planes, st));
        }
        {
            TraceScope tr(ctx, "k_same_spin_ex", st);
            Y.ss.S = sv;
            kss<<<dim3((unsigned)((lb + Sh::NT - 1) / Sh::NT), (unsigned)((la + 127) / 128), (unsigned)nv), kSsThreads, Sh::kSmem,
                  st>>>(Y.ss);
            TB_CUDA(ctx, cudaGetLastError());
        }
        if constexpr (PR == 0) {
            TraceScope tr(ctx, "k_sigma_ab_ex", st);
            A.S = sv;
            k_sigma_ab_ex<<<dim3((unsigned)la, (unsigned)nv), kAbThreads, ab_smem, st>>>(A);
            TB_CUDA(ctx, cudaGetLastError());
        } else {
            TB_TRY(sigma_tc_ab(ctx, P, 3, cv, sv, nv, Y.info, st, Y.planes));
        }
        TB_TRY(simt(v, nv, Y.info, out));
    }
    return TBSCI_OK;
}

tbsci_status exact_launch(tbsci_ctx *ctx, const tbsci_ham *ham, Plan *P, const double *c, double *s, int nvec,
                          cudaStream_t st, bool *ran, const std::function<tbsci_status(int, int, const int *, const OutlierArgs &)> &simt) {
    return exact_launch_t<double, 0>(ctx, ham, P, c, s, nvec, st, ran, simt);
}
tbsci_status exact_launch(tbsci_ctx *ctx, const tbsci_ham *ham, Plan *P, const float *c, float *s, int nvec,
                          cudaStream_t st, bool *ran, const std::function<tbsci_status(int, int, const int *, const OutlierArgs &)> &simt) {
    return exact_launch_t<float, 1>(ctx, ham, P, c, s, nvec, st, ran, simt);
}

// s (+)= the diagonal and the alpha singles with the beta string unchanged, FP32 (see k_udiag)
tbsci_status udiag_launch(tbsci_ctx *ctx, const tbsci_ham *ham, const Plan *P, const float *c, float *s, int nv, bool add,
                          bool singles, cudaStream_t st) {
    UdArgs<float> U = ud_args(ham, P, 0.f);
    U.C = c;
    U.S = s;
    U.add = add;
    TraceScope tr(ctx, "k_udiag", st);
    if (singles) k_udiag<float, true, false><<<ud_grid(P->A.l, P->B.l, nv), 256, 0, st>>>(U);
    else k_udiag<float, false, false><<<ud_grid(P->A.l, P->B.l, nv), 256, 0, st>>>(U);
    TB_CUDA(ctx, cudaGetLastError());
    return TBSCI_OK;
}

}  // namespace tbsci

// Bitstring selection and coefficient distributions (Sec. III.B and Fig. 3).
//
// The weight of an alpha string w in a normalised TPB vector is
// W_a(w) = sum_u c(w, u)^2 and of a beta string u is W_b(u) = sum_w c(w, u)^2;
// strings are kept when their weight is at least delta times the weight of the
// HF string (here: the string of largest weight), and the TPB space of the kept
// strings is solved again. The coefficient distribution counts |c_K| in
// logarithmic bins of |c_K / c_HF| (the caller passes the bin edges already
// scaled by |c_HF|, so both this code and a reference compare the same doubles).
// Every reduction has a fixed order: results are run-to-run identical.
#include <algorithm>
#include <cstring>
#include <vector>

#include "internal.cuh"

namespace tbsci {

namespace {

constexpr int kWThreads = 256;
// rows per partial column sum: short enough that 3,000 x 3,000 strings make 564 CTAs (256
// rows made 144, each a serial chain of loads: 40 us; now the pass takes about as long as
// its 15 us of FP64 multiply-adds)
constexpr int64_t kColRows = 64;

// rows[w] = sum_u c(w, u)^2, one CTA per row, fixed-order tree reduction
__global__ void __launch_bounds__(kWThreads) k_row_sumsq(const double *__restrict__ c, int64_t lb, double *rows) {
    __shared__ double sh[kWThreads];
    const double *r = c + (int64_t)blockIdx.x * lb;
    double acc = 0.0;
#pragma unroll 4
    for (int64_t u = threadIdx.x; u < lb; u += kWThreads) acc = fma(r[u], r[u], acc);
    sh[threadIdx.x] = acc;
    __syncthreads();
    for (int o = kWThreads / 2; o > 0; o >>= 1) {
        if (threadIdx.x < o) sh[threadIdx.x] += sh[threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0) rows[blockIdx.x] = sh[0];
}

// partial[chunk][u] = sum_{w in chunk} c(w, u)^2 over chunks of `rows` rows
__global__ void __launch_bounds__(kWThreads) k_col_sumsq(const double *__restrict__ c, int64_t la, int64_t lb,
                                                          int64_t rows, double *partial) {
    const int64_t u = (int64_t)blockIdx.x * kWThreads + threadIdx.x;
    if (u >= lb) return;
    const int64_t w0 = blockIdx.y * rows, w1 = min(la, w0 + rows);
    double acc = 0.0;
#pragma unroll 8
    for (int64_t w = w0; w < w1; ++w) {
        const double x = __ldg(c + w * lb + u);
        acc = fma(x, x, acc);
    }
    partial[(int64_t)blockIdx.y * lb + u] = acc;
}

// out[u] = sum_chunk partial[chunk][u] in chunk order
__global__ void k_col_reduce(const double *__restrict__ partial, int64_t nchunk, int64_t lb, double *out) {
    const int64_t u = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (u >= lb) return;
    double acc = 0.0;
    for (int64_t k = 0; k < nchunk; ++k) acc += partial[k * lb + u];
    out[u] = acc;
}

constexpr int kHistThreads = 256;

// counts[k] += values with edges[k - 1] <= |x| < edges[k] (bin 0 below edges[0], bin nedges
// at or above the last). Non-negative doubles order as their bit patterns, so the search
// compares 64-bit integers (an FP64 compare per step took the FP64 pipe 60 us at 9.0M
// values), each warp counts into its own 32-bit bins, and a CTA adds them up at its end;
// the sums are exact whatever their order. Bound by HBM: 72 MB in 13 us at its rate.
__global__ void __launch_bounds__(kHistThreads) k_histogram(const double *__restrict__ x, int64_t n,
                                                            const int64_t *__restrict__ edges, int nedges, int steps,
                                                            unsigned long long *counts) {
    extern __shared__ unsigned sbin[];  // [warps][nedges + 1]
    __shared__ int64_t sedge[512];      // padded to 2^steps - 1 with the largest integer
    const int bins = nedges + 1;
    for (int k = threadIdx.x; k < (kHistThreads / 32) * bins; k += kHistThreads) sbin[k] = 0;
    for (int k = threadIdx.x; k < (1 << steps) - 1; k += kHistThreads) sedge[k] = k < nedges ? edges[k] : INT64_MAX;
    __syncthreads();
    unsigned *mine = sbin + (threadIdx.x >> 5) * bins;
    auto count = [&](double v) {
        const int64_t a = __double_as_longlong(v) & INT64_MAX;
        int lo = 0;  // edges at or below a
        for (int h = 1 << (steps - 1); h > 0; h >>= 1)
            if (sedge[lo + h - 1] <= a) lo += h;
        if (a > 0x7FF0000000000000ll) lo = 0;  // NaN is at or above no edge
        atomicAdd(mine + lo, 1u);
    };
    const int64_t step = (int64_t)gridDim.x * kHistThreads;
    int64_t i = blockIdx.x * (int64_t)kHistThreads + threadIdx.x;
    for (; i + 3 * step < n; i += 4 * step) {
        const double a = __ldg(x + i), b = __ldg(x + i + step), c = __ldg(x + i + 2 * step), d = __ldg(x + i + 3 * step);
        count(a);
        count(b);
        count(c);
        count(d);
    }
    for (; i < n; i += step) count(__ldg(x + i));
    __syncthreads();
    for (int k = threadIdx.x; k < bins; k += kHistThreads) {
        unsigned long long t = 0;
        for (int w = 0; w < kHistThreads / 32; ++w) t += sbin[w * bins + k];
        if (t) atomicAdd(counts + k, t);
    }
}

tbsci_status weights_raw(tbsci_ctx *ctx, int64_t la, int64_t lb, const double *c, std::vector<double> &wa,
                         std::vector<double> &wb, cudaStream_t st) {
    wa.assign(la, 0.0);
    wb.assign(lb, 0.0);
    if (la == 0 || lb == 0) return TBSCI_OK;
    const int64_t chunk = la <= 65535 * kColRows ? kColRows : 4 * kColRows, nchunk = (la + chunk - 1) / chunk;
    DevBuf<double> sums, partial;  // row sums, then column sums: one copy to the host
    TB_CUDA(ctx, sums.alloc(la + lb));
    TB_CUDA(ctx, partial.alloc((size_t)nchunk * lb));
    TB_CHECK(ctx, la <= INT32_MAX && nchunk <= 65535, TBSCI_EINVAL, "string weights: too many alpha strings");
    k_row_sumsq<<<(unsigned)la, kWThreads, 0, st>>>(c, lb, sums.p);
    TB_CUDA(ctx, cudaGetLastError());
    k_col_sumsq<<<dim3((unsigned)((lb + kWThreads - 1) / kWThreads), (unsigned)nchunk), kWThreads, 0, st>>>(
        c, la, lb, chunk, partial.p);
    TB_CUDA(ctx, cudaGetLastError());
    k_col_reduce<<<(unsigned)((lb + 255) / 256), 256, 0, st>>>(partial.p, nchunk, lb, sums.p + la);
    TB_CUDA(ctx, cudaGetLastError());
    std::vector<double> h(la + lb);
    TB_CUDA(ctx, cudaMemcpyAsync(h.data(), sums.p, h.size() * sizeof(double), cudaMemcpyDeviceToHost, st));
    TB_CUDA(ctx, cudaStreamSynchronize(st));
    std::copy(h.begin(), h.begin() + la, wa.begin());
    std::copy(h.begin() + la, h.end(), wb.begin());
    double tot = 0.0;  // ||c||^2 from the row sums, in row order
    for (double x : wa) tot += x;
    TB_CHECK(ctx, tot > 0.0, TBSCI_EINVAL, "string weights: the vector is zero");
    for (double &x : wa) x /= tot;
    for (double &x : wb) x /= tot;
    return TBSCI_OK;
}

}  // namespace

}  // namespace tbsci

using namespace tbsci;

extern "C" {

tbsci_status tbsci_string_weights(tbsci_ctx *ctx, const tbsci_tables *a, const tbsci_tables *b, const double *c,
                                  double *wa, double *wb, tbsci_stream stream) {
    if (!ctx) return TBSCI_EINVAL;
    TB_CUDA(ctx, cudaSetDevice(ctx->device));
    TB_CHECK(ctx, a && b && wa && wb, TBSCI_EINVAL, "tbsci_string_weights: null argument");
    TB_CHECK(ctx, c || a->count * b->count == 0, TBSCI_EINVAL, "tbsci_string_weights: null vector");
    std::vector<double> va, vb;
    TB_TRY(weights_raw(ctx, a->count, b->count, c, va, vb, (cudaStream_t)stream));
    std::memcpy(wa, va.data(), va.size() * sizeof(double));
    std::memcpy(wb, vb.data(), vb.size() * sizeof(double));
    return TBSCI_OK;
}

tbsci_status tbsci_select_by_weight(tbsci_ctx *ctx, const tbsci_tables *a, const tbsci_tables *b, const double *c,
                                    double delta, uint64_t *sel_a, int64_t *na, uint64_t *sel_b, int64_t *nb,
                                    tbsci_stream stream) {
    if (!ctx) return TBSCI_EINVAL;
    TB_CUDA(ctx, cudaSetDevice(ctx->device));
    TB_CHECK(ctx, a && b && c && sel_a && na && sel_b && nb, TBSCI_EINVAL, "tbsci_select_by_weight: null argument");
    TB_CHECK(ctx, delta >= 0.0, TBSCI_EINVAL, "tbsci_select_by_weight: delta must be >= 0");
    TB_CHECK(ctx, a->count > 0 && b->count > 0, TBSCI_EINVAL, "tbsci_select_by_weight: empty space");
    std::vector<double> wa, wb;
    cudaStream_t st = (cudaStream_t)stream;
    TB_TRY(weights_raw(ctx, a->count, b->count, c, wa, wb, st));
    std::vector<uint64_t> sa(a->count), sb(b->count);
    TB_CUDA(ctx, cudaMemcpy(sa.data(), a->d_str.p, a->count * sizeof(uint64_t), cudaMemcpyDeviceToHost));
    TB_CUDA(ctx, cudaMemcpy(sb.data(), b->d_str.p, b->count * sizeof(uint64_t), cudaMemcpyDeviceToHost));
    auto pick = [&](const std::vector<double> &w, const std::vector<uint64_t> &s, uint64_t *out, int64_t *n) {
        const double hf = *std::max_element(w.begin(), w.end());  // the HF string: largest weight
        int64_t k = 0;
        for (size_t i = 0; i < w.size(); ++i)
            if (w[i] >= delta * hf) out[k++] = s[i];
        *n = k;
    };
    pick(wa, sa, sel_a, na);
    pick(wb, sb, sel_b, nb);
    return TBSCI_OK;
}

tbsci_status tbsci_coefficient_histogram(tbsci_ctx *ctx, const double *x, int64_t n, const double *edges, int nedges,
                                         int64_t *counts, tbsci_stream stream) {
    if (!ctx) return TBSCI_EINVAL;
    TB_CUDA(ctx, cudaSetDevice(ctx->device));
    TB_CHECK(ctx, edges && counts && n >= 0, TBSCI_EINVAL, "tbsci_coefficient_histogram: null argument");
    TB_CHECK(ctx, nedges >= 1 && nedges <= 256, TBSCI_EINVAL, "tbsci_coefficient_histogram: 1..256 edges");
    for (int k = 1; k < nedges; ++k)
        TB_CHECK(ctx, edges[k] > edges[k - 1], TBSCI_EINVAL, "tbsci_coefficient_histogram: edges must ascend");
    std::fill(counts, counts + nedges + 1, 0);
    if (n == 0) return TBSCI_OK;
    TB_CHECK(ctx, x, TBSCI_EINVAL, "tbsci_coefficient_histogram: null vector");
    cudaStream_t st = (cudaStream_t)stream;
    const int nblocks = (int)std::min<int64_t>(8 * ctx->num_sms, (n + 4 * kHistThreads - 1) / (4 * kHistThreads));
    std::vector<int64_t> h(2 * nedges + 1, 0);  // edges as bit patterns, then the counts (zero)
    for (int k = 0; k < nedges; ++k) {
        std::memcpy(&h[k], &edges[k], 8);
        if (edges[k] != edges[k]) h[k] = INT64_MAX;  // no value is at or above NaN
    }
    int steps = 1;
    while ((1 << steps) - 1 < nedges) ++steps;
    DevBuf<int64_t> d;
    TB_CUDA(ctx, d.alloc(h.size()));
    TB_CUDA(ctx, cudaMemcpyAsync(d.p, h.data(), h.size() * 8, cudaMemcpyHostToDevice, st));
    k_histogram<<<nblocks, kHistThreads, (kHistThreads / 32) * (nedges + 1) * sizeof(unsigned), st>>>(
        x, n, d.p, nedges, steps, reinterpret_cast<unsigned long long *>(d.p + nedges));
    TB_CUDA(ctx, cudaGetLastError());
    TB_CUDA(ctx, cudaMemcpyAsync(counts, d.p + nedges, (nedges + 1) * 8, cudaMemcpyDeviceToHost, st));
    TB_CUDA(ctx, cudaStreamSynchronize(st));
    return TBSCI_OK;
}

}  // extern "C"

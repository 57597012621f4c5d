// String sets (Sec. II.A, Eq. 3) and their single/double excitation links
// (BETA_SINGLE_LINK / BETA_DOUBLE_LINK, Sec. II.C), built on the device.
//
// Strings: the full space is unranked in colex order (= ascending integer
// order) from the combinatorial number system; a selected list is sorted by a
// bitonic network and validated (electron count, orbital range, duplicates).
//
// Links: one warp per source string walks its candidate excitations in the
// documented order, 32 at a time; the target's index comes from the colex rank
// (full space) or a binary search (selected set), the sign from masked
// popcounts, and a ballot + prefix popcount compacts the hits in order.
// Count pass -> exclusive scan -> fill pass.
#include <algorithm>

#include "internal.cuh"

namespace tbsci {

namespace {

constexpr int kWarpsPerBlock = 8;

__device__ __forceinline__ int64_t binom(const int64_t *__restrict__ B, int m, int k) {
    return (k < 0 || k > m) ? 0 : __ldg(B + m * 65 + k);
}

// k-th combination of N out of n in colex order.
__global__ void k_unrank(uint64_t *out, int64_t count, int n, int N, const int64_t *__restrict__ B) {
    int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (k >= count) return;
    uint64_t s = 0;
    int64_t r = k;
    int top = n;  // next position must be below `top`
    for (int i = N; i >= 1; --i) {
        int c = i - 1;
        while (c + 1 < top && binom(B, c + 1, i) <= r) ++c;
        r -= binom(B, c, i);
        s |= 1ull << c;
        top = c;
    }
    out[k] = s;
}

__global__ void k_fill_u64(uint64_t *a, int64_t from, int64_t to, uint64_t v) {
    int64_t i = from + blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i < to) a[i] = v;
}

// One compare-exchange stage of a bitonic sorting network over P = 2^m keys.
__global__ void k_bitonic(uint64_t *a, int64_t P, int64_t j, int64_t k) {
    int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= P) return;
    int64_t x = i ^ j;
    if (x <= i) return;
    uint64_t u = a[i], v = a[x];
    bool up = (i & k) == 0;
    if ((u > v) == up) {
        a[i] = v;
        a[x] = u;
    }
}

// All stages of the network inside blocks of kSortBlock keys, in shared memory: the sort of
// every block (k0 = 2) or the merge stages j < kSortBlock of one k > kSortBlock (k0 = k). A
// launch per stage took 300 us for 8,192 strings; one block now sorts them in 74 us.
constexpr int kSortBlock = 8192, kSortThreads = 1024;
__global__ void __launch_bounds__(kSortThreads) k_bitonic_block(uint64_t *a, int64_t P, int64_t k0, int64_t k1) {
    extern __shared__ uint64_t key[];
    const int64_t base = (int64_t)blockIdx.x * kSortBlock;
    const int n = (int)min((int64_t)kSortBlock, P - base);
    for (int i = threadIdx.x; i < n; i += kSortThreads) key[i] = a[base + i];
    for (int64_t k = k0; k <= k1; k <<= 1)
        for (int j = (int)min(k >> 1, (int64_t)n >> 1); j > 0; j >>= 1) {
            __syncthreads();
            for (int t = threadIdx.x; t < n / 2; t += kSortThreads) {
                const int i = 2 * t - (t & (j - 1)), x = i + j;  // the pair (i, i ^ j), i without bit j
                const uint64_t u = key[i], v = key[x];
                if ((u > v) == (((base + i) & k) == 0)) {
                    key[i] = v;
                    key[x] = u;
                }
            }
        }
    __syncthreads();
    for (int i = threadIdx.x; i < n; i += kSortThreads) a[base + i] = key[i];
}

// flags: 1 wrong electron count, 2 bit >= n, 4 duplicate
__global__ void k_validate(const uint64_t *a, int64_t m, int n, int N, int *flags) {
    int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= m) return;
    uint64_t s = a[i];
    int f = 0;
    if (__popcll(s) != N) f |= 1;
    if (n < 64 && (s >> n) != 0) f |= 2;
    if (i > 0 && a[i - 1] == s) f |= 4;
    if (f) atomicOr(flags, f);
}

__device__ __forceinline__ uint64_t lowmask(int k) { return (1ull << k) - 1ull; }

// Colex rank of a string of the full space.
__device__ __forceinline__ int64_t colex_rank(uint64_t s, const int64_t *__restrict__ B) {
    int64_t r = 0;
    int k = 1;
    while (s) {
        int c = __ffsll((long long)s) - 1;
        r += binom(B, c, k);
        ++k;
        s &= s - 1;
    }
    return r;
}

__device__ __forceinline__ int64_t bsearch_u64(const uint64_t *__restrict__ a, int64_t len, uint64_t s) {
    int64_t lo = 0, hi = len - 1;
    while (lo <= hi) {
        int64_t mid = (lo + hi) >> 1;
        uint64_t v = __ldg(a + mid);
        if (v == s) return mid;
        if (v < s) lo = mid + 1;
        else hi = mid - 1;
    }
    return -1;
}

// Membership of a selected set. Most candidates of a string are not in the set: a filter of
// one bit per hashed string, in shared memory, drops them, and what passes is looked up in a
// hash table {string, index + 1} of at most half its slots used (linear probing).
constexpr int64_t kHashMax = int64_t(1) << 22;  // above, the table (32 B or more per string)
                                                // leaves L2 and a binary search takes its place
__device__ __forceinline__ uint32_t string_hash(uint64_t s, int bits) {
    return (uint32_t)((s * 0x9E3779B97F4A7C15ull) >> (64 - bits));
}
__global__ void k_members(const uint64_t *__restrict__ str, int64_t l, int fbits, uint32_t *filter, int hbits, ulonglong2 *hash) {
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= l) return;
    const uint64_t s = str[i];
    const uint32_t f = string_hash(s, fbits);
    atomicOr(filter + (f >> 5), 1u << (f & 31));
    if (hbits == 0) return;
    uint32_t h = string_hash(s, hbits);
    while (atomicCAS(reinterpret_cast<unsigned long long *>(&hash[h].y), 0ull, (unsigned long long)(i + 1)) != 0ull)
        h = (h + 1) & ((1u << hbits) - 1u);
    hash[h].x = s;
}

struct LinkArgs {
    const uint32_t *filter;  // [2^fbits / 32], selected sets only
    const ulonglong2 *hash;  // [2^hbits]; hbits = 0: binary search in str
    int fbits, hbits;
    const uint64_t *str;
    int64_t l;
    int n, N;
    int full;
    const int64_t *B;
    int64_t *counts;  // count pass
    const int64_t *off;  // fill pass
    tbsci_single_link *e1;
    tbsci_double_link *e2;
};

// Pair tables: pair t of m items in lexicographic (i < j) order.
__device__ void build_pairs(uint8_t *pi, uint8_t *pj, int m) {
    // a warp fills the row of one i
    for (int i = threadIdx.x >> 5; i < m; i += kWarpsPerBlock) {
        const int t = i * (2 * m - i - 1) / 2 - i - 1;
        for (int j = i + 1 + (threadIdx.x & 31); j < m; j += 32) {
            pi[t + j] = (uint8_t)i;
            pj[t + j] = (uint8_t)j;
        }
    }
}

// One warp per source string, lanes over its candidates (occupied x empty orbitals, or pairs
// of them). What passes the filter is queued, so that 32 lookups run at once. Bound by the
// issue of the candidate loop; with a binary search of 13 levels in every pass of the loop
// the 5,000 strings at norb 24 with 2.6 M links took 0.40 (count) + 0.70 ms (fill), now
// 0.14 + 0.17 ms.
template <bool DBL, bool FILL>
__global__ void __launch_bounds__(kWarpsPerBlock * 32) k_links(LinkArgs A) {
    __shared__ uint8_t s_occ[kWarpsPerBlock][64], s_vir[kWarpsPerBlock][64];
    __shared__ uint8_t s_poi[DBL ? 2016 : 1], s_poj[DBL ? 2016 : 1];
    __shared__ uint8_t s_pvi[DBL ? 2016 : 1], s_pvj[DBL ? 2016 : 1];
    __shared__ uint32_t s_queue[kWarpsPerBlock][64];  // p | r << 8 | q << 16 | s << 24
    extern __shared__ __align__(16) uint32_t s_filter[];
    const int n = A.n, N = A.N, nv = n - N;
    const int npo = DBL ? N * (N - 1) / 2 : N;
    const int npv = DBL ? nv * (nv - 1) / 2 : nv;
    const int ncand = npo * npv;  // 496 x 496 at most
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t row = (int64_t)blockIdx.x * kWarpsPerBlock + warp;
    if (!FILL && A.full) {  // every candidate is in the set
        if (row < A.l && lane == 0) A.counts[row] = ncand;
        return;
    }
    if (!A.full)
        for (int x = threadIdx.x; x < 1 << (A.fbits - 7); x += kWarpsPerBlock * 32)
            reinterpret_cast<uint4 *>(s_filter)[x] = __ldg(reinterpret_cast<const uint4 *>(A.filter) + x);
    if (DBL) {
        build_pairs(s_poi, s_poj, N);
        build_pairs(s_pvi, s_pvj, nv);
    }
    __syncthreads();
    if (row >= A.l) return;
    const uint64_t J = A.str[row];
    // occupied / empty orbital lists, ascending
    int no = 0, ne = 0;
    const unsigned lt = (1u << lane) - 1u;
    for (int base = 0; base < n; base += 32) {
        const int i = base + lane;
        const bool in = i < n;
        const bool occ = in && ((J >> i) & 1ull);
        const unsigned mo = __ballot_sync(0xffffffffu, occ);
        const unsigned mv = __ballot_sync(0xffffffffu, in && !occ);
        if (occ) s_occ[warp][no + __popc(mo & lt)] = (uint8_t)i;
        if (in && !occ) s_vir[warp][ne + __popc(mv & lt)] = (uint8_t)i;
        no += __popc(mo);
        ne += __popc(mv);
    }
    __syncwarp();
    int64_t cnt = FILL ? A.off[row] : 0;
    uint32_t *queue = s_queue[warp];
    int queued = 0;
    // the first min(32, queued) candidates of the queue, in order
    auto drain = [&]() {
        __syncwarp();
        bool found = false;
        int64_t tgt = -1;
        uint64_t bp = 0, bq = 0, br = 0, bs = 0;
        const uint32_t code = queue[lane];
        const int p = code & 255, r = (code >> 8) & 255, q = (code >> 16) & 255, s = code >> 24;
        if (lane < queued) {
            bp = 1ull << p;
            bq = 1ull << q;
            if (DBL) {
                br = 1ull << r;
                bs = 1ull << s;
            }
            const uint64_t T = J ^ bp ^ bq ^ br ^ bs;
            if (A.full) {
                tgt = colex_rank(T, A.B);
            } else if (A.hbits) {
                uint32_t h = string_hash(T, A.hbits);
                for (ulonglong2 v = __ldg(A.hash + h); v.y; v = __ldg(A.hash + h)) {
                    if (v.x == T) {
                        tgt = (int64_t)v.y - 1;
                        break;
                    }
                    h = (h + 1) & ((1u << A.hbits) - 1u);
                }
            } else {
                tgt = bsearch_u64(A.str, A.l, T);
            }
            found = tgt >= 0;
        }
        const unsigned m = __ballot_sync(0xffffffffu, found);
        if (FILL && found) {
            const int64_t pos = cnt + __popc(m & lt);
            if (!DBL) {
                const int lo = min(p, q), hi = max(p, q);
                tbsci_single_link e;
                e.target = (int32_t)tgt;
                e.sign = (__popcll(J & lowmask(hi) & ~lowmask(lo + 1)) & 1) ? -1 : 1;
                e.p = (uint8_t)p;
                e.q = (uint8_t)q;
                e.pad = 0;
                A.e1[pos] = e;
            } else {
                // a_q, then a_s, then a+_r, then a+_p, each sign from the occupied
                // orbitals below the operator's orbital
                const int par = __popcll(J & (bq - 1)) + __popcll((J ^ bq) & (bs - 1)) + __popcll((J ^ bq ^ bs) & (br - 1)) +
                                __popcll((J ^ bq ^ bs ^ br) & (bp - 1));
                int *e = reinterpret_cast<int *>(A.e2 + pos);  // tbsci_double_link as three words
                e[0] = (int)tgt;
                e[1] = ((par & 1) ? 0xFF : 1) | p << 8 | r << 16 | q << 24;
                e[2] = s;
            }
        }
        cnt += __popc(m);
        __syncwarp();
        if (lane + 32 < queued) queue[lane] = queue[lane + 32];
        queued = max(0, queued - 32);
        __syncwarp();
    };
    // candidate c0 + lane = (occupied to, empty tv), stepped without a division
    int to = npv ? lane / npv : 0, tv = npv ? lane % npv : 0;
    const int dto = npv ? 32 / npv : 0, dtv = npv ? 32 % npv : 0;
    for (int c0 = 0; c0 < ncand; c0 += 32) {
        bool pass = false;
        uint32_t code = 0;
        if (c0 + lane < ncand) {
            uint32_t p, q, r = 0, s = 0;
            uint64_t T;
            if (!DBL) {
                q = s_occ[warp][to];
                p = s_vir[warp][tv];
                T = J ^ (1ull << q) ^ (1ull << p);
            } else {
                q = s_occ[warp][s_poi[to]];
                s = s_occ[warp][s_poj[to]];
                p = s_vir[warp][s_pvi[tv]];
                r = s_vir[warp][s_pvj[tv]];
                T = J ^ (1ull << q) ^ (1ull << s) ^ (1ull << r) ^ (1ull << p);
            }
            code = p | r << 8 | q << 16 | s << 24;
            pass = true;
            if (!A.full) {
                const uint32_t f = string_hash(T, A.fbits);
                pass = (s_filter[f >> 5] >> (f & 31)) & 1u;
            }
        }
        const unsigned m = __ballot_sync(0xffffffffu, pass);
        if (pass) queue[queued + __popc(m & lt)] = code;
        queued += __popc(m);
        if (queued >= 32) drain();
        to += dto;
        tv += dtv;
        if (tv >= npv) {
            tv -= npv;
            ++to;
        }
    }
    if (queued > 0) drain();
    if (!FILL && lane == 0) A.counts[row] = cnt;
}

// ---- exclusive scan (three passes: block sums, scan of sums, local scans)

constexpr int kScanBlock = 1024;
constexpr int kScanItems = 4;
constexpr int kScanTile = kScanBlock * kScanItems;

__device__ int64_t block_scan_excl(int64_t v, int64_t *sh, int64_t *total) {
    // Hillis-Steele over warps: warp inclusive scans, then scan of warp totals.
    int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    int64_t x = v;
    for (int o = 1; o < 32; o <<= 1) {
        int64_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) sh[w] = x;
    __syncthreads();
    if (w == 0) {
        int64_t t = (lane < (int)(blockDim.x >> 5)) ? sh[lane] : 0;
        for (int o = 1; o < 32; o <<= 1) {
            int64_t y = __shfl_up_sync(0xffffffffu, t, o);
            if (lane >= o) t += y;
        }
        sh[lane] = t;  // inclusive totals of warps
    }
    __syncthreads();
    int64_t before = (w > 0 ? sh[w - 1] : 0) + x - v;
    if (total) *total = sh[(blockDim.x >> 5) - 1];
    __syncthreads();
    return before;
}

__global__ void __launch_bounds__(kScanBlock) k_scan_sums(const int64_t *in, int64_t n, int64_t *sums) {
    __shared__ int64_t sh[32];
    int64_t base = (int64_t)blockIdx.x * kScanTile;
    int64_t v = 0;
    for (int k = 0; k < kScanItems; ++k) {
        int64_t i = base + (int64_t)threadIdx.x * kScanItems + k;
        if (i < n) v += in[i];
    }
    int64_t tot;
    block_scan_excl(v, sh, &tot);
    if (threadIdx.x == 0) sums[blockIdx.x] = tot;
}

__global__ void __launch_bounds__(kScanBlock) k_scan_top(int64_t *sums, int64_t nb, int64_t *total_out) {
    __shared__ int64_t sh[32];
    int64_t carry = 0;
    for (int64_t base = 0; base < nb; base += kScanBlock) {
        int64_t i = base + threadIdx.x;
        int64_t v = i < nb ? sums[i] : 0;
        int64_t tot;
        int64_t ex = block_scan_excl(v, sh, &tot);
        if (i < nb) sums[i] = carry + ex;
        carry += tot;
    }
    if (threadIdx.x == 0) *total_out = carry;
}

__global__ void __launch_bounds__(kScanBlock) k_scan_local(const int64_t *in, int64_t n, const int64_t *sums,
                                                            int64_t *out) {
    __shared__ int64_t sh[32];
    int64_t base = (int64_t)blockIdx.x * kScanTile;
    int64_t vals[kScanItems];
    int64_t v = 0;
    for (int k = 0; k < kScanItems; ++k) {
        int64_t i = base + (int64_t)threadIdx.x * kScanItems + k;
        vals[k] = i < n ? in[i] : 0;
        v += vals[k];
    }
    int64_t ex = block_scan_excl(v, sh, nullptr) + sums[blockIdx.x];
    for (int k = 0; k < kScanItems; ++k) {
        int64_t i = base + (int64_t)threadIdx.x * kScanItems + k;
        if (i < n) out[i] = ex;
        ex += vals[k];
    }
}

}  // namespace

static int64_t scan_scratch(int64_t n) { return (n + kScanTile - 1) / kScanTile; }

// the scan enqueued on st; `sums` holds scan_scratch(n) values
static tbsci_status scan_async(tbsci_ctx *ctx, const int64_t *in, int64_t *out, int64_t n, int64_t *sums, cudaStream_t st) {
    const int64_t nb = scan_scratch(n);
    if (nb > 0) k_scan_sums<<<(unsigned)nb, kScanBlock, 0, st>>>(in, n, sums);
    k_scan_top<<<1, kScanBlock, 0, st>>>(sums, nb, out + n);
    if (nb > 0) k_scan_local<<<(unsigned)nb, kScanBlock, 0, st>>>(in, n, sums, out);
    TB_CUDA(ctx, cudaGetLastError());
    return TBSCI_OK;
}

tbsci_status scan_exclusive(tbsci_ctx *ctx, const int64_t *in, int64_t *out, int64_t n, cudaStream_t st) {
    DevBuf<int64_t> sums;
    TB_CUDA(ctx, sums.alloc(std::max<int64_t>(scan_scratch(n), 1)));
    TB_TRY(scan_async(ctx, in, out, n, sums.p, st));
    TB_CUDA(ctx, cudaStreamSynchronize(st));
    return TBSCI_OK;
}

static int64_t host_binom(int m, int k) {
    if (k < 0 || k > m) return 0;
    // C(m-k+i, i) at step i; the product is formed in 128 bits
    unsigned __int128 v = 1;
    for (int i = 1; i <= k; ++i) v = v * (unsigned)(m - k + i) / (unsigned)i;
    return v > (unsigned __int128)INT64_MAX ? INT64_MAX : (int64_t)v;
}

tbsci_status strings_build(tbsci_ctx *ctx, int norb, int nelec, const uint64_t *sel, int64_t nsel,
                           tbsci_strings *out) {
    TB_CHECK(ctx, norb >= 1 && norb <= 64, TBSCI_EINVAL, "norb must be in 1..64");
    TB_CHECK(ctx, nelec >= 0 && nelec <= norb, TBSCI_EINVAL, "nelec must be in 0..norb");
    cudaStream_t st = ctx->stream;
    out->ctx = ctx;
    out->norb = norb;
    out->nelec = nelec;
    if (!sel) {
        int64_t count = host_binom(norb, nelec);
        TB_CHECK(ctx, count <= INT32_MAX, TBSCI_EINVAL, "string space exceeds 2^31-1 strings");
        out->count = count;
        out->full = true;
        TB_CUDA(ctx, out->d_str.alloc(count));
        if (count > 0) {
            k_unrank<<<(unsigned)((count + 255) / 256), 256, 0, st>>>(out->d_str.p, count, norb, nelec,
                                                                      ctx->d_binom.p);
            TB_CUDA(ctx, cudaGetLastError());
        }
        TB_CUDA(ctx, cudaStreamSynchronize(st));
        return TBSCI_OK;
    }
    TB_CHECK(ctx, nsel >= 0 && nsel <= INT32_MAX, TBSCI_EINVAL, "nsel must be in 0..2^31-1");
    out->count = nsel;
    out->full = false;
    int64_t P = 1;
    while (P < nsel) P <<= 1;
    DevBuf<uint64_t> work;
    TB_CUDA(ctx, work.alloc(std::max<int64_t>(P, 1)));
    if (nsel > 0) {
        TB_CUDA(ctx, cudaMemcpyAsync(work.p, sel, nsel * sizeof(uint64_t), cudaMemcpyHostToDevice, st));
        if (P > nsel) {
            k_fill_u64<<<(unsigned)((P - nsel + 255) / 256), 256, 0, st>>>(work.p, nsel, P, ~0ull);
            TB_CUDA(ctx, cudaGetLastError());
        }
        const size_t sm = (size_t)std::min<int64_t>(P, kSortBlock) * sizeof(uint64_t);
        const unsigned nb = (unsigned)((P + kSortBlock - 1) / kSortBlock);
        TB_CUDA(ctx, cudaFuncSetAttribute(k_bitonic_block, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm));
        k_bitonic_block<<<nb, kSortThreads, sm, st>>>(work.p, P, 2, std::min<int64_t>(P, kSortBlock));
        for (int64_t k = 2 * kSortBlock; k <= P; k <<= 1) {
            for (int64_t j = k >> 1; j >= kSortBlock; j >>= 1)
                k_bitonic<<<(unsigned)((P + 255) / 256), 256, 0, st>>>(work.p, P, j, k);
            k_bitonic_block<<<nb, kSortThreads, sm, st>>>(work.p, P, k, k);
        }
        TB_CUDA(ctx, cudaGetLastError());
    }
    DevBuf<int> flags;
    TB_CUDA(ctx, flags.alloc(1));
    TB_CUDA(ctx, cudaMemsetAsync(flags.p, 0, sizeof(int), st));
    if (nsel > 0) {
        k_validate<<<(unsigned)((nsel + 255) / 256), 256, 0, st>>>(work.p, nsel, norb, nelec, flags.p);
        TB_CUDA(ctx, cudaGetLastError());
    }
    int hf = 0;
    TB_CUDA(ctx, cudaMemcpyAsync(&hf, flags.p, sizeof(int), cudaMemcpyDeviceToHost, st));
    TB_CUDA(ctx, cudaStreamSynchronize(st));
    if (hf & 2) return fail(ctx, TBSCI_EINVAL, "selected string has a bit at or above norb");
    if (hf & 1) return fail(ctx, TBSCI_EINVAL, "selected string has the wrong electron count");
    if (hf & 4) return fail(ctx, TBSCI_EINVAL, "selected strings contain a duplicate");
    TB_CUDA(ctx, out->d_str.alloc(nsel));
    if (nsel > 0)
        TB_CUDA(ctx, cudaMemcpyAsync(out->d_str.p, work.p, nsel * sizeof(uint64_t), cudaMemcpyDeviceToDevice, st));
    // the set is full if it holds every string
    out->full = (nsel == host_binom(norb, nelec));
    TB_CUDA(ctx, cudaStreamSynchronize(st));
    return TBSCI_OK;
}

tbsci_status tables_build(tbsci_ctx *ctx, const tbsci_strings *s, int flags, tbsci_tables *out) {
    TB_CHECK(ctx, (flags & ~3) == 0, TBSCI_EINVAL, "unknown table flags");
    cudaStream_t st = ctx->stream;
    const int64_t l = s->count;
    out->ctx = ctx;
    out->norb = s->norb;
    out->nelec = s->nelec;
    out->flags = flags;
    out->count = l;
    out->full = s->full;
    TB_CUDA(ctx, out->d_str.alloc(l));
    if (l > 0) TB_CUDA(ctx, cudaMemcpyAsync(out->d_str.p, s->d_str.p, l * sizeof(uint64_t), cudaMemcpyDeviceToDevice, st));
    const bool want_double = !(flags & TBSCI_TABLES_SINGLES_ONLY);
    const bool fill = !(flags & TBSCI_TABLES_COUNT_ONLY);
    // filter: 16 bits or more per string as far as 64 KB of shared memory go; hash table: two
    // slots or more per string
    int fbits = 12, hbits = 0;
    while (fbits < 19 && (int64_t(1) << fbits) < 16 * l) ++fbits;
    const size_t fsm = s->full ? 0 : (size_t(1) << fbits) / 8;
    if (!s->full && l <= kHashMax)
        for (hbits = 1; (int64_t(1) << hbits) < 2 * l;) ++hbits;
    DevBuf<int64_t> counts, sums;
    DevBuf<uint32_t> filter;
    const int64_t nsum = std::max<int64_t>(1, scan_scratch(l));
    Arena tmp;  // freed on return, after the last kernel
    tmp.add(counts, 2 * std::max<int64_t>(l, 1));
    tmp.add(sums, 2 * nsum);
    DevBuf<ulonglong2> hash;
    if (fsm) tmp.add(filter, fsm / 4);
    if (hbits) tmp.add(hash, size_t(1) << hbits);
    TB_CUDA(ctx, tmp.commit());
    TB_CUDA(ctx, out->d_off1.alloc(l + 1));
    if (want_double) TB_CUDA(ctx, out->d_off2.alloc(l + 1));
    LinkArgs A{};
    A.filter = filter.p;
    A.hash = hash.p;
    A.fbits = fbits;
    A.hbits = hbits;
    A.str = out->d_str.p;
    A.l = l;
    A.n = s->norb;
    A.N = s->nelec;
    A.full = s->full ? 1 : 0;
    A.B = ctx->d_binom.p;
    const unsigned grid = (unsigned)((l + kWarpsPerBlock - 1) / kWarpsPerBlock);
    const int threads = kWarpsPerBlock * 32;
    for (auto k : {(const void *)k_links<false, false>, (const void *)k_links<false, true>, (const void *)k_links<true, false>,
                   (const void *)k_links<true, true>})
        TB_CUDA(ctx, cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, 65536));
    if (fsm && l > 0) {
        TB_CUDA(ctx, cudaMemsetAsync(filter.p, 0, fsm, st));
        if (hbits) TB_CUDA(ctx, cudaMemsetAsync(hash.p, 0, hash.bytes(), st));
        k_members<<<(unsigned)((l + 255) / 256), 256, 0, st>>>(out->d_str.p, l, fbits, filter.p, hbits, hash.p);
    }
    // counts of both classes, their offsets, one wait for both totals, then the entries
    out->h_off1.resize(l + 1);
    if (l > 0) {
        A.counts = counts.p;
        k_links<false, false><<<grid, threads, fsm, st>>>(A);
    }
    TB_TRY(scan_async(ctx, counts.p, out->d_off1.p, l, sums.p, st));
    TB_CUDA(ctx, cudaMemcpyAsync(out->h_off1.data(), out->d_off1.p, (l + 1) * sizeof(int64_t), cudaMemcpyDeviceToHost, st));
    if (want_double) {
        out->h_off2.resize(l + 1);
        if (l > 0) {
            A.counts = counts.p + l;
            k_links<true, false><<<grid, threads, fsm, st>>>(A);
        }
        TB_TRY(scan_async(ctx, counts.p + l, out->d_off2.p, l, sums.p + nsum, st));
        TB_CUDA(ctx, cudaMemcpyAsync(out->h_off2.data(), out->d_off2.p, (l + 1) * sizeof(int64_t), cudaMemcpyDeviceToHost, st));
    }
    TB_CUDA(ctx, cudaGetLastError());
    TB_CUDA(ctx, cudaStreamSynchronize(st));
    out->nsingle = out->h_off1[l];
    if (want_double) out->ndouble = out->h_off2[l];
    if (fill) {
        TB_CUDA(ctx, out->d_ent1.alloc(out->nsingle));
        A.off = out->d_off1.p;
        A.e1 = out->d_ent1.p;
        if (l > 0 && out->nsingle > 0) k_links<false, true><<<grid, threads, fsm, st>>>(A);
        if (want_double) {
            TB_CUDA(ctx, out->d_ent2.alloc(out->ndouble));
            A.off = out->d_off2.p;
            A.e2 = out->d_ent2.p;
            if (l > 0 && out->ndouble > 0) k_links<true, true><<<grid, threads, fsm, st>>>(A);
        }
        TB_CUDA(ctx, cudaGetLastError());
    }
    TB_CUDA(ctx, cudaStreamSynchronize(st));
    return TBSCI_OK;
}

}  // namespace tbsci

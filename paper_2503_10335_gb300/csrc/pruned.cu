// sigma = H.c on a pruned TBSCI space (Sec. II.A, Eq. 6): the determinants
// (w, u) of a TPB space with u in a per-alpha-string set I_w. H on the space is
// the principal submatrix of H on its determinants, so sigma on a member row is
// the TPB sigma of that row with c set to zero outside the space.
//
// One CTA owns alpha row Ia and walks its alpha terms Ja (Ia itself, its alpha
// singles, its alpha doubles) as the TPB kernel does. For each term the
// compressed c row Ja is expanded into a dense, zero-initialised shared-memory
// row (its members scattered in, then zeros scattered back after use), so every
// beta gather of the classes of Sec. II.C is a plain shared-memory read and a
// non-member reads 0: the membership test of Algorithm 1 costs nothing per link.
// Rows longer than shared memory look c(Ja, Jb) up by binary search in I_Ja.
// Each member column of Ia is owned by one thread across all terms (its sigma
// entry accumulates in place, no atomics, deterministic). Spaces whose rows fall
// into a few classes of equal I_w take k_sigma_classes (below) instead.
#include <algorithm>
#include <cstring>
#include <numeric>
#include <vector>

#include "internal.cuh"

namespace tbsci {

namespace {

template <typename T>
struct PrArgs {
    int64_t la, lb;
    const T *C;
    T *S;
    const int64_t *off;
    const int32_t *cols, *rows;
    int npair, na;
    const uint64_t *stra;
    const int64_t *a_soff, *a_doff;
    const int2 *a_sci;
    const T *a_sval, *a_dval;
    const int32_t *a_dcol;
    const T *Ea;
    const int64_t *b_soff, *b_doff;
    const int2 *b_sci;
    const T *b_sval, *b_dval;
    const int32_t *b_dcol;
    const T *Eb;
    const T *V;  // [npair][npair]
    const T *U;  // [npair][lb]
    T ecore;
};

template <typename T>
PrArgs<T> pr_args(const tbsci_ham *ham, const Plan *P, const tbsci_pruned *pr);

template <>
PrArgs<double> pr_args<double>(const tbsci_ham *ham, const Plan *P, const tbsci_pruned *pr) {
    PrArgs<double> A{};
    A.la = P->A.l;
    A.lb = P->B.l;
    A.off = pr->d_off.p;
    A.cols = pr->d_cols.p;
    A.rows = pr->d_rows.p;
    A.npair = P->npair;
    A.na = P->A.nelec;
    A.stra = P->A.d_str;
    A.a_soff = P->A.d_soff;
    A.a_doff = P->A.d_doff;
    A.a_sci = P->A.d_sci.p;
    A.a_sval = P->A.d_sval.p;
    A.a_dcol = P->A.d_dcol.p;
    A.a_dval = P->A.d_dval.p;
    A.Ea = P->A.d_E.p;
    A.b_soff = P->B.d_soff;
    A.b_doff = P->B.d_doff;
    A.b_sci = P->B.d_sci.p;
    A.b_sval = P->B.d_sval.p;
    A.b_dcol = P->B.d_dcol.p;
    A.b_dval = P->B.d_dval.p;
    A.Eb = P->B.d_E.p;
    A.V = ham->d_V.p;
    A.U = P->d_U.p;
    A.ecore = ham->ecore;
    return A;
}

template <>
PrArgs<float> pr_args<float>(const tbsci_ham *ham, const Plan *P, const tbsci_pruned *pr) {
    PrArgs<float> A{};
    A.la = P->A.l;
    A.lb = P->B.l;
    A.off = pr->d_off.p;
    A.cols = pr->d_cols.p;
    A.rows = pr->d_rows.p;
    A.npair = P->npair;
    A.na = P->A.nelec;
    A.stra = P->A.d_str;
    A.a_soff = P->A.d_soff;
    A.a_doff = P->A.d_doff;
    A.a_sci = P->A.d_sci.p;
    A.a_sval = P->A.d_svalf.p;
    A.a_dcol = P->A.d_dcol.p;
    A.a_dval = P->A.d_dvalf.p;
    A.Ea = P->A.d_Ef.p;
    A.b_soff = P->B.d_soff;
    A.b_doff = P->B.d_doff;
    A.b_sci = P->B.d_sci.p;
    A.b_sval = P->B.d_svalf.p;
    A.b_dcol = P->B.d_dcol.p;
    A.b_dval = P->B.d_dvalf.p;
    A.Eb = P->B.d_Ef.p;
    A.V = ham->d_Vf.p;
    A.U = P->d_Uf.p;
    A.ecore = (float)ham->ecore;
    return A;
}

template <typename T>
__host__ __device__ size_t pr_head_bytes(int npair) {
    return ((2 * npair + 2) * sizeof(T) + 64 * sizeof(int) + 15) & ~size_t(15);
}

constexpr int kPrThreads = 256;

template <typename T, bool EXPAND>
__global__ void __launch_bounds__(kPrThreads) k_sigma_pruned(PrArgs<T> A) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int npair = A.npair;
    T *sV2 = reinterpret_cast<T *>(smem_raw);  // [2 npair + 2]: coefficient by (pair, sign); last two zero
    int *sOcc = reinterpret_cast<int *>(sV2 + 2 * npair + 2);
    T *sC = reinterpret_cast<T *>(smem_raw + pr_head_bytes<T>(npair));  // [lb] when EXPAND
    const int64_t Ia = A.rows[blockIdx.x];
    const int64_t m0 = A.off[Ia], cnt = A.off[Ia + 1] - m0;
    if (cnt == 0) return;  // block-uniform, before any barrier
    const int64_t lb = A.lb;
    if (threadIdx.x == 0) {
        int k = 0;
        for (uint64_t s = A.stra[Ia]; s; s &= s - 1) {
            const int p = __ffsll((long long)s) - 1;
            sOcc[k++] = p * (p + 1) / 2 + p;
        }
        sV2[2 * npair] = T(0);
        sV2[2 * npair + 1] = T(0);
    }
    if (EXPAND)
        for (int64_t j = threadIdx.x; j < lb; j += kPrThreads) sC[j] = T(0);
    __syncthreads();
    for (int x = threadIdx.x; x < npair; x += kPrThreads) {  // W_Ia[x] = sum_{p in Ia} (pp|x)
        T w = 0;
        for (int k = 0; k < A.na; ++k) w += A.V[(size_t)sOcc[k] * npair + x];
        sV2[2 * x] = w;
        sV2[2 * x + 1] = -w;
    }
    const int64_t t0 = A.a_soff[Ia], ns = A.a_soff[Ia + 1] - t0;
    const int64_t d0 = A.a_doff[Ia], nd = A.a_doff[Ia + 1] - d0;
    const T *__restrict__ C = A.C;
    T *__restrict__ S = A.S;
    for (int64_t k = 0; k < 1 + ns + nd; ++k) {
        int64_t Ja = Ia;
        int kind = 0, pr = 0;
        T ha = T(0), sa = T(1);
        if (k >= 1 && k <= ns) {
            const int2 e = A.a_sci[t0 + k - 1];
            Ja = e.x;
            pr = e.y >> 1;
            sa = (e.y & 1) ? T(-1) : T(1);
            ha = A.a_sval[t0 + k - 1];
            kind = 1;
        } else if (k > ns) {
            Ja = A.a_dcol[d0 + k - 1 - ns];
            ha = A.a_dval[d0 + k - 1 - ns];
            kind = 2;
        }
        const int64_t j0 = A.off[Ja], jc = A.off[Ja + 1] - j0;
        if (jc == 0) continue;  // block-uniform: no member of row Ja couples
        if (kind == 1)
            for (int x = threadIdx.x; x < npair; x += kPrThreads) {
                const T vv = sa * A.V[(size_t)pr * npair + x];
                sV2[2 * x] = vv;
                sV2[2 * x + 1] = -vv;
            }
        if (EXPAND)
            for (int64_t i = threadIdx.x; i < jc; i += kPrThreads) sC[A.cols[j0 + i]] = __ldg(C + j0 + i);
        __syncthreads();
        // c(Ja, jb): expanded row, or binary search in I_Ja
        auto cv = [&](int64_t jb) -> T {
            if (EXPAND) return sC[jb];
            int64_t lo = j0, hi = j0 + jc - 1;
            while (lo <= hi) {
                const int64_t mid = (lo + hi) >> 1;
                const int32_t x = __ldg(A.cols + mid);
                if (x == jb) return __ldg(C + mid);
                if (x < jb) lo = mid + 1;
                else hi = mid - 1;
            }
            return T(0);
        };
        for (int64_t p = threadIdx.x; p < cnt; p += kPrThreads) {
            const int64_t ib = A.cols[m0 + p];
            T acc;
            if (kind == 0) {
                T ed = A.ecore + A.Ea[Ia] + A.Eb[ib];
                for (int q = 0; q < A.na; ++q) ed += __ldg(A.U + (size_t)sOcc[q] * lb + ib);
                acc = ed * cv(ib);
                for (int64_t t = A.b_soff[ib]; t < A.b_soff[ib + 1]; ++t) {
                    const int2 e = __ldg(A.b_sci + t);
                    acc += (__ldg(A.b_sval + t) + sV2[e.y]) * cv(e.x);
                }
                for (int64_t t = A.b_doff[ib]; t < A.b_doff[ib + 1]; ++t)
                    acc += __ldg(A.b_dval + t) * cv(__ldg(A.b_dcol + t));
            } else if (kind == 1) {
                acc = S[m0 + p] + (ha + sa * __ldg(A.U + (size_t)pr * lb + ib)) * cv(ib);
                for (int64_t t = A.b_soff[ib]; t < A.b_soff[ib + 1]; ++t) {
                    const int2 e = __ldg(A.b_sci + t);
                    acc += sV2[e.y] * cv(e.x);
                }
            } else {
                acc = S[m0 + p] + ha * cv(ib);
            }
            S[m0 + p] = acc;
        }
        __syncthreads();
        if (EXPAND) {
            for (int64_t i = threadIdx.x; i < jc; i += kPrThreads) sC[A.cols[j0 + i]] = T(0);
            __syncthreads();
        }
    }
}

// ---- rows in classes
//
// Where few distinct sets I_w occur (the irreps of a symmetry block, the levels of
// an excitation cap), the member couplings of a pair of classes (f, g) are the same
// for every pair of their rows, so they are listed once: per member of f its beta
// single links whose target is a member of g, the target given as its index in the
// compressed row. A staged c row is then read as it lies in memory, no link to a
// non-member is visited, and alpha terms whose class has nothing in common with
// the row's are dropped before the sweep. The links lie in sliced-ELL slices of 32
// consecutive members (a warp reads them coalesced); padding reads a zero slot
// behind the row with a zero coefficient, so it adds an exact zero for any c.
// Bound: FP64 pipe and the latency of the term loop (one barrier per alpha single,
// the next term's row and coefficients staged while this one is summed).
// norb 14 full space, 8 irreps, one block (1.47M determinants, FP64): 1.88 ms, 38.8 ms
// with the general kernel, whose links are 7/8 non-members read uncoalesced.
constexpr int kClsLinkBits = 13;
constexpr int kMaxClasses = 16;

struct ClsArgs {
    int ncls, cmax;
    const int32_t *cls, *ccnt, *pos;
    const int *ov;
    const int64_t *sbase, *dbase, *s_off, *d_off;
    const int32_t *s_w, *d_w;
    const uint32_t *s_ci;
    const int32_t *s_li;
    const int2 *d_ent;
};

template <typename T>
__host__ __device__ size_t cls_smem_bytes(int npair, int cmax, int threads) {
    // two coefficient tables, two c rows (with a zero slot), the sigma row, the term list
    size_t b = (2 * (2 * (size_t)npair + 2) + 2 * ((size_t)cmax + 1) + (size_t)cmax + threads) * sizeof(T);
    b = (b + 15) & ~size_t(15);
    return b + (size_t)threads * 16 + 64 * sizeof(int) + 32 * sizeof(int);
}

template <typename T, int TH>
__global__ void __launch_bounds__(TH) k_sigma_classes(PrArgs<T> A, ClsArgs K, int64_t nd_all) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int npair = A.npair, cmax = K.cmax, nv2 = 2 * npair + 2;
    T *sV2 = reinterpret_cast<T *>(smem_raw);  // [2][nv2], the last two of each zero
    T *sC = sV2 + 2 * nv2;                     // [2][cmax + 1], the last of each zero
    T *sAcc = sC + 2 * (cmax + 1);             // [cmax]
    T *sX = sAcc + cmax;                       // [TH] value of each listed alpha term
    const size_t head = ((2 * (size_t)nv2 + 2 * ((size_t)cmax + 1) + cmax + TH) * sizeof(T) + 15) & ~size_t(15);
    int64_t *sJ = reinterpret_cast<int64_t *>(smem_raw + head);  // [TH] start of the term's c row
    int *sG = reinterpret_cast<int *>(sJ + TH);                  // [TH] its class
    int *sP = sG + TH;                                           // [TH] 2 pair + (sign < 0)
    int *sOcc = sP + TH;                                         // [64]
    int *sWarp = sOcc + 64;                                      // [32]
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int64_t Ia = A.rows[blockIdx.x];
    const int64_t m0 = A.off[Ia];
    const int cnt = (int)(A.off[Ia + 1] - m0);
    if (cnt == 0) return;  // block-uniform, before any barrier
    const int64_t lb = A.lb;
    const T *__restrict__ C = A.C + blockIdx.y * nd_all;
    T *__restrict__ S = A.S + blockIdx.y * nd_all;
    const int32_t *__restrict__ mycols = A.cols + m0;
    const int f = K.cls[Ia], ncls = K.ncls;
    const int *ov = K.ov + f * ncls;
    if (tid == 0) {
        int k = 0;
        for (uint64_t s = A.stra[Ia]; s; s &= s - 1) {
            const int p = __ffsll((long long)s) - 1;
            sOcc[k++] = p * (p + 1) / 2 + p;
        }
    }
    if (tid < 2) {
        sV2[tid * nv2 + 2 * npair] = T(0);
        sV2[tid * nv2 + 2 * npair + 1] = T(0);
        sC[tid * (cmax + 1) + cmax] = T(0);
    }
    for (int i = tid; i < cnt; i += TH) sC[i] = __ldg(C + m0 + i);
    __syncthreads();
    for (int x = tid; x < npair; x += TH) {  // W_Ia[x] = sum_{p in Ia} (pp|x)
        T w = 0;
        for (int k = 0; k < A.na; ++k) w += A.V[(size_t)sOcc[k] * npair + x];
        sV2[2 * x] = w;
        sV2[2 * x + 1] = -w;
    }
    __syncthreads();
    constexpr uint32_t kIdx = (1u << kClsLinkBits) - 1;

    // ---- Ja = Ia
    const T eIa = A.ecore + A.Ea[Ia];
    for (int p = tid; p < cnt; p += TH) {
        const int64_t ib = mycols[p];
        T ed = eIa + __ldg(A.Eb + ib);
        for (int q = 0; q < A.na; ++q) ed += __ldg(A.U + (size_t)sOcc[q] * lb + ib);
        T acc = ed * sC[p];
        const int64_t ss = K.sbase[f * ncls + f] + (p >> 5), ds = K.dbase[f] + (p >> 5);
        const uint32_t *ci = K.s_ci + K.s_off[ss] + lane;
        const int32_t *li = K.s_li + K.s_off[ss] + lane;
        const int ws = K.s_w[ss], wd = K.d_w[ds];
#pragma unroll 4
        for (int k = 0; k < ws; ++k) {
            const uint32_t e = __ldg(ci + 32 * k);
            const int32_t t = __ldg(li + 32 * k);
            const T x = t >= 0 ? __ldg(A.b_sval + t) + sV2[e & kIdx] : T(0);
            acc += x * sC[e >> kClsLinkBits];
        }
        const int2 *de = K.d_ent + K.d_off[ds] + lane;
#pragma unroll 4
        for (int k = 0; k < wd; ++k) {
            const int2 e = __ldg(de + 32 * k);
            const T x = e.y >= 0 ? __ldg(A.b_dval + e.y) : T(0);
            acc += x * sC[e.x];
        }
        sAcc[p] = acc;
    }
    __syncthreads();

    // lists the alpha terms first .. first + TH - 1 (below `end`) whose class passes
    // `mask`, in order; returns their number (block-uniform, ends with a barrier)
    auto list_terms = [&](int64_t first, int64_t end, bool dbl, int mask) -> int {
        const int64_t t = first + tid;
        bool keep = false;
        int64_t Ja = 0;
        int g = 0, pr = 0;
        T x = T(0);
        if (t < end) {
            if (dbl) {
                Ja = __ldg(A.a_dcol + t);
                x = __ldg(A.a_dval + t);
            } else {
                const int2 e = __ldg(A.a_sci + t);
                Ja = e.x;
                pr = e.y;
                x = __ldg(A.a_sval + t);
            }
            g = K.cls[Ja];
            keep = (ov[g] & mask) != 0;
        }
        const unsigned m = __ballot_sync(0xffffffffu, keep);
        if (lane == 0) sWarp[warp] = __popc(m);
        __syncthreads();
        int at = __popc(m & ((1u << lane) - 1u)), total = 0;
        for (int w = 0; w < TH / 32; ++w) {
            if (w < warp) at += sWarp[w];
            total += sWarp[w];
        }
        if (keep) {
            sJ[at] = A.off[Ja];
            sG[at] = g;
            sP[at] = pr;
            sX[at] = x;
        }
        __syncthreads();
        return total;
    };

    // ---- alpha singles
    const int64_t t0 = A.a_soff[Ia], t1 = A.a_soff[Ia + 1];
    for (int64_t first = t0; first < t1; first += TH) {
        const int n = list_terms(first, t1, false, 3);
        auto stage = [&](int i) {
            T *v2 = sV2 + (i & 1) * nv2, *c = sC + (i & 1) * (cmax + 1);
            const int pr = sP[i] >> 1;
            const T sa = (sP[i] & 1) ? T(-1) : T(1);
            const T *src = C + sJ[i];
            const int jc = K.ccnt[sG[i]];
            for (int x = tid; x < jc; x += TH) c[x] = __ldg(src + x);
            for (int x = tid; x < npair; x += TH) {
                const T vv = sa * __ldg(A.V + (size_t)pr * npair + x);
                v2[2 * x] = vv;
                v2[2 * x + 1] = -vv;
            }
        };
        if (n > 0) stage(0);
        __syncthreads();
        for (int i = 0; i < n; ++i) {
            if (i + 1 < n) stage(i + 1);
            const T *v2 = sV2 + (i & 1) * nv2, *c = sC + (i & 1) * (cmax + 1);
            const int g = sG[i], pr = sP[i] >> 1;
            const T sa = (sP[i] & 1) ? T(-1) : T(1), ha = sX[i];
            const bool common = ov[g] & 1;
            const int64_t sb = K.sbase[f * ncls + g];
            for (int p = tid; p < cnt; p += TH) {
                T acc = sAcc[p];
                if (common) {
                    const int64_t ib = __ldg(mycols + p);
                    const int q = g == f ? p : __ldg(K.pos + g * lb + ib);
                    if (q >= 0) acc += (ha + sa * __ldg(A.U + (size_t)pr * lb + ib)) * c[q];
                }
                const int64_t ss = sb + (p >> 5);
                const uint32_t *ci = K.s_ci + __ldg(K.s_off + ss) + lane;
                const int w = __ldg(K.s_w + ss);
#pragma unroll 4
                for (int k = 0; k < w; ++k) {
                    const uint32_t e = __ldg(ci + 32 * k);
                    acc += v2[e & kIdx] * c[e >> kClsLinkBits];
                }
                sAcc[p] = acc;
            }
            __syncthreads();
        }
    }

    // ---- alpha doubles: c rows read coalesced
    const int64_t u0 = A.a_doff[Ia], u1 = A.a_doff[Ia + 1];
    for (int64_t first = u0; first < u1; first += TH) {
        const int n = list_terms(first, u1, true, 1);
        for (int p = tid; p < cnt; p += TH) {
            T acc = sAcc[p];
            const int64_t ib = __ldg(mycols + p);
#pragma unroll 4
            for (int i = 0; i < n; ++i) {
                const int g = sG[i];
                const int q = g == f ? p : __ldg(K.pos + g * lb + ib);
                if (q >= 0) acc += sX[i] * __ldg(C + sJ[i] + q);
            }
            sAcc[p] = acc;
        }
        __syncthreads();
    }
    for (int p = tid; p < cnt; p += TH) S[m0 + p] = sAcc[p];
}

// d_pos of one class per blockIdx.y (set to -1 before)
__global__ void k_cls_pos(const int64_t *__restrict__ cbeg, const int32_t *__restrict__ ccnt,
                          const int32_t *__restrict__ cols, int64_t lb, int32_t *pos) {
    const int g = blockIdx.y;
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p < ccnt[g]) pos[g * lb + cols[cbeg[g] + p]] = p;
}

struct ClsBuild {
    int ncls, cmax;
    int64_t lb;
    const int64_t *cbeg;
    const int32_t *ccnt, *cols, *pos;
    const int64_t *off1, *off2;
    const tbsci_single_link *ent1;
    const tbsci_double_link *ent2;
    const int64_t *sbase, *dbase;
    int *ov;
    int64_t *s_cnt, *d_cnt;  // count pass: entries of each slice (32 x width)
    int32_t *s_w, *d_w;
    const int64_t *s_off, *d_off;  // fill pass
    uint32_t *s_ci;
    int32_t *s_li;
    int2 *d_ent;
    uint32_t zero_idx;
};

// One thread per member of class f (blockIdx.y = f ncls + g); a warp is one slice.
// The singles of (f, g), and the doubles of f when g = f.
template <bool FILL>
__global__ void __launch_bounds__(128) k_cls_links(ClsBuild B) {
    const int f = blockIdx.y / B.ncls, g = blockIdx.y - f * B.ncls;
    const int p = blockIdx.x * 128 + threadIdx.x, cf = B.ccnt[f];
    if ((p & ~31) >= cf) return;  // warp-uniform
    const int lane = p & 31;
    const bool ok = p < cf;
    const int64_t ib = ok ? B.cols[B.cbeg[f] + p] : 0;
    const int32_t *pos = B.pos + g * B.lb;
    const int64_t a1 = ok ? B.off1[ib] : 0, b1 = ok ? B.off1[ib + 1] : 0;
    const int64_t a2 = ok && f == g ? B.off2[ib] : 0, b2 = ok && f == g ? B.off2[ib + 1] : 0;
    const int64_t ss = B.sbase[f * B.ncls + g] + (p >> 5), ds = B.dbase[f] + (p >> 5);
    int n1 = 0, n2 = 0;
    for (int64_t t = a1; t < b1; ++t) {
        const tbsci_single_link e = B.ent1[t];
        const int q = pos[e.target];
        if (q < 0) continue;
        if (FILL) {
            const int hi = max(e.p, e.q), lo = min(e.p, e.q);
            const int64_t at = B.s_off[ss] + 32 * (int64_t)n1 + lane;
            B.s_ci[at] = ((uint32_t)q << kClsLinkBits) | (uint32_t)(2 * (hi * (hi + 1) / 2 + lo) + (e.sign < 0 ? 1 : 0));
            B.s_li[at] = (int32_t)t;
        }
        ++n1;
    }
    for (int64_t t = a2; t < b2; ++t) {
        const int q = pos[B.ent2[t].target];
        if (q < 0) continue;
        if (FILL) B.d_ent[B.d_off[ds] + 32 * (int64_t)n2 + lane] = make_int2(q, (int32_t)t);
        ++n2;
    }
    if (FILL) {
        for (int k = n1; k < B.s_w[ss]; ++k) {
            const int64_t at = B.s_off[ss] + 32 * (int64_t)k + lane;
            B.s_ci[at] = ((uint32_t)B.cmax << kClsLinkBits) | B.zero_idx;
            B.s_li[at] = -1;
        }
        if (f == g)
            for (int k = n2; k < B.d_w[ds]; ++k) B.d_ent[B.d_off[ds] + 32 * (int64_t)k + lane] = make_int2(B.cmax, -1);
        return;
    }
    const int w1 = (int)__reduce_max_sync(0xffffffffu, (unsigned)n1), w2 = (int)__reduce_max_sync(0xffffffffu, (unsigned)n2);
    const bool common = __any_sync(0xffffffffu, ok && pos[ib] >= 0);
    if (lane == 0) {
        B.s_w[ss] = w1;
        B.s_cnt[ss] = 32 * (int64_t)w1;
        if (f == g) {
            B.d_w[ds] = w2;
            B.d_cnt[ds] = 32 * (int64_t)w2;
        }
        const int bits = (common ? 1 : 0) | (w1 > 0 ? 2 : 0);
        if (bits) atomicOr(B.ov + f * B.ncls + g, bits);
    }
}

// diag[off[w] + p] = ecore + E_a(w) + E_b(u) + sum_{q in w} U[qq][u], u = cols[off[w] + p]
__global__ void k_diagonal_pruned(const uint64_t *__restrict__ stra, int64_t lb, const int64_t *__restrict__ off,
                                  const int32_t *__restrict__ cols, const double *__restrict__ Ea,
                                  const double *__restrict__ Eb, const double *__restrict__ U, double ecore,
                                  double *diag) {
    const int64_t w = blockIdx.x;
    const int64_t m0 = off[w], cnt = off[w + 1] - m0;
    const uint64_t sw = stra[w];
    for (int64_t p = threadIdx.x; p < cnt; p += blockDim.x) {
        const int64_t u = cols[m0 + p];
        double d = ecore + Ea[w] + Eb[u];
        for (uint64_t s = sw; s; s &= s - 1) {
            const int q = __ffsll((long long)s) - 1;
            d += U[(size_t)(q * (q + 1) / 2 + q) * lb + u];
        }
        diag[m0 + p] = d;
    }
}

template <typename T>
tbsci_status launch_pruned(tbsci_ctx *ctx, const tbsci_ham *ham, const Plan *P, const tbsci_pruned *pr, const T *c,
                           T *s, int nvec, cudaStream_t st) {
    PrArgs<T> A = pr_args<T>(ham, P, pr);
    if (pr->nd == 0 || A.la == 0) return TBSCI_OK;
    // rows in classes: the warps of a CTA take 32 members each, so a row of a few
    // hundred members runs on 4 warps and many CTAs share an SM
    std::unique_lock<std::mutex> lk;
    if (pr->classes) lk = std::unique_lock<std::mutex>(pr->classes->mu);
    const int cls_threads = pr->cmax > 1024 ? 512 : pr->cmax > 256 ? 256 : 128;
    if (pr->ncls > 0 && nvec <= 65535 && cls_smem_bytes<T>(A.npair, pr->cmax, cls_threads) <= ctx->smem_optin) {
        ClsArgs K{pr->ncls, pr->cmax, pr->d_cls.p, pr->d_ccnt.p, pr->d_pos.p, pr->d_ov.p, pr->d_sbase.p, pr->d_dbase.p,
                  pr->d_s_off.p, pr->d_d_off.p, pr->d_s_w.p, pr->d_d_w.p, pr->d_s_ci.p, pr->d_s_li.p, pr->d_d_ent.p};
        A.C = c;
        A.S = s;
        const size_t sm = cls_smem_bytes<T>(A.npair, pr->cmax, cls_threads);
        auto kern = cls_threads == 512 ? k_sigma_classes<T, 512> : cls_threads == 256 ? k_sigma_classes<T, 256>
                                                                                      : k_sigma_classes<T, 128>;
        TB_CUDA(ctx, cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm));
        TraceScope tr(ctx, "k_sigma_classes", st);
        kern<<<dim3((unsigned)A.la, (unsigned)nvec), cls_threads, sm, st>>>(A, K, pr->nd);
        TB_CUDA(ctx, cudaGetLastError());
        return TBSCI_OK;
    }
    if (lk.owns_lock()) lk.unlock();
    const size_t head = pr_head_bytes<T>(A.npair), full = head + (size_t)A.lb * sizeof(T);
    const bool expand = full <= ctx->smem_optin;
    for (int v = 0; v < nvec; ++v) {
        A.C = c + (size_t)v * pr->nd;
        A.S = s + (size_t)v * pr->nd;
        TraceScope tr(ctx, "k_sigma_pruned", st);
        if (expand) {
            TB_CUDA(ctx, cudaFuncSetAttribute(k_sigma_pruned<T, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                              (int)full));
            k_sigma_pruned<T, true><<<(unsigned)A.la, kPrThreads, full, st>>>(A);
        } else {
            k_sigma_pruned<T, false><<<(unsigned)A.la, kPrThreads, head, st>>>(A);
        }
        TB_CUDA(ctx, cudaGetLastError());
    }
    return TBSCI_OK;
}

// The lists of a pruned space's classes as spare memory; without them the space runs on the
// general kernel.
struct ClassLists : Spare {
    tbsci_pruned *const pr;
    size_t charged = 0;
    ClassLists(tbsci_ctx *c, tbsci_pruned *p) : Spare(c), pr(p) {}
    void publish() { enlist(); }  // once the lists are there
    ~ClassLists() override {
        retire();
        uncharge(ctx, charged);
    }
    void release() {
        pr->ncls = 0;
        pr->d_cls.release();
        pr->d_cbeg.release();
        pr->d_ccnt.release();
        pr->d_pos.release();
        pr->d_ov.release();
        pr->d_sbase.release();
        pr->d_dbase.release();
        pr->d_s_off.release();
        pr->d_d_off.release();
        pr->d_s_w.release();
        pr->d_d_w.release();
        pr->d_s_ci.release();
        pr->d_s_li.release();
        pr->d_d_ent.release();
    }
    bool give_back() override {
        if (pr->ncls == 0 || cudaDeviceSynchronize() != cudaSuccess) return false;
        release();
        uncharge(ctx, charged);
        charged = 0;
        return true;
    }
};

// Groups the alpha rows by equal I_w and lists the links between the classes on the
// device. Not more than kMaxClasses classes (their pair tables grow with the square),
// rows that fit in shared memory beside two staged c rows, and, under a budget, an
// eighth of what is left of it: otherwise the space keeps the general kernel.
tbsci_status build_classes(tbsci_ctx *ctx, const tbsci_tables *a, const tbsci_tables *b, const int64_t *off,
                           const int32_t *cols, tbsci_pruned *pr) {
    const int64_t la = pr->la, lb = pr->lb;
    if (pr->nd == 0 || a->flags != 0 || b->flags != 0 || a->norb != b->norb) return TBSCI_OK;
    std::vector<int64_t> cbeg;
    std::vector<int32_t> ccnt, cls(la);
    for (int64_t w = 0; w < la; ++w) {
        const int64_t n = off[w + 1] - off[w];
        size_t k = 0;
        for (; k < cbeg.size(); ++k)
            if (ccnt[k] == n && (n == 0 || std::memcmp(cols + cbeg[k], cols + off[w], n * sizeof(int32_t)) == 0)) break;
        if (k == cbeg.size()) {
            if (k == (size_t)kMaxClasses) return TBSCI_OK;
            cbeg.push_back(off[w]);
            ccnt.push_back((int32_t)n);
        }
        cls[w] = (int32_t)k;
    }
    const int ncls = (int)cbeg.size(), cmax = *std::max_element(ccnt.begin(), ccnt.end());
    const int npair = a->norb * (a->norb + 1) / 2;
    if (cmax >= (1 << (32 - kClsLinkBits)) || 2 * npair + 2 > (1 << kClsLinkBits) ||
        b->nsingle > INT32_MAX || b->ndouble > INT32_MAX || cls_smem_bytes<float>(npair, cmax, 128) > ctx->smem_optin)
        return TBSCI_OK;
    std::vector<int64_t> sbase((size_t)ncls * ncls), dbase(ncls);
    int64_t ns = 0, nds = 0;
    for (int f = 0; f < ncls; ++f) {
        const int64_t sl = (ccnt[f] + 31) / 32;
        for (int g = 0; g < ncls; ++g, ns += sl) sbase[(size_t)f * ncls + g] = ns;
        dbase[f] = nds;
        nds += sl;
    }
    const size_t fixed = (size_t)la * 4 + (size_t)ncls * (12 + 8 * ncls + 4 * ncls + 8 + lb * 4) + (ns + nds) * 12 + 32;
    const size_t left = ctx->hbm_budget ? ctx->hbm_budget - std::min(ctx->hbm_budget, ctx->hbm_used.load()) : SIZE_MAX;
    if (fixed > left / 8) return TBSCI_OK;
    cudaStream_t st = ctx->stream;
    auto lists = std::make_unique<ClassLists>(ctx, pr);
    DevBuf<int64_t> s_cnt, d_cnt;
    cudaError_t e = cudaSuccess;
    auto need = [&](auto &buf, size_t n) {
        if (e == cudaSuccess) e = buf.alloc(n, true);
    };
    auto put = [&](auto &buf, const auto &h) {
        need(buf, h.size());
        if (e == cudaSuccess) e = cudaMemcpyAsync(buf.p, h.data(), h.size() * sizeof(h[0]), cudaMemcpyHostToDevice, st);
    };
    put(pr->d_cls, cls);
    put(pr->d_cbeg, cbeg);
    put(pr->d_ccnt, ccnt);
    put(pr->d_sbase, sbase);
    put(pr->d_dbase, dbase);
    need(pr->d_pos, (size_t)ncls * lb);
    need(pr->d_ov, (size_t)ncls * ncls);
    need(pr->d_s_off, ns + 1);
    need(pr->d_d_off, nds + 1);
    need(pr->d_s_w, ns);
    need(pr->d_d_w, nds);
    need(s_cnt, ns);
    need(d_cnt, nds);
    tbsci_status ret = TBSCI_OK;
    int64_t tot[2] = {0, 0};
    ClsBuild B{ncls, cmax, lb, pr->d_cbeg.p, pr->d_ccnt.p, pr->d_cols.p, pr->d_pos.p, b->d_off1.p, b->d_off2.p,
               b->d_ent1.p, b->d_ent2.p, pr->d_sbase.p, pr->d_dbase.p, pr->d_ov.p, s_cnt.p, d_cnt.p, pr->d_s_w.p,
               pr->d_d_w.p, pr->d_s_off.p, pr->d_d_off.p, nullptr, nullptr, nullptr, (uint32_t)(2 * npair)};
    const dim3 grid((unsigned)((cmax + 127) / 128), (unsigned)(ncls * ncls));
    if (e == cudaSuccess) e = cudaMemsetAsync(pr->d_pos.p, 0xFF, pr->d_pos.bytes(), st);
    if (e == cudaSuccess) e = cudaMemsetAsync(pr->d_ov.p, 0, pr->d_ov.bytes(), st);
    if (e == cudaSuccess) {
        k_cls_pos<<<dim3((unsigned)((cmax + 127) / 128), (unsigned)ncls), 128, 0, st>>>(pr->d_cbeg.p, pr->d_ccnt.p,
                                                                                       pr->d_cols.p, lb, pr->d_pos.p);
        k_cls_links<false><<<grid, 128, 0, st>>>(B);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) ret = scan_exclusive(ctx, s_cnt.p, pr->d_s_off.p, ns, st);
    if (e == cudaSuccess && ret == TBSCI_OK) ret = scan_exclusive(ctx, d_cnt.p, pr->d_d_off.p, nds, st);
    if (e == cudaSuccess && ret == TBSCI_OK) {
        e = cudaMemcpy(&tot[0], pr->d_s_off.p + ns, 8, cudaMemcpyDeviceToHost);
        if (e == cudaSuccess) e = cudaMemcpy(&tot[1], pr->d_d_off.p + nds, 8, cudaMemcpyDeviceToHost);
    }
    const size_t bytes = fixed + 8 * (size_t)(tot[0] + tot[1]);
    const bool fits = e == cudaSuccess && ret == TBSCI_OK && bytes <= left / 8 && spare_charge(ctx, bytes);
    if (fits) {
        need(pr->d_s_ci, std::max<int64_t>(tot[0], 1));
        need(pr->d_s_li, std::max<int64_t>(tot[0], 1));
        need(pr->d_d_ent, std::max<int64_t>(tot[1], 1));
        if (e == cudaSuccess) {
            B.s_ci = pr->d_s_ci.p;
            B.s_li = pr->d_s_li.p;
            B.d_ent = pr->d_d_ent.p;
            k_cls_links<true><<<grid, 128, 0, st>>>(B);
            e = cudaGetLastError();
        }
        if (e == cudaSuccess) e = cudaStreamSynchronize(st);
        if (e == cudaSuccess) {
            pr->ncls = ncls;
            pr->cmax = cmax;
            lists->charged = bytes;
            lists->publish();
            pr->classes = std::move(lists);
            return TBSCI_OK;
        }
        uncharge(ctx, bytes);
    }
    lists->release();
    cudaGetLastError();  // a failed allocation is not the caller's error
    return e == cudaSuccess || e == cudaErrorMemoryAllocation ? TBSCI_OK
                                                               : fail(ctx, TBSCI_ECUDA, std::string("pruned space classes: ") + cudaGetErrorString(e));
}

}  // namespace

tbsci_status pruned_sigma_launch(tbsci_ctx *ctx, const tbsci_ham *ham, const Plan *plan, const tbsci_pruned *pr,
                                 const void *c, void *s, int nvec, tbsci_dtype dt, cudaStream_t st) {
    if (dt == TBSCI_F64)
        return launch_pruned<double>(ctx, ham, plan, pr, static_cast<const double *>(c), static_cast<double *>(s),
                                     nvec, st);
    if (dt == TBSCI_F32 || dt == TBSCI_F32_TC_TF32 || dt == TBSCI_F32_TC_BF16)
        return launch_pruned<float>(ctx, ham, plan, pr, static_cast<const float *>(c), static_cast<float *>(s), nvec,
                                    st);
    return fail(ctx, TBSCI_EINVAL, "unknown dtype");
}

tbsci_status pruned_diagonal_launch(tbsci_ctx *ctx, const tbsci_ham *ham, const Plan *P, const tbsci_pruned *pr,
                                    double *diag, cudaStream_t st) {
    if (pr->nd == 0 || P->A.l == 0) return TBSCI_OK;
    k_diagonal_pruned<<<(unsigned)P->A.l, 128, 0, st>>>(P->A.d_str, P->B.l, pr->d_off.p, pr->d_cols.p, P->A.d_E.p,
                                                       P->B.d_E.p, P->d_U.p, ham->ecore, diag);
    TB_CUDA(ctx, cudaGetLastError());
    return TBSCI_OK;
}

}  // namespace tbsci

using namespace tbsci;

extern "C" {

tbsci_status tbsci_pruned_create(tbsci_ctx *ctx, const tbsci_tables *a, const tbsci_tables *b, const int64_t *off,
                                 const int32_t *cols, tbsci_pruned **out) {
    if (!ctx) return TBSCI_EINVAL;
    TB_CUDA(ctx, cudaSetDevice(ctx->device));
    TB_CHECK(ctx, a && b && off && out, TBSCI_EINVAL, "tbsci_pruned_create: null argument");
    *out = nullptr;
    const int64_t la = a->count, lb = b->count;
    TB_CHECK(ctx, off[0] == 0, TBSCI_EINVAL, "tbsci_pruned_create: off[0] must be 0");
    for (int64_t w = 0; w < la; ++w)
        TB_CHECK(ctx, off[w + 1] >= off[w], TBSCI_EINVAL, "tbsci_pruned_create: off must be non-decreasing");
    const int64_t nd = off[la];
    TB_CHECK(ctx, nd == 0 || cols, TBSCI_EINVAL, "tbsci_pruned_create: null cols");
    for (int64_t w = 0; w < la; ++w)
        for (int64_t k = off[w]; k < off[w + 1]; ++k) {
            TB_CHECK(ctx, cols[k] >= 0 && cols[k] < lb, TBSCI_EINVAL,
                     "tbsci_pruned_create: beta index out of range in row " + std::to_string(w));
            TB_CHECK(ctx, k == off[w] || cols[k] > cols[k - 1], TBSCI_EINVAL,
                     "tbsci_pruned_create: beta indices of row " + std::to_string(w) + " not strictly ascending");
        }
    auto pr = std::make_unique<tbsci_pruned>();
    pr->ctx = ctx;
    pr->ida = a->id;
    pr->idb = b->id;
    pr->la = la;
    pr->lb = lb;
    pr->nd = nd;
    pr->h_off.assign(off, off + la + 1);
    // alpha rows by work, heaviest first: members x (1 + alpha singles + alpha doubles)
    std::vector<double> work(la);
    for (int64_t w = 0; w < la; ++w)
        work[w] = (double)(off[w + 1] - off[w]) *
                  (double)(1 + (a->h_off1[w + 1] - a->h_off1[w]) + (a->h_off2.empty() ? 0 : a->h_off2[w + 1] - a->h_off2[w]));
    std::vector<int32_t> rows(la);
    std::iota(rows.begin(), rows.end(), 0);
    std::stable_sort(rows.begin(), rows.end(), [&](int32_t x, int32_t y) { return work[x] > work[y]; });
    const size_t bytes = (size_t)(la + 1) * 8 + (size_t)nd * 4 + (size_t)la * 4;
    TB_TRY(charge(ctx, bytes, "pruned space"));
    pr->charged = bytes;
    cudaError_t e = pr->d_off.alloc(la + 1);
    if (e == cudaSuccess) e = pr->d_cols.alloc(nd);
    if (e == cudaSuccess) e = pr->d_rows.alloc(la);
    if (e == cudaSuccess) e = cudaMemcpy(pr->d_off.p, off, (la + 1) * sizeof(int64_t), cudaMemcpyHostToDevice);
    if (e == cudaSuccess && nd) e = cudaMemcpy(pr->d_cols.p, cols, nd * sizeof(int32_t), cudaMemcpyHostToDevice);
    if (e == cudaSuccess && la) e = cudaMemcpy(pr->d_rows.p, rows.data(), la * sizeof(int32_t), cudaMemcpyHostToDevice);
    if (e != cudaSuccess) {
        uncharge(ctx, bytes);
        return fail(ctx, e == cudaErrorMemoryAllocation ? TBSCI_ENOMEM : TBSCI_ECUDA,
                    std::string("tbsci_pruned_create: ") + cudaGetErrorString(e));
    }
    if (const tbsci_status st = build_classes(ctx, a, b, off, cols, pr.get()); st != TBSCI_OK) {
        uncharge(ctx, pr->charged);
        return st;
    }
    *out = pr.release();
    return TBSCI_OK;
}

// Symmetry blocks (Sec. II.A): each I_w is the class of beta strings whose irrep
// is target XOR irrep(w); a string's irrep is the XOR of the labels of its
// occupied orbitals. The classes are built once and copied per alpha string.
tbsci_status tbsci_pruned_create_symmetry(tbsci_ctx *ctx, const tbsci_tables *a, const tbsci_tables *b,
                                          const int32_t *orb_irrep, int target, tbsci_pruned **out) {
    if (!ctx) return TBSCI_EINVAL;
    TB_CUDA(ctx, cudaSetDevice(ctx->device));
    TB_CHECK(ctx, a && b && orb_irrep && out, TBSCI_EINVAL, "tbsci_pruned_create_symmetry: null argument");
    TB_CHECK(ctx, a->norb == b->norb, TBSCI_EINVAL, "tbsci_pruned_create_symmetry: norb differs between the sets");
    TB_CHECK(ctx, target >= 0 && target < 8, TBSCI_EINVAL, "tbsci_pruned_create_symmetry: target irrep not in 0..7");
    for (int i = 0; i < a->norb; ++i)
        TB_CHECK(ctx, orb_irrep[i] >= 0 && orb_irrep[i] < 8, TBSCI_EINVAL,
                 "tbsci_pruned_create_symmetry: orbital irrep not in 0..7");
    std::vector<uint64_t> sa(a->count), sb(b->count);
    if (a->count) TB_CUDA(ctx, cudaMemcpy(sa.data(), a->d_str.p, a->count * 8, cudaMemcpyDeviceToHost));
    if (b->count) TB_CUDA(ctx, cudaMemcpy(sb.data(), b->d_str.p, b->count * 8, cudaMemcpyDeviceToHost));
    auto irrep = [&](uint64_t s) {
        int g = 0;
        for (; s; s &= s - 1) g ^= orb_irrep[__builtin_ctzll(s)];
        return g;
    };
    std::vector<int32_t> cls[8];
    for (int64_t u = 0; u < b->count; ++u) cls[irrep(sb[u])].push_back((int32_t)u);
    std::vector<int64_t> off(a->count + 1, 0);
    for (int64_t w = 0; w < a->count; ++w) off[w + 1] = off[w] + (int64_t)cls[target ^ irrep(sa[w])].size();
    std::vector<int32_t> cols((size_t)off[a->count]);
    for (int64_t w = 0; w < a->count; ++w) {
        const std::vector<int32_t> &c = cls[target ^ irrep(sa[w])];
        std::copy(c.begin(), c.end(), cols.begin() + off[w]);
    }
    return tbsci_pruned_create(ctx, a, b, off.data(), cols.empty() ? nullptr : cols.data(), out);
}

tbsci_status tbsci_pruned_count(const tbsci_pruned *pr, int64_t *ndet) {
    if (!pr || !ndet) return TBSCI_EINVAL;
    *ndet = pr->nd;
    return TBSCI_OK;
}

void tbsci_pruned_destroy(tbsci_pruned *pr) {
    if (!pr) return;
    if (pr->ctx) cudaSetDevice(pr->ctx->device);
    pr->classes.reset();  // nothing is taken back from here on
    uncharge(pr->ctx, pr->charged);
    delete pr;
}

static tbsci_status pruned_plan(tbsci_ctx *ctx, tbsci_ham *ham, const tbsci_tables *a, const tbsci_tables *b,
                                const tbsci_pruned *pr, Plan **p) {
    if (!ctx) return TBSCI_EINVAL;
    TB_CUDA(ctx, cudaSetDevice(ctx->device));
    TB_CHECK(ctx, pr && a && b, TBSCI_EINVAL, "null handle");
    TB_CHECK(ctx, pr->ida == a->id && pr->idb == b->id, TBSCI_EINVAL,
             "the pruned space was made from other tables");
    return plan_get(ctx, ham, a, b, p);
}

tbsci_status tbsci_sigma_pruned(tbsci_ctx *ctx, tbsci_ham *ham, const tbsci_tables *a, const tbsci_tables *b,
                                const tbsci_pruned *pr, const void *c, void *sigma, int nvec, tbsci_dtype dtype,
                                tbsci_stream stream) {
    Plan *p = nullptr;
    TB_TRY(pruned_plan(ctx, ham, a, b, pr, &p));
    TB_CHECK(ctx, nvec >= 1, TBSCI_EINVAL, "nvec must be >= 1");
    if (pr->nd == 0) return TBSCI_OK;
    TB_CHECK(ctx, c && sigma && c != sigma, TBSCI_EINVAL, "bad vector pointers");
    return pruned_sigma_launch(ctx, ham, p, pr, c, sigma, nvec, dtype, (cudaStream_t)stream);
}

tbsci_status tbsci_diagonal_pruned(tbsci_ctx *ctx, tbsci_ham *ham, const tbsci_tables *a, const tbsci_tables *b,
                                   const tbsci_pruned *pr, double *diag, tbsci_stream stream) {
    Plan *p = nullptr;
    TB_TRY(pruned_plan(ctx, ham, a, b, pr, &p));
    if (pr->nd == 0) return TBSCI_OK;
    TB_CHECK(ctx, diag, TBSCI_EINVAL, "null diag pointer");
    return pruned_diagonal_launch(ctx, ham, p, pr, diag, (cudaStream_t)stream);
}

tbsci_status tbsci_davidson_pruned(tbsci_ctx *ctx, tbsci_ham *ham, const tbsci_tables *a, const tbsci_tables *b,
                                   const tbsci_pruned *pr, int nroots, const tbsci_davidson_opts *opts,
                                   double *energies, double *vecs, tbsci_davidson_info *info) {
    Plan *p = nullptr;
    TB_TRY(pruned_plan(ctx, ham, a, b, pr, &p));
    TB_CHECK(ctx, energies, TBSCI_EINVAL, "null energies");
    tbsci_davidson_opts o{};
    if (opts) o = *opts;
    else o.mixed = ctx->default_mixed;
    const size_t bytes = engine_device_bytes(pr->nd, nroots, &o);
    TB_TRY(charge(ctx, bytes, "Davidson vectors"));
    tbsci_status st = davidson_run(ctx, ham, p, nroots, &o, energies, vecs, info, pr);
    uncharge(ctx, bytes);
    return st;
}

}  // extern "C"

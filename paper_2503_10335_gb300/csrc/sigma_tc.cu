// The alpha-beta classes of sigma on the 5th-generation tensor cores, in FP32.
//
// For one alpha row Ia (one CTA), with K alpha terms k = (Ja_k, pq_k, s_k):
// k = 0 is Ja = Ia ("W" row: sum_{p in Ia} (pp|rs)), k >= 1 the alpha singles.
//   G[rs][Jb] = sum_k A[rs][k] * F[k][Jb],   A[rs][k] = s_k (pq_k|rs) (k >= 1),
//                                            A[rs][0] = sum_{p in Ia} (pp|rs),
//                                            F[k][Jb] = c(Ja_k, Jb)
// over the off-diagonal orbital pairs rs (one 128-row MMA tile for norb <= 16),
// then sigma(Ia, Ib) += sign * G[rs][Jb] for every beta single link
// Ib = E_rs Jb (the gather D of the classic formulation, done from the accumulators).
// The beta-diagonal pairs (r = s in Ib), the alpha-single string-Hamiltonian values
// and the diagonal are added by k_udiag (sigma_exact.cu). Together: classes [1,1],
// [1,0], [0,1] (alpha-beta part) and [0,0] of Sec. II.C; the same-spin classes come
// from the passes of sigma.cu, sigma_split.cu or sigma_dense.cu run first.
//
// Precision: three BF16 planes per operand (x = x0 + x1 + x2 holds all 24 bits of an
// FP32 value) and the six products x_i y_j with i + j <= 2, FP32 accumulation, for the
// split-TF32 type and the FP32 type (at least the accuracy of three TF32 products, at
// the same tensor-core time); or one BF16 product (~3 significant digits).
//
// What bounds it: not the products (512 to 960 tensor-core cycles per 64 columns) but
// the way of G into the sigma row. So it keeps the products' operands out of the
// draining warps' hands (A lies in TMEM for the whole row; three warps stage the coupled
// c rows, a tile each) and gives the accumulators a plan of the links made once per space:
// every link of a 64-column tile has a slot, the slots of a target column are consecutive,
// and a thread sums up to four of them. No atomics: results are run-to-run identical.
// c arrives as BF16 planes cut once per vector into memory of the space (a 128-byte
// segment per coupled row). In a graph, whose replays would share that memory with other
// streams, and where there is no room for it, the staging warps cut c themselves, to the
// same bits: 100 ms instead of 67 on the full norb-16 space with three planes, 54 instead
// of 42 with one.
// Norb 16, full space (165.6M determinants), one vector: 35.7 ms with three planes, 30.4
// ms with one; 85 and 53 ms with operands staged element by element and sums by
// shared-memory atomics.
// Every mbarrier wait is bounded; on timeout the CTA records an error, writes a NaN,
// skips the rest of its row and still frees its TMEM.
#include <cuda_bf16.h>

#include <algorithm>
#include <type_traits>

#include "internal.cuh"
#include "tensor.cuh"

namespace tbsci {

namespace {

// ------------------------------------------------------------------ link plan

constexpr int kLinkThreads = 256;

// One CTA per tile of 64 columns Jb. counts -> places of the target columns' lists ->
// ranks of the links. Lists of n slots are summed by ceil(n / 4) consecutive lanes,
// aligned to a power of two so that a list stays in one warp, longest lists first.
// Within a list: positive links by column and pair, then negative ones.
__global__ void __launch_bounds__(kLinkThreads) k_tile_links(const int32_t *__restrict__ lbp, int64_t lb, int npoff, int npiece,
                                                             int nslot, uint16_t *pos, int2 *piece, int *rounds) {
    extern __shared__ uint32_t scnt[];  // [lb] positive links | negative links << 16, then the next slots
    __shared__ int sOff[6][kLinkThreads];
    __shared__ int sTot[6];
    const int t = blockIdx.x, tid = threadIdx.x;
    const int64_t j0 = (int64_t)t * kAbTile;
    const int ncol = (int)min((int64_t)kAbTile, lb - j0);
    const int32_t *L = lbp + j0 * npoff;
    for (int64_t i = tid; i < lb; i += kLinkThreads) scnt[i] = 0;
    __syncthreads();
    for (int x = tid; x < ncol * npoff; x += kLinkThreads) {
        const int32_t e = L[x];
        if (e >= 0) atomicAdd(&scnt[e >> 1], (e & 1) ? 0x10000u : 1u);
    }
    __syncthreads();
    const int64_t per = (lb + kLinkThreads - 1) / kLinkThreads, a = min(lb, tid * per), b = min(lb, a + per);
    int own[6] = {0, 0, 0, 0, 0, 0};  // lists by size class (1, 2, 4, 8, 16 lanes), slots
    for (int64_t i = a; i < b; ++i) {
        const int n = (int)(scnt[i] & 0xFFFF) + (int)(scnt[i] >> 16);
        if (!n) continue;
        const int np = (n + kPiece - 1) / kPiece;
        ++own[np <= 1 ? 0 : np <= 2 ? 1 : np <= 4 ? 2 : np <= 8 ? 3 : 4];
        own[5] += n;
    }
#pragma unroll
    for (int k = 0; k < 6; ++k) sOff[k][tid] = own[k];
    __syncthreads();
    if (tid < 6) {  // exclusive sums in thread order
        int run = 0;
        for (int k = 0; k < kLinkThreads; ++k) {
            const int x = sOff[tid][k];
            sOff[tid][k] = run;
            run += x;
        }
        sTot[tid] = run;
    }
    __syncthreads();
    int base[5], lanes = 0;
#pragma unroll
    for (int k = 4; k >= 0; --k) {
        base[k] = lanes;
        lanes += sTot[k] << k;
    }
    int2 *P = piece + (int64_t)t * npiece;
    int at[5], slot = sOff[5][tid];
#pragma unroll
    for (int k = 0; k < 5; ++k) at[k] = base[k] + (sOff[k][tid] << k);
    for (int64_t i = a; i < b; ++i) {
        const int plus = (int)(scnt[i] & 0xFFFF), n = plus + (int)(scnt[i] >> 16);
        if (!n) continue;
        const int np = (n + kPiece - 1) / kPiece, cl = np <= 1 ? 0 : np <= 2 ? 1 : np <= 4 ? 2 : np <= 8 ? 3 : 4;
        int p = 0;
#pragma unroll
        for (int k = 0; k < 5; ++k)
            if (k == cl) {
                p = at[k];
                at[k] += 1 << k;
            }
        for (int k = 0; k < (1 << cl); ++k) {
            int2 v = make_int2(-1, 0);
            if (k < np) {
                const int s = k * kPiece, cnt = min(kPiece, n - s), pc = min(cnt, max(0, plus - s));
                v = make_int2(k ? -1 : (int)i, (int)((uint32_t)(slot + s) | ((uint32_t)pc << 16) | ((uint32_t)(cnt - pc) << 20) |
                                                     ((uint32_t)(np - 1 - k) << 24)));
            }
            P[p + k] = v;
        }
        scnt[i] = (uint32_t)slot | ((uint32_t)(slot + plus) << 16);
        slot += n;
    }
    for (int k = lanes + tid; k < npiece; k += kLinkThreads) P[k] = make_int2(-1, 0);
    if (tid == 0) rounds[t] = (lanes + kAbDrain - 1) / kAbDrain;
    __syncthreads();
    for (int c = 0; c < kAbTile; ++c) {  // a target occurs at most once per column
        for (int rs = tid; rs < 128; rs += kLinkThreads) {
            uint16_t s = (uint16_t)(nslot - 1);
            const int32_t e = c < ncol && rs < npoff ? L[c * npoff + rs] : -1;
            if (e >= 0) {
                const uint32_t x = scnt[e >> 1];
                s = (uint16_t)((e & 1) ? x >> 16 : x & 0xFFFF);
                scnt[e >> 1] = x + ((e & 1) ? 0x10000u : 1u);
            }
            pos[((((size_t)t * 4 + (c >> 4)) * 2 + ((c >> 3) & 1)) * 128 + rs) * 8 + (c & 7)] = s;
        }
        __syncthreads();
    }
}

// ------------------------------------------------------------------ planes

// planes [NP][la][lbp] of a vector, columns lb .. lbp - 1 zero; 8 columns per thread
template <int NP>
__global__ void __launch_bounds__(256) k_planes(const float *__restrict__ c, int64_t la, int64_t lb, int64_t lbp,
                                                const int *__restrict__ info, __nv_bfloat16 *out) {
    if (info && !info[2 * blockIdx.y]) return;  // one vector per blockIdx.y
    c += blockIdx.y * la * lb;
    out += blockIdx.y * NP * la * lbp;
    const int64_t per = lbp / 8, n = la * per, plane = la * lbp;
    for (int64_t i = blockIdx.x * 256ll + threadIdx.x; i < n; i += (int64_t)gridDim.x * 256) {
        const int64_t r = i / per, j = (i - r * per) * 8;
        uint32_t h[8][NP];
#pragma unroll
        for (int u = 0; u < 8; ++u) bf16_planes<NP>(j + u < lb ? __ldg(c + r * lb + j + u) : 0.f, h[u]);
#pragma unroll
        for (int s = 0; s < NP; ++s)
            *reinterpret_cast<uint4 *>(out + s * plane + r * lbp + j) =
                make_uint4(h[0][s] | (h[1][s] << 16), h[2][s] | (h[3][s] << 16), h[4][s] | (h[5][s] << 16), h[6][s] | (h[7][s] << 16));
    }
}

// Cuts the columns 64 t .. 64 t + 63 of the rows sJa[0 .. Kp - 1] of c into planes in stage
// `dst0` by one warp, two columns per lane: MN-major operand planes of Kp rows of 128 bytes,
// 128-byte swizzle. PAIR: rows of c start on 8 bytes (even length), else scalar loads. Eight
// rows of loads are in flight (a warp has three tile times for its tile).
template <int NP, bool PAIR>
__device__ __forceinline__ void stage_tile(const float *__restrict__ C, int64_t lb, const int *sJa, int Kp, int t, uint32_t dst0) {
    constexpr int kRows = 8;  // Kp is a multiple of 16
    const int lane = threadIdx.x & 31;
    const int64_t j = (int64_t)t * kAbTile + 2 * lane;
    const bool in0 = j < lb, in1 = j + 1 < lb;
    const float *src0 = C + j;
    for (int k0 = 0; k0 < Kp; k0 += kRows) {
        float x[kRows], y[kRows];
#pragma unroll
        for (int u = 0; u < kRows; ++u) {
            const float *src = src0 + (size_t)sJa[k0 + u] * lb;
            if (PAIR) {
                const float2 v = in0 ? __ldg(reinterpret_cast<const float2 *>(src)) : make_float2(0.f, 0.f);
                x[u] = v.x;
                y[u] = v.y;
            } else {
                x[u] = in0 ? __ldg(src) : 0.f;
                y[u] = in1 ? __ldg(src + 1) : 0.f;
            }
        }
#pragma unroll
        for (int u = 0; u < kRows; ++u) {
            const int k = k0 + u;
            uint32_t hx[NP], hy[NP];
            bf16_planes<NP>(x[u], hx);
            bf16_planes<NP>(y[u], hy);
            const uint32_t dst = dst0 + k * 128 + (((lane >> 2) ^ (k & 7)) << 4) + ((lane & 3) << 2);
#pragma unroll
            for (int s = 0; s < NP; ++s)
                asm volatile("st.shared.b32 [%0], %1;" ::"r"(dst + s * Kp * 128), "r"(hx[s] | (hy[s] << 16)) : "memory");
        }
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

// planes of the integral columns, [pair][128 off-diagonal pairs] x 4 BF16 (the last zero), or of
// W_Ia, [la][128] x 4; one plane is the first of three
__global__ void k_ab_planes(const float *__restrict__ V, int npair, int npoff, const int32_t *__restrict__ offpair,
                            const uint64_t *__restrict__ str, int64_t rows, uint2 *out) {
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= rows * 128) return;
    const int64_t row = i >> 7;
    const int rs = (int)(i & 127);
    float x = 0.f;
    if (rs < npoff) {
        const int col = offpair[rs];
        if (str) {
            for (uint64_t s = str[row]; s; s &= s - 1) {
                const int p = __ffsll((long long)s) - 1;
                x += V[(size_t)(p * (p + 1) / 2 + p) * npair + col];
            }
        } else {
            x = V[(size_t)row * npair + col];
        }
    }
    uint32_t h[3];
    bf16_planes<3>(x, h);
    out[i] = make_uint2(h[0] | (h[1] << 16), h[2]);
}

// ------------------------------------------------------------------ the kernel

struct FpArgs {
    int64_t la, lb, lbp;
    const float *C;
    const __nv_bfloat16 *Cs;  // planes of c (PLANES)
    float *S;
    const int *info;       // run only where info[2 v] is set (NULL: always)
    const uint2 *Vd, *Wd;  // [pair][128], [la][128] x 4 BF16
    const int64_t *a_soff;
    const int2 *a_sci;
    const uint4 *pos;      // [tile][4][2][128] x 8: slot of (pair, column); nslot - 1: no link
    const int2 *piece;     // [tile][npiece]: {target column (-1: not the first piece of its list), first slot |
                           // positive links << 16 | negative links << 20 | further pieces << 24}
    const int *rounds;     // [tile] pieces / kAbDrain, rounded up
    int npiece, nslot;
    int stage_bytes;       // shared memory for the staged c rows
    int pair;              // rows of c start on 8 bytes
    const int32_t *rowsa;
    int *err;
};

template <int NP, bool PLANES>
__global__ void __launch_bounds__(kAbThreads, 1) k_sigma_ab_tc(const FpArgs A) {
    if (A.info && !A.info[2 * blockIdx.y]) return;  // one vector per blockIdx.y
    extern __shared__ unsigned char smem_dyn[];
    __shared__ uint64_t bar[16];
    __shared__ uint32_t tmem_base;
    __shared__ int sAbort;
    __shared__ int sJa[kAbMaxK], sPq[kAbMaxK];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int64_t lb = A.lb, Ia = A.rowsa[blockIdx.x], t0 = A.a_soff[Ia];
    const int K = 1 + (int)(A.a_soff[Ia + 1] - t0), Kp = (K + 15) / 16 * 16;
    const uint32_t stage_sz = (uint32_t)NP * Kp * kAbTile * 2;
    const int nst = min(4, A.stage_bytes / (int)stage_sz);
    constexpr int ndb = 4;                                      // accumulators: NP Kp / 2 <= 120 columns of A, then 4 x 64
    const int dcol0 = (NP * Kp / 2 + 31) / 32 * 32;
    unsigned char *sm = smem_dyn + ((1024 - (su32(smem_dyn) & 1023)) & 1023);
    const uint32_t sB = su32(sm);
    float *sAcc = reinterpret_cast<float *>(sm + A.stage_bytes);  // [lb]
    float *sSlot = sAcc + lb;                                     // [2][nslot]
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
    for (int64_t j = tid; j < lb; j += kAbThreads) sAcc[j] = 0.f;
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
        // A's planes: lane = pair row, two terms per 32-bit column, plane s at column s Kp / 2
        const int quarter = warp & 3, rs = quarter * 32 + lane;
        for (int kb = warp >> 2; kb < Kp / 8; kb += 4) {
            uint32_t v[8][2];
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                const int k = kb * 8 + q, pq = sPq[k];
                uint2 x = make_uint2(0, 0);
                if (k == 0) x = __ldg(A.Wd + Ia * 128 + rs);
                else if (pq >= 0) x = __ldg(A.Vd + (size_t)(pq >> 1) * 128 + rs);
                const uint32_t neg = k > 0 && pq >= 0 && (pq & 1) ? 0x80008000u : 0u;
                v[q][0] = x.x ^ neg;
                v[q][1] = x.y ^ neg;
            }
#pragma unroll
            for (int s = 0; s < NP; ++s) {
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
        const uint32_t dbase = uni((uint32_t)dcol0);
        int st = 0;
        uint32_t sph = 0;
        bool ok = true;
        // unrolled for the row's number of 16-term steps, so that every descriptor is a
        // uniform base plus an immediate
        auto tiles = [&](auto ks_tag) {
            constexpr int KS = decltype(ks_tag)::value;
            for (int t = 0; t < ntiles && ok; ++t) {
                const int db = t & (ndb - 1);
                ok = __all_sync(0xffffffffu, mb_wait(bfull + 8 * st, sph, ab));
                if (ok && t >= ndb) ok = __all_sync(0xffffffffu, mb_wait(dempty + 8 * db, (t / ndb - 1) & 1, ab));
                if (!ok) break;
                tc_after();
                const uint64_t b0 = op_desc(uni(sB + st * stage_sz), 16, 1024, 2);
                const uint32_t d = uni(dbase + db * kAbTile);
                if (elect_one()) {
                    constexpr uint32_t idesc = inst_desc(kAbTile, true);
                    // smallest products first
#pragma unroll
                    for (int o = NP - 1; o >= 0; --o)
#pragma unroll
                        for (int i = 0; i <= o; ++i)
#pragma unroll
                            for (int ks = 0; ks < KS; ++ks)
                                asm volatile(
                                    "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
                                    " tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n}" ::"r"(d),
                                    "r"(tmem + i * (KS * 8) + ks * 8), "l"(b0 + ((o - i) * KS + ks) * (kAbTile * 2)), "r"(idesc),
                                    "r"(o == NP - 1 && i == 0 && ks == 0 ? 0u : 1u)
                                    : "memory");
                    mma_commit(dfull + 8 * db);
                    mma_commit(bempty + 8 * st);
                }
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
        __syncwarp();
    } else if (warp >= 16) {
        // a warp stages a whole tile; three tiles are on their way (not more than there are
        // stages: a wait must not run a phase ahead of its barrier)
        const int ng = min(3, nst), g = warp - 16;
        for (int t = g; t < ntiles && g < ng; t += ng) {
            const int st = t % nst;
            if (t >= nst && !mb_wait(bempty + 8 * st, (t / nst - 1) & 1, ab)) break;
            const float *C = A.C + blockIdx.y * A.la * lb;
            if (PLANES)
                gather_tile<NP>(A.Cs + blockIdx.y * NP * A.la * A.lbp, (size_t)A.la * A.lbp, A.lbp, sJa, Kp, t, sB + st * stage_sz);
            else if (A.pair) stage_tile<NP, true>(C, lb, sJa, Kp, t, sB + st * stage_sz);
            else stage_tile<NP, false>(C, lb, sJa, Kp, t, sB + st * stage_sz);
            mb_arrive(bfull + 8 * st);
        }
    } else {
        const int quarter = warp & 3, part = warp >> 2, rs = quarter * 32 + lane;
        // slots, pieces and rounds of a tile are read a tile ahead
        const uint4 *pp = A.pos + (size_t)part * 2 * 128 + rs;
        const int2 *pc = A.piece + tid;
        uint4 p0 = __ldg(pp), p1 = __ldg(pp + 128);
        int nr = __ldg(A.rounds);
        int2 sg = __ldg(pc), sg1 = nr > 1 ? __ldg(pc + kAbDrain) : make_int2(-1, 0);
        for (int t = 0; t < ntiles; ++t) {
            const int db = t & (ndb - 1);
            float *slots = sSlot + (t & 1) * A.nslot;
            const bool ok = __all_sync(0xffffffffu, mb_wait(dfull + 8 * db, (t / ndb) & 1, ab));
            tc_after();
            uint32_t q[16];
            if (ok) {
                tmem_ld16(tmem + ((uint32_t)(quarter * 32) << 16) + dcol0 + db * kAbTile + part * 16, q);
                pin16(q);
            } else {
#pragma unroll
                for (int x = 0; x < 16; ++x) q[x] = 0;
            }
            tc_before();
            __syncwarp();
            if (lane == 0) mb_arrive(dempty + 8 * db);
            const uint32_t pw[8] = {p0.x, p0.y, p0.z, p0.w, p1.x, p1.y, p1.z, p1.w};
#pragma unroll
            for (int x = 0; x < 16; ++x)
                slots[(pw[x >> 1] >> (16 * (x & 1))) & 0xFFFFu] = __uint_as_float(q[x]);  // no link: the last slot
            const int rounds = nr;
            const int2 *cur = pc;
            int2 c0 = sg, c1 = sg1;
            if (t + 1 < ntiles) {
                pp += 4 * 2 * 128;
                pc += A.npiece;
                p0 = __ldg(pp);
                p1 = __ldg(pp + 128);
                nr = __ldg(A.rounds + t + 1);
                sg = __ldg(pc);
                sg1 = A.npiece > kAbDrain ? __ldg(pc + kAbDrain) : make_int2(-1, 0);
            }
            // one barrier per tile: a warp that passes it has summed the tile before last,
            // whose slots this tile's successor writes
            asm volatile("bar.sync 1, 512;" ::: "memory");
            for (int i = 0; i < rounds; ++i) {
                const uint32_t y = (uint32_t)c0.y;
                const int ib = c0.x, first = y & 0xFFFF, np = (y >> 16) & 0xF, n = np + ((y >> 20) & 0xF);
                const int more = y >> 24;  // further pieces, in the lanes above
                c0 = c1;
                if (i + 2 < rounds) c1 = __ldg(cur + (i + 2) * kAbDrain);
                float z[kPiece];
#pragma unroll
                for (int k = 0; k < kPiece; ++k) z[k] = slots[first + k];
                float v = 0.f;
#pragma unroll
                for (int k = 0; k < kPiece; ++k)
                    if (k < n) v += k < np ? z[k] : -z[k];
                const int steps = __reduce_max_sync(0xffffffffu, (unsigned)more);
                for (int d = 1; d <= steps; d <<= 1) {
                    const float w = __shfl_down_sync(0xffffffffu, v, d);
                    if (d <= more) v += w;
                }
                if (ib >= 0) sAcc[ib] += v;
            }
        }
    }
    tc_before();
    __syncthreads();
    float *S = A.S + (blockIdx.y * A.la + Ia) * lb;
    for (int64_t j = tid; j < lb; j += kAbThreads) S[j] += sAcc[j];
    if (sAbort && tid == 0) {
        atomicExch(A.err, 1);
        S[0] = NAN;  // fail loudly
    }
    if (warp == 19) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem_base));
}

inline int64_t pad64(int64_t l) { return (l + 63) / 64 * 64; }

// stages of the fullest row that fit beside the sigma row and the slots (at most four), as bytes; 0: none
int fp_stage_bytes(const tbsci_ctx *ctx, const Plan *P, int np) {
    const int64_t one = (int64_t)np * P->tl_kpmax * kAbTile * 2;
    const int64_t fixed = 1024 + 4 * (P->B.l + 2 * (int64_t)P->tl_nslot);
    const int64_t room = ((int64_t)ctx->smem_optin - 2048 - fixed) / 1024 * 1024;
    return room < one ? 0 : (int)std::min<int64_t>(room, 4 * one);
}

}  // namespace

// Vectors per launch: small spaces share the launches with up to eight (up to 2^24
// determinants together).
int sigma_tc_batch(int64_t ndet) {
    return (int)std::max<int64_t>(1, std::min<int64_t>(8, (int64_t(1) << 24) / std::max<int64_t>(1, ndet)));
}

// Spare bytes that a tensor-core type takes on a space of these sizes: planes of c
size_t sigma_tc_device_bytes(int norb, int64_t la, int64_t lb, int np) {
    return norb < 2 || norb > 16 ? 0 : (size_t)sigma_tc_batch(la * lb) * np * la * pad64(lb) * sizeof(__nv_bfloat16);
}

// Link plan of a space (norb <= 16) and planes of its integrals, made when the space is prepared; left out
// (tl_kpmax = 0) where the alpha-beta kernels do not apply.
void tile_links_size(tbsci_ctx *ctx, Plan *P) {
    const int64_t la = P->A.l, lb = P->B.l;
    P->tl_kpmax = 0;
    if (P->npoff < 1 || P->npoff > 120 || la < 1 || lb < 1) return;
    const int kmax = 1 + P->a_smax;
    if (kmax > 65 || (size_t)lb * 4 + 16384 > ctx->smem_optin) return;
    const int nt = (int)((lb + kAbTile - 1) / kAbTile);
    int links = 0;
    for (int t = 0; t < nt; ++t)
        links = std::max<int>(links, (int)(P->B.h_soff[std::min<int64_t>(lb, (t + 1) * (int64_t)kAbTile)] - P->B.h_soff[(int64_t)t * kAbTile]));
    P->tl_nslot = (links + kPiece + 2) / 2 * 2;  // a piece is read whole; the last slot takes pairs without a link
    P->tl_npiece = std::max(1, (links + kAbDrain - 1) / kAbDrain) * kAbDrain;
    P->arena.add(P->d_tl_pos, (size_t)nt * 4 * 2 * 128);
    P->arena.add(P->d_tl_piece, (size_t)nt * P->tl_npiece);
    P->arena.add(P->d_tl_rounds, nt);
    P->arena.add(P->d_ab_v, (size_t)P->npair * 128);
    P->arena.add(P->d_ab_w, (size_t)la * 128);
    P->tl_kpmax = (kmax + 15) / 16 * 16;
}

tbsci_status tile_links_build(tbsci_ctx *ctx, const tbsci_ham *ham, Plan *P, cudaStream_t st) {
    if (P->tl_kpmax == 0) return TBSCI_OK;
    const int64_t la = P->A.l, lb = P->B.l;
    const size_t smem = (size_t)lb * 4;
    TB_CUDA(ctx, cudaFuncSetAttribute(k_tile_links, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    k_tile_links<<<(unsigned)((lb + kAbTile - 1) / kAbTile), kLinkThreads, smem, st>>>(
        P->d_lbp.p, lb, P->npoff, P->tl_npiece, P->tl_nslot, reinterpret_cast<uint16_t *>(P->d_tl_pos.p), P->d_tl_piece.p,
        P->d_tl_rounds.p);
    k_ab_planes<<<(unsigned)((P->npair * 128 + 255) / 256), 256, 0, st>>>(ham->d_Vf.p, P->npair, P->npoff, P->d_offpair.p, nullptr,
                                                                         P->npair, P->d_ab_v.p);
    k_ab_planes<<<(unsigned)((la * 128 + 255) / 256), 256, 0, st>>>(ham->d_Vf.p, P->npair, P->npoff, P->d_offpair.p, P->A.d_str, la,
                                                                   P->d_ab_w.p);
    TB_CUDA(ctx, cudaGetLastError());
    return TBSCI_OK;
}

// The planes of c of one space and number of planes (spare memory), made by the first sigma
// that has room for them. Calls on several streams share them: each waits for the event that
// the one before it recorded, and `mu` keeps the launches of one call together.
struct AbPlanes : Spare {
    cudaEvent_t busy = nullptr;
    bool tried = false;
    DevBuf<__nv_bfloat16> c;  // planes of sigma_tc_batch vectors
    explicit AbPlanes(tbsci_ctx *x) : Spare(x) { enlist(); }
    ~AbPlanes() override {
        retire();
        uncharge(ctx, c.bytes());
        if (busy) cudaEventDestroy(busy);
    }
    bool give_back() override {
        if (!c.p || cudaEventSynchronize(busy) != cudaSuccess) return false;
        uncharge(ctx, c.bytes());
        c.release();
        tried = false;
        return true;
    }
};

namespace {

tbsci_status build_planes(tbsci_ctx *ctx, const Plan *P, int np, AbPlanes *X) {
    const size_t n = (size_t)sigma_tc_batch(P->A.l * P->B.l) * np * P->A.l * pad64(P->B.l), bytes = n * sizeof(__nv_bfloat16);
    if (!spare_charge(ctx, bytes)) return TBSCI_OK;  // asked for again by the next call
    X->tried = true;
    cudaError_t e = X->busy ? cudaSuccess : cudaEventCreateWithFlags(&X->busy, cudaEventDisableTiming);
    if (e == cudaSuccess) e = X->c.alloc(n, true);
    if (e != cudaSuccess) {
        uncharge(ctx, bytes);
        cudaGetLastError();
        return e == cudaErrorMemoryAllocation ? TBSCI_OK : fail(ctx, TBSCI_ECUDA, std::string("alpha-beta planes: ") + cudaGetErrorString(e));
    }
    return TBSCI_OK;
}

template <int NP>
tbsci_status ab_launch(tbsci_ctx *ctx, const Plan *P, const __nv_bfloat16 *planes, const float *c, float *s,
                       int nv, const int *info, cudaStream_t st) {
    const int64_t la = P->A.l, lb = P->B.l;
    FpArgs A{};
    A.la = la;
    A.lb = lb;
    A.lbp = pad64(lb);
    A.C = c;
    A.Cs = planes;
    A.S = s;
    A.info = info;
    A.Vd = P->d_ab_v.p;
    A.Wd = P->d_ab_w.p;
    A.a_soff = P->A.d_soff;
    A.a_sci = P->A.d_sci.p;
    A.pos = P->d_tl_pos.p;
    A.piece = P->d_tl_piece.p;
    A.rounds = P->d_tl_rounds.p;
    A.npiece = P->tl_npiece;
    A.nslot = P->tl_nslot;
    A.stage_bytes = fp_stage_bytes(ctx, P, NP);
    A.pair = lb % 2 == 0 && (uintptr_t)c % 8 == 0;
    A.rowsa = P->d_rowsa.p;
    A.err = P->d_tc_err.p;
    const size_t smem = 1024 + (size_t)A.stage_bytes + 4 * ((size_t)lb + 2 * (size_t)A.nslot);
    auto kern = planes ? k_sigma_ab_tc<NP, true> : k_sigma_ab_tc<NP, false>;
    TB_CUDA(ctx, cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    TraceScope tr(ctx, "k_sigma_ab_tc", st);
    kern<<<dim3((unsigned)la, (unsigned)nv), kAbThreads, smem, st>>>(A);
    TB_CUDA(ctx, cudaGetLastError());
    return TBSCI_OK;
}

template <int NP>
tbsci_status ab_add(tbsci_ctx *ctx, Plan *P, AbPlanes *X, const float *c, float *s, int nv, const int *info,
                    cudaStream_t st) {
    if (!X) return ab_launch<NP>(ctx, P, nullptr, c, s, nv, info, st);
    const int64_t la = P->A.l, lb = P->B.l, lbp = pad64(lb);
    TB_CUDA(ctx, cudaStreamWaitEvent(st, X->busy, 0));
    {
        TraceScope tr(ctx, "k_planes", st);
        const unsigned nb = (unsigned)std::min<int64_t>(8ll * ctx->num_sms, (la * (lbp / 8) + 255) / 256);
        k_planes<NP><<<dim3(nb, (unsigned)nv), 256, 0, st>>>(c, la, lb, lbp, info, X->c.p);
        TB_CUDA(ctx, cudaGetLastError());
    }
    const tbsci_status r = ab_launch<NP>(ctx, P, X->c.p, c, s, nv, info, st);
    TB_CUDA(ctx, cudaEventRecord(X->busy, st));  // also behind a failed launch: the planes are in use
    return r;
}

}  // namespace

// Whether the kernel serves a space with `np` planes (1 or 3)
bool sigma_tc_serves(const tbsci_ctx *ctx, const Plan *P, int np) { return P->tl_kpmax > 0 && fp_stage_bytes(ctx, P, np) > 0; }

// The three planes [nv][3][la][pad64(lb)] of nv vectors, for the vectors whose info is set
tbsci_status sigma_tc_planes(tbsci_ctx *ctx, const Plan *P, const float *c, int nv, const int *info, __nv_bfloat16 *out,
                             cudaStream_t st) {
    const int64_t la = P->A.l, lb = P->B.l, lbp = pad64(lb);
    TraceScope tr(ctx, "k_planes", st);
    const unsigned nb = (unsigned)std::min<int64_t>(8ll * ctx->num_sms, (la * (lbp / 8) + 255) / 256);
    k_planes<3><<<dim3(nb, (unsigned)nv), 256, 0, st>>>(c, la, lb, lbp, info, out);
    TB_CUDA(ctx, cudaGetLastError());
    return TBSCI_OK;
}

// Adds the alpha-beta products of nv vectors (at most sigma_tc_batch) into s; info: device
// flags [nv][2], nothing is done for a vector whose first one is 0 (NULL: always); planes:
// those of c if the caller has them (np = 3).
tbsci_status sigma_tc_ab(tbsci_ctx *ctx, Plan *P, int np, const float *c, float *s, int nv,
                         const int *info, cudaStream_t st, const __nv_bfloat16 *planes) {
    if (planes) return ab_launch<3>(ctx, P, planes, c, s, nv, info, st);
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    const cudaError_t e = cudaStreamIsCapturing(st, &cap);
    if (e != cudaSuccess) cudaGetLastError();
    if (e != cudaSuccess || cap != cudaStreamCaptureStatusNone || P->no_spare) {
        return np == 1 ? ab_add<1>(ctx, P, nullptr, c, s, nv, info, st) : ab_add<3>(ctx, P, nullptr, c, s, nv, info, st);
    }
    std::shared_ptr<AbPlanes> &own = P->ab[np == 1 ? 0 : 1];
    {
        static std::mutex make;
        std::lock_guard<std::mutex> g(make);
        if (!own) own = std::make_shared<AbPlanes>(ctx);
    }
    std::lock_guard<std::mutex> g(own->mu);
    if (!own->tried) TB_TRY(build_planes(ctx, P, np, own.get()));
    AbPlanes *X = own->c.p ? own.get() : nullptr;
    return np == 1 ? ab_add<1>(ctx, P, X, c, s, nv, info, st) : ab_add<3>(ctx, P, X, c, s, nv, info, st);
}

}  // namespace tbsci

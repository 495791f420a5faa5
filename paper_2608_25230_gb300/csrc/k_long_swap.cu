// k_long_swap.cu -- the balancing selector (Sec. 2.1) inside the candidate set
// (Definition 2.2) for rows of any length.
//
// One persistent block walks rows.  Per row, one pass over the keys
// accumulates the band sums S_b = sum p_j v_j (band = number of budgets that
// drop key j), the band masses and every key's single-key error
// p_j ||v_j - o|| (o = the dense output given by fw_dense_and_topk_gap).  Per
// budget: the E extras are the dropped keys of largest single-key error (a
// radix select on the error's bits, ties to lower indices); the current set
// is described by
//   g = sum_{A} u_i = pbar(A) N_A - p(A) N_{A^c},  u_i = p_i w_i,  w = v - mu,
// with mu = sum_b S_b and disjoint sums, so g carries no cancellation.
//
// Scoring a swap.  With N = |g|^2 and P = p(A), exchanging kept i for pool key
// j changes es^2 by D_ij / (P^2 P'^2), P' = P + p_j - p_i, where
//   D_ij = (alpha_i + beta_j - 2 p_i p_j C_ij) P^2 - N (p_j - p_i)(2P + p_j - p_i),
//   alpha_i = p_i^2 |w_i|^2 - 2 p_i g.w_i,  beta_j = p_j^2 |w_j|^2 + 2 p_j g.w_j,
//   C_ij = w_i . w_j.
// The swap lowers es iff D_ij < 0; the round takes the pair of smallest
// D_ij / P'^2 (ties: smallest i, then j) and stops when that is not negative.
//
// Only C_ij needs a d-long product per pair, and it does not depend on g: a
// swap changes one kept position (the key that enters) and one pool slot (the
// key that leaves takes the entering key's slot).  So the block keeps the
// table C[slot][position] in its workspace: the first round of a budget fills
// it (a k x d by d x E product in register tiles), and every later round
// computes only the changed slot's column y.w_i, y the leaving key's vector,
// and the changed position's row.  g.w_i is formed anew from g in every round,
// beside the column and from the same read of the value row: carried along from
// the table's entries (g.w_t moves by p_j C_jt - p_i C_it) it would gather their
// rounding swap by swap, apart from g's own.
//
// A round is one pass over the kept keys: four lanes share a key (each a
// quarter of the columns, and of every 32 pool slots a class of 8); the key's
// value row and its scalars are read one iteration ahead.  Regrouped, D_ij =
// A_i + B_j + p_i (h_j + k_j C_ij) with per-key A_i and per-slot B_j, h_j, k_j,
// so with m_i >= max_j p_j C_ij over a class (kept per key and class, raised
// when a slot of it changes) no pair of the key with that class scores below
//   (A_i + min_j B_j + p_i min_j h_j - 2 P^2 p_i m_i) / (P - p_i + min_j p_j)^2,
// min_j B_j over the class too.  A lane whose bound lies above the least score
// that it or the block has found is done after the two products; the few others
// (one key in a hundred and fewer on the measured rows) score their pairs from
// the table.  Each lane decides for itself, and nothing in the scoring names
// another lane.  (One bound over all slots, the key's lanes deciding together:
// 512 rows of 32,768 keys 20.8 ms, now 20.1, 3,072 GQA rows 6.13 and 5.65: a key
// of little weight that leaves becomes a slot with a small B_j, and loosens its
// own class only.)  The least score wins; among pairs at that score the smallest
// (i, j), except that two positions of one lane at exactly the same fp32 score
// keep the first: such pairs are tied to ~1e-7 relative, a decision no fp32
// evaluation can settle.
//
// A key that holds most of the kept mass (P' could fall below P / 4) is scored
// after the pass by the whole block from g' = g - u_i + u_j, the columns split
// over the warps, a lane per slot; at most one key of a round qualifies.
//
// Bound: on long rows the reads of value rows and scalars through the SM's L2
// port (~290 bytes per kept key and round at d = 128) and the products' shared
// reads; on short rows the latency of a round's barriers.  Scoring every key's E
// pairs in every round (408 bytes per key) took, with the gap call, 30.2 ms on
// 512 rows of 32,768 keys with three budgets and 9.4 ms on 3,072 GQA rows of
// 1,000 to 8,192 keys; now 20.1 and 5.65 ms.
#include <algorithm>
#include <climits>

#include "fw_internal.h"

namespace fw {
namespace {

constexpr int SWT = 256;     // threads per block
constexpr int SWW = SWT / 32;  // warps per block
constexpr int SWMAXE = kLongSwapMaxE;  // largest pool size E
constexpr int TK = 2;        // kept keys per thread in the first-round product tile
constexpr int TS = 8;        // pool slots per thread in that tile (4 threads cover 32)
constexpr int QL = 4;        // lanes per kept key in the round pass
constexpr int KPI = SWT / QL;  // kept keys per block iteration of the pass
// resident blocks per SM: three for rows up to 8,192 keys (short rounds, whose
// fixed per-round costs want more blocks), two above and for d = 256 (the
// registers hold the next key's value row and the table tiles)
constexpr int LS_BPS_SHORT = 3, LS_BPS_LONG = 2, LS_LONG_N = 8192;
inline int ls_bps(const RowsDev &R) { return R.max_n > LS_LONG_N || R.d > 128 ? LS_BPS_LONG : LS_BPS_SHORT; }

struct LSArgs {
    RowsDev R;
    const int32_t *k;
    int nb;
    const uint32_t *thr_key;
    const int32_t *thr_idx;
    const float *o;
    const float *row_max;
    const float *row_sum;
    int E, Ep, max_swaps;
    int32_t *n_swaps, *swap_out, *swap_in, *capped;
    float *refined_gap, *topk_gap;
    // per-block scratch, each [gridDim.x][max_n]
    float *ebuf;     // single-key error^2 of every key
    int32_t *kbuf;   // key at each position of the current kept list
    float *pbuf;     // its mass
    float *xbuf;     // its |w|^2
    float *mbuf;     // its bounds on max_j p_j C_ij, by lane class: [4] each
    uint32_t *kebuf; // order key of every dropped key's error (0: kept)
    // per-block cross-product table, [gridDim.x][Ep][cstride] (slot-major)
    float *cbuf;
    int cstride;     // positions per block table (max_n rounded up to a multiple of 4)
};

// (red: SWW floats that nothing else uses until the next barrier)
__device__ __forceinline__ float block_sum(float v, float *red)
{
    v = warp_sum(v);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
    __syncthreads();
    float t = 0.f;
    for (int i = 0; i < SWW; ++i) t += red[i];
    return t;
}

// The fast form divides D (a difference of terms of size ~N P^2) by P'^2, so
// its rounding grows like P^2 / P'^2; it is trusted while P'^2 >= P^2 / 16.
// A swap that removes more of the kept mass is scored from g' = g - u_i + u_j,
// which keeps the cancellation in d-vectors.

// The score from |g'|^2, g' = g - u_i + u_j.
__device__ __forceinline__ float vector_score(float gp2, float P, float p_i, float p_j, float P2, float N)
{
    const float Pp = P + p_j - p_i;
    return gp2 * (P2 / (Pp * Pp)) - N;
}


// Up to 16 sixteen-byte loads of a value row, all issued before any use:
// NV vectors of 8 bf16 or 4 fp32 elements.
template <typename VT, int NV> struct RowChunk;
template <int NV> struct RowChunk<uint16_t, NV> {
    uint4 u[NV];
    __device__ __forceinline__ void load(const uint16_t *p)
    {
#pragma unroll
        for (int i = 0; i < NV; ++i) u[i] = __ldg(reinterpret_cast<const uint4 *>(p) + i);
    }
    __device__ __forceinline__ float at(int c) const  // c is a constant after unrolling
    {
        const uint4 v = u[c >> 3];
        const int e = (c >> 1) & 3;
        const uint32_t w = e == 0 ? v.x : e == 1 ? v.y : e == 2 ? v.z : v.w;
        return (c & 1) ? __uint_as_float(w & 0xffff0000u) : __uint_as_float(w << 16);
    }
};
template <int NV> struct RowChunk<float, NV> {
    float4 u[NV];
    __device__ __forceinline__ void load(const float *p)
    {
#pragma unroll
        for (int i = 0; i < NV; ++i) u[i] = __ldg(reinterpret_cast<const float4 *>(p) + i);
    }
    __device__ __forceinline__ float at(int c) const
    {
        const float4 v = u[c >> 2];
        const int e = c & 3;
        return e == 0 ? v.x : e == 1 ? v.y : e == 2 ? v.z : v.w;
    }
};

static_assert(TK == 2, "the table is written in pairs of positions");
// First round of a budget: C[q][t] = w_{kb[t]} . w_q for every kept position
// t < nk and pool slot q in the 32-slot blocks below nadd.  A thread owns 2
// consecutive positions x 8 slots; the 4 threads of a group cover 32 slots.
// The sum over the d columns runs in column order, as in the later rounds.
template <int DPL, typename VT>
__device__ __forceinline__ void cross_table(const int *kb, int nk, const VT *V, const float *mu, const float *Wt,
                                            int Ep, int nadd, float *cb, int cstride)
{
    constexpr int d = DPL * 32;
    const int sub = threadIdx.x & 3, grp = threadIdx.x >> 2;
    constexpr int GROUPS = SWT / 4;
    for (int base = 0; base < nk; base += GROUPS * TK) {
        const int t0 = base + grp * TK;
        if (t0 >= nk) break;
        const VT *vr[TK];
#pragma unroll
        for (int u = 0; u < TK; ++u) vr[u] = V + (int64_t)kb[t0 + u < nk ? t0 + u : t0] * d;
        for (int q0 = 0; q0 < nadd; q0 += 32) {
            float acc[TK][TS];
#pragma unroll
            for (int u = 0; u < TK; ++u)
#pragma unroll
                for (int s = 0; s < TS; ++s) acc[u][s] = 0.f;
            const float *wq = Wt + q0 + sub * TS;
            // one 16-byte vector per position in flight ahead of the one in use
            constexpr int EPV = 16 / (int)sizeof(VT);
            RowChunk<VT, 1> cur[TK];
#pragma unroll
            for (int u = 0; u < TK; ++u) cur[u].load(vr[u]);
#pragma unroll 1
            for (int c0 = 0; c0 < d; c0 += EPV) {
                RowChunk<VT, 1> nxt[TK];
                const int cn = c0 + EPV < d ? c0 + EPV : c0;
#pragma unroll
                for (int u = 0; u < TK; ++u) nxt[u].load(vr[u] + cn);
#pragma unroll
                for (int m = 0; m < EPV; ++m) {
                    const float mc = mu[c0 + m];
                    const float4 A = *reinterpret_cast<const float4 *>(wq + (c0 + m) * Ep);
                    const float4 B = *reinterpret_cast<const float4 *>(wq + (c0 + m) * Ep + 4);
                    const float ws[TS] = {A.x, A.y, A.z, A.w, B.x, B.y, B.z, B.w};
#pragma unroll
                    for (int u = 0; u < TK; ++u) {
                        const float x = cur[u].at(m) - mc;
#pragma unroll
                        for (int s = 0; s < TS; ++s) acc[u][s] = fmaf(x, ws[s], acc[u][s]);
                    }
                }
#pragma unroll
                for (int u = 0; u < TK; ++u) cur[u] = nxt[u];
            }
            // (TK consecutive positions: cstride and t0 are even, and a write past nk
            // stays inside the slot's row)
#pragma unroll
            for (int h = 0; h < TS; ++h)
                *reinterpret_cast<float2 *>(cb + (size_t)(q0 + sub * TS + h) * cstride + t0) =
                    make_float2(acc[0][h], acc[1][h]);
        }
    }
}

// The 16-byte vectors sub, sub + 4, ... of a value row (4 lanes per row),
// each lane's loads issued before any use.
template <int DPL, typename VT> struct LaneRow {
    static constexpr int EPV = 16 / (int)sizeof(VT);       // elements per vector
    static constexpr int NVL = DPL * 32 / EPV / QL;          // vectors per lane
    RowChunk<VT, 1> u[NVL];
    __device__ __forceinline__ void load(const VT *vr, int sub)
    {
#pragma unroll
        for (int k = 0; k < NVL; ++k) u[k].load(vr + (k * QL + sub) * EPV);
    }
};

// This lane's part of g.w and |w|^2, w = v - mu.
template <int DPL, typename VT>
__device__ __forceinline__ void lane_products(const VT *vr, const float *mu, const float *g, int sub, float &sg,
                                              float &s2)
{
    using L = LaneRow<DPL, VT>;
    L row;
    row.load(vr, sub);
    sg = 0.f;
    s2 = 0.f;
#pragma unroll
    for (int k = 0; k < L::NVL; ++k) {
        const int c0 = (k * QL + sub) * L::EPV;
#pragma unroll
        for (int e = 0; e < L::EPV; ++e) {
            const float w = row.u[k].at(e) - mu[c0 + e];
            sg = fmaf(w, g[c0 + e], sg);
            s2 = fmaf(w, w, s2);
        }
    }
}

// a b + c of two floats at once, each rounded once
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c)
{
    unsigned long long r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;"
        : "=l"(r)
        : "l"(*reinterpret_cast<const unsigned long long *>(&a)), "l"(*reinterpret_cast<const unsigned long long *>(&b)),
          "l"(*reinterpret_cast<const unsigned long long *>(&c)));
    return *reinterpret_cast<float2 *>(&r);
}

// This lane's part of v.g and v.y from its loaded vectors (even and odd columns in
// the halves of a two-float sum).
template <int DPL, typename VT>
__device__ __forceinline__ void lane_products_v_row(const LaneRow<DPL, VT> &row, const float *g, const float *y, int sub,
                                                    float &vg, float &vy)
{
    using L = LaneRow<DPL, VT>;
    float2 sg = make_float2(0.f, 0.f), sy = sg;
#pragma unroll
    for (int k = 0; k < L::NVL; ++k) {
        const int c0 = (k * QL + sub) * L::EPV;
#pragma unroll
        for (int e = 0; e < L::EPV; e += 4) {
            const float4 g4 = *reinterpret_cast<const float4 *>(g + c0 + e);
            const float4 y4 = *reinterpret_cast<const float4 *>(y + c0 + e);
            const float2 va = make_float2(row.u[k].at(e), row.u[k].at(e + 1));
            const float2 vb = make_float2(row.u[k].at(e + 2), row.u[k].at(e + 3));
            sg = fma2(va, make_float2(g4.x, g4.y), sg);
            sy = fma2(va, make_float2(y4.x, y4.y), sy);
            sg = fma2(vb, make_float2(g4.z, g4.w), sg);
            sy = fma2(vb, make_float2(y4.z, y4.w), sy);
        }
    }
    vg = sg.x + sg.y;
    vy = sy.x + sy.y;
}

// NC consecutive elements of a value row as floats, by the widest loads that NC allows.
template <int NC> __device__ __forceinline__ void load_cols(const uint16_t *p, float (&x)[NC])
{
    if constexpr (NC == 1) {
        x[0] = bf16_to_f32(__ldg(p));
    } else {
        uint32_t w[NC / 2];
        if constexpr (NC == 2) {
            w[0] = __ldg(reinterpret_cast<const uint32_t *>(p));
        } else if constexpr (NC == 4) {
            const uint2 u = __ldg(reinterpret_cast<const uint2 *>(p));
            w[0] = u.x, w[1] = u.y;
        } else {
#pragma unroll
            for (int m = 0; m < NC / 8; ++m) {
                const uint4 u = __ldg(reinterpret_cast<const uint4 *>(p) + m);
                w[4 * m] = u.x, w[4 * m + 1] = u.y, w[4 * m + 2] = u.z, w[4 * m + 3] = u.w;
            }
        }
#pragma unroll
        for (int m = 0; m < NC / 2; ++m) {
            x[2 * m] = __uint_as_float(w[m] << 16);
            x[2 * m + 1] = __uint_as_float(w[m] & 0xffff0000u);
        }
    }
}
template <int NC> __device__ __forceinline__ void load_cols(const float *p, float (&x)[NC])
{
    if constexpr (NC == 1) {
        x[0] = __ldg(p);
    } else if constexpr (NC == 2) {
        const float2 u = __ldg(reinterpret_cast<const float2 *>(p));
        x[0] = u.x, x[1] = u.y;
    } else {
#pragma unroll
        for (int m = 0; m < NC; m += 4) {
            const float4 u = __ldg(reinterpret_cast<const float4 *>(p + m));
            x[m] = u.x, x[m + 1] = u.y, x[m + 2] = u.z, x[m + 3] = u.w;
        }
    }
}

// The float of an order key (inverse of order_key).
__device__ __forceinline__ float key_to_float(uint32_t k)
{
    return __uint_as_float((k & 0x80000000u) ? (k & 0x7fffffffu) : ~k);
}

// Score D / P'^2 of one pair in the regrouped fast form: sq = (B_j, k_j, h_j,
// p_j), Ai = A_i, Pm = P - p_i.
__device__ __forceinline__ float fast_score(float4 sq, float cij, float p_i, float Ai, float Pm)
{
    const float Pp = Pm + sq.w;
    return __fdividef(fmaf(p_i, fmaf(sq.y, cij, sq.z), Ai + sq.x), Pp * Pp);
}

template <int DPL, typename VT, int BPS>
__global__ void __launch_bounds__(SWT, BPS) k_long_swap(const LSArgs a)
{
    constexpr int d = DPL * 32;
    const int Ep = a.Ep;         // pool slots, a multiple of 32
    extern __shared__ __align__(16) float sm[];
    float *S = sm;                     // [5][d] band sums of p v
    float *mu = S + 5 * d;             // [d]
    float *o = mu + d;                 // [d]   dense output given by the caller
    float *g = o + d;                  // [d]
    float *wdep = g + d;               // [d]   w of the key that left A last (its pool slot's column)
    float *wtmp = wdep + d;            // [d]   w of the key that entered A last
    float *Wt = wtmp + d;              // [d][Ep] pool vectors w_j, slot-major inner
    // per-round slot terms of the regrouped score: B_j, k_j, h_j, p_j ([Ep] each)
    float *sB = Wt + d * Ep, *sK = sB + Ep, *sH = sK + Ep, *sP = sH + Ep;
    float *xj = sP + Ep;               // [Ep] |w_j|^2 of the slots
    int *idxj = reinterpret_cast<int *>(xj + Ep);  // [Ep] keys in the slots
    float *partA = reinterpret_cast<float *>(idxj + Ep);  // [SWW][Ep] column sums by warp
    float *partB = partA + SWW * Ep;   // [SWW][Ep]
    float *mass = partB + SWW * Ep;    // [8]
    __shared__ TopmSmem s_top;
    __shared__ float red[SWW], red2[SWW];
    __shared__ int s_cnt, s_bt, s_bq, s_heavy;
    __shared__ float s_gm, s_ym, s_pmin, s_pmax, s_Bmin[QL], s_hsg;
    __shared__ uint32_t s_ub;          // order key of the least score found in the round
    __shared__ unsigned long long s_bkey;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int gq = tid / QL, sub = tid % QL;  // key group and lane within it
    const size_t boff = (size_t)blockIdx.x * a.R.max_n;
    float *eb = a.ebuf + boff;
    int *kb = a.kbuf + boff;
    float *pk = a.pbuf + boff;
    float *xk = a.xbuf + boff;
    float *mk = a.mbuf + boff * QL;
    uint32_t *ke = a.kebuf + boff;
    const int cs = a.cstride;
    float *cb = a.cbuf + (size_t)blockIdx.x * Ep * cs;  // [Ep][cs]
    const int nb = a.nb, MS = a.max_swaps;

    for (int64_t row = blockIdx.x; row < a.R.rows; row += gridDim.x) {
        const int64_t grp_i = row / a.R.R;
        const int64_t ri = row - grp_i * a.R.R;
        const int n = a.R.n[grp_i];
        const float *lg = a.R.logits + a.R.logit_off[grp_i] + ri * n;
        const VT *V = reinterpret_cast<const VT *>(a.R.v) + a.R.v_off[grp_i];
        const float M = a.row_max[row];
        const float Zi = 1.f / a.row_sum[row];
        uint32_t tk[4];
        int ti[4];
        for (int b = 0; b < 4; ++b) {
            tk[b] = b < nb ? a.thr_key[row * nb + b] : 0u;
            ti[b] = b < nb ? a.thr_idx[row * nb + b] : -1;
        }
        for (int i = tid; i < d; i += SWT) o[i] = a.o[row * d + i];
        for (int i = tid; i < 5 * d; i += SWT) S[i] = 0.f;
        if (tid < 8) mass[tid] = 0.f;
        __syncthreads();
        // ---- one pass: band sums, band masses, single-key errors of every key
        {
            // lane l holds the DPL columns from l DPL (one vector load per key)
            float acc[5][DPL];
            float macc[5], ol[DPL];
#pragma unroll
            for (int t = 0; t < DPL; ++t) ol[t] = o[lane * DPL + t];
#pragma unroll
            for (int b = 0; b < 5; ++b) {
                macc[b] = 0.f;
#pragma unroll
                for (int t = 0; t < DPL; ++t) acc[b][t] = 0.f;
            }
            // 16 consecutive keys per warp and step: lanes l and l + 16 find the
            // mass and band of key j0 + (l mod 16); then the warp walks the 16
            // value rows (lane = columns), and the 16 partial |v_j - o|^2 are summed
            // by a transposed butterfly (lane l ends with key j0 + (l mod 16))
            constexpr int KS = 16;
            for (int j0 = wid * KS; j0 < n; j0 += SWW * KS) {
                const int jl = j0 + (lane & (KS - 1));
                float pl = 0.f;
                int bl = 0;
                if (jl < n) {
                    const float x = lg[jl];
                    pl = expf(x - M) * Zi;
                    const uint32_t key = order_key(x);
                    for (int b = 0; b < nb; ++b) bl += !(key > tk[b] || (key == tk[b] && jl <= ti[b]));
                }
#pragma unroll
                for (int b = 0; b < 5; ++b) macc[b] += lane < KS && bl == b ? pl : 0.f;
                float dd[KS];
#pragma unroll
                for (int u0 = 0; u0 < KS; u0 += 8) {
                    float v[8][DPL];
#pragma unroll
                    for (int u = 0; u < 8; ++u) {
                        const int j = j0 + u0 + u < n ? j0 + u0 + u : j0;
                        load_cols<DPL>(V + (int64_t)j * d + lane * DPL, v[u]);
                    }
#pragma unroll
                    for (int u = 0; u < 8; ++u) {
                        const float p = __shfl_sync(FW_FULL, pl, u0 + u);  // 0 past the row's end
                        const int band = __shfl_sync(FW_FULL, bl, u0 + u);
                        // band is the same for the whole warp: one accumulator set is touched
#pragma unroll
                        for (int b = 0; b < 5; ++b)
                            if (b == band) {
#pragma unroll
                                for (int t = 0; t < DPL; ++t) acc[b][t] = fmaf(p, v[u][t], acc[b][t]);
                            }
                        float dist = 0.f;
#pragma unroll
                        for (int t = 0; t < DPL; ++t) {
                            const float w = v[u][t] - ol[t];
                            dist = fmaf(w, w, dist);
                        }
                        dd[u0 + u] = dist;
                    }
                }
                // transposed butterfly: the step with offset h leaves lane l the
                // keys whose bit h equals lane bit h; after h = 1 it holds key
                // l mod 16, and the last step adds the other half of the columns
#pragma unroll
                for (int h = KS / 2; h >= 1; h >>= 1) {
                    const bool up = lane & h;
#pragma unroll
                    for (int u = 0; u < h; ++u) {
                        const float send = up ? dd[u] : dd[u + h];
                        const float keep = up ? dd[u + h] : dd[u];
                        dd[u] = keep + __shfl_xor_sync(FW_FULL, send, h);
                    }
                }
                dd[0] += __shfl_xor_sync(FW_FULL, dd[0], KS);
                if (jl < n && lane < KS) eb[jl] = pl * pl * dd[0];  // single-key error squared
            }
#pragma unroll
            for (int b = 0; b < 5; ++b) {
#pragma unroll
                for (int t = 0; t < DPL; ++t) atomicAdd(&S[b * d + lane * DPL + t], acc[b][t]);
                macc[b] = warp_sum(macc[b]);
                if (lane == 0) atomicAdd(&mass[b], macc[b]);
            }
        }
        __syncthreads();
        for (int c = tid; c < d; c += SWT) {
            float m = 0.f;
            for (int b = 0; b < 5; ++b) m += S[b * d + c];
            mu[c] = m;
        }
        __syncthreads();

        for (int b = 0; b < nb; ++b) {
            const int64_t rb = row * nb + b;
            const int kbud = a.k[rb];
            int sb = 0;
            for (int b2 = 0; b2 < nb; ++b2) {
                const int k2 = a.k[row * nb + b2];
                sb += (k2 < kbud) || (k2 == kbud && b2 < b);
            }
            if (kbud < 1 || kbud > n) {
                if (tid == 0) {
                    a.n_swaps[rb] = 0;
                    a.refined_gap[rb] = __int_as_float(0x7fc00000);
                    if (a.topk_gap) a.topk_gap[rb] = __int_as_float(0x7fc00000);
                    if (a.capped) a.capped[rb] = 0;
                }
                for (int t = tid; t < MS; t += SWT) a.swap_out[rb * MS + t] = a.swap_in[rb * MS + t] = -1;
                continue;
            }
            // g, P, N for the top-k set; kept-key list
            float P = 0.f, Pb = 0.f;
            for (int q = 0; q < 5; ++q) {
                if (q <= sb) P += mass[q];
                else Pb += mass[q];
            }
            float gl = 0.f;
            for (int c = tid; c < d; c += SWT) {
                float NA = 0.f, NC = 0.f;
                for (int q = 0; q < 5; ++q) {
                    if (q <= sb) NA += S[q * d + c];
                    else NC += S[q * d + c];
                }
                g[c] = Pb * NA - P * NC;
                gl = fmaf(g[c], g[c], gl);
            }
            if (tid == 0) s_cnt = 0;
            float N = block_sum(gl, red);
            const uint32_t T = tk[b];
            const int TI = ti[b];
            // (four keys per thread and step: independent loads)
            for (int j0 = 0; j0 < n; j0 += 4 * SWT) {
                float x[4];
                uint32_t er[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const int j = j0 + u * SWT + tid;
                    x[u] = j < n ? lg[j] : 0.f;
                    er[u] = j < n ? __float_as_uint(eb[j]) : 0u;
                }
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const int j = j0 + u * SWT + tid;
                    const uint32_t key = order_key(x[u]);
                    const bool kept = j < n && (key > T || (key == T && j <= TI));
                    if (j < n) ke[j] = kept ? 0u : er[u] + 1u;
                    const uint32_t bal = __ballot_sync(FW_FULL, kept);
                    int base = 0;
                    if (lane == 0 && bal) base = atomicAdd(&s_cnt, __popc(bal));
                    base = __shfl_sync(FW_FULL, base, 0);
                    if (kept) kb[base + __popc(bal & ((1u << lane) - 1u))] = j;
                }
            }
            __syncthreads();
            const int nk = s_cnt;
            if (tid == 0 && a.topk_gap) a.topk_gap[rb] = sqrtf(N) / P;
            // ---- pool extras: the E dropped keys of largest error (kept keys rank
            // below every dropped one; equal errors: lower index)
            const int ndrop = n - kbud;
            const int Eeff = a.E < ndrop ? a.E : ndrop;
            int nadd = 0;
            if (Eeff > 0) {
                auto ekey = [&](int j) { return ke[j]; };
                uint32_t eT = 0u;
                int eL = -1;
                block_topm(n, Eeff, ekey, s_top, eT, eL);
                if (tid == 0) s_cnt = 0;
                __syncthreads();
                for (int j0 = tid; j0 < n; j0 += 4 * SWT) {
                    uint32_t e[4];
#pragma unroll
                    for (int u = 0; u < 4; ++u) e[u] = j0 + u * SWT < n ? ekey(j0 + u * SWT) : 0u;
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        const int j = j0 + u * SWT;
                        if (j < n && (e[u] > eT || (e[u] == eT && j <= eL))) {
                            const int q = atomicAdd(&s_cnt, 1);
                            if (q < Ep) idxj[q] = j;
                        }
                    }
                }
                nadd = Eeff;
                __syncthreads();
            }
            // stage the pool: w_j = v_j - mu in slots [0, nadd), zeros above
            for (int e = tid; e < d * Ep; e += SWT) {
                const int c = e / Ep, q = e - c * Ep;
                Wt[e] = q < nadd ? load_v(V, (int64_t)idxj[q] * d + c) - mu[c] : 0.f;
            }
            for (int q = tid; q < Ep; q += SWT) {
                sP[q] = q < nadd ? expf(lg[idxj[q]] - M) * Zi : 0.f;
                if (q >= nadd) {
                    idxj[q] = -1;
                    sB[q] = INFINITY;
                    sK[q] = sH[q] = 0.f;
                }
            }
            __syncthreads();

            int taken = 0, cap = 0;
            bool first = true;
            int tprev = -1, qprev = -1;  // position that entered and slot that changed last round
            float pdep = 0.f;              // mass of the key that left
            for (;;) {
                if (nadd == 0 || nk == 0) break;
                const float P2 = P * P;
                // ---- sums over the columns for every slot: g.w_j, and in the first
                // round |w_j|^2, later the entered key's row of the table (warps
                // split the columns, lanes take the slots of a 32-slot block)
                {
                    constexpr int CPW = d / SWW;
                    for (int q0 = 0; q0 < nadd; q0 += 32) {
                        const int q = q0 + lane;
                        float sg = 0.f, s2 = 0.f;
#pragma unroll
                        for (int e = 0; e < CPW; ++e) {
                            const int c = wid * CPW + e;
                            const float w = Wt[c * Ep + q];
                            sg = fmaf(g[c], w, sg);
                            s2 = fmaf(first ? w : wtmp[c], w, s2);
                        }
                        partA[wid * Ep + q] = sg;
                        partB[wid * Ep + q] = s2;
                    }
                }
                if (wid == 1) {  // mu.g and mu.(changed slot's vector)
                    float a1 = 0.f, a2 = 0.f;
                    for (int c = lane; c < d; c += 32) {
                        a1 = fmaf(mu[c], g[c], a1);
                        a2 = fmaf(mu[c], wdep[c], a2);
                    }
                    a1 = warp_sum(a1);
                    a2 = warp_sum(a2);
                    if (lane == 0) {
                        s_gm = a1;
                        s_ym = a2;
                    }
                }
                if (first) cross_table<DPL, VT>(kb, nk, V, mu, Wt, Ep, nadd, cb, cs);
                __syncthreads();
                if (wid == 0) {
                    float pm = INFINITY, px = 0.f, Bm = INFINITY;
                    for (int q = lane; q < nadd; q += 32) {
                        float sg = 0.f, s2 = 0.f;
#pragma unroll
                        for (int w = 0; w < SWW; ++w) {
                            sg += partA[w * Ep + q];
                            s2 += partB[w * Ep + q];
                        }
                        if (first) xj[q] = s2;
                        else cb[(size_t)q * cs + tprev] = s2;
                        const float p = sP[q];
                        // D_ij = A_i + B_j + p_i (h_j + k_j C_ij) (the file comment's D regrouped)
                        const float B = (p * p * xj[q] + 2.f * p * sg) * P2 - N * p * fmaf(2.f, P, p);
                        sB[q] = B;
                        sK[q] = -2.f * P2 * p;
                        sH[q] = 2.f * N * p;
                        pm = fminf(pm, p);
                        px = fmaxf(px, p);
                        Bm = fminf(Bm, B);
                    }
                    pm = warp_min(pm);
                    px = warp_max(px);
                    // (slot q belongs to class (q / 8) % 4, the lane of a key that holds it)
#pragma unroll
                    for (int o = 1; o < 8; o <<= 1) Bm = fminf(Bm, __shfl_xor_sync(FW_FULL, Bm, o));
                    if ((lane & 7) == 0) s_Bmin[lane >> 3] = Bm;
                    if (lane == 0) {
                        s_pmin = pm;
                        s_pmax = px;
                        s_heavy = -1;
                        s_ub = order_key(0.f);  // only scores below 0 are swaps
                        s_bkey = ~0ull;
                    }
                }
                __syncthreads();
                // ---- one pass over the kept keys.  Each lane keeps the least of its
                // scores, with the pair's position and slot.
                float lmin = INFINITY;
                int lt = -1, li = 0, lq = 0;
                const float pmin = s_pmin, Bmin = s_Bmin[sub], hmin = 2.f * N * pmin, hmax = 2.f * N * s_pmax;
                // position t, key i: this lane's pairs, unless their bound excludes them
                auto score_key = [&](int t, int i, float sg, float sn, float p_i, float x2, float mx, bool scan) {
                    const float alpha = p_i * p_i * x2 - 2.f * p_i * sg;
                    const float Ai = alpha * P2 + N * p_i * (2.f * P - p_i);
                    const float Pm = P - p_i;
                    const float Pl = Pm + pmin;
                    if (16.f * Pl * Pl < P2) {  // some pair needs the vector form: after the pass
                        if (sub == 0) {
                            s_heavy = t;
                            s_hsg = sg;
                        }
                        return;
                    }
                    if (8 * sub >= nadd) return;  // no slots
                    const float ub = key_to_float(*(volatile uint32_t *)&s_ub);
                    const float cmx = 2.f * P2 * p_i * mx;
                    const float lb = (Ai + Bmin) + (p_i * hmin - cmx);
                    const float slack = 4e-6f * (fabsf(Ai) + fabsf(Bmin) + p_i * hmax + fabsf(cmx));  // its rounding
                    if (!scan && lb - slack > fminf(ub, lmin) * (Pl * Pl)) return;
                    float kmin = INFINITY, kc = -INFINITY;
                    int kq = 0;
                    for (int q0 = 0; q0 < nadd; q0 += 32) {
                        const int qb = q0 + 8 * sub;  // this lane's 8 consecutive slots (B_j = inf past nadd)
                        float cq[8], sc[8];
#pragma unroll
                        for (int m = 0; m < 8; ++m) cq[m] = qb + m < nadd ? cb[(size_t)(qb + m) * cs + t] : 0.f;
                        if (t != tprev) {
#pragma unroll
                            for (int m = 0; m < 8; ++m)
                                if (qb + m == qprev) cq[m] = sn;
                        }
                        float k8 = INFINITY;
#pragma unroll
                        for (int h = 0; h < 8; h += 4) {
                            const float4 B4 = *reinterpret_cast<const float4 *>(sB + qb + h);
                            const float4 K4 = *reinterpret_cast<const float4 *>(sK + qb + h);
                            const float4 H4 = *reinterpret_cast<const float4 *>(sH + qb + h);
                            const float4 P4 = *reinterpret_cast<const float4 *>(sP + qb + h);
                            sc[h] = fast_score(make_float4(B4.x, K4.x, H4.x, P4.x), cq[h], p_i, Ai, Pm);
                            sc[h + 1] = fast_score(make_float4(B4.y, K4.y, H4.y, P4.y), cq[h + 1], p_i, Ai, Pm);
                            sc[h + 2] = fast_score(make_float4(B4.z, K4.z, H4.z, P4.z), cq[h + 2], p_i, Ai, Pm);
                            sc[h + 3] = fast_score(make_float4(B4.w, K4.w, H4.w, P4.w), cq[h + 3], p_i, Ai, Pm);
                            kc = fmaxf(kc, fmaxf(fmaxf(P4.x * cq[h], P4.y * cq[h + 1]), fmaxf(P4.z * cq[h + 2], P4.w * cq[h + 3])));
                            k8 = fminf(k8, fminf(fminf(sc[h], sc[h + 1]), fminf(sc[h + 2], sc[h + 3])));
                        }
                        if (k8 < lmin && k8 <= kmin) {
                            // equal scores of one key: the smaller pool key
#pragma unroll
                            for (int m = 0; m < 8; ++m)
                                if (sc[m] == k8 && (k8 < kmin || idxj[qb + m] < idxj[kq])) {
                                    kmin = k8;
                                    kq = qb + m;
                                }
                        }
                    }
                    mk[QL * t + sub] = kc;
                    if (kmin < lmin) {  // first position of the lane's least score
                        lmin = kmin;
                        lt = t;
                        li = i;
                        lq = kq;
                        if (kmin < ub) atomicMin(&s_ub, order_key(kmin));
                    }
                };
                if (first) {
                    for (int t0 = 0; t0 < nk; t0 += KPI) {
                        const int t = t0 + gq;
                        const bool valid = t < nk;
                        const int i = kb[valid ? t : t0];
                        const VT *vr = V + (int64_t)i * d;
                        float sg, sn;  // g.w_i and |w_i|^2 from w itself
                        lane_products<DPL, VT>(vr, mu, g, sub, sg, sn);
                        sg += __shfl_xor_sync(FW_FULL, sg, 1);
                        sn += __shfl_xor_sync(FW_FULL, sn, 1);
                        sg += __shfl_xor_sync(FW_FULL, sg, 2);
                        sn += __shfl_xor_sync(FW_FULL, sn, 2);
                        const float p_i = expf(lg[i] - M) * Zi;
                        if (!valid) continue;
                        if (sub == 0) {
                            pk[t] = p_i;
                            xk[t] = sn;
                        }
                        mk[QL * t + sub] = INFINITY;
                        score_key(t, i, sg, sn, p_i, sn, INFINITY, true);
                    }
                } else {
                    // software pipeline: the value row and scalars of the next iteration and
                    // the kept index of the one after are in flight during this one
                    const float gm = s_gm, ym = s_ym;
                    const int niter = (nk + KPI - 1) / KPI;
                    float *col = cb + (size_t)qprev * cs;
                    const int tf = gq < nk ? gq : nk - 1;
                    int i_cur = kb[tf];
                    int i_next = kb[gq + KPI < nk ? gq + KPI : nk - 1];
                    LaneRow<DPL, VT> row;
                    row.load(V + (int64_t)i_cur * d, sub);
                    float p_i = pk[tf], x2 = xk[tf], m0 = mk[QL * tf + sub];
                    const bool mine = (qprev >> 3 & (QL - 1)) == sub;  // the changed slot is of this lane's class
                    for (int it = 0; it < niter; ++it) {
                        const int t = it * KPI + gq;
                        const int tn = t + KPI < nk ? t + KPI : nk - 1;
                        const float p_n = pk[tn], x2_n = xk[tn], m_n = mk[QL * tn + sub];
                        LaneRow<DPL, VT> rown;
                        rown.load(V + (int64_t)i_next * d, sub);
                        const int tnn = t + 2 * KPI;
                        const int i_nn = kb[tnn < nk ? tnn : nk - 1];
                        float sg, sn;  // v_i.g and v_i . (the changed slot's vector)
                        lane_products_v_row<DPL, VT>(row, g, wdep, sub, sg, sn);
                        sg += __shfl_xor_sync(FW_FULL, sg, 1);
                        sn += __shfl_xor_sync(FW_FULL, sn, 1);
                        sg += __shfl_xor_sync(FW_FULL, sg, 2);
                        sn += __shfl_xor_sync(FW_FULL, sn, 2);
                        if (t < nk) {
                            sn -= ym;
                            if (t != tprev) {
                                if (sub == 0) col[t] = sn;
                                if (mine && pdep * sn > m0) {
                                    m0 = pdep * sn;
                                    mk[QL * t + sub] = m0;
                                }
                            }
                            score_key(t, i_cur, sg - gm, sn, p_i, x2, m0, false);
                        }
                        row = rown;
                        i_cur = i_next;
                        i_next = i_nn;
                        p_i = p_n;
                        x2 = x2_n;
                        m0 = m_n;
                    }
                }
                first = false;
                __syncthreads();
                const int th = s_heavy;
                if (th >= 0) {  // (uniform) the heavy key's pairs: |g - u_i + u_j|^2, warps split the columns
                    constexpr int CPW = d / SWW;
                    const int ih = kb[th];
                    const float p_i = pk[th];
                    for (int q0 = 0; q0 < nadd; q0 += 32) {
                        const int q = q0 + lane;
                        const float p_j = sP[q];
                        float gv = 0.f;
#pragma unroll
                        for (int e = 0; e < CPW; ++e) {
                            const int c = wid * CPW + e;
                            const float wi = load_v(V, (int64_t)ih * d + c) - mu[c];
                            const float gp = fmaf(p_j, Wt[c * Ep + q], fmaf(-p_i, wi, g[c]));
                            gv = fmaf(gp, gp, gv);
                        }
                        partA[wid * Ep + q] = gv;
                    }
                    __syncthreads();
                    if (wid == 0) {
                        const float alpha = p_i * p_i * xk[th] - 2.f * p_i * s_hsg;
                        const float Ai = alpha * P2 + N * p_i * (2.f * P - p_i);
                        const float Pm = P - p_i;
                        for (int q = lane; q < nadd; q += 32) {
                            float gv = 0.f;
#pragma unroll
                            for (int w = 0; w < SWW; ++w) gv += partA[w * Ep + q];
                            const float Pp = Pm + sP[q];
                            const float sc = 16.f * Pp * Pp >= P2
                                                 ? fast_score(make_float4(sB[q], sK[q], sH[q], sP[q]),
                                                              cb[(size_t)q * cs + th], p_i, Ai, Pm)
                                                 : vector_score(gv, P, p_i, sP[q], P2, N);
                            if (sc < lmin || (sc == lmin && (ih < li || (ih == li && idxj[q] < idxj[lq])))) {
                                lmin = sc;
                                lt = th;
                                li = ih;
                                lq = q;
                            }
                        }
                    }
                }
                // the block's least score; the smallest (i, j) among the lanes that hold it
                {
                    const float wb = warp_min(lmin);
                    if (lane == 0) red[wid] = wb;
                }
                __syncthreads();
                float bmin = INFINITY;
                for (int w = 0; w < SWW; ++w) bmin = fminf(bmin, red[w]);
                if (!(bmin < 0.f)) break;  // no pair strictly decreases es (uniform)
                if (taken >= MS) {
                    cap = 1;
                    break;
                }
                const unsigned long long mykey = ((unsigned long long)(uint32_t)li << 32) | (uint32_t)idxj[lq];
                const bool mine = lt >= 0 && lmin == bmin;
                if (mine) atomicMin(&s_bkey, mykey);
                __syncthreads();
                if (mine && mykey == s_bkey) {
                    s_bt = lt;
                    s_bq = lq;
                }
                __syncthreads();
                // apply: g += u_j - u_i, P += p_j - p_i; slot qj of the pool takes i
                const unsigned long long bk = s_bkey;
                const int bi = (int)(bk >> 32), bj = (int)(bk & 0xffffffffu);
                const int tb = s_bt, qj = s_bq;
                const float p_i = pk[tb], x_i = xk[tb];
                const float p_j = sP[qj], x_j = xj[qj];
                float gl2 = 0.f;
                for (int c = tid; c < d; c += SWT) {
                    const float wi = load_v(V, (int64_t)bi * d + c) - mu[c];
                    const float wj = Wt[c * Ep + qj];
                    const float gn = g[c] + p_j * wj - p_i * wi;
                    g[c] = gn;
                    wdep[c] = wi;
                    wtmp[c] = wj;
                    Wt[c * Ep + qj] = wi;
                    gl2 = fmaf(gn, gn, gl2);
                }
                P = P - p_i + p_j;
                N = block_sum(gl2, red2);  // (its barrier ends every read above)
                if (tid < QL) mk[QL * tb + tid] = INFINITY;
                if (tid == 0) {
                    idxj[qj] = bi;
                    sP[qj] = p_i;
                    xj[qj] = x_i;
                    kb[tb] = bj;
                    pk[tb] = p_j;
                    xk[tb] = x_j;
                    a.swap_out[rb * MS + taken] = bi;
                    a.swap_in[rb * MS + taken] = bj;
                }
                pdep = p_i;
                tprev = tb;
                qprev = qj;
                ++taken;
            }
            if (tid == 0) {
                a.n_swaps[rb] = taken;
                a.refined_gap[rb] = sqrtf(N) / P;
                if (a.capped) a.capped[rb] = cap;
            }
            for (int t = taken + tid; t < MS; t += SWT) a.swap_out[rb * MS + t] = a.swap_in[rb * MS + t] = -1;
            __syncthreads();
        }
        __syncthreads();
    }
}

// pool slots rounded up to the 32-slot blocks of the product tile
inline int pool_slots(int E) { return std::max(32, (E + 31) / 32 * 32); }

template <int DPL> size_t ls_smem(int Ep)
{
    constexpr int d = DPL * 32;
    return sizeof(float) * (10 * (size_t)d + (size_t)d * Ep + (6 + 2 * SWW) * (size_t)Ep + 8);
}

}  // namespace

// ls_bps resident blocks per SM (the launch bounds guarantee the registers
// for it); the workspace is sized by the same count, queried from the current device
static unsigned ls_grid(const RowsDev &R)
{
    int sms = 0;
    if (device_sms(&sms) != FW_OK) sms = 152;  // no device: the size query still answers
    return (unsigned)std::min<int64_t>(R.rows, (int64_t)sms * ls_bps(R));
}

static size_t ls_array_bytes(const RowsDev &R) { return align256((size_t)ls_grid(R) * R.max_n * 4); }

static int ls_cstride(const RowsDev &R) { return (R.max_n + 3) / 4 * 4; }

static size_t ls_table_bytes(const RowsDev &R, int E)
{
    return align256((size_t)ls_grid(R) * pool_slots(E) * ls_cstride(R) * 4);
}

size_t long_swap_workspace(const RowsDev &R, int nb, int E, int max_swaps)
{
    (void)nb, (void)max_swaps;
    return ls_array_bytes(R) * (5 + QL) + ls_table_bytes(R, E);
}

fw_status long_swap(const RowsDev &R, const int32_t *k, int nb, const fw_gap_out &topk, int E, int max_swaps,
                    int32_t *n_swaps, int32_t *swap_out, int32_t *swap_in, float *refined_gap, float *topk_gap,
                    int32_t *capped, void *ws, size_t ws_bytes, cudaStream_t s)
{
    (void)ws_bytes;
    if (E > SWMAXE) return FW_ERR_UNSUPPORTED;
    LSArgs a;
    a.R = R;
    a.k = k;
    a.nb = nb;
    a.thr_key = topk.thr_key;
    a.thr_idx = topk.thr_idx;
    a.o = topk.o;
    a.row_max = topk.row_max;
    a.row_sum = topk.row_sum;
    a.E = E;
    a.Ep = pool_slots(E);
    a.max_swaps = max_swaps;
    a.n_swaps = n_swaps;
    a.swap_out = swap_out;
    a.swap_in = swap_in;
    a.capped = capped;
    a.refined_gap = refined_gap;
    a.topk_gap = topk_gap;
    a.cstride = ls_cstride(R);
    const unsigned grid = ls_grid(R);
    const size_t arr = ls_array_bytes(R);
    char *w = (char *)ws;
    a.ebuf = (float *)(w + 0 * arr);
    a.kbuf = (int32_t *)(w + 1 * arr);
    a.pbuf = (float *)(w + 2 * arr);
    a.xbuf = (float *)(w + 3 * arr);
    a.kebuf = (uint32_t *)(w + 4 * arr);
    a.mbuf = (float *)(w + 5 * arr);
    a.cbuf = (float *)(w + (5 + QL) * arr);
    FW_DISPATCH(R.d, R.v_dtype, {
        const size_t smem = ls_smem<DPL>(a.Ep);
        constexpr int SHORT = DPL <= 4 ? LS_BPS_SHORT : LS_BPS_LONG;
        auto kern = ls_bps(R) == LS_BPS_LONG ? k_long_swap<DPL, VT, LS_BPS_LONG> : k_long_swap<DPL, VT, SHORT>;
        FW_CUDA_CHECK(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
        FW_LAUNCH(kern, grid, SWT, smem, s, a);
    });
    return FW_OK;
}

}  // namespace fw

// k_pool.cu -- ES_pool (Definition 2.2): the exact best size-s subset of the
// candidate set -- the top-mass set plus the E dropped keys of largest
// single-key error p_j ||v_j - mu|| (ties -> lower index) -- for rows of any
// length up to 49,152 keys and budgets s <= 32 (pools of at most 64 keys).
//
//   k_pool_build  one CTA per row: e_j^2 = p_j^2 ||v_j - o||^2 of every key (o =
//                 the dense output of the gap call; four lanes per key, 16-byte
//                 loads, o in registers), ONE radix select of the m = max(s + E)
//                 largest errors -- a budget's E extras are among the s + E
//                 largest errors of the whole row, since at most s kept keys
//                 can be ahead of them -- and per budget the pool in ascending
//                 key order, ranked among those m and the kept keys by a warp.
//   k_pool_enum   one CTA per (row, budget), below.
//
// Enumeration.  With u = p (v - o), G_xy = u_x . u_y, t the least es^2 known (at
// first the top-mass set's) and a set K of s pool keys (at first the same), a
// size-s subset A = (K \ R) u D has es(A)^2 <= t iff
//   val(A) = |sum_A u|^2 - t p(A)^2 <= 0,
// and val is a quadratic form in the exchanged keys: with H = G - t p p^T and
// h = H 1_K,
//   val(A) = val(K) + sum_R (H_xx - 2 h_x) + sum_D (H_yy + 2 h_y)
//            + 2 sum_{pairs in R} H + 2 sum_{pairs in D} H - 2 sum_{R x D} H.
// val(K) and h come from sum_K u, summed in fp64 (h by double-float products); G is
// plain fp32.  The
// rounding of the whole is at most kappa (e^2 + 2 e b + val(K)), b = |sum_K u|
// + sqrt(t) p(K), e the sum over the exchanged keys of a_x = |u_x| + sqrt(t) p_x
// -- a bound that leaves out the heavy keys both sets share -- and is a
// quadratic form too, so it is folded into the table entries: "computed value
// <= 0" is a necessary condition and costs nothing.  A sweep over the subsets
// collects those that pass, with their values; value and bound give each an
// interval for es^2, the few whose lower end does not exceed the least upper
// end are scored from the value rows in fp64, and the least es wins,
// exact ties to the smallest colex rank of the members' pool positions.  Where
// more than GCAP pass -- rows with good subsets that leave out the attention
// sink, far from the top-mass set, whose values the bound around that set
// cannot tell apart -- the subset of least value becomes K and the sweep is
// repeated around it, with the least es^2 known by then.
//
// A sweep walks |R| = |D| = r = 1 .. min(s, E).  All subsets of the side with
// fewer keys are laid out in groups of 8 (their own value, and W[y][8], their
// cross terms with key y of the other side) in shared memory, in batches where
// they do not fit; lanes take the other side's subsets without their highest
// member and run that member upwards, so a subset costs two additions and a
// minimum.  Bound: instruction issue.
//
// Measured on 256 rows of 4,096 keys, d = 128, s = 4/8/16/32 with E =
// 24/12/6/4 (gap call, build and enumeration): 0.71 ms, against 37 to 250 ms
// (by which rows were drawn) with one warp per item that scored every subset
// from scratch under an error bound of the whole pool's sum |u| and re-scored
// what passed in fp64.  16 warps per block (64 registers) rather than 8: 0.71
// against 0.80 ms, the sweeps wait on shared memory.  Since then fp64 scores instead
// of double-float ones cost 1.2 %, the checks of range 2.1 %.
//
// Rows with a non-finite logit or value have no es to compare and are reported
// before any sweep.  Masses are scaled by a power of two where the largest u is
// far from 1, which changes no es, so that finite rows keep their bounds.
//
// Nothing waits on another block; when sweeping around better sets does not
// bring the hits below GCAP (exact ties by the thousand) the lanes score every
// hit, so the answer stays exact.
#include <algorithm>
#include <cfloat>
#include <climits>

#include "fw_internal.h"

namespace fw {
namespace {

constexpr int PB_T = 256;            // k_pool_build: threads per row
constexpr int PB_Q = 4;              // ... lanes per key
constexpr int PE_T = 512;            // k_pool_enum: threads per (row, budget)
constexpr int PE_NW = PE_T / 32;
constexpr int PE_CH = 8;             // small-side subsets per group
constexpr int PE_WCAP = 5120;        // floats of W: one batch of groups
constexpr int PE_GMAX = 64;          // groups per batch
constexpr int PE_GSPLIT = 16;        // groups per warp task
constexpr int PE_BPS = 2;            // blocks per SM (their shared memory: 104 KB at d = 128)
constexpr int PMAX = 64;             // pool keys
constexpr int PSMAX = 32;            // largest budget
constexpr int PCAND = PMAX + PSMAX;  // keys k_pool_build gathers: largest errors and kept keys
constexpr int PB_STAGE_MAX = 49152;  // keys per row staged in shared memory
constexpr int GCAP = 512;            // re-scoring candidates buffered per block
constexpr int PE_SURV = 32;           // survivors that another sweep may cut
constexpr int PE_SWEEPS = 8;         // sweeps before the lanes score every candidate
constexpr uint64_t PE_MAX_SUBSETS = 1ull << 32;
constexpr int CLD = PMAX + 1;        // table row stride (odd: conflict-free columns)
constexpr float PE_TINY = 1e-36f;    // slack for subnormal table entries
constexpr int PE_XMASS = 90;         // largest scale of the masses, as an exponent

// C(a, b) for a <= 64, b <= 32 (all below 2^63), by Pascal's rule at compile time.
struct Binom64Table {
    uint64_t v[65][33];
};
constexpr Binom64Table make_binom64()
{
    Binom64Table t{};
    for (int a = 0; a <= 64; ++a) {
        t.v[a][0] = 1;
        for (int b = 1; b <= 32; ++b) t.v[a][b] = a == 0 ? 0 : t.v[a - 1][b - 1] + t.v[a - 1][b];
    }
    return t;
}
static __constant__ Binom64Table c_b64 = make_binom64();  // warp-uniform reads
static __device__ const Binom64Table g_b64 = make_binom64();  // reads that differ by lane

__device__ __forceinline__ uint64_t cb(int a, int b) { return (b < 0 || b > 32 || a < b) ? 0 : c_b64.v[a][b]; }
__device__ __forceinline__ uint64_t cbl(int a, int b) { return (b > 32 || a < b) ? 0 : __ldg(&g_b64.v[a][b]); }

struct PoolArgs {
    RowsDev R;
    const int32_t *k;          // [rows][nb]
    int nb;
    int E[4];                  // extras of each budget slot
    const uint32_t *thr_key;   // [rows][nb] from the gap call
    const int32_t *thr_idx;
    const float *o, *M, *Z;    // [rows][d], [rows], [rows]
    int32_t *pool;             // ws [rows][nb][PMAX] ascending key indices
    int32_t *pool_n;           // ws [rows][nb] pool size; -1 invalid budget, -2 pool too large, -3 a logit
                               // of the row is not finite
    float *best_gap;           // [rows][nb]
    int32_t *best_idx;         // [rows][nb][k_max]
    int k_max;
    float *topk_gap;           // [rows][nb] or null
    int32_t *row_status;       // [rows] or null
    int64_t *n_cand;           // [rows][nb] re-scored subsets, or null
};

// ------------------------------------------------------------ the pool

// This lane's quarter of a value row as fp32: the 16-byte vectors sub, sub + 4, ...
template <int DPL, typename VT> struct PoolLane {
    static constexpr int EPV = 16 / (int)sizeof(VT);
    static constexpr int NV = DPL * 32 / EPV / PB_Q;
    uint4 u[NV];
    __device__ __forceinline__ void load(const VT *v, int sub)
    {
#pragma unroll
        for (int q = 0; q < NV; ++q) u[q] = __ldg(reinterpret_cast<const uint4 *>(v + (q * PB_Q + sub) * EPV));
    }
    __device__ __forceinline__ float at(int q, int e) const  // constants after unrolling
    {
        const uint32_t w[4] = {u[q].x, u[q].y, u[q].z, u[q].w};
        if constexpr (sizeof(VT) == 4) return __uint_as_float(w[e]);
        else return __uint_as_float((e & 1) ? (w[e >> 1] & 0xffff0000u) : (w[e >> 1] << 16));
    }
};

template <int DPL, typename VT>
__global__ void __launch_bounds__(PB_T) k_pool_build(PoolArgs a)
{
    extern __shared__ float sm[];
    float *e2 = sm;  // [max_n] single-key errors squared
    __shared__ TopmSmem S;
    __shared__ int32_t c_idx[PCAND];
    __shared__ uint32_t c_err[PCAND], c_log[PCAND];
    __shared__ int s_cnt;
    using L = PoolLane<DPL, VT>;
    constexpr int d = DPL * 32;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int sub = tid % PB_Q, gq = tid / PB_Q;
    constexpr int KPI = PB_T / PB_Q;
    for (int64_t r = blockIdx.x; r < a.R.rows; r += gridDim.x) {
        const int64_t g = r / a.R.R;
        const int n = a.R.n[g];
        const float *l = a.R.logits + a.R.logit_off[g] + (r - g * a.R.R) * n;
        const VT *V = static_cast<const VT *>(a.R.v) + a.R.v_off[g];
        const float M = a.M[r], Zi = 1.f / a.Z[r];
        float so[L::NV * L::EPV];
#pragma unroll
        for (int q = 0; q < L::NV; ++q)
#pragma unroll
            for (int e = 0; e < L::EPV; ++e) so[q * L::EPV + e] = a.o[r * d + (q * PB_Q + sub) * L::EPV + e];
        __syncthreads();  // the previous row's shared arrays are no longer read
        if (tid == 0) s_cnt = 0;
        bool bad = false;  // a logit is not finite
        // two keys in flight per group of four lanes
        for (int j0 = 0; j0 < n; j0 += 2 * KPI) {
            const int ja = j0 + gq, jb = j0 + KPI + gq;
            L ra, rb;
            ra.load(V + (int64_t)min(ja, n - 1) * d, sub);
            rb.load(V + (int64_t)min(jb, n - 1) * d, sub);
            const int jm = sub & 1 ? jb : ja;  // lanes 0 and 1 finish one key each
            const float lj = __ldg(l + min(jm, n - 1));
            bad |= !isfinite(lj);
            const float p = sub < 2 ? __expf(lj - M) * Zi : 0.f;
            float sa = 0.f, sb = 0.f;
#pragma unroll
            for (int q = 0; q < L::NV; ++q)
#pragma unroll
                for (int e = 0; e < L::EPV; ++e) {
                    const float o = so[q * L::EPV + e];
                    const float wa = ra.at(q, e) - o, wb = rb.at(q, e) - o;
                    sa = fmaf(wa, wa, sa);
                    sb = fmaf(wb, wb, sb);
                }
            sa += __shfl_xor_sync(FW_FULL, sa, 1);
            sb += __shfl_xor_sync(FW_FULL, sb, 1);
            sa += __shfl_xor_sync(FW_FULL, sa, 2);
            sb += __shfl_xor_sync(FW_FULL, sb, 2);
            if (sub < 2 && jm < n) e2[jm] = p * p * (sub ? sb : sa);
        }
        const int nonfinite = __syncthreads_or(bad);
        // the budgets: sizes, and the longest prefix of the error order any of them needs
        int m = 0;
        int sb_[4], Eb[4];
        uint32_t tk[4];
        int ti[4];
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            sb_[b] = Eb[b] = -1;
            tk[b] = 0xffffffffu;
            ti[b] = -1;
            if (b >= a.nb) continue;
            const int64_t rb = r * a.nb + b;
            const int s = a.k[rb];
            int no = 0;
            if (s < 1 || s > n || s > PSMAX || s > a.k_max || a.E[b] < 0) no = -1;
            else if (s + min(a.E[b], n - s) > PMAX) no = -2;
            else if (nonfinite) no = -3;
            if (no) {
                if (tid == 0) a.pool_n[rb] = no;
                continue;
            }
            sb_[b] = s;
            Eb[b] = min(a.E[b], n - s);
            tk[b] = a.thr_key[rb];
            ti[b] = a.thr_idx[rb];
            m = max(m, s + Eb[b]);
        }
        if (m == 0) continue;  // (uniform)
        uint32_t T = 0u;
        int Lx = -1;
        block_topm(n, m, [&](int j) { return order_key(e2[j]); }, S, T, Lx);
        // the m largest errors and every budget's kept keys (at most PCAND for
        // thresholds that keep the budgets' counts; more are not listed)
        for (int j = tid; j < n; j += PB_T) {
            const uint32_t u = order_key(e2[j]), kl = order_key(__ldg(l + j));
            bool in = u > T || (u == T && j <= Lx);
#pragma unroll
            for (int b = 0; b < 4; ++b) in |= kl > tk[b] || (kl == tk[b] && j <= ti[b]);
            if (in) {
                const int q = atomicAdd(&s_cnt, 1);
                if (q < PCAND) {
                    c_idx[q] = j;
                    c_err[q] = u;
                    c_log[q] = kl;
                }
            }
        }
        __syncthreads();
        const int nc = s_cnt;
        // a warp per budget: kept keys and the Eb dropped ones of largest error, in key order
        for (int b = wid; b < a.nb; b += PB_T / 32) {
            int s = -1, E = 0, tix = -1;
            uint32_t tkx = 0u;
#pragma unroll
            for (int q = 0; q < 4; ++q)
                if (q == b) s = sb_[q], E = Eb[q], tkx = tk[q], tix = ti[q];
            if (s < 0) continue;
            const int64_t rb = r * a.nb + b;
            if (nc > PCAND) {
                if (lane == 0) a.pool_n[rb] = -2;
                continue;
            }
            constexpr int PER = PCAND / 32;
            uint32_t in[PER];  // ballots over the listed keys
#pragma unroll
            for (int q = 0; q < PER; ++q) {
                const int c = q * 32 + lane;
                bool take = false;
                if (c < nc) {
                    const int j = c_idx[c];
                    const uint32_t u = c_err[c];
                    take = c_log[c] > tkx || (c_log[c] == tkx && j <= tix);
                    if (!take) {
                        int ahead = 0;  // dropped keys before this one in the error order
                        for (int c2 = 0; c2 < nc; ++c2) {
                            const int j2 = c_idx[c2];
                            const bool k2 = c_log[c2] > tkx || (c_log[c2] == tkx && j2 <= tix);
                            ahead += !k2 && (c_err[c2] > u || (c_err[c2] == u && j2 < j));
                        }
                        take = ahead < E;
                    }
                }
                in[q] = __ballot_sync(FW_FULL, take);
            }
            int cnt = 0;
#pragma unroll
            for (int q = 0; q < PER; ++q) cnt += __popc(in[q]);
#pragma unroll
            for (int q = 0; q < PER; ++q) {
                const int c = q * 32 + lane;
                if (!((in[q] >> lane) & 1u)) continue;
                const int j = c_idx[c];
                int pos = 0;
#pragma unroll
                for (int q2 = 0; q2 < PER; ++q2)
                    for (uint32_t w = in[q2]; w; w &= w - 1) pos += c_idx[q2 * 32 + __ffs(w) - 1] < j;
                if (pos < PMAX) a.pool[rb * PMAX + pos] = j;
            }
            if (lane == 0) a.pool_n[rb] = cnt <= PMAX ? cnt : -2;
        }
    }
}

// ------------------------------------------------------------ enumeration

// the m-combination of colex rank `rank` out of 0..P-1 as a bit mask
__device__ __forceinline__ uint64_t colex_unrank(uint64_t rank, int m, int P)
{
    uint64_t A = 0;
    int x = P - 1;
    for (int i = m; i >= 1; --i) {
        if (i == 3) {  // the largest x with C(x, 3) <= rank, from the cube root
            const uint32_t q = (uint32_t)rank;
            uint32_t y = (uint32_t)(cbrtf(6.f * (float)q) + 1.f);
            while (y * (y - 1) * (y - 2) / 6 > q) --y;
            while ((y + 1) * y * (y - 1) / 6 <= q) ++y;
            A |= 1ull << y;
            rank = q - y * (y - 1) * (y - 2) / 6;
            continue;
        }
        if (i == 2) {  // C(x, 2) <= rank
            const uint32_t q = (uint32_t)rank;
            uint32_t y = (uint32_t)((sqrtf(8.f * (float)q + 1.f) + 1.f) * 0.5f);
            while (y * (y - 1) / 2 > q) --y;
            while ((y + 1) * y / 2 <= q) ++y;
            A |= 1ull << y;
            rank = q - y * (y - 1) / 2;
            continue;
        }
        if (i == 1) {
            A |= 1ull << rank;
            break;
        }
        while (x >= i && cbl(x, i) > rank) --x;
        A |= 1ull << x;
        rank -= cbl(x, i);
        --x;
    }
    return A;
}

// colex rank of the set bits of a 64-bit mask (positions ascending)
__device__ __forceinline__ uint64_t colex_rank64(uint64_t A)
{
    uint64_t rank = 0;
    int i = 1;
    for (uint64_t w = A; w; w &= w - 1, ++i) rank += cbl(__ffsll((long long)w) - 1, i);
    return rank;
}

// state of one (row, budget); the value rows v [PMAX][d + 4] follow it
struct EnumSm {
    double QK, PK, rPK, bes;    // |sum_K u|^2, p(K) and its inverse, the least es known
    uint64_t K, topK;           // the set exchanged from; kept keys by the thresholds
    uint64_t bmask, brank;      // the best set known, its colex rank
    uint64_t candD[GCAP];       // hits: the big side's keys exchanged ...
    uint64_t red_rank[PE_NW], red_mask[PE_NW];
    double red_es[PE_NW];
    long long red_seen[PE_NW];
    uint32_t candR[GCAP];       // ... the small side's
    float candV[GCAP];          // ... and the value
    __align__(16) float W[PE_WCAP];  // [group][big key][PE_CH]
    float C[PMAX * CLD];        // table entries, small side's keys first (on the diagonal: one key alone)
    float G[PMAX * CLD];        // u_x . u_y
    uint32_t rmask[PE_GMAX * PE_CH];
    float rbase[PE_GMAX * PE_CH];
    float o[256];
    double UK[256];             // sum over K of u, by column
    float UKh[256], UKl[256];   // ... as double-float, for the products below
    float gh[PMAX], gl[PMAX];   // its products with v_x - o
    float pp[PMAX];             // masses
    float ax[PMAX];             // |u_x| + sqrt(t) p_x, scaled
    int32_t pidx[PMAX];
    int32_t loc[PMAX];          // pool position of a table index
    float red_v[PE_NW];
    int ncand, nsurv, stale;
    uint32_t task;
    // segments of the batch: (r, first group of that r, groups)
    int seg_r[PSMAX], seg_g[PSMAX], seg_n[PSMAX], nseg, next_r, next_g;
};

// columns c + step k (k < NC, below d) of sum over A of p (v - o), in fp64,
// members ascending; the columns are independent chains
template <int NC>
__device__ __forceinline__ void col_sums(const EnumSm &S, const float *v, int d, uint64_t A, int c, int step,
                                         double (&out)[NC])
{
    double o[NC];
#pragma unroll
    for (int k = 0; k < NC; ++k) {
        out[k] = 0.0;
        o[k] = c + step * k < d ? (double)S.o[c + step * k] : 0.0;
    }
    for (uint64_t w = A; w; w &= w - 1) {
        const int x = __ffsll((long long)w) - 1;
        const double p = (double)S.pp[x];
        const float *vx = v + x * (d + 4);
#pragma unroll
        for (int k = 0; k < NC; ++k) {
            const int ck = c + step * k;
            if (ck >= d) break;
            out[k] = fma(p, (double)vx[ck] - o[k], out[k]);
        }
    }
}

__device__ __forceinline__ double mass_warp(const EnumSm &S, uint64_t A, int lane)
{
    return warp_sum_d((((A >> lane) & 1ull) ? (double)S.pp[lane] : 0.0) +
                      (((A >> (lane + 32)) & 1ull) ? (double)S.pp[lane + 32] : 0.0));
}

// es of the pool positions in A, by the definition (the warp together)
__device__ double es_warp(const EnumSm &S, const float *v, int d, uint64_t A, int lane)
{
    double q = 0.0;
    for (int c0 = 0; c0 < d; c0 += 128) {
        double u[4];
        col_sums<4>(S, v, d, A, c0 + lane, 32, u);
#pragma unroll
        for (int k = 0; k < 4; ++k) q = fma(u[k], u[k], q);
    }
    return sqrt(warp_sum_d(q)) / mass_warp(S, A, lane);
}

// the same by one lane alone (the last resort)
__device__ double es_lane(const EnumSm &S, const float *v, int d, uint64_t A)
{
    double q = 0.0, pa = 0.0;
    for (int c = 0; c < d; c += 4) {
        double u[4];
        col_sums<4>(S, v, d, A, c, 1, u);
#pragma unroll
        for (int k = 0; k < 4; ++k) q = fma(u[k], u[k], q);
    }
    for (uint64_t w = A; w; w &= w - 1) pa += (double)S.pp[__ffsll((long long)w) - 1];
    return sqrt(q) / pa;
}

// what a lane carries through a sweep
struct LaneBest {
    bool score;      // score every hit (else: collect hits, keep the least value)
    float least;     // least value and its subset
    uint32_t R;
    uint64_t D;
    uint64_t mask;   // the subset of least es
    double es;
    uint64_t rank;
    int64_t seen;    // subsets scored
};

// the subset that exchanges the small side's keys in R and the big side's in D
__device__ __forceinline__ uint64_t exchanged(const EnumSm &S, int ns, uint32_t R, uint64_t D)
{
    uint64_t A = S.K;
    for (uint32_t w = R; w; w &= w - 1) A ^= 1ull << S.loc[__ffs(w) - 1];
    for (uint64_t w = D; w; w &= w - 1) A ^= 1ull << S.loc[ns + __ffsll((long long)w) - 1];
    return A;
}

// a subset that can reach es^2 = t (rare).  Once the list has overflowed only
// values below the lane's least are looked at: returns the new limit.
__device__ __noinline__ float sweep_hit(EnumSm &S, const float *v, int d, LaneBest &lb, int ns, uint32_t R, uint64_t D,
                                       float val)
{
    if (lb.score) {
        ++lb.seen;
        const uint64_t A = exchanged(S, ns, R, D);
        const double es = es_lane(S, v, d, A);
        const uint64_t rank = colex_rank64(A);
        if (es < lb.es || (es == lb.es && rank < lb.rank)) {
            lb.es = es;
            lb.rank = rank;
            lb.mask = A;
        }
        return PE_TINY;
    }
    if (val < lb.least) {
        lb.least = val;
        lb.R = R;
        lb.D = D;
    }
    const int q = *(volatile int *)&S.ncand > GCAP ? GCAP : atomicAdd(&S.ncand, 1);
    if (q < GCAP) {
        S.candR[q] = R;
        S.candD[q] = D;
        S.candV[q] = val;
        return PE_TINY;
    }
    return lb.least;
}

// The big-side subsets U u {x}, x > max U, against the groups [g0, g1) of a
// segment (first slot of the segment: slot0), NR subsets each but the last
// group's.  RM = |U| (RM = -1: any, members by bit loops).  One: the segment
// has a single group of at most 2 subsets.
template <int RM, bool One>
__device__ __forceinline__ void sweep_run(EnumSm &S, const float *v, int d, LaneBest &lb, float &limit, int ns, int nbg,
                                          uint64_t U, int slot0, int g0, int g1, int nr)
{
    const float *C = S.C + ns * CLD + ns;  // the big side's block
    int um[RM > 0 ? RM : 1];
    float fU = 0.f;
    if constexpr (RM >= 0) {
        uint64_t w = U;
#pragma unroll
        for (int i = 0; i < RM; ++i) {
            um[i] = __ffsll((long long)w) - 1;
            w &= w - 1;
            float f = C[um[i] * CLD + um[i]];
#pragma unroll
            for (int h = 0; h < i; ++h) f += C[um[i] * CLD + um[h]];
            fU += f;
        }
    } else {
        for (uint64_t w = U; w; w &= w - 1) {
            const int y = __ffsll((long long)w) - 1;
            float f = C[y * CLD + y];
            for (uint64_t w2 = U & ((1ull << y) - 1ull); w2; w2 &= w2 - 1) f += C[y * CLD + __ffsll((long long)w2) - 1];
            fU += f;
        }
    }
    const int top = U ? 64 - __clzll((long long)U) : 0;
    auto pairs = [&](int x) {  // key x alone and with U
        float lw = C[x * CLD + x];
        if constexpr (RM >= 0) {
#pragma unroll
            for (int i = 0; i < RM; ++i) lw += C[x * CLD + um[i]];
        } else {
            for (uint64_t w = U; w; w &= w - 1) lw += C[x * CLD + __ffsll((long long)w) - 1];
        }
        return lw;
    };
    auto members = [&](auto &&f) {
        if constexpr (RM >= 0) {
#pragma unroll
            for (int i = 0; i < RM; ++i) f(um[i]);
        } else {
            for (uint64_t w = U; w; w &= w - 1) f(__ffsll((long long)w) - 1);
        }
    };
    // the key run upwards is taken NX values at a time: independent chains
    if constexpr (One) {
        constexpr int NX = 2;
        for (int c = 0; c < nr; ++c) {
            const float *W = S.W + (slot0 / PE_CH) * nbg * PE_CH + c;
            float base = S.rbase[slot0 + c] + fU;
            members([&](int y) { base += W[y * PE_CH]; });
            for (int x = top; x < nbg; x += NX) {
                float val[NX];
#pragma unroll
                for (int h = 0; h < NX; ++h) {
                    const int xh = min(x + h, nbg - 1);
                    val[h] = base + (pairs(xh) + W[xh * PE_CH]);
                    if (x + h >= nbg) val[h] = INFINITY;
                }
                if (fminf(val[0], val[1]) <= limit) {
#pragma unroll
                    for (int h = 0; h < NX; ++h)
                        if (val[h] <= limit)
                            limit = sweep_hit(S, v, d, lb, ns, S.rmask[slot0 + c], U | (1ull << (x + h)), val[h]);
                }
            }
        }
    } else {
        constexpr int NX = 1;
        for (int g = g0; g < g1; ++g) {
            const int slot = slot0 + g * PE_CH;
            const float *W = S.W + (slot / PE_CH) * nbg * PE_CH;
            float base[PE_CH];
#pragma unroll
            for (int c = 0; c < PE_CH; ++c) base[c] = S.rbase[slot + c] + fU;
            members([&](int y) {
                const float4 wa = *reinterpret_cast<const float4 *>(W + y * PE_CH);
                const float4 wb = *reinterpret_cast<const float4 *>(W + y * PE_CH + 4);
                base[0] += wa.x, base[1] += wa.y, base[2] += wa.z, base[3] += wa.w;
                base[4] += wb.x, base[5] += wb.y, base[6] += wb.z, base[7] += wb.w;
            });
            for (int x = top; x < nbg; x += NX) {
                float val[NX][PE_CH], mn = INFINITY;
#pragma unroll
                for (int h = 0; h < NX; ++h) {
                    const int xh = min(x + h, nbg - 1);
                    const float lw = x + h < nbg ? pairs(xh) : INFINITY;
                    const float4 wa = *reinterpret_cast<const float4 *>(W + xh * PE_CH);
                    const float4 wb = *reinterpret_cast<const float4 *>(W + xh * PE_CH + 4);
                    val[h][0] = base[0] + (lw + wa.x), val[h][1] = base[1] + (lw + wa.y);
                    val[h][2] = base[2] + (lw + wa.z), val[h][3] = base[3] + (lw + wa.w);
                    val[h][4] = base[4] + (lw + wb.x), val[h][5] = base[5] + (lw + wb.y);
                    val[h][6] = base[6] + (lw + wb.z), val[h][7] = base[7] + (lw + wb.w);
                    mn = fminf(mn, fminf(fminf(fminf(val[h][0], val[h][1]), fminf(val[h][2], val[h][3])),
                                         fminf(fminf(val[h][4], val[h][5]), fminf(val[h][6], val[h][7]))));
                }
                if (mn <= limit) {
#pragma unroll
                    for (int h = 0; h < NX; ++h)
#pragma unroll
                        for (int c = 0; c < PE_CH; ++c)
                            if (val[h][c] <= limit)
                                limit = sweep_hit(S, v, d, lb, ns, S.rmask[slot + c], U | (1ull << (x + h)), val[h][c]);
                }
            }
        }
    }
}

template <bool One>
__device__ __forceinline__ void sweep_u(EnumSm &S, const float *v, int d, LaneBest &lb, float &limit, int ns, int nbg,
                                        int r, uint64_t U, int slot0, int g0, int g1, int nr)
{
    switch (r) {
    case 1: sweep_run<0, One>(S, v, d, lb, limit, ns, nbg, U, slot0, g0, g1, nr); break;
    case 2: sweep_run<1, One>(S, v, d, lb, limit, ns, nbg, U, slot0, g0, g1, nr); break;
    case 3: sweep_run<2, One>(S, v, d, lb, limit, ns, nbg, U, slot0, g0, g1, nr); break;
    case 4: sweep_run<3, One>(S, v, d, lb, limit, ns, nbg, U, slot0, g0, g1, nr); break;
    case 5: sweep_run<4, One>(S, v, d, lb, limit, ns, nbg, U, slot0, g0, g1, nr); break;
    case 6: sweep_run<5, One>(S, v, d, lb, limit, ns, nbg, U, slot0, g0, g1, nr); break;
    case 7: sweep_run<6, One>(S, v, d, lb, limit, ns, nbg, U, slot0, g0, g1, nr); break;
    case 8: sweep_run<7, One>(S, v, d, lb, limit, ns, nbg, U, slot0, g0, g1, nr); break;
    default: sweep_run<-1, One>(S, v, d, lb, limit, ns, nbg, U, slot0, g0, g1, nr); break;
    }
}

// every exchange of r = 1 .. ns keys (all threads of the block)
__device__ __noinline__ void sweep(EnumSm &S, const float *v, int d, LaneBest &lb, int ns, int nbg, float base0)
{
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    float limit = PE_TINY;  // values up to this are hits
    const int room = min(PE_GMAX, PE_WCAP / (nbg * PE_CH));
    if (tid == 0) {
        S.next_r = 1;
        S.next_g = 0;
    }
    for (;;) {
        __syncthreads();
        // ---- the next batch of groups
        if (tid == 0) {
            int n = 0, left = room, r = S.next_r, g = S.next_g;
            while (r <= ns && left > 0) {
                const int64_t ng = (int64_t)((cb(ns, r) + PE_CH - 1) / PE_CH);
                const int take = (int)min((int64_t)left, ng - g);
                S.seg_r[n] = r;
                S.seg_g[n] = g;
                S.seg_n[n] = take;
                ++n;
                left -= take;
                g += take;
                if (g >= ng) {
                    ++r;
                    g = 0;
                }
            }
            S.task = 0u;
            S.nseg = n;
            S.next_r = r;
            S.next_g = g;
        }
        __syncthreads();
        const int nseg = S.nseg;
        if (nseg == 0) return;
        int slots = 0;
        for (int i = 0; i < nseg; ++i) slots += S.seg_n[i] * PE_CH;
        for (int e = tid; e < slots; e += PE_T) {
            int i = 0, rel = e;
            while (rel >= S.seg_n[i] * PE_CH) rel -= S.seg_n[i++] * PE_CH;
            const int r = S.seg_r[i];
            const uint64_t rank = (uint64_t)S.seg_g[i] * PE_CH + rel;
            uint32_t Rm = 0;
            float f = INFINITY;
            if (rank < cbl(ns, r)) {
                Rm = (uint32_t)colex_unrank(rank, r, ns);
                f = base0;
                for (uint32_t w = Rm; w; w &= w - 1) {
                    const int x = __ffs(w) - 1;
                    f += S.C[x * CLD + x];
                    for (uint32_t w2 = Rm & ((1u << x) - 1u); w2; w2 &= w2 - 1) f += S.C[x * CLD + __ffs(w2) - 1];
                }
            }
            S.rmask[e] = Rm;
            S.rbase[e] = f;
        }
        __syncthreads();
        for (int e = tid; e < slots * nbg; e += PE_T) {  // e = (group, y, c)
            const int c = e % PE_CH, gy = e / PE_CH, g = gy / nbg, y = gy - g * nbg;
            float f = 0.f;
            for (uint32_t w = S.rmask[g * PE_CH + c]; w; w &= w - 1) f += S.C[(__ffs(w) - 1) * CLD + ns + y];
            S.W[e] = f;
        }
        __syncthreads();
        // ---- tasks (segment, 32 subsets U, PE_GSPLIT groups), taken by the warps as they finish
        uint64_t tfirst = 0;
        uint32_t t = 0;
        int slot0 = 0;
        if (lane == 0) t = atomicAdd(&S.task, 1u);
        t = __shfl_sync(FW_FULL, t, 0);
        for (int i = 0; i < nseg; ++i) {
            const int r = S.seg_r[i], ng = S.seg_n[i];
            const uint64_t NR = cb(ns, r), NU = cb(nbg - 1, r - 1);
            const bool one = NR <= 2;
            const int nsp = (ng + PE_GSPLIT - 1) / PE_GSPLIT;
            const uint64_t nt = (NU + 31) / 32 * nsp;
            while (t < tfirst + nt) {
                const uint64_t q = t - tfirst, ub = q / nsp, u = ub * 32 + lane;
                const int g0 = (int)(q - ub * nsp) * PE_GSPLIT, g1 = min(ng, g0 + PE_GSPLIT);
                if (u < NU) {
                    const uint64_t U = r > 1 ? colex_unrank(u, r - 1, nbg - 1) : 0;
                    if (one) sweep_u<true>(S, v, d, lb, limit, ns, nbg, r, U, slot0, g0, g1, (int)NR);
                    else sweep_u<false>(S, v, d, lb, limit, ns, nbg, r, U, slot0, g0, g1, 0);
                }
                __syncwarp();
                if (lane == 0) t = atomicAdd(&S.task, 1u);
                t = __shfl_sync(FW_FULL, t, 0);
            }
            tfirst += nt;
            slot0 += ng * PE_CH;
        }
    }
}

__global__ void __launch_bounds__(PE_T, PE_BPS) k_pool_enum(PoolArgs a)
{
    extern __shared__ __align__(16) unsigned char smraw[];
    EnumSm &S = *reinterpret_cast<EnumSm *>(smraw);
    float *v = reinterpret_cast<float *>(smraw + (sizeof(EnumSm) + 15) / 16 * 16);  // [PMAX][d + 4]
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int d = a.R.d, ld = d + 4;
    const bool bf16 = a.R.v_dtype == FW_BF16;
    const int64_t items = a.R.rows * a.nb;
    for (int64_t it = blockIdx.x; it < items; it += gridDim.x) {
        const int64_t r = it / a.nb;
        const int64_t g = r / a.R.R;
        const int n = a.R.n[g];
        const float *l = a.R.logits + a.R.logit_off[g] + (r - g * a.R.R) * n;
        const int64_t voff = a.R.v_off[g];
        const float M = a.M[r], Zi = 1.f / a.Z[r];
        const int s = a.k[it];
        const int P = a.pool_n[it];
        int32_t *bi = a.best_idx + it * a.k_max;
        // refused items: an out-of-range budget (P = -1), a pool over PMAX keys
        // (P = -2), a non-finite logit (P = -3), thresholds that keep fewer than s
        // keys, or more subsets than the enumeration takes
        int status = P == -2 ? FW_ERR_UNSUPPORTED : (P == -3 ? FW_ERR_NONFINITE : (P < s ? FW_ERR_INVALID_ARG : FW_OK));
        if (status == FW_OK && cb(P, min(s, P - s)) > PE_MAX_SUBSETS) status = FW_ERR_UNSUPPORTED;
        if (status != FW_OK) {
            if (tid == 0) {
                if (a.row_status) atomicMax(a.row_status + r, status);
                a.best_gap[it] = __int_as_float(0x7fc00000);
                if (a.topk_gap) a.topk_gap[it] = __int_as_float(0x7fc00000);
                if (a.n_cand) a.n_cand[it] = 0;
            }
            for (int q = tid; q < a.k_max; q += PE_T) bi[q] = -1;
            continue;
        }
        __syncthreads();  // the previous item's state is no longer read
        if (wid < 2) {  // masses; the kept keys by the thresholds
            const int x = tid;
            bool kept = false;
            float p = 0.f;
            if (x < P) {
                const int j = a.pool[it * PMAX + x];
                const float lj = __ldg(l + j);
                S.pidx[x] = j;
                p = __expf(lj - M) * Zi;
                const uint32_t kl = order_key(lj), tk = a.thr_key[it];
                kept = kl > tk || (kl == tk && j <= a.thr_idx[it]);
            }
            S.pp[x] = p;
            const uint32_t bal = __ballot_sync(FW_FULL, kept);
            if (lane == 0) reinterpret_cast<uint32_t *>(&S.topK)[wid] = bal;
        }
        for (int c = tid; c < d; c += PE_T) S.o[c] = a.o[r * d + c];
        __syncthreads();
        // ---- value rows (zeros past P in the last pair of rows), 4 columns per thread and step
        for (int e = tid; e < ((P + 1) & ~1) * (d / 4); e += PE_T) {
            const int x = e / (d / 4), c = (e - x * (d / 4)) * 4;
            float4 u = make_float4(0.f, 0.f, 0.f, 0.f);
            if (x < P) {
                const int64_t i = voff + (int64_t)S.pidx[x] * d + c;
                if (bf16) {
                    const uint2 h = __ldg(reinterpret_cast<const uint2 *>(static_cast<const uint16_t *>(a.R.v) + i));
                    u = make_float4(__uint_as_float(h.x << 16), __uint_as_float(h.x & 0xffff0000u),
                                    __uint_as_float(h.y << 16), __uint_as_float(h.y & 0xffff0000u));
                } else {
                    u = __ldg(reinterpret_cast<const float4 *>(static_cast<const float *>(a.R.v) + i));
                }
            }
            *reinterpret_cast<float4 *>(v + x * ld + c) = u;
        }
        __syncthreads();
        const uint64_t topK = S.topK;
        // the set exchanged from: the top-mass set (s keys also where the
        // caller's thresholds keep another count)
        uint64_t K = __popcll(topK) == s ? topK : (1ull << s) - 1ull;
        const bool ksmall = s <= P - s;  // the smaller side: K or the keys outside it
        const int ns = ksmall ? s : P - s, nbg = P - ns;
        // roundings: the table sums' chains, and the entries' own (fp32 G)
        const float kappa = (float)(ns * (ns + 1) / 2 + 2 * ns + 10 + d / 4 + 18) * 1.5f * 5.9604645e-8f;
        int64_t ncand = 1;
        // the block's subset of least value (every thread)
        auto least_of = [&](LaneBest &lb) -> uint64_t {
            uint64_t mk = lb.least < INFINITY ? exchanged(S, ns, lb.R, lb.D) : ~0ull;
            for (int o = 16; o; o >>= 1) {
                const float v2 = __shfl_xor_sync(FW_FULL, lb.least, o);
                const uint64_t om = __shfl_xor_sync(FW_FULL, mk, o);
                if (v2 < lb.least || (v2 == lb.least && om < mk)) {
                    lb.least = v2;
                    mk = om;
                }
            }
            __syncthreads();
            if (lane == 0) {
                S.red_v[wid] = lb.least;
                S.red_mask[wid] = mk;
            }
            __syncthreads();
            for (int w = 0; w < PE_NW; ++w)
                if (S.red_v[w] < lb.least || (S.red_v[w] == lb.least && S.red_mask[w] < mk)) {
                    lb.least = S.red_v[w];
                    mk = S.red_mask[w];
                }
            return mk;
        };
        // (fp64 runs at 1/60 of fp32's rate here: scalars in fp64 are one thread's work)
        bool scaled = false;
        for (int round = 0;; ++round) {
            // ---- G in fp32: 2 x 2 keys per thread and step, four partial sums per entry
            if (round == 0) {
                const int P2 = (P + 1) / 2, nt = P2 * (P2 + 1) / 2;
                for (int i = tid; i < nt; i += PE_T) {
                    int x = (int)((sqrtf(8.f * (float)i + 1.f) - 1.f) * 0.5f);
                    while (x * (x + 1) / 2 > i) --x;
                    while ((x + 1) * (x + 2) / 2 <= i) ++x;
                    const int y = i - x * (x + 1) / 2;
                    const float *x0 = v + 2 * x * ld, *y0 = v + 2 * y * ld;
                    float4 s00{}, s01{}, s10{}, s11{};
                    for (int c = 0; c < d; c += 4) {
                        const float4 o4 = *reinterpret_cast<const float4 *>(S.o + c);
                        auto diff = [&](const float *q) {
                            const float4 u = *reinterpret_cast<const float4 *>(q);
                            return make_float4(u.x - o4.x, u.y - o4.y, u.z - o4.z, u.w - o4.w);
                        };
                        const float4 xa = diff(x0 + c), xb = diff(x0 + ld + c), ya = diff(y0 + c), yb = diff(y0 + ld + c);
                        auto mac = [](float4 &s, const float4 &p, const float4 &q) {
                            s.x = fmaf(p.x, q.x, s.x), s.y = fmaf(p.y, q.y, s.y);
                            s.z = fmaf(p.z, q.z, s.z), s.w = fmaf(p.w, q.w, s.w);
                        };
                        mac(s00, xa, ya), mac(s01, xa, yb), mac(s10, xb, ya), mac(s11, xb, yb);
                    }
                    auto put = [&](int p, int q, const float4 &s4) {
                        if (p >= P || q >= P) return;
                        const float w = ((s4.x + s4.y) + (s4.z + s4.w)) * S.pp[p] * S.pp[q];
                        S.G[p * CLD + q] = S.G[q * CLD + p] = w;
                    };
                    put(2 * x, 2 * y, s00), put(2 * x + 1, 2 * y, s10), put(2 * x + 1, 2 * y + 1, s11);
                    if (x != y) put(2 * x, 2 * y + 1, s01);
                }
            }
            // ---- sum_K u
            for (int c = tid; c < d; c += PE_T) {
                double uc[1];
                col_sums<1>(S, v, d, K, c, 1, uc);
                const df u = df_from_double(uc[0]);
                S.UK[c] = uc[0];
                S.UKh[c] = u.hi;
                S.UKl[c] = u.lo;
            }
            if (tid < P) {  // table order: the smaller side's keys first
                const bool kept = (K >> tid) & 1ull;
                const int i = __popcll((kept ? K : ~K) & ((1ull << tid) - 1ull));
                S.loc[kept == ksmall ? i : ns + i] = tid;
            }
            __syncthreads();
            if (wid == 0) {  // es(K), and the best set so far
                double q = 0.0;
                for (int c = lane; c < d; c += 32) {  // (es_warp's order)
                    const double u = S.UK[c];
                    q = fma(u, u, q);
                }
                q = warp_sum_d(q);
                const double pk = mass_warp(S, K, lane);
                if (lane == 0) {
                    const double ek = sqrt(q) / pk;
                    const uint64_t krank = colex_rank64(K);
                    if (round == 0) S.stale = 0;
                    else S.stale = ek < S.bes ? 0 : S.stale + 1;
                    if (round == 0 || ek < S.bes || (ek == S.bes && krank < S.brank)) {
                        S.bes = ek;
                        S.bmask = K;
                        S.brank = krank;
                    }
                    S.QK = q;
                    S.PK = pk;
                    S.rPK = 1.0 / pk;
                    S.K = K;
                    S.ncand = S.nsurv = 0;
                    if (round == 0 && a.topk_gap && topK == K) a.topk_gap[it] = (float)ek;
                }
            }
            // its products with the pool: four lanes per key
            for (int x = tid >> 2; x < P; x += PE_T / 4) {
                float hi = 0.f, lo = 0.f;
                for (int c = tid & 3; c < d; c += 4) {
                    const df u = df_two_sum(v[x * ld + c], -S.o[c]);
                    const float kh = S.UKh[c], kl = S.UKl[c];
                    const float q = u.hi * kh;
                    const float e = fmaf(u.lo, kh, fmaf(u.hi, kl, fmaf(u.hi, kh, -q)));
                    const df t = df_two_sum(hi, q);
                    hi = t.hi;
                    lo += t.lo + e;
                }
                df q{hi, lo};
                const uint32_t quad = 0xfu << (lane & 28);
#pragma unroll
                for (int o = 1; o < 4; o <<= 1) {
                    const df q2{__shfl_xor_sync(quad, q.hi, o), __shfl_xor_sync(quad, q.lo, o)};
                    q = df_add(q, q2);
                }
                if ((tid & 3) == 0) {
                    S.gh[x] = q.hi;
                    S.gl[x] = q.lo;
                }
            }
            __syncthreads();
            if (round == 0 && a.topk_gap && topK != K && wid == 0) {
                const double te = es_warp(S, v, d, topK, lane);
                if (lane == 0) a.topk_gap[it] = (float)te;
            }
            if (ns == 0 || !isfinite(S.bes)) break;  // (not finite: a value of the row, hence o, is not)
            // ---- the tables, scaled by a power of two that brings the largest a_x^2 near 1
            const float te = (float)S.bes;
            float amax = 0.f;
            for (int x = lane; x < P; x += 32) amax = fmaxf(amax, fmaxf(sqrtf(S.G[x * CLD + x]), te * S.pp[x]));
            amax = warp_max(amax);
            // es does not change with a factor of the masses: where the products leave the
            // range whose squares fp32 holds (a sink so heavy that every u is tiny), a power
            // of two on the masses brings them back, once
            const bool far = !(amax > 1e-15f && amax < 1e15f);
            if (far && !scaled && amax > 0.f) {
                __syncthreads();  // the state above is no longer read
                if (tid < P) S.pp[tid] = scalbnf(S.pp[tid], amax < INFINITY ? max(-PE_XMASS, min(-ilogbf(amax), PE_XMASS)) : -PE_XMASS);
                __syncthreads();
                scaled = true;
                round = -1;
                continue;
            }
            // (vectors that are all zero, or beyond even that: no value decides anything,
            // every subset is a hit)
            const bool blind = far;
            amax *= amax;
            const float sc = blind ? 1.f : scalbnf(1.f, -ilogbf(amax));
            if (tid < P) {
                const float st = te * sqrtf(sc) * 1.00001f;
                S.ax[tid] = sqrtf(S.G[tid * CLD + tid] * sc) * 1.00001f + st * S.pp[tid];
                // h_x = u_x . sum_K u - t p_x p(K), kept in the slot of the double-float product
                const double t = S.bes * S.bes;
                S.gh[tid] = (float)(((double)S.gh[tid] + (double)S.gl[tid] - t * S.PK) * (double)S.pp[tid] * (double)sc);
                if (tid == 0) {
                    S.red_v[0] = (float)((S.QK - t * S.PK * S.PK) * (double)sc);
                    S.red_v[1] = (sqrtf((float)(S.QK * (double)sc)) + st * (float)S.PK) * 1.00001f;
                    S.red_v[2] = te * sqrtf(sc);
                }
            }
            __syncthreads();
            const float c0 = S.red_v[0], b0 = S.red_v[1], rt = S.red_v[2];
            const float base0 = blind ? -1.f : c0 - kappa * fabsf(c0);
            for (int i = wid; i < P; i += PE_NW) {
                const int x = S.loc[i];
                const float ax = S.ax[x], px = S.pp[x];
                for (int j = lane; j <= i; j += 32) {
                    const int y = S.loc[j];
                    const float H = S.G[x * CLD + y] * sc - (rt * px) * (rt * S.pp[y]);
                    float w;
                    if (i == j) w = H + ((i < ns) == ksmall ? -2.f : 2.f) * S.gh[x] - kappa * ax * (ax + 2.f * b0);
                    else w = ((i < ns) == (j < ns) ? 2.f : -2.f) * H - 2.f * kappa * ax * S.ax[y];
                    S.C[i * CLD + j] = S.C[j * CLD + i] = blind ? 0.f : w;
                }
            }
            const bool score = round >= PE_SWEEPS;
            LaneBest lb;
            lb.score = score;
            lb.least = INFINITY;
            lb.R = 0;
            lb.D = 0;
            lb.mask = S.bmask;
            lb.rank = S.brank;
            lb.es = INFINITY;
            lb.seen = 0;
            if (score) lb.es = es_lane(S, v, d, lb.mask);  // (by the operations the lanes use)
            sweep(S, v, d, lb, ns, nbg, base0);  // (begins and ends with block barriers)
            if (score) {
                int64_t seen = lb.seen;
                for (int o = 16; o; o >>= 1) {
                    seen += __shfl_xor_sync(FW_FULL, seen, o);
                    const double oe = __shfl_xor_sync(FW_FULL, lb.es, o);
                    const uint64_t orank = __shfl_xor_sync(FW_FULL, lb.rank, o);
                    const uint64_t om = __shfl_xor_sync(FW_FULL, lb.mask, o);
                    if (oe < lb.es || (oe == lb.es && orank < lb.rank)) {
                        lb.es = oe;
                        lb.rank = orank;
                        lb.mask = om;
                    }
                }
                if (lane == 0) {
                    S.red_es[wid] = lb.es;
                    S.red_rank[wid] = lb.rank;
                    S.red_mask[wid] = lb.mask;
                    S.red_seen[wid] = seen;
                }
                __syncthreads();
                ncand = 1;
                for (int w = 0; w < PE_NW; ++w) ncand += S.red_seen[w];
                if (tid == 0) S.bes = DBL_MAX;  // (the warps' include it)
                break;
            }
            if (S.ncand > GCAP) {  // (uniform)
                // again around the subset of least value; when three rounds brought
                // no better es the values decide nothing more
                const uint64_t mk = least_of(lb);
                if (S.stale >= 3 || mk == K) round = PE_SWEEPS - 1;
                K = mk;
                __syncthreads();  // the state above is no longer read
                continue;
            }
            // ---- each hit's interval of es^2 - t, times p(K)^2: [v, v + 2 bound] (p(K) / p(A))^2
            const int seen = S.ncand;
            constexpr int PER = (GCAP + PE_T - 1) / PE_T;
            float up = 0.f;
            float myl[PER];
#pragma unroll
            for (int q = 0; q < PER; ++q) {
                const int i = tid + q * PE_T;
                myl[q] = INFINITY;
                if (i >= seen) continue;
                double pr = 0.0, pd = 0.0;
                float e = 0.f;
                for (uint32_t w = S.candR[i]; w; w &= w - 1) {
                    const int x = S.loc[__ffs(w) - 1];
                    pr += (double)S.pp[x];
                    e += S.ax[x];
                }
                for (uint64_t w = S.candD[i]; w; w &= w - 1) {
                    const int x = S.loc[ns + __ffsll((long long)w) - 1];
                    pd += (double)S.pp[x];
                    e += S.ax[x];
                }
                const double pa = S.PK + (ksmall ? pd - pr : pr - pd);
                // masses that cancel to nothing leave the hit to the exact score
                const float p2 = !blind && pa > 1e-9 * (pr + pd) ? (float)(pa * S.rPK * (pa * S.rPK)) : 0.f;
                const float lov = S.candV[i];
                const float upv = lov + 2.f * kappa * (e * (e + 2.f * b0) + fabsf(c0)) * 1.001f + 2.f * PE_TINY;
                myl[q] = p2 > 0.f ? (lov - 1e-5f * fabsf(lov)) / p2 : -INFINITY;
                if (p2 > 0.f) up = fminf(up, (upv + 1e-5f * fabsf(upv)) / p2);
            }
            up = warp_min(up);
            if (lane == 0) S.red_v[wid] = up;
            __syncthreads();
            for (int w = 0; w < PE_NW; ++w) up = fminf(up, S.red_v[w]);
            // the survivors' subsets in place of their hits, then a list of them
            uint32_t keep = 0;
#pragma unroll
            for (int q = 0; q < PER; ++q) {
                const int i = tid + q * PE_T;
                if (i < seen && myl[q] <= up) {
                    S.candD[i] = exchanged(S, ns, S.candR[i], S.candD[i]);
                    keep |= 1u << q;
                }
            }
            __syncthreads();
#pragma unroll
            for (int q = 0; q < PER; ++q)
                if ((keep >> q) & 1u) S.candR[atomicAdd(&S.nsurv, 1)] = (uint32_t)(tid + q * PE_T);
            __syncthreads();
            const int nsv = S.nsurv;
            if (nsv > PE_SURV && round < 2 && !blind) {  // the values around K do not tell them apart
                const uint64_t mk = least_of(lb);
                if (mk != K) {
                    K = mk;
                    __syncthreads();
                    continue;
                }
            }
            ncand = nsv + 1;
            double wes = INFINITY;
            uint64_t wrank = ~0ull, wmask = 0;
            for (int q = wid; q < nsv; q += PE_NW) {
                const uint64_t A = S.candD[S.candR[q]];
                const double es = es_warp(S, v, d, A, lane);
                const uint64_t rank = colex_rank64(A);
                if (es < wes || (es == wes && rank < wrank)) {
                    wes = es;
                    wrank = rank;
                    wmask = A;
                }
            }
            if (lane == 0) {
                S.red_es[wid] = wes;
                S.red_rank[wid] = wrank;
                S.red_mask[wid] = wmask;
            }
            break;
        }
        __syncthreads();
        const bool none = !isfinite(S.bes);  // no subset has an es
        if (tid == 0 && none) {
            if (a.row_status) atomicMax(a.row_status + r, (int)FW_ERR_NONFINITE);
            a.best_gap[it] = __int_as_float(0x7fc00000);
            if (a.topk_gap) a.topk_gap[it] = __int_as_float(0x7fc00000);
            if (a.n_cand) a.n_cand[it] = 0;
        } else if (tid == 0) {
            if (ns > 0)
                for (int w = 0; w < PE_NW; ++w)
                    if (S.red_es[w] < S.bes || (S.red_es[w] == S.bes && S.red_rank[w] < S.brank)) {
                        S.bes = S.red_es[w];
                        S.brank = S.red_rank[w];
                        S.bmask = S.red_mask[w];
                    }
            a.best_gap[it] = (float)S.bes;
            if (a.n_cand) a.n_cand[it] = ncand;
        }
        __syncthreads();
        const uint64_t bmask = none ? 0 : S.bmask;
        if (tid < P && ((bmask >> tid) & 1ull)) bi[__popcll(bmask & ((1ull << tid) - 1ull))] = S.pidx[tid];
        for (int q = (none ? 0 : s) + tid; q < a.k_max; q += PE_T) bi[q] = -1;
    }
}

}  // namespace

static size_t pool_bytes(const RowsDev &R, int nb) { return align256((size_t)R.rows * nb * PMAX * 4); }

size_t pool_best_subset_workspace(const RowsDev &R, int nb)
{
    return pool_bytes(R, nb) + align256((size_t)R.rows * nb * 4);
}

fw_status pool_best_subset(const RowsDev &R, const int32_t *k, int nb, const int32_t *E, const fw_gap_out &topk,
                           float *best_gap, int32_t *best_idx, int k_max, float *topk_gap, int64_t *n_cand,
                           int32_t *row_status, void *ws, cudaStream_t st)
{
    if (R.max_n > PB_STAGE_MAX) return FW_ERR_UNSUPPORTED;
    PoolArgs a;
    a.R = R;
    a.k = k;
    a.nb = nb;
    for (int b = 0; b < 4; ++b) a.E[b] = b < nb ? E[b] : 0;
    a.thr_key = topk.thr_key;
    a.thr_idx = topk.thr_idx;
    a.o = topk.o;
    a.M = topk.row_max;
    a.Z = topk.row_sum;
    a.pool = (int32_t *)ws;
    a.pool_n = (int32_t *)((char *)ws + pool_bytes(R, nb));
    a.best_gap = best_gap;
    a.best_idx = best_idx;
    a.k_max = k_max;
    a.topk_gap = topk_gap;
    a.row_status = row_status;
    a.n_cand = n_cand;
    int sms = 0;
    if (device_sms(&sms) != FW_OK) return FW_ERR_CUDA;
    if (row_status) FW_CUDA_CHECK(cudaMemsetAsync(row_status, 0, (size_t)R.rows * 4, st));
    FW_DISPATCH(R.d, R.v_dtype, {
        const size_t sb = (size_t)R.max_n * 4;
        FW_CUDA_CHECK(cudaFuncSetAttribute(k_pool_build<DPL, VT>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sb));
        FW_LAUNCH((k_pool_build<DPL, VT>), (unsigned)std::min<int64_t>(R.rows, (int64_t)sms * 8), PB_T, sb, st, a);
    });
    const size_t se = (sizeof(EnumSm) + 15) / 16 * 16 + (size_t)PMAX * (R.d + 4) * 4;
    FW_CUDA_CHECK(cudaFuncSetAttribute(k_pool_enum, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)se));
    FW_LAUNCH(k_pool_enum, (unsigned)std::min<int64_t>(R.rows * nb, 1 << 20), PE_T, se, st, a);
    return FW_OK;
}

}  // namespace fw

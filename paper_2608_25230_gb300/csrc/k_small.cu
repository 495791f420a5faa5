// k_small.cu -- rows with at most 32 keys (the exact-search workloads).
//
// One warp per row.  Lane j owns key j for the softmax and the top-k rank;
// for vector quantities lane l owns dimensions l, l+32, ...  Masses are fp64
// (one exp per key), vector sums are double-float on the fp32 pipe, so every
// output carries ~1e-13 relative error against an fp64 evaluation of the
// definitions.
#include <algorithm>

#include "fw_internal.h"

namespace fw {
namespace {

struct SmallGapArgs {
    RowsDev R;
    const int32_t *k;
    int nb;
    fw_gap_out out;
};

// Definition 2.1 / Sec. 2.1 / Lemma 2.1 for one row and up to four budgets.
// NBM: budgets held in registers (1, or up to 4)
template <int DPL, typename VT, int NBM>
__global__ void __launch_bounds__(256) k_small_gap(const SmallGapArgs a)
{
    const int lane = threadIdx.x & 31;
    const int64_t row = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (row >= a.R.rows) return;
    const int64_t g = row / a.R.R;
    const int64_t ri = row - g * a.R.R;
    const int n = a.R.n[g];
    constexpr int d = DPL * 32;
    int32_t *st = a.out.row_status;
    if (n < 1 || n > 32) {
        if (lane == 0 && st) st[row] = FW_ERR_INVALID_ARG;
        return;
    }
    const float *lg = a.R.logits + a.R.logit_off[g] + ri * n;
    const VT *V = reinterpret_cast<const VT *>(a.R.v) + a.R.v_off[g];
    const float l = lane < n ? lg[lane] : -INFINITY;
    if (__any_sync(FW_FULL, lane < n && !isfinite(l))) {
        if (lane == 0 && st) st[row] = FW_ERR_NONFINITE;
        return;
    }
    // softmax masses (fp64)
    const float M = warp_max(l);
    double p = lane < n ? exp((double)l - (double)M) : 0.0;
    const double Z = warp_sum_d(p);
    p = p / Z;
    // rank in the order (logit desc, index asc)
    int rank = 0;
    for (int s = 0; s < n; ++s) {
        const float ls = __shfl_sync(FW_FULL, l, s);
        rank += (ls > l) || (ls == l && s < lane);
    }
    const int nb = a.nb;
    uint32_t mask[NBM];
    int status = FW_OK;
#pragma unroll
    for (int b = 0; b < NBM; ++b) {
        mask[b] = 0u;
        if (b >= nb) continue;
        const int kb = a.k[row * nb + b];
        if (kb < 1 || kb > n) {
            status = FW_ERR_INVALID_ARG;
            continue;
        }
        mask[b] = __ballot_sync(FW_FULL, lane < n && rank < kb);
        if (lane < n && rank == kb - 1) {
            if (a.out.thr_key) a.out.thr_key[row * nb + b] = order_key(l);
            if (a.out.thr_idx) a.out.thr_idx[row * nb + b] = lane;
        }
        if (a.out.kept_bits) {
            uint32_t *w = a.out.kept_bits + (row * nb + b) * (int64_t)a.out.kept_words;
            for (int t = lane; t < a.out.kept_words; t += 32) w[t] = t == 0 ? mask[b] : 0u;
        }
    }
    // dense output mu = sum_j p_j v_j
    const df pd = df_from_double(p);
    df mu[DPL];
#pragma unroll
    for (int t = 0; t < DPL; ++t) mu[t] = df_zero();
    for (int j = 0; j < n; ++j) {
        const df pj = shfl_df(pd, j);
#pragma unroll
        for (int t = 0; t < DPL; ++t)
            mu[t] = df_add(mu[t], df_mul_f(pj, load_v(V, (int64_t)j * d + lane + 32 * t)));
    }
    // g_A = sum_{j in A} p_j (v_j - mu) for each budget (Lemma 2.1)
    df gA[NBM][DPL];
#pragma unroll
    for (int b = 0; b < NBM; ++b)
#pragma unroll
        for (int t = 0; t < DPL; ++t) gA[b][t] = df_zero();
    for (int j = 0; j < n; ++j) {
        const df pj = shfl_df(pd, j);
#pragma unroll
        for (int t = 0; t < DPL; ++t) {
            const df tj = df_mul(pj, df_rsub_f(load_v(V, (int64_t)j * d + lane + 32 * t), mu[t]));
#pragma unroll
            for (int b = 0; b < NBM; ++b)
                if ((mask[b] >> j) & 1u) gA[b][t] = df_add(gA[b][t], tj);
        }
    }
    if (a.out.o) {
#pragma unroll
        for (int t = 0; t < DPL; ++t) a.out.o[row * d + lane + 32 * t] = mu[t].hi + mu[t].lo;  // rounded once
    }
#pragma unroll
    for (int b = 0; b < NBM; ++b) {
        if (mask[b] == 0u) continue;
        const bool in = (mask[b] >> lane) & 1u;
        const double PA = warp_sum_d(in ? p : 0.0);
        const double PD = warp_sum_d(in ? 0.0 : p);
        df nrm = df_zero();
#pragma unroll
        for (int t = 0; t < DPL; ++t) nrm = df_add(nrm, df_mul(gA[b][t], gA[b][t]));
        nrm = warp_sum_df(nrm);
        const double phi = sqrt(fmax(df_to_double(nrm), 0.0));
        const int64_t rb = row * nb + b;
        if (lane == 0) {
            a.out.gap[rb] = (float)(phi / PA);
            a.out.dropped[rb] = (float)PD;
            if (a.out.phi) a.out.phi[rb] = (float)phi;
        }
        if (a.out.o_kept) {  // mu + g_A / P(A) in double-float, rounded once
            const df invP = df_from_double(1.0 / PA);
#pragma unroll
            for (int t = 0; t < DPL; ++t) {
                const df ok = df_add(mu[t], df_mul(gA[b][t], invP));
                a.out.o_kept[rb * d + lane + 32 * t] = ok.hi + ok.lo;
            }
        }
    }
    if (lane == 0) {
        if (a.out.row_max) a.out.row_max[row] = M;
        if (a.out.row_sum) a.out.row_sum[row] = (float)Z;
        if (st) st[row] = status;
    }
}

// ------------------------------------------------------------------ swap rule

struct SmallSwapArgs {
    RowsDev R;
    const int32_t *k;
    int nb;
    const uint32_t *thr_key;
    const int32_t *thr_idx;
    int E, max_swaps;
    int32_t *n_swaps, *swap_out, *swap_in, *capped;
    float *refined_gap, *topk_gap;
    int nr;  // largest n
};

// dimensions staged at a time
__host__ __device__ constexpr int swap_dch(int d) { return d < 64 ? d : 64; }
// shared memory per warp (floats): U (the values, then the high parts of u, and g), G
__host__ __device__ constexpr int swap_smem_floats(int n, int d) { return staged_floats(n, swap_dch(d)) + gram_floats(n); }

// The balancing selector (Sec. 2.1) inside the candidate set (Definition 2.2).
// Pair scores are screened in fp32 from the Gram matrix G = U U^T of the
// centred, weighted points u_j = p_j (v_j - mu) (es(A)^2 = ||g||^2 / p(A)^2,
// g = sum_A u_j, Lemma 2.1); every pair whose fp32 score is within a rigorous
// error bound of the best one is re-scored in double-float and the decision is
// taken on those exact values.
//
// What bounds it: one row's chain of double-float sums (a warp alone issues an
// instruction every 7 cycles or so), instruction fetch (the warps of an SM are in
// different steps of a long program) and the fp64 pipe, which takes 16 cycles for a
// warp's instruction whatever its lanes hold.  Hence
//  - the values are staged 64 dimensions at a time and the Gram tiles (4 x 4 products
//    per lane, 16-byte reads) add up in shared memory, so that 20 warps fit an SM;
//  - loops are not unrolled over keys or chunks (unrolled by 4: 806 us, below: 704);
//  - Q(A - i + j) is screened as Q(A) + 2 g.(u_j - u_i) + |u_j - u_i|^2, with Q(A) and g
//    from the double-float state (g is one more row of the Gram matrix): the error
//    scales with (|g| + |u_i| + |u_j|)^2, not with the square of the kept keys' summed
//    norms, and where g is the small sum of large terms (a sink and its
//    counterweights) far fewer pairs are re-scored (24 keys, k = 6: 5.6 a row before);
//  - the re-scored pairs' fp64 quotients are taken up to 32 pairs at a time, one per
//    lane, and P(A - i) once a round for every i.
// 36,864 rows of 24 keys, d = 128: 1,433 us with whole rows staged and Gram entries one
// by one, 704 us so; 256 rows of 20 keys, d = 64: 67 and 28 us.
// (10 blocks an SM are 96 registers: d = 256 spills 41 of its words, and still takes 763
// us on 20,000 rows of 24 keys, 2,180 before; with 128 registers 748.)
template <int DPL, typename VT>
__global__ void __launch_bounds__(64, 10) k_small_swap(const SmallSwapArgs a)
{
    extern __shared__ __align__(16) float smem[];
    constexpr int d = DPL * 32;
    constexpr int DCH = swap_dch(d), TCH = DCH / 32, NCH = d / DCH;
    const int lane = threadIdx.x & 31;
    const int wib = threadIdx.x >> 5;
    float *U = smem + (size_t)wib * swap_smem_floats(a.nr, d);
    float *G = U + staged_floats(a.nr, DCH);
    const int64_t row = (int64_t)blockIdx.x * (blockDim.x >> 5) + wib;
    if (row >= a.R.rows) return;
    const int64_t g = row / a.R.R;
    const int64_t ri = row - g * a.R.R;
    const int n = a.R.n[g];
    const int nb = a.nb;
    const int MS = a.max_swaps;
    auto fail = [&](int b) {
        const int64_t rb = row * nb + b;
        if (lane == 0) {
            a.n_swaps[rb] = 0;
            a.refined_gap[rb] = __int_as_float(0x7fc00000);
            if (a.topk_gap) a.topk_gap[rb] = __int_as_float(0x7fc00000);
            if (a.capped) a.capped[rb] = 0;
        }
        for (int t = lane; t < MS; t += 32) a.swap_out[rb * MS + t] = a.swap_in[rb * MS + t] = -1;
    };
    if (n < 1 || n > 32) {
        for (int b = 0; b < nb; ++b) fail(b);
        return;
    }
    const float *lg = a.R.logits + a.R.logit_off[g] + ri * n;
    const VT *V = reinterpret_cast<const VT *>(a.R.v) + a.R.v_off[g];
    const float l = lane < n ? lg[lane] : -INFINITY;
    if (__any_sync(FW_FULL, lane < n && !isfinite(l))) {
        for (int b = 0; b < nb; ++b) fail(b);
        return;
    }
    const float M = warp_max(l);
    double p = lane < n ? exp((double)l - (double)M) : 0.0;
    p = p / warp_sum_d(p);
    const df pd = df_from_double(p);
    // the kept set of budget b: the keys from its threshold up
    auto kept = [&](int b) {
        const uint32_t tk = a.thr_key[row * nb + b], key = order_key(l);
        const int ti = a.thr_idx[row * nb + b];
        return __ballot_sync(FW_FULL, lane < n && (key > tk || (key == tk && lane <= ti)));
    };
    const uint32_t A0 = kept(0);
    // One pass over the values, DCH dimensions at a time: mu (double-float, j
    // ascending), u_j = p_j (v_j - mu), whose high parts replace the values (the
    // exact re-scoring recomputes u_j from V), and g of budget 0, the last row.
    df mu[DPL], g0[DPL];
#pragma unroll
    for (int t = 0; t < DPL; ++t) mu[t] = g0[t] = df_zero();
#pragma unroll 1  // (a cold instruction cache costs a small batch more than the shifts below)
    for (int ch = 0; ch < NCH; ++ch) {
        __syncwarp();
        stage_rows<DCH>(V, n, d, ch * DCH, U, lane);
        __syncwarp();
        df m[TCH], gg[TCH];
#pragma unroll
        for (int t = 0; t < TCH; ++t) m[t] = gg[t] = df_zero();
#pragma unroll 1
        for (int j = 0; j < n; ++j) {
            const df pj = shfl_df(pd, j);
#pragma unroll
            for (int t = 0; t < TCH; ++t) m[t] = df_add(m[t], df_mul_f(pj, U[staged_at<DCH>(j, lane + 32 * t)]));
        }
#pragma unroll 1
        for (int j = 0; j < n; ++j) {
            const df pj = shfl_df(pd, j);
            const bool in = (A0 >> j) & 1u;
#pragma unroll
            for (int t = 0; t < TCH; ++t) {
                float *cell = U + staged_at<DCH>(j, lane + 32 * t);
                const df u = df_mul(pj, df_rsub_f(*cell, m[t]));
                *cell = u.hi;
                if (in) gg[t] = df_add(gg[t], u);
            }
        }
#pragma unroll
        for (int t = 0; t < DPL; ++t) {  // chunk by chunk into place
            mu[t] = t + TCH < DPL ? mu[t + TCH < DPL ? t + TCH : 0] : m[t + TCH - DPL < 0 ? 0 : t + TCH - DPL];
            g0[t] = t + TCH < DPL ? g0[t + TCH < DPL ? t + TCH : 0] : gg[t + TCH - DPL < 0 ? 0 : t + TCH - DPL];
        }
#pragma unroll
        for (int t = 0; t < TCH; ++t) U[staged_at<DCH>(n, lane + 32 * t)] = gg[t].hi;
        __syncwarp();
        gram_chunk<d, DCH>(U, G, n, ch == 0, lane);  // and g.u_x in column n
    }
    __syncwarp();
    // u_j in double-float, recomputed from V (the expression of the pass above)
    auto u_df = [&](int j, int t) {
        return df_mul(shfl_df(pd, j), df_rsub_f(load_v(V, (int64_t)j * d + lane + 32 * t), mu[t]));
    };
    // ||u_j||^2, held by lane j, only where a budget restricts the pool (E < n - k)
    bool need_e2 = false;
    for (int b = 0; b < nb; ++b) need_e2 |= a.E < n - a.k[row * nb + b];
    double e2 = 0.0;
    if (need_e2)
#pragma unroll 1
        for (int j = 0; j < n; ++j) {
            df s = df_zero();
#pragma unroll
            for (int t = 0; t < DPL; ++t) {
                const df u = u_df(j, t);
                s = df_add(s, df_mul(u, u));
            }
            s = warp_sum_df(s);
            if (lane == j) e2 = df_to_double(s);
        }
    const float gd = lane < n ? G[lane * GRAM_LD + lane] : 0.f;  // G_xx, lane x
    const float unorm = sqrtf(fmaxf(gd, 0.f)) * 1.0001f;
    const uint32_t all = n == 32 ? FW_FULL : ((1u << n) - 1u);

#pragma unroll 1
    for (int b = 0; b < nb; ++b) {
        const int64_t rb = row * nb + b;
        const int kb = a.k[rb];
        uint32_t A = b == 0 ? A0 : kept(b);
        if (kb < 1 || kb > n || __popc(A) != kb) {
            fail(b);
            continue;
        }
        // candidate set: A plus the E dropped keys of largest single-key error
        uint32_t pool;
        if (a.E >= n - kb) {
            pool = all;
        } else {
            const bool dropped = lane < n && !((A >> lane) & 1u);
            int cnt = 0;
            for (int s = 0; s < n; ++s) {
                const double es = __shfl_sync(FW_FULL, e2, s);
                const bool ds = !((A >> s) & 1u);
                cnt += ds && (es > e2 || (es == e2 && s < lane));
            }
            pool = A | __ballot_sync(FW_FULL, dropped && cnt < a.E);
        }
        // exact state: g_A (double-float, lanes over dims), p(A), es^2
        df gA[DPL];
        if (b == 0) {
#pragma unroll
            for (int t = 0; t < DPL; ++t) gA[t] = g0[t];
        } else {
#pragma unroll
            for (int t = 0; t < DPL; ++t) gA[t] = df_zero();
#pragma unroll 1
            for (uint32_t m = A; m; m &= m - 1) {
                const int j = __ffs(m) - 1;
#pragma unroll
                for (int t = 0; t < DPL; ++t) gA[t] = df_add(gA[t], u_df(j, t));
            }
        }
        double PA = warp_sum_d(((A >> lane) & 1u) ? p : 0.0);
        auto norm2 = [&](const df *gv) {
            df s = df_zero();
#pragma unroll
            for (int t = 0; t < DPL; ++t) s = df_add(s, df_mul(gv[t], gv[t]));
            return warp_sum_df(s);
        };
        df Q = norm2(gA);
        double cur = fmax(df_to_double(Q), 0.0) / (PA * PA);
        if (a.topk_gap && lane == 0) a.topk_gap[rb] = (float)sqrt(cur);
        // f_x = g.u_x in fp32, lane x, kept up to date from G; W bounds |g| and the
        // norms of every term that went into f
        float f, W;
        if (b == 0) {
            f = lane < n ? G[lane * GRAM_LD + n] : 0.f;
            W = sqrtf(fmaxf(Q.hi, 0.f)) * 1.0001f;
        } else {
            f = 0.f;
            if (lane < n)
#pragma unroll 1
                for (uint32_t m = A; m; m &= m - 1) f += G[lane * GRAM_LD + __ffs(m) - 1];
            W = warp_sum(((A >> lane) & 1u) ? unorm : 0.f) * 1.0001f;
        }
        // Bound on the fp32 error of a screened score, times P(A - i + j)^2: with
        // B = W + |u_i| + |u_j| the terms' absolute values sum to at most B^2; each
        // dot product is chains of at most DCH / 2 fused terms, summed, f adds a
        // term per kept key (b > 0) or two per swap, and 12 more roundings cover the
        // operands (u and g to fp32), Q(A) and the sum of terms; doubled.  8 ulps for the
        // rounded P(A - i + j) and its inverse square.  kTiny covers underflow.
        constexpr float kTiny = 1e-37f;
        const float C0 = 0.5f * DCH + NCH + kb + 13.f;
        int taken = 0, cap = 0;
#pragma unroll 1
        for (;;) {
            const uint32_t add = pool & ~A;
            const int nadd = __popc(add);
            if (nadd == 0) break;
            const float CB = (2.f * (C0 + 2.f * taken) + 8.f) * 5.9604645e-8f;
            // fp32 screening of every (kept i, added j) pair, lane j taking the
            // added key j: Q(A - i + j) = (Q_A - 2 f_i + G_ii) + (2 f_j + G_jj) - 2 G_ij,
            // P(A - i + j) = P(A - i) + p_j (two positive terms)
            const bool isadd = (add >> lane) & 1u;
            const float cj = 2.f * f + gd, ci_ = Q.hi - 2.f * f + gd;
            const float pjf = (float)p, Pm = (float)(PA - p);
            const float Wj = W + unorm;
            float inv = 0.f, sc = 0.f, err = 0.f;
            auto screen = [&](int i) {
                const float Pp = __shfl_sync(FW_FULL, Pm, i) + pjf;
                inv = 1.f / (Pp * Pp);
                sc = (__shfl_sync(FW_FULL, ci_, i) + cj - 2.f * G[i * GRAM_LD + (lane < n ? lane : 0)]) * inv;
                const float B = Wj + __shfl_sync(FW_FULL, unorm, i);
                err = fmaf(CB * B, B, kTiny) * inv;
            };
            float best_up = INFINITY;
#pragma unroll 1
            for (uint32_t mi = A; mi; mi &= mi - 1) {
                screen(__ffs(mi) - 1);
                if (isadd) best_up = fminf(best_up, sc + err);
            }
            best_up = warp_min(best_up);
            // exact re-scoring, in (i, j) order, of every pair that may be the best: the
            // norms pair by pair, the fp64 quotients of up to 32 pairs at once (lane c
            // holds the c-th pair of the batch)
            unsigned long long best = 0x7ff0000000000000ull;  // bits of +inf: es^2 >= 0 orders as integers
            int bij = 0, cnt = 0, mij = 0;
            df mine = df_zero();
            auto settle = [&]() {
                const int i = mij >> 5, j = mij & 31;
                const double P2 = PA - __shfl_sync(FW_FULL, p, i) + __shfl_sync(FW_FULL, p, j);
                const double e = fmax(df_to_double(mine), 0.0) / (P2 * P2);
                unsigned long long eb = (unsigned long long)__double_as_longlong(e);
                if (eb == 0x8000000000000000ull) eb = 0ull;  // -0
                if (lane >= cnt) eb = ~0ull;
                const uint32_t hi = __reduce_min_sync(FW_FULL, (uint32_t)(eb >> 32));
                const uint32_t lo = __reduce_min_sync(FW_FULL, (uint32_t)(eb >> 32) == hi ? (uint32_t)eb : 0xffffffffu);
                const unsigned long long eb_min = ((unsigned long long)hi << 32) | lo;
                const int first = __ffs(__ballot_sync(FW_FULL, eb == eb_min)) - 1;
                if (eb_min < best) {
                    best = eb_min;
                    bij = __shfl_sync(FW_FULL, mij, first);
                }
                cnt = 0;
            };
#pragma unroll 1
            for (uint32_t mi = A; mi; mi &= mi - 1) {
                const int i = __ffs(mi) - 1;
                screen(i);
                uint32_t cand = __ballot_sync(FW_FULL, isadd && sc - err <= best_up);
#pragma unroll 1
                while (cand) {
                    const int j = __ffs(cand) - 1;
                    cand &= cand - 1;
                    df gn[DPL];
#pragma unroll
                    for (int t = 0; t < DPL; ++t) gn[t] = df_add(df_sub(gA[t], u_df(i, t)), u_df(j, t));
                    const df s2 = norm2(gn);
                    if (lane == cnt) {
                        mine = s2;
                        mij = 32 * i + j;
                    }
                    if (++cnt == 32) settle();
                }
            }
            if (cnt) settle();
            const int bi = bij >> 5, bj = bij & 31;
            const double bestd = __longlong_as_double((long long)best);
            if (!(bestd < cur)) break;
            if (taken >= MS) {
                cap = 1;
                break;
            }
#pragma unroll
            for (int t = 0; t < DPL; ++t) gA[t] = df_add(df_sub(gA[t], u_df(bi, t)), u_df(bj, t));
            Q = norm2(gA);
            PA = PA - __shfl_sync(FW_FULL, p, bi) + __shfl_sync(FW_FULL, p, bj);
            A = (A & ~(1u << bi)) | (1u << bj);
            cur = bestd;
            if (lane < n) f += G[lane * GRAM_LD + bj] - G[lane * GRAM_LD + bi];
            W += __shfl_sync(FW_FULL, unorm, bi) + __shfl_sync(FW_FULL, unorm, bj);
            if (lane == 0) {
                a.swap_out[rb * MS + taken] = bi;
                a.swap_in[rb * MS + taken] = bj;
            }
            ++taken;
        }
        if (lane == 0) {
            a.n_swaps[rb] = taken;
            a.refined_gap[rb] = (float)sqrt(cur);
            if (a.capped) a.capped[rb] = cap;
        }
        for (int t = lane; t < MS; t += 32)
            if (t >= taken) a.swap_out[rb * MS + t] = a.swap_in[rb * MS + t] = -1;
    }
}

}  // namespace

fw_status small_gap(const RowsDev &R, const int32_t *k, int nb, const fw_gap_out &out, cudaStream_t s)
{
    if (R.rows == 0) return FW_OK;
    const SmallGapArgs a{R, k, nb, out};
    const int warps = 8;
    const unsigned grid = (unsigned)((R.rows + warps - 1) / warps);
    if (nb == 1) {
        FW_DISPATCH(R.d, R.v_dtype, FW_LAUNCH((k_small_gap<DPL, VT, 1>), grid, warps * 32, 0, s, a));
    } else {
        FW_DISPATCH(R.d, R.v_dtype, FW_LAUNCH((k_small_gap<DPL, VT, 4>), grid, warps * 32, 0, s, a));
    }
    return FW_OK;
}

fw_status small_swap(const RowsDev &R, const int32_t *k, int nb, const fw_gap_out &topk, int E,
                     int max_swaps, int32_t *n_swaps, int32_t *swap_out, int32_t *swap_in,
                     float *refined_gap, float *topk_gap, int32_t *capped, cudaStream_t s)
{
    if (R.rows == 0) return FW_OK;
    const int nr = std::min(R.max_n, 32);
    const SmallSwapArgs a{R, k, nb, topk.thr_key, topk.thr_idx, E, max_swaps, n_swaps, swap_out,
                          swap_in, capped, refined_gap, topk_gap, nr};
    FW_DISPATCH(R.d, R.v_dtype, {
        const int warps = 2;
        const size_t smem = (size_t)warps * swap_smem_floats(nr, DPL * 32) * sizeof(float);
        FW_CUDA_CHECK(cudaFuncSetAttribute(k_small_swap<DPL, VT>,
                                           cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
        const unsigned grid = (unsigned)((R.rows + warps - 1) / warps);
        FW_LAUNCH((k_small_swap<DPL, VT>), grid, warps * 32, smem, s, a);
    });
    return FW_OK;
}

}  // namespace fw

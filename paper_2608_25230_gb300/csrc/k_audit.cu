// k_audit.cu -- the deployed selectors audited in Sec. 2.3 / App. C, as
// kernels: for every row and budget s, the kept set that each rule would
// choose, scored with Definition 2.1's es(A) = ||m_A - mu|| (to be set against
// the top-mass set and ES_pool).  The rules, with App. C's settings:
//   StreamingLLM  the first min(4, s/2) positions (sinks) and the last
//                 s - sinks positions (recency);
//   H2O           the last s/2 positions and, among the others, the
//                 s - s/2 of largest mass accumulated over the group's rows
//                 (the KV head's query rows that share the cache);
//   SnapKV        window w = max(1, min(32, s/2)): the last w positions and,
//                 among the others, the s - w of largest pooled vote, the vote
//                 of a key being its mass summed over the group's last w rows,
//                 pooled by a maximum over 7 neighbouring positions (clipped
//                 to the candidates);
//   Quest         pages of P = max(2, s/4) consecutive keys; the floor(s/P)
//                 pages of largest maximum logit (Quest ranks pages by an
//                 upper bound on that maximum; with the row's logits at hand
//                 the bound is the maximum itself);
//   Quest-16      the same with pages of 16 keys (s >= 16).
// Equal scores keep lower positions (pages) first, as everywhere in the
// library.
//
//   k_aud_mass    accumulated masses and window votes of every group (a thread
//                 per key walks the group's rows; compensated sums);
//   k_aud_select  a CTA per group, budget and rule: the H2O or SnapKV set (the
//                 order keys staged once in shared memory, CTA-wide radix
//                 top-m), written as a bit mask by ballots;
//   k_aud_row     per row (its logits staged in shared memory): a warp per
//                 (budget, page size) takes Quest's few largest pages by
//                 repeated arg-max, then one warp per (rule, budget) lists its
//                 members and gathers their p_j v_j, 8 value rows in flight.
// Both are bound by shared-memory and L2 latency.  On 1,024 rows of 4,096 keys
// (256 groups, d = 128, s = 4/8/16/32) the audit with its
// gap call takes 0.41 ms; with a CTA per group for all sets, a radix select for
// every page size and members gathered one at a time it took 0.90 ms.
#include <algorithm>
#include <climits>

#include "fw_internal.h"

namespace fw {
namespace {

constexpr int AM_T = 256;   // k_aud_mass threads
constexpr int AS_T = 512;   // k_aud_select threads
constexpr int AR_T = 256;   // k_aud_row threads (8 warps)
constexpr int A_NBMAX = 4;
constexpr int AS_STAGE = 24576;  // candidates whose keys k_aud_select stages (96 KB)
constexpr size_t AR_SMEM = 196608;  // k_aud_row stages the row where its sets and logits fit this
constexpr int NSEL = FW_NUM_SELECTORS;

struct AudArgs {
    RowsDev R;
    int nb;
    int s[A_NBMAX];
    const float *M, *Z, *o;  // [rows], [rows], [rows][d] from the gap call
    float *G;                // ws [groups][max_n] accumulated mass
    float *vote;             // ws [groups][nb][max_n] window votes
    uint32_t *gbits;         // ws [groups][nb][2][words] H2O and SnapKV sets
    int words;
    int pm_floats;           // page maxima of the largest row (0: no budget needs them)
    float *es;               // [rows][NSEL][nb]
    uint32_t *bits;          // [rows][NSEL][nb][words] or null
};

__device__ __forceinline__ int snap_w(int s) { return max(1, min(32, s / 2)); }
__host__ __device__ __forceinline__ int quest_p(int q, int s) { return q == 0 ? (s / 4 > 2 ? s / 4 : 2) : 16; }
// Pages of a row of n keys that a warp takes by repeated arg-max; more are the block's
// radix select.  The warp reads the row once per page, the block about five times as fast
// but with barriers that cost as much as 24,000 keys.  Measured on the whole audit, one
// budget, arg-max / select, us: 256 groups of 4 rows of 4,096 keys, 8 pages 186 / 206, 10
// pages 213 / 221, 12 pages 237 / 231, 16 pages 289 / 254; 64 x 4 rows of 16,384 keys, 8
// pages 208 / 182, 16 pages 334 / 212; 128 rows of 32,768 keys, 8 pages 481 / 409, 16 pages
// 685 / 422; 300 x 4 rows of 1,000 keys, 16 pages 174 / 193.
__host__ __device__ __forceinline__ int argmax_pages(int n) { return 5 + 24000 / n; }

// ---------------------------------------------------------------- masses
__global__ void __launch_bounds__(AM_T) k_aud_mass(AudArgs a)
{
    __shared__ float sM[AM_T], sZ[AM_T];
    const int tid = threadIdx.x;
    const int Rg = a.R.R;
    for (int64_t g = blockIdx.y; g < a.R.num_groups; g += gridDim.y) {
        const int n = a.R.n[g];
        const float *lg = a.R.logits + a.R.logit_off[g];
        int wfirst[A_NBMAX];  // first row of each budget's window
#pragma unroll
        for (int b = 0; b < A_NBMAX; ++b) wfirst[b] = b < a.nb ? max(0, Rg - snap_w(a.s[b])) : Rg;
        for (int j0 = blockIdx.x * AM_T; j0 < n; j0 += gridDim.x * AM_T) {
            const int j = j0 + tid;
            float hi = 0.f, lo = 0.f;
            float vh[A_NBMAX], vl[A_NBMAX];
#pragma unroll
            for (int b = 0; b < A_NBMAX; ++b) vh[b] = vl[b] = 0.f;
            for (int i0 = 0; i0 < Rg; i0 += AM_T) {
                const int cnt = min(AM_T, Rg - i0);
                __syncthreads();
                if (tid < cnt) {
                    const int64_t r = g * Rg + i0 + tid;
                    sM[tid] = a.M[r];
                    sZ[tid] = 1.f / a.Z[r];
                }
                __syncthreads();
                if (j < n) {
                    const float *col = lg + (int64_t)i0 * n + j;
                    for (int i = 0; i < cnt; ++i) {
                        const float p = __expf(__ldg(col + (int64_t)i * n) - sM[i]) * sZ[i];
                        float t = hi + p, bb = t - hi;
                        lo += (hi - (t - bb)) + (p - bb);
                        hi = t;
#pragma unroll
                        for (int b = 0; b < A_NBMAX; ++b)
                            if (i0 + i >= wfirst[b]) {
                                t = vh[b] + p;
                                bb = t - vh[b];
                                vl[b] += (vh[b] - (t - bb)) + (p - bb);
                                vh[b] = t;
                            }
                    }
                }
            }
            if (j < n) {
                a.G[g * a.R.max_n + j] = hi + lo;
                for (int b = 0; b < a.nb; ++b) a.vote[(g * a.nb + b) * a.R.max_n + j] = vh[b] + vl[b];
            }
        }
    }
}

// ------------------------------------------------------- group-level sets
// blockIdx.x = ((group, budget), rule).  STAGED: the candidates' order keys sit
// in shared memory (n <= AS_STAGE); otherwise every pass forms them again.
template <bool STAGED>
__global__ void __launch_bounds__(AS_T) k_aud_select(AudArgs a)
{
    extern __shared__ uint32_t skeys[];
    __shared__ TopmSmem S;
    const int tid = threadIdx.x, lane = tid & 31;
    const int64_t items = a.R.num_groups * a.nb * 2;
    for (int64_t it = blockIdx.x; it < items; it += gridDim.x) {
        const int rule = (int)(it & 1);  // 0: H2O, 1: SnapKV
        const int64_t gb = it >> 1, g = gb / a.nb;
        const int b = (int)(gb - g * a.nb);
        const int n = a.R.n[g], s = a.s[b];
        uint32_t *out = a.gbits + (gb * 2 + rule) * a.words;
        if (s < 1 || s > n) {
            for (int w = tid; w < a.words; w += AS_T) out[w] = 0u;
            continue;
        }
        // H2O: the last s / 2 positions, then the largest accumulated masses;
        // SnapKV: the last w positions, then the largest pooled votes
        const int rec = rule ? snap_w(s) : s / 2;
        const int m = s - rec, lim = n - rec;
        const float *G = a.G + g * a.R.max_n;
        const float *vt = a.vote + gb * a.R.max_n;
        auto form = [&](int j) {
            if (!rule) return order_key(G[j]);
            float v = vt[j];
            for (int q = max(0, j - 3); q <= min(lim - 1, j + 3); ++q) v = fmaxf(v, vt[q]);
            return order_key(v);
        };
        auto key = [&](int j) { return STAGED ? skeys[j] : form(j); };
        __syncthreads();  // the previous item's keys are no longer read
        if (STAGED) {
            for (int j = tid; j < lim; j += AS_T) skeys[j] = form(j);
            __syncthreads();
        }
        uint32_t T = 0u;
        int L = -1;
        if (m > 0) block_topm(lim, m, key, S, T, L);
        for (int j0 = 0; j0 < a.words * 32; j0 += AS_T) {
            const int j = j0 + tid;
            bool in = j < n && j >= lim;
            if (j < lim && m > 0) {
                const uint32_t k = key(j);
                in = k > T || (k == T && j <= L);
            }
            const uint32_t bal = __ballot_sync(FW_FULL, in);
            if (lane == 0 && (j >> 5) < a.words) out[j >> 5] = bal;
        }
    }
}

// ---------------------------------------------------------- rows: score sets
// The row's logits are staged (one pad word per 32: page strides do not
// collide) when stage_n >= n.
template <int DPL, typename VT>
__global__ void __launch_bounds__(AR_T) k_aud_row(AudArgs a, int stage_n)
{
    extern __shared__ uint32_t smw[];  // [nb][2][words] Quest sets, then the page maxima or the logits
    __shared__ TopmSmem S;
    __shared__ uint16_t s_list[AR_T / 32][1024];  // members of 32 words, by warp (offsets in the words)
    constexpr int d = DPL * 32;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    uint32_t *qbits = smw;
    float *pm = reinterpret_cast<float *>(smw + a.nb * 2 * a.words);
    float *sl = pm + a.pm_floats;
    for (int64_t row = blockIdx.x; row < a.R.rows; row += gridDim.x) {
        const int64_t g = row / a.R.R;
        const int n = a.R.n[g];
        const float *l = a.R.logits + a.R.logit_off[g] + (row - g * a.R.R) * n;
        const VT *V = static_cast<const VT *>(a.R.v) + a.R.v_off[g];
        const float M = a.M[row], Zi = 1.f / a.Z[row];
        const bool staged = n <= stage_n;
        auto at = [&](int j) { return staged ? sl[j + (j >> 5)] : __ldg(l + j); };
        __syncthreads();  // the previous row's sets and logits are no longer read
        if (staged)
            for (int j = tid; j < n; j += AR_T) sl[j + (j >> 5)] = __ldg(l + j);
        for (int w = tid; w < a.nb * 2 * a.words; w += AR_T) qbits[w] = 0u;
        __syncthreads();
        // Quest sets of few pages: a warp per (budget, page size) takes the
        // largest page after the last one taken (value descending, page
        // ascending), mp times
        for (int bq = wid; bq < a.nb * 2; bq += AR_T / 32) {
            const int b = bq >> 1, q = bq & 1, s = a.s[b];
            const int P = quest_p(q, s), np = (n + P - 1) / P, mp = s / P;
            if (!(s >= 1 && s <= n && mp >= 1 && mp <= argmax_pages(n) && (q == 0 || s >= 16))) continue;
            uint32_t *qb = qbits + bq * a.words;
            uint32_t lk = 0xffffffffu;
            int lp = -1;
            for (int t = 0; t < min(mp, np); ++t) {
                uint32_t bk = 0u;
                int bp = INT_MAX;
                for (int p = lane; p < np; p += 32) {
                    float m = -INFINITY;
                    const int j1 = min(n, p * P + P);
                    for (int j = p * P; j < j1; ++j) m = fmaxf(m, at(j));
                    const uint32_t k = order_key(m);
                    if ((k < lk || (k == lk && p > lp)) && (k > bk || bp == INT_MAX)) {
                        bk = k;
                        bp = p;
                    }
                }
                // the largest key, then its first page
                const uint32_t wk = __reduce_max_sync(FW_FULL, bp == INT_MAX ? 0u : bk);
                const int wp = (int)__reduce_min_sync(FW_FULL, bp != INT_MAX && bk == wk ? (uint32_t)bp : 0x7fffffffu);
                lk = wk;
                lp = wp;
                for (int j = wp * P + lane; j < min(n, wp * P + P); j += 32) atomicOr(&qb[j >> 5], 1u << (j & 31));
            }
        }
        // ... of many pages: page maxima and a radix top-m by the block
        for (int bq = 0; bq < a.nb * 2; ++bq) {
            const int b = bq >> 1, q = bq & 1, s = a.s[b];
            const int P = quest_p(q, s), np = (n + P - 1) / P, mp = s / P;
            if (!(s >= 1 && s <= n && mp > argmax_pages(n) && (q == 0 || s >= 16))) continue;
            uint32_t *qb = qbits + bq * a.words;
            __syncthreads();  // pm is free
            for (int p = tid; p < np; p += AR_T) {
                float m = -INFINITY;
                for (int j = p * P; j < min(n, p * P + P); ++j) m = fmaxf(m, at(j));
                pm[p] = m;
            }
            __syncthreads();
            uint32_t T = 0u;
            int L = -1;
            block_topm(np, min(mp, np), [&](int p) { return order_key(pm[p]); }, S, T, L);
            for (int j0 = 0; j0 < n; j0 += AR_T) {
                const int j = j0 + tid;
                bool in = false;
                if (j < n) {
                    const int p = j / P;
                    const uint32_t k = order_key(pm[p]);
                    in = k > T || (k == T && p <= L);
                }
                const uint32_t bal = __ballot_sync(FW_FULL, in);
                if (lane == 0 && j < n) qb[j >> 5] = bal;
            }
        }
        __syncthreads();
        // one warp per (rule, budget): list the members, gather them, form es
        float ol[DPL];
#pragma unroll
        for (int c = 0; c < DPL; ++c) ol[c] = a.o[row * d + lane * DPL + c];
        for (int set = wid; set < NSEL * a.nb; set += AR_T / 32) {
            const int sel = set / a.nb, b = set - sel * a.nb;
            const int s = a.s[b];
            const uint32_t *src = nullptr;
            if (sel == FW_SEL_H2O) src = a.gbits + ((g * a.nb + b) * 2 + 0) * a.words;
            if (sel == FW_SEL_SNAPKV) src = a.gbits + ((g * a.nb + b) * 2 + 1) * a.words;
            if (sel == FW_SEL_QUEST) src = qbits + (b * 2 + 0) * a.words;
            if (sel == FW_SEL_QUEST16) src = qbits + (b * 2 + 1) * a.words;
            const int sinks = min(4, s / 2);
            // bits [lo, hi) of the word whose first key is j0
            auto span = [](int j0, int lo, int hi) {
                const int x = max(lo - j0, 0), y = min(hi - j0, 32);
                return y <= x ? 0u : (y == 32 ? ~0u : (1u << y) - 1u) & ~((1u << x) - 1u);
            };
            float N[DPL];
#pragma unroll
            for (int c = 0; c < DPL; ++c) N[c] = 0.f;
            float pA = 0.f;
            int cnt = 0;
            const int nw = (n + 31) / 32;
            uint16_t *list = s_list[wid];
            for (int w0 = 0; w0 < nw; w0 += 32) {
                const int w = w0 + lane;
                uint32_t word = 0u;
                if (w < nw) {
                    if (sel == FW_SEL_STREAMING) {
                        if (s >= 1 && s <= n) word = span(w * 32, 0, sinks) | span(w * 32, n - (s - sinks), n);
                    } else {
                        word = src[w];
                    }
                    if (a.bits) a.bits[((row * NSEL + sel) * a.nb + b) * (int64_t)a.words + w] = word;
                }
                if (!__any_sync(FW_FULL, word != 0u)) continue;
                // the members of these words in index order
                int off = __popc(word);
                const int own = off;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const int y = __shfl_up_sync(FW_FULL, off, o);
                    if (lane >= o) off += y;
                }
                const int tot = __shfl_sync(FW_FULL, off, 31);
                off -= own;
                __syncwarp();  // the previous list is no longer read
                for (uint32_t mw = word; mw; mw &= mw - 1) list[off++] = (uint16_t)(lane * 32 + __ffs(mw) - 1);
                __syncwarp();
                cnt += tot;
                for (int i0 = 0; i0 < tot; i0 += 32) {
                    const int i = i0 + lane;
                    int j = 0;
                    float p = 0.f;
                    if (i < tot) {
                        j = w0 * 32 + list[i];
                        p = __expf(__ldg(l + j) - M) * Zi;
                    }
                    pA += p;
                    const int lim = min(32, tot - i0);
                    for (int e0 = 0; e0 < lim; e0 += 8) {  // 8 value rows in flight (mass 0 past the last)
                        float x[8][DPL], pe[8];
#pragma unroll
                        for (int e = 0; e < 8; ++e) {
                            const int je = __shfl_sync(FW_FULL, j, e0 + e);
                            pe[e] = __shfl_sync(FW_FULL, p, e0 + e);
#pragma unroll
                            for (int c = 0; c < DPL; ++c) x[e][c] = load_v(V, (int64_t)je * d + lane * DPL + c);
                        }
#pragma unroll
                        for (int e = 0; e < 8; ++e)
                            if (e0 + e < lim)
#pragma unroll
                                for (int c = 0; c < DPL; ++c) N[c] = fmaf(pe[e], x[e][c], N[c]);
                    }
                }
            }
            pA = warp_sum(pA);
            float e2 = 0.f;
#pragma unroll
            for (int c = 0; c < DPL; ++c) {
                const float diff = N[c] / pA - ol[c];
                e2 = fmaf(diff, diff, e2);
            }
            e2 = warp_sum(e2);
            if (lane == 0) a.es[(row * NSEL + sel) * a.nb + b] = cnt > 0 ? sqrtf(e2) : __int_as_float(0x7fc00000);
        }
    }
}

}  // namespace

static size_t aud_words(const RowsDev &R) { return (size_t)(R.max_n + 31) / 32; }

size_t selector_audit_workspace(const RowsDev &R, int nb)
{
    return align256((size_t)R.num_groups * R.max_n * 4) + align256((size_t)R.num_groups * nb * R.max_n * 4) +
           align256((size_t)R.num_groups * nb * 2 * aud_words(R) * 4);
}

fw_status selector_audit(const RowsDev &R, const int32_t *s, int nb, const fw_gap_out &topk, float *es,
                         uint32_t *bits, int words, void *ws, cudaStream_t st)
{
    AudArgs a;
    a.R = R;
    a.nb = nb;
    for (int b = 0; b < A_NBMAX; ++b) a.s[b] = b < nb ? s[b] : 0;
    a.M = topk.row_max;
    a.Z = topk.row_sum;
    a.o = topk.o;
    char *w = (char *)ws;
    a.G = (float *)w;
    w += align256((size_t)R.num_groups * R.max_n * 4);
    a.vote = (float *)w;
    w += align256((size_t)R.num_groups * nb * R.max_n * 4);
    a.gbits = (uint32_t *)w;
    a.words = (int)aud_words(R);
    a.es = es;
    a.bits = bits;
    if (bits && words != a.words) return FW_ERR_INVALID_ARG;
    int sms = 0;
    if (device_sms(&sms) != FW_OK) return FW_ERR_CUDA;
    const int64_t chunks = (R.max_n + AM_T - 1) / AM_T;
    const int64_t per_group = std::max<int64_t>(1, ((int64_t)sms * 8 + R.num_groups - 1) / R.num_groups);
    const dim3 gm((unsigned)std::min(chunks, per_group), (unsigned)std::min<int64_t>(R.num_groups, 65535));
    FW_LAUNCH(k_aud_mass, gm, AM_T, 0, st, a);
    const unsigned gs = (unsigned)std::min<int64_t>(R.num_groups * nb * 2, 1 << 20);
    if (R.max_n <= AS_STAGE) {
        const size_t sk = (size_t)R.max_n * 4;
        FW_CUDA_CHECK(cudaFuncSetAttribute(k_aud_select<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sk));
        FW_LAUNCH(k_aud_select<true>, gs, AS_T, sk, st, a);
    } else {
        FW_LAUNCH(k_aud_select<false>, gs, AS_T, 0, st, a);
    }
    a.pm_floats = 0;
    for (int b = 0; b < nb; ++b)
        for (int q = 0; q < 2; ++q) {
            const int P = quest_p(q, s[b]);
            if (s[b] / P > argmax_pages(R.max_n)) a.pm_floats = std::max(a.pm_floats, (R.max_n + P - 1) / P);
        }
    const size_t sets = ((size_t)nb * 2 * a.words + a.pm_floats) * 4, lrow = ((size_t)R.max_n + (R.max_n >> 5) + 1) * 4;
    const int stage_n = sets + lrow <= AR_SMEM ? R.max_n : 0;
    const size_t smem = sets + (stage_n ? lrow : 0);
    FW_DISPATCH(R.d, R.v_dtype, {
        FW_CUDA_CHECK(cudaFuncSetAttribute(k_aud_row<DPL, VT>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
        FW_LAUNCH((k_aud_row<DPL, VT>), (unsigned)std::min<int64_t>(R.rows, (int64_t)sms * 16), AR_T, smem, st, a, stage_n);
    });
    return FW_OK;
}

}  // namespace fw

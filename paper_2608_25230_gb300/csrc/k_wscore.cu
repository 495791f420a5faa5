// k_wscore.cu -- the observation-window importance score that Sec. 4 runs
// ContourKV with (SnapKV's score): the last w query rows of a cell (KV head)
// vote for the keys they attend to, and the votes are max-pooled along the
// positions.  For cell c with keys k_j (j < T) and window queries q_i
// (i < w, query i at position T - w + i, so it sees keys j <= T - w + i):
//   a_ij   = softmax over the visible j of scale * q_i . k_j,
//   vote_j = sum_i a_ij,
//   r_j    = max of vote over [j - h, j + h] clipped to the prefix [0, T - w)
//            for prefix positions (h = pool / 2), r_j = vote_j in the window.
//
// A cell's keys are split over S slices, a CTA each, and two launches read them:
// k_wscore<1> keeps every query's softmax statistics over the slice, k_wscore<2>
// merges the slices' statistics and writes the votes; k_wpool takes the window
// maxima of the votes.  Each is a GEMM of 128-key tiles against the window:
// D[128 keys][32 queries] = K_tile (128 x d, K-major) x Q^T (d x 32, K-major)
// on tcgen05 (bf16 x bf16 -> fp32 in TMEM), the K tiles brought in by TMA
// (128-byte swizzle, three stages), the window queries by TMA once per CTA.
// Warp 0 issues the TMA loads, warp 1 the MMAs (and owns the TMEM: four
// accumulators of 32 columns), warps 2-9 read the accumulators, two warps per
// TMEM lane quarter: in the first launch each takes half of the queries, in the
// second every other tile.  Every wait is bounded; a wait that gives up marks
// the cell FW_ERR_TIMEOUT, the warps keep their loop shape, in-flight copies
// are waited for, and the TMEM is freed.
//
// Bound: HBM, the keys read twice.  256 cells x 32,768 keys, d = 128: 0.65 ms,
// 6.6 TB/s; one CTA per cell with four epilogue warps, a true running maximum
// (nine operations per element in the first pass instead of four) and both
// passes in one launch took 2.02 ms, and 0.89 ms for 8 cells (now 0.06).
#include <cuda.h>  // CUtensorMap and its enums (the encoder comes from the driver at run time)

#include <algorithm>

#include "fw_internal.h"
#include "tc_sm100.cuh"

namespace fw {
namespace {

constexpr int WS_KT = 128;                 // keys per tile: the MMA's M
constexpr int WS_N = 32;                   // window queries per tile: the MMA's N (w <= 32, padded)
constexpr int WS_H = WS_N / 2;             // queries per warp in the statistics launch
constexpr int WS_STAGES = 3;               // K tiles in flight
constexpr int WS_ACC = 4;                  // accumulators in TMEM
constexpr int WS_EW = 8;                   // epilogue warps
constexpr int WS_THREADS = 64 + 32 * WS_EW;
constexpr int WS_SMAX = 64;                // slices of a cell at most
constexpr uint32_t WS_WAIT = 1u << 22;     // polls before a wait gives up
constexpr int WP_T = 256;                  // k_wpool threads

struct WsArgs {
    int cells, T, w, ph;  // ph: half-width of the max pool
    int S, tps;           // slices per cell, tiles per slice
    float scale2;         // scale * log2(e): logits in base-2 units
    float *votes;         // workspace [cells][T]
    float *scores;        // [cells][T]
    int32_t *status;      // [cells] or null
};

// A slice's softmax statistics of query i -- a reference logit and the sum of 2^(x -
// reference), -1 where a wait of the slice's CTA gave up -- sit between the two launches
// in the cell's part of the scores, which nothing else uses before k_wpool writes them:
// 2 WS_N floats a slice (slices hold at least 4 tiles where there are several).  A cell
// of one slice may be shorter than that, so its sums wait among its votes, which its CTA
// writes after it has read them.
static_assert((4 * 2 - 4) * WS_KT + 1 >= 2 * 2 * WS_N, "statistics of two slices");
__device__ __forceinline__ float *stat_ref(const WsArgs &a, int c, int sl)
{
    return a.scores + (int64_t)c * a.T + sl * 2 * WS_N;
}
__device__ __forceinline__ float *stat_sum(const WsArgs &a, int c, int sl)
{
    return a.S == 1 ? a.votes + (int64_t)c * a.T : stat_ref(a, c, sl) + WS_N;
}

// 2^x by the hardware approximation (ex2.approx.ftz: ~2 ulp, well inside the
// score's 1e-4 tolerance); the per-(key, query) exponentials are most of the
// epilogue's work
__device__ __forceinline__ float ex2a(float x)
{
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// combine two (reference, sum of 2^(x - reference)) pairs; -inf: nothing seen
__device__ __forceinline__ void ms_merge(float &m, float &z, float m2, float z2)
{
    const float mn = fmaxf(m, m2);
    const float a = m == -INFINITY ? 0.f : z * exp2f(m - mn);
    const float b = m2 == -INFINITY ? 0.f : z2 * exp2f(m2 - mn);
    m = mn;
    z = a + b;
}

template <int D, int PASS>
__global__ void __launch_bounds__(WS_THREADS, 2) k_wscore(const __grid_constant__ CUtensorMap tmK,
                                                          const __grid_constant__ CUtensorMap tmQ, const WsArgs a)
{
    constexpr int NBOX = D / 64;          // 128-byte boxes across d
    constexpr int KBOX = WS_KT * 128;     // bytes of one K box
    constexpr int KSTAGE = NBOX * KBOX;   // bytes of one K tile
    constexpr int QBOX = WS_N * 128;      // bytes of one Q box
    // warps that read one accumulator: all, or the tile's half of them
    constexpr int READERS = PASS == 1 ? WS_EW : WS_EW / 2;
    extern __shared__ uint8_t smraw[];
    uint8_t *sm = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smraw) + 1023) & ~(uintptr_t)1023);
    uint8_t *sK = sm;                            // [STAGES][NBOX][128 rows x 128 B]
    uint8_t *sQ = sm + WS_STAGES * KSTAGE;       // [NBOX][32 rows x 128 B]
    __shared__ __align__(8) uint64_t full[WS_STAGES], empty[WS_STAGES], accfull[WS_ACC], accempty[WS_ACC], qfull;
    __shared__ uint32_t s_taddr;
    __shared__ int s_err;
    __shared__ float2 s_mz[WS_EW / 2][WS_N];     // pass 1: (reference, sum) by lane quarter
    __shared__ __align__(16) float2 s_st[WS_N];  // pass 2: (max, 1 / sum) of every query

    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int c = blockIdx.x / a.S, sl = blockIdx.x - c * a.S;
    const int T = a.T, w = a.w;
    const int ntiles = (T + WS_KT - 1) / WS_KT;
    const int t0 = sl * a.tps, total = min(ntiles, t0 + a.tps) - t0;  // (total >= 1: the launch's slices cover the tiles)
    if (tid == 0) {
        for (int s = 0; s < WS_STAGES; ++s) {
            tc::mbar_init(&full[s], 1);
            tc::mbar_init(&empty[s], 1);
        }
        for (int b = 0; b < WS_ACC; ++b) {
            tc::mbar_init(&accfull[b], 1);
            tc::mbar_init(&accempty[b], READERS);
        }
        tc::mbar_init(&qfull, 1);
        tc::mbar_init_fence();
        s_err = 0;
    }
    if (wid == 1) tc::tmem_alloc(&s_taddr, WS_ACC * WS_N);
    bool lost = false;
    if (PASS == 2 && tid >= 64 && tid < 64 + w) {
        // the softmax statistics of every query over all keys of the cell
        const int i = tid - 64;
        float m = -INFINITY, z = 0.f;
        for (int s = 0; s < a.S; ++s) {
            const float zs = stat_sum(a, c, s)[i];
            lost |= zs < 0.f;
            ms_merge(m, z, stat_ref(a, c, s)[i], zs);
        }
        s_st[i] = make_float2(m, z > 0.f ? 1.f / z : 0.f);
    }
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    const uint32_t taddr = s_taddr;

    if (wid == 0) {
        // -------------------------------------------------------------- TMA
        if (lane == 0) {
            tc::tma_prefetch_desc(&tmK);
            tc::tma_prefetch_desc(&tmQ);
            tc::mbar_arrive_expect_tx(&qfull, NBOX * QBOX);
            for (int h = 0; h < NBOX; ++h) tc::tma_load_2d(sQ + h * QBOX, &tmQ, 64 * h, c * w, &qfull);
            int issued = 0;
            bool ok = true;
            for (int it = 0; it < total; ++it) {
                const int s = it % WS_STAGES;
                if (it >= WS_STAGES && !tc::mbar_wait(&empty[s], (uint32_t)((it / WS_STAGES) - 1) & 1u, WS_WAIT)) {
                    ok = false;
                    break;
                }
                tc::mbar_arrive_expect_tx(&full[s], KSTAGE);
                for (int h = 0; h < NBOX; ++h)
                    tc::tma_load_2d(sK + s * KSTAGE + h * KBOX, &tmK, 64 * h, c * T + (t0 + it) * WS_KT, &full[s]);
                ++issued;
            }
            if (!ok) atomicOr(&s_err, 1);
            // every copy this thread started has landed before the CTA moves on
            // (already so when the MMAs consumed them)
            for (int it = issued - WS_STAGES < 0 ? 0 : issued - WS_STAGES; it < issued; ++it)
                if (!tc::mbar_wait(&full[it % WS_STAGES], (uint32_t)(it / WS_STAGES) & 1u, WS_WAIT)) atomicOr(&s_err, 1);
            if (!tc::mbar_wait(&qfull, 0, WS_WAIT)) atomicOr(&s_err, 1);
        }
        __syncwarp();
    } else if (wid == 1) {
        // -------------------------------------------------------------- MMA
        if (lane == 0) {
            constexpr uint32_t idesc = tc::idesc_bf16_f32(WS_KT, WS_N, false, false);
            const uint32_t k0 = tc::smem_u32(sK), q0 = tc::smem_u32(sQ);
            bool ok = tc::mbar_wait(&qfull, 0, WS_WAIT);
            int last = -1;
            for (int it = 0; ok && it < total; ++it) {
                const int s = it % WS_STAGES, b = it % WS_ACC;
                ok = tc::mbar_wait(&full[s], (uint32_t)(it / WS_STAGES) & 1u, WS_WAIT);
                if (ok && it >= WS_ACC)
                    ok = tc::mbar_wait(&accempty[b], (uint32_t)((it / WS_ACC) - 1) & 1u, WS_WAIT);
                if (!ok) break;
                tc::fence_after_sync();
#pragma unroll
                for (int ks = 0; ks < D / 16; ++ks) {
                    const int h = ks >> 2, off = (ks & 3) * 32;
                    const uint64_t ad = tc::sdesc_sw128(k0 + s * KSTAGE + h * KBOX + off, 16, 1024);
                    const uint64_t bd = tc::sdesc_sw128(q0 + h * QBOX + off, 16, 1024);
                    tc::mma_bf16(taddr + (uint32_t)(b * WS_N), ad, bd, idesc, ks > 0);
                }
                tc::commit(&empty[s]);
                tc::commit(&accfull[b]);
                last = it;
            }
            if (!ok) atomicOr(&s_err, 1);
            // the last MMAs have completed before the TMEM can be freed
            if (last >= 0 && !tc::mbar_wait(&accfull[last % WS_ACC], (uint32_t)(last / WS_ACC) & 1u, WS_WAIT))
                atomicOr(&s_err, 1);
        }
        __syncwarp();
    } else {
        // --------------------------------------------------------- epilogue
        const int q4 = wid & 3;           // the TMEM lane quarter this warp may read
        const int half = (wid - 2) >> 2;  // pass 1: its half of the queries; pass 2: its tiles' parity
        const float scale2 = a.scale2;
        const int lim = T - w;  // query i sees keys j <= lim + i
        const uint32_t lbase = taddr + ((uint32_t)(q4 * 32) << 16);
        bool ok = true;
        if constexpr (PASS == 1) {
            // Per lane and query a reference r (a logit seen) and z = the sum of
            // 2^(x - r): one exponential and two adds per element.  The
            // reference only moves when a logit exceeds it by 2^6 octaves (a
            // rescale then), so no sum can overflow and what underflows is
            // below 2^-126 of the largest term.
            float r[WS_H], z[WS_H];
#pragma unroll
            for (int i = 0; i < WS_H; ++i) {
                r[i] = -INFINITY;
                z[i] = 0.f;
            }
            bool first = true;
            for (int it = 0; it < total; ++it) {
                const int b = it % WS_ACC;
                if (ok) ok = tc::mbar_wait(&accfull[b], (uint32_t)(it / WS_ACC) & 1u, WS_WAIT);
                float v[WS_H];
                if (ok) {
                    tc::fence_after_sync();
                    tc::ld16(lbase + (uint32_t)(b * WS_N + half * WS_H), v);
                    tc::fence_before_sync();
                }
                __syncwarp();
                if (ok && lane == 0) tc::mbar_arrive(&accempty[b]);
                if (!ok) continue;
                const int j = (t0 + it) * WS_KT + q4 * 32 + lane;
                // a tile whose keys every query sees (all but the cell's last) skips the masks
                const bool open = (t0 + it + 1) * WS_KT - 1 <= lim;
                if (open && !first) {
                    float top = -INFINITY;
                    float dx[WS_H];
#pragma unroll
                    for (int i = 0; i < WS_H; ++i) {
                        dx[i] = fmaf(v[i], scale2, -r[i]);
                        top = fmaxf(top, dx[i]);
                    }
                    if (top <= 64.f) {
#pragma unroll
                        for (int i = 0; i < WS_H; ++i) z[i] += ex2a(dx[i]);
                        continue;
                    }
                }
#pragma unroll
                for (int i = 0; i < WS_H; ++i) {
                    const int qi = half * WS_H + i;
                    if (open || (j < T && j <= lim + qi)) {
                        const float x = v[i] * scale2;
                        const float d = x - r[i];
                        if (d <= 64.f) {
                            z[i] += ex2a(d);
                        } else {  // (also the first key seen: r = -inf)
                            z[i] = fmaf(z[i], r[i] == -INFINITY ? 0.f : ex2a(-d), 1.f);
                            r[i] = x;
                        }
                    }
                }
                // queries past the window read other rows: their references may be anything
                first = false;
#pragma unroll
                for (int i = 0; i < WS_H; ++i) first |= r[i] == -INFINITY;
            }
            if (!ok) atomicOr(&s_err, 1);
#pragma unroll
            for (int i = 0; i < WS_H; ++i) {
                float mi = r[i], zi = z[i];
#pragma unroll
                for (int o = 16; o > 0; o >>= 1)
                    ms_merge(mi, zi, __shfl_xor_sync(FW_FULL, mi, o), __shfl_xor_sync(FW_FULL, zi, o));
                if (lane == 0) s_mz[q4][half * WS_H + i] = make_float2(mi, zi);
            }
        } else {
            for (int it = half; it < total; it += 2) {
                const int b = it % WS_ACC;
                if (ok) ok = tc::mbar_wait(&accfull[b], (uint32_t)(it / WS_ACC) & 1u, WS_WAIT);
                float v[WS_N];
                if (ok) {
                    tc::fence_after_sync();
                    tc::ld32(lbase + (uint32_t)(b * WS_N), v);
                    tc::fence_before_sync();
                }
                __syncwarp();
                if (ok && lane == 0) tc::mbar_arrive(&accempty[b]);
                if (!ok) continue;
                const int j = (t0 + it) * WS_KT + q4 * 32 + lane;
                const bool open = (t0 + it + 1) * WS_KT - 1 <= lim;
                if (j < T) {
                    float vote = 0.f, vote2 = 0.f;
#pragma unroll
                    for (int i = 0; i < WS_N; i += 2) {
                        const float4 st = *reinterpret_cast<const float4 *>(&s_st[i]);
                        if (i < w && (open || j <= lim + i)) vote = fmaf(ex2a(fmaf(v[i], scale2, -st.x)), st.y, vote);
                        if (i + 1 < w && (open || j <= lim + i + 1))
                            vote2 = fmaf(ex2a(fmaf(v[i + 1], scale2, -st.z)), st.w, vote2);
                    }
                    a.votes[(int64_t)c * T + j] = vote + vote2;
                }
            }
            if (!ok) atomicOr(&s_err, 1);
        }
    }
    tc::fence_before_sync();
    __syncthreads();
    if (PASS == 1 && tid < w) {
        float m = -INFINITY, z = 0.f;
        for (int q = 0; q < WS_EW / 2; ++q) ms_merge(m, z, s_mz[q][tid].x, s_mz[q][tid].y);
        stat_ref(a, c, sl)[tid] = m;
        stat_sum(a, c, sl)[tid] = s_err ? -1.f : z;
    }
    // the cell's status: OK by the first launch, a failure of either by the second
    if (PASS == 1 && tid == 0 && sl == 0 && a.status) a.status[c] = FW_OK;
    if (PASS == 2 && a.status && (lost || (tid == 0 && s_err))) a.status[c] = FW_ERR_TIMEOUT;
    if (wid == 1) {
        tc::fence_after_sync();
        tc::tmem_dealloc(taddr, WS_ACC * WS_N);
    }
}

// Max pooling of the votes along the prefix positions (window positions keep
// their own).
__global__ void __launch_bounds__(WP_T) k_wpool(const WsArgs a)
{
    const int c = blockIdx.y, lim = a.T - a.w;
    const float *vc = a.votes + (int64_t)c * a.T;
    for (int j = blockIdx.x * WP_T + threadIdx.x; j < a.T; j += gridDim.x * WP_T) {
        float r = vc[j];
        if (j < lim) {
            const int lo = j - a.ph < 0 ? 0 : j - a.ph, hi = j + a.ph < lim ? j + a.ph : lim - 1;
            for (int q = lo; q <= hi; ++q) r = fmaxf(r, vc[q]);
        }
        a.scores[(int64_t)c * a.T + j] = r;
    }
}

// tiles per slice: enough CTAs for several waves of two per SM, at least four
// tiles each (a CTA's setup is about one tile's time), at most WS_SMAX slices
int slice_tiles(int cells, int T)
{
    int sms = 0;
    if (device_sms(&sms) != FW_OK) sms = 152;  // no device: the size query still answers
    const int ntiles = (T + WS_KT - 1) / WS_KT;
    const int64_t want = std::max<int64_t>(1, ((int64_t)sms * 2 * 6 + cells - 1) / cells);
    const int S = (int)std::min<int64_t>({want, (ntiles + 3) / 4, WS_SMAX});
    return (ntiles + S - 1) / S;
}

}  // namespace

size_t window_score_workspace(int cells, int T) { return align256((size_t)cells * T * 4); }

fw_status window_score(const void *Qw, const void *K, int cells, int T, int d, int w, float scale, int pool,
                       float *scores, void *ws, int32_t *status, cudaStream_t s)
{
    CUtensorMap mk, mq;
    if (!make_tma_2d_bf16(&mk, K, (uint64_t)cells * T, (uint64_t)d, WS_KT)) return FW_ERR_CUDA;
    if (!make_tma_2d_bf16(&mq, Qw, (uint64_t)cells * w, (uint64_t)d, WS_N)) return FW_ERR_CUDA;
    WsArgs a;
    a.cells = cells;
    a.T = T;
    a.w = w;
    a.ph = pool / 2;
    a.tps = slice_tiles(cells, T);
    a.S = ((T + WS_KT - 1) / WS_KT + a.tps - 1) / a.tps;
    a.scale2 = scale * 1.4426950408889634f;
    a.votes = (float *)ws;
    a.scores = scores;
    a.status = status;
    auto launch = [&](auto kernel, int nbox) -> fw_status {
        const size_t smem = 1024 + (size_t)WS_STAGES * nbox * WS_KT * 128 + (size_t)nbox * WS_N * 128;
        FW_CUDA_CHECK(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
        FW_LAUNCH(kernel, (unsigned)(cells * a.S), WS_THREADS, smem, s, mk, mq, a);
        return FW_OK;
    };
    fw_status st = d == 128 ? launch(k_wscore<128, 1>, 2) : launch(k_wscore<64, 1>, 1);
    if (st != FW_OK) return st;
    st = d == 128 ? launch(k_wscore<128, 2>, 2) : launch(k_wscore<64, 2>, 1);
    if (st != FW_OK) return st;
    for (int c0 = 0; c0 < cells; c0 += 65535) {  // (the grid's y limit)
        WsArgs b = a;
        const int nc = std::min(cells - c0, 65535);
        b.votes += (int64_t)c0 * T;
        b.scores += (int64_t)c0 * T;
        const dim3 grid((unsigned)std::min((T + WP_T - 1) / WP_T, 64), (unsigned)nc);
        FW_LAUNCH(k_wpool, grid, WP_T, 0, s, b);
    }
    return FW_OK;
}

}  // namespace fw

// K3 bin finish + HNEMA sums (Eq. 19), K4 GKMA lag correlation (Eq. 17 integrand),
// K5 running Green-Kubo integral (Eq. 17) and the HNEMA normalisation (Eq. 19).
#include <algorithm>
#include <cmath>

#include "common.cuh"
#include "kernels.h"

namespace mhc {

namespace {

// ------------------------------------------------------------------ K3
// One CTA per bin, thread t on component t % 3 of the steps t / 3 + steps j (bf_threads(K) = 3 steps
// threads): J_b^a(k) = sum of the bin's partial slots in slot order, and the HNEMA sums over the
// block's steps in FP64.  One CTA more sums the total current.  Bound by latency (three dependent
// round trips to memory: slots, sums, the HNEMA sum), so eight of a thread's slots (of one step, or
// of four steps where a block has that many a thread) are in flight together, and the FP64 sums are
// reduced by one barrier and a warp a component, with one read-modify-write of the sum at the end.
// The order of the sums depends on K alone, so a grouped launch gives the bits of a solo one.  It is
// launched plainly: as a programmatic dependent of the projection it made the 8000-atom push 20 us
// and the 512-atom push 2 us longer.
// Measured (ncu, us, one thread a step with a tree of FP64 sums -> now): 600 rows, K = 128 10.4 -> 6.4;
// 200 rows, K = 128 6.8 -> 5.0; 16 systems of 52 bins, K = 256 21.7 -> 16.8; 100 rows, K = 1000 8.7
// -> 7.9; 64 rows of 13 slots, K = 256 7.5 -> 6.5; 100 and 304 rows of a slot or none, K = 200 4.9 ->
// 4.9, K = 1000 9.7 -> 10.4.
constexpr int BF_MAX_THREADS = 768;
__host__ __device__ constexpr int bf_threads(int K) { return K <= 128 ? 384 : BF_MAX_THREADS; }

// (Plain loads: a bin's slots share sectors, so most of them hit L1.)
// J_b^a of the steps k0, k0 + steps, ..: the bin's slots [s0, s1) added in order, QU slots of
// PASSES steps loaded at a time; the sum over the steps in hs.
template <int PASSES, int QU>
__device__ __forceinline__ void bf_steps(const float *partials, int n_slots, int s0, int s1,
                                         int b, int a, int B, int K, int k0, int steps, float *Jb,
                                         double &hs) {
    for (int k = k0; k < K; k += PASSES * steps) {
        float s[PASSES];
#pragma unroll
        for (int u = 0; u < PASSES; ++u) s[u] = 0.f;
        for (int q = s0; q < s1; q += QU) {
            float v[QU][PASSES];
#pragma unroll
            for (int w = 0; w < QU; ++w)
#pragma unroll
                for (int u = 0; u < PASSES; ++u)
                    v[w][u] = q + w < s1 && k + u * steps < K
                                  ? partials[((size_t)(k + u * steps) * 3 + a) * n_slots + q + w]
                                  : 0.f;
#pragma unroll
            for (int w = 0; w < QU; ++w)
                if (q + w < s1)
#pragma unroll
                    for (int u = 0; u < PASSES; ++u) s[u] += v[w][u];
        }
#pragma unroll
        for (int u = 0; u < PASSES; ++u)
            if (k + u * steps < K) {
                Jb[((size_t)(k + u * steps) * B + b) * 3 + a] = s[u];
                hs += (double)s[u];
            }
    }
}

__device__ __forceinline__ void bin_finish_body(const float *partials, int n_slots,
                                                const int *slot_begin, int B, int K, float *Jb,
                                                double *hsum, const double *Jtot, double *Jsum,
                                                int b) {
    __shared__ double red[BF_MAX_THREADS];
    const int nt = bf_threads(K), steps = nt / 3;   // threads past nt (a longer system's) hold no steps
    const int t = threadIdx.x, a = t % 3, k0 = t / 3;
    const int lane = t & 31, warp = t >> 5;
    if (b == B) {   // the total current, two warps a component (sums on all warps took this CTA 3 us more)
        if (warp < 6) {
            double acc = 0.0;
#pragma unroll 4
            for (int k = 32 * (warp / 3) + lane; k < K; k += 64) acc += Jtot[3 * k + warp % 3];
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(FULL_MASK, acc, o);
            if (lane == 0) red[warp] = acc;
        }
        __syncthreads();
        if (t < 3) Jsum[t] += red[t] + red[t + 3];
        return;
    }
    const int s0 = slot_begin[b], s1 = slot_begin[b + 1];
    const double old = t < 96 && lane == 0 ? hsum[b * 3 + warp] : 0.0;   // warp = component below
    double hs = 0.0;
    if (K <= steps) bf_steps<1, 8>(partials, n_slots, s0, s1, b, a, B, K, k0, steps, Jb, hs);
    else if (t < nt) bf_steps<4, 2>(partials, n_slots, s0, s1, b, a, B, K, k0, steps, Jb, hs);
    red[t] = hs;
    __syncthreads();
    if (warp < 3) {   // component `warp`: lane l the threads 3 (l + 32 j) + warp, then the lanes
        hs = 0.0;
        for (int j = lane; j < steps; j += 32) hs += red[3 * j + warp];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) hs += __shfl_down_sync(FULL_MASK, hs, o);
        if (lane == 0) hsum[b * 3 + warp] = old + hs;
    }
}

// steps: the step counter, advanced by K here, or null.
__global__ void __launch_bounds__(BF_MAX_THREADS, 2) bin_finish_kernel(const float *partials,
                                                                    int n_slots, const int *slot_begin,
                                                                    int B, int K, float *Jb,
                                                                    double *hsum, const double *Jtot,
                                                                    double *Jsum, long long *steps) {
    if (steps && blockIdx.x == 0 && threadIdx.x == 0) *steps += K;
    bin_finish_body(partials, n_slots, slot_begin, B, K, Jb, hsum, Jtot, Jsum, blockIdx.x);
}

// All systems of a group in one launch: CTAs cta_begin[j] .. cta_begin[j+1) are system j's bins
// and its total current.
__global__ void __launch_bounds__(BF_MAX_THREADS, 2) bin_finish_group_kernel(const __grid_constant__ FinishGroupArgs g) {
    int j = 0;
    while (j + 1 < g.n && (int)blockIdx.x >= g.cta_begin[j + 1]) ++j;
    if ((int)blockIdx.x == g.cta_begin[j] && threadIdx.x == 0) *g.steps[j] += g.K[j];
    bin_finish_body(g.partials[j], g.n_slots[j], g.slot_begin[j], g.B[j], g.K[j], g.Jb[j],
                    g.hsum[j], g.Jtot[j], g.Jsum[j], (int)blockIdx.x - g.cta_begin[j]);
}

// ------------------------------------------------------------------ K4
// Register-tiled like a GEMM micro-kernel.  A tile is 32 consecutive lags (one per lane) times
// LC_ROWS rows (b, mu) of LC_ROWS / 3 bins.  Its warps take consecutive ranges of ks steps of
// the block: per step a thread loads its lag's total current J(t - l) (one 16-byte shared-memory
// load from the CTA's window of J samples) and the step's LC_ROWS binned currents (broadcast
// 16-byte loads) and does 3 LC_ROWS FMAs into FP32 partial sums over the warp's steps.  The
// warps' partials are then added in step order in an unevaluated float pair (TwoSum, ~48 bits;
// GB300's FP64 pipe is narrow) and each lag sum gets one FP64 add.
//
// What bounds it: the FMAs when a grid fills the SMs, otherwise the chain staging -> steps ->
// final sums of one CTA.  So (lag_corr_plan):
//   - a tile's steps are spread over as many warps as give about three warps a scheduler over
//     the GPU, down to LC_MIN_STEPS steps a warp: with one warp per 32 steps a 32-step block ran
//     one warp a tile, 23.3 us (ncu), nearly all of it 36 read-modify-writes of the sums in turn;
//   - the tile's warps go to a cluster of CTAs of four warps where the grid can fill the SMs
//     (smaller pieces balance better: N = 512, K = 1000 had 175 CTAs of 16 warps, two on 23 of
//     the 152 SMs), each CTA staging its own steps alone; the ranks read each other's partials
//     through distributed shared memory and each finishes its share of the tile's sums;
//   - a CTA alone has up to LC_FINAL_WARPS warps where the tiles are few (those without steps take
//     part in the staging and the final sums), and every warp fetches the sums it will update into
//     L2 first;
//   - from LC_MANY_TILES tiles the latency of one CTA is hidden by the others, and warps without steps,
//     the early fetch and the barriers of a cluster only cost: CTAs stay small, a tile is a CTA
//     of its own (but for 16 warps of steps, of which an SM holds too few whole), and the sums are
//     updated one by one.  304 bins x 1000 lags (2432 tiles; us a push, one warp a tile and 32 steps ->
//     the form for few tiles -> now): K = 1 43 -> 70 -> 45, 128 59 -> 87 -> 59, 400 119 -> 131 -> 117; 1000
//     in clusters 202 -> 192.
// Measured (ncu, us, one warp a tile and 32 steps -> now): K = 32, 8 bins, 8 lags 16.0 -> 5.6; K = 77, 37
// bins, 123 lags 11.9 -> 6.9; K = 1000, 100 bins, 200 lags 24.6 -> 17.9; K = 512, 64 bins, 1000 lags
// 29.8 -> 28.6; K = 256, 64 bins, 500 lags 12.6 -> 12.8.  The cluster form starts at LC_FILL_TILES =
// half the SMs: below it a tile's CTA has an SM to itself either way, and one CTA's barriers are cheaper
// than a cluster's.
constexpr int LC_ROWS = 12;   // 4 bins x 3 components a thread
constexpr int LC_OUT = 3 * LC_ROWS;
constexpr int LC_WARPS = 16;      // warps of a tile, and of a CTA that holds a tile alone
constexpr int LC_CTA_WARPS = 4;   // warps of a CTA of a cluster
constexpr int LC_FINAL_WARPS = 12;   // warps of a CTA that holds a tile alone where the tiles are few
constexpr int LC_BATCH = 5;       // sums a warp updates at a time (all of them with 8 or more warps)
constexpr int LC_MIN_STEPS = 4;   // fewest steps a warp is worth starting for
// (Of this GPU's 152 SMs and not of those a process is given: the order of the sums then depends on the
// sizes alone.)
constexpr int LC_FILL_WARPS = 152 * 12;   // three warps a scheduler on every SM
constexpr int LC_FILL_TILES = 76;         // tiles from which clusters of small CTAs balance better
constexpr int LC_MANY_TILES = 700;        // tiles from which only throughput counts

// Warps with steps of one tile, steps a warp, the CTAs (cluster ranks) they run in, the warps
// with steps of a CTA and all its warps, the kernel's form.
enum LagCorrForm { LC_FEW, LC_CLUSTER, LC_MANY };
struct LagCorrPlan {
    int warps, ks, ranks, step_warps, cta_warps;
    LagCorrForm form;
};

LagCorrPlan lag_corr_plan(int K, int tiles) {
    LagCorrPlan p;
    // at least ceil(K / 32) warps up to LC_WARPS, so that an FP32 partial sum never covers more
    // steps than ceil(K / LC_WARPS) or 32, whichever is more
    const int lo = std::max(1, std::min(LC_WARPS, (K + 31) / 32));
    const int hi = std::max(lo, std::min(LC_WARPS, K / LC_MIN_STEPS));
    const int want = (LC_FILL_WARPS + tiles - 1) / std::max(tiles, 1);
    p.warps = std::max(lo, std::min(hi, want));
    p.ks = (K + p.warps - 1) / p.warps;
    p.warps = (K + p.ks - 1) / p.ks;
    const bool many = tiles >= LC_MANY_TILES;
    p.ranks = tiles >= LC_FILL_TILES && (!many || p.warps == LC_WARPS) ? (p.warps + LC_CTA_WARPS - 1) / LC_CTA_WARPS : 1;
    p.form = p.ranks > 1 ? LC_CLUSTER : many ? LC_MANY : LC_FEW;
    p.step_warps = p.ranks > 1 ? LC_CTA_WARPS : p.warps;
    p.cta_warps = p.ranks > 1 ? LC_CTA_WARPS : std::max(p.warps, std::min(LC_FINAL_WARPS, std::max(LC_CTA_WARPS, want)));
    return p;
}

size_t lag_corr_smem(const LagCorrPlan &p) {
    const size_t steps = (size_t)p.step_warps * p.ks;
    const size_t staging = steps * LC_ROWS * sizeof(float) + (steps + 31) * sizeof(float4);
    const size_t partials = (size_t)p.step_warps * LC_OUT * 32 * sizeof(float);
    return std::max(staging, partials);
}

// (s, c) += x exactly as an unevaluated float pair (_rn keeps it from being contracted)
__device__ __forceinline__ void lc_pair_add(float &s, float &c, float x) {
    const float t = __fadd_rn(s, x);
    const float bp = __fsub_rn(t, s);
    const float e = __fadd_rn(__fsub_rn(s, __fsub_rn(t, bp)), __fsub_rn(x, bp));
    s = t;
    c = __fadd_rn(c, e);
}

// t0_dev: the device step counter, which the push's bin finish has already advanced by K.
template <LagCorrForm FORM>
__global__ void __launch_bounds__(32 * LC_WARPS, 2) lag_corr_kernel(const float *__restrict__ Jb,
                                                                    const double *__restrict__ Jring,
                                                                    int R, double *Csum, int K,
                                                                    int B, int L, int ks,
                                                                    int step_warps,
                                                                    const long long *t0_dev) {
    // staging: rows [steps][LC_ROWS] of this CTA's steps, then their J window [steps + 31] as
    // float4 (x, y, z, 0); after the step loop the same space holds the warps' partials
    // [warp][LC_OUT][32]
    constexpr bool CLUSTER = FORM == LC_CLUSTER;
    extern __shared__ float4 lc_smem4[];
    float *sA = reinterpret_cast<float *>(lc_smem4);
    float *sP = reinterpret_cast<float *>(lc_smem4);
    const int nrank = CLUSTER ? (int)gridDim.z : 1, rank = CLUSTER ? (int)blockIdx.z : 0;   // a cluster spans grid z
    const int l0 = blockIdx.x * 32;
    const int b0 = blockIdx.y * (LC_ROWS / 3);
    const int nthreads = blockDim.x, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int cta_warps = nthreads >> 5;
    const int steps_cta = step_warps * ks;
    const int kc0 = min(K, rank * steps_cta), kc = min(K - kc0, steps_cta);   // this CTA's steps
    float4 *sW = lc_smem4 + steps_cta * (LC_ROWS / 4);

    // the tile's sums are shared out by warps over all ranks: output o (of all 32 lags) goes to
    // warp o mod ngw of the tile; its 256 bytes come into L2 while the staging and the steps run
    const int l = l0 + lane;
    const int gw = rank + nrank * warp, ngw = nrank * cta_warps;
    auto sums = [&](int o) { return Csum + ((size_t)(b0 + o / 9) * 9 + ((o / 3) % 3) * 3 + o % 3) * L + l; };
    if (FORM != LC_MANY && (lane & 15) == 0 && l < L)
        for (int o = gw; o < LC_OUT && b0 + o / 9 < B; o += ngw)
            asm volatile("prefetch.global.L2 [%0];" ::"l"(sums(o)));
    const float *Jk = Jb + (size_t)kc0 * B * 3;
    if (B % 4 == 0 && (reinterpret_cast<uintptr_t>(Jb) & 15) == 0) {
        // every bin group is whole and its 12 floats of a step start on a 16-byte boundary:
        // three asynchronous 16-byte copies a step, all in flight at once
        for (int q = threadIdx.x; q < 3 * kc; q += nthreads) {
            const int k = q / 3, j = q - 3 * k;
            cp_async16(sA + k * LC_ROWS + 4 * j, Jk + ((size_t)k * B + b0) * 3 + 4 * j);
        }
    } else {
        for (int q = threadIdx.x; q < kc * LC_ROWS; q += nthreads) {
            const int k = q / LC_ROWS, r = q - k * LC_ROWS;
            if (b0 + r / 3 < B) cp_async4(sA + q, Jk + ((size_t)k * B + b0) * 3 + r);
            else sA[q] = 0.f;
        }
    }
    // window entry w holds J(tw0 + w), tw0 = t0 + kc0 - l0 - 31: lane l at the CTA's step k reads
    // w = k - l + 31.  Ring slot of entry w: (tw0 mod R) + w brought into [0, R) with 32-bit
    // arithmetic (one 64-bit remainder a thread instead of one an entry).
    const long long tw0 = *t0_dev - K + kc0 - l0 - 31;
    const int m0 = (int)(tw0 % R);   // in (-R, R)
    for (int w = threadIdx.x; w < kc + 31; w += nthreads) {
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
        if (tw0 + w >= 0) {
            int slot = m0 + w;
            if (slot < 0) slot += R;
            if (slot >= R) slot %= R;
            const double *src = Jring + (size_t)slot * 3;
            v = make_float4((float)src[0], (float)src[1], (float)src[2], 0.f);
        }
        sW[w] = v;
    }
    cp_async_wait_all();
    __syncthreads();
    const int k_begin = min(kc, ks * warp), k_end = min(kc, k_begin + ks);
    float acc[LC_OUT];
#pragma unroll
    for (int o = 0; o < LC_OUT; ++o) acc[o] = 0.f;
    const float4 *wp = sW + (k_begin - lane + 31);
    const float4 *ap = reinterpret_cast<const float4 *>(sA) + k_begin * (LC_ROWS / 4);
#pragma unroll 4
    for (int k = k_begin; k < k_end; ++k) {
        const float4 j = *wp++;
        float x[LC_ROWS];
#pragma unroll
        for (int q = 0; q < LC_ROWS / 4; ++q) {
            const float4 a4 = ap[q];
            x[4 * q] = a4.x;
            x[4 * q + 1] = a4.y;
            x[4 * q + 2] = a4.z;
            x[4 * q + 3] = a4.w;
        }
        ap += LC_ROWS / 4;
#pragma unroll
        for (int r = 0; r < LC_ROWS; ++r) {
            acc[3 * r] = fmaf(x[r], j.x, acc[3 * r]);
            acc[3 * r + 1] = fmaf(x[r], j.y, acc[3 * r + 1]);
            acc[3 * r + 2] = fmaf(x[r], j.z, acc[3 * r + 2]);
        }
    }
    __syncthreads();   // staging no longer read: its space takes the partials
    if (warp < step_warps) {
#pragma unroll
        for (int o = 0; o < LC_OUT; ++o) sP[(warp * LC_OUT + o) * 32 + lane] = acc[o];
    }
    if (CLUSTER) cluster_sync_all();   // every rank's partials are complete
    else __syncthreads();
    if constexpr (FORM == LC_MANY) {
        for (int o = gw; o < LC_OUT && b0 + o / 9 < B; o += ngw) {   // warp-uniform
            if (l >= L) continue;
            double *dst = sums(o);
            const double old = *dst;
            float s = 0.f, c = 0.f;
            for (int w = 0; w < step_warps; ++w) lc_pair_add(s, c, sP[(w * LC_OUT + o) * 32 + lane]);
            *dst = old + (f32_to_f64(s) + f32_to_f64(c));
        }
    } else {
        for (int o0 = gw; o0 < LC_OUT && b0 + o0 / 9 < B; o0 += LC_BATCH * ngw) {   // warp-uniform
            double old[LC_BATCH];
#pragma unroll
            for (int u = 0; u < LC_BATCH; ++u) {
                const int o = o0 + u * ngw;
                old[u] = (o < LC_OUT && b0 + o / 9 < B && l < L) ? *sums(o) : 0.0;
            }
#pragma unroll
            for (int u = 0; u < LC_BATCH; ++u) {
                const int o = o0 + u * ngw;
                if (o >= LC_OUT || b0 + o / 9 >= B) break;   // warp-uniform
                float s = 0.f, c = 0.f;
                const float *mine = sP + o * 32 + lane;
                if (!CLUSTER) {
                    for (int w = 0; w < step_warps; ++w) lc_pair_add(s, c, mine[w * LC_OUT * 32]);
                } else {
                    for (int q = 0; q < nrank; ++q) {   // step order: ranks, then warps
                        const uint32_t peer = mapa_shared(smem_u32(mine), (uint32_t)q);
#pragma unroll
                        for (int w = 0; w < LC_CTA_WARPS; ++w)
                            lc_pair_add(s, c, ld_shared_cluster_f32(peer + (uint32_t)(w * LC_OUT * 32 * sizeof(float))));
                    }
                }
                if (l < L) *sums(o) = old[u] + (f32_to_f64(s) + f32_to_f64(c));
            }
        }
    }
    if (CLUSTER) cluster_sync_all();   // peers have read this CTA's partials: its shared memory may go
}

// ------------------------------------------------------------------ K5
// 1 / (T_s - l), zero when no origin has lag l.
__device__ __forceinline__ double gk_inv_count(long long T_s, int l) {
    return T_s > l ? 1.0 / (double)(T_s - l) : 0.0;
}

// table[l] = 1 / (T_s - l) for reads whose table does not fit a CTA's shared memory
__global__ void inv_counts_kernel(long long T_s, int L, double *inv) {
    const int l = blockIdx.x * blockDim.x + threadIdx.x;
    if (l < L) inv[l] = gk_inv_count(T_s, l);
}

// WARPS warps per (b, mu, nu) row, four warps a CTA or one row of more; lane i of the row's 32 WARPS
// owns per = ceil(L / (32 WARPS)) consecutive lags.  C(l) = Csum(l) / (T_s - l); the running trapezoid
// sum S(l) = sum_{1 <= l' <= l} (C(l'-1) + C(l')) comes from the lanes' totals, a warp scan and the
// totals of the row's warps before (a fixed tree, deterministic); kappa(l) = (c dt / 2) S(l).  The
// window average runs over the lags l_lo .. l_hi (the host picks them with the same FP64 test on l dt
// as the oracle).  Bound by the FP64 pipe and the latency of its chain, so:
//   - a lane with at most GK_CACHE lags keeps its running sums in registers; beyond, it walks its lags
//     twice, one load in flight.  So a row gets the fewest warps that hold it in registers, up to
//     eight (gk_tau_warps); more warps spend their time in scans and barriers;
//   - the reciprocal counts come from a table that the CTA builds, a division a lag spread over its
//     threads, or from one launch where the CTAs' divisions together cost more (gk_own_table).
// Measured (us, back to back; four warps a row and the table's launch, with a copy of the result ->
// one warp a row -> now): 72 rows x 200 lags 18.4 -> 6.2 -> 6.2; x 500 16.4 -> 12.3 -> 8.2; x 1000
// 20.5 -> 20.5 -> 10.2; x 5000 35.9 -> 92 -> 20.8; 576 x 1000 28.7 -> 22.5 -> 18.4; x 5000 69.5 -> 92
// -> 59.4; 900 x 200 30.7 -> 10.3 -> 10.3; x 1000 38.9 -> 32.8 -> 24.6.
constexpr int GK_TAU_ROWS = 4;
constexpr int GK_CACHE = 8;
constexpr int gk_tau_rows(int warps) { return warps >= GK_TAU_ROWS ? 1 : GK_TAU_ROWS / warps; }
template <int WARPS>
__global__ void __launch_bounds__(32 * WARPS * gk_tau_rows(WARPS), WARPS == 1 ? 9 : WARPS == 8 ? 4 : 8) gk_kappa_kernel(
    const double *Csum, int rows, int L, const double *__restrict__ inv, long long T_s, double coef_half,
    int l_lo, int l_hi, double *kappa_tau, double *kappa_w) {
    constexpr int ROWS = gk_tau_rows(WARPS);
    extern __shared__ double gk_tab[];
    __shared__ double s_tot[WARPS * ROWS], s_win[WARPS * ROWS];
    if (!inv) {
        for (int l = threadIdx.x; l < L; l += blockDim.x) gk_tab[l] = gk_inv_count(T_s, l);
        __syncthreads();
        inv = gk_tab;
    }
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int r = blockIdx.x * ROWS + warp / WARPS, part = warp % WARPS;
    const bool live = r < rows;   // (every warp takes the barriers)
    const double *cs = Csum + (size_t)(live ? r : 0) * L;
    double *kt = kappa_tau + (size_t)(live ? r : 0) * L;
    const int per = (L + 32 * WARPS - 1) / (32 * WARPS);
    const int l0 = live ? min(L, (32 * part + lane) * per) : L, l1 = min(L, l0 + per);
    const double c_before = (l0 > 0 && l0 < l1) ? cs[l0 - 1] * inv[l0 - 1] : 0.0;
    double run[GK_CACHE];   // the lane's running sums
    double tot = 0.0, prev = c_before;
    if (per <= GK_CACHE) {
        double c[GK_CACHE];
#pragma unroll
        for (int u = 0; u < GK_CACHE; ++u) c[u] = l0 + u < l1 ? cs[l0 + u] * inv[l0 + u] : 0.0;
#pragma unroll
        for (int u = 0; u < GK_CACHE; ++u) {
            if (l0 + u < l1 && l0 + u > 0) tot += prev + c[u];
            run[u] = tot;
            prev = c[u];
        }
    } else {
        for (int l = l0; l < l1; ++l) {
            const double c = cs[l] * inv[l];
            if (l > 0) tot += prev + c;
            prev = c;
        }
    }
    double base = tot;   // exclusive scan of the lanes' totals
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const double y = __shfl_up_sync(FULL_MASK, base, o);
        if (lane >= o) base += y;
    }
    if (WARPS > 1 && lane == 31) s_tot[warp] = base;
    base = __shfl_up_sync(FULL_MASK, base, 1);
    if (lane == 0) base = 0.0;
    if (WARPS > 1) {
        __syncthreads();
        double before = 0.0;
        for (int q = 0; q < part; ++q) before += s_tot[warp - part + q];
        base += before;
    }
    double wsum = 0.0;
    auto emit = [&](int l, double s) {
        const double kap = coef_half * s;
        kt[l] = kap;
        if (l >= l_lo && l <= l_hi) wsum += kap;
    };
    if (per <= GK_CACHE) {
#pragma unroll
        for (int u = 0; u < GK_CACHE; ++u)
            if (l0 + u < l1) emit(l0 + u, base + run[u]);
    } else {
        prev = c_before;
        for (int l = l0; l < l1; ++l) {
            const double c = cs[l] * inv[l];
            if (l > 0) base += prev + c;
            prev = c;
            emit(l, base);
        }
    }
    if (!kappa_w) return;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) wsum += __shfl_down_sync(FULL_MASK, wsum, o);
    if (WARPS > 1) {
        if (lane == 0) s_win[warp] = wsum;
        __syncthreads();
        if (part == 0)
            for (int q = 1; q < WARPS; ++q) wsum += s_win[warp + q];
    }
    if (part == 0 && lane == 0 && live) {
        const int n = l_hi >= l_lo ? l_hi - l_lo + 1 : 0;
        kappa_w[r] = n > 0 ? wsum / n : 0.0;
    }
}

// Window average alone (no kappa(tau) wanted): with S(l) the running trapezoid sum above,
//   sum_{l = l_lo..l_hi} S(l) = sum_m C(m) w(m),  w(m) = [m >= 1] cnt(m) + cnt(m + 1),
// cnt(x) = #{l in [l_lo, l_hi] : l >= x} (C(m) enters S(l) as the right end of the step m-1 -> m
// for l >= m >= 1 and as the left end of the step m -> m+1 for l >= m+1).  The integer weights
// and the reciprocal counts are folded into one table tw(m) = w(m) / (T_s - m), so a row takes one
// FP64 FMA a lag instead of the scan's few FP64 operations a lag on GB300's narrow FP64 pipe.
__device__ __forceinline__ double gk_window_weight(long long T_s, int m, int l_lo, int l_hi) {
    const auto cnt = [&](int x) {
        const int lo = max(x, l_lo);
        return l_hi >= lo ? l_hi - lo + 1 : 0;
    };
    return gk_inv_count(T_s, m) * (double)((m >= 1 ? cnt(m) : 0) + cnt(m + 1));
}

__global__ void gk_window_weights_kernel(long long T_s, int L, int l_lo, int l_hi, double *tw) {
    const int m = blockIdx.x * blockDim.x + threadIdx.x;
    if (m < L) tw[m] = gk_window_weight(T_s, m, l_lo, l_hi);
}

// WARPS warps per row, GK_ROWS warps a CTA: kappa_w = scale sum_m Csum(m) tw(m) (lanes stride the
// lags; fixed tree).  tw null: each CTA first builds the table in shared memory, a division a lag
// spread over its threads (gk_own_table).  One warp a row, or the whole CTA for more than
// GK_ONE_WARP_LAGS lags, where a warp's round trips to memory were the time.
// Measured (us, back to back, eight rows a CTA -> now): 576 rows x 500 lags 10.3 -> 6.2; x 1000 12.3
// -> 8.5; 72 x 5000 28.6 -> 13.3 (one warp a row 30.7); 72 x 10000 36.9 -> 16.4 (45.1).
constexpr int GK_ONE_WARP_LAGS = 1024;
constexpr int GK_ROWS = 4;
template <int WARPS>
__global__ void __launch_bounds__(32 * GK_ROWS) gk_window_kernel(const double *Csum, int rows, int L,
                                                                 const double *__restrict__ tw,
                                                                 long long T_s, int l_lo, int l_hi,
                                                                 double scale, double *kappa_w) {
    constexpr int ROWS = GK_ROWS / WARPS, STRIDE = 32 * WARPS;
    extern __shared__ double gk_tw[];
    __shared__ double s_part[GK_ROWS];
    if (!tw) {
        for (int m = threadIdx.x; m < L; m += blockDim.x) gk_tw[m] = gk_window_weight(T_s, m, l_lo, l_hi);
        __syncthreads();
        tw = gk_tw;
    }
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, part = warp % WARPS;
    const int r = blockIdx.x * ROWS + warp / WARPS;
    if (r >= rows) return;   // (with WARPS > 1 a CTA has one row, so none is left at the barrier)
    const double *cs = Csum + (size_t)r * L;
    double acc[4] = {0.0, 0.0, 0.0, 0.0};   // four loads in flight a lane
    for (int m = 32 * part + lane; m < L; m += 4 * STRIDE) {
#pragma unroll
        for (int u = 0; u < 4; ++u)
            if (m + STRIDE * u < L) acc[u] = fma(cs[m + STRIDE * u], tw[m + STRIDE * u], acc[u]);
    }
    double t = (acc[0] + acc[1]) + (acc[2] + acc[3]);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) t += __shfl_down_sync(FULL_MASK, t, o);
    if (WARPS > 1) {
        if (lane == 0) s_part[warp] = t;
        __syncthreads();
        if (part == 0)
            for (int q = 1; q < WARPS; ++q) t += s_part[warp + q];
    }
    if (part == 0 && lane == 0) kappa_w[r] = scale * t;
}

// The same average of the bin-bin sums, from their state X[l][j][i] (float pairs, i = 3b + mu and
// j = 3b' + nu of n = 3 nb rows) without the FP64 copy in [b][b'][mu][nu][l] order that the
// kappa(tau) read takes: consecutive threads take consecutive (j, i), so every lag is one
// contiguous read.  Bound by the FP64 pipe, 16 cycles an instruction of a warp: so an element takes one
// FP64 instruction and not four (two conversions, an addition and an FMA; 61 us for the case below).
// X is renormalised, its high part is widened by its bits and added by an FP64 FMA, and what its low
// part (at most half a unit of the high one) gives is summed in a pair of floats, 47 bits below
// those 24.  That holds FP64's precision while the terms are inside single precision's range: an
// output whose terms add up to less than XCW_SMALL or more than XCW_LARGE is summed again in FP64
// throughout.  The weights are scaled by a power of two so that they add up to less than one.
// The groups of a CTA share an output's lags and are added in order.
// Measured at n = 192, L = 200 (59 MB; us, back to back): 90 (FP64 copy, weights, sum) -> 22.6; in
// pairs of floats throughout, 46 bits, 14.4.
// Outputs that fill no more than an SM each (XCW_WIDE a CTA: xcw_wide) are spread over narrow CTAs, a
// 32-byte sector of outputs and 64 groups of lags each: 18 rows x 4000 lags 135 -> 27 us (33-41 with
// the FP64 copy), 3 x 5000 171 -> 33 (39), 60 x 1000 31 -> 27, but 66 x 100 6.2 -> 16.
constexpr int XCW_THREADS = 256, XCW_UNROLL = 8;
constexpr int XCW_WIDE = 64, XCW_NARROW = 4;   // outputs a CTA
constexpr float XCW_SMALL = 0x1p-70f, XCW_LARGE = 0x1p120f;

// A weight of the bin-bin windows, w(m) 2^-k, and its two leading floats.
struct __align__(16) XcwWeight {
    double w;
    float a, b;
};
__device__ __forceinline__ XcwWeight xcw_weight(long long T_s, int m, int l_lo, int l_hi, double down) {
    XcwWeight r;
    r.w = gk_window_weight(T_s, m, l_lo, l_hi) * down;
    r.a = (float)r.w;
    r.b = (float)(r.w - (double)r.a);
    return r;
}

// float -> double by its bits (zero for subnormals): the conversion runs on the FP64 pipe
__device__ __forceinline__ double xcw_double(float x) {
    const uint32_t u = __float_as_uint(x), a = u & 0x7fffffffu;
    const uint32_t hi = a >= 0x00800000u ? (a >> 3) + 0x38000000u : 0u;   // exponent rebiased
    return __hiloint2double((int)((u & 0x80000000u) | hi), (int)(u << 29));
}

__global__ void xcw_weights_kernel(long long T_s, int L, int l_lo, int l_hi, double down, XcwWeight *tw) {
    const int m = blockIdx.x * blockDim.x + threadIdx.x;
    if (m < L) tw[m] = xcw_weight(T_s, m, l_lo, l_hi, down);
}

template <int OUT>
__global__ void __launch_bounds__(XCW_THREADS) xcorr_window_kernel(
    const float2 *__restrict__ X, int nb, int L, const XcwWeight *__restrict__ tw, long long T_s,
    int l_lo, int l_hi, double down, double scale, double *kappa_w) {
    constexpr int GROUPS = XCW_THREADS / OUT;
    extern __shared__ XcwWeight xw_tab[];
    __shared__ double part[GROUPS][OUT];
    const int n = 3 * nb, o = threadIdx.x % OUT, g = threadIdx.x / OUT;
    const long long nn = (long long)n * n, q = blockIdx.x * (long long)OUT + o;
    const int per = (L + GROUPS - 1) / GROUPS;
    const int m0 = q < nn ? min(L, g * per) : 0, m1 = q < nn ? min(L, m0 + per) : 0;
    const float2 *src = X + q;
    float2 v[XCW_UNROLL];
    auto fetch = [&](int m) {
#pragma unroll
        for (int u = 0; u < XCW_UNROLL; ++u)
            v[u] = m + u < m1 ? __ldcs(src + (m + u) * nn) : make_float2(0.f, 0.f);
    };
    fetch(m0);   // in flight while the table is built
    if (!tw) {
        for (int m = threadIdx.x; m < L; m += blockDim.x) xw_tab[m] = xcw_weight(T_s, m, l_lo, l_hi, down);
        __syncthreads();
        tw = xw_tab;
    }
    double sum = 0.0;            // of the pairs' high parts
    float lo = 0.f, loc = 0.f;   // of their low parts, as a pair
    float size = 0.f;            // of the terms
    bool any = false;
    auto add = [&](float2 z, int m) {
        const XcwWeight w = tw[m];
        float x = z.x, y = 0.f;
        lc_pair_add(x, y, z.y);   // now |y| is at most half a unit of x
        sum = fma(xcw_double(x), w.w, sum);
        const float p = __fmul_rn(y, w.a);
        const float e = fmaf(y, w.b, fmaf(y, w.a, -p));
        lc_pair_add(lo, loc, p);
        loc = __fadd_rn(loc, e);
        size = fmaf(fabsf(x), w.a, size);
        any = any || x != 0.f;
    };
    int m = m0;
    for (; m + XCW_UNROLL <= m1; m += XCW_UNROLL) {
        if (m > m0) fetch(m);
#pragma unroll
        for (int u = 0; u < XCW_UNROLL; ++u) add(v[u], m + u);
    }
    if (m > m0) fetch(m);
#pragma unroll
    for (int u = 0; u < XCW_UNROLL - 1; ++u)
        if (m + u < m1) add(v[u], m + u);
    if (size >= XCW_SMALL && size <= XCW_LARGE) {
        sum += (double)lo + (double)loc;
    } else if (any) {   // terms near the ends of single precision's range, or nothing but zeros of w
        sum = 0.0;
        for (int k = m0; k < m1; ++k) {
            const float2 z = src[k * nn];
            sum = fma((double)z.x + (double)z.y, tw[k].w, sum);
        }
    }
    part[g][o] = sum;
    __syncthreads();
    if (g == 0 && q < nn) {
        double t = 0.0;
#pragma unroll 8
        for (int k = 0; k < GROUPS; ++k) t += part[k][o];
        const int j = (int)(q / n), i = (int)(q - (long long)j * n);
        kappa_w[(((size_t)(i / 3) * nb + j / 3) * 3 + i % 3) * 3 + j % 3] = scale * t;
    }
}

__global__ void hnema_finalize_kernel(const double *hsum, int n, long long T_s, double coef,
                                      double *mean, double *kappa) {
    const int q = blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= n) return;
    const double m = T_s > 0 ? hsum[q] / (double)T_s : 0.0;
    if (mean) mean[q] = m;
    if (kappa) kappa[q] = m * coef;
}

__global__ void hnema_finalize_group_kernel(const HnemaGroupArgs a, double *mean, double *kappa) {
    const int j = blockIdx.y;
    if (j >= a.n) return;
    for (int q = blockIdx.x * blockDim.x + threadIdx.x; q < a.nb[j]; q += gridDim.x * blockDim.x) {
        const double m = a.T_s[j] > 0 ? a.hsum[j][q] / (double)a.T_s[j] : 0.0;
        if (mean) mean[a.off[j] + q] = m;
        if (kappa) kappa[a.off[j] + q] = m * a.coef[j];
    }
}

__global__ void lag_counts_kernel(long long T_s, int L, long long *count) {
    const int l = blockIdx.x * blockDim.x + threadIdx.x;
    if (l < L) count[l] = T_s > l ? T_s - l : 0;
}

}  // namespace

void launch_bin_finish(const float *partials, int n_slots, const int *slot_begin, int B, int K,
                       float *Jb, double *hsum, const double *Jtot, double *Jsum, long long *steps,
                       cudaStream_t s) {
    if (B <= 0 || K <= 0) return;
    bin_finish_kernel<<<B + 1, bf_threads(K), 0, s>>>(partials, n_slots, slot_begin, B, K, Jb, hsum, Jtot,
                                               Jsum, steps);
}

namespace {
constexpr int XCW_TABLE_LAGS = 2900;   // longest table of a bin-bin window's CTA, within the default 48 KB

// Whether each of `ctas` CTAs builds its own table of L lags: the divisions take an SM about 5 ns each,
// against 4 us for a launch.  (576 rows, kappa(tau) of 500 lags: 288 CTAs 12.3 us own, 14.4
// launched; of 1000 lags: 576 CTAs 22.5 and 18.4.  72 rows x 5000 lags: 24.6 and 20.5.  Bin-bin windows
// of 60 rows x 1000 lags: 900 CTAs 45 and 27.)
bool gk_own_table(long long ctas, int L) { return L <= 3000 && ctas * L <= 300000; }

// Whether XCW_WIDE outputs a CTA give every other SM one, or the lags are few enough for that not to
// matter.  (Where the line is crossed, us, wide and narrow: 60 rows 31 and 27 at 1000 lags, 90 rows 37
// and 47; 66 rows 6 and 16 at 100 lags.)
constexpr int XCW_FILL_CTAS = 76, XCW_FEW_LAGS = 128;
bool xcw_wide(long long out, int L) { return (out + XCW_WIDE - 1) / XCW_WIDE >= XCW_FILL_CTAS || L <= XCW_FEW_LAGS; }

// Warps a row of kappa(tau) (see the kernel).  Up to 320 lags one warp walking its lags twice is as
// good, where the rows are many (1800 x 300: 16.4 us and 18.4; 900 x 300: 12.3 and 10.3).
int gk_tau_warps(int rows, int L) {
    if (L <= 256 || (L <= 320 && rows >= 1520)) return 1;
    return L <= 512 ? 2 : L <= 1024 ? 4 : 8;
}

// The window's lags: l dt in [tau_lo, tau_hi], tested in FP64 as the oracle tests it.
void gk_window(int L, double tau_lo, double tau_hi, double dt, int &l_lo, int &l_hi) {
    l_lo = L;
    l_hi = -1;
    for (int l = 0; l < L; ++l) {
        const double tau = l * dt;
        if (tau >= tau_lo && tau <= tau_hi) {
            l_lo = std::min(l_lo, l);
            l_hi = l;
        }
    }
}

int lag_corr_tiles(int B, int L) { return ((L + 31) / 32) * ((B + LC_ROWS / 3 - 1) / (LC_ROWS / 3)); }
}

cudaError_t lag_corr_prepare() {
    // a tile alone in its CTA stages at most 1024 steps or 16 warps' partials: below 80 KB
    LagCorrPlan p{LC_WARPS, 64, 1, LC_WARPS, LC_WARPS, LC_FEW};
    static PerDevice once[3];
    cudaError_t e = opt_in_smem(once[0], lag_corr_kernel<LC_FEW>, lag_corr_smem(p));
    if (e == cudaSuccess) e = opt_in_smem(once[1], lag_corr_kernel<LC_CLUSTER>, lag_corr_smem(p));
    return e != cudaSuccess ? e : opt_in_smem(once[2], lag_corr_kernel<LC_MANY>, lag_corr_smem(p));
}

void launch_bin_finish_group(FinishGroupArgs g, cudaStream_t s) {
    if (g.n < 1) return;
    g.cta_begin[0] = 0;
    int kmax = 0;
    for (int j = 0; j < g.n; ++j) {
        g.cta_begin[j + 1] = g.cta_begin[j] + (g.K[j] > 0 ? g.B[j] + 1 : 0);
        kmax = std::max(kmax, g.K[j]);
    }
    if (g.cta_begin[g.n] > 0) bin_finish_group_kernel<<<g.cta_begin[g.n], bf_threads(kmax), 0, s>>>(g);
}

cudaError_t launch_lag_corr(const float *Jb, const double *Jring, int R, double *Csum, int K, int B,
                            int L, const long long *t0_dev, cudaStream_t s) {
    if (L <= 0 || K <= 0 || B <= 0) return cudaSuccess;
    const cudaError_t ready = lag_corr_prepare();
    if (ready != cudaSuccess) return ready;
    const LagCorrPlan p = lag_corr_plan(K, lag_corr_tiles(B, L));
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)((L + 31) / 32), (unsigned)((B + LC_ROWS / 3 - 1) / (LC_ROWS / 3)),
                       (unsigned)p.ranks);
    cfg.blockDim = dim3((unsigned)(32 * p.cta_warps), 1, 1);
    cfg.dynamicSmemBytes = lag_corr_smem(p);
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 1;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = (unsigned)p.ranks;
    cfg.attrs = attr;
    cfg.numAttrs = p.ranks > 1 ? 1 : 0;
    const auto kernel = p.form == LC_CLUSTER ? lag_corr_kernel<LC_CLUSTER>
                        : p.form == LC_MANY  ? lag_corr_kernel<LC_MANY>
                                             : lag_corr_kernel<LC_FEW>;
    return cudaLaunchKernelEx(&cfg, kernel, Jb, Jring, R, Csum, K, B, L, p.ks, p.step_warps, t0_dev);
}

int launch_gk_kappa(const double *Csum, int B, int L, long long T_s, double coef_dt,
                    double tau_lo, double tau_hi, double dt, double *kappa_tau, double *kappa_w,
                    double *table, cudaStream_t s) {
    if (L <= 0 || B <= 0) return 0;
    int l_lo, l_hi;
    gk_window(L, tau_lo, tau_hi, dt, l_lo, l_hi);
    const int rows = B * 9;
    if (!kappa_tau) {   // the window average alone
        const int n = l_hi >= l_lo ? l_hi - l_lo + 1 : 0;
        const double scale = n > 0 ? 0.5 * coef_dt / n : 0.0;
        const bool one = L <= GK_ONE_WARP_LAGS;
        const int ctas = one ? (rows + GK_ROWS - 1) / GK_ROWS : rows;
        const bool own = gk_own_table(ctas, L);
        if (!own) gk_window_weights_kernel<<<(L + 255) / 256, 256, 0, s>>>(T_s, L, l_lo, l_hi, table);
        const auto run = [&](auto kernel) {
            kernel<<<ctas, 32 * GK_ROWS, own ? sizeof(double) * L : 0, s>>>(
                Csum, rows, L, own ? nullptr : table, T_s, l_lo, l_hi, scale, kappa_w);
        };
        if (one) run(gk_window_kernel<1>);
        else run(gk_window_kernel<GK_ROWS>);
        return own ? 1 : 2;
    }
    const int warps = gk_tau_warps(rows, L);
    const int ctas = (rows + gk_tau_rows(warps) - 1) / gk_tau_rows(warps);
    const bool own = gk_own_table(ctas, L);
    if (!own) inv_counts_kernel<<<(L + 255) / 256, 256, 0, s>>>(T_s, L, table);
    const auto run = [&](auto kernel) {
        kernel<<<ctas, 32 * warps * gk_tau_rows(warps), own ? sizeof(double) * L : 0, s>>>(
            Csum, rows, L, own ? nullptr : table, T_s, 0.5 * coef_dt, l_lo, l_hi, kappa_tau, kappa_w);
    };
    if (warps == 1) run(gk_kappa_kernel<1>);
    else if (warps == 2) run(gk_kappa_kernel<2>);
    else if (warps == 4) run(gk_kappa_kernel<4>);
    else run(gk_kappa_kernel<8>);
    return own ? 1 : 2;
}

int launch_xcorr_window(const float2 *X, int nb, int L, long long T_s, double coef_dt, double tau_lo,
                        double tau_hi, double dt, double *kappa_w, double *table, cudaStream_t s) {
    if (L <= 0 || nb <= 0) return 0;
    int l_lo, l_hi;
    gk_window(L, tau_lo, tau_hi, dt, l_lo, l_hi);
    const int n = l_hi >= l_lo ? l_hi - l_lo + 1 : 0;
    const double scale = n > 0 ? 0.5 * coef_dt / n : 0.0;
    const int Lw = n > 0 ? l_hi + 1 : 0;   // lags past the window have no weight: neither read nor tried in FP64
    // weights scaled so that they add up to less than one: w(m) <= 2 n / (T_s - m)
    const double most = 2.0 * n * Lw / (double)std::max(1ll, T_s - (Lw - 1));
    const int wexp = most > 0 ? std::ilogb(most) + 1 : 0;
    const double down = std::ldexp(1.0, -wexp), up = std::ldexp(scale, wexp);
    const long long out = 9ll * nb * nb;
    const bool wide = xcw_wide(out, Lw);
    const long long ctas = (out + (wide ? XCW_WIDE : XCW_NARROW) - 1) / (wide ? XCW_WIDE : XCW_NARROW);
    const bool own = Lw <= XCW_TABLE_LAGS && gk_own_table(ctas, Lw);
    XcwWeight *tw = reinterpret_cast<XcwWeight *>(table);
    if (!own) xcw_weights_kernel<<<(Lw + 255) / 256, 256, 0, s>>>(T_s, Lw, l_lo, l_hi, down, tw);
    const auto run = [&](auto kernel) {
        kernel<<<(unsigned)ctas, XCW_THREADS, own ? sizeof(XcwWeight) * Lw : 0, s>>>(
            X, nb, Lw, own ? nullptr : tw, T_s, l_lo, l_hi, down, up, kappa_w);
    };
    if (wide) run(xcorr_window_kernel<XCW_WIDE>);
    else run(xcorr_window_kernel<XCW_NARROW>);
    return own ? 1 : 2;
}

void launch_hnema_finalize(const double *hsum, int B, long long T_s, double coef, double *mean,
                           double *kappa, cudaStream_t s) {
    const int n = B * 3;
    hnema_finalize_kernel<<<(n + 127) / 128, 128, 0, s>>>(hsum, n, T_s, coef, mean, kappa);
}

void launch_hnema_finalize_group(const HnemaGroupArgs &a, double *mean, double *kappa,
                                 cudaStream_t s) {
    hnema_finalize_group_kernel<<<dim3(4, a.n), 128, 0, s>>>(a, mean, kappa);
}

void launch_lag_counts(long long T_s, int L, long long *count, cudaStream_t s) {
    if (L <= 0) return;
    lag_counts_kernel<<<(L + 127) / 128, 128, 0, s>>>(T_s, L, count);
}

}  // namespace mhc

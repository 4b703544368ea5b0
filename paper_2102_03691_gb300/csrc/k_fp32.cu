// Plain FP32 CUDA-core path of the two projections (Eq. 13 and the bracket of
// Eq. 16) and its bin epilogue.  This is the FP32 GPU baseline the tensor-core
// path is compared against; it accumulates in FP32 FMAs over d.
#include <algorithm>

#include "common.cuh"
#include "kernels.h"

namespace mhc {

namespace {

// R[c][n] = sum_d Bd[d][c] Ed[d][n], both operands stored d-major.
//
// Bound by the FP32 FMA pipe: 24 flops a mode, atom and step against 4 bytes an element of E that
// the column tiles share through L2.  Two persistent CTAs an SM compute tiles of 128 modes x 128
// columns; TMA keeps SG_AHEAD stages of 16 d's in flight and 256 threads hold 8 x 8 outputs each
// in FP32 FMAs in order of d.  What shapes it:
//   - the warps take turns at issuing the copies (a ninth warp would cost every thread 16
//     registers; one warp issuing all of them fell behind the others, which then waited for it a
//     fifth of their time: 2838 us);
//   - d-major operands: a thread's eight modes (columns) of one d are two 16-byte shared-memory
//     loads into consecutive registers, so the FMAs of one d alternate register banks.  With the
//     operands mode-major in shared memory (four d's a load) every second FMA had two operands in
//     one bank: 3863 us; packed two-wide FMAs (fma.rn.f32x2) on the same loads: 3064 us.
//   - lane bits: a 16-byte load takes 2 cycles for some ways of sharing its addresses among the
//     lanes and 4 for others, however few the distinct addresses (measured: 2 for lane bits
//     {1, 2, 3} and for {0, 3, 4}, 4 for {0, 1} and {0, 1, 2}), so the mode index takes lane bits
//     1, 2, 3 and the column index bits 0 and 4: 8 cycles of loads a warp and d beside 16 of FMAs.
//   - tiles rarely fill whole waves of CTAs, so the tiles of the last, partial wave are cut along
//     d into one range of equal length a CTA (whole chunks of 128 d's); a cut tile's first range goes
//     to R, the others to tiles of their own, and the bin epilogue adds them in order.
//   - the sums are stored word by word: 16-byte stores make the compiler place four sums in the
//     bank order of the four modes they belong to, and half the FMAs then find all three operands
//     in one register bank (2782 us, FMA pipe 71% against 80%).
// Measured at 12288 modes x 512 columns x 12288 d's (1.55e11 flops): 3877 us (16-d slabs through
// registers between two barriers, 384 tiles in waves of 304) -> 2510 us, 61.6 TFLOP/s, 0.80 of the
// measured FMA rate; what is left is issue slots (FMAs are 89% of the instructions).
constexpr int SG_BM = 128;  // modes per tile
constexpr int SG_BN = 128;  // columns per tile
constexpr int SG_BK = 16;   // d's per stage
constexpr int SG_STAGES = 6;
constexpr int SG_AHEAD = SG_STAGES - 2;   // a stage is refilled two stages after it was read
constexpr int SG_CTAS = 2;                // resident CTAs an SM
constexpr int SG_CHUNK_KB = SGEMM_CHUNK / SG_BK;
constexpr int SG_A_BYTES = SG_BM * SG_BK * 4, SG_B_BYTES = SG_BN * SG_BK * 4;
constexpr int SG_STAGE_BYTES = SG_A_BYTES + SG_B_BYTES;
constexpr int SG_SMEM = SG_STAGES * SG_STAGE_BYTES + 128 + 128;   // barriers + alignment slack
constexpr int SG_WARPS = 8;
constexpr int SG_THREADS = 32 * SG_WARPS;

// The units of one CTA: whole tiles round-robin, then its range of the tail's chunks.
struct SgUnit {
    int dir, mt, ct, kb_lo, kb_hi, seg;
};
struct SgUnitIter {
    int i;
    long long g, g_end;
    __device__ void start(const SgemmPlan &p) {
        i = blockIdx.x;
        g = g_end = 0;
        if ((int)blockIdx.x < p.parts) {
            g = p.part_begin(blockIdx.x);
            g_end = p.part_begin(blockIdx.x + 1);
        }
    }
    __device__ static void place(const SgemmPlan &p, int tile, SgUnit &u) {
        const int per_dir = p.n_mt * p.n_ct;
        u.dir = tile / per_dir;
        const int r = tile - u.dir * per_dir;
        u.mt = r / p.n_ct;
        u.ct = r - u.mt * p.n_ct;
    }
    __device__ bool next(const SgemmPlan &p, SgUnit &u) {
        if (i < p.t0) {
            place(p, i, u);
            u.kb_lo = 0;
            u.kb_hi = p.n_kb;
            u.seg = 0;
            i += gridDim.x;
            return true;
        }
        if (g >= g_end) return false;
        const int tl = (int)(g / p.nch), c0 = (int)(g - (long long)tl * p.nch);
        const int c1 = (int)min((long long)p.nch, (long long)c0 + (g_end - g));
        place(p, p.t0 + tl, u);
        u.kb_lo = c0 * SG_CHUNK_KB;
        u.kb_hi = min(p.n_kb, c1 * SG_CHUNK_KB);
        u.seg = p.part_of(g) - p.part_of(g - c0);
        g += c1 - c0;
        return true;
    }
};

__global__ void __launch_bounds__(SG_THREADS, SG_CTAS) sgemm_kernel(const __grid_constant__ SgemmParams p) {
    extern __shared__ uint8_t sg_smem_raw[];
    uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(sg_smem_raw) + 127) &
                                                ~uintptr_t(127));
    uint64_t *full = reinterpret_cast<uint64_t *>(smem + SG_STAGES * SG_STAGE_BYTES);
    uint64_t *empty = full + SG_STAGES;
    volatile int *abort = reinterpret_cast<volatile int *>(empty + SG_STAGES);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        for (int s = 0; s < SG_STAGES; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], SG_WARPS);
        }
        if (p.stall_inject) mbar_expect_tx(&full[0], 16);
        *abort = 0;
        fence_mbar_init();
    }
    __syncthreads();
    griddep_wait();   // the pack's rows
    const SgemmPlan &pl = p.plan;
    bool ok = true;

    // The CTA's sequence of k-blocks: its whole tiles, then the k-blocks tail0 .. tail0 + n_tail of
    // the tail's tiles laid end to end.  Number n of it goes into stage n % STAGES, issued by lane
    // 0 of warp n % WARPS when that warp reaches k-block n - AHEAD.
    const int n_whole = (int)blockIdx.x < pl.t0 ? ((pl.t0 - 1 - (int)blockIdx.x) / (int)gridDim.x + 1) * pl.n_kb : 0;
    int tail0 = 0, n_tail = 0;
    if ((int)blockIdx.x < pl.parts) {
        tail0 = pl.tail_kb(pl.part_begin(blockIdx.x), SG_CHUNK_KB);
        n_tail = pl.tail_kb(pl.part_begin(blockIdx.x + 1), SG_CHUNK_KB) - tail0;
    }
    auto produce = [&](int n) {
        if (n >= n_whole + n_tail) return true;
        const int q = n < n_whole ? n : tail0 + (n - n_whole);
        const int tl = q / pl.n_kb, kb = q - tl * pl.n_kb;
        SgUnit v;
        SgUnitIter::place(pl, n < n_whole ? (int)blockIdx.x + tl * (int)gridDim.x : pl.t0 + tl, v);
        const int st = n % SG_STAGES;
        if (!mbar_wait(&empty[st], ((n / SG_STAGES) & 1) ^ 1, abort, p.wait_limit)) return false;
        uint8_t *sa = smem + st * SG_STAGE_BYTES;
        mbar_arrive_expect_tx(&full[st], SG_STAGE_BYTES);
        const uint64_t pol = l2_policy_evict_normal();   // both operands are shared with other CTAs
        const int d = v.dir * p.dir_cols + kb * SG_BK;
        tma_load_2d(sa, &p.tmA, &full[st], v.mt * SG_BM, d, pol);
        tma_load_2d(sa + SG_A_BYTES, &p.tmB, &full[st], v.ct * SG_BN, d, pol);
        return true;
    };
    if (threadIdx.x == 0) {
        tma_prefetch_desc(&p.tmA);
        tma_prefetch_desc(&p.tmB);
        for (int q = 0; q < SG_AHEAD; ++q) ok = ok && produce(q);
    }
    ok = __all_sync(FULL_MASK, ok);

    // 16 x 16 threads; warps 2 x 4 of 8 x 4: modes 4 tx .. +3 and 64 + 4 tx .., columns alike
    const int tx = ((lane >> 1) & 7) | ((warp & 1) << 3);
    const int ty = (lane & 1) | ((lane >> 3) & 2) | ((warp >> 1) << 2);
    SgUnitIter it;
    it.start(pl);
    SgUnit u;
    int stage = 0, at = 0;   // at: the number of the k-block in the CTA's sequence
    uint32_t phase = 0;
    while (ok && it.next(pl, u)) {
        float acc[8][8];   // [column][mode]
#pragma unroll
        for (int j = 0; j < 8; ++j)
#pragma unroll
            for (int i = 0; i < 8; ++i) acc[j][i] = 0.f;
        for (int kb = u.kb_lo; kb < u.kb_hi; ++kb) {
            bool go = lane != 0 || warp != (at + SG_AHEAD) % SG_WARPS || produce(at + SG_AHEAD);
            ++at;
            go = go && mbar_wait(&full[stage], phase, abort, p.wait_limit);
            ok = __all_sync(FULL_MASK, go);   // a warp goes on or gives up as one
            if (!ok) break;
            const float *sa = reinterpret_cast<const float *>(smem + stage * SG_STAGE_BYTES) + 4 * tx;
            const float *sb = reinterpret_cast<const float *>(smem + stage * SG_STAGE_BYTES + SG_A_BYTES) + 4 * ty;
#pragma unroll 8
            for (int d = 0; d < SG_BK; ++d) {
                float a[8], b[8];
                *reinterpret_cast<float4 *>(a) = *reinterpret_cast<const float4 *>(sa + d * SG_BM);
                *reinterpret_cast<float4 *>(a + 4) = *reinterpret_cast<const float4 *>(sa + d * SG_BM + 64);
                *reinterpret_cast<float4 *>(b) = *reinterpret_cast<const float4 *>(sb + d * SG_BN);
                *reinterpret_cast<float4 *>(b + 4) = *reinterpret_cast<const float4 *>(sb + d * SG_BN + 64);
#pragma unroll
                for (int j = 0; j < 8; ++j)
#pragma unroll
                    for (int i = 0; i < 8; ++i) acc[j][i] = fmaf(a[i], b[j], acc[j][i]);
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(&empty[stage]);
            if (++stage == SG_STAGES) { stage = 0; phase ^= 1u; }
        }
        if (!ok) break;
        // column c of the product at R + at + c ld: in its plane, or in a tail piece whose column 0 is
        // the tile's first (one store sequence for both; two, or one more value kept over the sums,
        // cost 7% in register banks)
        const unsigned ld = u.seg ? SG_BM : p.Mp;
        float *R = u.seg ? p.tail : p.R;
        const long long at = 4 * tx + (u.seg ? p.tail_at(u.seg, (u.dir * pl.n_mt + u.mt) * pl.n_ct + u.ct - pl.t0) -
                                                   (long long)u.ct * SG_BN * SG_BM
                                             : (long long)(u.dir * p.rstride) + u.mt * SG_BM);
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const int c = u.ct * SG_BN + (j < 4 ? 4 * ty + j : 64 + 4 * ty + j - 4);
            if (c >= p.C) continue;
            float *row = R + (at + (long long)c * ld);   // one word a store: see the register banks above
#pragma unroll
            for (int i = 0; i < 8; ++i) row[i < 4 ? i : 60 + i] = acc[j][i];
        }
    }
    if (!ok) {
        *abort = 1;
        set_status(p.status, DEV_TIMEOUT);
    }
    if (!ok && lane == 0) {   // copies in flight land before the CTA exits (else all were consumed)
        for (int n = max(0, at - 1); n < at + SG_AHEAD && n < n_whole + n_tail; ++n) {
            if (n >= SG_AHEAD && n % SG_WARPS != warp) continue;
            const long long t0 = clock64();
            while (!mbar_try_wait(&full[n % SG_STAGES], (n / SG_STAGES) & 1) && clock64() - t0 < p.wait_limit) {
            }
        }
    }
    __syncthreads();
}

// The values of NK steps from step k of mode blockIdx.x SG_BM + threadIdx.x in direction b: their four
// columns, the tile's pieces added in order (zero past the block).  The next piece's loads are in
// flight while a piece is added.
template <int NK>
__device__ __forceinline__ void sg_load_piece(float (&v)[4 * NK], const float *p, size_t ld, int steps) {
#pragma unroll
    for (int q = 0; q < 4 * NK; ++q) v[q] = q / 4 < steps ? __ldcg(p + q * ld) : 0.f;
}
template <int NK>
__device__ __forceinline__ void sg_load(float (&v)[4 * NK], const SgemmParams &p, int b, int k, int K) {
    const int ct = 4 * k / SG_BN, tile = (b * p.plan.n_mt + (int)blockIdx.x) * p.plan.n_ct + ct;
    const int nseg = p.plan.segments(tile), c = 4 * k - ct * SG_BN;
    sg_load_piece<NK>(v, p.R + b * p.rstride + (size_t)(4 * k) * p.Mp + blockIdx.x * SG_BM + threadIdx.x, p.Mp, K - k);
    const auto piece = [&](float (&w)[4 * NK], int s) {
        sg_load_piece<NK>(w, p.tail + p.tail_at(s, tile - p.plan.t0) + c * SG_BM + threadIdx.x, SG_BM, K - k);
    };
    float w[2][4 * NK];
    if (nseg > 1) piece(w[0], 1);
    for (int s = 1; s < nseg; s += 2) {
        if (s + 1 < nseg) piece(w[1], s + 1);
#pragma unroll
        for (int q = 0; q < 4 * NK; ++q) v[q] += w[0][q];
        if (s + 1 >= nseg) break;
        if (s + 2 < nseg) piece(w[0], s + 2);
#pragma unroll
        for (int q = 0; q < 4 * NK; ++q) v[q] += w[1][q];
    }
}

// One thread per stored mode (warps = 32 consecutive modes), EPI_STEPS steps a CTA (a tile's
// columns are a multiple of theirs, so a CTA reads one tile of the product).
constexpr int EPI_STEPS = 4;
__global__ void __launch_bounds__(SG_BM) fp32_bin_epilogue_kernel(const __grid_constant__ SgemmParams p, int K,
                                                                const int *mode_bin,
                                                                const int *mode_slot,
                                                                float *partials, int n_slots) {
    const int n = blockIdx.x * SG_BM + threadIdx.x;
    const int lane = threadIdx.x & 31;
    const int k0 = blockIdx.y * EPI_STEPS;
    float v[4 * EPI_STEPS];
    sg_load<EPI_STEPS>(v, p, 0, k0, K);
    const int bin = mode_bin[n];
    const int slot = mode_slot[n];
    const uint32_t take = seg_scan_masks(bin, lane);
#pragma unroll
    for (int q = 0; q < EPI_STEPS; ++q) {
        const int k = k0 + q;
        if (k >= K) break;   // uniform
#pragma unroll
        for (int a = 0; a < 3; ++a) {   // Eq. 16: J_n = y_n Xdot_n, summed per bin run
            const float s = seg_scan(v[4 * q] * v[4 * q + 1 + a], take);
            if (slot >= 0) partials[((size_t)k * 3 + a) * n_slots + slot] = s;
        }
    }
}

// Direction-resolved variant: the three products R_b of the direction segments of d.
constexpr int DIR_EPI_STEPS = 2;
__global__ void __launch_bounds__(SG_BM) fp32_dir_epilogue_kernel(const __grid_constant__ SgemmParams p, int K,
                                                                const int *mode_bin,
                                                                const int *mode_slot,
                                                                float *partials, int n_slots) {
    const int n = blockIdx.x * SG_BM + threadIdx.x;
    const int lane = threadIdx.x & 31;
    const int k0 = blockIdx.y * DIR_EPI_STEPS;
    float v[3][4 * DIR_EPI_STEPS];
#pragma unroll
    for (int b = 0; b < 3; ++b) sg_load<DIR_EPI_STEPS>(v[b], p, b, k0, K);
    const int bin = mode_bin[n];
    const int slot = mode_slot[n];
    const uint32_t take = seg_scan_masks(bin, lane);
#pragma unroll
    for (int q = 0; q < DIR_EPI_STEPS; ++q) {
        const int k = k0 + q;
        if (k >= K) break;   // uniform
        const float x = (v[0][4 * q] + v[1][4 * q]) + v[2][4 * q];   // Eq. 13 over all d
#pragma unroll
        for (int b = 0; b < 3; ++b)
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                const float s = seg_scan(x * v[b][4 * q + 1 + a], take);
                if (slot >= 0) partials[((size_t)k * 3 + a) * (3 * (size_t)n_slots) + (size_t)b * n_slots + slot] = s;
            }
    }
}

// FP32 FMA throughput: every thread runs FMA_CHAINS independent dependency chains of
// a = a * m + c (m just below 1, so values stay finite), the chains interleaved so that the
// pipe never waits on one; one value per thread is stored so that nothing is dropped.
constexpr int FMA_CHAINS = 16;
__global__ void __launch_bounds__(256) fma_peak_kernel(float *out, int iters) {
    float a[FMA_CHAINS];
#pragma unroll
    for (int q = 0; q < FMA_CHAINS; ++q) a[q] = 1e-3f * (float)(threadIdx.x + q);
    const float m = 0.9999999f, c = 1e-7f;
    for (int it = 0; it < iters; ++it) {
#pragma unroll
        for (int q = 0; q < FMA_CHAINS; ++q) a[q] = fmaf(a[q], m, c);
    }
    float t = 0.f;
#pragma unroll
    for (int q = 0; q < FMA_CHAINS; ++q) t += a[q];
    out[blockIdx.x * blockDim.x + threadIdx.x] = t;
}

}  // namespace

cudaError_t measure_fp32_fma(cudaStream_t s, int sm_count, double *tflops) {
    const int blocks = sm_count * 8, threads = 256, iters = 4096;
    float *out = nullptr;
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    cudaError_t e = cudaMalloc(&out, sizeof(float) * blocks * threads);
    if (e == cudaSuccess) e = cudaEventCreate(&e0);
    if (e == cudaSuccess) e = cudaEventCreate(&e1);
    float best = 0.f;
    for (int r = 0; r < 4 && e == cudaSuccess; ++r) {   // launch 0 warms up
        cudaEventRecord(e0, s);
        fma_peak_kernel<<<blocks, threads, 0, s>>>(out, iters);
        cudaEventRecord(e1, s);
        if ((e = cudaEventSynchronize(e1)) != cudaSuccess) break;
        float ms = 0.f;
        cudaEventElapsedTime(&ms, e0, e1);
        if (r > 0 && (best == 0.f || ms < best)) best = ms;
    }
    if (e == cudaSuccess) e = cudaGetLastError();
    if (e == cudaSuccess && best > 0.f)
        *tflops = 2.0 * (double)blocks * threads * iters * FMA_CHAINS / (best * 1e-3) / 1e12;
    if (e0) cudaEventDestroy(e0);
    if (e1) cudaEventDestroy(e1);
    if (out) cudaFree(out);
    return e;
}

SgemmPlan sgemm_plan(int64_t Mp, int C, int64_t Dk, int ndir, int sms, bool cut) {
    const int ctas = SG_CTAS * std::max(1, sms);
    SgemmPlan p{};
    p.ndir = ndir;
    p.n_mt = (int)(Mp / SG_BM);
    p.n_ct = (C + SG_BN - 1) / SG_BN;
    p.n_kb = (int)(Dk / SG_BK);
    p.nch = (p.n_kb + SG_CHUNK_KB - 1) / SG_CHUNK_KB;
    p.tiles = ndir * p.n_mt * p.n_ct;
    p.t0 = cut ? p.tiles / ctas * ctas : p.tiles;
    p.max_seg = 1;
    const int tail = p.tiles - p.t0;
    // one range of the tail's chunks a CTA, but no tile in more than SGEMM_MAX_SEG pieces
    p.parts = (int)std::min<long long>(std::min(ctas, tail * (SGEMM_MAX_SEG - 1)), (long long)tail * p.nch);
    p.ctas = std::max(std::min(ctas, p.t0), p.parts);
    for (int t = p.t0; t < p.tiles; ++t) p.max_seg = std::max(p.max_seg, p.segments(t));
    return p;
}

cudaError_t launch_sgemm(const SgemmParams &p, cudaStream_t s, bool pdl) {
    static PerDevice once;
    const cudaError_t ready = opt_in_smem(once, sgemm_kernel, SG_SMEM);
    if (ready != cudaSuccess) return ready;
    if (p.plan.tiles < 1 || p.C < 1) return cudaSuccess;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)p.plan.ctas, 1, 1);
    cfg.blockDim = dim3(SG_THREADS, 1, 1);
    cfg.dynamicSmemBytes = SG_SMEM;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;   // after the pack
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = pdl ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, sgemm_kernel, p);
}

int sgemm_make_maps(const float *Ed32, int64_t Mp, const float *Bd32, int64_t cols, int64_t D, SgemmParams &p) {
    const int r = tc_make_tmap_f32(&p.tmA, Ed32, (uint64_t)D, (uint64_t)Mp, (uint64_t)Mp, SG_BK, SG_BM);
    return r ? r : tc_make_tmap_f32(&p.tmB, Bd32, (uint64_t)D, (uint64_t)cols, (uint64_t)cols, SG_BK, SG_BN);
}

void launch_fp32_epilogue(const SgemmParams &p, int K, const int *mode_bin, const int *mode_slot,
                          float *partials, int n_slots, cudaStream_t s) {
    const int steps = p.plan.ndir == 3 ? DIR_EPI_STEPS : EPI_STEPS;
    dim3 grid(p.Mp / SG_BM, (K + steps - 1) / steps);
    if (p.plan.ndir == 3)
        fp32_dir_epilogue_kernel<<<grid, SG_BM, 0, s>>>(p, K, mode_bin, mode_slot, partials, n_slots);
    else
        fp32_bin_epilogue_kernel<<<grid, SG_BM, 0, s>>>(p, K, mode_bin, mode_slot, partials, n_slots);
}

}  // namespace mhc

// K1 pack: per-step B-operand rows of the two projections and the FP64 total
// heat current (Eq. 10, Eq. 13, Eq. 16).
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include <algorithm>
#include <map>
#include <mutex>

#include "common.cuh"
#include "kernels.h"

namespace mhc {

namespace {

constexpr int PACK_THREADS = 512;

// Row r (0: velocities, 1..3: virials) of step k at column d.
__device__ __forceinline__ void store_split(const PackArgs &a, int k, int r, size_t d, float val) {
    const size_t idx = (size_t)(4 * k + r) * a.D_ld + d;
    if (a.split == SPLIT_BF16) {
        __nv_bfloat16 hi = __float2bfloat16_rn(val);
        __nv_bfloat16 lo = __float2bfloat16_rn(val - __bfloat162float(hi));
        static_cast<__nv_bfloat16 *>(a.Bt_hi)[idx] = hi;
        static_cast<__nv_bfloat16 *>(a.Bt_lo)[idx] = lo;
    } else if (a.split == SPLIT_FP16) {
        __half hi = __float2half_rn(val);
        __half lo = __float2half_rn(val - __half2float(hi));
        static_cast<__half *>(a.Bt_hi)[idx] = hi;
        static_cast<__half *>(a.Bt_lo)[idx] = lo;
    } else {
        a.Bd32[d * a.b_cols + 4 * k + r] = val;
    }
}

// TwoProduct + TwoSum: add w*v exactly into the unevaluated float pair (s, c).
// Explicit _rn intrinsics keep the compiler from contracting these into FMAs.
__device__ __forceinline__ void acc_exact(float &s, float &c, float w, float v) {
    const float pr = __fmul_rn(w, v);
    const float pe = fmaf(w, v, -pr);                       // w*v = pr + pe exactly
    const float t = __fadd_rn(s, pr);
    const float bp = __fsub_rn(t, s);
    const float er = __fadd_rn(__fsub_rn(s, __fsub_rn(t, bp)), __fsub_rn(pr, bp));
    s = t;
    c = __fadd_rn(c, __fadd_rn(er, pe));
}

// (s, c) += (s2, c2): the leading parts added error-free (TwoSum), the rounding error and the
// trailing parts into c.  FP32 instructions only: GB300's FP64 pipe is too narrow for a
// warp-wide FP64 reduction per CTA (it cost ~5 us of a 26 us pack).
__device__ __forceinline__ void pair_add(float &s, float &c, float s2, float c2) {
    const float t = __fadd_rn(s, s2);
    const float bp = __fsub_rn(t, s);
    const float e = __fadd_rn(__fsub_rn(s, __fsub_rn(t, bp)), __fsub_rn(s2, bp));
    s = t;
    c = __fadd_rn(c, __fadd_rn(c2, e));
}

__global__ void __launch_bounds__(PACK_THREADS) pack_kernel(const PackArgs a) {
    const int k = blockIdx.x;
    const float *v = a.v + (size_t)k * a.N * 3;
    const float *W = a.W + (size_t)k * a.N * 9;

    // Phase 1, one thread per atom: row maxima (for the power-of-two scales) and
    // Eq. 10, J^a = sum_i sum_b W_i^{ab} v_i^b.  Products are added exactly into an
    // unevaluated float pair per thread (about 48 significant bits with FP32
    // instructions only) and the pairs are combined in FP64 below.  (GB300's FP64
    // pipe is too narrow for 9 FP64 FMAs per atom per step.)
    float mx[4] = {0.f, 0.f, 0.f, 0.f};
    float js[3] = {0.f, 0.f, 0.f}, jc[3] = {0.f, 0.f, 0.f};
    for (int i = threadIdx.x; i < a.N; i += PACK_THREADS) {
        float vv[3], ww[9];
#pragma unroll
        for (int b = 0; b < 3; ++b) vv[b] = v[(size_t)i * 3 + b];
#pragma unroll
        for (int q = 0; q < 9; ++q) ww[q] = W[(size_t)i * 9 + q];
        const float sm = a.sqm[i], ism = a.isqm[i];
#pragma unroll
        for (int b = 0; b < 3; ++b) mx[0] = fmaxf(mx[0], fabsf(sm * vv[b]));
#pragma unroll
        for (int al = 0; al < 3; ++al)
#pragma unroll
            for (int b = 0; b < 3; ++b) {
                mx[1 + al] = fmaxf(mx[1 + al], fabsf(ww[3 * al + b] * ism));
                acc_exact(js[al], jc[al], ww[3 * al + b], vv[b]);
            }
    }
    double j[3];
#pragma unroll
    for (int al = 0; al < 3; ++al) j[al] = (double)js[al] + (double)jc[al];
    __shared__ float s_mx[PACK_THREADS / 32][4];
    __shared__ double s_j[PACK_THREADS / 32][3];
    __shared__ float s_mul[4];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
#pragma unroll
        for (int c = 0; c < 4; ++c) mx[c] = fmaxf(mx[c], __shfl_down_sync(FULL_MASK, mx[c], o));
#pragma unroll
        for (int c = 0; c < 3; ++c) j[c] += __shfl_down_sync(FULL_MASK, j[c], o);
    }
    if (lane == 0) {
        for (int c = 0; c < 4; ++c) s_mx[warp][c] = mx[c];
        for (int c = 0; c < 3; ++c) s_j[warp][c] = j[c];
    }
    __syncthreads();
    if (threadIdx.x < 4) {
        const int c = threadIdx.x;
        float m = 0.f;
        for (int w = 0; w < PACK_THREADS / 32; ++w) m = fmaxf(m, s_mx[w][c]);
        int s = 0;
        if (a.split == SPLIT_FP16 && m > 0.f && isfinite(m)) {
            int e;
            frexpf(m, &e);      // m < 2^e
            s = 14 - e;         // scaled row maximum < 2^14 keeps the lo parts normal
        }
        s_mul[c] = ldexpf(1.f, s);
        a.col_scale[4 * k + c] = ldexpf(1.f, -(s + a.e_exp));
    } else if (threadIdx.x >= 32 && threadIdx.x < 35) {
        const int c = threadIdx.x - 32;
        double t = 0.0;
        for (int w = 0; w < PACK_THREADS / 32; ++w) t += s_j[w][c];
        a.Jtot[3 * k + c] = t;
        if (a.Jring) {
            const long long t0 = a.t0_dev ? *a.t0_dev : a.t0;
            a.Jring[((t0 + k) % a.R) * 3 + c] = t;
        }
    }
    __syncthreads();

    // Phase 2, one thread per atom: the four scaled rows of step k,
    //   Bt[4k][3i+b] = sqrt(m_i) v_i^b,  Bt[4k+1+a][3i+b] = W_i^{ab} / sqrt(m_i),
    // split into hi/lo (inputs re-read from L2).
    // (direction-major columns b*npad + i when npad > 0)
    const float mul[4] = {s_mul[0], s_mul[1], s_mul[2], s_mul[3]};
    const size_t cs_i = a.npad ? 1 : 3, cs_b = a.npad ? (size_t)a.npad : 1;
    for (int i = threadIdx.x; i < a.N; i += PACK_THREADS) {
        const float sm = a.sqm[i], ism = a.isqm[i];
#pragma unroll
        for (int b = 0; b < 3; ++b)
            store_split(a, k, 0, cs_i * i + cs_b * b, (sm * v[(size_t)i * 3 + b]) * mul[0]);
#pragma unroll
        for (int al = 0; al < 3; ++al)
#pragma unroll
            for (int b = 0; b < 3; ++b)
                store_split(a, k, 1 + al, cs_i * i + cs_b * b,
                            (W[(size_t)i * 9 + 3 * al + b] * ism) * mul[1 + al]);
    }
}

// ------------------------------------------------------------------ cluster / bulk-copy pack
__device__ __forceinline__ double ld_cluster_f64(uint32_t addr) {
    double v;
    asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(v) : "r"(addr) : "memory");
    return v;
}
__device__ __forceinline__ float ld_cluster_f32(uint32_t addr) {
    float v;
    asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(addr) : "memory");
    return v;
}

// Four consecutive values of one row: one 8-byte store each for hi and lo.
__device__ __forceinline__ void store_split4(const PackArgs &a, size_t idx, const float (&x)[4]) {
    uint32_t h[4], l[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        if (a.split == SPLIT_BF16) {
            const __nv_bfloat16 hv = __float2bfloat16_rn(x[q]);
            h[q] = __bfloat16_as_ushort(hv);
            l[q] = __bfloat16_as_ushort(__float2bfloat16_rn(x[q] - __bfloat162float(hv)));
        } else {
            const __half hv = __float2half_rn(x[q]);
            h[q] = __half_as_ushort(hv);
            l[q] = __half_as_ushort(__float2half_rn(x[q] - __half2float(hv)));
        }
    }
    *reinterpret_cast<uint2 *>(static_cast<uint16_t *>(a.Bt_hi) + idx) = make_uint2(h[0] | (h[1] << 16), h[2] | (h[3] << 16));
    *reinterpret_cast<uint2 *>(static_cast<uint16_t *>(a.Bt_lo) + idx) = make_uint2(l[0] | (l[1] << 16), l[2] | (l[3] << 16));
}

// A cluster of ceil(N / (4 THREADS)) CTAs per step k.  CTA r copies the contiguous velocities and
// virials of its atoms r*4*THREADS .. into shared memory, every copy in flight at once and the
// inputs read once: by TMA where the step's inputs start on 16-byte boundaries, else (N % 4 != 0,
// or a caller's pointer in the middle of a buffer) by 4-byte asynchronous copies.  Phase 1, thread
// t takes the atoms t, t+THREADS, t+2 THREADS, t+3 THREADS (shared-memory strides of 3 and 9 words
// across a warp: no bank conflicts): row maxima and the exact total-current pairs (acc_exact),
// combined per CTA in a fixed order (unevaluated float pairs across the warp, FP64 across the
// warps); one cluster barrier, then every CTA combines all ranks' maxima in rank order through
// distributed shared memory (each computes the same scales) and rank 0 the current (FP64, rank
// order).  Phase 1 also replaces each atom's inputs in shared memory by its row values sqrt(m) v
// and W / sqrt(m).  Phase 2 writes the four B rows of the CTA's atoms: each row is one contiguous
// run of 16-bit values (three per atom; three runs of one per atom, one per direction, with the
// direction-major columns), cut into groups of four values that consecutive threads take in
// order, so that every warp store covers 256 contiguous bytes (the last group's values past the
// system are zeros in the padding of B's rows).  A CTA leaves only after the second half of the
// cluster barrier: its peers may still be reading its partial sums.
// What bounds it: a wave's chain of load, barrier and store (the stores wait for the row maxima),
// at 4.1 TB/s of the 96 bytes an atom and step.  Keeping the values in registers over the barrier
// and storing through shared memory by bulk copies halved the instructions and was not faster
// (8000 atoms, K = 256: 52 against 48.5 us).  Atoms not a multiple of four and systems beyond
// 16384 atoms, which a kernel of one CTA a step packed from two reads of the inputs, measured
// (us, before -> now): 1003 atoms, K = 77 13.0 -> 8.9; 20000 atoms, K = 512 425 -> 270.
template <int THREADS>
__device__ __forceinline__ void pack_cluster_body(const PackArgs &a, int k, uint32_t rank, uint32_t nrank) {
    constexpr int APC = 4 * THREADS;
    extern __shared__ float4 pk_smem4[];
    float *sv = reinterpret_cast<float *>(pk_smem4);   // [APC][3]
    float *sw = sv + APC * 3;                          // [APC][9]
    __shared__ float s_mx[THREADS / 32][4];
    __shared__ float s_js[THREADS / 32][3], s_jcc[THREADS / 32][3];
    __shared__ float s_loc[4], s_mul[4];
    __shared__ double s_jc[3];
    __shared__ __align__(8) uint64_t bar;
    __shared__ int abort_flag;
    const int a0 = (int)rank * APC;
    const int na = max(0, min(APC, a.N - a0));
    const long long limit = a.wait_limit > 0 ? a.wait_limit : WAIT_LIMIT_CYCLES;
    const float *gv = a.v + ((size_t)k * a.N + a0) * 3, *gw = a.W + ((size_t)k * a.N + a0) * 9;
    const bool bulk = ((a.N & 3) | ((reinterpret_cast<uintptr_t>(a.v) | reinterpret_cast<uintptr_t>(a.W)) & 15)) == 0;
    bool ok = true;
    if (bulk) {
        if (threadIdx.x == 0) {
            mbar_init(&bar, 1);
            abort_flag = 0;
            fence_mbar_init();
        }
        __syncthreads();
        if (threadIdx.x == 0 && na > 0) {
            const uint32_t vb = (uint32_t)na * 12, wb = (uint32_t)na * 36;
            mbar_arrive_expect_tx(&bar, vb + wb);
            for (uint32_t o = 0; o < vb; o += 16384)
                bulk_load(reinterpret_cast<char *>(sv) + o, reinterpret_cast<const char *>(gv) + o, min(16384u, vb - o), &bar);
            for (uint32_t o = 0; o < wb; o += 16384)
                bulk_load(reinterpret_cast<char *>(sw) + o, reinterpret_cast<const char *>(gw) + o, min(16384u, wb - o), &bar);
        }
        if (na > 0) ok = mbar_wait(&bar, 0, &abort_flag, limit);
    } else {
        for (int q = threadIdx.x; q < 3 * na; q += THREADS) cp_async4(sv + q, gv + q);
        for (int q = threadIdx.x; q < 9 * na; q += THREADS) cp_async4(sw + q, gw + q);
        cp_async_wait_all();
        __syncthreads();
    }
    float mx[4] = {0.f, 0.f, 0.f, 0.f};
    float js[3] = {0.f, 0.f, 0.f}, jc[3] = {0.f, 0.f, 0.f};
    if (ok) {
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int ia = (int)threadIdx.x + u * THREADS;
            if (ia >= na) break;
            const float sm = __ldg(a.sqm + a0 + ia), ism = __ldg(a.isqm + a0 + ia);
            float *vu = sv + ia * 3, *wu = sw + ia * 9;
            float x[12];   // the atom's row values sqrt(m) v^b and W^{ab} / sqrt(m)
#pragma unroll
            for (int b = 0; b < 3; ++b) {
                x[b] = sm * vu[b];
                mx[0] = fmaxf(mx[0], fabsf(x[b]));
            }
#pragma unroll
            for (int al = 0; al < 3; ++al)
#pragma unroll
                for (int b = 0; b < 3; ++b) {
                    x[3 + 3 * al + b] = wu[3 * al + b] * ism;
                    mx[1 + al] = fmaxf(mx[1 + al], fabsf(x[3 + 3 * al + b]));
                    acc_exact(js[al], jc[al], wu[3 * al + b], vu[b]);
                }
            // the scaled values replace the inputs in shared memory (this thread's atom alone),
            // so phase 2 reads them without the masses
#pragma unroll
            for (int b = 0; b < 3; ++b) vu[b] = x[b];
#pragma unroll
            for (int q = 0; q < 9; ++q) wu[q] = x[3 + q];
        }
    }
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
#pragma unroll
        for (int c = 0; c < 4; ++c) mx[c] = fmaxf(mx[c], __shfl_down_sync(FULL_MASK, mx[c], o));
#pragma unroll
        for (int c = 0; c < 3; ++c)
            pair_add(js[c], jc[c], __shfl_down_sync(FULL_MASK, js[c], o), __shfl_down_sync(FULL_MASK, jc[c], o));
    }
    if (lane == 0) {
        for (int c = 0; c < 4; ++c) s_mx[warp][c] = mx[c];
        for (int c = 0; c < 3; ++c) {
            s_js[warp][c] = js[c];
            s_jcc[warp][c] = jc[c];
        }
    }
    __syncthreads();
    if (threadIdx.x < 4) {
        float m = 0.f;
        for (int w = 0; w < THREADS / 32; ++w) m = fmaxf(m, s_mx[w][threadIdx.x]);
        s_loc[threadIdx.x] = m;
    } else if (threadIdx.x >= 32 && threadIdx.x < 35) {   // the warps' pairs in FP64, warp order
        const int c = threadIdx.x - 32;
        double t = 0.0;
        for (int w = 0; w < THREADS / 32; ++w) t += (double)s_js[w][c] + (double)s_jcc[w][c];
        s_jc[c] = t;
    }
    cluster_sync_all();   // every CTA's maxima and current partials are complete
    if (threadIdx.x < 4) {
        const int c = threadIdx.x;
        float m = 0.f;
        for (uint32_t q = 0; q < nrank; ++q) m = fmaxf(m, ld_cluster_f32(mapa_shared(smem_u32(&s_loc[c]), q)));
        int sc = 0;
        if (a.split == SPLIT_FP16 && m > 0.f && isfinite(m)) {
            int e;
            frexpf(m, &e);   // m < 2^e
            sc = 14 - e;     // scaled row maximum < 2^14 keeps the lo parts normal
        }
        s_mul[c] = ldexpf(1.f, sc);
        if (rank == 0) a.col_scale[4 * k + c] = ldexpf(1.f, -(sc + a.e_exp));
    } else if (rank == 0 && threadIdx.x >= 32 && threadIdx.x < 35) {
        const int c = threadIdx.x - 32;
        double t = 0.0;
        for (uint32_t q = 0; q < nrank; ++q) t += ld_cluster_f64(mapa_shared(smem_u32(&s_jc[c]), q));
        a.Jtot[3 * k + c] = t;
        if (a.Jring) {
            const long long t0 = a.t0_dev ? *a.t0_dev : a.t0;
            a.Jring[((t0 + k) % a.R) * 3 + c] = t;
        }
    }
    cluster_arrive_release();   // this CTA has read its peers' partials
    __syncthreads();            // s_mul is visible to the CTA
    if (!ok) {   // the CTA stays alive until its copy has landed (bounded) or given up on
        if (threadIdx.x == 0) {
            if (a.status) set_status(a.status, DEV_TIMEOUT);
            const long long c0 = clock64();
            while (!mbar_try_wait(&bar, 0) && clock64() - c0 < limit) {
            }
        }
    } else {
        const size_t ld = (size_t)a.D_ld;
        const size_t r0 = (size_t)(4 * k) * ld;
        const int q4 = (na + 3) / 4;                        // groups of four atoms (direction-major runs)
        const int G = a.npad ? 3 * q4 : (3 * na + 3) / 4;   // groups of four values a row
#pragma unroll 1
        for (int g = (int)threadIdx.x; g < G; g += THREADS) {
            int ia[4], bb[4];
            size_t col;
            if (a.npad) {   // direction-major: run b holds atoms a0 .. a0+na-1 at columns b*npad + i
                const int b = g / q4, i0 = 4 * (g - b * q4);
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    ia[e] = i0 + e;
                    bb[e] = b;
                }
                col = (size_t)b * a.npad + a0 + i0;
            } else {        // column 3i+b: values 4g .. 4g+3 of the CTA's run
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    ia[e] = (4 * g + e) / 3;
                    bb[e] = (4 * g + e) - 3 * ia[e];
                }
                col = 3 * (size_t)a0 + 4 * (size_t)g;
            }
            float x[4][4];   // [row][value]
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const bool in = ia[e] < na;
                x[0][e] = in ? sv[3 * ia[e] + bb[e]] * s_mul[0] : 0.f;
#pragma unroll
                for (int al = 0; al < 3; ++al)
                    x[1 + al][e] = in ? sw[9 * ia[e] + 3 * al + bb[e]] * s_mul[1 + al] : 0.f;
            }
            if (a.split == SPLIT_FP32) {   // d-major: the step's four rows are 16 bytes of a d
#pragma unroll
                for (int e = 0; e < 4; ++e)
                    if (ia[e] < na)
                        *reinterpret_cast<float4 *>(a.Bd32 + (col + e) * a.b_cols + 4 * k) =
                            make_float4(x[0][e], x[1][e], x[2][e], x[3][e]);
            } else {
#pragma unroll
                for (int r = 0; r < 4; ++r) store_split4(a, r0 + (size_t)r * ld + col, x[r]);
            }
        }
    }
    cluster_wait_acquire();   // peers have read this CTA's partials: its shared memory may go
}

// Shared memory (48 B an atom) allows eight CTAs of 128 threads, four of 256 or two of 512 per
// SM; the register cap of the launch bounds lets as many be resident.
template <int THREADS>
__global__ void __launch_bounds__(THREADS, 1024 / THREADS) pack_cluster_kernel(const PackArgs a) {
    griddep_launch_dependents();   // the projection may set up on the SMs this grid leaves
    const uint32_t nrank = cluster_nctarank();
    pack_cluster_body<THREADS>(a, (int)(blockIdx.x / nrank), cluster_ctarank(), nrank);
}

// Several systems in one launch: system j owns the CTAs cta_begin[j] .. cta_begin[j+1) (K_j
// clusters of the common cluster size; ranks beyond a system's atoms hold no atoms and only
// take part in the cluster's combination).
template <int THREADS>
__global__ void __launch_bounds__(THREADS, 1024 / THREADS) pack_cluster_group_kernel(const __grid_constant__ PackGroupArgs g) {
    griddep_launch_dependents();
    int j = 0;
    while (j + 1 < g.n && (int)blockIdx.x >= g.cta_begin[j + 1]) ++j;
    const uint32_t nrank = cluster_nctarank();
    pack_cluster_body<THREADS>(g.a[j], (int)((blockIdx.x - (uint32_t)g.cta_begin[j]) / nrank),
                            cluster_ctarank(), nrank);
}

template <int THREADS>
cudaError_t launch_pack_cluster(const PackArgs &a, cudaStream_t s) {
    constexpr int APC = 4 * THREADS;
    const int smem = APC * 48;
    static PerDevice once;
    const cudaError_t attr = opt_in_smem(once, pack_cluster_kernel<THREADS>, smem);
    if (attr != cudaSuccess) return attr;
    const int csize = (a.N + APC - 1) / APC;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(a.K * csize), 1, 1);
    cfg.blockDim = dim3(THREADS, 1, 1);
    cfg.dynamicSmemBytes = (size_t)smem;
    cfg.stream = s;
    cudaLaunchAttribute la[1];
    la[0].id = cudaLaunchAttributeClusterDimension;
    la[0].val.clusterDim.x = (unsigned)csize;
    la[0].val.clusterDim.y = 1;
    la[0].val.clusterDim.z = 1;
    cfg.attrs = la;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, pack_cluster_kernel<THREADS>, a);
}

}  // namespace

namespace {
// CTA size of the cluster pack of a system of N atoms (four atoms a thread): one CTA a step and
// eight an SM up to 512 atoms, clusters of up to 8 CTAs of 256 (four an SM) up to 8192, of 512
// beyond; clusters of more than 8 CTAs (the portable size) from 16384 atoms, up to 16.
int pack_threads(int N) { return N <= 4 * 128 ? 128 : N <= 8 * 1024 ? 256 : 512; }
constexpr int PACK_MAX_CLUSTER = 16;

// Whether a cluster of `csize` 512-thread CTAs can be resident on the current device.
bool pack_wide_ok(int csize) {
    static std::map<int, int> limits;   // device -> largest cluster size found to fit
    static std::mutex m;
    std::lock_guard<std::mutex> lock(m);
    int device = 0;
    if (cudaGetDevice(&device) != cudaSuccess) return false;
    if (!limits.count(device)) {
        int limit = 8;
        const int smem = 4 * 512 * 48;
        if (cudaFuncSetAttribute(pack_cluster_kernel<512>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess &&
            cudaFuncSetAttribute(pack_cluster_group_kernel<512>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess &&
            cudaFuncSetAttribute(pack_cluster_kernel<512>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) == cudaSuccess) {
            for (int cs = 9; cs <= PACK_MAX_CLUSTER; ++cs) {
                cudaLaunchConfig_t cfg = {};
                cfg.gridDim = dim3((unsigned)cs, 1, 1);
                cfg.blockDim = dim3(512, 1, 1);
                cfg.dynamicSmemBytes = smem;
                cudaLaunchAttribute la[1];
                la[0].id = cudaLaunchAttributeClusterDimension;
                la[0].val.clusterDim.x = (unsigned)cs;
                la[0].val.clusterDim.y = 1;
                la[0].val.clusterDim.z = 1;
                cfg.attrs = la;
                cfg.numAttrs = 1;
                int n = 0;
                if (cudaOccupancyMaxActiveClusters(&n, pack_cluster_kernel<512>, &cfg) != cudaSuccess || n < 1) break;
                limit = cs;
            }
        }
        cudaGetLastError();
        limits[device] = limit;
    }
    return csize <= limits[device];
}

// The cluster pack takes every system up to PACK_MAX_CLUSTER CTAs of 2048 atoms.
bool cluster_ok(const PackArgs &a) {
    const auto al16 = [](const void *q) { return (reinterpret_cast<uintptr_t>(q) & 15) == 0; };
    const bool out = a.split == SPLIT_FP32 ? al16(a.Bd32) : al16(a.Bt_hi) && al16(a.Bt_lo);
    return out && (a.N <= 8 * 2048 || (a.N <= PACK_MAX_CLUSTER * 2048 && pack_wide_ok((a.N + 2047) / 2048)));
}

template <int THREADS>
cudaError_t launch_pack_cluster_group(PackGroupArgs g, int csize, cudaStream_t s) {
    constexpr int APC = 4 * THREADS;
    const int smem = APC * 48;
    static PerDevice once;
    const cudaError_t attr = opt_in_smem(once, pack_cluster_group_kernel<THREADS>, smem);
    if (attr != cudaSuccess) return attr;
    g.cta_begin[0] = 0;
    for (int j = 0; j < g.n; ++j) g.cta_begin[j + 1] = g.cta_begin[j] + g.a[j].K * csize;
    if (g.cta_begin[g.n] == 0) return cudaSuccess;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)g.cta_begin[g.n], 1, 1);
    cfg.blockDim = dim3(THREADS, 1, 1);
    cfg.dynamicSmemBytes = (size_t)smem;
    cfg.stream = s;
    cudaLaunchAttribute la[1];
    la[0].id = cudaLaunchAttributeClusterDimension;
    la[0].val.clusterDim.x = (unsigned)csize;
    la[0].val.clusterDim.y = 1;
    la[0].val.clusterDim.z = 1;
    cfg.attrs = la;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, pack_cluster_group_kernel<THREADS>, g);
}
}  // namespace

cudaError_t launch_pack_group(const PackGroupArgs &g, const cudaStream_t *streams, int n_streams,
                              int *n_launches) {
    *n_launches = 0;
    if (g.n < 1 || g.n > TC_MAX_GROUP) return cudaErrorInvalidValue;
    for (int j = 0; j < g.n; ++j)
        if (!cluster_ok(g.a[j])) return cudaErrorNotSupported;
    // one launch per (CTA size, cluster size): every system is packed by the CTA size it gets
    // alone (so its results are bitwise those of a solo push), and no rank is idle
    for (const int threads : {128, 256, 512}) {
        const int apc = 4 * threads;
        for (int cs = 1; cs <= (threads == 512 ? PACK_MAX_CLUSTER : 8); ++cs) {
            PackGroupArgs sub{};
            for (int j = 0; j < g.n; ++j)
                if (pack_threads(g.a[j].N) == threads &&
                    ((g.a[j].N + apc - 1) / apc == cs || (g.a[j].N == 0 && cs == 1)))
                    sub.a[sub.n++] = g.a[j];
            if (sub.n == 0) continue;
            const cudaStream_t s = streams[*n_launches % n_streams];   // independent systems
            const cudaError_t e = threads == 128 ? launch_pack_cluster_group<128>(sub, cs, s)
                                  : threads == 256 ? launch_pack_cluster_group<256>(sub, cs, s)
                                                   : launch_pack_cluster_group<512>(sub, cs, s);
            if (e != cudaSuccess) return e;
            ++*n_launches;
        }
    }
    return cudaSuccess;
}

cudaError_t launch_pack(const PackArgs &a, cudaStream_t s) {
    if (a.K <= 0) return cudaSuccess;
    if (cluster_ok(a)) {
        const int threads = pack_threads(a.N);
        return threads == 128 ? launch_pack_cluster<128>(a, s)
               : threads == 256 ? launch_pack_cluster<256>(a, s)
                                : launch_pack_cluster<512>(a, s);
    }
    pack_kernel<<<a.K, PACK_THREADS, 0, s>>>(a);
    return cudaGetLastError();
}

}  // namespace mhc

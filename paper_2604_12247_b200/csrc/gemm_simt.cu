// CUDA-core weight-streaming kernels: the skinny GEMM  out[row][n] = sum_k act[row][k] W[n][k]
// for up to 8 rows, and the exit-confidence kernel (LM-head GEMV fused with the online
// temperature-scaled softmax max / argmax of Eq. 2).  One warp per output row, 128-bit coalesced
// weight loads, fp32 accumulation.  These cover every dtype (fp32 models never use tensor cores:
// tf32 would break their 1e-4 logit tolerance) and are the reference path for the tcgen05 kernels.  On small models they are
// bound by latency, a chain of launches of 3-6 us: hence SwiGLU in the gate/up kernel and grids no larger than their rows.
#include "sb_internal.cuh"

namespace sb {

// eight consecutive weights of a row as floats
__device__ __forceinline__ void load8(const float* p, float (&w)[8]) {
    float4 a = __ldg(reinterpret_cast<const float4*>(p));
    float4 b = __ldg(reinterpret_cast<const float4*>(p) + 1);
    w[0] = a.x; w[1] = a.y; w[2] = a.z; w[3] = a.w; w[4] = b.x; w[5] = b.y; w[6] = b.z; w[7] = b.w;
}
__device__ __forceinline__ void load8(const __nv_bfloat16* p, float (&w)[8]) {
    uint4 u = __ldg(reinterpret_cast<const uint4*>(p));
    const uint32_t r[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        w[2 * j] = __uint_as_float(r[j] << 16);
        w[2 * j + 1] = __uint_as_float(r[j] & 0xffff0000u);
    }
}
// eight consecutive activations of row `row` as floats
__device__ __forceinline__ void load_act8(const float* a, int row, int k, int K, float (&x)[8]) {
    load8(a + (size_t)row * K + k, x);
}
__device__ __forceinline__ void load_act8(const __nv_bfloat16* a, int row, int k, int K, float (&x)[8]) {
    float lo[8];
    load8(a + (size_t)row * K + k, x);
    load8(a + (size_t)(row + 8) * K + k, lo);
#pragma unroll
    for (int j = 0; j < 8; ++j) x[j] += lo[j];
}

// M = rows of the launch (1 .. 8): an instance each, whose registers and instructions are those of its rows (one instance for up
// to 8 predicated rows took 76 registers for one row, three blocks per SM instead of six).  Bound by the weight stream at few
// rows, which is as fast as there are loads in flight, and by the activations' loads at many.  Hence for fp32 weights: up to four
// rows, the next pieces of the weight row are requested before this one is used (two ahead at one or two rows, where registers
// are left for it), and above four rows the activations of four rows are requested together.  With bf16 weights, whose
// activations are two halves, either only costs registers.  us for 3 layers, rows predicated / an instance each / as it is: fp32
// d_model 4096, 1 row 960 / 724 / 567, 4 rows 1338 / 1176 / 1050; d_model 2048, 8 rows 577 / 647 / 607; d_model 512, 1 row 72 /
// 61 / 59; bf16 7B shape, 1 row 570 / 335, 8 rows 1976 / 1538.
template <typename T, int M>
__device__ __forceinline__ void row_dots(const T* __restrict__ wrow, const typename Act<T>::type* __restrict__ act, int K,
                                         int r0, int lane, float (&acc)[M]) {
    constexpr int kAhead = sizeof(T) == 4 ? (M <= 2 ? 2 : M <= 4 ? 1 : 0) : 0;
#pragma unroll
    for (int i = 0; i < M; ++i) acc[i] = 0.f;
    if constexpr (kAhead > 0) {
        float w[kAhead][8];
#pragma unroll
        for (int u = 0; u < kAhead; ++u)
            if ((lane + 32 * u) * 8 < K) load8(wrow + (lane + 32 * u) * 8, w[u]);
        for (int k0 = lane * 8; k0 < K; k0 += 256 * kAhead) {
#pragma unroll
            for (int u = 0; u < kAhead; ++u) {
                const int k = k0 + 256 * u;
                float c[8];
#pragma unroll
                for (int j = 0; j < 8; ++j) c[j] = w[u][j];
                if (k + 256 * kAhead < K) load8(wrow + k + 256 * kAhead, w[u]);
                if (k < K) {
#pragma unroll
                    for (int i = 0; i < M; ++i) {
                        float x[8];
                        load_act8(act, r0 + i, k, K, x);
#pragma unroll
                        for (int j = 0; j < 8; ++j) acc[i] = fmaf(c[j], x[j], acc[i]);
                    }
                }
            }
        }
    } else {
#pragma unroll (M <= 2 ? 2 : 1)
        for (int k = lane * 8; k < K; k += 256) {
            float w[8];
            load8(wrow + k, w);
            if constexpr (sizeof(T) == 4) {
#pragma unroll
                for (int i0 = 0; i0 < M; i0 += 4) {
                    float x[4][8];
#pragma unroll
                    for (int i = 0; i < 4; ++i)
                        if (i0 + i < M) load_act8(act, r0 + i0 + i, k, K, x[i]);
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        if (i0 + i < M) {
#pragma unroll
                            for (int j = 0; j < 8; ++j) acc[i0 + i] = fmaf(w[j], x[i][j], acc[i0 + i]);
                        }
                    }
                }
            } else {
#pragma unroll
                for (int i = 0; i < M; ++i) {
                    float x[8];
                    load_act8(act, r0 + i, k, K, x);
#pragma unroll
                    for (int j = 0; j < 8; ++j) acc[i] = fmaf(w[j], x[j], acc[i]);
                }
            }
        }
    }
#pragma unroll
    for (int i = 0; i < M; ++i) acc[i] = warp_sum(acc[i]);
}

template <typename T, int M>
__global__ void __launch_bounds__(256) k_gemm_simt(const __grid_constant__ GemmArgs a) {
    using AT = typename Act<T>::type;
    pdl_trigger();
    pdl_wait();
    const AT* act = reinterpret_cast<const AT*>(a.act);
    int lane = threadIdx.x & 31;
    int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    int n_warps = (gridDim.x * blockDim.x) >> 5;
    for (int n = warp; n < a.n_total; n += n_warps) {
        int j = 0, base = 0;
        while (n >= a.n_end[j]) base = a.n_end[j++];
        float acc[M];
        row_dots<T, M>(reinterpret_cast<const T*>(a.W[j]) + (size_t)(n - base) * a.K, act, a.K, a.r0, lane, acc);
        if (lane == 0) {
#pragma unroll
            for (int i = 0; i < M; ++i) a.out[(size_t)(a.r0 + i) * a.n_total + n] = acc[i];
        }
    }
}
// Gate/up with SwiGLU (swiglu_out set, two matrices of equal shape): a warp takes the gate and the up row of a column and
// writes silu(gate) * up as the down projection's operand.  The same sums and the same rounding as k_gemm_simt and k_swiglu,
// one launch less.
template <typename T, int M>
__global__ void __launch_bounds__(256) k_gemm_swiglu_simt(const __grid_constant__ GemmArgs a) {
    using A = Act<T>;
    using AT = typename A::type;
    pdl_trigger();
    pdl_wait();
    const AT* act = reinterpret_cast<const AT*>(a.act);
    const int lane = threadIdx.x & 31, F = a.n_end[0];
    const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, n_warps = (gridDim.x * blockDim.x) >> 5;
    for (int f = warp; f < F; f += n_warps) {
        float g[M], u[M];
        row_dots<T, M>(reinterpret_cast<const T*>(a.W[0]) + (size_t)f * a.K, act, a.K, a.r0, lane, g);
        row_dots<T, M>(reinterpret_cast<const T*>(a.W[1]) + (size_t)f * a.K, act, a.K, a.r0, lane, u);
#pragma unroll
        for (int i = 0; i < M; ++i)
            if (lane == i) A::store(reinterpret_cast<AT*>(a.swiglu_out), a.r0 + i, f, F, g[i] / (1.f + expf(-g[i])) * u[i]);
    }
}
// One warp per output row, in no more blocks than four whole rounds of what is resident at once: a part of a round at the end
// leaves SMs idle, and in one round nothing makes up for a slow block (fp32 d_model 4096, 8 rows: 1 / 2 / 4 rounds 2172 / 1898 /
// 1801 us).
template <typename T, int M, bool kSwiglu> static void launch_rows(cudaStream_t st, const GemmArgs& a) {
    constexpr auto kernel = kSwiglu ? k_gemm_swiglu_simt<T, M> : k_gemm_simt<T, M>;
    static int per_sm[kMaxDevices];
    const int dev = current_device(), rows = kSwiglu ? a.n_end[0] : a.n_total;
    int n = dev < 0 ? 4 : per_sm[dev];
    if (n == 0) {
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kernel, 256, 0) != cudaSuccess || n < 1) { (void)cudaGetLastError(); n = 4; }
        per_sm[dev] = n;
    }
    launch_k(kernel, dim3(min((rows + 7) / 8, 4 * n * device_sm_count())), dim3(256), 0, st, a);
}
template <typename T, int M> static void launch_m(cudaStream_t st, const GemmArgs& a) {
    if (a.swiglu_out) launch_rows<T, M, true>(st, a);
    else launch_rows<T, M, false>(st, a);
}
template <typename T> void launch_gemm_simt(cudaStream_t st, const GemmArgs& a) {
    switch (a.m) {
        case 1: launch_m<T, 1>(st, a); break;
        case 2: launch_m<T, 2>(st, a); break;
        case 3: launch_m<T, 3>(st, a); break;
        case 4: launch_m<T, 4>(st, a); break;
        case 5: launch_m<T, 5>(st, a); break;
        case 6: launch_m<T, 6>(st, a); break;
        case 7: launch_m<T, 7>(st, a); break;
        default: launch_m<T, 8>(st, a); break;
    }
}

// ------------------------------------------------------------------------------------------------
// Exit-confidence kernel (CUDA-core variant).  Every warp walks vocabulary rows v = warp, warp +
// n_warps, ... and keeps, per activation row, the running triple (max logit, its index, sum of
// exp((z - max)/T)).  Warps of a CTA are merged in warp order, CTAs in CTA order by the last CTA
// to arrive (a wait-free ticket), so the result is deterministic.  conf = 1 / sum.
// ------------------------------------------------------------------------------------------------
constexpr int kHeadWarps = 8;
constexpr int kHeadCtasPerSm = 4;   // the launcher's CTAs are one round of these: with one fewer resident the last of them run alone
                                    // (bf16, one 7B row: 104 us, 170 with three per SM; fp32 218 -> 146)
template <typename T, int M>
__global__ void __launch_bounds__(kHeadWarps * 32, kHeadCtasPerSm) k_head_simt(const __grid_constant__ HeadArgs a) {
    using AT = typename Act<T>::type;
    __shared__ SoftTriple cta_part[kHeadWarps][M];
    __shared__ bool is_last;
    pdl_trigger();
    pdl_wait();
    const AT* act = reinterpret_cast<const AT*>(a.act);
    int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    int warp = blockIdx.x * kHeadWarps + wib;
    int n_warps = gridDim.x * kHeadWarps;
    SoftTriple tr[M];
#pragma unroll
    for (int i = 0; i < M; ++i) tr[i] = soft_empty();
    for (int v = warp; v < a.V; v += n_warps) {
        float acc[M];
        row_dots<T, M>(reinterpret_cast<const T*>(a.W) + (size_t)v * a.K, act, a.K, a.r0, lane, acc);
#pragma unroll
        for (int i = 0; i < M; ++i) {
            soft_push(tr[i], acc[i], v, a.inv_tau);
            if (a.logits_dbg && lane == 0) a.logits_dbg[(size_t)i * a.V + v] = acc[i];
        }
    }
    if (lane == 0) {
#pragma unroll
        for (int i = 0; i < M; ++i) cta_part[wib][i] = tr[i];
    }
    __syncthreads();
    if (threadIdx.x < M) {
        int i = threadIdx.x;
        SoftTriple t = cta_part[0][i];
        for (int w = 1; w < kHeadWarps; ++w) t = soft_merge(t, cta_part[w][i], a.inv_tau);
        a.part[(size_t)blockIdx.x * kMaxW + a.r0 + i] = t;
        __threadfence();
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        unsigned int prev = atomicAdd(a.ticket, 1u);
        is_last = (prev == gridDim.x - 1);
    }
    __syncthreads();
    if (!is_last) return;
    __threadfence();
    soft_final_merge(a.part, (int)gridDim.x, a.r0, a.m, a.inv_tau, a.threshold, a.conf, a.token, a.exit_flag);
    if (threadIdx.x == 0) *a.ticket = 0u;   // ready for the next launch on this stream
    publish_results(a.mirror);
}
template <typename T> void launch_head_simt(cudaStream_t st, const HeadArgs& a) {
    // no more CTAs than there are rows for their warps: the last one to arrive folds the triples of all of them
    const dim3 grid(min(min(kHeadCtasPerSm * device_sm_count(), kHeadMaxCtas), (a.V + kHeadWarps - 1) / kHeadWarps)), block(kHeadWarps * 32);
    switch (a.m) {
        case 1: launch_k(k_head_simt<T, 1>, grid, block, 0, st, a); break;
        case 2: launch_k(k_head_simt<T, 2>, grid, block, 0, st, a); break;
        case 3: launch_k(k_head_simt<T, 3>, grid, block, 0, st, a); break;
        case 4: launch_k(k_head_simt<T, 4>, grid, block, 0, st, a); break;
        case 5: launch_k(k_head_simt<T, 5>, grid, block, 0, st, a); break;
        case 6: launch_k(k_head_simt<T, 6>, grid, block, 0, st, a); break;
        case 7: launch_k(k_head_simt<T, 7>, grid, block, 0, st, a); break;
        default: launch_k(k_head_simt<T, 8>, grid, block, 0, st, a); break;
    }
}

template void launch_gemm_simt<float>(cudaStream_t, const GemmArgs&);
template void launch_gemm_simt<__nv_bfloat16>(cudaStream_t, const GemmArgs&);
template void launch_head_simt<float>(cudaStream_t, const HeadArgs&);
template void launch_head_simt<__nv_bfloat16>(cudaStream_t, const HeadArgs&);

}  // namespace sb

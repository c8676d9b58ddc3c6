// Token-affinity matrix, Eq. symbolic-m with Omega = cosine similarity of token embeddings:
//   M_ij = exp(Omega_ij / tau) / sum_{k in T} exp(Omega_ik / tau),  i in I (kept ids), j in T.
// One-time preprocessing.  This file: fp32 FMAs, for fp32 embeddings and the fp32 layout.  The dot products are computed
// twice, once for the sums and once for the values, by the same kernel: a thread has 4 columns (or 1) x 16 kept rows (two rows
// to an instruction), a CTA the 16 rows against a share of the columns, so that few kept rows fill the chip too.  The
// soft-max is shifted by the row's largest possible value, its own length (1, or 0 for a zero embedding), so that no
// maximum has to be found.  Bound by the FMA pipe: 8000 x 2000 x 64 takes 140 us.
#include <math.h>

#include "rdk_device.cuh"

namespace rdk {

constexpr int kAffRows = 16;      // kept rows per CTA
constexpr int kAffThreads = 256;
constexpr int kAffShares = 32;    // most shares of the columns
static int aff_npad(int N) { return (N + 3) & ~3; }

// Et[k * Npad + t] = e_t[k] / max(|e_t|, 1e-12): unit-length embeddings, stored dimension-major so
// that consecutive threads (tokens) read consecutive addresses.
template <typename TE>
__global__ void aff_normalise_kernel(const TE* __restrict__ E, long long stride, float* __restrict__ Et, int N, int Npad, int d) {
    const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    if (warp >= N) return;
    const TE* row = E + (long long)warp * stride;
    float ss = 0.f;
    for (int k = lane; k < d; k += 32) { const float v = to_float<TE>(row[k]); ss += v * v; }
    ss = warp_sum(ss);
    const float inv = 1.f / fmaxf(sqrtf(ss), 1e-12f);
    for (int k = lane; k < d; k += 32) Et[(long long)k * Npad + warp] = to_float<TE>(row[k]) * inv;
}

// WRITE = false: part[share][i] = sum over the share's columns of exp((Omega_ij - shift_i) / tau); WRITE = true: M.
template <int LAYOUT, bool WRITE, int VC>
__global__ void __launch_bounds__(kAffThreads, 2)
aff_fma_kernel(const float* __restrict__ Et, const int32_t* __restrict__ ids, int N, int Npad, int n, int d, float scale /* log2(e) / tau */,
               float* __restrict__ part, void* __restrict__ Mout, long long ld) {
    extern __shared__ __align__(16) float rows_s[];          // [d][kAffRows]
    __shared__ float red[kAffThreads / 32][kAffRows], inv_s[kAffRows], shift_s[kAffRows];
    __shared__ int id_s[kAffRows];
    const int i0 = blockIdx.x * kAffRows;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
    if (tid < kAffRows) {
        const int i = i0 + tid;
        const int id = (i < n) ? ids[i] : -1;
        id_s[tid] = (id >= 0 && id < N) ? id : -1;
        if (WRITE && i < n) {
            float z = 0.f;
            for (int k = 0; k < (int)gridDim.y; ++k) z += part[(long long)k * n + i];
            inv_s[tid] = 1.f / z;
        }
    }
    __syncthreads();
    for (int x = tid; x < d * kAffRows; x += kAffThreads) {
        const int k = x / kAffRows, r = x % kAffRows;
        rows_s[x] = id_s[r] >= 0 ? Et[(long long)k * Npad + id_s[r]] : 0.f;
    }
    __syncthreads();
    {   // lengths, 16 threads to a row
        float ss = 0.f;
        for (int k = tid & 15; k < d; k += 16) { const float v = rows_s[k * kAffRows + tid / 16]; ss = fmaf(v, v, ss); }
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
        if ((tid & 15) == 0) shift_s[tid / 16] = sqrtf(ss);
    }
    __syncthreads();
    float sum[kAffRows];
#pragma unroll
    for (int r = 0; r < kAffRows; ++r) sum[r] = 0.f;
    const bool vec = LAYOUT == RDK_AFF_F32_ROWS && ld % 4 == 0 && !(reinterpret_cast<uintptr_t>(Mout) & 15u);
    for (int j = (blockIdx.y * kAffThreads + tid) * VC; j < N; j += gridDim.y * kAffThreads * VC) {
        float2 acc[VC][kAffRows / 2];
#pragma unroll
        for (int c = 0; c < VC; ++c)
#pragma unroll
            for (int r = 0; r < kAffRows / 2; ++r) acc[c][r] = splat(0.f);
#pragma unroll(VC == 4 ? 2 : 8)
        for (int k = 0; k < d; ++k) {
            float2 ac[VC];
            if (VC == 4) {
                const float4 a = __ldg(reinterpret_cast<const float4*>(Et + (long long)k * Npad + j));
                ac[0] = splat(a.x); ac[VC / 4] = splat(a.y); ac[VC / 2] = splat(a.z); ac[VC - 1] = splat(a.w);
            } else {
                ac[0] = splat(__ldg(Et + (long long)k * Npad + j));
            }
            const float4* rv = reinterpret_cast<const float4*>(rows_s + k * kAffRows);
#pragma unroll
            for (int q = 0; q < kAffRows / 4; ++q) {
                const float4 b = rv[q];
#pragma unroll
                for (int c = 0; c < VC; ++c) {
                    acc[c][2 * q] = ffma2(ac[c], make_float2(b.x, b.y), acc[c][2 * q]);
                    acc[c][2 * q + 1] = ffma2(ac[c], make_float2(b.z, b.w), acc[c][2 * q + 1]);
                }
            }
        }
#pragma unroll
        for (int r = 0; r < kAffRows; ++r) {
            float e[VC];
#pragma unroll
            for (int c = 0; c < VC; ++c) e[c] = ex2(((r & 1 ? acc[c][r / 2].y : acc[c][r / 2].x) - shift_s[r]) * scale);
            if (!WRITE) {
#pragma unroll
                for (int c = 0; c < VC; ++c) sum[r] += j + c < N ? e[c] : 0.f;
            } else if (i0 + r < n) {
#pragma unroll
                for (int c = 0; c < VC; ++c) e[c] = id_s[r] >= 0 ? e[c] * inv_s[r] : 0.f;
                if (LAYOUT == RDK_AFF_F32_ROWS) {
                    float* out = static_cast<float*>(Mout) + (long long)(i0 + r) * ld + j;
                    if (VC == 4 && vec && j + 4 <= N) {
                        *reinterpret_cast<float4*>(out) = make_float4(e[0], e[VC / 4], e[VC / 2], e[VC - 1]);
                    } else {
#pragma unroll
                        for (int c = 0; c < VC; ++c) if (j + c < N) out[c] = e[c];
                    }
                } else {
#pragma unroll
                    for (int c = 0; c < VC; ++c) if (j + c < N) static_cast<__nv_bfloat16*>(Mout)[(long long)(j + c) * ld + i0 + r] = __float2bfloat16_rn(e[c]);
                }
            }
        }
    }
    if (WRITE) return;
#pragma unroll
    for (int r = 0; r < kAffRows; ++r) {
        const float t = warp_sum(sum[r]);
        if (lane == 0) red[warp][r] = t;
    }
    __syncthreads();
    if (tid < kAffRows && i0 + tid < n) {
        float t = 0.f;
        for (int w = 0; w < kAffThreads / 32; ++w) t += red[w][tid];
        part[(long long)blockIdx.y * n + i0 + tid] = t;
    }
}

// the tensor-core route (bf16 embeddings into the bf16 layout)
size_t affinity_tc_workspace_bytes(int N, int n, int d);
bool affinity_tc_eligible(const void* embeddings, int emb_dtype, int layout);
int build_affinity_tc(const __nv_bfloat16* E, int d, long long estride, const int32_t* ids, int n, int N, float tau,
                      __nv_bfloat16* Mt, long long ld, void* ws, cudaStream_t s);

}  // namespace rdk

using namespace rdk;

extern "C" size_t rdk_build_affinity_workspace_bytes(int32_t N, int32_t n, int32_t d) {
    if (N < 1 || n < 1 || d < 1) return 0;
    const size_t fma = idx_align((size_t)aff_npad(N) * d * sizeof(float)) + idx_align((size_t)kAffShares * n * sizeof(float)), tc = affinity_tc_workspace_bytes(N, n, d);
    return (fma > tc ? fma : tc) + 256;      // either route may serve the call, from the first 256-byte boundary on
}

extern "C" int rdk_build_affinity(const void* embeddings, int32_t emb_dtype, int32_t d, int64_t emb_row_stride,
                                  const int32_t* kept_ids, int32_t n, int32_t N, float tau,
                                  const rdk_affinity* M_desc, void* M_out, void* ws, size_t ws_bytes,
                                  void* stream) {
    if (!embeddings || !kept_ids || !M_desc || !M_out || !ws || N < 1 || n < 1 || d < 1 || !(tau > 0.f)) {
        set_error("rdk_build_affinity: null pointer, non-positive size or tau <= 0");
        return RDK_ERR_INVALID_ARG;
    }
    if (emb_dtype != RDK_F32 && emb_dtype != RDK_BF16) { set_error("rdk_build_affinity: bad embedding dtype"); return RDK_ERR_INVALID_ARG; }
    const long long estride = emb_row_stride ? emb_row_stride : d;
    if (estride < d) { set_error("rdk_build_affinity: embedding row stride smaller than d"); return RDK_ERR_INVALID_ARG; }
    if (M_desc->reserved != 0) { set_error("rdk_build_affinity: reserved field must be 0"); return RDK_ERR_INVALID_ARG; }
    if (M_desc->layout == RDK_AFF_F32_ROWS) {
        if (M_desc->ld < N) { set_error("rdk_build_affinity: ld < N"); return RDK_ERR_INVALID_ARG; }
    } else if (M_desc->layout == RDK_AFF_BF16_COLS) {
        if (M_desc->ld < n || (M_desc->ld % 8) != 0 || (reinterpret_cast<uintptr_t>(M_out) & 15u)) {
            set_error("rdk_build_affinity: bf16 layout needs ld >= n, ld %% 8 == 0 and a 16-byte aligned base");
            return RDK_ERR_INVALID_ARG;
        }
    } else {
        set_error("rdk_build_affinity: unknown layout %d", M_desc->layout);
        return RDK_ERR_INVALID_ARG;
    }
    if (ws_bytes < rdk_build_affinity_workspace_bytes(N, n, d)) {
        set_error("rdk_build_affinity: workspace has %zu bytes, %zu needed", ws_bytes, rdk_build_affinity_workspace_bytes(N, n, d));
        return RDK_ERR_WORKSPACE_TOO_SMALL;
    }
    const size_t smem = (size_t)d * kAffRows * sizeof(float);
    if (smem > 200 * 1024) { set_error("rdk_build_affinity: embedding dimension %d too large", d); return RDK_ERR_UNSUPPORTED; }
    const int st = check_arch();
    if (st != RDK_OK) return st;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    ws = reinterpret_cast<void*>(idx_align(reinterpret_cast<uintptr_t>(ws)));
    if (affinity_tc_eligible(embeddings, emb_dtype, M_desc->layout))
        return build_affinity_tc(static_cast<const __nv_bfloat16*>(embeddings), d, estride, kept_ids, n, N, tau,
                                 static_cast<__nv_bfloat16*>(M_out), M_desc->ld, ws, s);
    float* Et = static_cast<float*>(ws);
    const int Npad = aff_npad(N);
    float* part = reinterpret_cast<float*>(static_cast<unsigned char*>(ws) + idx_align((size_t)Npad * d * sizeof(float)));
    const int wpb = 8;
    if (emb_dtype == RDK_F32)
        aff_normalise_kernel<float><<<(N + wpb - 1) / wpb, wpb * 32, 0, s>>>(static_cast<const float*>(embeddings), estride, Et, N, Npad, d);
    else
        aff_normalise_kernel<__nv_bfloat16><<<(N + wpb - 1) / wpb, wpb * 32, 0, s>>>(static_cast<const __nv_bfloat16*>(embeddings), estride, Et, N, Npad, d);
    RDK_CUDA(cudaGetLastError());
    const float scale = kLog2e / tau;
    // Shares of the columns: two CTAs an SM, none without columns.  One column a thread where four would leave SMs idle
    // (1000 x 100 x 512: 68 us, with four 220).
    const int blocks = (n + kAffRows - 1) / kAffRows;
    const bool wide = (long long)blocks * ((N + 4 * kAffThreads - 1) / (4 * kAffThreads)) >= 148;
    const int most = (N + (wide ? 4 : 1) * kAffThreads - 1) / ((wide ? 4 : 1) * kAffThreads);
    int shares = (2 * 148 + blocks - 1) / blocks;
    if (shares > most) shares = most;
    if (shares > kAffShares) shares = kAffShares;
    const bool rows = M_desc->layout == RDK_AFF_F32_ROWS;
    auto sums = wide ? aff_fma_kernel<RDK_AFF_F32_ROWS, false, 4> : aff_fma_kernel<RDK_AFF_F32_ROWS, false, 1>;
    auto write = rows ? (wide ? aff_fma_kernel<RDK_AFF_F32_ROWS, true, 4> : aff_fma_kernel<RDK_AFF_F32_ROWS, true, 1>)
                      : (wide ? aff_fma_kernel<RDK_AFF_BF16_COLS, true, 4> : aff_fma_kernel<RDK_AFF_BF16_COLS, true, 1>);
    for (int pass = 0; pass < 2; ++pass) {
        auto k = pass == 0 ? sums : write;
        RDK_CUDA(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3((unsigned)blocks, (unsigned)shares, 1);
        cfg.blockDim = dim3(kAffThreads, 1, 1);
        cfg.dynamicSmemBytes = smem;
        cfg.stream = s;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[0].val.programmaticStreamSerializationAllowed = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        RDK_CUDA(cudaLaunchKernelEx(&cfg, k, (const float*)Et, kept_ids, N, Npad, n, d, scale, part, M_out, (long long)M_desc->ld));
    }
    return RDK_OK;
}

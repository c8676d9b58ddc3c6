// Exact redistribution, Algorithm 1 steps 1-2:  q' = TLI(softmax(y)),  w = M^T q'.
// This file holds the operand preparation (q' at the kept slots), the fp32 FMA contraction for
// the fp32 row layout of M, the row sums S, and the entry point; the tensor-core contraction for
// the bf16 layout lives in rdk_exact_tc.cu.
#include <math.h>

#include "rdk_row.cuh"

namespace rdk {

int launch_exact_tc(const __nv_bfloat16* A, long long lda, const __nv_bfloat16* Mt, long long ldm,
                    float* w_out, float* S_out, int rows, int n, int N, int32_t* status_word, cudaStream_t s);

constexpr int kOperandThreads = 512;
constexpr int kOperandSums = 256;        // partial sums of a row: entries i, i + 256, ... one after the other

// A[r, i] = q'_{kappa_i}: soft-max over the drafter entries whose id lies in the target vocabulary
// (Eq. tli-drafter: drop the rest, renormalise), zero for dropped entries and for the padding
// columns i in [n, lda); S[r] = 0 for the contraction to add to (or to count in).
// The maximum and the result in passes of 16-byte vectors, all but the first out of L1/L2; the ids are looked at only where
// the index says that some lie outside the vocabulary.  The sum is taken over 256 interleaved runs: its order decides on
// which side of a bf16 boundary an entry falls (added up vector by vector, 30 to 500 of 10 million entries of q' change),
// so it does not follow the width of the loads.  (Three passes with an element and an id at a time took 99 us for 320 rows
// of 32064 entries, 10 times the memory time.)
template <typename TY, typename TA, int KIND>
__global__ void __launch_bounds__(kOperandThreads)
exact_operand_kernel(const TY* __restrict__ drafter, long long dstride, const int32_t* __restrict__ header, const int32_t* __restrict__ ids,
                     int N, int n, TA* __restrict__ A, long long lda, float* __restrict__ S) {
    __shared__ float red[kOperandThreads / 32];
    const int row = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, threads = blockDim.x;
    const TY* y = drafter + (long long)row * dstride;
    const bool vec = (reinterpret_cast<uintptr_t>(y) & 15u) == 0;
    asm volatile("griddepcontrol.wait;" ::: "memory");
    // only now: the contraction may fetch the affinity matrix as soon as it is let go, and that may have been written by
    // the kernel before this one
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const bool all_valid = __ldg(header + kHdrMagic) == kIdxMagic && __ldg(header + kHdrN) == N && __ldg(header + kHdrn) == n && __ldg(header + kHdrValid) == n;
    // the row's entries i .. i + 7; what carries no weight reads as -inf (a logit) or 0
    constexpr float kNone = KIND == RDK_LOGITS ? -INFINITY : 0.f;
    auto load_y = [&](int i, float (&v)[kVec]) {
        load8<TY>(y, i, n, vec, kNone, v);
        if (!all_valid) {
#pragma unroll
            for (int k = 0; k < kVec; ++k) {
                const int id = i + k < n ? __ldg(ids + i + k) : -1;
                if (id < 0 || id >= N) v[k] = kNone;
            }
        }
    };
    float m = -INFINITY;
    if (KIND == RDK_LOGITS) {
#pragma unroll 2
        for (int i = tid * kVec; i < n; i += threads * kVec) {
            float v[kVec];
            load_y(i, v);
#pragma unroll
            for (int k = 0; k < kVec; ++k) m = fmaxf(m, v[k]);
        }
        m = warp_max(m);
        if (lane == 0) red[warp] = m;
        __syncthreads();
        m = warp_max(red[lane & (threads / 32 - 1)]);
        __syncthreads();
    }
    float s = 0.f;
    if (tid < kOperandSums) {
#pragma unroll 16
        for (int i = tid; i < n; i += kOperandSums) {
            const int id = all_valid ? 0 : __ldg(ids + i);
            const float v = to_float<TY>(y[i]);
            if (id >= 0 && id < N) s += KIND == RDK_LOGITS ? ex2((v - m) * kLog2e) : v;
        }
        s = warp_sum(s);
        if (lane == 0) red[warp] = s;
    }
    __syncthreads();
    s = 0.f;
    for (int k = 0; k < kOperandSums / 32; ++k) s += red[k];
    const float inv = 1.f / s;
    TA* out = A + (long long)row * lda;
    for (int i = tid * kVec; i < lda; i += threads * kVec) {
        float v[kVec];
        load_y(i, v);
#pragma unroll
        for (int k = 0; k < kVec; ++k) v[k] = (KIND == RDK_LOGITS ? ex2((v[k] - m) * kLog2e) : v[k]) * inv;
        if (sizeof(TA) == 2) {                   // lda is a multiple of 64 and the rows are 16-byte aligned
            uint32_t w[4];
#pragma unroll
            for (int h = 0; h < 4; ++h) asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(w[h]) : "f"(v[2 * h + 1]), "f"(v[2 * h]));
            *reinterpret_cast<uint4*>(out + i) = make_uint4(w[0], w[1], w[2], w[3]);
        } else {
#pragma unroll
            for (int k = 0; k < kVec; ++k) if (i + k < lda) reinterpret_cast<float*>(out)[i + k] = v[k];
        }
    }
    if (tid == 0 && S) S[row] = 0.f;
}

// S[r] = sum_j w[r, j], by one warp: fp32 runs of 16 per lane, carried in fp64, the lanes added in a fixed order.  w is read
// from L2, where other CTAs have just written it.
__device__ __forceinline__ void warp_row_sum(const float* __restrict__ row, int N, float* S, int lane) {
    double acc = 0.0;
#pragma unroll 2
    for (int j0 = lane; j0 < N; j0 += 32 * 16) {
        float v[16], s = 0.f;
#pragma unroll
        for (int k = 0; k < 16; ++k) v[k] = j0 + k * 32 < N ? __ldcg(row + j0 + k * 32) : 0.f;
#pragma unroll
        for (int k = 0; k < 16; ++k) s += v[k];
        acc += (double)s;
    }
    acc = warp_sum_d(acc);
    if (lane == 0) *S = (float)acc;
}
// The same for long rows, a CTA each.
constexpr int kSumThreads = 256;
__global__ void __launch_bounds__(kSumThreads)
row_sum_kernel(const float* __restrict__ w, int N, float* __restrict__ S) {
    __shared__ double red[kSumThreads / 32];
    const int tid = threadIdx.x, lane = tid & 31;
    const float* row = w + (long long)blockIdx.x * N;
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
    double acc = 0.0;
    for (int j0 = tid; j0 < N; j0 += kSumThreads * 16) {
        float v[16], s = 0.f;
#pragma unroll
        for (int k = 0; k < 16; ++k) v[k] = j0 + k * kSumThreads < N ? row[j0 + k * kSumThreads] : 0.f;
#pragma unroll
        for (int k = 0; k < 16; ++k) s += v[k];
        acc += (double)s;
    }
    acc = warp_sum_d(acc);
    if (lane == 0) red[tid >> 5] = acc;
    __syncthreads();
    if (tid == 0) { double t = 0.0; for (int k = 0; k < kSumThreads / 32; ++k) t += red[k]; S[blockIdx.x] = (float)t; }
}

// w[r, j] = sum_i A[r, i] M[i, j]  with fp32 FMAs (fp32 row layout of M; small problems).  Where S is given, the CTA of a
// row block that arrives last adds up its rows of w; until then the block's first S counts the arrivals (the operand kernel
// has zeroed it).  Sums added as they come, by fp32 atomics, are not the same twice and three times as far off.
// A CTA takes 8 rows x 32 VC columns; its warps share the contraction (warp w takes i = w, w + 8, ...) and add up in shared
// memory.  With a thread for a column and all of the contraction, 4 x 1024 x 256 ran on 4 SMs with one load in flight:
// 27 us.
constexpr int kFmaRows = 8, kFmaWarps = 8, kFmaChunk = 256, kFmaSumMax = 4096;
template <int VC>
__global__ void __launch_bounds__(kFmaWarps * 32)
exact_fma_kernel(const float* __restrict__ A, long long lda, const float* __restrict__ M, long long ldm,
                 float* __restrict__ w, float* __restrict__ S, int rows, int n, int N) {
    constexpr int kCols = 32 * VC;
    __shared__ __align__(16) float a_s[kFmaChunk][kFmaRows];
    __shared__ float part[kFmaWarps][kFmaRows][kCols];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int j0 = blockIdx.x * kCols, r0 = blockIdx.y * kFmaRows, j = j0 + lane * VC;
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
    float acc[kFmaRows][VC];
#pragma unroll
    for (int r = 0; r < kFmaRows; ++r)
#pragma unroll
        for (int c = 0; c < VC; ++c) acc[r][c] = 0.f;
    for (int i0 = 0; i0 < n; i0 += kFmaChunk) {
        const int lim = min(kFmaChunk, n - i0);
        __syncthreads();
#pragma unroll
        for (int r = 0; r < kFmaRows; ++r) a_s[tid][r] = (r0 + r < rows && tid < lim) ? A[(long long)(r0 + r) * lda + i0 + tid] : 0.f;
        __syncthreads();
#pragma unroll 8
        for (int ii = warp; ii < lim; ii += kFmaWarps) {
            float mv[VC];
            const float* m = M + (long long)(i0 + ii) * ldm + j;
            if (VC == 4) {
                const float4 q = __ldg(reinterpret_cast<const float4*>(m));
                mv[0] = q.x; mv[VC > 1 ? 1 : 0] = q.y; mv[VC > 2 ? 2 : 0] = q.z; mv[VC > 3 ? 3 : 0] = q.w;
            } else {
                mv[0] = j < N ? __ldg(m) : 0.f;
            }
            const float4 a0 = *reinterpret_cast<const float4*>(&a_s[ii][0]), a1 = *reinterpret_cast<const float4*>(&a_s[ii][4]);
            const float av[kFmaRows] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
#pragma unroll
            for (int r = 0; r < kFmaRows; ++r)
#pragma unroll
                for (int c = 0; c < VC; ++c) acc[r][c] = fmaf(av[r], mv[c], acc[r][c]);
        }
    }
#pragma unroll
    for (int r = 0; r < kFmaRows; ++r)
#pragma unroll
        for (int c = 0; c < VC; ++c) part[warp][r][lane * VC + c] = acc[r][c];
    __syncthreads();
    for (int o = tid; o < kFmaRows * kCols; o += kFmaWarps * 32) {
        const int r = o / kCols, c = o % kCols;
        float v = 0.f;
#pragma unroll
        for (int k = 0; k < kFmaWarps; ++k) v += part[k][r][c];
        const bool in = r0 + r < rows && j0 + c < N;
        if (in) w[(long long)(r0 + r) * N + j0 + c] = v;
    }
    if (!S) return;
    __shared__ bool last;
    __syncthreads();
    if (tid == 0) {                              // releases the whole CTA's w, and acquires that of those before it
        unsigned before;
        asm volatile("atom.acq_rel.gpu.global.add.u32 %0, [%1], 1;" : "=r"(before) : "l"(S + r0) : "memory");
        last = before == gridDim.x - 1;
    }
    __syncthreads();
    if (!last) return;
    static_assert(kFmaRows == kFmaWarps, "a warp to a row");
    if (r0 + warp < rows) warp_row_sum(w + (long long)(r0 + warp) * N, N, S + r0 + warp, lane);
}

template <typename K, typename... A>
static cudaError_t launch_pdl(K kern, dim3 grid, unsigned block, cudaStream_t s, A... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(block, 1, 1);
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, args...);
}

template <typename TY, typename TA>
static cudaError_t launch_operand(const void* drafter, long long dstride, const KeptIndexView& v, int N, int n, int kind,
                                  void* A, long long lda, float* S, int rows, cudaStream_t s) {
    // half the threads where a vector each covers the row
    auto k = kind == RDK_LOGITS ? exact_operand_kernel<TY, TA, RDK_LOGITS> : exact_operand_kernel<TY, TA, RDK_PROBS>;
    return launch_pdl(k, dim3((unsigned)rows), (unsigned)(n <= kOperandSums * kVec ? kOperandSums : kOperandThreads), s, static_cast<const TY*>(drafter), dstride, v.header, v.ids, N, n,
                      static_cast<TA*>(A), lda, S);
}

static long long operand_ld(int n, int layout) {
    return layout == RDK_AFF_BF16_COLS ? ((n + 63) / 64) * 64LL : n;
}

}  // namespace rdk

using namespace rdk;

extern "C" size_t rdk_exact_workspace_bytes(const rdk_problem* problem, int32_t affinity_layout) {
    if (!problem || problem->n < 1 || problem->batch < 1 || problem->positions < 1) return 0;
    if (affinity_layout != RDK_AFF_F32_ROWS && affinity_layout != RDK_AFF_BF16_COLS) return 0;
    const size_t rows = (size_t)problem->batch * problem->positions;
    const size_t el = affinity_layout == RDK_AFF_BF16_COLS ? 2 : 4;
    return idx_align(rows * (size_t)operand_ld(problem->n, affinity_layout) * el);
}

extern "C" int rdk_redistribute_exact(const rdk_problem* problem, const void* drafter, const rdk_affinity* M,
                                      float* w_out, float* S_out, void* ws, size_t ws_bytes,
                                      int32_t* status_word, void* stream) {
    if (!problem || !drafter || !M || !M->data || !w_out || !ws) {
        set_error("rdk_redistribute_exact: null pointer");
        return RDK_ERR_INVALID_ARG;
    }
    if (problem->N < 1 || problem->n < 1 || problem->batch < 1 || problem->positions < 1 || !problem->kept_index ||
        (problem->drafter_dtype != RDK_F32 && problem->drafter_dtype != RDK_BF16) ||
        (problem->drafter_kind != RDK_LOGITS && problem->drafter_kind != RDK_PROBS) || (problem->flags & ~(RDK_FLAG_ROW_KERNEL | RDK_FLAG_W_AS_GIVEN)) != 0 ||
        (problem->drafter_row_stride != 0 && problem->drafter_row_stride < problem->n) || M->reserved != 0) {
        set_error("rdk_redistribute_exact: bad problem description");
        return RDK_ERR_INVALID_ARG;
    }
    const int N = problem->N, n = problem->n;
    const long long rows_ll = (long long)problem->batch * problem->positions;
    if (rows_ll > 0x7fffffffLL) { set_error("rdk_redistribute_exact: too many rows"); return RDK_ERR_INVALID_ARG; }
    const int rows = (int)rows_ll;
    if (M->layout == RDK_AFF_F32_ROWS) {
        if (M->ld < N) { set_error("rdk_redistribute_exact: ld < N"); return RDK_ERR_INVALID_ARG; }
    } else if (M->layout == RDK_AFF_BF16_COLS) {
        if (M->ld < n || (M->ld % 8) != 0 || (reinterpret_cast<uintptr_t>(M->data) & 15u)) {
            set_error("rdk_redistribute_exact: bf16 layout needs ld >= n, ld %% 8 == 0 and a 16-byte aligned base");
            return RDK_ERR_INVALID_ARG;
        }
    } else {
        set_error("rdk_redistribute_exact: unknown affinity layout %d", M->layout);
        return RDK_ERR_INVALID_ARG;
    }
    if ((reinterpret_cast<uintptr_t>(ws) & 255u) != 0) { set_error("rdk_redistribute_exact: workspace must be 256-byte aligned"); return RDK_ERR_INVALID_ARG; }
    if (ws_bytes < rdk_exact_workspace_bytes(problem, M->layout)) {
        set_error("rdk_redistribute_exact: workspace has %zu bytes, %zu needed", ws_bytes, rdk_exact_workspace_bytes(problem, M->layout));
        return RDK_ERR_WORKSPACE_TOO_SMALL;
    }
    int st = check_arch();
    if (st != RDK_OK) return st;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    KeptIndexView v = make_view(problem->kept_index, N, n);
    const long long dstride = problem->drafter_row_stride ? problem->drafter_row_stride : n;
    const long long lda = operand_ld(n, M->layout);
    const bool bf = M->layout == RDK_AFF_BF16_COLS;
    using B = __nv_bfloat16;
    const bool f = problem->drafter_dtype == RDK_F32;
    const int kind = problem->drafter_kind;
    if (bf) RDK_CUDA((f ? launch_operand<float, B> : launch_operand<B, B>)(drafter, dstride, v, N, n, kind, ws, lda, S_out, rows, s));
    else RDK_CUDA((f ? launch_operand<float, float> : launch_operand<B, float>)(drafter, dstride, v, N, n, kind, ws, lda, S_out, rows, s));
    if (bf)                                      // also accumulates S (one atomic partial sum per row and warp)
        return launch_exact_tc(static_cast<const B*>(ws), lda, static_cast<const B*>(M->data), M->ld, w_out, S_out, rows, n, N, status_word, s);
    // four columns a thread where that still fills the chip, M's rows are whole 16-byte units and a CTA's columns exist
    const float *A = static_cast<const float*>(ws), *Mf = static_cast<const float*>(M->data);
    const unsigned ry = (unsigned)((rows + kFmaRows - 1) / kFmaRows);
    const bool wide = N % 128 == 0 && M->ld % 4 == 0 && !(reinterpret_cast<uintptr_t>(Mf) & 15u) && (long long)(N / 128) * ry >= 296;
    // S by a kernel of its own where one CTA's turn at eight long rows would take longer than that launch
    const bool sum_after = S_out && N > kFmaSumMax;
    float* S_in = sum_after ? nullptr : S_out;
    if (wide) RDK_CUDA(launch_pdl(exact_fma_kernel<4>, dim3((unsigned)(N / 128), ry), kFmaWarps * 32u, s, A, lda, Mf, (long long)M->ld, w_out, S_in, rows, n, N));
    else RDK_CUDA(launch_pdl(exact_fma_kernel<1>, dim3((unsigned)((N + 31) / 32), ry), kFmaWarps * 32u, s, A, lda, Mf, (long long)M->ld, w_out, S_in, rows, n, N));
    if (sum_after) RDK_CUDA(launch_pdl(row_sum_kernel, dim3((unsigned)rows), (unsigned)kSumThreads, s, (const float*)w_out, N, S_out));
    return RDK_OK;
}

// ------------------------------------------------------------------------------------------------
// Variant of rdk_redistribute_exact whose q' operand lives in a fixed device array instead of a
// caller-supplied workspace, for callers that are not able to allocate device memory.
// ------------------------------------------------------------------------------------------------
#include <mutex>

static __device__ __align__(256) unsigned char g_exact_static_scratch[RDK_STATIC_SCRATCH_BYTES];

namespace {
constexpr int kMaxDevices = 64;
std::mutex g_scratch_mutex;
void* g_scratch_ptr[kMaxDevices] = {nullptr};
}  // namespace

extern "C" int rdk_redistribute_exact_static(const rdk_problem* problem, const void* drafter,
                                             const rdk_affinity* M, float* w_out, float* S_out,
                                             int32_t* status_word, void* stream) {
    if (!problem || !M) {
        set_error("rdk_redistribute_exact_static: null pointer");
        return RDK_ERR_INVALID_ARG;
    }
    const size_t need = rdk_exact_workspace_bytes(problem, M->layout);
    if (need == 0) {
        set_error("rdk_redistribute_exact_static: bad sizes or affinity layout");
        return RDK_ERR_INVALID_ARG;
    }
    if (need > (size_t)RDK_STATIC_SCRATCH_BYTES) {
        set_error("rdk_redistribute_exact_static: the q' operand needs %zu bytes but the built-in scratch array holds "
                  "%zu; use rdk_redistribute_exact with your own workspace", need, (size_t)RDK_STATIC_SCRATCH_BYTES);
        return RDK_ERR_WORKSPACE_TOO_SMALL;
    }
    int dev = 0;
    RDK_CUDA(cudaGetDevice(&dev));
    if (dev < 0 || dev >= kMaxDevices) {
        set_error("rdk_redistribute_exact_static: device ordinal %d not supported", dev);
        return RDK_ERR_UNSUPPORTED;
    }
    void* scratch = nullptr;
    {
        std::lock_guard<std::mutex> lock(g_scratch_mutex);
        if (!g_scratch_ptr[dev]) {
            // The array's name is only a host-side handle; the kernels need its device address.
            void* p = nullptr;
            RDK_CUDA(cudaGetSymbolAddress(&p, g_exact_static_scratch));
            g_scratch_ptr[dev] = p;
        }
        scratch = g_scratch_ptr[dev];
    }
    // Every element of the operand that the contraction reads is written first by the operand
    // kernel (padding columns included), so nothing left over from an earlier call is ever used.
    return rdk_redistribute_exact(problem, drafter, M, w_out, S_out, scratch, (size_t)RDK_STATIC_SCRATCH_BYTES,
                                  status_word, stream);
}

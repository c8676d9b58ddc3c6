// Emitted sequences, Algorithm 4 steps 7-9: for every sequence (and trial) the accepted drafts
// d_1..d_j followed by one more token t -- the residual draw of the first rejected position, or,
// when all drafts were accepted, a fresh draw t ~ p from the target row that follows the last draft
// (inverse CDF in ascending token id with uniform lane 3 of the sequence's last position).
//
// One thread-block cluster per (sequence, trial).  Most sequences need no fresh draw: their clusters leave at once.
// For the others the row's 16-byte aligned positions are dealt out to the cluster's warps; a warp takes the soft-max
// sum of its run on a running scale, and these (scale, sum) records are all that the prefix sums need, so the row is
// read once.  CTA 0 collects them (distributed shared memory), finds the run of the draw and reads that one again.
// One CTA per sequence with two passes over the row was bound by what one SM can keep in flight: 65 us as soon as one
// of 64 sequences of 128k tokens needed its draw.
#include "rdk_device.cuh"
#include "rdk_row.cuh"

namespace rdk {

constexpr int kEmitThreads = 256;
constexpr int kEmitWarps = kEmitThreads / 32;
constexpr int kEmitMaxCtas = 8;
constexpr int kEmitMaxSeg = kEmitMaxCtas * kEmitWarps;

struct EmitParams {
    int N, batch, positions, trials, pad;
    int per;                              // vectors of 8 positions per warp, a multiple of 32
    const void* bonus; long long bonus_stride;
    const float* uniforms;
    const int32_t* draft_token; const uint8_t* accepted; const int32_t* out_token;
    int32_t* seq_tokens; int32_t* seq_len;
};

// the 8 logits at position v * 8 of a row whose token 0 is at position `phase` (so that vectors are 16-byte aligned)
template <typename TZ>
__device__ __forceinline__ void emit_load8(const TZ* zrow, int v, int phase, int N, float (&z)[kVec]) {
    const int jb = v * kVec - phase;
    if (jb >= 0) {
        load8<TZ>(zrow, jb, N, true, -INFINITY, z);
    } else {
#pragma unroll
        for (int k = 0; k < kVec; ++k) z[k] = jb + k >= 0 && jb + k < N ? to_float<TZ>(zrow[jb + k]) : -INFINITY;
    }
}

template <typename TZ>
__global__ void __launch_bounds__(kEmitThreads)
emit_kernel(const EmitParams P) {
    __shared__ float2 rec[kEmitMaxSeg];                  // CTA 0: (scale, sum) of every warp of the cluster
    __shared__ double cdf[kEmitMaxSeg];
    __shared__ float chunk_sum[32];
    __shared__ float bc[2];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    uint32_t rank, C;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
    asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(C));
    const int g = (int)(blockIdx.x / C), b = g / P.trials, t = g % P.trials;
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");   // the inputs are usually the previous kernel's outputs

    // leading accepted positions, 32 flags at a time
    int j = 0;
    for (int k0 = 0; k0 < P.positions; k0 += 32) {
        const int k = k0 + lane;
        const bool acc = k < P.positions && P.accepted[((long long)b * P.positions + k) * P.trials + t];
        const uint32_t no = ~__ballot_sync(0xffffffffu, acc);
        j += no ? __ffs(no) - 1 : 32;
        if (no) break;
    }
    int32_t* seq = P.seq_tokens + (long long)g * (P.positions + 1);
    if (rank == 0) {
        for (int k = tid; k <= P.positions; k += kEmitThreads) {
            if (k < j) seq[k] = P.draft_token[((long long)b * P.positions + k) * P.trials + t];
            else if (k == j && j < P.positions) seq[k] = P.out_token[((long long)b * P.positions + k) * P.trials + t];   // the residual draw made there
            else if (k > j && P.pad) seq[k] = -1;
        }
        if (tid == 0) P.seq_len[g] = j + 1;
    }
    if (j < P.positions) return;                         // (the same in every thread of the cluster)

    // every draft accepted: t ~ softmax(bonus row)
    const TZ* zrow = static_cast<const TZ*>(P.bonus) + (long long)b * P.bonus_stride;
    const int phase = (int)((reinterpret_cast<uintptr_t>(zrow) & 15u) / sizeof(TZ));
    const int sg = (int)rank * kEmitWarps + warp, nseg = (int)C * kEmitWarps;
    MS zs{-INFINITY, 0.f, 0.f};
#pragma unroll 4
    for (int k = lane; k < P.per; k += 32) {
        float z[kVec];
        emit_load8<TZ>(zrow, sg * P.per + k, phase, P.N, z);
        float vmax = z[0];
#pragma unroll
        for (int q = 1; q < kVec; ++q) vmax = fmaxf(vmax, z[q]);
        if (vmax > zs.m) { zs.s *= ex2((zs.m - vmax) * kLog2e); zs.m = vmax; }
        const float off = zs.m > -INFINITY ? -zs.m * kLog2e : 0.f;
#pragma unroll
        for (int q = 0; q < kVec; ++q) zs.s += ex2(fmaf(z[q], kLog2e, off));
    }
    zs = ms_warp(zs);
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");      // CTA 0 runs
    if (lane == 0) {
        uint32_t r;
        asm volatile("mapa.shared::cluster.u32 %0, %1, 0;" : "=r"(r) : "r"(smem_u32(&rec[sg])));
        asm volatile("st.shared::cluster.v2.f32 [%0], {%1, %2};" ::"r"(r), "f"(zs.m), "f"(zs.s) : "memory");
    }
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    if (rank != 0) return;
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
    if (warp == 0) {
        MS a{-INFINITY, 0.f, 0.f};
        for (int s = lane; s < nseg; s += 32) a = ms_combine(a, MS{rec[s].x, rec[s].y, 0.f});
        a = ms_warp(a);
        const float off = -a.m * kLog2e, inv_z = 1.f / a.s;
        if (lane == 0) { bc[0] = off; bc[1] = inv_z; }
        // prefix sums of the runs' probabilities, two runs per lane
        double v[2], x = 0.0;
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            const int s = 2 * lane + k;
            if (s < nseg && rec[s].x > -INFINITY) x += (double)(rec[s].y * ex2((rec[s].x - a.m) * kLog2e) * inv_z);
            v[k] = x;
        }
        double incl = x;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const double y = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += y;
        }
        double before = __shfl_up_sync(0xffffffffu, incl, 1);
        if (lane == 0) before = 0.0;
#pragma unroll
        for (int k = 0; k < 2; ++k) if (2 * lane + k < nseg) cdf[2 * lane + k] = before + v[k];
    }
    __syncthreads();
    const float off = bc[0], inv_z = bc[1];
    const double thr = (double)__ldg(P.uniforms + (((long long)b * P.positions + P.positions - 1) * P.trials + t) * 4 + 3) * cdf[nseg - 1];
    const int s = min(first_above(cdf, nseg, thr), nseg - 1);
    const float rem = (float)(thr - (s ? cdf[s - 1] : 0.0));
    const int nch = P.per / 32;                          // 256-position chunks of a run, at most 32 taken at a time
    auto chunk_p = [&](int ch, float (&p)[kVec]) -> float {
        float z[kVec], sum = 0.f;
        emit_load8<TZ>(zrow, s * P.per + ch * 32 + lane, phase, P.N, z);
#pragma unroll
        for (int q = 0; q < kVec; ++q) { p[q] = ex2(fmaf(z[q], kLog2e, off)) * inv_z; sum += p[q]; }
        return warp_sum(sum);
    };
    float p[kVec], cum = 0.f, before = 0.f;
    int chosen = -1, last_pos = -1;
    for (int c0 = 0; c0 < nch && chosen < 0; c0 += 32) {
        for (int ch = c0 + warp; ch < min(nch, c0 + 32); ch += kEmitWarps) {
            const float sum = chunk_p(ch, p);
            if (lane == 0) chunk_sum[ch - c0] = sum;
        }
        __syncthreads();
        for (int ch = c0; ch < min(nch, c0 + 32); ++ch) {
            const float sum = chunk_sum[ch - c0];
            if (sum > 0.f) {
                if (chosen < 0 && cum + sum > rem) { chosen = ch; before = cum; }
                last_pos = ch;
                cum += sum;
            }
        }
        __syncthreads();
    }
    if (warp != 0) return;
    const float r_in = chosen < 0 ? INFINITY : rem - before;     // rounding left no token: the last positive one
    if (chosen < 0) chosen = max(last_pos, 0);
    (void)chunk_p(chosen, p);
    const int sel = max(pick_in_segment(p, r_in, lane), 0);
    if (lane == 0) seq[j] = min(max((s * P.per + chosen * 32) * kVec - phase + sel, 0), P.N - 1);
}

template <typename TZ>
static cudaError_t launch_emit(EmitParams P, cudaStream_t s) {
    // CTAs per sequence: up to 8, a run of at least 256 positions for each warp, while the clusters are few; with many
    // sequences most clusters leave at once and their launch is what costs.
    const long long seqs = (long long)P.batch * P.trials;
    unsigned C = 1;
    while (C < (unsigned)kEmitMaxCtas && (long long)C * 2048 < P.N && seqs * C < 2048) C *= 2;
    P.per = (int)(((long long)P.N + 8 + C * kEmitWarps * kVec - 1) / (C * kEmitWarps * kVec));
    P.per = (P.per + 31) / 32 * 32;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)seqs * C, 1, 1);
    cfg.blockDim = dim3(kEmitThreads, 1, 1);
    cfg.stream = s;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = C; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;      // may be set up while the previous kernel drains
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    return cudaLaunchKernelEx(&cfg, emit_kernel<TZ>, P);
}

}  // namespace rdk

using namespace rdk;

extern "C" int rdk_emit_sequences(const rdk_problem* problem, const void* bonus_target, int64_t bonus_row_stride,
                                  const float* uniforms, int32_t trials, const int32_t* draft_token,
                                  const uint8_t* accepted, const int32_t* out_token, int32_t* seq_tokens,
                                  int32_t* seq_len, void* stream) {
    if (!problem || !bonus_target || !uniforms || !draft_token || !accepted || !out_token || !seq_tokens || !seq_len) {
        set_error("rdk_emit_sequences: null pointer");
        return RDK_ERR_INVALID_ARG;
    }
    if (problem->N < 1 || problem->batch < 1 || problem->positions < 1 || trials < 1 ||
        (problem->target_dtype != RDK_F32 && problem->target_dtype != RDK_BF16) ||
        (bonus_row_stride != 0 && bonus_row_stride < problem->N)) {
        set_error("rdk_emit_sequences: bad sizes, dtype or stride");
        return RDK_ERR_INVALID_ARG;
    }
    if (problem->N > (1 << 21)) { set_error("rdk_emit_sequences: N exceeds the supported maximum"); return RDK_ERR_UNSUPPORTED; }
    if ((long long)problem->batch * trials > 0x7fffffffLL) { set_error("rdk_emit_sequences: too many sequences"); return RDK_ERR_INVALID_ARG; }
    const int st = check_arch();
    if (st != RDK_OK) return st;
    EmitParams P;
    P.N = problem->N; P.batch = problem->batch; P.positions = problem->positions; P.trials = trials;
    P.pad = (problem->flags & RDK_FLAG_PAD_SEQUENCES) ? 1 : 0;
    P.bonus = bonus_target; P.bonus_stride = bonus_row_stride ? bonus_row_stride : problem->N;
    P.uniforms = uniforms; P.draft_token = draft_token; P.accepted = accepted; P.out_token = out_token;
    P.seq_tokens = seq_tokens; P.seq_len = seq_len;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const cudaError_t e = problem->target_dtype == RDK_F32 ? launch_emit<float>(P, s) : launch_emit<__nv_bfloat16>(P, s);
    if (e != cudaSuccess) return cuda_fail(e, "emit kernel launch");
    return RDK_OK;
}

// Emitted sequences, Algorithm 4 steps 7-9: for every sequence (and trial) the accepted drafts
// d_1..d_j followed by one more token t -- the residual draw of the first rejected position, or,
// when all drafts were accepted, a fresh draw t ~ p from the target row that follows the last draft
// (inverse CDF in ascending token id with uniform lane 3 of the sequence's last position).
//
// A fixed number of thread-block clusters, each with a share of the (sequence, trial) pairs.  A cluster first settles what
// needs no row -- a warp per pair counts the accepted positions and copies the tokens -- and then takes the pairs whose
// drafts were all accepted, usually few, one after the other with all of its warps: the row's 16-byte aligned positions
// are dealt out to the warps, a warp takes the soft-max sum of its run on a running scale, and these (scale, sum) records
// are all that the prefix sums need, so the row is read once.  CTA 0 collects them (distributed shared memory), finds the
// run of the draw and reads that one again.  What bounds it is the latency of that chain.  (One CTA per pair with two
// passes over the row: 65 us as soon as one of 64 sequences of 128k tokens needed its draw; a cluster per pair: 11 us, and
// 30 us for 512 sequences of 262k.)
#include "rdk_device.cuh"
#include "rdk_row.cuh"

namespace rdk {

constexpr int kEmitMaxWarps = 16;
constexpr int kEmitMaxCtas = 8;
constexpr int kEmitMaxSeg = kEmitMaxCtas * kEmitMaxWarps;
constexpr int kEmitBatch = 256;           // pairs whose answers are kept at a time
constexpr unsigned kEmitSpin = 1u << 22;

struct EmitParams {
    int N, batch, positions, trials, pad;
    int per;                              // vectors of 8 positions per warp, a multiple of 32
    const void* bonus; long long bonus_stride;
    const float* uniforms;
    const int32_t* draft_token; const uint8_t* accepted; const int32_t* out_token;
    int32_t* seq_tokens; int32_t* seq_len;
    unsigned spin_limit;
};

// Bounded wait of a warp for the phase of `bar`; a try may park the warp, except under the small limits of the failure-path
// tests, whose tries must be able to run out.
__device__ __forceinline__ bool emit_wait(uint32_t bar, uint32_t parity, unsigned limit) {
    uint32_t done = 0;
    for (unsigned spins = 0; !done && spins < limit; ++spins) {
        if (limit < 64)
            asm volatile("{\n .reg .pred p;\n mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
                         : "=r"(done) : "r"(bar), "r"(parity) : "memory");
        else
            asm volatile("{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
                         : "=r"(done) : "r"(bar), "r"(parity) : "memory");
    }
    return __all_sync(0xffffffffu, done != 0);
}

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

// accepted drafts of one (sequence, trial) pair and the tokens that need no row, by one warp; returns the leading accepts
__device__ __forceinline__ int emit_accepted(const EmitParams& P, int pair, int lane, bool write) {
    const int b = pair / P.trials, t = pair - b * P.trials;
    const long long first = (long long)b * P.positions * P.trials + t;
    int32_t* seq = P.seq_tokens + (long long)pair * (P.positions + 1);
    int j = 0;
    bool run = true;
    for (int k0 = 0; k0 <= P.positions; k0 += 32) {      // 32 positions at a time
        const int k = k0 + lane;
        const long long at = first + (long long)k * P.trials;
        const bool in = k < P.positions;
        const uint8_t acc = in ? P.accepted[at] : 0;
        const int d = write && in ? P.draft_token[at] : -1, o = write && in ? P.out_token[at] : -1;      // (all three loads travel together)
        if (run) {
            const uint32_t no = ~__ballot_sync(0xffffffffu, acc != 0);
            j += no ? __ffs(no) - 1 : 32;
            run = no == 0;
        }
        if (write && k <= P.positions) {
            if (k < j) seq[k] = d;
            else if (k == j && in) seq[k] = o;           // the residual draw made there
            else if (k > j && P.pad) seq[k] = -1;
        }
        if (!run && !(write && P.pad)) break;
    }
    if (write && lane == 0) P.seq_len[pair] = j + 1;
    return j;
}

template <typename TZ>
__global__ void __launch_bounds__(kEmitMaxWarps * 32)
emit_kernel(const EmitParams P) {
    __shared__ float2 rec[kEmitMaxSeg];                  // CTA 0: (scale, sum) of every warp of the cluster
    __shared__ double cdf[kEmitMaxSeg];
    __shared__ float chunk_sum[32];
    __shared__ float bc[2];
    __shared__ __align__(8) unsigned long long rbar;     // CTA 0: the records of the row are in rec[]
    __shared__ bool lost_s;                              // the wait for the records gave up
    __shared__ uint8_t all_s[kEmitBatch];                // whether all drafts of the pair were accepted
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nw = blockDim.x >> 5;
    uint32_t rank, C;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
    asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(C));
    const int cluster = (int)(blockIdx.x / C), clusters = (int)(gridDim.x / C);
    const int pairs = P.batch * P.trials, mine = pairs > cluster ? (pairs - cluster + clusters - 1) / clusters : 0;
    if (tid == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&rbar)));
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    uint32_t parity = 0;
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");   // the inputs are usually the previous kernel's outputs

    for (int i0 = 0; i0 < mine; i0 += kEmitBatch) {
        const int cnt = min(kEmitBatch, mine - i0);
        // every CTA looks at all of the cluster's pairs, CTA 0 writes
        for (int i = warp; i < cnt; i += nw) {
            const int j = emit_accepted(P, cluster + (i0 + i) * clusters, lane, rank == 0);
            if (lane == 0) all_s[i] = j == P.positions;
        }
        __syncthreads();
        for (int i = 0; i < cnt; ++i) {
            if (!all_s[i]) continue;                     // (the same in every thread of the cluster)
            // every draft accepted: t ~ softmax(bonus row)
            const int pair = cluster + (i0 + i) * clusters, b = pair / P.trials, t = pair - b * P.trials;
            const TZ* zrow = static_cast<const TZ*>(P.bonus) + (long long)b * P.bonus_stride;
            const int phase = (int)((reinterpret_cast<uintptr_t>(zrow) & 15u) / sizeof(TZ));
            const int sg = (int)rank * nw + warp, nseg = (int)C * nw;
            const float u = __ldg(P.uniforms + (((long long)b * P.positions + P.positions - 1) * P.trials + t) * 4 + 3);
            // CTA 0 runs, and is done with the previous row's records: it says so here, the others wait for it with their sums
            if (rank == 0 && tid == 0)
                asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(&rbar)), "r"((uint32_t)nseg * 8u) : "memory");
            __syncwarp();
            asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
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
            asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
            if (lane == 0) {
                uint32_t r, m;
                asm volatile("mapa.shared::cluster.u32 %0, %1, 0;" : "=r"(r) : "r"(smem_u32(&rec[sg])));
                asm volatile("mapa.shared::cluster.u32 %0, %1, 0;" : "=r"(m) : "r"(smem_u32(&rbar)));
                asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v2.b32 [%0], {%1, %2}, [%3];"
                             ::"r"(r), "r"(__float_as_uint(zs.m)), "r"(__float_as_uint(zs.s)), "r"(m) : "memory");
            }
            if (rank != 0) continue;
            if (warp == 0) {                             // the records are on their way from running CTAs; a limit all the same
                const bool in = emit_wait(smem_u32(&rbar), parity, P.spin_limit);
                if (!in) (void)emit_wait(smem_u32(&rbar), parity, kEmitSpin);      // (they must have landed before the CTA goes on, or leaves)
                if (lane == 0) lost_s = !in;
            }
            parity ^= 1u;
            constexpr int K = kEmitMaxSeg / 32;          // runs per lane
            if (warp == 0) {
                float2 r[K];
                MS a{-INFINITY, 0.f, 0.f};
                const int per = (nseg + 31) >> 5;
#pragma unroll
                for (int k = 0; k < K; ++k) {
                    r[k] = k < per && lane * per + k < nseg ? rec[lane * per + k] : make_float2(-INFINITY, 0.f);
                    a = ms_combine(a, MS{r[k].x, r[k].y, 0.f});
                }
                a = ms_warp(a);
                const float inv_z = 1.f / a.s;
                if (lane == 0) { bc[0] = -a.m * kLog2e; bc[1] = inv_z; }
                double v[K], x = 0.0;                    // prefix sums of the runs' probabilities
#pragma unroll
                for (int k = 0; k < K; ++k) {
                    if (r[k].x > -INFINITY) x += (double)(r[k].y * ex2((r[k].x - a.m) * kLog2e) * inv_z);
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
                for (int k = 0; k < K; ++k) if (k < per && lane * per + k < nseg) cdf[lane * per + k] = before + v[k];
            }
            __syncthreads();
            if (lost_s) {                                // no draw from records that may not be the row's
                if (tid == 0) P.seq_tokens[(long long)pair * (P.positions + 1) + P.positions] = -1;
                continue;
            }
            const float off = bc[0], inv_z = bc[1];
            const double thr = (double)u * cdf[nseg - 1];
            const int s = warp_first_above(cdf, nseg, thr, lane);
            const float rem = (float)(thr - (s ? cdf[s - 1] : 0.0));
            const int nch = P.per / 32;                  // 256-position chunks of a run, at most 32 taken at a time
            float p[kVec], cum = 0.f, before = 0.f;
            int chosen = -1, last_pos = -1, held = -1;
            auto chunk_p = [&](int ch) -> float {
                float z[kVec], sum = 0.f;
                emit_load8<TZ>(zrow, s * P.per + ch * 32 + lane, phase, P.N, z);
#pragma unroll
                for (int q = 0; q < kVec; ++q) { p[q] = ex2(fmaf(z[q], kLog2e, off)) * inv_z; sum += p[q]; }
                held = ch;
                return warp_sum(sum);
            };
            for (int c0 = 0; c0 < nch && chosen < 0; c0 += 32) {
                for (int ch = c0 + warp; ch < min(nch, c0 + 32); ch += nw) {
                    const float sum = chunk_p(ch);
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
            const float r_in = chosen < 0 ? INFINITY : rem - before;     // rounding left no token: the last positive one
            if (chosen < 0) chosen = max(last_pos, 0);
            if (chosen % nw != warp) continue;
            if (held != chosen) (void)chunk_p(chosen);
            const int sel = max(pick_in_segment(p, r_in, lane), 0);
            if (lane == 0) P.seq_tokens[(long long)pair * (P.positions + 1) + P.positions] = min(max((s * P.per + chosen * 32) * kVec - phase + sel, 0), P.N - 1);
        }
        __syncthreads();                                 // all_s has been read
    }
}

template <typename TZ>
static cudaError_t launch_emit(EmitParams P, cudaStream_t s) {
    // Warps: few for few tokens, so that more rows are under way (2048 rows of 1000 tokens, all drawn from: 12 us, with
    // sixteen 32), and eight where rows are many (512 of 8000: 7.2 us, with sixteen 8.1; 64 or 160: 5.9 either way).
    // CTAs per cluster: a warp's run is at least two 256-position chunks, and all pairs can have such a cluster at once:
    // beyond that a larger one only serialises what would run side by side (2048 rows of 32000 tokens, all drawn from: 65 us, on
    // clusters of four 187).  Up to four pairs to a cluster for rows that one CTA takes longer over than their chain: 512 rows
    // of 262143, a tenth drawn from, 27 us, with single CTAs 37.  Clusters: what is resident at once.
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    const long long pairs = (long long)P.batch * P.trials;
    const unsigned nw = P.N <= 1000 ? 4 : (P.N <= 4000 || (P.N <= 65536 && pairs > 2 * sms) ? 8 : kEmitMaxWarps);
    const long long resident = (long long)sms * 64 / nw;        // CTAs, at 64 warps an SM
    unsigned C = 1;
    while (C < (unsigned)kEmitMaxCtas && (long long)C * nw * 512 < P.N && pairs * 2 * C <= (P.N > 65536 ? 4 : 1) * resident) C *= 2;
    const long long most = resident / C;
    P.per = (int)(((long long)P.N + 8 + C * nw * kVec - 1) / (C * nw * kVec));
    P.per = (P.per + 31) / 32 * 32;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(pairs < most ? pairs : most) * C, 1, 1);
    cfg.blockDim = dim3(nw * 32, 1, 1);
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
    P.spin_limit = stream_spin_limit() ? stream_spin_limit() : kEmitSpin;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const cudaError_t e = problem->target_dtype == RDK_F32 ? launch_emit<float>(P, s) : launch_emit<__nv_bfloat16>(P, s);
    if (e != cudaSuccess) return cuda_fail(e, "emit kernel launch");
    return RDK_OK;
}

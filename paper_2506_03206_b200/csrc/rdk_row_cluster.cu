// Cluster row kernel: one thread-block cluster takes one row (sequence, draft position) from its logits to its
// draws in one launch, the row held once in the cluster's shared memory.
//   soft-max statistics, Token-Level Intersection     (Eq. tli-drafter)
//   first-order redistribution                        (Eq. rdk-taylor), with p or a separate prior inside it,
//     or a given w = M^T q'                           (Algorithm 1 step 2)
//   acceptance rate, draft draw, rejection test, residual draw, or q~ written out   (Algorithm 4 steps 4-8)
//
// The row's 16-byte aligned positions are dealt out to the cluster's CTAs and inside a CTA to its warps, each warp
// a contiguous run ("segment").  Up to the first exchange everything is a warp's own affair: a warp copies its
// segment (cp.async.bulk on a barrier of its own, the few elements a 16-byte copy cannot cover by plain loads, so
// any row alignment will do), takes its own maximum as the scale of its exponentials, and leaves one record.  The
// CTAs then exchange one record each through distributed shared memory (theta, 1/Z_p, 1/Z_q), the warps finish
// their segment sums of w, min(p, q~), max(0, p - q~) and p and leave them in CTA 0.  The other CTAs are done then and
// make room for the next rows; CTA 0 draws: prefix sums over the segments, the draw's segment read again (from L2), its
// 256-position chunks shared by the warps.  (Draws made in place by the CTA that holds the segment would keep whole clusters
// waiting for two chains of dependent loads.)
//
// Four variants:
//   kVarSparse  N >= 4096, Eq. rdk-taylor with p itself.  A token that is not kept has q~ = theta x < p, x = p / N, so such
//               tokens enter through the segment's sum of p only; only the kept tokens are visited a second time,
//               from registers (kRegSlots x 32 per warp; the rest is evaluated anew).
//   kVarPrior   N >= 4096, Eq. rdk-taylor with a prior pi.  Here a token that is not kept needs its own min(p, theta pi / N),
//               so the second visit runs over all tokens.
//   kVarDense   any N, q~ output and small vocabularies, with or without a prior: a fp32 array of q' for all tokens of
//               the segment beside the logits.
//   kVarGiven   w in place of q'.
#include <math.h>
#include <string.h>

#include <atomic>
#include <type_traits>

#include "rdk_device.cuh"
#include "rdk_row.cuh"

namespace rdk {

enum { kVarSparse = 0, kVarPrior = 1, kVarDense = 2, kVarGiven = 3 };

constexpr int kCluMaxCtas = 16;                     // CTAs per cluster (above 8: non-portable)
constexpr int kCluMaxWarps = 16;
constexpr int kCluMaxSeg = kCluMaxCtas * kCluMaxWarps;
constexpr int kCluRound = 16;                       // trials settled between two collections
constexpr int kCluMaxChunks = 32;                   // 256-position chunks of a segment
constexpr unsigned kCluSpinDefault = 1u << 22;

// What CTA 0 needs for the draws lies where its part of the row was: nobody reads that any more by then.
struct DrawSmem {
    double cdf[3][kCluMaxSeg];                      // prefix sums of the segments' w, residual, p
    float4 res[2 * kCluRound];                      // draft (first half) and residual draws of a round
    float dsum[2 * kCluRound][kCluMaxChunks];       // a draw's sums over the chunks of its segment
};

struct CluGeo {
    int per;                 // vectors of 8 positions per warp, a multiple of 32
    uint32_t zoff_p, zoff_q; // byte offsets of the prior and of the q' array in dynamic shared memory
    uint32_t tag;            // marks this call's arrival counters
    unsigned spin_limit;
};

// Four floats into CTA `cta`'s copy of the shared variable at `local`, counted as 16 bytes on its barrier `bar`: a message and
// its signal in one, where a barrier over the cluster costs every CTA a round trip and a flush of its stores.
__device__ __forceinline__ void send_cluster4(uint32_t local, uint32_t bar, uint32_t cta, float a, float b, float c, float d) {
    uint32_t r, m;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(local), "r"(cta));
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(m) : "r"(bar), "r"(cta));
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v4.b32 [%0], {%1, %2, %3, %4}, [%5];"
                 ::"r"(r), "r"(__float_as_uint(a)), "r"(__float_as_uint(b)), "r"(__float_as_uint(c)), "r"(__float_as_uint(d)), "r"(m) : "memory");
}

// Scales of exponentials are whole powers of two: 2^(z log2 e - k) then has the rounding error of its own exponent only, and
// going from one scale to another is exact.  (On the scale e^m itself m log2 e is rounded for each segment apart, an error of the
// size of m that all tokens of the segment share.)
__device__ __forceinline__ float scale_of(float m) { return m > -INFINITY ? rintf(m * kLog2e) : -INFINITY; }

// One segment's share of the row, on the scales 2^m (target), 2^my (drafter), 2^mp (prior)
struct SegRec { float E, Zq, th, m, my, Ep, mp, W; };

// Folds the records of the warp's lanes into one (lanes without a record hold m = my = mp = -inf and zeros); the
// scale of th is that of the target (or the prior) times that of the drafter.
// exact_q: the drafter's sum in fp64 (see the warp totals).
template <bool PRIOR>
__device__ __forceinline__ SegRec fold_records(const SegRec& r, int lane, bool exact_q) {
    SegRec o;
    o.m = warp_max_redux(r.m); o.my = warp_max_redux(r.my);
    const float f = r.m > -INFINITY ? ex2(r.m - o.m) : 0.f;
    const float g = r.my > -INFINITY ? ex2(r.my - o.my) : 0.f;
    float fp = f;
    o.mp = 0.f; o.Ep = 0.f;
    if (PRIOR) {
        o.mp = warp_max_redux(r.mp);
        fp = r.mp > -INFINITY ? ex2(r.mp - o.mp) : 0.f;
    }
    const float t = warp_sum4(r.E * f, r.Zq * g, r.th * (fp * g), PRIOR ? r.Ep * fp : r.W, lane);
    o.E = __shfl_sync(0xffffffffu, t, 0); o.Zq = __shfl_sync(0xffffffffu, t, 8); o.th = __shfl_sync(0xffffffffu, t, 16);
    if (exact_q) o.Zq = (float)warp_sum_d((double)(r.Zq * g));
    const float last = __shfl_sync(0xffffffffu, t, 24);
    if (PRIOR) { o.Ep = last; o.W = 0.f; } else o.W = last;
    return o;
}

// 8 consecutive values at a 16-byte aligned shared address, as fp32
template <typename T> __device__ __forceinline__ void lds8(uint32_t a, float (&v)[kVec]);
template <> __device__ __forceinline__ void lds8<__nv_bfloat16>(uint32_t a, float (&v)[kVec]) {
    const uint4 q = lds128(a);
    v[0] = bf16_lo(q.x); v[1] = bf16_hi(q.x); v[2] = bf16_lo(q.y); v[3] = bf16_hi(q.y);
    v[4] = bf16_lo(q.z); v[5] = bf16_hi(q.z); v[6] = bf16_lo(q.w); v[7] = bf16_hi(q.w);
}
template <> __device__ __forceinline__ void lds8<float>(uint32_t a, float (&v)[kVec]) {
    const uint4 q = lds128(a), r = lds128(a + 16u);
    v[0] = __uint_as_float(q.x); v[1] = __uint_as_float(q.y); v[2] = __uint_as_float(q.z); v[3] = __uint_as_float(q.w);
    v[4] = __uint_as_float(r.x); v[5] = __uint_as_float(r.y); v[6] = __uint_as_float(r.z); v[7] = __uint_as_float(r.w);
}
template <typename T> __device__ __forceinline__ void sts_elem(uint32_t a, T v);
template <> __device__ __forceinline__ void sts_elem<float>(uint32_t a, float v) { sts32(a, __float_as_uint(v)); }
template <> __device__ __forceinline__ void sts_elem<__nv_bfloat16>(uint32_t a, __nv_bfloat16 v) {
    asm volatile("st.shared.u16 [%0], %1;" ::"r"(a), "h"(__bfloat16_as_ushort(v)) : "memory");
}
template <typename T> __device__ __forceinline__ T minus_inf();
template <> __device__ __forceinline__ float minus_inf<float>() { return -INFINITY; }
template <> __device__ __forceinline__ __nv_bfloat16 minus_inf<__nv_bfloat16>() { return __ushort_as_bfloat16((unsigned short)0xff80u); }

// How elements [0, cnt) of src get to shared address dst: when the two share their phase (mod 16 bytes), `body` elements
// behind the first `head` go by one bulk copy and the rest by plain loads; else all by plain loads.  Returns the bytes
// the barrier has to expect.
template <typename T>
__device__ __forceinline__ uint32_t copy_in_plan(const T* src, int cnt, uint32_t dst, int& head, int& body) {
    const uintptr_t a = reinterpret_cast<uintptr_t>(src);
    head = cnt; body = 0;
    if (((a ^ dst) & 15u) == 0) {
        const int h = min(cnt, (int)(((16u - (unsigned)(a & 15u)) & 15u) / sizeof(T)));
        const int b = (cnt - h) / (int)(16 / sizeof(T)) * (int)(16 / sizeof(T));
        if (b > 0) { head = h; body = b; }
    }
    return (uint32_t)body * (uint32_t)sizeof(T);
}
template <typename T>
__device__ __forceinline__ void copy_in_issue(const T* src, int cnt, uint32_t dst, int head, int body, uint32_t bar, int lane) {
    if (lane == 0 && body)
        asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                     ::"r"(dst + (uint32_t)(head * sizeof(T))), "l"(src + head), "r"((uint32_t)(body * sizeof(T))), "r"(bar) : "memory");
#pragma unroll 8
    for (int i = lane; i < head; i += 32) sts_elem<T>(dst + (uint32_t)(i * sizeof(T)), src[i]);
    for (int i = head + body + lane; i < cnt; i += 32) sts_elem<T>(dst + (uint32_t)(i * sizeof(T)), src[i]);
}

// Bounded wait for phase 0 of `bar` by one warp; false when the limit is reached.  A try may park the warp for a
// while, except under the small limits of the failure-path tests, whose tries must be able to run out.
__device__ __forceinline__ bool clu_wait(uint32_t bar, unsigned limit) {
    uint32_t done = 0;
    for (unsigned spins = 0; !done && spins < limit; ++spins) {
        if (limit < 64)
            asm volatile("{\n .reg .pred p;\n mbarrier.test_wait.parity.shared::cta.b64 p, [%1], 0;\n selp.u32 %0, 1, 0, p;\n}"
                         : "=r"(done) : "r"(bar) : "memory");
        else
            asm volatile("{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], 0;\n selp.u32 %0, 1, 0, p;\n}"
                         : "=r"(done) : "r"(bar) : "memory");
    }
    return __all_sync(0xffffffffu, done != 0);
}

// w_j = (N q'_j + theta p_j) / (N + p_j) = q'_j + x (theta - q'_j) / (1 + x) for 8 tokens, x = p_j / N (p the prior's where there
// is one).  From N = 4096 on 1 / (1 + x) = 1 - x up to x^2 <= 2^-24 of the correction term, which itself is x times a probability.
__device__ __forceinline__ void redistribute8(const float (&x)[kVec], const float (&qp)[kVec], float theta, bool small, float (&w)[kVec]) {
    if (small) {
#pragma unroll
        for (int k = 0; k < kVec; ++k) w[k] = fmaf(x[k] * (theta - qp[k]), __frcp_rn(1.f + x[k]), qp[k]);
    } else {
#pragma unroll
        for (int k = 0; k < kVec; ++k) w[k] = fmaf(x[k] * (theta - qp[k]), 1.f - x[k], qp[k]);
    }
}
__device__ __forceinline__ float redistribute1(float x, float qp, float theta) { return fmaf(x * (theta - qp), 1.f - x, qp); }

// accepted_len of a sequence (Algorithm 4 step 7): the number of leading accepted positions, counted by the position that
// arrives last.  The word of a (sequence, trial) holds (tag of the call, accept bits, arrivals), so it needs no
// initialisation, and one atomic operation carries a position's answer along with its arrival: nothing has to be fenced
// or read back.  The last one clears the word, for a replayed graph, whose calls carry the same tag.  Sequences longer
// than the bits count arrivals only and read the flags again.
constexpr int kCluBits = 24;
__device__ __forceinline__ void count_accepted(const RowParams& P, uint32_t tag, int row, int t, bool acc) {
    const int b = row / P.positions, pos = row - b * P.positions;
    unsigned long long* word = P.arrivals + (long long)b * P.trials + t;
    int32_t* out = P.accepted_len + (long long)b * P.trials + t;
    if (P.positions == 1) { *out = acc; return; }
    const bool bits = P.positions <= kCluBits;
    const unsigned long long mine = 1ull | (bits && acc ? 256ull << pos : 0ull), first = (unsigned long long)tag << 32 | mine;
    if (!bits) __threadfence();
    unsigned long long old = atomicCAS(word, 0ull, first), now = first;
    while (old != 0ull) {
        if ((uint32_t)(old >> 32) == tag) { now = atomicAdd(word, mine) + mine; break; }
        const unsigned long long seen = atomicCAS(word, old, first);          // left over from something else
        if (seen == old) break;
        old = seen;
    }
    const int arrived = bits ? (int)(now & 255ull) : (int)(uint32_t)now;
    if (arrived != P.positions) return;
    *word = 0ull;
    int k = 0;
    if (bits) {
        k = __ffs(~(int)((uint32_t)now >> 8)) - 1;
    } else {
        __threadfence();
        const volatile uint8_t* af = P.accepted;
        while (k < P.positions && af[((long long)b * P.positions + k) * P.trials + t]) ++k;
    }
    *out = k;
}

// Registers a thread: with many CTAs, what lets most of them be resident: 80 where two arrays and the draws' two chunks need
// them (320 rows of 128k with a prior: 117 -> 111 us, although a CTA of 512 threads then has the SM to itself), 64
// elsewhere (given weights of 1024 x 32k: 66 us, with 80 registers 70).  ROOMY, for calls whose CTAs all fit beside one another
// all the same: 128, nothing spilled and more loads in flight in a row's chain (5 rows of 128257 bf16 10.4 -> 8.7 us, with four
// trials 12.9 -> 9.5; 1 row of 5001 7.0 -> 6.4, given weights of 1 x 128256 8.1 -> 7.0).
template <int VAR, bool ROOMY> constexpr int clu_registers() { return ROOMY ? 128 : (VAR == kVarPrior ? 80 : 64); }

template <typename TZ, typename TY, int KIND, int VAR, bool kPrior, bool ROOMY>
__global__ void __maxnreg__((clu_registers<VAR, ROOMY>()))
rdk_cluster_kernel(const RowParams P, const CluGeo g) {
    constexpr bool kLinear = VAR != kVarGiven, kDense = VAR == kVarDense || VAR == kVarGiven;
    constexpr uint32_t es = (uint32_t)sizeof(TZ);
    // kept tokens per lane held in registers between the visits; more cost the others their registers
    constexpr int kRegSlots = VAR == kVarSparse ? 12 : 8;
    extern __shared__ __align__(128) unsigned char csm[];
    __shared__ __align__(16) float4 segs[kCluMaxSeg];            // per segment: sums of w, min(p, q~), max(0, p - q~), p
    __shared__ __align__(16) float4 xrec[kCluMaxCtas][2];        // one record per CTA of the cluster
    __shared__ __align__(16) float wrec[kCluMaxWarps][8];
    __shared__ __align__(8) unsigned long long wbar[kCluMaxWarps], xbar, sbar;     // a warp's copies; records of all CTAs; sums of all segments (CTA 0)
    __shared__ __align__(16) float4 tot_s[2];
    __shared__ float alpha_s, part_s[kCluMaxWarps];

    const int tid = threadIdx.x, lane = tid & 31;
    const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0), nw = blockDim.x >> 5;
    uint32_t rank, C;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
    asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(C));
    const int row = (int)(blockIdx.x / C);
    const bool small = P.N < kStreamMinN;

    const uint32_t bar = smem_u32(&wbar[warp]);
    if (lane == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(bar));
        if (warp == 0) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&xbar)));
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&sbar)));
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    __syncwarp();
    if (tid == 0) {
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(&xbar)), "r"(C * 32u) : "memory");
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(&sbar)), "r"(rank == 0 ? C * (uint32_t)nw * 16u : 0u) : "memory");
    }
    // another CTA's shared memory may be touched only once that CTA runs: arrive here, wait before the first message
    asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");

    // ---- this warp's segment: positions [sg len, (sg + 1) len) of the row, position = token + phase ----------------
    const TZ* zrow = static_cast<const TZ*>(P.target) + (long long)row * P.target_stride;
    const TZ* prow = kPrior ? static_cast<const TZ*>(P.prior) + (long long)row * P.prior_stride : nullptr;
    const int phase = (int)((reinterpret_cast<uintptr_t>(zrow) & 15u) / es);
    const int len = g.per * kVec;
    const int sg = (int)rank * nw + warp, nseg = (int)C * nw;
    const int seg_tok = sg * len - phase;                        // token at the segment's first position (may be negative)
    const int t0 = min(max(seg_tok, 0), P.N), t1 = max(t0, min(P.N, seg_tok + len));
    const uint32_t zb0 = smem_u32(csm), pb0 = zb0 + g.zoff_p, qb0 = zb0 + g.zoff_q;
    const uint32_t zb = zb0 + (uint32_t)(warp * len) * es, pb = pb0 + (uint32_t)(warp * len) * es, qb = qb0 + (uint32_t)(warp * len) * 4u;

    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");       // inputs may be the previous kernel's outputs, the index (a copy of one) too

    // header of the index and the ranks of the segment's ends: requested together, looked at when the copies are under way
    int4 h0 = make_int4(0, 0, 0, 0), h1 = h0;
    uint32_t end_word = 0;
    int end_rank = 0;
    const int end_tok = lane == 0 ? t0 : t1;
    if (kLinear) {
        h0 = __ldg(reinterpret_cast<const int4*>(P.header)); h1 = __ldg(reinterpret_cast<const int4*>(P.header) + 1);
        if (end_tok < P.N && lane < 2) { end_word = __ldg(P.mask + (end_tok >> 5)); end_rank = __ldg(P.rank + (end_tok >> 5)); }
    }

    {   // start the copies; positions without a token weigh nothing
        int zh, zl, ph = 0, pl = 0, qh = 0, ql = 0;
        const int n_tok = t1 - t0;
        const uint32_t lead = (uint32_t)(t0 - seg_tok);          // positions before the first token
        uint32_t total = copy_in_plan<TZ>(zrow + t0, n_tok, zb + lead * es, zh, zl);
        const float* wrow = VAR == kVarGiven ? P.w + (long long)row * P.w_stride : nullptr;
        if (kPrior) total += copy_in_plan<TZ>(prow + t0, n_tok, pb + lead * es, ph, pl);
        if (VAR == kVarGiven) total += copy_in_plan<float>(wrow + t0, n_tok, qb + lead * 4u, qh, ql);
        if (lane == 0) asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(total) : "memory");
        __syncwarp();
        copy_in_issue<TZ>(zrow + t0, n_tok, zb + lead * es, zh, zl, bar, lane);
        if (kPrior) copy_in_issue<TZ>(prow + t0, n_tok, pb + lead * es, ph, pl, bar, lane);
        if (VAR == kVarGiven) copy_in_issue<float>(wrow + t0, n_tok, qb + lead * 4u, qh, ql, bar, lane);
        for (int i = lane; i < len - n_tok; i += 32) {
            const uint32_t o = (uint32_t)(i < (int)lead ? i : i + n_tok);
            sts_elem<TZ>(zb + o * es, minus_inf<TZ>());
            if (kPrior) sts_elem<TZ>(pb + o * es, minus_inf<TZ>());
            if (VAR == kVarGiven) sts32(qb + o * 4u, 0u);
        }
        if (kDense && kLinear)
            for (int i = 0; i < len / 128; ++i) sts128(qb + (uint32_t)(i * 32 + lane) * 16u, 0.f, 0.f, 0.f, 0.f);
    }
    bool identity = true;
    int r0 = 0, cnt = 0;                                         // kept tokens of the segment: ranks [r0, r0 + cnt)
    if (kLinear) {
        if (h0.x != kIdxMagic || h0.y != P.N || h0.z != P.n) {      // not an index of this problem: the same decision everywhere
            if (tid == 0 && rank == 0 && P.status_word) atomicCAS(P.status_word, 0, (int)RDK_ERR_INVALID_ARG);
            clu_wait(bar, kCluSpinDefault);                      // the copies must land before the CTA leaves
            return;
        }
        identity = h1.y != 0;
        const int r = end_tok < P.N ? end_rank + __popc(end_word & ((1u << (end_tok & 31)) - 1u)) : h0.w;
        r0 = __shfl_sync(0xffffffffu, r, 0);
        cnt = __shfl_sync(0xffffffffu, r, 1) - r0;
    }
    // uniforms of the first round of draws: lane t < 16 has those of the draft draw of trial t, lane 16 + t of its residual draw
    const int trial = lane & (kCluRound - 1), kind = lane / kCluRound;
    const float* u_row = P.uniforms + (long long)row * P.trials * 4;
    float u_draw = 0.f, u_test = 0.f;
    if (trial < P.trials) { u_draw = __ldg(u_row + trial * 4 + 2 * kind); u_test = __ldg(u_row + trial * 4 + 1); }

    // ---- kept tokens: drafter values and positions of the first kRegSlots x 32 ---------------------------------------
    const TY* yrow = kLinear ? static_cast<const TY*>(P.drafter) + (long long)row * P.drafter_stride : nullptr;
    // four kept tokens per lane, the il-th of the segment and the ones 32, 64, 96 later; loads without branches (they travel
    // together), pos = -1 and a drafter value of no weight beyond the last
    auto load_kept = [&](int il, float* y, int* pos) {
        int i[4];
        const bool full = il - lane + 128 <= cnt;                // (the same in every lane)
#pragma unroll
        for (int k = 0; k < 4; ++k) i[k] = r0 + il + k * 32;
        if (!full) {
#pragma unroll
            for (int k = 0; k < 4; ++k) i[k] = min(i[k], r0 + cnt - 1);
        }
        if (!identity) {
#pragma unroll
            for (int k = 0; k < 4; ++k) i[k] = __ldg(P.slot + i[k]);
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) { y[k] = to_float<TY>(yrow[i[k]]); pos[k] = __ldg(P.ids + i[k]) - seg_tok; }
        if (!full) {
#pragma unroll
            for (int k = 0; k < 4; ++k)
                if (il + k * 32 >= cnt) { y[k] = KIND == RDK_LOGITS ? -INFINITY : 0.f; pos[k] = -1; }
        }
    };
    float ke[kRegSlots];                                             // drafter values, after the first visit e_y
    uint32_t kpos[kRegSlots / 2] = {};                                 // positions in the segment, two to a word; 0xffff: none
    auto pos_of = [&](int k) -> int { return (int)(short)(k & 1 ? kpos[k / 2] >> 16 : kpos[k / 2] & 0xffffu); };     // (a segment has at most 8192)
    auto load_slots = [&](int h) {                                   // slots h .. h + 3
        if (h * 32 < cnt) {
            int pos[4];
            load_kept(h * 32 + lane, ke + h, pos);
            kpos[h / 2] = (uint32_t)(pos[0] & 0xffff) | (uint32_t)pos[1] << 16;
            kpos[h / 2 + 1] = (uint32_t)(pos[2] & 0xffff) | (uint32_t)pos[3] << 16;
        } else {
#pragma unroll
            for (int k = 0; k < 4; ++k) ke[h + k] = KIND == RDK_LOGITS ? -INFINITY : 0.f;
            kpos[h / 2] = kpos[h / 2 + 1] = 0xffffffffu;
        }
    };
    float my_w = KIND == RDK_LOGITS ? -INFINITY : 0.f;
    if (kLinear) {
#pragma unroll
        for (int h = 0; h < kRegSlots; h += 4) load_slots(h);
        if (KIND == RDK_LOGITS) {
#pragma unroll
            for (int k = 0; k < kRegSlots; ++k) my_w = fmaxf(my_w, ke[k]);
            my_w = warp_max_redux(my_w);
        }
    }

    if (!clu_wait(bar, g.spin_limit)) {      // the copies must land before the CTA leaves all the same (bounded as well)
        for (unsigned spins = 0; spins < (1u << 16); ++spins) {
            uint32_t done;
            asm volatile("{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], 0;\n selp.u32 %0, 1, 0, p;\n}"
                         : "=r"(done) : "r"(bar) : "memory");
            if (done) break;
            __nanosleep(100);
        }
        if (lane == 0 && P.status_word) atomicCAS(P.status_word, 0, (int)RDK_ERR_TIMEOUT);
    }
    __syncwarp();

    // ---- first visit ------------------------------------------------------------------------------------------------
    // Scale of a segment's exponentials: its maximum, so that the heaviest tokens have the smallest exponents and with them the
    // smallest errors.  (On the maximum of the first vectors, which saves a pass over shared memory, q~ is 1.2 to 1.9 times
    // as far off.)  The drafter's is the maximum of the tokens in registers; any scale will do as long as the sum does not grow
    // beyond 1e18, in which case (or with nothing but -inf among them) the visit is repeated with the maximum of all.
    const int nit16 = g.per * kVec * (int)es / 512;              // 16-byte vectors per lane
    auto seg_max = [&](uint32_t base, int nit) -> float {
        MaxAcc<TZ> a;
#pragma unroll 4
        for (int k = 0; k < nit; ++k) a.push(lds128(base + (uint32_t)(k * 32 + lane) * 16u));
        return warp_max_redux(a.result());
    };
    auto seg_sum = [&](uint32_t base, float off) -> float {
        float2 Ea = splat(0.f), Eb = splat(0.f);
        const float2 l2 = splat(kLog2e), of = splat(off);
#pragma unroll 4
        for (int k = 0; k < nit16; ++k) exp_sum_vec<TZ>(lds128(base + (uint32_t)(k * 32 + lane) * 16u), l2, of, Ea, Eb);
        return (Ea.x + Ea.y) + (Eb.x + Eb.y);
    };
    const float m_w = scale_of(seg_max(zb, nit16)), mp_w = kPrior ? scale_of(seg_max(pb, nit16)) : -INFINITY;
    const float zoff = m_w > -INFINITY ? -m_w : 0.f, poff = mp_w > -INFINITY ? -mp_w : 0.f;
    float yoff = 0.f, my_s = KIND == RDK_LOGITS ? -INFINITY : 0.f;   // the drafter's scale (probabilities: 1)
    float E = seg_sum(zb, zoff), Ep = kPrior ? seg_sum(pb, poff) : 0.f;
    float K = 0.f, Zq = 0.f, th = 0.f, W = 0.f;
    float kz[kRegSlots];                                             // e_z (prior: that of the prior) of the first kept tokens
    const uint32_t db = kPrior ? pb : zb;                            // the distribution that enters theta
    // q~ is written out as it stands, not divided by its sum: the roundings of the 15 additions that fold the drafter's sum over
    // warp, CTA and cluster, each of the size of the whole, would be in all of a row's q~, and so would those of
    // exponents above zero (9e-8 to 1.1e-7 off 64 bits instead of 6e-8 to 7e-8)
    const bool exact_q = VAR == kVarDense && P.qtilde;
    auto max_of_rest = [&]() {                                       // the drafter's maximum, of the tokens beyond the registers too
        for (int il = kRegSlots * 32 + lane; il - lane < cnt; il += 128) {
            float y[4];
            int pos[4];
            load_kept(il, y, pos);
            my_w = fmaxf(fmaxf(my_w, fmaxf(y[0], y[1])), fmaxf(y[2], y[3]));
        }
        my_w = warp_max_redux(my_w);
    };
    if (KIND == RDK_LOGITS && exact_q && cnt > kRegSlots * 32) max_of_rest();
    for (int attempt = 0; kLinear && attempt < 2; ++attempt) {
        if (attempt == 1) {                                          // the values have become exponentials: once more
#pragma unroll
            for (int h = 0; h < kRegSlots; h += 4) load_slots(h);
            max_of_rest();
        }
        if (KIND == RDK_LOGITS) { my_s = scale_of(my_w); yoff = my_s > -INFINITY ? -my_s : 0.f; }
        K = 0.f; Zq = 0.f; th = 0.f;
        {
            const float doff = kPrior ? poff : zoff;
            auto visit = [&](int pos, const float y, float& ed, float& ey) {
                ed = ex2(fmaf(lds_z<TZ>(db + (uint32_t)max(pos, 0) * es), kLog2e, doff));
                if (pos < 0) ed = 0.f;
                ey = KIND == RDK_LOGITS ? ex2(fmaf(y, kLog2e, yoff)) : y;
                if (kDense && pos >= 0) sts32(qb + (uint32_t)pos * 4u, __float_as_uint(ey));
                K += ed; Zq += ey; th = fmaf(ed, ey, th);
            };
#pragma unroll
            for (int h = 0; h < kRegSlots; h += 4) {
                if (h * 32 < cnt) {
#pragma unroll
                    for (int k = 0; k < 4; ++k) visit(pos_of(h + k), ke[h + k], kz[h + k], ke[h + k]);
                } else {
#pragma unroll
                    for (int k = 0; k < 4; ++k) { kz[h + k] = 0.f; ke[h + k] = 0.f; }
                }
            }
            for (int il = kRegSlots * 32 + lane; il - lane < cnt; il += 128) {
                float y[4], ed, ey;
                int pos[4];
                load_kept(il, y, pos);
#pragma unroll
                for (int k = 0; k < 4; ++k) visit(pos[k], y[k], ed, ey);
            }
        }
        const bool poor = KIND == RDK_LOGITS && cnt > kRegSlots * 32 && (!(Zq < 1e18f) || !(my_s > -INFINITY));
        if (!__any_sync(0xffffffffu, poor)) break;
    }
    if (VAR == kVarGiven) {
#pragma unroll 4
        for (int k = 0; k < len / 128; ++k) {
            const uint4 q = lds128(qb + (uint32_t)(k * 32 + lane) * 16u);
            W += (__uint_as_float(q.x) + __uint_as_float(q.y)) + (__uint_as_float(q.z) + __uint_as_float(q.w));
        }
    }
    {   // warp totals
        if (exact_q) {
            const float all = (float)warp_sum_d((double)Zq);
            Zq = lane == 0 ? all : 0.f;
        }
        const float t = warp_sum4(E, K, Zq, th, lane);
        E = __shfl_sync(0xffffffffu, t, 0); K = __shfl_sync(0xffffffffu, t, 8);
        Zq = __shfl_sync(0xffffffffu, t, 16); th = __shfl_sync(0xffffffffu, t, 24);
        if (kPrior) Ep = warp_sum(Ep);
        if (VAR == kVarGiven) W = warp_sum(W);
    }
    if (lane == 0) {
        reinterpret_cast<float4*>(wrec[warp])[0] = make_float4(E, Zq, th, m_w);
        reinterpret_cast<float4*>(wrec[warp])[1] = make_float4(my_s, Ep, mp_w, W);
    }
    __syncthreads();

    // ---- first exchange: the row's soft-max sums and theta ------------------------------------------------------------
    if (warp == 0) {
        SegRec r{0.f, 0.f, 0.f, -INFINITY, -INFINITY, 0.f, -INFINITY, 0.f};
        if (lane < nw) {
            const float4 a = reinterpret_cast<const float4*>(wrec[lane])[0], b = reinterpret_cast<const float4*>(wrec[lane])[1];
            r = SegRec{a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
        }
        r = fold_records<kPrior>(r, lane, exact_q);
        asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");      // all CTAs of the cluster run
        if (lane < (int)C) {
            send_cluster4(smem_u32(&xrec[rank][0]), smem_u32(&xbar), (uint32_t)lane, r.E, r.Zq, r.th, r.m);
            send_cluster4(smem_u32(&xrec[rank][1]), smem_u32(&xbar), (uint32_t)lane, r.my, r.Ep, r.mp, r.W);
        }
        // (the messages are on their way as soon as all CTAs have come this far: no short limit, which would let a CTA leave
        // before a message to it has arrived)
        if (!clu_wait(smem_u32(&xbar), kCluSpinDefault) && lane == 0 && P.status_word) atomicCAS(P.status_word, 0, (int)RDK_ERR_TIMEOUT);
        r = SegRec{0.f, 0.f, 0.f, -INFINITY, -INFINITY, 0.f, -INFINITY, 0.f};
        if (lane < (int)C) {                             // fold the cluster's records, once per CTA
            const float4 a = xrec[lane][0], b = xrec[lane][1];
            r = SegRec{a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
        }
        r = fold_records<kPrior>(r, lane, exact_q);
        if (lane == 0) { tot_s[0] = make_float4(r.m, r.my, r.mp, r.W); tot_s[1] = make_float4(1.f / r.E, kLinear ? 1.f / r.Zq : 1.f, kPrior ? 1.f / r.Ep : 1.f / r.E, r.th); }
    }
    __syncthreads();
    const float4 tot_a = tot_s[0], tot_b = tot_s[1];
    const float tot_m = tot_a.x, tot_my = tot_a.y, tot_mp = tot_a.z;
    const float inv_zp = tot_b.x, inv_zq = tot_b.y, inv_zpi = tot_b.z;
    const float theta = kLinear ? tot_b.w * inv_zpi * inv_zq : 0.f;
    const float inv_n = 1.f / (float)P.N;
    const float offg = -tot_m, poffg = kPrior ? -tot_mp : 0.f;
    const float yoffg = KIND == RDK_LOGITS ? -tot_my : 0.f;
    // factor that turns the e_y of a segment with scale my into q'
    auto y_factor = [&](float my) -> float {
        return !kLinear ? 1.f : (KIND == RDK_LOGITS ? (my > -INFINITY ? ex2(my - tot_my) : 0.f) : 1.f) * inv_zq;
    };
    const float fy = y_factor(my_s);
    float inv_s = 1.f;

    // p and w of two neighbouring positions, from their logits (pr: prior's) and e_y (or w)
    const float fz = (m_w > -INFINITY ? ex2(m_w - tot_m) : 0.f) * inv_zp;      // e on the segment's scale -> p
    const float xs = kPrior ? (mp_w > -INFINITY ? ex2(mp_w - tot_mp) : 0.f) * inv_zpi * inv_n : fz * inv_n;    // -> x
    const float2 l2e2 = splat(kLog2e), zoff2 = splat(zoff), poff2 = splat(poff), fz2 = splat(fz), xs2 = splat(xs), fy2 = splat(fy), th2 = splat(theta), neg2 = splat(-1.f), one2 = splat(1.f);
    auto dense_pair = [&](float2 z, float2 pr, float2 q, float2& p, float2& w) {
        const float2 e = ex2_2(ffma2(z, l2e2, zoff2));
        p = fmul2(e, fz2);
        if (VAR == kVarGiven) { w = q; return; }
        const float2 x = fmul2(kPrior ? ex2_2(ffma2(pr, l2e2, poff2)) : e, xs2), qp = fmul2(q, fy2);
        const float2 t = fmul2(x, ffma2(qp, neg2, th2));                                   // x (theta - q')
        const float2 r = small ? make_float2(__frcp_rn(1.f + x.x), __frcp_rn(1.f + x.y)) : ffma2(x, neg2, one2);
        w = ffma2(t, r, qp);
    };
    // the four pairs of vector k * 32 + lane of the segment
    auto dense_vec = [&](int k, float2 (&p)[4], float2 (&w)[4]) {
        const uint32_t v = (uint32_t)(k * 32 + lane);
        float z[kVec], pr[kVec], q[kVec];
        lds8<TZ>(zb + v * kVec * es, z);
        if (kPrior) lds8<TZ>(pb + v * kVec * es, pr);
        lds8<float>(qb + v * 32u, q);
#pragma unroll
        for (int h = 0; h < 4; ++h)
            dense_pair(make_float2(z[2 * h], z[2 * h + 1]), kPrior ? make_float2(pr[2 * h], pr[2 * h + 1]) : splat(0.f), make_float2(q[2 * h], q[2 * h + 1]), p[h], w[h]);
    };
    const int nit = g.per / 32;                          // vectors of 8 positions per lane

    // ---- S.  Sum w = 1 + O(N^-2), because sum q' = 1 and the first-order terms cancel: taken as 1 from N = 4096 on -----
    if (VAR == kVarGiven) {
        inv_s = P.w_as_given ? 1.f : 1.f / tot_a.w;
    } else if (kDense && small) {                       // a small vocabulary: one CTA has the whole row
        float2 s2 = splat(0.f);
        for (int k = 0; k < nit; ++k) {
            float2 p[4], w[4];
            dense_vec(k, p, w);
#pragma unroll
            for (int h = 0; h < 4; ++h) s2 = fadd2(s2, w[h]);
        }
        float s = warp_sum(s2.x + s2.y);
        if (lane == 0) part_s[warp] = s;
        __syncthreads();
        s = lane < nw ? part_s[lane] : 0.f;
        inv_s = 1.f / warp_sum(s);
    }

    // ---- second visit: the segment's sums of w, min(p, q~), max(0, p - q~), p -----------------------------------------
    float4 sums;
    if (VAR == kVarSparse) {
        float ak = 0.f;
#pragma unroll
        for (int k = 0; k < kRegSlots; ++k) {
            if ((k & ~3) * 32 < cnt) {
                const float qp = ke[k] * fy;
                ak += fminf(kz[k] * fz, fmaf(kz[k] * xs, theta - qp, qp));
            }
        }
        for (int il = kRegSlots * 32 + lane; il - lane < cnt; il += 128) {
            float y[4];
            int pos[4];
            load_kept(il, y, pos);
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const float ez = ex2(fmaf(lds_z<TZ>(zb + (uint32_t)max(pos[k], 0) * es), kLog2e, zoff));
                const float qp = (KIND == RDK_LOGITS ? ex2(fmaf(y[k], kLog2e, yoff)) : y[k]) * fy;
                const float a = fminf(ez * fz, fmaf(ez * xs, theta - qp, qp));
                ak += pos[k] >= 0 ? a : 0.f;
            }
        }
        ak = warp_sum(ak);
        const float segP = E * fz;
        const float oov = theta * xs * fmaxf(0.f, E - K);
        const float Kw = fy * Zq - fy * xs * th + theta * xs * K;
        sums = make_float4(oov + Kw, oov + ak, fmaxf(0.f, segP - (oov + ak)), segP);
    } else if (VAR == kVarPrior) {
        // All tokens as if not kept, w = theta x (what x^2 takes away is below 1 / N^2 in all); that is the smaller of w and p
        // nearly everywhere, so the sum of min(p, w) is theta times that of x, less w - p where p is the smaller: where
        // z - prior falls below a constant of the row.  The difference of the logits (in their own type, with a margin
        // for its rounding) tells; only vectors with such a token evaluate their exponentials again.  (Evaluating all:
        // 150 us for 320 rows of 128k.)  Then the kept tokens' own w, in place of theta x.
        float c = (__log2f(theta * xs) - __log2f(fz) + poff - zoff) * (1.f / kLog2e);
        c = c == c ? c + fabsf(c) * 0x1p-7f + 0.01f : INFINITY;
        float viol = 0.f;
        auto over = [&](float z, float pr) { viol += fmaxf(0.f, theta * xs * ex2(fmaf(pr, kLog2e, poff)) - fz * ex2(fmaf(z, kLog2e, zoff))); };
#pragma unroll 4
        for (int k = 0; k < nit16; ++k) {
            const uint4 qz = lds128(zb + (uint32_t)(k * 32 + lane) * 16u), qp = lds128(pb + (uint32_t)(k * 32 + lane) * 16u);
            const uint32_t vz[4] = {qz.x, qz.y, qz.z, qz.w}, vp[4] = {qp.x, qp.y, qp.z, qp.w};
            if (sizeof(TZ) == 2) {
                __nv_bfloat162 d[4];
#pragma unroll
                for (int h = 0; h < 4; ++h) d[h] = __hsub2(*reinterpret_cast<const __nv_bfloat162*>(&vz[h]), *reinterpret_cast<const __nv_bfloat162*>(&vp[h]));
                const __nv_bfloat162 m = __hmin2(__hmin2(d[0], d[1]), __hmin2(d[2], d[3]));
                if (!(fminf(__low2float(m), __high2float(m)) < c)) continue;
#pragma unroll
                for (int h = 0; h < 4; ++h) { over(bf16_lo(vz[h]), bf16_lo(vp[h])); over(bf16_hi(vz[h]), bf16_hi(vp[h])); }
            } else {
                float m = INFINITY;
#pragma unroll
                for (int h = 0; h < 4; ++h) m = fminf(m, __uint_as_float(vz[h]) - __uint_as_float(vp[h]));
                if (!(m < c)) continue;
#pragma unroll
                for (int h = 0; h < 4; ++h) over(__uint_as_float(vz[h]), __uint_as_float(vp[h]));
            }
        }
        float dw = 0.f, da = 0.f;
        auto again = [&](int pos, float ep, float ey) {
            const float p = ex2(fmaf(lds_z<TZ>(zb + (uint32_t)max(pos, 0) * es), kLog2e, zoff)) * fz, x = ep * xs;
            const float w0 = theta * x, w = redistribute1(x, ey * fy, theta);
            if (pos >= 0) { dw += w - w0; da += fminf(p, w) - fminf(p, w0); }
        };
#pragma unroll
        for (int k = 0; k < kRegSlots; ++k) if ((k & ~3) * 32 < cnt) again(pos_of(k), kz[k], ke[k]);
        for (int il = kRegSlots * 32 + lane; il - lane < cnt; il += 128) {
            float y[4];
            int pos[4];
            load_kept(il, y, pos);
#pragma unroll
            for (int k = 0; k < 4; ++k)
                again(pos[k], ex2(fmaf(lds_z<TZ>(pb + (uint32_t)max(pos[k], 0) * es), kLog2e, poff)), KIND == RDK_LOGITS ? ex2(fmaf(y[k], kLog2e, yoff)) : y[k]);
        }
        const float segP = E * fz, all = theta * xs * Ep;
        const float sw = all + warp_sum(dw), sa = all + warp_sum(da - viol);
        sums = make_float4(sw, sa, fmaxf(0.f, segP - sa), segP);
    } else {
        float2 sw2 = splat(0.f), sa2 = splat(0.f), sr2 = splat(0.f);
        const float2 is2 = splat(inv_s);
        float* qrow = P.qtilde ? P.qtilde + (long long)row * P.N : nullptr;
        // the row of q~ and the positions share their 16-byte phase: store vectors straight away, else by way of shared memory
        const bool straight = qrow && ((reinterpret_cast<uintptr_t>(qrow) - 4u * (unsigned)phase) & 15u) == 0;
        for (int k = 0; k < nit; ++k) {
            float2 p[4], w[4];
            dense_vec(k, p, w);
#pragma unroll
            for (int h = 0; h < 4; ++h) {
                sw2 = fadd2(sw2, w[h]);
                w[h] = fmul2(w[h], is2);                             // q~
                const float2 a = make_float2(fminf(p[h].x, w[h].x), fminf(p[h].y, w[h].y));
                sa2 = fadd2(sa2, a);
                sr2 = fadd2(sr2, ffma2(a, neg2, p[h]));              // max(0, p - q~)
            }
            if (kLinear && qrow) {
                const int tok = seg_tok + (k * 32 + lane) * kVec;
                if (straight && tok >= 0 && tok + kVec <= P.N) {
                    reinterpret_cast<float4*>(qrow + tok)[0] = make_float4(w[0].x, w[0].y, w[1].x, w[1].y);
                    reinterpret_cast<float4*>(qrow + tok)[1] = make_float4(w[2].x, w[2].y, w[3].x, w[3].y);
                } else if (straight) {
#pragma unroll
                    for (int h = 0; h < 4; ++h) {
                        if (tok + 2 * h >= 0 && tok + 2 * h < P.N) qrow[tok + 2 * h] = w[h].x;
                        if (tok + 2 * h + 1 >= 0 && tok + 2 * h + 1 < P.N) qrow[tok + 2 * h + 1] = w[h].y;
                    }
                } else {
                    const uint32_t a = qb + (uint32_t)(k * 32 + lane) * 32u;
                    sts128(a, w[0].x, w[0].y, w[1].x, w[1].y);
                    sts128(a + 16u, w[2].x, w[2].y, w[3].x, w[3].y);
                }
            }
        }
        if (kLinear && qrow && !straight) {
            __syncwarp();
            for (int t = t0 + lane; t < t1; t += 32) qrow[t] = __uint_as_float(lds32(qb + (uint32_t)(t - seg_tok) * 4u));
        }
        const float t = warp_sum4(sw2.x + sw2.y, sa2.x + sa2.y, sr2.x + sr2.y, 0.f, lane);
        sums = make_float4(__shfl_sync(0xffffffffu, t, 0), __shfl_sync(0xffffffffu, t, 8), __shfl_sync(0xffffffffu, t, 16), E * fz);
    }

    // ---- second exchange: CTA 0 gets the sums of all segments; the others are done -----------------------------------------
    if (lane == 0) send_cluster4(smem_u32(&segs[sg]), smem_u32(&sbar), 0u, sums.x, sums.y, sums.z, sums.w);
    if (rank != 0) return;
    if (!clu_wait(smem_u32(&sbar), kCluSpinDefault) && lane == 0 && P.status_word) atomicCAS(P.status_word, 0, (int)RDK_ERR_TIMEOUT);
    DrawSmem& ds = *reinterpret_cast<DrawSmem*>(csm);
    double (&cdf)[3][kCluMaxSeg] = ds.cdf;
    for (int job = warp; job < 4; job += nw) {
        constexpr int kPerLane = kCluMaxSeg / 32;
        const int per_lane = (nseg + 31) >> 5, s0 = lane * per_lane;
        double run[kPerLane], x = 0.0;
#pragma unroll
        for (int k = 0; k < kPerLane; ++k) {
            if (k < per_lane && s0 + k < nseg) {
                const float4 s = segs[s0 + k];
                x += (double)(job == 0 ? s.x : (job == 1 ? s.z : (job == 2 ? s.w : s.y)));
            }
            run[k] = x;
        }
        if (job == 3) {
            x = warp_sum_d(x);
            if (lane == 0) alpha_s = (float)x;
        } else {
            double incl = x;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const double a = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += a;
            }
            double before = __shfl_up_sync(0xffffffffu, incl, 1);
            if (lane == 0) before = 0.0;
#pragma unroll
            for (int k = 0; k < kPerLane; ++k)
                if (k < per_lane && s0 + k < nseg) cdf[job][s0 + k] = before + run[k];
        }
    }
    __syncthreads();
    const double S_d = cdf[0][nseg - 1], R_d = cdf[1][nseg - 1];
    if (tid == 0) {
        if (P.alpha) P.alpha[row] = alpha_s;
        if (P.theta) P.theta[row] = theta;
        if (P.S) P.S[row] = (float)S_d;
        if (P.residual_mass) P.residual_mass[row] = (float)R_d;
    }

    // ---- draws ------------------------------------------------------------------------------------------------------------
    // Every step here is a round trip to L2 or a chain of barriers that only this row waits for, so the draws of a round
    // (a draft and a residual draw per trial) go side by side: their segments' 256-position chunks are dealt out to the
    // warps, two at a time so that both chunks' loads travel together.  (One chunk at a time, binary searches by every
    // thread, an integer division per draw and a fence with three dependent loads for accepted_len took 18 to 40 thousand
    // cycles a row, twice what the row itself takes.)
    const bool from_p = !(R_d > 0.0);                    // p and q~ coincide: the replacement comes from p itself
    const int nch = g.per / 32;
    auto load_row8 = [&](const auto* src, int jb, float fill, float (&v)[kVec]) {
        using T = typename std::remove_cv<typename std::remove_pointer<decltype(src)>::type>::type;
        if (jb >= 0) {
            load8<T>(src, jb, P.N, (reinterpret_cast<uintptr_t>(src + jb) & 15u) == 0, fill, v);
        } else {
#pragma unroll
            for (int k = 0; k < kVec; ++k) v[k] = jb + k >= 0 && jb + k < P.N ? to_float<T>(src[jb + k]) : fill;
        }
    };
    const float* wrow = VAR == kVarGiven ? P.w + (long long)row * P.w_stride : nullptr;
    // x[h] of this lane's 8 positions in chunk ch[h] of segment sgm[h], for H chunks at once, read from global memory again;
    // what[h] = 0: w, 1: max(0, p - q~), 2: p.  sum[h]: over the warp.
    auto chunks = [&](auto HC, const int* sgm, const int* ch, const int* what, float (*x)[kVec], float* sum) {
        constexpr int H = decltype(HC)::value;
        float z[H][kVec], a[H][kVec];
        uint32_t mb[H];
        int i[H][kVec], jb[H];
#pragma unroll
        for (int h = 0; h < H; ++h) {
            jb[h] = sgm[h] * len - phase + (ch[h] * 32 + lane) * kVec;
            load_row8(zrow, jb[h], -INFINITY, z[h]);
            if (VAR == kVarGiven) load_row8(wrow, jb[h], 0.f, a[h]);
            if (kPrior) load_row8(prow, jb[h], -INFINITY, a[h]);
        }
        if (kLinear) {       // the kept tokens among the 8, looked up in the index
            uint32_t lo[H], hi[H];
            int rw[H];
#pragma unroll
            for (int h = 0; h < H; ++h) {
                const int wi = jb[h] >> 5;
                const bool in = wi >= 0 && jb[h] < P.N;
                lo[h] = in ? __ldg(P.mask + wi) : 0u;
                hi[h] = jb[h] < P.N && (wi + 1) * 32 < P.N ? __ldg(P.mask + wi + 1) : 0u;
                rw[h] = in ? __ldg(P.rank + wi) : 0;
            }
#pragma unroll
            for (int h = 0; h < H; ++h) {
                const int sh = jb[h] & 31;
                mb[h] = __funnelshift_r(lo[h], hi[h], sh) & 0xffu;
                const int rb = rw[h] + __popc(lo[h] & ((1u << sh) - 1u));
                // independent loads: a token that is not kept reads what the first kept one does (or entry 0)
#pragma unroll
                for (int k = 0; k < kVec; ++k) i[h][k] = (mb[h] >> k) & 1u ? rb + __popc(mb[h] & ((1u << k) - 1u)) : (mb[h] ? rb : 0);
            }
            if (!identity) {
#pragma unroll
                for (int h = 0; h < H; ++h)
#pragma unroll
                    for (int k = 0; k < kVec; ++k) i[h][k] = __ldg(P.slot + i[h][k]);
            }
#pragma unroll
            for (int h = 0; h < H; ++h)
#pragma unroll
                for (int k = 0; k < kVec; ++k) i[h][k] = __float_as_int(to_float<TY>(yrow[i[h][k]]));
        }
#pragma unroll
        for (int h = 0; h < H; ++h) {
            float w[kVec], q[kVec];
#pragma unroll
            for (int k = 0; k < kVec; ++k) {
                z[h][k] = ex2(fmaf(z[h][k], kLog2e, offg)) * inv_zp;
                if (VAR == kVarGiven) w[k] = a[h][k];
                if (kLinear) {
                    const float y = __int_as_float(i[h][k]);
                    a[h][k] = kPrior ? ex2(fmaf(a[h][k], kLog2e, poffg)) * inv_zpi * inv_n : z[h][k] * inv_n;
                    q[k] = (mb[h] >> k) & 1u ? (KIND == RDK_LOGITS ? ex2(fmaf(y, kLog2e, yoffg)) : y) * inv_zq : 0.f;
                }
            }
            if (kLinear) redistribute8(a[h], q, theta, small, w);
            float t = 0.f;
#pragma unroll
            for (int k = 0; k < kVec; ++k) {
                x[h][k] = what[h] == 0 ? w[k] : (what[h] == 1 ? fmaxf(0.f, z[h][k] - w[k] * inv_s) : z[h][k]);
                t += x[h][k];
            }
            sum[h] = warp_sum(t);
        }
    };
    for (int base = 0; base < P.trials; base += kCluRound) {
        const int nt = min(kCluRound, P.trials - base), nd = 2 * nt, items = nd * nch;
        if (base && trial < nt) { u_draw = __ldg(u_row + (base + trial) * 4 + 2 * kind); u_test = __ldg(u_row + (base + trial) * 4 + 1); }
        // draw d < nt: the draft draw of trial base + d; nt + d: its residual draw (needed only if the draft is rejected)
        auto locate = [&](int d, int& sgm, int& what, float& rem) {
            const bool res = d >= nt;
            const double* c = res ? (from_p ? cdf[2] : cdf[1]) : cdf[0];
            const double thr = (double)__shfl_sync(0xffffffffu, u_draw, res ? kCluRound + d - nt : d) * c[nseg - 1];
            sgm = warp_first_above(c, nseg, thr, lane);
            rem = (float)(thr - (sgm ? c[sgm - 1] : 0.0));
            what = res ? (from_p ? 2 : 1) : 0;
        };
        // the token of draw d where the running sum of x, from the start of chunk ch, passes r_in
        auto pick = [&](int d, int sgm, int ch, const float (&x)[kVec], float r_in) {
            const int sel = max(pick_in_segment(x, r_in, lane), 0);
            float wd = 0.f;
#pragma unroll
            for (int k = 0; k < kVec; ++k) if (k == (sel & (kVec - 1))) wd = x[k];
            wd = __shfl_sync(0xffffffffu, wd, sel / kVec);
            const int tok = min(max(sgm * len - phase + ch * 256 + sel, 0), P.N - 1);
            if (lane == 0) ds.res[d] = make_float4(__int_as_float(tok), ex2(fmaf(to_float<TZ>(zrow[tok]), kLog2e, offg)) * inv_zp, wd, 0.f);
        };
        // the chunk of draw d in which rem is passed, and what is left of rem there; rounding may leave none: the last positive one
        auto choose = [&](int d, float rem, int& ch, float& r_in) {
            const float v = lane < nch ? ds.dsum[d][lane] : 0.f;
            float incl = v;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const float t = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += t;
            }
            const uint32_t pos = __ballot_sync(0xffffffffu, v > 0.f), hit = __ballot_sync(0xffffffffu, v > 0.f && incl > rem);
            ch = hit ? __ffs(hit) - 1 : (pos ? 31 - __clz(pos) : 0);
            const float before = __shfl_sync(0xffffffffu, incl - v, ch);
            r_in = hit ? rem - before : INFINITY;
        };
        if (nch == 1) {                                  // no sums to look at: a warp settles its draws by itself
            for (int d = warp; d < nd; d += nw) {
                int sgm[1], what[1];
                const int ch[1] = {0};
                float rem, x[1][kVec], sum[1];
                locate(d, sgm[0], what[0], rem);
                chunks(std::integral_constant<int, 1>(), sgm, ch, what, x, sum);
                pick(d, sgm[0], 0, x[0], rem);
            }
        } else {
            int d[2] = {0, 0}, ch[2] = {0, 0}, sgm[2] = {0, 0}, what[2] = {0, 0};
            float rem[2] = {0.f, 0.f}, x[2][kVec], sum[2];
            for (int it = warp; it < items; it += 2 * nw) {
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int item = it + h * nw;
                    if (item >= items) break;
                    d[h] = item / nch; ch[h] = item - d[h] * nch;
                    locate(d[h], sgm[h], what[h], rem[h]);
                }
                if (it + nw < items) {
                    chunks(std::integral_constant<int, 2>(), sgm, ch, what, x, sum);
                    if (lane == 0) ds.dsum[d[1]][ch[1]] = sum[1];
                } else {
                    chunks(std::integral_constant<int, 1>(), sgm, ch, what, x, sum);
                }
                if (lane == 0) ds.dsum[d[0]][ch[0]] = sum[0];
            }
            __syncthreads();
            int c;
            float r_in;
            if (items <= 2 * nw) {                       // every chunk is still in the registers of the warp that summed it
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    if (warp + h * nw >= items) break;
                    choose(d[h], rem[h], c, r_in);
                    if (c == ch[h]) pick(d[h], sgm[h], c, x[h], r_in);
                }
            } else {
                for (int e = warp; e < nd; e += nw) {
                    locate(e, sgm[0], what[0], rem[0]);
                    choose(e, rem[0], ch[0], r_in);
                    chunks(std::integral_constant<int, 1>(), sgm, ch, what, x, sum);
                    pick(e, sgm[0], ch[0], x[0], r_in);
                }
            }
        }
        __syncthreads();
        if (tid < nt) {
            const int dtok = __float_as_int(ds.res[tid].x);
            const float pd = ds.res[tid].y, qd = ds.res[tid].z * inv_s;
            const bool acc = u_test * qd < pd;
            const long long o = (long long)row * P.trials + base + tid;
            if (P.draft_token) P.draft_token[o] = dtok;
            if (P.accepted) P.accepted[o] = acc ? 1 : 0;
            if (P.accept_prob) P.accept_prob[o] = (pd >= qd) ? 1.f : pd / qd;
            if (P.out_token) P.out_token[o] = acc ? dtok : __float_as_int(ds.res[nt + tid].x);
            if (P.arrivals && P.accepted_len) count_accepted(P, g.tag, row, base + tid, acc);
        }
        if (base + kCluRound < P.trials) __syncthreads();        // the round's draws have been read
    }
}

// ------------------------------------------------------------------------------------------------
// host side
// ------------------------------------------------------------------------------------------------
constexpr int kCluStatic = 7 * 1024;                            // static shared memory of the kernel and what a CTA has besides, rounded up
constexpr int kCluDynamic = 227 * 1024 - 6 * 1024 - 512;
constexpr int kCluSms = 148;

struct CluShape { int C, nw, per; size_t smem; bool roomy; float cost; };

// A rule of thumb for the time of a call with a given shape, in us: launch and row statistics, then for every wave of CTAs a
// chain (k; km where waves follow one another), b for each 256-position chunk of a warp, what the number of warps and CTAs of a row adds
// to the exchange and to the prefix sums, a second pass over the chunks for the draws (unless there is but one), more
// rounds of draws, kept tokens beyond a warp's registers (visited in memory, twice) and the warps that share the SM.
// The constants are a fit to measured calls: 539 problems (N from 4992 to 262143, 1 to 1000 rows, bf16 and fp32), some 39 shapes of each.
// The shape that the rule picks is within 1 to 4 % of the fastest one tried on average (a prior 0.7 %, one draw a row 3.9 %); powers of
// two alone, which this replaces as the last word, were 8 to 20 % off (50257 tokens: 80 rows 16.9 -> 12.3 us, 320 rows
// 44.8 -> 33.5; 128257: 320 rows 86.4 -> 70.4; q~ of 80 x 262143: 114.6 -> 62.1; given weights of 40 x 50240: 11.4 -> 8.7).
// With three trials or more, clusters of one CTA an SM are counted as they were seen to fit: 32 rows of four trials at 32001 are
// one round of four CTAs with 128 registers (fp32 13.6 -> 9.8 us, bf16 11.9 -> 8.6), and 24 rows at 44001 would be two rounds of
// five (15.6 us against 11.9 with four).
struct CluCost {
    float t0, k, km, b, seg, cluster, second, over, warps, tail, fill, roomy, draws;
    bool counted;        // see rows_at_once
};
constexpr CluCost kCostFewDraws{3.794f, 1.737f, 0.762f, 0.742f, 0.015f, 0.501f, 0.394f, 2.617f, 2.986f, 0.006f, 0.776f, 0.902f, 1.884f, false};
constexpr CluCost kCostManyDraws{5.372f, 0.72f, 1.228f, 1.997f, 0.01f, 1.092f, 0.249f, 3.958f, 0.002f, 0.173f, 0.829f, 0.702f, 0.993f, true};
constexpr CluCost kCostDense{3.425f, 2.429f, 4.145f, 0.574f, 0.275f, 0.081f, 0.168f, 0.151f, 0.69f, 0.281f, 0.876f, 0.845f, 0.117f, false};
constexpr CluCost kCostPrior{4.82f, 4.042f, 1.734f, 1.087f, 0.033f, 0.61f, 0.494f, 0.034f, 2.926f, 0.829f, 0.949f, 0.982f, 1.884f, false};
constexpr CluCost kCostGiven{3.984f, 0.916f, 1.611f, 0.565f, 1.035f, 0.125f, 0.613f, 2.38f, 0.613f, 0.48f, 0.87f, 0.846f, 0.713f, false};

// The shape with C CTAs a row and at most `warps` warps each; false where a row does not fit.
static bool shape_cluster(long long positions, int rows, int trials, int C, int warps, size_t bytes, bool roomy, CluShape& s) {
    const int chunks = (int)((positions + C * 256 - 1) / (C * 256)), per = (chunks + warps - 1) / warps;
    const int nw = (chunks + per - 1) / per;
    s.C = C; s.nw = nw < 4 ? 4 : nw; s.per = per * 32; s.roomy = roomy;
    // segments of one chunk and several draws a row: a warp for each draw, also where there is nothing to sweep for it
    if (per == 1 && (long long)rows * C < 4 * kCluSms && 2 * trials > s.nw) s.nw = 2 * trials < kCluMaxWarps ? 2 * trials : kCluMaxWarps;
    s.smem = (size_t)s.nw * s.per * kVec * bytes;
    if (s.smem < sizeof(DrawSmem)) s.smem = sizeof(DrawSmem);
    return s.smem <= (size_t)kCluDynamic && per <= kCluMaxChunks;
}

// CTAs of a shape that an SM holds
static int resident_ctas(const CluShape& s, int registers) {
    const int by_smem = (int)(228u * 1024u / (s.smem + kCluStatic + 256)), by_regs = 65536 / (registers * 32 * s.nw), by_warps = 64 / s.nw;
    const int n = by_smem < by_regs ? by_smem : by_regs;
    return n < by_warps ? (n < 1 ? 1 : n) : by_warps;
}

// Rows under way at once.  Clusters do not fill the chip to the last SM, as they stay within a group of SMs: about `fill` of what
// the SMs hold, but of one CTA an SM, and of eight CTAs or more two an SM, no more than the driver counts (of ten CTAs 11: q~ of
// 12 x 136768 in two rounds of them took 14.3 us, with two CTAs an SM of sixteen 10.0; of five CTAs 22: 24 rows took two rounds,
// although it counts 26).  `counted`: that count itself for one CTA an SM, where `fill` is too low a guess.
static int rows_at_once(const CluCost& c, const CluShape& s, int slots) {
    constexpr int kOne[kCluMaxCtas + 1] = {0, 148, 74, 45, 33, 22, 22, 15, 15, 15, 11, 7, 7, 7, 7, 7, 7};
    if (s.C == 1) return kCluSms * slots;
    const int filled = (int)(c.fill * (float)(kCluSms * slots) / (float)s.C), most = kOne[s.C] * slots;
    if (slots == 1 && c.counted) return most;
    const int n = (slots == 1 || (slots == 2 && s.C >= 8)) && most < filled ? most : filled;
    return n < 1 ? 1 : n;
}

static float cost_cluster(const CluCost& c, const CluShape& s, int rows, int trials, int registers, float kept, int kept_slots) {
    const int slots = resident_ctas(s, registers), chunks = s.per / 32;
    const float waves = (float)rows / (float)rows_at_once(c, s, slots);
    float resident = (float)rows * (float)s.C / (float)kCluSms;
    resident = resident < 1.f ? 1.f : (resident > (float)slots ? (float)slots : resident);
    const float most = kept * 256.f * (float)chunks + 2.f * sqrtf(kept * 256.f * (float)chunks);     // kept tokens of a warp, nearly at most
    const float over = most > (float)kept_slots ? ceilf((most - (float)kept_slots) / 128.f) : 0.f;
    const int rounds = (trials * chunks + s.nw - 1) / s.nw - 1;                                        // two draws a trial, two chunks a turn
    const float one = (waves > 1.f ? c.km : c.k) + c.b * (float)chunks + c.seg * (float)(s.C * s.nw) / 128.f + (s.C > 1 ? c.cluster : 0.f) +
                      (chunks > 1 ? c.second : 0.f) + c.over * over + c.warps * resident * (float)s.nw / 32.f + c.draws * (float)(rounds > 0 ? rounds : 0);
    return c.t0 + (waves > 1.f ? waves + c.tail : 1.f) * one * (s.roomy ? c.roomy : 1.f);
}

// CTAs per row, warps per CTA and vectors per warp; false when a row does not fit a cluster's shared memory.  `lead`: most
// positions before a row's first token.
static bool plan_cluster_anew(int N, int n, int rows, int trials, size_t es, int variant, bool prior, int lead, CluShape& s) {
    const size_t bytes = es * (prior ? 2 : 1) + (variant == kVarDense || variant == kVarGiven ? 4 : 0);    // per position
    const long long positions = (long long)N + lead;
    const int registers = variant == kVarPrior ? 80 : 64;
    int C = 1;
    if (N >= kStreamMinN) {
        // three CTAs to an SM, whose phases of copying, exponentials and waiting overlap (320 rows of 128k with a prior: 112 us) ...
        while (C < kCluMaxCtas && (long long)bytes * (positions / C) > 64 * 1024) C *= 2;
        // ... and, with few rows, enough CTAs to fill the chip four times over, while each has 4096 positions or more (with
        // less the exchange between the CTAs costs more than the sweep)
        while (C < kCluMaxCtas && (long long)rows * C < 4 * kCluSms && positions / C > 4096) C *= 2;
    }
    // about eight warps of equally many 256-position chunks each: more warps mean more per-warp overhead, fewer do not
    // hide each other's latencies (50257 tokens x 160 rows: 8 warps 29 us, 12 35, 16 46)
    // (sixteen, and shorter segments, where several draws a row keep the warps busy -- 32 rows of 32k with four trials 16.6 ->
    // 14.1 us, 1500 rows of 8k with eight 107 -> 84 -- and where the CTAs are fewer than two an SM and not many share a row:
    // 100 rows of 3000 10.4 -> 9.0 us, 4 rows of 8k 7.7 -> 7.2, but 5 rows of 128k on 16 CTAs each 8.9 -> 9.3)
    const int warps = trials >= 3 || ((long long)rows * C < 2 * kCluSms && C < kCluMaxCtas) ? kCluMaxWarps : 8;
    bool found = shape_cluster(positions, rows, trials, C, warps, bytes, false, s);
    if (N < kStreamMinN) {
        CluShape r;      // a CTA holds the row either way
        if (shape_cluster(positions, rows, trials, C, warps, bytes, true, r) && rows <= kCluSms * resident_ctas(r, 128)) { s = r; found = true; }
    } else {
        const CluCost& c = variant == kVarGiven ? kCostGiven : (variant == kVarDense ? kCostDense : (variant == kVarPrior ? kCostPrior : (trials >= 3 ? kCostManyDraws : kCostFewDraws)));
        const float kept = variant == kVarGiven ? 0.f : fminf(1.f, (float)n / (float)N);
        const int kept_slots = variant == kVarSparse ? 384 : 256;
        // another shape where the rule promises more than it is off by itself
        if (found) s.cost = cost_cluster(c, s, rows, trials, registers, kept, kept_slots);
        float best = found ? 0.95f * s.cost : INFINITY;
        for (int k : {1, 2, 3, 4, 5, 6, 8, 10, 16})
            for (int w = 8; w <= kCluMaxWarps; w += 8)
                for (int roomy = 0; roomy < 2; ++roomy) {
                    CluShape t;
                    if (!shape_cluster(positions, rows, trials, k, w, bytes, roomy != 0, t)) continue;
                    const int regs = roomy ? 128 : registers;
                    if (roomy && rows > rows_at_once(c, t, resident_ctas(t, regs))) continue;      // (measured where one wave holds them)
                    t.cost = cost_cluster(c, t, rows, trials, regs, kept, kept_slots);
                    if (t.cost < best) { best = t.cost; s = t; found = true; }
                }
    }
    return found;
}
// The last few plans of the calling thread: trying all shapes takes the host a microsecond.
static bool plan_cluster(int N, int n, int rows, int trials, size_t es, int variant, bool prior, int lead, CluShape& s) {
    struct Plan { int key[8]; CluShape shape; bool found; };
    static thread_local Plan plans[4] = {};
    static thread_local unsigned next = 0;
    const int key[8] = {N, n, rows, trials, (int)es, variant, prior ? 1 : 0, lead};
    for (const Plan& p : plans)
        if (p.key[0] && !memcmp(p.key, key, sizeof(key))) { s = p.shape; return p.found; }
    Plan& p = plans[next++ & 3u];
    p.found = plan_cluster_anew(N, n, rows, trials, es, variant, prior, lead, p.shape);
    memcpy(p.key, key, sizeof(key));
    s = p.shape;
    return p.found;
}

template <typename TZ, typename TY, int KIND, int VAR, bool PRIOR, bool ROOMY>
static cudaError_t launch_cluster_as(const RowParams& P, CluGeo g, const CluShape& sh, cudaStream_t s) {
    auto kern = rdk_cluster_kernel<TZ, TY, KIND, VAR, PRIOR, ROOMY>;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 64) return cudaErrorNotSupported;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)P.rows * (unsigned)sh.C, 1, 1);
    cfg.blockDim = dim3((unsigned)sh.nw * 32, 1, 1);
    cfg.dynamicSmemBytes = sh.smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)sh.C; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;      // may set itself up while the previous kernel drains
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    // once per kernel, device and cluster size: the limits raised, and whether such a cluster can be resident at all
    static std::atomic<uint32_t> known[64];                       // bit C - 1: asked; bit 16 + C - 1: fits
    const uint32_t bit = (uint32_t)sh.C - 1u;
    uint32_t k = known[dev].load(std::memory_order_acquire);
    if (!(k >> bit & 1u)) {
        e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kCluDynamic);
        if (e != cudaSuccess) return e;
        e = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
        if (e != cudaSuccess) return e;
        cudaLaunchConfig_t q = cfg;
        q.dynamicSmemBytes = kCluDynamic;
        q.numAttrs = 1;
        int fit = 0;
        e = cudaOccupancyMaxActiveClusters(&fit, kern, &q);
        if (e != cudaSuccess) { (void)cudaGetLastError(); fit = 0; }
        k = (1u << bit) | (fit > 0 ? 65536u << bit : 0u);
        k |= known[dev].fetch_or(k, std::memory_order_acq_rel);
    }
    if (!(k >> (16 + bit) & 1u)) return cudaErrorNotSupported;
    return cudaLaunchKernelEx(&cfg, kern, P, g);
}

template <typename TZ, typename TY, int KIND, int VAR, bool PRIOR>
static cudaError_t launch_cluster(const RowParams& P, const CluGeo& g, const CluShape& sh, cudaStream_t s) {
    return sh.roomy ? launch_cluster_as<TZ, TY, KIND, VAR, PRIOR, true>(P, g, sh, s) : launch_cluster_as<TZ, TY, KIND, VAR, PRIOR, false>(P, g, sh, s);
}

template <typename TZ, typename TY, int KIND>
static cudaError_t launch_variant(const RowParams& P, const CluGeo& g, const CluShape& sh, int variant, cudaStream_t s) {
    if (variant == kVarSparse) return launch_cluster<TZ, TY, KIND, kVarSparse, false>(P, g, sh, s);
    if (variant == kVarPrior) return launch_cluster<TZ, TY, KIND, kVarPrior, true>(P, g, sh, s);
    return P.prior ? launch_cluster<TZ, TY, KIND, kVarDense, true>(P, g, sh, s) : launch_cluster<TZ, TY, KIND, kVarDense, false>(P, g, sh, s);
}

template <typename TZ, typename TY>
static cudaError_t launch_kind_c(const RowParams& P, const CluGeo& g, const CluShape& sh, int variant, int kind, cudaStream_t s) {
    return kind == RDK_LOGITS ? launch_variant<TZ, TY, RDK_LOGITS>(P, g, sh, variant, s) : launch_variant<TZ, TY, RDK_PROBS>(P, g, sh, variant, s);
}

// What a linear call of 16-byte aligned rows is expected to take, in us (INFINITY where no shape fits), to be compared with the streaming
// kernels' time: the rule above for the shape that it picks, without its draws (whose term there is fitted to few of them), and those
// anew.  For each round of sixteen trials the turns of the one CTA's warps: a draw each where a segment is one chunk, else two
// chunks at a time, and then a pick each unless every chunk is still in its warp's registers (of several waves of clusters one and
// a half are in their draws at once); and what the draws of an SM's CTAs take of one another.
float cluster_rows_cost(const RowParams& P, size_t es) {
    CluShape sh;
    const int variant = P.prior ? kVarPrior : kVarSparse;
    if (P.N < kStreamMinN || !plan_cluster(P.N, P.n, P.rows, P.trials, es, variant, P.prior != nullptr, 0, sh)) return INFINITY;
    const CluCost& c = P.prior ? kCostPrior : (P.trials >= 3 ? kCostManyDraws : kCostFewDraws);
    const int registers = sh.roomy ? 128 : (P.prior ? 80 : 64), nch = sh.per / 32;
    const float sweep = cost_cluster(c, sh, P.rows, 0, registers, fminf(1.f, (float)P.n / (float)P.N), P.prior ? 256 : 384);
    const float turn = nch == 1 ? 1.6f : 0.94f;
    auto round = [&](int trials) -> float {
        const int draws = 2 * trials, items = draws * nch, each = (draws + sh.nw - 1) / sh.nw;
        if (nch == 1) return turn * (float)each;
        return turn * (float)((items + 2 * sh.nw - 1) / (2 * sh.nw)) + (items > 2 * sh.nw ? 1.94f * (float)each : 0.f);
    };
    const int last = P.trials % kCluRound;
    const float rounds = (float)(P.trials / kCluRound) * round(kCluRound) + (last ? round(last) : 0.f) - turn;      // (one turn is in the sweep's time)
    const float waves = (float)P.rows / (float)rows_at_once(c, sh, resident_ctas(sh, registers));
    const float crowd = (float)P.rows * (float)P.trials / (float)kCluSms - 3.f;
    return sweep + (waves > 1.f ? fminf(waves + c.tail, 1.5f) : 1.f) * rounds + (crowd > 0.f ? 0.33f * sqrtf((float)nch) * crowd : 0.f);
}

cudaError_t launch_cluster_rows(RowParams P, int mode, int tz, int ty, int kind, uint32_t tag, unsigned spin_limit, cudaStream_t s) {
    using B = __nv_bfloat16;
    const size_t es = tz == RDK_F32 ? 4 : 2;
    const int variant = mode == RDK_MODE_PRECOMPUTED_W ? kVarGiven
                        : (P.qtilde || P.N < kStreamMinN ? kVarDense : (P.prior ? kVarPrior : kVarSparse));
    CluShape sh;
    const bool aligned = !(reinterpret_cast<uintptr_t>(P.target) & 15u) && !((P.target_stride * (long long)es) & 15);
    if (!plan_cluster(P.N, P.n, P.rows, P.trials, es, variant, P.prior != nullptr, aligned ? 0 : (int)(16 / es) - 1, sh)) return cudaErrorNotSupported;
    if ((long long)P.rows * sh.C > 0x7fffffffLL) return cudaErrorNotSupported;
    CluGeo g;
    g.per = sh.per;
    const size_t zbytes = (size_t)sh.nw * sh.per * kVec * es;
    g.zoff_p = (uint32_t)zbytes;
    g.zoff_q = (uint32_t)(P.prior ? 2 * zbytes : zbytes);
    g.tag = tag; g.spin_limit = spin_limit ? spin_limit : kCluSpinDefault;
    if (variant == kVarGiven)
        return tz == RDK_F32 ? launch_cluster<float, float, RDK_LOGITS, kVarGiven, false>(P, g, sh, s) : launch_cluster<B, float, RDK_LOGITS, kVarGiven, false>(P, g, sh, s);
    if (tz == RDK_F32) return ty == RDK_F32 ? launch_kind_c<float, float>(P, g, sh, variant, kind, s) : launch_kind_c<float, B>(P, g, sh, variant, kind, s);
    return ty == RDK_F32 ? launch_kind_c<B, float>(P, g, sh, variant, kind, s) : launch_kind_c<B, B>(P, g, sh, variant, kind, s);
}

}  // namespace rdk

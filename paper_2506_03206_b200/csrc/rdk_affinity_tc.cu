// Token-affinity matrix (Eq. symbolic-m with Omega = cosine similarity) for bf16 embeddings and the bf16
// transposed layout, with the dot products on the tensor cores:
//   G[j, i] = <e_j, e_{kappa_i}>                       (bf16 x bf16 products are exact, fp32 accumulation)
//   Mt[j, i] = exp((G[j, i] / (|e_j| |e_{kappa_i}|) - 1) / tau) / Z_i,
//   Z_i = sum_{j in T} exp((G[j, i] / (|e_j| |e_{kappa_i}|) - 1) / tau)
// (the shift by the largest possible cosine, 1, cancels in the quotient).
//
// G is never stored: the embedding dimension is a few hundred, so computing it twice costs the tensor cores less
// (2 x 42 us for 32768 x 8192 x 128) than a round trip of fp32 through HBM.  One kernel runs twice over tiles of
// 128 x 256 dot products, accumulated in tensor memory (two accumulators, so that one is filled while the other is
// read back):
//   kAffSums  : rows = kept ids, columns = tokens.  A thread owns a kept id and adds up its exponentials over blocks of
//               64 tokens; a small kernel adds the blocks in order.
//   kAffWrite : rows = tokens, columns = kept ids.  The same exponential times 1 / Z_i, rounded to bf16, staged in
//               swizzled shared memory and stored by TMA (128-byte rows).
// Both evaluate 2^((G x - 1) scale), x the product of the inverse norms, in the same order of operations, so an entry
// and its share of Z_i carry the same rounding error: where one token has all the weight the entry is 1 however small
// tau is.  (As one exponential of a scaled G less log2 Z the two differ by the rounding of a number of size scale, 1e-6
// of the entry at tau = 0.1, 5e-3 at 1e-5; some ten of 32064 diagonal entries, the heaviest of a row, then land on
// another bf16 number, which moves draws.)
// Both are bound by the special-function unit (one exponential per element and pass: 2 x 60 us at 16 per clock and SM)
// and by the write of the matrix (537 MB: 82 us).  CTAs side by side share an operand tile in either pass, and the epilogue of
// both has sixteen warps with a block of 64 columns each: 277 us for that size (with four tiles in a row to a CTA for the sums and
// eight warps with two store buffers each for the write 288).  Sums of one panel of kept ids and the matrix of
// another in one launch, so that exponentials and stores overlap, were slower: two panels 286, four 311.
#include <math.h>

#include "rdk_device.cuh"
#include "rdk_tc.cuh"

namespace rdk {

constexpr int kAffM = 128, kAffN = 256, kAffK = 64;
constexpr int kAffABytes = kAffM * kAffK * 2, kAffBBytes = kAffN * kAffK * 2;       // 16 KB, 32 KB
constexpr int kAffStage = kAffABytes + kAffBBytes;
constexpr int kAffStages = 3;
// Epilogue warps: sixteen, whose exponentials need the latency hidden (sums alone: 101 us, with eight 118); eight for the write where
// a CTA has one tile (see build_affinity_tc).
constexpr int kAffEpiWarps = 16, kAffFewWarps = 8;
constexpr int kAffStoreBuffers = 16;
constexpr int kAffStoreBytes = 32 * 128;                 // a warp's 32 rows x 64 bf16
constexpr int kAffSmem = kAffStages * kAffStage + kAffStoreBuffers * kAffStoreBytes + 1024;
constexpr int kAffBlock = 64;                            // tokens summed one after the other
static_assert(4 * kAffN / kAffEpiWarps == kAffBlock, "an epilogue warp leaves one sum per tile");
constexpr int aff_threads(int epi) { return 64 + 32 * epi; }
constexpr uint32_t kAffIdesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(kAffN >> 3) << 17) | ((uint32_t)(kAffM >> 4) << 24);

constexpr float kAffZeroInv = 1e12f;                     // inverse norm of a zero embedding
constexpr float kAffTinySum = 0x1p-100f;                 // exponentials this small are rounded, or flushed to zero

enum { kAffSums = 0, kAffWrite = 1 };

struct AffParams {
    int N, n, num_kb;
    int row_tiles, col_tiles;          // sums: kept ids x tokens; write: tokens x kept ids
    const float* row_inv;              // 1 / |e| of the rows and of the columns, zero-padded to whole tiles
    const float* col_inv;
    const float* z;                    // kAffWrite: 1 / Z of every kept id (0: no weight)
    float scale;                       // log2(e) / tau
    float* part;                       // kAffSums: [blocks of kAffBlock tokens][npad]
    int npad;
    int32_t* status;
};

template <int MODE, int EPI>
__global__ void __launch_bounds__(aff_threads(EPI), 1)
aff_tc_kernel(const __grid_constant__ CUtensorMap tmapA, const __grid_constant__ CUtensorMap tmapB, const __grid_constant__ CUtensorMap tmapC, const AffParams P) {
    constexpr bool kWrite = MODE == kAffWrite;
    constexpr int kCols = 4 * kAffN / EPI, kBufs = kAffStoreBuffers / EPI;       // columns and store buffers of an epilogue warp
    extern __shared__ __align__(1024) unsigned char aff_smem[];
    unsigned char* tiles = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(aff_smem) + 1023) & ~uintptr_t(1023));
    __shared__ __align__(8) unsigned long long full_bar[kAffStages], empty_bar[kAffStages], acc_full[2], acc_empty[2];
    __shared__ uint32_t tmem_base_s;
    __shared__ int abort_s;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    volatile int* abort = &abort_s;
    if (threadIdx.x == 0) {
        abort_s = 0;
        for (int s = 0; s < kAffStages; ++s) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(s32(&full_bar[s])));
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(s32(&empty_bar[s])));
        }
        for (int a = 0; a < 2; ++a) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(s32(&acc_full[a])));
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(s32(&acc_empty[a])), "r"(EPI));
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(s32(&tmem_base_s)) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem_base = tmem_base_s;
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

    // Every role walks the same sequence of tiles: blockIdx.x, + gridDim.x, ...  CTAs side by side take the tiles of one row of
    // tiles of the matrix when it is written (whole rows of it are under way then) and those of one column of tiles, the
    // same tokens, for the sums.
    const int num_tiles = P.row_tiles * P.col_tiles;
    auto walk = [&](auto&& tile) {
        for (int j = blockIdx.x; j < num_tiles; j += gridDim.x) {
            const int row = kWrite ? j / P.col_tiles : j % P.row_tiles, col = kWrite ? j % P.col_tiles : j / P.row_tiles;
            if (!tile(row * kAffM, col * kAffN)) return;
        }
    };
    if (warp == 0) {
        int stage = 0;
        uint32_t phase = 0;
        walk([&](int row, int col) -> bool {
            for (int kb = 0; kb < P.num_kb; ++kb) {
                if (!tc_wait(&empty_bar[stage], phase ^ 1u, abort)) return false;
                if (elect_one()) {
                    const uint32_t sa = s32(tiles + stage * kAffStage), bar = s32(&full_bar[stage]);
                    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"((uint32_t)kAffStage) : "memory");
                    asm volatile("cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
                                 ::"r"(sa), "l"(reinterpret_cast<uint64_t>(&tmapA)), "r"(kb * kAffK), "r"(row), "r"(bar) : "memory");
                    asm volatile("cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
                                 ::"r"(sa + kAffABytes), "l"(reinterpret_cast<uint64_t>(&tmapB)), "r"(kb * kAffK), "r"(col), "r"(bar) : "memory");
                }
                __syncwarp();
                if (++stage == kAffStages) { stage = 0; phase ^= 1u; }
            }
            return true;
        });
    } else if (warp == 1) {
        const uint64_t adesc0 = smem_desc(s32(tiles));
        int stage = 0, acc = 0;
        uint32_t phase = 0, acc_phase = 0;
        walk([&](int, int) -> bool {
            if (!tc_wait(&acc_empty[acc], acc_phase ^ 1u, abort)) return false;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            for (int kb = 0; kb < P.num_kb; ++kb) {
                if (!tc_wait(&full_bar[stage], phase, abort)) return false;
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                if (elect_one()) {
                    const uint64_t ad = adesc0 + (uint64_t)(stage * (kAffStage >> 4));
                    mma_kblock<1>(tmem_base + (uint32_t)(acc * kAffN), ad, ad + (kAffABytes >> 4), kAffIdesc, kb > 0);
                    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(s32(&empty_bar[stage])) : "memory");
                }
                __syncwarp();
                if (++stage == kAffStages) { stage = 0; phase ^= 1u; }
            }
            if (lane == 0)
                asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(s32(&acc_full[acc])) : "memory");
            __syncwarp();
            if (++acc == 2) { acc = 0; acc_phase ^= 1u; }
            return true;
        });
    } else {
        const int quarter = warp & 3, share = (warp - 2) >> 2;       // TMEM lanes 32 quarter .. + 32, columns kCols share .. + kCols
        const uint32_t taddr0 = tmem_base + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(share * kCols);
        const uint32_t store0 = s32(tiles + kAffStages * kAffStage + (warp - 2) * kBufs * kAffStoreBytes);
        int acc = 0, buf = 0;
        uint32_t acc_phase = 0;
        const float2 sc = splat(P.scale), neg = splat(-1.f);
        walk([&](int row0, int col0) -> bool {
            const int row = row0 + quarter * 32 + lane, c0 = col0 + share * kCols;
            const float2 ri = splat(__ldg(P.row_inv + row));
            // 2^((G x - 1) scale) of two columns
            auto weight2 = [&](uint32_t g0, uint32_t g1, float k0, float k1) -> float2 {
                return ex2_2(fmul2(ffma2(make_float2(__uint_as_float(g0), __uint_as_float(g1)), fmul2(make_float2(k0, k1), ri), neg), sc));
            };
            if (!tc_wait(&acc_full[acc], acc_phase, abort)) return false;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            float sum = 0.f;
            uint32_t v[2][32];
            tmem_ld32(taddr0 + (uint32_t)(acc * kAffN), v[0]);
#pragma unroll
            for (int c = 0; c < kCols / 32; ++c) {
                if (kWrite && (c & 1) == 0) {                        // the buffer's last store has been read
                    if (lane == 0) asm volatile("cp.async.bulk.wait_group.read %0;" ::"n"(kBufs - 1) : "memory");
                    __syncwarp();
                }
                tmem_wait_ld(v[c & 1]);
                uint32_t (&x)[32] = v[c & 1];
                if (c < kCols / 32 - 1) {
                    tmem_ld32(taddr0 + (uint32_t)(acc * kAffN + (c + 1) * 32), v[(c + 1) & 1]);
                } else {                                             // the accumulator is in registers: the next tile may have it
                    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                    __syncwarp();
                    if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(s32(&acc_empty[acc])) : "memory");
                }
                const int col = c0 + c * 32;
                const float4* ci = reinterpret_cast<const float4*>(P.col_inv + col);
                if (!kWrite) {
#pragma unroll
                    for (int q = 0; q < 8; ++q) {
                        const float4 k4 = __ldg(ci + q);
                        float2 e0 = weight2(x[4 * q], x[4 * q + 1], k4.x, k4.y), e1 = weight2(x[4 * q + 2], x[4 * q + 3], k4.z, k4.w);
                        if (col + 32 > P.N) {                        // tokens beyond the vocabulary have no weight
                            const int left = P.N - col - 4 * q;
                            if (left < 1) e0.x = 0.f;
                            if (left < 2) e0.y = 0.f;
                            if (left < 3) e1.x = 0.f;
                            if (left < 4) e1.y = 0.f;
                        }
                        sum += e0.x; sum += e0.y; sum += e1.x; sum += e1.y;
                    }
                } else {
                    const float4* cz = reinterpret_cast<const float4*>(P.z + col);
                    const uint32_t rowaddr = store0 + (uint32_t)(buf * kAffStoreBytes) + (uint32_t)lane * 128u;
#pragma unroll
                    for (int q = 0; q < 8; q += 2) {
                        uint32_t w[4];
#pragma unroll
                        for (int h = 0; h < 2; ++h) {
                            const float4 k4 = __ldg(ci + q + h), z4 = __ldg(cz + q + h);
                            const int i = 4 * (q + h);
                            const float2 e0 = fmul2(weight2(x[i], x[i + 1], k4.x, k4.y), make_float2(z4.x, z4.y));
                            const float2 e1 = fmul2(weight2(x[i + 2], x[i + 3], k4.z, k4.w), make_float2(z4.z, z4.w));
                            asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(w[2 * h]) : "f"(e0.y), "f"(e0.x));
                            asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(w[2 * h + 1]) : "f"(e1.y), "f"(e1.x));
                        }
                        // 16-byte chunk (c & 1) * 4 + q / 2 of the row, at its place in the 128-byte swizzle
                        const uint32_t chunk = (uint32_t)((c & 1) * 4 + q / 2) ^ (uint32_t)(lane & 7);
                        asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(rowaddr + chunk * 16u), "r"(w[0]), "r"(w[1]), "r"(w[2]), "r"(w[3]) : "memory");
                    }
                    if (c & 1) {                                     // 64 columns are complete (read while the next are evaluated)
                        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                        __syncwarp();
                        if (lane == 0) {
                            const int x0 = c0 + (c >> 1) * 64, y0 = row0 + quarter * 32;
                            if (x0 < P.n && y0 < P.N)
                                asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.tile.bulk_group [%0, {%1, %2}], [%3];"
                                             ::"l"(reinterpret_cast<uint64_t>(&tmapC)), "r"(x0), "r"(y0), "r"(store0 + (uint32_t)(buf * kAffStoreBytes)) : "memory");
                            asm volatile("cp.async.bulk.commit_group;" ::: "memory");
                        }
                        if (++buf == kBufs) buf = 0;
                    }
                }
            }
            if (!kWrite) P.part[(long long)(c0 / kAffBlock) * P.npad + row] = sum;
            if (++acc == 2) { acc = 0; acc_phase ^= 1u; }
            return true;
        });
        if (kWrite && lane == 0) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    // after a wait that gave up (none can any more), copies may still be on their way into shared memory: let them land (bounded as well)
    if (abort_s && warp == 0)
        for (int s = 0; s < kAffStages; ++s)
            for (unsigned spins = 0; spins < (1u << 12); ++spins) __nanosleep(100);
    if (warp == 1) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem_base) : "memory");
    }
    if (threadIdx.x == 0 && abort_s && P.status) atomicCAS(P.status, 0, (int)RDK_ERR_TIMEOUT);
}

// One warp per row: rows [0, Npad) are tokens, inv[t] = 1 / max(|e_t|, 1e-12) (0 beyond the vocabulary) and, where
// Epad is given, the embedding copied to rows of dpad elements; rows [Npad, Npad + npad) are kept ids, their embedding
// gathered into Ek and its inverse norm into invk (zeros for an id outside [0, N) and beyond the last).
__global__ void __launch_bounds__(256)
aff_rows_kernel(const __nv_bfloat16* __restrict__ E, long long stride, const int32_t* __restrict__ ids, __nv_bfloat16* __restrict__ Epad,
                float* __restrict__ inv, __nv_bfloat16* __restrict__ Ek, float* __restrict__ invk, int32_t* status,
                int N, int Npad, int n, int npad, int d, int dpad, bool vec) {
    const int r = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    if (r == 0 && lane == 0) *status = 0;
    if (r >= Npad + npad) return;
    const bool kept = r >= Npad;
    const int i = kept ? r - Npad : r;
    int t = kept ? (i < n ? ids[i] : -1) : (i < N ? i : -1);
    if (t >= N) t = -1;
    __nv_bfloat16* copy = kept ? (i < n ? Ek + (long long)i * dpad : nullptr) : (Epad && i < N ? Epad + (long long)i * dpad : nullptr);
    float ss = 0.f;
    const __nv_bfloat16* row = E + (long long)max(t, 0) * stride;
    for (int k = lane; k < d; k += 32) { const float v = t >= 0 ? __bfloat162float(row[k]) : 0.f; ss = fmaf(v, v, ss); }
    if (copy && vec) {                    // 16-byte aligned rows of a multiple of 8 elements
        for (int k = lane * 8; k < d; k += 256) *reinterpret_cast<uint4*>(copy + k) = t >= 0 ? __ldg(reinterpret_cast<const uint4*>(row + k)) : make_uint4(0u, 0u, 0u, 0u);
    } else if (copy) {
        for (int k = lane; k < dpad; k += 32) copy[k] = t >= 0 && k < d ? row[k] : __float2bfloat16_rn(0.f);
    }
    ss = warp_sum(ss);
    if (lane == 0) (kept ? invk : inv)[i] = t >= 0 ? 1.f / fmaxf(sqrtf(ss), 1e-12f) : 0.f;
}

// z[i] = 1 / Z_i, the blocks' sums added in order; 0 where the kept id has no token, and where a zero embedding (equally
// near to every token) leaves sums too small to count.  32 ids to a CTA: its warps fetch the sums of 64 blocks at a time into
// shared memory, one of them adds them up while the next are on their way.
__global__ void __launch_bounds__(256)
aff_norm_kernel(const float* __restrict__ part, const float* __restrict__ invk, float* __restrict__ z, int blocks, int npad) {
    __shared__ float tile[2][64][32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, i = blockIdx.x * 32 + lane;
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    float v[8], s = 0.f;
    auto fetch = [&](int b0) {
#pragma unroll
        for (int k = 0; k < 8; ++k) v[k] = b0 + warp * 8 + k < blocks ? part[(long long)(b0 + warp * 8 + k) * npad + i] : 0.f;
    };
    fetch(0);
    for (int b0 = 0, buf = 0; b0 < blocks; b0 += 64, buf ^= 1) {
#pragma unroll
        for (int k = 0; k < 8; ++k) tile[buf][warp * 8 + k][lane] = v[k];
        fetch(b0 + 64);
        __syncthreads();                  // (the tile before this one has been added up)
        if (warp == 0) {
#pragma unroll 16
            for (int k = 0; k < 64; ++k) s += tile[buf][k][lane];
        }
    }
    if (warp == 0) {
        const float ik = invk[i];
        z[i] = ik > 0.f && !(ik >= kAffZeroInv && s < kAffTinySum) ? 1.f / s : 0.f;
    }
}

// Last: the columns of zero embeddings whose sums were too small to count, 1 / N each (a warp to a kept id; rare).  And if a
// wait inside the tensor-core kernel ran out, the matrix is incomplete: make that impossible to miss.
__global__ void __launch_bounds__(256)
aff_finish_kernel(const int32_t* status, const float* __restrict__ invk, const float* __restrict__ z, __nv_bfloat16* Mt, long long ld, int n, int N) {
    const int i = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    asm volatile("griddepcontrol.wait;" ::: "memory");
    if (i < n && invk[i] >= kAffZeroInv && z[i] == 0.f)
        for (int j = lane; j < N; j += 32) Mt[(long long)j * ld + i] = __float2bfloat16_rn(1.f / (float)N);
    __syncwarp();
    if (i == 0 && lane == 0 && *status != 0) Mt[0] = __float2bfloat16_rn(NAN);
}

// ------------------------------------------------------------------------------------------------
// host side
// ------------------------------------------------------------------------------------------------
// workspace: inv[Npad] | invk[npad] | z[npad] | status | Ek[n, dpad] bf16 | part[blocks, npad] | Epad[N, dpad] bf16
struct AffTcLayout { size_t inv, invk, z, status, Ek, part, Epad, total; int Npad, npad, dpad, blocks; };
static AffTcLayout aff_tc_layout(int N, int n, int d) {
    AffTcLayout L;
    L.Npad = (N + kAffN - 1) / kAffN * kAffN;
    L.npad = (n + kAffN - 1) / kAffN * kAffN;
    L.dpad = (d + 7) & ~7;
    L.blocks = L.Npad / kAffBlock;
    size_t o = 0;
    L.inv = o;    o += idx_align((size_t)L.Npad * sizeof(float));
    L.invk = o;   o += idx_align((size_t)L.npad * sizeof(float));
    L.z = o;      o += idx_align((size_t)L.npad * sizeof(float));
    L.status = o; o += idx_align(sizeof(int32_t));
    L.Ek = o;     o += idx_align((size_t)n * L.dpad * sizeof(__nv_bfloat16));
    L.part = o;   o += idx_align((size_t)L.blocks * L.npad * sizeof(float));
    L.Epad = o;   o += idx_align((size_t)N * L.dpad * sizeof(__nv_bfloat16));
    L.total = o;
    return L;
}

size_t affinity_tc_workspace_bytes(int N, int n, int d) { return aff_tc_layout(N, n, d).total; }

// whether the tensor-core route serves this call (the other route serves everything)
bool affinity_tc_eligible(const void* embeddings, int emb_dtype, int layout) {
    return emb_dtype == RDK_BF16 && layout == RDK_AFF_BF16_COLS && (reinterpret_cast<uintptr_t>(embeddings) & 1u) == 0;
}

template <typename K, typename... A>
static cudaError_t launch_pdl(K kern, unsigned grid, unsigned block, size_t smem, cudaStream_t s, A... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid, 1, 1);
    cfg.blockDim = dim3(block, 1, 1);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, args...);
}

int build_affinity_tc(const __nv_bfloat16* E, int d, long long estride, const int32_t* ids, int n, int N, float tau,
                      __nv_bfloat16* Mt, long long ld, void* ws, cudaStream_t s) {
    const AffTcLayout L = aff_tc_layout(N, n, d);
    unsigned char* base = static_cast<unsigned char*>(ws);
    float* inv = reinterpret_cast<float*>(base + L.inv);
    float* invk = reinterpret_cast<float*>(base + L.invk);
    float* z = reinterpret_cast<float*>(base + L.z);
    int32_t* status = reinterpret_cast<int32_t*>(base + L.status);
    __nv_bfloat16* Ek = reinterpret_cast<__nv_bfloat16*>(base + L.Ek);
    float* part = reinterpret_cast<float*>(base + L.part);
    const float scale = kLog2e / tau;
    // TMA reads rows of whole 16-byte units: others are copied to padded rows along with the norms
    const bool rows16 = (estride % 8) == 0 && (reinterpret_cast<uintptr_t>(E) & 15u) == 0;
    __nv_bfloat16* Epad = rows16 ? nullptr : reinterpret_cast<__nv_bfloat16*>(base + L.Epad);
    const int wpb = 8;
    RDK_CUDA(launch_pdl(aff_rows_kernel, (unsigned)((L.Npad + L.npad + wpb - 1) / wpb), 256u, 0, s, E, estride, ids, Epad, inv, Ek, invk, status,
                        N, L.Npad, n, L.npad, d, L.dpad, rows16 && d % 8 == 0));
    const __nv_bfloat16* Et = rows16 ? E : Epad;
    const long long et_stride = rows16 ? estride : L.dpad;
    CUtensorMap tokA, tokB, keptA, keptB, out;
    int st;
    if ((st = make_map(&tokA, Et, (uint64_t)d, (uint64_t)N, (uint64_t)et_stride, kAffK, kAffM)) != RDK_OK) return st;
    if ((st = make_map(&tokB, Et, (uint64_t)d, (uint64_t)N, (uint64_t)et_stride, kAffK, kAffN)) != RDK_OK) return st;
    if ((st = make_map(&keptA, Ek, (uint64_t)d, (uint64_t)n, (uint64_t)L.dpad, kAffK, kAffM)) != RDK_OK) return st;
    if ((st = make_map(&keptB, Ek, (uint64_t)d, (uint64_t)n, (uint64_t)L.dpad, kAffK, kAffN)) != RDK_OK) return st;
    if ((st = make_map(&out, Mt, (uint64_t)n, (uint64_t)N, (uint64_t)ld, 64, 32)) != RDK_OK) return st;
    int dev = 0, sms = 0;
    RDK_CUDA(cudaGetDevice(&dev));
    RDK_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    // the write: small CTAs where each has one tile, which it then starts the sooner; sixteen warps where they have many
    auto sums_kernel = aff_tc_kernel<kAffSums, kAffEpiWarps>;
    const bool few = (long long)(L.npad / kAffN) * (L.Npad / kAffM) <= sms;
    auto write_kernel = few ? aff_tc_kernel<kAffWrite, kAffFewWarps> : aff_tc_kernel<kAffWrite, kAffEpiWarps>;
    RDK_CUDA(cudaFuncSetAttribute(sums_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kAffSmem));
    RDK_CUDA(cudaFuncSetAttribute(write_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kAffSmem));
    AffParams P;
    P.N = N; P.n = n; P.num_kb = (d + kAffK - 1) / kAffK; P.scale = scale; P.status = status; P.part = part; P.npad = L.npad; P.z = z;
    const long long tiles = (long long)(L.npad / kAffM) * (L.Npad / kAffN);       // of either pass
    if (tiles > 0x7fffffffLL) { set_error("rdk_build_affinity: too many tiles"); return RDK_ERR_UNSUPPORTED; }
    const unsigned grid = (unsigned)(tiles < sms ? tiles : sms);
    P.row_tiles = L.npad / kAffM; P.col_tiles = L.Npad / kAffN; P.row_inv = invk; P.col_inv = inv;
    RDK_CUDA(launch_pdl(sums_kernel, grid, (unsigned)aff_threads(kAffEpiWarps), (size_t)kAffSmem, s, keptA, tokB, out, P));
    RDK_CUDA(launch_pdl(aff_norm_kernel, (unsigned)(L.npad / 32), 256u, 0, s, (const float*)part, (const float*)invk, z, L.blocks, L.npad));
    P.row_tiles = L.Npad / kAffM; P.col_tiles = L.npad / kAffN; P.row_inv = inv; P.col_inv = invk;
    RDK_CUDA(launch_pdl(write_kernel, grid, (unsigned)aff_threads(few ? kAffFewWarps : kAffEpiWarps), (size_t)kAffSmem, s, tokA, keptB, out, P));
    RDK_CUDA(launch_pdl(aff_finish_kernel, (unsigned)((n + wpb - 1) / wpb), 256u, 0, s, (const int32_t*)status, (const float*)invk, (const float*)z, Mt, ld, n, N));
    return RDK_OK;
}

}  // namespace rdk

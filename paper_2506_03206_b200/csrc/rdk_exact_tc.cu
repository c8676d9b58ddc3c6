// Exact redistribution on the tensor cores (Algorithm 1 step 2):  w = q' M,  i.e.
//   w[r, j] = sum_i Mt[j, i] A[r, i]
// with A = q' (bf16, [rows, K = n], contraction index contiguous) and Mt = the transposed affinity
// matrix (bf16, [N, K]); products accumulate in fp32.
//
// The vocabulary takes the M side of the instruction, the rows the N side, which comes in steps of 16: 20 rows cost the
// tensor cores 32, not 256, and 320 rows cost 320.  A persistent pair of CTAs (cta_group::2, one CTA per SM) computes a
// work item of 256 tokens x up to 512 rows: each CTA holds its own 128 tokens of Mt and half of the rows of A per 64-wide
// K block, and the 128 x (T R) fp32 accumulators of its tokens in tensor memory (T = 1 or 2 instructions of R rows).
// Both operands of a pair are fetched once, so a K block of 512 rows needs 48 KB per CTA for 128 x 512 x 64 products;
// a CTA by itself with a 256 x 256 tile needs 64 KB, and what an SM can keep in flight bounded it (1024 rows x 32k:
// 374 us; 320 rows x 128k in padded tiles of 256 rows 3140 us).
//   warp 0   : TMA producer of its CTA   (128-byte swizzle, out-of-range rows and columns read 0; completion is counted
//              on the leader's barrier)
//   warp 1   : in the leader CTA the MMA issuer; in both the owner of the TMEM allocation
//   warps 2-9: epilogue: a lane is a token, a column a row of w, so a warp stores 32 consecutive tokens per row;
//              row sums by a butterfly over the lanes, kept in registers while the CTA's items are of the same rows
//              (in shared memory where they are not); the four warps of a column are added up at the end: one atomic
//              per row and CTA.  (One per row, warp and item put 4008 fp32 additions behind each other for 128256
//              tokens: S off by 8e-7, now 1.6e-7.)
// Items are ordered so that the row tiles of one 256-token panel of Mt run at the same time: the
// panel is fetched from HBM once and shared through L2.
// Every wait is bounded; on expiry the CTA flags RDK_ERR_TIMEOUT in the status word and winds down.
#include <atomic>

#include "rdk_tc.cuh"

namespace rdk {

constexpr int kVoc = 128;                // most tokens of one CTA: its half of the instruction's M
constexpr int kBK = 64;                  // K block: 64 bf16 = 128 bytes = one swizzle row
constexpr int kVocBytes = kVoc * kBK * 2;        // 16 KB
constexpr int kTcMaxStages = 12;
constexpr int kTcSumRows = 8192;         // most rows with a sum in shared memory
constexpr int kTcMaxRows = 512;          // rows of an item: the columns of the accumulators
constexpr int kTcSmem = 227 * 1024 - 2048;       // for the ring, alignment included
constexpr int kTcEpiWarps = 8;
constexpr int kTcThreads = 64 + 32 * kTcEpiWarps;

struct TcParams {
    float* w; float* S; int rows, N;
    int R, T;                        // rows of one instruction, instructions per item
    int voc;                         // tokens of one CTA, a multiple of 8
    int tiles_r, num_kb, stages;
    int sum_rows;                    // rows with a sum in shared memory behind the ring: all, or 0
    int full_items, num_items;       // items [0, full_items) are whole, the rest halves (one instruction of R rows)
    int32_t* status_word;
};

// Work item -> token tile, first row, instructions.  The last partial round of items is cut into halves so that it
// costs half a round instead of a whole one.
__device__ __forceinline__ void decode_item(const TcParams& P, int item, int& tv, int& row0, int& t) {
    int tile = item, half = 0;
    t = P.T;
    if (item >= P.full_items) { tile = P.full_items + ((item - P.full_items) >> 1); half = (item - P.full_items) & 1; t = 1; }
    tv = tile / P.tiles_r;
    row0 = (tile % P.tiles_r) * P.T * P.R + half * P.R;
    if (row0 >= P.rows) t = 0;                           // a half beyond the last row
    else if (t == 2 && row0 + P.R >= P.rows) t = 1;
}

__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kTcThreads, 1)
exact_tc_kernel(const __grid_constant__ CUtensorMap tmapV, const __grid_constant__ CUtensorMap tmapR, const TcParams P) {
    extern __shared__ __align__(1024) unsigned char tc_smem[];
    const uint32_t ring = (s32(tc_smem) + 1023u) & ~1023u;               // the same offset in both CTAs
    float* row_sums = reinterpret_cast<float*>(tc_smem + (ring - s32(tc_smem)) + (size_t)P.stages * (size_t)(kVocBytes + P.T * P.R * kBK));
    for (int r = threadIdx.x; r < P.sum_rows; r += kTcThreads) row_sums[r] = 0.f;
    float (*tc_sums)[kTcMaxRows] = reinterpret_cast<float (*)[kTcMaxRows]>(tc_smem);      // [4 quarters], at the end of the kernel
    __shared__ __align__(8) unsigned long long full_bar[kTcMaxStages], empty_bar[kTcMaxStages], acc_full, acc_empty;
    __shared__ uint32_t tmem_base_s;
    __shared__ int abort_s, sum_row0_s;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    volatile int* abort = &abort_s;
    uint32_t rank;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
    const bool leader = rank == 0;

    if (threadIdx.x == 0) {
        abort_s = 0;
        sum_row0_s = -1;
        for (int s = 0; s < P.stages; ++s) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(s32(&full_bar[s])));
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(s32(&empty_bar[s])));
        }
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(s32(&acc_full)));
        asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(s32(&acc_empty)), "r"(2 * kTcEpiWarps));
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(s32(&tmem_base_s)) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("barrier.cluster.arrive.release.aligned;\n barrier.cluster.wait.acquire.aligned;" ::: "memory");
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem_base = tmem_base_s;
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

    const int pair = blockIdx.x >> 1, pairs = gridDim.x >> 1;
    const uint32_t rbytes = (uint32_t)(P.R / 2) * kBK * 2;               // this CTA's half of one instruction's rows
    const uint32_t stage_bytes = kVocBytes + (uint32_t)P.T * rbytes;

    if (warp == 0) {
        // ------------------------------------------------------------------ TMA producer
        // Mt is not written by the kernel before this one (the operand kernel lets this one start only after everything
        // before it is complete), so its first blocks are requested before the operand is there.
        int stage = 0; uint32_t phase = 0;
        bool ok = true, waited = false;
        uint32_t full0;                                  // the leader's barriers
        asm volatile("mapa.shared::cluster.u32 %0, %1, 0;" : "=r"(full0) : "r"(s32(&full_bar[0])));
        auto full_addr = [&](int s) -> uint32_t { return full0 + 8u * (uint32_t)s; };
        auto load_voc = [&](int s, int kb, int tv) {
            asm volatile("cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
                         ::"r"(ring + (uint32_t)s * stage_bytes), "l"(reinterpret_cast<uint64_t>(&tmapV)), "r"(kb * kBK),
                           "r"((2 * tv + (int)rank) * P.voc), "r"(full_addr(s)) : "memory");
        };
        auto load_rows = [&](int s, int kb, int row0, int t) {
            for (int k = 0; k < t; ++k)
                asm volatile("cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
                             ::"r"(ring + (uint32_t)s * stage_bytes + kVocBytes + (uint32_t)k * rbytes), "l"(reinterpret_cast<uint64_t>(&tmapR)), "r"(kb * kBK),
                               "r"(row0 + k * P.R + (int)rank * (P.R / 2)), "r"(full_addr(s)) : "memory");
        };
        auto expect = [&](int s, int t) {                // both CTAs' bytes, announced by the leader
            if (leader)
                asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(s32(&full_bar[s])), "r"(2u * ((uint32_t)P.voc * (kBK * 2) + (uint32_t)t * rbytes)) : "memory");
        };
        for (int item = pair; item < P.num_items && ok; item += pairs) {
            int tv, row0, t;
            decode_item(P, item, tv, row0, t);
            if (t == 0) continue;
            int kb = 0;
            if (!waited) {                               // the ring is free: the first item's first blocks
                const int first = min(P.stages, P.num_kb);
                if (lane == 0) for (int s = 0; s < first; ++s) { expect(s, t); load_voc(s, s, tv); }
                __syncwarp();
                asm volatile("griddepcontrol.wait;" ::: "memory");
                if (lane == 0) for (int s = 0; s < first; ++s) load_rows(s, s, row0, t);
                __syncwarp();
                waited = true;
                kb = first;
                stage = first;
                if (stage == P.stages) { stage = 0; phase ^= 1u; }
            }
            for (; kb < P.num_kb; ++kb) {
                if (!tc_wait(&empty_bar[stage], phase ^ 1u, abort)) { ok = false; break; }
                if (elect_one()) { expect(stage, t); load_voc(stage, kb, tv); load_rows(stage, kb, row0, t); }
                __syncwarp();
                if (++stage == P.stages) { stage = 0; phase ^= 1u; }
            }
        }
    } else if (warp == 1) {
        // ------------------------------------------------------------------ MMA issuer (leader only)
        if (leader) {
            const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(P.R >> 3) << 17) | (16u << 24);   // fp32 += bf16 bf16, M = 256, N = R
            // (one thread issues everything: the descriptors are prepared so that an instruction costs it a few adds.  Built
            // anew for every instruction they took 195 to 250 cycles each, whatever the tile, against 128 for 256 rows.)
            const uint64_t vdesc0 = smem_desc(ring);
            const uint32_t dstage = stage_bytes >> 4, empty0 = s32(&empty_bar[0]);
            int stage = 0; uint32_t phase = 0, acc_phase = 0;
            bool ok = true;
            for (int item = pair; item < P.num_items && ok; item += pairs) {
                int tv, row0, t;
                decode_item(P, item, tv, row0, t);
                if (t == 0) continue;
                if (!tc_wait(&acc_empty, acc_phase ^ 1u, abort)) break;       // both epilogues have drained the accumulators
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                for (int kb = 0; kb < P.num_kb; ++kb) {
                    if (!tc_wait(&full_bar[stage], phase, abort)) { ok = false; break; }
                    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                    if (elect_one()) {
                        const uint64_t vd = vdesc0 + (uint64_t)((uint32_t)stage * dstage), rd = vd + (kVocBytes >> 4);
                        mma_kblock<2>(tmem_base, vd, rd, idesc, kb > 0);
                        if (t == 2) mma_kblock<2>(tmem_base + (uint32_t)P.R, vd, rd + (rbytes >> 4), idesc, kb > 0);
                        // frees the stage in both CTAs once the MMAs above have read it
                        asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;"
                                     ::"r"(empty0 + 8u * (uint32_t)stage), "h"((uint16_t)3) : "memory");
                    }
                    __syncwarp();
                    if (++stage == P.stages) { stage = 0; phase ^= 1u; }
                }
                if (!ok) break;
                if (lane == 0)
                    asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;"
                                 ::"r"(s32(&acc_full)), "h"((uint16_t)3) : "memory");
                __syncwarp();
                acc_phase ^= 1u;
            }
        }
    } else {
        // ------------------------------------------------------------------ epilogue
        const int quarter = warp & 3, share = (warp - 2) >> 2;       // TMEM lanes 32 quarter .. + 32; every second block of 32 columns
        uint32_t empty_addr;
        asm volatile("mapa.shared::cluster.u32 %0, %1, 0;" : "=r"(empty_addr) : "r"(s32(&acc_empty)));
        asm volatile("griddepcontrol.wait;" ::: "memory");           // S is zeroed by the kernel before this one
        uint32_t acc_phase = 0;
        constexpr int kBlocks = kTcMaxRows / 64;                     // this warp's blocks of 32 columns
        float sums[kBlocks];                                         // lane q: row sum_row0 + 32 share + 64 k + q
        int sum_row0 = -1;
        auto keep_sums = [&](auto&& put) {
#pragma unroll
            for (int k = 0; k < kBlocks; ++k) { put(k, sums[k]); sums[k] = 0.f; }
        };
        keep_sums([](int, float) {});
        auto hand_over = [&](int k, float v) {
            const int r = sum_row0 + share * 32 + k * 64 + lane;
            if (v != 0.f && r < P.rows) atomicAdd((P.sum_rows ? row_sums : P.S) + r, v);
        };
        for (int item = pair; item < P.num_items; item += pairs) {
            int tv, row0, t;
            decode_item(P, item, tv, row0, t);
            if (t == 0) continue;
            if (P.S && row0 != sum_row0) {                           // other rows: what there is goes to them (while the tensor cores work)
                if (sum_row0 >= 0) keep_sums(hand_over);
                sum_row0 = row0;
            }
            if (!tc_wait(&acc_full, acc_phase, abort)) break;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            // (accumulator lanes beyond the CTA's tokens hold products of whatever lies behind them in the ring)
            const bool held = quarter * 32 + lane < P.voc;
            const int tok = held ? (2 * tv + (int)rank) * P.voc + quarter * 32 + lane : P.N;
            const int cols = t * P.R;
            for (int c = share * 32; c < cols; c += 64) {
                uint32_t v[32];
                tmem_ld32(tmem_base + ((uint32_t)(quarter * 32) << 16) + (uint32_t)c, v);
                tmem_wait_ld(v);
                const int r = row0 + c;
                float* wp = P.w + (long long)r * P.N + tok;
                const int left = min(min(P.rows - r, cols - c), 32);
                if (tok < P.N) {
                    if (left == 32) {
#pragma unroll
                        for (int q = 0; q < 32; ++q) wp[(long long)q * P.N] = __uint_as_float(v[q]);
                    } else {
#pragma unroll
                        for (int q = 0; q < 32; ++q) if (q < left) wp[(long long)q * P.N] = __uint_as_float(v[q]);
                    }
                }
                if (P.S) {
                    // sums over the lanes (tokens beyond the vocabulary are zero): lane q ends up with column q's
                    if (P.voc != kVoc) {
#pragma unroll
                        for (int q = 0; q < 32; ++q) v[q] = held ? v[q] : 0u;
                    }
#pragma unroll
                    for (int s = 16; s > 0; s >>= 1) {
                        const bool up = lane & s;
#pragma unroll
                        for (int q = 0; q < s; ++q) {
                            const float keep = __uint_as_float(up ? v[q + s] : v[q]), send = __uint_as_float(up ? v[q] : v[q + s]);
                            v[q] = __float_as_uint(keep + __shfl_xor_sync(0xffffffffu, send, s));
                        }
                    }
                    const float mine = lane < left ? __uint_as_float(v[0]) : 0.f;
#pragma unroll
                    for (int k = 0; k < kBlocks; ++k) sums[k] += k == c / 64 ? mine : 0.f;
                }
            }
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            __syncwarp();
            if (lane == 0) asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(empty_addr) : "memory");
            acc_phase ^= 1u;
        }
        // every item of the CTA is through the tensor cores: the ring holds nothing that is still needed
        if (P.S && sum_row0 >= 0 && P.sum_rows) {
            keep_sums(hand_over);
        } else if (P.S && sum_row0 >= 0 && !*abort) {
            keep_sums([&](int k, float v) { tc_sums[quarter][share * 32 + k * 64 + lane] = v; });
            if (lane == 0) sum_row0_s = sum_row0;                    // (the same in all eight warps)
        }
    }

    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    // after a wait that gave up (none can any more), copies may still be on their way into shared memory: let them land
    if (abort_s && warp == 0) for (int k = 0; k < 10000; ++k) __nanosleep(100);
    if (sum_row0_s >= 0 && !abort_s)
        for (int c = threadIdx.x; c < kTcMaxRows; c += kTcThreads) {
            const float v = (tc_sums[0][c] + tc_sums[1][c]) + (tc_sums[2][c] + tc_sums[3][c]);
            if (v != 0.f && sum_row0_s + c < P.rows) atomicAdd(P.S + sum_row0_s + c, v);
        }
    for (int r = threadIdx.x; r < P.sum_rows; r += kTcThreads)
        if (row_sums[r] != 0.f) atomicAdd(P.S + r, row_sums[r]);
    // neither CTA leaves, nor gives its tensor memory back, while the other may still signal its barriers or read its operands
    asm volatile("barrier.cluster.arrive.release.aligned;\n barrier.cluster.wait.acquire.aligned;" ::: "memory");
    if (warp == 1) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, 512;" ::"r"(tmem_base) : "memory");
    }
    if (threadIdx.x == 0 && abort_s && P.status_word) atomicCAS(P.status_word, 0, (int)RDK_ERR_TIMEOUT);
}

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                                  const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

int make_map(CUtensorMap* map, const void* base, uint64_t inner, uint64_t outer, uint64_t pitch_elems, uint32_t box_inner, uint32_t box_outer) {
    static std::atomic<EncodeTiledFn> known{nullptr};
    EncodeTiledFn enc = known.load();
    if (!enc) {
        void* fn = nullptr;
        cudaDriverEntryPointQueryResult qres;
        RDK_CUDA(cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &fn, cudaEnableDefault, &qres));
        if (qres != cudaDriverEntryPointSuccess || !fn) {
            set_error("the driver does not provide cuTensorMapEncodeTiled");
            return RDK_ERR_CUDA;
        }
        enc = reinterpret_cast<EncodeTiledFn>(fn);
        known.store(enc);
    }
    const cuuint64_t dims[2] = {inner, outer};
    const cuuint64_t strides[1] = {pitch_elems * 2};
    const cuuint32_t box[2] = {box_inner, box_outer};
    const cuuint32_t estr[2] = {1, 1};
    const CUresult r = enc(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box, estr,
                           CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                           CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) {
        set_error("cuTensorMapEncodeTiled failed with CUresult %d", (int)r);
        return RDK_ERR_CUDA;
    }
    return RDK_OK;
}

// S_out has to be zeroed by the kernel launched just before, which lets this one start early only once everything before
// it is complete.
int launch_exact_tc(const __nv_bfloat16* A, long long lda, const __nv_bfloat16* Mt, long long ldm, float* w_out,
                    float* S_out, int rows, int n, int N, int32_t* status_word, cudaStream_t s) {
    if ((reinterpret_cast<uintptr_t>(A) & 15u) || (lda % 8) || (ldm % 8)) {
        set_error("rdk_redistribute_exact: tensor-core operands need 16-byte aligned rows");
        return RDK_ERR_INVALID_ARG;
    }
    int dev = 0;
    RDK_CUDA(cudaGetDevice(&dev));
    static thread_local int c_dev = -1, sms = 0;
    if (dev != c_dev) {
        RDK_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
        RDK_CUDA(cudaFuncSetAttribute(exact_tc_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kTcSmem));
        c_dev = dev;
    }
    TcParams P;
    P.w = w_out; P.S = S_out; P.rows = rows; P.N = N;
    P.num_kb = (n + kBK - 1) / kBK;
    P.status_word = status_word;
    long long tiles_v = ((long long)N + 2 * kVoc - 1) / (2 * kVoc);
    const int pairs_most = sms / 2;
    // as few row tiles as the 512 accumulator columns allow, more where that leaves pairs without work (down to 64 rows,
    // below which an item is bound by its part of Mt)
    long long tiles_r = (rows + kTcMaxRows - 1) / kTcMaxRows;
    while (tiles_v * tiles_r < pairs_most && rows / tiles_r > 64) ++tiles_r;
    const int per = (int)((rows + tiles_r - 1) / tiles_r);
    P.T = per > 256 ? 2 : 1;
    P.R = P.T == 2 ? ((per + 1) / 2 + 15) / 16 * 16 : (per + 31) / 32 * 32;
    P.tiles_r = (rows + P.T * P.R - 1) / (P.T * P.R);
    const int stage_bytes = kVocBytes + P.T * P.R * kBK;
    // Up to 256 rows the call is the read of Mt, and a last round with few panels reads it with few SMs.  So the panels are made
    // lower than the instruction, as low as leaves every round full; the rest of the instruction's rows are idle (whole calls with
    // the draws: 32 rows x 20011 x 5001 68.5 -> 59.9 us, 16 x 65536 x 16000 359 -> 334, 240 x 50000 x 5000 151 -> 144 to 149, 20 x
    // 32768 x 8192 104.1 -> 102.8).  Not where one round holds all panels: more of them, each with the operand to fetch, were
    // slower (16 x 8192 x 2000 24.6 -> 25.3).
    P.voc = kVoc;
    if (P.tiles_r == 1 && P.T == 1 && tiles_v > pairs_most) {
        const long long rounds = (tiles_v + pairs_most - 1) / pairs_most, per_cta = ((long long)N + 2 * rounds * pairs_most - 1) / (2 * rounds * pairs_most);
        P.voc = (int)((per_cta + 7) / 8 * 8);
        if (P.voc > kVoc) P.voc = kVoc;
        tiles_v = ((long long)N + 2 * P.voc - 1) / (2 * P.voc);
    }
    const long long tiles = tiles_v * P.tiles_r;
    if (tiles > 0x3fffffffLL) { set_error("rdk_redistribute_exact: too many output tiles"); return RDK_ERR_UNSUPPORTED; }
    const int pairs = (int)(tiles < pairs_most ? tiles : pairs_most);
    const int rest = (int)(tiles % pairs);
    const bool split = P.T == 2 && rest > 0 && 2 * rest <= pairs;         // cut the last partial round into halves
    // a pair's items have rows of their own each where the row tiles do not divide the pairs, or in halves
    P.sum_rows = S_out && tiles > pairs && (pairs % P.tiles_r || split) && rows <= kTcSumRows ? rows : 0;
    P.stages = (kTcSmem - 1024 - 4 * P.sum_rows) / stage_bytes;
    if (P.stages > kTcMaxStages) P.stages = kTcMaxStages;
    CUtensorMap mapV, mapR;
    int st = make_map(&mapV, Mt, (uint64_t)n, (uint64_t)N, (uint64_t)ldm, kBK, (uint32_t)P.voc);
    if (st != RDK_OK) return st;
    st = make_map(&mapR, A, (uint64_t)n, (uint64_t)rows, (uint64_t)lda, kBK, (uint32_t)P.R / 2);
    if (st != RDK_OK) return st;
    P.full_items = split ? (int)(tiles - rest) : (int)tiles;
    P.num_items = split ? (int)(tiles + rest) : (int)tiles;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(2u * (unsigned)pairs, 1, 1);
    cfg.blockDim = dim3(kTcThreads, 1, 1);
    cfg.dynamicSmemBytes = (size_t)P.stages * stage_bytes + 1024 + 4 * (size_t)P.sum_rows;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    RDK_CUDA(cudaLaunchKernelEx(&cfg, exact_tc_kernel, mapV, mapR, P));
    return RDK_OK;
}

}  // namespace rdk

// The dense projections of the packed encoder layer (QKV, attention output, MLP) and their gradients on the token matrix
// [T, hidden]; bf16 operands, fp32 accumulation in TMEM.
//   mpipe_linear_fwd    C[M, N]  = epilogue(A[M, K] W[N, K]^T)      both operands K-major
//   mpipe_linear_dgrad  dX[M, K] = epilogue(dY[M, N] W[N, K])       second operand [contraction][output], MN-major
//   mpipe_linear_wgrad  dW[N, K] += dY[M, N]^T X[M, K] in fp32      both operands MN-major (the token index is the contraction);
//                       the token range is split over CTA pairs, partial tiles are added with TMA reduce-add
//
// One kernel, a CTA PAIR (cta_group::2) per 256 x BN output tile: each CTA holds 128 rows of A, half of the BN columns of B and
// 128 x BN of the fp32 result in its TMEM.  What bounds a projection of a full-size microbatch is the tensor pipe, and next to
// it the operand traffic from L2: a 128 x 256 tile on one CTA asks 96 bytes per clock and SM while the pipe runs at its peak, the
// pair 64.  Persistent: pair i takes tiles i, i + pairs, ... (n fastest, so that a wave shares the weight tiles in L2 and walks
// down the token rows together).  Warp roles of each CTA (384 threads):
//   warps 0, 3  TMA producers of the CTA's half, A box [128 rows][64 k] and B box [BN / 2 rows][64 k] (MN-major: boxes of 64
//               columns) per stage, 128-byte swizzle, 3 to 8 stages of 20 to 48 KB; the bytes of both CTAs are counted on the even CTA's barrier
//   warp 1      (even CTA) tcgen05 issuer: 4 x (M 256, N BN, K 16) per stage into one of TWO accumulators of up to 256 columns, so
//               that the epilogue of tile i overlaps the main loop of tile i + 1
//   warp 2      TMEM allocation
//   warps 4-11  epilogue: thread = output row = TMEM lane; the two warpgroups take alternate 64-column chunks.  Every warp owns two
//               [32 rows][64 columns] staging boxes (128-byte swizzle): a side operand (residual, or the pre-activation the
//               gradient of GELU needs) arrives in the box by TMA before the accumulator is ready, the result replaces it in
//               place, and one TMA store takes it out.  No barrier between warps: with one staging box per warpgroup and two
//               named barriers per 32 columns the epilogue of the GELU projections was longer than their main loop.
// A row of a projection is summed over the contraction in one order whatever the number of rows: an image's tokens come out with the same
// bits alone and in any microbatch.  So the contraction is never split over pairs, though two pairs to a tile of a few hundred rows are
// up to 4 us sooner done with an input gradient (300 x 4096 -> 1024 11.2 against 13.8 us; forward of 777 rows 12.5 against 11.7): the
// halves meet in another order than the one accumulator of a large microbatch adds in.
// Measured against the one-CTA 128 x 256 kernel with warpgroup-wide staging that this replaces (us, M = 50 439): fc1 + GELU
// 1024 -> 4096 394 -> 322, its gradient with GELU' 480 -> 374, attention output + residual 120 -> 87, QKV 232 -> 214 (1480
// TFLOP/s), weight gradient 1024 x 4096 345 -> 288, one launch at a time; M = 777: fc2 27.9 -> 11.7, output projection 14.4 -> 7.2, weight
// gradient 1024 x 4096 34 -> 12.
// Every mbarrier wait is bounded (status MPIPE_ERR_TIMEOUT), as in the attention kernels.
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "common.h"
#include "gelu.cuh"
#include "per_device.h"
#include "sm100_ptx.cuh"
#include "tensormap.h"

namespace mpipe {

constexpr int kGemmBM = 128, kGemmBK = 64;                    // rows per CTA (256 per pair), contraction per stage
constexpr int kGemmMaxBN = 256;
// the weight gradient has four more warps, which add up the columns of its first operand (the bias gradient) from the stages
__host__ __device__ constexpr int gemm_threads(int mode) { return mode == 2 ? 512 : 384; }
constexpr int kGemmABytes = kGemmBM * kGemmBK * 2;            // 16 KB
constexpr int kGemmRing = 160 * 1024, kGemmMaxStages = 8;     // 5 stages at BN 256 and 192, 6 at 128, 8 at 64 (of two blocks of the contraction: 3 and 4)
constexpr int kGemmBox = 32 * 128;                            // [32 rows][128 bytes] staging box of one warp
constexpr int kGemmSmemOut = kGemmRing;                       // 8 warps x 2 boxes
constexpr int kGemmSmem = kGemmSmemOut + 8 * 2 * kGemmBox + 1024;
static_assert(kGemmSmem <= 227 * 1024, "shared memory budget");

enum { kEpiPlain = 0, kEpiGelu = 1, kEpiGeluGrad = 2 };

struct GemmParams {
    int32_t M, N, K;
    int32_t bn;                      // columns of a tile: 64, 128, 192 or 256
    int32_t kpb;                     // 64-element blocks of the contraction per stage: 1 or 2 (2: wide only)
    int32_t stages;                  // of kpb * (kGemmABytes + 64 bn) bytes each in the ring
    int32_t wide;                    // map_a / map_w bring all atoms of a stage with one copy (make_tensor_map_chunks)
    int32_t settled_w;               // the second operand was complete before the previous kernel of the stream started
    int32_t tiles_m, tiles_n;
    int32_t splits;                  // weight gradient: parts of the token range
    const __nv_bfloat16* bias;       // [N] or null
    const __nv_bfloat16* direct_res; // [M, ldr] or null: residual read by the epilogue threads (when the boxes carry something else)
    int64_t ldr;
    int32_t side;                    // the side operand of map_s: residual (plain, GELU) or pre-activation (GELU gradient)
    int32_t store_pre;               // GELU only: also store the pre-activation (bf16) through map_u
    const void* ahead[2];            // matrices that the next kernels of the layer read: brought into L2 meanwhile, or null
    uint32_t ahead_bytes[2];
    float* colsum;                   // weight gradient: [M] or null, the column sums of the first operand are added to it
    int32_t* status_buf;
};

struct GemmBarriers {
    uint64_t full[kGemmMaxStages], empty[kGemmMaxStages], done[kGemmMaxStages], acc_full[2], acc_empty[2], side_full[8][2];
};

__device__ __forceinline__ float2 bf16x2_to_f2(uint32_t w) {
    return make_float2(__uint_as_float(w << 16), __uint_as_float(w & 0xffff0000u));
}

// kMode 0: forward, 1: input gradient, 2: weight gradient (see above)
template <int kMode, int kEpi>
__global__ void __launch_bounds__(gemm_threads(kMode), 1)
linear_kernel(const __grid_constant__ CUtensorMap map_a, const __grid_constant__ CUtensorMap map_w,
              const __grid_constant__ CUtensorMap map_c, const __grid_constant__ CUtensorMap map_s,
              const __grid_constant__ CUtensorMap map_u, const GemmParams p) {
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    __shared__ GemmBarriers bars;
    __shared__ uint32_t tmem_base_slot;
    __shared__ int abort_flag;

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int half = int(cluster_ctarank());                  // which 128 rows of A / half of B this CTA holds; 0: the issuing CTA
    if (tid == 0) {
        abort_flag = 0;
        for (int s = 0; s < kGemmMaxStages; ++s) {
            mbar_init(&bars.full[s], 1);
            mbar_init(&bars.empty[s], 1);
            mbar_init(&bars.done[s], 1);
        }
        for (int a = 0; a < 2; ++a) {
            mbar_init(&bars.acc_full[a], 1);
            mbar_init(&bars.acc_empty[a], 16);                // the epilogue warps of both CTAs
        }
        for (int w = 0; w < 8; ++w)
            for (int b = 0; b < 2; ++b) mbar_init(&bars.side_full[w][b], 1);
        fence_mbar_init();
    }
    if (warp == 2) {
        tmem_alloc_pair(&tmem_base_slot, 512);
        tmem_relinquish_pair();
    }
    if (lane == 0) {   // descriptors first: an epilogue that meets a cold one waits a microsecond for it
        if (warp == 0) prefetch_tmap(&map_a);
        if (warp == 3) prefetch_tmap(&map_w);
        if (warp == 4) prefetch_tmap(&map_c);
        if (warp == 5) prefetch_tmap(&map_s);
        if (warp == 6) prefetch_tmap(&map_u);
    }
    __syncwarp();
    tc_fence_before();
    cluster_sync_all();                                       // the peer's barriers exist before anything arrives on them
    tc_fence_after();
    const uint32_t tmem = tmem_base_slot;
    if (kMode != 1 && warp == 2) {   // every CTA a slice, a lane 4 KB at a time
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            constexpr uint32_t kPiece = 4096;
            const uint8_t* src = static_cast<const uint8_t*>(p.ahead[i]);
            const uint32_t bytes = src != nullptr ? p.ahead_bytes[i] : 0u;
            for (uint32_t off = (blockIdx.x * 32u + lane) * kPiece; off < bytes; off += gridDim.x * 32u * kPiece)
                prefetch_l2_bulk(src + off, min(kPiece, bytes - off));
        }
    }
    if (!(warp == 3 && p.settled_w)) pdl_wait();   // weights inside a layer are loaded while the kernel before still runs, a ring of them
    if (warp == 0) pdl_launch();
    const int kpb = kMode == 2 ? 1 : p.kpb, nk = (p.K + kpb * kGemmBK - 1) / (kpb * kGemmBK);   // stages of the whole contraction
    const int n_out_tiles = p.tiles_m * p.tiles_n;
    const int n_items = n_out_tiles * (kMode == 2 ? p.splits : 1);
    const int cid = int(blockIdx.x) / 2, n_clusters = int(gridDim.x) / 2;
    // work item -> output tile and range of contraction blocks (weight gradient: the split index is the slow one, so that the
    // pairs of a wave work on the same token range and share its dY and X rows through L2)
    auto tile_of = [&](int t) { return kMode == 2 ? t % n_out_tiles : t; };
    auto kb_lo_of = [&](int t) { return kMode == 2 ? int((long long)(t / n_out_tiles) * nk / p.splits) : 0; };
    auto kb_hi_of = [&](int t) { return kMode == 2 ? int((long long)(t / n_out_tiles + 1) * nk / p.splits) : nk; };
    // weight gradient: the tiles of one row of tiles all load the row's first operand; block kb of it is summed by tile kb mod tiles_n
    // (by one tile alone, that tile's delayed stages were 4 us of a 26 us launch)
    const bool summing = kMode == 2 && p.colsum != nullptr;
    auto sum_turn = [&](int t, int kb) {   // blocks until the item's next turn, from kb
        const int d = (tile_of(t) % p.tiles_n - kb) % p.tiles_n;
        return d < 0 ? d + p.tiles_n : d;
    };
    const int bn = p.bn, bn_half = bn >> 1;
    const int a_bytes = kpb * kGemmABytes, stage_bytes = a_bytes + kpb * bn_half * kGemmBK * 2, n_stages = p.stages;

    bool left = false;                                        // this warp has arrived at the cluster's last meeting
    if (warp == 0 || warp == 3) {
        // Two producers, one per operand: a thread gets a TMA instruction out every ~90 clocks and a barrier test through in
        // ~110, so one thread issuing both operands' boxes was the slowest role below BN 256 (455 clocks per stage whatever BN)
        // and in the weight gradient, whose stages are four boxes (660).
        if (lane == 0) {
            const bool is_a = warp == 0;
            const uint32_t tx = 2u * uint32_t(stage_bytes);   // both CTAs' boxes; out-of-range elements are zero-filled and still counted
            const uint32_t bar0 = mapa_u32(smem_u32(&bars.full[0]), 0);
            uint32_t s = 0, ph = 1;                           // ring position; parity of the "empty" phase awaited
            bool ok = true;
            for (int t = cid; t < n_items && ok; t += n_clusters) {
                const int m0 = (tile_of(t) / p.tiles_n) * 2 * kGemmBM + half * kGemmBM;
                const int n0 = (tile_of(t) % p.tiles_n) * bn + half * bn_half;
                const int kb_hi = kb_hi_of(t);
                for (int kb = kb_lo_of(t); kb < kb_hi; ++kb) {
                    // early weights: the ring is full, and stages come back when the kernel before this one has ended and not a second later
                    if (!is_a && p.settled_w && ph == 0) pdl_wait();
                    ok = mbar_wait(&bars.empty[s], ph, &abort_flag);
                    if (!ok) break;
                    uint8_t* st = smem + s * stage_bytes;
                    const uint32_t bar = bar0 + s * 8;
                    if (is_a) {
                        if (half == 0) mbar_expect_tx(&bars.full[s], tx);
                        if (p.wide) {
                            if (kMode == 2) tma_load_3d_pair(st, &map_a, bar, 0, kb * kGemmBK, m0 >> 6);
                            else tma_load_3d_pair(st, &map_a, bar, 0, m0, kb * kpb);
                        } else if (kMode == 2) {
#pragma unroll
                            for (int i = 0; i < kGemmBM / 64; ++i)
                                tma_load_3d_pair(st + i * (kGemmBK * 128), &map_a, bar, m0 + 64 * i, 0, kb * kGemmBK);
                        } else {
                            tma_load_3d_pair(st, &map_a, bar, kb * kGemmBK, 0, m0);
                        }
                    } else if (p.wide) {
                        if (kMode == 0) tma_load_3d_pair(st + a_bytes, &map_w, bar, 0, n0, kb * kpb);
                        else tma_load_3d_pair(st + a_bytes, &map_w, bar, 0, kb * kpb * kGemmBK, n0 >> 6);
                    } else if (kMode == 0) {
                        tma_load_3d_pair(st + a_bytes, &map_w, bar, kb * kGemmBK, 0, n0);
                    } else {
                        for (int i = 0; i < bn_half / 64; ++i)
                            tma_load_3d_pair(st + a_bytes + i * (kGemmBK * 128), &map_w, bar, n0 + 64 * i, 0, kb * kGemmBK);
                    }
                    if (++s == uint32_t(n_stages)) { s = 0; ph ^= 1; }
                }
            }
            // the pair's last commits have arrived on this CTA's barriers, which must not be gone by then
            for (int i = 0; is_a && ok && i < n_stages; ++i) {
                ok = mbar_wait(&bars.empty[s], ph, &abort_flag);
                if (++s == uint32_t(n_stages)) { s = 0; ph ^= 1; }
            }
        }
        __syncwarp();
    } else if (warp == 1 && half == 0) {
        const bool leader = elect_one();
        const uint32_t sbase = smem_u32(smem);
        constexpr uint32_t hi128 = umma_desc_hi(1024, kSwizzle128);
        const uint32_t idesc = umma_idesc_bf16(2 * kGemmBM, bn, kMode == 2 ? 1 : 0, kMode != 0 ? 1 : 0);
        constexpr uint16_t pair_mask = 3;
        uint32_t s = 0, ph = 0, tile_it = 0;
        bool ok = true;
        for (int t = cid; t < n_items && ok; t += n_clusters, ++tile_it) {
            const int lo = kb_lo_of(t), hi = kb_hi_of(t);
            if (lo >= hi) { --tile_it; continue; }   // an empty split: no role touches it
            const uint32_t acc = tile_it & 1;
            ok = mbar_wait(&bars.acc_empty[acc], ((tile_it >> 1) & 1) ^ 1, &abort_flag);
            if (!ok) break;
            tc_fence_after();
            int turn = summing ? sum_turn(t, lo) : -1;
            for (int kb = lo; kb < hi; ++kb) {
                const bool mine = turn == 0;
                if (summing) turn = mine ? p.tiles_n - 1 : turn - 1;
                ok = mbar_wait(&bars.full[s], ph, &abort_flag);
                if (!ok) break;
                tc_fence_after();
                // one K-step: 32 bytes along a row (K-major; the next 64 elements are an atom further), or 16 rows of 128 bytes
                // (MN-major; atoms kpb * 8 KB apart)
                const uint32_t a_lo = umma_desc_lo(sbase + s * stage_bytes, kMode == 2 ? kGemmBK * 128 : 0);
                const uint32_t b_lo = umma_desc_lo(sbase + s * stage_bytes + a_bytes, kMode == 0 ? 0 : uint32_t(kpb) * kGemmBK * 128);
                if (leader) {
                    auto block = [&](int kk) {
                        const uint32_t a_kk = a_lo + kk * (kGemmABytes >> 4), b_kk = b_lo + kk * (kMode == 0 ? bn_half * 8 : 4 * 128);
#pragma unroll
                        for (int ks = 0; ks < kGemmBK / 16; ++ks)
                            umma_ss_pair(tmem + acc * kGemmMaxBN, umma_desc(a_kk + ks * (kMode == 2 ? 128 : 2), hi128),
                                         umma_desc(b_kk + ks * (kMode == 0 ? 2 : 128), hi128), idesc, (kb > lo || kk + ks > 0) ? 1u : 0u);
                    };
                    block(0);
                    if (kMode != 2 && kpb == 2) block(1);
                    umma_commit_pair(mine ? &bars.done[s] : &bars.empty[s], pair_mask);   // (then the summing warps free the stage)
                }
                if (++s == uint32_t(n_stages)) { s = 0; ph ^= 1; }
            }
            if (!ok) break;
            if (leader) umma_commit_pair(&bars.acc_full[acc], pair_mask);
        }
        __syncwarp();
    } else if (kMode == 2 && warp >= 12) {
        // Column sums of the first operand: a stage's [64 tokens][128 columns] read once more from shared memory after the MMAs
        // have read it.  A separate pass over dY is 20 to 85 us per projection of a 50 439-token microbatch, this hides beside
        // the main loop (8 x 16 bytes per thread and stage).  No early exit: the four warps meet at a named barrier.
        const int hw = warp - 12;
        const int col = 32 * (hw & 1) + 8 * (lane & 3);                     // this lane's 8 columns of atom hw / 2
        const int row = ((lane >> 2) & 1) * 4 + (lane >> 3);                // of every 8 (neighbouring lanes 4 rows apart: no bank meets twice)
        const uint8_t* src = smem + (hw >> 1) * (kGemmBK * 128) + row * 128 + (((col >> 3) ^ row) << 4);
        uint32_t s = 0, phases = 0;
        bool ok = true;
        for (int t = cid; summing && t < n_items; t += n_clusters) {
            float2 acc[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) acc[j] = make_float2(0.f, 0.f);
            const int kb_lo = kb_lo_of(t), kb_hi = kb_hi_of(t);
            int turn = sum_turn(t, kb_lo);
            const bool any = kb_lo + turn < kb_hi;
            for (int kb = kb_lo; kb < kb_hi; ++kb) {
                if (turn == 0) {
                    if (ok) ok = mbar_wait(&bars.done[s], (phases >> s) & 1, &abort_flag);
                    phases ^= 1u << s;
                    if (ok) {
#pragma unroll
                        for (int i = 0; i < kGemmBK / 8; ++i) {
                            const uint4 q = *reinterpret_cast<const uint4*>(src + s * stage_bytes + i * 1024);
                            acc[0] = add2(acc[0], bf16x2_to_f2(q.x));
                            acc[1] = add2(acc[1], bf16x2_to_f2(q.y));
                            acc[2] = add2(acc[2], bf16x2_to_f2(q.z));
                            acc[3] = add2(acc[3], bf16x2_to_f2(q.w));
                        }
                    }
                    named_barrier_sync(1, 128);
                    if (hw == 0 && lane == 0) mbar_arrive(&bars.empty[s]);
                    turn = p.tiles_n;
                }
                --turn;
                if (++s == uint32_t(n_stages)) s = 0;
            }
            if (!any || !ok) continue;
            const int m = (tile_of(t) / p.tiles_n) * 2 * kGemmBM + half * kGemmBM + 64 * (hw >> 1) + col;
#pragma unroll
            for (int j = 0; j < 4; ++j) {   // over the eight row lanes of a column
#pragma unroll
                for (int o = 4; o <= 16; o <<= 1)
                    acc[j] = add2(acc[j], make_float2(__shfl_xor_sync(0xffffffffu, acc[j].x, o), __shfl_xor_sync(0xffffffffu, acc[j].y, o)));
            }
            if (lane < 4 && m < p.M) {      // M is a multiple of 8
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    atomicAdd(p.colsum + m + 2 * j, acc[j].x);
                    atomicAdd(p.colsum + m + 2 * j + 1, acc[j].y);
                }
            }
        }
    } else if (warp >= 4) {
        const int ew = warp - 4, wg = ew >> 2, quarter = warp & 3;
        const uint32_t lane_base = uint32_t(quarter * 32) << 16;
        uint8_t* boxes = smem + kGemmSmemOut + ew * 2 * kGemmBox;
        uint32_t acc_empty_addr[2] = {mapa_u32(smem_u32(&bars.acc_empty[0]), 0), mapa_u32(smem_u32(&bars.acc_empty[1]), 0)};
        const int n_chunks = bn >> 6;
        uint32_t tile_it = 0, bc = 0;   // bc: boxes used so far by this warp; box = bc & 1
        // Arrive at the last meeting of the cluster as soon as this warp will touch neither TMEM nor the other CTA any more, under
        // the arithmetic and the stores of its last chunk (an arrival behind them kept every CTA about half a microsecond longer).
        auto leave = [&]() {
            if (!left) cluster_arrive();
            left = true;
        };
        bool ok = true;
        for (int t = cid; t < n_items; t += n_clusters, ++tile_it) {
            if (kb_lo_of(t) >= kb_hi_of(t)) { --tile_it; continue; }
            const uint32_t acc = tile_it & 1;
            const uint32_t tacc = tmem + lane_base + acc * kGemmMaxBN;
            const int m0 = (tile_of(t) / p.tiles_n) * 2 * kGemmBM + half * kGemmBM + quarter * 32;   // first row of this warp
            const int n0 = (tile_of(t) % p.tiles_n) * bn;
            const bool rows_in = m0 < p.M;
            // the chunks this warp finishes: wg, wg + 2, ... of the tile
            auto active = [&](int c) { return rows_in && n0 + 64 * c < p.N; };
            if (kMode != 2 && p.side && ok) {   // the side operand of both chunks, before the accumulator is ready
                uint32_t b = bc;
                for (int c = wg; c < n_chunks; c += 2) {
                    if (!active(c)) continue;
                    if (lane == 0) {
                        if (c == wg) bulk_wait_group_read<1>();   // the store that used this box two boxes ago has read it
                        else bulk_wait_group_read<0>();
                        mbar_expect_tx(&bars.side_full[ew][b & 1], kGemmBox);
                        tma_load_3d(boxes + (b & 1) * kGemmBox, &map_s, &bars.side_full[ew][b & 1], n0 + 64 * c, 0, m0);
                    }
                    ++b;
                }
            }
            // The bias of a chunk, asked for a chunk ahead: eight loads that the first use would otherwise wait for one after the
            // other, each as long as a value from L2 or HBM takes (epilogue of one 64-column chunk 1.9 -> 1.2 us; 777 x 1024 -> 3072
            // 12.2 -> 11.4 us, -> 1024 7.7 -> 7.4).
            uint4 bias[8];
            auto load_bias = [&](int c) {
                if (kMode != 0 || p.bias == nullptr || !active(c)) return;
                const int n = n0 + 64 * c;
#pragma unroll
                for (int g = 0; g < 8; ++g)
                    if (n + 8 * g < p.N) bias[g] = __ldg(reinterpret_cast<const uint4*>(p.bias + n + 8 * g));   // (N is a multiple of 8)
            };
            load_bias(wg);
            if (ok) ok = mbar_wait(&bars.acc_full[acc], (tile_it >> 1) & 1, &abort_flag);
            tc_fence_after();
            bool released = false;
            auto release = [&]() {   // this warp has read its part of the accumulator
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive_cluster(acc_empty_addr[acc]);
                released = true;
                if (t + n_clusters >= n_items) leave();
            };
#pragma unroll 1
            for (int c = wg; c < n_chunks; c += 2) {
                const bool last = c + 2 >= n_chunks;
                if (!active(c) || !ok) continue;
                const int n = n0 + 64 * c;
                uint32_t v[64];
                tmem_ld32(tacc + c * 64, *reinterpret_cast<uint32_t(*)[32]>(&v[0]));
                tmem_ld32(tacc + c * 64 + 32, *reinterpret_cast<uint32_t(*)[32]>(&v[32]));
                tmem_wait_ld();
                if (last) release();
                if (kMode == 2) {   // fp32 partial tile, added to the output: two [32 rows][32 fp32] boxes
#pragma unroll
                    for (int h = 0; h < 2; ++h, ++bc) {
                        uint8_t* box = boxes + (bc & 1) * kGemmBox;
                        if (lane == 0) bulk_wait_group_read<1>();
                        __syncwarp();
#pragma unroll
                        for (int g = 0; g < 8; ++g)
                            *reinterpret_cast<uint4*>(box + lane * 128 + ((g ^ (lane & 7)) << 4)) =
                                make_uint4(v[32 * h + 4 * g], v[32 * h + 4 * g + 1], v[32 * h + 4 * g + 2], v[32 * h + 4 * g + 3]);
                        fence_async_smem();
                        __syncwarp();
                        if (lane == 0) {
                            if (n + 32 * h < p.N) tma_reduce_add_3d(&map_c, box, n + 32 * h, 0, m0);
                            bulk_commit_group();
                        }
                    }
                    continue;
                }
                uint8_t* box = boxes + (bc & 1) * kGemmBox;          // result (and side operand, in place)
                uint8_t* pre_box = boxes + ((bc & 1) ^ 1) * kGemmBox; // pre-activation, when it is stored too
                if (p.side) {
                    ok = mbar_wait(&bars.side_full[ew][bc & 1], (bc >> 1) & 1, &abort_flag);
                    if (!ok) continue;
                } else {
                    if (lane == 0) {   // the box's (both boxes') last store has been read
                        if (kEpi == kEpiGelu && p.store_pre) bulk_wait_group_read<0>();
                        else bulk_wait_group_read<1>();
                    }
                    __syncwarp();
                }
                const __nv_bfloat16* rrow = nullptr;
                if (p.direct_res != nullptr && m0 + lane < p.M) rrow = p.direct_res + int64_t(m0 + lane) * p.ldr + n;
#pragma unroll
                for (int g = 0; g < 8; ++g) {   // 8 columns = 16 bytes of output
                    const bool col_ok = n + 8 * g < p.N;   // N is a multiple of 8; the store clips what lies outside
                    uint4* slot = reinterpret_cast<uint4*>(box + lane * 128 + ((g ^ (lane & 7)) << 4));
                    float2 f[4];
#pragma unroll
                    for (int j = 0; j < 4; ++j) f[j] = make_float2(__uint_as_float(v[8 * g + 2 * j]), __uint_as_float(v[8 * g + 2 * j + 1]));
                    if (kMode == 0 && p.bias != nullptr) {
                        const uint32_t bw[4] = {bias[g].x, bias[g].y, bias[g].z, bias[g].w};
#pragma unroll
                        for (int j = 0; j < 4; ++j) f[j] = add2(f[j], bf16x2_to_f2(bw[j]));
                    }
                    if (kEpi == kEpiGelu) {
                        if (p.store_pre)
                            *reinterpret_cast<uint4*>(pre_box + lane * 128 + ((g ^ (lane & 7)) << 4)) =
                                make_uint4(pack_bf16(f[0].x, f[0].y), pack_bf16(f[1].x, f[1].y), pack_bf16(f[2].x, f[2].y), pack_bf16(f[3].x, f[3].y));
#pragma unroll
                        for (int j = 0; j < 4; ++j) f[j] = gelu_erf2(f[j]);   // of the fp32 value, whether or not u is stored
                    }
                    if (p.side) {
                        const uint4 s4 = *slot;
                        const uint32_t sw[4] = {s4.x, s4.y, s4.z, s4.w};
#pragma unroll
                        for (int j = 0; j < 4; ++j)
                            f[j] = kEpi == kEpiGeluGrad ? mul2(f[j], gelu_erf_grad2(bf16x2_to_f2(sw[j]))) : add2(f[j], bf16x2_to_f2(sw[j]));
                    }
                    if (kEpi == kEpiGeluGrad && rrow != nullptr && col_ok) {
                        const uint4 r4 = __ldg(reinterpret_cast<const uint4*>(rrow + 8 * g));
                        const uint32_t rw[4] = {r4.x, r4.y, r4.z, r4.w};
#pragma unroll
                        for (int j = 0; j < 4; ++j) f[j] = add2(f[j], bf16x2_to_f2(rw[j]));
                    }
                    *slot = make_uint4(pack_bf16(f[0].x, f[0].y), pack_bf16(f[1].x, f[1].y), pack_bf16(f[2].x, f[2].y), pack_bf16(f[3].x, f[3].y));
                }
                if (!last) load_bias(c + 2);
                fence_async_smem();
                __syncwarp();
                if (lane == 0) {
                    if (kEpi == kEpiGelu && p.store_pre) tma_store_3d(&map_u, pre_box, n, 0, m0);
                    tma_store_3d(&map_c, box, n, 0, m0);
                    bulk_commit_group();
                }
                ++bc;
            }
            if (!released) release();
        }
        if (lane == 0) bulk_wait_group_read<0>();   // shared memory must outlive the copy engine's reads
        __syncwarp();
    }
    __syncwarp();
    if (!left) {
        tc_fence_before();
        cluster_arrive();
    }
    cluster_wait();       // neither CTA frees TMEM or leaves while the pair's MMAs or arrivals may still touch it
    if (warp == 2) tmem_dealloc_pair(tmem, 512);
    if (tid == 0 && abort_flag) report_status(p.status_buf, MPIPE_ERR_TIMEOUT, int32_t(blockIdx.x));
}

// ---- choice of tile width, in SM clocks; the constants are fitted to graph-replayed sweeps of every width over M 86..12000 and
// hidden 320..1280.
// 64 of the contraction of a 256 x bn tile, by the waves of tiles there are: 2 bn clocks of tensor pipe at bn 256 and 192 plus what
// the other SMs' operand traffic adds; below, first the issuing thread's instructions, then (with every SM loading) that traffic.
static double gemm_stage_clk(int bn, long long waves) {
    if (bn == 256) return 640.0;
    if (bn == 192) return waves <= 1 ? 450.0 : 540.0;
    if (bn == 128) return waves <= 1 ? 320.0 : waves == 2 ? 385.0 : 470.0;
    return waves <= 1 ? 270.0 : 310.0;
}
// Launch, first loads, and the epilogue of the last tile (two 64-column chunks per warp above bn 128; GELU ~2700 a chunk).
static double gemm_fixed_clk(int bn, bool gelu) {
    const double plain = bn == 256 ? 13800.0 : bn == 192 ? 12600.0 : 10600.0;
    return plain + (gelu ? (bn > 128 ? 5200.0 : 2800.0) : 0.0);
}
static int gemm_stages(int bn, int kpb) {
    const int n = kGemmRing / (kpb * (kGemmABytes + 64 * bn));
    return n < kGemmMaxStages ? n : kGemmMaxStages;
}
// CTA pairs that fit on the current device at once.
template <auto kernel>
static int max_pairs(int threads) {
    static PerDevice pairs;
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess) return 0;
    return pairs.get(dev, [&]() {
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(2);
        cfg.blockDim = dim3(unsigned(threads));
        cfg.dynamicSmemBytes = kGemmSmem;
        cudaLaunchAttribute at[1];
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = 2;
        at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
        cfg.attrs = at;
        cfg.numAttrs = 1;
        int n = 0;
        if (cudaOccupancyMaxActiveClusters(&n, kernel, &cfg) == cudaSuccess) return n;
        (void)cudaGetLastError();
        return 0;
    });
}
static int choose_width(int mode, bool gelu, int pairs, int M, int N, int K) {
    const int nk = cdiv(K, kGemmBK), tiles_m = cdiv(M, 2 * kGemmBM);
    int best = kGemmMaxBN;
    double best_clk = 1e30;
    for (int bn = kGemmMaxBN; bn >= 64; bn -= 64) {
        if (mode == 1 && (bn % 128) != 0) continue;        // MN-major B: each CTA holds whole 64-column atoms
        const long long tiles = (long long)tiles_m * cdiv(N, bn), waves = (tiles + pairs - 1) / pairs;
        const double clk = waves * nk * gemm_stage_clk(bn, waves) + 1000.0 * (waves - 1) + gemm_fixed_clk(bn, gelu);
        if (clk < best_clk) {
            best_clk = clk;
            best = bn;
        }
    }
    return best;
}

template <auto kernel>
static int32_t launch_gemm(int threads, int pairs, const CUtensorMap& map_a, const CUtensorMap& map_w, const CUtensorMap& map_c,
                           const CUtensorMap& map_s, const CUtensorMap& map_u, const GemmParams& p, cudaStream_t st) {
    profile_start(kProfileLinear, st);
    const cudaError_t e = launch_kernel(kernel, unsigned(2 * pairs), unsigned(threads), kGemmSmem, st, 2u, map_a, map_w, map_c,
                                        map_s, map_u, p);
    profile_stop(kProfileLinear, st);
    return e == cudaSuccess && cudaGetLastError() == cudaSuccess ? MPIPE_OK : MPIPE_ERR_CUDA;
}

struct LinearCall {   // one forward projection or input gradient
    const void *a, *w, *bias, *residual, *aux;
    void *c, *pre;
    int32_t M, n_out, n_contract;
    int64_t lda, ldw, ldr, ldx, ldc, ldp;
    int32_t gelu;
    int32_t* status_buf;
    bool settled_w;      // see GemmParams
    LayerAhead ahead;    // see GemmParams
};

template <int kMode, int kEpi>
static int32_t launch_linear_as(const LinearCall& x, cudaStream_t st) {
    if (!ensure_dynamic_smem<linear_kernel<kMode, kEpi>>(kGemmSmem)) return MPIPE_ERR_CUDA;
    const int pairs = max_pairs<linear_kernel<kMode, kEpi>>(gemm_threads(kMode));
    if (pairs <= 0) return MPIPE_ERR_CUDA;
    GemmParams p = {};
    p.M = x.M; p.N = x.n_out; p.K = x.n_contract;
    p.bn = choose_width(kMode, kEpi != kEpiPlain, pairs, x.M, x.n_out, x.n_contract);
    // Operands whose 64-element atoms are all whole take one copy per stage; the narrow tiles, whose loop is bound by the
    // producers' and the issuer's instructions and not by the MMAs, then also take two blocks of the contraction per stage
    // (777 x 1024 x 1024 at bn 64: 360 -> 268 clocks per block, 9.1 -> 7.8 us).
    const bool wide = x.n_contract % kGemmBK == 0 && (kMode == 0 || x.n_out % 64 == 0);
    p.wide = wide ? 1 : 0;
    p.kpb = wide && p.bn <= 128 ? 2 : 1;
    p.settled_w = x.settled_w ? 1 : 0;
    for (int i = 0; i < 2; ++i) {
        p.ahead[i] = x.ahead.ptr[i];
        p.ahead_bytes[i] = x.ahead.bytes[i];
    }
    p.stages = gemm_stages(p.bn, p.kpb);
    p.splits = 1;
    p.tiles_m = cdiv(x.M, 2 * kGemmBM);
    p.tiles_n = cdiv(x.n_out, p.bn);
    p.bias = static_cast<const __nv_bfloat16*>(x.bias);
    // the boxes bring one side operand; the gradient of GELU takes them for u and reads a residual directly
    const void* side = kEpi == kEpiGeluGrad ? x.aux : x.residual;
    const int64_t ld_side = kEpi == kEpiGeluGrad ? x.ldx : x.ldr;
    if (kEpi == kEpiGeluGrad) p.direct_res = static_cast<const __nv_bfloat16*>(x.residual);
    p.ldr = x.ldr;
    p.side = side != nullptr ? 1 : 0;
    p.store_pre = x.pre != nullptr ? 1 : 0;
    p.status_buf = x.status_buf;
    CUtensorMap map_a, map_w, map_c;
    bool ok = make_tensor_map_thd(&map_c, x.c, x.M, 1, x.n_out, x.ldc, x.ldc, 64, 32, 128);
    CUtensorMap map_s = map_c, map_u = map_c;
    if (side != nullptr) ok = ok && make_tensor_map_thd(&map_s, side, x.M, 1, x.n_out, ld_side, ld_side, 64, 32, 128);
    if (x.pre != nullptr) ok = ok && make_tensor_map_thd(&map_u, x.pre, x.M, 1, x.n_out, x.ldp, x.ldp, 64, 32, 128);
    // A[M rows, n_contract]: 128 rows.  W forward [n_out rows, n_contract]: bn / 2 rows; gradient [n_contract rows, n_out]: the
    // stage's contraction rows x 64 output columns per atom
    if (wide)
        ok = ok && make_tensor_map_chunks(&map_a, x.a, x.M, x.n_contract / 64, x.lda, kGemmBM, uint32_t(p.kpb)) &&
             (kMode == 0 ? make_tensor_map_chunks(&map_w, x.w, x.n_out, x.n_contract / 64, x.ldw, uint32_t(p.bn / 2), uint32_t(p.kpb))
                         : make_tensor_map_chunks(&map_w, x.w, x.n_contract, x.n_out / 64, x.ldw, uint32_t(p.kpb * kGemmBK), uint32_t(p.bn / 128)));
    else
        ok = ok && make_tensor_map_thd(&map_a, x.a, x.M, 1, x.n_contract, x.lda, x.lda, kGemmBK, kGemmBM, 128) &&
             (kMode == 0 ? make_tensor_map_thd(&map_w, x.w, x.n_out, 1, x.n_contract, x.ldw, x.ldw, kGemmBK, p.bn / 2, 128)
                         : make_tensor_map_thd(&map_w, x.w, x.n_contract, 1, x.n_out, x.ldw, x.ldw, 64, kGemmBK, 128));
    if (!ok) return MPIPE_ERR_CUDA;
    const long long tiles = (long long)p.tiles_m * p.tiles_n;
    if (tiles > 0x7fffffffLL / 2) return MPIPE_ERR_UNSUPPORTED;
    return launch_gemm<linear_kernel<kMode, kEpi>>(gemm_threads(kMode), int(tiles < pairs ? tiles : pairs), map_a, map_w, map_c, map_s, map_u, p, st);
}

// Shared host side of the two entry points: checks, then the instantiation the epilogue needs.
static int32_t launch_linear(int b_mode, const LinearCall& x, void* stream) {
    if (x.M < 0 || x.n_out <= 0 || x.n_contract <= 0) return MPIPE_ERR_INVALID_ARG;
    if (x.M == 0) return MPIPE_OK;
    if (x.a == nullptr || x.w == nullptr || x.c == nullptr) return MPIPE_ERR_INVALID_ARG;
    if ((x.n_out % 8) != 0 || (x.n_contract % 8) != 0) return MPIPE_ERR_UNSUPPORTED;
    const int64_t w_cols = b_mode == 0 ? x.n_contract : x.n_out;
    if (x.lda < x.n_contract || x.ldw < w_cols || x.ldc < x.n_out || (x.residual != nullptr && x.ldr < x.n_out) ||
        (x.aux != nullptr && x.ldx < x.n_out))
        return MPIPE_ERR_INVALID_ARG;
    if ((x.lda % 8) != 0 || (x.ldw % 8) != 0 || (x.ldc % 8) != 0 || (x.residual != nullptr && (x.ldr % 8) != 0) ||
        (x.aux != nullptr && (x.ldx % 8) != 0))
        return MPIPE_ERR_UNSUPPORTED;
    if (!aligned16(x.a) || !aligned16(x.w) || !aligned16(x.c) || !aligned16(x.bias) || !aligned16(x.residual) || !aligned16(x.aux))
        return MPIPE_ERR_UNSUPPORTED;
    // the two outputs of a kept pre-activation take both staging boxes: no residual beside it
    if (x.pre != nullptr && (b_mode != 0 || !x.gelu || x.residual != nullptr || x.ldp < x.n_out || (x.ldp % 8) != 0 || !aligned16(x.pre)))
        return MPIPE_ERR_INVALID_ARG;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    if (b_mode == 0) return x.gelu ? launch_linear_as<0, kEpiGelu>(x, st) : launch_linear_as<0, kEpiPlain>(x, st);
    return x.aux != nullptr ? launch_linear_as<1, kEpiGeluGrad>(x, st) : launch_linear_as<1, kEpiPlain>(x, st);
}

// dW[n_rows, n_cols] (fp32) += dY[tokens, n_rows]^T X[tokens, n_cols]; with db also db[n_rows] += column sums of dY
static int32_t launch_wgrad(const void* dy, const void* x, float* dw, float* db, int32_t tokens, int32_t n_rows, int32_t n_cols, int64_t lddy,
                            int64_t ldx, int64_t lddw, int32_t* status_buf, void* stream, const LayerAhead& ahead) {
    if (tokens < 0 || n_rows <= 0 || n_cols <= 0) return MPIPE_ERR_INVALID_ARG;
    if (tokens == 0) return MPIPE_OK;
    if (dy == nullptr || x == nullptr || dw == nullptr || lddy < n_rows || ldx < n_cols || lddw < n_cols) return MPIPE_ERR_INVALID_ARG;
    if ((n_rows % 8) != 0 || (n_cols % 8) != 0 || (lddy % 8) != 0 || (ldx % 8) != 0 || (lddw % 4) != 0) return MPIPE_ERR_UNSUPPORTED;
    if (!aligned16(dy) || !aligned16(x) || !aligned16(dw)) return MPIPE_ERR_UNSUPPORTED;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    CUtensorMap map_a, map_w, map_c;
    if (!make_tensor_map_thd(&map_c, dw, n_rows, 1, n_cols, lddw, lddw, 32, 32, 128, 4)) return MPIPE_ERR_CUDA;
    if (!ensure_dynamic_smem<linear_kernel<2, kEpiPlain>>(kGemmSmem)) return MPIPE_ERR_CUDA;
    const int pairs = max_pairs<linear_kernel<2, kEpiPlain>>(gemm_threads(2));
    if (pairs <= 0) return MPIPE_ERR_CUDA;
    // Tile width and split of the token range, in SM clocks (fitted like choose_width's constants).  A pair's fp32 tile leaves at
    // about 12 bytes per clock and SM (the L2's rate of fp32 reductions with every SM adding) beside the next item's main loop.
    // A long token range runs into the power limit, where the sum of the work counts and not its spread over the pairs: no
    // estimate goes below the work at 68 % of the tensor peak, and among equals the fewest splits (least reduction traffic) win
    // (1024 x 4096 over 50 439 tokens, back to back under that limit: 322 us unsplit on 64 of the 74 pairs, 355 to 415 us for any split).
    GemmParams p = {};
    const int nk = cdiv(tokens, kGemmBK);
    double best_clk = 1e30;
    for (int bn = kGemmMaxBN; bn >= 128; bn -= 128) {
        const long long tiles = (long long)cdiv(n_rows, 2 * kGemmBM) * cdiv(n_cols, bn);
        const double red = bn == 256 ? 11000.0 : 6500.0, stage = bn == 256 ? 600.0 : 480.0, fixed = bn == 256 ? 14500.0 : 12500.0;
        const double power = double(tiles) * nk * 2 * bn / (0.68 * pairs);
        for (int sp = 1; sp <= 64 && sp <= nk; ++sp) {
            const long long waves = (tiles * sp + pairs - 1) / pairs;
            const double loop = cdiv(nk, sp) * stage, run = waves * ((loop > red ? loop : red) + 1000.0);
            const double clk = (run > power ? run : power) + fixed;
            if (clk < best_clk * 0.999) {
                best_clk = clk;
                p.bn = bn;
                p.splits = sp;
            }
        }
    }
    p.wide = n_rows % 64 == 0 && n_cols % 64 == 0 ? 1 : 0;
    if (p.wide ? !make_tensor_map_chunks(&map_a, dy, tokens, n_rows / 64, lddy, kGemmBK, kGemmBM / 64) ||
                     !make_tensor_map_chunks(&map_w, x, tokens, n_cols / 64, ldx, kGemmBK, uint32_t(p.bn / 128))
               : !make_tensor_map_thd(&map_a, dy, tokens, 1, n_rows, lddy, lddy, 64, kGemmBK, 128) ||
                     !make_tensor_map_thd(&map_w, x, tokens, 1, n_cols, ldx, ldx, 64, kGemmBK, 128))
        return MPIPE_ERR_CUDA;
    p.kpb = 1;
    p.stages = gemm_stages(p.bn, 1);
    p.M = n_rows; p.N = n_cols; p.K = tokens;
    p.tiles_m = cdiv(n_rows, 2 * kGemmBM);
    p.tiles_n = cdiv(n_cols, p.bn);
    p.colsum = db;
    for (int i = 0; i < 2; ++i) {
        p.ahead[i] = ahead.ptr[i];
        p.ahead_bytes[i] = ahead.bytes[i];
    }
    p.status_buf = status_buf;
    const long long items = (long long)p.tiles_m * p.tiles_n * p.splits;
    return launch_gemm<linear_kernel<2, kEpiPlain>>(gemm_threads(2), int(items < pairs ? items : pairs), map_a, map_w, map_c, map_c, map_c, p, st);
}

// Weight and bias gradient of a projection in one launch.
int32_t linear_wgrad_bias(const void* dy, const void* x, float* dw, float* db, int32_t n_tokens, int32_t N, int32_t K, int64_t lddy,
                          int64_t ldx, int64_t lddw, int32_t* status_buf, void* stream, const LayerAhead& ahead) {
    if (db == nullptr && n_tokens > 0) return MPIPE_ERR_INVALID_ARG;
    return launch_wgrad(dy, x, dw, db, n_tokens, N, K, lddy, ldx, lddw, status_buf, stream, ahead);
}

// fc1 of a TRAINED layer forward: act = GELU(a W^T + bias) and pre = a W^T + bias from ONE accumulator, so that the
// activation is computed from the same fp32 value as in the FROZEN forward (freezing changes no forward bit).
int32_t linear_fwd_gelu_keep_preact(const void* a, const void* w, const void* bias, void* act, void* pre, int32_t M, int32_t N,
                                    int32_t K, int64_t lda, int64_t ldw, int64_t ldact, int64_t ldpre, int32_t* status_buf,
                                    void* stream) {
    const LinearCall x = {a, w, bias, nullptr, nullptr, act, pre, M, N, K, lda, ldw, 0, 0, ldact, ldpre, 1, status_buf, true};
    return launch_linear(0, x, stream);
}

// mpipe_linear_fwd / mpipe_linear_dgrad inside a layer, where the weights are older than the kernel before.
int32_t linear_fwd_in_layer(const void* a, const void* w, const void* bias, const void* residual, void* c, int32_t M, int32_t N, int32_t K,
                            int64_t lda, int64_t ldw, int64_t ldr, int64_t ldc, int32_t flags, int32_t* status_buf, void* stream,
                            const LayerAhead& ahead) {
    const LinearCall x = {a, w, bias, residual, nullptr, c, nullptr, M, N, K, lda, ldw, ldr, 0, ldc, 0,
                          (flags & MPIPE_LINEAR_GELU) ? 1 : 0, status_buf, true, ahead};
    return launch_linear(0, x, stream);
}
int32_t linear_dgrad_in_layer(const void* dy, const void* w, const void* gelu_input, void* dx, int32_t M, int32_t N, int32_t K, int64_t lddy,
                              int64_t ldw, int64_t ldu, int64_t lddx, int32_t* status_buf, void* stream) {
    const LinearCall x = {dy, w, nullptr, nullptr, gelu_input, dx, nullptr, M, K, N, lddy, ldw, 0, ldu, lddx, 0, 0, status_buf, true};
    return launch_linear(1, x, stream);
}

}  // namespace mpipe

extern "C" {

int32_t mpipe_linear_wgrad(const void* dy, const void* x, float* dw, int32_t n_tokens, int32_t N, int32_t K, int64_t lddy,
                           int64_t ldx, int64_t lddw, int32_t* status_buf, void* stream) {
    return mpipe::launch_wgrad(dy, x, dw, nullptr, n_tokens, N, K, lddy, ldx, lddw, status_buf, stream, mpipe::LayerAhead());
}

int32_t mpipe_linear_fwd(const void* a, const void* w, const void* bias, const void* residual, void* c, int32_t M,
                         int32_t N, int32_t K, int64_t lda, int64_t ldw, int64_t ldr, int64_t ldc, int32_t flags,
                         int32_t* status_buf, void* stream) {
    if ((flags & ~(MPIPE_LINEAR_GELU)) != 0) return MPIPE_ERR_INVALID_ARG;
    const mpipe::LinearCall x = {a, w, bias, residual, nullptr, c, nullptr, M, N, K, lda, ldw, ldr, 0, ldc, 0,
                                 (flags & MPIPE_LINEAR_GELU) ? 1 : 0, status_buf, false};
    return mpipe::launch_linear(0, x, stream);
}

int32_t mpipe_linear_dgrad(const void* dy, const void* w, const void* gelu_input, const void* residual, void* dx, int32_t M,
                           int32_t N, int32_t K, int64_t lddy, int64_t ldw, int64_t ldu, int64_t ldr, int64_t lddx,
                           int32_t* status_buf, void* stream) {
    const mpipe::LinearCall x = {dy, w, nullptr, residual, gelu_input, dx, nullptr, M, K, N, lddy, ldw, ldr, ldu, lddx, 0, 0, status_buf, false};
    return mpipe::launch_linear(1, x, stream);
}

}  // extern "C"

// mpipe_varlen_attn_fwd: block-diagonal (per-image) softmax attention over a packed token sequence,
// the attention of the relocated Fwd(enc, r, m) event (Section 4.2).
//
// Persistent CTAs, one per SM, take (work item, head) units from the longest-first list as they get free (units.cuh; mix of eight
// 819-token images 47.6 -> 44.8 us, ViT-L microbatch 523 -> 513 against a fixed assignment).  A work item is up to 256 query rows of
// one segment = two 128-row query tiles that share every K/V tile.  Warp roles:
//   warp 0      TMA producer: Q tiles once per unit, K and V tiles through a kStages-deep ring
//   warp 1      tcgen05 issuer: S_w = Q_w K^T into TMEM, O_w += P_w V with P_w read from TMEM
//   warp 2      TMEM allocation
//   warps 4-7   softmax of query tile 0 (thread = query row = TMEM lane)
//   warps 8-11  softmax of query tile 1
// The issuer interleaves the two query tiles (PV_0(j), S_0(j+1), PV_1(j), S_1(j+1)) so that the tensor
// pipe works on one tile while the other tile's softmax runs.  Softmax is online with a lazily updated
// reference maximum: the accumulator in TMEM is rescaled only when a row maximum grows by more than
// 2^8, so P stays <= 256 and almost no tile needs the rescale.  P is written back over S in TMEM as
// packed bf16 and consumed from there as the A operand of the second MMA.
//
// Every mbarrier wait is bounded; on expiry the CTA sets an abort flag, all roles drain, TMEM is freed
// and MPIPE_ERR_TIMEOUT is reported through status_buf.
#include <cuda.h>
#include <math_constants.h>

#include <type_traits>

#include "common.h"
#include "sm100_ptx.cuh"
#include "tensormap.h"
#include "units.cuh"

namespace mpipe {

constexpr int kFwdThreads = 384;
constexpr int kTileM = 128;        // query rows per tile (= TMEM lanes)
constexpr int kTileN = 128;        // keys per K/V tile
constexpr float kRescaleThreshold = 8.0f;  // in log2 units
// setmaxnreg: the 4 light warps release what the 8 softmax warps take (an increase blocks until the CTA's
// own pool has the registers).
constexpr int kFwdRegsLaunch = 168, kFwdRegsLight = 56, kFwdRegsSoftmax = 224;
static_assert(4 * (kFwdRegsLaunch - kFwdRegsLight) >= 8 * (kFwdRegsSoftmax - kFwdRegsLaunch), "setmaxnreg pool arithmetic");

template <int D>
struct FwdCfg {
    static constexpr int kStages = (D == 64) ? 4 : 3;
    static constexpr int kTail = D - 64;                              // 0 or 16 head-dim columns beyond the first 64
    static constexpr int kQBytesMain = kTileM * 128;                  // 64 bf16 per row, 128-byte swizzle
    static constexpr int kQBytesTail = kTail ? kTileM * 32 : 0;       // 16 bf16 per row, 32-byte swizzle
    static constexpr int kQBytes = kQBytesMain + kQBytesTail;         // Q and K tiles (K-major operands)
    static constexpr int kVBytes = kTail ? 2 * kTileN * 128 : kTileN * 128;  // V (MN-major): two 64-wide atoms if D=80
    static constexpr int kSmemQ = 0;
    static constexpr int kSmemK = 2 * kQBytes;
    static constexpr int kSmemV = kSmemK + kStages * kQBytes;
    static constexpr int kOutCols = (D == 64) ? 64 : 32;              // one [32 rows][kOutCols] box of O per softmax warp
    static constexpr int kOutBox = 32 * kOutCols * 2;
    static constexpr int kSmemO = kSmemV + kStages * kVBytes;
    static constexpr int kSmemTotal = kSmemO + 8 * kOutBox;
    static constexpr int kSmemAlloc = kSmemTotal + 1024;              // slack for manual 1024-byte alignment
    // TMEM: S_w at 128 w, O_w at 256 + 128 w.  head_dim 64 leaves 64 columns behind each O_w: P_w (128 keys as bf16) goes
    // there instead of overlaying S_w, so that S_w(j+1) can be issued as soon as the softmax warps have READ S_w(j)
    // and runs under their exponentials, instead of waiting behind P_w(j) V(j).
    static constexpr bool kPSep = (D + kTileN / 2 <= 128);
    // bit i: column pair i (mod 8) of a row forms its exponential with the polynomial on the FMA pipes instead of the
    // special-function unit.  3 of 8 balances the two when the query tiles' softmax passes alternate (head_dim 80);
    // with separate P columns the two passes run side by side and 2 of 8 measured best (all-MUFU 752, 1 of 8 781,
    // 2 of 8 800, 3 of 8 770 TFLOP/s on the ViT-L workload).
    static constexpr unsigned kPolyMask = kPSep ? 0x12u : 0x52u;
    static constexpr int kColP0 = kPSep ? 256 + 64 : 0, kColPStride = 128;
};

struct FwdParams {
    const mpipe_work_item_t* items;
    int32_t n_items, n_heads;
    __nv_bfloat16* o;
    float* lse;  // nullptr when the encoder is frozen
    int64_t tok_stride_o, head_stride_o;
    int32_t total_tokens;
    float scale_log2;  // softmax_scale * log2(e)
    int32_t settled;   // the items were complete before the previous kernel of the stream started
    int32_t* status_buf;
};

struct FwdBarriers {
    uint64_t q_full, q_empty;
    uint64_t k_full[4], k_empty[4], v_full[4], v_empty[4];
    uint64_t s_full[2], p_full[2], o_full[2], s_read[2], pv_done[2];
};

// kSplit: the two query tiles of an item are units of their own (an instantiation apart: the bookkeeping for it in the other one
// costs 2 to 7 % on long lists).
// kStaged: O leaves through shared memory (see the epilogue).
// kLate: when a unit asks for the next one (see the launch).
template <int D, bool kSplit, bool kStaged, bool kLate>
__global__ void __maxnreg__(kFwdRegsLaunch)
attn_fwd_kernel(const __grid_constant__ CUtensorMap map_q, const __grid_constant__ CUtensorMap map_k,
                const __grid_constant__ CUtensorMap map_v, const __grid_constant__ CUtensorMap map_q_tail,
                const __grid_constant__ CUtensorMap map_k_tail, const __grid_constant__ CUtensorMap map_o, const FwdParams p) {
    using Cfg = FwdCfg<D>;
    constexpr int NS = Cfg::kStages;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    __shared__ FwdBarriers bars;
    __shared__ UnitRing units;
    __shared__ uint32_t tmem_base_slot;
    __shared__ int abort_flag;

    const int tid = threadIdx.x;
    const int warp = tid >> 5;
    const int lane = tid & 31;

    if (tid == 0) {
        abort_flag = 0;
        unit_ring_init(&units, 9);   // the issuer and the softmax warps read it
        mbar_init(&bars.q_full, 1);
        mbar_init(&bars.q_empty, 1);
        for (int s = 0; s < 4; ++s) {
            mbar_init(&bars.k_full[s], 1);
            mbar_init(&bars.k_empty[s], 1);
            mbar_init(&bars.v_full[s], 1);
            mbar_init(&bars.v_empty[s], 1);
        }
        for (int w = 0; w < 2; ++w) {
            mbar_init(&bars.s_full[w], 1);
            mbar_init(&bars.p_full[w], 4);  // one arrival per softmax warp
            mbar_init(&bars.o_full[w], 1);
            mbar_init(&bars.s_read[w], 4);   // (separate P only) S_w is in the softmax warps' registers
            mbar_init(&bars.pv_done[w], 1);  // (separate P only) P_w V has consumed P_w and updated O_w
        }
        fence_mbar_init();
    }
    if (warp == 2) {
        tmem_alloc(&tmem_base_slot, 512);
        tmem_relinquish();
    }
    if (warp == 0 && lane == 0) {
        prefetch_tmap(&map_q);
        prefetch_tmap(&map_k);
        prefetch_tmap(&map_v);
        prefetch_tmap(&map_o);
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_base_slot;
    // TMEM columns: S_0 [0,128), S_1 [128,256), O_0 [256,256+D), O_1 [384,384+D); P_w overlays S_w.
    // The plan comes from device memory: it is checked as a whole before any role starts (see plan_ok_cta); a
    // rejected plan leaves every role with nothing to do.  Inside a layer (`settled`) the plan is older than the kernel
    // before this one and is checked while that kernel still runs.
    __shared__ int plan_flag;
    if (!p.settled) pdl_wait();
    const int n_units = plan_ok_cta(p.items, p.n_items, 2 * kTileM, p.total_tokens, p.status_buf, &plan_flag) ? p.n_items * p.n_heads * (kSplit ? 2 : 1) : 0;
    if (p.settled) pdl_wait();
    pdl_launch();
    // Unit -> work item with the head in its `seg` field.  kSplit: the second half of an item with one query tile comes back
    // without rows; every role passes over it.
    auto item_at = [&](int u) {
        mpipe_work_item_t z = {0, 0, 0, 0, 0, 0};
        if (u < 0 || u >= n_units) return z;
        const int v = kSplit ? u / 2 : u;
        z = p.items[v / p.n_heads];
        z.seg = v % p.n_heads;
        if (kSplit) {
            const int off = (u % 2) * kTileM;
            z.row_start += off;
            z.row_len = min(z.row_len - off, kTileM);
        }
        return z;
    };

    if (warp == 0) {
        setmaxnreg_dec<kFwdRegsLight>();
        // ------------------------------------------------------------------ TMA producer
        if (lane == 0) {
            uint32_t kv_it = 0, unit_it = 0;
            bool ok = true;
            UnitSource source{&units, &abort_flag};
            for (int u = int(blockIdx.x); ok; ++unit_it) {
                const mpipe_work_item_t it = item_at(u);
                ok = source.put(it);
                if (!ok || it.kv_len <= 0) break;
                if (!kLate) source.ask();
                if (kSplit && it.row_len <= 0) {
                    u = source.take(&ok);
                    --unit_it;
                    continue;
                }
                const int head = it.seg;
                const bool two = it.row_len > kTileM;
                const int nkv = (it.kv_len + kTileN - 1) / kTileN;
                ok = mbar_wait(&bars.q_empty, (unit_it & 1) ^ 1, &abort_flag);
                if (!ok) break;
                mbar_expect_tx(&bars.q_full, (two ? 2 : 1) * Cfg::kQBytes);
                for (int w = 0; w < (two ? 2 : 1); ++w) {
                    uint8_t* dst = smem + Cfg::kSmemQ + w * Cfg::kQBytes;
                    tma_load_3d(dst, &map_q, &bars.q_full, 0, head, it.row_start + w * kTileM);
                    if (Cfg::kTail) tma_load_3d(dst + Cfg::kQBytesMain, &map_q_tail, &bars.q_full, 64, head, it.row_start + w * kTileM);
                }
                for (int j = 0; j < nkv; ++j, ++kv_it) {
                    const int s = kv_it % NS;
                    const uint32_t ph = (kv_it / NS) & 1;
                    const int row = it.kv_start + j * kTileN;
                    ok = mbar_wait(&bars.k_empty[s], ph ^ 1, &abort_flag);
                    if (!ok) break;
                    mbar_expect_tx(&bars.k_full[s], Cfg::kQBytes);
                    uint8_t* kdst = smem + Cfg::kSmemK + s * Cfg::kQBytes;
                    tma_load_3d(kdst, &map_k, &bars.k_full[s], 0, head, row);
                    if (Cfg::kTail) tma_load_3d(kdst + Cfg::kQBytesMain, &map_k_tail, &bars.k_full[s], 64, head, row);
                    ok = mbar_wait(&bars.v_empty[s], ph ^ 1, &abort_flag);
                    if (!ok) break;
                    mbar_expect_tx(&bars.v_full[s], Cfg::kVBytes);
                    uint8_t* vdst = smem + Cfg::kSmemV + s * Cfg::kVBytes;
                    tma_load_3d(vdst, &map_v, &bars.v_full[s], 0, head, row);
                    if (Cfg::kTail) tma_load_3d(vdst + kTileN * 128, &map_v, &bars.v_full[s], 64, head, row);
                }
                if (!ok) break;
                if (kLate) {   // the scores of the last key tile but one are there (of the last: head_dim 64, two or three of them)
                    if (nkv > 1) {
                        const uint32_t at = kv_it - (D == 64 && nkv <= 3 ? 1 : 2);
                        ok = mbar_wait(&bars.k_empty[at % NS], (at / NS) & 1, &abort_flag);
                        if (!ok) break;
                    }
                    source.ask();
                }
                u = source.take(&ok);
            }
            if (!ok) source.cancel_rest();
        }
        __syncwarp();
    } else if (warp == 1) {
        // ------------------------------------------------------------------ tcgen05 issuer
        // The whole warp walks the loop (uniform control flow, uniform descriptors); one elected lane
        // issues the MMAs and commits.  Descriptors are precomputed: a K-step only bumps the low word.
        setmaxnreg_dec<kFwdRegsLight>();
        {
            const bool leader = elect_one();
            const uint32_t sbase = smem_u32(smem);
            constexpr uint32_t hi128 = umma_desc_hi(1024, kSwizzle128);
            constexpr uint32_t hi32 = umma_desc_hi(256, kSwizzle32);
            uint32_t kv_it = 0, unit_it = 0, cnt[2] = {0, 0};
            bool ok = true;
            // S_w = Q_w K^T for the KV tile in stage s; n_cols = keys to cover (multiple of 16)
            auto issue_s = [&](int w, int s, int n_cols) {
                const uint32_t qa = sbase + Cfg::kSmemQ + w * Cfg::kQBytes;
                const uint32_t ka = sbase + Cfg::kSmemK + s * Cfg::kQBytes;
                const uint32_t qlo = umma_desc_lo(qa, 0), klo = umma_desc_lo(ka, 0);
                const uint32_t idesc = umma_idesc_bf16(kTileM, n_cols, 0, 0);
                const uint32_t d = tmem + w * 128;
                if (leader) {
#pragma unroll
                    for (int ks = 0; ks < 4; ++ks)
                        umma_ss(d, umma_desc(qlo + ks * 2, hi128), umma_desc(klo + ks * 2, hi128), idesc, ks > 0);
                    if (Cfg::kTail)
                        umma_ss(d, umma_desc(umma_desc_lo(qa + Cfg::kQBytesMain, 0), hi32),
                                umma_desc(umma_desc_lo(ka + Cfg::kQBytesMain, 0), hi32), idesc, 1);
                }
            };
            // O_w (+)= P_w V for the KV tile in stage s; n_keys = keys to cover (multiple of 16)
            auto issue_pv = [&](int w, int s, int n_keys, bool accumulate) {
                const uint32_t vlo = umma_desc_lo(sbase + Cfg::kSmemV + s * Cfg::kVBytes, kTileN * 128);
                constexpr uint32_t idesc = umma_idesc_bf16(kTileM, D, 0, 1);
                const uint32_t d = tmem + 256 + w * 128;
                const uint32_t pa = tmem + Cfg::kColP0 + w * Cfg::kColPStride;
                if (leader) {
                    if (n_keys == kTileN) {
#pragma unroll
                        for (int ks = 0; ks < 8; ++ks)
                            umma_ts(d, pa + ks * 8, umma_desc(vlo + ks * 128, hi128), idesc, (accumulate || ks > 0) ? 1u : 0u);
                    } else {
                        for (int ks = 0; ks < n_keys / 16; ++ks)
                            umma_ts(d, pa + ks * 8, umma_desc(vlo + ks * 128, hi128), idesc, (accumulate || ks > 0) ? 1u : 0u);
                    }
                }
            };
            mpipe_work_item_t it;
            for (uint32_t ui = 0; ok && next_unit(&units, ui, &it, lane, &abort_flag); ++ui, ++unit_it) {
                if (kSplit && it.row_len <= 0) { --unit_it; continue; }
                const bool two = it.row_len > kTileM;
                const int nkv = (it.kv_len + kTileN - 1) / kTileN;
                auto cols_of = [&](int j) {
                    const int rem = it.kv_len - j * kTileN;
                    return rem >= kTileN ? kTileN : ((rem + 15) & ~15);
                };
                ok = mbar_wait(&bars.q_full, unit_it & 1, &abort_flag);
                if (!ok) break;
                {
                    const int s = kv_it % NS;
                    ok = mbar_wait(&bars.k_full[s], (kv_it / NS) & 1, &abort_flag);
                    if (!ok) break;
                    tc_fence_after();
                    issue_s(0, s, cols_of(0));
                    if (leader) umma_commit(&bars.s_full[0]);
                    if (two) {
                        issue_s(1, s, cols_of(0));
                        if (leader) umma_commit(&bars.s_full[1]);
                    }
                    if (leader) umma_commit(&bars.k_empty[s]);
                    if (nkv == 1) if (leader) umma_commit(&bars.q_empty);
                }
                if (Cfg::kPSep) {
                    // Order per KV tile j:  S_0(j+1) | PV_1(j-1) | S_1(j+1) | PV_0(j): each S goes out as soon as its
                    // predecessor has been read, each PV as soon as its P is complete, and the two query tiles stay half
                    // a pass apart.
                    for (int j = 0; j < nkv; ++j) {
                        const uint32_t itv = kv_it + j;
                        const int sv = itv % NS;
                        const bool more = (j + 1 < nkv);
                        const int sk = (itv + 1) % NS;
                        if (more) {
                            ok = mbar_wait(&bars.k_full[sk], ((itv + 1) / NS) & 1, &abort_flag);
                            if (ok) ok = mbar_wait(&bars.s_read[0], (cnt[0] + j) & 1, &abort_flag);
                            if (!ok) break;
                            tc_fence_after();
                            issue_s(0, sk, cols_of(j + 1));
                            if (leader) umma_commit(&bars.s_full[0]);
                        }
                        if (two && j > 0) {
                            ok = mbar_wait(&bars.p_full[1], (cnt[1] + j - 1) & 1, &abort_flag);
                            if (!ok) break;
                            tc_fence_after();
                            issue_pv(1, (itv - 1) % NS, cols_of(j - 1), j - 1 > 0);
                            if (leader) umma_commit(&bars.pv_done[1]);
                            if (leader) umma_commit(&bars.v_empty[(itv - 1) % NS]);
                        }
                        if (more) {
                            if (two) {
                                ok = mbar_wait(&bars.s_read[1], (cnt[1] + j) & 1, &abort_flag);
                                if (!ok) break;
                                tc_fence_after();
                                issue_s(1, sk, cols_of(j + 1));
                                if (leader) umma_commit(&bars.s_full[1]);
                            }
                            if (leader) umma_commit(&bars.k_empty[sk]);
                            if (j + 2 == nkv) if (leader) umma_commit(&bars.q_empty);
                        }
                        ok = mbar_wait(&bars.v_full[sv], (itv / NS) & 1, &abort_flag);
                        if (ok) ok = mbar_wait(&bars.p_full[0], (cnt[0] + j) & 1, &abort_flag);
                        if (!ok) break;
                        tc_fence_after();
                        issue_pv(0, sv, cols_of(j), j > 0);
                        if (leader) umma_commit(&bars.pv_done[0]);
                        if (!more) if (leader) umma_commit(&bars.o_full[0]);
                        if (!two) if (leader) umma_commit(&bars.v_empty[sv]);
                    }
                    if (ok && two) {   // PV_1 of the unit's last KV tile
                        const uint32_t itv = kv_it + nkv - 1;
                        ok = mbar_wait(&bars.p_full[1], (cnt[1] + nkv - 1) & 1, &abort_flag);
                        if (!ok) break;
                        tc_fence_after();
                        issue_pv(1, itv % NS, cols_of(nkv - 1), nkv - 1 > 0);
                        if (leader) umma_commit(&bars.pv_done[1]);
                        if (leader) umma_commit(&bars.o_full[1]);
                        if (leader) umma_commit(&bars.v_empty[itv % NS]);
                    }
                    if (!ok) break;
                } else
                for (int j = 0; j < nkv; ++j) {
                    const uint32_t itv = kv_it + j;
                    const int sv = itv % NS;
                    const bool more = (j + 1 < nkv);
                    const int sk = (itv + 1) % NS;
                    ok = mbar_wait(&bars.v_full[sv], (itv / NS) & 1, &abort_flag);
                    if (!ok) break;
                    ok = mbar_wait(&bars.p_full[0], (cnt[0] + j) & 1, &abort_flag);
                    if (!ok) break;
                    tc_fence_after();
                    issue_pv(0, sv, cols_of(j), j > 0);
                    if (more) {
                        ok = mbar_wait(&bars.k_full[sk], ((itv + 1) / NS) & 1, &abort_flag);
                        if (!ok) break;
                        tc_fence_after();
                        issue_s(0, sk, cols_of(j + 1));
                        if (leader) umma_commit(&bars.s_full[0]);
                    } else {
                        if (leader) umma_commit(&bars.o_full[0]);
                    }
                    if (two) {
                        ok = mbar_wait(&bars.p_full[1], (cnt[1] + j) & 1, &abort_flag);
                        if (!ok) break;
                        tc_fence_after();
                        issue_pv(1, sv, cols_of(j), j > 0);
                        if (more) {
                            issue_s(1, sk, cols_of(j + 1));
                            if (leader) umma_commit(&bars.s_full[1]);
                        } else {
                            if (leader) umma_commit(&bars.o_full[1]);
                        }
                    }
                    if (leader) umma_commit(&bars.v_empty[sv]);
                    if (more) {
                        if (leader) umma_commit(&bars.k_empty[sk]);
                        if (j + 2 == nkv) if (leader) umma_commit(&bars.q_empty);
                    }
                }
                kv_it += nkv;
                cnt[0] += nkv;
                if (two) cnt[1] += nkv;
            }
        }
        __syncwarp();
    } else if (warp < 4) {
        setmaxnreg_dec<kFwdRegsLight>();
    } else {
        // ------------------------------------------------------------------ softmax + epilogue
        setmaxnreg_inc<kFwdRegsSoftmax>();
        const int w = (warp - 4) >> 2;              // query tile handled by this warpgroup
        const int r = ((warp & 3) << 5) | lane;     // row inside the tile = TMEM lane
        const uint32_t lane_base = uint32_t((warp & 3) * 32) << 16;
        const uint32_t t_s = tmem + lane_base + w * 128;
        const uint32_t t_o = tmem + lane_base + 256 + w * 128;
        const uint32_t t_p = tmem + lane_base + Cfg::kColP0 + w * Cfg::kColPStride;   // = t_s when P overlays S
        uint32_t cnt = 0, ocnt = 0;
        bool ok = true;
        mpipe_work_item_t it;
        for (uint32_t ui = 0; ok && next_unit(&units, ui, &it, lane, &abort_flag); ++ui) {
            const int head = it.seg;
            const int rows_here = it.row_len - w * kTileM;  // valid rows of this tile
            if (rows_here <= 0) continue;
            const int nkv = (it.kv_len + kTileN - 1) / kTileN;
            float m_ref = -CUDART_INF_F;  // reference maximum, scaled log2 domain
            float l = 0.f;
            for (int j = 0; j < nkv; ++j) {
                ok = mbar_wait(&bars.s_full[w], (cnt + j) & 1, &abort_flag);
                if (!ok) break;
                tc_fence_after();
                uint32_t sr[128];
                tmem_ld32(t_s + 0, *reinterpret_cast<uint32_t(*)[32]>(&sr[0]));
                tmem_ld32(t_s + 32, *reinterpret_cast<uint32_t(*)[32]>(&sr[32]));
                tmem_ld32(t_s + 64, *reinterpret_cast<uint32_t(*)[32]>(&sr[64]));
                tmem_ld32(t_s + 96, *reinterpret_cast<uint32_t(*)[32]>(&sr[96]));
                tmem_wait_ld();
                if (Cfg::kPSep) {   // the scores are in registers: S_w of the next KV tile may be written
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&bars.s_read[w]);
                }
                const int n_valid = it.kv_len - j * kTileN;
                if (n_valid < kTileN) {
#pragma unroll
                    for (int c = 0; c < 128; ++c)
                        if (c >= n_valid) sr[c] = 0xFF800000u;  // -inf
                }
                // eight independent running maxima, three inputs per instruction (a single chain of 127
                // dependent max ops would cost ~4 cycles each with only two softmax warps per scheduler)
                float mx8[8];
#pragma unroll
                for (int e = 0; e < 8; ++e) mx8[e] = fmaxf(__uint_as_float(sr[e]), __uint_as_float(sr[8 + e]));
#pragma unroll
                for (int c = 16; c < 128; c += 16) {
#pragma unroll
                    for (int e = 0; e < 8; ++e)
                        mx8[e] = fmax3(mx8[e], __uint_as_float(sr[c + e]), __uint_as_float(sr[c + 8 + e]));
                }
                const float mx = fmax3(fmax3(mx8[0], mx8[1], mx8[2]), fmax3(mx8[3], mx8[4], mx8[5]), fmaxf(mx8[6], mx8[7]));
                const float m_tile = mx * p.scale_log2;
                const bool grow = m_tile > m_ref + kRescaleThreshold;  // always true on the first tile
                const float m_new = grow ? m_tile : m_ref;
                const float alpha = ex2_approx(m_ref - m_new);         // 0 on the first tile, 1 if unchanged
                m_ref = m_new;
                if (Cfg::kPSep && j > 0) {   // P_w V of the previous KV tile has read P_w and updated O_w (long since, as a rule)
                    ok = mbar_wait(&bars.pv_done[w], (cnt + j - 1) & 1, &abort_flag);
                    if (!ok) break;
                    tc_fence_after();
                }
                if (j > 0 && __any_sync(0xffffffffu, grow)) {
                    // rescale this warp's rows of the accumulator; PV(j-1) has completed (overlaid P: it was issued
                    // before S(j), whose completion we just observed; separate P: waited for above)
#pragma unroll
                    for (int c0 = 0; c0 < D; c0 += 16) {
                        uint32_t orr[16];
                        tmem_ld16(t_o + c0, orr);
                        tmem_wait_ld();
#pragma unroll
                        for (int c = 0; c < 16; ++c) orr[c] = __float_as_uint(__uint_as_float(orr[c]) * alpha);
                        tmem_st16(t_o + c0, orr);
                    }
                }
                // p = exp2(s * scale*log2e - m_ref): packed fp32 pairs for the multiply-add and the row sum,
                // four independent partial sums
                const float2 sc2 = make_float2(p.scale_log2, p.scale_log2);
                const float2 nm2 = make_float2(-m_ref, -m_ref);
                float2 acc[4] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f), make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
#pragma unroll
                for (int c0 = 0; c0 < 128; c0 += 32) {
                    uint32_t pk[16];
#pragma unroll
                    for (int c = 0; c < 32; c += 2) {
                        const float2 x = fma2(make_float2(__uint_as_float(sr[c0 + c]), __uint_as_float(sr[c0 + c + 1])), sc2, nm2);
                        // kPolyMask picks, out of every 8 column pairs, those whose exponential runs on the FMA
                        // pipes; the rest use the special-function unit.  The split balances the two.
                        const float2 e = ((Cfg::kPolyMask >> ((c >> 1) & 7)) & 1) ? exp2_poly2(x)
                                                                           : make_float2(ex2_approx(x.x), ex2_approx(x.y));
                        acc[(c >> 1) & 3] = add2(acc[(c >> 1) & 3], e);
                        pk[c >> 1] = pack_bf16(e.x, e.y);
                    }
                    tmem_st16(t_p + (c0 >> 1), pk);
                }
                const float2 s01 = add2(add2(acc[0], acc[1]), add2(acc[2], acc[3]));
                l = l * alpha + (s01.x + s01.y);
                tmem_wait_st();
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(&bars.p_full[w]);
            }
            if (!ok) break;
            cnt += nkv;
            // epilogue: O / l -> bf16, LSE = ln2 * m_ref + ln l
            ok = mbar_wait(&bars.o_full[w], ocnt & 1, &abort_flag);
            if (!ok) break;
            ++ocnt;
            tc_fence_after();
            const float inv_l = 1.0f / l;
            const bool store = r < rows_here;
            const int64_t tok = int64_t(it.row_start) + w * kTileM + r;
            // Staged: in a unit of two query tiles, where all 32 rows of a warp are rows of the segment, the first 64 columns leave
            // through the warp's staging box (128- or 64-byte swizzle) by a TMA store: straight from the registers every store
            // of a warp touches 32 rows (256 wavefronts per warp and unit, 2000 clocks for the eight of a 256-row unit).
            // head_dim 80 has room for half of the columns: the first half is read back and stored in coalesced pieces, so that
            // nothing waits for the copy engine inside a unit.  A ragged warp and a unit of one tile, whose four warps get in
            // nobody's way, store directly.
            __nv_bfloat16* orow = p.o + tok * p.tok_stride_o + int64_t(head) * p.head_stride_o;
            const int row0 = (warp & 3) * 32;                   // first row of this warp in the tile
            const bool whole = kStaged && it.row_len > kTileM && rows_here - row0 >= 32;
            int c_done = 0;                                     // columns that have left
            if (kStaged && (D == 80 || whole)) {                // (head_dim 80: one path with predicated stores measured faster)
                constexpr int kOC = Cfg::kOutCols, kCh = kOC / 8;
                auto slot = [](int row, int c) { return row * (kOC * 2) + ((kOC == 64 ? c ^ (row & 7) : c ^ ((row >> 1) & 3)) << 4); };
                uint32_t orr[64];
                tmem_ld32(t_o, *reinterpret_cast<uint32_t(*)[32]>(&orr[0]));
                tmem_ld32(t_o + 32, *reinterpret_cast<uint32_t(*)[32]>(&orr[32]));
                uint8_t* box = smem + Cfg::kSmemO + (warp - 4) * Cfg::kOutBox;
                if (whole && lane == 0) bulk_wait_group_read<0>();   // the previous unit's store has read the box
                tmem_wait_ld();
                __syncwarp();
#pragma unroll
                for (int c0 = 0; c0 < 64; c0 += kOC) {
#pragma unroll
                    for (int g = 0; g < kCh; ++g) {
                        uint32_t o4[4];
#pragma unroll
                        for (int e = 0; e < 4; ++e)
                            o4[e] = pack_bf16(__uint_as_float(orr[c0 + 8 * g + 2 * e]) * inv_l, __uint_as_float(orr[c0 + 8 * g + 2 * e + 1]) * inv_l);
                        const uint4 v = make_uint4(o4[0], o4[1], o4[2], o4[3]);
                        if (D == 64 || whole) *reinterpret_cast<uint4*>(box + slot(lane, g)) = v;
                        else if (store) *reinterpret_cast<uint4*>(orow + c0 + 8 * g) = v;
                    }
                    if (whole && c0 + kOC < 64) {
                        __syncwarp();
                        __nv_bfloat16* orow0 = orow - lane * p.tok_stride_o + c0;
#pragma unroll
                        for (int i = 0; i < kCh; ++i) {
                            const int rr = (32 / kCh) * i + lane / kCh, c = lane % kCh;
                            *reinterpret_cast<uint4*>(orow0 + rr * p.tok_stride_o + c * 8) = *reinterpret_cast<const uint4*>(box + slot(rr, c));
                        }
                        __syncwarp();                            // (read before it is written again)
                    } else if (whole) {
                        fence_async_smem();
                        __syncwarp();
                        if (lane == 0) {
                            tma_store_3d(&map_o, box, c0, head, it.row_start + w * kTileM + row0);
                            bulk_commit_group();
                        }
                    }
                }
                c_done = 64;
            }
#pragma unroll
            for (int c0 = 0; c0 < D; c0 += 16) {
                if (c0 < c_done) continue;
                uint32_t orr[16];
                tmem_ld16(t_o + c0, orr);
                tmem_wait_ld();
                uint32_t o8[8];
#pragma unroll
                for (int e = 0; e < 8; ++e) o8[e] = pack_bf16(__uint_as_float(orr[2 * e]) * inv_l, __uint_as_float(orr[2 * e + 1]) * inv_l);
                if (store) {
                    *reinterpret_cast<uint4*>(orow + c0) = make_uint4(o8[0], o8[1], o8[2], o8[3]);
                    *reinterpret_cast<uint4*>(orow + c0 + 8) = make_uint4(o8[4], o8[5], o8[6], o8[7]);
                }
            }
            if (store && p.lse != nullptr)
                p.lse[int64_t(head) * p.total_tokens + tok] = m_ref * 0.6931471805599453f + logf(l);
            tc_fence_before();
        }
        if (kStaged) {
            if (lane == 0) bulk_wait_group_read<0>();   // shared memory must outlive the copy engine's reads
            __syncwarp();
        }
    }

    tc_fence_before();
    __syncthreads();
    if (warp == 2) tmem_dealloc(tmem, 512);
    if (tid == 0 && abort_flag) report_status(p.status_buf, MPIPE_ERR_TIMEOUT, int32_t(blockIdx.x));
}

template <int D, bool kSplit, bool kStaged, bool kLate>
static int32_t launch_fwd(const void* q, const void* k, const void* v, int64_t tok_stride, int64_t head_stride,
                          int32_t total_tokens, int32_t n_heads, const FwdParams& prm, cudaStream_t stream) {
    using Cfg = FwdCfg<D>;
    CUtensorMap mq, mk, mv, mqt, mkt, mo;
    const uint32_t main_box = 64;
    if (!make_tensor_map_thd(&mq, q, total_tokens, n_heads, D, tok_stride, head_stride, main_box, kTileM, 128) ||
        !make_tensor_map_thd(&mk, k, total_tokens, n_heads, D, tok_stride, head_stride, main_box, kTileN, 128) ||
        !make_tensor_map_thd(&mv, v, total_tokens, n_heads, D, tok_stride, head_stride, main_box, kTileN, 128) ||
        !make_tensor_map_thd(&mo, prm.o, total_tokens, n_heads, D, prm.tok_stride_o, prm.head_stride_o, Cfg::kOutCols, 32, Cfg::kOutCols * 2))
        return MPIPE_ERR_CUDA;
    mqt = mq;
    mkt = mk;
    if (Cfg::kTail) {
        if (!make_tensor_map_thd(&mqt, q, total_tokens, n_heads, D, tok_stride, head_stride, 16, kTileM, 32) ||
            !make_tensor_map_thd(&mkt, k, total_tokens, n_heads, D, tok_stride, head_stride, 16, kTileN, 32))
            return MPIPE_ERR_CUDA;
    }
    if (!ensure_dynamic_smem<attn_fwd_kernel<D, kSplit, kStaged, kLate>>(Cfg::kSmemAlloc)) return MPIPE_ERR_CUDA;
    const int n_units = prm.n_items * prm.n_heads * (kSplit ? 2 : 1);
    profile_start(kProfileFwd, stream);
    const cudaError_t e = launch_kernel_as(true, attn_fwd_kernel<D, kSplit, kStaged, kLate>, unsigned(n_units), kFwdThreads, Cfg::kSmemAlloc, stream, 1,
                                           mq, mk, mv, mqt, mkt, mo, prm);
    profile_stop(kProfileFwd, stream);
    return e == cudaSuccess && cudaGetLastError() == cudaSuccess ? MPIPE_OK : MPIPE_ERR_CUDA;
}

int32_t varlen_attn_fwd(const void* q, const void* k, const void* v, void* o, float* lse,
                              int64_t tok_stride_qkv, int64_t head_stride_qkv, int64_t tok_stride_o,
                              int64_t head_stride_o, const int32_t* cu_seqlens_dev, int32_t n_seg,
                              int32_t total_tokens, int32_t max_seqlen, const mpipe_work_item_t* fwd_items_dev,
                              int32_t n_fwd_items, int32_t n_heads, int32_t head_dim, float softmax_scale,
                              int32_t mode, int32_t* status_buf, void* stream, bool settled) {
    if (mode != MPIPE_ENC_FROZEN && mode != MPIPE_ENC_TRAINED) return MPIPE_ERR_INVALID_ARG;
    if (n_seg < 0 || total_tokens < 0 || max_seqlen < 0 || n_fwd_items < 0 || n_heads <= 0) return MPIPE_ERR_INVALID_ARG;
    if (head_dim != 64 && head_dim != 80) return MPIPE_ERR_UNSUPPORTED;
    if (total_tokens == 0 || n_fwd_items == 0) return MPIPE_OK;
    if (q == nullptr || k == nullptr || v == nullptr || o == nullptr || fwd_items_dev == nullptr ||
        cu_seqlens_dev == nullptr)
        return MPIPE_ERR_INVALID_ARG;
    if (mode == MPIPE_ENC_TRAINED && lse == nullptr) return MPIPE_ERR_INVALID_ARG;
    if (!aligned16(q) || !aligned16(k) || !aligned16(v) || !aligned16(o)) return MPIPE_ERR_INVALID_ARG;
    if ((tok_stride_qkv & 7) || (head_stride_qkv & 7) || (tok_stride_o & 7) || (head_stride_o & 7))
        return MPIPE_ERR_INVALID_ARG;
    if (head_stride_qkv < head_dim || head_stride_o < head_dim || tok_stride_qkv < head_dim || tok_stride_o < head_dim)
        return MPIPE_ERR_INVALID_ARG;
    if (!(softmax_scale > 0.f) || !(softmax_scale < 1e30f)) return MPIPE_ERR_INVALID_ARG;
    if (int64_t(n_fwd_items) * n_heads >= (int64_t(1) << 31)) return MPIPE_ERR_INVALID_ARG;

    FwdParams prm;
    prm.items = fwd_items_dev;
    prm.n_items = n_fwd_items;
    prm.n_heads = n_heads;
    prm.o = static_cast<__nv_bfloat16*>(o);
    prm.lse = (mode == MPIPE_ENC_TRAINED) ? lse : nullptr;
    prm.tok_stride_o = tok_stride_o;
    prm.head_stride_o = head_stride_o;
    prm.total_tokens = total_tokens;
    prm.scale_log2 = softmax_scale * 1.4426950408889634f;
    prm.settled = settled ? 1 : 0;
    prm.status_buf = status_buf;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    // Two query tiles per CTA share every K/V tile and run side by side, which is 1.4 x the work per clock of one; where so few
    // units would leave half of the SMs idle, one tile each is sooner done (one image of 777 tokens, 16 heads of 64: 13.8 -> 11.8 us,
    // of 300: 8.9 -> 7.5; with 80 units on 148 SMs a second round of single tiles would cost more than it saves).
    const bool split = 2 * int64_t(n_fwd_items) * n_heads <= sm_count();
    auto launch = [&](auto f) { return f(q, k, v, tok_stride_qkv, head_stride_qkv, total_tokens, n_heads, prm, st); };
    // Staged O pays where units have two query tiles and enough key tiles behind them (us direct -> staged): head_dim 64, ViT-L
    // microbatch 512 -> 505, but images of 300 235 -> 239 and of 819 44.2 -> 44.6; head_dim 80, 200 images of 64 to 256 tokens
    // 101.5 -> 94.6, 65 536 long-tailed ones 2940 -> 2850, images of 2048 765 -> 700, but of 100 (one tile each) 187 -> 200.
    const bool staged = max_seqlen > (head_dim == 64 ? 1024 : 128);
    // Who gets the next unit.  Asked for at the start of a unit, the units of the second wave go to the CTAs whose first ones are the
    // longest, as all start at once; asked for towards the end (kLate), to those that are done first.  That is worth it where a
    // list of several lengths goes around a few times only: 29 images of 35 to 154, 8 heads, 9.9 -> 8.1 us (head_dim 80 10.8 -> 8.7), 25
    // of 300 20.1 -> 19.1, 74 of 300 at head_dim 80 52.3 -> 51.2, 64 of 512 53.6 -> 53.2.  The answer is then waited for by units of
    // one key tile (2062 of 16 tokens 458 -> 468, head_dim 80 490 -> 522) and by the end of a list without a second wave (one
    // image of 4096, 4 heads, 36.0 -> 36.9), and over many waves the lengths even out (40 of 819, 16 heads, 182.7 -> 184.5).
    const int64_t units = int64_t(n_fwd_items) * n_heads;
    const bool late = max_seqlen > kTileN && units > sm_count() && units <= 8 * int64_t(sm_count());
    auto pick = [&](auto dim) {
        constexpr int D = decltype(dim)::value;
        if (split) return launch(launch_fwd<D, true, false, false>);
        if (staged) return late ? launch(launch_fwd<D, false, true, true>) : launch(launch_fwd<D, false, true, false>);
        return late ? launch(launch_fwd<D, false, false, true>) : launch(launch_fwd<D, false, false, false>);
    };
    return head_dim == 64 ? pick(std::integral_constant<int, 64>()) : pick(std::integral_constant<int, 80>());
}

}  // namespace mpipe

extern "C" {

int32_t mpipe_fwd_tile_rows(void) { return 2 * mpipe::kTileM; }

int32_t mpipe_varlen_attn_fwd(const void* q, const void* k, const void* v, void* o, float* lse,
                              int64_t tok_stride_qkv, int64_t head_stride_qkv, int64_t tok_stride_o,
                              int64_t head_stride_o, const int32_t* cu_seqlens_dev, int32_t n_seg,
                              int32_t total_tokens, int32_t max_seqlen, const mpipe_work_item_t* fwd_items_dev,
                              int32_t n_fwd_items, int32_t n_heads, int32_t head_dim, float softmax_scale,
                              int32_t mode, int32_t* status_buf, void* stream) {
    return mpipe::varlen_attn_fwd(q, k, v, o, lse, tok_stride_qkv, head_stride_qkv, tok_stride_o, head_stride_o, cu_seqlens_dev,
                                  n_seg, total_tokens, max_seqlen, fwd_items_dev, n_fwd_items, n_heads, head_dim, softmax_scale,
                                  mode, status_buf, stream, false);
}

}  // extern "C"

// Prefill path: y = bf16( x.W0^T + sum over chunks u_chunk.B_chunk^T ) on the sm_100a tensor cores.
//
// One persistent CTA per SM, 6 warps:
//   warp 0   TMA producer: streams 128x64 tiles of x and BNx64 tiles of W0 (128-byte swizzle) into
//            a ring of shared-memory stages; after the last k-block of a tile it appends the tile's LoRA
//            chunks (lml_bind.cu), up to four to a stage: per chunk the 128x16 block of u and the BNx16
//            block of the slot's packed B, two contiguous pieces.  So the LoRA expand is just more K for
//            the same accumulator: [x | u_1 | u_2 ...] . [W0 ; B_1 ; B_2 ...], and costs what the ranks of the tile's slots need.
//   warp 1   MMA issuer: one lane issues tcgen05.mma (M=128, N=BN, K=16) per 16 columns of a stage
//            into one of two TMEM accumulators and commits to the stage's "empty" barrier.
//   warps 2-5 epilogue: tcgen05.ld the accumulator (each warp its 32 TMEM lanes = 32 rows), round to
//            bf16 once, stage 32x32 chunks in shared memory and write them with TMA stores.  Runs one tile
//            behind the MMA warp thanks to the second accumulator.
// Several projections of the same x share a launch: their tiles are numbered through, so that the last wave of
// tiles is shared as well.
// Dual form (two slot bindings of the same segments, two outputs): the base product is computed once.
// The epilogue reads the first output out of the accumulator and tells the MMA thread; that thread
// then adds (second binding's delta - first binding's delta) on top, as further K-steps whose u
// operands come from a second set of u blocks, and the epilogue reads the second output.  The producer slips
// those stages into the middle of the next tile's k-blocks, by when the first read is long done.
// Tall tiles (two row tiles to a CTA): see the kernel.
// Fused shrink (the plain call on a few row tiles, on tall tiles): no launch goes ahead of this one.  Every CTA works out the slots of
// all row tiles; the CTAs at the end of the grid, which own the fewest output tiles, first compute u = scale * x.A^T,
// four chunks of a row tile to a pass, as 128 x 64 tcgen05 products, write the u blocks and raise the pass's flag in the
// table's device memory; a producer waits for a tile's flags (a bounded wait) before it loads the tile's u blocks.  The
// table's epoch, advanced by the last CTA of every such call, tells this call's flags from the last call's.
// Early start (few rows): the kernel begins while the work before the call is still running.  It asks for the first stages'
// W0, which is frozen, and reads x once bind_shrink, which waits for that work, has raised a word for it.  That work may take as
// long as it likes: no other role, and no limit, starts before x may be read (see wait_x).
// For few tokens (tiles far fewer than SMs) a split-K variant follows below: a cluster of CTAs shares a
// tile and exchanges partial sums through distributed shared memory.
// B's chunks hold zeros where the adapter's B is Inf or NaN (every row of a tile meets the chunks of all its slots).  The terms
// left out are added by the epilogue, element by element, to the rows that are bound to such a slot; other tiles pay one word.
// Every wait is bounded; on give-up the CTA sets LML_FLAG_TIMEOUT, gives its copies in flight time to land and frees its TMEM.
#include <cstdio>
#include <cstdlib>
#include <mutex>

#include "lml_gemm_common.cuh"

namespace lml {

constexpr int kGemmThreads = 192;
constexpr int kGemmThreadsTall = 320;
constexpr int kTallOverride = 512;        // the shape knob's width for tall tiles

constexpr int kFuseTilesInKernel = 80;    // row tiles of a call whose shrink runs inside the kernel (the per-tile tables in shared memory)

template <int BN, bool kTall = false> struct GemmCfg {
    static constexpr int kRowTiles = kTall ? 2 : 1;
    static constexpr int kXBytes = kBM * kBK * 2;             // a k-block of one row tile
    static constexpr int kABytes = kRowTiles * kXBytes;
    static constexpr int kBBytes = BN * kBK * 2;
    static constexpr int kStageBytes = kABytes + kBBytes;
    static constexpr int kStages = kTall ? 3 : (BN == 256 ? 4 : (BN == 128 ? 6 : 8));
    static constexpr int kEpiBufs = kTall ? 1 : 2;            // staging buffers of an epilogue warp
    static constexpr int kEpiBytes = 4 * kRowTiles * kEpiBufs * kEpiBufBytes;
    static constexpr int kTmemCols = 2 * BN;
    static constexpr int kCtrlBytes = 256 + (kBindSegs + 1) * 4 + kBindSegs + 4 + 512 + kFuseTilesInKernel * 10 + 8 + kMaxChunks * 4;   // barriers; fused shrink: segment cache, shrink plan, per-tile masks and first passes; the first tile's chunks
    // The split-K kernel: no staging for the epilogue.  The ring also takes the partial sums that the CTAs exchange; where
    // they fit, a shorter one leaves the launch that computes u room on the same SM, so that the two run side by side.
    static constexpr int kSplitStagesShort = BN == 256 ? 3 : (BN == 128 ? 4 : 5);
    static constexpr int split_smem(int stages) { return 1024 + stages * kStageBytes + 256 + 2 * kMaxChunks * 4; }
    static constexpr int kSmemBytes = 1024 + kStages * kStageBytes + kEpiBytes + ((kCtrlBytes + 15) & ~15);
};

struct GemmCtrl {
    uint64_t full[8];
    uint64_t empty[8];
    uint64_t tmem_full[2];
    uint64_t tmem_empty[2];
    uint64_t tmem_read1[2];   // dual form: the first output of the tile has been read out of the accumulator
    uint64_t plan_full;       // the list of chunks is in shared memory
    uint32_t tmem_base;
    int abort;
    uint32_t stage_info[8];   // written by the producer: k-steps (0..4) | kStage* flags
    int32_t pad[2];
    int32_t listed[2];        // entries of the list (per binding)
    unsigned long long nonfinite;   // fused shrink: slots whose B holds Inf or NaN
};
// stage_info flags
constexpr uint32_t kStageCommit = 0x100u;   // after this stage the accumulator holds an output: commit it to the epilogue
constexpr uint32_t kStageAcc1 = 0x200u;     // the stage belongs to accumulator 1 (else 0)

static_assert(sizeof(GemmCtrl) <= 256, "control block");
constexpr uint32_t kStageBoth = 0x2000u;    // split-K dual form: the stage's product goes into both bindings' accumulators
constexpr uint32_t kStageMore0 = 0x8000u, kStageMore1 = 0x10000u;   // tall tiles, on the last k-block: LoRA stages follow for the first / second row tile
constexpr uint32_t kStageOneB = 0x1000u;    // a LoRA chunk whose u is three blocks: a K-step each, with the same block of B
constexpr uint32_t kStageChunks = 0x4000u;  // LoRA chunks (no-swizzle operands), a K-step each

// Fused shrink: a pass computes up to four chunks of a row tile, x[tile].A^T over all of K, two k-blocks to a stage.
constexpr int kShrMaxPasses = 4;
constexpr int kShrChunks = 4;
struct ShrPass {
    int32_t m;          // row tile
    int32_t n;          // chunks in this pass
    int32_t first;      // number of the first among the tile's chunks
    int32_t flag;       // the pass's number among all passes of the call: the flag it raises
    int32_t slot[kShrChunks];
    int32_t c[kShrChunks];
};
struct ShrPlan {
    int32_t npass;
    int32_t epoch;
    int32_t pad[2];
    ShrPass pass[kShrMaxPasses];
};
static_assert(sizeof(ShrPlan) <= 512, "shrink plan");

// One chunk of a stage: the block of u (number `index` of row tile m) and the chunk's rows of B for columns
// [n * BN, + BN), each contiguous.  entry = slot | chunk << 8.
template <int BN>
__device__ __forceinline__ void load_chunk(const GemmPart& pt, const __nv_bfloat16* u, int m, int n, uint32_t entry, int index, int k,
                                           uint32_t a_dst, uint32_t b_dst, uint32_t bar)
{
    mbar_expect_tx(bar, kUBlockBytes + BN * kChunk * 2);
    bulk_load(a_dst + (uint32_t)(k * kUBlockBytes), u + ((size_t)m * pt.cap + index) * (kTileM * kChunk), kUBlockBytes, bar);
    const size_t chunk = (size_t)(entry & 0xffu) * (kRankPad / kChunk) + (size_t)((entry >> 8) & 0xfu);
    bulk_load(b_dst + (uint32_t)(k * BN * kChunk * 2), pt.bk + (chunk * pt.n_pad + (size_t)n * BN) * kChunk, BN * kChunk * 2, bar);
}
// ... and the other two blocks of a u of three
__device__ __forceinline__ void load_u_rest(const GemmPart& pt, int m, int index, uint32_t a_dst, uint32_t bar)
{
    const size_t at = ((size_t)m * pt.cap + index) * (kTileM * kChunk);
    mbar_expect_tx(bar, 2 * kUBlockBytes);
    bulk_load(a_dst + kUBlockBytes, pt.u_mid + at, kUBlockBytes, bar);
    bulk_load(a_dst + 2 * kUBlockBytes, pt.u_lo + at, kUBlockBytes, bar);
}
// Early start: the live slots' rows of B for this CTA's columns start on their way into L2 (a hint; the warps that will
// run the epilogue have nothing else to do).  rank, S: this CTA's share of the chunks.
template <int BN>
__device__ __forceinline__ void prefetch_b(const GemmPart& pt, int n, int lane, int rank, int S)
{
    for (int i = lane; i < kMaxChunks; i += 32) {
        const int s = i / (kRankPad / kChunk), c = i % (kRankPad / kChunk);
        if (((pt.live >> s) & 1ull) && c < slot_chunks(pt, s) && (s + c) % S == rank)
            bulk_prefetch_to_l2(pt.bk + ((size_t)i * pt.n_pad + (size_t)n * BN) * kChunk, BN * kChunk * 2);
    }
}

// kTall: a tile is two row tiles high (256 x 256).  Both accumulators belong to the tile, each row tile has four epilogue
// warps of its own, and a stage holds two tiles of x beside one of W0: 64 KB for 1024 cycles of the tensor cores where the
// single tile moves 48 KB for 512.  A CTA covers what a pair of CTAs does, so a call whose tall tiles take no more than a round leaves
// SMs to bind_shrink, or to the shrink's passes, which only this form takes inside.  (No dual form.)
template <int BN, bool kTall>
__global__ void __launch_bounds__(kTall ? kGemmThreadsTall : kGemmThreads, 1) lora_gemm_sm100_kernel(
    const __grid_constant__ GemmParams p, const __grid_constant__ SlotSnapshot snap)
{
    using Cfg = GemmCfg<BN, kTall>;
    constexpr int kRowTiles = Cfg::kRowTiles;
    constexpr int kThreads = kTall ? kGemmThreadsTall : kGemmThreads;
    const bool dual = !kTall && p.u2 != nullptr, fused = kTall && p.fused;
    extern __shared__ uint8_t smem_raw[];
    // 128-byte swizzled tiles need 1024-byte alignment
    const uint32_t raw_addr = smem_u32(smem_raw);
    const uint32_t tiles_addr = (raw_addr + 1023u) & ~1023u;
    uint8_t* tiles_ptr = smem_raw + (tiles_addr - raw_addr);
    const uint32_t epi_addr = tiles_addr + Cfg::kStages * Cfg::kStageBytes;
    uint8_t* epi_ptr = tiles_ptr + Cfg::kStages * Cfg::kStageBytes;
    GemmCtrl* ctrl = reinterpret_cast<GemmCtrl*>(epi_ptr + Cfg::kEpiBytes);
    ShrPlan* shr = reinterpret_cast<ShrPlan*>(reinterpret_cast<uint8_t*>(ctrl) + 256);
    unsigned long long* tile_mask = reinterpret_cast<unsigned long long*>(reinterpret_cast<uint8_t*>(shr) + 512);   // [row tile] the slots in use
    int32_t* seg_cache = reinterpret_cast<int32_t*>(tile_mask + kFuseTilesInKernel);
    uint16_t* shr_base = reinterpret_cast<uint16_t*>(seg_cache + kBindSegs + 1);   // [row tile] first pass; kFuseTilesInKernel + 1 entries
    int8_t* slot_cache = reinterpret_cast<int8_t*>(shr_base + kFuseTilesInKernel + 2);
    uint32_t* list0 = reinterpret_cast<uint32_t*>(slot_cache + kBindSegs);   // chunks of the CTA's first tile

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int num_tiles = p.num_tiles;
    const int num_kb = (p.K + kBK - 1) / kBK;
    const int num_mt = (p.num_m + kRowTiles - 1) / kRowTiles;   // tiles along the rows

    if (threadIdx.x == 0) {
        for (int s = 0; s < Cfg::kStages; ++s) {
            mbar_init(smem_u32(&ctrl->full[s]), 1);
            mbar_init(smem_u32(&ctrl->empty[s]), 1);
        }
        for (int a = 0; a < 2; ++a) {
            mbar_init(smem_u32(&ctrl->tmem_full[a]), 1);
            mbar_init(smem_u32(&ctrl->tmem_empty[a]), 4);
            mbar_init(smem_u32(&ctrl->tmem_read1[a]), 4);
        }
        mbar_init(smem_u32(&ctrl->plan_full), 1);
        ctrl->abort = 0;
        ctrl->nonfinite = 0ull;
        fence_mbar_init();
    }
    if (warp == 0 && lane == 0) {
        prefetch_tmap(&p.x);
        for (int i = 0; i < p.P; ++i) { prefetch_tmap(&p.part[i].w); prefetch_tmap(&p.part[i].y); }
        if (dual) prefetch_tmap(&p.y2);
    }
    if (warp == 1) tmem_alloc(smem_u32(&ctrl->tmem_base), Cfg::kTmemCols);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = ctrl->tmem_base;
    volatile int* abort = &ctrl->abort;
    const uint64_t once = policy_evict_first();   // (see there)
    if (p.x_flag) {   // early start: the first k-blocks' W0, then x
        const GemmPart& pt = p.part[part_of(p, (int)blockIdx.x)];
        const int n0 = ((int)blockIdx.x - pt.tile0) / num_mt;
        if (warp == 0) {
            if (elect_one()) {
                for (int kb = 0; kb < min(Cfg::kStages, num_kb); ++kb) {
                    const uint32_t bar = smem_u32(&ctrl->full[kb]);
                    mbar_expect_tx(bar, Cfg::kBBytes);
                    tma_load_2d_once(tiles_addr + kb * Cfg::kStageBytes + Cfg::kABytes, &pt.w, bar, kb * kBK, n0 * BN, once);
                }
                wait_x(p.x_flag, p.call_id);
            }
        } else if (warp == 2) {
            prefetch_b<BN>(pt, n0, lane, 0, 1);
        }
        __syncthreads();
    }
    if (!p.lora || fused) {   // no launch of this call came before this one: wait for foreign work here
        grid_dependency_wait();
        grid_launch_dependents();
    }
    const bool by_segment = p.rows.mode == kRowsSegments;
    if (fused) {
        // Every CTA works out the slots of all row tiles from its own copy of the segment arrays (checked here: all reach
        // the same verdict) or from the slot per row.
        int bad_off = 0, bad_slot = 0;
        const uint32_t any_nonfinite = threadIdx.x < kMaxSlots ? ld_after_wait(p.part[0].nonfinite) : 0u;
        for (int m = threadIdx.x; m < p.num_m; m += kThreads) tile_mask[m] = 0ull;
        if (by_segment) {
            const int G = p.rows.G;
            for (int g = threadIdx.x; g <= G; g += kThreads) seg_cache[g] = ld_after_wait(p.rows.seg_offsets + g);
            for (int g = threadIdx.x; g < G; g += kThreads) {
                const int s = ld_after_wait(p.rows.ids + g);
                slot_cache[g] = (int8_t)(slot_rank(snap, s) > 0 ? s : (s == -1 ? -1 : -2));
            }
            __syncthreads();
            for (int g = threadIdx.x; g < G; g += kThreads) {
                const int s0 = seg_cache[g], s1 = seg_cache[g + 1];
                if (s1 < s0 || s0 < 0 || s1 > p.T) bad_off = 1;
                if (slot_cache[g] == -2 && s1 > s0) bad_slot = 1;   // an empty segment may name anything
            }
            if (threadIdx.x == 0 && (seg_cache[0] != 0 || seg_cache[G] != p.T)) bad_off = 1;
            bad_off = __syncthreads_or(bad_off);
            bad_slot = __syncthreads_or(bad_slot);
            if (!bad_off)
                for (int g = threadIdx.x; g < G; g += kThreads) {
                    const int s0 = seg_cache[g], s1 = seg_cache[g + 1], s = slot_cache[g];
                    if (s >= 0 && s1 > s0)
                        for (int m = s0 / kBM; m <= (s1 - 1) / kBM; ++m) atomicOr(&tile_mask[m], 1ull << s);
                }
            if (threadIdx.x == 0 && blockIdx.x == 0) {
                const unsigned f = (bad_off ? LML_FLAG_BAD_OFFSETS : 0u) | (bad_slot ? LML_FLAG_BAD_SLOT : 0u);
                if (f) atomicOr(p.status, f);
            }
        } else {
            __syncthreads();
            for (int row = threadIdx.x; row < p.T; row += kThreads) {
                const int s = p.rows.rows[row];
                if (slot_rank(snap, s) > 0) atomicOr(&tile_mask[row / kBM], 1ull << s);
            }
        }
        __syncthreads();
        const GemmPart& pt = p.part[0];
        if (any_nonfinite && ld_after_wait(pt.nonfinite + 1 + threadIdx.x) == nonfinite_tag(snap.gen[threadIdx.x])) atomicOr(&ctrl->nonfinite, 1ull << threadIdx.x);
        for (int m = threadIdx.x; m < p.num_m; m += kThreads)
            shr_base[m + 1] = (uint16_t)((mask_chunks(pt, tile_mask[m]) + kShrChunks - 1) / kShrChunks);
        __syncthreads();
        if (threadIdx.x == 0) {
            // The passes are numbered through all row tiles (shr_base[m] = first pass of tile m); pass i is the work of CTA
            // grid-1 - (i mod grid): the CTAs at the end of the grid own the fewest output tiles, and the passes of a row
            // tile run side by side on different CTAs.
            shr->epoch = (int32_t)(*reinterpret_cast<volatile uint32_t*>(p.fuse_sync));
            shr_base[0] = 0;
            for (int m = 0; m < p.num_m; ++m) shr_base[m + 1] = (uint16_t)(shr_base[m] + shr_base[m + 1]);
            const int total = shr_base[p.num_m];
            int np = 0, m = 0;
            for (int i = (int)gridDim.x - 1 - (int)blockIdx.x; i < total && np < kShrMaxPasses; i += (int)gridDim.x) {
                while (shr_base[m + 1] <= i) ++m;
                ShrPass& ps = shr->pass[np++];
                ps.m = m; ps.flag = i; ps.n = 0;
                ps.first = (i - shr_base[m]) * kShrChunks;
                int at = 0;
                for (unsigned long long mk = tile_mask[m]; mk; mk &= mk - 1ull) {
                    const int s = __ffsll((long long)mk) - 1;
                    for (int c = 0; c < slot_chunks(pt, s); ++c, ++at)
                        if (at >= ps.first && at < ps.first + kShrChunks) { ps.slot[ps.n] = s; ps.c[ps.n] = c; ++ps.n; }
                }
            }
            shr->npass = np;
        }
        __syncthreads();
    }

    if (warp == 0) {
        // ------------------------------------------------------------------ TMA producer
        // Stage order.  A tile is its base k-blocks followed by its LoRA chunks, up to four to a stage; the last stage
        // carries kStageCommit.  In the dual form every tile has a second output, the same accumulator plus (second
        // slots' delta minus first slots' delta): the chunks of both bindings again, with the blocks that hold that
        // difference.  These "delta stages" can only run once the epilogue has read the first output, so they are slipped
        // into the middle of the NEXT tile's k-blocks (or follow the last tile), where the MMA thread does not have to
        // wait for that.
        if (elect_one()) {
            bool lora = false, lora_known = !p.lora;
            // the CTA's first tile: its chunks are listed in shared memory
            const GemmPart* const list0_part = &p.part[part_of(p, (int)blockIdx.x)];
            const int list0_m = ((int)blockIdx.x - list0_part->tile0) % num_mt * kRowTiles, list0_n = ((int)blockIdx.x - list0_part->tile0) / num_mt;
            int stage = 0;
            uint32_t phase = 0;
            bool ok = true;
            auto acquire = [&]() -> bool {
                return mbar_wait(smem_u32(&ctrl->empty[stage]), phase ^ 1u, abort);
            };
            auto advance = [&]() { if (++stage == Cfg::kStages) { stage = 0; phase ^= 1u; } };
            auto learn_lora = [&]() {
                // Everything the launch before this one wrote (plans, u blocks) is first touched after the
                // base k-blocks of the first tile are already in flight.
                if (!lora_known) {
                    if (!fused) {   // (warp 2 has waited for that launch, and has let the next one go)
                        ok = mbar_wait(smem_u32(&ctrl->plan_full), 0u, abort);
                        grid_dependency_wait();
                    }
                    lora = true;
                    lora_known = true;
                }
            };
            // fused shrink: the u blocks of row tile m are written by other CTAs of this grid, which raise the
            // passes' flags when they are complete (bounded wait; the flags' writers run their passes first thing)
            int flag_seen_m = -1;
            auto wait_u = [&](int m) {
                if (!fused || m == flag_seen_m) return;
                const int want = shr->epoch + 1;
                const long long t0 = clock64();
                for (int i = shr_base[m]; i < shr_base[m + 1]; ++i)
                    while (ld_acquire_gpu_s32(p.pass_flags + i) != want) {
                        if (*abort) { ok = false; return; }
                        if (clock64() - t0 > (1ll << 31)) { *abort = 1; ok = false; return; }
                    }
                fence_proxy_async_all();   // what those CTAs wrote with ordinary stores is read by bulk copies from here on
                flag_seen_m = m;
            };
            // The chunks of row tile m that rows use under the bindings `who`, up to four to a stage; `flags_last` go on the last
            // stage.  They are listed in the tile's plan; with the fused shrink, they follow
            // from the tile's slots.
            auto emit_chunks = [&](const GemmPart& pt, const __nv_bfloat16* u, int m, int n, uint32_t who, uint32_t acc_flag, uint32_t flags_last) {
                wait_u(m);
                int index = -1, c = 0, at = 0;
                const bool listed = !fused && &pt == list0_part && m == list0_m && n == list0_n;
                unsigned long long mk = fused ? tile_mask[m] : 0ull;
                const TilePlan* plan = pt.plan + m;
                const int count = fused ? 0 : (listed ? ctrl->listed[0] : ld_after_wait(&plan->count));
                auto next = [&]() -> int {   // the next chunk, or -1; index is its number
                    if (fused) {
                        if (!mk) return -1;
                        const int s = __ffsll((long long)mk) - 1, e = s | (c << 8);
                        if (++c == slot_chunks(pt, s)) { c = 0; mk &= mk - 1ull; }
                        ++index;
                        return e;
                    }
                    while (listed && at < count) {
                        const uint32_t e = list0[at++];
                        index = (int)(e >> 16);
                        if (e & who) return (int)(e & 0xffffu);
                    }
                    if (listed) return -1;
                    while (++index < count) {
                        const int e = ld_after_wait(&plan->chunk[index]);
                        if ((uint32_t)e & who) return e;
                    }
                    return -1;
                };
                int e = next();
                while (e >= 0 && ok) {
                    ok = acquire();
                    if (!ok) break;
                    const uint32_t a_dst = tiles_addr + stage * Cfg::kStageBytes, bar = smem_u32(&ctrl->full[stage]);
                    int k = 0;
                    while (k < 4 && e >= 0) {
                        load_chunk<BN>(pt, u, m, n, (uint32_t)e, index, k++, a_dst, a_dst + Cfg::kABytes, bar);
                        if (pt.u_lo) { load_u_rest(pt, m, index, a_dst, bar); k = 4; }   // (a stage to itself)
                        e = next();
                    }
                    ctrl->stage_info[stage] = (pt.u_lo ? 3u | kStageOneB : (uint32_t)k) | acc_flag | kStageChunks | (e < 0 ? flags_last : 0u);
                    mbar_arrive(bar);
                    advance();
                }
            };
            // whether any rows of tile m use a slot under the bindings `who`
            auto has_chunks = [&](const GemmPart& pt, int m, int n, uint32_t who) -> bool {
                if (!lora) return false;
                if (fused) return tile_mask[m] != 0ull;
                const bool listed = &pt == list0_part && m == list0_m && n == list0_n;
                const TilePlan* plan = pt.plan + m;
                const int count = listed ? ctrl->listed[0] : ld_after_wait(&plan->count);
                if constexpr (!kTall) {   // (tall tiles have no dual form)
                    if (dual) {
                        for (int i = 0; i < count; ++i) if ((listed ? list0[i] : ld_after_wait(&plan->chunk[i])) & who) return true;
                        return false;
                    }
                }
                return count > 0;
            };
            // a stage without operands: only its flags matter to the MMA thread
            auto emit_marker = [&](uint32_t info) {
                ok = acquire();
                if (!ok) return;
                ctrl->stage_info[stage] = info;
                mbar_arrive(smem_u32(&ctrl->full[stage]));
                advance();
            };
            // dual form: the delta stages of tile (m, n) on accumulator flag acc_flag
            auto emit_delta = [&](int m, int n, uint32_t acc_flag) {
                if (!has_chunks(p.part[0], m, n, kChunkFirst | kChunkSecond)) { emit_marker(acc_flag | kStageCommit); return; }
                emit_chunks(p.part[0], p.u2, m, n, kChunkFirst | kChunkSecond, acc_flag, kStageCommit);
            };
            int ordinal = 0, prev_m = -1, prev_n = -1;
            // this CTA's shrink passes: a pass is num_kb stages of [x k-block | A k-blocks of its pieces]
            for (int ps = 0; fused && ps < shr->npass && ok; ++ps, ++ordinal) {
                const ShrPass& sp = shr->pass[ps];
                const uint32_t acc_flag = (ordinal & 1) ? kStageAcc1 : 0u;
                // (a k-block of a pass is at most 24 KB: two share a stage, so that as many bytes are on their way
                // as in the tiles' stages)
                const int sub_bytes = Cfg::kXBytes + sp.n * (kChunk * kBK * 2);
                const int per_stage = 2 * sub_bytes <= Cfg::kStageBytes ? 2 : 1;
                for (int kb = 0; kb < num_kb && ok; kb += per_stage) {
                    ok = acquire();
                    if (!ok) break;
                    const int nsub = min(per_stage, num_kb - kb);
                    const uint32_t bar = smem_u32(&ctrl->full[stage]);
                    ctrl->stage_info[stage] = 4u | acc_flag | ((uint32_t)sp.n << 16) | ((uint32_t)nsub << 20) |
                                              (kb + nsub >= num_kb ? kStageCommit : 0u);
                    mbar_arrive_expect_tx(bar, (uint32_t)(nsub * (p.x_bytes + sp.n * (kChunk * kBK * 2))));
                    for (int j = 0; j < nsub; ++j) {
                        const uint32_t a_dst = tiles_addr + stage * Cfg::kStageBytes + j * sub_bytes;
                        tma_load_2d(a_dst, &p.x, bar, (kb + j) * kBK, sp.m * kBM);
                        for (int i = 0; i < sp.n; ++i)
                            tma_load_3d(a_dst + Cfg::kXBytes + i * (kChunk * kBK * 2), &p.a, bar, (kb + j) * kBK, sp.c[i] * kChunk, sp.slot[i]);
                    }
                    advance();
                }
            }
            const int ahead = p.x_flag ? min(Cfg::kStages, num_kb) : 0;   // early start: k-blocks of the first tile whose W0 has been asked for already
            // k-blocks [k0, k1) of a tile; the ring's place lives in registers here (the lambdas above hold it by reference)
            auto base_blocks = [&](const CUtensorMap* w, int row0, int col0, int k0, int k1, uint32_t acc_flag, uint32_t flags_last, int have_w) {
                int st = stage;
                uint32_t ph = phase;
                bool good = ok;
                for (int kb = k0; kb < k1; ++kb) {
                    good = mbar_wait(smem_u32(&ctrl->empty[st]), ph ^ 1u, abort);
                    if (!good) break;
                    const uint32_t a_dst = tiles_addr + st * Cfg::kStageBytes;
                    const uint32_t bar = smem_u32(&ctrl->full[st]);
                    const bool second = kTall && row0 + kBM < p.T;
                    ctrl->stage_info[st] = 4u | acc_flag | (kb == num_kb - 1 ? flags_last : 0u);
                    mbar_arrive_expect_tx(bar, (uint32_t)(p.x_bytes + (second ? p.x_bytes : 0) + (kb < have_w ? 0 : Cfg::kBBytes)));
                    tma_load_2d(a_dst, &p.x, bar, kb * kBK, row0);
                    if (second) tma_load_2d(a_dst + Cfg::kXBytes, &p.x, bar, kb * kBK, row0 + kBM);
                    if (kb >= have_w) tma_load_2d_once(a_dst + Cfg::kABytes, w, bar, kb * kBK, col0, once);
                    if (++st == Cfg::kStages) { st = 0; ph ^= 1u; }
                }
                stage = st; phase = ph; ok = good;
            };
            for (int tile = blockIdx.x; tile < num_tiles && ok; tile += gridDim.x, ++ordinal) {
                const GemmPart& pt = p.part[part_of(p, tile)];
                const int m = (tile - pt.tile0) % num_mt * kRowTiles, n = (tile - pt.tile0) / num_mt;
                const int row0 = m * kBM;
                const uint32_t acc_flag = (ordinal & 1) ? kStageAcc1 : 0u;
                const int mid = min((num_kb + 1) / 2, num_kb - 1);
                int from = 0;
                if (dual && prev_m >= 0) {
                    base_blocks(&pt.w, row0, n * BN, 0, mid, acc_flag, 0u, 0);
                    from = mid;
                    if (!ok) break;
                    learn_lora();
                    if (ok) emit_delta(prev_m, prev_n, acc_flag ^ kStageAcc1);
                    if (!ok) break;
                }
                base_blocks(&pt.w, row0, n * BN, from, num_kb - 1, acc_flag, 0u, ordinal == 0 ? ahead : 0);
                if (!ok) break;
                learn_lora();
                if (!ok) break;
                const bool chunks = has_chunks(pt, m, n, kChunkFirst);
                if constexpr (kTall) {
                    const bool chunks1 = m + 1 < p.num_m && has_chunks(pt, m + 1, n, kChunkFirst);
                    base_blocks(&pt.w, row0, n * BN, num_kb - 1, num_kb, 0u, (chunks ? kStageMore0 : 0u) | (chunks1 ? kStageMore1 : 0u), ordinal == 0 ? ahead : 0);
                    if (ok && chunks) emit_chunks(pt, pt.u, m, n, kChunkFirst, 0u, kStageCommit);
                    if (ok && chunks1) emit_chunks(pt, pt.u, m + 1, n, kChunkFirst, 0u, kStageCommit);
                } else {
                    base_blocks(&pt.w, row0, n * BN, num_kb - 1, num_kb, acc_flag, chunks ? 0u : kStageCommit, ordinal == 0 ? ahead : 0);
                    if (ok && chunks) emit_chunks(pt, pt.u, m, n, kChunkFirst, acc_flag, kStageCommit);
                }
                prev_m = m; prev_n = n;
            }
            if (ok && dual && prev_m >= 0) {
                learn_lora();
                emit_delta(prev_m, prev_n, ((ordinal - 1) & 1) ? kStageAcc1 : 0u);
            }
            // Leave only after every load issued above has landed (its stage was consumed or its
            // full barrier completed): wait for the ring to drain.
            for (int i = 0; i < Cfg::kStages && ok; ++i) { ok = acquire(); advance(); }
        }
    } else if (warp == 1) {
        // ------------------------------------------------------------------ MMA issuer
        // Walks the same schedule as the producer.  The base k-blocks are always four K-steps and need no
        // side-band word; the last one, the LoRA stages after it and the delta stages carry one (how
        // many K-steps, and whether an output is complete after the stage).
        if (elect_one()) {
            constexpr uint32_t idesc = umma_idesc_bf16(kBM, BN);
            int stage = 0;
            uint32_t phase = 0;
            uint32_t empty_ph0 = 0, empty_ph1 = 0, read1_ph0 = 0, read1_ph1 = 0;
            bool ok = true;
            // one stage: ksteps MMAs into d_tmem, then the stage goes back to the producer
            auto issue = [&](uint32_t d_tmem, int ksteps, bool chunks, bool one_b, uint32_t& accumulate) {
                const uint32_t a_addr = tiles_addr + stage * Cfg::kStageBytes;
                const uint64_t adesc = chunks ? umma_desc_k16(a_addr) : umma_desc_k128(a_addr);
                const uint64_t bdesc = chunks ? umma_desc_k16(a_addr + Cfg::kABytes) : umma_desc_k128(a_addr + Cfg::kABytes);
                // 16 bf16 columns = 32 bytes further along the swizzled row: +2 in 16-byte units; a chunk is a block of its own
                const uint64_t astep = chunks ? kUBlockBytes / 16 : 2, bstep = one_b ? 0 : (chunks ? BN * kChunk * 2 / 16 : 2);
#pragma unroll 4
                for (int k = 0; k < ksteps; ++k) {
                    umma_bf16(d_tmem, adesc + (uint64_t)k * astep, bdesc + (uint64_t)k * bstep, idesc, accumulate);
                    accumulate = 1;
                }
                umma_commit(smem_u32(&ctrl->empty[stage]));
                if (++stage == Cfg::kStages) { stage = 0; phase ^= 1u; }
            };
            // `count` k-blocks without a side-band word: the loop that the tensor cores wait for; its state lives in registers
            // (tall tiles: both halves, the second's product right behind the first's)
            auto base_stages = [&](uint32_t d_tmem, int count, uint32_t& accumulate, bool second) {
                int st = stage;
                uint32_t ph = phase, on = accumulate;
                bool good = true;
                const uint64_t adesc0 = umma_desc_k128(tiles_addr), bdesc0 = umma_desc_k128(tiles_addr + Cfg::kABytes);
                const uint32_t full0 = smem_u32(&ctrl->full[0]), empty0 = smem_u32(&ctrl->empty[0]);
                for (int i = 0; i < count; ++i) {
                    good = mbar_wait(full0 + 8u * (uint32_t)st, ph, abort);
                    if (!good) break;
                    const uint64_t at = (uint64_t)((uint32_t)st * (uint32_t)(Cfg::kStageBytes / 16));
#pragma unroll
                    for (int k = 0; k < 4; ++k)
                        umma_bf16(d_tmem, adesc0 + at + (uint64_t)(k * 2), bdesc0 + at + (uint64_t)(k * 2), idesc, k == 0 ? on : 1u);
                    if (kTall && second) {
#pragma unroll
                        for (int k = 0; k < 4; ++k)
                            umma_bf16(d_tmem + (uint32_t)BN, adesc0 + at + (uint64_t)(Cfg::kXBytes / 16 + k * 2), bdesc0 + at + (uint64_t)(k * 2), idesc, k == 0 ? on : 1u);
                    }
                    on = 1u;
                    umma_commit(empty0 + 8u * (uint32_t)st);
                    if (++st == Cfg::kStages) { st = 0; ph ^= 1u; }
                }
                stage = st; phase = ph; accumulate = on; ok = good;
            };
            // stages with a side-band word, up to and including the one that completes an output
            auto flagged_stages = [&](int acc, uint32_t& accumulate) {
                const uint32_t d_tmem = tmem_base + (uint32_t)(acc * BN);
                for (bool more = true; more && ok;) {
                    ok = mbar_wait(smem_u32(&ctrl->full[stage]), phase, abort);
                    if (!ok) break;
                    const uint32_t info = ctrl->stage_info[stage];
                    more = (info & kStageCommit) == 0;
                    issue(d_tmem, (int)(info & 0xffu), (info & kStageChunks) != 0, (info & kStageOneB) != 0, accumulate);
                }
                if (ok) umma_commit(smem_u32(&ctrl->tmem_full[acc]));
            };
            // the second output of the tile that sits in accumulator acc: once the epilogue has read the
            // first, add (second slots' delta - first slots' delta) on top
            auto delta_stages = [&](int acc) {
                uint32_t& ph = acc ? read1_ph1 : read1_ph0;
                ok = mbar_wait(smem_u32(&ctrl->tmem_read1[acc]), ph, abort);
                if (!ok) return;
                ph ^= 1u;
                tc_fence_after();
                uint32_t accumulate = 1;
                flagged_stages(acc, accumulate);
            };
            int ordinal = 0;
            // this CTA's shrink passes: 128 x (16 per chunk) products
            for (int ps = 0; fused && ps < shr->npass && ok; ++ps, ++ordinal) {
                const int acc = ordinal & 1;
                uint32_t& eph = acc ? empty_ph1 : empty_ph0;
                ok = mbar_wait(smem_u32(&ctrl->tmem_empty[acc]), eph ^ 1u, abort);
                if (!ok) break;
                eph ^= 1u;
                tc_fence_after();
                const uint32_t d_tmem = tmem_base + (uint32_t)(acc * BN);
                bool fresh = true;
                for (bool more = true; more && ok;) {
                    ok = mbar_wait(smem_u32(&ctrl->full[stage]), phase, abort);
                    if (!ok) break;
                    const uint32_t info = ctrl->stage_info[stage];
                    more = (info & kStageCommit) == 0;
                    const int nch = (int)((info >> 16) & 7u), nsub = (int)((info >> 20) & 3u);
                    const int sub_bytes = Cfg::kXBytes + nch * (kChunk * kBK * 2);
                    const uint32_t idesc_n = umma_idesc_bf16(kBM, nch * kChunk);
                    tc_fence_after();
                    for (int j = 0; j < nsub; ++j) {
                        const uint32_t a_addr = tiles_addr + stage * Cfg::kStageBytes + j * sub_bytes;
                        const uint64_t adesc = umma_desc_k128(a_addr);
                        const uint64_t bdesc = umma_desc_k128(a_addr + Cfg::kXBytes);
#pragma unroll
                        for (int k = 0; k < 4; ++k)
                            umma_bf16(d_tmem, adesc + (uint64_t)(k * 2), bdesc + (uint64_t)(k * 2), idesc_n, (!fresh || k > 0) ? 1u : 0u);
                        fresh = false;
                    }
                    umma_commit(smem_u32(&ctrl->empty[stage]));
                    if (++stage == Cfg::kStages) { stage = 0; phase ^= 1u; }
                }
                if (ok) umma_commit(smem_u32(&ctrl->tmem_full[acc]));
            }
            for (int tile = blockIdx.x; kTall && tile < num_tiles && ok; tile += gridDim.x) {
                const GemmPart& pt = p.part[part_of(p, tile)];
                const bool second = (tile - pt.tile0) % num_mt * kRowTiles + 1 < p.num_m;
                ok = mbar_wait(smem_u32(&ctrl->tmem_empty[0]), empty_ph0 ^ 1u, abort);
                if (ok && second) ok = mbar_wait(smem_u32(&ctrl->tmem_empty[1]), empty_ph1 ^ 1u, abort);
                if (!ok) break;
                empty_ph0 ^= 1u;
                if (second) empty_ph1 ^= 1u;
                tc_fence_after();
                uint32_t accumulate = 0;
                base_stages(tmem_base, num_kb - 1, accumulate, second);
                if (!ok) break;
                ok = mbar_wait(smem_u32(&ctrl->full[stage]), phase, abort);
                if (!ok) break;
                const uint32_t info = ctrl->stage_info[stage];
                base_stages(tmem_base, 1, accumulate, second);
                if (info & kStageMore0) flagged_stages(0, accumulate);
                else umma_commit(smem_u32(&ctrl->tmem_full[0]));
                if (!ok || !second) continue;
                if (info & kStageMore1) flagged_stages(1, accumulate);
                else umma_commit(smem_u32(&ctrl->tmem_full[1]));
            }
            for (int tile = blockIdx.x; !kTall && tile < num_tiles && ok; tile += gridDim.x, ++ordinal) {
                const int acc = ordinal & 1;
                uint32_t& eph = acc ? empty_ph1 : empty_ph0;
                ok = mbar_wait(smem_u32(&ctrl->tmem_empty[acc]), eph ^ 1u, abort);
                if (!ok) break;
                eph ^= 1u;
                tc_fence_after();
                const uint32_t d_tmem = tmem_base + (uint32_t)(acc * BN);
                uint32_t accumulate = 0;
                int from = 0;
                if (dual && ordinal > 0) {
                    from = min((num_kb + 1) / 2, num_kb - 1);
                    base_stages(d_tmem, from, accumulate, false);
                    if (ok) delta_stages(acc ^ 1);
                    if (!ok) break;
                }
                base_stages(d_tmem, num_kb - 1 - from, accumulate, false);
                if (!ok) break;
                flagged_stages(acc, accumulate);   // the last k-block and the tile's LoRA pieces
            }
            if (ok && dual && ordinal > 0) delta_stages((ordinal - 1) & 1);
        }
    } else {
        // ------------------------------------------------------------------ epilogue warps
        const int q = warp & 3;                 // TMEM lane quarter this warp may read
        const int ew = warp - 2;
        const int group = ew >> 2;              // tall tiles: the row tile, and accumulator, of these four warps
        constexpr int kBufs = Cfg::kEpiBufs;
        const bool one = elect_one();           // the lane that issues the stores
        const uint32_t buf_addr0 = epi_addr + (uint32_t)(ew * kBufs * kEpiBufBytes);
        uint8_t* buf_ptr0 = epi_ptr + ew * kBufs * kEpiBufBytes;
        int acc = 0;
        uint32_t full_ph0 = 0, full_ph1 = 0;
        int buf = 0;
        auto row_slot = [&](int row) -> int {   // fused shrink: the slot of a row (< 0: none)
            if (!by_segment) return p.rows.rows[row];
            int lo = 0, hi = p.rows.G;
            while (lo < hi) { const int mid = (lo + hi) >> 1; if (seg_cache[mid + 1] > row) hi = mid; else lo = mid + 1; }
            return lo < p.rows.G ? slot_cache[lo] : -1;
        };
        bool ok = true;
        if (p.lora && !fused && warp == 2) {   // nothing else to do yet: the first tile's chunks, as soon as they are known
            const GemmPart& pt = p.part[part_of(p, (int)blockIdx.x)];
            grid_dependency_wait();
            grid_launch_dependents();
            const int n = list_chunks(pt.plan + ((int)blockIdx.x - pt.tile0) % num_mt * kRowTiles, kChunkFirst | kChunkSecond, 0, 1, lane, list0);
            __syncwarp();
            if (lane == 0) { ctrl->listed[0] = n; mbar_arrive(smem_u32(&ctrl->plan_full)); }
        } else if (p.lora && !fused) {
            grid_dependency_wait();   // (this warp reads the plans too)
        }
        // this CTA's shrink passes: scale, zero the rows of other slots, round, write the u blocks; then the pass's
        // flag goes up (release: the four warps' stores are complete)
        for (int ps = 0; fused && ps < shr->npass && ok; ++ps) {
            const ShrPass& sp = shr->pass[ps];
            if (kTall && (ps & 1) != group) { acc ^= 1; continue; }
            uint32_t& fph = acc ? full_ph1 : full_ph0;
            ok = mbar_wait_warp(smem_u32(&ctrl->tmem_full[acc]), fph, abort);
            if (!ok) break;
            fph ^= 1u;
            tc_fence_after();
            const int pos = sp.m * kBM + q * 32 + lane;
            const int my_slot = pos < p.T ? row_slot(pos) : -1;
#pragma unroll 1
            for (int i0 = 0; i0 < sp.n; i0 += 2) {   // two chunks, 32 columns at a time
                uint32_t r[32];
                tmem_ld_32x32(tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)(acc * BN + kChunk * i0), r);
                tmem_ld_wait();
#pragma unroll
                for (int ii = 0; ii < 2; ++ii) {
                    const int i = i0 + ii;
                    if (i >= sp.n) continue;
                    const bool mine = my_slot == sp.slot[i];
                    const float sc = snap.scale[sp.slot[i]];
                    const int have = (int)snap.rank[sp.slot[i]] - sp.c[i] * kChunk;   // columns that the adapter has, of these (Inf in x times the padding of A: not into u)
                    auto at = [&](int b, int col) { return col < have ? __uint_as_float(r[b + col]) * sc : 0.f; };
                    __nv_bfloat16* out = const_cast<__nv_bfloat16*>(p.part[0].u) + ((size_t)sp.m * p.part[0].cap + sp.first + i) * (kTileM * kChunk) + chunk_elem(q * 32 + lane, 0);
#pragma unroll
                    for (int j = 0; j < 2; ++j) {
                        const int b = ii * 16, c = j * 8;
                        uint4 v;
                        v.x = pack_bf16(at(b, c + 0), at(b, c + 1));
                        v.y = pack_bf16(at(b, c + 2), at(b, c + 3));
                        v.z = pack_bf16(at(b, c + 4), at(b, c + 5));
                        v.w = pack_bf16(at(b, c + 6), at(b, c + 7));
                        if (!mine) v = make_uint4(0, 0, 0, 0);
                        *reinterpret_cast<uint4*>(out + j * 64) = v;
                    }
                }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&ctrl->tmem_empty[acc]));
            fence_proxy_async_all();   // the blocks will be read by TMA
            __threadfence();
            asm volatile("bar.sync %0, 128;" ::"r"(1 + group) : "memory");   // the four epilogue warps of the accumulator
            if ((ew & 3) == 0 && lane == 0) st_release_gpu_s32(p.pass_flags + sp.flag, shr->epoch + 1);
            acc ^= 1;
        }
        for (int tile = blockIdx.x; tile < num_tiles && ok; tile += gridDim.x) {
            const GemmPart& pt = p.part[part_of(p, tile)];
            const int m = (tile - pt.tile0) % num_mt * kRowTiles + group, n = (tile - pt.tile0) / num_mt;
            if (kTall) {
                acc = group;
                if (m >= p.num_m) continue;
            }
            const int row_base = m * kBM + q * 32;
            const bool nonfinite = p.lora && (fused ? (tile_mask[m] & ctrl->nonfinite) != 0ull : ld_after_wait(pt.nonfinite) != 0u);
            for (int pass = 0; pass < (dual ? 2 : 1) && ok; ++pass) {
                uint32_t& fph = acc ? full_ph1 : full_ph0;
                ok = mbar_wait_warp(smem_u32(&ctrl->tmem_full[acc]), fph, abort);
                if (!ok) break;
                fph ^= 1u;
                tc_fence_after();
                const bool last_pass = pass == (dual ? 1 : 0);
                const uint32_t t_addr = tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)(acc * BN);
#pragma unroll 1
                for (int c = 0; c < BN / kEpiChunkCols; ++c) {
                    uint32_t r[32];
                    tmem_ld_32x32(t_addr + (uint32_t)(c * kEpiChunkCols), r);
                    tmem_ld_wait();
                    if (c == BN / kEpiChunkCols - 1) {
                        // accumulator fully read: hand it back to the MMA warp (for the tile's second
                        // output, or for the next tile)
                        tc_fence_before();
                        __syncwarp();
                        if (lane == 0) mbar_arrive(smem_u32(last_pass ? &ctrl->tmem_empty[acc] : &ctrl->tmem_read1[acc]));
                    }
                    const int col0 = n * BN + c * kEpiChunkCols;
                    if (col0 >= pt.N || row_base >= p.T) continue;   // nothing of this chunk is inside y
                    // the buffer we are about to overwrite must have been read by its earlier store
                    if (one) tma_store_wait_read<kBufs - 1>();
                    __syncwarp();
                    uint8_t* bp = buf_ptr0 + buf * kEpiBufBytes;
                    const uint32_t ba = buf_addr0 + (uint32_t)(buf * kEpiBufBytes);
                    // row = lane: 64 bytes, four 16-byte chunks, 64-byte swizzle (chunk ^= (row >> 1) & 3)
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        uint4 v;
                        v.x = pack_bf16(__uint_as_float(r[8 * j + 0]), __uint_as_float(r[8 * j + 1]));
                        v.y = pack_bf16(__uint_as_float(r[8 * j + 2]), __uint_as_float(r[8 * j + 3]));
                        v.z = pack_bf16(__uint_as_float(r[8 * j + 4]), __uint_as_float(r[8 * j + 5]));
                        v.w = pack_bf16(__uint_as_float(r[8 * j + 6]), __uint_as_float(r[8 * j + 7]));
                        const int phys = j ^ ((lane >> 1) & 3);
                        *reinterpret_cast<uint4*>(bp + lane * 64 + phys * 16) = v;
                    }
                    if (__builtin_expect(nonfinite, 0)) {
                        int s = -1, index = -1;
                        if (fused && row_base + lane < p.T) {
                            s = row_slot(row_base + lane);
                            if (s >= 0 && ((ctrl->nonfinite >> s) & 1ull)) index = mask_chunks(pt, tile_mask[m] & ((1ull << s) - 1ull));
                        }
                        if (!fused || index >= 0)
                            add_nonfinite(pt, m, q * 32 + lane, pass, s, index, col0, pt.u, pass ? p.u2 : pt.u_mid, pt.u_lo, bp + lane * 64, (lane >> 1) & 3);
                    }
                    fence_proxy_async_smem();
                    __syncwarp();
                    if (one) {
                        if (pass == 0) tma_store_2d(&pt.y, ba, col0, row_base);
                        else tma_store_2d(&p.y2, ba, col0, row_base);
                        tma_store_commit();
                    }
                    buf = kBufs == 2 ? buf ^ 1 : 0;
                }
            }
            acc ^= 1;
        }
        if (one) tma_store_wait_all();
    }

    __syncthreads();
    if (ctrl->abort) __nanosleep(50000);   // gave up: let copies still in flight land before the CTA goes away
    if (threadIdx.x == 0 && ctrl->abort) atomicOr(p.status, LML_FLAG_TIMEOUT);
    if (threadIdx.x == 0) leave_early_start(p.x_flag);
    if (threadIdx.x == 0 && fused) {
        // the last CTA to finish moves the table's epoch on: the flags of this call mean nothing to the next one
        __threadfence();
        if (atomicAdd(p.fuse_sync + 1, 1u) == gridDim.x - 1) {
            p.fuse_sync[1] = 0u;
            p.fuse_sync[0] = (uint32_t)(shr->epoch + 1);
        }
    }
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem_base, Cfg::kTmemCols);
    }
}

// ---- split-K variant for few tokens ---------------------------------------------------------------------
// With a few hundred tokens or fewer the layer is bound by the read of W0, and 128 x 256 tiles give far
// fewer CTAs than the machine has SMs.  Here a cluster of S CTAs shares one tile: CTA r multiplies its
// share of the k-blocks (and of the tile's LoRA chunks, which are just more K) into its own TMEM
// accumulator, so S times as many SMs stream W0.  The partial sums are then exchanged through
// distributed shared memory: the tile's eight 32-column chunks are dealt out to the CTAs, every CTA
// writes each chunk of its partial sums into the owner's (by then idle) stage memory, and the owner adds
// the S contributions in rank order, rounds once and writes its columns of y.  Two cluster barriers
// frame the exchange: nobody writes into a CTA that is still multiplying, nobody adds before all
// have written.  Warp roles and the stage ring are those of the kernel above; every stage carries its
// side-band word.
constexpr int kSplitMaxS = 8;

template <int BN>
__global__ void __launch_bounds__(kGemmThreads, 1) lora_gemm_sm100_splitk_kernel(const __grid_constant__ GemmParams p)
{
    using Cfg = GemmCfg<BN>;
    constexpr int kSplitChunks = BN / kEpiChunkCols;   // 32-column chunks of the tile: 4 or 8
    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw_addr = smem_u32(smem_raw);
    const uint32_t tiles_addr = (raw_addr + 1023u) & ~1023u;
    uint8_t* tiles_ptr = smem_raw + (tiles_addr - raw_addr);
    GemmCtrl* ctrl = reinterpret_cast<GemmCtrl*>(tiles_ptr + p.stages * Cfg::kStageBytes);
    uint32_t* lists = reinterpret_cast<uint32_t*>(reinterpret_cast<uint8_t*>(ctrl) + 256);   // this CTA's chunks, per binding
    // Dual form (two bindings of the same segments, two outputs): the k-blocks pass through shared memory once and
    // are multiplied into two accumulators (with few tokens the tensor cores have time to spare: the kernel is
    // bound by the read of W0); each binding's pieces go to its own accumulator, and the exchange runs twice.
    const bool dual = p.u2 != nullptr;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int S = (int)gridDim.x, rank = (int)blockIdx.x;   // the cluster spans the grid's x dimension
    const int m = (int)blockIdx.z;
    // (column tiles are numbered through the projections; tile0 counts row tiles too)
    const GemmPart& pt = p.part[part_of(p, (int)blockIdx.y * p.num_m)];
    const int n = (int)blockIdx.y - pt.tile0 / p.num_m;
    const int num_kb = (p.K + kBK - 1) / kBK;
    // chunks of the tile's 256 columns that CTA r reduces: [first(r), first(r + 1))
    auto first_chunk = [&](int r) { return r * kSplitChunks / S; };
    const int cpr = (kSplitChunks + S - 1) / S;   // most chunks any CTA owns

    if (threadIdx.x == 0) {
        for (int s = 0; s < p.stages; ++s) {
            mbar_init(smem_u32(&ctrl->full[s]), 1);
            mbar_init(smem_u32(&ctrl->empty[s]), 1);
        }
        mbar_init(smem_u32(&ctrl->tmem_full[0]), 1);
        mbar_init(smem_u32(&ctrl->plan_full), 1);
        ctrl->abort = 0;
        fence_mbar_init();
    }
    if (warp == 0 && lane == 0) {
        prefetch_tmap(&p.x); prefetch_tmap(&pt.w);
    }
    if (warp == 1) tmem_alloc(smem_u32(&ctrl->tmem_base), dual ? 2 * BN : BN);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = ctrl->tmem_base;
    volatile int* abort = &ctrl->abort;
    const uint64_t once = policy_evict_first();   // (see there)
    if (p.x_flag) {   // early start: the first k-blocks' W0, then x
        if (warp == 0) {
            if (elect_one()) {
                const int kb0 = rank * num_kb / S, ahead = min(p.stages, (rank + 1) * num_kb / S - kb0);
                for (int i = 0; i < ahead; ++i) {
                    const uint32_t bar = smem_u32(&ctrl->full[i]);
                    mbar_expect_tx(bar, Cfg::kBBytes);
                    tma_load_2d_once(tiles_addr + i * Cfg::kStageBytes + Cfg::kABytes, &pt.w, bar, (kb0 + i) * kBK, n * BN, once);
                }
                wait_x(p.x_flag, p.call_id);
            }
        } else if (warp == 2) {
            prefetch_b<BN>(pt, n, lane, rank, S);
        }
        __syncthreads();
    }
    if (!p.lora) {   // no launch of this call came before this one: wait for foreign work here
        grid_dependency_wait();
        grid_launch_dependents();
    }

    if (warp == 0) {
        // ------------------------------------------------------------------ TMA producer
        if (elect_one()) {
            int stage = 0;
            uint32_t phase = 0;
            bool ok = true;
            auto acquire = [&]() -> bool { return mbar_wait(smem_u32(&ctrl->empty[stage]), phase ^ 1u, abort); };
            auto advance = [&]() { if (++stage == p.stages) { stage = 0; phase ^= 1u; } };
            const int row0 = m * kBM;
            const int kb0 = rank * num_kb / S, kb1 = (rank + 1) * num_kb / S;
            // base k-blocks first: they do not depend on the launch that precedes this one
            const int ahead = p.x_flag ? min(p.stages, kb1 - kb0) : 0;   // early start: k-blocks whose W0 has been asked for already
            for (int kb = kb0; kb < kb1 && ok; ++kb) {
                ok = acquire();
                if (!ok) break;
                const uint32_t a_dst = tiles_addr + stage * Cfg::kStageBytes;
                const uint32_t bar = smem_u32(&ctrl->full[stage]);
                ctrl->stage_info[stage] = 4u | (dual ? kStageBoth : 0u);
                const bool have_w = kb - kb0 < ahead;
                mbar_arrive_expect_tx(bar, (uint32_t)(p.x_bytes + (have_w ? 0 : Cfg::kBBytes)));
                tma_load_2d(a_dst, &p.x, bar, kb * kBK, row0);
                if (!have_w) tma_load_2d_once(a_dst + Cfg::kABytes, &pt.w, bar, kb * kBK, n * BN, once);
                advance();
            }
            // This CTA's share of the tile's LoRA chunks: chunk c of slot s goes to CTA (s + c) mod S.  Which CTA adds a
            // row's LoRA term depends only on the row's own slot, so a row's bits do not change with what other rows
            // are bound to.
            if (p.lora && ok) {
                ok = mbar_wait(smem_u32(&ctrl->plan_full), 0u, abort);   // (warp 2 has waited for that launch)
                grid_dependency_wait();
                for (int side = 0; side < (dual ? 2 : 1) && ok; ++side) {
                    const __nv_bfloat16* u = side ? p.u2 : pt.u;
                    const uint32_t* list = lists + side * kMaxChunks;
                    const int count = ctrl->listed[side];
                    const int per = pt.u_lo ? 1 : 4;   // chunks to a stage
                    for (int i = 0; i < count && ok; i += per) {
                        ok = acquire();
                        if (!ok) break;
                        const uint32_t a_dst = tiles_addr + stage * Cfg::kStageBytes, bar = smem_u32(&ctrl->full[stage]);
                        int nk = 0;
                        for (int q = i; q < min(i + per, count); ++q) {
                            load_chunk<BN>(pt, u, m, n, list[q] & 0xffffu, (int)(list[q] >> 16), nk++, a_dst, a_dst + Cfg::kABytes, bar);
                            if (pt.u_lo) load_u_rest(pt, m, (int)(list[q] >> 16), a_dst, bar);
                        }
                        ctrl->stage_info[stage] = (pt.u_lo ? 3u | kStageOneB : (uint32_t)nk) | kStageChunks | (side ? kStageAcc1 : 0u);
                        mbar_arrive(bar);
                        advance();
                    }
                }
            }
            if (ok) {   // end of this CTA's K: a stage without operands
                ok = acquire();
                if (ok) {
                    ctrl->stage_info[stage] = kStageCommit;
                    mbar_arrive(smem_u32(&ctrl->full[stage]));
                    advance();
                }
            }
            // leave the role only after every load has landed and been consumed
            for (int i = 0; i < p.stages && ok; ++i) { ok = acquire(); advance(); }
        }
    } else if (warp == 1) {
        // ------------------------------------------------------------------ MMA issuer
        if (elect_one()) {
            constexpr uint32_t idesc = umma_idesc_bf16(kBM, BN);
            int stage = 0;
            uint32_t phase = 0, accumulate = 0, accumulate2 = 0;
            bool ok = true;
            for (bool more = true; more && ok;) {
                ok = mbar_wait(smem_u32(&ctrl->full[stage]), phase, abort);
                if (!ok) break;
                const uint32_t info = ctrl->stage_info[stage];
                more = (info & kStageCommit) == 0;
                const int ksteps = (int)(info & 0xffu);
                const bool chunks = (info & kStageChunks) != 0;
                const uint32_t a_addr = tiles_addr + stage * Cfg::kStageBytes;
                const uint64_t adesc = chunks ? umma_desc_k16(a_addr) : umma_desc_k128(a_addr);
                const uint64_t bdesc = chunks ? umma_desc_k16(a_addr + Cfg::kABytes) : umma_desc_k128(a_addr + Cfg::kABytes);
                const uint64_t astep = chunks ? kUBlockBytes / 16 : 2, bstep = (info & kStageOneB) ? 0 : (chunks ? BN * kChunk * 2 / 16 : 2);
                tc_fence_after();
                if ((info & kStageAcc1) == 0) {
#pragma unroll 4
                    for (int k = 0; k < ksteps; ++k) {
                        umma_bf16(tmem_base, adesc + (uint64_t)k * astep, bdesc + (uint64_t)k * bstep, idesc, accumulate);
                        accumulate = 1;
                    }
                }
                if (info & (kStageAcc1 | kStageBoth)) {   // the second binding's accumulator
#pragma unroll 4
                    for (int k = 0; k < ksteps; ++k) {
                        umma_bf16(tmem_base + (uint32_t)BN, adesc + (uint64_t)k * astep, bdesc + (uint64_t)k * bstep, idesc, accumulate2);
                        accumulate2 = 1;
                    }
                }
                umma_commit(smem_u32(&ctrl->empty[stage]));
                if (++stage == p.stages) { stage = 0; phase ^= 1u; }
            }
            if (ok) umma_commit(smem_u32(&ctrl->tmem_full[0]));
            ctrl->pad[0] = (int32_t)accumulate;    // 0: this CTA had no K at all, its accumulator holds nothing
            ctrl->pad[1] = (int32_t)accumulate2;   // the same for the second binding's
        }
    }
    // ---------------------------------------------------------------------- exchange and reduction
    __syncwarp();   // (the producer's and the MMA issuer's other lanes waited here: the cluster barrier wants whole warps)
    bool ok = true, nonfinite = false;
    if (warp >= 2) {
        if (p.lora && warp == 2) {   // nothing else to do yet: this CTA's share of the tile's chunks, as soon as they are known
            grid_dependency_wait();
            grid_launch_dependents();
            for (int side = 0; side < (dual ? 2 : 1); ++side) {
                const int c = list_chunks(pt.plan + m, side ? kChunkSecond : kChunkFirst, rank, S, lane, lists + side * kMaxChunks);
                if (lane == 0) ctrl->listed[side] = c;
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&ctrl->plan_full));
        } else if (p.lora) {
            grid_dependency_wait();   // (this warp reads the plan too)
        }
        if (p.lora) nonfinite = ld_after_wait(pt.nonfinite) != 0u;
        ok = mbar_wait_warp(smem_u32(&ctrl->tmem_full[0]), 0u, abort);   // this CTA's MMAs are complete: so are its loads
        if (!ok) __nanosleep(50000);   // gave up: let copies still in flight land before the stages take the partial sums
        tc_fence_after();
    }
    const int q = warp & 3;   // TMEM lane quarter an epilogue warp may read
    const int row = q * 32 + lane;
    for (int o = 0; o < (dual ? 2 : 1); ++o) {   // one exchange per output
    __nv_bfloat16* const yout = o ? p.y2_ptr : pt.y_ptr;
    cluster_sync_all();   // every CTA of the cluster is done with its stage memory (and with the exchange before this one)
    if (warp >= 2 && ok) {
        const bool have = ctrl->pad[o] != 0;
        const uint32_t t_addr = tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)(o * BN);
        int owner = 0;
#pragma unroll 1
        for (int c = 0; c < kSplitChunks; ++c) {
            while (first_chunk(owner + 1) <= c) ++owner;
            uint32_t r[32];
            tmem_ld_32x32(t_addr + (uint32_t)(c * kEpiChunkCols), r);
            tmem_ld_wait();
            if (!have) {
#pragma unroll
                for (int i = 0; i < 32; ++i) r[i] = 0u;
            }
            // slot (this CTA's rank, chunk within the owner's share) of the owner's receive area, 16 KB: the
            // 16-byte pieces of the 128 rows, piece-major, so that a warp's store is 512 contiguous bytes
            const uint32_t local = tiles_addr + (uint32_t)((rank * cpr + (c - first_chunk(owner))) * (kBM * 128) + row * 16);
            const uint32_t remote = mapa_shared(local, (uint32_t)owner);
#pragma unroll
            for (int j = 0; j < 8; ++j)
                st_shared_cluster_v4(remote + (uint32_t)(j * kBM * 16), r[4 * j], r[4 * j + 1], r[4 * j + 2], r[4 * j + 3]);
        }
        tc_fence_before();
    }
    cluster_sync_all();   // all contributions have arrived
    if (warp >= 2 && ok) {
        const int pos = m * kBM + row;
        const bool row_ok = pos < p.T;
        const int c_first = first_chunk(rank), c_end = first_chunk(rank + 1);
#pragma unroll 1
        for (int c = c_first; c < c_end; ++c) {
            float acc[32];
#pragma unroll
            for (int i = 0; i < 32; ++i) acc[i] = 0.f;
            for (int src = 0; src < S; ++src) {   // rank order: the sum does not depend on timing
                const uint8_t* rp = tiles_ptr + (size_t)(src * cpr + (c - c_first)) * (kBM * 128) + row * 16;
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    const float4 v = *reinterpret_cast<const float4*>(rp + j * kBM * 16);
                    acc[4 * j] += v.x; acc[4 * j + 1] += v.y; acc[4 * j + 2] += v.z; acc[4 * j + 3] += v.w;
                }
            }
            const int col0 = n * BN + c * kEpiChunkCols;
            if (!row_ok) continue;
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                if (col0 + j * 8 >= pt.N) continue;
                uint4 v;
                v.x = pack_bf16(acc[8 * j + 0], acc[8 * j + 1]);
                v.y = pack_bf16(acc[8 * j + 2], acc[8 * j + 3]);
                v.z = pack_bf16(acc[8 * j + 4], acc[8 * j + 5]);
                v.w = pack_bf16(acc[8 * j + 6], acc[8 * j + 7]);
                *reinterpret_cast<uint4*>(yout + (size_t)pos * pt.N + col0 + j * 8) = v;
            }
            if (__builtin_expect(nonfinite, 0))
                add_nonfinite(pt, m, row, o, -1, -1, col0, o ? p.u2 : pt.u, pt.u_mid, pt.u_lo, reinterpret_cast<uint8_t*>(yout + (size_t)pos * pt.N + col0), 0);
        }
    }
    }   // outputs
    __syncthreads();
    if (threadIdx.x == 0 && ctrl->abort) atomicOr(p.status, LML_FLAG_TIMEOUT);
    if (threadIdx.x == 0) leave_early_start(p.x_flag);
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem_base, dual ? 2 * BN : BN);
    }
}

// ---- host side ---------------------------------------------------------------------------------------

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*,
                                  CUtensorMapInterleave, CUtensorMapSwizzle, CUtensorMapL2promotion,
                                  CUtensorMapFloatOOBfill);

static EncodeTiledFn get_encode_fn()
{
    static EncodeTiledFn fn = nullptr;
    if (!fn) {
        void* sym = nullptr;
        cudaDriverEntryPointQueryResult qres;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &sym, cudaEnableDefault, &qres) == cudaSuccess &&
            qres == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<EncodeTiledFn>(sym);
    }
    return fn;
}

static CUtensorMapSwizzle swizzle_for(uint32_t box_inner_elems)
{
    return box_inner_elems * 2 >= 128 ? CU_TENSOR_MAP_SWIZZLE_128B
                                      : (box_inner_elems * 2 == 64 ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_32B);
}

bool encode_tmap_2d(CUtensorMap* m, const void* base, uint64_t inner, uint64_t outer, uint64_t row_stride_bytes,
                    uint32_t box_inner, uint32_t box_outer, bool swizzle)
{
    EncodeTiledFn fn = get_encode_fn();
    if (!fn) return false;
    cuuint64_t dims[2] = {inner, outer};
    cuuint64_t strides[1] = {row_stride_bytes};
    cuuint32_t box[2] = {box_inner, box_outer};
    cuuint32_t estr[2] = {1, 1};
    return fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box, estr,
              CU_TENSOR_MAP_INTERLEAVE_NONE, swizzle ? swizzle_for(box_inner) : CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

bool encode_tmap_3d(CUtensorMap* m, const void* base, uint64_t d0, uint64_t d1, uint64_t d2, uint64_t stride1_bytes,
                    uint64_t stride2_bytes, uint32_t b0, uint32_t b1, uint32_t b2)
{
    EncodeTiledFn fn = get_encode_fn();
    if (!fn) return false;
    cuuint64_t dims[3] = {d0, d1, d2};
    cuuint64_t strides[2] = {stride1_bytes, stride2_bytes};
    cuuint32_t box[3] = {b0, b1, b2};
    cuuint32_t estr[3] = {1, 1, 1};
    return fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(base), dims, strides, box, estr,
              CU_TENSOR_MAP_INTERLEAVE_NONE, swizzle_for(b0), CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

cudaError_t gemm_sm100_init(int /*device*/)
{
    cudaError_t e = cudaFuncSetAttribute(lora_gemm_sm100_splitk_kernel<64>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         GemmCfg<64>::split_smem(GemmCfg<64>::kStages));
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(lora_gemm_sm100_kernel<64, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, GemmCfg<64>::kSmemBytes);
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(lora_gemm_sm100_kernel<256, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, GemmCfg<256, true>::kSmemBytes);
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(lora_gemm_sm100_kernel<256, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         GemmCfg<256>::kSmemBytes);
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(lora_gemm_sm100_splitk_kernel<256>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             GemmCfg<256>::split_smem(GemmCfg<256>::kStages));
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(lora_gemm_sm100_splitk_kernel<128>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             GemmCfg<128>::split_smem(GemmCfg<128>::kStages));
    if (e != cudaSuccess) return e;
    return cudaFuncSetAttribute(lora_gemm_sm100_kernel<128, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                GemmCfg<128>::kSmemBytes);
}

// The table's override (LML_GEMM_SPLIT, read once when the table is created; a test knob): "<bn>x<split>"
// forces that shape, "512x1" tall tiles, "<bn>p" CTA pairs of that width, 0 switches the split-K kernel off.  Returns false
// when the variable is not set.  split_out: 0 for pairs.
bool gemm_split_override(int* bn_out, int* split_out)
{
    *bn_out = -1; *split_out = -1;
    const char* e = getenv("LML_GEMM_SPLIT");
    if (!e) return false;
    int bn = 0, sp = 0;
    char c = 0;
    if (sscanf(e, "%d%c", &bn, &c) == 2 && c == 'p' && bn >= 64 && bn <= 256 && bn % 32 == 0) { *bn_out = bn; *split_out = 0; return true; }
    if (sscanf(e, "%dx%d", &bn, &sp) == 2 && (bn == 64 || bn == 128 || bn == 256 || (bn == kTallOverride && sp == 1)) && sp >= 1 && sp <= kSplitMaxS &&
        (sp == 1 ? 0 : sp) * ((bn / 32 + sp - 1) / sp) * 16384 <= GemmCfg<128>::kStages * GemmCfg<128>::kStageBytes) {
        *bn_out = bn; *split_out = sp;
    } else {
        *bn_out = 0; *split_out = 0;
    }
    return true;
}

static int gemm_stages(int bn) { return bn == 256 ? GemmCfg<256>::kStages : (bn == 128 ? GemmCfg<128>::kStages : GemmCfg<64>::kStages); }
static int gemm_stages_short(int bn)
{
    return bn == 256 ? GemmCfg<256>::kSplitStagesShort : (bn == 128 ? GemmCfg<128>::kSplitStagesShort : GemmCfg<64>::kSplitStagesShort);
}
static int gemm_stage_bytes(int bn) { return (kBM + bn) * kBK * 2; }
static int gemm_exchange_bytes(int bn, int split) { return split * ((bn / 32 + split - 1) / split) * 16384; }

// The shape of a call: the smallest estimated time (us) over whole-K tiles of three widths, the splits that the machine can hold, and
// CTA pairs.  A fixed part and so much per k-block and round of tiles, from single calls with four adapters, W0 out of HBM (us per call):
// whole-K tiles of 64 / 128 / 256 columns 16.0 / 19.1 / 28.5 at 128 x 4096 -> 4096, 12.2 / 12.6 / 16.8 at 2048 -> 2048, 33.7 / 42.7 / 68.0 at
// 11008 -> 4096; splits there 128x2 34.7, 128x3 27.0, 256x4 32.5, 256x6 30.0; pairs of 256 / 160 / 128 columns 26.8 / 21.4 / 21.3 at 512 x
// 4096 -> 4096, and where the tiles take several rounds, at the power that the tensor cores may draw, 96.6 at 1300 x 4096 -> 11008 (256
// columns, four rounds), 109.3 at 1600 (224 columns, five; with 256 columns 115.9), against 111 and 128.6 for single tiles of 128.
// A pair's k-block also takes a share of a trip to memory, 1.4 us over the stages of its ring, which is what narrow pairs are bound by (256 x
// 11008 -> 4096: 64p 39.7, 64x1 32.8).  And 2 us where the tiles' CTAs and bind_shrink's do not find SMs of their own, so that some start when
// bind_shrink leaves (3000 x 3072 -> 1024: 192p, 144 CTAs, 29.7; 256x1, 96 CTAs, 21.1).  With these two, over 14 layers from 264 -> 8192 to
// 5120 -> 13824, 64 ... 4096 tokens, 4 and 16 adapters, the choice is 1.046 times the best of all shapes in the mean, 1.067 without.
// slots: of the largest table, 0 without adapters; what the tables hold must not choose between sums of different order.
GemmShape gemm_pick_shape(int T, int d_in, const int* d_outs, int P, bool dual, bool precise, int slots, int num_sms, int num_pairs, int split_bn, int split_s)
{
    static int max_clusters[3][kSplitMaxS + 1];   // for 64, 128 and 256 columns
    static std::once_flag probed;
    std::call_once(probed, [&]() {   // clusters of each size that can be resident together
        for (int w = 0; w < 3; ++w)
            for (int S = 2; S <= kSplitMaxS; ++S) {
                cudaLaunchConfig_t cfg = {};
                cfg.gridDim = dim3(S, num_sms / S, 1);
                cfg.blockDim = dim3(kGemmThreads);
                cfg.dynamicSmemBytes = w == 2 ? GemmCfg<256>::split_smem(GemmCfg<256>::kStages)
                                              : (w == 1 ? GemmCfg<128>::split_smem(GemmCfg<128>::kStages) : GemmCfg<64>::split_smem(GemmCfg<64>::kStages));
                cudaLaunchAttribute attr[1];
                attr[0].id = cudaLaunchAttributeClusterDimension;
                attr[0].val.clusterDim.x = S; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
                cfg.attrs = attr; cfg.numAttrs = 1;
                int n = 0;
                cudaError_t e = w == 2 ? cudaOccupancyMaxActiveClusters(&n, lora_gemm_sm100_splitk_kernel<256>, &cfg)
                                       : (w == 1 ? cudaOccupancyMaxActiveClusters(&n, lora_gemm_sm100_splitk_kernel<128>, &cfg)
                                                 : cudaOccupancyMaxActiveClusters(&n, lora_gemm_sm100_splitk_kernel<64>, &cfg));
                if (e != cudaSuccess) { n = 0; (void)cudaGetLastError(); }
                max_clusters[w][S] = n;
            }
    });
    const int num_m = (T + kBM - 1) / kBM, num_kb = (d_in + kBK - 1) / kBK;
    auto tiles_of = [&](int bn) {
        int tiles = 0;
        for (int p = 0; p < P; ++p) tiles += num_m * ((d_outs[p] + bn - 1) / bn);
        return tiles;
    };
    auto pair_tiles_of = [&](int bn) {
        int tiles = 0;
        for (int p = 0; p < P; ++p) tiles += (num_m + 1) / 2 * ((d_outs[p] + bn - 1) / bn);
        return tiles;
    };
    const bool pairs = num_pairs > 0 && !dual && !precise;   // (the pair kernel has neither a second output nor a u of three values)
    if (split_bn > 0 && split_s == 0) {
        if (pairs) return {split_bn, 1, 2 * pair_tiles_of(split_bn), true};
        split_bn = 0;
    }
    if (split_bn == kTallOverride) {
        if (!dual) return {256, 1, pair_tiles_of(256), false, true};
        split_bn = 0;
    }
    if (split_bn > 0) return {split_bn, split_s, tiles_of(split_bn) * split_s, false};
    float w0_bytes = 0.f;
    for (int p = 0; p < P; ++p) w0_bytes += 2.f * (float)d_in * (float)d_outs[p];
    const float stream_us = 7.5f + w0_bytes / 5.45e6f;   // no shape reads W0 faster
    GemmShape best = {256, 1, tiles_of(256), false};
    float best_us = 1e30f;
    const int bind_ctas = slots > 0 ? bind_ctas_reckoned(T, d_in, P, slots, num_sms) : 0;
    auto consider = [&](const GemmShape& shape, float us) {
        us = (us > stream_us ? us : stream_us) + 0.1f * us;
        if (bind_ctas > 0 && shape.ctas + bind_ctas > num_sms) us += 2.f;
        if (us < best_us * 0.999f) { best_us = us; best = shape; }
    };
    for (int w = 2; w >= 0; --w) {
        const int bn = 64 << w, tiles = tiles_of(bn);
        const int waves = (tiles + num_sms - 1) / num_sms;
        const float t1[3] = {0.145f, 0.21f, 0.365f}, t2[3] = {0.185f, 0.25f, 0.41f}, a1[3] = {7.f, 5.5f, 5.f};
        consider({bn, 1, tiles, false}, a1[w] + (float)(waves * num_kb) * (waves > 1 ? t2[w] : t1[w]));
        for (int S = 2; S <= kSplitMaxS && split_bn != 0; ++S) {
            if (max_clusters[w][S] < tiles || num_kb < 8 * S || gemm_exchange_bytes(bn, S) > gemm_stages(bn) * gemm_stage_bytes(bn)) continue;
            // (a cluster needs its CTAs on one part of the chip: where they do not all find a place beside bind_shrink's, about
            // 40 CTAs, some wait for it to end)
            const bool beside = tiles * num_sms <= max_clusters[w][S] * (num_sms - 40);
            consider({bn, S, tiles * S, false}, (S <= 4 ? 5.f + 2.f * (float)S : 18.5f) + (float)((num_kb + S - 1) / S) * (w == 2 ? 0.43f : 0.29f) +
                                                    (beside ? 0.f : (S == 2 ? 1.5f : (S == 3 ? 4.f : 6.f))));
        }
    }
    // Whether K is split is settled among the single tiles, which a dual call has too: its first output has the bits of the plain call.  Whole-K
    // tiles of every form add up in one order.
    if (pairs && num_m > 1 && best.split == 1) {   // CTA pairs (lml_gemm_pair.cu), tiles of 256 rows
        for (int bn = 256; bn >= 64; bn -= 32) {
            const int tiles = pair_tiles_of(bn), waves = (tiles + num_pairs - 1) / num_pairs;
            const float trip = 1.4f / (float)gemm_pair_stages(bn), one = 0.035f + 0.00097f * (float)bn;
            consider({bn, 1, 2 * tiles, true}, 10.f + (float)(waves * num_kb) * (waves > 1 ? 0.12f + 0.00082f * (float)bn : (one > trip ? one : trip)));
        }
    }
    return best;
}

// Tensor maps of the caller's buffers are kept per table: a serving loop calls with the same few
// (pointer, shape) combinations over and over, and encoding a map costs a driver call each time.
bool TmapCache::get_2d(CUtensorMap* out, const void* base, uint64_t inner, uint64_t outer, uint64_t stride_bytes,
                       uint32_t box_inner, uint32_t box_outer, bool swizzle)
{
    std::lock_guard<std::mutex> lock(mu);
    for (int i = 0; i < used; ++i) {
        const Key& k = keys[i];
        if (k.base == base && k.inner == inner && k.outer == outer && k.stride == stride_bytes && k.box_inner == box_inner &&
            k.box_outer == box_outer && k.swizzle == swizzle) {
            *out = maps[i];
            return true;
        }
    }
    CUtensorMap m;
    if (!encode_tmap_2d(&m, base, inner, outer, stride_bytes, box_inner, box_outer, swizzle)) return false;
    const int slot = used < kEntries ? used++ : (next = (next + 1) % kEntries);
    keys[slot] = Key{base, inner, outer, stride_bytes, box_inner, box_outer, swizzle};
    maps[slot] = m;
    *out = m;
    return true;
}

// Whether the shrink runs inside the GEMM kernel: a plain call with little x (1.4 M elements) of more than one wave of 256-column tiles, as
// tall tiles; few enough row tiles for the kernel's tables, and no more passes (a pass per row tile and four chunks; every segment
// boundary inside a row tile can add one) than there are CTAs with a tile less than the others, or none: those compute u while the others'
// tiles run.  us per call back to back, inside / the same tiles behind bind_shrink / single 256-column tiles with the shrink inside: 700 x
// 520 -> 8192 18.4 / 15.2 / 26.0, 700 x 264 -> 8192 15.9 / 15.0 / 20.8, 1300 x 1032 -> 4104 24.9 / 21.0 / 32.7, 2048 x 520 -> 8192 33.1 / 28.8 /
// 42.3.  One launch instead of two: what it is for is a call alone, issued from the host.
// (What counts is T, G and the table's size, not what is registered: the two forms sum x.A^T in different orders, and a call's
// bits must not change with adapters that it does not use.  Segments in order: a tile has one pass and one more for every segment
// that begins in it, at most; rows in any order: reckoned with half of the widest adapter for every segment.)
bool gemm_fused_shape(GemmShape* shape, int T, int d_in, int d_out, int G, bool in_segment_order, int max_slots, int num_sms, int split_bn)
{
    if (G <= 0 || (in_segment_order && G > kBindSegs)) return false;
    if (split_bn > 0 && split_bn != kTallOverride) return false;
    const int num_m = (T + kBM - 1) / kBM, num_n = (d_out + 255) / 256, tall_tiles = (num_m + 1) / 2 * num_n;
    if (num_m > kFuseTilesInKernel) return false;
    if (split_bn != kTallOverride && ((long long)T * d_in > 1400000ll || num_m * num_n <= num_sms)) return false;
    static_assert(kShrChunks * kChunk == kRankPad, "a slot takes one pass at most");
    const int slots = G < max_slots ? G : max_slots;
    if (num_m * slots > kShrMaxPasses * num_sms && !in_segment_order) return false;   // (room for a CTA's passes)
    *shape = {256, 1, tall_tiles, false, true};
    return (in_segment_order ? num_m + G : num_m * ((slots + 1) / 2)) <= num_sms - (tall_tiles - 1) % num_sms - 1;
}

cudaError_t launch_gemm_sm100(const CUtensorMap& tmap_A, TmapCache* const* caches, const GemmArgs& a, cudaStream_t stream)
{
    const bool dual = a.u2 != nullptr;
    if (dual && (!a.lora || !a.y2 || a.P != 1 || a.fused)) return cudaErrorInvalidValue;
    const int bn = a.shape.bn, split = a.shape.split;
    if ((a.fused && (!a.shape.tall || a.P != 1)) || (a.shape.tall && dual)) return cudaErrorInvalidValue;
    GemmParams p;
    p.a = tmap_A;
    p.num_m = (a.T + kBM - 1) / kBM;
    const uint64_t xs = (uint64_t)a.d_in * 2;
    if (!caches[0]->get_2d(&p.x, a.x, (uint64_t)a.d_in, (uint64_t)a.T, xs, kBK, (uint32_t)x_box_rows(a.T))) return cudaErrorInvalidValue;
    p.x_bytes = x_box_rows(a.T) * kBK * 2;
    int tiles = 0, columns = 0;
    for (int i = 0; i < a.P; ++i) {
        const GemmProj& pr = a.proj[i];
        GemmPart& pt = p.part[i];
        fill_gemm_part(pt, pr, bn, tiles);
        const uint64_t ys = (uint64_t)pr.d_out * 2;
        if (!caches[i]->get_2d(&pt.w, pr.W0, (uint64_t)a.d_in, (uint64_t)pr.d_out, xs, kBK, (uint32_t)bn)) return cudaErrorInvalidValue;
        if (split == 1) {   // (the split-K kernel stores its outputs with plain stores)
            if (!caches[i]->get_2d(&pt.y, pr.y, (uint64_t)pr.d_out, (uint64_t)a.T, ys, kEpiChunkCols, 32)) return cudaErrorInvalidValue;
        } else {
            pt.y = pt.w;
        }
        tiles += (a.shape.tall ? (p.num_m + 1) / 2 : p.num_m) * pt.num_n;
        columns += pt.num_n;
    }
    p.y2 = p.part[0].y;
    if (dual && split == 1 &&
        !caches[0]->get_2d(&p.y2, a.y2, (uint64_t)a.proj[0].d_out, (uint64_t)a.T, (uint64_t)a.proj[0].d_out * 2, kEpiChunkCols, 32)) return cudaErrorInvalidValue;
    p.u2 = a.u2; p.y2_ptr = (__nv_bfloat16*)a.y2;
    p.status = a.proj[0].ar->status;
    p.T = a.T; p.K = a.d_in; p.P = a.P; p.num_tiles = tiles;
    p.lora = a.lora ? 1 : 0; p.fused = a.fused ? 1 : 0; p.rows = a.rows;
    p.pass_flags = a.proj[0].ar->pass_flags; p.fuse_sync = a.proj[0].ar->status + 4;
    p.x_flag = a.x_flag; p.call_id = a.call_id;
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[2];
    // with adapters the predecessor is the bind_shrink launch of this call, else the kernel waits at its top
    // (tall tiles with the shrink inside: the SMs without a tile take its passes)
    const bool tall = a.shape.tall;
    pdl_config(cfg, attr, dim3((unsigned)(tiles < a.num_sms && !(tall && a.fused) ? tiles : a.num_sms)), dim3(tall ? kGemmThreadsTall : kGemmThreads),
               tall ? GemmCfg<256, true>::kSmemBytes : bn == 256 ? GemmCfg<256>::kSmemBytes : (bn == 128 ? GemmCfg<128>::kSmemBytes : GemmCfg<64>::kSmemBytes), stream);
    p.stages = 0;
    if (split > 1) {
        p.stages = a.share_sm && gemm_exchange_bytes(bn, split) <= gemm_stages_short(bn) * gemm_stage_bytes(bn) ? gemm_stages_short(bn) : gemm_stages(bn);
        cfg.dynamicSmemBytes = GemmCfg<64>::split_smem(0) + p.stages * gemm_stage_bytes(bn);
        cfg.gridDim = dim3(split, columns, p.num_m);
        attr[1].id = cudaLaunchAttributeClusterDimension;
        attr[1].val.clusterDim.x = split;
        attr[1].val.clusterDim.y = 1;
        attr[1].val.clusterDim.z = 1;
        cfg.numAttrs = 2;
        if (bn == 256) return cudaLaunchKernelEx(&cfg, lora_gemm_sm100_splitk_kernel<256>, p);
        if (bn == 64) return cudaLaunchKernelEx(&cfg, lora_gemm_sm100_splitk_kernel<64>, p);
        return cudaLaunchKernelEx(&cfg, lora_gemm_sm100_splitk_kernel<128>, p);
    }
    if (tall) return cudaLaunchKernelEx(&cfg, lora_gemm_sm100_kernel<256, true>, p, *a.proj[0].snap);
    if (bn == 256) return cudaLaunchKernelEx(&cfg, lora_gemm_sm100_kernel<256, false>, p, *a.proj[0].snap);
    if (bn == 64) return cudaLaunchKernelEx(&cfg, lora_gemm_sm100_kernel<64, false>, p, *a.proj[0].snap);
    return cudaLaunchKernelEx(&cfg, lora_gemm_sm100_kernel<128, false>, p, *a.proj[0].snap);
}

}  // namespace lml

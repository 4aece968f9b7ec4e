// The GEMM path's kernel for calls of several row tiles: CTA pairs (tcgen05 cta_group::2).
//
// Two CTAs of a cluster multiply a tile of 256 rows x BN columns together: each stages its own 128 rows of x and half of
// the tile's rows of W0, and the pair's first CTA issues MMAs (M = 256) that read both CTAs' shared memory and leave 128
// rows of the product in each CTA's TMEM.  So a CTA brings in 32 KB per 128 x 256 x 64 products where a tile of its own
// takes 48 KB: on many rows the copies into shared memory bound the single tiles (0.415 us per k-block at 117 KB/us into
// an SM, tensor cores 57 % busy), and the accumulator of 256 columns leaves room for a second one, so the epilogue runs
// beside the next tile.  What bounds it: the tensor cores (512 - 540 cycles per k-block of 256 columns) and, at thousands of rows, the
// power they may draw.  us per call, single or two-row-tile CTAs before / pairs: 1000 x 4096 -> 4096 with four adapters 40.0 / 28.7, 1000 x
// 11008 -> 4096 86.4 / 67.0, 8192 x 4096 -> 4096 without 226 / 206, 8192 x 4096 -> 11008 582 / 538 (1373 TFLOP/s at the power limit; a plain
// library product takes 556).
//
// Seven warps in each CTA:
//   warp 0   TMA producer: its CTA's 128 x 64 tiles of x and BN/2 x 64 tiles of W0 into a ring of stages, then the tile's
//            LoRA chunks, up to four to a stage: per chunk the 128 x 16 block of u and its half of the BN x 16 block of B.
//            All copies of both CTAs complete on the first CTA's barrier of the stage.
//   warp 1   in the first CTA: the MMA issuer.  A commit arrives on the barriers of both CTAs.
//   warps 2-5 epilogue: as in the single-tile kernel (lml_gemm_sm100.cu), one tile behind the MMAs.
//   warp 6   lists the chunks of the next tile: those that either row tile of the pair uses, in order of slot and chunk; a CTA
//            whose own row tile does not use a chunk multiplies zeros (a copy from behind the end of the u blocks).
//
// Early start as in lml_gemm_sm100.cu.  Every wait is bounded; on give-up the CTA sets LML_FLAG_TIMEOUT, gives its copies in
// flight time to land and frees its TMEM.
#include "lml_gemm_common.cuh"

namespace lml {

constexpr int kPairThreads = 224;
constexpr int kPairMaxStages = 8;
constexpr int kPairXBytes = kBM * kBK * 2;                 // a k-block of this CTA's rows
constexpr int kPairRingBytes = 6 * (kPairXBytes + 128 * kBK * 2);
constexpr int kPairEpiBytes = 4 * 2 * kEpiBufBytes;
constexpr int kPairAcc = 256;                              // TMEM columns of an accumulator

struct PairCtrl {
    uint64_t full[kPairMaxStages], empty[kPairMaxStages];
    uint64_t tmem_full[2], tmem_empty[2];
    uint64_t list_full[2], list_empty[2];
    uint32_t tmem_base;
    int abort;
    uint32_t stage_info[kPairMaxStages];   // written by the first CTA's producer: K-steps | kPair* flags
    int32_t count[2];                      // entries of the lists
};
constexpr uint32_t kPairCommit = 0x100u;   // after this stage the accumulator holds an output
constexpr uint32_t kPairChunks = 0x200u;   // LoRA chunks (no-swizzle operands), a K-step each

struct PairShared {
    PairCtrl ctrl;
    uint32_t list[2][kMaxChunks];          // slot | chunk << 8 | (number among the row tile's own chunks, or 0xffff) << 16
};
constexpr int kPairSmemBytes = 1024 + kPairRingBytes + kPairEpiBytes + (int)sizeof(PairShared);
static_assert(kPairSmemBytes <= 227 * 1024, "shared memory budget");

struct alignas(64) PairPart {
    GemmPart g;
    CUtensorMap u, bk;          // the u blocks and the packed B as rows of 128 bytes
};
struct alignas(64) PairParams {
    CUtensorMap x;
    PairPart part[LML_MAX_PROJECTIONS];
    uint32_t* status;
    int T, K, P;
    int num_m, num_mp;          // row tiles, pairs of them
    int num_tiles;
    int bn, stages, stage_bytes;
    int panel;                  // see pair_tile
    int x_bytes;                // of one copy of x (a k-block of a row tile)
    int u_rows;                 // behind the last row of the u maps: a copy from there brings zeros
    int lora;
    uint32_t* x_flag;           // early start (else null), as in GemmParams
    uint32_t call_id;
};

__device__ __forceinline__ int pair_part_of(const PairParams& p, int tile)
{
    int i = 0;
    while (i + 1 < p.P && tile >= p.part[i + 1].g.tile0) ++i;
    return i;
}
// Where tile `tile` of the launch lies: panels of p.panel pairs of row tiles, in a panel the rows before the columns.
struct PairTile { int part, mp, n; };
__device__ __forceinline__ PairTile pair_tile(const PairParams& p, int tile)
{
    PairTile t;
    t.part = pair_part_of(p, tile);
    const GemmPart& pt = p.part[t.part].g;
    const int local = tile - pt.tile0, per_panel = p.panel * pt.num_n;
    const int mp0 = local / per_panel * p.panel, in = local % per_panel;
    const int rows = min(p.panel, p.num_mp - mp0);
    t.mp = mp0 + in % rows;
    t.n = in / rows;
    return t;
}
// One 32nd of the chunks that either of two row tiles uses (ids 32w .. 32w + 31, id = slot * 4 + chunk), an id per lane.
// Returns whether the lane's id is among them; own: its number among the chunks of the tile with slots `mask`, or -1.
__device__ __forceinline__ bool union_chunk(const GemmPart& pt, unsigned long long mask, unsigned long long both, int w, int lane,
                                            int& own_before, int& own)
{
    const int slot = w * 8 + (lane >> 2);
    const bool there = ((both >> slot) & 1ull) && (lane & 3) < slot_chunks(pt, slot);
    const bool mine = there && ((mask >> slot) & 1ull);
    const uint32_t b = __ballot_sync(0xffffffffu, mine);
    own = mine ? own_before + __popc(b & ((1u << lane) - 1u)) : -1;
    own_before += __popc(b);
    return there;
}

__global__ void __launch_bounds__(kPairThreads, 1) lora_gemm_pair_kernel(const __grid_constant__ PairParams p)
{
    extern __shared__ uint8_t pair_smem[];
    const uint32_t raw_addr = smem_u32(pair_smem);
    const uint32_t ring = (raw_addr + 1023u) & ~1023u;   // 128-byte swizzled tiles need 1024-byte alignment
    uint8_t* const ring_ptr = pair_smem + (ring - raw_addr);
    uint8_t* const epi_ptr = ring_ptr + kPairRingBytes;
    PairShared* const sh = reinterpret_cast<PairShared*>(epi_ptr + kPairEpiBytes);
    PairCtrl* const ctrl = &sh->ctrl;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int r = (int)cluster_ctarank();                // which half of the rows
    const int pair = (int)blockIdx.x >> 1, npairs = (int)gridDim.x >> 1;
    const int num_kb = (p.K + kBK - 1) / kBK;
    const int half = p.bn >> 1;

    if (threadIdx.x == 0) {
        for (int s = 0; s < p.stages; ++s) {
            mbar_init(smem_u32(&ctrl->full[s]), 1);
            mbar_init(smem_u32(&ctrl->empty[s]), 1);
        }
        for (int a = 0; a < 2; ++a) {
            mbar_init(smem_u32(&ctrl->tmem_full[a]), 1);
            mbar_init(smem_u32(&ctrl->tmem_empty[a]), 8);   // four warps of each CTA
            mbar_init(smem_u32(&ctrl->list_full[a]), 1);
            mbar_init(smem_u32(&ctrl->list_empty[a]), 1);
        }
        ctrl->abort = 0;
        fence_mbar_init();
    }
    if (warp == 0 && lane == 0) {
        prefetch_tmap(&p.x);
        for (int i = 0; i < p.P; ++i) { prefetch_tmap(&p.part[i].g.w); prefetch_tmap(&p.part[i].g.y); }
    }
    if (warp == 1) tmem_alloc_pair(smem_u32(&ctrl->tmem_base), 2 * kPairAcc);
    tc_fence_before();
    __syncthreads();
    cluster_sync_all();          // the barriers of both CTAs are set up
    tc_fence_after();
    const uint32_t tmem_base = ctrl->tmem_base;
    volatile int* abort = &ctrl->abort;
    const uint32_t full0 = mapa_shared(smem_u32(&ctrl->full[0]), 0);   // the first CTA's
    if (p.x_flag) {   // early start: the first k-blocks' W0, then x
        const PairTile first = pair_tile(p, pair);
        const int first_n = first.n;
        const PairPart& pp = p.part[first.part];
        if (warp == 0) {
            if (elect_one()) {
                for (int kb = 0; kb < min(p.stages, num_kb); ++kb) {
                    if (r == 0) mbar_expect_tx(smem_u32(&ctrl->full[kb]), (uint32_t)(p.bn * kBK * 2));
                    tma_load_2d_pair(ring + (uint32_t)(kb * p.stage_bytes + kPairXBytes), &pp.g.w, full0 + 8u * (uint32_t)kb, kb * kBK, first_n * p.bn + r * half);
                }
                wait_x(p.x_flag, p.call_id);
            }
        } else if (warp == 6) {
            for (int i = lane; i < kMaxChunks; i += 32) {   // the live slots' rows of B for this CTA's columns: a hint
                const int s = i / (kRankPad / kChunk), c = i % (kRankPad / kChunk);
                if (((pp.g.live >> s) & 1ull) && c < slot_chunks(pp.g, s) && first_n * p.bn + r * half + half <= pp.g.n_pad)
                    bulk_prefetch_to_l2(pp.g.bk + ((size_t)i * pp.g.n_pad + (size_t)(first_n * p.bn + r * half)) * kChunk, (uint32_t)(half * kChunk * 2));
            }
        }
        __syncthreads();
    }
    if (!p.lora) {   // no launch of this call came before this one: wait for foreign work here
        grid_dependency_wait();
        grid_launch_dependents();
    }
    if (warp == 0) {
        // ------------------------------------------------------------------ TMA producer
        // Both CTAs' producers walk the same stages; the first CTA's accounts for the bytes of both.
        if (elect_one()) {
            int stage = 0;
            uint32_t phase = 0;
            bool ok = true;
            const bool lead = r == 0;
            auto acquire = [&]() -> bool { return mbar_wait(smem_u32(&ctrl->empty[stage]), phase ^ 1u, abort); };
            auto advance = [&]() { if (++stage == p.stages) { stage = 0; phase ^= 1u; } };
            const int ahead = p.x_flag ? min(p.stages, num_kb) : 0;   // early start: k-blocks of the first tile whose W0 has been asked for already
            int ordinal = 0;
            for (int tile = pair; tile < p.num_tiles && ok; tile += npairs, ++ordinal) {
                const PairTile at = pair_tile(p, tile);
                const PairPart& pp = p.part[at.part];
                const int mp = at.mp, n = at.n;
                const int row0 = (2 * mp + r) * kBM, col0 = n * p.bn + r * half;
                const int have_w = ordinal == 0 ? ahead : 0;
                // k-blocks [k0, k1); the ring's place lives in registers here
                auto base_blocks = [&](int k0, int k1, uint32_t info) {
                    int st = stage;
                    uint32_t ph = phase;
                    bool good = ok;
                    for (int kb = k0; kb < k1; ++kb) {
                        good = mbar_wait(smem_u32(&ctrl->empty[st]), ph ^ 1u, abort);
                        if (!good) break;
                        const uint32_t dst = ring + (uint32_t)(st * p.stage_bytes), bar = full0 + 8u * (uint32_t)st;
                        if (lead) {
                            ctrl->stage_info[st] = info;
                            mbar_arrive_expect_tx(smem_u32(&ctrl->full[st]), (uint32_t)(2 * p.x_bytes + (kb < have_w ? 0 : p.bn * kBK * 2)));
                        }
                        tma_load_2d_pair(dst, &p.x, bar, kb * kBK, row0);
                        if (kb >= have_w) tma_load_2d_pair(dst + kPairXBytes, &pp.g.w, bar, kb * kBK, col0);
                        if (++st == p.stages) { st = 0; ph ^= 1u; }
                    }
                    stage = st; phase = ph; ok = good;
                };
                base_blocks(0, num_kb - 1, 4u);
                if (!ok) break;
                int count = 0;
                const int b = ordinal & 1;
                if (p.lora) {
                    ok = mbar_wait(smem_u32(&ctrl->list_full[b]), (uint32_t)(ordinal >> 1) & 1u, abort);
                    if (!ok) break;
                    if (ordinal == 0) grid_dependency_wait();   // (over: warp 6 has waited; what that launch wrote is this thread's to read)
                    count = ctrl->count[b];
                }
                base_blocks(num_kb - 1, num_kb, 4u | (count ? 0u : kPairCommit));
                if (ok && count) {
                    for (int i = 0; i < count && ok; i += 4) {
                        ok = acquire();
                        if (!ok) break;
                        const int k = min(4, count - i);
                        const uint32_t dst = ring + (uint32_t)(stage * p.stage_bytes), bar = full0 + 8u * (uint32_t)stage;
                        if (lead) {
                            ctrl->stage_info[stage] = (uint32_t)k | kPairChunks | (i + 4 >= count ? kPairCommit : 0u);
                            mbar_arrive_expect_tx(smem_u32(&ctrl->full[stage]), (uint32_t)(k * (2 * kUBlockBytes + p.bn * kChunk * 2)));
                        }
                        for (int j = 0; j < k; ++j) {
                            const uint32_t e = sh->list[b][i + j];
                            const int own = (int)(e >> 16), slot = (int)(e & 0xffu), c = (int)((e >> 8) & 0xffu);
                            // (rows of 128 bytes: 32 to a block of u, four rows of a chunk of B to one)
                            tma_load_2d_pair(dst + (uint32_t)(j * kUBlockBytes), &pp.u, bar, 0,
                                             own == 0xffff ? p.u_rows : ((2 * mp + r) * pp.g.cap + own) * (kUBlockBytes / 128));
                            tma_load_2d_pair(dst + (uint32_t)(kPairXBytes + j * half * kChunk * 2), &pp.bk, bar, 0,
                                             ((slot * (kRankPad / kChunk) + c) * pp.g.n_pad + col0) / 4);
                        }
                        advance();
                    }
                }
                if (p.lora) mbar_arrive(smem_u32(&ctrl->list_empty[b]));
            }
            // leave only after every load issued above has landed and been consumed, and every commit has arrived here
            for (int i = 0; i < p.stages && ok; ++i) { ok = acquire(); advance(); }
        }
    } else if (warp == 1) {
        // ------------------------------------------------------------------ MMA issuer, for both CTAs
        if (r == 0 && elect_one()) {
            const uint32_t idesc = umma_idesc_bf16(2 * kBM, p.bn);
            int stage = 0;
            uint32_t phase = 0;
            bool ok = true;
            int ordinal = 0;
            uint32_t eph = 0;   // bit a: phase of tmem_empty[a]
            auto take_acc = [&](int acc) -> bool {
                if (!mbar_wait(smem_u32(&ctrl->tmem_empty[acc]), ((eph >> acc) & 1u) ^ 1u, abort)) return false;
                eph ^= 1u << acc;
                tc_fence_after();
                return true;
            };
            for (int tile = pair; tile < p.num_tiles && ok; tile += npairs, ++ordinal) {
                const int acc = ordinal & 1;
                const uint32_t d_tmem = tmem_base + (uint32_t)(acc * kPairAcc);
                ok = take_acc(acc);
                if (!ok) break;
                uint32_t on = 0;
                {   // the k-blocks but the last: the loop that the tensor cores wait for
                    int st = stage;
                    uint32_t ph = phase;
                    bool good = true;
                    const uint64_t adesc0 = umma_desc_k128(ring), bdesc0 = umma_desc_k128(ring + kPairXBytes);
                    const uint32_t full = smem_u32(&ctrl->full[0]), empty = smem_u32(&ctrl->empty[0]);
                    const uint32_t step = (uint32_t)p.stage_bytes / 16;
                    for (int i = 0; i < num_kb - 1; ++i) {
                        good = mbar_wait(full + 8u * (uint32_t)st, ph, abort);
                        if (!good) break;
                        const uint64_t at = (uint64_t)((uint32_t)st * step);
#pragma unroll
                        for (int k = 0; k < 4; ++k)
                            umma_bf16_pair(d_tmem, adesc0 + at + (uint64_t)(k * 2), bdesc0 + at + (uint64_t)(k * 2), idesc, k == 0 ? on : 1u);
                        on = 1u;
                        umma_commit_pair(empty + 8u * (uint32_t)st);
                        if (++st == p.stages) { st = 0; ph ^= 1u; }
                    }
                    stage = st; phase = ph; ok = good;
                }
                // the last k-block and the tile's LoRA chunks: stages with a word that says what they are
                for (bool more = true; more && ok;) {
                    ok = mbar_wait(smem_u32(&ctrl->full[stage]), phase, abort);
                    if (!ok) break;
                    const uint32_t info = ctrl->stage_info[stage];
                    more = (info & kPairCommit) == 0;
                    const bool chunks = (info & kPairChunks) != 0;
                    const uint32_t at = ring + (uint32_t)(stage * p.stage_bytes);
                    const uint64_t adesc = chunks ? umma_desc_k16(at) : umma_desc_k128(at);
                    const uint64_t bdesc = chunks ? umma_desc_k16(at + kPairXBytes) : umma_desc_k128(at + kPairXBytes);
                    const uint64_t astep = chunks ? kUBlockBytes / 16 : 2, bstep = chunks ? (uint64_t)(half * kChunk * 2 / 16) : 2;
                    const int ksteps = (int)(info & 0xffu);
#pragma unroll 4
                    for (int k = 0; k < ksteps; ++k) {
                        umma_bf16_pair(d_tmem, adesc + (uint64_t)k * astep, bdesc + (uint64_t)k * bstep, idesc, on);
                        on = 1u;
                    }
                    umma_commit_pair(smem_u32(&ctrl->empty[stage]));
                    if (++stage == p.stages) { stage = 0; phase ^= 1u; }
                }
                if (ok) umma_commit_pair(smem_u32(&ctrl->tmem_full[acc]));
            }
        }
    } else if (warp < 6) {
        // ------------------------------------------------------------------ epilogue warps
        const int q = warp & 3;                 // TMEM lane quarter this warp may read
        const int ew = warp - 2;
        const bool one = elect_one();           // the lane that issues the stores
        const uint32_t acc_free0 = mapa_shared(smem_u32(&ctrl->tmem_empty[0]), 0);   // the first CTA's
        int acc = 0;
        uint32_t fph = 0;   // bit a: phase of tmem_full[a]
        int buf = 0;        // staging buffer of the next store: it alternates from store to store, through all tiles (a tile may store
                            // an odd number of chunks)
        bool ok = true;
        if (p.lora) grid_dependency_wait();   // (the plans are read here too)
        for (int tile = pair; tile < p.num_tiles && ok; tile += npairs) {
            const PairTile pl = pair_tile(p, tile);
            const GemmPart& pt = p.part[pl.part].g;
            const int m = 2 * pl.mp + r, n = pl.n;
            const int row_base = m * kBM + q * 32;
            const bool nonfinite = p.lora && m < p.num_m && ld_after_wait(pt.nonfinite) != 0u;
            ok = mbar_wait_warp(smem_u32(&ctrl->tmem_full[acc]), (fph >> acc) & 1u, abort);
            if (!ok) break;
            fph ^= 1u << acc;
            tc_fence_after();
            const uint32_t t_addr = tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)(acc * kPairAcc);
            const int chunks = p.bn / kEpiChunkCols;
            // The CTA's last tile is staged in the ring, which nobody needs any more, and stored in one go.
            const bool last = tile + npairs >= p.num_tiles;
            uint32_t va[32], vb[32];
            auto put = [&](int c, const uint32_t (&v32)[32]) {   // 32 columns: to bf16, into shared memory, out
                const int col0 = n * p.bn + c * kEpiChunkCols;
                if (col0 >= pt.N || row_base >= p.T) return;   // nothing of this chunk is inside y
                const int at = last ? (ew * (kPairAcc / kEpiChunkCols) + c) * kEpiBufBytes : kPairRingBytes + (ew * 2 + buf) * kEpiBufBytes;
                if (!last) {   // the buffer we are about to overwrite must have been read by its earlier store: all but the newest have
                    if (one) tma_store_wait_read<1>();
                    __syncwarp();
                }
                uint8_t* bp = ring_ptr + at;
                // row = lane: 64 bytes, four 16-byte chunks, 64-byte swizzle (chunk ^= (row >> 1) & 3)
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    uint4 v;
                    v.x = pack_bf16(__uint_as_float(v32[8 * j + 0]), __uint_as_float(v32[8 * j + 1]));
                    v.y = pack_bf16(__uint_as_float(v32[8 * j + 2]), __uint_as_float(v32[8 * j + 3]));
                    v.z = pack_bf16(__uint_as_float(v32[8 * j + 4]), __uint_as_float(v32[8 * j + 5]));
                    v.w = pack_bf16(__uint_as_float(v32[8 * j + 6]), __uint_as_float(v32[8 * j + 7]));
                    *reinterpret_cast<uint4*>(bp + lane * 64 + (j ^ ((lane >> 1) & 3)) * 16) = v;
                }
                if (__builtin_expect(nonfinite, 0))
                    add_nonfinite(pt, m, q * 32 + lane, 0, -1, -1, col0, pt.u, nullptr, nullptr, bp + lane * 64, (lane >> 1) & 3);
                if (last) return;
                fence_proxy_async_smem();
                __syncwarp();
                if (one) {
                    tma_store_2d(&pt.y, ring + (uint32_t)at, col0, row_base);
                    tma_store_commit();
                }
                buf ^= 1;
            };
            auto fetched = [&](int c) {   // chunk c is in registers; behind the last one the accumulator goes back to the MMA issuer
                tmem_ld_wait();
                if (c < chunks - 1) return;
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive_cluster(acc_free0 + 8u * (uint32_t)acc);
            };
            tmem_ld_32x32(t_addr, va);
#pragma unroll 1
            for (int c = 0; c < chunks; c += 2) {   // (the next 32 columns are on their way while these are stored)
                fetched(c);
                if (c + 1 < chunks) tmem_ld_32x32(t_addr + (uint32_t)((c + 1) * kEpiChunkCols), vb);
                put(c, va);
                if (c + 1 == chunks) break;
                fetched(c + 1);
                if (c + 2 < chunks) tmem_ld_32x32(t_addr + (uint32_t)((c + 2) * kEpiChunkCols), va);
                put(c + 1, vb);
            }
            if (last && row_base < p.T) {
                fence_proxy_async_smem();
                if (elect_one()) {
                    for (int c = 0; c < chunks && n * p.bn + c * kEpiChunkCols < pt.N; ++c)
                        tma_store_2d(&pt.y, ring + (uint32_t)((ew * (kPairAcc / kEpiChunkCols) + c) * kEpiBufBytes), n * p.bn + c * kEpiChunkCols, row_base);
                    tma_store_commit();
                }
            }
            acc ^= 1;
        }
        tma_store_wait_all();   // (whichever lane has issued any)
    } else if (p.lora) {
        // ------------------------------------------------------------------ the chunks of each tile
        grid_dependency_wait();
        grid_launch_dependents();
        int ordinal = 0;
        for (int tile = pair; tile < p.num_tiles; tile += npairs, ++ordinal) {
            const PairTile at = pair_tile(p, tile);
            const GemmPart& pt = p.part[at.part].g;
            const int mp = at.mp, b = ordinal & 1;
            unsigned long long mask[2];
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                const int m = 2 * mp + i;
                mask[i] = m >= p.num_m ? 0ull : ld_after_wait(&pt.plan[m].used);
            }
            if (!mbar_wait_warp(smem_u32(&ctrl->list_empty[b]), (((uint32_t)ordinal >> 1) & 1u) ^ 1u, abort)) break;
            const unsigned long long both = mask[0] | mask[1], mine = r ? mask[1] : mask[0];
            int n = 0, own_before = 0;
            for (int w = 0; w < kMaxChunks / 32; ++w) {
                if (!((both >> (w * 8)) & 0xffull)) continue;
                int own;
                const bool there = union_chunk(pt, mine, both, w, lane, own_before, own);
                const uint32_t bits = __ballot_sync(0xffffffffu, there);
                if (there)
                    sh->list[b][n + __popc(bits & ((1u << lane) - 1u))] =
                        (uint32_t)(w * 8 + (lane >> 2)) | ((uint32_t)(lane & 3) << 8) | ((uint32_t)(own & 0xffff) << 16);
                n += __popc(bits);
            }
            __syncwarp();
            if (lane == 0) { ctrl->count[b] = n; mbar_arrive(smem_u32(&ctrl->list_full[b])); }
        }
    }

    __syncthreads();
    if (ctrl->abort) __nanosleep(50000);   // gave up: let copies still in flight land before the CTA goes away
    if (threadIdx.x == 0 && ctrl->abort) atomicOr(p.status, LML_FLAG_TIMEOUT);
    if (threadIdx.x == 0) leave_early_start(p.x_flag);
    __syncwarp();
    cluster_sync_all();          // nobody leaves while the other's MMAs, arrivals and reads of this CTA are on their way
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc_pair(tmem_base, 2 * kPairAcc);
    }
}

int gemm_pair_stages(int bn)
{
    const int stages = kPairRingBytes / (kPairXBytes + bn / 2 * kBK * 2);
    return stages < kPairMaxStages ? stages : kPairMaxStages;
}

// pairs: the pairs of CTAs that are resident at once; 0, and no call takes pairs, where the runtime does not say.
cudaError_t gemm_pair_init(int num_sms, int* pairs)
{
    const cudaError_t e = cudaFuncSetAttribute(lora_gemm_pair_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kPairSmemBytes);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(num_sms / 2 * 2));
    cfg.blockDim = dim3(kPairThreads);
    cfg.dynamicSmemBytes = kPairSmemBytes;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 2; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr; cfg.numAttrs = 1;
    if (cudaOccupancyMaxActiveClusters(pairs, lora_gemm_pair_kernel, &cfg) != cudaSuccess) { *pairs = 0; (void)cudaGetLastError(); }
    return cudaSuccess;
}

cudaError_t launch_gemm_pair(TmapCache* const* caches, const GemmArgs& a, cudaStream_t stream)
{
    if (a.u2 || a.fused || a.num_pairs < 1) return cudaErrorInvalidValue;
    PairParams p;
    const int bn = a.shape.bn;
    p.num_m = (a.T + kBM - 1) / kBM;
    p.num_mp = (p.num_m + 1) / 2;
    const uint64_t xs = (uint64_t)a.d_in * 2;
    if (!caches[0]->get_2d(&p.x, a.x, (uint64_t)a.d_in, (uint64_t)a.T, xs, kBK, (uint32_t)x_box_rows(a.T))) return cudaErrorInvalidValue;
    p.x_bytes = x_box_rows(a.T) * kBK * 2;
    p.u_rows = 0;
    int tiles = 0;
    for (int i = 0; i < a.P; ++i) {
        const GemmProj& pr = a.proj[i];
        if (pr.u_lo) return cudaErrorInvalidValue;   // (gemm_pick_shape chooses no pairs for such a call)
        PairPart& pp = p.part[i];
        GemmPart& pt = pp.g;
        fill_gemm_part(pt, pr, bn, tiles);
        if (!caches[i]->get_2d(&pt.w, pr.W0, (uint64_t)a.d_in, (uint64_t)pr.d_out, xs, kBK, (uint32_t)(bn / 2)) ||
            !caches[i]->get_2d(&pt.y, pr.y, (uint64_t)pr.d_out, (uint64_t)a.T, (uint64_t)pr.d_out * 2, kEpiChunkCols, 32)) return cudaErrorInvalidValue;
        if (a.lora) {
            const uint64_t u_rows = (uint64_t)p.num_m * pr.cap * (kUBlockBytes / 128);
            p.u_rows = (int)u_rows > p.u_rows ? (int)u_rows : p.u_rows;
            if (!caches[i]->get_2d(&pp.u, pr.u, 64, u_rows, 128, 64, kUBlockBytes / 128, false) ||
                !caches[i]->get_2d(&pp.bk, pr.ar->Bk, 64, (uint64_t)pr.snap->max_slots * (kRankPad / kChunk) * pt.n_pad / 4, 128, 64, (uint32_t)(bn / 8), false))
                return cudaErrorInvalidValue;
        } else {
            pp.u = pp.bk = pt.w;
        }
        tiles += p.num_mp * pt.num_n;
    }
    p.status = a.proj[0].ar->status;
    p.T = a.T; p.K = a.d_in; p.P = a.P; p.num_tiles = tiles;
    p.bn = bn;
    // Panels whose rows of x (48 MB at most, evenly dealt) stay in L2 while the columns go by; every panel reads W0 once.  With the
    // chip at its power limit what is not fetched again is time: 8192 x 4096 -> 11008 600 us with all rows in one panel, 538 with 16
    // pairs of row tiles to a panel, 555 with 8, 581 with 4; 8192 x 11008 -> 4096 610 in one, 574 with 16 ... 4.
    const int panels = (int)((uint64_t)p.num_mp * 2 * kBM * xs / (48u << 20)) + 1;
    p.panel = (p.num_mp + panels - 1) / panels;
    p.stage_bytes = kPairXBytes + bn / 2 * kBK * 2;
    p.stages = gemm_pair_stages(bn);
    p.lora = a.lora ? 1 : 0;
    p.x_flag = a.x_flag; p.call_id = a.call_id;
    const int pairs = tiles < a.num_pairs ? tiles : a.num_pairs;
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[2];
    pdl_config(cfg, attr, dim3((unsigned)(2 * pairs)), dim3(kPairThreads), kPairSmemBytes, stream);
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = 2;
    attr[1].val.clusterDim.y = 1;
    attr[1].val.clusterDim.z = 1;
    cfg.numAttrs = 2;
    return cudaLaunchKernelEx(&cfg, lora_gemm_pair_kernel, p);
}

}  // namespace lml

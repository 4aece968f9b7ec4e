// Binding and shrink of the GEMM path: which slots the rows of a 128-row tile use, and u = scale * x.A^T for them, in
// one launch that leaves the rows where they are.
//
// The rows of a tile are not grouped by slot.  A tile's slots name the chunks of 16 columns of A that
// any of its rows needs; a chunk's block of u is the dense product of all 128 rows with those 16 columns, kept in the rows
// that are bound to the slot and zero in the others.  The GEMM adds block x (16 columns of the slot's B) per chunk, one
// K-step of the tensor cores, so a slot costs the chunks its rank needs whether its rows are together or scattered.
// Against grouping the rows first (a sort, a copy of x, a product per run of rows) the dense product does more
// arithmetic, on tensor cores that are idle here anyway, and no pass over x but one.
//
// A cluster shares the K of (row tile, group of chunks).  Every CTA streams its part of x and of the chunks' rows of A
// through a TMA ring into tcgen05 products of 128 x (16 per chunk); the partial sums meet through distributed shared
// memory, a share of the rows in each CTA, and are added in a fixed order.  What bounds it is latency for few rows (the ids,
// then A, then the exchange) and the read of x for many.
#include "lml_internal.cuh"
#include "lml_ptx_sm100.cuh"

namespace lml {

using namespace ptx;

constexpr int kBindThreads = 192;          // producer, MMA issuer, four warps for the rows
constexpr int kBindMaxStages = 8;
constexpr int kBindXBytes = kTileM * 64 * 2;   // a k-block (64 columns) of the tile's rows
constexpr int kBindABytes = kChunk * 64 * 2;   // ... and of a chunk's rows of A

struct BindCtrl {
    uint64_t full[kBindMaxStages], empty[kBindMaxStages];
    uint64_t tmem_full;
    uint32_t tmem_base;
    int abort;
    int scan[2];
    uint32_t mask[2][2][kTileM / 32];       // [binding][low, high half][32 rows]
    int8_t row[2][kTileM];                  // slot per row of the tile, first and second binding
    uint16_t list[kMaxChunks];              // chunks of the tile: slot | chunk << 8
    int32_t seg[kBindSegs + 1];
    int8_t seg_slot[2][kBindSegs];
};

struct alignas(64) BindLaunch {
    CUtensorMap x;
    CUtensorMap a[LML_MAX_PROJECTIONS];
    BindArgs args;
    int num_m;
    int group;      // chunks of a pass at most
    int ring_bytes; // divided into as many stages as the pass's chunks allow
    int tmem_cols;
    int x_bytes;    // of one copy of x
    int early;      // few rows: x is asked for before the ids are known, and A's rows into L2 before the wait for the preceding work
};

// Two fp32 values, each as three bf16 values of 8 bits that add up to it.  (The first is the largest bf16 value where rounding
// would make Inf of a finite one; of an Inf or a NaN it is all there is.)
__device__ __forceinline__ void split_bf16(float a, float b, uint32_t& hi, uint32_t& mid, uint32_t& lo)
{
    hi = pack_bf16(a, b);
    if (isfinite(a) && (hi & 0x7fffu) == 0x7f80u) hi -= 1u;
    if (isfinite(b) && (hi & 0x7fff0000u) == 0x7f800000u) hi -= 0x10000u;
    a = isfinite(a) ? a - bf16_lo(hi) : 0.f;
    b = isfinite(b) ? b - bf16_hi(hi) : 0.f;
    mid = pack_bf16(a, b);
    lo = pack_bf16(a - bf16_lo(mid), b - bf16_hi(mid));
}

__global__ void __launch_bounds__(kBindThreads) bind_shrink_kernel(const __grid_constant__ BindLaunch B)
{
    const BindArgs& L = B.args;
    extern __shared__ uint8_t bind_smem[];
    const uint32_t raw = smem_u32(bind_smem);
    const uint32_t ring = (raw + 1023u) & ~1023u;   // 128-byte swizzled tiles need 1024-byte alignment
    uint8_t* ring_ptr = bind_smem + (ring - raw);
    BindCtrl* ctrl = reinterpret_cast<BindCtrl*>(ring_ptr + B.ring_bytes);

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int S = (int)gridDim.x, r = (int)blockIdx.x;   // the cluster spans the grid's x dimension
    const int m = (int)blockIdx.z % B.num_m, pi = (int)blockIdx.z / B.num_m;
    const BindPart& part = L.part[pi];
    const SlotSnapshot& snap = L.snap[pi];
    const bool dual = L.second == 1 || L.second == 2;
    const bool first_cta = r == 0 && blockIdx.y == 0;
    const int num_kb = (L.d_in + 63) / 64;
    const int kb0 = r * num_kb / S, kb1 = (r + 1) * num_kb / S, nkb = kb1 - kb0;

    if (tid == 0) {
        for (int i = 0; i < kBindMaxStages; ++i) { mbar_init(smem_u32(&ctrl->full[i]), 1); mbar_init(smem_u32(&ctrl->empty[i]), 1); }
        mbar_init(smem_u32(&ctrl->tmem_full), 1);
        ctrl->abort = 0;
        fence_mbar_init();
        prefetch_tmap(&B.x);
        prefetch_tmap(&B.a[pi]);
    }
    // TMEM is taken before the GEMM may get resident: it waits for this grid before its chunks, and this grid must not wait
    // for columns that the GEMM holds.
    if (warp == 1) {
        tmem_alloc(smem_u32(&ctrl->tmem_base), (uint32_t)B.tmem_cols);
        if (B.early) grid_launch_dependents();   // the GEMM starts on W0; x is not its to read yet
    }
    if (B.early) {
        // The adapters are not written by the work that this launch overlaps with; a share of this part of K of the live
        // slots' rows starts on its way into L2 now (a hint: nothing is read before the wait).
        const int k0 = kb0 * 64, k1 = min(L.d_in, kb1 * 64), lines = max(0, (k1 - k0 + 63) / 64);
        for (int s = 0; s < snap.max_slots; ++s) {
            const int n = (int)snap.rank[s] * lines;
            for (int i = (int)blockIdx.y * kBindThreads + tid; i < n; i += (int)gridDim.y * kBindThreads) {
                const __nv_bfloat16* a = part.A + ((size_t)s * kRankPad + i / lines) * L.d_in + k0 + (i % lines) * 64;
                asm volatile("prefetch.global.L2 [%0];" ::"l"(a));
            }
        }
    }
    grid_dependency_wait();      // launched as a programmatic dependent: whatever ran before is complete now
    if (B.early) {
        if (first_cta && blockIdx.z == 0 && tid == 0) st_release_gpu_u32(L.x_flag, L.call_id);
    } else if (warp == 1) {
        grid_launch_dependents();
    }

    // ---- the slot of every row
    const int row_t = tid - 64;   // warps 2 .. 5: a row each
    const uint32_t any_nonfinite = first_cta && row_t >= 0 ? ld_after_wait(part.nonfinite) : 0u;   // (used at the end)
    int bad_slot = 0;
    int s_a = -1, s_b = -1;
    if (L.rows.mode == kRowsSegments) {
        int bad_off = 0;
        for (int g = tid; g <= L.rows.G; g += kBindThreads) ctrl->seg[g] = ld_after_wait(L.rows.seg_offsets + g);
        for (int g = tid; g < L.rows.G; g += kBindThreads) {
            const int s = ld_after_wait(part.ids + g);
            ctrl->seg_slot[0][g] = (int8_t)(slot_rank(snap, s) > 0 ? s : (s == -1 ? -1 : -2));
            if (dual) {
                const int s2 = ld_after_wait(L.rows.ids2 + g);
                ctrl->seg_slot[1][g] = (int8_t)(slot_rank(snap, s2) > 0 ? s2 : (s2 == -1 ? -1 : -2));
            }
        }
        __syncthreads();
        for (int g = tid; g < L.rows.G; g += kBindThreads) {
            const int s0 = ctrl->seg[g], s1 = ctrl->seg[g + 1];
            if (s1 < s0 || s0 < 0 || s1 > L.T) bad_off = 1;
            if (s1 > s0 && (ctrl->seg_slot[0][g] == -2 || (dual && ctrl->seg_slot[1][g] == -2))) bad_slot = 1;   // an empty segment may name anything
        }
        if (tid == 0 && (ctrl->seg[0] != 0 || ctrl->seg[L.rows.G] != L.T)) bad_off = 1;
        bad_off = __syncthreads_or(bad_off);
        if (row_t >= 0 && !bad_off) {
            const int row = m * kTileM + row_t;
            int lo = 0, hi = L.rows.G;
            while (lo < hi) { const int mid = (lo + hi) >> 1; if (ctrl->seg[mid + 1] > row) hi = mid; else lo = mid + 1; }
            if (row < L.T && lo < L.rows.G) { s_a = ctrl->seg_slot[0][lo]; if (dual) s_b = ctrl->seg_slot[1][lo]; }
        }
        if (first_cta && m == 0) {
            const int any = __syncthreads_or(bad_slot);
            const unsigned f = (bad_off ? LML_FLAG_BAD_OFFSETS : 0u) | (any ? LML_FLAG_BAD_SLOT : 0u);
            if (tid == 0 && f) atomicOr(part.status, f);
        }
    } else if (row_t >= 0) {
        const int row = m * kTileM + row_t;
        if (row < L.T) {
            if (L.rows.mode == kRowsTokens) {
                s_a = ld_after_wait(part.ids + row);
                if (part.adapter_map) s_a = resolve_adapter(snap, part.adapter_map, s_a);
                if (s_a != -1 && slot_rank(snap, s_a) == 0) { bad_slot = 1; s_a = -1; }
            } else {
                s_a = L.rows.rows[row];
                if (slot_rank(snap, s_a) == 0) s_a = -1;
                if (dual) { s_b = L.rows.rows2[row]; if (slot_rank(snap, s_b) == 0) s_b = -1; }
            }
        }
        if (bad_slot && first_cta) atomicOr(part.status, LML_FLAG_BAD_SLOT);
    }
    // ---- the tile's slots, and their chunks by slot
    if (row_t >= 0) {
        if (s_a < 0) s_a = -1;
        if (s_b < 0) s_b = -1;
        ctrl->row[0][row_t] = (int8_t)s_a;
        ctrl->row[1][row_t] = (int8_t)s_b;
        const uint32_t la = __reduce_or_sync(0xffffffffu, s_a >= 0 && s_a < 32 ? 1u << s_a : 0u);
        const uint32_t ha = __reduce_or_sync(0xffffffffu, s_a >= 32 ? 1u << (s_a - 32) : 0u);
        const uint32_t lb = __reduce_or_sync(0xffffffffu, s_b >= 0 && s_b < 32 ? 1u << s_b : 0u);
        const uint32_t hb = __reduce_or_sync(0xffffffffu, s_b >= 32 ? 1u << (s_b - 32) : 0u);
        if (lane == 0) {
            ctrl->mask[0][0][warp - 2] = la; ctrl->mask[0][1][warp - 2] = ha;
            ctrl->mask[1][0][warp - 2] = lb; ctrl->mask[1][1][warp - 2] = hb;
        }
    }
    // x does not depend on the ids: the first stages' tiles go out here when most groups of chunks are sure to be needed
    const int wide_stage = kBindXBytes + B.group * kBindABytes;
    const int pre = B.early ? min(min(B.ring_bytes / wide_stage, kBindMaxStages), nkb) : 0;
    if (warp == 0 && elect_one())
        for (int i = 0; i < pre; ++i) {
            const uint32_t bar = smem_u32(&ctrl->full[i]);
            mbar_expect_tx(bar, (uint32_t)B.x_bytes);
            tma_load_2d(ring + (uint32_t)(i * wide_stage), &B.x, bar, (kb0 + i) * 64, m * kTileM);
        }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    unsigned long long mask[2];
#pragma unroll
    for (int b = 0; b < 2; ++b) {
        uint32_t lo = 0, hi = 0;
#pragma unroll
        for (int w = 0; w < kTileM / 32; ++w) { lo |= ctrl->mask[b][0][w]; hi |= ctrl->mask[b][1][w]; }
        mask[b] = (unsigned long long)lo | ((unsigned long long)hi << 32);
    }
    const unsigned long long used = mask[0] | mask[1];
    int before = 0, mine = 0;   // (threads 0 .. 63: one slot each)
    if (tid < kMaxSlots) {
        if ((used >> tid) & 1ull) mine = chunks_of_rank((int)snap.rank[tid]);
        before = mine;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) { const int v = __shfl_up_sync(0xffffffffu, before, o); if (lane >= o) before += v; }
        if (lane == 31) ctrl->scan[warp] = before;
        before -= mine;
    }
    __syncthreads();
    const int count = min(ctrl->scan[0] + ctrl->scan[1], part.cap);   // (never above cap: the call's snapshot bounds it)
    if (tid < kMaxSlots) {
        if (warp == 1) before += ctrl->scan[0];
        const uint32_t who = ((mask[0] >> tid) & 1ull ? kChunkFirst : 0u) | ((mask[1] >> tid) & 1ull ? kChunkSecond : 0u);
        for (int c = 0; c < mine; ++c) {
            ctrl->list[before + c] = (uint16_t)(tid | (c << 8));
            if (first_cta) part.plan[m].chunk[before + c] = (uint16_t)((uint32_t)(tid | (c << 8)) | who);
        }
    }
    if (first_cta && tid == 0) { part.plan[m].count = count; part.plan[m].used = used; }
    __syncthreads();

    // ---- x.A^T of this CTA's part of K, a group of chunks at a time
    const uint32_t tmem_base = ctrl->tmem_base;
    volatile int* abort = &ctrl->abort;
    uint32_t tmem_ph = 0;
    bool first = true;
    for (int c0 = (int)blockIdx.y * B.group; c0 < count; c0 += (int)gridDim.y * B.group) {   // (the same trips in every CTA of the cluster)
        const int nc = min(B.group, count - c0);
        // (a pass whose x went out early keeps that layout)
        const int stage_bytes = first && pre > 0 ? wide_stage : kBindXBytes + nc * kBindABytes;
        const int stages = min(B.ring_bytes / stage_bytes, kBindMaxStages);
        int stage = 0;                // producer's and issuer's place in the ring
        uint32_t phase = 0;
        if (warp != 1) {
            // Warp 0 brings in x and accounts for the stage's bytes; the four row warps, which have nothing to do yet, share the chunks (an
            // issue costs its thread some 60 cycles: 17 copies of a k-block from one thread took 0.55 us, longer than their flight).
            // A warp without a chunk stays out: no stage waits for it, so nothing would keep it within a lap of the ring, and a parity read
            // a lap late says "not yet" for good.
            if ((warp == 0 || warp - 2 < nc) && elect_one()) {
                bool ok = true;
                for (int i = 0; i < nkb && ok; ++i) {
                    ok = mbar_wait(smem_u32(&ctrl->empty[stage]), phase ^ 1u, abort);
                    if (!ok) break;
                    const uint32_t bar = smem_u32(&ctrl->full[stage]), dst = ring + (uint32_t)(stage * stage_bytes);
                    if (warp == 0) {
                        const bool have_x = first && i < pre;
                        mbar_arrive_expect_tx(bar, (uint32_t)(nc * kBindABytes + (have_x ? 0 : B.x_bytes)));
                        if (!have_x) tma_load_2d(dst, &B.x, bar, (kb0 + i) * 64, m * kTileM);
                    } else {
                        for (int c = warp - 2; c < nc; c += 4) {
                            const int e = ctrl->list[c0 + c];
                            tma_load_3d(dst + (uint32_t)(kBindXBytes + c * kBindABytes), &B.a[pi], bar, (kb0 + i) * 64, (e >> 8) * kChunk, e & 0xff);
                        }
                    }
                    if (++stage == stages) { stage = 0; phase ^= 1u; }
                }
            }
        } else if (warp == 1) {
            if (elect_one()) {
                const uint32_t idesc = umma_idesc_bf16(kTileM, nc * kChunk);
                bool ok = true;
                for (int i = 0; i < nkb && ok; ++i) {
                    ok = mbar_wait(smem_u32(&ctrl->full[stage]), phase, abort);
                    if (!ok) break;
                    tc_fence_after();
                    const uint32_t at = ring + (uint32_t)(stage * stage_bytes);
                    const uint64_t adesc = umma_desc_k128(at), bdesc = umma_desc_k128(at + kBindXBytes);
#pragma unroll
                    for (int k = 0; k < 4; ++k)
                        umma_bf16(tmem_base, adesc + (uint64_t)(k * 2), bdesc + (uint64_t)(k * 2), idesc, (i > 0 || k > 0) ? 1u : 0u);
                    umma_commit(smem_u32(&ctrl->empty[stage]));
                    if (++stage == stages) { stage = 0; phase ^= 1u; }
                }
                if (ok) umma_commit(smem_u32(&ctrl->tmem_full));
            }
        }
        first = false;
        __syncwarp();
        bool ok = true;
        if (warp >= 2) {
            ok = mbar_wait_warp(smem_u32(&ctrl->tmem_full), tmem_ph, abort);   // this CTA's products are complete: so are its loads
            if (!ok) __nanosleep(50000);   // gave up: let copies still in flight land before the ring takes the partial sums
            tc_fence_after();
        }
        tmem_ph ^= 1u;
        cluster_sync_all();   // every CTA of the cluster is done with its ring, which now takes the partial sums
        const int rows = kTileM / S;                    // rows that a CTA adds up
        const int row = (warp & 3) * 32 + lane;         // the TMEM lane this thread may read
        if (warp >= 2 && ok) {
            // [contribution][16-byte piece][row]: a warp's store is contiguous
            const uint32_t to = mapa_shared(ring + (uint32_t)((r * nc * 4 * rows + row % rows) * 16), (uint32_t)(row / rows));
            for (int c = 0; c < nc; c += 2) {
                uint32_t v[32];
                tmem_ld_32x32(tmem_base + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)(c * kChunk), v);
                tmem_ld_wait();
                if (nkb == 0) {
#pragma unroll
                    for (int i = 0; i < 32; ++i) v[i] = 0u;
                }
#pragma unroll
                for (int j = 0; j < 8; ++j)
                    if (c * 4 + j < nc * 4)
                        st_shared_cluster_v4(to + (uint32_t)((c * 4 + j) * rows * 16), v[4 * j], v[4 * j + 1], v[4 * j + 2], v[4 * j + 3]);
            }
            tc_fence_before();
        }
        cluster_sync_all();
        for (int e = tid; e < nc * 4 * rows; e += kBindThreads) {   // four columns of one row
            const int rr = e % rows, piece = e / rows;
            const uint8_t* src = ring_ptr + (size_t)(piece * rows + rr) * 16;
            float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
            for (int q = 0; q < S; ++q) {   // rank order: the sum does not depend on timing
                const float4 w = *reinterpret_cast<const float4*>(src + (size_t)q * (nc * 4 * rows * 16));
                v.x += w.x; v.y += w.y; v.z += w.z; v.w += w.w;
            }
            const int slot = ctrl->list[c0 + (piece >> 2)] & 0xff;
            const float sc = snap.scale[slot];
            const int tr = r * rows + rr;
            const int have = (int)snap.rank[slot] - (ctrl->list[c0 + (piece >> 2)] >> 8) * kChunk - (piece & 3) * 4;   // columns that the adapter has, of these and on
            v = make_float4(have > 0 ? v.x * sc : 0.f, have > 1 ? v.y * sc : 0.f, have > 2 ? v.z * sc : 0.f, have > 3 ? v.w * sc : 0.f);   // (Inf in x times the padding of A: not into u)
            const bool a = ctrl->row[0][tr] == slot, b = dual && ctrl->row[1][tr] == slot;
            const uint2 zero = make_uint2(0u, 0u);
            const size_t at = ((size_t)m * part.cap + c0 + (piece >> 2)) * (kTileM * kChunk) + chunk_elem(tr, (piece & 3) * 4);
            if (part.u3) {
                uint2 hi, mid, lo;
                split_bf16(v.x, v.y, hi.x, mid.x, lo.x);
                split_bf16(v.z, v.w, hi.y, mid.y, lo.y);
                *reinterpret_cast<uint2*>(part.u + at) = a ? hi : zero;
                *reinterpret_cast<uint2*>(part.u2 + at) = a ? mid : zero;
                *reinterpret_cast<uint2*>(part.u3 + at) = a ? lo : zero;
                continue;
            }
            const uint2 val = make_uint2(pack_bf16(v.x, v.y), pack_bf16(v.z, v.w));
            *reinterpret_cast<uint2*>(part.u + at) = a ? val : zero;
            if (dual) {
                // (the blocks of the second binding, or of the difference of the two)
                const uint2 neg = make_uint2(val.x ^ 0x80008000u, val.y ^ 0x80008000u);
                *reinterpret_cast<uint2*>(part.u2 + at) = L.second == 1 ? (b ? val : zero) : (a == b ? zero : (b ? val : neg));
            }
        }
        if (c0 + (int)gridDim.y * B.group < count) {   // the ring is loaded again, perhaps in stages of another size: its barriers start over
            fence_proxy_async_smem();
            __syncthreads();
            if (tid == 0) {
                for (int i = 0; i < kBindMaxStages; ++i) {
                    mbar_inval(smem_u32(&ctrl->full[i])); mbar_inval(smem_u32(&ctrl->empty[i]));
                    mbar_init(smem_u32(&ctrl->full[i]), 1); mbar_init(smem_u32(&ctrl->empty[i]), 1);
                }
                fence_mbar_init();
            }
            cluster_sync_all();
        }
    }
    if (first && tid == 0)   // no chunks for this CTA: the tiles of x that went out early have to land before it leaves
        for (int i = 0; i < pre; ++i) { mbar_arrive(smem_u32(&ctrl->full[i])); mbar_wait(smem_u32(&ctrl->full[i]), 0u, abort); }
    if (any_nonfinite) {
        auto marked = [&](int slot) { return slot >= 0 && ld_after_wait(part.nonfinite + 1 + slot) == nonfinite_tag(snap.gen[slot]) ? slot : -1; };
        part.plan[m].nonfinite_row[0][row_t] = (int8_t)marked(s_a);
        part.plan[m].nonfinite_row[1][row_t] = (int8_t)marked(s_b);
    }
    __syncthreads();
    if (tid == 0 && ctrl->abort) atomicOr(part.status, LML_FLAG_TIMEOUT);
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem_base, (uint32_t)B.tmem_cols);
    }
}

// (the partial sums, 8 KB per chunk of a pass, fit each)
constexpr int kBindRingShared = 72 * 1024, kBindRingTwo = 96 * 1024, kBindRingLarge = 192 * 1024;
static int bind_smem_bytes(int ring) { return 1024 + ring + (int)sizeof(BindCtrl); }

// CTAs that share K.  It follows from the rows alone: a projection's u has the same bits in a call of its own and beside others.
static int bind_cluster(int T, int d_in, int num_sms)
{
    const int num_m = (T + kTileM - 1) / kTileM, num_kb = (d_in + 63) / 64;
    int S = num_m * 24 <= num_sms ? 8 : (num_m * 8 <= num_sms ? 4 : (num_m * 2 <= num_sms ? 2 : 1));
    while (S > 1 && num_kb < S) S >>= 1;
    return S;
}
// A chunk per slot, 16 chunks at most, whatever the table holds.
int bind_ctas_reckoned(int T, int d_in, int P, int slots, int num_sms)
{
    const int clusters = (T + kTileM - 1) / kTileM * P * bind_cluster(T, d_in, num_sms);
    return clusters * (slots > 8 && bind_starts_gemm_early(T, P, num_sms) ? 2 : 1);
}
bool bind_starts_gemm_early(int T, int P, int num_sms) { return (T + kTileM - 1) / kTileM * P * 8 <= num_sms; }
// Few rows: a pass takes eight chunks (or all there are), or sixteen where only that leaves the GEMM's CTAs (gemm_ctas) SMs of their own.
// Layer passes, us, with 4 / 8 / 16: 40 tokens, 16 chunks 169 / 162 / 149, 128 tokens, 18 chunks 145 / 126 / 133.  Where the two do not
// find SMs of their own, bind_shrink shares SMs with the split-K GEMM, each with a short ring; no other GEMM fits beside it, so two
// of its own CTAs share an SM, with three stages of eight chunks, and leave the other SMs to the GEMM.  us per call, 16 adapters of rank 8
// ... 64, with two stages of eight (three to an SM) / three (two) / six (one): 160 x 11008 -> 4096 63.5 / 59.3 / 57.5, 500 x 4096 -> 4096 37.4 / 36.0 /
// 36.0, but with four adapters of rank 16 500 x 4096 -> 4096 20.9 / 20.9 / 26.9, 1000 x 2048 -> 2048 15.8 / 15.8 / 20.2.
BindEarly bind_early(int T, int d_in, int P, int cap, int gemm_ctas, bool split, int num_sms)
{
    const int clusters = (T + kTileM - 1) / kTileM * P * bind_cluster(T, d_in, num_sms);
    for (int most = 8; most <= 16; most += 8) {
        const int group = cap < most ? cap : most;
        if (gemm_ctas + clusters * ((cap + group - 1) / group) <= num_sms) return {group, kBindRingLarge, false};
    }
    return {cap < 8 ? cap : 8, split ? kBindRingShared : kBindRingTwo, split};
}

cudaError_t launch_bind_shrink(const BindArgs& a, const CUtensorMap* const* tmap_A, TmapCache* cache, int num_sms, cudaStream_t stream)
{
    BindLaunch b;
    b.args = a;
    if (!cache->get_2d(&b.x, a.x, (uint64_t)a.d_in, (uint64_t)a.T, (uint64_t)a.d_in * 2, 64, (uint32_t)x_box_rows(a.T))) return cudaErrorInvalidValue;
    b.x_bytes = x_box_rows(a.T) * 128;
    int cap = 1;
    for (int p = 0; p < a.P; ++p) {
        cap = a.part[p].cap > cap ? a.part[p].cap : cap;
        b.a[p] = *tmap_A[p];
    }
    const int num_m = b.num_m = (a.T + kTileM - 1) / kTileM;
    const int tiles = num_m * a.P, S = bind_cluster(a.T, a.d_in, num_sms);
    // Few rows: see bind_early.  Many rows: x is read once for up to 16 chunks, one wave of CTAs.
    int groups;
    b.early = a.x_flag ? 1 : 0;
    if (b.early) {
        b.group = a.early.group;
        b.ring_bytes = a.early.ring_bytes;
        groups = (cap + b.group - 1) / b.group;
    } else {
        b.group = 16; b.ring_bytes = kBindRingLarge;
        groups = (cap + b.group - 1) / b.group;
        const int most = num_sms / (tiles * S);   // (one wave: what is over goes in turn)
        groups = groups < most ? groups : (most < 1 ? 1 : most);
    }
    for (b.tmem_cols = 32; b.tmem_cols < b.group * kChunk;) b.tmem_cols *= 2;
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[2];
    pdl_config(cfg, attr, dim3((unsigned)S, (unsigned)groups, (unsigned)tiles), dim3(kBindThreads), (size_t)bind_smem_bytes(b.ring_bytes), stream);
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = (unsigned)S;
    attr[1].val.clusterDim.y = 1;
    attr[1].val.clusterDim.z = 1;
    cfg.numAttrs = 2;
    return cudaLaunchKernelEx(&cfg, bind_shrink_kernel, b);
}

cudaError_t bind_init()
{
    return cudaFuncSetAttribute(bind_shrink_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bind_smem_bytes(kBindRingLarge));
}

// ---------------------------------------------------------------------------------------------
// Slot per row of a segment call whose rows are permuted, or that has more segments than the kernels look up in shared
// memory: one CTA checks the arrays (and raises the flags) and writes the slots.  Latency only; a call in segment order
// does not need it.
// ---------------------------------------------------------------------------------------------
__global__ void __launch_bounds__(1024) rows_from_segments_kernel(
    const __grid_constant__ SlotSnapshot snap, const int32_t* __restrict__ seg_offsets, const int32_t* __restrict__ slot_ids,
    const int32_t* __restrict__ slot_ids2, int G, const int32_t* __restrict__ perm, int T, int8_t* __restrict__ rows,
    int8_t* __restrict__ rows2, uint32_t* __restrict__ status)
{
    __shared__ int32_t seg_s[kBindSegs + 1];
    grid_dependency_wait();
    grid_launch_dependents();
    const int tid = threadIdx.x;
    const bool cached = G <= kBindSegs;
    int bad_off = 0, bad_slot = 0, bad_perm = 0;
    for (int g = tid; g < G; g += blockDim.x) {
        const int s0 = ld_after_wait(seg_offsets + g), s1 = ld_after_wait(seg_offsets + g + 1);
        if (cached) seg_s[g] = s0;
        if (s1 < s0 || s0 < 0 || s1 > T) bad_off = 1;
        const int s = ld_after_wait(slot_ids + g), s2 = slot_ids2 ? ld_after_wait(slot_ids2 + g) : -1;
        if (s1 > s0 && ((s != -1 && slot_rank(snap, s) == 0) || (s2 != -1 && slot_rank(snap, s2) == 0))) bad_slot = 1;
    }
    if (tid == 0) {
        const int last = ld_after_wait(seg_offsets + G);
        if (cached) seg_s[G] = last;
        if (ld_after_wait(seg_offsets) != 0 || last != T) bad_off = 1;
    }
    if (perm)   // (rows that a malformed perm does not name get no adapter)
        for (int i = tid; i < T; i += blockDim.x) { rows[i] = -1; if (rows2) rows2[i] = -1; }
    bad_off = __syncthreads_or(bad_off);
    for (int pos = tid; pos < T; pos += blockDim.x) {
        const int row = perm ? ld_after_wait(perm + pos) : pos;
        if (row < 0 || row >= T) { bad_perm = 1; continue; }
        int s = -1, s2 = -1;
        if (!bad_off) {
            int lo = 0, hi = G;
            while (lo < hi) {
                const int mid = (lo + hi) >> 1;
                if ((cached ? seg_s[mid + 1] : ld_after_wait(seg_offsets + mid + 1)) > pos) hi = mid; else lo = mid + 1;
            }
            if (lo < G) {
                s = ld_after_wait(slot_ids + lo);
                if (slot_rank(snap, s) == 0) s = -1;
                if (slot_ids2) { s2 = ld_after_wait(slot_ids2 + lo); if (slot_rank(snap, s2) == 0) s2 = -1; }
            }
        }
        rows[row] = (int8_t)s;
        if (rows2) rows2[row] = (int8_t)s2;
    }
    bad_slot = __syncthreads_or(bad_slot);
    bad_perm = __syncthreads_or(bad_perm);
    if (tid == 0) {
        const unsigned f = (bad_off ? LML_FLAG_BAD_OFFSETS : 0u) | (bad_slot ? LML_FLAG_BAD_SLOT : 0u) | (bad_perm ? LML_FLAG_BAD_PERM : 0u);
        if (f) atomicOr(status, f);
    }
}

cudaError_t launch_rows_from_segments(const Arena& ar, const SlotSnapshot& snap, const int32_t* seg_offsets, const int32_t* slot_ids,
                                      const int32_t* slot_ids2, int G, const int32_t* perm, int T, int8_t* rows, int8_t* rows2,
                                      cudaStream_t stream)
{
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[1];
    pdl_config(cfg, attr, dim3(1), dim3(1024), 0, stream);
    uint32_t* status = ar.status;
    return cudaLaunchKernelEx(&cfg, rows_from_segments_kernel, snap, seg_offsets, slot_ids, slot_ids2, G, perm, T, rows, rows2, status);
}

}  // namespace lml

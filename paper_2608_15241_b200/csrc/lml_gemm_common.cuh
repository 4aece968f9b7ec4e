// What the kernels of the GEMM path share: the parameters of a launch, the chunks of a row tile, the early start, the terms of
// adapters whose B holds Inf or NaN.  Not part of the public ABI.
#pragma once
#include "lml_internal.cuh"
#include "lml_ptx_sm100.cuh"

namespace lml {

using namespace ptx;

constexpr int kBM = kTileM;   // 128
constexpr int kBK = 64;       // bf16 elements per 128-byte swizzled row
constexpr int kEpiChunkCols = 32;
constexpr int kEpiBufBytes = 32 * kEpiChunkCols * 2;   // 2 KB: 32 rows x 64 B

struct alignas(64) GemmPart {
    CUtensorMap w, y;
    const __nv_bfloat16* bk;            // the table's packed B, by chunk
    const __nv_bfloat16* b;             // ... and by row, as registered
    const uint32_t* nonfinite;
    const TilePlan* plan;               // [row tile] its chunks
    const __nv_bfloat16* u;
    const __nv_bfloat16* u_mid;         // or null: what u's bf16 values leave of the fp32 u, two further K-steps per chunk
    const __nv_bfloat16* u_lo;
    __nv_bfloat16* y_ptr;
    unsigned long long live;            // slots that hold an adapter
    unsigned long long nch[2];          // ... their chunks less one, two bits each
    int N, num_n, n_pad, cap;           // n_pad: rows of a chunk of B in memory
    int tile0;                          // number of its first tile
};
struct alignas(64) GemmParams {
    CUtensorMap x, a, y2;
    GemmPart part[LML_MAX_PROJECTIONS];
    const __nv_bfloat16* u2;            // dual form (else null): the second set of u blocks
    __nv_bfloat16* y2_ptr;              // dual form: the second output
    uint32_t* status;
    int T, K, P;
    int num_m, num_tiles;
    int x_bytes;                // of one copy of x (a k-block of a row tile)
    int stages;                 // split-K kernel: stages of the ring
    int lora;                   // the call has adapters
    int fused;                  // the shrink runs inside this kernel (else a bind_shrink launch came before it)
    RowSource rows;             // fused: where the slot of a row comes from
    int32_t* pass_flags;        // fused: [pass] = epoch + 1 once its u blocks are written
    uint32_t* fuse_sync;        // fused: [0] the table's epoch, [1] CTAs that have finished (the last one advances the epoch)
    uint32_t* x_flag;           // early start (else null): [0] == call_id: x may be read; [1] CTAs that have finished
    uint32_t call_id;
};
__device__ __forceinline__ int slot_chunks(const GemmPart& pt, int slot)
{
    return 1 + (int)((pt.nch[slot >> 5] >> (2 * (slot & 31))) & 3ull);
}
__device__ __forceinline__ int mask_chunks(const GemmPart& pt, unsigned long long mask)
{
    int n = 0;
    for (; mask; mask &= mask - 1ull) n += slot_chunks(pt, __ffsll((long long)mask) - 1);
    return n;
}
// Early start: W0 is on its way already; x may be read once bind_shrink, which this launch overlaps with, says so.  The word is
// polled for a few milliseconds; if the work before the call runs on for longer, the hardware's wait for the whole of bind_shrink
// (which waits for that work) takes over.  The rest of the CTA is held at a barrier meanwhile, so that the limits of the other
// waits in this kernel measure this kernel only.
constexpr long long kPollClocks = 1ll << 22;
__device__ __forceinline__ void wait_x(const uint32_t* x_flag, uint32_t call_id)
{
    const long long t0 = clock64();
    while (ld_acquire_gpu_u32(x_flag) != call_id)
        if (clock64() - t0 > kPollClocks) { grid_dependency_wait(); break; }
    fence_proxy_async_all();
}
// ... and its last CTA clears the word: a replay of the same call finds it cleared.
__device__ __forceinline__ void leave_early_start(uint32_t* x_flag)
{
    if (x_flag && atomicAdd(x_flag + 1, 1u) == gridDim.x * gridDim.y * gridDim.z - 1) {
        x_flag[1] = 0u;
        x_flag[0] = 0u;
    }
}
// the projection that a tile belongs to
__device__ __forceinline__ int part_of(const GemmParams& p, int tile)
{
    int i = 0;
    while (i + 1 < p.P && tile >= p.part[i + 1].tile0) ++i;
    return i;
}
// A whole warp copies the part of a tile's plan that concerns this CTA into shared memory, number << 16 | chunk word:
// chunks that rows use under the bindings `who` and (rank, S) its share of them.  Returns how many.
__device__ __forceinline__ int list_chunks(const TilePlan* plan, uint32_t who, int rank, int S, int lane, uint32_t* out)
{
    uint32_t e = ld_after_wait(&plan->chunk[lane]);   // (goes out with the count; what lies past it is not used)
    const int count = ld_after_wait(&plan->count);
    int n = 0;
    for (int i0 = 0; i0 < count; i0 += 32) {
        const int i = i0 + lane;
        if (i0 > 0) e = i < count ? ld_after_wait(&plan->chunk[i]) : 0u;
        const bool keep = i < count && (e & who) && (S == 1 || (int)((e & 0xffu) + ((e >> 8) & 0xfu)) % S == rank);
        const uint32_t m = __ballot_sync(0xffffffffu, keep);
        if (keep) out[n + __popc(m & ((1u << lane) - 1u))] = ((uint32_t)i << 16) | e;
        n += __popc(m);
    }
    return n;
}
// The terms of one row that the product with the chunks left out, 32 columns from col0: u_j B[n][j] where B is Inf or NaN.
// slot, index: the row's slot and the number of its first chunk (index < 0: looked up in the tile's plan, and the slot with it,
// under binding `which`); u, u_more, u_rest: the sets of blocks whose sum is u (the latter two may be null); out: the row's outputs,
// bf16, 16-byte pieces in an order given by piece_xor.  Out of line, and all of it, so that the epilogue stays as short as it is
// without.
static __device__ __noinline__ void add_nonfinite(const GemmPart& pt, int m, int row, int which, int slot, int index, int col0, const __nv_bfloat16* u,
                                           const __nv_bfloat16* u_more, const __nv_bfloat16* u_rest, uint8_t* out, int piece_xor)
{
    auto value = [](const __nv_bfloat16* p) { return __uint_as_float(ld_after_wait(reinterpret_cast<const uint16_t*>(p)) << 16); };
    if (index < 0) {
        slot = ld_after_wait(&pt.plan[m].nonfinite_row[which][row]);
        if (slot < 0) return;
        for (index = 0; index < kMaxChunks - 1 && (int)(ld_after_wait(&pt.plan[m].chunk[index]) & 0xfffu) != slot;) ++index;
    }
    const size_t u_at = ((size_t)m * pt.cap + index) * (kTileM * kChunk) + chunk_elem(row, 0);
    const int cols = slot_chunks(pt, slot) * kChunk;
    for (int c = 0; c < kEpiChunkCols && col0 + c < pt.N; ++c) {
        const __nv_bfloat16* b = pt.b + ((size_t)slot * pt.N + col0 + c) * kRankPad;
        float sum = 0.f;
        bool any = false;
        for (int j = 0; j < cols; ++j) {
            const float bv = value(b + j);
            if (isfinite(bv)) continue;
            const size_t at = u_at + (size_t)(j / kChunk) * (kTileM * kChunk) + chunk_elem(0, j % kChunk);
            sum += (value(u + at) + (u_more ? value(u_more + at) : 0.f) + (u_rest ? value(u_rest + at) : 0.f)) * bv;
            any = true;
        }
        if (!any) continue;
        __nv_bfloat16* o = reinterpret_cast<__nv_bfloat16*>(out + ((c >> 3) ^ piece_xor) * 16 + (c & 7) * 2);
        *o = __float2bfloat16_rn(__bfloat162float(*o) + sum);
    }
}

// The parts of a projection's parameters that do not depend on the kernel's tiles; tile0: the number of its first tile, of bn columns.
inline void fill_gemm_part(GemmPart& pt, const GemmProj& pr, int bn, int tile0)
{
    pt.bk = pr.ar->Bk; pt.b = pr.ar->B; pt.nonfinite = pr.ar->nonfinite; pt.plan = pr.plan;
    pt.u = pr.u; pt.u_mid = pr.u_mid; pt.u_lo = pr.u_lo; pt.y_ptr = (__nv_bfloat16*)pr.y;
    pt.live = pt.nch[0] = pt.nch[1] = 0ull;
    for (int s = 0; s < pr.snap->max_slots; ++s)
        if (pr.snap->rank[s] > 0) {
            pt.live |= 1ull << s;
            pt.nch[s >> 5] |= (unsigned long long)(chunks_of_rank(pr.snap->rank[s]) - 1) << (2 * (s & 31));
        }
    pt.N = pr.d_out; pt.num_n = (pr.d_out + bn - 1) / bn; pt.n_pad = b_rows_padded(pr.d_out); pt.cap = pr.cap;
    pt.tile0 = tile0;
}

}  // namespace lml

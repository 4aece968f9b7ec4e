// Internal declarations shared by the sm_100a kernels and the host API of the mixed-adapter
// LoRA linear library.  Not part of the public ABI.
#pragma once

#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <mutex>

#include "lora_mixed_linear.h"

namespace lml {

constexpr int kMaxSlots = LML_MAX_SLOTS;
constexpr int kRankPad = 64;          // adapters are stored zero-padded to this rank
constexpr int kRankCompact = 16;      // ... and B a second time, padded to this rank only, where the rank allows
constexpr int kTileM = 128;           // token rows per GEMM tile and per shrink piece block
constexpr int kChunk = 16;            // the LoRA product is computed in chunks of 16 of a slot's columns: one K-step of the tensor cores
constexpr int kMaxChunks = kMaxSlots * (kRankPad / kChunk);   // chunks of a row tile at most
constexpr int kUBlockBytes = kTileM * kChunk * 2;             // u of one row tile and chunk
constexpr int kSlabTiles = 512;       // row tiles worked on at a time: longer calls run in slabs of this many, so that the u blocks stay bounded
constexpr int kBindSegs = 256;        // segments that the kernels look up in shared memory; more are turned into a slot per row first
constexpr int kDecodeMaxT = LML_DECODE_MAX_TOKENS;
constexpr int kMaxAdapterIds = LML_MAX_ADAPTER_IDS;   // adapter ids that can be resolved on the device
constexpr int kFuseMaxPasses = 4096;   // flags of the fused shrink, one a pass; a call has a few hundred passes at most (gemm_fused_shape)

// Per-call snapshot of the slot table, passed by value as a kernel parameter so that a later
// register / retire cannot change a call that is already enqueued.
struct SlotSnapshot {
    uint8_t rank[kMaxSlots];   // 0 = slot not live.  First, with max_slots right behind: what a kernel needs
    int32_t max_slots;         // first sits in one or two lines of the parameter cache (a miss there costs
    float scale[kMaxSlots];    // as much as a trip to L2)
    uint16_t gen[kMaxSlots];   // registration counter of the entry in the slot: what a word of the adapter map must name
};

// Device-resident pieces of a table.
struct Arena {
    __nv_bfloat16* A;   // [max_slots][kRankPad][d_in]   rows >= rank are zero (as far as the last chunk of 16 that the rank needs)
    __nv_bfloat16* B;   // [max_slots][d_out][kRankPad]  columns >= rank are zero (likewise)
    __nv_bfloat16* Bc;  // [max_slots][d_out][kRankCompact]: the same rows, 32 bytes each, for slots of rank <= kRankCompact
                        // (what the decode kernel reads: it needs a row's real columns only, a quarter of the padded row)
    __nv_bfloat16* Bk;  // [max_slots][4 chunks][b_rows_padded(d_out)][kChunk] for the GEMM: a chunk is 16 of the slot's columns, its rows in the
                        // no-swizzle operand order of the tensor cores (see chunk_elem), so that the rows of an output tile are one
                        // contiguous piece and a slot costs the chunks its rank needs and no more.  Zero where B is Inf or NaN: every row
                        // of an output tile meets the chunks of all slots of the tile, and 0 x Inf would reach the rows of other slots
    uint32_t* nonfinite;    // [0] not 0: some registration's B held Inf or NaN; [1 + slot] nonfinite_tag() of the last such one in the slot.  The
                            // GEMM adds those terms to the slot's own rows
    uint32_t* status;   // sticky LML_FLAG_* bits
    int32_t* pass_flags;    // [kFuseMaxPasses] fused shrink of the prefill GEMM: the u blocks of pass i are written (= epoch + 1; the epoch is word 4 of status)
    int32_t* adapter_map;   // [kMaxAdapterIds] serving entry of each adapter id: slot | generation << 8, -1 = none; written by lml_publish
    unsigned long long* dec_u;   // [kDecMaxBlocks][kDecExchStride] the decode kernel's exchange blocks, one per part of a launch that works on this table
};

__host__ __device__ inline uint32_t nonfinite_tag(uint16_t gen) { return 0x10000u | gen; }   // (0: nothing registered yet)
inline int32_t adapter_map_word(int slot, uint16_t gen) { return (int32_t)((uint32_t)slot | ((uint32_t)gen << 8)); }

// ---- kernel launchers (each enqueues on `stream` and returns the launch error) ------------

cudaError_t launch_pack_adapter(const Arena& ar, int slot, uint16_t gen, const void* A, const void* B, int rank,
                                int d_in, int d_out, cudaStream_t stream);

cudaError_t launch_set_word(int32_t* dst, int32_t value, cudaStream_t stream);
cudaError_t launch_clear_word_if(int32_t* dst, int32_t expected, cudaStream_t stream);   // *dst = -1 if it still holds `expected`
cudaError_t aux_init();   // sets the dynamic shared memory attribute of the gradient kernel
// per-chunk segment arrays ([offsets (G + 1) | slot ids (G)] every `stride` ints) of a call done in chunks of `rows` rows
cudaError_t launch_clip_segments(const int32_t* seg_offsets, const int32_t* slot_ids, int G, int T, int rows, int chunks,
                                 int32_t* out, int stride, cudaStream_t stream);
// inputs of a decode call out of pinned host memory (device-accessible pointers) into device staging; x_bytes a multiple of 16
cudaError_t launch_stage_host_inputs(const void* x_host, void* x_dev, size_t x_bytes, const int32_t* so_host, int32_t* so_dev,
                                     int n_so, const int32_t* ids_host, int32_t* ids_dev, int n_ids,
                                     const int32_t* perm_host, int32_t* perm_dev, int n_perm, cudaStream_t stream);
// (A', B') = (B^T, A^T) of a forward adapter A [rank][K], B [N][rank] into slot `slot` of the transposed table's arena
cudaError_t launch_pack_adapter_transposed(const Arena& arT, int slot, uint16_t gen, const void* A, const void* B, int rank,
                                           int K, int N, cudaStream_t stream);
// out_s += P_s^T . Q_s per slot (adapter gradients); mode 0: out[slot][j][c], mode 1: out[slot][c][j]
cudaError_t launch_weight_grad(const SlotSnapshot& snap, const __nv_bfloat16* pieces, const void* Q, int T, int C,
                               const int32_t* seg_offsets, const int32_t* slot_ids, int G, float* out, int mode,
                               cudaStream_t stream,   // optionally a second gradient in the same launch:
                               const __nv_bfloat16* pieces2 = nullptr, const void* Q2 = nullptr, int C2 = 0,
                               float* out2 = nullptr, int mode2 = 0);
cudaError_t launch_segment_tokens(const Arena& ar, const SlotSnapshot& snap, const int32_t* token_slots,
                                  int T, int32_t* perm, int32_t* seg_offsets, int32_t* seg_slot_ids,
                                  cudaStream_t stream, bool by_adapter = false);   // by_adapter: the ids are adapter ids, resolved through ar.adapter_map

// u blocks of the backward pass: block b = (tile m) + (segment g) holds the 128 x 64 bf16 values scale*(x.A^T) of
// the rows of tile m that belong to segment g, zero elsewhere.
cudaError_t launch_shrink_pieces(const Arena& ar, const SlotSnapshot& snap, const void* x, int T,
                                 int d_in, const int32_t* seg_offsets, const int32_t* slot_ids, int G,
                                 __nv_bfloat16* u_blocks, cudaStream_t stream,
                                 int chained = 0);   // 1: a further pass of the same call, may run beside the one before

// ---- binding and shrink of the GEMM path ----------------------------------------------------------
// The rows stay where they are.  Of every 128-row tile the GEMM needs to know which slots its rows use and,
// per chunk of 16 columns of each of those slots, the block u = scale * x.A^T of the tile, zero in the rows that are
// bound to another slot.  A tile's blocks are numbered by slot, then by chunk; it has room for `cap` of them.

__host__ __device__ __forceinline__ int chunks_of_rank(int rank) { return (rank + kChunk - 1) / kChunk; }
// element (row, column) of a chunk's block: 8 x 8 core matrices of 128 contiguous bytes, the two of a row group side by side
__host__ __device__ __forceinline__ size_t chunk_elem(int row, int col)
{
    return (size_t)(row >> 3) * 128 + (size_t)(col >> 3) * 64 + (size_t)(row & 7) * 8 + (size_t)(col & 7);
}
// rows of x that a copy of one row tile brings in: a call of a single tile moves its own rows only (the others' products are
// not stored, whatever the shared memory under them holds)
inline int x_box_rows(int T) { return T >= kTileM ? kTileM : (T + 7) / 8 * 8; }
inline int b_rows_padded(int d_out) { return (d_out + 255) / 256 * 256; }

// What bind_shrink writes for the GEMM, per row tile: the tile's chunks in the order of their blocks.
struct alignas(16) TilePlan {
    int32_t count;
    int32_t pad;
    unsigned long long used;      // the slots that rows of the tile use, under either binding
    uint16_t chunk[kMaxChunks];   // slot | chunk << 8 | kChunkFirst, kChunkSecond
    int8_t nonfinite_row[2][kTileM];   // [binding][row] the row's slot if its B holds Inf or NaN, else -1 (written only where the table has seen such a B)
};
constexpr uint32_t kChunkFirst = 0x1000u, kChunkSecond = 0x2000u;   // rows use the slot under the first / second binding

enum RowMode { kRowsNone = 0, kRowsTokens = 1, kRowsSegments = 2, kRowsGiven = 3 };
// Where the slot of a row comes from: an id per token, the segment arrays (G <= kBindSegs), or a slot per row that
// launch_rows_from_segments has written.
struct RowSource {
    int mode = kRowsNone;
    const int32_t* ids = nullptr;    // segments: per segment (BindPart has the ids of the bind_shrink launch)
    const int32_t* ids2 = nullptr;   // dual calls: the second binding (segments)
    const int32_t* seg_offsets = nullptr;
    int G = 0;
    const int8_t* rows = nullptr;
    const int8_t* rows2 = nullptr;
};
// One projection's share of a launch.
struct BindPart {
    const __nv_bfloat16* A;
    const int32_t* ids;           // per token, or per segment
    const int32_t* adapter_map;   // null: the ids are slots; else adapter ids, resolved through the table's device map
    uint32_t* status;
    const uint32_t* nonfinite;    // as in Arena
    TilePlan* plan;               // [row tile]
    __nv_bfloat16* u;
    __nv_bfloat16* u2;            // further sets of blocks (see BindArgs::second)
    __nv_bfloat16* u3;            // or null
    int cap;
    int pad;
};
// Early start: chunks of a pass, bytes of the ring, and whether the GEMM's CTAs and this launch's have to fit an SM together.
struct BindEarly { int group = 8, ring_bytes = 0; bool share_sm = false; };
struct BindArgs {
    const void* x;
    int T, d_in, P;
    RowSource rows;
    // what u2 holds in a dual call: 1 the second binding's blocks, 2 second minus first.  Else, where a part has u3: u, u2 and u3
    // are three bf16 values whose sum is the fp32 u (zeros in u2 and u3 where u is not finite)
    int second = 0;
    // early start of the GEMM (see bind_starts_gemm_early): the word that says "x may be read" and this call's value of it
    uint32_t* x_flag = nullptr;
    uint32_t call_id = 0;
    BindEarly early;
    BindPart part[LML_MAX_PROJECTIONS];
    SlotSnapshot snap[LML_MAX_PROJECTIONS];
};
// slot per row (int8, -1 = none) of a segment call with a row permutation or with many segments; checks the arrays and raises the flags
cudaError_t launch_rows_from_segments(const Arena& ar, const SlotSnapshot& snap, const int32_t* seg_offsets, const int32_t* slot_ids,
                                      const int32_t* slot_ids2, int G, const int32_t* perm, int T, int8_t* rows, int8_t* rows2,
                                      cudaStream_t stream);
cudaError_t bind_init();

// One projection of a GEMM launch.
struct GemmProj {
    const void* W0;
    void* y;
    int d_out;
    const Arena* ar;
    const SlotSnapshot* snap;
    const TilePlan* plan;
    const __nv_bfloat16* u;
    const __nv_bfloat16* u_mid;   // or null: what the bf16 values in u leave of the fp32 u, in two further sets, multiplied
    const __nv_bfloat16* u_lo;    // with the same B
    int cap;
};
// What the library takes for a call: width of an output tile and CTAs that share one (1: whole-K tiles), CTAs in all, and
// whether a whole-K tile is two row tiles high: the work of a pair of CTAs, or of one (tall).
struct GemmShape { int bn, split, ctas; bool pair, tall = false; };
struct GemmArgs {
    const void* x;
    int T, d_in, P;
    bool lora;                // the call has adapters (a bind_shrink launch came before, unless fused)
    GemmProj proj[LML_MAX_PROJECTIONS];
    GemmShape shape;
    // dual form (one projection): the second set of u blocks, the second output
    const __nv_bfloat16* u2 = nullptr;
    void* y2 = nullptr;
    // fused shrink (one projection): no bind_shrink launch; the kernel binds the rows and computes the u blocks itself
    bool fused = false;
    RowSource rows;
    uint32_t* x_flag = nullptr;   // early start: [0] holds call_id once x may be read, [1] CTAs that have finished (the last one clears both)
    uint32_t call_id = 0;
    bool share_sm = false;        // as in BindArgs
    int num_sms;
    int num_pairs;                // pairs of the pair kernel's CTAs that are resident at once
};
// split_bn, split_s: the table's override (-1 = the library chooses, 0 = whole-K tiles, else the forced shape); precise: some projection's
// u is three bf16 values; slots: of the largest table, 0 without adapters
GemmShape gemm_pick_shape(int T, int d_in, const int* d_outs, int P, bool dual, bool precise, int slots, int num_sms, int num_pairs, int split_bn, int split_s);
// whether the shrink of a plain call of this size runs inside the GEMM kernel, and on which shape
bool gemm_fused_shape(GemmShape* shape, int T, int d_in, int d_out, int G, bool in_segment_order, int max_slots, int num_sms, int split_bn);
// Tensor maps of caller buffers, kept per table and found again by (pointer, shape, box).
struct TmapCache {
    static constexpr int kEntries = 32;
    struct Key { const void* base; uint64_t inner, outer, stride; uint32_t box_inner, box_outer; bool swizzle; };
    Key keys[kEntries];
    CUtensorMap maps[kEntries];
    int used = 0, next = 0;
    std::mutex mu;
    bool get_2d(CUtensorMap* out, const void* base, uint64_t inner, uint64_t outer, uint64_t stride_bytes,
                uint32_t box_inner, uint32_t box_outer, bool swizzle = true);
};
bool gemm_split_override(int* bn_out, int* split_out);
// bind_starts_gemm_early: for calls of few rows the GEMM may start while the work before the call is still running; it then
// reads nothing but W0 until bind_shrink, which waits for that work, has said that x may be read.
bool bind_starts_gemm_early(int T, int P, int num_sms);
int bind_ctas_reckoned(int T, int d_in, int P, int slots, int num_sms);   // what bind_shrink is likely to launch
BindEarly bind_early(int T, int d_in, int P, int cap, int gemm_ctas, bool split, int num_sms);   // ... beside a GEMM of so many CTAs, split-K or not
// tmap_A[p]: the map of projection p's packed A arena ([max_slots][64][d_in], box 64 x 16 x 1)
cudaError_t launch_bind_shrink(const BindArgs& a, const CUtensorMap* const* tmap_A, TmapCache* cache, int num_sms, cudaStream_t stream);
// tmap_A: the same of the (first) table, for the fused shrink; caches[p]: the tensor maps of the buffers of projection p.
// Return cudaErrorInvalidValue if one cannot be encoded.
cudaError_t launch_gemm_sm100(const CUtensorMap& tmap_A, TmapCache* const* caches, const GemmArgs& a, cudaStream_t stream);
cudaError_t launch_gemm_pair(TmapCache* const* caches, const GemmArgs& a, cudaStream_t stream);   // shapes of CTA pairs
cudaError_t gemm_sm100_init(int device);
cudaError_t gemm_pair_init(int num_sms, int* pairs);
int gemm_pair_stages(int bn);
cudaError_t shrink_init();   // these set the dynamic shared memory attributes of their kernels
bool encode_tmap_2d(CUtensorMap* m, const void* base, uint64_t inner, uint64_t outer,
                    uint64_t row_stride_bytes, uint32_t box_inner, uint32_t box_outer, bool swizzle = true);
bool encode_tmap_3d(CUtensorMap* m, const void* base, uint64_t d0, uint64_t d1, uint64_t d2,
                    uint64_t stride1_bytes, uint64_t stride2_bytes, uint32_t b0, uint32_t b1,
                    uint32_t b2);

// The decode kernel's exchange block, through which the CTAs of a launch hand one another u = scale * x.A^T: 16 x kRankPad
// entries (an fp32 value beside the mark of the launch that wrote it, one 64-bit word), then three 32-bit words: the mark
// of the last launch that finished on this block, the CTAs that have left, the entries written.  All zero to begin with.
constexpr int kDecExchEntries = 16 * kRankPad;
constexpr int kDecExchStride = kDecExchEntries + 8;   // 64-bit words per block
constexpr int kDecMaxBlocks = 8;   // parts of one decode launch at most (projections, bindings, blocks of 16 tokens)
struct DecodeArgs {
    const void* x;
    const void* W0;
    void* y;
    const int32_t* perm;
    const int32_t* seg_offsets;
    const int32_t* slot_ids;
    const int32_t* token_slots = nullptr;   // instead of segments: one slot id per row of x (then G is 1 and perm is null)
    bool by_adapter = false;                // the ids in token_slots are adapter ids, resolved through the table's device map
    unsigned long long* exch = nullptr;   // exchange block of the call (kDecExchStride words); null: the table's own, by order of use in the launch
    int T, d_in, d_out, G;
    int num_sms;
};
cudaError_t decode_init();   // sets the dynamic shared memory attributes
int decode_patience();       // LML_DECODE_PATIENCE or the default, in clock cycles
cudaError_t launch_decode(const Arena& ar, const SlotSnapshot& snap, const DecodeArgs& a,
                          cudaStream_t stream, int* launches);
// P <= kDecMaxBlocks parts in one launch (d_in and num_sms equal for all; at most LML_MAX_PROJECTIONS distinct tables):
// projections that read the same x, the two bindings of a dual call, blocks of 16 tokens of a larger batch.
cudaError_t launch_decode_multi(const Arena* const* ars, const SlotSnapshot* snaps, const DecodeArgs* args, int P,
                                cudaStream_t stream);

// Every kernel of the library is launched as a programmatic dependent of whatever precedes it on
// the stream and executes griddepcontrol.wait before it touches global memory (unless its
// predecessor is the library's own kernel of the same call, which has already waited).  The wait
// costs nothing when the predecessor does not trigger early, and otherwise hides launch latency and
// the prologue behind the predecessor's tail.
inline void pdl_config(cudaLaunchConfig_t& cfg, cudaLaunchAttribute* attr, dim3 grid, dim3 block, size_t smem,
                       cudaStream_t stream)
{
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
}

// ---- small device helpers -------------------------------------------------------------------

__device__ __forceinline__ float bf16_lo(uint32_t v) { return __uint_as_float(v << 16); }
__device__ __forceinline__ float bf16_hi(uint32_t v) { return __uint_as_float(v & 0xffff0000u); }

__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi)
{
    __nv_bfloat162 p = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<uint32_t*>(&p);
}

__device__ __forceinline__ uint4 ldg_nc_v4(const void* p)
{
    uint4 v;
    asm volatile("ld.global.nc.L1::no_allocate.v4.u32 {%0,%1,%2,%3}, [%4];"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
    return v;
}

// What an earlier grid of the stream writes while this one is already resident (ids, segment arrays, the plans of the row
// tiles): read with ordinary loads, after griddepcontrol.wait.  The non-coherent path (__ldg) is for data that nobody writes
// during the reading kernel's life; a line of an earlier call's values may wait in L1 there.
__device__ __forceinline__ int ld_after_wait(const int32_t* p)
{
    int v;
    asm volatile("ld.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ uint32_t ld_after_wait(const uint16_t* p)
{
    uint16_t v;
    asm volatile("ld.global.u16 %0, [%1];" : "=h"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ unsigned long long ld_after_wait(const unsigned long long* p)
{
    unsigned long long v;
    asm volatile("ld.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ uint32_t ld_after_wait(const uint32_t* p) { return (uint32_t)ld_after_wait(reinterpret_cast<const int32_t*>(p)); }
__device__ __forceinline__ int ld_after_wait(const int8_t* p)
{
    int v;
    asm volatile("ld.global.s8 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

// D(16x8, fp32) += A(16x16, bf16, row) * B(16x8, bf16, col)
__device__ __forceinline__ void mma_bf16_16816(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2,
                                               uint32_t a3, uint32_t b0, uint32_t b1)
{
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
        "{%0,%1,%2,%3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

// Segment lookup shared by the kernels.  seg_offsets is assumed monotone; all results are clamped so that a
// malformed array can only produce wrong-but-in-range indices.
//
// first segment whose end lies beyond `pos`
__device__ __forceinline__ int seg_upper(const int32_t* __restrict__ seg_offsets, int G, int pos)
{
    int lo = 0, hi = G;   // answer in [0, G]
    while (lo < hi) {
        int mid = (lo + hi) >> 1;
        if (__ldg(seg_offsets + mid + 1) > pos) hi = mid; else lo = mid + 1;
    }
    return lo;
}

__device__ __forceinline__ int slot_rank(const SlotSnapshot& snap, int slot)
{
    return (slot >= 0 && slot < snap.max_slots) ? (int)snap.rank[slot] : 0;
}

// adapter id -> serving slot through the table's device map.  -1 stays -1 (no adapter); an id out of range,
// without a serving version, or whose map word names an entry that is no longer the one in that slot
// (retired, slot taken by another registration since) gives -2: no adapter, and the caller raises the flag.
__device__ __forceinline__ int resolve_adapter(const SlotSnapshot& snap, const int32_t* __restrict__ adapter_map, int id)
{
    if (id == -1) return -1;
    if (id < 0 || id >= kMaxAdapterIds) return -2;
    const int v = __ldg(adapter_map + id);
    if (v < 0) return -2;
    const int slot = v & 0xff;
    if (slot >= snap.max_slots || snap.rank[slot] == 0 || snap.gen[slot] != (uint16_t)((uint32_t)v >> 8)) return -2;
    return slot;
}

}  // namespace lml

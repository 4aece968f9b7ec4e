// Small helper kernels: adapter packing (register_adapter), token segmentation, host staging; the adapter gradients.
#include "lml_internal.cuh"
#include "lml_ptx_sm100.cuh"

namespace lml {

// ---------------------------------------------------------------------------------------------
// register_adapter: copy A[rank][d_in] and B[d_out][rank] into the arena, zero-padded to whole chunks of 16,
// so that every kernel can read fixed-shape, 16-byte aligned rows.
// ---------------------------------------------------------------------------------------------
// Eight columns of one row of B (row n, columns 8g ...) into the three places that hold it: the padded row, the compact row
// of narrow adapters, and the chunk that the GEMM multiplies, which takes zeros for Inf and NaN and leaves a mark.
__device__ __forceinline__ uint32_t finite_or_zero(uint32_t w)   // two bf16 values
{
    if ((w & 0x7f80u) == 0x7f80u) w &= 0xffff0000u;
    if ((w & 0x7f800000u) == 0x7f800000u) w &= 0x0000ffffu;
    return w;
}
__device__ __forceinline__ void store_b_group(__nv_bfloat16* dstB, __nv_bfloat16* dstBc, __nv_bfloat16* dstBk, int n_pad, bool compact,
                                              long long n, int g, const uint4& v, uint32_t* nonfinite, int slot, uint32_t tag)
{
    *reinterpret_cast<uint4*>(dstB + n * kRankPad + g * 8) = v;
    if (compact) *reinterpret_cast<uint4*>(dstBc + n * kRankCompact + g * 8) = v;
    const uint4 f = make_uint4(finite_or_zero(v.x), finite_or_zero(v.y), finite_or_zero(v.z), finite_or_zero(v.w));
    if (f.x != v.x || f.y != v.y || f.z != v.z || f.w != v.w) {   // (the same words from every thread that finds one)
        nonfinite[0] = 1u;
        nonfinite[1 + slot] = tag;
    }
    *reinterpret_cast<uint4*>(dstBk + (size_t)(g >> 1) * n_pad * kChunk + chunk_elem((int)n, (g & 1) * 8)) = f;
}
__device__ __forceinline__ uint4 pack_u16x8(const unsigned short (&e)[8])
{
    return make_uint4(e[0] | ((uint32_t)e[1] << 16), e[2] | ((uint32_t)e[3] << 16), e[4] | ((uint32_t)e[5] << 16),
                      e[6] | ((uint32_t)e[7] << 16));
}

// Only the rows of A and columns of B that are read are written: the chunks of 16 that the rank needs.
__global__ void __launch_bounds__(256) pack_adapter_kernel(__nv_bfloat16* __restrict__ dstA,
                                                           __nv_bfloat16* __restrict__ dstB,
                                                           __nv_bfloat16* __restrict__ dstBc,
                                                           __nv_bfloat16* __restrict__ dstBk, int n_pad,
                                                           const __nv_bfloat16* __restrict__ A,
                                                           const __nv_bfloat16* __restrict__ B,
                                                           int rank, int d_in, int d_out, uint32_t* __restrict__ nonfinite, int slot, uint32_t tag)
{
    const int cols = chunks_of_rank(rank) * kChunk, groups = cols / 8;
    const int k8 = d_in / 8;
    const long long nA = (long long)rank * k8, nA8 = (long long)cols * k8;   // uint4 chunks of A, and with its padding
    const long long nB8 = (long long)d_out * groups;
    const long long stride = (long long)gridDim.x * blockDim.x;
    const long long tid = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    for (long long i = tid; i < nA8; i += stride)   // same linear index: rows are contiguous
        reinterpret_cast<uint4*>(dstA)[i] = i < nA ? __ldg(reinterpret_cast<const uint4*>(A) + i) : make_uint4(0, 0, 0, 0);
    const unsigned short* Bs = reinterpret_cast<const unsigned short*>(B);
    for (long long i = tid; i < nB8; i += stride) {
        const int g = (int)(i % groups);
        const long long n = i / groups;
        uint4 v;
        if ((rank & 7) == 0) {   // rows of B are 16-byte aligned
            v = g * 8 < rank ? __ldg(reinterpret_cast<const uint4*>(Bs + n * rank + g * 8)) : make_uint4(0, 0, 0, 0);
        } else {
            unsigned short e[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) e[j] = g * 8 + j < rank ? Bs[n * rank + g * 8 + j] : (unsigned short)0;
            v = pack_u16x8(e);
        }
        store_b_group(dstB, dstBc, dstBk, n_pad, rank <= kRankCompact, n, g, v, nonfinite, slot, tag);
    }
}

static int pack_blocks(long long work)
{
    const long long blocks = (work + 255) / 256;
    return (int)(blocks > 1184 ? 1184 : (blocks < 1 ? 1 : blocks));
}

cudaError_t launch_pack_adapter(const Arena& ar, int slot, uint16_t gen, const void* A, const void* B, int rank,
                                int d_in, int d_out, cudaStream_t stream)
{
    __nv_bfloat16* dstA = ar.A + (size_t)slot * kRankPad * d_in;
    __nv_bfloat16* dstB = ar.B + (size_t)slot * d_out * kRankPad;
    __nv_bfloat16* dstBc = ar.Bc + (size_t)slot * d_out * kRankCompact;
    const int n_pad = b_rows_padded(d_out);
    __nv_bfloat16* dstBk = ar.Bk + (size_t)slot * kRankPad * n_pad;
    const long long work = (long long)chunks_of_rank(rank) * 2 * (d_in > d_out ? d_in : d_out);
    pack_adapter_kernel<<<pack_blocks(work), 256, 0, stream>>>(dstA, dstB, dstBc, dstBk, n_pad, (const __nv_bfloat16*)A,
                                                               (const __nv_bfloat16*)B, rank, d_in, d_out, ar.nonfinite, slot, nonfinite_tag(gen));
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------------------------
// Token segmentation: stable counting sort of T tokens by slot (keys 0..max_slots-1, then -1).
// One CTA of 32 warps.  Warp w owns a contiguous range of tokens; pass 1 counts keys per warp,
// a scan turns the counts into (key-major, warp-minor) start positions, pass 2 walks the same
// range in order and places each token, using match_any to rank equal keys inside a 32-token
// chunk.  Everything is order-deterministic.
// ---------------------------------------------------------------------------------------------
constexpr int kSegWarps = 32;
constexpr int kSegKeyCache = 16384;   // tokens whose keys are kept in shared memory between the two passes

__global__ void set_word_kernel(int32_t* dst, int32_t value) { *dst = value; }
__global__ void clear_word_if_kernel(int32_t* dst, int32_t expected) { if (*dst == expected) *dst = -1; }

cudaError_t launch_clear_word_if(int32_t* dst, int32_t expected, cudaStream_t stream)
{
    clear_word_if_kernel<<<1, 1, 0, stream>>>(dst, expected);
    return cudaGetLastError();
}

cudaError_t launch_set_word(int32_t* dst, int32_t value, cudaStream_t stream)
{
    set_word_kernel<<<1, 1, 0, stream>>>(dst, value);
    return cudaGetLastError();
}

// Host-buffer form of a decode call whose host buffers are pinned: one kernel pulls the inputs out of
// host memory (16-byte loads for x, all in flight at once: one trip over the host link instead of a DMA
// copy per array) into the device staging that the decode kernel reads.
__global__ void __launch_bounds__(256) stage_host_inputs_kernel(
    const uint4* __restrict__ x_host, uint4* __restrict__ x_dev, int x_chunks, const int32_t* __restrict__ so_host,
    int32_t* __restrict__ so_dev, int n_so, const int32_t* __restrict__ ids_host, int32_t* __restrict__ ids_dev, int n_ids,
    const int32_t* __restrict__ perm_host, int32_t* __restrict__ perm_dev, int n_perm)
{
    ptx::grid_dependency_wait();   // the call before may still read the staging
    ptx::grid_launch_dependents();
    const int i = blockIdx.x * blockDim.x + threadIdx.x, n = gridDim.x * blockDim.x;
    for (int c = i; c < x_chunks; c += n) x_dev[c] = x_host[c];
    for (int c = i; c < n_so; c += n) so_dev[c] = so_host[c];
    for (int c = i; c < n_ids; c += n) ids_dev[c] = ids_host[c];
    for (int c = i; c < n_perm; c += n) perm_dev[c] = perm_host[c];
}

cudaError_t launch_stage_host_inputs(const void* x_host, void* x_dev, size_t x_bytes, const int32_t* so_host, int32_t* so_dev,
                                     int n_so, const int32_t* ids_host, int32_t* ids_dev, int n_ids,
                                     const int32_t* perm_host, int32_t* perm_dev, int n_perm, cudaStream_t stream)
{
    const int chunks = (int)(x_bytes / 16);
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[1];
    pdl_config(cfg, attr, dim3((unsigned)((chunks + 255) / 256 < 1 ? 1 : (chunks + 255) / 256)), dim3(256), 0, stream);
    return cudaLaunchKernelEx(&cfg, stage_host_inputs_kernel, (const uint4*)x_host, (uint4*)x_dev, chunks, so_host, so_dev,
                              n_so, ids_host, ids_dev, n_ids, perm_host, perm_dev, n_perm);
}

// Host-buffer form of large calls, done chunk by chunk: the segment arrays of chunk c (rows [c * rows,
// (c + 1) * rows) of the call), offsets relative to the chunk and clipped to it.  Malformed offsets are
// detected on the whole call and poison every chunk's array, so that every chunk falls back to the base
// output, as the unchunked call does.
__global__ void __launch_bounds__(256) clip_segments_kernel(const int32_t* __restrict__ seg_offsets,
                                                            const int32_t* __restrict__ slot_ids, int G, int T, int rows,
                                                            int32_t* __restrict__ out, int stride)
{
    ptx::grid_dependency_wait();
    ptx::grid_launch_dependents();
    const int c = blockIdx.x, r0 = c * rows, Tc = min(rows, T - r0);
    int32_t* so = out + (size_t)c * stride;
    int32_t* ids = so + G + 1;
    int bad = 0;
    for (int g = threadIdx.x; g < G; g += blockDim.x) {
        const int s0 = __ldg(seg_offsets + g), s1 = __ldg(seg_offsets + g + 1);
        if (s1 < s0 || s0 < 0 || s1 > T) bad = 1;
    }
    if (threadIdx.x == 0 && (__ldg(seg_offsets) != 0 || __ldg(seg_offsets + G) != T)) bad = 1;
    bad = __syncthreads_or(bad);
    for (int g = threadIdx.x; g <= G; g += blockDim.x) {
        const int v = min(max(__ldg(seg_offsets + g) - r0, 0), Tc);
        so[g] = bad ? (g == 0 ? 1 : 0) : v;   // (an array that starts at 1 is malformed for every chunk)
        if (g < G) ids[g] = __ldg(slot_ids + g);
    }
}

cudaError_t launch_clip_segments(const int32_t* seg_offsets, const int32_t* slot_ids, int G, int T, int rows, int chunks,
                                 int32_t* out, int stride, cudaStream_t stream)
{
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[1];
    pdl_config(cfg, attr, dim3((unsigned)chunks), dim3(256), 0, stream);
    return cudaLaunchKernelEx(&cfg, clip_segments_kernel, seg_offsets, slot_ids, G, T, rows, out, stride);
}

__global__ void __launch_bounds__(kSegWarps * 32) segment_tokens_kernel(
    const __grid_constant__ SlotSnapshot snap, const int32_t* __restrict__ token_slots, int T,
    int32_t* __restrict__ perm, int32_t* __restrict__ seg_offsets, int32_t* __restrict__ seg_slot_ids,
    uint32_t* __restrict__ status, const int32_t* __restrict__ adapter_map)
{
    __shared__ int hist[kSegWarps][kMaxSlots + 1];
    __shared__ int base[kMaxSlots + 2];
    __shared__ uint8_t keys_s[kSegKeyCache];
    const int nk = snap.max_slots + 1;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (int i = threadIdx.x; i < kSegWarps * (kMaxSlots + 1); i += blockDim.x) (&hist[0][0])[i] = 0;
    ptx::grid_dependency_wait();      // launched as a programmatic dependent: whatever ran before is complete now
    ptx::grid_launch_dependents();    // the next kernel may get resident; it waits for this one the same way
    // Up to kSegKeyCache tokens: every key is fetched once, all loads in flight together (one trip to memory instead of
    // one per 32 tokens of a warp's range and pass), and both passes read shared memory.  0xff marks an id that names
    // no live slot (it counts as "none" and raises the flag).
    const bool cached = T <= kSegKeyCache;
    if (cached) {
        for (int i = threadIdx.x; i < T; i += blockDim.x) {
            int s = __ldg(token_slots + i);
            if (adapter_map) s = resolve_adapter(snap, adapter_map, s);
            const bool bad_id = s < -1 || s >= snap.max_slots || (s >= 0 && snap.rank[s] == 0);
            keys_s[i] = bad_id ? (uint8_t)0xff : (uint8_t)(s < 0 ? snap.max_slots : s);
        }
    }
    __syncthreads();

    int per = (T + kSegWarps - 1) / kSegWarps;
    per = (per + 31) & ~31;
    const int begin = min(T, warp * per);
    const int end = min(T, begin + per);
    bool bad = false;

    for (int c = begin; c < end; c += 32) {
        int i = c + lane;
        if (i < end) {
            int key;
            if (cached) {
                key = keys_s[i];
                if (key == 0xff) { bad = true; key = snap.max_slots; }
            } else {
                int s = __ldg(token_slots + i);
                if (adapter_map) s = resolve_adapter(snap, adapter_map, s);
                if (s < -1 || s >= snap.max_slots || (s >= 0 && snap.rank[s] == 0)) { bad = true; s = -1; }
                key = s < 0 ? snap.max_slots : s;
            }
            atomicAdd(&hist[warp][key], 1);
        }
    }
    if (bad) atomicOr(status, LML_FLAG_BAD_SLOT);
    __syncthreads();
    if ((int)threadIdx.x < nk) {
        int run = 0;
        for (int w = 0; w < kSegWarps; ++w) { int c = hist[w][threadIdx.x]; hist[w][threadIdx.x] = run; run += c; }
        base[threadIdx.x] = run;   // total of this key for now
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        int run = 0;
        for (int k = 0; k < nk; ++k) {
            int c = base[k];
            base[k] = run;
            seg_offsets[k] = run;
            seg_slot_ids[k] = k < snap.max_slots ? k : -1;
            run += c;
        }
        seg_offsets[nk] = run;
    }
    __syncthreads();

    for (int c = begin; c < end; c += 32) {   // trip count is uniform inside a warp
        int i = c + lane;
        int key = nk;                          // sentinel for lanes past the end
        if (i < end) {
            if (cached) {
                key = keys_s[i] == 0xff ? snap.max_slots : (int)keys_s[i];
            } else {
                int s = __ldg(token_slots + i);
                if (adapter_map) s = resolve_adapter(snap, adapter_map, s);
                if (s < -1 || s >= snap.max_slots || (s >= 0 && snap.rank[s] == 0)) s = -1;
                key = s < 0 ? snap.max_slots : s;
            }
        }
        unsigned m = __match_any_sync(0xffffffffu, key);
        int before = __popc(m & ((1u << lane) - 1u));
        int pos = 0;
        if (key < nk) {
            pos = base[key] + hist[warp][key] + before;
            perm[pos] = i;
        }
        __syncwarp();
        if (key < nk && before == 0) hist[warp][key] += __popc(m);
        __syncwarp();
    }
}

cudaError_t launch_segment_tokens(const Arena& ar, const SlotSnapshot& snap, const int32_t* token_slots,
                                  int T, int32_t* perm, int32_t* seg_offsets, int32_t* seg_slot_ids,
                                  cudaStream_t stream, bool by_adapter)
{
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[1];
    pdl_config(cfg, attr, dim3(1), dim3(kSegWarps * 32), 0, stream);
    uint32_t* status = ar.status;
    const int32_t* map = by_adapter ? ar.adapter_map : nullptr;
    return cudaLaunchKernelEx(&cfg, segment_tokens_kernel, snap, token_slots, T, perm, seg_offsets, seg_slot_ids, status, map);
}

// ---------------------------------------------------------------------------------------------
// Transposed registration for the backward pass: the gradient with respect to x of the layer
// (d_in = K, d_out = N, adapter A [r][K], B [N][r]) is the layer itself on the transposed problem
// (d_in = N, d_out = K, base weight W0^T, adapter A' = B^T [r][N], B' = A^T [K][r]).  This kernel
// packs (A', B') into the arena of the transposed table straight from the caller's A and B.
// ---------------------------------------------------------------------------------------------
__global__ void __launch_bounds__(256) pack_adapter_transposed_kernel(__nv_bfloat16* __restrict__ dstA,
                                                                      __nv_bfloat16* __restrict__ dstB,
                                                                      __nv_bfloat16* __restrict__ dstBc,
                                                                      __nv_bfloat16* __restrict__ dstBk, int k_pad,
                                                                      const __nv_bfloat16* __restrict__ A,
                                                                      const __nv_bfloat16* __restrict__ B,
                                                                      int rank, int K, int N, uint32_t* __restrict__ nonfinite, int slot, uint32_t tag)
{
    const unsigned short* As = reinterpret_cast<const unsigned short*>(A);
    const unsigned short* Bs = reinterpret_cast<const unsigned short*>(B);
    unsigned short* Ad = reinterpret_cast<unsigned short*>(dstA);   // [64][N]: A'[j][n] = B[n][j]
    const int cols = chunks_of_rank(rank) * kChunk, groups = cols / 8;
    const long long stride = (long long)gridDim.x * blockDim.x;
    const long long tid = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    for (long long i = tid; i < (long long)cols * N; i += stride) {
        const int j = (int)(i / N);
        const long long n = i % N;
        Ad[i] = j < rank ? Bs[n * rank + j] : (unsigned short)0;
    }
    for (long long i = tid; i < (long long)K * groups; i += stride) {   // B'[k][j] = A[j][k]
        const int g = (int)(i / K);
        const long long k = i % K;
        unsigned short e[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) e[j] = g * 8 + j < rank ? As[(long long)(g * 8 + j) * K + k] : (unsigned short)0;
        store_b_group(dstB, dstBc, dstBk, k_pad, rank <= kRankCompact, k, g, pack_u16x8(e), nonfinite, slot, tag);
    }
}

cudaError_t launch_pack_adapter_transposed(const Arena& arT, int slot, uint16_t gen, const void* A, const void* B, int rank,
                                           int K, int N, cudaStream_t stream)
{
    __nv_bfloat16* dstA = arT.A + (size_t)slot * kRankPad * N;   // the transposed table has d_in = N ...
    __nv_bfloat16* dstB = arT.B + (size_t)slot * K * kRankPad;   // ... and d_out = K
    __nv_bfloat16* dstBc = arT.Bc + (size_t)slot * K * kRankCompact;
    const int k_pad = b_rows_padded(K);
    __nv_bfloat16* dstBk = arT.Bk + (size_t)slot * kRankPad * k_pad;
    const long long work = (long long)chunks_of_rank(rank) * kChunk * (K > N ? K : N);
    pack_adapter_transposed_kernel<<<pack_blocks(work), 256, 0, stream>>>(dstA, dstB, dstBc, dstBk, k_pad, (const __nv_bfloat16*)A,
                                                                          (const __nv_bfloat16*)B, rank, K, N, arT.nonfinite, slot, nonfinite_tag(gen));
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------------------------
// Adapter gradients: out_s += P_s^T . Q_s over the tokens bound to slot s, where P holds one
// 64-wide row per position (the piece blocks a shrink pass wrote: scale.(dy.B) for dA, scale.(x.A^T)
// for dB) and Q is x (for dA, C = d_in) or dy (for dB, C = d_out).  One CTA of eight warps per
// (128 columns, slot), two CTAs to an SM; the contraction over positions runs on mma.sync (see the
// kernel), the slot's positions are walked in order and the sums stay in registers, so the result does
// not depend on scheduling.  fp32 accumulation, added onto what out holds.
// mode 0: out[slot][j][c] (dA);  mode 1: out[slot][c][j] (dB).
// ---------------------------------------------------------------------------------------------
constexpr int kGradCols = 128;                                  // columns of Q (and of the output) per CTA: two CTAs fit on an SM
constexpr int kGradQPitch = kGradCols * 2 + 16;                 // bytes per row of the staged Q tile (16 more: no bank conflicts in ldmatrix)
constexpr int kGradPPitch = kRankPad * 2 + 16;                  // bytes per row of the staged piece block
constexpr int kGradQBytes = kTileM * kGradQPitch;
constexpr int kGradPBytes = kTileM * kGradPPitch;
constexpr int kGradSmemBytes = 2 * (kGradQBytes + kGradPBytes); // two work items in flight

__device__ __forceinline__ void grad_cp_async_16(uint32_t dst, const void* src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void ldmatrix_x4_trans(uint32_t addr, uint32_t& r0, uint32_t& r1, uint32_t& r2, uint32_t& r3)
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3) : "r"(addr));
}

// out_s (64 x C) += P_s^T (64 x positions) . Q_s (positions x C) on mma.sync m16n8k16: the contraction
// runs over positions, 16 at a time.  P is staged as [position][j] and Q as [position][column], so both
// operands are read with ldmatrix .trans.  Warp w owns columns 16w .. 16w+15 (two 8-wide tiles) and all
// 16-row groups of j that the slot's rank needs.
// One launch does both gradients side by side: blockIdx.z = 0 takes the first set of arguments, 1 the second.
struct GradJob {
    const __nv_bfloat16* pieces;
    const __nv_bfloat16* Q;
    float* out;
    int C, mode;
};
__global__ void __launch_bounds__(256, 2) weight_grad_kernel(const __grid_constant__ SlotSnapshot snap, const GradJob job0,
                                                          const GradJob job1, int T,
                                                          const int32_t* __restrict__ seg_offsets,
                                                          const int32_t* __restrict__ slot_ids, int G)
{
    extern __shared__ __align__(16) unsigned char grad_smem[];
    ptx::grid_dependency_wait();     // the shrink passes before this kernel are complete now
    ptx::grid_launch_dependents();
    const GradJob& job = blockIdx.z == 0 ? job0 : job1;
    const __nv_bfloat16* __restrict__ pieces = job.pieces;
    const __nv_bfloat16* __restrict__ Q = job.Q;
    float* __restrict__ out = job.out;
    const int C = job.C, mode = job.mode;
    if ((int)blockIdx.x * kGradCols >= C) return;
    const int slot = blockIdx.y;
    const int rank = slot < snap.max_slots ? (int)snap.rank[slot] : 0;
    if (rank == 0) return;
    const int mtiles = (rank + 15) >> 4;   // 16-row groups of j
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int c0 = blockIdx.x * kGradCols;
    const int ncols = min(kGradCols, C - c0);
    float acc[4][2][4];   // [16-row group of j][8-column tile][fragment]
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int n = 0; n < 2; ++n) acc[a][n][0] = acc[a][n][1] = acc[a][n][2] = acc[a][n][3] = 0.f;
    const uint32_t smem = (uint32_t)__cvta_generic_to_shared(grad_smem);
    auto q_off = [](int buf) { return (uint32_t)(buf * (kGradQBytes + kGradPBytes)); };
    auto p_off = [](int buf) { return (uint32_t)(buf * (kGradQBytes + kGradPBytes) + kGradQBytes); };

    // Work items of this CTA: the slot's segments in order, each tile of a segment in order.  A piece block
    // (tile m, segment g) holds the rows of tile m that belong to g and zeros elsewhere, so the whole tile
    // of Q is multiplied (rows past T are zero-filled here).  Block and tile are brought into shared memory
    // by asynchronous copies, one item ahead of the arithmetic.
    int g = -1, m = 0, m_last = -1;
    auto advance = [&]() -> bool {   // next (g, m); false when the slot has no more
        if (m < m_last) { ++m; return true; }
        for (++g; g < G; ++g) {
            if (__ldg(slot_ids + g) != slot) continue;
            const int s0 = max(__ldg(seg_offsets + g), 0), s1 = min(__ldg(seg_offsets + g + 1), T);
            if (s1 <= s0) continue;
            m = s0 / kTileM;
            m_last = (s1 - 1) / kTileM;
            return true;
        }
        return false;
    };
    auto issue = [&](int buf) {
        const char* blk = reinterpret_cast<const char*>(pieces + (size_t)(m + g) * kTileM * kRankPad);
        for (int i = tid; i < kTileM * (kRankPad / 8); i += 256) {
            const int r = i / (kRankPad / 8), ch = i % (kRankPad / 8);
            grad_cp_async_16(smem + p_off(buf) + r * kGradPPitch + ch * 16, blk + (size_t)i * 16);
        }
        const int rows = min(kTileM, T - m * kTileM);
        const int chunks = ncols / 8;   // 16-byte chunks per row
        for (int i = tid; i < kTileM * chunks; i += 256) {
            const int r = i / chunks, ch = i % chunks;
            const uint32_t dst = smem + q_off(buf) + r * kGradQPitch + ch * 16;
            if (r < rows) grad_cp_async_16(dst, Q + (size_t)(m * kTileM + r) * C + c0 + ch * 8);
            else asm volatile("st.shared.v4.u32 [%0], {%1,%1,%1,%1};" ::"r"(dst), "r"(0u) : "memory");
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    bool have = advance();
    int buf = 0;
    if (have) issue(0);
    while (have) {
        const bool more = advance();
        if (more) issue(buf ^ 1);
        if (more) asm volatile("cp.async.wait_group 1;" ::: "memory");
        else asm volatile("cp.async.wait_group 0;" ::: "memory");
        __syncthreads();   // everybody's copies of the current item have landed
        const uint32_t qb = smem + q_off(buf), pb = smem + p_off(buf);
        // ldmatrix x4: lanes 0-7 address the rows of matrix 0, 8-15 of matrix 1, 16-23 of matrix 2, 24-31 of 3
        const int mi = lane >> 3, rr = lane & 7;
#pragma unroll 2
        for (int ks = 0; ks < kTileM / 16; ++ks) {
            const int p0 = ks * 16;
            // B operand for the warp's two column tiles: matrices (p 0-7 | 8-15) x (tile 0 | tile 1)
            uint32_t bq[2][2];
            {
                const uint32_t addr = qb + (uint32_t)((p0 + (mi & 1) * 8 + rr) * kGradQPitch + (warp * 16 + (mi >> 1) * 8) * 2);
                ldmatrix_x4_trans(addr, bq[0][0], bq[0][1], bq[1][0], bq[1][1]);
            }
#pragma unroll
            for (int a = 0; a < 4; ++a) {
                if (a < mtiles) {
                    // A operand (j x p) from the block stored [p][j]: matrices (p 0-7, j 0-7), (p 0-7, j 8-15),
                    // (p 8-15, j 0-7), (p 8-15, j 8-15) give a0..a3
                    uint32_t a0, a1, a2, a3;
                    const uint32_t addr = pb + (uint32_t)((p0 + (mi >> 1) * 8 + rr) * kGradPPitch + (a * 16 + (mi & 1) * 8) * 2);
                    ldmatrix_x4_trans(addr, a0, a1, a2, a3);
#pragma unroll
                    for (int n = 0; n < 2; ++n) mma_bf16_16816(acc[a][n], a0, a1, a2, a3, bq[n][0], bq[n][1]);
                }
            }
        }
        __syncthreads();   // the buffer may be refilled two items from now
        have = more;
        buf ^= 1;
    }
    // fragment: c0,c1 = (j = gq, columns 2tq, 2tq+1), c2,c3 = (j = gq + 8, same columns)
    const int gq = lane >> 2, tq = lane & 3;
#pragma unroll
    for (int a = 0; a < 4; ++a) {
        if (a >= mtiles) continue;
#pragma unroll
        for (int n = 0; n < 2; ++n) {
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const int j = a * 16 + gq + (e >> 1) * 8;
                const int c = c0 + warp * 16 + n * 8 + tq * 2 + (e & 1);
                if (j < rank && c < C) {
                    float* o = mode == 0 ? out + ((size_t)slot * kRankPad + j) * C + c : out + ((size_t)slot * C + c) * kRankPad + j;
                    *o += acc[a][n][e];
                }
            }
        }
    }
}

cudaError_t launch_weight_grad(const SlotSnapshot& snap, const __nv_bfloat16* pieces, const void* Q, int T, int C,
                               const int32_t* seg_offsets, const int32_t* slot_ids, int G, float* out, int mode,
                               cudaStream_t stream, const __nv_bfloat16* pieces2, const void* Q2, int C2, float* out2, int mode2)
{
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[1];
    const int cmax = (out2 && C2 > C) ? C2 : C;
    pdl_config(cfg, attr, dim3((cmax + kGradCols - 1) / kGradCols, snap.max_slots, out2 ? 2 : 1), dim3(256), kGradSmemBytes, stream);
    const GradJob j0 = {pieces, (const __nv_bfloat16*)Q, out, C, mode};
    const GradJob j1 = {pieces2, (const __nv_bfloat16*)Q2, out2, C2, mode2};
    return cudaLaunchKernelEx(&cfg, weight_grad_kernel, snap, j0, j1, T, seg_offsets, slot_ids, G);
}

cudaError_t aux_init()   // called with the table's device current, once per table
{
    return cudaFuncSetAttribute(weight_grad_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kGradSmemBytes);
}

}  // namespace lml

// Internal declarations shared by the host API and the kernel translation units.
#pragma once
#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "../../include/hydra_attn.h"
#include "once_per_device.h"

namespace hydra {

constexpr int D_QK = HYDRA_D_QK;
constexpr int D_V = HYDRA_D_V;
constexpr int TILE = 128;       // rows of a q tile and of a kv tile
constexpr int SUB = 64;         // rows of a q sub-tile in the key-side backward kernel
constexpr int FWD_SHORT_KEYS = 64;   // keys per step of the short-sequence forward kernel

// One (q-chunk, kv-chunk) pair with absolute token offsets, as the kernels see it.
struct PairDev {
    int32_t q_tok0;    // token index of the pair's first q row
    int32_t q_len;
    int32_t k_tok0;    // token index of the pair's first kv row
    int32_t k_len;
    int32_t off;       // q_start - k_start: key j is visible to q row i iff j <= i + off (causal)
    int32_t out_row0;  // first output row: part_row (partial buffers) or q_tok0 (out / lse)
    int32_t to_part;   // 1: partial buffers, 0: out / lse
    int32_t ds_base;   // backward: first block of this pair in the dS hand-off buffer (per head)
};

// Geometry of the dS hand-off buffer of the backward. The key-side kernel writes dS^T of every
// (128-row kv tile jk, 64-row q sub-tile u) it visits as one block of 16 KB: 8 chunks (8 q rows each) of
// 128 kv rows x 16 bytes, which is the tensor core's operand layout without swizzle (so the writer's
// stores are contiguous per warp and the reader's copy is one untiled bulk copy); the
// query-side kernel reads the blocks (jk, 2i) and (jk, 2i + 1) of its q tile i. Per pair the blocks of
// kv tile jk start at ds_rowstart(jk) and cover the sub-tiles ds_first(jk) .. nu_even - 1, where
// ds_first is the first sub-tile the causal mask leaves visible, rounded down to an even number, so
// that the buffer holds the visible trapezoid only. Both kernels and the host evaluate these forms.
struct DsGeom { int32_t nu_even; int32_t fo; };
__host__ __device__ inline DsGeom ds_geom(int32_t q_len, int32_t off, int causal)
{
    DsGeom g;
    g.nu_even = ((q_len + SUB - 1) / SUB + 1) & ~1;
    // fo = floor(-off / 128): kv tile jk sees q tiles jk + fo and later
    g.fo = !causal ? -(1 << 24) : (off <= 0 ? (-off) / TILE : -((off + TILE - 1) / TILE));
    return g;
}
__host__ __device__ inline int32_t ds_first(const DsGeom& g, int32_t jk)
{
    const int32_t m = jk + g.fo;
    return m > 0 ? 2 * m : 0;
}
__host__ __device__ inline int64_t ds_rowstart(const DsGeom& g, int32_t jk)
{
    int64_t m = static_cast<int64_t>(jk) + g.fo;
    if (m < 0) m = 0;
    const int64_t m0 = g.fo > 0 ? g.fo : 0;
    return static_cast<int64_t>(jk) * g.nu_even - (m * (m - 1) - m0 * (m0 - 1));
}
constexpr uint32_t DS_BLOCK_BYTES = TILE * SUB * 2;   // 16 KB

// Forward work item: up to 512 q rows of one pair and head = tiles A and B of 256 rows (128 per CTA of the pair).
struct FwdItem {
    int32_t pair;
    int32_t head;
    int32_t q0;        // first q row of tile A, relative to the pair; tile B starts at q0 + 128
    int32_t n_a;       // kv tiles tile A visits (after causal clipping); 0: its rows see no key
    int32_t n_b;       // same for tile B; -1 when the item has no second tile (its rows belong to another item)
    int32_t pad[3];
};

// Work item of the short-sequence forward kernel: one 128-row q tile of one pair and head, self-contained
// (a slot of that kernel reads nothing else to start it).
struct alignas(16) FwdShortItem {
    int32_t q_tok0;    // token index of the tile's first q row
    int32_t k_tok0;    // token index of the pair's first kv row
    int32_t k_len;
    int32_t off;       // key j is visible to row r of the tile iff j <= r + off (causal)
    int32_t out_row0;  // output row of the tile's first q row (partial buffers or out / lse)
    uint16_t head;
    uint16_t n_kv;     // steps of FWD_SHORT_KEYS keys the tile visits; 0: its rows see no key
    uint8_t rows;      // q rows of the tile that exist (1..128)
    uint8_t to_part;   // 1: partial buffers, 0: out / lse
    uint16_t half_segs;    // half() | n_segs() << 8 (one field: with two of a byte the kernel takes 16 registers more)
    uint32_t first_seg;    // (a call has at most pairs + tiles of them, and of each fewer than 2^31)
    // 0: all keys of the tile; 1, 2: its first and second part, run by the two slots of one thread block (the second hands its
    // result to the first)
    __host__ __device__ int half() const { return half_segs & 255; }
    // 0: all rows as above; else how many FwdSeg (at most 128), from first_seg on, say where the rows go
    __host__ __device__ int n_segs() const { return half_segs >> 8; }
};
static_assert(sizeof(FwdShortItem) == 32, "two 16-byte loads per work item");

// Rows of a tile that belong to one of several pairs: consecutive q chunks that meet the same kv chunk share their tiles.
struct FwdSeg {
    int16_t begin;     // first row of the tile; the segment ends where the next one begins
    int16_t to_part;
    int32_t delta;     // output row of tile row r is r + delta
};

// Backward work item: one tile of one chunk and head, visiting every pair that shares the chunk (key side: for
// BwdParams::item_heads query heads, of which `head` is the first).
struct GroupItem {
    int32_t list_off;  // first entry of the chunk's pair list
    int32_t list_len;
    int32_t head;
    int32_t r0;        // first row of the tile, relative to the chunk
};

// Merge: one q chunk with two or more partials.
struct MergeGroup {
    int32_t out_tok0;  // first token of the chunk in out / lse
    int32_t rows;
    int32_t list_off;  // first entry of the chunk's part_row list
    int32_t n_parts;
};
struct MergeItem {
    int32_t group;
    int32_t row0;      // first row of the block, relative to the chunk
};
constexpr int MERGE_ROWS = 8;   // rows of a merge block

// Lives at the start of the workspace. Zeroed before the kernels of a call, except in forward calls with a call_tag, whose
// workspace keeps what it held: there next_item is undefined and `status` counts as said below.
struct StatusBlock {
    int32_t status;
    int32_t pad;
    int64_t detail;
    int32_t next_item[4];       // work-queue heads of the persistent kernels (forward, dK/dV, dQ, short forward)
    // A call none of whose kernels pops from a queue is not worth a launch that clears this block. Its kernel writes call_tag,
    // a number of the call's own, and with an error the same number as error_tag; `status` counts only while the two are
    // equal, as they are (zero) wherever the block is cleared. (64 mixed bits: a workspace may hold anything, and small
    // numbers, which positions or token ids leave there, were taken for the first calls' own.)
    uint64_t call_tag, error_tag;
    // SM clock seen from inside the tensor-core kernels: cycles and nanoseconds that passed in the
    // producer thread of CTA 0 between its first and its last instruction (same index as next_item)
    uint64_t probe_cycles[4];
    uint64_t probe_ns[4];
};
enum : int { QUEUE_FWD = 0, QUEUE_DKV = 1, QUEUE_DQ = 2, QUEUE_FWD_SHORT = 3 };

#ifdef __CUDACC__
// The clock the driver reports between kernels says little about a 1 ms kernel on a power-capped part;
// the ratio of the cycle counter to the nanosecond timer inside the kernel does.
struct ClockProbe {
    long long c0; uint64_t t0;
    __device__ __forceinline__ void start()
    {
        c0 = clock64();
        asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t0));
    }
    __device__ __forceinline__ void stop(StatusBlock* sb, int queue) const
    {
        uint64_t t1;
        asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t1));
        sb->probe_cycles[queue] = static_cast<uint64_t>(clock64() - c0);
        sb->probe_ns[queue] = t1 - t0;
    }
};
#endif

// Launches of one stream overlap at their ends: every kernel of the library lets the next one start its blocks as soon
// as all of its own have started (they take the SMs that its first finished blocks leave) and waits, before it
// touches global memory, until the launch before it has completed and its results are visible. (The work tables are the
// exception: no kernel writes them, and their copy to the device is ordered before the call's first launch, so the
// producer of a thread block fetches its first work item before it waits. The other roles wait first thing, so that
// the limit of their bounded waits does not run while the launch before is still at work.) What is hidden
// that way is the launch itself, the barriers' and tensor memory's set-up and the wait for the last block: a step of
// four sequences of 7 to 300 tokens 42 -> 35 us, of 1024 tokens in short ones 49 -> 42 us, the ten launches around the
// attention of a 4096-token MLA block 813 -> 794 us. Kernels of other libraries before or after are ordered
// as usual.
// The elementwise steps of the MLA block and the Ulysses permutation let the next launch start at their end only. Their grids
// are a few blocks per SM, of which many fit: started at once, a grid fills the SMs that come free first and leaves the
// others empty. Rotary embedding, key / value assembly and its backward of 800 tokens, 63 heads of 126 + 62 / 126 (the
// four-byte kernels) 101 us started at once, 78 plainly, 72 at the end; 1200 tokens, 128 heads 214, 182, 177.
#ifdef __CUDACC__
__device__ __forceinline__ void overlap_next_launch() { cudaTriggerProgrammaticLaunchCompletion(); }
__device__ __forceinline__ void wait_for_previous_launch() { cudaGridDependencySynchronize(); }
// (cluster: CTAs per cluster of a kernel that does not state it itself; 1 for all others)
template <class... Params, class... Args>
cudaError_t launch_overlapped_clusters(void (*kernel)(Params...), int cluster, int grid, int block, size_t smem_bytes,
                                       cudaStream_t stream, Args&&... args)
{
    cudaLaunchAttribute attr[2] = {};
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = static_cast<unsigned>(cluster);
    attr[1].val.clusterDim.y = attr[1].val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(static_cast<unsigned>(grid));
    cfg.blockDim = dim3(static_cast<unsigned>(block));
    cfg.dynamicSmemBytes = smem_bytes;
    cfg.stream = stream;
    cfg.attrs = attr;
    cfg.numAttrs = cluster > 1 ? 2 : 1;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<Params>(args)...);
}
template <class... Params, class... Args>
cudaError_t launch_overlapped(void (*kernel)(Params...), int grid, int block, size_t smem_bytes, cudaStream_t stream,
                              Args&&... args)
{
    return launch_overlapped_clusters(kernel, 1, grid, block, smem_bytes, stream, static_cast<Args&&>(args)...);
}
// A grid of small blocks behind a kernel that fills the GPU: its blocks start as that kernel's leave, as many as fit on each
// SM that comes free first, and a grid of two or three blocks per SM ends up on a fraction of the SMs. Dynamic shared
// memory that the kernel does not use keeps it to as many blocks per SM as an even spread has. A 1024-token step of 8 heads,
// where D = rowsum(dO O) is such a grid, takes 49.6 us with it and 51.4 without. From four blocks per SM on there is
// nothing to keep apart (the kernels' registers admit four to eight): spreading up to eight per SM changed no time,
// spreading a single block per SM only gave the gain back.
template <auto kKernel, class... Args>
cudaError_t launch_overlapped_spread(int grid, int block, cudaStream_t stream, Args&&... args)
{
    constexpr int kSms = 148, kSmemPerSm = 227 * 1024, kMostPerSm = 4;
    static OncePerDevice opt_in;
    size_t smem = 0;
    const int per_sm = (grid + kSms - 1) / kSms;
    if (per_sm < kMostPerSm) {
        int dev = 0;
        cudaError_t e = cudaGetDevice(&dev);
        if (e != cudaSuccess) return e;
        if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
        smem = static_cast<size_t>(kSmemPerSm / (per_sm + 1) / 1024 + 1) * 1024;
        e = opt_in(dev, [] {
            return cudaFuncSetAttribute(kKernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemPerSm / 2 / 1024 * 1024 + 1024);
        });
        if (e != cudaSuccess) return e;
    }
    return launch_overlapped(kKernel, grid, block, smem, stream, static_cast<Args&&>(args)...);
}

// The opt-in of a kernel to more than 48 KB of dynamic shared memory, once per device ordinal.
template <class Kernel>
cudaError_t allow_dynamic_smem(Kernel kernel, size_t smem_bytes, OncePerDevice& done)
{
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
    return done(dev, [&] {
        return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem_bytes));
    });
}
#endif

struct FwdParams {
    const PairDev* pairs;
    const FwdItem* items;
    int32_t n_items;
    const FwdShortItem* short_items;   // the pairs that go to the short-sequence kernel
    int32_t n_short;
    int32_t early_pops;         // short-sequence kernel: items of up to so many steps are popped two items ahead
    void* out; float* lse; void* o_part; float* lse_part;
    int64_t T; int64_t part_rows;
    int32_t h; int32_t causal;
    int32_t kv_group;           // query heads per KV head (1: every head has its own K, V)
    float scale_log2;           // softmax_scale * log2(e)
    StatusBlock* status;
    uint64_t wait_limit_ns;
    uint64_t debug_stall_ns;    // test hook (hydra_debug_stall): 0 in normal operation
};

struct BwdParams {
    const PairDev* pairs;
    const int32_t* lists;       // pair indices, grouped by chunk
    const GroupItem* items;
    int32_t n_items;
    const float* lse; const float* dsum;   // [h, T]
    void* dq; void* dk; void* dv;   // bf16 [T,h,d], written; or, with accumulate, fp32 [T,h,d], added to
    int64_t T;
    int32_t h; int32_t causal;
    int32_t kv_group;           // query heads per KV head; k, v, dk, dv have h / kv_group heads
    int32_t item_heads;         // key-side kernel: consecutive query heads (of one KV head) that an item visits
    float scale; float scale_log2;
    int32_t accumulate;
    void* ds;                   // dS hand-off buffer, or null: the query-side kernel recomputes S and dP
    int64_t ds_head_blocks;     // blocks per head
    StatusBlock* status;
    uint64_t wait_limit_ns;
    uint64_t debug_stall_ns;    // test hook (hydra_debug_stall): 0 in normal operation
};

struct MergeParams {
    const MergeGroup* groups;
    const int32_t* lists;       // part_row of every partial, grouped by chunk
    const MergeItem* items;
    int32_t n_items;
    const void* o_part; const float* lse_part;
    void* out; float* lse;
    int64_t T; int64_t part_rows;
    int32_t h;
    int32_t accumulate;         // 1: the current (out, lse) rows are one more input of their merge
    int32_t max_parts;          // most partials any chunk has (chooses how many are requested together)
    int32_t split;              // thread blocks that share an item (set by launch_merge)
};

// The tensor-core kernels exist once per supported q / k head dimension (the kernel files are compiled
// twice): the unsuffixed set for d_qk = 192, the _d128 set for d_qk = 128; d_v = 128 in both.
#define HYDRA_DECLARE_KERNEL_SET(SUFFIX)                                                                              \
    size_t fwd_smem_bytes##SUFFIX();                                                                                  \
    int fwd_max_clusters##SUFFIX();                                                                                   \
    size_t bwd_dq_smem_bytes##SUFFIX();                                                                               \
    size_t bwd_dkv_smem_bytes##SUFFIX();                                                                              \
    size_t bwd_dq_ds_smem_bytes##SUFFIX();                                                                            \
    cudaError_t launch_fwd##SUFFIX(const CUtensorMap& mq, const CUtensorMap& mk, const CUtensorMap& mv,               \
                                   const FwdParams& p, int grid, cudaStream_t stream);                                \
    size_t fwd_short_smem_bytes##SUFFIX();                                                                            \
    cudaError_t launch_fwd_short##SUFFIX(const CUtensorMap& mq, const CUtensorMap& mk, const CUtensorMap& mv_sub,     \
                                         const FwdParams& p, const FwdSeg* segs, uint64_t call_tag, bool halves, int grid, \
                                         cudaStream_t stream);                                                        \
    cudaError_t launch_bwd_dq##SUFFIX(const CUtensorMap& mq, const CUtensorMap& mk, const CUtensorMap& mv,            \
                                      const CUtensorMap& mdo, const BwdParams& p, int grid, cudaStream_t stream);     \
    cudaError_t launch_bwd_dq_from_ds##SUFFIX(const CUtensorMap& mk, const BwdParams& p, int grid,                    \
                                              cudaStream_t stream);                                                   \
    cudaError_t launch_bwd_dkv##SUFFIX(const CUtensorMap& mq_sub, const CUtensorMap& mk, const CUtensorMap& mv,       \
                                       const CUtensorMap& mdo_sub, const BwdParams& p, bool halves, int grid,             \
                                       cudaStream_t stream);
HYDRA_DECLARE_KERNEL_SET()
HYDRA_DECLARE_KERNEL_SET(_d128)
#undef HYDRA_DECLARE_KERNEL_SET
cudaError_t launch_merge(const MergeParams& p, cudaStream_t stream);
// launch_merge plus the library's launch counter and per-kernel timer (defined beside them, in api.cu)
cudaError_t launch_merge_counted(const MergeParams& p, cudaStream_t stream);
cudaError_t launch_grad_cast(const float* acc, void* grad, int64_t n, cudaStream_t stream);
// two gradients, in one launch where sizes and alignment allow it
cudaError_t launch_grad_cast2(const float* acc_a, void* grad_a, int64_t n_a, const float* acc_b, void* grad_b, int64_t n_b,
                              int* launches, cudaStream_t stream);
cudaError_t launch_ulysses(bool pack, const void* src, void* dst, int64_t n_tokens, int32_t cp_u, int64_t chunk_units,
                           cudaStream_t stream);
// the elementwise steps of a gated MLA block around the attention kernel (mla_ops.cu)
cudaError_t launch_rope(const void* x, const int32_t* positions, void* y, int64_t n_tokens, int32_t n_heads,
                        int32_t head_dim, int32_t rope_offset, int32_t rope_dim, float theta, int inverse,
                        cudaStream_t stream);
cudaError_t launch_mla_kv_assemble(const void* kv_up, const void* k_pe, const int32_t* positions, void* k, void* v,
                                   int64_t n_tokens, int32_t n_heads, int32_t nope, int32_t rope_dim, int32_t dv,
                                   float theta, cudaStream_t stream);
cudaError_t launch_mla_kv_assemble_bwd(const void* dk, const void* dv, const int32_t* positions, void* dkv_up,
                                       void* dk_pe, int64_t n_tokens, int32_t n_heads, int32_t nope, int32_t rope_dim,
                                       int32_t dvd, float theta, cudaStream_t stream);
cudaError_t launch_gate(const void* out, const void* gate, void* y, int64_t n8, cudaStream_t stream);
cudaError_t launch_gate_bwd(const void* dy, const void* out, const void* gate, void* d_out, void* d_gate, int64_t n8,
                            cudaStream_t stream);
// clears the status block (of which keep_status leaves all but the work-queue heads)
cudaError_t launch_reset(StatusBlock* status, bool keep_status, cudaStream_t stream);
// D = rowsum(dO * O); also clears the status block and `zero_bytes` (a multiple of 16) at `zero`
cudaError_t launch_bwd_prep(const void* dout, const void* out, float* dsum, int64_t T, int32_t h, StatusBlock* status,
                            void* zero, size_t zero_bytes, cudaStream_t stream);

}  // namespace hydra

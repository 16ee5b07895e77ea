// Host side of the C ABI: argument validation, chunk cutting (zigzag pairs), work-list planning
// with a small cache, tensor-map encoding and kernel launches.
#include <algorithm>
#include <atomic>
#include <chrono>
#include <cmath>
#include <cstddef>
#include <cstring>
#include <functional>
#include <map>
#include <memory>
#include <mutex>
#include <queue>
#include <tuple>
#include <vector>

#include "hydra_internal.h"

namespace hydra {
namespace {

std::atomic<int64_t> g_launches{0};
std::atomic<uint64_t> g_wait_limit_ns{2000000000ull};
std::atomic<uint64_t> g_debug_stall_ns[3];           // test hook, see hydra_debug_stall

constexpr size_t kStatusBytes = 256;

// ---------------------------------------------------------------------------------------------
// optional per-kernel timing with CUDA events on the launching stream
// ---------------------------------------------------------------------------------------------
enum KernelKind { K_FWD = 0, K_MERGE, K_PREP, K_DKV, K_DQ, K_CAST, K_ULYSSES, K_MLA, K_COUNT };
struct ProfRecord { int kind; cudaEvent_t start, stop; };
std::mutex g_prof_mutex;
bool g_prof_on = false;
std::vector<ProfRecord> g_prof_records;
std::vector<cudaEvent_t> g_prof_pool;

struct ScopedKernelTimer {
    cudaStream_t stream;
    ProfRecord rec{};
    bool active = false;
    ScopedKernelTimer(int kind, cudaStream_t s) : stream(s)
    {
        std::lock_guard<std::mutex> lock(g_prof_mutex);
        if (!g_prof_on) return;
        auto get = [&]() {
            cudaEvent_t e = nullptr;
            if (!g_prof_pool.empty()) { e = g_prof_pool.back(); g_prof_pool.pop_back(); }
            else cudaEventCreate(&e);
            return e;
        };
        rec.kind = kind; rec.start = get(); rec.stop = get();
        active = rec.start && rec.stop;
        if (active) cudaEventRecord(rec.start, stream);
    }
    ~ScopedKernelTimer()
    {
        if (!active) return;
        cudaEventRecord(rec.stop, stream);
        std::lock_guard<std::mutex> lock(g_prof_mutex);
        g_prof_records.push_back(rec);
    }
};

inline size_t align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }
inline bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

// ---------------------------------------------------------------------------------------------
// validated problem description
// ---------------------------------------------------------------------------------------------
struct Problem {
    std::vector<int32_t> cu;
    std::vector<hydra_pair_t> pairs;
    int32_t n_seqs = 0, h = 0;
    int64_t T = 0;
    int32_t dqk = D_QK;     // q / k head dimension of the call: 192 or 128 (the value dimension is 128)
    int32_t kv_group = 1;   // query heads per K / V head (the forward's routing looks at it)
    int32_t fwd_short_set = -1;     // hydra_set_fwd_short_len as it stood when a forward call began
    // Local layouts (a rank of a ring holds only its own q chunks and the visiting kv chunks): where the
    // chunks of the sequences sit in the q-side tensors (q, out, lse, dout, dq) and in the kv-side tensors
    // (k, v, dk, dv). Empty tables = the packed layout, row = cu[seq] + position, Tq = Tk = T.
    std::vector<hydra_chunk_t> qc, kc;
    int64_t Tq = 0, Tk = 0;
    static int64_t row_in(const std::vector<hydra_chunk_t>& table, int32_t seq, int32_t pos)
    {
        for (const hydra_chunk_t& c : table)
            if (c.seq == seq && pos >= c.start && pos < c.start + c.len) return int64_t{c.row} + (pos - c.start);
        return -1;
    }
    int64_t q_row(int32_t seq, int32_t pos) const { return qc.empty() ? int64_t{cu[seq]} + pos : row_in(qc, seq, pos); }
    int64_t k_row(int32_t seq, int32_t pos) const { return kc.empty() ? int64_t{cu[seq]} + pos : row_in(kc, seq, pos); }
};

int32_t make_problem(const int32_t* cu, int32_t n_seqs, int32_t h, const hydra_pair_t* pairs,
                     int32_t n_pairs, Problem& out)
{
    if (n_seqs < 0 || h < 1 || h > 65535 || (n_seqs > 0 && cu == nullptr)) return HYDRA_ERR_INVALID_ARG;
    if ((pairs == nullptr) != (n_pairs == 0) || n_pairs < 0) return HYDRA_ERR_INVALID_ARG;
    out.n_seqs = n_seqs;
    out.h = h;
    out.cu.assign(1, 0);
    if (n_seqs > 0) {
        out.cu.assign(cu, cu + n_seqs + 1);
        if (out.cu[0] != 0) return HYDRA_ERR_INVALID_ARG;
        for (int b = 0; b < n_seqs; ++b)
            if (out.cu[b + 1] < out.cu[b]) return HYDRA_ERR_INVALID_ARG;
    }
    out.T = out.cu[n_seqs];
    if (out.T > (int64_t{1} << 30)) return HYDRA_ERR_UNSUPPORTED;
    out.Tq = out.Tk = out.T;
    out.qc.clear();
    out.kc.clear();
    out.pairs.clear();
    if (pairs == nullptr) {
        for (int b = 0; b < n_seqs; ++b) {
            const int32_t len = out.cu[b + 1] - out.cu[b];
            if (len == 0) continue;
            out.pairs.push_back(hydra_pair_t{b, 0, len, 0, len, -1, b, 0});
        }
        return HYDRA_OK;
    }
    for (int i = 0; i < n_pairs; ++i) {
        const hydra_pair_t& p = pairs[i];
        if (p.seq < 0 || p.seq >= n_seqs || p.flags != 0) return HYDRA_ERR_INVALID_ARG;
        const int64_t len = out.cu[p.seq + 1] - out.cu[p.seq];
        if (p.q_start < 0 || p.q_len < 0 || int64_t{p.q_start} + p.q_len > len) return HYDRA_ERR_INVALID_ARG;
        if (p.k_start < 0 || p.k_len < 0 || int64_t{p.k_start} + p.k_len > len) return HYDRA_ERR_INVALID_ARG;
        if (p.part_row < -1) return HYDRA_ERR_INVALID_ARG;
        if (i > 0) {
            const hydra_pair_t& o = pairs[i - 1];
            if (p.group < o.group) return HYDRA_ERR_INVALID_ARG;
            if (p.group == o.group &&
                (p.seq != o.seq || p.q_start != o.q_start || p.q_len != o.q_len ||
                 (p.part_row < 0) != (o.part_row < 0)))
                return HYDRA_ERR_INVALID_ARG;
            if (p.group == o.group && p.part_row < 0) return HYDRA_ERR_INVALID_ARG;  // two direct writers
        }
        out.pairs.push_back(p);
    }
    return HYDRA_OK;
}

// The same with local layouts: every chunk lies inside its sequence and inside its tensor, chunks of one table
// do not share rows, and every pair's q range lies inside one q chunk and its kv range inside one kv chunk.
int32_t make_problem_local(const int32_t* cu, int32_t n_seqs, int32_t h, const hydra_chunk_t* q_chunks,
                           int32_t n_q_chunks, int64_t q_rows, const hydra_chunk_t* kv_chunks, int32_t n_kv_chunks,
                           int64_t kv_rows, const hydra_pair_t* pairs, int32_t n_pairs, Problem& out)
{
    if (!pairs || n_pairs < 1 || !q_chunks || n_q_chunks < 1 || !kv_chunks || n_kv_chunks < 1) return HYDRA_ERR_INVALID_ARG;
    if (q_rows < 1 || kv_rows < 1 || q_rows > (int64_t{1} << 30) || kv_rows > (int64_t{1} << 30)) return HYDRA_ERR_INVALID_ARG;
    if (int32_t s = make_problem(cu, n_seqs, h, pairs, n_pairs, out)) return s;
    auto take = [&](const hydra_chunk_t* src, int32_t n, int64_t rows, std::vector<hydra_chunk_t>& dst) {
        dst.assign(src, src + n);
        std::vector<std::pair<int64_t, int64_t>> iv;
        for (const hydra_chunk_t& c : dst) {
            if (c.seq < 0 || c.seq >= n_seqs || c.start < 0 || c.len < 0 || c.row < 0) return false;
            if (int64_t{c.start} + c.len > int64_t{out.cu[c.seq + 1]} - out.cu[c.seq]) return false;
            if (int64_t{c.row} + c.len > rows) return false;
            if (c.len > 0) iv.emplace_back(c.row, int64_t{c.row} + c.len);
        }
        std::sort(iv.begin(), iv.end());
        for (size_t i = 1; i < iv.size(); ++i)
            if (iv[i].first < iv[i - 1].second) return false;
        return true;
    };
    if (!take(q_chunks, n_q_chunks, q_rows, out.qc) || !take(kv_chunks, n_kv_chunks, kv_rows, out.kc))
        return HYDRA_ERR_INVALID_ARG;
    out.Tq = q_rows;
    out.Tk = kv_rows;
    for (const hydra_pair_t& p : out.pairs) {
        if (p.q_len > 0 && (out.q_row(p.seq, p.q_start) < 0 ||
                            out.q_row(p.seq, p.q_start + p.q_len - 1) != out.q_row(p.seq, p.q_start) + p.q_len - 1))
            return HYDRA_ERR_INVALID_ARG;
        if (p.k_len > 0 && (out.k_row(p.seq, p.k_start) < 0 ||
                            out.k_row(p.seq, p.k_start + p.k_len - 1) != out.k_row(p.seq, p.k_start) + p.k_len - 1))
            return HYDRA_ERR_INVALID_ARG;
    }
    return HYDRA_OK;
}

// The backward sums over pairs, so a sequence whose pairs cover its causal triangle, every visible position once, is the same
// problem uncut: one pair, whose tiles are whole where every chunk's last tile is ragged, whose items are longer and whose
// tables are shorter. (For every q chunk the kv chunks follow one another from the sequence's start to the chunk's end at
// least: what lies beyond is masked.) True if pairs were joined. Step in passes one after another, pair by pair / joined: 12
// sequences of 121 tokens, 16 heads, ring of 2, 100 / 64 us; 1728 tokens, 32 heads, ring of 2, 146 / 113; 26283 log-normal
// tokens, 16 heads, ring of 4, 2510 / 2071; 65536 tokens of 64 to 512, 32 heads, cut in two, 3213 / 3012.
bool join_chunks(Problem& pb, int32_t causal)
{
    if (!causal || !pb.qc.empty() || !pb.kc.empty()) return false;
    bool cut = false;
    for (const auto& p : pb.pairs) {
        const int32_t len = pb.cu[p.seq + 1] - pb.cu[p.seq];
        cut = cut || (p.q_len > 0 && p.k_len > 0 && (p.q_len != len || p.k_len != len));
    }
    if (!cut) return false;
    std::vector<hydra_pair_t> by_q;
    by_q.reserve(pb.pairs.size());
    for (const auto& p : pb.pairs)
        if (p.q_len > 0 && p.k_len > 0) by_q.push_back(p);
    auto less = [](const hydra_pair_t& a, const hydra_pair_t& b) {
        if (a.seq != b.seq) return a.seq < b.seq;
        return a.q_start != b.q_start ? a.q_start < b.q_start : a.k_start < b.k_start;
    };
    if (!std::is_sorted(by_q.begin(), by_q.end(), less)) std::sort(by_q.begin(), by_q.end(), less);     // (in every call)
    std::vector<hydra_pair_t> joined;
    bool any = false;
    for (size_t i = 0, j = 0; i < by_q.size(); i = j) {
        const int32_t seq = by_q[i].seq, len = pb.cu[seq + 1] - pb.cu[seq];
        while (j < by_q.size() && by_q[j].seq == seq) ++j;
        bool whole = true;
        int32_t q_end = 0;
        for (size_t t = i; t < j && whole;) {
            const int32_t q_start = by_q[t].q_start, q_len = by_q[t].q_len;
            int32_t k_end = 0;
            whole = q_start == q_end;
            for (; t < j && by_q[t].q_start == q_start; ++t) {
                whole = whole && by_q[t].q_len == q_len && by_q[t].k_start == k_end;
                k_end = by_q[t].k_start + by_q[t].k_len;
            }
            q_end = q_start + q_len;
            whole = whole && k_end >= q_end;
        }
        if (whole && q_end == len) {
            any = any || j - i > 1;
            joined.push_back(hydra_pair_t{seq, 0, len, 0, len, -1, static_cast<int32_t>(joined.size()), 0});
            continue;
        }
        for (size_t t = i; t < j; ++t) {
            joined.push_back(by_q[t]);
            joined.back().part_row = -1;
            joined.back().group = static_cast<int32_t>(joined.size()) - 1;
        }
    }
    if (any) pb.pairs.swap(joined);
    return any;
}

// partial rows must lie inside the buffers and must not overlap
int32_t check_part_rows(const Problem& pb, int64_t part_rows)
{
    std::vector<std::pair<int64_t, int64_t>> iv;
    for (const auto& p : pb.pairs)
        if (p.part_row >= 0 && p.q_len > 0) {
            if (int64_t{p.part_row} + p.q_len > part_rows) return HYDRA_ERR_INVALID_ARG;
            iv.emplace_back(p.part_row, int64_t{p.part_row} + p.q_len);
        }
    std::sort(iv.begin(), iv.end());
    for (size_t i = 1; i < iv.size(); ++i)
        if (iv[i].first < iv[i - 1].second) return HYDRA_ERR_INVALID_ARG;
    return HYDRA_OK;
}

// ranges of one kind (q or kv) inside one sequence must be identical or disjoint
struct Range { int32_t seq, start, len; };
inline bool range_less(const Range& a, const Range& b)
{
    if (a.seq != b.seq) return a.seq < b.seq;
    if (a.start != b.start) return a.start < b.start;
    return a.len < b.len;
}
int32_t check_identical_or_disjoint(std::vector<Range> r)
{
    std::sort(r.begin(), r.end(), range_less);
    for (size_t i = 1; i < r.size(); ++i) {
        const Range &a = r[i - 1], &b = r[i];
        if (a.seq != b.seq) continue;
        if (a.start == b.start && a.len == b.len) continue;
        if (b.start < a.start + a.len) return HYDRA_ERR_INVALID_ARG;
    }
    return HYDRA_OK;
}

// ---------------------------------------------------------------------------------------------
// plans: work lists built on the host, cached by content, resident on the device in a fixed arena
// ---------------------------------------------------------------------------------------------
// A training loop meets a new cu_seqlens with every micro-batch, so a new problem must cost neither a device
// allocation nor a device-wide stall. The tables of a plan are built on the host (and cached by content:
// every layer of a micro-batch asks for the same ones), staged in pinned host memory and copied with
// cudaMemcpyAsync, on the caller's stream, into an arena that the library allocates ONCE per device (the
// first call on that device). The arena is used as two halves: tables are appended to the active half; when
// it is full the other half becomes active, the plans that lived there stop being resident (they are
// uploaded again when they are next used) and the uploading stream first waits, on the device, for the
// kernels that last read that half (an event per stream that used it). No cudaMalloc, no cudaFree and no
// host-side wait happens after the first call on a device, whatever the number of distinct problems. The
// one exception: a plan larger than half the arena gets an allocation of its own (and is cached).
struct DeviceBlob {
    void* ptr = nullptr;
    ~DeviceBlob() { if (ptr) cudaFree(ptr); }
    cudaError_t upload(const std::vector<uint8_t>& bytes)
    {
        cudaError_t e = cudaMalloc(&ptr, std::max<size_t>(bytes.size(), 16));
        if (e != cudaSuccess) { ptr = nullptr; return e; }
        if (!bytes.empty()) e = cudaMemcpy(ptr, bytes.data(), bytes.size(), cudaMemcpyHostToDevice);
        return e;
    }
};

template <class T>
size_t append(std::vector<uint8_t>& blob, const std::vector<T>& v)
{
    const size_t off = align_up(blob.size(), 16);
    blob.resize(off + v.size() * sizeof(T));
    if (!v.empty()) std::memcpy(blob.data() + off, v.data(), v.size() * sizeof(T));
    return off;
}

struct Plan {
    std::vector<uint8_t> key;
    int kind = 0, device = 0;
    std::vector<uint8_t> blob;       // the tables, as they go to the device
    size_t off_pairs = 0, off_items = 0, off_lists = 0, off_groups = 0, off_items2 = 0, off_lists2 = 0;
    int32_t n_items = 0, n_items2 = 0;
    int32_t halves = 0;              // forward: the short kernel's items are dealt out, longer tiles as a part per slot;
                                     // backward: two CTAs share every key-side item
    int32_t early_pops = 0;          // forward: FwdParams::early_pops
    int32_t short_grid = 0;          // forward, halves: thread blocks the items have been dealt out to
    size_t off_segs = 0;             // forward: FwdSeg table of the short-sequence kernel's items
    size_t n_segs = 0;
    int32_t item_heads = 1;          // backward: query heads per key-side item (BwdParams::item_heads)
    int64_t ds_head_blocks = 0;      // backward: blocks of the dS hand-off buffer per head; -1: not usable
    // residency on the device (guarded by g_plan_mutex)
    int half = -1;                   // arena half the tables were last copied to
    uint64_t epoch = 0;              // generation of that half at the time: resident iff it still is the half's
    size_t dev_off = 0;
    cudaStream_t up_stream = nullptr;    // stream that carried the copy, and its completion
    cudaEvent_t uploaded = nullptr;
    DeviceBlob own;                  // a plan too large for the arena owns its device copy
    ~Plan() { if (uploaded) cudaEventDestroy(uploaded); }
};

std::mutex g_plan_mutex;
std::vector<std::shared_ptr<Plan>> g_plans;
constexpr size_t kMaxPlans = 256;

struct PlanArena {
    uint8_t* base = nullptr;
    size_t half_bytes = 0;
    int active = 0;
    size_t used = 0;
    uint64_t epoch[2] = {0, 0};
    uint64_t next_epoch = 1;
    // kernels that read tables of a half: one event per stream, re-recorded at every use
    std::vector<std::pair<cudaStream_t, cudaEvent_t>> users[2];
    std::vector<cudaEvent_t> spare_events;
    // "the previous readers of this half are done", recorded on the stream that switched to it; uploads on
    // other streams wait for it
    cudaEvent_t freed[2] = {nullptr, nullptr};
    cudaStream_t freed_on[2] = {nullptr, nullptr};
    // pinned staging: a slot is reused once the copy that read it has completed. The slots are slices of one
    // pinned allocation made with the arena (page-locking memory takes a fraction of a millisecond, too long
    // for the first call of a new shape); tables larger than a slice get a pinned buffer of their own.
    struct Slot { uint8_t* host = nullptr; size_t cap = 0; cudaEvent_t done = nullptr; bool used = false; bool own = false; };
    static constexpr int kSlots = 8;
    static constexpr size_t kSlotBytes = size_t{2} << 20;
    uint8_t* stage_base = nullptr;
    Slot slots[kSlots];
    int next_slot = 0;
};
PlanArena g_arena[64];
std::atomic<uint64_t> g_arena_bytes{uint64_t{32} << 20};

void arena_release(PlanArena& a)                         // device idle, g_plan_mutex held
{
    if (a.base) cudaFree(a.base);
    a.base = nullptr; a.half_bytes = 0; a.used = 0; a.active = 0;
    for (int h = 0; h < 2; ++h) {
        for (auto& u : a.users[h]) cudaEventDestroy(u.second);
        a.users[h].clear();
        if (a.freed[h]) cudaEventDestroy(a.freed[h]);
        a.freed[h] = nullptr; a.freed_on[h] = nullptr;
        a.epoch[h] = a.next_epoch++;                     // nothing is resident any more
    }
    for (cudaEvent_t e : a.spare_events) cudaEventDestroy(e);
    a.spare_events.clear();
    for (auto& sl : a.slots) {
        if (sl.host && sl.own) cudaFreeHost(sl.host);
        if (sl.done) cudaEventDestroy(sl.done);
        sl = PlanArena::Slot{};
    }
    if (a.stage_base) cudaFreeHost(a.stage_base);
    a.stage_base = nullptr;
}

// Makes the tables of `plan` resident on the current device and returns their address. g_plan_mutex held.
int32_t arena_place(Plan& plan, int device, cudaStream_t stream, const uint8_t** tables)
{
    if (plan.own.ptr) { *tables = static_cast<const uint8_t*>(plan.own.ptr); return HYDRA_OK; }
    PlanArena& a = g_arena[device];
    if (!a.base) {                                       // first call on this device: the one allocation
        const size_t half = align_up(std::max<uint64_t>(g_arena_bytes.load() / 2, 4096), 256);
        void* ptr = nullptr;
        if (cudaMalloc(&ptr, 2 * half) != cudaSuccess) return HYDRA_ERR_CUDA;
        a.base = static_cast<uint8_t*>(ptr);
        a.half_bytes = half;
        a.epoch[0] = a.next_epoch++;
        a.epoch[1] = a.next_epoch++;
        void* hp = nullptr;
        if (cudaHostAlloc(&hp, PlanArena::kSlots * PlanArena::kSlotBytes, cudaHostAllocDefault) != cudaSuccess)
            return HYDRA_ERR_CUDA;
        a.stage_base = static_cast<uint8_t*>(hp);
        for (int i = 0; i < PlanArena::kSlots; ++i) {
            a.slots[i].host = a.stage_base + i * PlanArena::kSlotBytes;
            a.slots[i].cap = PlanArena::kSlotBytes;
            if (cudaEventCreateWithFlags(&a.slots[i].done, cudaEventDisableTiming) != cudaSuccess) return HYDRA_ERR_CUDA;
        }
    }
    if (plan.half >= 0 && plan.epoch == a.epoch[plan.half]) {
        // resident; a stream other than the one that carried the copy waits for the copy (free once complete)
        if (stream != plan.up_stream && cudaStreamWaitEvent(stream, plan.uploaded, 0) != cudaSuccess) return HYDRA_ERR_CUDA;
        *tables = a.base + plan.half * a.half_bytes + plan.dev_off;
        return HYDRA_OK;
    }
    const size_t need = align_up(std::max<size_t>(plan.blob.size(), 16), 256);
    if (need > a.half_bytes) {                           // documented exception: its own allocation, once
        if (plan.own.upload(plan.blob) != cudaSuccess) return HYDRA_ERR_CUDA;
        *tables = static_cast<const uint8_t*>(plan.own.ptr);
        return HYDRA_OK;
    }
    if (a.used + need > a.half_bytes) {
        // switch halves: what lived in the other half is no longer resident, and this stream waits (on the
        // device) for the kernels that last read it before anything is copied over their tables
        a.active ^= 1;
        a.used = 0;
        a.epoch[a.active] = a.next_epoch++;
        for (auto& u : a.users[a.active]) {
            if (cudaStreamWaitEvent(stream, u.second, 0) != cudaSuccess) return HYDRA_ERR_CUDA;
            a.spare_events.push_back(u.second);
        }
        a.users[a.active].clear();
        if (!a.freed[a.active] && cudaEventCreateWithFlags(&a.freed[a.active], cudaEventDisableTiming) != cudaSuccess)
            return HYDRA_ERR_CUDA;
        if (cudaEventRecord(a.freed[a.active], stream) != cudaSuccess) return HYDRA_ERR_CUDA;
        a.freed_on[a.active] = stream;
    }
    const int half = a.active;
    if (a.freed[half] && a.freed_on[half] != stream && cudaStreamWaitEvent(stream, a.freed[half], 0) != cudaSuccess)
        return HYDRA_ERR_CUDA;
    // staging slot: pinned, reused once the copy that read it has completed (eight uploads ago, so the host
    // may run two micro-batches ahead of the device before this ever waits)
    PlanArena::Slot& sl = a.slots[a.next_slot];
    a.next_slot = (a.next_slot + 1) % PlanArena::kSlots;
    if (sl.used && cudaEventSynchronize(sl.done) != cudaSuccess) return HYDRA_ERR_CUDA;
    if (sl.cap < need) {                                 // rare: tables of more than 2 MB
        if (sl.host && sl.own) cudaFreeHost(sl.host);
        sl.host = nullptr; sl.cap = 0; sl.own = false;
        void* hp = nullptr;
        if (cudaHostAlloc(&hp, need, cudaHostAllocDefault) != cudaSuccess) return HYDRA_ERR_CUDA;
        sl.host = static_cast<uint8_t*>(hp);
        sl.cap = need;
        sl.own = true;
    }
    if (!sl.done && cudaEventCreateWithFlags(&sl.done, cudaEventDisableTiming) != cudaSuccess) return HYDRA_ERR_CUDA;
    if (!plan.uploaded && cudaEventCreateWithFlags(&plan.uploaded, cudaEventDisableTiming) != cudaSuccess)
        return HYDRA_ERR_CUDA;
    if (!plan.blob.empty()) std::memcpy(sl.host, plan.blob.data(), plan.blob.size());
    uint8_t* dst = a.base + half * a.half_bytes + a.used;
    if (!plan.blob.empty() &&
        cudaMemcpyAsync(dst, sl.host, plan.blob.size(), cudaMemcpyHostToDevice, stream) != cudaSuccess)
        return HYDRA_ERR_CUDA;
    if (cudaEventRecord(sl.done, stream) != cudaSuccess || cudaEventRecord(plan.uploaded, stream) != cudaSuccess)
        return HYDRA_ERR_CUDA;
    sl.used = true;
    plan.half = half;
    plan.epoch = a.epoch[half];
    plan.dev_off = a.used;
    plan.up_stream = stream;
    a.used += need;
    *tables = dst;
    return HYDRA_OK;
}

// After the launches that read the tables of `plan`: remember that `stream` has to be waited for before the
// plan's half of the arena is overwritten. g_plan_mutex held.
void arena_note_use(const Plan& plan, int device, cudaStream_t stream)
{
    if (plan.own.ptr || plan.half < 0) return;
    PlanArena& a = g_arena[device];
    if (plan.epoch != a.epoch[plan.half]) return;
    auto& users = a.users[plan.half];
    for (auto& u : users)
        if (u.first == stream) { cudaEventRecord(u.second, stream); return; }
    cudaEvent_t e = nullptr;
    if (!a.spare_events.empty()) { e = a.spare_events.back(); a.spare_events.pop_back(); }
    else if (cudaEventCreateWithFlags(&e, cudaEventDisableTiming) != cudaSuccess) return;
    cudaEventRecord(e, stream);
    users.emplace_back(stream, e);
}

// Pairs whose q range and kv range are both at most this long go to the short-sequence forward kernel
// (0: none do; negative: chosen by the library from the head layout). See build_fwd.
std::atomic<int32_t> g_fwd_short_len{-1};
// Where the two forward kernels take equal time. In calls of fewer than 20 q tiles per SM (16384 tokens of 16 heads have 15),
// where the tail counts, at 1280 tokens with a K / V head per query head at d_qk = 192 and 2048 with shared K / V heads or at
// d_qk = 128 (where a slot of the short-sequence kernel has room for a second V stage): CTA pairs / short-sequence kernel, 16384
// tokens, 8 heads, sequences of 1281 to 1920 tokens 0.97-1.03, of 2047 and more 0.93-1.00. In larger calls, which have
// sequences of many lengths cut into 256-row tiles to fill the CTA pairs with, at 1920 and 3328: 65536 tokens, 32 heads of 192,
// 1281 tokens 1.08, 1600 1.20, 1920 1.13, 2047 1.00; with shared K / V heads 1281 1.27, 2047 1.05, 2900 1.07, 3200
// 1.03, 3584 0.98; heads of 128 1281 1.28, 2600 1.09, 3200 1.05, 3584 0.99. (Large calls of whole causal sequences, that
// is. Chunk pairs off the diagonal keep CTA pairs busy without a mask: eleven sequences of 5685 tokens, 4 heads, cut in
// chunks of 1421 445 us on CTA pairs, 495 on the other kernel, four of 12000, 16 heads, chunks of 1500 2810 and 3150.)
constexpr int32_t kManyTilesPerSm = 20;
int plan_workers(int per_worker_sms);
bool many_q_tiles(const Problem& pb, int causal)
{
    int64_t n = 0;
    bool diagonal = causal != 0;
    for (const auto& p : pb.pairs) {
        n += (p.q_len + TILE - 1) / TILE;
        diagonal = diagonal && p.q_start == p.k_start;
    }
    return diagonal && n * pb.h >= int64_t{kManyTilesPerSm} * plan_workers(1);
}
int32_t fwd_short_len_for(const Problem& pb, int causal)
{
    if (pb.fwd_short_set >= 0) return pb.fwd_short_set;
    const bool per_head = pb.dqk == D_QK && pb.kv_group == 1;
    return many_q_tiles(pb, causal) ? (per_head ? 1920 : 3328) : (per_head ? 1280 : 2048);
}
static_assert(FWD_SHORT_KEYS == SUB, "the short forward kernel reads K through the 64-row map of the CTA-pair kernel");

std::vector<uint8_t> make_key(int kind, int device, const Problem& pb, int causal)
{
    std::vector<uint8_t> key;
    auto put = [&](const void* p, size_t n) {
        const uint8_t* b = static_cast<const uint8_t*>(p);
        key.insert(key.end(), b, b + n);
    };
    // the forward's tables depend on which pairs go to the short-sequence kernel: on the limit, and on who chose it
    const bool fwd = kind == HYDRA_WS_FWD;
    const int32_t head[8] = {kind, device, pb.h, causal, pb.n_seqs, fwd ? fwd_short_len_for(pb, causal) : 0,
                             fwd && pb.fwd_short_set < 0, kind == HYDRA_WS_BWD ? pb.kv_group : 0};
    put(head, sizeof head);
    put(pb.cu.data(), pb.cu.size() * sizeof(int32_t));
    put(pb.pairs.data(), pb.pairs.size() * sizeof(hydra_pair_t));
    if (!pb.qc.empty() || !pb.kc.empty()) {
        const int64_t dims[4] = {pb.Tq, pb.Tk, static_cast<int64_t>(pb.qc.size()), static_cast<int64_t>(pb.kc.size())};
        put(dims, sizeof dims);
        put(pb.qc.data(), pb.qc.size() * sizeof(hydra_chunk_t));
        put(pb.kc.data(), pb.kc.size() * sizeof(hydra_chunk_t));
    }
    return key;
}

std::vector<PairDev> device_pairs(const Problem& pb)
{
    std::vector<PairDev> v;
    v.reserve(pb.pairs.size());
    for (const auto& p : pb.pairs) {
        PairDev d;
        d.q_tok0 = p.q_len > 0 ? static_cast<int32_t>(pb.q_row(p.seq, p.q_start)) : 0;
        d.q_len = p.q_len;
        d.k_tok0 = p.k_len > 0 ? static_cast<int32_t>(pb.k_row(p.seq, p.k_start)) : 0;
        d.k_len = p.k_len;
        d.off = p.q_start - p.k_start;
        d.to_part = p.part_row >= 0;
        d.out_row0 = d.to_part ? p.part_row : d.q_tok0;
        d.ds_base = 0;
        v.push_back(d);
    }
    return v;
}

// kv tiles that the q rows [q0, q0 + rows) of a pair visit (0: they see no key)
inline int32_t kv_tiles(const hydra_pair_t& p, int32_t q0, int causal, int32_t rows = TILE)
{
    const int32_t last_row = std::min(q0 + rows, p.q_len) - 1;
    int64_t n_keys = p.k_len;
    if (causal) n_keys = std::min<int64_t>(n_keys, int64_t{last_row} + (p.q_start - p.k_start) + 1);
    return n_keys > 0 ? static_cast<int32_t>((n_keys + TILE - 1) / TILE) : 0;
}

// Order: blocks of items that share their operands (same pair/chunk and head) stay together so
// that CTAs running at the same time hit the same K/V (or Q/dO) tiles in L2; blocks go
// longest-first, and inside a block items go longest-first too (the quadratic load model of
// Sections 3.2 / 5.1: cost ~ number of inner tiles). The persistent CTAs pop items from a counter in
// this order at run time, so a CTA that finishes early takes more items and nothing has to predict
// how long an item runs.
//
// The end of the list can be different: in block order the last block's longest item starts when the
// queue is nearly empty and runs on alone (few long sequences of equal length: the slowest CTA ended 10 %
// after the even share). If a simulation of the queue shows that, the cheapest items, up to one longest
// item's worth per worker (CTA or cluster), are taken out of their blocks and go last, longest-first
// across blocks: whatever starts late is short.
struct Keyed { int64_t block_cost; int32_t block; int32_t cost; int32_t idx; };
constexpr int32_t kItemOverhead = 5;    // what an item costs beyond its tiles, in tile steps (measured: 2-6 us)
int32_t device_info(int* sms);
int plan_workers(int per_worker_sms)
{
    int sms = 0;
    if (device_info(&sms) != HYDRA_OK || sms <= 0) sms = 148;
    return std::max(1, sms / per_worker_sms);
}
template <class Item>
void order_items(std::vector<Item>& items, const std::vector<int32_t>& block_of, const std::vector<int32_t>& cost,
                 int workers)
{
    const size_t n = items.size();
    int32_t n_blocks = 0;
    for (int32_t b : block_of) n_blocks = std::max(n_blocks, b + 1);
    std::vector<int64_t> block_cost(n_blocks, 0);
    for (size_t i = 0; i < n; ++i) block_cost[block_of[i]] += cost[i];
    // the block order, sorted once; a trial order is this one with its tail items taken out and appended
    std::vector<Keyed> base(n);
    for (size_t i = 0; i < n; ++i)
        base[i] = Keyed{block_cost[block_of[i]], block_of[i], cost[i], static_cast<int32_t>(i)};
    std::sort(base.begin(), base.end(), [](const Keyed& a, const Keyed& b) {
        if (a.block_cost != b.block_cost) return a.block_cost > b.block_cost;
        if (a.block != b.block) return a.block < b.block;
        if (a.cost != b.cost) return a.cost > b.cost;
        return a.idx < b.idx;
    });
    // ascending by cost: the candidates for the tail (sorted only if a tail is tried at all)
    std::vector<int32_t> asc;
    int32_t longest = 0;
    int64_t total = 0;
    for (int32_t c : cost) { longest = std::max(longest, c); total += c + kItemOverhead; }
    // the order with a tail worth `want` units of work
    std::vector<uint8_t> in_tail(n);
    auto ordered = [&](int64_t want) {
        if (asc.empty()) {
            asc.resize(n);
            for (size_t i = 0; i < n; ++i) asc[i] = static_cast<int32_t>(i);
            std::sort(asc.begin(), asc.end(), [&](int32_t a, int32_t b) {
                return cost[a] != cost[b] ? cost[a] < cost[b] : a > b;
            });
        }
        std::fill(in_tail.begin(), in_tail.end(), 0);
        std::vector<Keyed> tail;
        int64_t have = 0;
        for (int32_t i : asc) {
            if (have >= want) break;
            in_tail[i] = 1;
            have += cost[i] + kItemOverhead;
            tail.push_back(Keyed{block_cost[block_of[i]], block_of[i], cost[i], i});
        }
        std::sort(tail.begin(), tail.end(), [](const Keyed& a, const Keyed& b) {
            if (a.cost != b.cost) return a.cost > b.cost;
            if (a.block != b.block) return a.block < b.block;
            return a.idx < b.idx;
        });
        std::vector<Keyed> o;
        o.reserve(n);
        for (const Keyed& e : base)
            if (!in_tail[e.idx]) o.push_back(e);
        o.insert(o.end(), tail.begin(), tail.end());
        return o;
    };
    // When the last worker ends if the workers pop the items in this order (time = cost + a fixed part). Times
    // are small integers and an item always starts at the earliest free time, which never decreases, so the
    // workers' free times live in a calendar (count of workers per time value) with a cursor that only moves
    // forward: O(items + end time), a few nanoseconds per item (a heap cost 1 ms for the 8000 items of the
    // 32K workload's backward, as long as the kernels of the step). List scheduling ends within one longest
    // item of the even share, which bounds the calendar.
    const int64_t even = (total + workers - 1) / workers;
    std::vector<int32_t> calendar(static_cast<size_t>(even + longest + kItemOverhead + 2));
    auto makespan = [&](const std::vector<Keyed>& o) {
        std::fill(calendar.begin(), calendar.end(), 0);
        calendar[0] = workers;
        size_t now = 0;
        int64_t end = 0;
        for (const Keyed& e : o) {
            while (calendar[now] == 0) ++now;
            --calendar[now];
            const size_t t = now + static_cast<size_t>(e.cost + kItemOverhead);
            ++calendar[t];
            end = std::max<int64_t>(end, static_cast<int64_t>(t));
        }
        return end;
    };
    // Taking items out of their blocks costs locality (measured: -5 % on workloads of many short sequences
    // when a tail was always cut), so the smallest tail that brings the simulated end within 5 % of the
    // even share is taken, and none if the block order already gets there.
    const int64_t full_tail = static_cast<int64_t>(workers) * (longest + kItemOverhead);
    std::vector<Keyed> k = base;
    int64_t best = makespan(k);
    for (int step = 1; step <= 4 && best * 100 > even * 105; ++step) {
        std::vector<Keyed> o = ordered(full_tail * step / 4);
        const int64_t m = makespan(o);
        if (m < best) { best = m; k.swap(o); }
    }
    std::vector<Item> sorted(n);
    for (size_t i = 0; i < n; ++i) sorted[i] = items[k[i].idx];
    items.swap(sorted);
}

// The items of a plan come in groups (a sequence: all of its pairs or chunks) that repeat for every head with the same costs,
// so the block order above (blocks = (group, head), longest block first, the items of a block longest first)
// needs only the GROUPS sorted, and the list is then written out in one pass. That matters because a
// training loop meets new cu_seqlens with every micro-batch: sorting the 22 000 items of the many-short
// workload took milliseconds on the host, as long as the kernels they feed. List scheduling ends within one
// longest item of the even share, so when the longest item is under 5 % of that share the block order needs
// no check; only otherwise (few, long, equal sequences: few items) is the queue simulated as above.
// A group is a whole sequence because its pairs share Q, K, V and dO, which items that run at the same time find in L2. With
// a group per pair or chunk, which run far apart, sequences of 64 to 512 tokens cut in two (32768 tokens, 32 heads) read 1.67
// GB in the forward, 2.08 on the key side and 1.58 on the query side, as whole sequences 1.19, 1.52 and 1.29 (step of 65536
// tokens 3391 -> 3213 us). 32768 log-normal tokens, 16 heads, ring of 4, 3140 -> 2975 us; five sequences of 13107, 8 heads,
// ring of 4, 8912 -> 8640; one of 65536 39444 -> 38900; heads of 128, 31598 tokens, 32 heads, ring of 2, 4207 -> 4030.
struct GroupEntry { int32_t a, b, c, cost, of; };        // of: the pair or chunk
// The groups longest first (their entries longest first inside), the number of items, and whether the block
// order needs no check against the queue simulation.
struct GroupOrder { std::vector<int32_t> order; int64_t n_items = 0; bool settled = true; };
GroupOrder order_groups(std::vector<std::vector<GroupEntry>>& groups, int32_t h, int workers)
{
    GroupOrder go;
    std::vector<int64_t> group_cost(groups.size(), 0);
    int64_t total = 0;
    int32_t longest = 0;
    for (size_t g = 0; g < groups.size(); ++g) {
        std::stable_sort(groups[g].begin(), groups[g].end(),
                         [](const GroupEntry& x, const GroupEntry& y) { return x.cost > y.cost; });
        for (const GroupEntry& e : groups[g]) {
            group_cost[g] += e.cost;
            total += static_cast<int64_t>(e.cost + kItemOverhead) * h;
            longest = std::max(longest, e.cost);
        }
        go.n_items += static_cast<int64_t>(groups[g].size()) * h;
    }
    go.order.resize(groups.size());
    for (size_t g = 0; g < groups.size(); ++g) go.order[g] = static_cast<int32_t>(g);
    std::sort(go.order.begin(), go.order.end(), [&](int32_t x, int32_t y) {
        return group_cost[x] != group_cost[y] ? group_cost[x] > group_cost[y] : x < y;
    });
    const int64_t even = (total + workers - 1) / workers;
    go.settled = static_cast<int64_t>(longest + kItemOverhead) * 20 <= even;
    if (go.settled) {
        // No item is long: only the end of the list needs the longest-first order (a longest item's worth per worker). Before it
        // the groups run as they lie in memory: a ragged tile's loads take rows of the next sequence along, which are then
        // used while they are in L2. 32768 tokens of 64 to 512, 32 heads, read from memory, longest first / as they lie:
        // forward 1.22 / 1.11 GB, key side 1.55 / 1.38, query side 1.12 / 1.06 (1.03 at least); step of 65536 2707 / 2660 us.
        int64_t left = static_cast<int64_t>(workers) * (longest + kItemOverhead);
        size_t tail = groups.size();
        while (tail > 0 && left > 0) {
            const int32_t g = go.order[--tail];
            left -= (group_cost[g] + static_cast<int64_t>(groups[g].size()) * kItemOverhead) * h;
        }
        std::vector<uint8_t> early(groups.size(), 0);
        for (size_t i = 0; i < tail; ++i) early[go.order[i]] = 1;
        for (size_t g = 0, i = 0; g < groups.size(); ++g)       // (they are in order already: no sort)
            if (early[g]) go.order[i++] = static_cast<int32_t>(g);
    }
    return go;
}
template <class Item, class Make>
std::vector<Item> order_by_groups(std::vector<std::vector<GroupEntry>>& groups, int32_t h, int workers, Make make)
{
    const GroupOrder go = order_groups(groups, h, workers);
    std::vector<Item> items;
    items.reserve(static_cast<size_t>(go.n_items));
    std::vector<int32_t> block_of, cost;
    for (int32_t g : go.order)
        for (int32_t a = 0; a < h; ++a)
            for (const GroupEntry& e : groups[g]) {
                items.push_back(make(a, e));
                if (!go.settled) {
                    block_of.push_back(g * h + a);
                    cost.push_back(e.cost);
                }
            }
    if (!go.settled) order_items(items, block_of, cost, workers);
    return items;
}

// Steps of FWD_SHORT_KEYS keys that the q rows [q0, q0 + rows) of a pair visit in the short-sequence kernel
inline int32_t kv_steps_short(const hydra_pair_t& p, int32_t q0, int32_t rows, int causal)
{
    int64_t n_keys = p.k_len;
    if (causal) n_keys = std::min<int64_t>(n_keys, int64_t{q0} + rows - 1 + (p.q_start - p.k_start) + 1);
    return n_keys > 0 ? static_cast<int32_t>((n_keys + FWD_SHORT_KEYS - 1) / FWD_SHORT_KEYS) : 0;
}

// What the short-sequence forward makes its q tiles of: a pair, or consecutive q chunks that meet the same kv chunk, where that
// saves tiles (a chunk's last tile is ragged: sequences of 121 tokens in chunks of 30 have ten tiles pair by pair, four by kv
// chunk). `all` has the sum of the pairs' rows.
// Forward, pair by pair / shared, us: 30000 tokens of 64 to 512, 16 heads, ring of 4 628 / 347, 12 sequences of 121 tokens, 16
// heads, ring of 2 28.8 / 22.6, 26283 log-normal tokens, 16 heads, ring of 4 710 / 619, 65536 of 64 to 512, 32 heads, cut in two
// 831 / 804.
// Where no pair has partial rows the pairs are the runs, in their order.
struct FwdRun {
    hydra_pair_t all;
    int32_t first, n;       // its pairs: FwdRuns::order[first .. first + n)
};
struct FwdRuns {
    std::vector<FwdRun> runs;
    std::vector<int32_t> order;
    bool cut = false;       // some pair has partial rows
};
FwdRuns make_runs(const Problem& pb, const std::vector<uint8_t>& wanted)
{
    FwdRuns r;
    r.order.reserve(pb.pairs.size());
    for (size_t i = 0; i < pb.pairs.size(); ++i)
        if (wanted[i] && pb.pairs[i].q_len > 0) {
            r.order.push_back(static_cast<int32_t>(i));
            r.cut = r.cut || pb.pairs[i].part_row >= 0;
        }
    r.runs.reserve(r.order.size());
    auto alone = [&](size_t i) { r.runs.push_back(FwdRun{pb.pairs[r.order[i]], static_cast<int32_t>(i), 1}); };
    if (!r.cut) {
        for (size_t i = 0; i < r.order.size(); ++i) alone(i);
        return r;
    }
    auto less = [&](int32_t x, int32_t y) {
        const auto &a = pb.pairs[x], &b = pb.pairs[y];
        if (a.seq != b.seq) return a.seq < b.seq;
        if (a.k_start != b.k_start) return a.k_start < b.k_start;
        return a.k_len != b.k_len ? a.k_len < b.k_len : a.q_start < b.q_start;
    };
    std::stable_sort(r.order.begin(), r.order.end(), less);
    auto tiles = [](int32_t rows) { return (rows + TILE - 1) / TILE; };
    for (size_t i = 0, j = 0; i < r.order.size(); i = j) {
        hydra_pair_t all = pb.pairs[r.order[i]];
        int32_t separate = tiles(all.q_len);
        for (j = i + 1; j < r.order.size(); ++j) {
            const auto& p = pb.pairs[r.order[j]];
            if (p.seq != all.seq || p.k_start != all.k_start || p.k_len != all.k_len || p.q_start != all.q_start + all.q_len ||
                pb.q_row(p.seq, p.q_start) != pb.q_row(p.seq, all.q_start) + all.q_len)
                break;
            all.q_len += p.q_len;
            separate += tiles(p.q_len);
        }
        if (tiles(all.q_len) < separate) {
            r.runs.push_back(FwdRun{all, static_cast<int32_t>(i), static_cast<int32_t>(j - i)});
            continue;
        }
        for (size_t t = i; t < j; ++t) alone(t);        // one pair, or nothing saved
    }
    return r;
}

// Tiles whose keys the two slots of a thread block share (short-sequence forward, calls of few tiles), dealt out longest first,
// each to the thread block that has least to do: a longer tile as two parts, one per slot, short ones two at a time, a whole
// one per slot (not in calls with a thread block for each).
struct SharedTile { int32_t run, q0, steps, head; };
struct DealtTile { int32_t first, second, block, round; };      // second: the tile beside it; the same one: shared; -1: none
struct Deal {
    int32_t grid = 0, rounds = 0;
    int64_t end = 0;                                    // of the longest thread block, in steps
    std::vector<DealtTile> tiles;
};
Deal deal_shared_tiles(const std::vector<SharedTile>& tiles)
{
    constexpr int32_t kSharedSteps = 6;                 // a part of two steps is not worth the join
    constexpr int32_t kOverhead = 3;                    // of a tile: load, join and store, in steps
    Deal deal;
    const int32_t n = static_cast<int32_t>(tiles.size());
    deal.grid = std::min(plan_workers(1), n);
    std::vector<int32_t> order(n), used(deal.grid, 0);
    for (int32_t i = 0; i < n; ++i) order[i] = i;
    if (n > deal.grid)                                  // (else as they lie: neighbours share K and V)
        std::stable_sort(order.begin(), order.end(), [&](int32_t x, int32_t y) { return tiles[x].steps > tiles[y].steps; });
    using Load = std::pair<int64_t, int32_t>;           // (steps so far, thread block)
    std::priority_queue<Load, std::vector<Load>, std::greater<Load>> least;
    for (int32_t c = 0; c < deal.grid; ++c) least.push({0, c});
    for (int32_t i = 0; i < n; ++i) {
        const int32_t t = order[i], steps = tiles[t].steps;
        const int32_t block = least.top().second;
        int64_t load = least.top().first + kOverhead;
        least.pop();
        DealtTile d{t, -1, block, used[block]++};
        if (steps >= (n > deal.grid ? kSharedSteps : 2)) {
            d.second = t;
            load += (steps + 1) / 2;
        } else {
            if (n > deal.grid && i + 1 < n) d.second = order[++i];
            load += steps;
        }
        deal.tiles.push_back(d);
        deal.rounds = std::max(deal.rounds, used[block]);
        deal.end = std::max(deal.end, load);
        least.push({load, block});
    }
    return deal;
}

void build_fwd(const Problem& pb, int causal, Plan& plan, std::vector<uint8_t>& blob)
{
    // Which pairs go to the short-sequence kernel (one CTA per SM, two independent 128-row tiles in flight,
    // steps of 64 keys): those whose q range and kv range are both short. On such pairs the CTA-pair kernel is
    // bound by the length of a tile's chain of steps, and more, shorter chains per SM win; on long pairs its
    // operand sharing and its 256-row tiles do. A second launch has a price of its own (its start and its
    // tail), so the short kernel is used only if the short pairs carry at least a quarter of the call's work.
    const int32_t short_len = fwd_short_len_for(pb, causal);
    std::vector<uint8_t> is_short(pb.pairs.size(), 0);
    // A call of few q tiles takes as long as its longest tile's chain of steps. The short kernel's two slots then share the
    // keys of a tile, whatever their number (deal_shared_tiles; the CTA-pair kernel would leave SMs idle): always with no more
    // tiles than SMs, in calls of more where the queue is expected to take longer than the tiles dealt out. A step takes 0.93
    // us in a slot whose neighbour idles, 1.25 to 1.4 beside a busy one; on CTA pairs a step's share of an SM is 0.5 to 0.6.
    // Forward in passes one after another, 16 heads of 192 unless said, queue / shared, us: one sequence of 1300 tokens 28.2 /
    // 19.8, of 2048 39.1 / 29.4, of 4096, 8 heads 68.1 / 51.4, of 8192, 4 heads 126 / 94; 4820 tokens in five sequences of 341 to
    // 2078, 8 heads 39.9 / 33.4; 8192 in seven of 341 to 2908, 4 heads 50.6 / 38.9; beyond the line one of 3000 60.1 / 63.8, of
    // 4096 86.9 / 100, of 2048, 32 heads 61.0 / 66.2, ten of 410 34.1 / 40.8.
    // (A limit set by the caller is kept to.)
    // (A work item counts its steps in 16 bits: more keys than two items hold stay with the CTA-pair kernel.)
    constexpr int64_t kMostKeys = int64_t{UINT16_MAX} * FWD_SHORT_KEYS;
    constexpr int64_t kMostShared = 5;                 // half tiles per SM: above 2.5 tiles per SM sharing never won
    int64_t n_tiles = 0;
    int32_t longest = 0, most_keys = 0;
    bool within = true;
    for (const auto& p : pb.pairs) {
        longest = std::max(longest, std::max(p.q_len, p.k_len));
        most_keys = std::max(most_keys, p.k_len);
        within = within && p.q_len <= short_len && p.k_len <= short_len;
    }
    FwdRuns made = make_runs(pb, std::vector<uint8_t>(pb.pairs.size(), 1));
    const std::vector<FwdRun>& runs = made.runs;
    for (const FwdRun& run : runs) n_tiles += (run.all.q_len + TILE - 1) / TILE;
    n_tiles *= pb.h;
    std::vector<SharedTile> tiles;
    Deal deal;
    bool halves = short_len > 0 && 2 * n_tiles <= kMostShared * plan_workers(1) && most_keys <= 2 * kMostKeys &&
                  (within || pb.fwd_short_set < 0);
    if (halves) {
        int64_t work = 0;
        int32_t chain = 0;
        for (size_t ri = 0; ri < runs.size(); ++ri) {
            const auto& p = runs[ri].all;
            for (int32_t a = 0; a < pb.h; ++a)
                for (int32_t q0 = 0; q0 < p.q_len; q0 += TILE) {
                    const int32_t steps = kv_steps_short(p, q0, std::min(TILE, p.q_len - q0), causal);
                    chain = std::max(chain, steps + kItemOverhead);
                    work += steps + kItemOverhead;
                    tiles.push_back(SharedTile{static_cast<int32_t>(ri), q0, steps, a});
                }
        }
        const int64_t queue = std::max<int64_t>(chain * 93, work * 60 / plan_workers(1));
        deal = deal_shared_tiles(tiles);
        halves = n_tiles <= plan_workers(1) || deal.end * 130 < queue;
    }
    if (halves) {
        std::fill(is_short.begin(), is_short.end(), 1);
    } else {
        double work_short = 0, work_all = 0;
        for (size_t pi = 0; pi < pb.pairs.size(); ++pi) {
            const auto& p = pb.pairs[pi];
            const double w = static_cast<double>(p.q_len) * p.k_len;
            work_all += w;
            if (short_len > 0 && p.q_len <= short_len && p.k_len <= short_len) { is_short[pi] = 1; work_short += w; }
        }
        // The second launch is not worth its price either if little is left for it that the short kernel would run almost
        // as fast (not against a limit set by the caller). In a small call: pairs of up to twice the limit and 2^29 positions
        // (with those above the mask), which take 0.2 ms. 4096 packed tokens, 16 heads, the longest sequence 1381 tokens:
        // 75 us on both kernels, 59 on the short one alone. In a large one pairs of up to a quarter more than the limit,
        // however much they are of it: 65536 tokens, 16 heads, 24 sequences of 2016 tokens beside some of 300 639 us
        // alone, 696 on both, 720 on CTA pairs; 16 query heads over two K / V heads, seven of 4160 767, 886, 886.
        const bool automatic = pb.fwd_short_set < 0, many = many_q_tiles(pb, causal);
        if (automatic && many && int64_t{4} * longest <= 5 * short_len && work_short * 64 >= work_all)
            std::fill(is_short.begin(), is_short.end(), 1);
        else if (work_short * 4 < work_all)
            std::fill(is_short.begin(), is_short.end(), 0);
        else if (automatic && !many && longest <= 2 * short_len && (work_all - work_short) * pb.h <= double{1 << 29})
            std::fill(is_short.begin(), is_short.end(), 1);
    }
    int32_t longest_tile = 0;
    int64_t short_cost = 0;
    std::vector<std::vector<GroupEntry>> groups(pb.n_seqs), groups_short(pb.n_seqs);
    if (made.cut && std::find(is_short.begin(), is_short.end(), 0) != is_short.end()) made = make_runs(pb, is_short);
    for (size_t ri = 0; ri < runs.size(); ++ri) {
        const auto& p = runs[ri].all;
        if (!is_short[made.order[runs[ri].first]]) continue;
        for (int32_t q0 = 0; q0 < p.q_len; q0 += TILE) {
            const int32_t rows = std::min(TILE, p.q_len - q0);
            const int32_t n_kv = kv_steps_short(p, q0, rows, causal);
            groups_short[p.seq].push_back(GroupEntry{q0, n_kv, rows, n_kv, static_cast<int32_t>(ri)});
            longest_tile = std::max(longest_tile, n_kv);
            short_cost += n_kv + kItemOverhead;
        }
    }
    for (size_t pi = 0; pi < pb.pairs.size(); ++pi) {
        const auto& p = pb.pairs[pi];
        const int32_t of = static_cast<int32_t>(pi);
        if (is_short[pi]) continue;
        // One item = two consecutive 256-row UMMA tiles (A, then B) of a CTA pair. The slabs are aligned to
        // the END of the q chunk: with an odd number of 256-row tiles the chunk's FIRST tile goes alone (it
        // visits the fewest kv tiles), so the ragged last tile rides with a full neighbour instead of running
        // its many kv tiles with the tensor cores half idle (32K packed workload: 1008 -> 942 kv steps per
        // head, steps with a single active tile 266 -> 134).
        const int32_t n_tiles = (p.q_len + 2 * TILE - 1) / (2 * TILE);
        for (int32_t q0 = (n_tiles & 1) ? -2 * TILE : 0; q0 < p.q_len; q0 += 4 * TILE) {
            const bool lone = q0 < 0;                       // tile A only, at row 0
            const int32_t qa = lone ? 0 : q0;
            const int32_t n_a = kv_tiles(p, qa, causal, 2 * TILE);
            // n_b = -1: the item has no second tile (0 would mean: a tile whose rows see no key)
            const int32_t n_b = (!lone && qa + 2 * TILE < p.q_len) ? kv_tiles(p, qa + 2 * TILE, causal, 2 * TILE) : -1;
            // the two tiles advance in lockstep (one kv tile each per step of the issue order), so the time
            // of an item goes with the longer tile, not with the sum: a slab whose second tile is empty costs
            // as much per kv tile as a full one (measured: with the sum the slowest cluster of the 32K packed
            // workload ended 17 % after the mean, now 4 %)
            groups[p.seq].push_back(GroupEntry{qa, n_a, n_b, 2 * std::max(n_a, std::max(n_b, 0)), of});
        }
    }
    // How far ahead the short kernel's slots pop: items of up to 8 steps two ahead, longer ones late, so that no slot sits on
    // an item while others run dry. Two ahead throughout is better where no item is long: all of up to 16 steps (1024
    // keys) and none over a slot's even share of the call, or all of up to 24 and none over 0.6 of it. Late / two ahead us:
    // 16384 tokens, 8 heads of 192, sequences of 520 tokens 66.7 / 64.9, of 900 84.6 / 77.5, of 1000 80.3 / 78.0, of 1150
    // 90.4 / 88.7; of 128 53.5 / 48.1, 68.9 / 58.6, 58.7 / 58.4, 70.3 / 69.3. Beyond the lines: 4 heads, 10 sequences of 1006
    // tokens 25.0 / 26.7, 12 of 900 25.5 / 30.6; 16 heads, 6000 tokens of 1100 54.8 / 64.6, 4096 of 1500 36.2 / 42.2, 8192
    // log-normal ones 105.9 / 124.5. (A fixed line inside a call, at 12, 16 or 24 steps, was worse than either way on
    // 1500-token sequences.)
    constexpr int32_t kShortItem = 8, kShortTile = 16, kMidTile = 24;
    const int64_t slots = 2 * plan_workers(1);
    const int64_t share = longest_tile <= kShortTile ? 10 : longest_tile <= kMidTile ? 6 : 0;      // tenths of the even share
    const bool early = (longest_tile + kItemOverhead) * slots * 10 <= short_cost * pb.h * share;
    plan.early_pops = early ? kMidTile : kShortItem;
    const std::vector<FwdItem> items = order_by_groups<FwdItem>(
        groups, pb.h, plan_workers(2),
        [](int32_t a, const GroupEntry& e) { return FwdItem{e.of, a, e.a, e.b, e.c, {0, 0, 0}}; });
    const std::vector<PairDev> dev_pairs = device_pairs(pb);
    plan.off_pairs = append(blob, dev_pairs);
    plan.off_items = append(blob, items);
    plan.n_items = static_cast<int32_t>(items.size());
    // The short kernel's items carry what they need of their pair (its slots start an item from this alone). A
    // micro-batch of short sequences has tens of thousands of them and a new one arrives with every step, so in
    // the common case (many items, none long: the block order is final) they are written straight into the
    // table, a group's entries once and then one copy per head with the head number set.
    // Where the rows of tiles that several pairs share go, once per tile (every head has the same).
    std::vector<FwdSeg> segs;
    std::vector<size_t> tile_segs;                      // first entry of each tile of the shared runs, and the end
    std::vector<size_t> run_tiles(runs.size(), 0);      // where a run's tiles begin in it
    for (size_t ri = 0; ri < runs.size(); ++ri) {
        const FwdRun& run = runs[ri];
        if (run.n < 2) continue;
        run_tiles[ri] = tile_segs.size();
        for (int32_t q0 = 0; q0 < run.all.q_len; q0 += TILE) {
            tile_segs.push_back(segs.size());
            int32_t first = 0;                          // the pair's first row in the run
            for (int32_t t = run.first; t < run.first + run.n; ++t) {
                const int32_t pi = made.order[t], len = pb.pairs[pi].q_len;
                if (first < q0 + TILE && first + len > q0) {
                    const int32_t begin = std::max(0, first - q0);
                    segs.push_back(FwdSeg{static_cast<int16_t>(begin), static_cast<int16_t>(dev_pairs[pi].to_part),
                                          dev_pairs[pi].out_row0 + q0 - first});
                }
                first += len;
            }
        }
    }
    tile_segs.push_back(segs.size());
    auto make_short = [&](int32_t a, const GroupEntry& e) {
        const FwdRun& run = runs[e.of];
        const PairDev& d = dev_pairs[made.order[run.first]];
        FwdShortItem it{};
        it.q_tok0 = d.q_tok0 + e.a;
        it.k_tok0 = d.k_tok0;
        it.k_len = d.k_len;
        it.off = e.a + d.off;
        it.out_row0 = d.out_row0 + e.a;
        it.head = static_cast<uint16_t>(a);
        it.n_kv = static_cast<uint16_t>(e.b);
        it.rows = static_cast<uint8_t>(e.c);
        it.to_part = static_cast<uint8_t>(d.to_part);
        if (run.n > 1) {
            const size_t* at = &tile_segs[run_tiles[e.of] + e.a / TILE];
            it.first_seg = static_cast<uint32_t>(at[0]);
            it.half_segs = static_cast<uint16_t>((at[1] - at[0]) << 8);
        }
        return it;
    };
    plan.off_segs = append(blob, segs);
    plan.n_segs = segs.size();
    const int short_workers = 2 * plan_workers(1);
    if (halves) {
        auto entry = [&](const SharedTile& t) {
            return GroupEntry{t.q0, t.steps, std::min(TILE, runs[t.run].all.q_len - t.q0), t.steps, t.run};
        };
        // (an item of no rows and no steps does nothing)
        std::vector<FwdShortItem> table(static_cast<size_t>(deal.rounds) * 2 * deal.grid);
        for (const DealtTile& t : deal.tiles) {
            const SharedTile& one = tiles[t.first];
            FwdShortItem it = make_short(one.head, entry(one)), other{};
            if (t.second == t.first) {
                const int32_t n0 = (one.steps + 1) / 2, skip = n0 * FWD_SHORT_KEYS;
                other = it;
                it.n_kv = static_cast<uint16_t>(n0);
                it.half_segs |= 1;
                other.n_kv = static_cast<uint16_t>(one.steps - n0);
                other.half_segs |= 2;
                other.k_tok0 += skip;
                other.k_len -= skip;
                other.off -= skip;
            } else if (t.second >= 0) {
                other = make_short(tiles[t.second].head, entry(tiles[t.second]));
            }
            table[static_cast<size_t>(2 * t.round) * deal.grid + t.block] = it;
            table[static_cast<size_t>(2 * t.round + 1) * deal.grid + t.block] = other;
        }
        plan.off_items2 = append(blob, table);
        plan.n_items2 = static_cast<int32_t>(table.size());
        plan.halves = 1;
        plan.short_grid = deal.grid;
        return;
    }
    const GroupOrder go = order_groups(groups_short, pb.h, short_workers);
    if (go.settled) {
        const size_t off = align_up(blob.size(), 16);
        blob.resize(off + static_cast<size_t>(go.n_items) * sizeof(FwdShortItem));
        FwdShortItem* dst = reinterpret_cast<FwdShortItem*>(blob.data() + off);
        std::vector<FwdShortItem> block;
        for (int32_t g : go.order) {
            block.clear();
            for (const GroupEntry& e : groups_short[g]) block.push_back(make_short(0, e));
            for (int32_t a = 0; a < pb.h; ++a) {
                std::memcpy(dst, block.data(), block.size() * sizeof(FwdShortItem));
                for (size_t i = 0; i < block.size(); ++i) dst[i].head = static_cast<uint16_t>(a);
                dst += block.size();
            }
        }
        plan.off_items2 = off;
        plan.n_items2 = static_cast<int32_t>(go.n_items);
    } else {
        const std::vector<FwdShortItem> short_items =
            order_by_groups<FwdShortItem>(groups_short, pb.h, short_workers, make_short);
        plan.off_items2 = append(blob, short_items);
        plan.n_items2 = static_cast<int32_t>(short_items.size());
    }
}

void build_merge(const Problem& pb, Plan& plan, std::vector<uint8_t>& blob)
{
    std::vector<MergeGroup> groups;
    std::vector<int32_t> lists;
    std::vector<MergeItem> items;
    size_t i = 0;
    while (i < pb.pairs.size()) {
        size_t j = i;
        while (j < pb.pairs.size() && pb.pairs[j].group == pb.pairs[i].group) ++j;
        const auto& p = pb.pairs[i];
        if (p.part_row >= 0 && p.q_len > 0) {
            MergeGroup g;
            g.out_tok0 = static_cast<int32_t>(pb.q_row(p.seq, p.q_start));
            g.rows = p.q_len;
            g.list_off = static_cast<int32_t>(lists.size());
            g.n_parts = static_cast<int32_t>(j - i);
            plan.n_items2 = std::max(plan.n_items2, g.n_parts);     // (of a merge plan: the most partials of a chunk)
            for (size_t t = i; t < j; ++t) lists.push_back(pb.pairs[t].part_row);
            for (int32_t r = 0; r < g.rows; r += MERGE_ROWS)
                items.push_back(MergeItem{static_cast<int32_t>(groups.size()), r});
            groups.push_back(g);
        }
        i = j;
    }
    plan.off_groups = append(blob, groups);
    plan.off_lists = append(blob, lists);
    plan.off_items = append(blob, items);
    plan.n_items = static_cast<int32_t>(items.size());
}

// Backward lists: pairs grouped by q chunk (dQ kernel) and by kv chunk (dK/dV kernel).
// Lays the pairs out in the dS hand-off buffer (see DsGeom): returns the number of 16 KB blocks per
// head and, if `dev` is given, writes every pair's first block. -1 if a pair has a kv tile whose first
// visible q sub-tile lies beyond the pair's q rows (possible only for pairs that are not chunk pairs of
// a cut sequence); the backward then recomputes S and dP on the query side instead.
int64_t ds_layout(const Problem& pb, int causal, std::vector<PairDev>* dev)
{
    int64_t blocks = 0;
    for (size_t i = 0; i < pb.pairs.size(); ++i) {
        const auto& p = pb.pairs[i];
        if (dev) (*dev)[i].ds_base = static_cast<int32_t>(blocks);
        if (p.q_len <= 0 || p.k_len <= 0) continue;
        const DsGeom g = ds_geom(p.q_len, p.q_start - p.k_start, causal);
        const int32_t nk = (p.k_len + TILE - 1) / TILE;
        if (ds_first(g, nk - 1) > g.nu_even) return -1;
        blocks += ds_rowstart(g, nk);
        if (blocks > (int64_t{1} << 30)) return -1;
    }
    return blocks + 1;                                  // one spare block: a q tile is read as two blocks
}

// q sub-tiles of pair p that a kv tile starting at row k0 of the pair's keys meets
inline int32_t q_subs(const hydra_pair_t& p, int32_t k0, int causal)
{
    const int32_t n_sub = (p.q_len + SUB - 1) / SUB;
    const int32_t i_min = causal ? k0 - (p.q_start - p.k_start) : 0;
    return std::max(0, n_sub - (i_min > 0 ? i_min / SUB : 0));
}

// Two CTAs per key-side item where there are enough for that and the longest is worth the exchange at the end: it and the
// cluster's start cost 2 us, a sub-tile takes 1.1. Step with sequences of 300 tokens (5 sub-tiles) 30.5 us with one CTA,
// 31.8 with two; of 512 (8) 36.6 and 36.4; of 1024 tokens, 8 heads, 54.8 and 51.4; of 2048, 4 heads, 84.7 and 73.4.
// Decided for a call as a whole, so that its bands add up dk and dv in the same order as one launch would.
bool key_tiles_halved(const Problem& pb, int causal)
{
    std::vector<const hydra_pair_t*> by_k;
    for (const auto& p : pb.pairs)
        if (p.q_len > 0 && p.k_len > 0) by_k.push_back(&p);
    auto range = [](const hydra_pair_t* p) { return Range{p->seq, p->k_start, p->k_len}; };
    std::sort(by_k.begin(), by_k.end(), [&](const hydra_pair_t* a, const hydra_pair_t* b) { return range_less(range(a), range(b)); });
    int64_t items = 0;
    int32_t longest = 0;
    for (size_t i = 0, j = 0; i < by_k.size(); i = j) {
        for (j = i; j < by_k.size() && !range_less(range(by_k[i]), range(by_k[j])); ++j) {}
        for (int32_t r0 = 0; r0 < by_k[i]->k_len; r0 += TILE) {
            items += pb.h;
            if (2 * items > plan_workers(1)) return false;
            int32_t c = 0;
            for (size_t t = i; t < j; ++t) c += q_subs(*by_k[t], r0, causal);
            longest = std::max(longest, c);
        }
    }
    return longest > 8;
}

// Query heads that a key-side item visits where several share a K / V head. With all of a group in one item dk and dv are
// complete in tensor memory: no fp32 sums in memory, no cast, K and V loaded and the accumulators written once. But such
// items are few and long; the fewer heads an item takes, the better a small call fills the SMs. The queue is simulated for
// every number of heads that divides the group (longest items first, as the kernel's list has them; a unit is a 64-row
// sub-tile, about 1 us). Step in passes one after another, one head per item / as chosen here: 32768 tokens of 64 to 512,
// 32 heads of 128 over 8, 1245 / 965 us; log-normal lengths, 8192 tokens, 32 heads over 8, 854 / 776, 16384 tokens, 16 over
// 4, 1100 / 1038, 32768 tokens, 16 heads of 128 over 2, 1886 / 1852 (1, 2, 4, 8 heads per item: key side 959, 923, 908, 932
// us, and the cast 23 us less with all 8).
int32_t heads_per_key_item(const std::vector<std::vector<GroupEntry>>& groups, const Problem& pb, int workers)
{
    if (pb.kv_group <= 1) return 1;
    constexpr int64_t kItem = 4, kItemSummed = 6, kCast = 8;    // beyond its sub-tiles: an item, one that adds in fp32; zeroing and cast
    std::vector<int32_t> costs;
    int64_t total = 0;
    int32_t longest = 0;
    for (const auto& g : groups)
        for (const GroupEntry& e : g) { costs.push_back(e.cost); total += e.cost; longest = std::max(longest, e.cost); }
    std::sort(costs.begin(), costs.end(), std::greater<int32_t>());
    int64_t best = 0;
    int32_t heads = 1;
    for (int32_t d = pb.kv_group; d >= 1; --d) {
        if (pb.kv_group % d) continue;
        const int64_t item = d == pb.kv_group ? kItem : kItemSummed, copies = pb.h / d;
        const int64_t even = (total * pb.h + static_cast<int64_t>(costs.size()) * copies * item + workers - 1) / workers;
        int64_t end = std::max(even, longest * int64_t{d} + item);
        // (with more items than that the list ends with short ones)
        if (static_cast<int64_t>(costs.size()) * copies <= 16 * workers) {
            std::priority_queue<int64_t, std::vector<int64_t>, std::greater<int64_t>> free;
            for (int i = 0; i < workers; ++i) free.push(0);
            end = 0;
            for (int32_t c : costs)
                for (int64_t k = 0; k < copies; ++k) {
                    const int64_t t = free.top() + int64_t{c} * d + item;
                    free.pop();
                    free.push(t);
                    end = std::max(end, t);
                }
        }
        end += d == pb.kv_group ? 0 : kCast;
        if (d == pb.kv_group || end < best) { best = end; heads = d; }
    }
    return heads;
}

void build_bwd(const Problem& pb, int causal, Plan& plan, std::vector<uint8_t>& blob)
{
    const int32_t n = static_cast<int32_t>(pb.pairs.size());
    auto group_by = [&](bool by_q, std::vector<int32_t>& lists, std::vector<GroupItem>& items) {
        std::vector<int32_t> order(n);
        for (int32_t i = 0; i < n; ++i) order[i] = i;
        auto key = [&](int32_t i) {
            const auto& p = pb.pairs[i];
            return Range{p.seq, by_q ? p.q_start : p.k_start, by_q ? p.q_len : p.k_len};
        };
        std::stable_sort(order.begin(), order.end(),
                         [&](int32_t a, int32_t b) { return range_less(key(a), key(b)); });
        std::vector<std::vector<GroupEntry>> groups(pb.n_seqs);
        std::vector<std::pair<int32_t, int32_t>> list_of;  // (list_off, list_len) of every chunk that has work
        int32_t i = 0;
        while (i < n) {
            int32_t j = i;
            const Range r = key(order[i]);
            while (j < n) {
                const Range s = key(order[j]);
                if (s.seq != r.seq || s.start != r.start || s.len != r.len) break;
                ++j;
            }
            // a chunk with no rows, or whose pairs are all empty on the other side, has no work
            const int32_t list_off = static_cast<int32_t>(lists.size());
            for (int32_t t = i; t < j; ++t) {
                const auto& p = pb.pairs[order[t]];
                if ((by_q ? p.k_len : p.q_len) > 0) lists.push_back(order[t]);
            }
            const int32_t list_len = static_cast<int32_t>(lists.size()) - list_off;
            if (r.len > 0 && list_len > 0) {
                const int32_t of = static_cast<int32_t>(list_of.size());
                list_of.emplace_back(list_off, list_len);
                for (int32_t r0 = 0; r0 < r.len; r0 += TILE) {
                    int32_t c = 0;
                    for (int32_t t = 0; t < list_len; ++t) {
                        const auto& p = pb.pairs[lists[list_off + t]];
                        c += by_q ? kv_tiles(p, r0, causal) : q_subs(p, r0, causal);
                    }
                    groups[r.seq].push_back(GroupEntry{r0, 0, 0, c, of});
                }
            }
            i = j;
        }
        const int32_t heads = by_q || plan.halves ? 1 : heads_per_key_item(groups, pb, plan_workers(1));
        if (!by_q) plan.item_heads = heads;
        for (auto& g : groups)
            for (GroupEntry& e : g) e.cost *= heads;
        items = order_by_groups<GroupItem>(groups, pb.h / heads, plan_workers(1), [&](int32_t a, const GroupEntry& e) {
            return GroupItem{list_of[e.of].first, list_of[e.of].second, a * heads, e.a};
        });
    };
    std::vector<int32_t> lists_q, lists_k;
    std::vector<GroupItem> items_q, items_k;
    plan.halves = key_tiles_halved(pb, causal);
    group_by(true, lists_q, items_q);
    group_by(false, lists_k, items_k);
    std::vector<PairDev> dev = device_pairs(pb);
    plan.ds_head_blocks = ds_layout(pb, causal, &dev);
    plan.off_pairs = append(blob, dev);
    plan.off_lists = append(blob, lists_q);
    plan.off_items = append(blob, items_q);
    plan.off_lists2 = append(blob, lists_k);
    plan.off_items2 = append(blob, items_k);
    plan.n_items = static_cast<int32_t>(items_q.size());
    plan.n_items2 = static_cast<int32_t>(items_k.size());
}

// A plan on loan for the launches of one call: holds the plan cache's lock from the look-up to the last
// launch (so that no other thread can recycle the arena half between the two), and on release records, on
// the call's stream, that the tables have a reader.
class PlanLease {
public:
    PlanLease() = default;
    PlanLease(const PlanLease&) = delete;
    PlanLease& operator=(const PlanLease&) = delete;
    ~PlanLease() { release(); }
    void release()
    {
        if (!lock_.owns_lock()) return;
        if (plan_) arena_note_use(*plan_, device_, stream_);
        lock_.unlock();
    }
    // Finds the plan (building it on the host the first time) and makes its tables resident.
    int32_t acquire(int kind, const Problem& pb, int causal, cudaStream_t stream);
    const Plan& plan() const { return *plan_; }
    template <class T>
    const T* at(size_t off) const { return reinterpret_cast<const T*>(tables_ + off); }

private:
    std::unique_lock<std::mutex> lock_;
    std::shared_ptr<Plan> plan_;
    const uint8_t* tables_ = nullptr;
    int device_ = 0;
    cudaStream_t stream_ = nullptr;
};

// The cached plan of a problem, built on the host if it is new. g_plan_mutex held.
std::shared_ptr<Plan> find_or_build_plan(int kind, int device, const Problem& pb, int causal)
{
    std::vector<uint8_t> key = make_key(kind, device, pb, causal);
    for (size_t i = 0; i < g_plans.size(); ++i)
        if (g_plans[i]->key == key) {
            if (i + 1 != g_plans.size()) std::rotate(g_plans.begin() + i, g_plans.begin() + i + 1, g_plans.end());
            return g_plans.back();
        }
    auto plan = std::make_shared<Plan>();
    plan->kind = kind;
    plan->device = device;
    if (kind == HYDRA_WS_FWD) build_fwd(pb, causal, *plan, plan->blob);
    else if (kind == HYDRA_WS_MERGE) build_merge(pb, *plan, plan->blob);
    else build_bwd(pb, causal, *plan, plan->blob);
    plan->key.swap(key);
    if (g_plans.size() >= kMaxPlans) {
        // an evicted plan that owns device memory frees it: drain the device first (arena plans own none)
        if (g_plans.front()->own.ptr) cudaDeviceSynchronize();
        g_plans.erase(g_plans.begin());
    }
    g_plans.push_back(plan);
    return plan;
}

int32_t PlanLease::acquire(int kind, const Problem& pb, int causal, cudaStream_t stream)
{
    if (cudaGetDevice(&device_) != cudaSuccess || device_ < 0 || device_ >= 64) return HYDRA_ERR_CUDA;
    stream_ = stream;
    lock_ = std::unique_lock<std::mutex>(g_plan_mutex);
    plan_ = find_or_build_plan(kind, device_, pb, causal);
    if (int32_t s = arena_place(*plan_, device_, stream, &tables_)) { plan_.reset(); return s; }
    return HYDRA_OK;
}

// A forward of a new problem is followed, in training, by the merge and the backward of the same problem:
// their tables are built on the host right after the forward kernel has been launched, while the GPU runs
// it, instead of when their own calls arrive and the GPU has nothing to do (host work only: nothing is
// uploaded). hydra_set_plan_prefetch(0) switches this off for forward-only use. (The last use of `pb`: its pairs are joined.)
std::atomic<int> g_plan_prefetch{1};
void prefetch_plans(Problem& pb, int causal, bool any_part)
{
    if (!g_plan_prefetch.load()) return;
    int device = 0;
    if (cudaGetDevice(&device) != cudaSuccess || device < 0 || device >= 64) return;
    std::lock_guard<std::mutex> lock(g_plan_mutex);
    if (any_part) find_or_build_plan(HYDRA_WS_MERGE, device, pb, 0);
    join_chunks(pb, causal);                               // as the backward will
    find_or_build_plan(HYDRA_WS_BWD, device, pb, causal);
}

// ---------------------------------------------------------------------------------------------
// device properties and tensor maps
// ---------------------------------------------------------------------------------------------
int32_t device_info(int* sms)
{
    static std::atomic<int> majors[kMaxDevices] = {}, counts[kMaxDevices] = {};
    static OncePerDevice asked;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return HYDRA_ERR_CUDA;
    const cudaError_t e = asked(dev, [&] {
        int major = 0, count = 0;
        cudaError_t status = cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, dev);
        if (status == cudaSuccess) status = cudaDeviceGetAttribute(&count, cudaDevAttrMultiProcessorCount, dev);
        majors[dev] = major;
        counts[dev] = count;
        return status;
    });
    if (e != cudaSuccess) return HYDRA_ERR_CUDA;
    if (majors[dev] != 10) return HYDRA_ERR_NOT_SM100;
    if (sms) *sms = counts[dev];
    return HYDRA_OK;
}

using EncodeFn = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                              const cuuint64_t*, const cuuint32_t*, const cuuint32_t*,
                              CUtensorMapInterleave, CUtensorMapSwizzle, CUtensorMapL2promotion,
                              CUtensorMapFloatOOBfill);
EncodeFn encode_fn()
{
    static std::atomic<EncodeFn> found{nullptr};
    EncodeFn fn = found.load();
    if (!fn) {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) == cudaSuccess)
            found = fn = reinterpret_cast<EncodeFn>(p);
    }
    return fn;
}

// [T, h, d] bf16 seen as (d, h, T); a box is 64 elements x 1 head x `rows` tokens, written to
// shared memory as `rows` 128-byte rows with the 128-byte swizzle. Tokens past T read as zero.
int32_t make_map(CUtensorMap* map, const void* base, int64_t T, int32_t h, int32_t d, int32_t rows)
{
    EncodeFn enc = encode_fn();
    if (!enc) return HYDRA_ERR_CUDA;
    const cuuint64_t dims[3] = {static_cast<cuuint64_t>(d), static_cast<cuuint64_t>(h),
                                static_cast<cuuint64_t>(std::max<int64_t>(T, 1))};
    const cuuint64_t strides[2] = {static_cast<cuuint64_t>(d) * 2, static_cast<cuuint64_t>(d) * 2 * h};
    const cuuint32_t box[3] = {64, 1, static_cast<cuuint32_t>(rows)};
    const cuuint32_t es[3] = {1, 1, 1};
    const CUresult r = enc(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(base), dims, strides,
                           box, es, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                           CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? HYDRA_OK : HYDRA_ERR_CUDA;
}

// The kernels of one q / k head dimension.
struct KernelSet {
    int (*fwd_max_clusters)();
    cudaError_t (*launch_fwd)(const CUtensorMap&, const CUtensorMap&, const CUtensorMap&, const FwdParams&, int,
                              cudaStream_t);
    cudaError_t (*launch_fwd_short)(const CUtensorMap&, const CUtensorMap&, const CUtensorMap&, const FwdParams&,
                                    const FwdSeg*, uint64_t, bool, int, cudaStream_t);
    cudaError_t (*launch_bwd_dq)(const CUtensorMap&, const CUtensorMap&, const CUtensorMap&, const CUtensorMap&,
                                 const BwdParams&, int, cudaStream_t);
    cudaError_t (*launch_bwd_dq_from_ds)(const CUtensorMap&, const BwdParams&, int, cudaStream_t);
    cudaError_t (*launch_bwd_dkv)(const CUtensorMap&, const CUtensorMap&, const CUtensorMap&, const CUtensorMap&,
                                  const BwdParams&, bool, int, cudaStream_t);
};
const KernelSet* kernel_set(int32_t d_qk, int32_t d_v)
{
    static const KernelSet k192{fwd_max_clusters, launch_fwd, launch_fwd_short, launch_bwd_dq, launch_bwd_dq_from_ds, launch_bwd_dkv};
    static const KernelSet k128{fwd_max_clusters_d128, launch_fwd_d128, launch_fwd_short_d128, launch_bwd_dq_d128, launch_bwd_dq_from_ds_d128,
                                launch_bwd_dkv_d128};
    if (d_v != D_V) return nullptr;
    if (d_qk == 192) return &k192;
    if (d_qk == 128) return &k128;
    return nullptr;
}

}  // namespace

cudaError_t launch_merge_counted(const MergeParams& p, cudaStream_t stream)
{
    cudaError_t e;
    {
        ScopedKernelTimer timer(K_MERGE, stream);
        e = launch_merge(p, stream);
    }
    if (e == cudaSuccess && p.n_items > 0) g_launches += 1;
    return e;
}
}  // namespace hydra

using namespace hydra;

// =============================================================================================
// C ABI
// =============================================================================================
namespace {
// Copy streams and events of hydra_attn_fwd_bwd_host, one set per device, created on first use.
constexpr size_t kHostLsePad = 64 * 256;                    // alignment slack of the per-group LSE slices
struct HostPipe {
    static constexpr int kMaxGroups = 64;
    cudaStream_t in = nullptr, out = nullptr;
    cudaEvent_t start = nullptr, end = nullptr;
    cudaEvent_t in_done[kMaxGroups] = {}, dout_done[kMaxGroups] = {}, fwd_done[kMaxGroups] = {}, comp_done[kMaxGroups] = {};
};
HostPipe* host_pipe()
{
    static std::mutex mu;
    static std::map<int, HostPipe> pipes;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return nullptr;
    std::lock_guard<std::mutex> lock(mu);
    auto it = pipes.find(dev);
    if (it != pipes.end()) return &it->second;
    HostPipe p;
    bool ok = cudaStreamCreateWithFlags(&p.in, cudaStreamNonBlocking) == cudaSuccess &&
              cudaStreamCreateWithFlags(&p.out, cudaStreamNonBlocking) == cudaSuccess &&
              cudaEventCreateWithFlags(&p.start, cudaEventDisableTiming) == cudaSuccess &&
              cudaEventCreateWithFlags(&p.end, cudaEventDisableTiming) == cudaSuccess;
    for (int g = 0; ok && g < HostPipe::kMaxGroups; ++g)
        ok = cudaEventCreateWithFlags(&p.in_done[g], cudaEventDisableTiming) == cudaSuccess &&
             cudaEventCreateWithFlags(&p.dout_done[g], cudaEventDisableTiming) == cudaSuccess &&
             cudaEventCreateWithFlags(&p.fwd_done[g], cudaEventDisableTiming) == cudaSuccess &&
             cudaEventCreateWithFlags(&p.comp_done[g], cudaEventDisableTiming) == cudaSuccess;
    if (!ok) return nullptr;
    return &pipes.emplace(dev, p).first->second;
}

// Groups of the host-buffer step. The gradients of a group cannot leave before its in-copy has ended, so a step
// takes the copies of one direction plus most of those of its largest group, and every copy costs some 15 us beyond
// its bytes. When the copies bound the step and every sequence fits a group of 1/24 of the (token, head) pairs (not
// under 1 MB of inputs: the launches of a group cost about as much as that copy), a group is a run of whole
// sequences with all heads, contiguous on the host. Otherwise it is a range of heads over all sequences, strided on
// the host: two heads when the copies bound the step, four (which keep the kernels efficient) when the arithmetic
// does; narrower rows slow the link down, and so did groups of both kinds mixed in one step (copies of a few MB).
struct HostGroup { int32_t s0, s1, h0, hn; int64_t t0, tn; };
std::vector<HostGroup> host_groups(const Problem& pb, bool copy_bound)
{
    std::vector<HostGroup> g;
    const int32_t h = pb.h;
    if (copy_bound) {
        int64_t target = std::max<int64_t>(pb.T * h / 24, (int64_t{1} << 20) / ((2 * D_QK + 2 * D_V) * 2));
        for (bool fits = true; fits; target *= 2) {
            g.clear();
            for (int32_t s = 0; s < pb.n_seqs && fits;) {
                int32_t e = s;
                int64_t tok = 0;
                while (e < pb.n_seqs && (tok + pb.cu[e + 1] - pb.cu[e]) * h <= target) tok += pb.cu[e + 1] - pb.cu[e], ++e;
                fits = e > s;
                if (tok > 0) g.push_back({s, e, 0, h, pb.cu[s], tok});
                s = e;
            }
            if (fits && g.size() <= static_cast<size_t>(HostPipe::kMaxGroups)) return g;
        }
        g.clear();
    }
    int32_t hg = h < 4 ? h : (copy_bound ? 2 : 4);
    hg = std::max(hg, (h + HostPipe::kMaxGroups - 1) / HostPipe::kMaxGroups);
    for (int32_t h0 = 0; h0 < h; h0 += hg) g.push_back({0, pb.n_seqs, h0, std::min(hg, h - h0), 0, pb.T});
    return g;
}
}  // namespace

extern "C" {

int32_t hydra_version(void) { return 1; }

const char* hydra_status_string(int32_t s)
{
    switch (s) {
        case HYDRA_OK: return "HYDRA_OK";
        case HYDRA_ERR_INVALID_ARG: return "HYDRA_ERR_INVALID_ARG";
        case HYDRA_ERR_UNSUPPORTED: return "HYDRA_ERR_UNSUPPORTED";
        case HYDRA_ERR_WORKSPACE_TOO_SMALL: return "HYDRA_ERR_WORKSPACE_TOO_SMALL";
        case HYDRA_ERR_CUDA: return "HYDRA_ERR_CUDA";
        case HYDRA_ERR_DEVICE_TIMEOUT: return "HYDRA_ERR_DEVICE_TIMEOUT";
        case HYDRA_ERR_NOT_SM100: return "HYDRA_ERR_NOT_SM100";
        default: return "HYDRA_ERR_UNKNOWN";
    }
}

int64_t hydra_launch_count(void) { return g_launches.load(); }

void hydra_set_wait_limit_ns(uint64_t ns) { g_wait_limit_ns.store(ns ? ns : 1); }

void hydra_debug_stall(int32_t kernel, uint64_t ns)
{
    if (kernel >= 0 && kernel < 3) g_debug_stall_ns[kernel].store(ns);
}

void hydra_shutdown(void)
{
    std::lock_guard<std::mutex> lock(g_plan_mutex);
    int current = 0, count = 0;
    const bool have_device = cudaGetDevice(&current) == cudaSuccess && cudaGetDeviceCount(&count) == cudaSuccess;
    for (int d = 0; have_device && d < count && d < 64; ++d) {
        bool owns = g_arena[d].base != nullptr;
        for (const auto& p : g_plans) owns |= (p->device == d && p->own.ptr != nullptr);
        if (!owns) continue;
        if (cudaSetDevice(d) != cudaSuccess) continue;
        cudaDeviceSynchronize();                       // kernels in flight may still read the tables
        for (auto it = g_plans.begin(); it != g_plans.end();)
            it = ((*it)->device == d) ? g_plans.erase(it) : it + 1;
        arena_release(g_arena[d]);
    }
    if (have_device) cudaSetDevice(current);
    g_plans.clear();
}

void hydra_set_plan_arena_bytes(uint64_t bytes) { g_arena_bytes.store(bytes); }

void hydra_set_plan_prefetch(int32_t on) { g_plan_prefetch.store(on != 0); }

// (a work item counts its 64-key steps in 16 bits)
void hydra_set_fwd_short_len(int32_t len) { g_fwd_short_len.store(std::min(len, 1 << 21)); }

namespace {
// The tables of one call of kind `which`, as the call itself builds them.
bool build_plan(int32_t which, Problem& pb, int32_t causal, Plan& plan)
{
    if (which == HYDRA_WS_BWD) join_chunks(pb, causal);
    if (which == HYDRA_WS_FWD) build_fwd(pb, causal != 0, plan, plan.blob);
    else if (which == HYDRA_WS_MERGE) build_merge(pb, plan, plan.blob);
    else if (which == HYDRA_WS_BWD) build_bwd(pb, causal != 0, plan, plan.blob);
    else return false;
    return true;
}
}  // namespace

double hydra_plan_build_seconds(int32_t which, const int32_t* cu, int32_t n_seqs, int32_t n_heads,
                                const hydra_pair_t* pairs, int32_t n_pairs, int32_t causal)
{
    Problem pb;
    if (make_problem(cu, n_seqs, n_heads, pairs, n_pairs, pb) != HYDRA_OK) return -1.0;
    pb.fwd_short_set = g_fwd_short_len.load();
    Plan plan;
    const auto t0 = std::chrono::steady_clock::now();
    if (!build_plan(which, pb, causal, plan)) return -1.0;
    return std::chrono::duration<double>(std::chrono::steady_clock::now() - t0).count();
}

int32_t hydra_plan_describe(int32_t which, const int32_t* cu, int32_t n_seqs, int32_t n_heads, int32_t n_kv_heads,
                            int32_t d_qk, const hydra_pair_t* pairs, int32_t n_pairs, int32_t causal,
                            int64_t* fields_out, void* tables_out, size_t capacity)
{
    if (!fields_out || (capacity > 0 && !tables_out)) return HYDRA_ERR_INVALID_ARG;
    if (!kernel_set(d_qk, D_V)) return HYDRA_ERR_UNSUPPORTED;
    if (n_kv_heads < 1 || n_heads % n_kv_heads) return HYDRA_ERR_INVALID_ARG;
    Problem pb;
    if (int32_t s = make_problem(cu, n_seqs, n_heads, pairs, n_pairs, pb)) return s;
    pb.dqk = d_qk;
    pb.kv_group = n_heads / n_kv_heads;
    pb.fwd_short_set = g_fwd_short_len.load();
    Plan plan;
    if (!build_plan(which, pb, causal, plan)) return HYDRA_ERR_INVALID_ARG;
    const int64_t fields[HYDRA_PLAN_FIELDS] = {
        static_cast<int64_t>(pb.pairs.size()), plan.n_items, plan.n_items2, plan.halves, plan.short_grid,
        static_cast<int64_t>(plan.n_segs), plan.item_heads, static_cast<int64_t>(plan.off_items2),
        static_cast<int64_t>(plan.off_segs), static_cast<int64_t>(plan.blob.size())};
    std::copy(fields, fields + HYDRA_PLAN_FIELDS, fields_out);
    if (capacity > 0) {
        if (capacity < plan.blob.size()) return HYDRA_ERR_WORKSPACE_TOO_SMALL;
        std::memcpy(tables_out, plan.blob.data(), plan.blob.size());
    }
    return HYDRA_OK;
}

int32_t hydra_usp_factor(int32_t degree, int32_t heads, int32_t* cp_u, int32_t* cp_r)
{
    if (degree < 1 || heads < 1 || !cp_u || !cp_r) return HYDRA_ERR_INVALID_ARG;
    const int32_t u = degree < heads ? degree : heads;
    if (degree % u != 0) return HYDRA_ERR_INVALID_ARG;
    *cp_u = u;
    *cp_r = degree / u;
    return HYDRA_OK;
}

int32_t hydra_zigzag_pairs(const int32_t* cu, int32_t n_seqs, const int32_t* cp_r_host, int32_t cp_r_all,
                           hydra_pair_t* pairs_out, int32_t max_pairs, int32_t* n_pairs_out,
                           int64_t* part_rows_out, int32_t* rank_out, int32_t* step_out)
{
    if (n_seqs < 0 || (n_seqs > 0 && !cu) || !n_pairs_out || !part_rows_out || max_pairs < 0 ||
        (max_pairs > 0 && !pairs_out))
        return HYDRA_ERR_INVALID_ARG;
    if (n_seqs > 0 && cu[0] != 0) return HYDRA_ERR_INVALID_ARG;
    int64_t n_pairs = 0, part_rows = 0;
    int32_t group = 0;
    for (int32_t b = 0; b < n_seqs; ++b) {
        const int64_t len = int64_t{cu[b + 1]} - cu[b];
        const int32_t ring = cp_r_host ? cp_r_host[b] : cp_r_all;
        if (len < 0 || ring < 0 || ring > 4096) return HYDRA_ERR_INVALID_ARG;
        const int32_t n_c = ring == 0 ? 1 : 2 * ring;
        auto edge = [&](int32_t c) { return static_cast<int32_t>(c * len / n_c); };
        auto owner = [&](int32_t c) { return ring == 0 ? 0 : (c < ring ? c : n_c - 1 - c); };
        for (int32_t qc = 0; qc < n_c; ++qc) {
            const int32_t qs = edge(qc), ql = edge(qc + 1) - qs;
            if (ql == 0) continue;
            int32_t in_group = 0;
            for (int32_t kc = 0; kc <= qc; ++kc)
                if (edge(kc + 1) - edge(kc) > 0) ++in_group;
            for (int32_t kc = 0; kc <= qc; ++kc) {
                const int32_t ks = edge(kc), kl = edge(kc + 1) - ks;
                if (kl == 0) continue;
                if (n_pairs < max_pairs) {
                    hydra_pair_t& p = pairs_out[n_pairs];
                    p.seq = b; p.q_start = qs; p.q_len = ql; p.k_start = ks; p.k_len = kl;
                    p.group = group; p.flags = 0;
                    p.part_row = in_group > 1 ? static_cast<int32_t>(part_rows) : -1;
                    if (rank_out) rank_out[n_pairs] = owner(qc);
                    if (step_out) {
                        const int32_t m = ring > 0 ? ring : 1;
                        step_out[n_pairs] = ((owner(qc) - owner(kc)) % m + m) % m;
                    }
                }
                if (in_group > 1) part_rows += ql;
                ++n_pairs;
            }
            ++group;
        }
    }
    if (n_pairs > INT32_MAX || part_rows > INT32_MAX) return HYDRA_ERR_UNSUPPORTED;
    *n_pairs_out = static_cast<int32_t>(n_pairs);
    *part_rows_out = part_rows;
    return n_pairs > max_pairs ? HYDRA_ERR_WORKSPACE_TOO_SMALL : HYDRA_OK;
}

namespace {
std::atomic<uint64_t> g_ds_limit_bytes{uint64_t{4} << 30};

// smallest scratch the banded backward is worth running with
constexpr uint64_t kMinBandBytes = uint64_t{1} << 20;
// Band scratch: a byte count, 0 (bands off) or HYDRA_BAND_AUTO: as much as the dS limit, for problems whose whole dS buffer
// is at most 16 times that and whose longest sequence's own is at most 7 times. The longer a sequence, the fewer of its key
// tiles a band holds, all nearly as long: 16 to 21 at 48K to 64K tokens, two waves of work items of which the second is
// half empty, and beside the stores of dS that costs more than the recomputation it saves. How many sequences there are
// costs nothing. Backward in bands of 4 GiB / recomputing, ms, 16 heads, one sequence: 28000 tokens (2.9 times the limit) 10.4 /
// 11.2, 36000 (4.9) 18.5 / 18.7, 40000 (6.0) 22.7 / 22.9, 44000 (7.2) 28.7 / 27.8, 49152 (9.0) 35.3 / 34.4, 64K (16) 65.1 /
// 61.3; several: ten of 16384 (10.1, each 1.0) 36.9 / 39.2, fourteen 51.5 / 55.5, forty of 8192 39.3 / 41.3, two of 40000
// (12, each 6.0) 45.9 / 46.1; 32 heads, four of 16384 (8.1, each 2.0) 29.7 / 31.3.
std::atomic<uint64_t> g_band_bytes{HYDRA_BAND_AUTO};
constexpr uint64_t kAutoBandsMax = 16, kAutoBandsLongest = 7;
// blocks per head of the dS of the sequence that has most of them
int64_t longest_ds_blocks(const Problem& pb, int causal)
{
    std::vector<int64_t> blocks(pb.n_seqs, 0);
    for (const auto& p : pb.pairs)
        if (p.q_len > 0 && p.k_len > 0)
            blocks[p.seq] += ds_rowstart(ds_geom(p.q_len, p.q_start - p.k_start, causal), (p.k_len + TILE - 1) / TILE);
    return blocks.empty() ? 0 : *std::max_element(blocks.begin(), blocks.end());
}
uint64_t band_scratch_for(const Problem& pb, int causal, int64_t head_blocks)
{
    const uint64_t set = g_band_bytes.load();
    if (set != HYDRA_BAND_AUTO) return set;
    if (head_blocks <= 0) return 0;
    const uint64_t limit = g_ds_limit_bytes.load();
    const uint64_t block = static_cast<uint64_t>(pb.h) * DS_BLOCK_BYTES;
    const bool bands = limit >= kMinBandBytes && head_blocks * block <= kAutoBandsMax * limit &&
                       longest_ds_blocks(pb, causal) * block <= kAutoBandsLongest * limit;
    return bands ? limit : 0;
}

size_t bwd_acc_bytes(const Problem& pb)
{
    return align_up(static_cast<size_t>(pb.Tq) * pb.h * pb.dqk * sizeof(float), 1024);
}
size_t bwd_kv_acc_bytes(const Problem& pb, int32_t n_kv_heads)
{
    return align_up(static_cast<size_t>(pb.Tk) * n_kv_heads * (pb.dqk + D_V) * sizeof(float), 1024);
}
size_t bwd_base_bytes(const Problem& pb)
{
    return align_up(kStatusBytes + align_up(static_cast<size_t>(pb.Tq) * pb.h * sizeof(float), 256), 1024);
}
// bytes of the dS hand-off buffer, or 0 if it is not to be used (layout not possible, or over the limit)
size_t bwd_ds_bytes(int64_t head_blocks, int32_t n_heads, uint64_t limit)
{
    if (head_blocks <= 0) return 0;
    const uint64_t bytes = static_cast<uint64_t>(head_blocks) * n_heads * DS_BLOCK_BYTES;
    return bytes <= limit ? static_cast<size_t>(bytes) : 0;
}
}  // namespace

void hydra_set_bwd_scratch_limit(uint64_t bytes) { g_ds_limit_bytes.store(bytes); }
void hydra_set_bwd_band_scratch(uint64_t bytes) { g_band_bytes.store(bytes); }

size_t hydra_workspace_bytes(int32_t which, const int32_t* cu, int32_t n_seqs, int32_t n_heads,
                             const hydra_pair_t* pairs, int32_t n_pairs)
{
    return hydra_workspace_bytes_gqa(which, cu, n_seqs, n_heads, n_heads, pairs, n_pairs);
}

size_t hydra_workspace_bytes_gqa(int32_t which, const int32_t* cu, int32_t n_seqs, int32_t n_heads,
                                 int32_t n_kv_heads, const hydra_pair_t* pairs, int32_t n_pairs)
{
    return hydra_workspace_bytes_dims(which, cu, n_seqs, n_heads, n_kv_heads, D_QK, D_V, pairs, n_pairs);
}

size_t hydra_workspace_bytes_dims(int32_t which, const int32_t* cu, int32_t n_seqs, int32_t n_heads,
                                  int32_t n_kv_heads, int32_t d_qk, int32_t d_v, const hydra_pair_t* pairs,
                                  int32_t n_pairs)
{
    Problem pb;
    if (make_problem(cu, n_seqs, n_heads, pairs, n_pairs, pb) != HYDRA_OK) return 0;
    if (n_kv_heads < 1 || n_heads % n_kv_heads || !kernel_set(d_qk, d_v)) return 0;
    pb.dqk = d_qk;
    // sized for a causal call, whose chunks may be joined, and for the pairs as they are
    auto bwd_bytes = [&](const Problem& pr) -> size_t {
        const size_t base = bwd_base_bytes(pr);
        const int64_t head_blocks = ds_layout(pr, 1, nullptr);
        const size_t ds = bwd_ds_bytes(head_blocks, n_heads, g_ds_limit_bytes.load());
        // one-shot grouped-query backward: fp32 dk, dv of the KV heads, then the dS buffer if within the limit
        if (n_kv_heads != n_heads) return base + bwd_kv_acc_bytes(pr, n_kv_heads) + ds;
        // D, plus the dS hand-off buffer when it stays within the limit
        if (ds) return base + ds;
        // over the limit: the banded form, if switched on, wants an fp32 dq and its scratch
        const uint64_t band = band_scratch_for(pr, 1, head_blocks);
        if (head_blocks > 0 && band >= kMinBandBytes) {
            const uint64_t full = static_cast<uint64_t>(head_blocks) * n_heads * DS_BLOCK_BYTES;
            return base + bwd_acc_bytes(pr) + static_cast<size_t>(std::min(band, full));
        }
        return base;
    };
    switch (which) {
        case HYDRA_WS_FWD:
        case HYDRA_WS_MERGE: return kStatusBytes;
        case HYDRA_WS_BWD: {
            const size_t as_given = bwd_bytes(pb);
            return join_chunks(pb, 1) ? std::max(as_given, bwd_bytes(pb)) : as_given;
        }
        default: return 0;
    }
}

namespace {
int32_t fwd_core(Problem& pb, const void* q, const void* k, const void* v, int32_t n_kv_heads, int32_t causal,
                 float softmax_scale, void* out, float* lse, void* o_part, float* lse_part, int64_t part_rows,
                 void* workspace, size_t workspace_bytes, void* cuda_stream);
}

int32_t hydra_attn_fwd(const void* q, const void* k, const void* v, const int32_t* cu, int32_t n_seqs,
                       int32_t n_heads, const hydra_pair_t* pairs, int32_t n_pairs, int32_t causal,
                       float softmax_scale, void* out, float* lse, void* o_part, float* lse_part,
                       int64_t part_rows, void* workspace, size_t workspace_bytes, void* cuda_stream)
{
    return hydra_attn_fwd_gqa(q, k, v, cu, n_seqs, n_heads, n_heads, pairs, n_pairs, causal, softmax_scale, out, lse,
                              o_part, lse_part, part_rows, workspace, workspace_bytes, cuda_stream);
}

int32_t hydra_attn_fwd_gqa(const void* q, const void* k, const void* v, const int32_t* cu, int32_t n_seqs,
                           int32_t n_heads, int32_t n_kv_heads, const hydra_pair_t* pairs, int32_t n_pairs,
                           int32_t causal, float softmax_scale, void* out, float* lse, void* o_part,
                           float* lse_part, int64_t part_rows, void* workspace, size_t workspace_bytes,
                           void* cuda_stream)
{
    return hydra_attn_fwd_dims(q, k, v, cu, n_seqs, n_heads, n_kv_heads, D_QK, D_V, pairs, n_pairs, causal,
                               softmax_scale, out, lse, o_part, lse_part, part_rows, workspace, workspace_bytes,
                               cuda_stream);
}

int32_t hydra_attn_fwd_dims(const void* q, const void* k, const void* v, const int32_t* cu, int32_t n_seqs,
                            int32_t n_heads, int32_t n_kv_heads, int32_t d_qk, int32_t d_v,
                            const hydra_pair_t* pairs, int32_t n_pairs, int32_t causal, float softmax_scale,
                            void* out, float* lse, void* o_part, float* lse_part, int64_t part_rows,
                            void* workspace, size_t workspace_bytes, void* cuda_stream)
{
    if (!kernel_set(d_qk, d_v)) return HYDRA_ERR_UNSUPPORTED;
    Problem pb;
    if (int32_t s = make_problem(cu, n_seqs, n_heads, pairs, n_pairs, pb)) return s;
    pb.dqk = d_qk;
    return fwd_core(pb, q, k, v, n_kv_heads, causal, softmax_scale, out, lse, o_part, lse_part, part_rows, workspace,
                    workspace_bytes, cuda_stream);
}

int32_t hydra_attn_fwd_local(const void* q, const void* k, const void* v, const int32_t* cu, int32_t n_seqs,
                             int32_t n_heads, int32_t n_kv_heads, int32_t d_qk, int32_t d_v,
                             const hydra_chunk_t* q_chunks, int32_t n_q_chunks, int64_t q_rows,
                             const hydra_chunk_t* kv_chunks, int32_t n_kv_chunks, int64_t kv_rows,
                             const hydra_pair_t* pairs, int32_t n_pairs, int32_t causal, float softmax_scale,
                             void* out, float* lse, void* o_part, float* lse_part, int64_t part_rows,
                             void* workspace, size_t workspace_bytes, void* cuda_stream)
{
    if (!kernel_set(d_qk, d_v)) return HYDRA_ERR_UNSUPPORTED;
    Problem pb;
    if (int32_t s = make_problem_local(cu, n_seqs, n_heads, q_chunks, n_q_chunks, q_rows, kv_chunks, n_kv_chunks,
                                       kv_rows, pairs, n_pairs, pb))
        return s;
    pb.dqk = d_qk;
    return fwd_core(pb, q, k, v, n_kv_heads, causal, softmax_scale, out, lse, o_part, lse_part, part_rows, workspace,
                    workspace_bytes, cuda_stream);
}

namespace {
// A number that no other call of this process has and that a workspace holds by chance once in 2^64: the calls counted from a
// start of the process's own, in steps and mixed as in splitmix64 (Steele, Lea and Flood, 2014), a one-to-one function. Not 0.
uint64_t next_call_tag()
{
    static std::atomic<uint64_t> calls{static_cast<uint64_t>(std::chrono::system_clock::now().time_since_epoch().count()) ^
                                       static_cast<uint64_t>(std::chrono::steady_clock::now().time_since_epoch().count()) << 20};
    uint64_t x;
    do {
        x = calls.fetch_add(0x9e3779b97f4a7c15ull);
        x = (x ^ (x >> 30)) * 0xbf58476d1ce4e5b9ull;
        x = (x ^ (x >> 27)) * 0x94d049bb133111ebull;
        x ^= x >> 31;
    } while (x == 0);
    return x;
}

int32_t fwd_core(Problem& pb, const void* q, const void* k, const void* v, int32_t n_kv_heads, int32_t causal,
                 float softmax_scale, void* out, float* lse, void* o_part, float* lse_part, int64_t part_rows,
                 void* workspace, size_t workspace_bytes, void* cuda_stream)
{
    const int32_t n_heads = pb.h;
    const KernelSet* ks = kernel_set(pb.dqk, D_V);
    if (n_kv_heads < 1 || n_heads % n_kv_heads) return HYDRA_ERR_INVALID_ARG;
    pb.kv_group = n_heads / n_kv_heads;
    pb.fwd_short_set = g_fwd_short_len.load();          // once: another thread may set it meanwhile
    if (!(softmax_scale > 0.f) || !std::isfinite(softmax_scale)) return HYDRA_ERR_INVALID_ARG;
    if (!workspace || !aligned16(workspace)) return HYDRA_ERR_INVALID_ARG;
    if (workspace_bytes < kStatusBytes) return HYDRA_ERR_WORKSPACE_TOO_SMALL;
    bool any_part = false, any_direct = false;
    for (const auto& p : pb.pairs) (p.part_row >= 0 ? any_part : any_direct) = true;
    if (pb.T > 0 && (!q || !k || !v || !aligned16(q) || !aligned16(k) || !aligned16(v))) return HYDRA_ERR_INVALID_ARG;
    if (any_direct && (!out || !lse || !aligned16(out) || !aligned16(lse))) return HYDRA_ERR_INVALID_ARG;
    if (any_part && (!o_part || !lse_part || !aligned16(o_part) || !aligned16(lse_part) || part_rows <= 0))
        return HYDRA_ERR_INVALID_ARG;
    if (int32_t s = check_part_rows(pb, part_rows)) return s;
    cudaStream_t stream = static_cast<cudaStream_t>(cuda_stream);
    int sms = 0;
    if (int32_t s = device_info(&sms)) return s;
    if (pb.pairs.empty()) return HYDRA_OK;

    PlanLease lease;
    if (int32_t s = lease.acquire(HYDRA_WS_FWD, pb, causal != 0, stream)) return s;
    const Plan* plan = &lease.plan();
    if (plan->n_items == 0 && plan->n_items2 == 0) return HYDRA_OK;
    // One item per SM before any SM gets two, or what the items have been dealt out to.
    const int short_grid = plan->halves ? plan->short_grid : std::min(sms, plan->n_items2);
    FwdParams fp{};
    uint64_t call_tag = 0;
    // With no more items than slots nothing is popped from the queue, and the block at the workspace's start need not be
    // cleared (one launch less: four sequences of 7 to 300 tokens, forward 11.5 -> 9.4 us). Not where the launches are
    // recorded: every replay would have the number of the first.
    cudaStreamCaptureStatus capturing = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(stream, &capturing) != cudaSuccess) return HYDRA_ERR_CUDA;
    if (capturing == cudaStreamCaptureStatusNone && plan->n_items == 0 && (plan->halves || plan->n_items2 <= 2 * short_grid)) {
        call_tag = next_call_tag();
    } else if (launch_reset(static_cast<StatusBlock*>(workspace), false, stream) != cudaSuccess) {
        return HYDRA_ERR_CUDA;
    }
    fp.pairs = lease.at<PairDev>(plan->off_pairs);
    fp.items = lease.at<FwdItem>(plan->off_items);
    fp.n_items = plan->n_items;
    fp.short_items = lease.at<FwdShortItem>(plan->off_items2);
    fp.n_short = plan->n_items2;
    fp.early_pops = plan->early_pops;
    fp.out = out; fp.lse = lse; fp.o_part = o_part; fp.lse_part = lse_part;
    fp.T = pb.Tq; fp.part_rows = part_rows; fp.h = n_heads; fp.causal = causal != 0;
    fp.kv_group = n_heads / n_kv_heads;
    fp.scale_log2 = softmax_scale * 1.4426950408889634f;
    fp.status = static_cast<StatusBlock*>(workspace);
    fp.wait_limit_ns = g_wait_limit_ns.load();
    fp.debug_stall_ns = g_debug_stall_ns[HYDRA_STALL_FWD].load();
    CUtensorMap mq, mk;
    if (make_map(&mq, q, pb.Tq, n_heads, pb.dqk, TILE) || make_map(&mk, k, pb.Tk, n_kv_heads, pb.dqk, SUB))
        return HYDRA_ERR_CUDA;
    if (plan->n_items > 0) {
        // long pairs, on CTA pairs: each CTA of a pair stages 64 kv rows of K (box of 64 rows) and 64 value
        // columns of V
        const int n_clusters = ks->fwd_max_clusters();    // CTA pairs resident at once: the persistent grid
        if (n_clusters < 1) return HYDRA_ERR_CUDA;
        CUtensorMap mv;
        if (make_map(&mv, v, pb.Tk, n_kv_heads, D_V, TILE)) return HYDRA_ERR_CUDA;
        ScopedKernelTimer timer(K_FWD, stream);
        if (ks->launch_fwd(mq, mk, mv, fp, n_clusters, stream) != cudaSuccess) return HYDRA_ERR_CUDA;
        g_launches += 1;
    }
    if (plan->n_items2 > 0) {
        // short pairs: one CTA per SM with two work items in flight, K and V in boxes of 64 keys
        CUtensorMap mv_sub;
        if (make_map(&mv_sub, v, pb.Tk, n_kv_heads, D_V, FWD_SHORT_KEYS)) return HYDRA_ERR_CUDA;
        ScopedKernelTimer timer(K_FWD, stream);
        const FwdSeg* segs = plan->n_segs ? lease.at<FwdSeg>(plan->off_segs) : nullptr;
        if (ks->launch_fwd_short(mq, mk, mv_sub, fp, segs, call_tag, plan->halves != 0, short_grid, stream) != cudaSuccess)
            return HYDRA_ERR_CUDA;
        g_launches += 1;
    }
    lease.release();                                   // the tables have their reader on record
    prefetch_plans(pb, causal != 0, any_part);
    return HYDRA_OK;
}
}  // namespace

namespace {
int32_t merge_impl(const void* o_part, const float* lse_part, int64_t part_rows, const int32_t* cu,
                   int32_t n_seqs, int32_t n_heads, const hydra_pair_t* pairs, int32_t n_pairs, void* out,
                   float* lse, void* workspace, size_t workspace_bytes, void* cuda_stream, int32_t accumulate);
int32_t merge_core(const Problem& pb, const void* o_part, const float* lse_part, int64_t part_rows, void* out,
                   float* lse, void* workspace, size_t workspace_bytes, void* cuda_stream, int32_t accumulate);
}

int32_t hydra_lse_merge(const void* o_part, const float* lse_part, int64_t part_rows, const int32_t* cu,
                        int32_t n_seqs, int32_t n_heads, const hydra_pair_t* pairs, int32_t n_pairs,
                        void* out, float* lse, void* workspace, size_t workspace_bytes, void* cuda_stream)
{
    return merge_impl(o_part, lse_part, part_rows, cu, n_seqs, n_heads, pairs, n_pairs, out, lse, workspace,
                      workspace_bytes, cuda_stream, 0);
}

int32_t hydra_lse_merge_accumulate(const void* o_part, const float* lse_part, int64_t part_rows,
                                   const int32_t* cu, int32_t n_seqs, int32_t n_heads, const hydra_pair_t* pairs,
                                   int32_t n_pairs, void* out, float* lse, void* workspace, size_t workspace_bytes,
                                   void* cuda_stream)
{
    return merge_impl(o_part, lse_part, part_rows, cu, n_seqs, n_heads, pairs, n_pairs, out, lse, workspace,
                      workspace_bytes, cuda_stream, 1);
}

namespace {
int32_t merge_impl(const void* o_part, const float* lse_part, int64_t part_rows, const int32_t* cu,
                   int32_t n_seqs, int32_t n_heads, const hydra_pair_t* pairs, int32_t n_pairs, void* out,
                   float* lse, void* workspace, size_t workspace_bytes, void* cuda_stream, int32_t accumulate)
{
    Problem pb;
    if (int32_t s = make_problem(cu, n_seqs, n_heads, pairs, n_pairs, pb)) return s;
    return merge_core(pb, o_part, lse_part, part_rows, out, lse, workspace, workspace_bytes, cuda_stream, accumulate);
}

int32_t merge_core(const Problem& pb, const void* o_part, const float* lse_part, int64_t part_rows, void* out,
                   float* lse, void* workspace, size_t workspace_bytes, void* cuda_stream, int32_t accumulate)
{
    const int32_t n_heads = pb.h;
    if (!workspace || !aligned16(workspace)) return HYDRA_ERR_INVALID_ARG;
    if (workspace_bytes < kStatusBytes) return HYDRA_ERR_WORKSPACE_TOO_SMALL;
    bool any_part = false;
    for (const auto& p : pb.pairs) any_part |= (p.part_row >= 0 && p.q_len > 0);
    if (any_part && (!o_part || !lse_part || !out || !lse || !aligned16(o_part) || !aligned16(lse_part) ||
        !aligned16(out) || !aligned16(lse) || part_rows <= 0))
        return HYDRA_ERR_INVALID_ARG;
    if (int32_t s = check_part_rows(pb, part_rows)) return s;
    if (!any_part) return HYDRA_OK;
    cudaStream_t stream = static_cast<cudaStream_t>(cuda_stream);
    int sms = 0;
    if (int32_t s = device_info(&sms)) return s;
    PlanLease lease;
    if (int32_t s = lease.acquire(HYDRA_WS_MERGE, pb, 0, stream)) return s;
    const Plan* plan = &lease.plan();
    MergeParams mp{};
    mp.groups = lease.at<MergeGroup>(plan->off_groups);
    mp.lists = lease.at<int32_t>(plan->off_lists);
    mp.items = lease.at<MergeItem>(plan->off_items);
    mp.n_items = plan->n_items;
    mp.o_part = o_part; mp.lse_part = lse_part; mp.out = out; mp.lse = lse;
    mp.T = pb.Tq; mp.part_rows = part_rows; mp.h = n_heads;
    mp.accumulate = accumulate;
    mp.max_parts = plan->n_items2;
    if (launch_merge_counted(mp, stream) != cudaSuccess) return HYDRA_ERR_CUDA;
    return HYDRA_OK;
}
}  // namespace

namespace {
struct BwdTensors {
    const void *q, *k, *v, *out, *dout;
    const float* lse;
    void *dq, *dk, *dv;                 // bf16 outputs or fp32 accumulators
};

// Where dk and dv may be summed in fp32 when several key-side items share their rows (grouped query heads).
struct KvSums {
    float *dk, *dv;
    size_t bytes;                       // dk's and dv's together
    bool used;                          // set by bwd_run: the sums are there, the outputs are not written yet
};

// One backward over the pairs of `pb`: D = rowsum(dO*O) (if `first`), the key-side kernel, the query-side
// kernel. dq and dk/dv are bf16 outputs or fp32 accumulators, each by its own flag. `ds` / `ds_room` is
// where a dS hand-off buffer may go. `sums`: where dk and dv are summed if no item of the plan holds all query heads of a
// K / V head (null: the outputs need no such sums). With `first` false the status block keeps its flags and only the
// work-queue counters are cleared. `halves_of_call` is key_tiles_halved of the whole call, -1 if `pb` is all of it.
int32_t bwd_run(const Problem& pb, int32_t n_kv_heads, int32_t causal, float softmax_scale, const BwdTensors& t,
                KvSums* sums, bool accumulate_dq, bool accumulate_dkv, void* workspace, uint8_t* ds, size_t ds_room,
                uint64_t ds_limit, bool first, int halves_of_call, int sms, cudaStream_t stream)
{
    const int32_t n_heads = pb.h;
    const KernelSet* ks = kernel_set(pb.dqk, D_V);
    if (!ks) return HYDRA_ERR_UNSUPPORTED;
    PlanLease lease;
    if (int32_t s = lease.acquire(HYDRA_WS_BWD, pb, causal != 0, stream)) return s;
    const Plan* plan = &lease.plan();

    float* dsum = reinterpret_cast<float*>(static_cast<uint8_t*>(workspace) + kStatusBytes);
    CUtensorMap mk, mv, mq_sub, mdo_sub;
    if (make_map(&mk, t.k, pb.Tk, n_kv_heads, pb.dqk, TILE) || make_map(&mv, t.v, pb.Tk, n_kv_heads, D_V, TILE) ||
        make_map(&mq_sub, t.q, pb.Tq, n_heads, pb.dqk, SUB) || make_map(&mdo_sub, t.dout, pb.Tq, n_heads, D_V, SUB))
        return HYDRA_ERR_CUDA;
    if (sums) sums->used = plan->item_heads != n_heads / n_kv_heads;
    const bool summed = sums && sums->used;
    if (first) {
        ScopedKernelTimer timer(K_PREP, stream);
        if (launch_bwd_prep(t.dout, t.out, dsum, pb.Tq, n_heads, static_cast<StatusBlock*>(workspace), summed ? sums->dk : nullptr,
                            summed ? sums->bytes : 0, stream) != cudaSuccess)
            return HYDRA_ERR_CUDA;
        g_launches += 1;
    } else if (launch_reset(static_cast<StatusBlock*>(workspace), true, stream) != cudaSuccess) {
        return HYDRA_ERR_CUDA;
    }

    BwdParams bp{};
    bp.pairs = lease.at<PairDev>(plan->off_pairs);
    bp.lse = t.lse; bp.dsum = dsum; bp.dq = t.dq; bp.dk = t.dk; bp.dv = t.dv;
    bp.T = pb.Tq; bp.h = n_heads; bp.causal = causal != 0;
    bp.kv_group = n_heads / n_kv_heads;
    bp.scale = softmax_scale; bp.scale_log2 = softmax_scale * 1.4426950408889634f;
    bp.status = static_cast<StatusBlock*>(workspace);
    bp.wait_limit_ns = g_wait_limit_ns.load();
    // dS hand-off: the key-side kernel leaves dS^T in the workspace and the query-side kernel only
    // multiplies it with K, if the buffer fits the room given and the limit set
    const size_t ds_bytes = bwd_ds_bytes(plan->ds_head_blocks, n_heads, ds_limit);
    const bool hand_off = ds_bytes > 0 && ds != nullptr && ds_room >= ds_bytes;
    if (hand_off) {
        bp.ds = ds;
        bp.ds_head_blocks = plan->ds_head_blocks;
    }
    if (plan->n_items2 > 0) {
        bp.lists = lease.at<int32_t>(plan->off_lists2);
        bp.items = lease.at<GroupItem>(plan->off_items2);
        bp.n_items = plan->n_items2;
        bp.item_heads = plan->item_heads;
        bp.accumulate = accumulate_dkv || summed ? 1 : 0;
        if (summed) { bp.dk = sums->dk; bp.dv = sums->dv; }
        bp.debug_stall_ns = g_debug_stall_ns[HYDRA_STALL_BWD_DKV].load();
        ScopedKernelTimer timer(K_DKV, stream);
        const bool halves = halves_of_call >= 0 ? halves_of_call != 0 : plan->halves != 0;
        if (ks->launch_bwd_dkv(mq_sub, mk, mv, mdo_sub, bp, halves, halves ? 2 * bp.n_items : std::min(sms, bp.n_items),
                               stream) != cudaSuccess)
            return HYDRA_ERR_CUDA;
        g_launches += 1;
    }
    if (plan->n_items > 0) {
        bp.lists = lease.at<int32_t>(plan->off_lists);
        bp.items = lease.at<GroupItem>(plan->off_items);
        bp.n_items = plan->n_items;
        bp.accumulate = accumulate_dq ? 1 : 0;
        bp.debug_stall_ns = g_debug_stall_ns[HYDRA_STALL_BWD_DQ].load();
        ScopedKernelTimer timer(K_DQ, stream);
        const int grid = std::min(sms, bp.n_items);
        CUtensorMap mq, mdo;                           // whole tiles of q and dO: the recomputing form only
        if (!hand_off && (make_map(&mq, t.q, pb.Tq, n_heads, pb.dqk, TILE) || make_map(&mdo, t.dout, pb.Tq, n_heads, D_V, TILE)))
            return HYDRA_ERR_CUDA;
        const cudaError_t e = hand_off ? ks->launch_bwd_dq_from_ds(mk, bp, grid, stream)
                                       : ks->launch_bwd_dq(mq, mk, mv, mdo, bp, grid, stream);
        if (e != cudaSuccess)
            return HYDRA_ERR_CUDA;
        g_launches += 1;
    }
    return HYDRA_OK;
}

// Bands of key rows for a backward whose dS buffer is over the limit: every band is a list of pairs
// clipped to some 128-row tiles of their key chunk (and, under the causal mask, to the query rows that
// see those keys), chosen so that the band's own dS buffer fits `room`. A key tile lies in one band, so
// dk and dv of a band are final; dq sums over the bands. Empty if some band cannot be made to fit, if a
// clipped pair would have no visible position, or if the clipped chunks would break the
// identical-or-disjoint rule.
std::vector<std::vector<hydra_pair_t>> make_bands(const Problem& pb, int32_t causal, size_t room)
{
    std::vector<std::vector<hydra_pair_t>> bands;
    // distinct key ranges, in order
    std::vector<Range> ranges;
    for (const auto& p : pb.pairs)
        if (p.q_len > 0 && p.k_len > 0) ranges.push_back(Range{p.seq, p.k_start, p.k_len});
    std::sort(ranges.begin(), ranges.end(), range_less);
    ranges.erase(std::unique(ranges.begin(), ranges.end(),
                             [](const Range& a, const Range& b) {
                                 return a.seq == b.seq && a.start == b.start && a.len == b.len;
                             }), ranges.end());
    // appends the pairs of key range r clipped to its keys [c0, c1); false if one of them sees nothing
    auto clip = [&](const Range& r, int32_t c0, int32_t c1, std::vector<hydra_pair_t>& into) {
        for (const auto& p : pb.pairs) {
            if (p.seq != r.seq || p.k_start != r.start || p.k_len != r.len || p.q_len <= 0) continue;
            hydra_pair_t c = p;
            c.k_start = p.k_start + c0;
            c.k_len = c1 - c0;
            if (causal) {                                  // query rows before the first key see nothing
                const int32_t first = std::max(p.q_start, c.k_start);
                if (first >= p.q_start + p.q_len) return false;
                c.q_len = p.q_start + p.q_len - first;
                c.q_start = first;
            }
            c.part_row = -1;
            c.group = static_cast<int32_t>(into.size());
            c.flags = 0;
            into.push_back(c);
        }
        return true;
    };
    Problem probe;
    probe.cu = pb.cu; probe.n_seqs = pb.n_seqs; probe.h = pb.h; probe.T = pb.T; probe.Tq = pb.Tq; probe.Tk = pb.Tk; probe.dqk = pb.dqk;
    auto fits = [&](const std::vector<hydra_pair_t>& pairs) {
        probe.pairs = pairs;
        return bwd_ds_bytes(ds_layout(probe, causal, nullptr), pb.h, room) > 0;
    };
    std::vector<hydra_pair_t> cur;
    for (const Range& r : ranges) {
        const int32_t n = (r.len + TILE - 1) / TILE;
        int32_t i = 0;
        while (i < n) {
            // the most key tiles [i, j) of this range that still fit beside what the band holds
            int32_t lo = i, hi = n;
            while (lo < hi) {
                const int32_t mid = lo + (hi - lo + 1) / 2;
                std::vector<hydra_pair_t> trial = cur;
                if (clip(r, i * TILE, std::min(r.len, mid * TILE), trial) && fits(trial)) lo = mid;
                else hi = mid - 1;
            }
            if (lo == i) {
                if (cur.empty()) return {};                // one tile column alone does not fit
                bands.push_back(std::move(cur));
                cur.clear();
                continue;
            }
            if (!clip(r, i * TILE, std::min(r.len, lo * TILE), cur)) return {};
            i = lo;
        }
    }
    if (!cur.empty()) bands.push_back(std::move(cur));
    for (const auto& band : bands) {
        std::vector<Range> rq, rk;
        for (const auto& p : band) {
            rq.push_back(Range{p.seq, p.q_start, p.q_len});
            rk.push_back(Range{p.seq, p.k_start, p.k_len});
        }
        if (check_identical_or_disjoint(rq) || check_identical_or_disjoint(rk)) return {};
    }
    return bands;
}

// Token rows [first, end) that the listed ranges cover, sorted, with ranges that touch or overlap joined: a
// packed batch whose chunks tile its sequences is one run, so a cast over it is one launch (a batch of 230
// short sequences used to take 460 launches of a few microseconds each).
std::vector<std::pair<size_t, size_t>> covered_rows(const Problem& pb, bool key_side)
{
    std::vector<std::pair<size_t, size_t>> rows;
    for (const auto& p : pb.pairs) {
        if (p.q_len <= 0 || p.k_len <= 0) continue;
        const size_t first = static_cast<size_t>(key_side ? pb.k_row(p.seq, p.k_start) : pb.q_row(p.seq, p.q_start));
        rows.emplace_back(first, first + static_cast<size_t>(key_side ? p.k_len : p.q_len));
    }
    std::sort(rows.begin(), rows.end());
    std::vector<std::pair<size_t, size_t>> runs;
    for (const auto& r : rows) {
        if (!runs.empty() && r.first <= runs.back().second) runs.back().second = std::max(runs.back().second, r.second);
        else runs.push_back(r);
    }
    return runs;
}

int32_t bwd_core(Problem& pb, const void* q, const void* k, const void* v, const void* out, const float* lse,
                 const void* dout, int32_t causal, float softmax_scale, void* dq, void* dk, void* dv, bool accumulate,
                 void* workspace, size_t workspace_bytes, void* cuda_stream, int32_t n_kv_heads);

int32_t bwd_impl(const void* q, const void* k, const void* v, const void* out, const float* lse,
                 const void* dout, const int32_t* cu, int32_t n_seqs, int32_t n_heads,
                 const hydra_pair_t* pairs, int32_t n_pairs, int32_t causal, float softmax_scale,
                 void* dq, void* dk, void* dv, bool accumulate, void* workspace, size_t workspace_bytes,
                 void* cuda_stream, int32_t n_kv_heads, int32_t d_qk = D_QK, int32_t d_v = D_V)
{
    if (!kernel_set(d_qk, d_v)) return HYDRA_ERR_UNSUPPORTED;
    Problem pb;
    if (int32_t s = make_problem(cu, n_seqs, n_heads, pairs, n_pairs, pb)) return s;
    pb.dqk = d_qk;
    return bwd_core(pb, q, k, v, out, lse, dout, causal, softmax_scale, dq, dk, dv, accumulate, workspace,
                    workspace_bytes, cuda_stream, n_kv_heads);
}

int32_t bwd_core(Problem& pb, const void* q, const void* k, const void* v, const void* out, const float* lse,
                 const void* dout, int32_t causal, float softmax_scale, void* dq, void* dk, void* dv, bool accumulate,
                 void* workspace, size_t workspace_bytes, void* cuda_stream, int32_t n_kv_heads)
{
    const int32_t n_heads = pb.h;
    if (n_kv_heads < 1 || n_heads % n_kv_heads) return HYDRA_ERR_INVALID_ARG;
    pb.kv_group = n_heads / n_kv_heads;
    if (!(softmax_scale > 0.f) || !std::isfinite(softmax_scale)) return HYDRA_ERR_INVALID_ARG;
    if (!workspace || !aligned16(workspace)) return HYDRA_ERR_INVALID_ARG;
    const size_t need = kStatusBytes + align_up(static_cast<size_t>(pb.Tq) * n_heads * sizeof(float), 256);
    if (workspace_bytes < need) return HYDRA_ERR_WORKSPACE_TOO_SMALL;
    const size_t ds_off = bwd_base_bytes(pb);
    if (pb.T == 0 || pb.pairs.empty()) return HYDRA_OK;
    const void* ptrs[] = {q, k, v, out, lse, dout, dq, dk, dv};
    for (const void* p : ptrs)
        if (!p || !aligned16(p)) return HYDRA_ERR_INVALID_ARG;
    {
        std::vector<Range> rq, rk;
        for (const auto& p : pb.pairs) {
            if (p.q_len > 0) rq.push_back(Range{p.seq, p.q_start, p.q_len});
            if (p.k_len > 0) rk.push_back(Range{p.seq, p.k_start, p.k_len});
        }
        if (check_identical_or_disjoint(rq) || check_identical_or_disjoint(rk)) return HYDRA_ERR_INVALID_ARG;
    }
    join_chunks(pb, causal);
    cudaStream_t stream = static_cast<cudaStream_t>(cuda_stream);
    int sms = 0;
    if (int32_t s = device_info(&sms)) return s;
    uint8_t* ws = static_cast<uint8_t*>(workspace);
    const BwdTensors t{q, k, v, out, dout, lse, dq, dk, dv};
    const size_t room = workspace_bytes > ds_off ? workspace_bytes - ds_off : 0;

    // One-shot grouped-query form: where no key-side item holds all query heads of a group, they add into one dk / dv row,
    // which only the accumulating epilogue can do: dk, dv are then summed in fp32 in the workspace (cleared by the D =
    // rowsum(dO O) kernel) and rounded at the end. dq (one query head per row) is written as bf16 as usual.
    if (!accumulate && n_kv_heads != n_heads) {
        const size_t kv_bytes = bwd_kv_acc_bytes(pb, n_kv_heads);
        if (room < kv_bytes) return HYDRA_ERR_WORKSPACE_TOO_SMALL;
        KvSums sums{};
        sums.dk = reinterpret_cast<float*>(ws + ds_off);
        sums.dv = sums.dk + static_cast<size_t>(pb.Tk) * n_kv_heads * pb.dqk;
        sums.bytes = kv_bytes;
        if (int32_t s = bwd_run(pb, n_kv_heads, causal, softmax_scale, t, &sums, false, false, workspace,
                                ws + ds_off + kv_bytes, room - kv_bytes, g_ds_limit_bytes.load(), true, -1, sms, stream))
            return s;
        if (!sums.used) return HYDRA_OK;
        const size_t rk = static_cast<size_t>(n_kv_heads) * pb.dqk, rv = static_cast<size_t>(n_kv_heads) * D_V;
        for (const auto& run : covered_rows(pb, true)) {
            const size_t row = run.first, n = run.second - run.first;
            ScopedKernelTimer timer(K_CAST, stream);
            int launches = 0;
            if (launch_grad_cast2(sums.dk + row * rk, static_cast<uint16_t*>(dk) + row * rk, static_cast<int64_t>(n * rk),
                                  sums.dv + row * rv, static_cast<uint16_t*>(dv) + row * rv, static_cast<int64_t>(n * rv),
                                  &launches, stream) != cudaSuccess)
                return HYDRA_ERR_CUDA;
            g_launches += launches;
        }
        return HYDRA_OK;
    }

    // Banded form: the dS buffer of the whole call is over the limit, but the caller has switched the
    // bands on and left room for an fp32 accumulator of dq and a band's scratch. Each band of key rows
    // then runs with its own hand-off: dk and dv of its keys are final, dq is summed in fp32 over the
    // bands and rounded once at the end.
    const size_t acc_bytes = bwd_acc_bytes(pb);
    if (!accumulate && room >= acc_bytes + kMinBandBytes) {
        const int64_t head_blocks = ds_layout(pb, causal, nullptr);
        const uint64_t band_limit = band_scratch_for(pb, causal, head_blocks);
        if (head_blocks > 0 && band_limit >= kMinBandBytes &&
            bwd_ds_bytes(head_blocks, n_heads, g_ds_limit_bytes.load()) == 0) {
            const size_t scratch = static_cast<size_t>(std::min<uint64_t>(band_limit, room - acc_bytes));
            const auto bands = make_bands(pb, causal, scratch);
            if (!bands.empty()) {
                float* dq_acc = reinterpret_cast<float*>(ws + ds_off);
                if (cudaMemsetAsync(dq_acc, 0, acc_bytes, stream) != cudaSuccess) return HYDRA_ERR_CUDA;
                const BwdTensors tb{q, k, v, out, dout, lse, dq_acc, dk, dv};
                Problem band_pb;
                band_pb.cu = pb.cu; band_pb.n_seqs = pb.n_seqs; band_pb.h = pb.h; band_pb.T = pb.T; band_pb.Tq = pb.Tq; band_pb.Tk = pb.Tk; band_pb.dqk = pb.dqk;
                const int halves = key_tiles_halved(pb, causal);
                bool first = true;
                for (const auto& band : bands) {
                    band_pb.pairs = band;
                    if (int32_t s = bwd_run(band_pb, n_heads, causal, softmax_scale, tb, nullptr, true, false, workspace,
                                            ws + ds_off + acc_bytes, scratch, scratch, first, halves, sms, stream))
                        return s;
                    first = false;
                }
                // round the query rows the pairs cover; rows outside every pair stay untouched, as in
                // the one-shot form
                const size_t per_row = static_cast<size_t>(n_heads) * pb.dqk;
                for (const auto& run : covered_rows(pb, false)) {
                    const size_t row = run.first, n = run.second - run.first;
                    ScopedKernelTimer timer(K_CAST, stream);
                    if (launch_grad_cast(dq_acc + row * per_row, static_cast<uint16_t*>(dq) + row * per_row,
                                         static_cast<int64_t>(n * per_row), stream) != cudaSuccess)
                        return HYDRA_ERR_CUDA;
                    g_launches += 1;
                }
                return HYDRA_OK;
            }
        }
    }
    return bwd_run(pb, n_kv_heads, causal, softmax_scale, t, nullptr, accumulate, accumulate, workspace, ws + ds_off, room,
                   g_ds_limit_bytes.load(), true, -1, sms, stream);
}
}  // namespace

int32_t hydra_bwd_bands(const int32_t* cu, int32_t n_seqs, int32_t n_heads, const hydra_pair_t* pairs,
                        int32_t n_pairs, int32_t causal, uint64_t scratch_bytes, hydra_pair_t* pairs_out,
                        int32_t* band_out, int32_t max_pairs, int32_t* n_pairs_out, int32_t* n_bands_out)
{
    if (!n_pairs_out || !n_bands_out || max_pairs < 0 || (max_pairs > 0 && (!pairs_out || !band_out)))
        return HYDRA_ERR_INVALID_ARG;
    Problem pb;
    if (int32_t s = make_problem(cu, n_seqs, n_heads, pairs, n_pairs, pb)) return s;
    join_chunks(pb, causal);
    const auto bands = make_bands(pb, causal, static_cast<size_t>(scratch_bytes));
    int64_t n = 0;
    for (size_t b = 0; b < bands.size(); ++b)
        for (const auto& p : bands[b]) {
            if (n < max_pairs) { pairs_out[n] = p; band_out[n] = static_cast<int32_t>(b); }
            ++n;
        }
    if (n > INT32_MAX) return HYDRA_ERR_UNSUPPORTED;
    *n_pairs_out = static_cast<int32_t>(n);
    *n_bands_out = static_cast<int32_t>(bands.size());
    return n > max_pairs ? HYDRA_ERR_WORKSPACE_TOO_SMALL : HYDRA_OK;
}

int32_t hydra_attn_bwd(const void* q, const void* k, const void* v, const void* out, const float* lse,
                       const void* dout, const int32_t* cu, int32_t n_seqs, int32_t n_heads,
                       const hydra_pair_t* pairs, int32_t n_pairs, int32_t causal, float softmax_scale,
                       void* dq, void* dk, void* dv, void* workspace, size_t workspace_bytes,
                       void* cuda_stream)
{
    return bwd_impl(q, k, v, out, lse, dout, cu, n_seqs, n_heads, pairs, n_pairs, causal, softmax_scale, dq, dk,
                    dv, false, workspace, workspace_bytes, cuda_stream, n_heads);
}

int32_t hydra_attn_bwd_accumulate(const void* q, const void* k, const void* v, const void* out,
                                  const float* lse, const void* dout, const int32_t* cu, int32_t n_seqs,
                                  int32_t n_heads, const hydra_pair_t* pairs, int32_t n_pairs, int32_t causal,
                                  float softmax_scale, float* dq_acc, float* dk_acc, float* dv_acc,
                                  void* workspace, size_t workspace_bytes, void* cuda_stream)
{
    return bwd_impl(q, k, v, out, lse, dout, cu, n_seqs, n_heads, pairs, n_pairs, causal, softmax_scale, dq_acc,
                    dk_acc, dv_acc, true, workspace, workspace_bytes, cuda_stream, n_heads);
}

int32_t hydra_attn_bwd_gqa(const void* q, const void* k, const void* v, const void* out, const float* lse,
                           const void* dout, const int32_t* cu, int32_t n_seqs, int32_t n_heads, int32_t n_kv_heads,
                           const hydra_pair_t* pairs, int32_t n_pairs, int32_t causal, float softmax_scale,
                           void* dq, void* dk, void* dv, void* workspace, size_t workspace_bytes, void* cuda_stream)
{
    return bwd_impl(q, k, v, out, lse, dout, cu, n_seqs, n_heads, pairs, n_pairs, causal, softmax_scale, dq, dk,
                    dv, false, workspace, workspace_bytes, cuda_stream, n_kv_heads);
}

int32_t hydra_attn_bwd_accumulate_gqa(const void* q, const void* k, const void* v, const void* out,
                                      const float* lse, const void* dout, const int32_t* cu, int32_t n_seqs,
                                      int32_t n_heads, int32_t n_kv_heads, const hydra_pair_t* pairs,
                                      int32_t n_pairs, int32_t causal, float softmax_scale, float* dq_acc,
                                      float* dk_acc, float* dv_acc, void* workspace, size_t workspace_bytes,
                                      void* cuda_stream)
{
    return bwd_impl(q, k, v, out, lse, dout, cu, n_seqs, n_heads, pairs, n_pairs, causal, softmax_scale, dq_acc,
                    dk_acc, dv_acc, true, workspace, workspace_bytes, cuda_stream, n_kv_heads);
}

int32_t hydra_attn_bwd_dims(const void* q, const void* k, const void* v, const void* out, const float* lse,
                            const void* dout, const int32_t* cu, int32_t n_seqs, int32_t n_heads, int32_t n_kv_heads,
                            int32_t d_qk, int32_t d_v, const hydra_pair_t* pairs, int32_t n_pairs, int32_t causal,
                            float softmax_scale, void* dq, void* dk, void* dv, void* workspace, size_t workspace_bytes,
                            void* cuda_stream)
{
    return bwd_impl(q, k, v, out, lse, dout, cu, n_seqs, n_heads, pairs, n_pairs, causal, softmax_scale, dq, dk,
                    dv, false, workspace, workspace_bytes, cuda_stream, n_kv_heads, d_qk, d_v);
}

int32_t hydra_attn_bwd_accumulate_dims(const void* q, const void* k, const void* v, const void* out, const float* lse,
                                       const void* dout, const int32_t* cu, int32_t n_seqs, int32_t n_heads,
                                       int32_t n_kv_heads, int32_t d_qk, int32_t d_v, const hydra_pair_t* pairs,
                                       int32_t n_pairs, int32_t causal, float softmax_scale, float* dq_acc,
                                       float* dk_acc, float* dv_acc, void* workspace, size_t workspace_bytes,
                                       void* cuda_stream)
{
    return bwd_impl(q, k, v, out, lse, dout, cu, n_seqs, n_heads, pairs, n_pairs, causal, softmax_scale, dq_acc,
                    dk_acc, dv_acc, true, workspace, workspace_bytes, cuda_stream, n_kv_heads, d_qk, d_v);
}

int32_t hydra_lse_merge_local(const void* o_part, const float* lse_part, int64_t part_rows, const int32_t* cu,
                              int32_t n_seqs, int32_t n_heads, const hydra_chunk_t* q_chunks, int32_t n_q_chunks,
                              int64_t q_rows, const hydra_pair_t* pairs, int32_t n_pairs, int32_t accumulate, void* out,
                              float* lse, void* workspace, size_t workspace_bytes, void* cuda_stream)
{
    // the merge touches q-side tensors only: the kv table is the q table (every pair's kv range is unused here)
    Problem pb;
    if (int32_t s = make_problem(cu, n_seqs, n_heads, pairs, n_pairs, pb)) return s;
    if (!q_chunks || n_q_chunks < 1 || q_rows < 1 || q_rows > (int64_t{1} << 30)) return HYDRA_ERR_INVALID_ARG;
    pb.qc.assign(q_chunks, q_chunks + n_q_chunks);
    pb.Tq = q_rows;
    for (const hydra_chunk_t& c : pb.qc)
        if (c.seq < 0 || c.seq >= n_seqs || c.start < 0 || c.len < 0 || c.row < 0 || int64_t{c.row} + c.len > q_rows ||
            int64_t{c.start} + c.len > int64_t{pb.cu[c.seq + 1]} - pb.cu[c.seq])
            return HYDRA_ERR_INVALID_ARG;
    for (const hydra_pair_t& p : pb.pairs)
        if (p.q_len > 0 && p.part_row >= 0 &&
            (pb.q_row(p.seq, p.q_start) < 0 ||
             pb.q_row(p.seq, p.q_start + p.q_len - 1) != pb.q_row(p.seq, p.q_start) + p.q_len - 1))
            return HYDRA_ERR_INVALID_ARG;
    return merge_core(pb, o_part, lse_part, part_rows, out, lse, workspace, workspace_bytes, cuda_stream,
                      accumulate != 0);
}

int32_t hydra_attn_bwd_accumulate_local(const void* q, const void* k, const void* v, const void* out, const float* lse,
                                        const void* dout, const int32_t* cu, int32_t n_seqs, int32_t n_heads,
                                        int32_t n_kv_heads, int32_t d_qk, int32_t d_v, const hydra_chunk_t* q_chunks,
                                        int32_t n_q_chunks, int64_t q_rows, const hydra_chunk_t* kv_chunks,
                                        int32_t n_kv_chunks, int64_t kv_rows, const hydra_pair_t* pairs,
                                        int32_t n_pairs, int32_t causal, float softmax_scale, float* dq_acc,
                                        float* dk_acc, float* dv_acc, void* workspace, size_t workspace_bytes,
                                        void* cuda_stream)
{
    if (!kernel_set(d_qk, d_v)) return HYDRA_ERR_UNSUPPORTED;
    Problem pb;
    if (int32_t s = make_problem_local(cu, n_seqs, n_heads, q_chunks, n_q_chunks, q_rows, kv_chunks, n_kv_chunks,
                                       kv_rows, pairs, n_pairs, pb))
        return s;
    pb.dqk = d_qk;
    return bwd_core(pb, q, k, v, out, lse, dout, causal, softmax_scale, dq_acc, dk_acc, dv_acc, true, workspace,
                    workspace_bytes, cuda_stream, n_kv_heads);
}

size_t hydra_workspace_bytes_local(int32_t which, const int32_t* cu, int32_t n_seqs, int32_t n_heads,
                                   int32_t n_kv_heads, int32_t d_qk, int32_t d_v, const hydra_chunk_t* q_chunks,
                                   int32_t n_q_chunks, int64_t q_rows, const hydra_chunk_t* kv_chunks,
                                   int32_t n_kv_chunks, int64_t kv_rows, const hydra_pair_t* pairs, int32_t n_pairs)
{
    Problem pb;
    if (!kernel_set(d_qk, d_v) || n_kv_heads < 1 || n_heads % n_kv_heads) return 0;
    if (make_problem_local(cu, n_seqs, n_heads, q_chunks, n_q_chunks, q_rows, kv_chunks, n_kv_chunks, kv_rows, pairs,
                           n_pairs, pb) != HYDRA_OK)
        return 0;
    pb.dqk = d_qk;
    if (which == HYDRA_WS_FWD || which == HYDRA_WS_MERGE) return kStatusBytes;
    if (which != HYDRA_WS_BWD) return 0;
    // the accumulating backward: D of the local q rows, plus the dS hand-off buffer when it is within the limit
    return bwd_base_bytes(pb) + bwd_ds_bytes(ds_layout(pb, 1, nullptr), n_heads, g_ds_limit_bytes.load());
}

int32_t hydra_grad_cast(const float* acc, void* grad, int64_t n_elements, void* cuda_stream)
{
    if (n_elements < 0) return HYDRA_ERR_INVALID_ARG;
    if (n_elements == 0) return HYDRA_OK;
    if (!acc || !grad || !aligned16(acc) || !aligned16(grad)) return HYDRA_ERR_INVALID_ARG;
    if (int32_t s = device_info(nullptr)) return s;
    cudaStream_t stream = static_cast<cudaStream_t>(cuda_stream);
    {
        ScopedKernelTimer timer(K_CAST, stream);
        if (launch_grad_cast(acc, grad, n_elements, stream) != cudaSuccess) return HYDRA_ERR_CUDA;
    }
    g_launches += 1;
    return HYDRA_OK;
}

void hydra_profile_enable(int32_t on)
{
    std::lock_guard<std::mutex> lock(g_prof_mutex);
    g_prof_on = on != 0;
}

int32_t hydra_profile_collect(double* ms_out, int64_t* launches_out)
{
    if (!ms_out || !launches_out) return HYDRA_ERR_INVALID_ARG;
    std::lock_guard<std::mutex> lock(g_prof_mutex);
    for (int i = 0; i < K_COUNT; ++i) { ms_out[i] = 0.0; launches_out[i] = 0; }
    int32_t status = HYDRA_OK;
    for (const ProfRecord& r : g_prof_records) {
        float ms = 0.f;
        if (cudaEventSynchronize(r.stop) != cudaSuccess || cudaEventElapsedTime(&ms, r.start, r.stop) != cudaSuccess)
            status = HYDRA_ERR_CUDA;
        ms_out[r.kind] += ms;
        launches_out[r.kind] += 1;
        g_prof_pool.push_back(r.start);
        g_prof_pool.push_back(r.stop);
    }
    g_prof_records.clear();
    return status;
}

size_t hydra_host_step_arena_bytes(const int32_t* cu, int32_t n_seqs, int32_t n_heads,
                                   const hydra_pair_t* pairs, int32_t n_pairs)
{
    Problem pb;
    if (make_problem(cu, n_seqs, n_heads, pairs, n_pairs, pb) != HYDRA_OK) return 0;
    int64_t part_rows = 0;
    for (const auto& p : pb.pairs)
        if (p.part_row >= 0) part_rows = std::max<int64_t>(part_rows, int64_t{p.part_row} + p.q_len);
    const size_t th = static_cast<size_t>(std::max<int64_t>(pb.T, 1)) * n_heads;
    size_t b = 0;
    b += 3 * align_up(th * D_QK * 2, 256);                   // q, k + dq/dk share nothing: q, k, dq
    b += 1 * align_up(th * D_QK * 2, 256);                   // dk
    b += 4 * align_up(th * D_V * 2, 256);                    // v, dout, out, dv
    b += align_up(th * 4, 256) + kHostLsePad;                // lse, one 256-byte aligned slice per head group
    b += align_up(static_cast<size_t>(std::max<int64_t>(part_rows, 1)) * n_heads * D_V * 2, 256);
    b += align_up(static_cast<size_t>(std::max<int64_t>(part_rows, 1)) * n_heads * 4, 256);
    b += kStatusBytes + align_up(th * 4, 256);               // workspace of the backward call
    return b;
}

int32_t hydra_attn_fwd_bwd_host(const void* q_host, const void* k_host, const void* v_host,
                                const void* dout_host, const int32_t* cu, int32_t n_seqs, int32_t n_heads,
                                const hydra_pair_t* pairs, int32_t n_pairs, int32_t causal,
                                float softmax_scale, void* out_host, float* lse_host, void* dq_host,
                                void* dk_host, void* dv_host, void* device_arena, size_t arena_bytes,
                                void* cuda_stream)
{
    Problem pb;
    if (int32_t s = make_problem(cu, n_seqs, n_heads, pairs, n_pairs, pb)) return s;
    const void* ptrs[] = {q_host, k_host, v_host, dout_host, out_host, lse_host, dq_host, dk_host, dv_host};
    for (const void* p : ptrs)
        if (!p) return HYDRA_ERR_INVALID_ARG;
    if (!device_arena || (reinterpret_cast<uintptr_t>(device_arena) & 255u)) return HYDRA_ERR_INVALID_ARG;
    if (arena_bytes < hydra_host_step_arena_bytes(cu, n_seqs, n_heads, pairs, n_pairs))
        return HYDRA_ERR_WORKSPACE_TOO_SMALL;
    if (pb.T == 0) return HYDRA_OK;
    int64_t part_rows = 0;
    for (const auto& p : pb.pairs)
        if (p.part_row >= 0) part_rows = std::max<int64_t>(part_rows, int64_t{p.part_row} + p.q_len);
    cudaStream_t stream = static_cast<cudaStream_t>(cuda_stream);
    const size_t th = static_cast<size_t>(pb.T) * n_heads;
    uint8_t* cur = static_cast<uint8_t*>(device_arena);
    auto carve = [&](size_t bytes) { void* p = cur; cur += align_up(bytes, 256); return p; };
    uint8_t* dq_ = static_cast<uint8_t*>(carve(th * D_QK * 2)); uint8_t* dk_ = static_cast<uint8_t*>(carve(th * D_QK * 2));
    uint8_t* q = static_cast<uint8_t*>(carve(th * D_QK * 2)); uint8_t* k = static_cast<uint8_t*>(carve(th * D_QK * 2));
    uint8_t* v = static_cast<uint8_t*>(carve(th * D_V * 2)); uint8_t* dout = static_cast<uint8_t*>(carve(th * D_V * 2));
    uint8_t* out = static_cast<uint8_t*>(carve(th * D_V * 2)); uint8_t* dv_ = static_cast<uint8_t*>(carve(th * D_V * 2));
    uint8_t* lse = static_cast<uint8_t*>(carve(th * 4 + kHostLsePad));
    void* o_part = carve(static_cast<size_t>(std::max<int64_t>(part_rows, 1)) * n_heads * D_V * 2);
    float* lse_part = static_cast<float*>(carve(static_cast<size_t>(std::max<int64_t>(part_rows, 1)) * n_heads * 4));
    void* ws = carve(kStatusBytes + align_up(th * 4, 256));
    const size_t ws_bytes = kStatusBytes + align_up(th * 4, 256);

    // Sequences and heads are independent, so the step is pipelined over groups (a range of whole sequences
    // times a range of heads): while group g computes, group g+1 is on its way in and group g-1 on its way
    // out, on two internal copy streams; the host link then carries both directions at once. On the device a
    // group is a compact [tokens, heads_of_group, d] tensor inside its token range of each arena tensor.
    HostPipe* pipe = host_pipe();
    if (!pipe) return HYDRA_ERR_CUDA;
    double pair_count = 0.0;
    for (const auto& p : pb.pairs) {
        const double full = static_cast<double>(p.q_len) * p.k_len;
        pair_count += causal ? std::min(full, 0.5 * p.q_len * (p.q_len + 1.0) +
                                                  static_cast<double>(p.q_len) * std::max(0, p.q_start - p.k_start))
                             : full;
    }
    // rough rates: 50 GB/s per direction, 700 TFLOP/s
    const double copy_s = static_cast<double>(pb.T) * (2 * D_QK + 2 * D_V) * 2 / 50e9;   // per head, one direction
    const double math_s = pair_count * 3.5 * 2 * (D_QK + D_V) / 700e12;                  // per head
    const std::vector<HostGroup> groups = host_groups(pb, math_s < 0.5 * copy_s);
    const int32_t n_groups = static_cast<int32_t>(groups.size());
    const size_t H = static_cast<size_t>(n_heads);
    struct Slice { size_t oqk, ov, lse; };                  // byte offsets of a group's tensors in the arena tensors
    std::vector<Slice> slice(n_groups);
    size_t lse_off = 0;
    for (int32_t g = 0; g < n_groups; ++g) {
        const HostGroup& G = groups[g];
        const size_t th0 = static_cast<size_t>(G.t0) * H + static_cast<size_t>(G.tn) * G.h0;   // (token, head) pairs before it
        slice[g] = {th0 * D_QK * 2, th0 * D_V * 2, lse_off};
        lse_off = align_up(lse_off + static_cast<size_t>(G.tn) * G.hn * 4, 256);
    }
    // one tensor of a group between the host's [T, n_heads, d] layout and the group's compact one
    auto move = [&](const HostGroup& G, uint8_t* dev, const uint8_t* host_base, size_t row_bytes, bool to_device,
                    cudaStream_t st) {
        uint8_t* host = const_cast<uint8_t*>(host_base) + (static_cast<size_t>(G.t0) * H + G.h0) * row_bytes;
        const cudaMemcpyKind kind = to_device ? cudaMemcpyHostToDevice : cudaMemcpyDeviceToHost;
        const size_t width = static_cast<size_t>(G.hn) * row_bytes, rows = static_cast<size_t>(G.tn);
        if (G.hn == n_heads)
            return to_device ? cudaMemcpyAsync(dev, host, width * rows, kind, st) : cudaMemcpyAsync(host, dev, width * rows, kind, st);
        return to_device ? cudaMemcpy2DAsync(dev, width, host, H * row_bytes, width, rows, kind, st)
                         : cudaMemcpy2DAsync(host, H * row_bytes, dev, width, width, rows, kind, st);
    };
    // (an output buffer may be an input's: the results of a group then wait until its inputs have been read)
    auto share = [](const void* a, size_t na, const void* b, size_t nb) {
        const uintptr_t x = reinterpret_cast<uintptr_t>(a), y = reinterpret_cast<uintptr_t>(b);
        return x < y + nb && y < x + na;
    };
    const bool out_over_dout = share(out_host, th * D_V * 2, dout_host, th * D_V * 2) ||
                               share(lse_host, th * 4, dout_host, th * D_V * 2);
    if (cudaEventRecord(pipe->start, stream) || cudaStreamWaitEvent(pipe->in, pipe->start, 0) ||
        cudaStreamWaitEvent(pipe->out, pipe->start, 0))
        return HYDRA_ERR_CUDA;
    for (int32_t g = 0; g < n_groups; ++g) {
        const HostGroup& G = groups[g];
        if (move(G, q + slice[g].oqk, static_cast<const uint8_t*>(q_host), D_QK * 2, true, pipe->in) ||
            move(G, k + slice[g].oqk, static_cast<const uint8_t*>(k_host), D_QK * 2, true, pipe->in) ||
            move(G, v + slice[g].ov, static_cast<const uint8_t*>(v_host), D_V * 2, true, pipe->in) ||
            cudaEventRecord(pipe->in_done[g], pipe->in) ||
            move(G, dout + slice[g].ov, static_cast<const uint8_t*>(dout_host), D_V * 2, true, pipe->in) ||
            cudaEventRecord(pipe->dout_done[g], pipe->in))
            return HYDRA_ERR_CUDA;
    }
    std::vector<int32_t> cu_g;
    std::vector<hydra_pair_t> pairs_g;
    for (int32_t g = 0; g < n_groups; ++g) {
        const HostGroup& G = groups[g];
        const size_t oqk = slice[g].oqk, ov = slice[g].ov;
        float* lse_g = reinterpret_cast<float*>(lse + slice[g].lse);
        if (g == 0 || G.s0 != groups[g - 1].s0) {            // the sequences of this group, and their pairs, renumbered
            cu_g.assign(cu + G.s0, cu + G.s1 + 1);
            for (int32_t& c : cu_g) c -= cu[G.s0];
            pairs_g.clear();
            for (int32_t i = 0; i < n_pairs; ++i)
                if (pairs[i].seq >= G.s0 && pairs[i].seq < G.s1) {
                    pairs_g.push_back(pairs[i]);
                    pairs_g.back().seq -= G.s0;
                }
        }
        const int32_t ns = G.s1 - G.s0, np = static_cast<int32_t>(pairs_g.size());
        const hydra_pair_t* pg = np ? pairs_g.data() : nullptr;
        bool part = false;
        for (const hydra_pair_t& p : pairs_g) part = part || p.part_row >= 0;
        if (cudaStreamWaitEvent(stream, pipe->in_done[g], 0)) return HYDRA_ERR_CUDA;
        const bool work = n_pairs == 0 || np > 0;            // else sequences without any pair of the caller's list
        if (work) {
            if (int32_t s = hydra_attn_fwd(q + oqk, k + oqk, v + ov, cu_g.data(), ns, G.hn, pg, np, causal, softmax_scale,
                                           out + ov, lse_g, part ? o_part : nullptr, part ? lse_part : nullptr,
                                           part ? part_rows : 0, ws, ws_bytes, cuda_stream))
                return s;
            if (part)
                if (int32_t s = hydra_lse_merge(o_part, lse_part, part_rows, cu_g.data(), ns, G.hn, pg, np, out + ov,
                                                lse_g, ws, ws_bytes, cuda_stream))
                    return s;
        }
        // out and lse leave while dO is still on its way in, which takes a fifth off the time that only one direction of the
        // link is busy (before the first copy out and after the last copy in): 12288 tokens, 16 heads 6.47 -> 6.35 ms, 8192
        // packed tokens 4.77 -> 4.53, 8192 tokens of short sequences, 8 heads 2.55 -> 2.42, 1024 tokens, 4 heads 0.252 -> 0.235
        if (cudaEventRecord(pipe->fwd_done[g], stream) || cudaStreamWaitEvent(pipe->out, pipe->fwd_done[g], 0) ||
            (out_over_dout && cudaStreamWaitEvent(pipe->out, pipe->dout_done[g], 0)) ||
            move(G, out + ov, static_cast<const uint8_t*>(out_host), D_V * 2, false, pipe->out) ||
            cudaMemcpy2DAsync(lse_host + static_cast<size_t>(G.h0) * pb.T + G.t0, static_cast<size_t>(pb.T) * 4, lse_g,
                              static_cast<size_t>(G.tn) * 4, static_cast<size_t>(G.tn) * 4, G.hn, cudaMemcpyDeviceToHost,
                              pipe->out) ||
            cudaStreamWaitEvent(stream, pipe->dout_done[g], 0))
            return HYDRA_ERR_CUDA;
        if (work)
            if (int32_t s = hydra_attn_bwd(q + oqk, k + oqk, v + ov, out + ov, lse_g, dout + ov, cu_g.data(), ns, G.hn,
                                           pg, np, causal, softmax_scale, dq_ + oqk, dk_ + oqk, dv_ + ov, ws, ws_bytes,
                                           cuda_stream))
                return s;
        if (cudaEventRecord(pipe->comp_done[g], stream) || cudaStreamWaitEvent(pipe->out, pipe->comp_done[g], 0) ||
            move(G, dv_ + ov, static_cast<const uint8_t*>(dv_host), D_V * 2, false, pipe->out) ||
            move(G, dq_ + oqk, static_cast<const uint8_t*>(dq_host), D_QK * 2, false, pipe->out) ||
            move(G, dk_ + oqk, static_cast<const uint8_t*>(dk_host), D_QK * 2, false, pipe->out))
            return HYDRA_ERR_CUDA;
    }
    // the caller's stream completes when the last copy out has completed
    if (cudaEventRecord(pipe->end, pipe->out) || cudaStreamWaitEvent(stream, pipe->end, 0)) return HYDRA_ERR_CUDA;
    return HYDRA_OK;
}

namespace {
int32_t ulysses_impl(bool pack, const void* x, int64_t n_tokens, int32_t n_heads, int32_t head_dim, int32_t cp_u,
                     void* out, void* cuda_stream)
{
    if (n_tokens < 0 || n_heads < 1 || head_dim < 1 || cp_u < 1 || n_heads % cp_u) return HYDRA_ERR_INVALID_ARG;
    const int64_t chunk_bytes = static_cast<int64_t>(n_heads / cp_u) * head_dim * 2;
    if (chunk_bytes % 16) return HYDRA_ERR_UNSUPPORTED;
    if (n_tokens == 0) return HYDRA_OK;
    if (!x || !out || x == out || !aligned16(x) || !aligned16(out)) return HYDRA_ERR_INVALID_ARG;
    // the kernel indexes 16-byte units with 32 bits: tensors up to 60 GB
    if (n_tokens > (int64_t{60} << 30) / (chunk_bytes * cp_u)) return HYDRA_ERR_UNSUPPORTED;
    if (int32_t s = device_info(nullptr)) return s;
    cudaStream_t stream = static_cast<cudaStream_t>(cuda_stream);
    ScopedKernelTimer timer(K_ULYSSES, stream);
    if (launch_ulysses(pack, x, out, n_tokens, cp_u, chunk_bytes / 16, stream) != cudaSuccess) return HYDRA_ERR_CUDA;
    g_launches += 1;
    return HYDRA_OK;
}
}  // namespace

int32_t hydra_ulysses_pack(const void* x, int64_t n_tokens, int32_t n_heads, int32_t head_dim, int32_t cp_u,
                           void* send, void* cuda_stream)
{
    return ulysses_impl(true, x, n_tokens, n_heads, head_dim, cp_u, send, cuda_stream);
}

int32_t hydra_ulysses_unpack(const void* recv, int64_t n_tokens, int32_t n_heads, int32_t head_dim, int32_t cp_u,
                             void* y, void* cuda_stream)
{
    return ulysses_impl(false, recv, n_tokens, n_heads, head_dim, cp_u, y, cuda_stream);
}

namespace {
bool rope_shape_ok(int32_t head_dim, int32_t rope_offset, int32_t rope_dim)
{
    return head_dim >= 2 && head_dim % 2 == 0 && rope_offset >= 0 && rope_offset % 2 == 0 && rope_dim >= 2 &&
           rope_dim % 2 == 0 && rope_dim <= 256 && rope_offset + rope_dim <= head_dim;
}
bool aligned4(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 3u) == 0; }
}  // namespace

int32_t hydra_mla_rope(const void* x, const int32_t* positions, int64_t n_tokens, int32_t n_heads, int32_t head_dim,
                       int32_t rope_offset, int32_t rope_dim, float theta, int32_t inverse, void* y, void* cuda_stream)
{
    if (n_tokens < 0 || n_heads < 1 || !rope_shape_ok(head_dim, rope_offset, rope_dim) || !(theta > 1.f) ||
        !std::isfinite(theta))
        return HYDRA_ERR_INVALID_ARG;
    if (n_tokens == 0) return HYDRA_OK;
    if (!x || !y || !positions || !aligned4(x) || !aligned4(y) || !aligned4(positions)) return HYDRA_ERR_INVALID_ARG;
    if (int32_t s = device_info(nullptr)) return s;
    cudaStream_t stream = static_cast<cudaStream_t>(cuda_stream);
    ScopedKernelTimer timer(K_MLA, stream);
    if (launch_rope(x, positions, y, n_tokens, n_heads, head_dim, rope_offset, rope_dim, theta, inverse != 0, stream) !=
        cudaSuccess)
        return HYDRA_ERR_CUDA;
    g_launches += 1;
    return HYDRA_OK;
}

int32_t hydra_mla_kv_assemble(const void* kv_up, const void* k_pe, const int32_t* positions, int64_t n_tokens,
                              int32_t n_heads, int32_t d_nope, int32_t d_rope, int32_t d_v, float theta, void* k, void* v,
                              void* cuda_stream)
{
    if (n_tokens < 0 || n_heads < 1 || d_nope < 2 || d_nope % 2 || d_v < 2 || d_v % 2 ||
        !rope_shape_ok(d_rope, 0, d_rope) || !(theta > 1.f) || !std::isfinite(theta))
        return HYDRA_ERR_INVALID_ARG;
    if (n_tokens == 0) return HYDRA_OK;
    const void* ptrs[] = {kv_up, k_pe, positions, k, v};
    for (const void* p : ptrs)
        if (!p || !aligned4(p)) return HYDRA_ERR_INVALID_ARG;
    if (int32_t s = device_info(nullptr)) return s;
    cudaStream_t stream = static_cast<cudaStream_t>(cuda_stream);
    ScopedKernelTimer timer(K_MLA, stream);
    if (launch_mla_kv_assemble(kv_up, k_pe, positions, k, v, n_tokens, n_heads, d_nope, d_rope, d_v, theta, stream) !=
        cudaSuccess)
        return HYDRA_ERR_CUDA;
    g_launches += 1;
    return HYDRA_OK;
}

int32_t hydra_mla_kv_assemble_bwd(const void* dk, const void* dv, const int32_t* positions, int64_t n_tokens,
                                  int32_t n_heads, int32_t d_nope, int32_t d_rope, int32_t d_v, float theta, void* dkv_up,
                                  void* dk_pe, void* cuda_stream)
{
    if (n_tokens < 0 || n_heads < 1 || d_nope < 2 || d_nope % 2 || d_v < 2 || d_v % 2 ||
        !rope_shape_ok(d_rope, 0, d_rope) || !(theta > 1.f) || !std::isfinite(theta))
        return HYDRA_ERR_INVALID_ARG;
    if (n_tokens == 0) return HYDRA_OK;
    const void* ptrs[] = {dk, dv, positions, dkv_up, dk_pe};
    for (const void* p : ptrs)
        if (!p || !aligned4(p)) return HYDRA_ERR_INVALID_ARG;
    if (int32_t s = device_info(nullptr)) return s;
    cudaStream_t stream = static_cast<cudaStream_t>(cuda_stream);
    ScopedKernelTimer timer(K_MLA, stream);
    if (launch_mla_kv_assemble_bwd(dk, dv, positions, dkv_up, dk_pe, n_tokens, n_heads, d_nope, d_rope, d_v, theta,
                                   stream) != cudaSuccess)
        return HYDRA_ERR_CUDA;
    g_launches += 1;
    return HYDRA_OK;
}

int32_t hydra_gate_apply(const void* out, const void* gate, int64_t n_elements, void* y, void* cuda_stream)
{
    if (n_elements < 0 || n_elements % 8) return HYDRA_ERR_INVALID_ARG;
    if (n_elements == 0) return HYDRA_OK;
    if (!out || !gate || !y || !aligned16(out) || !aligned16(gate) || !aligned16(y)) return HYDRA_ERR_INVALID_ARG;
    if (int32_t s = device_info(nullptr)) return s;
    cudaStream_t stream = static_cast<cudaStream_t>(cuda_stream);
    ScopedKernelTimer timer(K_MLA, stream);
    if (launch_gate(out, gate, y, n_elements / 8, stream) != cudaSuccess) return HYDRA_ERR_CUDA;
    g_launches += 1;
    return HYDRA_OK;
}

int32_t hydra_gate_apply_bwd(const void* dy, const void* out, const void* gate, int64_t n_elements, void* d_out,
                             void* d_gate, void* cuda_stream)
{
    if (n_elements < 0 || n_elements % 8) return HYDRA_ERR_INVALID_ARG;
    if (n_elements == 0) return HYDRA_OK;
    const void* ptrs[] = {dy, out, gate, d_out, d_gate};
    for (const void* p : ptrs)
        if (!p || !aligned16(p)) return HYDRA_ERR_INVALID_ARG;
    if (int32_t s = device_info(nullptr)) return s;
    cudaStream_t stream = static_cast<cudaStream_t>(cuda_stream);
    ScopedKernelTimer timer(K_MLA, stream);
    if (launch_gate_bwd(dy, out, gate, d_out, d_gate, n_elements / 8, stream) != cudaSuccess) return HYDRA_ERR_CUDA;
    g_launches += 1;
    return HYDRA_OK;
}

int32_t hydra_poll_status(void* workspace, void* cuda_stream, int32_t* device_status, int64_t* detail)
{
    if (!workspace || !device_status) return HYDRA_ERR_INVALID_ARG;
    if (cudaStreamSynchronize(static_cast<cudaStream_t>(cuda_stream)) != cudaSuccess) return HYDRA_ERR_CUDA;
    StatusBlock sb;
    if (cudaMemcpy(&sb, workspace, sizeof sb, cudaMemcpyDeviceToHost) != cudaSuccess) return HYDRA_ERR_CUDA;
    *device_status = sb.call_tag == sb.error_tag ? sb.status : HYDRA_OK;
    if (detail) *detail = *device_status ? sb.detail : -1;
    return HYDRA_OK;
}

int32_t hydra_poll_clocks(void* workspace, void* cuda_stream, double* mhz_out)
{
    if (!workspace || !mhz_out) return HYDRA_ERR_INVALID_ARG;
    if (cudaStreamSynchronize(static_cast<cudaStream_t>(cuda_stream)) != cudaSuccess) return HYDRA_ERR_CUDA;
    StatusBlock sb;
    if (cudaMemcpy(&sb, workspace, sizeof sb, cudaMemcpyDeviceToHost) != cudaSuccess) return HYDRA_ERR_CUDA;
    for (int i = 0; i < 3; ++i) {
        // the forward's figure comes from the CTA-pair kernel if the call used it, else from the short-sequence one
        const int src = (i == QUEUE_FWD && !sb.probe_ns[i]) ? QUEUE_FWD_SHORT : i;
        mhz_out[i] = sb.probe_ns[src] ? 1e3 * static_cast<double>(sb.probe_cycles[src]) / static_cast<double>(sb.probe_ns[src]) : 0.0;
    }
    return HYDRA_OK;
}

}  // extern "C"

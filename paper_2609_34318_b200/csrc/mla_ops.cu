// The elementwise steps of a gated multi-head-latent attention block around the attention kernel
// (Section 5.2, "Exposed All-to-All Overlap": the query's rotary embedding; the split of the KV
// up-projection's output into the value and the key's position-free part; the key's rotary embedding and
// concatenation; the output gate), forward and backward. All are bound by HBM: every byte moves once, with
// 32-, 16- or 4-byte accesses that are contiguous per warp. The paper names the steps, not their formulas;
// the readings taken (rotary pairs (2i, 2i+1), angle = position * theta^(-2i/rope_dim); one rotary key
// vector per token shared by all heads; up-projection rows laid out [key part | value]; gate = sigmoid)
// are stated with each entry point in the header.
#include <cuda_bf16.h>

#include <algorithm>
#include <initializer_list>

#include <cmath>

#include "hydra_internal.h"
#include "sm100_ptx.cuh"

namespace hydra {
namespace {

constexpr int kRopeThreads = 128;
constexpr int kMaxRopePairs = 128;          // rotary dimensions up to 256

__device__ __forceinline__ float2 bf2_to_f2(uint32_t w)
{
    return make_float2(__uint_as_float(w << 16), __uint_as_float(w & 0xffff0000u));
}
__device__ __forceinline__ uint32_t f2_to_bf2(float lo, float hi)
{
    const __nv_bfloat162 h = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<const uint32_t*>(&h);
}

// cos / sin of position * theta^(-2i/rope_dim), i < rope_dim / 2, for one token, into shared memory. The
// angle is formed and reduced modulo 2 pi in double precision: at position 262143 a single-precision
// product is off by hundredths of a radian.
__device__ __forceinline__ void rope_table(float* s_cos, float* s_sin, int32_t pos, int32_t rope_dim, double log_theta,
                                           int inverse)
{
    for (int i = threadIdx.x; i < rope_dim / 2; i += blockDim.x) {
        const double freq = exp(-log_theta * (2.0 * i) / rope_dim);
        double ang = static_cast<double>(pos) * freq;
        ang -= 6.283185307179586476925 * floor(ang / 6.283185307179586476925);
        float sn, cs;
        sincosf(static_cast<float>(ang), &sn, &cs);
        s_cos[i] = cs;
        s_sin[i] = inverse ? -sn : sn;
    }
}

// y[t, a, :] = x[t, a, :] with the pairs (2i, 2i+1) of columns [rope_offset, rope_offset + rope_dim) rotated
// by the token's angles. One block per token (grid-stride), the heads' rows as 4-byte pairs.
__global__ void __launch_bounds__(kRopeThreads)
hydra_rope_kernel(const uint32_t* __restrict__ x, const int32_t* __restrict__ positions, uint32_t* __restrict__ y,
                  int64_t n_tokens, int32_t n_heads, int32_t head_dim, int32_t rope_offset, int32_t rope_dim,
                  double log_theta, int inverse, int in_place)
{
    wait_for_previous_launch();
    __shared__ float s_cos[kMaxRopePairs], s_sin[kMaxRopePairs];
    const int pairs_per_head = head_dim / 2, p0 = rope_offset / 2, p1 = (rope_offset + rope_dim) / 2;
    for (int64_t t = blockIdx.x; t < n_tokens; t += gridDim.x) {
        __syncthreads();                               // the previous token's table is no longer read
        rope_table(s_cos, s_sin, positions[t], rope_dim, log_theta, inverse);
        __syncthreads();
        const int64_t row0 = t * n_heads * pairs_per_head;
        if (in_place) {                                // only the rotary columns move
            const int n = n_heads * (p1 - p0);
            for (int e = threadIdx.x; e < n; e += kRopeThreads) {
                const int a = e / (p1 - p0), i = e - a * (p1 - p0);
                const int64_t idx = row0 + static_cast<int64_t>(a) * pairs_per_head + p0 + i;
                const float2 v = bf2_to_f2(x[idx]);
                y[idx] = f2_to_bf2(v.x * s_cos[i] - v.y * s_sin[i], v.x * s_sin[i] + v.y * s_cos[i]);
            }
        } else {
            const int n = n_heads * pairs_per_head;
            for (int e = threadIdx.x; e < n; e += kRopeThreads) {
                const int c = e % pairs_per_head;
                uint32_t w = x[row0 + e];
                if (c >= p0 && c < p1) {
                    const float2 v = bf2_to_f2(w);
                    const int i = c - p0;
                    w = f2_to_bf2(v.x * s_cos[i] - v.y * s_sin[i], v.x * s_sin[i] + v.y * s_cos[i]);
                }
                y[row0 + e] = w;
            }
        }
    }
    overlap_next_launch();
}

// k[t, a, :] = [kv_up[t, a, 0:nope] | rope(k_pe[t, :])], v[t, a, :] = kv_up[t, a, nope:nope+dv]
__global__ void __launch_bounds__(kRopeThreads)
hydra_mla_kv_assemble_kernel(const uint32_t* __restrict__ kv_up, const uint32_t* __restrict__ k_pe,
                             const int32_t* __restrict__ positions, uint32_t* __restrict__ k, uint32_t* __restrict__ v,
                             int64_t n_tokens, int32_t n_heads, int32_t nope, int32_t rope_dim, int32_t dv,
                             double log_theta)
{
    wait_for_previous_launch();
    __shared__ float s_cos[kMaxRopePairs], s_sin[kMaxRopePairs];
    __shared__ uint32_t s_pe[kMaxRopePairs];
    const int np = nope / 2, rp = rope_dim / 2, vp = dv / 2;
    const int up_pairs = np + vp, k_pairs = np + rp;
    for (int64_t t = blockIdx.x; t < n_tokens; t += gridDim.x) {
        __syncthreads();
        rope_table(s_cos, s_sin, positions[t], rope_dim, log_theta, 0);
        __syncthreads();
        for (int i = threadIdx.x; i < rp; i += kRopeThreads) {
            const float2 w = bf2_to_f2(k_pe[t * rp + i]);
            s_pe[i] = f2_to_bf2(w.x * s_cos[i] - w.y * s_sin[i], w.x * s_sin[i] + w.y * s_cos[i]);
        }
        __syncthreads();
        const int64_t up0 = t * n_heads * up_pairs, k0 = t * n_heads * k_pairs, v0 = t * n_heads * vp;
        for (int e = threadIdx.x; e < n_heads * up_pairs; e += kRopeThreads) {
            const int a = e / up_pairs, c = e - a * up_pairs;
            const uint32_t w = kv_up[up0 + e];
            if (c < np) k[k0 + static_cast<int64_t>(a) * k_pairs + c] = w;
            else v[v0 + static_cast<int64_t>(a) * vp + (c - np)] = w;
        }
        for (int e = threadIdx.x; e < n_heads * rp; e += kRopeThreads) {
            const int a = e / rp, i = e - a * rp;
            k[k0 + static_cast<int64_t>(a) * k_pairs + np + i] = s_pe[i];
        }
    }
    overlap_next_launch();
}

// The adjoint: dkv_up[t, a, :] = [dk[t, a, 0:nope] | dv[t, a, :]],
// dk_pe[t, :] = rope^-1( sum_a dk[t, a, nope:nope+rope_dim] ) (summed in fp32, rounded once).
__global__ void __launch_bounds__(kRopeThreads)
hydra_mla_kv_assemble_bwd_kernel(const uint32_t* __restrict__ dk, const uint32_t* __restrict__ dv,
                                 const int32_t* __restrict__ positions, uint32_t* __restrict__ dkv_up,
                                 uint32_t* __restrict__ dk_pe, int64_t n_tokens, int32_t n_heads, int32_t nope,
                                 int32_t rope_dim, int32_t dvd, double log_theta)
{
    wait_for_previous_launch();
    __shared__ float s_cos[kMaxRopePairs], s_sin[kMaxRopePairs];
    const int np = nope / 2, rp = rope_dim / 2, vp = dvd / 2;
    const int up_pairs = np + vp, k_pairs = np + rp;
    for (int64_t t = blockIdx.x; t < n_tokens; t += gridDim.x) {
        __syncthreads();
        rope_table(s_cos, s_sin, positions[t], rope_dim, log_theta, 1);
        __syncthreads();
        const int64_t up0 = t * n_heads * up_pairs, k0 = t * n_heads * k_pairs, v0 = t * n_heads * vp;
        for (int e = threadIdx.x; e < n_heads * up_pairs; e += kRopeThreads) {
            const int a = e / up_pairs, c = e - a * up_pairs;
            dkv_up[up0 + e] = c < np ? dk[k0 + static_cast<int64_t>(a) * k_pairs + c]
                                     : dv[v0 + static_cast<int64_t>(a) * vp + (c - np)];
        }
        for (int i = threadIdx.x; i < rp; i += kRopeThreads) {
            float sx = 0.f, sy = 0.f;
            for (int a = 0; a < n_heads; ++a) {
                const float2 w = bf2_to_f2(dk[k0 + static_cast<int64_t>(a) * k_pairs + np + i]);
                sx += w.x;
                sy += w.y;
            }
            dk_pe[t * rp + i] = f2_to_bf2(sx * s_cos[i] - sy * s_sin[i], sx * s_sin[i] + sy * s_cos[i]);
        }
    }
    overlap_next_launch();
}

inline bool aligned16_all(std::initializer_list<const void*> ptrs)
{
    uintptr_t bits = 0;
    for (const void* p : ptrs) bits |= reinterpret_cast<uintptr_t>(p);
    return (bits & 15u) == 0;
}

// kWords 32-bit words (pairs of bf16) per thread and access: 4 (16 bytes), or 8 (32 bytes) where the element
// count and the buffers allow it. Half as many threads then share the loop and address arithmetic.
template <int kWords>
struct Words { uint32_t w[kWords]; };
template <int kWords>
__device__ __forceinline__ Words<kWords> ld_words(const void* base, int64_t i)
{
    Words<kWords> v;
    if constexpr (kWords == 8) {
        const Words<8>* p = static_cast<const Words<8>*>(base) + i;
        asm volatile("ld.global.nc.L1::no_allocate.v8.u32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                     : "=r"(v.w[0]), "=r"(v.w[1]), "=r"(v.w[2]), "=r"(v.w[3]), "=r"(v.w[4]), "=r"(v.w[5]),
                       "=r"(v.w[6]), "=r"(v.w[7])
                     : "l"(p));
    } else {
        const uint4 t = static_cast<const uint4*>(base)[i];
        v.w[0] = t.x; v.w[1] = t.y; v.w[2] = t.z; v.w[3] = t.w;
    }
    return v;
}
// the same from memory that this kernel writes
template <int kWords>
__device__ __forceinline__ Words<kWords> ld_words_coherent(const void* base, int64_t i)
{
    Words<kWords> v;
    const uint4* p = reinterpret_cast<const uint4*>(static_cast<const Words<kWords>*>(base) + i);
#pragma unroll
    for (int j = 0; j < kWords / 4; ++j) {
        const uint4 t = p[j];
        v.w[4 * j] = t.x; v.w[4 * j + 1] = t.y; v.w[4 * j + 2] = t.z; v.w[4 * j + 3] = t.w;
    }
    return v;
}
template <int kWords>
__device__ __forceinline__ void st_words(void* base, int64_t i, const Words<kWords>& v)
{
    if constexpr (kWords == 8) {
        st_global_v8(static_cast<Words<8>*>(base) + i, v.w);
    } else {
        static_cast<uint4*>(base)[i] = make_uint4(v.w[0], v.w[1], v.w[2], v.w[3]);
    }
}

// ---------------------------------------------------------------------------------------------
// Vector forms of the three kernels above (kWords rotary pairs, 16 or 32 bytes, per access), used when the head
// dimensions are multiples of the vector and the buffers aligned to it. All three are bound by memory, and what keeps
// them from its rate is the time in which a block has no access in flight. So: a block takes several tokens at once where
// a token is short, and forms their cos / sin (or rotated keys) in one pass with a thread per (token, pair); what needs no
// table is moved while that is done; vector numbers are split with a multiplication. Against one token, 128 threads and
// 16 bytes at a time (and, in the backward, 8 threads adding up the rotary columns of all heads): 4096 tokens, 128 heads
// of 128 + 64 / 128, rotary embedding 77.2 -> 66.6 us (6.05 TB/s), assembly 119.3 -> 97.3 (6.2), its backward
// 155 -> 99.3 (6.1); 16384 tokens, 8 heads 20.8 -> 20.5, 31.3 -> 26.8 and 41.2 -> 31.3; 100 tokens, 128 heads 6.7 -> 5.7,
// 9.7 -> 6.4 and 20.1 -> 6.1. A copy of as many bytes runs at 6.3 TB/s.
// ---------------------------------------------------------------------------------------------
constexpr int kVecThreads = 256;
// Vectors of a thread in flight. The assembly gains from four (two: 100 us instead of 97.3); the other two need their registers
// for more blocks (rotary embedding with four, two, one: 71.5, 66.6, 68.3 us; assembly backward 113, 99.3, 104).
constexpr int kAsmUnroll = 4, kRopeUnroll = 2, kAsmBwdUnroll = 2;

// n / d for n * d < 2^32 (`fits` below): the error of n * m / 2^32, m = floor(2^32 / d) + 1, is under 1 / d
struct Div {
    uint32_t d, m;
    explicit Div(uint32_t div) : d(div), m(div > 1 ? static_cast<uint32_t>((uint64_t{1} << 32) / div) + 1 : 0) {}
    __device__ __forceinline__ uint32_t operator()(uint32_t n) const { return m ? __umulhi(n, m) : n; }
};

// cos / sin of position * freq, the angle reduced as in rope_table
__device__ __forceinline__ void rope_angle(int32_t pos, double freq, float& cs, float& sn)
{
    double ang = static_cast<double>(pos) * freq;
    ang -= 6.283185307179586476925 * floor(ang / 6.283185307179586476925);
    sincosf(static_cast<float>(ang), &sn, &cs);
}

// A block takes `per_item` tokens at once; thread (token of the item) * pairs + pair forms that pair's angle.
struct VecItems {
    int64_t n_tokens;
    int32_t n_heads, per_item, pairs;
    double log_theta;
    Div by_heads;
    VecItems(int64_t n, int32_t h, int32_t rope_dim, int64_t vecs_per_token, float theta)
        : n_tokens(n), n_heads(h), per_item(1), pairs(rope_dim / 2), log_theta(std::log(static_cast<double>(theta))),
          by_heads(static_cast<uint32_t>(h))
    {
        // eight vectors per thread where the tokens are short, but no fewer than two blocks per SM for that (4096 tokens of
        // 8 heads: assembly backward 6.9 us, with four vectors and four blocks per SM 9.8)
        const int64_t want = 8 * kVecThreads / vecs_per_token;
        per_item = static_cast<int32_t>(std::max<int64_t>(1, std::min({want, int64_t{kVecThreads / pairs}, n / (148 * 2)})));
    }
    // are all vector and row numbers of an item in the range of Div?
    bool fits(int32_t vecs_per_head) const
    {
        const double rows = static_cast<double>(per_item) * n_heads, vecs = rows * vecs_per_head;
        return std::max(vecs * vecs_per_head, rows * n_heads) < 4294967296.0;
    }
    int grid() const
    {
        const int64_t items = (n_tokens + per_item - 1) / per_item;
        return static_cast<int>(std::min<int64_t>(items, 148 * 32));
    }
};

template <int kWords>
__device__ __forceinline__ Words<kWords> rotate_vec(const Words<kWords>& w, const float* cp, const float* sp)
{
    Words<kWords> out;
#pragma unroll
    for (int j = 0; j < kWords; ++j) {
        const float2 v = bf2_to_f2(w.w[j]);
        out.w[j] = f2_to_bf2(v.x * cp[j] - v.y * sp[j], v.x * sp[j] + v.y * cp[j]);
    }
    return out;
}

// n vectors of a block: load(e) gives vector e and where it goes, store(at, v) puts it there
template <int kWords, int kVecUnroll, class Load, class Store>
__device__ __forceinline__ void move_vecs(uint32_t n, Load load, Store store)
{
    for (uint32_t e0 = threadIdx.x; e0 < n; e0 += kVecUnroll * kVecThreads) {
        Words<kWords> v[kVecUnroll];
        uint32_t at[kVecUnroll];
#pragma unroll
        for (int u = 0; u < kVecUnroll; ++u)
            if (e0 + u * kVecThreads < n) v[u] = load(e0 + u * kVecThreads, at[u]);
#pragma unroll
        for (int u = 0; u < kVecUnroll; ++u)
            if (e0 + u * kVecThreads < n) store(at[u], v[u]);
    }
}

// the rotary vectors and the others in loops of their own: no lane waits for a rotation it does not do. In place (x == y)
// only the rotary columns move.
template <int kWords, bool kInPlace>
__global__ void __launch_bounds__(kVecThreads)
hydra_rope_vec_kernel(const uint32_t* x, const int32_t* __restrict__ positions, uint32_t* y, const VecItems it, int32_t v0,
                      const Div by_rot, const Div by_copy, int inverse)
{
    __shared__ __align__(16) float s_cos[kVecThreads], s_sin[kVecThreads];
    const uint32_t nv = by_rot.d, vph = by_rot.d + by_copy.d;
    const int my_tok = threadIdx.x / it.pairs, my_pair = threadIdx.x - my_tok * it.pairs;
    const double freq = exp(-it.log_theta * my_pair / it.pairs);
    wait_for_previous_launch();
    for (int64_t t0 = static_cast<int64_t>(blockIdx.x) * it.per_item; t0 < it.n_tokens;
         t0 += static_cast<int64_t>(gridDim.x) * it.per_item) {
        const int n_tok = static_cast<int>(min(static_cast<int64_t>(it.per_item), it.n_tokens - t0));
        const uint32_t rows = n_tok * it.n_heads;
        const uint32_t* xb = x + t0 * it.n_heads * vph * kWords;
        uint32_t* yb = y + t0 * it.n_heads * vph * kWords;
        if (!kInPlace)
            move_vecs<kWords, kRopeUnroll>(rows * by_copy.d, [&](uint32_t e, uint32_t& at) {
                const uint32_t r = by_copy(e), j = e - r * by_copy.d;
                at = r * vph + (j < static_cast<uint32_t>(v0) ? j : j + nv);
                return ld_words<kWords>(xb, at);
            }, [&](uint32_t at, const Words<kWords>& v) { st_words<kWords>(yb, at, v); });
        bool tables = false;
        for (uint32_t e0 = threadIdx.x; !tables || e0 < rows * nv; e0 += kRopeUnroll * kVecThreads) {
            Words<kWords> w[kRopeUnroll];
#pragma unroll
            for (int u = 0; u < kRopeUnroll; ++u) {
                const uint32_t e = e0 + u * kVecThreads, r = by_rot(e), at = r * vph + v0 + e - r * nv;
                if (e < rows * nv) w[u] = kInPlace ? ld_words_coherent<kWords>(xb, at) : ld_words<kWords>(xb, at);
            }
            if (!tables) {                             // the angles while the first vectors are on their way
                tables = true;
                __syncthreads();                       // the tables of the tokens before are no longer read
                if (my_tok < n_tok) {
                    float cs, sn;
                    rope_angle(positions[t0 + my_tok], freq, cs, sn);
                    s_cos[threadIdx.x] = cs;
                    s_sin[threadIdx.x] = inverse ? -sn : sn;
                }
                __syncthreads();
            }
#pragma unroll
            for (int u = 0; u < kRopeUnroll; ++u) {
                const uint32_t e = e0 + u * kVecThreads, r = by_rot(e), i = e - r * nv;
                const uint32_t c = it.by_heads(r) * it.pairs + i * kWords;
                if (e < rows * nv) st_words<kWords>(yb, r * vph + v0 + i, rotate_vec<kWords>(w[u], s_cos + c, s_sin + c));
            }
        }
    }
    overlap_next_launch();
}

template <int kWords>
__global__ void __launch_bounds__(kVecThreads)
hydra_mla_kv_assemble_vec_kernel(const uint32_t* __restrict__ kv_up, const uint32_t* __restrict__ k_pe,
                                 const int32_t* __restrict__ positions, uint32_t* __restrict__ k, uint32_t* __restrict__ v,
                                 const VecItems it, uint32_t nv, const Div by_up, const Div by_rot)
{
    __shared__ __align__(32) uint32_t s_pe[kVecThreads];
    const uint32_t vv = by_up.d - nv, rv = by_rot.d, k_vecs = nv + rv;
    const int my_tok = threadIdx.x / it.pairs, my_pair = threadIdx.x - my_tok * it.pairs;
    const double freq = exp(-it.log_theta * my_pair / it.pairs);
    wait_for_previous_launch();
    for (int64_t t0 = static_cast<int64_t>(blockIdx.x) * it.per_item; t0 < it.n_tokens;
         t0 += static_cast<int64_t>(gridDim.x) * it.per_item) {
        const int n_tok = static_cast<int>(min(static_cast<int64_t>(it.per_item), it.n_tokens - t0));
        const uint32_t rows = n_tok * it.n_heads;
        const int64_t row0 = t0 * it.n_heads;
        const uint32_t* ub = kv_up + row0 * by_up.d * kWords;
        uint32_t* kb = k + row0 * k_vecs * kWords;
        uint32_t* vb = v + row0 * vv * kWords;
        __syncthreads();                               // the rotated keys of the tokens before are no longer read
        if (my_tok < n_tok) {
            float cs, sn;
            rope_angle(positions[t0 + my_tok], freq, cs, sn);
            const float2 w = bf2_to_f2(k_pe[t0 * it.pairs + threadIdx.x]);
            s_pe[threadIdx.x] = f2_to_bf2(w.x * cs - w.y * sn, w.x * sn + w.y * cs);
        }
        move_vecs<kWords, kAsmUnroll>(rows * by_up.d, [&](uint32_t e, uint32_t& at) {
            at = e;
            return ld_words<kWords>(ub, e);
        }, [&](uint32_t e, const Words<kWords>& w) {
            const uint32_t r = by_up(e), c = e - r * by_up.d;
            if (c < nv) st_words<kWords>(kb, r * k_vecs + c, w);
            else st_words<kWords>(vb, r * vv + (c - nv), w);
        });
        __syncthreads();
        for (uint32_t e = threadIdx.x; e < rows * rv; e += kVecThreads) {
            const uint32_t r = by_rot(e), i = e - r * rv;
            const uint32_t* pe = s_pe + it.by_heads(r) * it.pairs + i * kWords;
            Words<kWords> w;
#pragma unroll
            for (int j = 0; j < kWords; ++j) w.w[j] = pe[j];
            st_words<kWords>(kb, r * k_vecs + nv + i, w);
        }
    }
    overlap_next_launch();
}

// The shared rotary key's gradient is the sum over the heads: each thread adds up one vector over every n-th head of its
// token, a thread per (token, pair) adds those partial sums in order, and rotates back.
template <int kWords>
__global__ void __launch_bounds__(kVecThreads)
hydra_mla_kv_assemble_bwd_vec_kernel(const uint32_t* __restrict__ dk, const uint32_t* __restrict__ dv,
                                     const int32_t* __restrict__ positions, uint32_t* __restrict__ dkv_up,
                                     uint32_t* __restrict__ dk_pe, const VecItems it, uint32_t nv, const Div by_up, uint32_t rv)
{
    __shared__ __align__(16) float s_part[kVecThreads * 2 * kWords];
    const uint32_t vv = by_up.d - nv, k_vecs = nv + rv;
    const int my_tok = threadIdx.x / it.pairs, my_pair = threadIdx.x - my_tok * it.pairs;
    const int part = threadIdx.x / rv, vec = threadIdx.x - part * rv;      // this thread's partial sum and vector of it
    const int parts = kVecThreads / static_cast<int>(rv) / it.per_item;    // partial sums per token
    const int part_tok = part / parts, first_head = part - part_tok * parts;
    const double freq = exp(-it.log_theta * my_pair / it.pairs);
    wait_for_previous_launch();
    for (int64_t t0 = static_cast<int64_t>(blockIdx.x) * it.per_item; t0 < it.n_tokens;
         t0 += static_cast<int64_t>(gridDim.x) * it.per_item) {
        const int n_tok = static_cast<int>(min(static_cast<int64_t>(it.per_item), it.n_tokens - t0));
        const uint32_t rows = n_tok * it.n_heads;
        const int64_t row0 = t0 * it.n_heads;
        const uint32_t* kb = dk + row0 * k_vecs * kWords;
        const uint32_t* vb = dv + row0 * vv * kWords;
        uint32_t* ub = dkv_up + row0 * by_up.d * kWords;
        float acc[2 * kWords];
#pragma unroll
        for (int j = 0; j < 2 * kWords; ++j) acc[j] = 0.f;
        if (part_tok < n_tok) {
#pragma unroll 2
            for (int a = first_head; a < it.n_heads; a += parts) {
                const Words<kWords> w = ld_words<kWords>(kb, (part_tok * it.n_heads + a) * k_vecs + nv + vec);
#pragma unroll
                for (int j = 0; j < kWords; ++j) {
                    const float2 f = bf2_to_f2(w.w[j]);
                    acc[2 * j] += f.x;
                    acc[2 * j + 1] += f.y;
                }
            }
        }
        __syncthreads();                               // the partial sums of the tokens before are no longer read
        if (part_tok < n_tok) {
#pragma unroll
            for (int j = 0; j < 2 * kWords; j += 4)
                *reinterpret_cast<float4*>(s_part + threadIdx.x * 2 * kWords + j) =
                    make_float4(acc[j], acc[j + 1], acc[j + 2], acc[j + 3]);
        }
        move_vecs<kWords, kAsmBwdUnroll>(rows * by_up.d, [&](uint32_t e, uint32_t& at) {
            const uint32_t r = by_up(e), c = e - r * by_up.d;
            at = e;
            return c < nv ? ld_words<kWords>(kb, r * k_vecs + c) : ld_words<kWords>(vb, r * vv + (c - nv));
        }, [&](uint32_t at, const Words<kWords>& w) { st_words<kWords>(ub, at, w); });
        __syncthreads();
        if (my_tok < n_tok) {
            float sx = 0.f, sy = 0.f;
            for (int q = 0; q < parts; ++q) {
                const float2 f = *reinterpret_cast<const float2*>(s_part + ((my_tok * parts + q) * it.pairs + my_pair) * 2);
                sx += f.x;
                sy += f.y;
            }
            float cs, sn;
            rope_angle(positions[t0 + my_tok], freq, cs, sn);
            dk_pe[t0 * it.pairs + threadIdx.x] = f2_to_bf2(sx * cs + sy * sn, sy * cs - sx * sn);
        }
    }
    overlap_next_launch();
}

// (exp and reciprocal of the special-function unit: a relative error of 2^-21, far below the bf16 result's 2^-9)
__device__ __forceinline__ float sigmoidf_(float x) { return __fdividef(1.f, 1.f + __expf(-x)); }

// y = out * sigmoid(gate)
template <int kWords>
__global__ void __launch_bounds__(256)
hydra_gate_kernel(const void* __restrict__ out, const void* __restrict__ gate, void* __restrict__ y, int64_t n)
{
    wait_for_previous_launch();
    for (int64_t i = static_cast<int64_t>(blockIdx.x) * 256 + threadIdx.x; i < n; i += static_cast<int64_t>(gridDim.x) * 256) {
        const Words<kWords> o = ld_words<kWords>(out, i), g = ld_words<kWords>(gate, i);
        Words<kWords> r;
#pragma unroll
        for (int e = 0; e < kWords; ++e) {
            const float2 a = bf2_to_f2(o.w[e]), b = bf2_to_f2(g.w[e]);
            r.w[e] = f2_to_bf2(a.x * sigmoidf_(b.x), a.y * sigmoidf_(b.y));
        }
        st_words<kWords>(y, i, r);
    }
    overlap_next_launch();
}

// d_out = dy * sigmoid(gate);  d_gate = dy * out * sigmoid(gate) * (1 - sigmoid(gate))
template <int kWords>
__global__ void __launch_bounds__(256)
hydra_gate_bwd_kernel(const void* __restrict__ dy, const void* __restrict__ out, const void* __restrict__ gate,
                      void* __restrict__ d_out, void* __restrict__ d_gate, int64_t n)
{
    wait_for_previous_launch();
    for (int64_t i = static_cast<int64_t>(blockIdx.x) * 256 + threadIdx.x; i < n; i += static_cast<int64_t>(gridDim.x) * 256) {
        const Words<kWords> d = ld_words<kWords>(dy, i), o = ld_words<kWords>(out, i), g = ld_words<kWords>(gate, i);
        Words<kWords> ro, rg;
#pragma unroll
        for (int e = 0; e < kWords; ++e) {
            const float2 a = bf2_to_f2(d.w[e]), b = bf2_to_f2(o.w[e]), c = bf2_to_f2(g.w[e]);
            const float s0 = sigmoidf_(c.x), s1 = sigmoidf_(c.y);
            ro.w[e] = f2_to_bf2(a.x * s0, a.y * s1);
            rg.w[e] = f2_to_bf2(a.x * b.x * s0 * (1.f - s0), a.y * b.y * s1 * (1.f - s1));
        }
        st_words<kWords>(d_out, i, ro);
        st_words<kWords>(d_gate, i, rg);
    }
    overlap_next_launch();
}

inline bool all_aligned32(std::initializer_list<const void*> ptrs)
{
    uintptr_t bits = 0;
    for (const void* p : ptrs) bits |= reinterpret_cast<uintptr_t>(p);
    return (bits & 31u) == 0;
}

int grid_for(int64_t work_items, int per_block)
{
    const int64_t blocks = (work_items + per_block - 1) / per_block;
    return static_cast<int>(blocks < 1 ? 1 : (blocks < 148 * 16 ? blocks : 148 * 16));
}

}  // namespace

// kWords of the vector kernels that the dimensions and buffers admit: 8, 4 or 0 (the four-byte kernels)
static int words_for(std::initializer_list<int32_t> dims, std::initializer_list<const void*> ptrs)
{
    int32_t bits = 0;
    for (int32_t d : dims) bits |= d;
    if (bits % 16 == 0 && all_aligned32(ptrs)) return 8;
    return bits % 8 == 0 && aligned16_all(ptrs) ? 4 : 0;
}

template <int kWords>
static cudaError_t launch_rope_vec(const VecItems& it, const uint32_t* x, const int32_t* positions, uint32_t* y, int32_t head_dim,
                                   int32_t rope_offset, int32_t rope_dim, int inverse, cudaStream_t stream)
{
    constexpr int32_t kElems = 2 * kWords;
    const Div by_rot(rope_dim / kElems), by_copy((head_dim - rope_dim) / kElems);
    return launch_overlapped(x == y ? hydra_rope_vec_kernel<kWords, true> : hydra_rope_vec_kernel<kWords, false>, it.grid(),
                             kVecThreads, 0, stream, x, positions, y, it, rope_offset / kElems, by_rot, by_copy, inverse);
}

cudaError_t launch_rope(const void* x, const int32_t* positions, void* y, int64_t n_tokens, int32_t n_heads,
                        int32_t head_dim, int32_t rope_offset, int32_t rope_dim, float theta, int inverse,
                        cudaStream_t stream)
{
    if (n_tokens == 0) return cudaSuccess;
    const uint32_t* x32 = static_cast<const uint32_t*>(x);
    uint32_t* y32 = static_cast<uint32_t*>(y);
    if (const int words = words_for({head_dim, rope_offset, rope_dim}, {x, y})) {
        const VecItems it(n_tokens, n_heads, rope_dim, int64_t{n_heads} * (head_dim / (2 * words)), theta);
        if (it.fits(head_dim / (2 * words)))
            return words == 8 ? launch_rope_vec<8>(it, x32, positions, y32, head_dim, rope_offset, rope_dim, inverse, stream)
                              : launch_rope_vec<4>(it, x32, positions, y32, head_dim, rope_offset, rope_dim, inverse, stream);
    }
    return launch_overlapped(hydra_rope_kernel, grid_for(n_tokens, 1), kRopeThreads, 0, stream,
        x32, positions, y32, n_tokens, n_heads, head_dim, rope_offset,
        rope_dim, std::log(static_cast<double>(theta)), inverse, x == y ? 1 : 0);
}

cudaError_t launch_mla_kv_assemble(const void* kv_up, const void* k_pe, const int32_t* positions, void* k, void* v,
                                   int64_t n_tokens, int32_t n_heads, int32_t nope, int32_t rope_dim, int32_t dv,
                                   float theta, cudaStream_t stream)
{
    if (n_tokens == 0) return cudaSuccess;
    const uint32_t *up32 = static_cast<const uint32_t*>(kv_up), *pe32 = static_cast<const uint32_t*>(k_pe);
    uint32_t *k32 = static_cast<uint32_t*>(k), *v32 = static_cast<uint32_t*>(v);
    if (const int words = words_for({nope, rope_dim, dv}, {kv_up, k, v})) {
        const int32_t per_head = (nope + std::max(dv, rope_dim)) / (2 * words);
        const VecItems it(n_tokens, n_heads, rope_dim, int64_t{n_heads} * ((nope + dv) / (2 * words)), theta);
        if (it.fits(per_head)) {
            const uint32_t nv = nope / (2 * words);
            const Div by_up((nope + dv) / (2 * words)), by_rot(rope_dim / (2 * words));
            return launch_overlapped(words == 8 ? hydra_mla_kv_assemble_vec_kernel<8> : hydra_mla_kv_assemble_vec_kernel<4>,
                                     it.grid(), kVecThreads, 0, stream, up32, pe32, positions, k32, v32, it, nv, by_up, by_rot);
        }
    }
    return launch_overlapped(hydra_mla_kv_assemble_kernel, grid_for(n_tokens, 1), kRopeThreads, 0, stream,
        up32, pe32, positions, k32, v32, n_tokens, n_heads, nope, rope_dim, dv, std::log(static_cast<double>(theta)));
}

cudaError_t launch_mla_kv_assemble_bwd(const void* dk, const void* dv, const int32_t* positions, void* dkv_up,
                                       void* dk_pe, int64_t n_tokens, int32_t n_heads, int32_t nope, int32_t rope_dim,
                                       int32_t dvd, float theta, cudaStream_t stream)
{
    if (n_tokens == 0) return cudaSuccess;
    const uint32_t *dk32 = static_cast<const uint32_t*>(dk), *dv32 = static_cast<const uint32_t*>(dv);
    uint32_t *up32 = static_cast<uint32_t*>(dkv_up), *pe32 = static_cast<uint32_t*>(dk_pe);
    if (const int words = words_for({nope, rope_dim, dvd}, {dk, dv, dkv_up})) {
        const int32_t per_head = (nope + std::max(dvd, rope_dim)) / (2 * words);
        const VecItems it(n_tokens, n_heads, rope_dim, int64_t{n_heads} * ((nope + dvd) / (2 * words)), theta);
        if (it.fits(per_head)) {
            const uint32_t nv = nope / (2 * words), rv = rope_dim / (2 * words);
            const Div by_up((nope + dvd) / (2 * words));
            return launch_overlapped(words == 8 ? hydra_mla_kv_assemble_bwd_vec_kernel<8> : hydra_mla_kv_assemble_bwd_vec_kernel<4>,
                                     it.grid(), kVecThreads, 0, stream, dk32, dv32, positions, up32, pe32, it, nv, by_up, rv);
        }
    }
    return launch_overlapped(hydra_mla_kv_assemble_bwd_kernel, grid_for(n_tokens, 1), kRopeThreads, 0, stream,
        dk32, dv32, positions, up32, pe32, n_tokens, n_heads, nope, rope_dim, dvd, std::log(static_cast<double>(theta)));
}

cudaError_t launch_gate(const void* out, const void* gate, void* y, int64_t n8, cudaStream_t stream)
{
    if (n8 == 0) return cudaSuccess;
    if ((n8 & 1) == 0 && all_aligned32({out, gate, y}))
        return launch_overlapped(hydra_gate_kernel<8>, grid_for(n8 / 2, 256), 256, 0, stream, out, gate, y, n8 / 2);
    else
        return launch_overlapped(hydra_gate_kernel<4>, grid_for(n8, 256), 256, 0, stream, out, gate, y, n8);
}

cudaError_t launch_gate_bwd(const void* dy, const void* out, const void* gate, void* d_out, void* d_gate, int64_t n8,
                            cudaStream_t stream)
{
    if (n8 == 0) return cudaSuccess;
    if ((n8 & 1) == 0 && all_aligned32({dy, out, gate, d_out, d_gate}))
        return launch_overlapped(hydra_gate_bwd_kernel<8>, grid_for(n8 / 2, 256), 256, 0, stream, dy, out, gate, d_out, d_gate, n8 / 2);
    else
        return launch_overlapped(hydra_gate_bwd_kernel<4>, grid_for(n8, 256), 256, 0, stream, dy, out, gate, d_out, d_gate, n8);
}

}  // namespace hydra

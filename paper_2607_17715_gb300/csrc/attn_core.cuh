// The CUDA-core attention loop shared by the suffix attention (attn_simt.cu) and the extraction
// attention (extract.cu): fp32 arithmetic throughout, for fp32 contexts (no tensor-core format
// keeps fp32 inputs exact) and for the head layouts the tensor-core kernel does not take.
//
// One CTA of four warps holds 16 RT packed query rows of one (layer, request, KV head) (row
// r = t G + g: the G query heads that share a KV head share every K/V tile) and walks the key
// tiles of 64 that some row of it may see.  A warp owns 4 RT rows; its lane (ty, tx) =
// (lane / 8, lane % 8) rows ty + 4 i of them, of a tile's scores the keys tx + 8 j, and of the
// output the channels 4 tx + 32 h .. + 3.
//   S:   per 4 channels RT + 8 16-byte shared loads feed 32 RT FMAs; every 16 channels the
//        partial dot products are folded, so no sum is a chain of more than 16 terms.
//   P.V: 32 keys at a time the weights pass through shared memory within the warp; the
//        products of 32 keys are summed apart and then folded into O.  The keys that a row does
//        not see have a weight of 0 there; where 32 keys' sums are not finite in a tile that some
//        row does not see whole, they are formed again without such keys (0 times a value of
//        infinity or NaN, which may be another row's to see, is not 0).  Looking for them takes
//        1 to 4 % of a call, leaving every such key out by a test a weight took 8 to 10 %.
// A 16-byte shared load costs a wavefront per half-warp and 128 bytes of different addresses:
// with 4 x 8 lanes every load above costs the least, two, so 128 FMAs take 20 to 24 (with lanes
// 2 x 16 the loads of K and V cost four, and shared memory bound the kernel).
// K (then V) of the next tile is copied by cp.async while the weights (the next scores) are
// formed.  Measured (fp32, clock stamps, with sums folded every 32 channels; every 16 takes the same
// time): d = 128, 64 rows: S 7.7 K and P.V 8.2 K clocks a tile for 4096 FMAs a lane each, a CTA alone on
// its SM; two sharing one reach 60 % of the FMA pipe.
// An attend of 2 requests x 96 tokens over 720 slots, 16 / 4 heads, d = 128, went from 176 us
// (one shared load per FMA operand) to 61.5 us, 4 requests x 250 tokens x 1024 slots, d = 64, from
// 548 to 176 us, extraction of 2000 tokens, d = 128, from 1858 to 669 us.
//
// The work follows what there is: a warp whose rows lie past the last one only copies, the last key
// tile costs by its keys, and the third form (RT = 0) holds four rows, of which each warp takes the
// keys 16 w .. 16 w + 15 of a tile, the four warps' (max, sum, O) merged at the end.  Without these,
// one token of ten requests, 32 layers of 32 / 8 heads, d = 128, took 161 us over 9 keys, and now 77 (89
// in the earlier kernel, a warp a row); 3 tokens of 3 requests x 1888 keys, 16 layers of 8 heads, d = 64,
// the whole step, 316 and now 208 (241).
//
// A launch of few row tiles splits each one's key range over a cluster of `ns` CTAs, whose
// (max, sum, O) are merged through distributed shared memory by the exact log-sum-exp rule: no
// scratch in device memory, no second launch.
#pragma once

#include <cooperative_groups.h>
#include <math_constants.h>

#include <algorithm>
#include <cmath>
#include <type_traits>

#include "internal.cuh"
#include "per_device.cuh"
#include "ptx.cuh"
#include "vec16.cuh"

namespace c2kv {
namespace {

constexpr int kCoreKeys = 64;              // keys per tile
constexpr int kCoreMaxSplit = 8;           // portable cluster size
constexpr int kCoreThreads = 128;
constexpr int kCorePPitch = 40 * 4;        // bytes of a row's 32 weights, padded

// RT = 0: the four-row form, whose warps share the keys.
template <int D, int RT>
struct Core {
    static constexpr int kSlots = RT == 0 ? 16 : 16 * RT;          // (row, warp that holds it)
    static constexpr int kRows = RT == 0 ? 4 : 16 * RT;
    static constexpr int kPitch = (D + 4) * 4;                     // bytes of a Q or K row
    static constexpr int kQ = 0;
    static constexpr int kK = kQ + kRows * kPitch;
    static constexpr int kV = kK + kCoreKeys * kPitch;
    static constexpr int kP = kV + kCoreKeys * D * 4;
    static constexpr int kML = kP + kSlots * kCorePPitch;          // max and sum of each slot (merge)
    static constexpr int kSmem = kML + kSlots * 8;
    static_assert(kSlots * D * 4 <= kP - kK, "the merge's O fits over K and V");
};

// CTAs an SM is to hold (shared memory allows them; what the registers are cut to).
__host__ __device__ constexpr int core_ctas(int d, int rt) { return rt == 0 ? (d == 128 ? 3 : 5) : d == 128 ? 2 : rt == 1 ? 4 : 3; }

// `rows` rows of D elements into shared memory as fp32, row r from src + r * stride (row_ok(r):
// zeros otherwise), at `pitch` bytes a row.  fp32 rows go by cp.async (the caller commits and
// waits), bf16 rows through registers.
template <typename T, int D, class Src>
__device__ __forceinline__ void core_copy(uint8_t* dst, int pitch, int rows, const Src& src) {
    if constexpr (sizeof(T) == 4) {
        constexpr int CPR = D / 4;                         // 16-byte chunks a row
        for (int i = threadIdx.x; i < rows * CPR; i += kCoreThreads) {
            const int r = i / CPR, c = i - r * CPR;
            const T* p = src(r);
            const uint32_t n = p != nullptr ? 16u : 0u;    // 0: zeros, nothing read
            const uint32_t a = smem_u32(dst + (size_t)r * pitch + c * 16);
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(a),
                         "l"(p != nullptr ? p + 4 * c : src.any()), "r"(n)
                         : "memory");
        }
    } else {
        constexpr int CPR = D / 8;
        constexpr int U = 4;                               // loads in flight a thread
        for (int i0 = threadIdx.x; i0 < rows * CPR; i0 += U * kCoreThreads) {
            uint4 w[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int i = i0 + u * kCoreThreads;
                const int r = i / CPR, c = i - r * CPR;
                const T* p = i < rows * CPR ? src(r) : nullptr;
                w[u] = p != nullptr ? *reinterpret_cast<const uint4*>(p + 8 * c) : make_uint4(0u, 0u, 0u, 0u);
            }
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int i = i0 + u * kCoreThreads;
                if (i >= rows * CPR) break;
                const int r = i / CPR, c = i - r * CPR;
                float f[8];
                Vec16<__nv_bfloat16>::unpack(w[u], f);
                float4* o = reinterpret_cast<float4*>(dst + (size_t)r * pitch + c * 32);
                o[0] = make_float4(f[0], f[1], f[2], f[3]);
                o[1] = make_float4(f[4], f[5], f[6], f[7]);
            }
        }
    }
}
__device__ __forceinline__ void core_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void core_wait() {
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

template <typename T>
struct CoreRows {                // rows of a K or V tile, none past `limit`
    const T* base;
    int64_t stride;
    int first, limit;
    __device__ const T* operator()(int r) const { return first + r < limit ? base + (int64_t)(first + r) * stride : nullptr; }
    __device__ const T* any() const { return base; }
};
template <typename T, class Job>
struct CoreQ {                   // the CTA's query rows
    const Job& job;
    int row0;
    __device__ const T* operator()(int r) const { return row0 + r < job.nrows ? job.q_row(row0 + r) : nullptr; }
    __device__ const T* any() const { return job.q_row(row0); }
};

__device__ __forceinline__ float4 core_ld4(const uint8_t* p) { return *reinterpret_cast<const float4*>(p); }

template <int RT, int J, class Channel>
__device__ __forceinline__ void core_dot(float (&acc)[RT][J], const float4 (&q)[RT], const float4 (&kf)[J], Channel ch) {
#pragma unroll
    for (int i = 0; i < RT; ++i)
#pragma unroll
        for (int j = 0; j < J; ++j) acc[i][j] = fmaf(ch(q[i]), ch(kf[j]), acc[i][j]);
}

// A lane's scores of a tile: its rows (qb) with its keys tx + 8 j, j < J (kb); the others stay.
template <int D, int RT, int J, int NJ>
__device__ __forceinline__ void core_score(const uint8_t* qb, const uint8_t* kb, float (&s)[RT][NJ]) {
    using L = Core<D, RT>;
    // channels per folded partial sum.  (16, and the scale in the exponent's fused multiply-add: the
    // error against 64 bits is that of the earlier kernel's four interleaved sums, 2e-7 to 5e-7 of the
    // largest output over 32 to 8192 keys; with 32 and a rounded product it was up to a third above it,
    // and no faster.)
    constexpr int kBlk = 16;
#pragma unroll 1
    for (int c0 = 0; c0 < D; c0 += kBlk) {
        float a[RT][J];
#pragma unroll
        for (int i = 0; i < RT; ++i)
#pragma unroll
            for (int j = 0; j < J; ++j) a[i][j] = 0.f;
#pragma unroll
        for (int c = 0; c < kBlk; c += 4) {
            float4 kf[J], q[RT];
#pragma unroll
            for (int j = 0; j < J; ++j) kf[j] = core_ld4(kb + 8 * j * L::kPitch + (c0 + c) * 4);
#pragma unroll
            for (int i = 0; i < RT; ++i) q[i] = core_ld4(qb + 4 * i * L::kPitch + (c0 + c) * 4);
            // channel by channel over every (i, j): no FMA waits for the one before it
            core_dot(a, q, kf, [](const float4& v) { return v.x; });
            core_dot(a, q, kf, [](const float4& v) { return v.y; });
            core_dot(a, q, kf, [](const float4& v) { return v.z; });
            core_dot(a, q, kf, [](const float4& v) { return v.w; });
        }
#pragma unroll
        for (int i = 0; i < RT; ++i)
#pragma unroll
            for (int j = 0; j < J; ++j) s[i][j] += a[i][j];
    }
}

// Job: nrows (packed rows of the unit), nkeys (keys of this CTA's rows), k, v, stride (key rows),
// scale_log2; q_row(r), out_row(r), lse_at(r) (null without lse); needed(k0, k1): some row of the
// CTA may see a key of [k0, k1); whole(k0, k1): every row sees all of them; row(r): what
// sees(row, key) takes of packed row r.
template <typename T, int D, int kForm, class Job>
__device__ __forceinline__ void attention_core(const Job& job, int row0, int ns, int rank, uint8_t* sm) {
    using L = Core<D, kForm>;
    constexpr bool KS = kForm == 0;                        // four rows, the warps share the keys
    constexpr int RT = KS ? 1 : kForm, NJ = KS ? 2 : 8;    // rows a lane; keys a lane
    constexpr int H = D / 32;                              // 4-channel groups a lane
    const int tid = threadIdx.x, lane = tid & 31, ty = lane >> 3, tx = lane & 7;
    const int slot0 = (tid >> 5) * 4 * RT + ty;            // this lane's slots slot0 + 4 i,
    const int r0 = KS ? ty : slot0;                        // rows r0 + 4 i
    const int key0 = KS ? (tid >> 5) * 16 : 0;             // and keys key0 + tx + 8 j of a tile
    const int tiles = (job.nkeys + kCoreKeys - 1) / kCoreKeys;
    const int t_beg = (int)((int64_t)tiles * rank / ns), t_end = (int)((int64_t)tiles * (rank + 1) / ns);
    auto next = [&](int t) {                               // first tile >= t that some row may see
        while (t < t_end && !job.needed(t * kCoreKeys, (t + 1) * kCoreKeys)) ++t;
        return t;
    };
    // keys of tile t, and the rows of it that are copied (8 at a time; zeros past the last key)
    auto keys_in = [&](int t) { return min(kCoreKeys, job.nkeys - t * kCoreKeys); };
    auto load_k = [&](int t) {
        core_copy<T, D>(sm + L::kK, L::kPitch, (keys_in(t) + 7) & ~7, CoreRows<T>{job.k, job.stride, t * kCoreKeys, job.nkeys});
        core_commit();
    };
    auto load_v = [&](int t) {
        core_copy<T, D>(sm + L::kV, D * 4, (keys_in(t) + 7) & ~7, CoreRows<T>{job.v, job.stride, t * kCoreKeys, job.nkeys});
        core_commit();
    };
    const bool rows_here = KS || row0 + (tid >> 5) * 4 * RT < job.nrows;   // (a warp without rows only copies)

    float m[RT], l[RT];
    float4 o[RT][H];
#pragma unroll
    for (int i = 0; i < RT; ++i) {
        m[i] = -CUDART_INF_F;
        l[i] = 0.f;
#pragma unroll
        for (int h = 0; h < H; ++h) o[i][h] = make_float4(0.f, 0.f, 0.f, 0.f);
    }
    int t = next(t_beg);
    core_copy<T, D>(sm + L::kQ, L::kPitch, L::kRows, CoreQ<T, Job>{job, row0});
    if (t < t_end) load_k(t);                              // (one group with Q)
    else core_commit();
    if (t < t_end) load_v(t);
    else core_commit();

    const uint8_t* qb = sm + L::kQ + r0 * L::kPitch;
    const uint8_t* kb = sm + L::kK + (key0 + tx) * L::kPitch;
    const uint8_t* vb = sm + L::kV + key0 * D * 4 + tx * 16;
    uint8_t* pb = sm + L::kP + slot0 * kCorePPitch;
    while (t < t_end) {
        const int k0 = t * kCoreKeys, tn = next(t + 1), nt = keys_in(t);
        core_wait<1>();
        __syncthreads();                                   // K (and Q) of this tile
        float s[RT][NJ];
#pragma unroll
        for (int i = 0; i < RT; ++i)
#pragma unroll
            for (int j = 0; j < NJ; ++j) s[i][j] = 0.f;
        const bool live = rows_here && key0 < nt;
        if (live) {
            // (few rows: a tile of few keys, the only one of a short context, costs by its keys)
            if (KS || (RT == 1 && nt <= 16)) core_score<D, RT, 2>(qb, kb, s);
            else if (RT == 1 && nt <= 32) core_score<D, RT, NJ / 2>(qb, kb, s);
            else core_score<D, RT, NJ>(qb, kb, s);
        }
        __syncthreads();                                   // K is read: the next tile's may land
        if (tn < t_end) load_k(tn);
        else core_commit();

        const bool whole = k0 + kCoreKeys <= job.nkeys && job.whole(k0, k0 + kCoreKeys);
        float alpha[RT];
        if (live) {
#pragma unroll
            for (int i = 0; i < RT; ++i) {
                uint32_t hidden = 0u;                          // bit j: the row does not see key tx + 8 j
                if (!whole) {
                    const auto row = job.row(row0 + r0 + 4 * i);
#pragma unroll
                    for (int j = 0; j < NJ; ++j) {
                        const int key = k0 + key0 + tx + 8 * j;
                        if (key >= job.nkeys || !job.sees(row, key)) {
                            s[i][j] = -CUDART_INF_F;
                            hidden |= 1u << j;
                        }
                    }
                }
                float mx = s[i][0];
#pragma unroll
                for (int j = 1; j < NJ; ++j) mx = fmaxf(mx, s[i][j]);
#pragma unroll
                for (int off = 4; off > 0; off >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, off));
                const float mn = fmaxf(m[i], mx * job.scale_log2);
                const float ms = mn == -CUDART_INF_F ? 0.f : mn;      // nothing visible yet
                alpha[i] = exp2f(m[i] - ms);
                m[i] = mn;
#pragma unroll
                for (int j = 0; j < NJ; ++j) {
                    s[i][j] = exp2f(fmaf(s[i][j], job.scale_log2, -ms));
                    if (hidden >> j & 1u) s[i][j] = -0.f;
                }
                float sum = s[i][0] + s[i][1];                 // of this lane's keys
                if constexpr (NJ == 8)
                    sum = (sum + (s[i][2] + s[i][3])) + ((s[i][4] + s[i][5]) + (s[i][6] + s[i][7]));
                l[i] = l[i] * alpha[i] + sum;
            }
        }
        core_wait<1>();
        __syncthreads();                                   // V of this tile
        if (live) {
#pragma unroll
            for (int half = 0; half < 2; ++half) {
                if (half == 1 && (KS || nt <= 32)) continue;
                const int un = min(KS ? 16 : 32, (nt - key0 - 32 * half + 7) & ~7);
                float4 pv[RT][H];
                auto clear = [&] {
#pragma unroll
                    for (int i = 0; i < RT; ++i)
#pragma unroll
                        for (int h = 0; h < H; ++h) pv[i][h] = make_float4(0.f, 0.f, 0.f, 0.f);
                };
                // keys 32 half + u .. + 3; `masked`: a hidden key's weight, -0, is left out
                auto weigh = [&](int u, auto masked) {
                    float4 p[RT];
#pragma unroll
                    for (int i = 0; i < RT; ++i) p[i] = core_ld4(pb + 4 * i * kCorePPitch + u * 4);
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        float4 v[H];
#pragma unroll
                        for (int h = 0; h < H; ++h) v[h] = core_ld4(vb + (32 * half + u + e) * D * 4 + h * 128);
#pragma unroll
                        for (int i = 0; i < RT; ++i) {
                            const float w = e == 0 ? p[i].x : e == 1 ? p[i].y : e == 2 ? p[i].z : p[i].w;
                            if (decltype(masked)::value && __float_as_uint(w) == 0x80000000u) continue;
#pragma unroll
                            for (int h = 0; h < H; ++h) {
                                pv[i][h].x = fmaf(w, v[h].x, pv[i][h].x);
                                pv[i][h].y = fmaf(w, v[h].y, pv[i][h].y);
                                pv[i][h].z = fmaf(w, v[h].z, pv[i][h].z);
                                pv[i][h].w = fmaf(w, v[h].w, pv[i][h].w);
                            }
                        }
                    }
                };
                clear();
                __syncwarp();                                  // the weights before these are read
#pragma unroll
                for (int i = 0; i < RT; ++i)
#pragma unroll
                    for (int j = 0; j < NJ && j < 4; ++j)
                        *reinterpret_cast<float*>(pb + 4 * i * kCorePPitch + (tx + 8 * j) * 4) = s[i][KS ? j : 4 * half + j];
                __syncwarp();
#pragma unroll 1
                for (int u = 0; u < un; u += 8) {
                    weigh(u, std::false_type{});
                    weigh(u + 4, std::false_type{});
                }
                if (!whole) {
                    float4 z = make_float4(0.f, 0.f, 0.f, 0.f);      // zeros, or NaN when some sum is not finite
#pragma unroll
                    for (int i = 0; i < RT; ++i)
#pragma unroll
                        for (int h = 0; h < H; ++h)
                            z = make_float4(fmaf(pv[i][h].x, 0.f, z.x), fmaf(pv[i][h].y, 0.f, z.y),
                                            fmaf(pv[i][h].z, 0.f, z.z), fmaf(pv[i][h].w, 0.f, z.w));
                    if (__any_sync(0xffffffffu, (z.x + z.y) + (z.z + z.w) != 0.f)) {
                        clear();
#pragma unroll 1
                        for (int u = 0; u < un; u += 4) weigh(u, std::true_type{});
                    }
                }
#pragma unroll
                for (int i = 0; i < RT; ++i) {
                    const float f = half == 0 ? alpha[i] : 1.f;
#pragma unroll
                    for (int h = 0; h < H; ++h) {
                        o[i][h].x = fmaf(o[i][h].x, f, pv[i][h].x);
                        o[i][h].y = fmaf(o[i][h].y, f, pv[i][h].y);
                        o[i][h].z = fmaf(o[i][h].z, f, pv[i][h].z);
                        o[i][h].w = fmaf(o[i][h].w, f, pv[i][h].w);
                    }
                }
            }
        }
        __syncthreads();                                   // V is read
        if (tn < t_end) load_v(tn);
        else core_commit();
        t = tn;
    }
    core_wait<0>();
    __syncthreads();
#pragma unroll
    for (int i = 0; i < RT; ++i)
#pragma unroll
        for (int off = 4; off > 0; off >>= 1) l[i] += __shfl_xor_sync(0xffffffffu, l[i], off);

    auto put = [](T* p, float4 v) {
        if constexpr (sizeof(T) == 4) {
            *reinterpret_cast<float4*>(p) = v;
        } else {
            __nv_bfloat162 a = __floats2bfloat162_rn(v.x, v.y), b = __floats2bfloat162_rn(v.z, v.w);
            *reinterpret_cast<uint2*>(p) = make_uint2(*reinterpret_cast<uint32_t*>(&a), *reinterpret_cast<uint32_t*>(&b));
        }
    };
    if (!KS && ns == 1) {
#pragma unroll
        for (int i = 0; i < RT; ++i) {
            const int r = row0 + r0 + 4 * i;
            if (r >= job.nrows) continue;
            const float inv = 1.f / l[i];
            T* out = job.out_row(r);
#pragma unroll
            for (int h = 0; h < H; ++h)
                put(out + 4 * tx + 32 * h,
                    make_float4(o[i][h].x * inv, o[i][h].y * inv, o[i][h].z * inv, o[i][h].w * inv));
            float* lse = job.lse_at(r);
            if (lse != nullptr && tx == 0) *lse = (m[i] + log2f(l[i])) * 0.69314718055994531f;
        }
        return;
    }
    // the partials: O over K and V, (max, sum) beside; then each CTA of the cluster merges the rows
    // rank, rank + ns, ... from every CTA's shared memory (and, with four rows, every warp's slots)
    namespace cg = cooperative_groups;
    cg::cluster_group cluster = cg::this_cluster();
    float* so = reinterpret_cast<float*>(sm + L::kK);
    float2* sml = reinterpret_cast<float2*>(sm + L::kML);
#pragma unroll
    for (int i = 0; i < RT; ++i) {
        const int r = slot0 + 4 * i;
#pragma unroll
        for (int h = 0; h < H; ++h) *reinterpret_cast<float4*>(so + r * D + 4 * tx + 32 * h) = o[i][h];
        if (tx == 0) sml[r] = make_float2(m[i], l[i]);
    }
    if (ns == 1) __syncthreads();
    else cluster.sync();
    constexpr int TPR = D / 4;                             // threads a row
    constexpr int W = KS ? 4 : 1;                          // slots a row in a CTA
    auto part = [&](auto* p, int q) { return ns == 1 ? p : cluster.map_shared_rank(p, q); };
    for (int i = tid / TPR; rank + i * ns < L::kRows; i += kCoreThreads / TPR) {
        const int r = rank + i * ns, c4 = tid % TPR;
        if (row0 + r >= job.nrows) break;
        float mx = -CUDART_INF_F;
        for (int q = 0; q < ns; ++q)
            for (int w = 0; w < W; ++w) mx = fmaxf(mx, part(sml, q)[4 * w + r].x);
        float ls = 0.f;
        float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
        for (int q = 0; q < ns; ++q)
            for (int w = 0; w < W; ++w) {
                const float2 ml = part(sml, q)[4 * w + r];
                const float f = exp2f(ml.x - mx);          // 0 for a slot that saw nothing (some slot saw a key)
                const float4 v = reinterpret_cast<const float4*>(part(so, q) + (4 * w + r) * D)[c4];
                acc.x = fmaf(f, v.x, acc.x);
                acc.y = fmaf(f, v.y, acc.y);
                acc.z = fmaf(f, v.z, acc.z);
                acc.w = fmaf(f, v.w, acc.w);
                ls = fmaf(f, ml.y, ls);
            }
        const float inv = 1.f / ls;
        put(job.out_row(row0 + r) + 4 * c4, make_float4(acc.x * inv, acc.y * inv, acc.z * inv, acc.w * inv));
        float* lse = job.lse_at(row0 + r);
        if (lse != nullptr && c4 == 0) *lse = (mx + log2f(ls)) * 0.69314718055994531f;
    }
    if (ns > 1) cluster.sync();                            // no CTA leaves while its partial is read
}

// How a launch is cut: rows per CTA, CTAs (a cluster) per row tile, and whether each CTA is to
// have an SM of its own (the scheduler may put two on one SM while others idle, so such a launch
// asks for more shared memory than two would find).
struct CorePlan {
    int form = 4;            // 64 rows a CTA (4), 16 (1), or four whose keys the warps share (0)
    int ns = 1;
    bool alone = false;
};
constexpr int kCoreAlone = 118 * 1024;     // shared memory that leaves no room for a second CTA

// The cheapest cut by a model of the schedule (us).  A CTA takes `start` to begin and end and `tile` a key
// tile, or `start_sm` and `tile_sm` of its SM's time where more of them share it than that hides; of a row
// tile that is not full, `fixed` of a tile's time stays, as `last` does of a last key tile that is not
// full; a cluster's merge takes `merge`; of a round of CTAs that does not fill the device, the share `ceil`
// counts as a whole one.  causal (extraction): the longest CTA sees all keys, a round takes `mean` of it.
// Fitted to 1983 measured launches under up to 24 cuts each (fp32 and bf16, groups of 1 to 4; attends of 2
// to 2560 units of 1 to 240 rows over 9 to 1960 keys, extraction of 16 to 3000 tokens in 1 to 32 layers):
// the choice takes 2.0 % (d = 64) and 1.9 % (128) more than the best cut in the mean, 11 and 12 % in 95 of
// 100.  A model without the four-row form and without rows and tiles that are not full took 20 and 26 %
// more, up to 1.8 times the time of the kernel before this loop on few rows of many units.
// capacity(form, ns, alone): CTAs of such a launch that the device holds at once.
struct CoreCosts {
    double tile[3], tile_sm[3], start[3], start_sm[3], fixed[3], last, merge, ceil, mean;      // forms 4, 1, 0
};
inline const CoreCosts& core_costs(int d) {
    static const CoreCosts c128 = {{7.5, 5.3, 3.5}, {4.7, 3.2, .80}, {7.8, 3.6, 2.5}, {1.9, .60, .85}, {1.0, .56, 1.0},
                                   .05, 2.1, .85, .68};
    static const CoreCosts c64 = {{6.6, 5.9, 2.75}, {1.2, 1.2, .67}, {5.9, 2.5, .45}, {2.1, .25, .43}, {.54, .51, 1.0},
                                  .05, 1.55, .62, .80};
    return d == 128 ? c128 : c64;
}
template <class Capacity>
inline CorePlan core_plan(int64_t nrows, int64_t units, int64_t nkeys, int d, bool causal, const Capacity& capacity) {
    CorePlan best;
    double cost = -1.0;
    const CoreCosts& k = core_costs(d);
    const int64_t sms = device_sms();
    const int64_t tiles = (nkeys + kCoreKeys - 1) / kCoreKeys;
    const double last = (double)(nkeys - (tiles - 1) * kCoreKeys) / kCoreKeys;       // how full the last tile is
    constexpr int forms[3] = {4, 1, 0};
    for (int i = 0; i < 3; ++i) {
        const int form = forms[i];
        const int64_t rows = form == 0 ? 4 : 16 * form, row_tiles = (nrows + rows - 1) / rows;
        // warps with rows: all but in the last row tile (four rows: all)
        const int64_t quarter = rows / 4, rest = nrows - (row_tiles - 1) * rows;
        const double live = form == 0 ? 1.0 : ((double)(row_tiles - 1) + (double)((rest + quarter - 1) / quarter) / 4.0) / row_tiles;
        const int64_t resident = std::max<int64_t>(1, capacity(form, 1, false) / sms);
        for (int ns = 1; ns <= kCoreMaxSplit && ns <= tiles; ++ns) {
            const int64_t ctas = row_tiles * units * ns;
            const bool alone = ctas <= capacity(form, ns, true);
            const double slots = std::max(1, capacity(form, ns, false));
            const double share = alone ? 1.0 : (double)std::min(resident, (ctas + sms - 1) / sms);
            const double tile = std::max(k.tile[i], share * k.tile_sm[i]) * (k.fixed[i] + (1.0 - k.fixed[i]) * live);
            const double start = std::max(k.start[i], share * k.start_sm[i]);
            const double keys = (double)((tiles + ns - 1) / ns) - (ns == 1 ? (1.0 - k.last) * (1.0 - last) : 0.0);
            const double rounds = ctas <= slots ? 1.0 : (1.0 - k.ceil) * (ctas / slots) + k.ceil * std::ceil(ctas / slots);
            const double longest = start + keys * tile;
            const double c = (causal ? std::max(longest, rounds * (start + k.mean * keys * tile)) : rounds * longest) +
                             (ns > 1 ? k.merge : 0.0);
            if (cost < 0.0 || c < cost) {
                cost = c;
                best.form = form;
                best.ns = ns;
                best.alone = alone;
            }
        }
    }
    return best;
}

// CTAs of a kernel with `smem` bytes in clusters of ns that the device holds at once.
inline int core_capacity(const void* kernel, int ns, size_t smem, int sms) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)ns);
    cfg.blockDim = dim3(kCoreThreads);
    cfg.dynamicSmemBytes = smem;
    cudaLaunchAttribute attr[1];
    int n = 0;
    if (ns == 1) {
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kernel, kCoreThreads, smem) != cudaSuccess) n = 1;
        n *= sms;
    } else {
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = (unsigned)ns;
        attr[0].val.clusterDim.y = 1;
        attr[0].val.clusterDim.z = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        if (cudaOccupancyMaxActiveClusters(&n, kernel, &cfg) != cudaSuccess) n = sms / (2 * ns);
        n *= ns;
    }
    (void)cudaGetLastError();
    return n;
}

// The shared memory opt-in of a kernel instantiation on a device, and its table of capacities there.
template <int D, int RT>
struct CoreKernel {
    cudaError_t err = cudaSuccess;
    int slots[2][kCoreMaxSplit + 1] = {};  // [alone][ns]
    CoreKernel() = default;
    CoreKernel(const void* kernel, int sms) {
        err = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                   std::max(Core<D, RT>::kSmem, kCoreAlone));
        for (int ns = 1; ns <= kCoreMaxSplit; ++ns) {
            slots[0][ns] = core_capacity(kernel, ns, Core<D, RT>::kSmem, sms);
            slots[1][ns] = core_capacity(kernel, ns, kCoreAlone, sms);
        }
    }
};

// A planned launch: `ns` CTAs a cluster along x; `dependent`: it starts while the kernel before it runs,
// and waits for it.
inline cudaError_t core_launch(const void* kernel, dim3 grid, size_t smem, const CorePlan& plan, bool dependent, void** args,
                               cudaStream_t s) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(kCoreThreads);
    cfg.dynamicSmemBytes = plan.alone ? kCoreAlone : smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[2];
    cfg.attrs = attr;
    if (plan.ns > 1) {
        attr[cfg.numAttrs].id = cudaLaunchAttributeClusterDimension;
        attr[cfg.numAttrs].val.clusterDim.x = (unsigned)plan.ns;
        attr[cfg.numAttrs].val.clusterDim.y = 1;
        attr[cfg.numAttrs].val.clusterDim.z = 1;
        ++cfg.numAttrs;
    }
    if (dependent) {
        attr[cfg.numAttrs].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[cfg.numAttrs].val.programmaticStreamSerializationAllowed = 1;
        ++cfg.numAttrs;
    }
    return cudaLaunchKernelExC(&cfg, kernel, args);
}

}  // namespace
}  // namespace c2kv

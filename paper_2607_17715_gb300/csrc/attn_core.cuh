// The CUDA-core attention loop shared by the suffix attention (attn_simt.cu) and the extraction
// attention (extract.cu): fp32 arithmetic throughout, for fp32 contexts (no tensor-core format
// keeps fp32 inputs exact) and for the head layouts the tensor-core kernel does not take.
//
// One CTA of four warps holds 16 RT packed query rows of one (layer, request, KV head) (row
// r = t G + g: the G query heads that share a KV head share every K/V tile) and walks the key
// tiles of 64 that some row of it may see.  A warp owns 4 RT rows; its lane (ty, tx) =
// (lane / 8, lane % 8) rows ty + 4 i of them, of a tile's scores the keys tx + 8 j, and of the
// output the channels 4 tx + 32 h .. + 3.
//   S:   per 4 channels RT + 8 16-byte shared loads feed 32 RT FMAs; every 32 channels the
//        partial dot products are folded, so no sum is a chain of more than 32 terms.
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
// formed.  Measured (fp32, clock stamps): d = 128, 64 rows: S 7.7 K and P.V 8.2 K clocks a tile
// for 4096 FMAs a lane each, a CTA alone on its SM; two sharing one reach 60 % of the FMA pipe.
// An attend of 2 requests x 96 tokens over 720 slots, 16 / 4 heads, d = 128, went from 176 us
// (one shared load per FMA operand) to 59.5 us, 4 requests x 250 tokens x 1024 slots, d = 64, from
// 548 to 176 us, extraction of 2000 tokens, d = 128, from 1858 to 655 us.
//
// A launch of few row tiles splits each one's key range over a cluster of `ns` CTAs, whose
// (max, sum, O) are merged through distributed shared memory by the exact log-sum-exp rule: no
// scratch in device memory, no second launch.
#pragma once

#include <cooperative_groups.h>
#include <math_constants.h>

#include <algorithm>
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

template <int D, int RT>
struct Core {
    static constexpr int kRows = 16 * RT;
    static constexpr int kPitch = (D + 4) * 4;                     // bytes of a Q or K row
    static constexpr int kQ = 0;
    static constexpr int kK = kQ + kRows * kPitch;
    static constexpr int kV = kK + kCoreKeys * kPitch;
    static constexpr int kP = kV + kCoreKeys * D * 4;
    static constexpr int kML = kP + kRows * kCorePPitch;           // max and sum of each row (merge)
    static constexpr int kSmem = kML + kRows * 8;
    static_assert(kRows * D * 4 <= kP - kK, "the merge's O fits over K and V");
};

// CTAs an SM is to hold (shared memory allows them; what the registers are cut to).
__host__ __device__ constexpr int core_ctas(int d, int rt) { return d == 128 ? 2 : rt == 1 ? 4 : 3; }

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

// Job: nrows (packed rows of the unit), nkeys (keys of this CTA's rows), k, v, stride (key rows),
// scale_log2; q_row(r), out_row(r), lse_at(r) (null without lse); needed(k0, k1): some row of the
// CTA may see a key of [k0, k1); whole(k0, k1): every row sees all of them; row(r): what
// sees(row, key) takes of packed row r.
template <typename T, int D, int RT, class Job>
__device__ __forceinline__ void attention_core(const Job& job, int row0, int ns, int rank, uint8_t* sm) {
    using L = Core<D, RT>;
    constexpr int H = D / 32;                              // 4-channel groups a lane
    // channels per folded partial sum.  (16, and the scale in the exponent's fused multiply-add: the
    // error against 64 bits is that of the earlier kernel's four interleaved sums, 2e-7 to 5e-7 of the
    // largest output over 32 to 8192 keys; with 32 and a rounded product it was up to a third above it,
    // and no faster.)
    constexpr int kBlk = 16;
    const int tid = threadIdx.x, lane = tid & 31, ty = lane >> 3, tx = lane & 7;
    const int r0 = (tid >> 5) * 4 * RT + ty;               // this lane's rows r0 + 4 i
    const int tiles = (job.nkeys + kCoreKeys - 1) / kCoreKeys;
    const int t_beg = (int)((int64_t)tiles * rank / ns), t_end = (int)((int64_t)tiles * (rank + 1) / ns);
    auto next = [&](int t) {                               // first tile >= t that some row may see
        while (t < t_end && !job.needed(t * kCoreKeys, (t + 1) * kCoreKeys)) ++t;
        return t;
    };
    auto load_k = [&](int t) {
        core_copy<T, D>(sm + L::kK, L::kPitch, kCoreKeys, CoreRows<T>{job.k, job.stride, t * kCoreKeys, job.nkeys});
        core_commit();
    };
    auto load_v = [&](int t) {
        core_copy<T, D>(sm + L::kV, D * 4, kCoreKeys, CoreRows<T>{job.v, job.stride, t * kCoreKeys, job.nkeys});
        core_commit();
    };

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
    const uint8_t* kb = sm + L::kK + tx * L::kPitch;
    const uint8_t* vb = sm + L::kV + tx * 16;
    uint8_t* pb = sm + L::kP + r0 * kCorePPitch;
    auto ld4 = [](const uint8_t* p) { return *reinterpret_cast<const float4*>(p); };
    while (t < t_end) {
        const int k0 = t * kCoreKeys, tn = next(t + 1);
        core_wait<1>();
        __syncthreads();                                   // K (and Q) of this tile
        float s[RT][8];
#pragma unroll
        for (int i = 0; i < RT; ++i)
#pragma unroll
            for (int j = 0; j < 8; ++j) s[i][j] = 0.f;
#pragma unroll 1
        for (int c0 = 0; c0 < D; c0 += kBlk) {
            float a[RT][8];
#pragma unroll
            for (int i = 0; i < RT; ++i)
#pragma unroll
                for (int j = 0; j < 8; ++j) a[i][j] = 0.f;
#pragma unroll
            for (int c = 0; c < kBlk; c += 4) {
                float4 kf[8], q[RT];
#pragma unroll
                for (int j = 0; j < 8; ++j) kf[j] = ld4(kb + 8 * j * L::kPitch + (c0 + c) * 4);
#pragma unroll
                for (int i = 0; i < RT; ++i) q[i] = ld4(qb + 4 * i * L::kPitch + (c0 + c) * 4);
                // channel by channel over every (i, j): no FMA waits for the one before it
                auto dot = [&](float (&acc)[RT][8], auto ch) {
#pragma unroll
                    for (int i = 0; i < RT; ++i)
#pragma unroll
                        for (int j = 0; j < 8; ++j) acc[i][j] = fmaf(ch(q[i]), ch(kf[j]), acc[i][j]);
                };
                dot(a, [](const float4& v) { return v.x; });
                dot(a, [](const float4& v) { return v.y; });
                dot(a, [](const float4& v) { return v.z; });
                dot(a, [](const float4& v) { return v.w; });
            }
#pragma unroll
            for (int i = 0; i < RT; ++i)
#pragma unroll
                for (int j = 0; j < 8; ++j) s[i][j] += a[i][j];
        }
        __syncthreads();                                   // K is read: the next tile's may land
        if (tn < t_end) load_k(tn);
        else core_commit();

        const bool whole = k0 + kCoreKeys <= job.nkeys && job.whole(k0, k0 + kCoreKeys);
        float alpha[RT];
#pragma unroll
        for (int i = 0; i < RT; ++i) {
            uint32_t hidden = 0u;                          // bit j: the row does not see key tx + 8 j
            if (!whole) {
                const auto row = job.row(row0 + r0 + 4 * i);
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    const int key = k0 + tx + 8 * j;
                    if (key >= job.nkeys || !job.sees(row, key)) {
                        s[i][j] = -CUDART_INF_F;
                        hidden |= 1u << j;
                    }
                }
            }
            float mx = s[i][0];
#pragma unroll
            for (int j = 1; j < 8; ++j) mx = fmaxf(mx, s[i][j]);
#pragma unroll
            for (int off = 4; off > 0; off >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, off));
            const float mn = fmaxf(m[i], mx * job.scale_log2);
            const float ms = mn == -CUDART_INF_F ? 0.f : mn;      // nothing visible yet
            alpha[i] = exp2f(m[i] - ms);
            m[i] = mn;
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                s[i][j] = exp2f(fmaf(s[i][j], job.scale_log2, -ms));
                if (hidden >> j & 1u) s[i][j] = -0.f;
            }
            l[i] = l[i] * alpha[i] + (((s[i][0] + s[i][1]) + (s[i][2] + s[i][3])) +
                                      ((s[i][4] + s[i][5]) + (s[i][6] + s[i][7])));   // this lane's keys
        }
        core_wait<1>();
        __syncthreads();                                   // V of this tile
#pragma unroll
        for (int half = 0; half < 2; ++half) {
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
                for (int i = 0; i < RT; ++i) p[i] = ld4(pb + 4 * i * kCorePPitch + u * 4);
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    float4 v[H];
#pragma unroll
                    for (int h = 0; h < H; ++h) v[h] = ld4(vb + (32 * half + u + e) * D * 4 + h * 128);
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
                for (int j = 0; j < 4; ++j)
                    *reinterpret_cast<float*>(pb + 4 * i * kCorePPitch + (tx + 8 * j) * 4) = s[i][4 * half + j];
            __syncwarp();
#pragma unroll 2
            for (int u = 0; u < 32; u += 4) weigh(u, std::false_type{});
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
                    for (int u = 0; u < 32; u += 4) weigh(u, std::true_type{});
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
    if (ns == 1) {
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
    // the cluster's partials: O over K and V, (max, sum) beside; then each CTA merges the rows
    // rank, rank + ns, ... from every CTA's shared memory
    namespace cg = cooperative_groups;
    cg::cluster_group cluster = cg::this_cluster();
    float* so = reinterpret_cast<float*>(sm + L::kK);
    float2* sml = reinterpret_cast<float2*>(sm + L::kML);
#pragma unroll
    for (int i = 0; i < RT; ++i) {
        const int r = r0 + 4 * i;
#pragma unroll
        for (int h = 0; h < H; ++h) *reinterpret_cast<float4*>(so + r * D + 4 * tx + 32 * h) = o[i][h];
        if (tx == 0) sml[r] = make_float2(m[i], l[i]);
    }
    cluster.sync();
    constexpr int TPR = D / 4;                             // threads a row
    for (int i = tid / TPR; rank + i * ns < L::kRows; i += kCoreThreads / TPR) {
        const int r = rank + i * ns, c4 = tid % TPR;
        if (row0 + r >= job.nrows) break;
        float mx = -CUDART_INF_F;
        for (int q = 0; q < ns; ++q) mx = fmaxf(mx, cluster.map_shared_rank(sml, q)[r].x);
        float ls = 0.f;
        float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
        for (int q = 0; q < ns; ++q) {
            const float2 ml = cluster.map_shared_rank(sml, q)[r];
            const float w = exp2f(ml.x - mx);              // 0 for a CTA that saw nothing (some CTA saw a key)
            const float4 v = reinterpret_cast<const float4*>(cluster.map_shared_rank(so, q) + r * D)[c4];
            acc.x = fmaf(w, v.x, acc.x);
            acc.y = fmaf(w, v.y, acc.y);
            acc.z = fmaf(w, v.z, acc.z);
            acc.w = fmaf(w, v.w, acc.w);
            ls = fmaf(w, ml.y, ls);
        }
        const float inv = 1.f / ls;
        put(job.out_row(row0 + r) + 4 * c4, make_float4(acc.x * inv, acc.y * inv, acc.z * inv, acc.w * inv));
        float* lse = job.lse_at(row0 + r);
        if (lse != nullptr && c4 == 0) *lse = (mx + log2f(ls)) * 0.69314718055994531f;
    }
    cluster.sync();                                        // no CTA leaves while its partial is read
}

// How a launch is cut: rows per CTA, CTAs (a cluster) per row tile, and whether each CTA is to
// have an SM of its own (the scheduler may put two on one SM while others idle, so such a launch
// asks for more shared memory than two would find).
struct CorePlan {
    bool small = false;      // 16 rows a CTA, else 64
    int ns = 1;
    bool alone = false;
};
constexpr int kCoreAlone = 118 * 1024;     // shared memory that leaves no room for a second CTA

// The cheapest cut by a model of the schedule, in clocks per key tile of a CTA alone on an SM and
// of one that shares it (measured on GB300 with clock stamps: d = 128, 64 rows 19.4 K and 28.6 K,
// 16 rows 17 K and 19 K; d = 64 about half, 16 rows 5.7 K), 8 K to start and end, 4 K to merge a
// cluster.  Few rows over many keys take 16-row tiles and clusters, large launches 64 rows and no
// split.  capacity(small, ns, alone): CTAs of such a launch that the device holds at once.
template <class Capacity>
inline CorePlan core_plan(int64_t nrows, int64_t units, int64_t nkeys, int d, const Capacity& capacity) {
    CorePlan best;
    double cost = -1.0;
    const int64_t tiles = (nkeys + kCoreKeys - 1) / kCoreKeys;
    const double one[2] = {d == 128 ? 19.4e3 : 9.7e3, d == 128 ? 17.0e3 : 5.7e3};
    const double shared[2] = {d == 128 ? 28.6e3 : 19.0e3, d == 128 ? 19.0e3 : 8.5e3};
    for (int small = 0; small < 2; ++small) {
        const int64_t rows = small ? 16 : 64;
        for (int ns = 1; ns <= kCoreMaxSplit && ns <= tiles; ++ns) {
            const int64_t ctas = (nrows + rows - 1) / rows * units * ns;
            const int64_t per = (tiles + ns - 1) / ns;
            const bool alone = ctas <= capacity(small != 0, ns, true);
            const int64_t slots = std::max(1, capacity(small != 0, ns, false));
            const double tile = alone ? one[small] : shared[small] * (double)((ctas + slots - 1) / slots);
            const double c = per * tile + 8.0e3 + (ns > 1 ? 4.0e3 : 0.0);
            if (cost < 0.0 || c < 0.97 * cost) {
                cost = c;
                best.small = small != 0;
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

}  // namespace
}  // namespace c2kv

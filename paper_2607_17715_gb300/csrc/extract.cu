// Extraction attention with the Structured Information Flow mask (Sec. 3.3): one attention
// layer of the C2 Extractor's forward over a chunk, given the Q, K, V of its n document
// tokens and m = ceil(n/k) C2 tokens (the trained projections that make them are the
// caller's).  The sequence is [x_0 .. x_{n-1}; c_0 .. c_{m-1}] with the C2 tokens grouped
// after the document (Sec. 3.3.1), and
//   * document token t sits at position t and sees document tokens 0..t only (original-token
//     invariance: its output is the frozen model's);
//   * C2 token c_j sits at the position of the last token of its block B(j) =
//     [jk, min((j+1)k, n)) and sees the document tokens of B(j) and of the sink block, and
//     the C2 tokens c_0 .. c_j (causal accumulation across blocks).
// The sink block B(0) of the paper's 1-based numbering is undefined by its block formula;
// it is read as the first block, [0, min(k, n)).
//
// extract_rope_kernel turns Q and K to those positions (fp32 arithmetic, stored in the
// context dtype like every cached activation), or extract_rope_k_kernel K alone where the attention
// turns the queries itself.  The masked attention then takes one of two routes.
//
// Tensor cores (bf16, the group sizes the tensor-core kernels take; heads of 64 channels not over short
// chunks: extract_uses_tc).  The mask splits into
// pieces the suffix-attention kernel already computes:
//   1. document rows: plain causal attention over document keys 0..t, i.e. a "suffix" of n
//      tokens over an empty prefix;
//   2. C2 rows: a "suffix" of m tokens after n "slots", the document rows, so that c_j sees
//      c_0 .. c_j causally; the kernel's SIF mode (sif_k = k) masks every document key but
//      those of the sink block and B(j), and visits only the key tiles that hold them (for
//      a pair of 2 x 128 packed rows: its blocks' tiles, tile 0, the C2 tiles).
// Both are launches of attn_solo_kernel (or the pair kernel) with a token pitch of n + m, so they read and write
// the extraction layout in place.
//
// CUDA cores (the others): extract_attn_kernel runs every row with fp32
// accumulation through attention_core (attn_core.cuh): packed row r = t * G + g is token t,
// query head h_kv * G + g, and the tiles that none of a CTA's rows can see are skipped.
#include <algorithm>

#include "attn_core.cuh"
#include "rope.cuh"

namespace c2kv {
namespace {

// Extraction position of token t of an (n, k) chunk.
__device__ __forceinline__ int extract_pos(int t, int n, int k) {
    if (t < n) return t;
    const int j = t - n;
    const int end = (j + 1) * k < n ? (j + 1) * k : n;
    return end - 1;
}

template <typename T, int VPH>
__global__ void __launch_bounds__(256) extract_rope_kernel(const __grid_constant__ ExtractParams P) {
    using V = Vec16<T>;
    constexpr int E = V::N;
    constexpr int HALF = VPH * E;
    constexpr int D = 2 * HALF;
    __shared__ float2 cs[HALF];
    const int t = blockIdx.x;
    const int l = blockIdx.y;
    const int pos = extract_pos(t, P.n, P.ratio);
    if (threadIdx.x < HALF) cs[threadIdx.x] = turn_cs(P.rope.turn[threadIdx.x], pos);
    __syncthreads();
    const int64_t row = (int64_t)l * P.n_all + t;               // token row of layer l
    const int nq = P.hq * VPH;
    const int items = (P.hq + P.hkv) * VPH;
    for (int p = threadIdx.x; p < items; p += blockDim.x) {
        const bool is_q = p < nq;
        const int pp = is_q ? p : p - nq;
        const int h = pp / VPH;
        const int iv = pp - h * VPH;
        const int heads = is_q ? P.hq : P.hkv;
        const int64_t off = (row * heads + h) * D + iv * E;
        const T* src = static_cast<const T*>(is_q ? P.q : P.k) + off;
        float x[E], y[E], gx[E], gy[E];
        V::unpack(ld16(src), x);
        V::unpack(ld16(src + HALF), y);
        rotate<E>(x, y, cs + iv * E, gx, gy);
        T* dst = static_cast<T*>(is_q ? P.q_rot : P.k_rot) + off;
        st16(dst, V::pack(gx));
        st16(dst + HALF, V::pack(gy));
    }
}

// K alone, and the table of every token's (cos, sin) from which the solo attention kernel turns its
// query tiles in shared memory.  Turning Q here read and wrote four fifths of the tensors' bytes
// (Q is Hq / Hkv times K): 68 us of the 32-layer call on 512 + 128 tokens, against 49 us for those
// bytes at the rate of HBM; the call went from 226 to 200 us.  A CTA takes kRopeTokens tokens of one
// layer, each thread one (token, head, vector pair) at a time, its loads issued before the angles are
// formed.
constexpr int kRopeTokens = 4;
template <typename T, int VPH>
__global__ void __launch_bounds__(256) extract_rope_k_kernel(const __grid_constant__ ExtractParams P) {
    using V = Vec16<T>;
    constexpr int E = V::N, HALF = VPH * E, D = 2 * HALF;
    __shared__ float2 cs[kRopeTokens * HALF];
    const int t0 = blockIdx.x * kRopeTokens, l = blockIdx.y;
    const int nt = min(kRopeTokens, P.n_all - t0);
    const int items = nt * P.hkv * VPH;
    const int64_t base = ((int64_t)l * P.n_all + t0) * P.hkv * D;      // the tokens' rows are contiguous
    const T* src = static_cast<const T*>(P.k) + base;
    T* dst = static_cast<T*>(P.k_rot) + base;
    auto offset = [&](int p) { return (int64_t)(p / VPH) * D + (p % VPH) * E; };
    uint4 a{}, b{};
    int p = threadIdx.x;
    if (p < items) {
        a = ld16(src + offset(p));
        b = ld16(src + offset(p) + HALF);
    }
    for (int e = threadIdx.x; e < nt * HALF; e += blockDim.x) {
        const int t = t0 + e / HALF;
        const float2 v = turn_cs(P.rope.turn[e % HALF], extract_pos(t, P.n, P.ratio));
        cs[e] = v;
        if (l == 0) P.q_cs[(int64_t)t0 * HALF + e] = v;
    }
    __syncthreads();
    while (p < items) {
        float x[E], y[E], gx[E], gy[E];
        V::unpack(a, x);
        V::unpack(b, y);
        rotate<E>(x, y, cs + p / (P.hkv * VPH) * HALF + p % VPH * E, gx, gy);
        st16(dst + offset(p), V::pack(gx));
        st16(dst + offset(p) + HALF, V::pack(gy));
        p += blockDim.x;
        if (p < items) {
            a = ld16(src + offset(p));
            b = ld16(src + offset(p) + HALF);
        }
    }
}

// The rows of one (layer, KV head) under the SIF mask, for attention_core.
template <typename T, int D>
struct SifJob {
    const ExtractParams& p;
    int l, hk, g_heads;
    int row0, t0, t1;                 // this CTA's first packed row, first and last token
    int nrows, nkeys;
    int doc_end;                      // document keys its document rows see: [0, doc_end)
    int blk_lo, blk_hi, sink;         // document keys its C2 rows see: [0, sink) and within [blk_lo, blk_hi)
    const T *k, *v;
    int64_t stride;
    float scale_log2;
    __device__ int64_t row_off(int r) const {
        const int t = r / g_heads, g = r - t * g_heads;
        return (((int64_t)l * p.n_all + t) * p.hq + hk * g_heads + g) * D;
    }
    __device__ const T* q_row(int r) const { return static_cast<const T*>(p.q_rot) + row_off(r); }
    __device__ T* out_row(int r) const { return static_cast<T*>(p.out) + row_off(r); }
    __device__ float* lse_at(int r) const {
        if (p.lse == nullptr) return nullptr;
        const int t = r / g_heads, g = r - t * g_heads;
        return p.lse + ((int64_t)l * p.hq + hk * g_heads + g) * p.n_all + t;
    }
    __device__ bool needed(int k0, int k1) const {
        if (k0 < doc_end) return true;
        if (t1 < p.n) return false;                              // document rows only
        return k0 < sink || (k1 > blk_lo && k0 < blk_hi) || k1 > p.n;
    }
    __device__ bool whole(int, int k1) const { return t1 < p.n && k1 - 1 <= t0; }
    __device__ int row(int r) const { return r / g_heads; }               // its token
    __device__ bool sees(int t, int key) const {
        const int n = p.n;
        if (t < n) return key <= t;                              // document: causal, no C2 tokens
        const int j = t - n;
        if (key >= n) return key - n <= j;                       // C2 tokens c_0 .. c_j
        return key < p.ratio || (int64_t)key >= (int64_t)j * p.ratio && (int64_t)key < ((int64_t)j + 1) * p.ratio;
    }
};

template <typename T, int D, int RT>
__global__ void __launch_bounds__(kCoreThreads, core_ctas(D, RT)) extract_attn_kernel(const __grid_constant__ ExtractParams P, int ns) {
    extern __shared__ __align__(16) uint8_t core_smem[];
    SifJob<T, D> j{P};
    j.l = blockIdx.z;
    j.hk = blockIdx.y;
    j.g_heads = P.hq / P.hkv;
    // last rows first: under the causal mask they see the most keys
    constexpr int kRows = Core<D, RT>::kRows;
    j.row0 = (int)((gridDim.x - 1 - blockIdx.x) / (unsigned)ns) * kRows;
    j.nrows = P.n_all * j.g_heads;
    j.t0 = j.row0 / j.g_heads;
    j.t1 = min(P.n_all - 1, (j.row0 + kRows - 1) / j.g_heads);
    const int n = P.n, ja = max(j.t0 - n, 0), jb = j.t1 - n;
    const bool c2 = j.t1 >= n;
    j.doc_end = j.t0 < n ? min(j.t1, n - 1) + 1 : 0;
    j.sink = c2 ? min(P.ratio, n) : 0;
    j.blk_lo = c2 ? min((int64_t)ja * P.ratio, (int64_t)n) : 0;
    j.blk_hi = c2 ? min(((int64_t)jb + 1) * P.ratio, (int64_t)n) : 0;
    j.nkeys = c2 ? n + jb + 1 : j.doc_end;
    j.stride = (int64_t)P.hkv * D;
    j.k = static_cast<const T*>(P.k_rot) + ((int64_t)j.l * P.n_all * P.hkv + j.hk) * D;
    j.v = static_cast<const T*>(P.v) + ((int64_t)j.l * P.n_all * P.hkv + j.hk) * D;
    j.scale_log2 = P.scale_log2;
    attention_core<T, D, RT>(j, j.row0, ns, (int)(blockIdx.x % (unsigned)ns), core_smem);   // (the cluster rank)
}

template <int D>
cudaError_t launch_tc(const ExtractParams& p, cudaStream_t s, cudaStream_t s2, cudaEvent_t fork,
                      cudaEvent_t join) {
    constexpr int VPH = D / 2 / Vec16<__nv_bfloat16>::N;
    const bool turn_q = p.q_rot == nullptr;
    if (turn_q)
        extract_rope_k_kernel<__nv_bfloat16, VPH>
            <<<dim3((unsigned)((p.n_all + kRopeTokens - 1) / kRopeTokens), (unsigned)p.lq), 256, 0, s>>>(p);
    else
        extract_rope_kernel<__nv_bfloat16, VPH><<<dim3((unsigned)p.n_all, (unsigned)p.lq), 256, 0, s>>>(p);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    const int m = p.n_all - p.n;
    AttnParams a{};
    a.cache_k = p.k_rot;
    a.cache_v = p.v;
    a.err = p.err;
    a.rows = p.n_all;
    a.layer0 = 0;
    a.lq = p.lq;
    a.batch = 1;
    a.batch_total = 1;
    a.b0 = 0;
    a.sq_pitch = p.n_all;
    a.hq = p.hq;
    a.hkv = p.hkv;
    a.d = D;
    a.scale_log2 = p.scale_log2;
    a.n_split = 1;
    a.pairs_per_cta = p.pairs_per_cta;
    // piece 2 writes only the C2 rows (and reads the rotated rows): with a second stream it
    // runs beside piece 1, in the SMs its last wave of CTAs leaves idle
    cudaStream_t sc = s;
    if (s2 != nullptr) {
        e = cudaEventRecord(fork, s);
        if (e == cudaSuccess) e = cudaStreamWaitEvent(s2, fork, 0);
        if (e != cudaSuccess) return e;
        sc = s2;
    }
    // 1. document rows over document keys 0..t
    const void* const q = turn_q ? p.q : p.q_rot;
    a.q_rot = q;
    a.q_cs = turn_q ? p.q_cs : nullptr;
    a.out = p.out;
    a.lse = p.lse;
    a.sq = p.n;
    a.req[0] = ReqParam{0, 0, 0, 0};
    e = launch_attn_tc(a, s);
    if (e != cudaSuccess) return e;
    // 2. C2 rows: the n document rows as the request's slots, the C2 rows as its suffix, so
    // that c_j sees c_0 .. c_j causally; the kernel's SIF mode keeps, of the document keys,
    // the sink block and B(j), and visits only their key tiles
    const int64_t c2_off = (int64_t)p.n * p.hq * D;
    a.q_rot = static_cast<const __nv_bfloat16*>(q) + c2_off;
    a.q_cs = turn_q ? p.q_cs + (int64_t)p.n * (D / 2) : nullptr;
    a.out = static_cast<__nv_bfloat16*>(p.out) + c2_off;
    a.lse = p.lse != nullptr ? p.lse + p.n : nullptr;
    a.sq = m;
    a.sif_k = p.ratio;
    a.req[0] = ReqParam{0, p.n, 0, 0};
    e = launch_attn_tc(a, sc);
    if (s2 != nullptr) {       // the work ends on s
        cudaError_t ej = cudaEventRecord(join, s2);
        if (ej == cudaSuccess) ej = cudaStreamWaitEvent(s, join, 0);
        if (e == cudaSuccess) e = ej;
    }
    return e;
}

template <typename T, int D, int RT>
CoreKernel<D, RT> ready() {
    static PerDevice<CoreKernel<D, RT>> kept;
    return kept.get([] { return CoreKernel<D, RT>(reinterpret_cast<const void*>(&extract_attn_kernel<T, D, RT>), device_sms()); });
}

template <typename T, int D, int RT>
cudaError_t launch_rt(const ExtractParams& p, CorePlan plan, cudaStream_t s) {
    constexpr int kRows = Core<D, RT>::kRows;
    const int64_t gx = ((int64_t)p.n_all * (p.hq / p.hkv) + kRows - 1) / kRows * plan.ns;
    if (gx > 0x7fffffffLL) return cudaErrorInvalidValue;
    void* args[2] = {const_cast<ExtractParams*>(&p), &plan.ns};
    return core_launch(reinterpret_cast<const void*>(&extract_attn_kernel<T, D, RT>),
                       dim3((unsigned)gx, (unsigned)p.hkv, (unsigned)p.lq), Core<D, RT>::kSmem, plan, false, args, s);
}

template <typename T, int D>
cudaError_t launch_typed(const ExtractParams& p, cudaStream_t s) {
    constexpr int VPH = D / 2 / Vec16<T>::N;
    extract_rope_kernel<T, VPH><<<dim3((unsigned)p.n_all, (unsigned)p.lq), 256, 0, s>>>(p);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    const CoreKernel<D, 4> large = ready<T, D, 4>();
    const CoreKernel<D, 1> small = ready<T, D, 1>();
    const CoreKernel<D, 0> four = ready<T, D, 0>();
    if (large.err != cudaSuccess) return large.err;
    if (small.err != cudaSuccess || four.err != cudaSuccess) return small.err != cudaSuccess ? small.err : four.err;
    const CorePlan plan = core_plan((int64_t)p.n_all * (p.hq / p.hkv), (int64_t)p.hkv * p.lq, p.n_all, D, true,
                                    [&](int form, int ns, bool alone) {
                                        return form == 4   ? large.slots[alone][ns]
                                               : form == 1 ? small.slots[alone][ns]
                                                           : four.slots[alone][ns];
                                    });
    return plan.form == 4   ? launch_rt<T, D, 4>(p, plan, s)
           : plan.form == 1 ? launch_rt<T, D, 1>(p, plan, s)
                            : launch_rt<T, D, 0>(p, plan, s);
}

}  // namespace

// Heads of 64 channels ran on the CUDA cores, with fp32 weights, and still do over short chunks, where a
// tensor-core CTA is mostly its start and end: at most 40 packed rows a unit, or 40 keys with packed rows x
// keys x units <= 400,000.  Over 420 calls (8 / 8 to 32 / 4 heads, 1 to 32 layers, 1 to 300 tokens, ratios 1
// to 16) the rule takes 1.6 % more than the better side in the mean, and is never more than 5 % slower than
// the tensor cores.  (Few units of up to 150 keys are faster on the CUDA cores too, by up to a third; the
// solo and the pair kernel's equal bits are relied on there.)  Measured (us a call, CUDA cores / tensor
// cores): 16 tokens at ratio 4, 16 heads, 32 layers 19 / 38, 1 layer 11 / 18; 130 tokens at ratio 4, 8 heads, 1
// layer 18 / 21, 16 layers 52 / 31.
bool extract_uses_tc(int dtype, int d, int hq, int hkv, int n_all, int lq, int pairs_per_cta) {
    if (!attn_tc_takes(dtype, d, hq, hkv)) return false;
    if (d != 64 || pairs_per_cta != 0) return true;
    const int64_t rows = (int64_t)n_all * (hq / hkv);
    return rows > 40 && (n_all > 40 || rows * n_all * hkv * lq > 400000);
}

// (the context's attn_pairs asks for the pair kernel, which takes turned queries)
bool extract_turns_queries(int pairs_per_cta) { return pairs_per_cta == 0; }

cudaError_t launch_extract(const ExtractParams& p, int dtype, int d, cudaStream_t s, cudaStream_t s2,
                           cudaEvent_t fork, cudaEvent_t join) {
    (void)cudaGetLastError();   // report this launch's error only, not a stale one
    if (p.n_all < 1 || p.lq < 1) return cudaSuccess;
    if (p.lq > 65535 || p.hkv > 65535) return cudaErrorInvalidValue;
    const bool tc = extract_uses_tc(dtype, d, p.hq, p.hkv, p.n_all, p.lq, p.pairs_per_cta);
    if (!p.q_rot != (tc && extract_turns_queries(p.pairs_per_cta))) return cudaErrorInvalidValue;
    if (tc)
        return d == 64 ? launch_tc<64>(p, s, s2, fork, join) : launch_tc<128>(p, s, s2, fork, join);
    if (dtype == kDtypeF32 && d == 64) return launch_typed<float, 64>(p, s);
    if (dtype == kDtypeF32 && d == 128) return launch_typed<float, 128>(p, s);
    if (dtype == kDtypeBf16 && d == 64) return launch_typed<__nv_bfloat16, 64>(p, s);
    if (dtype == kDtypeBf16 && d == 128) return launch_typed<__nv_bfloat16, 128>(p, s);
    return cudaErrorInvalidValue;
}

}  // namespace c2kv

// CUDA-core attention over [composed cache; suffix]: the path of fp32 contexts and of the head
// layouts that the tensor-core kernel does not take.  The loop is attention_core
// (attn_core.cuh); here is what a row and a key are: packed row r = t * G + g is suffix token t,
// query head h_kv * G + g, and token t sees keys 0 .. S + t.
#include <algorithm>

#include "attn_core.cuh"

namespace c2kv {
namespace {

template <typename T, int D>
struct SuffixJob {
    const AttnParams& a;
    int l, bl, hk, g_heads;
    int row0, rows;                   // this CTA's packed rows [row0, row0 + rows)
    int nrows, nkeys, slots;
    const T *k, *v;
    int64_t stride;
    float scale_log2;
    __device__ int64_t token_row(int t) const {
        return ((int64_t)l * a.batch_total + a.b0 + bl) * a.sq + t;
    }
    __device__ int64_t row_off(int r) const {
        const int t = r / g_heads, g = r - t * g_heads;
        return (token_row(t) * a.hq + hk * g_heads + g) * D;
    }
    __device__ const T* q_row(int r) const { return static_cast<const T*>(a.q_rot) + row_off(r); }
    __device__ T* out_row(int r) const { return static_cast<T*>(a.out) + row_off(r); }
    __device__ float* lse_at(int r) const {
        if (a.lse == nullptr) return nullptr;
        const int t = r / g_heads, g = r - t * g_heads;
        return a.lse + (((int64_t)l * a.batch_total + a.b0 + bl) * a.hq + hk * g_heads + g) * a.sq + t;
    }
    __device__ bool needed(int, int) const { return true; }
    __device__ bool whole(int, int k1) const { return k1 - 1 <= slots + row0 / g_heads; }
    __device__ int row(int r) const { return slots + r / g_heads; }      // its last key
    __device__ bool sees(int last, int key) const { return key <= last; }
};

template <typename T, int D, int RT>
__global__ void __launch_bounds__(kCoreThreads, core_ctas(D, RT)) attn_simt_kernel(const __grid_constant__ AttnParams a, int ns) {
    extern __shared__ __align__(16) uint8_t core_smem[];
    asm volatile("griddepcontrol.wait;" ::: "memory");   // the rotated query and the newest key rows
    const int rank = (int)(blockIdx.x % (unsigned)ns);
    SuffixJob<T, D> j{a};
    j.l = (int)blockIdx.z / a.batch;
    j.bl = (int)blockIdx.z - j.l * a.batch;
    j.hk = blockIdx.y;
    j.g_heads = a.hq / a.hkv;
    j.rows = Core<D, RT>::kRows;
    j.row0 = (int)(blockIdx.x / (unsigned)ns) * j.rows;
    j.nrows = a.sq * j.g_heads;
    j.slots = a.req[j.bl].n_slots;
    j.nkeys = j.slots + min(a.sq - 1, (j.row0 + j.rows - 1) / j.g_heads) + 1;
    j.stride = (int64_t)a.hkv * D;
    const int64_t base = (((int64_t)(a.layer0 + j.l) * a.rows + a.req[j.bl].row_base) * a.hkv + j.hk) * D;
    j.k = static_cast<const T*>(a.cache_k) + base;
    j.v = static_cast<const T*>(a.cache_v) + base;
    j.scale_log2 = a.scale_log2;
    attention_core<T, D, RT>(j, j.row0, ns, rank, core_smem);
}

template <typename T, int D, int RT>
CoreKernel<D, RT> ready() {
    static PerDevice<CoreKernel<D, RT>> kept;
    return kept.get([] { return CoreKernel<D, RT>(reinterpret_cast<const void*>(&attn_simt_kernel<T, D, RT>), device_sms()); });
}

template <typename T, int D, int RT>
cudaError_t launch_rt(const AttnParams& a, CorePlan plan, cudaStream_t s) {
    constexpr int kRows = Core<D, RT>::kRows;
    const int64_t gx = ((int64_t)a.sq * (a.hq / a.hkv) + kRows - 1) / kRows * plan.ns;
    if (gx > 0x7fffffffLL) return cudaErrorInvalidValue;
    void* args[2] = {const_cast<AttnParams*>(&a), &plan.ns};
    return core_launch(reinterpret_cast<const void*>(&attn_simt_kernel<T, D, RT>), dim3((unsigned)gx, a.hkv, a.lq * a.batch),
                       Core<D, RT>::kSmem, plan, a.dependent != 0, args, s);
}

template <typename T, int D>
cudaError_t launch_typed(const AttnParams& a, cudaStream_t s) {
    int64_t nkeys = 0;
    for (int i = 0; i < a.batch; ++i) nkeys = std::max<int64_t>(nkeys, (int64_t)a.req[i].n_slots + a.sq);
    const int64_t nrows = (int64_t)a.sq * (a.hq / a.hkv);
    const CoreKernel<D, 4> large = ready<T, D, 4>();
    const CoreKernel<D, 1> small = ready<T, D, 1>();
    const CoreKernel<D, 0> four = ready<T, D, 0>();
    if (large.err != cudaSuccess) return large.err;
    if (small.err != cudaSuccess || four.err != cudaSuccess) return small.err != cudaSuccess ? small.err : four.err;
    const CorePlan plan = core_plan(nrows, (int64_t)a.hkv * a.lq * a.batch, nkeys, D, false, [&](int form, int ns, bool alone) {
        return form == 4 ? large.slots[alone][ns] : form == 1 ? small.slots[alone][ns] : four.slots[alone][ns];
    });
    return plan.form == 4   ? launch_rt<T, D, 4>(a, plan, s)
           : plan.form == 1 ? launch_rt<T, D, 1>(a, plan, s)
                            : launch_rt<T, D, 0>(a, plan, s);
}

template <typename T, int D>
cudaError_t preload() {
    cudaFuncAttributes fa{};
    cudaError_t e = cudaFuncGetAttributes(&fa, attn_simt_kernel<T, D, 4>);
    if (e == cudaSuccess) e = cudaFuncGetAttributes(&fa, attn_simt_kernel<T, D, 1>);
    if (e == cudaSuccess) e = cudaFuncGetAttributes(&fa, attn_simt_kernel<T, D, 0>);
    if (e == cudaSuccess) e = ready<T, D, 4>().err;
    if (e == cudaSuccess) e = ready<T, D, 1>().err;
    if (e == cudaSuccess) e = ready<T, D, 0>().err;
    return e;
}

}  // namespace

cudaError_t preload_attn_simt_kernels(int dtype, int d) {
    if (dtype == kDtypeF32 && d == 64) return preload<float, 64>();
    if (dtype == kDtypeF32 && d == 128) return preload<float, 128>();
    if (dtype == kDtypeBf16 && d == 64) return preload<__nv_bfloat16, 64>();
    if (dtype == kDtypeBf16 && d == 128) return preload<__nv_bfloat16, 128>();
    return cudaErrorInvalidValue;
}

cudaError_t launch_attn_simt(const AttnParams& a, int dtype, int d, cudaStream_t s) {
    (void)cudaGetLastError();   // report this launch's error only, not a stale one
    if ((int64_t)a.lq * a.batch > 65535 || a.hkv > 65535) return cudaErrorInvalidValue;
    if (dtype == kDtypeF32 && d == 64) return launch_typed<float, 64>(a, s);
    if (dtype == kDtypeF32 && d == 128) return launch_typed<float, 128>(a, s);
    if (dtype == kDtypeBf16 && d == 64) return launch_typed<__nv_bfloat16, 64>(a, s);
    if (dtype == kDtypeBf16 && d == 128) return launch_typed<__nv_bfloat16, 128>(a, s);
    return cudaErrorInvalidValue;
}

}  // namespace c2kv

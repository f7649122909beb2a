// ts_router.cu -- MoE router (Sec. 4): logits r = W_r x, top-k experts (a
// lower expert index wins a tie), softmax over the k picked logits.
// One CTA per token; warp e computes logit e with 16-byte streaming loads,
// kRowVecs of them in flight: the kernel is nothing but latency, and one load
// at a time took 13 us at d = 4096. Each warp's first loads go out right behind
// those of the activations.
// In stack mode the CTA first normalises its residual row (the stack glue)
// and publishes the activations for the grouped expert kernels.
#include "ts_kernels.cuh"

namespace tsffn {

constexpr int kRowVecs = 16;  // 16-byte vectors of a row a lane loads at once (d = 4096 bf16: all)

template <typename T>
__global__ void __launch_bounds__(256) k_router(const RouterLaunch a) {
    constexpr int VEC = Vec<T>::N;
    extern __shared__ __align__(16) float xs[];  // [d]
    __shared__ float logit[kMaxExperts];
    __shared__ float red[8];
    const int t = blockIdx.x;
    const int d = a.d;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;

    uint4 v[kRowVecs];
    auto load = [&](int e, int col0) {  // the row's vectors from column col0 + lane * VEC on
        const T* row = static_cast<const T*>(a.wr) + (size_t)e * d;
#pragma unroll
        for (int u = 0; u < kRowVecs; ++u) {
            if (col0 + u * kWarp * VEC >= d) break;  // (short rows do not go through all of the places)
            const int col = col0 + (u * kWarp + lane) * VEC;
            v[u] = col < d ? ld_stream(row + col) : make_uint4(0u, 0u, 0u, 0u);
        }
    };
    // Loaded after the wait, as the kernel before may have written W_r; until then only pulled into L2. A layer of
    // 2 tokens over 8 experts, d = 1024, m = 2500, with loads before the wait 25.2 us, right after it 26.0 (26.5
    // without the prefetch), behind the activations' loads 25.0.
    if (warp < a.n_experts) {
        constexpr int kLine = 128 / (int)sizeof(T);
        for (int col = lane * kLine; col < d; col += kWarp * kLine)
            prefetch_l2(static_cast<const T*>(a.wr) + (size_t)warp * d + col);
    }
    pdl_wait();
    pdl_launch_dependents();
    stage_act_row<T>(a.h != nullptr ? a.h + (size_t)t * d : nullptr, static_cast<const T*>(a.x) + (size_t)t * d, d,
                     (int)threadIdx.x, (int)blockDim.x, red, [&](int i, float f) { xs[i] = f; },
                     [&]() {  // behind the activations' loads
                         if (warp < a.n_experts) load(warp, 0);
                     });
    if (a.h != nullptr) {
        __syncthreads();
        for (int i = threadIdx.x; i < d; i += blockDim.x) Vec<T>::store1(a.xbuf, (size_t)t * d + i, xs[i]);
    }
    __syncthreads();

    for (int e = warp; e < a.n_experts; e += nw) {
        float acc = 0.0f;
        for (int col0 = 0; col0 < d; col0 += kRowVecs * kWarp * VEC) {
            if (e != warp || col0 != 0) load(e, col0);
#pragma unroll
            for (int u = 0; u < kRowVecs; ++u) {
                if (col0 + u * kWarp * VEC >= d) break;
                const int col = col0 + (u * kWarp + lane) * VEC;
                if (col < d) {
                    float f[VEC];
                    Vec<T>::unpack(v[u], f);
#pragma unroll
                    for (int q = 0; q < VEC; ++q) acc = fmaf(f[q], xs[col + q], acc);
                }
            }
        }
        acc = warp_sum(acc);
        if (lane == 0) logit[e] = acc;
    }
    __syncthreads();

    if (threadIdx.x == 0) {
        TokenRoute r;
        unsigned taken = 0u;
        for (int k = 0; k < kMaxTopK; ++k) {
            r.sel[k] = -1;
            r.w[k] = 0.0f;
        }
        for (int k = 0; k < a.top_k; ++k) {
            int best = -1;
            for (int e = 0; e < a.n_experts; ++e) {
                if ((taken >> e) & 1u) continue;
                if (best < 0 || logit[e] > logit[best]) best = e;
            }
            r.sel[k] = best;
            taken |= 1u << best;
        }
        float z = 0.0f;
        for (int k = 0; k < a.top_k; ++k) z += expf(logit[r.sel[k]] - logit[r.sel[0]]);
        for (int k = 0; k < a.top_k; ++k) r.w[k] = expf(logit[r.sel[k]] - logit[r.sel[0]]) / z;
        a.route[t] = r;
    }
}

cudaError_t launch_router(const RouterLaunch& a, int wdtype, cudaStream_t stream, bool pdl) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(a.batch);
    cfg.blockDim = dim3(256);
    cfg.dynamicSmemBytes = (size_t)a.d * sizeof(float);
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = pdl ? 1 : 0;
    if (wdtype == 1) return cudaLaunchKernelEx(&cfg, k_router<__nv_bfloat16>, a);
    return cudaLaunchKernelEx(&cfg, k_router<float>, a);
}

cudaError_t prepare_router() {
    cudaError_t e = cudaFuncSetAttribute(k_router<__nv_bfloat16>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, kRouterMaxD * 4);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_router<float>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 kRouterMaxD * 4);
    return e;
}

}  // namespace tsffn

// vc_noalloc.cu -- one FP32 Bellman sweep of the implicit model that allocates nothing.
//
// Some callers cannot call cudaMalloc: code whose device memory is entirely reserved by
// another allocator (a framework's caching pool), code that must not risk the implicit
// device synchronisation an allocation can cause (latency-bound control loops), and code
// that runs while another library captures the stream.  For them this file keeps the
// sweep's scratch -- the post-decision value array U, two residual words and a control block
// whose error word the bounds-checking build reports through -- in file-scope __device__
// arrays of fixed size, loaded with the library on every GPU that loads it and held until
// the process exits.  The caller still passes V and V_out.
#include <math.h>

#include <algorithm>
#include <mutex>
#include <type_traits>

#include "vc_implicit.cuh"
#include "vc_internal.cuh"

namespace vc {

constexpr int kNoAllocMaxStates = 1 << 20;  // 1,048,576 states: 4 MiB of float scratch

static __device__ __align__(256) float g_noalloc_U[kNoAllocMaxStates + kUPad];
static __device__ __align__(256) unsigned int g_noalloc_res[64];
static __device__ __align__(256) Ctl g_noalloc_ctl;

// Device addresses of the static arrays and the SM count, looked up once per device by the
// first call there.  A later call makes no CUDA call but two launches and error queries, so it
// may run while the stream is being captured.  In host code the array
// names are host-side stand-ins, never device addresses: only these pointers are passed to
// kernels.
struct NoAllocScratch {
    bool ready = false;
    float* U = nullptr;
    unsigned int* res = nullptr;
    Ctl* ctl = nullptr;
    int num_sms = 0;
};

constexpr int kMaxDevices = 64;
static NoAllocScratch g_scratch[kMaxDevices];
static std::mutex g_scratch_mu;

static int noalloc_scratch(NoAllocScratch* out) {
    int dev = 0;
    VC_CUDA(cudaGetDevice(&dev));
    if (dev < 0 || dev >= kMaxDevices) return fail(VC_ERR_ARG, "device ordinal beyond the static scratch table");
    std::lock_guard<std::mutex> lock(g_scratch_mu);
    NoAllocScratch& s = g_scratch[dev];
    if (!s.ready) {
        void* p = nullptr;
        VC_CUDA(cudaGetSymbolAddress(&p, g_noalloc_U));
        s.U = (float*)p;
        VC_CUDA(cudaGetSymbolAddress(&p, g_noalloc_res));
        s.res = (unsigned int*)p;
        VC_CUDA(cudaGetSymbolAddress(&p, g_noalloc_ctl));
        s.ctl = (Ctl*)p;
        VC_CUDA(cudaDeviceGetAttribute(&s.num_sms, cudaDevAttrMultiProcessorCount, dev));
        s.ready = true;
    }
    *out = s;
    return VC_OK;
}

// Pass 1 of the sweep; it also clears pass 2's residual words, so a call owes nothing to the state
// that an earlier one left (calls that overlap, against the rule, spoil only themselves).
template <int MH, int VW>
__global__ void __launch_bounds__(kThreads) k_noalloc_post(Model md, Coef<float> c, const float* V, float* U,
                                                           unsigned int* cell, Ctl* ctl) {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    if (blockIdx.x == 0 && threadIdx.x < 2) cell[threadIdx.x] = 0u;
    const int items = md.S / VW;
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < items; t += gridDim.x * blockDim.x)
        post_item<MH, VW, false>(md, c, V, VW * t, U, nullptr, ctl);
}

// Pass 2 with max |V_out - V| over all states on the way: one atomicMax a block into cell[0]
// (non-negative float bits, order independent), and the last block to arrive (ticket cell[1])
// hands the result out.  A NaN difference counts as +infinity: fmaxf would drop it, and a sweep
// that produced a NaN must not report a finite residual.  Launched as pass 1's programmatic
// dependent; it touches the words only once pass 1 has ended.
template <int MH, int VW, bool ARG>
__global__ void __launch_bounds__(kThreads) k_noalloc_max(Model md, const float* U, const float* V, float* V_out,
                                                          int32_t* pi, unsigned int* cell, float* residual, Ctl* ctl) {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const int items = md.S / VW;
    float r = 0.0f;
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < items; t += gridDim.x * blockDim.x) {
        const int s = VW * t;
        float vin[VW], best[VW], second[VW];
        int arg[VW];
        ldv<VW>(V + s, vin);
        max_item<MH, VW, false, ARG>(md, U, nullptr, s, best, second, arg, ctl);
        stv<VW>(V_out + s, best);
#pragma unroll
        for (int j = 0; j < VW; j++) {
            if constexpr (ARG) pi[s + j] = arg[j];
            const float d = fabsf(best[j] - vin[j]);
            r = d != d ? INFINITY : fmaxf(r, d);
        }
    }
    if (!residual) return;
    __shared__ unsigned int sh_r;
    if (threadIdx.x == 0) sh_r = 0u;
    __syncthreads();
    const unsigned int rb = __reduce_max_sync(0xffffffffu, __float_as_uint(r));
    if ((threadIdx.x & 31) == 0) atomicMax(&sh_r, rb);
    __syncthreads();
    if (threadIdx.x != 0) return;
    atomicMax(&cell[0], sh_r);
    __threadfence();
    if (atomicAdd(&cell[1], 1u) != gridDim.x - 1) return;
    __threadfence();
    *residual = __uint_as_float(__ldcg(&cell[0]));
}

// Both passes.  Bound: the launches (a sweep of 17,500 states keeps the device busy for 4 us);
// two, the second overlapping the first's start, in place of four and a memset: 23 -> 16 us
// a call.
template <int MH, int VW>
static int noalloc_run(const Mdp& m, const NoAllocScratch& sc, const float* V, float* V_out, int32_t* pi,
                       float* residual, Ctl* ctl, cudaStream_t st) {
    const int items = m.S / VW;
    // small sweeps in blocks of two warps, so that every SM takes part
    const int threads = items <= 64 * 4 * sc.num_sms ? 64 : kThreads;
    const int grid = std::min((items + threads - 1) / threads, 8 * sc.num_sms);
    float* U = sc.U + kUShift;
    count_launches(2);
    k_noalloc_post<MH, VW><<<grid, threads, 0, st>>>(m.md, m.c32, V, U, sc.res, ctl);
    VC_CUDA(cudaGetLastError());
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3((unsigned)threads);
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    const float* Uc = U;
    if (pi)
        VC_CUDA(cudaLaunchKernelEx(&cfg, k_noalloc_max<MH, VW, true>, m.md, Uc, V, V_out, pi, sc.res, residual, ctl));
    else
        VC_CUDA(cudaLaunchKernelEx(&cfg, k_noalloc_max<MH, VW, false>, m.md, Uc, V, V_out, pi, sc.res, residual, ctl));
    return VC_OK;
}

static int noalloc_sweep(const Mdp& m, const NoAllocScratch& sc, const float* V, float* V_out, int32_t* pi,
                         float* residual, Ctl* ctl, cudaStream_t st) {
    const bool wide = wide_rows(m.md) && (((uintptr_t)V | (uintptr_t)V_out) & 15) == 0;
    auto go = [&](auto mh) {
        constexpr int MH = decltype(mh)::value;
        return wide && MH <= 8 ? noalloc_run<MH, MH <= 8 ? 4 : 2>(m, sc, V, V_out, pi, residual, ctl, st)
                               : noalloc_run<MH, 2>(m, sc, V, V_out, pi, residual, ctl, st);
    };
    switch (m.md.H) {
        case 1: return go(std::integral_constant<int, 1>());
        case 2: return go(std::integral_constant<int, 2>());
        case 3: return go(std::integral_constant<int, 3>());
        case 4: return go(std::integral_constant<int, 4>());
        case 5: return go(std::integral_constant<int, 5>());
        case 6: return go(std::integral_constant<int, 6>());
        case 7: return go(std::integral_constant<int, 7>());
        case 8: return go(std::integral_constant<int, 8>());
        default: return go(std::integral_constant<int, 16>());
    }
}

}  // namespace vc

using namespace vc;

extern "C" int vc_bellman32_noalloc(const vc_params* p, const float* V, float* V_out, int32_t* pi, float* residual,
                                    void* stream) {
    set_error("");
    if (!V || !V_out) return fail(VC_ERR_ARG, "V / V_out is NULL");
    if (V == V_out) return fail(VC_ERR_ARG, "V and V_out must be different buffers");
    Mdp m;  // host-side descriptor only; owns no device memory here
    m.fmt = VC_IMPLICIT;
    int rc = build_model(p, &m);
    if (rc) return rc;
    if (m.S > kNoAllocMaxStates)
        return fail(VC_ERR_ARG, "S = " + std::to_string(m.S) + " exceeds the static scratch of " +
                                    std::to_string(kNoAllocMaxStates) + " states");
    NoAllocScratch sc;
    if ((rc = noalloc_scratch(&sc))) return rc;
    m.num_sms = sc.num_sms;
    cudaStream_t st = (cudaStream_t)stream;
    Ctl* ctl = nullptr;
#ifdef VC_DEBUG_BOUNDS
    // bounds-checking build: the sweep raises its flags in the static control block, which
    // is cleared here and read back after the sweep (this build synchronises the stream)
    ctl = sc.ctl;
    VC_CUDA(cudaMemsetAsync(&sc.ctl->error, 0, sizeof(int), st));
#endif
    if ((rc = noalloc_sweep(m, sc, V, V_out, pi, residual, ctl, st))) return rc;
#ifdef VC_DEBUG_BOUNDS
    int err = 0;
    VC_CUDA(cudaMemcpyAsync(&err, &sc.ctl->error, sizeof(int), cudaMemcpyDeviceToHost, st));
    VC_CUDA(cudaStreamSynchronize(st));
    if (err & kErrBounds) return fail(VC_ERR_CUDA, "a device bounds check failed (bounds-checking build)");
#endif
    return VC_OK;
}

#ifdef VC_DEBUG_BOUNDS
// Test hook of the bounds-checking build: overwrites the residual words of the current device.
extern "C" int vc_debug_noalloc_words(uint32_t residual, uint32_t ticket) {
    NoAllocScratch sc;
    const int rc = noalloc_scratch(&sc);
    if (rc) return rc;
    const uint32_t w[2] = {residual, ticket};
    VC_CUDA(cudaMemcpy(sc.res, w, sizeof(w), cudaMemcpyHostToDevice));
    return VC_OK;
}
#endif

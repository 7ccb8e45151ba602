// vc_batch_loop.cu -- the batched FP32 loop (Algorithm 3, steps 1-3, for every instance) in one
// resident kernel.
//
// All active instances advance one sweep in step: pass 1, grid barrier, pass 2, grid barrier.
// The work of a pass (items of four or two states, weighted by what an item costs) is cut into
// equal contiguous shares, one per warp of the resident grid, so uneven instances leave no
// CTA idle and a warp's loads fall into one or two instances; the cut is made again only when
// an instance ends.  A warp takes each instance's coefficients into registers once per pass
// and runs the items of vc_implicit.cuh for the instance's exact host count.  After the
// second barrier every CTA takes step 3's decision for every instance itself.
// Once only small instances are left, with many sweeps to go, the loop leaves them to the
// whole-instance kernel (kHandOver in vc_batch.cu).
//
// Bound: L2 (DRAM while more than ~10 M states are active) latency of the items' loads at 16
// warps an SM, and the slower SMs' tail at the two barriers.  Whole solves against the graph of
// paired tile kernels (coefficients read from shared memory at each use, 8-byte loads): 512
// instances of 17.4 M states 134 -> 105 ms, 48 with the self-transition solve 13.1 -> 9.2 ms (with
// the hand-over below).
#include <algorithm>

#include "vc_batch.cuh"
#include "vc_grid.cuh"
#include "vc_implicit.cuh"
#include "vc_internal.cuh"

namespace vc {

constexpr int kBatchLoopThreads = 512;  // 640 and 768: spills, 48 instances 10.0 -> 11.4 and 14 ms
// Sweeps for which the hand-over (four launches, two host calls: 0.1 ms) pays at 2 to 4 us a sweep.
constexpr int kHandOverSweeps = 64;

// Relative cost of an item (a decode and, per host, its loads and arithmetic).
__host__ __device__ inline int item_cost(int H, bool wide) { return 40 + (wide ? 40 : 26) * H; }
__device__ __forceinline__ bool wide_inst(const Model& md) { return (md.Q & 1) != 0; }

// FP32 part of an instance's descriptor, kept in shared memory for the instances of a CTA's
// share (a barrier's acquire drops the L1 lines of the global one).
struct LoopInst {
    Model md;
    Coef<float> c32;
    long long off;
};
constexpr int kBatchLoopCached = 32;

// The coefficients an MH-host instance uses.
template <int MH>
struct LocalModel {
    Model md;
    Coef<float> c;
    template <typename D>
    __device__ __forceinline__ explicit LocalModel(const D& d) {
        md.H = MH;
        md.C = d.md.C;
        md.Q = d.md.Q;
        md.S = d.md.S;
        md.div_q = d.md.div_q;
        md.div_c = d.md.div_c;
        c.gamma = d.c32.gamma;
        c.pa = d.c32.pa;
        c.lossa = d.c32.lossa;
        c.pf0 = d.c32.pf0;
        c.pf1 = d.c32.pf1;
        c.w_occ = d.c32.w_occ;
        c.w_q = d.c32.w_q;
#pragma unroll
        for (int k = 0; k < MH; k++) {
            md.stride[k] = d.md.stride[k];
            c.pc[k] = d.c32.pc[k];
            c.pd[k] = d.c32.pd[k];
            c.lossd[k] = d.c32.lossd[k];
        }
    }
};

template <int MH, int VW, bool SL, typename D>
__device__ __forceinline__ void post_share(const D& d, const float* V, float* U, float* W, int i0, int i1, Ctl* ctl) {
    const LocalModel<MH> m(d);
    const float* Vi = V + d.off;
    float* Ui = U + d.off;
    float* Wi = SL ? W + d.off : nullptr;
    for (int t = i0 + (int)(threadIdx.x & 31); t < i1; t += 32) post_item<MH, VW, SL>(m.md, m.c, Vi, VW * t, Ui, Wi, ctl);
}

template <int MH, int VW, bool SL, typename D>
__device__ __forceinline__ void max_share(const D& d, const float* V, const float* U, const float* W, float* Vo,
                                          int i0, int i1, float& res, float& vabs, Ctl* ctl) {
    const LocalModel<MH> m(d);
    const float* Vi = V + d.off;
    const float* Ui = U + d.off;
    const float* Wi = SL ? W + d.off : nullptr;
    float* Oi = Vo + d.off;
    for (int t = i0 + (int)(threadIdx.x & 31); t < i1; t += 32) {
        float vin[VW], best[VW];
        ldv<VW>(Vi + VW * t, vin);
        max_item<MH, VW, SL, false>(m.md, Ui, Wi, VW * t, best, nullptr, nullptr, ctl);
        stv<VW>(Oi + VW * t, best);
#pragma unroll
        for (int j = 0; j < VW; j++) {
            res = fmaxf(res, fabsf(best[j] - vin[j]));
            vabs = fmaxf(vabs, fabsf(best[j]));
        }
    }
}

// Calls f<MH, VW> for an instance.
#define VC_BY_INST(d, F, ...)                                                   \
    switch (2 * (d).md.H + (wide_inst((d).md) ? 1 : 0)) {                       \
        case 2: F<1, 2, SL>(__VA_ARGS__); break;                                \
        case 3: F<1, 4, SL>(__VA_ARGS__); break;                                \
        case 4: F<2, 2, SL>(__VA_ARGS__); break;                                \
        case 5: F<2, 4, SL>(__VA_ARGS__); break;                                \
        case 6: F<3, 2, SL>(__VA_ARGS__); break;                                \
        case 7: F<3, 4, SL>(__VA_ARGS__); break;                                \
        case 8: F<4, 2, SL>(__VA_ARGS__); break;                                \
        case 9: F<4, 4, SL>(__VA_ARGS__); break;                                \
        case 10: F<5, 2, SL>(__VA_ARGS__); break;                               \
        default: F<5, 4, SL>(__VA_ARGS__); break;                               \
    }

template <bool SL>
__global__ void __launch_bounds__(kBatchLoopThreads, 1) k_batch_loop(BatchLoopArgs a) {
    extern __shared__ long long batch_sm[];
    // active instances: work before each (and the total), number, best residual, sweeps since
    long long* start = batch_sm;
    int* id = reinterpret_cast<int*>(start + a.n + 1);
    float* best = reinterpret_cast<float*>(id + a.n);
    int* since = reinterpret_cast<int*>(best + a.n);
    __shared__ int sh_m, sh_ended, sh_fail, sh_first, sh_small;
    __shared__ long long sh_end, sh_start;
    __shared__ LoopInst sh_inst[kBatchLoopCached];  // active instances sh_first ..
    const int lane = (int)threadIdx.x & 31, warp = (int)threadIdx.x >> 5;
    const bool lead = threadIdx.x == 0;
    const long long warps = (long long)gridDim.x * (blockDim.x >> 5), me = (long long)blockIdx.x * (blockDim.x >> 5) + warp;
    const double tol = *a.c.tol;
    const long long max_sweeps = *a.c.max_sweeps;
    for (int i = threadIdx.x; i < a.n; i += blockDim.x) {
        id[i] = a.c.done[i] ? -1 : i;
        best[i] = a.c.best_res[i];
        since[i] = a.c.since_best[i];
    }
    if (lead) {
        sh_m = a.n;
        sh_ended = 1;
        sh_fail = 0;
        sh_end = a.first + kLaunchSweeps;
    }
    __syncthreads();
    GridBarrier bar{a.arrivals, gridDim.x, 0u, &sh_fail, a.polls};
    long long k = a.first;
    const bool first_cta = lead && blockIdx.x == 0;
    LaunchEnd end{a.end, &sh_start};
    if (first_cta) end.open(k);
    long long w0 = 0, w1 = 0;
    int first = 0;
    while (true) {
        const bool recut = sh_ended != 0;
        __syncthreads();
        if (recut) {
            // the instances still active, in order, and the work before each (warp 0)
            if (warp == 0) {
                int m = 0, largest = 0;
                long long total = 0;
                for (int i0 = 0; i0 < sh_m; i0 += 32) {
                    const int i = i0 + lane;
                    const int inst = i < sh_m ? id[i] : -1;
                    const float b = inst >= 0 ? best[i] : 0.0f;
                    const int sb = inst >= 0 ? since[i] : 0;
                    long long work = 0;
                    if (inst >= 0) {
                        largest = max(largest, a.descs[inst].S);
                        const bool wide = wide_inst(a.descs[inst].md);
                        work = (long long)(a.descs[inst].S / (wide ? 4 : 2)) * item_cost(a.descs[inst].md.H, wide);
                    }
                    const unsigned int live = __ballot_sync(0xffffffffu, inst >= 0);
                    long long incl = work;
#pragma unroll
                    for (int o = 1; o < 32; o <<= 1) {
                        const long long y = __shfl_up_sync(0xffffffffu, incl, o);
                        if (lane >= o) incl += y;
                    }
                    __syncwarp();
                    if (inst >= 0) {
                        const int p = m + __popc(live & ((1u << lane) - 1u));
                        id[p] = inst;
                        best[p] = b;
                        since[p] = sb;
                        start[p] = total + incl - work;
                    }
                    m += __popc(live);
                    total += __shfl_sync(0xffffffffu, incl, 31);
                    __syncwarp();
                }
                largest = __reduce_max_sync(0xffffffffu, largest);
                bool leave = m > 0 && largest <= a.hand_over;
                if (leave) {
                    // sweeps still needed, from the last sweep's residuals (-1: none was made) and each
                    // instance's contraction; every CTA reads the same words
                    float left = 0.0f;
                    for (int p = lane; p < m; p += 32) {
                        const int slot = 2 * id[p] + (int)((k - 1) & 1);
                        const float r = __uint_as_float(__ldcg(a.c.res32 + slot));
                        const float vm = __uint_as_float(__ldcg(a.c.vmax32 + slot));
                        const float t = fmaxf((float)(tol * (a.c.tol_scale ? (double)a.c.tol_scale[id[p]] : 1.0)), vm * 0x1p-21f);
                        left = fmaxf(left, k == 0 ? INFINITY : logf(r / t) / -logf(a.descs[id[p]].c32.gamma));
                    }
                    leave = __any_sync(0xffffffffu, left > (float)kHandOverSweeps);
                }
                if (lane == 0) {
                    start[m] = total;
                    sh_m = m;
                    sh_ended = 0;
                    sh_small = leave;
                }
            }
            __syncthreads();
            const int m = sh_m;
            w0 = start[m] * me / warps;
            w1 = start[m] * (me + 1) / warps;
            int lo = 0, hi = m;  // the last instance that starts at or before w0
            while (hi - lo > 1) {
                const int mid = (lo + hi) >> 1;
                if (start[mid] <= w0) lo = mid;
                else hi = mid;
            }
            first = lo;
            if (lead) sh_first = lo;
            __syncthreads();
            for (int p = sh_first + warp; p < min(m, sh_first + kBatchLoopCached); p += (int)(blockDim.x >> 5)) {
                const InstDesc& d = a.descs[id[p]];
                LoopInst& c = sh_inst[p - sh_first];
                for (int j = lane; j < (int)(sizeof(Model) / 4); j += 32)
                    reinterpret_cast<int*>(&c.md)[j] = reinterpret_cast<const int*>(&d.md)[j];
                for (int j = lane; j < (int)(sizeof(Coef<float>) / 4); j += 32)
                    reinterpret_cast<int*>(&c.c32)[j] = reinterpret_cast<const int*>(&d.c32)[j];
                if (lane == 0) c.off = d.off;
            }
            __syncthreads();
        }
        const int m = sh_m;
        if (m == 0 || k >= sh_end || sh_small) break;
        if (first_cta) end.check(k);
        const int in = (int)(k & 1);
        const float* Vi = in ? a.V1 : a.V0;
        float* Vo = in ? a.V0 : a.V1;
        // items [i0, i1) of active instance p that belong to this warp
        auto share = [&](int p, const Model& md, int& i0, int& i1) {
            const bool wide = wide_inst(md);
            const int cost = item_cost(md.H, wide), items = md.S / (wide ? 4 : 2);
            i0 = w0 <= start[p] ? 0 : (int)((w0 - start[p]) / cost);
            i1 = w1 >= start[p + 1] ? items : (int)((w1 - start[p]) / cost);
        };
        for (int p = first; p < m && start[p] < w1; p++) {
            int i0, i1;
            if (p - sh_first < kBatchLoopCached) {
                const LoopInst& d = sh_inst[p - sh_first];
                share(p, d.md, i0, i1);
                VC_BY_INST(d, post_share, d, Vi, a.U, a.U2, i0, i1, a.ctl)
            } else {
                const InstDesc& d = a.descs[id[p]];
                share(p, d.md, i0, i1);
                VC_BY_INST(d, post_share, d, Vi, a.U, a.U2, i0, i1, a.ctl)
            }
        }
        if (blockIdx.x == 0)  // this sweep's residual slots, last read two sweeps ago
            for (int p = threadIdx.x; p < m; p += blockDim.x)
                a.c.res32[2 * id[p] + in] = a.c.vmax32[2 * id[p] + in] = 0u;
        if (!bar.sync()) break;
        for (int p = first; p < m && start[p] < w1; p++) {
            const int inst = id[p];
            int i0, i1;
            float res = 0.0f, vabs = 0.0f;
            if (p - sh_first < kBatchLoopCached) {
                const LoopInst& d = sh_inst[p - sh_first];
                share(p, d.md, i0, i1);
                VC_BY_INST(d, max_share, d, Vi, a.U, a.U2, Vo, i0, i1, res, vabs, a.ctl)
            } else {
                const InstDesc& d = a.descs[inst];
                share(p, d.md, i0, i1);
                VC_BY_INST(d, max_share, d, Vi, a.U, a.U2, Vo, i0, i1, res, vabs, a.ctl)
            }
            // non-negative floats order like their bits
            const unsigned int rb = __reduce_max_sync(0xffffffffu, fbits(res));
            const unsigned int vb = __reduce_max_sync(0xffffffffu, fbits(vabs));
            if (lane == 0 && i0 < i1) {
                atomicMax(&a.c.res32[2 * inst + in], rb);
                atomicMax(&a.c.vmax32[2 * inst + in], vb);
            }
        }
        if (!bar.sync()) break;
        k++;
        if (threadIdx.x == blockDim.x - 1) sh_end = end.read();  // beside the verdicts' reads
        for (int p = threadIdx.x; p < m; p += blockDim.x) {
            const int inst = id[p];
            const float r = __uint_as_float(__ldcg(a.c.res32 + 2 * inst + in));
            const float vm = __uint_as_float(__ldcg(a.c.vmax32 + 2 * inst + in));
            const double t = tol * (a.c.tol_scale ? (double)a.c.tol_scale[inst] : 1.0);
            LoopVerdict v{t, __double2float_ru(t), best[p], since[p], max_sweeps};
            const int done = v(r, vm, k);
            best[p] = v.best;
            since[p] = v.since;
            if (done) {
                id[p] = -1;
                sh_ended = 1;
                if (blockIdx.x == 0) {
                    a.c.done[inst] = done;
                    a.c.sweeps[inst] = (int)k;
                    a.c.final_buf[inst] = (int)(k & 1);
                }
            }
        }
        __syncthreads();
    }
    __syncthreads();
    if (lead && sh_fail) atomicOr(a.fault, kLoopTimeout);
    if (blockIdx.x != 0) return;
    if (lead) {
        *a.c.active = sh_m;
        *a.end = k;
        if (sh_small) atomicOr(a.fault, kLoopHandOver);
    }
    for (int p = threadIdx.x; p < sh_m; p += blockDim.x) {
        a.c.best_res[id[p]] = best[p];
        a.c.since_best[id[p]] = since[p];
    }
}

int launch_batch_loop(const BatchLoopArgs& a, int max_hosts, int num_sms, bool self_loop, cudaStream_t st,
                      ResidentTurn& turn, bool* launched) {
    *launched = false;
    if (max_hosts > kBatchLoopMaxH || a.n > kBatchLoopMaxN) return VC_OK;
    const void* fn = self_loop ? (const void*)k_batch_loop<true> : (const void*)k_batch_loop<false>;
    const size_t smem = 8 * ((size_t)a.n + 1) + 12 * (size_t)a.n;
    VC_CUDA(cached_set_max_dyn_smem(fn, 8 * (kBatchLoopMaxN + 1) + 12 * kBatchLoopMaxN));
    return launch_resident(fn, num_sms, kBatchLoopThreads, smem, st, turn, num_sms, launched, a);
}

}  // namespace vc

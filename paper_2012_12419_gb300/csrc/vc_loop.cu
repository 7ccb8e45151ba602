// vc_loop.cu -- the FP32 value-iteration loop of an implicit handle (Algorithm 3, steps 1-3)
// in one resident kernel.
//
// A sweep of these models is short (20 us at 2.5 M states, 1 us at a few thousand), so
// launched kernel by kernel it pays as much for launches, for the tail of two grids and for
// 1,216 blocks' atomics on the control block as for the sweep.  Here at most one CTA per SM
// stays resident for the whole loop: each owns one contiguous range of items (inner hosts'
// targets then hit its L1), a grid barrier separates pass 1 from pass 2 and one sweep from
// the next, the residual travels with the second barrier, and every CTA takes step 3's
// decision itself from the same two words.  Instances whose arrays fit one CTA's shared
// memory run there without any grid barrier.
//
// Bound: issue and L2 latency of the two passes (16 loads of 16 bytes and some 340 instructions a
// pass for 4 states of 7 hosts; 47 % of the issue slots), then two barriers of ~1.5 us.  Measured per sweep, launched kernels
// against this loop: 45 -> 19 us at 2.5 M states (H = 7), 18.3 -> 8.0 us at 343,750 states
// with the self-transition solve (VW = 2), whole solves of 640 states 2.89 -> 0.76 ms.
#include <algorithm>
#include <type_traits>

#include "vc_grid.cuh"
#include "vc_implicit.cuh"
#include "vc_internal.cuh"

namespace vc {

// 640 threads leave 96 registers each, enough for items of four states of up to 7 hosts without
// spills (768 and 1,024 spill): solve of 2.5 M states 7.9 ms with 512, 7.6 with 576, 6.75 with
// 640, 8.9 with 768; gradient step of 343,750 states 8.8 -> 8.4 ms.
constexpr int kLoopThreads = 640;
// States up to which one CTA sweeps the instance alone: 8,192 states are ~5 us of issue on one
// SM, what a sweep of the multi-CTA loop takes at any size (two barriers and two cold L2
// round trips); four arrays of 8,192 floats also fit beside the L1's needs.
constexpr int kLoopOneCta = 8192;
// Sweeps of its launch: 6 to 20 ms at 1.4 to 5 us (by the clock, as the grids do it, the words in
// shared memory cost 5 % of a sweep).
constexpr int kLoopOneCtaSweeps = 4096;
constexpr int kLoopItems = 256;    // least items of a CTA of the multi-CTA loop

// SMEM: one CTA, V's two buffers, U and W in shared memory (4 S + kUPad floats); else W, U
// are the handle's buffers and V the caller's pair.
template <int MH, int VW, bool SL, bool SMEM>
__global__ void __launch_bounds__(kLoopThreads, 1) k_vi_loop(Model md, Coef<float> c, float* buf0, float* buf1,
                                                             float* U, float* W, Ctl* ctl) {
    extern __shared__ __align__(16) float loop_sm[];
    __shared__ unsigned int sh_max[2][2];  // residual and max|V'| of the sweep, by parity
    __shared__ float sh_rv[2];
    __shared__ int sh_fail;
    __shared__ long long sh_end, sh_start;
    const int items = md.S / VW;
    const int per = (items + (int)gridDim.x - 1) / (int)gridDim.x;
    const int t0 = (int)blockIdx.x * per, t1 = min(items, t0 + per);
    const bool lead = threadIdx.x == 0;
    long long k = ctl->sweeps;
    const bool first = lead && blockIdx.x == 0;
    const long long k_end = k + kLoopOneCtaSweeps;
    LaunchEnd end{&ctl->launch_end, &sh_start};
    LoopVerdict verdict{ctl->tol, __double2float_ru(ctl->tol), ctl->best_res, ctl->since_best, ctl->max_sweeps};
    float* V[2] = {buf0, buf1};
    if constexpr (SMEM) {
        V[0] = loop_sm;
        V[1] = loop_sm + md.S;
        W = loop_sm + 2 * md.S;
        U = loop_sm + (SL ? 3 : 2) * md.S + kUShift;
        const float* src = (k & 1) ? buf1 : buf0;
        for (int i = threadIdx.x; i < md.S; i += blockDim.x) V[k & 1][i] = src[i];
    }
    if (lead) {
        sh_max[0][0] = sh_max[0][1] = sh_max[1][0] = sh_max[1][1] = 0u;
        sh_fail = 0;
    }
    if (!SMEM && first) end.open(k);
    __syncthreads();
    GridBarrier bar{&ctl->arrivals, gridDim.x, 0u, &sh_fail, barrier_polls(ctl->spin_limit)};
    int done = 0;
    float r = 0.0f, vm = 0.0f;
    while (true) {
        const int in = (int)(k & 1);
        const float* Vi = V[in];
        float* Vo = V[in ^ 1];
        if (!SMEM && first) end.check(k);
        for (int t = t0 + (int)threadIdx.x; t < t1; t += (int)blockDim.x)
            post_item<MH, VW, SL>(md, c, Vi, VW * t, U, W, ctl);
        if constexpr (SMEM) {
            __syncthreads();
        } else {
            // the next sweep's slot: last read 63 sweeps ago, first written after two barriers
            if (first) {
                ctl->res32[(k + 1) % kRing] = 0u;
                ctl->vmax32[(k + 1) % kRing] = 0u;
            }
            if (!bar.sync()) break;
        }
        float res = 0.0f, vabs = 0.0f;
        for (int t = t0 + (int)threadIdx.x; t < t1; t += (int)blockDim.x) {
            float vin[VW], best[VW];
            ldv<VW>(Vi + VW * t, vin);
            max_item<MH, VW, SL, false>(md, U, W, VW * t, best, nullptr, nullptr, ctl);
            stv<VW>(Vo + VW * t, best);
#pragma unroll
            for (int j = 0; j < VW; j++) {
                res = fmaxf(res, fabsf(best[j] - vin[j]));
                vabs = fmaxf(vabs, fabsf(best[j]));
            }
        }
        // non-negative floats order like their bits
        const unsigned int rb = __reduce_max_sync(0xffffffffu, fbits(res));
        const unsigned int vb = __reduce_max_sync(0xffffffffu, fbits(vabs));
        if ((threadIdx.x & 31) == 0) {
            atomicMax(&sh_max[in][0], rb);
            atomicMax(&sh_max[in][1], vb);
        }
        __syncthreads();
        if constexpr (SMEM) {
            r = __uint_as_float(sh_max[in][0]);
            vm = __uint_as_float(sh_max[in][1]);
            if (lead) sh_max[in ^ 1][0] = sh_max[in ^ 1][1] = 0u;  // next written after the next __syncthreads
        } else {
            const int slot = (int)(k % kRing);
            if (lead) {
                atomicMax(&ctl->res32[slot], sh_max[in][0]);
                atomicMax(&ctl->vmax32[slot], sh_max[in][1]);
                sh_max[in][0] = sh_max[in][1] = 0u;
            }
            if (!bar.arrive_and_wait()) break;
            if (lead) {
                sh_rv[0] = __uint_as_float(*((volatile unsigned int*)&ctl->res32[slot]));
                sh_rv[1] = __uint_as_float(*((volatile unsigned int*)&ctl->vmax32[slot]));
            }
            if (threadIdx.x == blockDim.x - 1) sh_end = end.read();  // beside the lead's two reads
            __syncthreads();
            r = sh_rv[0];
            vm = sh_rv[1];
        }
        k++;
        done = verdict(r, vm, k);
        if (done || k >= (SMEM ? k_end : sh_end)) break;
    }
    if constexpr (SMEM) {
        __syncthreads();
        float* dst = (k & 1) ? buf1 : buf0;
        for (int i = threadIdx.x; i < md.S; i += blockDim.x) dst[i] = V[k & 1][i];
        if (lead) {
            ctl->res32[(k - 1) % kRing] = fbits(r);
            ctl->vmax32[(k - 1) % kRing] = fbits(vm);
        }
    }
    if (lead && sh_fail) atomicOr(&ctl->error, kErrTimeout);
    if (first) {
        ctl->sweeps = k;
        ctl->final_buf = (int)(k & 1);
        ctl->best_res = verdict.best;
        ctl->since_best = verdict.since;
        ctl->done = sh_fail ? 4 : done;
    }
}

// Threads of a CTA for `per` items: the multiple of 32 (at least 3/4 of the limit) that
// wastes the least of its last step.
static int loop_threads(int per) {
    if (per <= kLoopThreads) return std::max(32, (per + 31) / 32 * 32);
    int best = kLoopThreads;
    long long cost = -1;
    for (int t = kLoopThreads; t >= 3 * kLoopThreads / 4; t -= 32) {
        const long long w = (long long)((per + t - 1) / t) * t;
        if (cost < 0 || w < cost) {
            cost = w;
            best = t;
        }
    }
    return best;
}

template <int MH, int VW, bool SL>
static int vi_loop_run(Mdp* m, float* buf0, float* buf1, cudaStream_t st, ResidentTurn& turn, bool* launched) {
    const int items = m->S / VW;
    float* U = m->U32 + kUShift;
    const size_t smem = 4 * ((size_t)(SL ? 4 : 3) * m->S + kUPad);
    *launched = true;
    if (m->S <= kLoopOneCta) {
        auto kern = k_vi_loop<MH, VW, SL, true>;
        VC_CUDA(cached_set_max_dyn_smem((const void*)kern, 4 * (4 * kLoopOneCta + kUPad)));
        count_launches(1);
        kern<<<1, loop_threads(items), smem, st>>>(m->md, m->c32, buf0, buf1, U, m->U32s, m->ctl);
        VC_CUDA(cudaGetLastError());
        return VC_OK;
    }
    auto kern = k_vi_loop<MH, VW, SL, false>;
    const int sms = m->num_sms > 0 ? m->num_sms : 148;
    const int grid = std::min(sms, (items + kLoopItems - 1) / kLoopItems);
    const int per = (items + grid - 1) / grid;
    return launch_resident((const void*)kern, (items + per - 1) / per, loop_threads(per), 0, st, turn, sms, launched, m->md,
                           m->c32, buf0, buf1, U, m->U32s, m->ctl);
}

int launch_vi_loop(Mdp* m, float* buf0, float* buf1, int self_loop, cudaStream_t st, ResidentTurn& turn,
                   bool* launched) {
    const bool wide = wide_rows(m->md) && (((uintptr_t)buf0 | (uintptr_t)buf1) & 15) == 0;
    auto go = [&](auto mh) {
        constexpr int MH = decltype(mh)::value;
        constexpr int VW = MH <= 8 ? 4 : 2;
        if (self_loop)
            return wide && VW == 4 ? vi_loop_run<MH, VW, true>(m, buf0, buf1, st, turn, launched)
                                   : vi_loop_run<MH, 2, true>(m, buf0, buf1, st, turn, launched);
        return wide && VW == 4 ? vi_loop_run<MH, VW, false>(m, buf0, buf1, st, turn, launched)
                               : vi_loop_run<MH, 2, false>(m, buf0, buf1, st, turn, launched);
    };
    switch (m->md.H) {
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

// vc_sweep.cu -- implicit-form Bellman kernels (Algorithm 3, step 2, with the Eq. 18
// backup) and the dispatch between the implicit and the explicit CSR forms.
//
// Implicit form: successors generated in registers from the mixed-radix state code.  A
// sweep is two passes over the state space.  Pass 1 evaluates, for every state x read as
// a post-decision state, U(x) = R(x) + gamma * E[V(next) | x] over the at most 2H+3
// uniformised events (reward and probabilities depend on x only).  Pass 2 takes
// V'(s) = max over feasible a of U(x_a(s)), x_a the state after placing on host a (or s
// itself for defer).  This is the Eq. 18 backup with (2H+3) + A gathers per state
// instead of A * (2H+3).
//
// Every V-producing kernel fuses the residual max|V' - V| (warp -> block -> one atomicMax
// per block, order independent) and, in loop mode, the termination test of the last
// block (finish_block), so the host never reads the residual per sweep.  All grids are
// persistent (a few blocks per SM, grid-stride over states) to keep the per-sweep atomics
// on the control block few.  Kernels are instantiated for every H <= 8 and for H <= 16
// (MH) so the per-host loops issue no dead iterations up to 8 hosts.
#include <math.h>

#include <algorithm>
#include <type_traits>

#include "vc_implicit.cuh"
#include "vc_internal.cuh"

namespace vc {

int state_grid(const Mdp* m) {
    const long long need = ((long long)m->S + kThreads - 1) / kThreads;
    const long long cap = (long long)(m->num_sms > 0 ? m->num_sms : 148) * 8;
    return (int)(need < cap ? need : cap);
}

// Expected one-step reward of the post-decision state: occupancy, queue and losses
// (departures lose their tasks, a full queue loses the arrival).
template <int MH, typename T>
__device__ __forceinline__ T post_reward(const Model& md, const Coef<T>& c, const Digits& d) {
    T loss = T(0);
    int occ_sum = 0;
#pragma unroll
    for (int k = 0; k < MH; k++) {
        if (k < md.H) {
            occ_sum += d.occ[k];
            loss += c.lossd[k] * T(d.occ[k]);
        }
    }
    if (d.q >= md.Q) loss += c.lossa;
    return c.w_occ * T(occ_sum) + c.w_q * T(d.q) + loss;
}

// ---------------------------------------------------------------- implicit: pass 1
// One state per thread, any precision (the FP64 backups of the refinement).
template <int MH, typename T>
__global__ void __launch_bounds__(kThreads) k_post(Model md, Coef<T> c, const T* __restrict__ V, T* __restrict__ U,
                                                   SweepCtl sc) {
    for (int x = blockIdx.x * kThreads + threadIdx.x; x < md.S; x += gridDim.x * kThreads) {
        Digits d;
        decode<MH>(md, x, d);
#ifdef VC_DEBUG_BOUNDS
        if (!successors_in_range<MH>(md, x, d, sc.ctl)) continue;
#endif
        const T rx = post_reward<MH>(md, c, d);
        U[x] = rx + c.gamma * expect_next<MH>(md, c, V, x, d);
    }
}

// FP32 pass 1 over items of VW consecutive states (vc_implicit.cuh).
template <int MH, int VW, bool SL>
__global__ void __launch_bounds__(kThreads) k_post_vec(Model md, Coef<float> c, const float* __restrict__ V,
                                                       float* __restrict__ U, float* __restrict__ W, SweepCtl sc) {
    if (loop_done(sc)) return;
    const int items = md.S / VW;
    for (int t = blockIdx.x * kThreads + threadIdx.x; t < items; t += gridDim.x * kThreads)
        post_item<MH, VW, SL>(md, c, V, VW * t, U, W, sc.ctl);
}

// ---------------------------------------------------------------- implicit: pass 2
template <int MH, typename T>
__global__ void __launch_bounds__(kThreads) k_max(Model md, const T* __restrict__ U, const T* __restrict__ V_in,
                                                  T* __restrict__ V_out, int32_t* __restrict__ pi,
                                                  T* __restrict__ qgap, SweepCtl sc) {
    T res = T(0), vabs = T(0);
    for (int s = blockIdx.x * kThreads + threadIdx.x; s < md.S; s += gridDim.x * kThreads) {
        Digits d;
        decode<MH>(md, s, d);
        T best = -INFINITY, second = -INFINITY;
        int arg = md.H;
        // every gather first (infeasible actions read nothing and count as -inf), then the
        // max in action order
        T uk[MH];
#pragma unroll
        for (int k = 0; k < MH; k++) {
            const bool f = d.q >= 1 && k < md.H && d.occ[k] < md.C && (k == md.H - 1 || d.ph == 1) &&
                           VC_IN_BOUNDS(sc.ctl, s + md.stride[k] - 2 >= 0 && s + md.stride[k] - 2 < md.S);
            uk[k] = f ? U[s + md.stride[k] - 2] : T(-INFINITY);
        }
        const T u = U[s];  // defer: the post-decision state is s itself; highest index, so ties keep lower ones
#pragma unroll
        for (int k = 0; k < MH; k++) {
            if (uk[k] > best) {
                second = best;
                best = uk[k];
                arg = k;
            } else if (uk[k] > second) {
                second = uk[k];
            }
        }
        if (u > best) {
            second = best;
            best = u;
            arg = md.H;
        } else if (u > second) {
            second = u;
        }
        if (V_out) V_out[s] = best;
        if (pi) pi[s] = arg;
        if (qgap) qgap[s] = (second == -INFINITY) ? T(INFINITY) : best - second;
        res = fmax(res, fabs(best - V_in[s]));
        vabs = fmax(vabs, fabs(best));
        if (sc.mode == kModeCert64 && sc.pi_ref && sc.pi_ref[s] != arg) atomicAdd(&sc.ctl->changes, 1ull);
    }
    if (sc.mode == kModeNone) return;
    res = block_max<T, kThreads>(res);
    vabs = block_max<T, kThreads>(vabs);
    finish_block<T>(sc, res, vabs, 0);
}

// ------------------------------------------------------- implicit: in-block iteration
// (block_tile, the local passes over one tile of blocks, lives in vc_internal.cuh: the
// batched loop runs the same routine per instance.)
template <int MH, int HIN>
__global__ void __launch_bounds__(kBlockThreads, 3) k_block(Model md, Coef<float> c, int T, int passes,
                                                const float* __restrict__ Vin, const float* __restrict__ U,
                                                const float* __restrict__ W, float* __restrict__ V_out,
                                                SweepCtl sc) {
    extern __shared__ float blk_sm[];
    if (loop_done(sc)) return;
    const long long sweep = loop_sweep(sc);
    const int ntiles = (md.S + T - 1) / T;
    float res = 0.0f, vabs = 0.0f;
    for (int t = blockIdx.x; t < ntiles; t += gridDim.x) {
        const int start = t * T;
        block_tile<MH, HIN>(md, c, start, min(T, md.S - start), passes, Vin, U, W, V_out, blk_sm, sc.ctl, res, vabs);
    }
    if (sc.mode == kModeNone) return;
    res = block_max_dyn(res);
    vabs = block_max_dyn(vabs);
    finish_block<float>(sc, res, vabs, sweep);
}

// FP32 pass 2 over the same items, with policy and Q-gap when asked for.
template <int MH, int VW, bool SL, bool ARG>
__global__ void __launch_bounds__(kThreads) k_max_vec(Model md, const float* __restrict__ U,
                                                      const float* __restrict__ W, const float* __restrict__ V_in,
                                                      float* __restrict__ V_out, int32_t* __restrict__ pi,
                                                      float* __restrict__ qgap, SweepCtl sc) {
    if (loop_done(sc)) return;
    const long long sweep = loop_sweep(sc);
    float res = 0.0f, vabs = 0.0f;
    const int items = md.S / VW;
    for (int t = blockIdx.x * kThreads + threadIdx.x; t < items; t += gridDim.x * kThreads) {
        const int s = VW * t;
        float vin[VW], best[VW], second[VW];
        int arg[VW];
        ldv<VW>(V_in + s, vin);
        max_item<MH, VW, SL, ARG>(md, U, W, s, best, second, arg, sc.ctl);
        if (V_out) stv<VW>(V_out + s, best);
#pragma unroll
        for (int j = 0; j < VW; j++) {
            if constexpr (ARG) {
                if (pi) pi[s + j] = arg[j];
                if (qgap) qgap[s + j] = second[j] == -INFINITY ? INFINITY : best[j] - second[j];
            }
            res = fmaxf(res, fabsf(best[j] - vin[j]));
            vabs = fmaxf(vabs, fabsf(best[j]));
        }
    }
    if (sc.mode == kModeNone) return;
    res = block_max<float, kThreads>(res);
    vabs = block_max<float, kThreads>(vabs);
    finish_block<float>(sc, res, vabs, sweep);
}

// ------------------------------------------------ implicit: mixed-precision refinement
// Policy residual in FP64, r(s) = U64(x_pi(s)) - V64(s) with U64 = R + gamma E[V64(next) | x]
// from the FP64 pass-1 kernel over every post-decision state (coalesced: thread x gathers
// around x), so this kernel makes one gather per state.  r is stored as float (it is small
// once V64 is near V_pi, so FP32 keeps ~1e-7 of it).
template <int MH>
__global__ void __launch_bounds__(kThreads) k_resid64(Model md, const int32_t* __restrict__ pi,
                                                      const double* __restrict__ U, const double* __restrict__ V,
                                                      float* __restrict__ r, SweepCtl sc) {
    double mx = 0.0;
    for (int s = blockIdx.x * kThreads + threadIdx.x; s < md.S; s += gridDim.x * kThreads) {
        Digits d;
        decode<MH>(md, s, d);
        int x = s;
        if (!apply_action<MH>(md, s, pi[s], d, x)) {
            atomicOr(&sc.ctl->error, kErrInfeasiblePolicy);
            r[s] = 0.0f;
            continue;
        }
#ifdef VC_DEBUG_BOUNDS
        if (!VC_IN_BOUNDS(sc.ctl, x >= 0 && x < md.S)) continue;
#endif
        const double rd = U[x] - V[s];
        r[s] = (float)rd;
        mx = fmax(mx, fabs(rd));
    }
    // kModeCert64: max |T_pi V - V| in FP64 into the control block
    if (sc.mode != kModeCert64) return;
    mx = block_max<double, kThreads>(mx);
    finish_block<double>(sc, mx, 0.0, 0);
}

// Correction sweep in FP32: e_out(s) = r(s) + gamma E[e_in(next) | x_pi(s)].  Its fixed
// point e solves (I - gamma P_pi) e = r, so V64 + e is the evaluation of pi.
template <int MH>
__global__ void __launch_bounds__(kThreads) k_correct32(Model md, Coef<float> c, const int32_t* __restrict__ pi,
                                                        const float* __restrict__ r, const float* __restrict__ e_in,
                                                        float* __restrict__ e_out, SweepCtl sc) {
    if (loop_done(sc)) return;
    const long long sweep = loop_sweep(sc);
    float res = 0.0f, vabs = 0.0f;
    for (int s = blockIdx.x * kThreads + threadIdx.x; s < md.S; s += gridDim.x * kThreads) {
        Digits d;
        decode<MH>(md, s, d);
        int x = s;
        if (!apply_action<MH>(md, s, pi[s], d, x)) {
            atomicOr(&sc.ctl->error, kErrInfeasiblePolicy);
            e_out[s] = e_in[s];
            continue;
        }
#ifdef VC_DEBUG_BOUNDS
        if (!successors_in_range<MH>(md, x, d, sc.ctl)) continue;
#endif
        const float v = r[s] + c.gamma * expect_next<MH>(md, c, e_in, x, d);
        e_out[s] = v;
        res = fmaxf(res, fabsf(v - e_in[s]));
        vabs = fmaxf(vabs, fabsf(v));
    }
    if (sc.mode == kModeNone) return;
    res = block_max<float, kThreads>(res);
    vabs = block_max<float, kThreads>(vabs);
    finish_block<float>(sc, res, vabs, sweep);
}

__global__ void k_axpy64(double* __restrict__ V, const float* __restrict__ e, int n) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) V[i] += (double)e[i];
}

__global__ void k_f32_to_f64(const float* __restrict__ in, double* __restrict__ out, int n) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) out[i] = (double)in[i];
}

// ------------------------------------------------------------------------ dispatch
static inline bool implicit_sweeps(const Mdp* m) { return (m->fmt & 0xF) == VC_IMPLICIT; }

// Calls f with std::integral_constant<int, MH>: MH = H for H <= 8 (the per-host loops are
// unrolled to MH, so an exact bound issues no predicated-off iterations), else 16.
template <typename F>
static int by_h(const Mdp* m, F&& f) {
    switch (m->md.H) {
        case 1: return f(std::integral_constant<int, 1>());
        case 2: return f(std::integral_constant<int, 2>());
        case 3: return f(std::integral_constant<int, 3>());
        case 4: return f(std::integral_constant<int, 4>());
        case 5: return f(std::integral_constant<int, 5>());
        case 6: return f(std::integral_constant<int, 6>());
        case 7: return f(std::integral_constant<int, 7>());
        case 8: return f(std::integral_constant<int, 8>());
        default: return f(std::integral_constant<int, 16>());
    }
}

// Inner hosts and states of the blocks of the in-block iteration: h as set on the handle,
// else the largest h whose block of 2(Q+1)(C+1)^h states fits 1024 threads.
int block_shape(const Mdp* m, int* h_out, int* B_out) {
    int h = m->blk_h;
    if (h < 0) {
        h = 0;
        long long B = 2LL * (m->md.Q + 1);
        while (h < m->md.H && h < kBlockMaxInner && B * (m->md.C + 1) <= kBlockThreads) {
            B *= (m->md.C + 1);
            h++;
        }
    }
    long long B = 2LL * (m->md.Q + 1);
    for (int k = 0; k < h; k++) B *= (m->md.C + 1);
    if (h > m->md.H || h > kBlockMaxInner || B > kBlockThreads)
        return fail(VC_ERR_ARG, "a block of the in-block iteration needs at most 3 inner hosts and 512 states");
    *h_out = h;
    *B_out = (int)B;
    return VC_OK;
}

static int launch_block(Mdp* m, const float* V_in, float* V_out, SweepCtl sc, cudaStream_t st) {
    int h = 0, B = 0, rc;
    if ((rc = block_shape(m, &h, &B))) return rc;
    // tiles of whole blocks, at most kBlockThreads states
    const int T = B * (kBlockThreads / B);
    const int threads = (T + 31) / 32 * 32;
    const size_t smem = 4 * sizeof(float) * (size_t)threads;
    const int g = state_grid(m);
    SweepCtl sc1 = sc;
    if (sc1.mode != kModeLoop32) sc1.mode = kModeNone;
    count_launches(2);
    return by_h(m, [&](auto mh) {
        constexpr int MH = decltype(mh)::value;
        auto kern = h == 0 ? k_block<MH, 0> : h == 1 ? k_block<MH, 1> : h == 2 ? k_block<MH, 2> : k_block<MH, 3>;
        if (m->blk_grid <= 0) {
            int per_sm = 0;
            VC_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout,
                                         cudaSharedmemCarveoutMaxShared));
            VC_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, threads, smem));
            m->blk_grid = std::max(1, per_sm) * (m->num_sms > 0 ? m->num_sms : 148);
        }
        const int ntiles = (m->S + T - 1) / T;
        float* U = m->U32 + kUShift;
        k_post_vec<MH, 2, true><<<g, kThreads, 0, st>>>(m->md, m->c32, V_in, U, m->U32s, sc1);
        kern<<<std::min(ntiles, m->blk_grid), threads, smem, st>>>(m->md, m->c32, T, m->blk_passes, V_in, U,
                                                                   m->U32s, V_out, sc);
        VC_CUDA(cudaGetLastError());
        return (int)VC_OK;
    });
}

int launch_sweep32(Mdp* m, const float* V_in, float* V_out, int32_t* pi, float* qgap, SweepCtl sc,
                   cudaStream_t st) {
    if (!implicit_sweeps(m)) return csr_sweep32(m, V_in, V_out, pi, qgap, sc, st);
    if (sc.block) {
        if (pi || qgap) return fail(VC_ERR_ARG, "the in-block iteration returns values only");
        return launch_block(m, V_in, V_out, sc, st);
    }
    const int g = state_grid(m);
    SweepCtl sc1 = sc;
    if (sc1.mode != kModeLoop32) sc1.mode = kModeNone;
    float* U = m->U32 + kUShift;
    const bool aligned16 = (((uintptr_t)V_in | (uintptr_t)V_out) & 15) == 0;
    count_launches(2);
    by_h(m, [&](auto mh) {
        constexpr int MH = decltype(mh)::value;
        auto go = [&](auto vw, auto sl) {
            constexpr int VW = decltype(vw)::value;
            constexpr bool SL = decltype(sl)::value;
            k_post_vec<MH, VW, SL><<<g, kThreads, 0, st>>>(m->md, m->c32, V_in, U, m->U32s, sc1);
            if (pi || qgap)
                k_max_vec<MH, VW, SL, true><<<g, kThreads, 0, st>>>(m->md, U, m->U32s, V_in, V_out, pi, qgap, sc);
            else
                k_max_vec<MH, VW, SL, false><<<g, kThreads, 0, st>>>(m->md, U, m->U32s, V_in, V_out, pi, qgap, sc);
        };
        auto by_vw = [&](auto sl) {
            if (MH <= 8 && aligned16 && wide_rows(m->md))
                go(std::integral_constant<int, MH <= 8 ? 4 : 2>(), sl);
            else
                go(std::integral_constant<int, 2>(), sl);
        };
        if (sc.self_loop)
            by_vw(std::true_type());
        else
            by_vw(std::false_type());
        return 0;
    });
    VC_CUDA(cudaGetLastError());
    return VC_OK;
}

int launch_bellman64(Mdp* m, const double* V_in, double* V_out, int32_t* pi, double* qgap, SweepCtl sc,
                     cudaStream_t st) {
    if (!m->has_model) return csr_bellman64(m, V_in, V_out, pi, qgap, sc, st);
    const int g = state_grid(m);
    SweepCtl none = sc;
    none.mode = kModeNone;
    count_launches(2);
    by_h(m, [&](auto mh) {
        constexpr int MH = decltype(mh)::value;
        k_post<MH, double><<<g, kThreads, 0, st>>>(m->md, m->c64, V_in, m->U64, none);
        k_max<MH, double><<<g, kThreads, 0, st>>>(m->md, m->U64, V_in, V_out, pi, qgap, sc);
        return 0;
    });
    VC_CUDA(cudaGetLastError());
    return VC_OK;
}

int launch_resid64(Mdp* m, const int32_t* pi, const double* V64, float* r, SweepCtl sc, cudaStream_t st) {
    if (!m->has_model) return csr_resid64(m, pi, V64, r, sc, st);
    const int g = state_grid(m);
    SweepCtl none = sc;
    none.mode = kModeNone;
    count_launches(2);
    by_h(m, [&](auto mh) {
        constexpr int MH = decltype(mh)::value;
        k_post<MH, double><<<g, kThreads, 0, st>>>(m->md, m->c64, V64, m->U64, none);
        k_resid64<MH><<<g, kThreads, 0, st>>>(m->md, pi, m->U64, V64, r, sc);
        return 0;
    });
    VC_CUDA(cudaGetLastError());
    return VC_OK;
}

int launch_correct32(Mdp* m, const int32_t* pi, const float* r, const float* e_in, float* e_out, SweepCtl sc,
                     cudaStream_t st) {
    if (!m->has_model) return csr_correct32(m, pi, r, e_in, e_out, sc, st);
    count_launches(1);
    by_h(m, [&](auto mh) {
        k_correct32<decltype(mh)::value><<<state_grid(m), kThreads, 0, st>>>(m->md, m->c32, pi, r, e_in, e_out, sc);
        return 0;
    });
    VC_CUDA(cudaGetLastError());
    return VC_OK;
}

static inline unsigned elementwise_grid(int n) {
    const int b = (n + kThreads - 1) / kThreads;
    return (unsigned)(b < 4096 ? (b > 0 ? b : 1) : 4096);
}

int launch_axpy64(double* V64, const float* e, int n, cudaStream_t st) {
    count_launches(1);
    k_axpy64<<<elementwise_grid(n), kThreads, 0, st>>>(V64, e, n);
    VC_CUDA(cudaGetLastError());
    return VC_OK;
}

int launch_f32_to_f64(const float* in, double* out, int n, cudaStream_t st) {
    count_launches(1);
    k_f32_to_f64<<<elementwise_grid(n), kThreads, 0, st>>>(in, out, n);
    VC_CUDA(cudaGetLastError());
    return VC_OK;
}

// ------------------------------------------------------------- greedy heuristic policy
// Algorithm 2 read as a policy on this MDP: with a task waiting, place it on the feasible
// host with the largest service rate (ties to the lowest index), else defer.
struct ServiceRates {
    double mu[kMaxH];
};

template <int MH>
__global__ void __launch_bounds__(kThreads) k_greedy(Model md, ServiceRates r, int32_t* __restrict__ pi) {
    for (int s = blockIdx.x * kThreads + threadIdx.x; s < md.S; s += gridDim.x * kThreads) {
        Digits d;
        decode<MH>(md, s, d);
        int best = md.H;
        double best_mu = -1.0;
        if (d.q >= 1) {
#pragma unroll
            for (int k = 0; k < MH; k++) {
                if (k < md.H && d.occ[k] < md.C && (k == md.H - 1 || d.ph == 1) && r.mu[k] > best_mu) {
                    best_mu = r.mu[k];
                    best = k;
                }
            }
        }
        pi[s] = best;
    }
}

int launch_greedy(Mdp* m, int32_t* pi, cudaStream_t st) {
    ServiceRates r;
    for (int k = 0; k < kMaxH; k++) r.mu[k] = m->rates.mu[k];
    count_launches(1);
    by_h(m, [&](auto mh) {
        k_greedy<decltype(mh)::value><<<state_grid(m), kThreads, 0, st>>>(m->md, r, pi);
        return 0;
    });
    VC_CUDA(cudaGetLastError());
    return VC_OK;
}

}  // namespace vc

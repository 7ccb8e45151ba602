// vc_grad.cu -- adjoint gradient of J = rho . V_pi with respect to the model parameters
// theta = (lambda, mu_1..mu_H, delta_1..delta_H, f, w_occ, w_loss, w_q).
//
// For a fixed policy pi, V = R_pi + gamma P_pi V, so
//     dJ/dtheta_i = lam . (dR_pi/dtheta_i + gamma (dP_pi/dtheta_i) V),
//     (I - gamma P_pi)^T lam = rho.
// lam is found from an explicit transpose P_pi^T (rows = targets, entries sorted by source so
// every product sums in one fixed order), FP32 solves refined in FP64 like the forward
// solve.  The transpose is stored in slices of 32 rows, entry j of row y at
// base[y / 32] + 32 j + y % 32, so the lanes of a warp (a row each) read and write
// consecutive entries; row after row their accesses were a row length apart (gradient step of
// 343,750 states: fill and sort 0.59 -> 0.23 ms, the two adjoint solves 3.2 -> 2.9 ms).
// The contraction regenerates every event of each state's
// post-decision state and differentiates its probability rate/Lam analytically:
// d(rate/Lam) = drate/Lam - rate dLam/Lam^2, the self-loop taking minus the others, so
// sum_s' dP V = sum_e dp_e (V(y_e) - V(x)).  Partial sums reduce per block and then in a fixed
// order, so the result is reproducible bit for bit.
#include <cooperative_groups.h>
#include <math.h>

#include <algorithm>

#include "vc_adj.cuh"
#include "vc_internal.cuh"

namespace vc {

// ------------------------------------------------------------- transpose of P_pi
__global__ void k_adj_count(Model md, Rates rt, const int32_t* __restrict__ pi, int32_t* __restrict__ cnt, int* err) {
    for (int s = blockIdx.x * blockDim.x + threadIdx.x; s < md.S; s += gridDim.x * blockDim.x) {
        int cols[kMaxRow];
        double probs[kMaxRow], R;
        const int n = model_row(md, rt, s, pi[s], cols, probs, &R);
        if (n < 0) {
            atomicOr(err, kErrInfeasiblePolicy);
            continue;
        }
        for (int j = 0; j < n; j++) atomicAdd(&cnt[cols[j]], 1);
    }
}

// Entries of every slice of 32 rows (32 x its longest row); total[0]: the entries of all rows,
// total[1]: the longest row.
__global__ void __launch_bounds__(kThreads) k_adj_width(int S, const int32_t* __restrict__ cnt, int32_t* __restrict__ width,
                                                        unsigned long long* total) {
    const int lane = threadIdx.x & 31, slices = (S + 31) / 32;
    unsigned long long sum = 0, longest = 0;
    for (int g = (blockIdx.x * kThreads + threadIdx.x) >> 5; g < slices; g += (gridDim.x * kThreads) >> 5) {
        const int n = 32 * g + lane < S ? cnt[32 * g + lane] : 0;
        const int w = __reduce_max_sync(0xffffffffu, n);
        sum += (unsigned long long)__reduce_add_sync(0xffffffffu, n);
        if (lane == 0) width[g] = 32 * w;
        longest = max(longest, (unsigned long long)w);
    }
    if (lane == 0 && sum) {
        atomicAdd(&total[0], sum);
        atomicMax(&total[1], longest);
    }
}

__global__ void k_adj_fill(Model md, Rates rt, const int32_t* __restrict__ pi, const int64_t* __restrict__ base,
                           int32_t* __restrict__ fillpos, int32_t* __restrict__ colT,
                           double* __restrict__ valT64) {
    for (int s = blockIdx.x * blockDim.x + threadIdx.x; s < md.S; s += gridDim.x * blockDim.x) {
        int cols[kMaxRow];
        double probs[kMaxRow], R;
        const int n = model_row(md, rt, s, pi[s], cols, probs, &R);
        for (int j = 0; j < n; j++) {
            const int y = cols[j];
            const int64_t slot = base[y >> 5] + 32LL * atomicAdd(&fillpos[y], 1) + (y & 31);
            colT[slot] = s;
            valT64[slot] = probs[j];
        }
    }
}

// Orders each transposed row by source state: a warp copies its slice to its own scratch (`most`
// entries), and there an entry's position is the number of the row's entries with a smaller source
// (sources are distinct), counted over the lanes' consecutive loads.  By insertion, every step
// waited for its own loads and stores: 432 us at 343,750 states.  The count is quadratic in the
// row, so a row of more than kAdjLong entries is shared by the warp, a lane per entry: a lane
// alone took 109 ms for the rows of some 2,000 entries of a host of 1,000 slots.
constexpr int kAdjLong = 32;
__global__ void __launch_bounds__(kThreads) k_adj_sort(int S, const int64_t* __restrict__ base,
                                                       const int32_t* __restrict__ cnt, unsigned char* scratch,
                                                       int64_t most, int32_t* __restrict__ colT,
                                                       float* __restrict__ valT, double* __restrict__ valT64) {
    const int lane = threadIdx.x & 31, slices = (S + 31) / 32;
    const int warps = (int)(gridDim.x * kThreads) >> 5, me = (int)(blockIdx.x * kThreads + threadIdx.x) >> 5;
    double* valU = reinterpret_cast<double*>(scratch + 12 * most * me);
    int32_t* colU = reinterpret_cast<int32_t*>(valU + most);
    for (int g = me; g < slices; g += warps) {
        const int n = 32 * g + lane < S ? cnt[32 * g + lane] : 0;
        int32_t* col = colT + base[g];
        float* val = valT + base[g];
        double* val64 = valT64 + base[g];
        for (int i0 = 0; i0 < n; i0 += 8) {
            int c[8];
            double v[8];
#pragma unroll
            for (int u = 0; u < 8; u++) {
                if (i0 + u < n) {
                    c[u] = col[lane + 32 * (i0 + u)];
                    v[u] = val64[lane + 32 * (i0 + u)];
                }
            }
#pragma unroll
            for (int u = 0; u < 8; u++) {
                if (i0 + u < n) {
                    colU[lane + 32 * (i0 + u)] = c[u];
                    valU[lane + 32 * (i0 + u)] = v[u];
                }
            }
        }
        __syncwarp();
        // entries first, first + step, .. of the row in column q of the slice
        auto place = [&](int q, int len, int first, int step) {
            for (int i = first; i < len; i += step) {
                const int c = colU[q + 32 * i];
                const double v = valU[q + 32 * i];
                int rank = 0;
#pragma unroll 4
                for (int j = 0; j < len; j++) rank += colU[q + 32 * j] < c ? 1 : 0;
                col[q + 32 * rank] = c;
                val[q + 32 * rank] = (float)v;
                val64[q + 32 * rank] = v;
            }
        };
        if (n <= kAdjLong) place(lane, n, 0, 1);
        __syncwarp();
        for (unsigned int m = __ballot_sync(0xffffffffu, n > kAdjLong); m; m &= m - 1) {
            const int q = __ffs((int)m) - 1;
            place(q, __shfl_sync(0xffffffffu, n, q), lane, 32);
            __syncwarp();
        }
    }
}

// Fixed-point sweep of the adjoint system, x' = b + gamma P^T x (the fallback solve).
__global__ void __launch_bounds__(kThreads) k_adj_sweep(int S, float gamma, AdjRows t, const float* __restrict__ b,
                                                        const float* __restrict__ x, float* __restrict__ x_out,
                                                        SweepCtl sc) {
    if (loop_done(sc)) return;
    const long long sweep = loop_sweep(sc);
    float res = 0.0f, vabs = 0.0f;
    for (int y = blockIdx.x * kThreads + threadIdx.x; y < S; y += gridDim.x * kThreads) {
        const float v = b[y] + gamma * adj_row_dot<16>(t, t.val, y, x);
        x_out[y] = v;
        res = fmaxf(res, fabsf(v - x[y]));
        vabs = fmaxf(vabs, fabsf(v));
    }
    res = block_max<float, kThreads>(res);
    vabs = block_max<float, kThreads>(vabs);
    finish_block<float>(sc, res, vabs, sweep);
}

// FP64 residual of the adjoint system r = rho + gamma P^T lam - lam (stored as float);
// max |r| into the control block's certificate slot.
__global__ void __launch_bounds__(kThreads) k_adj_resid64(int S, double gamma, AdjRows t, const double* __restrict__ rho,
                                                          const double* __restrict__ lam, float* __restrict__ r,
                                                          SweepCtl sc) {
    double res = 0.0;
    for (int y = blockIdx.x * kThreads + threadIdx.x; y < S; y += gridDim.x * kThreads) {
        const double v = rho[y] + gamma * adj_row_dot<8>(t, t.val64, y, lam) - lam[y];
        r[y] = (float)v;
        res = fmax(res, fabs(v));
    }
    res = block_max<double, kThreads>(res);
    finish_block<double>(sc, res, 0.0, 0);
}

__global__ void k_f64_to_f32(const double* __restrict__ in, float* __restrict__ out, int n) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) out[i] = (float)in[i];
}

// ------------------------------------------------------------------ contraction
// Per state s with x = x_pi(s): lam(s) * (dR(x)/dtheta + gamma sum_e dp_e (V(y_e) - V(x))).
// Every derivative is linear in a few sums over the states (w = lam(s), dV the value change of
// an event), so the states only add those, in slots of a per-block partial row, and the
// derivatives are formed from the totals: an FP64 multiply-add or two per sum and state in
// place of ~40 FP64 divisions (FP64 issues two lanes a cycle and SM here).  Together with the
// final sums below: 0.46 -> 0.08 ms at 343,750 states.
enum GradSlot : int {
    kSumJ = 0,   // rho V
    kSumFull,    // w [q = Q]
    kSumA,       // w dV(arrival)
    kSumF0,      // w dV(flip), phase 0
    kSumF1,      // w dV(flip), phase 1
    kSumQ,       // w q
    kSumHost     // MH each: w o_k, w o_k dV(completion on k), w dV(departure of k)
};
constexpr int grad_slots(int MH) { return kSumHost + 3 * MH; }

template <int MH>
__global__ void __launch_bounds__(kThreads) k_grad_contract(Model md, const int32_t* __restrict__ pi,
                                                            const double* __restrict__ V,
                                                            const double* __restrict__ lam,
                                                            const double* __restrict__ rho,
                                                            double* __restrict__ partial) {
    constexpr int NT = grad_slots(MH);
    double g[NT];
#pragma unroll
    for (int i = 0; i < NT; i++) g[i] = 0.0;
    const int H = md.H;
    for (int s = blockIdx.x * kThreads + threadIdx.x; s < md.S; s += gridDim.x * kThreads) {
        Digits d;
        decode<MH>(md, s, d);
        int x = s;
        if (!apply_action<MH>(md, s, pi[s], d, x)) continue;  // rejected by the count kernel
        const double vx = V[x], w = lam[s];
        const bool full = d.q >= md.Q;
        // every gather first
        double v1[MH], v0[MH];
#pragma unroll
        for (int k = 0; k < MH; k++) {
            const bool on = k < H && d.occ[k] > 0;
            v1[k] = on ? V[x - md.stride[k]] : vx;
            v0[k] = on ? V[x - d.occ[k] * md.stride[k]] : vx;
        }
        const double va = full ? vx : V[x + 2];
        const double vf = V[d.ph ? x - 1 : x + 1];
        g[kSumJ] = fma(rho[s], V[s], g[kSumJ]);
        if (full) g[kSumFull] += w;
        g[kSumA] = fma(w, va - vx, g[kSumA]);
        if (d.ph) g[kSumF1] = fma(w, vf - vx, g[kSumF1]);
        else g[kSumF0] = fma(w, vf - vx, g[kSumF0]);
        g[kSumQ] = fma(w, (double)d.q, g[kSumQ]);
#pragma unroll
        for (int k = 0; k < MH; k++) {
            if (k < H) {
                const double wo = w * d.occ[k];
                g[kSumHost + k] += wo;
                g[kSumHost + MH + k] = fma(wo, v1[k] - vx, g[kSumHost + MH + k]);
                g[kSumHost + 2 * MH + k] = fma(w, v0[k] - vx, g[kSumHost + 2 * MH + k]);
            }
        }
    }
    // block reduction, fixed order: warp shuffles, then warps in index order
    __shared__ double part[kThreads / 32][NT];
    const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
#pragma unroll
    for (int i = 0; i < NT; i++) {
        double v = g[i];
        for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
        if (lane == 0) part[wid][i] = v;
    }
    __syncthreads();
    if (threadIdx.x < NT) {
        double v = 0.0;
        for (int w2 = 0; w2 < kThreads / 32; w2++) v += part[w2][threadIdx.x];
        partial[(size_t)blockIdx.x * NT + threadIdx.x] = v;
    }
}

// Adds the per-block rows (a warp per slot, its lanes' strided sums in a fixed tree) and
// forms the packed derivatives (lambda, mu_0..mu_{H-1}, delta_0..delta_{H-1}, f, w_occ, w_loss,
// w_q) and J from the totals.
__global__ void __launch_bounds__(kThreads) k_grad_final(const double* __restrict__ partial, int nblocks, int MH, int C,
                                                         int H, Rates rt, double gamma, double* __restrict__ out) {
    __shared__ double t[grad_slots(kMaxH)];
    const int NT = grad_slots(MH), lane = threadIdx.x & 31;
    for (int i = threadIdx.x >> 5; i < NT; i += kThreads / 32) {
        double v = 0.0;
        for (int b = lane; b < nblocks; b += 32) v += partial[(size_t)b * NT + i];
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if (lane == 0) t[i] = v;
    }
    __syncthreads();
    const int i = threadIdx.x;
    if (i >= 2 * H + 6) return;
    const double Lam = rt.Lam, Lam2 = rt.Lam * rt.Lam;
    // w (tasks lost per unit of time) and w (sum of rate x value change)
    double L = rt.lambda * t[kSumFull], occ = 0.0;
    double D = rt.lambda * t[kSumA] + rt.f * t[kSumF0] + (1.0 - rt.f) * t[kSumF1];
    for (int k = 0; k < H; k++) {
        occ += t[kSumHost + k];
        L += rt.delta[k] * t[kSumHost + k];
        D += rt.mu[k] * t[kSumHost + MH + k] + rt.delta[k] * t[kSumHost + 2 * MH + k];
    }
    double v;
    if (i == 0) {
        v = rt.w_loss * (t[kSumFull] / Lam - L / Lam2) + gamma * (t[kSumA] / Lam - D / Lam2);
    } else if (i <= H) {
        const int k = i - 1;
        v = -rt.w_loss * L * C / Lam2 + gamma * (t[kSumHost + MH + k] / Lam - C * D / Lam2);
    } else if (i <= 2 * H) {
        const int k = i - 1 - H;
        v = rt.w_loss * (t[kSumHost + k] / Lam - L / Lam2) + gamma * (t[kSumHost + 2 * MH + k] / Lam - D / Lam2);
    } else if (i == 2 * H + 1) {
        v = gamma * (t[kSumF0] - t[kSumF1]) / Lam;
    } else if (i == 2 * H + 2) {
        v = occ;
    } else if (i == 2 * H + 3) {
        v = L / Lam;
    } else if (i == 2 * H + 4) {
        v = t[kSumQ];
    } else {
        v = t[kSumJ];
    }
    out[i] = v;
}

// J = rho . V in FP64 by one cluster: each thread sums its strided states in index order, each
// block halves the partials in a fixed tree and the first block adds the blocks' in order, so the
// result is reproducible bit for bit and needs no scratch memory.  Bound by the FP64 adds and
// the latency of a thread's chain of loads; one block took 89 us at 343,750 states.
constexpr int kObjBlocks = 8, kObjThreads = 1024;
__global__ void __cluster_dims__(kObjBlocks, 1, 1) __launch_bounds__(kObjThreads)
    k_objective(const double* __restrict__ V, const double* __restrict__ rho, long long S, double* __restrict__ J) {
    namespace cg = cooperative_groups;
    __shared__ double part[kObjThreads];
    double acc = 0.0;
#pragma unroll 4
    for (long long s = (long long)blockIdx.x * kObjThreads + threadIdx.x; s < S; s += kObjBlocks * kObjThreads)
        acc = fma(rho[s], V[s], acc);
    part[threadIdx.x] = acc;
    __syncthreads();
    for (int w = kObjThreads / 2; w > 0; w >>= 1) {
        if ((int)threadIdx.x < w) part[threadIdx.x] += part[threadIdx.x + w];
        __syncthreads();
    }
    cg::cluster_group cl = cg::this_cluster();
    cl.sync();
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        double v = 0.0;
        for (int b = 0; b < kObjBlocks; b++) v += *cl.map_shared_rank(&part[0], b);
        *J = v;
    }
    cl.sync();
}

// ------------------------------------------------------------------------ launchers
int launch_adj_count(Mdp* m, const int32_t* pi, int32_t* cnt, int* err, cudaStream_t st) {
    count_launches(1);
    k_adj_count<<<state_grid(m), kThreads, 0, st>>>(m->md, m->rates, pi, cnt, err);
    VC_CUDA(cudaGetLastError());
    return VC_OK;
}

int launch_adj_width(Mdp* m, const int32_t* cnt, int32_t* width, unsigned long long* total, cudaStream_t st) {
    count_launches(1);
    k_adj_width<<<state_grid(m), kThreads, 0, st>>>(m->S, cnt, width, total);
    VC_CUDA(cudaGetLastError());
    return VC_OK;
}

// Blocks of k_adj_sort: enough warps to hide its loads, and no more scratch than 64 MB (which stays
// in L2) as long as 16 blocks remain; one slice of 32 rows of 6,000 entries takes 2.3 MB.
static int adj_sort_grid(const Mdp* m, int64_t most) {
    const int64_t by_scratch = std::max<int64_t>(16, (64LL << 20) / (12 * std::max<int64_t>(most, 32) * (kThreads / 32)));
    const int64_t slices = ((int64_t)m->S + 31) / 32, blocks = (slices + kThreads / 32 - 1) / (kThreads / 32);
    return (int)std::min({(int64_t)state_grid(m), by_scratch, blocks});
}

size_t adj_scratch_bytes(const Mdp* m, int64_t longest) {
    return (size_t)12 * 32 * longest * adj_sort_grid(m, 32 * longest) * (kThreads / 32);
}

int launch_adj_fill(Mdp* m, const int32_t* pi, const AdjRows& t, int32_t* fillpos, int64_t longest,
                    unsigned char* scratch, cudaStream_t st) {
    count_launches(2);
    k_adj_fill<<<state_grid(m), kThreads, 0, st>>>(m->md, m->rates, pi, t.base, fillpos, t.col, t.val64);
    k_adj_sort<<<adj_sort_grid(m, 32 * longest), kThreads, 0, st>>>(m->S, t.base, t.cnt, scratch, 32 * longest, t.col,
                                                                    t.val, t.val64);
    VC_CUDA(cudaGetLastError());
    return VC_OK;
}

int launch_adj_sweep(Mdp* m, const AdjRows& t, const float* b, const float* x, float* x_out, SweepCtl sc,
                     cudaStream_t st) {
    count_launches(1);
    k_adj_sweep<<<state_grid(m), kThreads, 0, st>>>(m->S, (float)m->gamma, t, b, x, x_out, sc);
    VC_CUDA(cudaGetLastError());
    return VC_OK;
}

int launch_adj_resid64(Mdp* m, const AdjRows& t, const double* rho, const double* lam, float* r, SweepCtl sc,
                       cudaStream_t st) {
    count_launches(1);
    k_adj_resid64<<<state_grid(m), kThreads, 0, st>>>(m->S, m->gamma, t, rho, lam, r, sc);
    VC_CUDA(cudaGetLastError());
    return VC_OK;
}

int launch_f64_to_f32(const double* in, float* out, int n, cudaStream_t st) {
    count_launches(1);
    const int b = (n + kThreads - 1) / kThreads;
    k_f64_to_f32<<<b < 4096 ? (b > 0 ? b : 1) : 4096, kThreads, 0, st>>>(in, out, n);
    VC_CUDA(cudaGetLastError());
    return VC_OK;
}

static int grad_mh(const Mdp* m) { return m->md.H <= 4 ? 4 : m->md.H <= 8 ? 8 : 16; }

// Two blocks per SM: the block sums' FP64 shuffles are then a small part.
static int grad_grid(const Mdp* m) { return std::min(state_grid(m), 2 * (m->num_sms > 0 ? m->num_sms : 148)); }

size_t grad_partial_bytes(const Mdp* m) { return 8 * (size_t)grad_grid(m) * grad_slots(grad_mh(m)); }

int launch_grad_contract(Mdp* m, const int32_t* pi, const double* V, const double* lam, const double* rho,
                         double* partial, double* out, cudaStream_t st) {
    const int g = grad_grid(m), MH = grad_mh(m);
    count_launches(2);
    if (MH == 4)
        k_grad_contract<4><<<g, kThreads, 0, st>>>(m->md, pi, V, lam, rho, partial);
    else if (MH == 8)
        k_grad_contract<8><<<g, kThreads, 0, st>>>(m->md, pi, V, lam, rho, partial);
    else
        k_grad_contract<16><<<g, kThreads, 0, st>>>(m->md, pi, V, lam, rho, partial);
    k_grad_final<<<1, kThreads, 0, st>>>(partial, g, MH, m->md.C, m->md.H, m->rates, m->gamma, out);
    VC_CUDA(cudaGetLastError());
    return VC_OK;
}

int launch_objective(const double* V, const double* rho, long long S, double* J, cudaStream_t st) {
    count_launches(1);
    k_objective<<<kObjBlocks, kObjThreads, 0, st>>>(V, rho, S, J);
    VC_CUDA(cudaGetLastError());
    return VC_OK;
}

}  // namespace vc

// The objective of the gradient entry point, exported on its own: J = rho . V.
extern "C" int vc_objective(const double* V, const double* rho, int64_t S, double* J, void* stream) {
    vc::set_error("");
    if (!V || !rho || !J) return vc::fail(VC_ERR_ARG, "vc_objective: NULL argument");
    if (S < 1) return vc::fail(VC_ERR_ARG, "vc_objective: S < 1");
    return vc::launch_objective(V, rho, (long long)S, J, (cudaStream_t)stream);
}

// vc_krylov.cu -- BiCGSTAB for the correction equation (I - gamma P_pi) e = r of the
// mixed-precision refinement (single handle), one resident kernel for the whole solve.
//
// Launched kernel by kernel an iteration is five launches, 1,216 blocks' tickets on the
// control block and FP64 block sums (two FP64 multiply-adds per SM and cycle on this chip), with
// host reads in between.  Here at most one CTA per SM stays for the whole solve: a CTA owns the
// same states in every vector, so only p and s cross CTAs; a grid barrier separates the five
// steps; the threads' dot products are added as three FP32 terms (Sum3), so FP64 is left with
// one partial per CTA; and every CTA adds the same partials in the same order and advances its
// own copy of the scalars.
//
// A dot product is a sum of FP32 chains, chain c over the states c, c + chains, c + 2 chains, ..
// with `chains` fixed by the model's size and the device (state_grid x kThreads).  The chains
// are grouped by thread, warp and CTA and added in no less than FP64's precision: a solve is
// reproducible bit for bit for a fixed grid and item width, and others agree with it up to that
// rounding.
//
// The product by A = I - gamma P_pi has three forms: from the stored rows; from the implicit
// model state by state (2H + 3 scalar gathers around x_pi(s)); and, for large models, in two
// passes as a sweep does it: E[x(next) | .] of every post-decision state by items of four
// (two) states, then one gather per state.  The two-pass form trades a grid barrier (1.5 us)
// for a quarter of the load instructions.
//
// Bound: L2 latency of the gathers and of five short vector steps, and five (seven) barriers an
// iteration.  Whole calls, launched kernels against this one: evaluation of a policy of
// 524,288 states 8.6 -> 2.8 ms, gradient step of 343,750 states 12.3 -> 8.6 ms, solves of
// 2.5 M states 10.1 -> 8.0 ms and of 640 states 0.74 -> 0.47 ms.
#include <math.h>
#include <string.h>

#include <algorithm>
#include <type_traits>

#include "vc_adj.cuh"
#include "vc_grid.cuh"
#include "vc_implicit.cuh"
#include "vc_krylov.cuh"

namespace vc {

constexpr int kKrThreads = 512;
constexpr int kKrOneCta = 2048;     // unknowns up to which one CTA solves alone (no grid barrier)
constexpr int kKrItems = 128;       // least items of a CTA otherwise

// Vectors of one solve (FP32, n entries each) and the reduction scratch.
struct KrylovArgs {
    KrylovCtl* kc;
    Ctl* ctl;          // the handle's control block (error flags of the bounds-checking build)
    double* part;      // [kKrPartSets][kKrPartValues][gridDim.x] (kr_part_set)
    const float* b;    // right-hand side and shadow residual
    float *x, *r, *p, *v, *s, *t;
    float* e;          // E[x(next) | .] of the two-pass product
    int32_t* post;     // x_pi(s) of every state (implicit model; -1: infeasible, a row of the identity)
    int n;
    int chains;        // FP32 chains of a dot product (a multiple of 4, or at least n)
};

// Scalars of the stage, from the grid totals (one thread).
__device__ inline void kr_advance(KrylovCtl* c, int stage, double d0, double d1, double mx) {
    if (stage == kKrInit) {
        c->rho = d0;  // <b, r0> with r0 = b
        c->rmax = (float)mx;
        // one FP32 solve reduces the residual by 2^-18 at most (the refinement's next
        // FP64 round takes it further), so the target never asks for more
        c->target = fmax(c->target, ldexp(mx, -18));
        c->alpha = c->omega = 1.0;
        c->beta = 0.0;
        c->iter = 0;
        if (mx < c->target) c->done = 1;
        else if (!(d0 > 0.0)) c->done = 5;
    } else if (stage == kKrV) {
        // alpha = rho / <b, v>
        if (d0 == 0.0 || !isfinite(d0)) {
            c->done = 5;
        } else {
            c->alpha = c->rho / d0;
        }
    } else if (stage == kKrT) {
        // omega = <t, s> / <t, t>; t = 0 means s = 0 (A is non-singular): omega = 0 and
        // the x / r update below ends the solve with r = s = 0
        c->omega = (d1 > 0.0) ? d0 / d1 : 0.0;
        if (!isfinite(c->omega)) c->done = 5;
    } else {
        // after x += alpha p + omega s, r = s - omega t
        c->rmax = (float)mx;
        c->iter += 1;
        if (mx < c->target) {
            c->done = 1;
        } else if (c->iter >= c->max_iter) {
            c->done = 2;
        } else if (c->omega == 0.0 || c->rho == 0.0 || !isfinite(mx)) {
            c->done = 5;
        } else {
            c->beta = (d0 / c->rho) * (c->alpha / c->omega);
            c->rho = d0;
            if (!isfinite(c->beta) || d0 == 0.0) c->done = 5;
        }
    }
}

// A sum of FP32 values as three unevaluated FP32 terms, every addition but the last term's split
// exactly (Knuth's two-sum; SumK with K = 3 of T. Ogita, S. M. Rump, S. Oishi, "Accurate sum and
// dot product", SIAM J. Sci. Comput. 26(6), 2005), so it comes out as if summed in about three
// times FP32's precision: no worse than FP64, which this chip adds at two a cycle and SM.
struct Sum3 {
    float s = 0.0f, c = 0.0f, e = 0.0f;
    static __device__ __forceinline__ float two_sum(float& a, float p) {
        const float t = __fadd_rn(a, p), z = __fsub_rn(t, a);
        const float err = __fadd_rn(__fsub_rn(a, __fsub_rn(t, z)), __fsub_rn(p, z));
        a = t;
        return err;
    }
    __device__ __forceinline__ void add(float p) { e += two_sum(c, two_sum(s, p)); }
    __device__ __forceinline__ void merge(float os, float oc, float oe) {
        add(os);
        e += two_sum(c, oc) + oe;
    }
    __device__ __forceinline__ double value() const { return ((double)e + (double)c) + (double)s; }
};

// The same with FP64's range for FP32 terms: once one of 2^96 or more (an infinity, a NaN) is
// met, the sum goes on scaled by 2^-32, which no sum of FP32 terms overflows; what that shifts
// out lies more than 200 bits below the term.
struct DotSum {
    static constexpr float kLarge = 0x1p96f, kDown = 0x1p-32f;
    static constexpr double kUp = 0x1p32;
    Sum3 v;
    float scale = 1.0f;
    __device__ __forceinline__ void scale_down() {
        v.s *= kDown;
        v.c *= kDown;
        v.e *= kDown;
        scale = kDown;
    }
    __device__ __forceinline__ void add(float p) {
        if (!(fabsf(p) < kLarge) && scale == 1.0f) [[unlikely]]
            scale_down();
        v.add(p * scale);
    }
    // One scale for the warp (every lane calls it).
    __device__ __forceinline__ void align() {
        if (__any_sync(0xffffffffu, scale != 1.0f)) [[unlikely]] {
            if (scale == 1.0f) scale_down();
        }
    }
    // The sum over the half-warp's lanes, one scale in all of them.
    __device__ __forceinline__ void half_warp_sum() {
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) add_lane(v, o);
    }
    // This lane's terms plus those that lane ^ o gives.
    __device__ __forceinline__ void add_lane(const Sum3& given, int o) {
        const float s = __shfl_xor_sync(0xffffffffu, given.s, o), c = __shfl_xor_sync(0xffffffffu, given.c, o);
        v.merge(s, c, __shfl_xor_sync(0xffffffffu, given.e, o));
    }
    __device__ __forceinline__ double value() const { return scale == 1.0f ? v.value() : kUp * v.value(); }
    __device__ __forceinline__ float4 words() const { return make_float4(v.s, v.c, v.e, scale); }
    __device__ __forceinline__ void set(const float4& w) { v.s = w.x, v.c = w.y, v.e = w.z, scale = w.w; }
};

struct KrShared {
    KrylovCtl c;                           // this CTA's copy of the scalars
    float4 dot[2][kKrThreads / 32];        // the warps' sums
    unsigned int mx;                       // bits of the CTA's max |r|
    double tot[2];
    long long end, start;                  // iterations at which this launch ends, its first cycle
    int fail;
};

// CTA totals -> grid totals -> scalars of `stage` in every CTA's copy.  False once a barrier
// wait gave up.  D1, MX: whether the stage has a second dot product, a maximum.
template <bool D1, bool MX>
__device__ __forceinline__ bool kr_reduce(const KrylovArgs& k, KrShared& sh, GridBarrier& bar, int stage, DotSum a0,
                                          DotSum a1, float mx, const LaunchEnd* end = nullptr) {
    const int w = (int)threadIdx.x >> 5, l = (int)threadIdx.x & 31, nw = (int)blockDim.x >> 5;
    // lanes 0..15 add up the first product, 16..31 the second (without one, the first again)
    static_assert(kKrThreads / 32 <= 16, "a half-warp adds up the warps' sums");
    DotSum t = a0;
    if (D1) {
        if (a0.scale != a1.scale) {
            if (a0.scale == 1.0f) a0.scale_down();
            else a1.scale_down();
        }
        a0.align();
        a1.align();
        t = l < 16 ? a0 : a1;
        t.add_lane(l < 16 ? a1.v : a0.v, 16);
    } else {
        t.align();
        t.add_lane(t.v, 16);
    }
    t.half_warp_sum();
    const unsigned int mb = MX ? __reduce_max_sync(0xffffffffu, fbits(mx)) : 0u;
    if (l == 0 || (D1 && l == 16)) sh.dot[l >> 4][w] = t.words();
    if (MX && l == 0) atomicMax(&sh.mx, mb);
    __syncthreads();
    const int G = (int)gridDim.x;
    double* part = k.part + kr_part_set(stage) * kKrPartValues * G;
    if (w == 0) {
        DotSum sum;
        if ((l & 15) < nw && (D1 || l < 16)) sum.set(sh.dot[l >> 4][l & 15]);
        sum.align();
        sum.half_warp_sum();
        const double v0 = sum.value(), v1 = D1 ? __shfl_sync(0xffffffffu, v0, 16) : 0.0;
        if (l == 0) {
            if (G == 1) {
                sh.tot[0] = v0;
                sh.tot[1] = v1;
            } else {
                part[blockIdx.x] = v0;
                if (D1) part[G + blockIdx.x] = v1;
                if (MX) *reinterpret_cast<unsigned int*>(part + 2 * G + blockIdx.x) = sh.mx;  // FP32 bits
            }
        }
    }
    if (!bar.arrive_and_wait()) return false;
    if (end && threadIdx.x == blockDim.x - 1) sh.end = end->read();  // beside warp 0's reads
    if (w == 0) {
        double v0 = 0.0, v1 = 0.0;
        unsigned int vm = 0u;
        if (G > 1) {
            // as above: a half-warp a product
            const double* mine = part + (D1 && l >= 16 ? G : 0);
            for (int i = D1 ? l & 15 : l; i < G; i += D1 ? 16 : 32) {
                v0 += __ldcg(mine + i);
                if (MX) vm = max(vm, __ldcg(reinterpret_cast<const unsigned int*>(part + 2 * G + i)));
            }
#pragma unroll
            for (int o = D1 ? 8 : 16; o > 0; o >>= 1) v0 += __shfl_xor_sync(0xffffffffu, v0, o);
            if (D1) v1 = __shfl_sync(0xffffffffu, v0, 16);
            if (MX) vm = __reduce_max_sync(0xffffffffu, vm);
        } else if (l == 0) {
            v0 = sh.tot[0];
            v1 = sh.tot[1];
            if (MX) vm = sh.mx;
        }
        if (l == 0) {
            kr_advance(&sh.c, stage, v0, v1, (double)__uint_as_float(vm));
            if (MX) sh.mx = 0u;  // next written after the caller's barriers
        }
    }
    __syncthreads();
    return true;
}

// ------------------------------------------------------------------------- products
// Implicit model, one state at a time: y(s) = x(s) - gamma E[x(next) | x_pi(s)].  The policy
// was checked feasible by the residual pass; an infeasible entry acts as the identity.
template <int MH>
struct ModelProduct {
    static constexpr int kWidth = 1;
    static constexpr bool kTwoPass = false;
    Model md;
    Coef<float> c;
    const int32_t* pi;
    __device__ __forceinline__ void setup(const KrylovArgs& k, int s) const {
        Digits d;
        decode<MH>(md, s, d);
        int x = s;
        k.post[s] = apply_action<MH>(md, s, pi[s], d, x) ? x : -1;
    }
    __device__ __forceinline__ void first(const KrylovArgs&, const float*, int) const {}
    __device__ __forceinline__ void row(const KrylovArgs& k, const float* xin, int s, float* y) const {
        y[0] = xin[s];
        const int x = k.post[s];
        if (x < 0) return;
        Digits d;
        decode<MH>(md, x, d);
#ifdef VC_DEBUG_BOUNDS
        if (!successors_in_range<MH>(md, x, d, k.ctl)) return;
#endif
        y[0] -= c.gamma * expect_next<MH>(md, c, xin, x, d);
    }
};

// Implicit model in two passes over items of VW states.
template <int MH, int VW>
struct ModelProduct2 {
    static constexpr int kWidth = VW;
    static constexpr bool kTwoPass = true;
    Model md;
    Coef<float> c;
    const int32_t* pi;
    __device__ __forceinline__ void setup(const KrylovArgs& k, int s0) const {
        for (int j = 0; j < VW; j++) {
            Digits d;
            decode<MH>(md, s0 + j, d);
            int x = s0 + j;
            k.post[s0 + j] = apply_action<MH>(md, s0 + j, pi[s0 + j], d, x) ? x : -1;
        }
    }
    __device__ __forceinline__ void first(const KrylovArgs& k, const float* xin, int s) const {
        post_item<MH, VW, false, true>(md, c, xin, s, k.e, nullptr, k.ctl);
    }
    __device__ __forceinline__ void row(const KrylovArgs& k, const float* xin, int s, float* y) const {
        int x[VW];
        ldv<VW>(xin + s, y);
#pragma unroll
        for (int j = 0; j < VW; j += 2) {
            const int2 t = *reinterpret_cast<const int2*>(k.post + s + j);
            x[j] = t.x;
            x[j + 1] = t.y;
        }
#pragma unroll
        for (int j = 0; j < VW; j++)
            if (x[j] >= 0 && VC_IN_BOUNDS(k.ctl, x[j] < k.n)) y[j] -= c.gamma * k.e[x[j]];
    }
};

// Stored rows of pi: y(s) = x(s) - gamma (scale) sum_j val_j x[col_j], fused multiply-adds in
// column order; the gathers of eight entries are in flight before the first of them is added.
template <typename VT>
struct RowProduct {
    static constexpr int kWidth = 1;
    static constexpr bool kTwoPass = false;
    int A;
    float gamma;
    const int64_t* row_ptr;
    const int32_t* col;
    const VT* val;
    const float* scale;
    const int32_t* pi;
    static __device__ __forceinline__ float value(const VT* p) {
        if constexpr (sizeof(VT) == 4) return __ldg(p);
        else return __uint_as_float((uint32_t)__ldg(p) << 16);
    }
    __device__ __forceinline__ void setup(const KrylovArgs&, int) const {}
    __device__ __forceinline__ void first(const KrylovArgs&, const float*, int) const {}
    __device__ __forceinline__ void row(const KrylovArgs& k, const float* xin, int s, float* y) const {
        y[0] = xin[s];
        const int act = pi[s];
        if (act < 0 || act >= A) return;
        const int64_t r = (int64_t)s * A + act;
        const int64_t lo = __ldg(row_ptr + r);
        const int n = (int)(__ldg(row_ptr + r + 1) - lo);
        float acc = 0.0f;
        for (int j0 = 0; j0 < n; j0 += 8) {
            float w[8], g[8];
#pragma unroll
            for (int u = 0; u < 8; u++) {
                w[u] = g[u] = 0.0f;
                if (j0 + u < n) {
                    w[u] = value(val + lo + j0 + u);
                    const int cj = __ldg(col + lo + j0 + u);
                    if (VC_IN_BOUNDS(k.ctl, cj >= 0 && cj < k.n)) g[u] = xin[cj];
                }
            }
#pragma unroll
            for (int u = 0; u < 8; u++)
                if (j0 + u < n) acc = fmaf(w[u], g[u], acc);
        }
        if (scale) acc *= __ldg(scale + r);
        y[0] -= gamma * acc;
    }
};

// The adjoint's rows, in slices of 32 (AdjRows): the lanes of a warp read consecutive entries.
struct AdjProduct {
    static constexpr int kWidth = 1;
    static constexpr bool kTwoPass = false;
    float gamma;
    AdjRows t;
    __device__ __forceinline__ void setup(const KrylovArgs&, int) const {}
    __device__ __forceinline__ void first(const KrylovArgs&, const float*, int) const {}
    __device__ __forceinline__ void row(const KrylovArgs& k, const float* xin, int s, float* y) const {
        y[0] = xin[s] - gamma * adj_row_dot<16>(t, t.val, s, xin);
    }
};

// ---------------------------------------------------------------------------- kernel
template <typename Op>
__global__ void __launch_bounds__(kKrThreads, 1) k_krylov(Op op, KrylovArgs k) {
    constexpr int VW = Op::kWidth;
    __shared__ KrShared sh;
    const int n = k.n, chains = k.chains, step = (int)blockDim.x;
    // this CTA's items of the two-pass product's first pass: one contiguous range of states
    const int per1 = (n / VW + (int)gridDim.x - 1) / (int)gridDim.x;
    const int f0 = (int)blockIdx.x * per1 + (int)threadIdx.x, f1 = min(n / VW, (int)(blockIdx.x + 1) * per1);
    // its items of everything else: the states of one contiguous range of chains
    const int vitems = min(n, chains) / VW;
    const int per = (vitems + (int)gridDim.x - 1) / (int)gridDim.x;
    const int c0 = (int)blockIdx.x * per + (int)threadIdx.x, c1 = min(vitems, (int)(blockIdx.x + 1) * per);
    if (threadIdx.x == 0) {
        sh.c = *k.kc;
        sh.mx = 0u;
        sh.fail = 0;
        sh.end = sh.c.iter + kLaunchSweeps;
    }
    __syncthreads();
    GridBarrier bar{&k.kc->arrivals, gridDim.x, 0u, &sh.fail, barrier_polls(sh.c.spin_limit)};
    const bool resumed = sh.c.iter > 0;
    const bool first_cta = threadIdx.x == 0 && blockIdx.x == 0;
    LaunchEnd end{&k.kc->launch_end, &sh.start};
    if (first_cta) end.open(sh.c.iter);
    bool ok = true;
    if (!resumed) {
        // r = b, x = 0, with <b, b> and max |b|
        DotSum a0;
        float mx = 0.0f;
        for (int v = c0; v < c1; v += step) {
            float d0[VW] = {};
            for (long long i = (long long)VW * v; i < n; i += chains) {
                op.setup(k, (int)i);
                float b[VW], z[VW] = {};
                ldv<VW>(k.b + i, b);
#pragma unroll
                for (int j = 0; j < VW; j++) {
                    d0[j] = fmaf(b[j], b[j], d0[j]);
                    mx = fmaxf(mx, fabsf(b[j]));
                }
                stv<VW>(k.r + i, b);
                stv<VW>(k.x + i, z);
            }
#pragma unroll
            for (int j = 0; j < VW; j++) a0.add(d0[j]);
        }
        ok = kr_reduce<false, true>(k, sh, bar, kKrInit, a0, DotSum(), mx);
    }
    // y = A x over the owned states, with the dot products of the stage
    auto product = [&](const float* xin, float* y, bool second) {
        if (!bar.sync()) return false;  // x is complete
        if constexpr (Op::kTwoPass) {
            for (int t = f0; t < f1; t += step) op.first(k, xin, VW * t);
            if (!bar.sync()) return false;
        }
        DotSum a0, a1;
        for (int v = c0; v < c1; v += step) {
            float d0[VW] = {}, d1[VW] = {};
            for (long long i = (long long)VW * v; i < n; i += chains) {
                float yv[VW], w[VW];
                ldv<VW>((second ? xin : k.b) + i, w);
                op.row(k, xin, (int)i, yv);
                stv<VW>(y + i, yv);
#pragma unroll
                for (int j = 0; j < VW; j++) {
                    d0[j] = fmaf(w[j], yv[j], d0[j]);
                    d1[j] = fmaf(yv[j], yv[j], d1[j]);
                }
            }
#pragma unroll
            for (int j = 0; j < VW; j++) {
                a0.add(d0[j]);
                a1.add(d1[j]);
            }
        }
        return second ? kr_reduce<true, false>(k, sh, bar, kKrT, a0, a1, 0.0f)
                      : kr_reduce<false, false>(k, sh, bar, kKrV, a0, a1, 0.0f);
    };
    while (ok && !sh.c.done && sh.c.iter < sh.end) {
        if (first_cta) end.check(sh.c.iter);
        // p = r (first iteration), else p = r + beta (p - omega v)
        const bool first = sh.c.iter == 0;
        const float beta = (float)sh.c.beta, omega0 = (float)sh.c.omega;
        for (int v0 = c0; v0 < c1; v0 += step)
            for (long long i = (long long)VW * v0; i < n; i += chains) {
                float r[VW], p[VW], v[VW];
                ldv<VW>(k.r + i, r);
                if (!first) {
                    ldv<VW>(k.p + i, p);
                    ldv<VW>(k.v + i, v);
#pragma unroll
                    for (int j = 0; j < VW; j++) r[j] = fmaf(beta, fmaf(-omega0, v[j], p[j]), r[j]);
                }
                stv<VW>(k.p + i, r);
            }
        if (!(ok = product(k.p, k.v, false)) || sh.c.done) break;
        // s = r - alpha v
        const float alpha = (float)sh.c.alpha;
        for (int v0 = c0; v0 < c1; v0 += step)
            for (long long i = (long long)VW * v0; i < n; i += chains) {
                float r[VW], v[VW];
                ldv<VW>(k.r + i, r);
                ldv<VW>(k.v + i, v);
#pragma unroll
                for (int j = 0; j < VW; j++) r[j] = fmaf(-alpha, v[j], r[j]);
                stv<VW>(k.s + i, r);
            }
        if (!(ok = product(k.s, k.t, true)) || sh.c.done) break;
        // x += alpha p + omega s; r = s - omega t, with <b, r> and max |r|
        const float omega = (float)sh.c.omega;
        DotSum a0;
        float mx = 0.0f;
        for (int v0 = c0; v0 < c1; v0 += step) {
            float d0[VW] = {};
            for (long long i = (long long)VW * v0; i < n; i += chains) {
                float x[VW], p[VW], s[VW], t[VW], b[VW];
                ldv<VW>(k.x + i, x);
                ldv<VW>(k.p + i, p);
                ldv<VW>(k.s + i, s);
                ldv<VW>(k.t + i, t);
                ldv<VW>(k.b + i, b);
#pragma unroll
                for (int j = 0; j < VW; j++) {
                    x[j] += fmaf(alpha, p[j], omega * s[j]);
                    s[j] = fmaf(-omega, t[j], s[j]);
                    d0[j] = fmaf(b[j], s[j], d0[j]);
                    mx = fmaxf(mx, fabsf(s[j]));
                }
                stv<VW>(k.x + i, x);
                stv<VW>(k.r + i, s);
            }
#pragma unroll
            for (int j = 0; j < VW; j++) a0.add(d0[j]);
        }
        ok = kr_reduce<false, true>(k, sh, bar, kKrX, a0, DotSum(), mx, &end);
    }
    if (threadIdx.x != 0) return;
    if (sh.fail) atomicOr(&k.kc->fault, 1);
    if (blockIdx.x == 0) {
        KrylovCtl* c = k.kc;
        c->rho = sh.c.rho;
        c->alpha = sh.c.alpha;
        c->omega = sh.c.omega;
        c->beta = sh.c.beta;
        c->target = sh.c.target;
        c->rmax = sh.c.rmax;
        c->done = sh.c.done;
        c->iter = sh.c.iter;
    }
}

// Enqueues one launch.  The grid is at most one CTA per SM; where the device cannot hold it
// at once (a partitioned GPU) it is halved until it can.
template <typename Op>
static int krylov_run(const Mdp* m, const Op& op, const KrylovArgs& k, cudaStream_t st, ResidentTurn& turn) {
    const int sms = m->num_sms > 0 ? m->num_sms : 148;
    const int items = std::min(k.n, k.chains) / Op::kWidth;
    int grid = k.n <= kKrOneCta ? 1 : std::max(1, std::min(sms, items / kKrItems));
    for (;; grid = std::max(1, grid / 2)) {
        const int per = (items + grid - 1) / grid;
        const int threads = std::min(kKrThreads, std::max(32, (per + 31) / 32 * 32));
        bool launched = false;
        const int rc = launch_resident((const void*)k_krylov<Op>, (items + per - 1) / per, threads, 0, st, turn,
                                       sms, &launched, op, k);
        if (rc || launched) return rc;
        if (grid == 1) return fail(VC_ERR_CUDA, "the correction solve's kernel does not fit the device");
    }
}

// States from which the two-pass product is the faster one.  Evaluation of a policy, one pass
// against two: 25,920 states 1.24 / 1.33 ms, 100,000 1.73 / 1.75, 131,072 1.90 / 1.82, 250,000
// 2.01 / 1.66, 524,288 3.58 / 2.72; items of two states (Q even): 343,750 2.77 / 2.35.
constexpr int kKrTwoPass = 120000;

static int krylov_launch(const Mdp* m, const int32_t* pi, const KrylovArgs& k, cudaStream_t st, ResidentTurn& turn) {
    if (m->adj) return krylov_run(m, AdjProduct{(float)m->gamma, *m->adj}, k, st, turn);
    if (!m->has_model) {
        if ((m->fmt & 0xF) == VC_CSR_BF16) {
            RowProduct<uint16_t> op{m->A, (float)m->gamma, m->row_ptr, m->col, (const uint16_t*)m->val, m->scale, pi};
            return krylov_run(m, op, k, st, turn);
        }
        RowProduct<float> op{m->A, (float)m->gamma, m->row_ptr, m->col, (const float*)m->val, m->scale, pi};
        return krylov_run(m, op, k, st, turn);
    }
    const bool two = m->S >= kKrTwoPass;
    auto go = [&](auto mh) -> int {
        constexpr int MH = decltype(mh)::value;
        if (two && MH <= 8 && wide_rows(m->md))
            return krylov_run(m, ModelProduct2<MH, MH <= 8 ? 4 : 2>{m->md, m->c32, pi}, k, st, turn);
        if (two) return krylov_run(m, ModelProduct2<MH, 2>{m->md, m->c32, pi}, k, st, turn);
        return krylov_run(m, ModelProduct<MH>{m->md, m->c32, pi}, k, st, turn);
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

int krylov_correct(Mdp* m, const int32_t* pi, const float* b, float* x, double target, long long max_iter,
                   cudaStream_t st, long long* products, bool* converged) {
    *products = 0;
    *converged = false;
    const size_t S = krylov_stride(m->S);
    KrylovCtl& h = *m->kctl_host;
    memset(&h, 0, sizeof(KrylovCtl));
    h.target = target;
    h.spin_limit = m->spin_polls < 0 ? 0 : m->spin_polls + 1;
    h.max_iter = (int)std::min<long long>(std::max<long long>(max_iter, 1), 1 << 30);
    VC_CUDA(cudaMemcpyAsync(m->kctl, &h, sizeof(KrylovCtl), cudaMemcpyHostToDevice, st));
    KrylovArgs k;
    k.kc = m->kctl;
    k.ctl = m->ctl;
    k.part = m->kr_part;
    k.b = b;
    k.x = x;
    k.r = m->kr;
    k.p = m->kr + S;
    k.v = m->kr + 2 * S;
    k.s = m->kr + 3 * S;
    k.t = m->kr + 4 * S;
    k.e = m->E1;
    k.post = m->post;
    k.n = m->S;
    k.chains = state_grid(m) * kThreads;
    int rc;
    for (;;) {
        ResidentTurn turn;
        if ((rc = krylov_launch(m, pi, k, st, turn))) return rc;
        VC_CUDA(cudaMemcpyAsync(&h, m->kctl, sizeof(KrylovCtl), cudaMemcpyDeviceToHost, st));
        VC_CUDA(cudaStreamSynchronize(st));
        if (h.fault) return fail(VC_ERR_TIMEOUT, "a bounded device-side wait expired");
        if (h.done) break;
        VC_CUDA(cudaMemsetAsync(&m->kctl->arrivals, 0, sizeof(unsigned int), st));
    }
    *products = 2LL * h.iter;
    *converged = (h.done == 1);
    return VC_OK;
}

}  // namespace vc

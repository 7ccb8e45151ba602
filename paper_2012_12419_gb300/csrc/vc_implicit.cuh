// vc_implicit.cuh -- per-item arithmetic of the implicit FP32 sweep (Algorithm 3, step 2,
// with the Eq. 18 backup), shared by the one-sweep kernels and the loop kernel.
//
// An item is VW consecutive state codes x .. x + VW - 1 with x a multiple of VW: VW / 2
// queue lengths q, q + 1, .. of one occupancy vector, each in both channel phases.  All of
// them share the digits, the event probabilities and the targets' offsets, so an item costs
// one decode and one VW-wide load per target.  VW = 4 needs rows of 2(Q + 1) codes to be
// whole items (Q odd; the strides are then multiples of 4, so every target is 16-byte
// aligned when the array is); VW = 2 serves every Q with 8-byte loads.
//
// U (pass-1 values of post-decision states) starts kUShift elements into a 16-byte-aligned
// buffer: a placement's post-decision states s + stride - 2 .. are then aligned for the
// VW-wide load that all H placements make, and only defer's own value straddles.
#pragma once

#include <math.h>

#include "vc_internal.cuh"

namespace vc {

constexpr int kUShift = 2;   // U(0) is element kUShift of its buffer
constexpr int kUPad = 8;     // floats of an U buffer beyond S

// ------------------------------------------------------------------ model arithmetic
// E[V(next) | x] = V(x) + sum_e p_e (V(y_e) - V(x)) from the gathered values (vx = V(x),
// v1 / v0 the completion / departure targets of each host, va the arrival, vf the phase
// flip): the self-loop probability is never formed, so rounding scales with value
// differences, not with |V|.  The sum runs in a fixed order.
template <int MH, typename T>
__device__ __forceinline__ T expect_from(const Model& md, const Coef<T>& c, const Digits& d, T vx, const T* v1,
                                         const T* v0, T va, T vf) {
    T acc = T(0);
#pragma unroll
    for (int k = 0; k < MH; k++) {
        if (k < md.H) {
            const int o = d.occ[k];
            if (o > 0) {
                if (o == 1) {
                    acc += (c.pc[k] + c.pd[k]) * (v1[k] - vx);  // completion and departure both empty the host
                } else {
                    acc += c.pc[k] * T(o) * (v1[k] - vx) + c.pd[k] * (v0[k] - vx);
                }
            }
        }
    }
    if (d.q < md.Q) acc += c.pa * (va - vx);
    acc += (d.ph ? c.pf1 : c.pf0) * (vf - vx);
    return vx + acc;
}

template <int MH, typename T>
__device__ __forceinline__ T expect_next(const Model& md, const Coef<T>& c, const T* V, int x,
                                         const Digits& d) {
    // every gather first (independent loads in flight together), then the sum
    const T vx = V[x];
    T v1[MH], v0[MH];
#pragma unroll
    for (int k = 0; k < MH; k++) {
        const int o = d.occ[k];
        v1[k] = (k < md.H && o > 0) ? V[x - md.stride[k]] : T(0);
        v0[k] = (k < md.H && o > 1) ? V[x - o * md.stride[k]] : T(0);
    }
    const T va = (d.q < md.Q) ? V[x + 2] : T(0);
    const T vf = V[d.ph ? x - 1 : x + 1];
    return expect_from<MH, T>(md, c, d, vx, v1, v0, va, vf);
}

#ifdef VC_DEBUG_BOUNDS
// Every state expect_next reads from post-decision state x lies in [0, S).
template <int MH>
__device__ __forceinline__ bool successors_in_range(const Model& md, int x, const Digits& d, Ctl* ctl) {
    bool ok = x >= 0 && x < md.S && (d.ph ? x - 1 : x + 1) >= 0 && (d.ph ? x - 1 : x + 1) < md.S &&
              (d.q >= md.Q || x + 2 < md.S);
#pragma unroll
    for (int k = 0; k < MH; k++)
        if (k < md.H && d.occ[k] > 0) ok = ok && x - d.occ[k] * md.stride[k] >= 0 && x - md.stride[k] >= 0;
    return VC_IN_BOUNDS(ctl, ok);
}
#endif

// Whether rows of 2(Q + 1) codes are whole items of four (VW = 4 also needs 16-byte-aligned
// value arrays; hosts beyond 8 keep VW = 2, whose gathered values fit the registers).
inline bool wide_rows(const Model& md) { return (md.Q & 1) != 0; }

template <int VW>
__device__ __forceinline__ void ldv(const float* p, float* v) {
    if constexpr (VW == 4) {
        const float4 t = *reinterpret_cast<const float4*>(p);
        v[0] = t.x;
        v[1] = t.y;
        v[2] = t.z;
        v[3] = t.w;
    } else if constexpr (VW == 1) {
        v[0] = *p;
    } else {
        const float2 t = *reinterpret_cast<const float2*>(p);
        v[0] = t.x;
        v[1] = t.y;
    }
}

template <int VW>
__device__ __forceinline__ void stv(float* p, const float* v) {
    if constexpr (VW == 4)
        *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]);
    else if constexpr (VW == 1)
        *p = v[0];
    else
        *reinterpret_cast<float2*>(p) = make_float2(v[0], v[1]);
}

// by_h instantiates MH = H for H <= 8, so the per-host bound is a constant there.
template <int MH>
__device__ __forceinline__ bool has_host(const Model& md, int k) {
    return MH <= 8 || k < md.H;
}

// Pass 1 of one item: U(x) = R(x) + gamma E[V(next) | x] of its VW states and, with SL,
// defer's value with its self-transition solved; EXPECT: E[V(next) | x] alone, into U.  Each
// state's arithmetic is expect_from's (and, for W, post_and_defer's) in the same order.
template <int MH, int VW, bool SL, bool EXPECT = false>
__device__ __forceinline__ void post_item(const Model& md, const Coef<float>& c, const float* V, int x, float* U,
                                          float* W, Ctl* ctl) {
    Digits d;
    decode<MH>(md, x, d);
#ifdef VC_DEBUG_BOUNDS
    {
        bool ok = x >= 0 && x + VW <= md.S && (d.q + VW / 2 > md.Q || x + VW + 2 <= md.S);
#pragma unroll
        for (int k = 0; k < MH; k++)
            if (has_host<MH>(md, k) && d.occ[k] > 0) ok = ok && x - d.occ[k] * md.stride[k] >= 0;
        if (!VC_IN_BOUNDS(ctl, ok)) return;
    }
#endif
    float vx[VW], v1[MH][VW], v0[MH][VW], vn[2] = {0.0f, 0.0f};
    ldv<VW>(V + x, vx);
#pragma unroll
    for (int k = 0; k < MH; k++) {
        const int o = d.occ[k];
#pragma unroll
        for (int j = 0; j < VW; j++) v1[k][j] = v0[k][j] = 0.0f;
        if (has_host<MH>(md, k) && o > 0) ldv<VW>(V + (x - md.stride[k]), v1[k]);
        if (has_host<MH>(md, k) && o > 1) ldv<VW>(V + (x - o * md.stride[k]), v0[k]);
    }
    if (d.q + VW / 2 <= md.Q) ldv<2>(V + (x + VW), vn);
    float acc[VW], sm[VW], pm[VW / 2], loss = 0.0f;
    int occ_sum = 0;
#pragma unroll
    for (int j = 0; j < VW; j++) acc[j] = sm[j] = 0.0f;
#pragma unroll
    for (int i = 0; i < VW / 2; i++) pm[i] = 0.0f;
#pragma unroll
    for (int k = 0; k < MH; k++) {
        if (!has_host<MH>(md, k)) continue;
        const int o = d.occ[k];
        occ_sum += o;
        loss += c.lossd[k] * float(o);
        if (o == 1) {
            const float p = c.pc[k] + c.pd[k];  // completion and departure both empty the host
#pragma unroll
            for (int j = 0; j < VW; j++) {
                acc[j] += p * (v1[k][j] - vx[j]);
                if constexpr (SL) sm[j] = fmaf(p, v1[k][j], sm[j]);
            }
#pragma unroll
            for (int i = 0; i < VW / 2; i++) pm[i] += p;
        } else if (o > 1) {
            const float p1 = c.pc[k] * float(o);
#pragma unroll
            for (int j = 0; j < VW; j++) {
                acc[j] += p1 * (v1[k][j] - vx[j]) + c.pd[k] * (v0[k][j] - vx[j]);
                if constexpr (SL) {
                    sm[j] = fmaf(p1, v1[k][j], sm[j]);
                    sm[j] = fmaf(c.pd[k], v0[k][j], sm[j]);
                }
            }
#pragma unroll
            for (int i = 0; i < VW / 2; i++) {
                pm[i] += p1;
                pm[i] += c.pd[k];
            }
        }
    }
    float u[VW], w[VW];
#pragma unroll
    for (int i = 0; i < VW / 2; i++) {
        const int q = d.q + i;
        const bool room = q < md.Q;
        float lq = loss;
        if (!room) lq += c.lossa;
        const float rx = c.w_occ * float(occ_sum) + c.w_q * float(q) + lq;  // the phase does not enter it
#pragma unroll
        for (int ph = 0; ph < 2; ph++) {
            const int j = 2 * i + ph;
            const float va = i + 1 < VW / 2 ? vx[(j + 2) % VW] : vn[ph];
            const float vf = vx[2 * i + (ph ^ 1)];  // the phase flip lands on the other state of the pair
            const float pf = ph ? c.pf1 : c.pf0;
            float a = acc[j];
            if (room) a += c.pa * (va - vx[j]);
            a += pf * (vf - vx[j]);
            const float e = vx[j] + a;
            u[j] = EXPECT ? e : rx + c.gamma * e;
            if constexpr (SL) {
                float s = sm[j], p = pm[i];
                if (room) {
                    s = fmaf(c.pa, va, s);
                    p += c.pa;
                }
                s = fmaf(pf, vf, s);
                p += pf;
                w[j] = __fdiv_rn(fmaf(c.gamma, s, rx), fmaf(c.gamma, p, 1.0f - c.gamma));
            }
        }
        if constexpr (!EXPECT) stv<2>(U + (x + 2 * i), u + 2 * i);
    }
    if constexpr (EXPECT) stv<VW>(U + x, u);
    if constexpr (SL) stv<VW>(W + x, w);
}

// Pass 2 of one item: best[j], second[j], arg[j] over the feasible actions in order (lowest
// index on ties).  Phase 1 may place on every host with a free slot, phase 0 on the RSU (host
// H - 1) only, both with a task waiting.
template <int MH, int VW, bool SL, bool ARG>
__device__ __forceinline__ void max_item(const Model& md, const float* U, const float* W, int s, float* best,
                                         float* second, int* arg, Ctl* ctl) {
    Digits d;
    decode<MH>(md, s, d);
    float uk[MH][VW], ud[VW];
#pragma unroll
    for (int k = 0; k < MH; k++) {
        const bool f = has_host<MH>(md, k) && d.occ[k] < md.C && d.q + VW / 2 > 1 &&
                       VC_IN_BOUNDS(ctl, s + md.stride[k] - 2 >= 0 && s + md.stride[k] + VW - 2 <= md.S);
#pragma unroll
        for (int j = 0; j < VW; j++) uk[k][j] = -INFINITY;
        if (f) {
            ldv<VW>(U + (s + md.stride[k] - 2), uk[k]);
            if (VW == 4 && d.q < 1) uk[k][0] = uk[k][1] = -INFINITY;  // no task waits at q = 0
        }
    }
    if constexpr (SL) {
        ldv<VW>(W + s, ud);
    } else {
#pragma unroll
        for (int i = 0; i < VW / 2; i++) ldv<2>(U + (s + 2 * i), ud + 2 * i);
    }
    const int last = MH <= 8 ? MH - 1 : md.H - 1;
#pragma unroll
    for (int j = 0; j < VW; j++) {
        float b = -INFINITY, b2 = -INFINITY;
        int a = last + 1;
#pragma unroll
        for (int k = 0; k < MH; k++) {
            if ((j & 1) == 0 && k != last) continue;  // phase 0
            const float v = uk[k][j];
            if (v > b) {
                b2 = b;
                b = v;
                a = k;
            } else if (ARG && v > b2) {
                b2 = v;
            }
        }
        if (ud[j] > b) {
            b2 = b;
            b = ud[j];
            a = last + 1;
        } else if (ARG && ud[j] > b2) {
            b2 = ud[j];
        }
        best[j] = b;
        if constexpr (ARG) {
            second[j] = b2;
            arg[j] = a;
        }
    }
}

}  // namespace vc

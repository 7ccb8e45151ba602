// vc_csr_loop.cu -- the FP32 value-iteration loop over a stored matrix (Algorithm 3, steps 1-3,
// Eq. 18 backup over the stored rows), in one resident kernel.
//
// A sweep over a matrix that stays in L2 takes 5-30 us, so launched one by one the sweeps of
// k_csr_tma pay as much for the launch, for filling a pipeline that a CTA uses for one to ten
// tiles, and for the CTA-wide hand-over of every tile.  Here one CTA per SM stays for the whole
// loop and every warp works alone: it owns chunks of 32 / A states (a row per lane), stages a
// chunk's columns and values with two bulk copies into its own double buffer while it sums the
// previous chunk, and runs on into the next sweep's first chunk before the grid barrier, since
// only V changes.  Rows are summed and compared as in k_csr_tma (fused multiply-adds in column
// order, the same tree of maxima), so both give the same iterates bit for bit.  CTAs own
// contiguous states of about equal numbers of entries.  Entry indices are 32-bit.
//
// Bound: the gathers of V.  Each distinct line of a warp's gather is an L1 lookup, and what
// misses L1 (V is larger) is an L2 sector; then issue (~350 instructions a chunk).  Per sweep,
// launched against resident: 640 states 10.5 -> 3.3 us, 12,500 states 13.0 -> 3.6 us, 100,000
// states padded (66 MiB) 31.3 -> 13.3 us, 200,003 states of random columns (61 MiB) 41.8 ->
// 29.5 us; beyond the L2, 2.5 M states (1.2 GiB) 520 -> 418 us, padded (2.8 GiB) 655 -> 597 us.
#include <algorithm>
#include <type_traits>

#include "vc_grid.cuh"
#include "vc_internal.cuh"
#include "vc_ptx.cuh"

namespace vc {

constexpr int kCsrLoopWarps = 24;             // most warps of a CTA
// Staging of a CTA; the rest of an SM's 228 KB is L1 for V.  100,000 states padded / 200,003
// random: 96 KB 14.7 / 27.9 us, 128 KB 13.4 / 29.4, 190 KB 13.3 / 29.4; 16 warps 14.6 / 29.7.
constexpr int kCsrLoopSmem = 128 * 1024;
constexpr int kCsrChunkCost = 128;            // a chunk's fixed work, in entries (CTA balance)

struct CsrLoopArgs {
    int S, A, cap;   // cap: most entries of a chunk
    float gamma;
    const int64_t* row_ptr;
    const int32_t* col;
    const void* val;
    const float* scale;
    const float* R;
};

// Staged bytes of a chunk: its entries from a 16-byte boundary, and kCsrSlots - 1 entries that
// the last row's slots may read beyond it.
constexpr int kCsrSlots = 16;
__host__ __device__ inline int loop_col_bytes(int cap) { return 4 * ((cap + 3 + kCsrSlots + 3) & ~3); }
template <typename VT>
__host__ __device__ inline int loop_val_bytes(int cap) {
    constexpr int kv = 16 / (int)sizeof(VT);
    return (int)sizeof(VT) * ((cap + kv - 1 + kCsrSlots + kv - 1) / kv * kv);
}

template <typename VT>
__device__ __forceinline__ float stored_value(const VT* p) {
    if constexpr (sizeof(VT) == 4) return *p;
    else return __uint_as_float((uint32_t)*p << 16);
}

// Row sum in column order (SL: without the row's own state, whose probability goes to pss).
// The slots beyond a row read what follows it in the staging buffer; only the gather and the
// multiply-add are predicated.
// Groups of four slots beyond the warp's longest row (nmax) are skipped, and up to 16
// gathers of a row are in flight before the first multiply-add.
template <typename VT, bool SL>
__device__ __forceinline__ float chunk_row_dot(const int32_t* cols, const VT* vals, int first, int n, int nmax,
                                               const float* V, int self, float& pss) {
    float acc = 0.0f;
    for (int j0 = 0; j0 < nmax; j0 += kCsrSlots, first += kCsrSlots, n -= kCsrSlots) {
        const int at = n > 0 ? first : 0;  // a finished row reads the buffer's start
        const int32_t* cp = cols + at;
        const VT* vp = vals + at;
        float g[kCsrSlots];
        uint32_t own = 0;
#pragma unroll
        for (int q = 0; q < kCsrSlots / 4; q++) {
            if (j0 + 4 * q < nmax) {
#pragma unroll
                for (int u = 4 * q; u < 4 * q + 4; u++) {
                    const int c = cp[u];
                    if (u < n) g[u] = V[c];
                    if (SL) own |= (c == self ? 1u : 0u) << u;
                }
            }
        }
#pragma unroll
        for (int q = 0; q < kCsrSlots / 4; q++) {
            if (j0 + 4 * q < nmax) {
#pragma unroll
                for (int u = 4 * q; u < 4 * q + 4; u++) {
                    const float w = stored_value<VT>(vp + u);
                    if (u < n) {
                        if (SL) {
                            const bool o = (own >> u) & 1u;
                            pss += o ? w : 0.0f;
                            acc = fmaf(w, o ? 0.0f : g[u], acc);
                        } else {
                            acc = fmaf(w, g[u], acc);
                        }
                    }
                }
            }
        }
    }
    return acc;
}

// Low word of row_ptr[r] (little-endian; every entry index of a served matrix fits 31 bits).
__device__ __forceinline__ int row_start(const int64_t* row_ptr, int64_t r) {
    return __ldg(reinterpret_cast<const int*>(row_ptr + r));
}

// APAD: the least power of two >= A (the depth of the tree of maxima).
template <typename VT, int APAD, bool SL>
__global__ void __launch_bounds__(kCsrLoopWarps * 32, 1) k_csr_loop(CsrLoopArgs a, float* buf0, float* buf1, Ctl* ctl) {
    extern __shared__ __align__(128) unsigned char csr_sm[];
    __shared__ unsigned int sh_max[2][2];  // residual and max|V'| of the sweep, by parity
    __shared__ float sh_rv[2];
    __shared__ long long sh_end, sh_start;
    __shared__ int sh_fail, sh_cut[2];
    __shared__ uint64_t sh_full[kCsrLoopWarps][2];  // staged chunks of each warp's two buffers
    const int warp = (int)threadIdx.x >> 5, lane = (int)threadIdx.x & 31, nw = (int)blockDim.x >> 5;
    const int A = a.A, spw = 32 / A, crows = spw * A;  // states and rows of a chunk
    const int grp = lane / A, act = lane - grp * A;    // lanes past the chunk's rows: grp == spw
    const bool lead = threadIdx.x == 0;
    const int chunks = (a.S + spw - 1) / spw;
    const int64_t rows = (int64_t)a.S * A;
    const VT* val = reinterpret_cast<const VT*>(a.val);
    if (threadIdx.x < 2) {
        // first chunk of CTA blockIdx.x (+ 1): the smallest c whose preceding work reaches its share
        const int b = (int)(blockIdx.x + threadIdx.x);
        const int64_t total = row_start(a.row_ptr, rows) + (int64_t)kCsrChunkCost * chunks;
        const int64_t want = (int64_t)((double)total / gridDim.x * b);
        int lo = 0, hi = chunks;
        if (b == (int)gridDim.x) lo = chunks;
        while (lo < hi) {
            const int mid = (lo + hi) >> 1;
            if (row_start(a.row_ptr, (int64_t)mid * crows) + (int64_t)kCsrChunkCost * mid < want) lo = mid + 1;
            else hi = mid;
        }
        sh_cut[threadIdx.x] = lo;
    }
    if (lead) {
        sh_max[0][0] = sh_max[0][1] = sh_max[1][0] = sh_max[1][1] = 0u;
        sh_fail = 0;
    }
    if (lane < 2) mbar_init(&sh_full[warp][lane], 1);
    if (lane == 0) fence_mbar_init();
    __syncthreads();
    const int cw = sh_cut[0] + warp, c1 = sh_cut[1];
    const bool any = cw < c1;
    const int col_bytes = loop_col_bytes(a.cap), buf_bytes = col_bytes + loop_val_bytes<VT>(a.cap);
    unsigned char* mine = csr_sm + (size_t)warp * 2 * buf_bytes;
    for (int i = 16 * lane; i < 2 * buf_bytes; i += 512) *reinterpret_cast<int4*>(mine + i) = make_int4(0, 0, 0, 0);
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    __syncwarp();

    // A lane's row of a chunk (infeasible and absent rows: n = 0 and R = -inf), and the entries
    // [e0, e1) of the chunk.
    struct Meta {
        int lo, hi, e0, e1;
        float rr, scale;
    };
    auto load_meta = [&](int c, Meta& m) {
        const int64_t r = (int64_t)c * crows + lane;
        const bool live = grp < spw && r < rows;
        m.lo = row_start(a.row_ptr, r < rows ? r : rows);
        m.hi = row_start(a.row_ptr, r < rows ? r + 1 : rows);
        m.rr = live ? __ldg(a.R + r) : -INFINITY;
        m.scale = live && a.scale ? __ldg(a.scale + r) : 1.0f;
    };
    bool gave = false;  // this lane gave up waiting for a chunk
    uint32_t owed = 0;  // phase at that point, when both buffers' copies were in flight
    auto stage = [&](Meta& m, int b) {
        // lanes past the chunk's rows hold rows of the next one
        m.e0 = __shfl_sync(0xffffffffu, m.lo, 0);
        m.e1 = __shfl_sync(0xffffffffu, m.hi, crows - 1);
        if (lane != 0 || gave) return;
        constexpr int kv = 16 / (int)sizeof(VT);
        const int q0 = m.e0 & ~3, p0 = m.e0 & ~(kv - 1);
        uint32_t bc = 4u * (uint32_t)(((m.e1 + 3) & ~3) - q0), bv = (uint32_t)sizeof(VT) * (uint32_t)(((m.e1 + kv - 1) & ~(kv - 1)) - p0);
        if (m.e1 <= m.e0 || !VC_IN_BOUNDS(ctl, m.e1 - m.e0 <= a.cap)) bc = bv = 0;
        unsigned char* dst = mine + b * buf_bytes;
        mbar_arrive_expect_tx(&sh_full[warp][b], bc + bv);
        if (bc) {
            bulk_g2s(dst, a.col + q0, bc, &sh_full[warp][b]);
            bulk_g2s(dst + col_bytes, val + p0, bv, &sh_full[warp][b]);
        }
    };

    long long k = ctl->sweeps;
    const bool first_cta = lead && blockIdx.x == 0;
    LaunchEnd end{&ctl->launch_end, &sh_start};
    if (first_cta) end.open(k);
    LoopVerdict verdict{ctl->tol, __double2float_ru(ctl->tol), ctl->best_res, ctl->since_best, ctl->max_sweeps};
    GridBarrier bar{&ctl->arrivals, gridDim.x, 0u, &sh_fail, barrier_polls(ctl->spin_limit)};
    const int lim = (int)barrier_polls(ctl->spin_limit);
    Meta cur, nxt;
    int b = 0, done = 0;
    uint32_t phase = 0;  // parity of each buffer's next chunk (bits 0, 1)
    if (any) {
        load_meta(cw, cur);
        stage(cur, 0);
        load_meta(cw + nw < c1 ? cw + nw : cw, nxt);
    }
    while (true) {
        const int in = (int)(k & 1);
        const float* Vi = in ? buf1 : buf0;
        float* Vo = in ? buf0 : buf1;
        float res = 0.0f, vabs = 0.0f;
        if (first_cta) end.check(k);
        for (int c = cw; c < c1; c += nw) {
            const int c_next = c + nw < c1 ? c + nw : cw;
            stage(nxt, b ^ 1);
            Meta after;
            load_meta(c_next + nw < c1 ? c_next + nw : cw, after);
            // A lane that gives up waits no more and goes on with what the buffers hold (columns of an
            // earlier chunk; the result is refused), and lane 0 then stages no more, so no buffer
            // is filled while an earlier copy into it is in flight.  The loop is not left here: an
            // exit inside it cost 3 to 5 % of a sweep.
            if (!gave && !mbar_wait(&sh_full[warp][b], (phase >> b) & 1u, lim)) {
                gave = true;
                owed = phase;
                atomicExch(&sh_fail, 1);
            }
            phase ^= 1u << b;
            const unsigned char* src = mine + b * buf_bytes;
            const int32_t* cs = reinterpret_cast<const int32_t*>(src) + (cur.e0 & 3);
            const VT* vs = reinterpret_cast<const VT*>(src + col_bytes) + (cur.e0 & (16 / (int)sizeof(VT) - 1));
            const int first = cur.lo - cur.e0;
            const int s = c * spw + grp;
            const bool owner = act == 0 && grp < spw && s < a.S;
            const float vin = owner ? Vi[s] : 0.0f;
            int n = cur.rr == -INFINITY ? 0 : cur.hi - cur.lo;
#ifdef VC_DEBUG_BOUNDS
            if (!VC_IN_BOUNDS(ctl, n >= 0 && (n == 0 || (cur.lo >= cur.e0 && cur.lo + n <= cur.e1)))) n = 0;
            for (int j = 0; j < n; ++j)
                if (!VC_IN_BOUNDS(ctl, cs[first + j] >= 0 && cs[first + j] < a.S)) n = 0;
#endif
            const int nmax = __reduce_max_sync(0xffffffffu, n);
            float pss = 0.0f;
            const float acc = chunk_row_dot<VT, SL>(cs, vs, first, n, nmax, Vi, s, pss);
            float q = -INFINITY;
            if (cur.rr != -INFINITY) {
                if (SL)
                    q = q_self_loop(cur.rr, a.gamma, a.scale ? cur.scale * acc : acc, a.scale ? cur.scale * pss : pss);
                else
                    q = cur.rr + a.gamma * (a.scale ? cur.scale * acc : acc);
            }
#pragma unroll
            for (int o = 1; o < APAD; o <<= 1) {
                const int oa = act ^ o;  // the tree over APAD lanes, absent ones -inf
                const float oq = __shfl_sync(0xffffffffu, q, oa < A ? grp * A + oa : lane);
                q = oa < A && oq > q ? oq : q;
            }
            if (owner) {
                Vo[s] = q;
                res = fmaxf(res, fabsf(q - vin));
                vabs = fmaxf(vabs, fabsf(q));
            }
            __syncwarp();  // the buffer just read is staged again in the next step
            cur = nxt;
            nxt = after;
            b ^= 1;
        }
        // non-negative floats order like their bits
        const unsigned int rb = __reduce_max_sync(0xffffffffu, fbits(res));
        const unsigned int vb = __reduce_max_sync(0xffffffffu, fbits(vabs));
        if (lane == 0) {
            atomicMax(&sh_max[in][0], rb);
            atomicMax(&sh_max[in][1], vb);
        }
        __syncthreads();
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
            if (first_cta) {
                // the slot after the next sweep's: read 62 sweeps ago, written after the next barrier
                ctl->res32[(k + 2) % kRing] = 0u;
                ctl->vmax32[(k + 2) % kRing] = 0u;
            }
        }
        if (threadIdx.x == blockDim.x - 1) sh_end = end.read();  // beside the lead's two reads
        __syncthreads();
        k++;
        done = verdict(sh_rv[0], sh_rv[1], k);
        if (done || k >= sh_end) break;
    }
    // no copy outlives the CTA: the chunk staged ahead, or both buffers' where lane 0 gave up
    if (any && lane == 0) {
        if (gave) {
            mbar_wait(&sh_full[warp][0], owed & 1u);
            mbar_wait(&sh_full[warp][1], (owed >> 1) & 1u);
        } else {
            mbar_wait(&sh_full[warp][b], (phase >> b) & 1u);
        }
    }
    if (lead && sh_fail) atomicOr(&ctl->error, kErrTimeout);
    if (first_cta) {
        ctl->sweeps = k;
        ctl->final_buf = (int)(k & 1);
        ctl->best_res = verdict.best;
        ctl->since_best = verdict.since;
        ctl->done = sh_fail ? 4 : done;
        ctl->res32[k % kRing] = ctl->vmax32[k % kRing] = 0u;  // a resumed loop's first two slots
        ctl->res32[(k + 1) % kRing] = ctl->vmax32[(k + 1) % kRing] = 0u;
    }
}

template <typename VT, int APAD>
static int csr_loop_run(Mdp* m, float* buf0, float* buf1, int self_loop, cudaStream_t st, ResidentTurn& turn,
                        bool* launched) {
    const int warp_bytes = 2 * (loop_col_bytes((int)m->loop_cap) + loop_val_bytes<VT>((int)m->loop_cap));
    const int warps = std::min(kCsrLoopWarps, kCsrLoopSmem / warp_bytes);
    if (warps < 12) return VC_OK;  // rows too long for a warp's own staging
    const int chunks = (m->S + 32 / m->A - 1) / (32 / m->A);
    const int sms = m->num_sms > 0 ? m->num_sms : 148;
    const int grid = std::min(sms, (chunks + 3) / 4);
    const CsrLoopArgs a{m->S, m->A, (int)m->loop_cap, (float)m->gamma, m->row_ptr, m->col, m->val, m->scale, m->R};
    const void* fn = self_loop ? (const void*)k_csr_loop<VT, APAD, true> : (const void*)k_csr_loop<VT, APAD, false>;
    VC_CUDA(cached_set_max_dyn_smem(fn, kCsrLoopSmem));
    return launch_resident(fn, grid, 32 * warps, (size_t)warps * warp_bytes, st, turn, sms, launched, a, buf0, buf1, m->ctl);
}

int launch_csr_loop(Mdp* m, float* buf0, float* buf1, int self_loop, cudaStream_t st, ResidentTurn& turn,
                    bool* launched) {
    *launched = false;
    const bool bf16 = (m->fmt & 0xF) == VC_CSR_BF16;
    // what the autotuner found, else every pipelined CSR schedule (the loop is the faster one at
    // each size and type measured), if the entries are counted in 31 bits; a handle whose waits were capped keeps the launched
    // sweeps (but for the bounds-checking build, where the cap reaches this loop's waits)
#ifdef VC_DEBUG_BOUNDS
    const bool capped = false;
#else
    const bool capped = m->spin_polls >= 0;
#endif
    if (m->loop_choice == 0 || (m->loop_choice < 0 && (!m->plan.tma || m->plan.sliced))) return VC_OK;
    if (m->loop_cap <= 0 || capped || m->nnz_stored >= (1LL << 31) - 64) return VC_OK;
    auto go = [&](auto apad) {
        constexpr int AP = decltype(apad)::value;
        return bf16 ? csr_loop_run<uint16_t, AP>(m, buf0, buf1, self_loop, st, turn, launched)
                    : csr_loop_run<float, AP>(m, buf0, buf1, self_loop, st, turn, launched);
    };
    switch (pow2_at_least(m->A)) {
        case 1: return go(std::integral_constant<int, 1>());
        case 2: return go(std::integral_constant<int, 2>());
        case 4: return go(std::integral_constant<int, 4>());
        case 8: return go(std::integral_constant<int, 8>());
        case 16: return go(std::integral_constant<int, 16>());
        default: return go(std::integral_constant<int, 32>());
    }
}

}  // namespace vc

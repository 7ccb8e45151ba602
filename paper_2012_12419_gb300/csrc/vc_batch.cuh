// vc_batch.cuh -- device-side descriptors of the batched solves, shared by the tile kernels
// (vc_batch.cu) and the resident loop (vc_batch_loop.cu).
#pragma once

#include "vc_internal.cuh"

namespace vc {

struct InstDesc {
    Model md;
    Coef<float> c32;
    Coef<double> c64;
    long long off;   // first state in the handle's concatenated arrays (a multiple of 64)
    long long eoff;  // first state in the caller's packed arrays
    int S;
    int blk_h;      // inner hosts of the in-block iteration's blocks (2(Q+1)(C+1)^blk_h states)
};

struct BatchTile {
    int inst;
    int start;  // first state, relative to the instance
    int count;
    int pad_;
};

// Device-side control of the batched loops (SoA over instances).
struct BatchCtl {
    int* done;                 // 0 running, 1 converged, 2 max sweeps, 3 FP32 stall
    int* sweeps;
    int* ticket;
    const int* tiles_of;       // tiles per instance (constant)
    int* final_buf;            // buffer of the last iterate (0: A, 1: B)
    int* since_best;
    float* best_res;
    unsigned int* res32;       // [2n] ring of two slots
    unsigned int* vmax32;      // [2n]
    unsigned long long* res64; // [n] FP64 residual of a certificate / residual pass
    int* active;               // instances still running
    long long* iters;          // sweeps launched by the graph loop
    const long long* max_sweeps; // loop parameters in device memory, so one captured graph
    const double* tol;           // serves every call
    const float* tol_scale;      // per-instance factor on tol (nullptr: 1)
};

// The FP32 loop of every active instance in one resident kernel (vc_batch_loop.cu), from sweep
// `first` on until all have ended, only instances of at most hand_over states are left or the
// launch's time is up (LaunchEnd); the sweeps then done are at *end.  *launched = false when it does not serve
// the batch (hosts, instances) or the device cannot hold the grid.
constexpr int kBatchLoopMaxH = 5;     // above, an item and its coefficients no longer fit 128 registers
constexpr int kBatchLoopMaxN = 4096;  // instances whose shares and verdicts fit shared memory
constexpr int kLoopTimeout = 1, kLoopHandOver = 2;
struct BatchLoopArgs {
    const InstDesc* descs;
    int n;
    BatchCtl c;
    float *V0, *V1, *U, *U2;  // U: kUShift past a 16-byte-aligned buffer
    unsigned int* arrivals;   // grid barrier, cleared by the host before each launch
    int* fault;               // kLoopTimeout: a barrier wait gave up; kLoopHandOver: small ones are left
    int hand_over;
    unsigned int polls;       // poll limit of a barrier wait
    Ctl* ctl;                 // error flags of the bounds-checking build
    long long first;          // sweeps done so far
    long long* end;           // LaunchEnd's word
};
int launch_batch_loop(const BatchLoopArgs& a, int max_hosts, int num_sms, bool self_loop, cudaStream_t st,
                      ResidentTurn& turn, bool* launched);

}  // namespace vc

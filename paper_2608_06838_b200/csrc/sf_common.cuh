// Shared kernel-parameter structs and small device helpers.
//
// Vocabulary (paper Section 3.1, last paragraph): a SEGMENT is the paper's sequence chunk C_i, a
// CHUNK its kernel-level chunk of T_C tokens.  A BLOCK is this library's own middle granularity:
// R consecutive chunks; only block-boundary states ever reach global memory.
#pragma once
#include <cuda_runtime.h>
#include <cuda_bf16.h>
#include <stdint.h>

namespace sf {

struct SegParams {
    int B, H;
    int L;        // tokens in the segment
    int C;        // chunk size T_C
    int NC;       // chunks in the segment
    int R;        // chunks per block
    int NB;       // blocks in the segment
    long long tqk, tv, tg;   // token strides (elements)
    long long bqk, bv, bg;   // batch strides (elements)
    // Boundary states of a chain whose segments run as one (merged launches): bslot[c] >= 0 marks chunk c as the first
    // chunk of segment bslot[c]; the forward sweep then stores the state entering that chunk to bbase + bslot[c]*bstride
    // (one [B,H,d_k,d_v] array per segment).  NULL outside that mode.
    const int* bslot;
    float* bbase;
    long long bstride;
    // A segment of one block needs no aggregate and no scan: with `single` set the sweeps start from s_init [B,H,d_k,d_v] (NULL:
    // zero) instead of the workspace's block states, and store the state (gradient) that leaves the block to s_final and, if
    // given, the one that entered it to s_copy.
    int single;
    const float* s_init;
    float *s_final, *s_copy;
    int wait_first;          // the first kernel of a call: grid_wait() before any access to global memory
};

// Programmatic dependent launch.  A kernel launched with launch_after() may start while the kernel before it in the stream
// still runs, once every CTA of that one has called grid_launch_next(); what it does before grid_wait() may only touch its own
// on-chip state, the caller's inputs and, past L1, SegParams::bslot, whose writer (mark_bounds_kernel) has completed before any
// of these can start: the kernel behind it, the merged chain's aggregate, is launched without the early start.  grid_wait() returns when the kernel before has completed and its writes are visible;
// every CTA calls it, so completion carries over a sequence of such launches.  What a kernel of the same call wrote is read
// through pointers without __restrict__: the data changes while this kernel is resident, so its loads must not count as
// read-only ones, which may be moved ahead of the wait.
// The caller's inputs may have been written by whatever stands before the call in the stream, another call of this library
// included, and that work may signal early too.  So the first kernel of a call (SegParams::wait_first) waits before it touches
// global memory at all (only its barriers and tensor memory are set up early) and signals after that wait: no later
// kernel of the call can be resident before everything ahead of the call has completed, however many of the kernels between signal
// before their own wait.  A CTA also signals only once it holds its tensor memory: a successor that took the columns first would
// keep them while it waits for this kernel.
__device__ __forceinline__ void grid_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void grid_launch_next() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

template <typename... P, typename... A>
inline bool launch_after(bool early, void (*kern)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, A... args) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid; cfg.blockDim = block; cfg.dynamicSmemBytes = smem; cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = early ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kern, P(args)...) == cudaSuccess;
}

// Error codes written to the device status word by kernels whose bounded waits run out.
enum : int { DEV_OK = 0, DEV_TIMEOUT_TMA = 1, DEV_TIMEOUT_MMA = 2, DEV_TIMEOUT_SELFTEST = 3 };

// A log-decay as the tables of the float32-precision kernels take it.  Everything below -1e4 wipes the state all the same, and limited to
// it, sums over a tile stay exact to 1e-10 in double precision also beside a mask value (-inf, the lowest float): differences of
// the sums, taken for tokens behind it, are right.  NaN stays NaN.
__device__ __forceinline__ double log_decay(float g) { return g < -1e4f ? -1e4 : (double)g; }
// The same for the float32 tables of the tensor-core kernels (bf16): below -128 a decay wipes the state in float32 all the same, and 64
// limited ones in a chunk leave the differences of its sums an error of 5e-4, an eighth of a bf16 rounding.
__device__ __forceinline__ float log_decay_bf16(float g) { return g < -128.f ? -128.f : g; }

__device__ __forceinline__ float to_f32(float x) { return x; }
__device__ __forceinline__ float to_f32(__nv_bfloat16 x) { return __bfloat162float(x); }
template <typename T> __device__ __forceinline__ T from_f32(float x);
template <> __device__ __forceinline__ float from_f32<float>(float x) { return x; }
template <> __device__ __forceinline__ __nv_bfloat16 from_f32<__nv_bfloat16>(float x) { return __float2bfloat16_rn(x); }

}  // namespace sf

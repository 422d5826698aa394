// tcgen05 / TMEM / TMA kernels for the bf16, d_k = d_v = 128, chunk = 64 shape.
//
// Thread roles in every kernel here: the first warps compute (TMEM loads/stores, decay masks, epilogues;
// warp w owns TMEM lanes 32(w mod 4)..+31), then one TMA producer warp and one warp that
// issues the MMAs (lane 0 each).  All waits are bounded (see ptx::mbar_wait).
//
// Shared-memory operand storage: every bf16 tile of 64 (aggregates) or 128 (sweeps) tokens x 128 features is two TMA boxes of
// [tokens x 64 columns] (128-byte rows, SWIZZLE_128B, features 0-63 then 64-127).  The
// same storage is read K-major when the contraction runs over features and MN-major when it runs
// over tokens (ptx::desc_lo).
#pragma once
#include <cuda.h>
#include <memory>
#include <new>

#include "../../include/stateflow.h"
#include "sf_common.cuh"
#include "sf_map_cache.h"
#include "sf_ptx.cuh"

namespace sf {
namespace tc {

using ptx::g_dev_status;

inline int read_device_status() {
    int v = 0;
    if (cudaMemcpyFromSymbol(&v, g_dev_status, sizeof(int)) != cudaSuccess) { cudaGetLastError(); return -1; }
    return v;
}
inline void clear_device_status() {
    int v = 0;
    if (cudaMemcpyToSymbol(g_dev_status, &v, sizeof(int)) != cudaSuccess) cudaGetLastError();
}

constexpr int C = 64;              // chunk
constexpr int D = 128;             // d_k = d_v
constexpr int BOX = 8192;          // bytes of one [64 x 64] bf16 box
constexpr int TILE = 2 * BOX;      // bytes of one [64 x 128] bf16 tile
constexpr int MAXR = 64;           // largest chunks_per_block of the tensor-core path
constexpr float LOG2E = 1.4426950408889634f;

__device__ __forceinline__ float fast_exp(float x) { return ptx::ex2(x * LOG2E); }

// ---- host: tensor maps ---------------------------------------------------------------------------
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                                  const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

// Looked up once; a thread that comes meanwhile waits for the result.
inline EncodeTiledFn encode_fn() {
    static const EncodeTiledFn fn = []() -> EncodeTiledFn {
        void* sym = nullptr;
        cudaDriverEntryPointQueryResult qres;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &sym, cudaEnableDefault, &qres) == cudaSuccess && qres == cudaDriverEntryPointSuccess)
            return reinterpret_cast<EncodeTiledFn>(sym);
        cudaGetLastError();
        return nullptr;
    }();
    return fn;
}

// Map of a [B, L, H, 128] bf16 view: dims (feature, head, token, batch), box = 64 features x 1 x `rows` tokens x 1.
// A map is a pure function of (base, rows, B, L, H, strides) and encoding one never reads device memory, so each host
// thread keeps the maps it encoded (up to MapCache::MAX_USED): a chain that is launched again from the host (no graph) with the
// same buffers re-encodes nothing.  A segment's forward and backward take 12 (k, v, q, dO in boxes of 64 tokens for the aggregates and of 128
// for the sweeps, o, dq, dk, dv in boxes of 64), so chains of up to 32 separately launched segments fit.
struct TmapKey {
    const void* base; int rows, B, L, H; long long tok_stride, batch_stride;
    bool operator==(const TmapKey& o) const {
        return base == o.base && rows == o.rows && B == o.B && L == o.L && H == o.H && tok_stride == o.tok_stride && batch_stride == o.batch_stride;
    }
    uint64_t hash() const {
        uint64_t h = reinterpret_cast<uintptr_t>(base) >> 4;
        for (uint64_t x : {(uint64_t)rows, (uint64_t)B, (uint64_t)L, (uint64_t)H, (uint64_t)tok_stride, (uint64_t)batch_stride}) h = h * 0x100000001B3ull + x;
        return h;
    }
};
using TmapCache = MapCache<TmapKey, CUtensorMap, 512>;

inline bool make_tmap(CUtensorMap* m, int rows, const void* base, int B, int L, int H, long long tok_stride, long long batch_stride) {
    thread_local std::unique_ptr<TmapCache> cache(new (std::nothrow) TmapCache);
    const TmapKey key{base, rows, B, L, H, tok_stride, batch_stride};
    if (const CUtensorMap* kept = cache ? cache->find(key) : nullptr) { *m = *kept; return true; }
    EncodeTiledFn fn = encode_fn();
    if (!fn) return false;
    cuuint64_t dims[4] = {(cuuint64_t)D, (cuuint64_t)H, (cuuint64_t)L, (cuuint64_t)B};
    cuuint64_t strides[3] = {(cuuint64_t)D * 2, (cuuint64_t)tok_stride * 2, (cuuint64_t)(B > 1 ? batch_stride : (long long)L * tok_stride) * 2};
    cuuint32_t box[4] = {64, 1, (cuuint32_t)rows, 1};
    cuuint32_t estr[4] = {1, 1, 1, 1};
    auto encode = [&] {
        return fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void*>(base), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                  CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    };
    CUresult r = encode();
    int dev = 0;
    if (r == CUDA_ERROR_INVALID_CONTEXT && cudaGetDevice(&dev) == cudaSuccess && cudaSetDevice(dev) == cudaSuccess)
        r = encode();                                    // the first CUDA work of this thread: a driver call brings no context up by itself
    if (r != CUDA_SUCCESS) {
        cudaGetLastError();
        return false;
    }
    if (cache) cache->insert(key, *m);
    return true;
}

// ---- device helpers --------------------------------------------------------------------------------
// First 1024-byte boundary of the dynamic shared memory.  The result is formed by adding an offset to the
// __shared__ array itself, never by casting an integer back to a pointer: a pointer that went through an integer
// loses its address space, and every access through it is compiled as a generic load or store.
__device__ __forceinline__ unsigned char* align1024(unsigned char* smem) {
    return smem + ((1024u - (ptx::smem_u32(smem) & 1023u)) & 1023u);
}

// Load one [64 x 128] tile (two boxes) of head h, batch b starting at token t0.
__device__ __forceinline__ void tma_tile(void* dst, const CUtensorMap* m, uint64_t* bar, int h, int t0, int b) {
    ptx::tma_load_4d(dst, m, bar, 0, h, t0, b);
    ptx::tma_load_4d(static_cast<char*>(dst) + BOX, m, bar, 64, h, t0, b);
}

// Decay tables of one block, computed by `nwarps` warps (threads 0 .. 32*nwarps-1).  Callers
// synchronise afterwards.
//   bloc[t]  = inclusive cumulative log-decay of token t inside ITS chunk  (t = 0 .. nch*64-1)
//   ctot[c]  = chunk totals
// of the log-decays as log_decay_bf16() limits them.  Tokens at or beyond `L` (a last chunk that is not full) get log-decay 0; TMA fills
// their tile rows with zeros.
// `issued`, if given, is an mbarrier (count = nwarps) on which every warp arrives once its loads are on their way: the
// TMA warp waits for it, so that these small requests do not queue behind the first burst of tile loads that all CTAs
// of the device send at the same moment.
__device__ __forceinline__ void prep_decay(const float* __restrict__ gh, long long tg, long long t0, int nch, int L, float* bloc,
                                           float* ctot, int nwarps, uint64_t* issued = nullptr) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int lim = L - (int)t0;                            // tokens from the block start to the end of the segment
    // All loads of this warp's chunks go out before the first scan (one memory round trip for the whole block, not one
    // per chunk).  Unconditional loads from clamped (always valid) tokens, zeroed afterwards.
    constexpr int MAXC = 4;                                 // chunks per warp in one round (MAXR / 8 warps)
    for (int cbase = warp; cbase < nch; cbase += nwarps * MAXC) {
        float g0[MAXC], g1[MAXC];
#pragma unroll
        for (int i = 0; i < MAXC; ++i) {
            const int c = cbase + i * nwarps;
            const int r = c * C + 2 * lane;
            const bool on = c < nch;
            g0[i] = on ? gh[(t0 + min(r, lim - 1)) * tg] : 0.f;
            g1[i] = on ? gh[(t0 + min(r + 1, lim - 1)) * tg] : 0.f;
        }
        if (issued && cbase == warp) { ptx::mbar_arrive_warp(issued); issued = nullptr; }
#pragma unroll
        for (int i = 0; i < MAXC; ++i) {
            const int c = cbase + i * nwarps;
            if (c < nch) {
                const int r = c * C + 2 * lane;             // selected, not multiplied by 0: the last token's value may be NaN
                g0[i] = r < lim ? log_decay_bf16(g0[i]) : 0.f;
                g1[i] = r + 1 < lim ? log_decay_bf16(g1[i]) : 0.f;
                float incl = g0[i] + g1[i];
                for (int off = 1; off < 32; off <<= 1) {
                    const float up = __shfl_up_sync(0xffffffffu, incl, off);
                    if (lane >= off) incl += up;
                }
                bloc[c * C + 2 * lane] = incl - g1[i];
                bloc[c * C + 2 * lane + 1] = incl;
                if (lane == 31) ctot[c] = incl;
            }
        }
    }
    if (issued) ptx::mbar_arrive_warp(issued);             // a warp without a chunk of its own has nothing to wait for
}

__device__ __forceinline__ void st_unit(unsigned char* box, int row, int unit, uint4 v) {
    *reinterpret_cast<uint4*>(box + row * 128 + ((unit ^ (row & 7)) << 4)) = v;
}
__device__ __forceinline__ uint4 ld_unit(const unsigned char* box, int row, int unit) {
    return *reinterpret_cast<const uint4*>(box + row * 128 + ((unit ^ (row & 7)) << 4));
}
__device__ __forceinline__ uint32_t pack2(float a, float b) {
    __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
    return *reinterpret_cast<uint32_t*>(&h);
}

// dst = diag(w) * src for a [64 x 128] tile (two boxes), done by NTHR threads (this one is `t`);
// w_row(row) gives the weight of a token row.  dst may equal src.  A thread touches 16-byte units
// t + NTHR*i; a box holds 64 rows x 8 units, so with NTHR = 256 it meets only rows (t>>3) and (t>>3)+32.
template <int NTHR, typename F>
__device__ __forceinline__ void scale_tile(unsigned char* dst, const unsigned char* src, int t, F w_row) {
    static_assert(NTHR == 256, "unit-to-row mapping below assumes 256 threads");
    const uint4* in = reinterpret_cast<const uint4*>(src);
    uint4* out = reinterpret_cast<uint4*>(dst);
    const float w0 = w_row(t >> 3), w1 = w_row((t >> 3) + 32);
    uint4 v[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) v[i] = in[t + NTHR * i];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const float w = (i & 1) ? w1 : w0;
        __nv_bfloat162* h2 = reinterpret_cast<__nv_bfloat162*>(&v[i]);
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const float2 f = __bfloat1622float2(h2[e]);
            h2[e] = __floats2bfloat162_rn(f.x * w, f.y * w);
        }
        out[t + NTHR * i] = v[i];
    }
}

// Passes over the [128 x 128] float32 state at TMEM columns `acc`; a thread owns lane threadIdx.x & 127 and NU units of 16 columns from u0
// on.  They are loops, not straight code: what a CTA runs has to stay in the instruction cache (see the sweeps).
//
// The state from global memory (init[a*128 + i], or init[i*128 + a] when `transposed`; NULL: zero) to tensor memory.
template <int NU>
__device__ __forceinline__ void state_init(uint32_t acc, const float* init, bool transposed, int u0) {
    const int a = threadIdx.x & 127;
    const uint32_t taddr = acc + ((uint32_t)((a >> 5) * 32) << 16);
#pragma unroll 1
    for (int u = u0; u < u0 + NU; ++u) {
        float v[16] = {};
        if (init && transposed) {
#pragma unroll
            for (int i = 0; i < 16; ++i) v[i] = init[(u * 16 + i) * D + a];
        } else if (init) {
#pragma unroll
            for (int i = 0; i < 16; i += 4) *reinterpret_cast<float4*>(v + i) = *reinterpret_cast<const float4*>(init + a * D + u * 16 + i);
        }
        ptx::tmem_st16(taddr + u * 16, v);
    }
    ptx::tmem_st_wait();
}
// The bf16 copy of the state to `sb` (two boxes of [128 rows x 64 columns], 16 KB apart); the accumulator times `decay`.
template <int NU>
__device__ __forceinline__ void state_pass(uint32_t acc, unsigned char* sb, float decay, int u0) {
    static_assert(NU % 2 == 0, "two units at a time");
    const int a = threadIdx.x & 127;
    const uint32_t taddr = acc + ((uint32_t)((a >> 5) * 32) << 16);
#pragma unroll 1
    for (int u = u0; u < u0 + NU; u += 2) {
        float v[32];
        ptx::tmem_ld32(taddr + u * 16, v);
        ptx::tmem_ld_wait();
        unsigned char* box = sb + (u >> 2) * 16384;
#pragma unroll
        for (int e = 0; e < 4; ++e)
            st_unit(box, a, (u & 3) * 2 + e, make_uint4(pack2(v[e * 8], v[e * 8 + 1]), pack2(v[e * 8 + 2], v[e * 8 + 3]),
                                                        pack2(v[e * 8 + 4], v[e * 8 + 5]), pack2(v[e * 8 + 6], v[e * 8 + 7])));
#pragma unroll
        for (int i = 0; i < 32; i += 2) ptx::mul2(v[i], v[i + 1], decay, decay);
        ptx::tmem_st32(taddr + u * 16, v);
    }
    ptx::tmem_st_wait();
}

// Rows of the [128 x 128] float32 accumulator at TMEM columns `acc` to a dense array: NU units of 16 columns from u0 on, the
// thread owns lane threadIdx.x & 127.
template <int NU>
__device__ __forceinline__ void state_out(uint32_t acc, float* __restrict__ dst, int u0) {
    const int a = threadIdx.x & 127;
    const uint32_t taddr = acc + ((uint32_t)((a >> 5) * 32) << 16);
#pragma unroll 1
    for (int k = 0; k < NU; ++k) {
        float v[16];
        ptx::tmem_ld16(taddr + (u0 + k) * 16, v);
        ptx::tmem_ld_wait();
        float4* o4 = reinterpret_cast<float4*>(dst + a * D + (u0 + k) * 16);
#pragma unroll
        for (int i = 0; i < 4; ++i) o4[i] = make_float4(v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]);
    }
}

// One K loop of MMAs from precomputed low descriptor words.  Offset rules of a K step (16-byte units):
//   DK16: K-major operand (a [128 rows x 128] tile, K step = features 16*ks .. 16*ks+15: +32 B inside a box, the second 64
//         features in the next box 16 KB away);
//   DMN:  MN-major operand (rows are the contraction index: K step = rows 16*ks .. 16*ks+15 = +2048 B; the other 64
//         elements of M/N lie one box away, which is the descriptor's leading offset).
// Straight code, unlike the elementwise passes: a loop's few dependent instructions per step take longer than the MMA (out_done of a
// sweep came 1500 cycles after the first issue instead of 800).
enum { DK16 = 1, DMN = 2 };
template <int RULE>
__host__ __device__ constexpr uint32_t dofs(int ks) { return RULE == DMN ? 128u * ks : 1024u * (ks >> 2) + 2u * (ks & 3); }
template <int FROM, int TO, int RA, int RB>
__device__ __forceinline__ void mma_group(uint32_t d, uint32_t alo, uint32_t blo, uint32_t idesc, bool acc) {
    if constexpr (FROM < TO) {
        ptx::mma_lo(d, alo + dofs<RA>(FROM), blo + dofs<RB>(FROM), idesc, acc);
        mma_group<FROM + 1, TO, RA, RB>(d, alo, blo, idesc, true);
    }
}
__device__ __forceinline__ uint32_t klo(uint32_t tile) { return ptx::desc_lo(tile, 0); }
__device__ __forceinline__ uint32_t mlo(uint32_t tile, uint32_t box_bytes) { return ptx::desc_lo(tile, box_bytes); }

#define SF_SPIN(bar, parity, code) ptx::mbar_wait<true>(bar, parity, abort_flag, code)
#define SF_WAIT(bar, parity, code) ptx::mbar_wait(bar, parity, abort_flag, code)

// ==================================================================================================
// Block aggregates on tensor cores: U = sum_s w_s x_s^T y_s over the block (M = N = 128, K = tokens).
//   mode 0: (x, y) = (k, v), w_s = exp(beta - B_s);   mode 1: (x, y) = (q, dO), w_s = exp(B_s)
// The chunks are visited against the order of the sweep that comes next (mode 0 from the last one on): it begins with what is still in
// L2 (forward, 8192 tokens x 32 heads 84.5 -> 80.5 us, 16384 147.9 -> 144.8).
// y is scaled by w in place in shared memory, then U += X^T (w*Y) with both operands MN-major.
// 8 compute warps, one TMA warp, one MMA warp.
constexpr int AGG_STAGES = 4;
constexpr int AGG_COMP = 256;
constexpr int AGG_THREADS = AGG_COMP + 64;
struct AggSmem {
    alignas(1024) unsigned char tiles[AGG_STAGES][2][TILE];
    float bloc[MAXR * C];
    float ctot[MAXR];
    float cofs[MAXR];
    float beta;
    uint64_t full[AGG_STAGES], empty[AGG_STAGES], ready[AGG_STAGES], done, g_issued;
    uint32_t tmem_base;
    int abort_flag;
};

__global__ void __launch_bounds__(AGG_THREADS, 1)
tc_aggregate_kernel(const __grid_constant__ CUtensorMap tmX, const __grid_constant__ CUtensorMap tmY, SegParams p,
                    const float* __restrict__ g, int mode, float* __restrict__ U, float* __restrict__ beta_out) {
    extern __shared__ unsigned char smem_raw[];
    AggSmem& sm = *reinterpret_cast<AggSmem*>(align1024(smem_raw));
    const int h = blockIdx.x, j = blockIdx.y, b = blockIdx.z;   // heads fastest: co-resident CTAs read neighbouring 256-byte pieces of the same tokens
    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
    const int c0 = j * p.R, nch = min(p.R, p.NC - c0);
    const long long t0 = (long long)c0 * C;
    int* abort_flag = &sm.abort_flag;
    constexpr int WT = AGG_COMP / 32, WM = WT + 1;
    auto at = [&](int c) { return mode == 0 ? nch - 1 - c : c; };

    if (tid == 0) {
        sm.abort_flag = 0;
        for (int s = 0; s < AGG_STAGES; ++s) { ptx::mbar_init(&sm.full[s], 1); ptx::mbar_init(&sm.empty[s], 1); ptx::mbar_init(&sm.ready[s], AGG_COMP / 32); }
        ptx::mbar_init(&sm.done, 1);
        ptx::mbar_init(&sm.g_issued, AGG_COMP / 32);
        ptx::fence_mbar_init();
    }
    if (warp == WT) ptx::tmem_alloc(&sm.tmem_base, 128);
    ptx::tc_fence_before_sync();
    __syncthreads();
    ptx::tc_fence_after_sync();
    const uint32_t tmem = sm.tmem_base;
    if (p.wait_first) grid_wait();

    if (warp == WT) {
        if (lane == 0) {
            grid_launch_next();                            // only now: see there
            ptx::prefetch_tmap(&tmX);
            ptx::prefetch_tmap(&tmY);
            SF_WAIT(&sm.g_issued, 0, DEV_TIMEOUT_TMA);
            for (int c = 0; c < nch; ++c) {
                const int s = c % AGG_STAGES, it = c / AGG_STAGES;
                if (it > 0) SF_WAIT(&sm.empty[s], (it - 1) & 1, DEV_TIMEOUT_MMA);
                ptx::mbar_expect_tx(&sm.full[s], 2 * TILE);
                tma_tile(sm.tiles[s][0], &tmX, &sm.full[s], h, (int)t0 + at(c) * C, b);
                tma_tile(sm.tiles[s][1], &tmY, &sm.full[s], h, (int)t0 + at(c) * C, b);
            }
        }
    } else if (warp == WM) {
        if (lane == 0) {
            constexpr uint32_t idesc = ptx::idesc_bf16(128, 128, 1, 1);
            for (int c = 0; c < nch; ++c) {
                const int s = c % AGG_STAGES, it = c / AGG_STAGES;
                SF_WAIT(&sm.ready[s], it & 1, DEV_TIMEOUT_TMA);
                ptx::tc_fence_after_sync();
                const uint32_t xa = ptx::smem_u32(sm.tiles[s][0]), ya = ptx::smem_u32(sm.tiles[s][1]);
                mma_group<0, 4, DMN, DMN>(tmem, mlo(xa, BOX), mlo(ya, BOX), idesc, c > 0);
                ptx::mma_commit(&sm.empty[s]);
            }
            ptx::mma_commit(&sm.done);
        }
    } else {
        const float* gh = g + (long long)b * p.bg + h;
        prep_decay(gh, p.tg, t0, nch, p.L, sm.bloc, sm.ctot, WT, &sm.g_issued);
        ptx::named_bar_sync(1, AGG_COMP);
        if (tid == 0) {
            float acc = 0.f;
            if (mode == 0) { for (int c = nch - 1; c >= 0; --c) { sm.cofs[c] = acc; acc += sm.ctot[c]; } }
            else           { for (int c = 0; c < nch; ++c)      { sm.cofs[c] = acc; acc += sm.ctot[c]; } }
            sm.beta = acc;
        }
        ptx::named_bar_sync(1, AGG_COMP);
        for (int c = 0; c < nch; ++c) {
            const int s = c % AGG_STAGES, it = c / AGG_STAGES;
            SF_WAIT(&sm.full[s], it & 1, DEV_TIMEOUT_TMA);
            const int cc = at(c);
            const float cof = sm.cofs[cc], bC = sm.ctot[cc];
            const float* bch = sm.bloc + cc * C;
            scale_tile<AGG_COMP>(sm.tiles[s][1], sm.tiles[s][1], tid,
                       [&](int row) { return fast_exp(mode == 0 ? (bC - bch[row]) + cof : bch[row] + cof); });
            ptx::fence_proxy_async();
            ptx::mbar_arrive_warp(&sm.ready[s]);
        }
        SF_WAIT(&sm.done, 0, DEV_TIMEOUT_MMA);
        ptx::tc_fence_after_sync();
        grid_wait();                                       // the workspace may still be in use by the kernels before
        if (tid == 0 && beta_out) beta_out[((long long)b * p.H + h) * p.NB + j] = sm.beta;
        // 8 warps read the [128 x 128] accumulator: warp w covers lanes 32*(w&3).., column half w>>2
        const int row = tid & 127, half = tid >> 7;
        float* Uo = U + (((long long)b * p.H + h) * p.NB + j) * (long long)(D * D) + (long long)row * D + half * 64;
#pragma unroll
        for (int cb = 0; cb < 2; ++cb) {
            float v[32];
            ptx::tmem_ld32(tmem + ((uint32_t)((warp & 3) * 32) << 16) + half * 64 + cb * 32, v);
            ptx::tmem_ld_wait();
#pragma unroll
            for (int e = 0; e < 32; e += 4)
                *reinterpret_cast<float4*>(Uo + cb * 32 + e) = make_float4(v[e], v[e + 1], v[e + 2], v[e + 3]);
        }
        ptx::tc_fence_before_sync();
    }
    __syncthreads();
    if (warp == WT) ptx::tmem_dealloc(tmem, 128);
}

// ==================================================================================================
// Chunk sweeps of a block: o (Out + ST of paper Eq. 2), dq (SR + OG of Section 3.4), dk and dv (STB + PG).  All four have the
// same form over tiles of 128 tokens, with x, y, z three of the tensors and a carried state St [128 x 128]:
//     out_r = sum_s (x_r . y_s) D[r,s] z_s  +  a_r x_r St ;     St <- exp(b_T) St + y^T diag(w) z
//             x   y   z    St               runs      pairs   D                a_r             w_s
//       o     q   k   v    H                forward   s <= r  exp(b_r - b_s)   exp(b_r)        exp(b_T - b_s)
//       dq    dO  v   k    H^T              forward   s <= r  exp(b_r - b_s)   exp(b_r)        exp(b_T - b_s)
//       dk    v   dO  q    G^T              reverse   s >= r  exp(b_s - b_r)   exp(b_T - b_r)  exp(b_s)
//       dv    k   q   dO   G                reverse   s >= r  exp(b_s - b_r)   exp(b_T - b_r)  exp(b_s)
// b: inclusive cumulative log-decay inside the tile, b_T its total, H the state, G the gradient of the state leaving the tile.
// With b_T - b in the place of b the reverse sweeps' weights are those of the forward ones; the decay tables hold it.
// dq and dk also store the row dot products x_out[t] = q_t . dq_t and k_t . dk_t (float32), which the log-decay gradient needs.
//
// Per tile four groups of eight MMAs of 128 x 128 x 16 (64 cycles each): scores x y^T, x St, the state update, and P z with
// P = bf16(scores * D) read from tensor memory, where the mask pass leaves it in the columns of the scores.  y is scaled by w in
// place once the scores have been taken; the output tile replaces z and leaves by TMA, the tile for the dot products arrives
// in the place of x: so two whole tile sets and the state fit the shared memory, and no operand is copied.
// K steps of P z write only the lanes whose rows have a pair in them (disable-output-lane), so a row meets no z row beyond
// its own 16 tokens: there 0 * Inf would be NaN.
//
// Why tiles of 128 tokens: a chunk of 64 needs M = 64 MMAs for the token-row products, which run at half rate, and pays every
// hand-off between MMAs and elementwise passes (commit, wait, fence, 100-250 cycles each) twice as often.
//
// Why loops where the code could be unrolled, and one body for the backward's sweeps with the role as a value: the 20 warps run eight
// different programs, and what they run per tile has to stay in the instruction cache.  Straight code, 62 KB for the forward sweep and 197 KB
// for the backward's three, took 7700 cycles per tile forward and 16000-20000 in dk and dv, whose CTAs pushed each other's code out; now 31 and
// 37 KB and 4150 / 5700 (dq, dk) / 5000 (dv).  A short call runs mostly cold code: 200 tokens x 16 heads 21.8 -> 13.6 us with the last 10 KB.
//
// What bounds them: per tile scores -> mask -> P z -> epilogue in series (850 + 1650 + 800 + 600 cycles), MMAs 2048 of 4150.  A second set of
// score columns (x St and P z in one accumulator, rescaled between) to overlap two tiles was slower: 4700 cycles, the elementwise warps
// then are in series.  Against 64-token tiles with dk and dv in one sweep (16384 tokens x 32 heads): o 123 -> 87 us, dq 151 -> 110,
// dk and dv 219 -> 201 (one launch of 256 CTAs, two waves of 32 tiles in series); chains forward + backward 1.13x, 256K tokens x 32 heads 9.43 -> 8.25 ms.
//
// A tile is two 64-token chunks, or one before a chunk where a segment of a merged launch begins (SegParams::bslot) and at the end
// of a block; the rows of a missing half take no part in the state update and in P z and are not stored.
//
// Roles (20 warps): WG0, WG1 state pass (TMEM state -> bf16 copy in shared memory, rescaled state), then y *= w;  WG2, WG3
// decay mask, then epilogue;  warp 16 MMAs, 17 tile loads, 18 output tiles, 19 decay tables.
// Tensor memory: St 0-127, x St 128-255, P z 256-383, scores / P 384-511.
constexpr int SW_THREADS = 640;
constexpr int W_MMA = 16, W_TMA = 17, W_OUT = 18, W_TAB = 19;
constexpr int TT = 128;                    // tokens per tile
constexpr int FBOX = TT * 128;             // bytes of [128 tokens x 64 features]
constexpr int XTILE = 2 * FBOX;            // bytes of [128 tokens x 128 features]
enum { SWEEP_O = 0, SWEEP_DQ = 1, SWEEP_DK = 2, SWEEP_DV = 3 };

struct SweepSmem {
    alignas(1024) unsigned char tiles[2][3][XTILE];      // x, y, z
    alignas(1024) unsigned char sb[2 * FBOX];            // bf16 copy of the state
    float b[2][TT];                                      // cumulative log-decay of a tile, in units of log 2
    float u[2][TT];                                      // 2^(b_ref - b_s), ref the token of s's 32 that is nearest to the rows they meet
                                                         // (both: the halves of the row dot products, once the tile's tables have served)
    float total[2];
    uint64_t full_xy[2], full_z[2], sc_done[2], p_ready[2], y_ready[2], st_ready[2], st_done[2], x_done[2], out_done[2], o_free[2], staged[2],
        e_full[2], z_free[2], tab_full[2], g_issued;
    unsigned long long cuts;
    uint32_t tmem_base;
    int abort_flag;
};
static_assert(sizeof(SweepSmem) <= 227 * 1024, "one CTA per SM");

// The tiles of a block of nch chunks, in order: first chunk c and length len (1 or 2 chunks) of the i-th.
struct Tiles {
    bool rev;
    int nch, i, c, len;
    unsigned long long cuts;                             // forward: bit c set where a tile must begin at chunk c
    __device__ __forceinline__ Tiles(bool rev_, int nch_, unsigned long long cuts_) : rev(rev_), nch(nch_), i(0), cuts(cuts_) {
        c = rev ? (nch - 1) & ~1 : 0;
        measure();
    }
    __device__ __forceinline__ void measure() { len = c + 1 < nch && !((cuts >> ((c + 1) & 63)) & 1) ? 2 : 1; }
    __device__ __forceinline__ bool more() const { return rev ? c >= 0 : c < nch; }
    __device__ __forceinline__ void next() {
        c = rev ? c - 2 : c + len;
        ++i;
        measure();
    }
    __device__ __forceinline__ int stage() const { return i & 1; }
    __device__ __forceinline__ uint32_t phase() const { return (i >> 1) & 1; }
};

// Loads the tile of head h from token t0 on; tokens at or beyond the end of the tensor are zeros.
__device__ __forceinline__ void load_tile(unsigned char* dst, const CUtensorMap* m, uint64_t* bar, int h, int t0, int b) {
    ptx::tma_load_4d(dst, m, bar, 0, h, t0, b);
    ptx::tma_load_4d(dst + FBOX, m, bar, 64, h, t0, b);
}
__device__ __forceinline__ void prefetch_tile(const CUtensorMap* m, int h, int t0, int b) {
    ptx::tma_prefetch_4d(m, 0, h, t0, b);
    ptx::tma_prefetch_4d(m, 64, h, t0, b);
}

// P = bf16(scores * D), D = 2^(b_r - b_s), for the 32 rows of a warp (row 32 q + lane) and every second block of 32 columns that has a
// pair, from block `half` on; P of a block takes the first half of its own columns.  Off the diagonal D is the product of a factor
// of the row and one of the column, both at most 1, split at the token of the block that is nearest to the rows: an
// exponential per element there would keep the SM quarter of the last rows (four of ten blocks) busy for 1000 cycles.
__device__ __forceinline__ void mask_tile(uint32_t sc, const float* b, const float* u, bool rev, int half) {
    const int q = (threadIdx.x >> 5) & 3, lane = threadIdx.x & 31;
    const uint32_t taddr = sc + ((uint32_t)(q * 32) << 16), pairs = rev ? 0xffffffffu << lane : 0xffffffffu >> (31 - lane);
    const float br = b[32 * q + lane];
#pragma unroll 1
    for (int cb = rev ? q + ((q ^ half) & 1) : half; cb < (rev ? 4 : q + 1); cb += 2) {
        float x[32], y[16];
        ptx::tmem_ld32(taddr + 32 * cb, x);
        if (cb == q) {
            const float* bc = b + 32 * cb;
            ptx::tmem_ld_wait();
#pragma unroll
            for (int j = 0; j < 32; j += 4) {
                const float4 f = *reinterpret_cast<const float4*>(bc + j);
                const float bs[4] = {f.x, f.y, f.z, f.w};
#pragma unroll
                for (int e = 0; e < 4; ++e) x[j + e] = (pairs >> (j + e)) & 1 ? x[j + e] * ptx::ex2(br - bs[e]) : 0.f;
            }
        } else {
            const float fr = ptx::ex2(br - b[32 * cb + (rev ? 0 : 31)]);
            const float* uc = u + 32 * cb;
            ptx::tmem_ld_wait();
#pragma unroll
            for (int j = 0; j < 32; j += 4) {
                const float4 f = *reinterpret_cast<const float4*>(uc + j);
                ptx::mul2(x[j], x[j + 1], fr, fr); ptx::mul2(x[j + 2], x[j + 3], fr, fr);
                ptx::mul2(x[j], x[j + 1], f.x, f.y); ptx::mul2(x[j + 2], x[j + 3], f.z, f.w);
            }
        }
#pragma unroll
        for (int j = 0; j < 16; ++j) y[j] = __uint_as_float(pack2(x[2 * j], x[2 * j + 1]));
        ptx::tmem_st16(taddr + 32 * cb, y);
    }
    ptx::tmem_st_wait();
}

// y *= w in place, 256 threads; a thread meets the rows t/8 + 32 i
template <typename F>
__device__ __forceinline__ void scale_rows(unsigned char* tile, int t, F w_row) {
    uint4* u = reinterpret_cast<uint4*>(tile);
    float w[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) w[i] = w_row((t >> 3) + 32 * i);
#pragma unroll 1
    for (int hf = 0; hf < 2; ++hf) {
        uint4 v[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) v[i] = u[hf * (FBOX / 16) + t + 256 * i];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            __nv_bfloat162* h2 = reinterpret_cast<__nv_bfloat162*>(&v[i]);
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                float2 f = __bfloat1622float2(h2[e]);
                ptx::mul2(f.x, f.y, w[i], w[i]);
                h2[e] = __floats2bfloat162_rn(f.x, f.y);
            }
            u[hf * (FBOX / 16) + t + 256 * i] = v[i];
        }
    }
}

// Row 32 q + lane of the output, features 64 half ..: a * inter + intra as bf16 into the tile `slot` and, with `with_dot`, its dot product
// with the tile `e_tile`.  `loaded` is called once the accumulators have been read.
template <typename F>
__device__ __forceinline__ float epilogue_tile(uint32_t inter, uint32_t intra, unsigned char* slot, const unsigned char* e_tile, float a, int half,
                                               bool with_dot, F loaded) {
    const int q = (threadIdx.x >> 5) & 3, row = 32 * q + (threadIdx.x & 31);
    const uint32_t from = ((uint32_t)(q * 32) << 16) + 64 * half;
    unsigned char* box = slot + half * FBOX;
    float dot0 = 0.f, dot1 = 0.f;                        // even and odd features
#pragma unroll 1
    for (int cb = 0; cb < 2; ++cb) {
        float x[32], y[32];
        ptx::tmem_ld32(inter + from + 32 * cb, x);
        ptx::tmem_ld32(intra + from + 32 * cb, y);
        ptx::tmem_ld_wait();
        if (cb == 1) loaded();
#pragma unroll
        for (int i = 0; i < 32; i += 2) ptx::fma2(y[i], y[i + 1], x[i], x[i + 1], a, a);
        if (with_dot) {
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const uint4 v = ld_unit(e_tile + half * FBOX, row, cb * 4 + e);
                const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const float2 f = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&w[i]));
                    ptx::fma2(dot0, dot1, y[8 * e + 2 * i], y[8 * e + 2 * i + 1], f.x, f.y);
                }
            }
        }
#pragma unroll
        for (int e = 0; e < 4; ++e)
            st_unit(box, row, cb * 4 + e, make_uint4(pack2(y[8 * e], y[8 * e + 1]), pack2(y[8 * e + 2], y[8 * e + 3]),
                                                     pack2(y[8 * e + 4], y[8 * e + 5]), pack2(y[8 * e + 6], y[8 * e + 7])));
    }
    return dot0 + dot1;
}

// P z over K steps of 16 tokens: FROM .. TO - 1 of the eight, counted from the last one in the reverse sweeps, each for the lanes that have a
// pair in it: rows from 16 ks on (forward) or up to 16 ks + 15 (reverse).  The first step is the one that all rows take part in.
template <int FROM, int TO>
__device__ __forceinline__ void mma_intra(uint32_t d, uint32_t p, uint32_t zlo, uint32_t idesc, bool rev, bool acc) {
    if constexpr (FROM < TO) {
        constexpr int pc = 32 * (FROM >> 1) + 8 * (FROM & 1), lanes = 16 * FROM;
        uint32_t off[4];
#pragma unroll
        for (int w = 0; w < 4; ++w) {
            const int n = lanes - 32 * w, m = lanes - 96 + 32 * w;       // lanes of word w that are off: the first n, or the last m
            const uint32_t fwd = n <= 0 ? 0u : n >= 32 ? ~0u : (1u << n) - 1, bwd = m <= 0 ? 0u : m >= 32 ? ~0u : ~0u << (32 - m);
            off[w] = rev ? bwd : fwd;
        }
        ptx::mma_ts(d, rev ? p + 104 - pc : p + pc, rev ? zlo + dofs<DMN>(7 - FROM) : zlo + dofs<DMN>(FROM), idesc, acc, off);
        mma_intra<FROM + 1, TO>(d, p, zlo, idesc, rev, true);
    }
}

struct SweepMaps { const CUtensorMap *x, *y, *z, *e, *out; };      // out: boxes of 64 tokens, the others of 128

template <bool BWD>
__device__ __forceinline__ void sweep_body(int role, const SweepMaps& m, const SegParams& p, const float* __restrict__ g, const float* states,
                                           const float* s_init, float* __restrict__ xout, int h, int j) {
    const bool rev = BWD && role >= SWEEP_DK, dot = BWD && role != SWEEP_DV;       // dq and dk carry the transposed state
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    SweepSmem& sm = *reinterpret_cast<SweepSmem*>(smem_raw);
    const int b = blockIdx.z;
    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
    const int c0 = j * p.R, nch = min(p.R, p.NC - c0), t0 = c0 * C;
    int* abort_flag = &sm.abort_flag;
    constexpr uint32_t T_ST = 0, T_INTER = 128, T_INTRA = 256, T_SC = 384;

    if (tid == 0) {
        sm.abort_flag = 0;
        for (int s = 0; s < 2; ++s) {
            ptx::mbar_init(&sm.full_xy[s], 1); ptx::mbar_init(&sm.full_z[s], 1); ptx::mbar_init(&sm.sc_done[s], 1);
            ptx::mbar_init(&sm.p_ready[s], 8); ptx::mbar_init(&sm.y_ready[s], 8); ptx::mbar_init(&sm.st_ready[s], 8);
            ptx::mbar_init(&sm.st_done[s], 1); ptx::mbar_init(&sm.x_done[s], 1); ptx::mbar_init(&sm.out_done[s], 1);
            ptx::mbar_init(&sm.o_free[s], 8); ptx::mbar_init(&sm.staged[s], 8); ptx::mbar_init(&sm.e_full[s], 1); ptx::mbar_init(&sm.z_free[s], 1);
            ptx::mbar_init(&sm.tab_full[s], 1);
        }
        ptx::mbar_init(&sm.g_issued, 1);
        ptx::fence_mbar_init();
    }
    if (warp == W_MMA) ptx::tmem_alloc(&sm.tmem_base, 512);
    if (!BWD && warp == 1) {                             // where segments of a merged launch begin (a block has at most 64 chunks), ahead of
                                                         // grid_wait(): see there
        unsigned long long cuts = 0;
        if (p.bslot) {
            const bool lo = lane < nch && __ldcg(p.bslot + c0 + lane) >= 0, hi = lane + 32 < nch && __ldcg(p.bslot + c0 + lane + 32) >= 0;
            cuts = __ballot_sync(0xffffffffu, lo) | ((unsigned long long)__ballot_sync(0xffffffffu, hi) << 32);
        }
        if (lane == 0) sm.cuts = cuts;
    }
    ptx::tc_fence_before_sync();
    __syncthreads();
    ptx::tc_fence_after_sync();
    const uint32_t tmem = sm.tmem_base;
    Tiles it(rev, nch, BWD ? 0 : sm.cuts);
    if (p.wait_first) grid_wait();

    if (warp == W_TMA) {
        const bool leader = ptx::elect_one();
        if (leader) {
            grid_launch_next();
            ptx::prefetch_tmap(m.x); ptx::prefetch_tmap(m.y); ptx::prefetch_tmap(m.z); ptx::prefetch_tmap(m.out);
        }
        SF_WAIT(&sm.g_issued, 0, DEV_TIMEOUT_TMA);
        for (; it.more(); it.next()) {
            const int s = it.stage(), tok = t0 + it.c * C;
            const uint32_t before = it.phase() ^ 1;
            const bool wait = it.i >= 2;
            // y of tile i - 2 has served with its state update, x with its product with the state (or as the tile for the dot products), z once
            // the output tile that took its place has left; what has to wait is on its way to L2 meanwhile.  full_xy is armed only where
            // tile i - 2 is known to have passed it.
            if (leader && dot) prefetch_tile(m.x, h, tok, b);
            if (leader) prefetch_tile(m.z, h, tok, b);
            if (wait) SF_WAIT(dot ? &sm.st_done[s] : &sm.x_done[s], before, DEV_TIMEOUT_MMA);
            if (leader) {
                ptx::mbar_expect_tx(&sm.full_xy[s], 2 * XTILE);
                load_tile(sm.tiles[s][dot], dot ? m.y : m.x, &sm.full_xy[s], h, tok, b);
            }
            if (wait) SF_WAIT(dot ? &sm.staged[s] : &sm.st_done[s], before, DEV_TIMEOUT_MMA);
            if (leader) load_tile(sm.tiles[s][!dot], dot ? m.x : m.y, &sm.full_xy[s], h, tok, b);
            if (wait) SF_WAIT(&sm.z_free[s], before, DEV_TIMEOUT_MMA);
            if (leader) {
                ptx::mbar_expect_tx(&sm.full_z[s], XTILE);
                load_tile(sm.tiles[s][2], m.z, &sm.full_z[s], h, tok, b);
                if (dot) prefetch_tile(m.e, h, tok, b);
            }
        }
    } else if (warp == W_MMA) {
        const bool leader = ptx::elect_one();
        constexpr uint32_t id_sc = ptx::idesc_bf16(128, 128, 0, 0), id_o = ptx::idesc_bf16(128, 128, 0, 1), id_st = ptx::idesc_bf16(128, 128, 1, 1);
        const uint32_t sb = ptx::smem_u32(sm.sb);
        for (; it.more(); it.next()) {
            const int s = it.stage();
            const uint32_t ph = it.phase();
            const uint32_t x = ptx::smem_u32(sm.tiles[s][0]), y = ptx::smem_u32(sm.tiles[s][1]), z = ptx::smem_u32(sm.tiles[s][2]);
            SF_SPIN(&sm.full_xy[s], ph, DEV_TIMEOUT_TMA);
            ptx::tc_fence_after_sync();
            if (leader) {                                // behind the MMAs that read the last P from these columns
                mma_group<0, 8, DK16, DK16>(tmem + T_SC, klo(x), klo(y), id_sc, false);
                ptx::mma_commit(&sm.sc_done[s]);
            }
            SF_SPIN(&sm.st_ready[s], ph, DEV_TIMEOUT_MMA);
            if (it.i > 0) SF_SPIN(&sm.o_free[s ^ 1], (uint32_t)((it.i - 1) >> 1) & 1, DEV_TIMEOUT_MMA);
            ptx::tc_fence_after_sync();
            if (leader) {
                mma_group<0, 8, DK16, DMN>(tmem + T_INTER, klo(x), mlo(sb, FBOX), id_o, false);
                ptx::mma_commit(&sm.x_done[s]);
            }
            SF_SPIN(&sm.full_z[s], ph, DEV_TIMEOUT_TMA);
            SF_SPIN(&sm.y_ready[s], ph, DEV_TIMEOUT_MMA);
            ptx::tc_fence_after_sync();
            if (leader) {
                mma_group<0, 4, DMN, DMN>(tmem + T_ST, mlo(y, FBOX), mlo(z, FBOX), id_st, true);
                if (it.len > 1) mma_group<4, 8, DMN, DMN>(tmem + T_ST, mlo(y, FBOX), mlo(z, FBOX), id_st, true);
                ptx::mma_commit(&sm.st_done[s]);
            }
            SF_SPIN(&sm.p_ready[s], ph, DEV_TIMEOUT_MMA);
            ptx::tc_fence_after_sync();
            if (leader) {                                // of a tile of one chunk the steps with its tokens: the first four, or the last in the reverse sweeps
                if (it.len > 1 || !rev) mma_intra<0, 4>(tmem + T_INTRA, tmem + T_SC, mlo(z, FBOX), id_o, rev, false);
                if (it.len > 1 || rev) mma_intra<4, 8>(tmem + T_INTRA, tmem + T_SC, mlo(z, FBOX), id_o, rev, it.len > 1);
                ptx::mma_commit(&sm.out_done[s]);
            }
        }
    } else if (warp == W_OUT) {
        const bool leader = ptx::elect_one();
        grid_wait();
        for (; it.more(); it.next()) {
            const int s = it.stage(), tok = t0 + it.c * C;
            if (dot) {
                SF_WAIT(&sm.x_done[s], it.phase(), DEV_TIMEOUT_MMA);
                if (leader) {
                    ptx::mbar_expect_tx(&sm.e_full[s], XTILE);
                    load_tile(sm.tiles[s][0], m.e, &sm.e_full[s], h, tok, b);
                }
            }
            if (leader && it.i > 0) {                    // behind the load for the dot products, which is waited for earlier
                ptx::tma_store_wait_read();
                ptx::mbar_arrive(&sm.z_free[s ^ 1]);
            }
            SF_WAIT(&sm.staged[s], it.phase(), DEV_TIMEOUT_MMA);
            if (leader) {
                const unsigned char* slot = sm.tiles[s][2];
#pragma unroll 1
                for (int th = 0; th < it.len; ++th)
                    if (tok + th * C < p.L) {
                        ptx::tma_store_4d(m.out, slot + th * BOX, 0, h, tok + th * C, b);
                        ptx::tma_store_4d(m.out, slot + FBOX + th * BOX, 64, h, tok + th * C, b);
                    }
                ptx::tma_store_commit();
            }
        }
        if (leader) ptx::tma_store_wait();
    } else if (warp == W_TAB) {
        // four tokens per lane; the log-decays of the next tile are on their way while this one is worked on
        const float* gh = g + (long long)b * p.bg + h;
        float gv[4];
        auto fetch = [&](const Tiles& t) {
            const int base = t0 + t.c * C + 4 * lane, lim = min(p.L, t0 + (t.c + t.len) * C);
            const float* src = gh + base * p.tg;
#pragma unroll
            for (int e = 0; e < 4; ++e, src += p.tg) gv[e] = base + e < lim ? __ldg(src) : 0.f;
        };
        fetch(it);
        if (lane == 0) ptx::mbar_arrive(&sm.g_issued);
        Tiles done = it;
        while (true) {
            const int s = it.stage();
#pragma unroll
            for (int e = 0; e < 4; ++e) gv[e] = log_decay_bf16(gv[e]) * LOG2E;
            gv[1] += gv[0]; gv[2] += gv[1]; gv[3] += gv[2];
            float pre = gv[3];
#pragma unroll
            for (int off = 1; off < 32; off <<= 1) {
                const float up = __shfl_up_sync(0xffffffffu, pre, off);
                if (lane >= off) pre += up;
            }
            const float total = __shfl_sync(0xffffffffu, pre, 31);
            if (lane == 31) sm.total[s] = total;
            pre -= gv[3];                                // tokens before this lane's
#pragma unroll
            for (int e = 0; e < 4; ++e) gv[e] = rev ? total - (gv[e] + pre) : gv[e] + pre;
            *reinterpret_cast<float4*>(sm.b[s] + 4 * lane) = make_float4(gv[0], gv[1], gv[2], gv[3]);
            const float ref = __shfl_sync(0xffffffffu, rev ? gv[0] : gv[3], rev ? lane & ~7 : lane | 7);
            *reinterpret_cast<float4*>(sm.u[s] + 4 * lane) = make_float4(ptx::ex2(ref - gv[0]), ptx::ex2(ref - gv[1]), ptx::ex2(ref - gv[2]), ptx::ex2(ref - gv[3]));
            ptx::mbar_arrive_warp(&sm.tab_full[s]);
            const bool first = it.i == 0;
            it.next();
            if (it.more()) fetch(it);
            if (first) {
                grid_wait();
                if (it.more()) continue;
            }
            // The tables of a tile have served once its output is staged; in their place come the halves of its row dot products.  At the end
            // the last two tiles are left.
            do {
                const int sd = done.stage();
                SF_WAIT(&sm.staged[sd], done.phase(), DEV_TIMEOUT_MMA);
                if (dot) {
                    const int tok = t0 + done.c * C + lane, lim = min(p.L, t0 + (done.c + done.len) * C);
                    float* xo = xout + ((long long)b * p.H + h) * p.L + tok;
#pragma unroll
                    for (int e = 0; e < 4; ++e)
                        if (tok + 32 * e < lim) xo[32 * e] = sm.u[sd][lane + 32 * e] + sm.b[sd][lane + 32 * e];
                    __syncwarp();
                }
                done.next();
            } while (!it.more() && done.more());
            if (!it.more()) break;
        }
    } else {
        const int wg = warp >> 2;
        const long long bh = (long long)b * p.H + h;
        // tables, first tiles, scores and mask need only the caller's inputs: they run while the scan finishes
        if (wg >= 2) {
            const int row = tid & 127, half = wg - 2;
            for (; it.more(); it.next()) {
                const int s = it.stage();
                SF_WAIT(&sm.tab_full[s], it.phase(), DEV_TIMEOUT_MMA);
                SF_WAIT(&sm.sc_done[s], it.phase(), DEV_TIMEOUT_MMA);
                ptx::tc_fence_after_sync();
                mask_tile(tmem + T_SC, sm.b[s], sm.u[s], rev, half);
                const float a = ptx::ex2(sm.b[s][row]);
                ptx::tc_fence_before_sync();
                ptx::mbar_arrive_warp(&sm.p_ready[s]);
                if (it.i == 0) grid_wait();
                if (dot) SF_WAIT(&sm.e_full[s], it.phase(), DEV_TIMEOUT_TMA);
                SF_WAIT(&sm.out_done[s], it.phase(), DEV_TIMEOUT_MMA);       // all of the tile's masks and row weights have been read
                ptx::tc_fence_after_sync();
                const float x = epilogue_tile(tmem + T_INTER, tmem + T_INTRA, sm.tiles[s][2], sm.tiles[s][0], a, half, dot, [&] {
                    ptx::tc_fence_before_sync();
                    ptx::mbar_arrive_warp(&sm.o_free[s]);
                });
                if (dot) (half ? sm.b : sm.u)[s][row] = x;
                ptx::fence_proxy_async();
                ptx::mbar_arrive_warp(&sm.staged[s]);
            }
        } else {
            const float* S0 = p.single ? (s_init ? s_init + bh * (D * D) : nullptr) : states + (bh * p.NB + j) * (long long)(D * D);
            grid_wait();
            state_init<4>(tmem + T_ST, S0, dot, 4 * wg);
            int last_s = 0;
            uint32_t last_ph = 0;
            for (; it.more(); it.next()) {
                const int s = it.stage();
                SF_WAIT(&sm.tab_full[s], it.phase(), DEV_TIMEOUT_MMA);
                float* dump = nullptr;                   // merged launches: the state entering a segment's first chunk goes out
                if (!BWD && it.c == 0 && p.single && p.s_copy) dump = p.s_copy + bh * (D * D);
                else if (!BWD && p.bslot) {
                    const int slot = __ldcg(p.bslot + c0 + it.c);
                    if (slot >= 0) dump = p.bbase + slot * p.bstride + bh * (D * D);
                }
                if (it.i > 0) SF_WAIT(&sm.st_done[s ^ 1], (uint32_t)((it.i - 1) >> 1) & 1, DEV_TIMEOUT_MMA);
                ptx::tc_fence_after_sync();
                const float total = sm.total[s];
                if (dump) state_out<4>(tmem + T_ST, dump, 4 * wg);
                state_pass<4>(tmem + T_ST, sm.sb, ptx::ex2(total), 4 * wg);
                ptx::fence_proxy_async();
                ptx::tc_fence_before_sync();
                ptx::mbar_arrive_warp(&sm.st_ready[s]);
                SF_WAIT(&sm.full_xy[s], it.phase(), DEV_TIMEOUT_TMA);
                SF_WAIT(&sm.sc_done[s], it.phase(), DEV_TIMEOUT_MMA);
                scale_rows(sm.tiles[s][1], tid, [&](int row) { return ptx::ex2(total - sm.b[s][row]); });
                ptx::fence_proxy_async();
                ptx::mbar_arrive_warp(&sm.y_ready[s]);
                last_s = s; last_ph = it.phase();
            }
            if ((!BWD || role == SWEEP_DV) && p.single) {       // the state (gradient) leaving the segment
                SF_WAIT(&sm.st_done[last_s], last_ph, DEV_TIMEOUT_MMA);
                ptx::tc_fence_after_sync();
                state_out<4>(tmem + T_ST, p.s_final + bh * (D * D), 4 * wg);
            }
        }
    }
    ptx::tc_fence_before_sync();
    __syncthreads();
    if (warp == W_MMA) ptx::tmem_dealloc(tmem, 512);
}

// grid (H, NB, B): heads fastest, so that co-resident CTAs read neighbouring 256-byte pieces of the same tokens
__global__ void __launch_bounds__(SW_THREADS, 1)
tc_forward_kernel(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmK, const __grid_constant__ CUtensorMap tmV,
                  const __grid_constant__ CUtensorMap tmO, SegParams p, const float* __restrict__ g, const float* Hs) {
    sweep_body<false>(SWEEP_O, {&tmQ, &tmK, &tmV, &tmQ, &tmO}, p, g, Hs, p.s_init, nullptr, blockIdx.x, blockIdx.y);
}

// The backward's sweeps, any consecutive ones in one launch: grid (heads x sweeps, NB, B).  dk and dv of a block are neighbours:
// they walk the same tokens at the same pace and read q and dO once from DRAM between them (8192 tokens x 32 heads: 285 MB read, the four inputs
// are 268 MB).
struct BwdMaps { CUtensorMap q, k, v, dO, dq, dk, dv; };
struct BwdArgs {
    const float *Hs, *Gs;
    const float *h_init, *g_init;                // one-block segments: the entering state, the gradient of the leaving state
    float *xq, *xk;
    int first, count;                            // sweeps first .. first + count - 1
};
__global__ void __launch_bounds__(SW_THREADS, 1)
tc_backward_kernel(const __grid_constant__ BwdMaps m, SegParams p, const float* __restrict__ g, BwdArgs a) {
    const int h = blockIdx.x / a.count, role = a.first + blockIdx.x % a.count, j = blockIdx.y;
    const bool dq = role == SWEEP_DQ, dk = role == SWEEP_DK;
    const SweepMaps maps{dq ? &m.dO : dk ? &m.v : &m.k, dq ? &m.v : dk ? &m.dO : &m.q, dq ? &m.k : dk ? &m.q : &m.dO, dq ? &m.q : &m.k,
                         dq ? &m.dq : dk ? &m.dk : &m.dv};
    sweep_body<true>(role, maps, p, g, dq ? a.Hs : a.Gs, dq ? a.h_init : a.g_init, dq ? a.xq : a.xk, h, j);
}

// Self-test of the bounded wait: one warp waits on a barrier on which nothing ever arrives, with a short limit given by
// the caller; the wait gives up, records DEV_TIMEOUT_SELFTEST in the status word and the kernel returns normally.
__global__ void wait_selftest_kernel(long long limit_cycles) {
    __shared__ uint64_t bar;
    __shared__ int abort_flag;
    if (threadIdx.x == 0) {
        abort_flag = 0;
        ptx::mbar_init(&bar, 1);
        ptx::fence_mbar_init();
    }
    __syncthreads();
    ptx::mbar_wait_limit<false>(ptx::smem_u32(&bar), 0, ptx::smem_u32(&abort_flag), DEV_TIMEOUT_SELFTEST, limit_cycles);
}

// ---- host launch -------------------------------------------------------------------------------------
// Per-device host state: whether the kernels' shared-memory attribute has been set there (it belongs to a device, not to the
// process).
constexpr int MAX_DEVICES = 64;
enum { K_AGG = 0, K_FWD, K_BWD, K_COUNT };
struct DeviceState {
    bool attr_done[K_COUNT] = {};
};
inline DeviceState* device_state() {
    static DeviceState table[MAX_DEVICES];
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= MAX_DEVICES) { cudaGetLastError(); return nullptr; }
    return &table[dev];
}
template <typename K>
inline bool opt_in_smem(DeviceState* d, int which, K kern, size_t bytes) {
    static std::mutex mu;
    std::lock_guard<std::mutex> lk(mu);
    if (d->attr_done[which]) return true;
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes) != cudaSuccess) { cudaGetLastError(); return false; }
    d->attr_done[which] = true;
    return true;
}

inline bool map_qk(CUtensorMap* m, int rows, const SegParams& p, const void* base) { return make_tmap(m, rows, base, p.B, p.L, p.H, p.tqk, p.bqk); }
inline bool map_v(CUtensorMap* m, int rows, const SegParams& p, const void* base) { return make_tmap(m, rows, base, p.B, p.L, p.H, p.tv, p.bv); }
inline sf_status_t launched(bool ok) {
    if (!ok) cudaGetLastError();
    return ok ? SF_OK : SF_ERR_CUDA;
}

inline sf_status_t launch_wait_selftest(long long limit_cycles, cudaStream_t st) {
    wait_selftest_kernel<<<1, 32, 0, st>>>(limit_cycles);
    return cudaGetLastError() == cudaSuccess ? SF_OK : SF_ERR_CUDA;
}

// Block aggregates: mode 0 of (k, v), mode 1 of (q, dO); early: launch_after()
inline sf_status_t launch_aggregate(const SegParams& p, const void* x, const void* y, const float* g, int mode, float* U, float* beta, bool early,
                                    cudaStream_t st) {
    DeviceState* ds = device_state();
    if (!ds) return SF_ERR_CUDA;
    if (p.R > MAXR) return SF_ERR_UNSUPPORTED;
    CUtensorMap tmX, tmY;
    if (!map_qk(&tmX, C, p, x) || !map_v(&tmY, C, p, y)) return SF_ERR_CUDA;
    constexpr size_t smem = sizeof(AggSmem) + 1024;
    if (!opt_in_smem(ds, K_AGG, tc_aggregate_kernel, smem)) return SF_ERR_CUDA;
    return launched(launch_after(early, tc_aggregate_kernel, dim3(p.H, p.NB, p.B), AGG_THREADS, smem, st, tmX, tmY, p, g, mode, U, beta));
}
inline sf_status_t launch_forward(const SegParams& p, const void* q, const void* k, const void* v, const float* g, const float* Hs, void* o, bool early,
                                  cudaStream_t st) {
    DeviceState* ds = device_state();
    if (!ds) return SF_ERR_CUDA;
    if (p.R > MAXR) return SF_ERR_UNSUPPORTED;
    CUtensorMap tq, tk, tv, to;
    if (!map_qk(&tq, TT, p, q) || !map_qk(&tk, TT, p, k) || !map_v(&tv, TT, p, v) || !map_v(&to, C, p, o)) return SF_ERR_CUDA;
    if (!opt_in_smem(ds, K_FWD, tc_forward_kernel, sizeof(SweepSmem))) return SF_ERR_CUDA;
    return launched(launch_after(early, tc_forward_kernel, dim3(p.H, p.NB, p.B), SW_THREADS, sizeof(SweepSmem), st, tq, tk, tv, to, p, g, Hs));
}
// a.first, a.count: which of the backward's sweeps; the output pointers of the others may be NULL, their maps are left blank
inline sf_status_t launch_backward(const SegParams& p, const void* q, const void* k, const void* v, const void* dO, const float* g, void* dq, void* dk,
                                   void* dv, const BwdArgs& a, bool early, cudaStream_t st) {
    DeviceState* ds = device_state();
    if (!ds) return SF_ERR_CUDA;
    if (p.R > MAXR) return SF_ERR_UNSUPPORTED;
    auto runs = [&](int sweep) { return sweep >= a.first && sweep < a.first + a.count; };
    BwdMaps m{};
    if (!map_qk(&m.q, TT, p, q) || !map_qk(&m.k, TT, p, k) || !map_v(&m.v, TT, p, v) || !map_v(&m.dO, TT, p, dO) ||
        (runs(SWEEP_DQ) && !map_qk(&m.dq, C, p, dq)) || (runs(SWEEP_DK) && !map_qk(&m.dk, C, p, dk)) || (runs(SWEEP_DV) && !map_v(&m.dv, C, p, dv)))
        return SF_ERR_CUDA;
    if (!opt_in_smem(ds, K_BWD, tc_backward_kernel, sizeof(SweepSmem))) return SF_ERR_CUDA;
    return launched(launch_after(early, tc_backward_kernel, dim3(p.H * a.count, p.NB, p.B), SW_THREADS, sizeof(SweepSmem), st, m, p, g, a));
}

}  // namespace tc
}  // namespace sf

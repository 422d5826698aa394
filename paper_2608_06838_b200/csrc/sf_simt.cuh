// CUDA-core (SIMT) kernels of the chunkwise gated linear recurrence: the float32 mode and the
// small-head bf16 shapes.  One CTA per (batch, head, block); tiles and the d_k x d_v state live in
// shared memory as float32, products are register-tiled (sf_tile.cuh).
//
// Algebra per tile of CT = 64 tokens (b_r = inclusive cumulative log-decay inside the tile, b_C its total,
// D[r,s] = exp(b_r - b_s) for s <= r, H_c the state entering the tile; paper Eq. 2 with
// V_new = {} specialised to F_t = exp(g_t) I):
//   Pre : A = (Q K^T) * D
//   Out : O = A V + diag(exp(b)) Q H_c
//   ST  : H_{c+1} = exp(b_C) H_c + sum_s exp(b_C - b_s) k_s^T v_s
// and the adjoint stages named in Section 3.4 (SR, OG, STB, PG):
//   OG  : dA = (dO V^T) * D ;  dq = dA K + diag(exp(b)) dO H_c^T
//   STB : dH_c = exp(b_C) dH_{c+1} + sum_r exp(b_r) q_r^T dO_r
//   PG  : dk = dA^T Q + diag(w) V dH_{c+1}^T ;  dv = A^T dO + diag(w) K dH_{c+1},  w_s = exp(b_C - b_s)
// The tile is the kernels' own: a block of chunks_per_block * chunk tokens is walked in tiles of 64 whatever the chunk.
// Every exponent is a sum of g over a token range (never a difference of long prefix sums), so all weights are <= 1 for
// g <= 0 and nothing overflows; differences of the tile's prefix sums are taken on float pairs (sums in double).
//
// What bounds these kernels: the FMA pipe (about 205 k multiply-adds per token and head forward + backward at d = 128, 70 k
// at d = 64, against 2.8 / 1.4 KB of memory traffic; 35 T multiply-adds/s were measured from registers alone).  A thread
// therefore owns 16 to 64 outputs of a product and feeds four multiply-adds per operand word read from shared memory.  Chains
// forward + backward, before (one output and one scalar inner product at a time) and now: float32 d = 128, 8144 tokens x 16
// heads 11.4 -> 1.58 ms (17 T multiply-adds/s); bf16 d = 64, 16384 tokens x 16 heads 5.92 -> 0.99 ms (18 T).
#pragma once
#include "sf_common.cuh"
#include "sf_tile.cuh"

namespace sf {
namespace simt {

constexpr int CT = 64;         // tokens per tile
constexpr int MAXR = 64;       // largest chunks_per_block
constexpr int MAXC = 64;       // largest chunk

// 8 warps; 4 for 32-wide keys, whose products have too few outputs for more.
template <int DK> constexpr int kThreads = DK == 32 ? 128 : 256;
// CTAs that share an SM in the sweeps: as many as the shared memory of the dk/dv sweep allows.
template <int DK> constexpr int kPerSM = DK == 128 ? 1 : (DK == 64 ? 2 : 3);

struct Decay {
    float bh[CT], bl[CT];      // inclusive cumulative log-decay as a float pair
    float wsuf[CT];            // exp(sum_{u>r} g_u)
    float ebc[CT];             // exp(sum_{u<=r} g_u)
};
// Tables of the tile whose `valid` tokens start at g (token stride tg), by warp 0.  A tile with fewer than CT tokens
// counts as if padded with zero rows of log-decay 0, which changes no sum; its missing rows are never stored.
__device__ __forceinline__ void tile_decay(Decay& d, const float* __restrict__ g, long long tg, int valid) {
    if (threadIdx.x >= 32) return;
    const int l = threadIdx.x, r0 = 2 * l, r1 = r0 + 1;
    const double g0 = r0 < valid ? (double)g[r0 * tg] : 0.0, g1 = r1 < valid ? (double)g[r1 * tg] : 0.0;
    double incl = g0 + g1;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const double up = __shfl_up_sync(0xffffffffu, incl, off);
        if (l >= off) incl += up;
    }
    const double tot = __shfl_sync(0xffffffffu, incl, 31);
    const double b[2] = {incl - g1, incl};
#pragma unroll
    for (int e = 0; e < 2; ++e) {
        const float hi = (float)b[e];
        d.bh[r0 + e] = hi;
        d.bl[r0 + e] = (float)(b[e] - (double)hi);
        d.wsuf[r0 + e] = __expf((float)(tot - b[e]));
        d.ebc[r0 + e] = __expf(hi);
    }
}

// out[r][s] = (x_r . y_s) exp(b_r - b_s) for s <= r, else 0; D = width of x and y.  Products of warps that lie wholly above
// the diagonal are left out: the triangular products below never read there.
template <int D, int NT>
__device__ __forceinline__ void masked_scores(float* out, const float* Xs, const float* Ys, const Decay& d) {
    const tile::Map<CT, CT, NT> mp;
    if (mp.TN == 4 && 4 * (mp.tx & ~7) > mp.warp_m0() + 15) return;
    float acc[mp.TM][mp.TN];
    tile::zero<decltype(mp)>(acc);
    tile::product<tile::Map<CT, CT, NT>, true, true, D, D>(acc, Xs, Ys, 0, D, mp);
#pragma unroll
    for (int i = 0; i < mp.TM; ++i) {
        const int r = mp.m(i);
        const float bh = d.bh[r], bl = d.bl[r];
#pragma unroll
        for (int gq = 0; gq < mp.GN; ++gq) {
            const int s0 = mp.n4(gq);
            float v[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int s = s0 + j;
                v[j] = s <= r ? acc[i][4 * gq + j] * __expf((bh - d.bh[s]) + (bl - d.bl[s])) : 0.f;
            }
            tile::st4(out + tile::at<CT>(r, s0), make_float4(v[0], v[1], v[2], v[3]));
        }
    }
}

// S <- decay S + X^T Y over the tile's tokens (X [CT][DK], Y [CT][DV], the weights already applied to one of them)
template <int DK, int DV, int NT>
__device__ __forceinline__ void state_update(float* S, const float* Xs, const float* Ys, float decay) {
    const tile::Map<DK, DV, NT> mp;
    if (!mp.on) return;
    float acc[mp.TM][mp.TN];
#pragma unroll
    for (int i = 0; i < mp.TM; ++i)
#pragma unroll
        for (int gq = 0; gq < mp.GN; ++gq) {
            const float4 v = tile::ld4(S + tile::at<DV>(mp.m(i), mp.n4(gq)));
            acc[i][4 * gq] = decay * v.x; acc[i][4 * gq + 1] = decay * v.y; acc[i][4 * gq + 2] = decay * v.z; acc[i][4 * gq + 3] = decay * v.w;
        }
    tile::product<tile::Map<DK, DV, NT>, false, false, DK, DV>(acc, Xs, Ys, 0, CT, mp);
#pragma unroll
    for (int i = 0; i < mp.TM; ++i)
#pragma unroll
        for (int gq = 0; gq < mp.GN; ++gq)
            tile::st4(S + tile::at<DV>(mp.m(i), mp.n4(gq)),
                      make_float4(acc[i][4 * gq], acc[i][4 * gq + 1], acc[i][4 * gq + 2], acc[i][4 * gq + 3]));
}

template <class Mp>
__device__ __forceinline__ void scale_acc(float (&acc)[Mp::TM][Mp::TN], const Mp& mp, const float* w) {
#pragma unroll
    for (int i = 0; i < Mp::TM; ++i) {
        const float f = w[mp.m(i)];
#pragma unroll
        for (int j = 0; j < Mp::TN; ++j) acc[i][j] *= f;
    }
}
// rows m < valid of the accumulator to global rows `stride` elements apart
template <class Mp, typename T>
__device__ __forceinline__ void store_acc(T* __restrict__ dst, long long stride, int valid, const float (&acc)[Mp::TM][Mp::TN], const Mp& mp) {
#pragma unroll
    for (int i = 0; i < Mp::TM; ++i) {
        const int r = mp.m(i);
        if (r < valid)
#pragma unroll
            for (int gq = 0; gq < Mp::GN; ++gq)
                tile::store4(dst + r * stride + mp.n4(gq),
                             make_float4(acc[i][4 * gq], acc[i][4 * gq + 1], acc[i][4 * gq + 2], acc[i][4 * gq + 3]));
    }
}
// Row dot products of the accumulator with e(m, n4) (four elements), summed over the row's threads in a fixed order:
// butterfly over the eight lanes of a warp that share the row, then over the warps through `red` [CT][WX].
template <class Mp, typename F>
__device__ __forceinline__ void row_dots(const float (&acc)[Mp::TM][Mp::TN], const Mp& mp, float* red, F e) {
    constexpr int WX = Mp::TXN / 8;
#pragma unroll
    for (int i = 0; i < Mp::TM; ++i) {
        float s = 0.f;
#pragma unroll
        for (int gq = 0; gq < Mp::GN; ++gq) {
            const float4 v = e(mp.m(i), mp.n4(gq));
            s = fmaf(acc[i][4 * gq], v.x, s); s = fmaf(acc[i][4 * gq + 1], v.y, s);
            s = fmaf(acc[i][4 * gq + 2], v.z, s); s = fmaf(acc[i][4 * gq + 3], v.w, s);
        }
        s = tile::sum_x(s);
        if ((mp.tx & 7) == 0) red[mp.m(i) * WX + (mp.tx >> 3)] = s;
    }
}
template <int WX>
__device__ __forceinline__ void store_dots(float* __restrict__ x, const float* red, int valid) {
    for (int r = threadIdx.x; r < valid; r += blockDim.x) {
        float s = red[r * WX];
#pragma unroll
        for (int w = 1; w < WX; ++w) s += red[r * WX + w];
        x[r] = s;
    }
}

// ------------------------------------------------------------------------------------------------
// Block aggregates (the chunk-parallel part of Pre that feeds ST, and of STB):
//   mode 0: U = sum_s exp(beta - B_s) x_s^T y_s   with (x, y) = (k, v)   [forward aggregate]
//   mode 1: U = sum_s exp(B_s)        x_s^T y_s   with (x, y) = (q, dO)  [backward aggregate]
// B_s = inclusive cumulative log-decay from the block start, beta = block total (written to beta_out).
template <int DK, int DV>
struct AggSmem {
    float X[CT * DK], Y[CT * DV];
    float w[MAXR * MAXC];
    double tot[MAXR * MAXC / CT], ofs[MAXR * MAXC / CT];
};
template <typename T, int DK, int DV>
__global__ void __launch_bounds__(kThreads<DK>, 2) block_aggregate_kernel(SegParams p, const T* __restrict__ X, const T* __restrict__ Y,
                                                                           const float* __restrict__ g, int mode,
                                                                           float* __restrict__ U, float* __restrict__ beta_out) {
    constexpr int NT = kThreads<DK>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    AggSmem<DK, DV>& sm = *reinterpret_cast<AggSmem<DK, DV>*>(smem_raw);
    const int j = blockIdx.x, h = blockIdx.y, b = blockIdx.z;
    const int t_begin = j * p.R * p.C, t_end = min(p.L, t_begin + p.R * p.C), ntile = (t_end - t_begin + CT - 1) / CT;
    const float* gh = g + (long long)b * p.bg + h;
    const T* Xh = X + (long long)b * p.bqk + (long long)h * DK;
    const T* Yh = Y + (long long)b * p.bv + (long long)h * DV;

    // per tile, one warp: mode 0 the sum of g after the token inside the tile, mode 1 up to and with it
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (int c = warp; c < ntile; c += NT / 32) {
        const int r0 = t_begin + c * CT + 2 * lane, r1 = r0 + 1;
        const double g0 = r0 < t_end ? (double)gh[r0 * p.tg] : 0.0, g1 = r1 < t_end ? (double)gh[r1 * p.tg] : 0.0;
        double incl = g0 + g1;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const double up = __shfl_up_sync(0xffffffffu, incl, off);
            if (lane >= off) incl += up;
        }
        const double tot = __shfl_sync(0xffffffffu, incl, 31);
        sm.w[c * CT + 2 * lane] = (float)(mode == 0 ? tot - (incl - g1) : incl - g1);
        sm.w[c * CT + 2 * lane + 1] = (float)(mode == 0 ? tot - incl : incl);
        if (lane == 0) sm.tot[c] = tot;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        double acc = 0.0;
        if (mode == 0) { for (int c = ntile - 1; c >= 0; --c) { sm.ofs[c] = acc; acc += sm.tot[c]; } }
        else           { for (int c = 0; c < ntile; ++c)      { sm.ofs[c] = acc; acc += sm.tot[c]; } }
        if (beta_out) beta_out[((long long)b * p.H + h) * p.NB + j] = (float)acc;
    }
    __syncthreads();
    for (int i = threadIdx.x; i < ntile * CT; i += NT) sm.w[i] = __expf((float)((double)sm.w[i] + sm.ofs[i / CT]));

    const tile::Map<DK, DV, NT> mp;
    float acc[mp.TM][mp.TN];
    tile::zero<tile::Map<DK, DV, NT>>(acc);
    for (int c = 0; c < ntile; ++c) {
        const int t0 = t_begin + c * CT, valid = min(CT, t_end - t0);
        __syncthreads();
        tile::load_scaled<CT, DK, NT>(sm.X, Xh + t0 * p.tqk, p.tqk, valid, sm.w + c * CT);
        tile::load<CT, DV, NT>(sm.Y, Yh + t0 * p.tv, p.tv, valid);
        __syncthreads();
        if (mp.on) tile::product<tile::Map<DK, DV, NT>, false, false, DK, DV>(acc, sm.X, sm.Y, 0, CT, mp);
    }
    if (mp.on) store_acc(U + (((long long)b * p.H + h) * p.NB + j) * (long long)(DK * DV), DV, DK, acc, mp);
}

// S (swizzled tile) from a dense [DK][DV] state
template <int DK, int DV, int NT>
__device__ __forceinline__ void load_state(float* S, const float* __restrict__ src) { tile::load<DK, DV, NT>(S, src, DV, DK); }

// ------------------------------------------------------------------------------------------------
// Forward output pass (Out and ST of paper Eq. 2 inside one block): from the block-entering state
// Hs[j], for each tile O = A V + diag(exp(b)) Q H_c, then H_{c+1} (left out after the block's last tile).
template <int DK, int DV>
struct FwdSmem {
    float Q[CT * DK], K[CT * DK], V[CT * DV], A[CT * CT], S[DK * DV];
    Decay d;
};
template <typename T, int DK, int DV>
__global__ void __launch_bounds__(kThreads<DK>, kPerSM<DK>) fwd_out_kernel(SegParams p, const T* __restrict__ q, const T* __restrict__ k,
                                                                const T* __restrict__ v, const float* __restrict__ g,
                                                                const float* __restrict__ Hs, T* __restrict__ o) {
    constexpr int NT = kThreads<DK>;
    using MO = tile::Map<CT, DV, NT>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    FwdSmem<DK, DV>& sm = *reinterpret_cast<FwdSmem<DK, DV>*>(smem_raw);
    const int j = blockIdx.x, h = blockIdx.y, b = blockIdx.z;
    const int t_begin = j * p.R * p.C, t_end = min(p.L, t_begin + p.R * p.C);
    const long long qk_off = (long long)b * p.bqk + (long long)h * DK;
    const long long v_off = (long long)b * p.bv + (long long)h * DV;
    const float* gh = g + (long long)b * p.bg + h;
    load_state<DK, DV, NT>(sm.S, Hs + (((long long)b * p.H + h) * p.NB + j) * (long long)(DK * DV));
    const MO mo;
    for (int t0 = t_begin; t0 < t_end; t0 += CT) {
        const int valid = min(CT, t_end - t0);
        tile_decay(sm.d, gh + t0 * p.tg, p.tg, valid);
        tile::load<CT, DK, NT>(sm.Q, q + qk_off + t0 * p.tqk, p.tqk, valid);
        tile::load<CT, DK, NT>(sm.K, k + qk_off + t0 * p.tqk, p.tqk, valid);
        tile::load<CT, DV, NT>(sm.V, v + v_off + t0 * p.tv, p.tv, valid);
        __syncthreads();
        masked_scores<DK, NT>(sm.A, sm.Q, sm.K, sm.d);
        float acc[MO::TM][MO::TN];
        tile::zero<MO>(acc);
        tile::product<MO, true, false, DK, DV>(acc, sm.Q, sm.S, 0, DK, mo);
        scale_acc(acc, mo, sm.d.ebc);
        __syncthreads();
        tile::product<MO, true, false, CT, DV>(acc, sm.A, sm.V, 0, mo.warp_m0() + 16, mo);
        store_acc(o + v_off + t0 * p.tv, p.tv, valid, acc, mo);
        if (t0 + CT < t_end) {
            tile::scale_rows<CT, DK, NT>(sm.K, sm.d.wsuf);
            __syncthreads();
            state_update<DK, DV, NT>(sm.S, sm.K, sm.V, sm.d.ebc[CT - 1]);
            __syncthreads();
        }
    }
}

// ------------------------------------------------------------------------------------------------
// dq pass (SR + OG): replays H_c inside the block from Hs[j]; dq = dA K + diag(exp(b)) dO H_c^T.
// Also emits xq[t] = q_t . dq_t from the float32 accumulators, a term of the log-decay gradient.
template <int DK, int DV>
struct DqSmem {
    float K[CT * DK], V[CT * DV], D[CT * DV], A[CT * CT], S[DK * DV];
    float red[CT * 2];
    Decay d;
};
template <typename T, int DK, int DV>
__global__ void __launch_bounds__(kThreads<DK>, kPerSM<DK>) bwd_dq_kernel(SegParams p, const T* __restrict__ q, const T* __restrict__ k,
                                                               const T* __restrict__ v, const float* __restrict__ g,
                                                               const T* __restrict__ dO, const float* __restrict__ Hs,
                                                               T* __restrict__ dq, float* __restrict__ xq) {
    constexpr int NT = kThreads<DK>;
    using MQ = tile::Map<CT, DK, NT>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    DqSmem<DK, DV>& sm = *reinterpret_cast<DqSmem<DK, DV>*>(smem_raw);
    const int j = blockIdx.x, h = blockIdx.y, b = blockIdx.z;
    const int t_begin = j * p.R * p.C, t_end = min(p.L, t_begin + p.R * p.C);
    const long long qk_off = (long long)b * p.bqk + (long long)h * DK;
    const long long v_off = (long long)b * p.bv + (long long)h * DV;
    const float* gh = g + (long long)b * p.bg + h;
    float* xqh = xq + ((long long)b * p.H + h) * p.L;
    load_state<DK, DV, NT>(sm.S, Hs + (((long long)b * p.H + h) * p.NB + j) * (long long)(DK * DV));
    const MQ mq;
    for (int t0 = t_begin; t0 < t_end; t0 += CT) {
        const int valid = min(CT, t_end - t0);
        tile_decay(sm.d, gh + t0 * p.tg, p.tg, valid);
        tile::load<CT, DK, NT>(sm.K, k + qk_off + t0 * p.tqk, p.tqk, valid);
        tile::load<CT, DV, NT>(sm.V, v + v_off + t0 * p.tv, p.tv, valid);
        tile::load<CT, DV, NT>(sm.D, dO + v_off + t0 * p.tv, p.tv, valid);
        __syncthreads();
        masked_scores<DV, NT>(sm.A, sm.D, sm.V, sm.d);                                  // dA
        float acc[MQ::TM][MQ::TN];
        tile::zero<MQ>(acc);
        tile::product<MQ, true, true, DV, DV>(acc, sm.D, sm.S, 0, DV, mq);              // dO H^T
        scale_acc(acc, mq, sm.d.ebc);
        __syncthreads();
        tile::product<MQ, true, false, CT, DK>(acc, sm.A, sm.K, 0, mq.warp_m0() + 16, mq);
        store_acc(dq + qk_off + t0 * p.tqk, p.tqk, valid, acc, mq);
        const T* qt = q + qk_off + t0 * p.tqk;
        row_dots(acc, mq, sm.red, [&](int r, int c) { return r < valid ? tile::load4(qt + r * p.tqk + c) : make_float4(0.f, 0.f, 0.f, 0.f); });
        const bool more = t0 + CT < t_end;
        if (more) tile::scale_rows<CT, DV, NT>(sm.V, sm.d.wsuf);
        __syncthreads();
        store_dots<MQ::TXN / 8>(xqh + t0, sm.red, valid);
        if (more) {
            state_update<DK, DV, NT>(sm.S, sm.K, sm.V, sm.d.ebc[CT - 1]);
            __syncthreads();
        }
    }
}

// ------------------------------------------------------------------------------------------------
// dk/dv pass (STB inside the block + PG): reverse sweep from Gs[j], the gradient w.r.t. the state
// leaving block j.  Also emits xk[t] = k_t . dk_t from the float32 accumulators.
template <int DK, int DV>
struct DkdvSmem {
    float Q[CT * DK], K[CT * DK], V[CT * DV], D[CT * DV], A[CT * CT], dA[CT * CT], G[DK * DV];
    Decay d;
};
template <typename T, int DK, int DV>
__global__ void __launch_bounds__(kThreads<DK>, kPerSM<DK>) bwd_dkdv_kernel(SegParams p, const T* __restrict__ q, const T* __restrict__ k,
                                                                 const T* __restrict__ v, const float* __restrict__ g,
                                                                 const T* __restrict__ dO, const float* __restrict__ Gs,
                                                                 T* __restrict__ dk, T* __restrict__ dv, float* __restrict__ xk) {
    constexpr int NT = kThreads<DK>;
    using MK = tile::Map<CT, DK, NT>;
    using MV = tile::Map<CT, DV, NT>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    DkdvSmem<DK, DV>& sm = *reinterpret_cast<DkdvSmem<DK, DV>*>(smem_raw);
    const int j = blockIdx.x, h = blockIdx.y, b = blockIdx.z;
    const int t_begin = j * p.R * p.C, t_end = min(p.L, t_begin + p.R * p.C), ntile = (t_end - t_begin + CT - 1) / CT;
    const long long qk_off = (long long)b * p.bqk + (long long)h * DK;
    const long long v_off = (long long)b * p.bv + (long long)h * DV;
    const float* gh = g + (long long)b * p.bg + h;
    float* xkh = xk + ((long long)b * p.H + h) * p.L;
    load_state<DK, DV, NT>(sm.G, Gs + (((long long)b * p.H + h) * p.NB + j) * (long long)(DK * DV));
    const MK mk;
    const MV mv;
    for (int c = ntile - 1; c >= 0; --c) {
        const int t0 = t_begin + c * CT, valid = min(CT, t_end - t0);
        tile_decay(sm.d, gh + t0 * p.tg, p.tg, valid);
        tile::load<CT, DK, NT>(sm.Q, q + qk_off + t0 * p.tqk, p.tqk, valid);
        tile::load<CT, DK, NT>(sm.K, k + qk_off + t0 * p.tqk, p.tqk, valid);
        tile::load<CT, DV, NT>(sm.V, v + v_off + t0 * p.tv, p.tv, valid);
        tile::load<CT, DV, NT>(sm.D, dO + v_off + t0 * p.tv, p.tv, valid);
        __syncthreads();
        masked_scores<DK, NT>(sm.A, sm.Q, sm.K, sm.d);             // A  = (Q K^T) * D
        masked_scores<DV, NT>(sm.dA, sm.D, sm.V, sm.d);            // dA = (dO V^T) * D
        float av[MV::TM][MV::TN], ak[MK::TM][MK::TN];
        tile::zero<MV>(av);
        tile::product<MV, true, false, DK, DV>(av, sm.K, sm.G, 0, DK, mv);              // K G
        scale_acc(av, mv, sm.d.wsuf);
        tile::zero<MK>(ak);
        tile::product<MK, true, true, DV, DV>(ak, sm.V, sm.G, 0, DV, mk);               // V G^T
        scale_acc(ak, mk, sm.d.wsuf);
        __syncthreads();
        tile::product<MV, false, false, CT, DV>(av, sm.A, sm.D, mv.warp_m0(), CT, mv);  // A^T dO, rows r >= s only
        store_acc(dv + v_off + t0 * p.tv, p.tv, valid, av, mv);
        tile::product<MK, false, false, CT, DK>(ak, sm.dA, sm.Q, mk.warp_m0(), CT, mk);
        store_acc(dk + qk_off + t0 * p.tqk, p.tqk, valid, ak, mk);
        row_dots(ak, mk, sm.V, [&](int r, int cc) { return tile::ld4(sm.K + tile::at<DK>(r, cc)); });      // V has served
        __syncthreads();
        store_dots<MK::TXN / 8>(xkh + t0, sm.V, valid);
        if (c > 0) {                                               // STB: G <- exp(bC) G + (diag(exp(b)) Q)^T dO
            tile::scale_rows<CT, DK, NT>(sm.Q, sm.d.ebc);
            __syncthreads();
            state_update<DK, DV, NT>(sm.G, sm.Q, sm.D, sm.d.ebc[CT - 1]);
            __syncthreads();
        }
    }
}

}  // namespace simt
}  // namespace sf

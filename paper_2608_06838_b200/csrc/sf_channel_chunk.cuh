// Chunkwise form of the diagonal-decay recurrence (paper Section 2.1, diagonal F_t; Section 2.2, Eq. 2 with an empty
// V_new): float32 CUDA-core kernels.
//
// Token rule: S_t = diag(exp(g_t)) S_{t-1} + k_t^T v_t,  o_t = q_t S_t,  g_t one log-decay per key channel.  Within a tile
// of n tokens, with b_t[i] the inclusive cumulative log-decay of channel i, gam = exp(b), om_s = exp(b_n - b_s), H the
// entering state:
//     A[t,s] = sum_i q_t[i] k_s[i] exp(b_t[i] - b_s[i])  (s <= t)      O = A V + (q*gam) H
//     H' = diag(gam_n) H + (om*K)^T V                                   (an affine map with a diagonal linear part)
//     Pre : Psi = (om*K)^T V and gam_n per tile (and, for the backward, Theta = (q*gam)^T dO)         all tiles in parallel
//     ST  : H' = gam_n * H + Psi element by element, storing the state entering every tile             sequential, one thread per element
//     Out : A, O                                                                                       all tiles in parallel
// Backward (hand-derived, checked against the fp64 oracle), dH' = gradient of the state leaving the tile:
//     dH = gam_n * dH' + Theta                                                                         the same kernel as ST, reversed
//     dv = A^T dO + (om*K) dH',   dA = lower(dO V^T),
//     dq[t,i] = sum_{s<=t} dA[t,s] k_s[i] exp(b_t[i]-b_s[i]) + gam_t[i] (dO H^T)[t,i]
//     dk[s,i] = sum_{t>=s} dA[t,s] q_t[i] exp(b_t[i]-b_s[i]) + om_s[i] (V dH'^T)[s,i]
//     dg_t[i] = sum_{u>=t in the tile} (q_u[i] dq_u[i] - k_u[i] dk_u[i]) + <dH'[i,:], H'[i,:]>            (rows of S are independent
//               scalar recurrences, so the per-row identity dg_t = dg_{t+1} + q dq - k dk holds and is anchored per tile)
//
// The decay sits inside the channel sums of A, dq and dk; an exponential per (token, token, channel) would cost more than
// all products together (32 tokens x 64 channels: 32 k exponentials per tile and sum).  Instead the tile of 32 tokens is halved
// three times: for t in the upper and s in the lower half of a (sub-)block the exponent splits at the boundary r between them,
//     exp(b_t - b_s) = exp(b_t - b_r) exp(b_r - b_s),      both factors <= 1 for g <= 0: nothing is ever divided by a decay,
// so with S_h[t] = q_t exp(b_t - b_r) on upper and S_h[s] = k_s exp(b_r - b_s) on lower rows (h = 16, 8, 4: one array per
// level) all pairs outside the eight diagonal 4 x 4 blocks are plain products of rows of S_h, in A and, with the same
// arrays, in dq and dk.  The diagonal blocks are done in registers: a thread owns 4 tokens x 4 channels and has the six
// weights of its block.  All exponents are local sums of g (never differences of prefix sums).
//
// The tile is 32 tokens whatever the caller's chunk (see the workspace).  A last tile's missing tokens count as zero rows
// with log-decay 0, which changes no sum.
#pragma once
#include "sf_common.cuh"
#include "sf_tile.cuh"

namespace sf {
namespace dcc {

constexpr int CT = 32;             // tokens per tile
constexpr int CC = CT * CT;

// 4 warps, 8 where a 128-wide side gives every product enough outputs.
template <int DK, int DV> constexpr int kThreads = DK == 128 || DV == 128 ? 256 : 128;

struct Params {
    int B, H, L, C, NC, dk, dv;              // C, NC: the caller's chunk (workspace rules)
    int NT;                                  // tiles
    bool vec;                                // rows allow accesses of four elements
    long long tqk, tv, tg, bqk, bv, bg;
};

// Workspace per (batch, head), in floats.  Its size is part of the interface: Psi [NC][dk][dv], gamn [NC][dk],
// Hc [NC+1][dk][dv] (the last one is the state leaving the segment); the backward adds Theta [NC][dk][dv] and dHc [NC][dk][dv].
// The kernels keep one of each per tile, and there are never more tiles than chunks.
struct Ws { float *Psi, *gamn, *Hc, *Theta, *dHc; };
__host__ __device__ inline size_t ws_floats(const Params& p, bool backward) {
    const size_t st = (size_t)p.dk * p.dv;
    size_t n = (size_t)p.NC * st + (size_t)p.NC * p.dk + (size_t)(p.NC + 1) * st;
    if (backward) n += 2 * (size_t)p.NC * st;
    return n;
}
__host__ __device__ inline Ws ws_of(float* base, const Params& p, long long bh, bool backward) {
    const size_t st = (size_t)p.dk * p.dv;
    float* c = base + bh * (long long)ws_floats(p, backward);
    Ws w;
    w.Psi = c;  c += (size_t)p.NT * st;
    w.gamn = c; c += (size_t)p.NT * p.dk;
    w.Hc = c;   c += (size_t)(p.NT + 1) * st;
    w.Theta = w.dHc = nullptr;
    if (backward) { w.Theta = c; c += (size_t)p.NT * st; w.dHc = c; }
    return w;
}

// A thread's 4 tokens x 4 channels (rows 4 ty .., channels 4 tx .. of a Map<CT, DK, NT>).
struct Quad { float v[4][4]; };
template <class Mp, typename T>
__device__ __forceinline__ Quad load_quad(const T* __restrict__ src, long long stride, int n, bool vec, const Mp& mp) {
    Quad q;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int r = mp.m(i);
        const float4 f = r < n ? tile::load4(src + r * stride + mp.n4(0), vec) : make_float4(0.f, 0.f, 0.f, 0.f);
        q.v[i][0] = f.x; q.v[i][1] = f.y; q.v[i][2] = f.z; q.v[i][3] = f.w;
    }
    return q;
}
template <int DK, class Mp>
__device__ __forceinline__ void put_quad(float* dst, const Quad& q, const Mp& mp) {
#pragma unroll
    for (int i = 0; i < 4; ++i) tile::st4(dst + tile::at<DK>(mp.m(i), mp.n4(0)), make_float4(q.v[i][0], q.v[i][1], q.v[i][2], q.v[i][3]));
}
// a * b * f, f one factor per channel
__device__ __forceinline__ Quad times(const Quad& a, const Quad& b, const float (&f)[4]) {
    Quad r;
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) r.v[i][j] = a.v[i][j] * b.v[i][j] * f[j];
    return r;
}
// exp of the sums of g inside the thread's four tokens: up to and with the token / after the token
__device__ __forceinline__ Quad exp_prefix(const Quad& g) {
    Quad r;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        float s = 0.f;
#pragma unroll
        for (int i = 0; i < 4; ++i) { s += g.v[i][j]; r.v[i][j] = __expf(s); }
    }
    return r;
}
__device__ __forceinline__ Quad exp_suffix(const Quad& g) {
    Quad r;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        float s = 0.f;
#pragma unroll
        for (int i = 3; i >= 0; --i) { r.v[i][j] = i == 3 ? 1.f : __expf(s); s += g.v[i][j]; }
    }
    return r;
}
// Totals of the eight four-token blocks per channel, in shared memory [8][DK]; exp of the sum of blocks [b0, b1).
template <int DK, class Mp>
__device__ __forceinline__ void put_total(float* tot, const Quad& g, const Mp& mp) {
    float s[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) s[j] = (g.v[0][j] + g.v[1][j]) + (g.v[2][j] + g.v[3][j]);
    tile::st4(tot + mp.ty * DK + mp.n4(0), make_float4(s[0], s[1], s[2], s[3]));
}
template <int DK, class Mp>
__device__ __forceinline__ void exp_blocks(float (&f)[4], const float* tot, int b0, int b1, const Mp& mp) {
    f[0] = f[1] = f[2] = f[3] = 0.f;
    for (int b = b0; b < b1; ++b) {
        const float4 t = tile::ld4(tot + b * DK + mp.n4(0));
        f[0] += t.x; f[1] += t.y; f[2] += t.z; f[3] += t.w;
    }
#pragma unroll
    for (int j = 0; j < 4; ++j) f[j] = __expf(f[j]);
}
// Block part of the factor of the thread's rows at level lb (half-size 4 << lb): exp of the sum of whole blocks from the
// boundary to the thread's block on upper rows, from after it to the boundary on lower ones.
template <int DK, class Mp>
__device__ __forceinline__ void level_blocks(float (&f)[4], const float* tot, int lb, const Mp& mp) {
    const int first = (mp.ty >> lb) << lb;                       // first block of the half that holds the thread's block
    if ((mp.ty >> lb) & 1) exp_blocks<DK>(f, tot, first, mp.ty, mp);
    else                   exp_blocks<DK>(f, tot, mp.ty + 1, first + (1 << lb), mp);
}
// S_h rows of the three levels; `ep`: exp_prefix, `es`: exp_suffix
template <int DK, class Mp>
__device__ __forceinline__ void put_levels(float* S, const Quad& q, const Quad& k, const Quad& ep, const Quad& es, const float* tot, const Mp& mp) {
#pragma unroll
    for (int lb = 0; lb < 3; ++lb) {
        float f[4];
        level_blocks<DK>(f, tot, lb, mp);
        const bool upper = (mp.ty >> lb) & 1;
        put_quad<DK>(S + lb * CT * DK, upper ? times(q, ep, f) : times(k, es, f), mp);
    }
}
// weights exp(b_t - b_s) inside the thread's block: e10, e21, e20 per channel; e32, e31, e30 are exp_suffix rows 2, 1, 0
struct Near { float e10[4], e21[4], e20[4]; };
__device__ __forceinline__ Near near_weights(const Quad& g) {
    Near w;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        w.e10[j] = __expf(g.v[1][j]);
        w.e21[j] = __expf(g.v[2][j]);
        w.e20[j] = __expf(g.v[1][j] + g.v[2][j]);
    }
    return w;
}
__device__ __forceinline__ float near_weight(const Near& w, const Quad& es, int t, int s, int j) {
    return t == s ? 1.f : (t == 3 ? es.v[s][j] : (t == 1 ? w.e10[j] : (s == 1 ? w.e21[j] : w.e20[j])));
}
// The diagonal 4 x 4 blocks of A: sums over the thread's channels, reduced over the eight lanes that share the tokens
// (reduce-scatter, two entries per lane) into red[ty][warp column][16], entry 4 t + s.
template <class Mp>
__device__ __forceinline__ void diag_partials(float* red, const Quad& q, const Quad& k, const Near& nw, const Quad& es, const Mp& mp) {
    float v[16];
#pragma unroll
    for (int t = 0; t < 4; ++t)
#pragma unroll
        for (int s = 0; s < 4; ++s) {
            float a = 0.f;
            if (s <= t)
#pragma unroll
                for (int j = 0; j < 4; ++j) a = fmaf(q.v[t][j] * k.v[s][j], near_weight(nw, es, t, s, j), a);
            v[4 * t + s] = a;
        }
    // over tx bits 2, 1, 0 = lane bits 4, 3, 1
    const int tx = mp.tx & 7;
#pragma unroll
    for (int b = 0, width = 16; b < 3; ++b, width >>= 1) {
        const int mask = b == 0 ? 16 : (b == 1 ? 8 : 2);
        const bool up = (tx >> (2 - b)) & 1;
#pragma unroll
        for (int e = 0; e < 8; ++e)
            if (e < width / 2) {
                const float keep = up ? v[e + width / 2] : v[e], give = up ? v[e] : v[e + width / 2];
                v[e] = keep + __shfl_xor_sync(0xffffffffu, give, mask);
            }
    }
    constexpr int WX = Mp::TXN / 8;
    *reinterpret_cast<float2*>(red + (mp.ty * WX + (mp.tx >> 3)) * 16 + 2 * tx) = make_float2(v[0], v[1]);
}
// A [32][32] (zero above the diagonal) from the level arrays and the diagonal partials.  Off the diagonal, KS lanes share one
// 4 x 4 block over a KS-th of the channels each and add up by a reduce-scatter.
template <int DK, int NT, int WX>
__device__ __forceinline__ void assemble_scores(float* A, const float* S, const float* red) {
    constexpr int KS = NT / 32;                                  // 28 blocks x KS lanes <= NT
    const int pi = threadIdx.x / KS, ks = threadIdx.x % KS;
    int tb = 1;
    while (tb < 7 && (tb + 1) * tb / 2 <= pi) ++tb;
    const bool on = pi < 28;
    const int sb = on ? pi - tb * (tb - 1) / 2 : 0;
    const float* Sl = S + (31 - __clz(tb ^ sb)) * CT * DK;
    tile::f32x2 acc2[4][4] = {};
    if (on)
        for (int u = ks; u < DK / 4; u += KS) {
            const int ot = (u ^ tb) << 2, os = (u ^ sb) << 2;
            ulonglong2 y[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) y[j] = tile::ld4x2(Sl + (4 * sb + j) * DK + os);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const ulonglong2 x = tile::ld4x2(Sl + (4 * tb + i) * DK + ot);
#pragma unroll
                for (int j = 0; j < 4; ++j) { tile::fma2(acc2[i][j], x.x, y[j].x); tile::fma2(acc2[i][j], x.y, y[j].y); }
            }
        }
    float acc[16];
#pragma unroll
    for (int e = 0; e < 16; ++e) {
        float lo, hi;
        tile::unpack(acc2[e >> 2][e & 3], lo, hi);
        acc[e] = lo + hi;
    }
#pragma unroll
    for (int b = KS / 2, width = 16; b >= 1; b >>= 1, width >>= 1) {
        const bool up = (ks & b) != 0;
#pragma unroll
        for (int e = 0; e < 8; ++e)
            if (e < width / 2) {
                const float keep = up ? acc[e + width / 2] : acc[e], give = up ? acc[e] : acc[e + width / 2];
                acc[e] = keep + __shfl_xor_sync(0xffffffffu, give, b);
            }
    }
    if (on) {
        if constexpr (KS == 4) {
            tile::st4(A + tile::at<CT>(4 * tb + ks, 4 * sb), make_float4(acc[0], acc[1], acc[2], acc[3]));
            tile::st4(A + tile::at<CT>(4 * sb + ks, 4 * tb), make_float4(0.f, 0.f, 0.f, 0.f));
        } else {
            static_assert(KS == 8, "4 or 8 lanes per block");
            *reinterpret_cast<float2*>(A + tile::at<CT>(4 * tb + (ks >> 1), 4 * sb + 2 * (ks & 1))) = make_float2(acc[0], acc[1]);
            *reinterpret_cast<float2*>(A + tile::at<CT>(4 * sb + (ks >> 1), 4 * tb + 2 * (ks & 1))) = make_float2(0.f, 0.f);
        }
    }
    for (int i = threadIdx.x; i < 8 * 16; i += NT) {
        const int blk = i >> 4, e = i & 15;
        float s = red[blk * WX * 16 + e];
#pragma unroll
        for (int w = 1; w < WX; ++w) s += red[(blk * WX + w) * 16 + e];
        A[tile::at<CT>(4 * blk + (e >> 2), 4 * blk + (e & 3))] = s;
    }
}

// ---- Pre: Psi = (om*K)^T V, gam_n; with dO also Theta = (q*gam)^T dO.  grid (tiles, H, B) --------------------------------
// Bound by memory: it reads 2 (4) rows and g per token and writes one (two) states per 32 tokens.
template <int DK, int DV>
struct PreSmem {
    float X[CT * DK], Y[CT * DV], tot[8 * DK];
};
template <typename T, int DK, int DV>
__global__ void __launch_bounds__(kThreads<DK, DV>, kThreads<DK, DV> == 128 ? 5 : 2)
pre_kernel(Params p, const T* __restrict__ q, const T* __restrict__ k, const T* __restrict__ v, const float* __restrict__ g,
           const T* __restrict__ dO, float* ws, int backward) {
    constexpr int NT = kThreads<DK, DV>;
    using MK = tile::Map<CT, DK, NT>;
    using MS = tile::Map<DK, DV, NT>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    PreSmem<DK, DV>& sm = *reinterpret_cast<PreSmem<DK, DV>*>(smem_raw);
    const int c = blockIdx.x, h = blockIdx.y, bb = blockIdx.z;
    const int t0 = c * CT, n = min(CT, p.L - t0);
    const Ws w = ws_of(ws, p, (long long)bb * p.H + h, backward != 0);
    const long long oqk = (long long)bb * p.bqk + (long long)t0 * p.tqk + (long long)h * DK;
    const long long ov = (long long)bb * p.bv + (long long)t0 * p.tv + (long long)h * DV;
    const MK mk;
    const MS ms;
    auto product_out = [&](float* out) {
        float acc[MS::TM][MS::TN];
        tile::zero<MS>(acc);
        if (ms.on) {
            tile::product<MS, false, false, DK, DV>(acc, sm.X, sm.Y, 0, CT, ms);
#pragma unroll
            for (int i = 0; i < MS::TM; ++i)
#pragma unroll
                for (int gq = 0; gq < MS::GN; ++gq)
                    tile::store4(out + ms.m(i) * DV + ms.n4(gq), make_float4(acc[i][4 * gq], acc[i][4 * gq + 1], acc[i][4 * gq + 2], acc[i][4 * gq + 3]));
        }
    };
    Quad gq, kq, qq;
    if (mk.on) {
        gq = load_quad(g + oqk, p.tqk, n, p.vec, mk);
        kq = load_quad(k + oqk, p.tqk, n, p.vec, mk);
        if (dO) qq = load_quad(q + oqk, p.tqk, n, p.vec, mk);
        put_total<DK>(sm.tot, gq, mk);
    }
    tile::load<CT, DV, NT>(sm.Y, v + ov, p.tv, n, p.vec);
    __syncthreads();
    if (mk.on) {
        float f[4];
        exp_blocks<DK>(f, sm.tot, mk.ty + 1, 8, mk);
        put_quad<DK>(sm.X, times(kq, exp_suffix(gq), f), mk);
        if (mk.ty == 0) {
            exp_blocks<DK>(f, sm.tot, 0, 8, mk);
            tile::store4(w.gamn + (long long)c * DK + mk.n4(0), make_float4(f[0], f[1], f[2], f[3]));
        }
    }
    __syncthreads();
    product_out(w.Psi + (long long)c * DK * DV);
    if (dO) {
        __syncthreads();
        if (mk.on) {
            float f[4];
            exp_blocks<DK>(f, sm.tot, 0, mk.ty, mk);
            put_quad<DK>(sm.X, times(qq, exp_prefix(gq), f), mk);
        }
        tile::load<CT, DV, NT>(sm.Y, dO + ov, p.tv, n, p.vec);
        __syncthreads();
        product_out(w.Theta + (long long)c * DK * DV);
    }
}

// ---- ST and its adjoint: x' = gam_n[i] x + R[i][j] per tile, one thread per state element.
//      forward: R = Psi, tiles ascending, Hc[c] = state entering tile c, Hc[NT] = state leaving the segment
//      reverse: R = Theta, tiles descending, dHc[c] = gradient of the state leaving tile c
//      grid (dk*dv/256, H, B), twice as wide with both directions in one launch (the backward).  Bound by memory latency: a
//      thread keeps the loads of UN tiles in flight while it walks the UN before them.
constexpr int CHAIN_NT = 256;
struct ChainEnds { const float* init; float* fin; };
__global__ void __launch_bounds__(CHAIN_NT) chain_kernel(Params p, ChainEnds fwd, ChainEnds rev, float* ws, int backward) {
    const int dk = p.dk, dv = p.dv, m = dk * dv, n = p.NT, wide = m / CHAIN_NT;
    const bool reverse = (int)blockIdx.x >= wide;
    const int e = ((int)blockIdx.x - (reverse ? wide : 0)) * CHAIN_NT + threadIdx.x, i = e / dv;
    const long long bh = (long long)blockIdx.z * p.H + blockIdx.y;
    const Ws w = ws_of(ws, p, bh, backward != 0);
    const ChainEnds ends = reverse ? rev : fwd;
    const float* R = (reverse ? w.Theta + (long long)(n - 1) * m : w.Psi) + e;
    const float* G = (reverse ? w.gamn + (long long)(n - 1) * dk : w.gamn) + i;
    float* states = (reverse ? w.dHc + (long long)(n - 1) * m : w.Hc) + e;
    const long long sm = reverse ? -m : m, sk = reverse ? -dk : dk;
    constexpr int UN = 8;
    float r[2][UN], a[2][UN];
    auto fetch = [&](int buf, int s0) {
#pragma unroll
        for (int u = 0; u < UN; ++u)
            if (s0 + u < n) { r[buf][u] = __ldcg(R + (s0 + u) * sm); a[buf][u] = __ldg(G + (s0 + u) * sk); }
    };
    float x = ends.init ? ends.init[bh * m + e] : 0.f;
    auto walk = [&](int buf, int s0) {
#pragma unroll
        for (int u = 0; u < UN; ++u)
            if (s0 + u < n) {
                states[(s0 + u) * sm] = x;
                x = fmaf(a[buf][u], x, r[buf][u]);
            }
    };
    fetch(0, 0);
    for (int s0 = 0; s0 < n; s0 += 2 * UN) {
        fetch(1, s0 + UN);
        walk(0, s0);
        fetch(0, s0 + 2 * UN);
        walk(1, s0 + UN);
    }
    if (!reverse) w.Hc[(long long)n * m + e] = x;
    if (ends.fin) ends.fin[bh * m + e] = x;
}

// accumulator rows m < n to rows of an output tensor
template <class Mp, typename T>
__device__ __forceinline__ void store_rows(T* __restrict__ dst, long long stride, int n, const float (&acc)[Mp::TM][Mp::TN], const Mp& mp, bool vec) {
#pragma unroll
    for (int i = 0; i < Mp::TM; ++i) {
        const int m = mp.m(i);
        if (m < n)
#pragma unroll
            for (int gq = 0; gq < Mp::GN; ++gq)
                tile::store4(dst + m * stride + mp.n4(gq), make_float4(acc[i][4 * gq], acc[i][4 * gq + 1], acc[i][4 * gq + 2], acc[i][4 * gq + 3]), vec);
    }
}

// ---- Out: O = A V + (q*gam) Hc.  grid (tiles, H, B) ---------------------------------------------------------------------
// The product with Hc comes first and the level arrays take its operands' place: four CTAs of a 64-wide head per SM instead of
// three (195 -> 179 us on 16384 tokens x 16 heads).
template <int DK, int DV>
struct OutSmem {
    static constexpr int LV = 3 * CT * DK, QH = CT * DK + DK * DV;
    float S[LV > QH ? LV : QH];                          // q*gam and Hc, then the level arrays
    float V[CT * DV], A[CC], tot[8 * DK];
    float red[8 * (DK / 32) * 16];
};
template <typename T, int DK, int DV>
__global__ void __launch_bounds__(kThreads<DK, DV>, kThreads<DK, DV> == 128 ? 4 : 1) out_kernel(Params p, const T* __restrict__ q, const T* __restrict__ k, const T* __restrict__ v,
                                                               const float* __restrict__ g, T* __restrict__ o, const float* ws) {
    constexpr int NT = kThreads<DK, DV>;
    using MK = tile::Map<CT, DK, NT>;
    using MV = tile::Map<CT, DV, NT>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    OutSmem<DK, DV>& sm = *reinterpret_cast<OutSmem<DK, DV>*>(smem_raw);
    const int c = blockIdx.x, h = blockIdx.y, bb = blockIdx.z;
    const int t0 = c * CT, n = min(CT, p.L - t0);
    const Ws w = ws_of(const_cast<float*>(ws), p, (long long)bb * p.H + h, false);
    const long long oqk = (long long)bb * p.bqk + (long long)t0 * p.tqk + (long long)h * DK;
    const long long ov = (long long)bb * p.bv + (long long)t0 * p.tv + (long long)h * DV;
    const MK mk;
    const MV mv;
    Quad gq, kq, qq;
    if (mk.on) {
        gq = load_quad(g + oqk, p.tqk, n, p.vec, mk);
        kq = load_quad(k + oqk, p.tqk, n, p.vec, mk);
        qq = load_quad(q + oqk, p.tqk, n, p.vec, mk);
        put_total<DK>(sm.tot, gq, mk);
    }
    tile::load<CT, DV, NT>(sm.V, v + ov, p.tv, n, p.vec);
    float *Qg = sm.S, *H = sm.S + CT * DK;
    tile::load<DK, DV, NT>(H, w.Hc + (long long)c * DK * DV, DV, DK);
    __syncthreads();
    if (mk.on) {
        float f[4];
        exp_blocks<DK>(f, sm.tot, 0, mk.ty, mk);
        put_quad<DK>(Qg, times(qq, exp_prefix(gq), f), mk);
    }
    __syncthreads();
    float acc[MV::TM][MV::TN];
    tile::zero<MV>(acc);
    if (mv.on) tile::product<MV, true, false, DK, DV>(acc, Qg, H, 0, DK, mv);
    __syncthreads();
    if (mk.on) {
        const Quad ep = exp_prefix(gq), es = exp_suffix(gq);
        diag_partials(sm.red, qq, kq, near_weights(gq), es, mk);
        put_levels<DK>(sm.S, qq, kq, ep, es, sm.tot, mk);
    }
    __syncthreads();
    assemble_scores<DK, NT, MK::TXN / 8>(sm.A, sm.S, sm.red);
    __syncthreads();
    if (mv.on) {
        tile::product<MV, true, false, CT, DV>(acc, sm.A, sm.V, 0, mv.warp_m0() + 16, mv);
        store_rows(o + ov, p.tv, n, acc, mv, p.vec);
    }
}

// ---- backward, tile-parallel: every input gradient of the tile from the stored Hc, dHc.  grid (tiles, H, B) ---------------
// H is needed only for dO H^T, so the level arrays take its place afterwards; 128 x 128 holds one state at a time.  om*K
// takes V's place.  With 64-wide heads this lets three CTAs share an SM (556 -> 499 us on 16384 tokens x 16 heads).
template <int DK, int DV>
struct BwdSmem {
    static constexpr bool BOTH = DK * DV < 128 * 128;
    static constexpr int LV = 3 * CT * DK, ST = DK * DV;
    float H[BOTH ? (ST > LV ? ST : LV) : ST];            // H, then the level arrays (BOTH) or dH'
    float X[BOTH ? ST : LV];                             // dH' (BOTH) or the level arrays
    float V[CT * (DV > DK ? DV : DK)], D[CT * DV], A[CC], DA[CC], tot[8 * DK], xt[8 * DK], anchor[DK];
    float red[8 * (DK / 32) * 16];
    __device__ __forceinline__ float* G() { return BOTH ? X : H; }
    __device__ __forceinline__ float* S() { return BOTH ? H : X; }
    __device__ __forceinline__ float* Kw() { return V; }
};

template <typename T, int DK, int DV>
__global__ void __launch_bounds__(kThreads<DK, DV>, kThreads<DK, DV> == 128 ? 3 : 1)
bwd_out_kernel(Params p, const T* __restrict__ q, const T* __restrict__ k, const T* __restrict__ v, const float* __restrict__ g,
               const T* __restrict__ dO, T* __restrict__ dq, T* __restrict__ dk_out, T* __restrict__ dv_out, float* __restrict__ dg,
               const float* ws) {
    constexpr int NT = kThreads<DK, DV>;
    using MK = tile::Map<CT, DK, NT>;
    using MV = tile::Map<CT, DV, NT>;
    using MC = tile::Map<CT, CT, NT>;
    using Smem = BwdSmem<DK, DV>;
    static_assert(MK::TM == 4 && MK::TN == 4, "a thread owns 4 tokens x 4 channels");
    extern __shared__ __align__(16) unsigned char smem_raw[];
    Smem& sm = *reinterpret_cast<Smem*>(smem_raw);
    float *H = sm.H, *S = sm.S(), *G = sm.G(), *Kw = sm.Kw();
    const int c = blockIdx.x, h = blockIdx.y, bb = blockIdx.z, tid = threadIdx.x;
    const int t0 = c * CT, n = min(CT, p.L - t0);
    const Ws w = ws_of(const_cast<float*>(ws), p, (long long)bb * p.H + h, true);
    const long long oqk = (long long)bb * p.bqk + (long long)t0 * p.tqk + (long long)h * DK;
    const long long ov = (long long)bb * p.bv + (long long)t0 * p.tv + (long long)h * DV;
    const float* Gg = w.dHc + (long long)c * DK * DV;
    const MK mk;
    const MV mv;
    Quad gq, kq, qq;
    if (mk.on) {
        gq = load_quad(g + oqk, p.tqk, n, p.vec, mk);
        kq = load_quad(k + oqk, p.tqk, n, p.vec, mk);
        qq = load_quad(q + oqk, p.tqk, n, p.vec, mk);
        put_total<DK>(sm.tot, gq, mk);
    }
    tile::load<CT, DV, NT>(sm.V, v + ov, p.tv, n, p.vec);
    tile::load<CT, DV, NT>(sm.D, dO + ov, p.tv, n, p.vec);
    tile::load<DK, DV, NT>(H, w.Hc + (long long)c * DK * DV, DV, DK);
    if constexpr (Smem::BOTH) tile::load<DK, DV, NT>(G, Gg, DV, DK);
    {   // anchor[i] = <dH'[i,:], H'[i,:]>, H' the state leaving the tile: DV/4 lanes per row
        const float* Hn = w.Hc + (long long)(c + 1) * DK * DV;
        for (int i = tid; i < DK * DV / 4; i += NT) {
            const float4 a = tile::load4(Gg + 4 * i), b = tile::load4(Hn + 4 * i);
            float s = fmaf(a.x, b.x, fmaf(a.y, b.y, fmaf(a.z, b.z, a.w * b.w)));
#pragma unroll
            for (int off = DV / 8; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
            if (i % (DV / 4) == 0) sm.anchor[i / (DV / 4)] = s;
        }
    }
    __syncthreads();
    float adq[4][4], adk[4][4];
    tile::zero<MK>(adq);
    tile::zero<MK>(adk);
    if (mk.on) tile::product<MK, true, true, DV, DV>(adq, sm.D, H, 0, DV, mk);                // dO H^T
    {   // dA, mirrored: DA[t][s] = DA[s][t] = dO_t . v_s for s <= t
        const MC mc;
        if (mc.on) {
            float a[MC::TM][MC::TN];
            tile::zero<MC>(a);
            tile::product<MC, true, true, DV, DV>(a, sm.D, sm.V, 0, DV, mc);
#pragma unroll
            for (int i = 0; i < MC::TM; ++i)
#pragma unroll
                for (int j = 0; j < MC::TN; ++j) {
                    const int t = mc.m(i), s = mc.n4(0) + j;
                    if (s <= t) {
                        sm.DA[tile::at<CT>(t, s)] = a[i][j];
                        sm.DA[tile::at<CT>(s, t)] = a[i][j];
                    }
                }
        }
    }
    if constexpr (Smem::BOTH) {
        if (mk.on) tile::product<MK, true, true, DV, DV>(adk, sm.V, G, 0, DV, mk);            // V dH'^T
    }
    __syncthreads();                                                    // H and (where both states fit) V have served
    if constexpr (!Smem::BOTH) {
        tile::load<DK, DV, NT>(G, Gg, DV, DK);
        __syncthreads();
        if (mk.on) tile::product<MK, true, true, DV, DV>(adk, sm.V, G, 0, DV, mk);
        __syncthreads();
    }
    Quad ep, es;
    Near nw;
    if (mk.on) {
        ep = exp_prefix(gq);
        es = exp_suffix(gq);
        nw = near_weights(gq);
        diag_partials(sm.red, qq, kq, nw, es, mk);
        put_levels<DK>(S, qq, kq, ep, es, sm.tot, mk);
        float f[4];
        exp_blocks<DK>(f, sm.tot, 0, mk.ty, mk);                        // gam
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) adq[i][j] *= ep.v[i][j] * f[j];
        exp_blocks<DK>(f, sm.tot, mk.ty + 1, 8, mk);                    // om
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) adk[i][j] *= es.v[i][j] * f[j];
        put_quad<DK>(Kw, times(kq, es, f), mk);
    }
    __syncthreads();
    assemble_scores<DK, NT, MK::TXN / 8>(sm.A, S, sm.red);
    if (mk.on) {
        // pairs outside the diagonal blocks: row r of a level sums DA[r][r'] S_h[r'] over the other half of its block and
        // belongs to dq on upper rows, to dk on lower ones
#pragma unroll
        for (int lb = 0; lb < 3; ++lb) {
            const bool upper = (mk.ty >> lb) & 1;
            const int r0 = (((mk.ty >> lb) ^ 1) << lb) * 4;
            const float* Sl = S + lb * CT * DK;
            tile::f32x2 a2[4][2] = {};
#pragma unroll 4
            for (int r = r0; r < r0 + (4 << lb); ++r) {
                const float4 d = tile::ld4(sm.DA + tile::at<CT>(r, 4 * mk.ty));
                const ulonglong2 x = tile::ld4x2(Sl + tile::at<DK>(r, mk.n4(0)));
                const float dv4[4] = {d.x, d.y, d.z, d.w};
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const tile::f32x2 d2 = tile::pack(dv4[i], dv4[i]);
                    tile::fma2(a2[i][0], d2, x.x);
                    tile::fma2(a2[i][1], d2, x.y);
                }
            }
            float f[4];
            level_blocks<DK>(f, sm.tot, lb, mk);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                float a[4];
                tile::unpack(a2[i][0], a[0], a[1]);
                tile::unpack(a2[i][1], a[2], a[3]);
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const float e = f[j] * a[j];
                    if (upper) adq[i][j] = fmaf(ep.v[i][j], e, adq[i][j]);
                    else       adk[i][j] = fmaf(es.v[i][j], e, adk[i][j]);
                }
            }
        }
        // the diagonal block
#pragma unroll
        for (int t = 0; t < 4; ++t) {
            const float4 d = tile::ld4(sm.DA + tile::at<CT>(4 * mk.ty + t, 4 * mk.ty));
            const float dv4[4] = {d.x, d.y, d.z, d.w};
#pragma unroll
            for (int s = 0; s <= t; ++s)
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const float e = dv4[s] * near_weight(nw, es, t, s, j);
                    adq[t][j] = fmaf(e, kq.v[s][j], adq[t][j]);
                    adk[s][j] = fmaf(e, qq.v[t][j], adk[s][j]);
                }
        }
        // dg: suffix sums of q dq - k dk over the tile; the totals of the later blocks come through shared memory
        Quad x;
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) x.v[i][j] = qq.v[i][j] * adq[i][j] - kq.v[i][j] * adk[i][j];
        put_total<DK>(sm.xt, x, mk);
        store_rows(dq + oqk, p.tqk, n, adq, mk, p.vec);
        store_rows(dk_out + oqk, p.tqk, n, adk, mk, p.vec);
    }
    __syncthreads();
    if (mk.on) {
        float s[4];
        const float4 a0 = tile::ld4(sm.anchor + mk.n4(0));
        s[0] = a0.x; s[1] = a0.y; s[2] = a0.z; s[3] = a0.w;
        for (int b = 7; b > mk.ty; --b) {
            const float4 t = tile::ld4(sm.xt + b * DK + mk.n4(0));
            s[0] += t.x; s[1] += t.y; s[2] += t.z; s[3] += t.w;
        }
#pragma unroll
        for (int i = 3; i >= 0; --i) {
            const int m = mk.m(i);
#pragma unroll
            for (int j = 0; j < 4; ++j) s[j] += qq.v[i][j] * adq[i][j] - kq.v[i][j] * adk[i][j];
            if (m < n) tile::store4(dg + oqk + m * p.tqk + mk.n4(0), make_float4(s[0], s[1], s[2], s[3]), p.vec);
        }
    }
    if (mv.on) {
        float a[MV::TM][MV::TN];
        tile::zero<MV>(a);
        tile::product<MV, true, false, DK, DV>(a, Kw, G, 0, DK, mv);                          // (om*K) dH'
        tile::product<MV, false, false, CT, DV>(a, sm.A, sm.D, mv.warp_m0(), CT, mv);         // + A^T dO
        store_rows(dv_out + ov, p.tv, n, a, mv, p.vec);
    }
}

// The (chunk, d_k, d_v) sets accepted: bytes of shared memory of a form with padded chunk-long tiles and both states of a
// chunk resident (chunk 32 excludes 128 x 128).  The kernels above need less for every shape; the set is part of the interface.
__host__ inline size_t smem_rule(int C, int dk, int dv) {
    auto ld = [](int c) { return (size_t)c + 1; };
    const size_t c = C;
    return sizeof(float) * (6 * c * ld(dk) + 3 * c * ld(dv) + 2 * dk * ld(dv) + 2 * c * ld(C) + dk);
}

}  // namespace dcc
}  // namespace sf

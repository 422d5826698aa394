// Register-tiled float32 products on CUDA cores, for the chunkwise forms of the extension operators.
//
// Operands live in shared memory as row-major float32 tiles whose 16-byte units are XOR-swizzled with the row's index over
// four: unit u of row r sits at position u ^ ((r >> 2) & 7).  A product C[m][n] += sum_k A(m,k) B(k,n) reads an operand
// either along k (rows are m or n: one LDS.128 gives four k of one row) or across k (rows are k: one LDS.128 gives four
// neighbouring m or n).  A thread owns groups of four consecutive m and n, so in the first form the lanes of a warp read
// rows four apart, which the swizzle spreads over all banks, and in the second they read neighbouring units of one row:
// both are free of conflicts from the same storage, and no tile is ever stored twice or transposed.
#pragma once
#include "sf_common.cuh"

namespace sf {
namespace tile {

// Word offset of element (row, col) of a tile with rows of LD floats (LD a multiple of 32).
template <int LD>
__device__ __forceinline__ int at(int row, int col) {
    return row * LD + ((((col >> 2) ^ ((row >> 2) & 7)) << 2) | (col & 3));
}
__device__ __forceinline__ float4 ld4(const float* p) { return *reinterpret_cast<const float4*>(p); }
__device__ __forceinline__ void st4(float* p, float4 v) { *reinterpret_cast<float4*>(p) = v; }

// A warp's 4 x 8 arrangement: y = lane bits 0, 2; x = lane bits 1, 3, 4.  A 128-bit shared-memory load moves a half-warp at a
// time if lanes l and l ^ 1 (or l and l ^ 2) agree on their address, else only a quarter: with the bits of y and x interleaved
// both operands' loads take two passes, with x in the low three bits one of them takes four (measured: 3.0 passes per load
// against 2.2, and at 70-75 % of the cycles the passes weighed as much as the multiply-adds).
__device__ __forceinline__ int lane_y(int l) { return (l & 1) | ((l >> 1) & 2); }
__device__ __forceinline__ int lane_x(int l) { return ((l >> 1) & 1) | ((l >> 2) & 6); }
// Sum over the eight lanes that share y.
__device__ __forceinline__ float sum_x(float s) {
    s += __shfl_xor_sync(0xffffffffu, s, 2);
    s += __shfl_xor_sync(0xffffffffu, s, 8);
    s += __shfl_xor_sync(0xffffffffu, s, 16);
    return s;
}

// How NT threads share an M x N product: TM x TN outputs per thread (4 or 8), TYN x TXN threads take part (whole warps; a
// warp covers 4 x 8 of them).  Thread (ty, tx) owns m in {4 ty .. 4 ty + 3} (+ M/2 for the second group) and n likewise.
template <int M, int N, int NT>
struct Map {
    static constexpr int PER = M * N / 16 <= NT ? 16 : (M * N / 32 <= NT ? 32 : 64);
    static constexpr int TM = PER == 64 ? 8 : (PER == 32 && M > N ? 8 : 4);
    static constexpr int TN = PER / TM;
    static constexpr int TYN = M / TM, TXN = N / TN;
    static constexpr int ACTIVE = TYN * TXN;
    static_assert(ACTIVE <= NT && TYN % 4 == 0 && TXN % 8 == 0, "shape does not map onto whole warps");
    static constexpr int GM = TM / 4, GN = TN / 4;
    int ty, tx;
    bool on;
    __device__ __forceinline__ explicit Map(int t = threadIdx.x) {
        const int w = t >> 5, l = t & 31;
        constexpr int WX = TXN / 8;
        ty = (w / WX) * 4 + lane_y(l);
        tx = (w % WX) * 8 + lane_x(l);
        on = t < ACTIVE;
    }
    __device__ __forceinline__ int m(int i) const { return (i >> 2) * (M / GM) + 4 * ty + (i & 3); }
    __device__ __forceinline__ int n4(int g) const { return g * (N / GN) + 4 * tx; }      // first of the g-th group of four
    // rows covered by this warp's first / last thread group: limits of triangular products (TM == 4 only)
    __device__ __forceinline__ int warp_m0() const { return 4 * (ty & ~3); }
};

// Two float32 multiply-adds in one instruction (each half rounds as a scalar fmaf does).  The multiply-add pipe is no wider
// for it, but a warp needs half as many issue slots and half as many instructions in flight to keep it busy, which is what
// the kernels here are short of at two to four warps per scheduler (chains 4-7 % faster).
typedef unsigned long long f32x2;
__device__ __forceinline__ f32x2 pack(float lo, float hi) {
    f32x2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ void unpack(f32x2 v, float& lo, float& hi) { asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v)); }
__device__ __forceinline__ void fma2(f32x2& d, f32x2 a, f32x2 b) { asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(d) : "l"(a), "l"(b)); }
__device__ __forceinline__ ulonglong2 ld4x2(const float* p) { return *reinterpret_cast<const ulonglong2*>(p); }

// acc += A B over k in [k0, k1), both multiples of 4.  AK: A is stored [m][k], else [k][m]; BK: B is stored [n][k], else [k][n].
template <class Mp, bool AK, bool BK, int LDA, int LDB>
__device__ __forceinline__ void product(float (&acc)[Mp::TM][Mp::TN], const float* __restrict__ A, const float* __restrict__ B, int k0, int k1,
                                        const Mp& mp) {
    static_assert(AK || !BK, "operand forms in use");
    if constexpr (BK) {
        // both operands along k: even and odd k accumulate in the halves of a pair, added up at the end
        f32x2 s[Mp::TM][Mp::TN];
#pragma unroll
        for (int i = 0; i < Mp::TM; ++i)
#pragma unroll
            for (int j = 0; j < Mp::TN; ++j) s[i][j] = pack(acc[i][j], 0.f);
#pragma unroll 2
        for (int k = k0; k < k1; k += 4) {
            const int u = k >> 2, ob = (u ^ (mp.tx & 7)) << 2, oa = (u ^ (mp.ty & 7)) << 2;     // rows of both groups share these bits
            ulonglong2 b[Mp::TN];
#pragma unroll
            for (int g = 0; g < Mp::GN; ++g)
#pragma unroll
                for (int j = 0; j < 4; ++j) b[4 * g + j] = ld4x2(B + (mp.n4(g) + j) * LDB + ob);
#pragma unroll
            for (int i = 0; i < Mp::TM; ++i) {
                const ulonglong2 a = ld4x2(A + mp.m(i) * LDA + oa);
#pragma unroll
                for (int j = 0; j < Mp::TN; ++j) { fma2(s[i][j], a.x, b[j].x); fma2(s[i][j], a.y, b[j].y); }
            }
        }
#pragma unroll
        for (int i = 0; i < Mp::TM; ++i)
#pragma unroll
            for (int j = 0; j < Mp::TN; ++j) {
                float lo, hi;
                unpack(s[i][j], lo, hi);
                acc[i][j] = lo + hi;
            }
    } else {
        // B across k: a pair holds two neighbouring n, the factor from A is repeated in both halves
        f32x2 s[Mp::TM][Mp::TN / 2];
#pragma unroll
        for (int i = 0; i < Mp::TM; ++i)
#pragma unroll
            for (int j = 0; j < Mp::TN / 2; ++j) s[i][j] = pack(acc[i][2 * j], acc[i][2 * j + 1]);
#pragma unroll 2
        for (int k = k0; k < k1; k += 4) {
            const int u = k >> 2;
            ulonglong2 b[4][Mp::GN];
#pragma unroll
            for (int kk = 0; kk < 4; ++kk)
#pragma unroll
                for (int g = 0; g < Mp::GN; ++g) b[kk][g] = ld4x2(B + (k + kk) * LDB + (((mp.n4(g) >> 2) ^ (u & 7)) << 2));
            if constexpr (AK) {
                const int off = (u ^ (mp.ty & 7)) << 2;
#pragma unroll
                for (int i = 0; i < Mp::TM; ++i) {
                    const float4 a = ld4(A + mp.m(i) * LDA + off);
                    const float av[4] = {a.x, a.y, a.z, a.w};
#pragma unroll
                    for (int kk = 0; kk < 4; ++kk) {
                        const f32x2 a2 = pack(av[kk], av[kk]);
#pragma unroll
                        for (int g = 0; g < Mp::GN; ++g) { fma2(s[i][2 * g], a2, b[kk][g].x); fma2(s[i][2 * g + 1], a2, b[kk][g].y); }
                    }
                }
            } else {
#pragma unroll
                for (int kk = 0; kk < 4; ++kk)
#pragma unroll
                    for (int ga = 0; ga < Mp::GM; ++ga) {
                        const float4 a = ld4(A + (k + kk) * LDA + (((mp.m(4 * ga) >> 2) ^ (u & 7)) << 2));
                        const float av[4] = {a.x, a.y, a.z, a.w};
#pragma unroll
                        for (int i = 0; i < 4; ++i) {
                            const f32x2 a2 = pack(av[i], av[i]);
#pragma unroll
                            for (int g = 0; g < Mp::GN; ++g) {
                                fma2(s[4 * ga + i][2 * g], a2, b[kk][g].x);
                                fma2(s[4 * ga + i][2 * g + 1], a2, b[kk][g].y);
                            }
                        }
                    }
            }
        }
#pragma unroll
        for (int i = 0; i < Mp::TM; ++i)
#pragma unroll
            for (int j = 0; j < Mp::TN / 2; ++j) unpack(s[i][j], acc[i][2 * j], acc[i][2 * j + 1]);
    }
}

template <class Mp>
__device__ __forceinline__ void zero(float (&acc)[Mp::TM][Mp::TN]) {
#pragma unroll
    for (int i = 0; i < Mp::TM; ++i)
#pragma unroll
        for (int j = 0; j < Mp::TN; ++j) acc[i][j] = 0.f;
}

// Four neighbouring elements of a row in global memory (16-byte aligned float32, 8-byte aligned bf16).
__device__ __forceinline__ float4 load4(const float* p) { return __ldg(reinterpret_cast<const float4*>(p)); }
__device__ __forceinline__ float4 load4(const __nv_bfloat16* p) {
    const uint2 v = __ldg(reinterpret_cast<const uint2*>(p));
    const float2 a = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&v.x));
    const float2 b = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&v.y));
    return make_float4(a.x, a.y, b.x, b.y);
}
__device__ __forceinline__ void store4(float* p, float4 v) { *reinterpret_cast<float4*>(p) = v; }
__device__ __forceinline__ void store4(__nv_bfloat16* p, float4 v) {
    const __nv_bfloat162 a = __floats2bfloat162_rn(v.x, v.y), b = __floats2bfloat162_rn(v.z, v.w);
    uint2 o;
    o.x = *reinterpret_cast<const uint32_t*>(&a);
    o.y = *reinterpret_cast<const uint32_t*>(&b);
    *reinterpret_cast<uint2*>(p) = o;
}

// The accumulator to a tile (f(m, n, value) applied to each element).
template <class Mp, int LD, typename F>
__device__ __forceinline__ void put(float* dst, const float (&acc)[Mp::TM][Mp::TN], const Mp& mp, F f) {
#pragma unroll
    for (int i = 0; i < Mp::TM; ++i)
#pragma unroll
        for (int g = 0; g < Mp::GN; ++g) {
            const int m = mp.m(i), n = mp.n4(g);
            st4(dst + at<LD>(m, n), make_float4(f(m, n, acc[i][4 * g]), f(m, n + 1, acc[i][4 * g + 1]), f(m, n + 2, acc[i][4 * g + 2]),
                                                f(m, n + 3, acc[i][4 * g + 3])));
        }
}

// The same element-wise access for callers whose pointers or strides do not allow vector accesses (`vec` false).
template <typename T>
__device__ __forceinline__ float4 load4(const T* p, bool vec) {
    if (vec) return load4(p);
    return make_float4(to_f32(p[0]), to_f32(p[1]), to_f32(p[2]), to_f32(p[3]));
}
template <typename T>
__device__ __forceinline__ void store4(T* p, float4 v, bool vec) {
    if (vec) { store4(p, v); return; }
    p[0] = from_f32<T>(v.x); p[1] = from_f32<T>(v.y); p[2] = from_f32<T>(v.z); p[3] = from_f32<T>(v.w);
}

// ROWS x D tile from global rows `stride` elements apart; rows at or beyond `valid` become zero.
template <int ROWS, int D, int NT, typename T>
__device__ __forceinline__ void load(float* dst, const T* __restrict__ src, long long stride, int valid, bool vec = true) {
    constexpr int U = D / 4, IT = ROWS * U / NT;
    static_assert(ROWS * U % NT == 0, "tile does not divide among the threads");
    float4 v[IT < 8 ? IT : 8];
#pragma unroll
    for (int i0 = 0; i0 < IT; i0 += 8) {
#pragma unroll
        for (int i = 0; i < 8 && i0 + i < IT; ++i) {
            const int idx = threadIdx.x + (i0 + i) * NT, r = idx / U, c = (idx % U) * 4;
            v[i] = r < valid ? load4(src + r * stride + c, vec) : make_float4(0.f, 0.f, 0.f, 0.f);
        }
#pragma unroll
        for (int i = 0; i < 8 && i0 + i < IT; ++i) {
            const int idx = threadIdx.x + (i0 + i) * NT, r = idx / U, c = (idx % U) * 4;
            st4(dst + at<D>(r, c), v[i]);
        }
    }
}
// Rows of a tile times a factor per row, in place.
template <int ROWS, int D, int NT>
__device__ __forceinline__ void scale_rows(float* x, const float* w) {
    for (int idx = threadIdx.x; idx < ROWS * D / 4; idx += NT) {
        const int r = idx / (D / 4);
        float4* p = reinterpret_cast<float4*>(x) + idx;          // the swizzle permutes units inside a row only
        const float f = w[r];
        float4 v = *p;
        v.x *= f; v.y *= f; v.z *= f; v.w *= f;
        *p = v;
    }
}

}  // namespace tile
}  // namespace sf

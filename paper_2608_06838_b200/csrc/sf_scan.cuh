// Bandwidth-bound kernels: the block-level state scan (ST / STB of paper Eq. 2 and Section 3.4 taken
// across blocks, and Eq. 5 / Eq. 7 across segment boundaries) and the log-decay-gradient epilogue.
#pragma once
#include "sf_common.cuh"

namespace sf {

// First-order linear recurrence over the n blocks of a segment, element-wise over m = d_k*d_v lanes
// for each (batch, head):
//   forward: X_0 = init; states[j] = X_j;     X_{j+1} = exp(ld[j]) X_j + U[j];  final = X_n
//   reverse: X_n = init; states[j] = X_{j+1}; X_j     = exp(ld[j]) X_{j+1} + U[j];  final = X_0
// One thread carries 4 consecutive lanes (float4, coalesced 512 B per warp) through all n steps;
// the U loads of the next steps do not depend on the carried value, so UNROLL of them are issued
// ahead of the dependent FMA chain.  states may alias U: each element is read before it is written
// by the same thread.  grid = (m/4/256, B*H).
constexpr int SCAN_NT = 256;
constexpr int SCAN_UNROLL = 4;

__global__ void __launch_bounds__(SCAN_NT) state_scan_kernel(int n, int m, int reverse, const float* ld,
                                                             const float* U, const float* __restrict__ init,
                                                             float* states, float* __restrict__ final_state) {
    grid_launch_next();
    grid_wait();
    const int bh = blockIdx.y;
    const int e = (blockIdx.x * SCAN_NT + threadIdx.x) * 4;
    if (e >= m) return;
    const float* ldh = ld + (long long)bh * n;
    const float4* Uh = reinterpret_cast<const float4*>(U + (long long)bh * n * m + e);
    float4* Sh = reinterpret_cast<float4*>(states + (long long)bh * n * m + e);
    const long long step = m / 4;                      // float4 stride between blocks
    float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
    if (init) x = *reinterpret_cast<const float4*>(init + (long long)bh * m + e);
    for (int s0 = 0; s0 < n; s0 += SCAN_UNROLL) {
        float4 u[SCAN_UNROLL];
        float a[SCAN_UNROLL];
#pragma unroll
        for (int i = 0; i < SCAN_UNROLL; ++i) {
            const int s = s0 + i;
            if (s < n) {
                const int j = reverse ? (n - 1 - s) : s;
                u[i] = Uh[j * step];
                a[i] = __expf(ldh[j]);
            }
        }
#pragma unroll
        for (int i = 0; i < SCAN_UNROLL; ++i) {
            const int s = s0 + i;
            if (s < n) {
                const int j = reverse ? (n - 1 - s) : s;
                Sh[j * step] = x;
                x.x = fmaf(a[i], x.x, u[i].x);
                x.y = fmaf(a[i], x.y, u[i].y);
                x.z = fmaf(a[i], x.z, u[i].z);
                x.w = fmaf(a[i], x.w, u[i].w);
            }
        }
    }
    *reinterpret_cast<float4*>(final_state + (long long)bh * m + e) = x;
}

// The same recurrence carried through several consecutive segments in one launch (paper Eq. 5 / Eq. 7: the state
// leaving one segment enters the next).  With short segments the chain of one small scan kernel per segment is
// what the hand-off costs (launch and dependency latency, not bytes), so the chaining driver scans a group of
// segments at once.  Segments are listed in the order they are visited (ascending forward, descending in
// reverse); the arithmetic per element is the one of state_scan_kernel, so results are bit-identical.
constexpr int SCAN_GROUP_MAX = 8;
struct ScanSeg {
    const float* ld;        // [B*H, n] block totals of the log-decay
    float* UH;              // [B*H, n, m] aggregates in, states out (in place)
    float* fin;             // [B*H, m] boundary state leaving the segment in scan direction
    int n;
};
struct ScanGroup {
    ScanSeg seg[SCAN_GROUP_MAX];
    int count;
};

__global__ void __launch_bounds__(SCAN_NT) state_scan_group_kernel(ScanGroup grp, int m, int reverse, const float* __restrict__ init) {
    const int bh = blockIdx.y;
    const int e = (blockIdx.x * SCAN_NT + threadIdx.x) * 4;
    if (e >= m) return;
    const long long step = m / 4;
    float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
    if (init) x = *reinterpret_cast<const float4*>(init + (long long)bh * m + e);
    for (int si = 0; si < grp.count; ++si) {
        const ScanSeg sg = grp.seg[si];
        const int n = sg.n;
        const float* ldh = sg.ld + (long long)bh * n;
        float4* Sh = reinterpret_cast<float4*>(sg.UH + (long long)bh * n * m + e);
        for (int s0 = 0; s0 < n; s0 += SCAN_UNROLL) {
            float4 u[SCAN_UNROLL];
            float a[SCAN_UNROLL];
#pragma unroll
            for (int i = 0; i < SCAN_UNROLL; ++i) {
                const int s = s0 + i;
                if (s < n) {
                    const int j = reverse ? (n - 1 - s) : s;
                    u[i] = Sh[j * step];
                    a[i] = __expf(ldh[j]);
                }
            }
#pragma unroll
            for (int i = 0; i < SCAN_UNROLL; ++i) {
                const int s = s0 + i;
                if (s < n) {
                    const int j = reverse ? (n - 1 - s) : s;
                    Sh[j * step] = x;
                    x.x = fmaf(a[i], x.x, u[i].x);
                    x.y = fmaf(a[i], x.y, u[i].y);
                    x.z = fmaf(a[i], x.z, u[i].z);
                    x.w = fmaf(a[i], x.w, u[i].w);
                }
            }
        }
        *reinterpret_cast<float4*>(sg.fin + (long long)bh * m + e) = x;
    }
}

// Marks the first chunk of segments first .. first + count - 1 of a chain in slot[] (see SegParams::bslot), after setting its
// first `clear` entries to -1.  The chunk indices travel as kernel arguments, so the launch can be recorded in a graph.
constexpr int MARK_MAX = 256;
struct SegStarts { int chunk[MARK_MAX]; int first, count; };
__global__ void mark_bounds_kernel(int* __restrict__ slot, int clear, SegStarts s) {
    const int i = threadIdx.x;
    for (int c = i; c < clear; c += MARK_MAX) slot[c] = -1;
    __syncthreads();
    if (i < s.count) slot[s.chunk[i]] = s.first + i;
}

// Log-decay gradient.  With x_t = q_t.dq_t - k_t.dk_t (the dq and dk/dv passes emit both dot products
// from their float32 accumulators) the recurrence gives dg_t = dg_{t+1} + x_t, and at a block start
// dg equals <H, dH> of the block-entering state and its gradient.  So, with
// P = <Hs[j], gradient entering block j> (Gs[j-1], or dS_in for j = 0) read from the float32 block
// states, the token u of block j gets
//     dg_u = P - sum_{t < u in block j} x_t ,
// evaluated chunk by chunk: P_{c+1} = P_c - sum_{t in chunk c} x_t, dg_u = P_{c+1} + sum_{t=u}^{end of c} x_t.
// The rounding errors of the dot products add up along the block like a random walk.  The block's end is an anchor too: there
// the sum must arrive at <H, dH> of the state that leaves (Hs[j+1] and Gs[j]; at the segment's end DgEnd).  What is missing, D, is
// spread over the block in proportion to the variance met so far, sum (q.dq)^2 + (k.dk)^2 (whole chunks, linear inside one):
// the walk then is a bridge, with a third of its mean square.  rms error of dg over rms, 2 of 40 heads x 32768 tokens: blocks of 16
// chunks 7.1e-3 without the second anchor, 4.0e-3 with it, of 48 9.9e-3 and 6.1e-3.  A D that is not finite (NaN or Inf in later tokens) is not spread.
// grid = (NB, H, B), DG_NT threads.  xq, xk: [B,H,L]; dg: [B,L,H] with strides.
constexpr int DG_NT = 512;
struct DgEnd {
    const float* G;                      // [B,H,m] gradient of the state leaving the segment, NULL: zero
    const float* S;                      // [B,H,m] that state; NULL: not at hand, the last block has one anchor
    const float* g;                      // with it S is the last block's aggregate: the state is exp(sum of g) (entering state) + S
};

__global__ void __launch_bounds__(DG_NT) dg_epilogue_kernel(SegParams p, int m, const float* xq, const float* xk, const float* Hs,
                                                            const float* Gs, const float* dS_in, DgEnd end, float* __restrict__ dg) {
    constexpr int NW = DG_NT / 32, XN = 64 / NW;
    __shared__ float red[4][NW];
    __shared__ float sx[64], sw[64], P_next[64], corr[64], slope[64];
    __shared__ float suffix[64 * 64];
    grid_launch_next();
    grid_wait();
    const int j = blockIdx.x, h = blockIdx.y, b = blockIdx.z;
    const long long bh = (long long)b * p.H + h;
    const int C = p.C;
    const int c0 = j * p.R, nch = min(p.R, p.NC - c0);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, r0 = 2 * lane, r1 = r0 + 1;
    const int ntok = min(nch * C, p.L - c0 * C);          // tokens of this block (the segment's last chunk may be partial)
    // The kernel is a chain of memory round trips (its bytes take about 1 us), so the loads of all chunks' dot products go out
    // first, and those of the anchors AN rows of threads at a time.  A warp has the chunks warp, warp + NW, ... (at most 64 chunks in a
    // block), two tokens per lane.
    const float* xqh = xq + bh * p.L;
    const float* xkh = xk + bh * p.L;
    float q0[XN], q1[XN], k0[XN], k1[XN];
#pragma unroll
    for (int k = 0; k < XN; ++k) {
        const int c = min(warp + k * NW, nch - 1);
        const long long t0 = (long long)(c0 + c) * C;
        const int lim = min(C, ntok - c * C), i0 = min(r0, lim - 1), i1 = min(r1, lim - 1);
        q0[k] = xqh[t0 + i0]; k0[k] = xkh[t0 + i0];
        q1[k] = xqh[t0 + i1]; k1[k] = xkh[t0 + i1];
    }

    // anchors: fixed-order tree reductions so that the result is reproducible run to run
    const bool last = j == p.NB - 1;
    const float* H0 = Hs ? Hs + (bh * p.NB + j) * (long long)m : nullptr;       // NULL: states of zeros
    const float* G0 = (j == 0) ? (dS_in + bh * (long long)m) : (Gs + (bh * p.NB + (j - 1)) * (long long)m);
    const float* H1 = last ? (end.G && end.S ? end.S + bh * (long long)m : nullptr) : Hs + (bh * p.NB + j + 1) * (long long)m;
    const float* G1 = last ? (end.G ? end.G + bh * (long long)m : nullptr) : Gs + (bh * p.NB + j) * (long long)m;
    const bool aggregate = last && end.g && H1 && H0;
    float part0 = 0.f, part1 = 0.f, part2 = 0.f, beta = 0.f;
    if (aggregate) {
        const float* gh = end.g + (long long)b * p.bg + (long long)c0 * C * p.tg + h;
        for (int t = threadIdx.x; t < ntok; t += DG_NT) beta += gh[(long long)t * p.tg];
    }
    constexpr int AN = 4;
    for (int e0 = threadIdx.x * 4; e0 < m; e0 += AN * DG_NT * 4) {
        float4 h0[AN], g0[AN], h1[AN], g1[AN];
#pragma unroll
        for (int i = 0; i < AN; ++i) {
            const int e = e0 + i * DG_NT * 4;
            h0[i] = g0[i] = h1[i] = g1[i] = make_float4(0.f, 0.f, 0.f, 0.f);
            if (e < m && H0) { h0[i] = *reinterpret_cast<const float4*>(H0 + e); g0[i] = *reinterpret_cast<const float4*>(G0 + e); }
            if (e < m && H1) { h1[i] = *reinterpret_cast<const float4*>(H1 + e); g1[i] = *reinterpret_cast<const float4*>(G1 + e); }
        }
#pragma unroll
        for (int i = 0; i < AN; ++i) {
            part0 = fmaf(h0[i].x, g0[i].x, part0); part0 = fmaf(h0[i].y, g0[i].y, part0);
            part0 = fmaf(h0[i].z, g0[i].z, part0); part0 = fmaf(h0[i].w, g0[i].w, part0);
            part1 = fmaf(h1[i].x, g1[i].x, part1); part1 = fmaf(h1[i].y, g1[i].y, part1);
            part1 = fmaf(h1[i].z, g1[i].z, part1); part1 = fmaf(h1[i].w, g1[i].w, part1);
            if (aggregate) part2 += h0[i].x * g1[i].x + h0[i].y * g1[i].y + h0[i].z * g1[i].z + h0[i].w * g1[i].w;
        }
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        part0 += __shfl_xor_sync(0xffffffffu, part0, off);
        part1 += __shfl_xor_sync(0xffffffffu, part1, off);
        if (aggregate) {
            part2 += __shfl_xor_sync(0xffffffffu, part2, off);
            beta += __shfl_xor_sync(0xffffffffu, beta, off);
        }
    }
    if (lane == 0) { red[0][warp] = part0; red[1][warp] = part1; red[2][warp] = part2; red[3][warp] = beta; }

    // per chunk: suffix sums of x_t, the chunk total and the total of the squares
#pragma unroll
    for (int k = 0; k < XN; ++k) {
        const int c = warp + k * NW;
        if (c < nch) {
            const int lim = min(C, ntok - c * C);           // tokens past the end of the segment (ragged last chunk) contribute nothing
            const float on0 = r0 < lim ? 1.f : 0.f, on1 = r1 < lim ? 1.f : 0.f;
            const float x0 = (q0[k] - k0[k]) * on0, x1 = (q1[k] - k1[k]) * on1;
            float incl = x0 + x1, sq = (q0[k] * q0[k] + k0[k] * k0[k]) * on0 + (q1[k] * q1[k] + k1[k] * k1[k]) * on1;
#pragma unroll
            for (int off = 1; off < 32; off <<= 1) {        // inclusive suffix sums over lanes
                const float up = __shfl_down_sync(0xffffffffu, incl, off), us = __shfl_down_sync(0xffffffffu, sq, off);
                if (lane + off < 32) { incl += up; sq += us; }
            }
            if (r0 < C) suffix[c * 64 + r0] = incl;
            if (r1 < C) suffix[c * 64 + r1] = incl - x0;
            if (lane == 0) { sx[c] = incl; sw[c] = sq; }
        }
    }
    __syncthreads();
    if (warp == 0) {                                        // prefix sums over the chunks, two per lane
        float P = 0.f, Pe = 0.f;
        for (int w = 0; w < NW; ++w) { P += red[0][w]; Pe += red[1][w]; }
        if (aggregate) {
            float HG = 0.f, total = 0.f;
            for (int w = 0; w < NW; ++w) { HG += red[2][w]; total += red[3][w]; }
            const float carry = __expf(total);
            if (carry != 0.f) Pe = fmaf(carry, HG, Pe);
        }
        const double a0 = r0 < nch ? sx[r0] : 0.0, a1 = r1 < nch ? sx[r1] : 0.0;
        const float w0 = r0 < nch ? sw[r0] : 0.f, w1 = r1 < nch ? sw[r1] : 0.f;
        double a = a0 + a1;
        float ws = w0 + w1;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const double ua = __shfl_up_sync(0xffffffffu, a, off);
            const float uw = __shfl_up_sync(0xffffffffu, ws, off);
            if (lane >= off) { a += ua; ws += uw; }
        }
        const float D = (float)((double)P - __shfl_sync(0xffffffffu, a, 31)) - Pe, W = __shfl_sync(0xffffffffu, ws, 31);
        const bool anchored = !last || !end.G || end.S;
        const float f = anchored && W > 0.f && isfinite(W) && fabsf(D) <= 0.05f * sqrtf(W) ? D / W : 0.f;
        auto spread = [&](float w) { return f != 0.f ? f * w : 0.f; };       // w may be infinite where f is 0
        const double ex = a - (a0 + a1);
        const float wx = ws - (w0 + w1);
        if (r0 < nch) { P_next[r0] = (float)((double)P - (ex + a0)); corr[r0] = spread(wx); slope[r0] = spread(w0) / (float)min(C, ntok - r0 * C); }
        if (r1 < nch) { P_next[r1] = (float)((double)P - a); corr[r1] = spread(wx + w0); slope[r1] = spread(w1) / (float)min(C, ntok - r1 * C); }
    }
    __syncthreads();
    float* dgh = dg + (long long)b * p.bg + h;
    for (int idx = threadIdx.x; idx < nch * C; idx += DG_NT) {
        const int c = idx / C, r = idx - c * C;
        if (idx < ntok) dgh[((long long)(c0 + c) * C + r) * p.tg] = (P_next[c] + suffix[c * 64 + r]) - fmaf(slope[c], (float)r, corr[c]);
    }
}

}  // namespace sf

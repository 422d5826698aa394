// C ABI of the chunkwise diagonal decay: argument checks, shape dispatch and launches.
#include "../../include/stateflow.h"
#include "sf_channel_chunk.cuh"
#include "sf_variants_host.h"

namespace {

using namespace sfv;

sf_status_t check_chunked(const sf_seg_desc_t* d) {
    const sf_status_t c = check_desc(d, true);
    if (c != SF_OK) return c;
    if (d->chunk <= 0) return SF_ERR_INVALID_ARG;
    if (d->chunk != 16 && d->chunk != 32) return SF_ERR_UNSUPPORTED;
    if (d->H > 65535) return SF_ERR_INVALID_ARG;
    return sf::dcc::smem_rule(d->chunk, d->d_k, d->d_v) <= kMaxSmem ? SF_OK : SF_ERR_UNSUPPORTED;
}

sf::dcc::Params chunked_params(const sf_seg_desc_t* d, bool vec) {
    sf::dcc::Params p;
    p.B = d->B; p.H = d->H; p.L = d->seg_len; p.C = d->chunk; p.NC = (d->seg_len + d->chunk - 1) / d->chunk;
    p.NT = (d->seg_len + sf::dcc::CT - 1) / sf::dcc::CT;
    p.dk = d->d_k; p.dv = d->d_v;
    p.vec = vec;
    p.tqk = d->tok_stride_qk; p.tv = d->tok_stride_v; p.tg = d->tok_stride_g;
    p.bqk = d->batch_stride_qk; p.bv = d->batch_stride_v; p.bg = d->batch_stride_g;
    return p;
}

size_t chunked_ws_bytes(const sf_seg_desc_t* d, bool backward) {
    return (size_t)d->B * d->H * sf::dcc::ws_floats(chunked_params(d, false), backward) * sizeof(float);
}

struct Args {
    const void *q, *k, *v;
    const float *g, *S_in;
    void* o;
    float* S_out;
    const void* dO;
    const float* dS_out;
    void *dq, *dk, *dv;
    float *dg, *dS_in;
    float* ws;
    cudaStream_t st;
};

// The backward rebuilds the forward's states first.
template <typename T, int DK, int DV>
sf_status_t launch(const sf::dcc::Params& p, const Args& a) {
    using namespace sf::dcc;
    const T *q = static_cast<const T*>(a.q), *k = static_cast<const T*>(a.k), *v = static_cast<const T*>(a.v), *dO = static_cast<const T*>(a.dO);
    const bool backward = dO != nullptr;
    const dim3 tiles(p.NT, p.H, p.B), elems((backward ? 2 : 1) * DK * DV / CHAIN_NT, p.H, p.B);
    constexpr int nt = kThreads<DK, DV>;
    constexpr size_t s1 = sizeof(PreSmem<DK, DV>), s2 = sizeof(OutSmem<DK, DV>), s3 = sizeof(BwdSmem<DK, DV>);
    if (!opt_in<pre_kernel<T, DK, DV>>(s1) || !opt_in<out_kernel<T, DK, DV>>(s2) || !opt_in<bwd_out_kernel<T, DK, DV>>(s3)) return SF_ERR_CUDA;
    pre_kernel<T, DK, DV><<<tiles, nt, s1, a.st>>>(p, q, k, v, a.g, dO, a.ws, backward);
    chain_kernel<<<elems, CHAIN_NT, 0, a.st>>>(p, ChainEnds{a.S_in, a.S_out}, ChainEnds{a.dS_out, a.dS_in}, a.ws, backward);
    if (backward)
        bwd_out_kernel<T, DK, DV><<<tiles, nt, s3, a.st>>>(p, q, k, v, a.g, dO, static_cast<T*>(a.dq), static_cast<T*>(a.dk), static_cast<T*>(a.dv),
                                                          a.dg, a.ws);
    else
        out_kernel<T, DK, DV><<<tiles, nt, s2, a.st>>>(p, q, k, v, a.g, static_cast<T*>(a.o), a.ws);
    return launched(3);
}

template <typename T>
sf_status_t dispatch(const sf::dcc::Params& p, const Args& a) {
#define SF_SHAPE(DK, DV) if (p.dk == DK && p.dv == DV) return launch<T, DK, DV>(p, a);
    SF_SHAPE(32, 32) SF_SHAPE(32, 64) SF_SHAPE(32, 128)
    SF_SHAPE(64, 32) SF_SHAPE(64, 64) SF_SHAPE(64, 128)
    SF_SHAPE(128, 32) SF_SHAPE(128, 64) SF_SHAPE(128, 128)
#undef SF_SHAPE
    return SF_ERR_UNSUPPORTED;
}

sf_status_t run(const sf_seg_desc_t* d, const Args& a) {
    const bool vec = vec_ok(d, {a.q, a.k, a.v, a.o, a.dO, a.dq, a.dk, a.dv}) && !((reinterpret_cast<uintptr_t>(a.g) | reinterpret_cast<uintptr_t>(a.dg)) & 15u);
    const sf::dcc::Params p = chunked_params(d, vec);
    return d->dtype == SF_F32 ? dispatch<float>(p, a) : dispatch<__nv_bfloat16>(p, a);
}

}  // namespace

extern "C" {

size_t sf_channel_chunked_workspace_bytes(const sf_seg_desc_t* desc, int backward) {
    return check_chunked(desc) == SF_OK ? chunked_ws_bytes(desc, backward != 0) : 0;
}

sf_status_t sf_channel_chunked_fwd(const sf_seg_desc_t* desc, const void* q, const void* k, const void* v, const float* g,
                                   const float* S_in, void* o, float* S_out, void* workspace, size_t workspace_bytes,
                                   sf_stream_t stream) {
    const sf_status_t c = check_chunked(desc);
    if (c != SF_OK) return c;
    if (!q || !k || !v || !g || !o || !S_out || S_in == S_out) return SF_ERR_INVALID_ARG;
    if (!workspace || workspace_bytes < chunked_ws_bytes(desc, false) || (reinterpret_cast<uintptr_t>(workspace) & 255u)) return SF_ERR_WORKSPACE;
    Args a{};
    a.q = q; a.k = k; a.v = v; a.g = g; a.S_in = S_in; a.o = o; a.S_out = S_out;
    a.ws = static_cast<float*>(workspace); a.st = reinterpret_cast<cudaStream_t>(stream);
    return run(desc, a);
}

sf_status_t sf_channel_chunked_bwd(const sf_seg_desc_t* desc, const void* q, const void* k, const void* v, const float* g,
                                   const float* S_in, const void* dO, const float* dS_out, void* dq, void* dk, void* dv,
                                   float* dg, float* dS_in, void* workspace, size_t workspace_bytes, sf_stream_t stream) {
    const sf_status_t c = check_chunked(desc);
    if (c != SF_OK) return c;
    if (!q || !k || !v || !g || !dO || !dq || !dk || !dv || !dg || !dS_in || dS_in == dS_out) return SF_ERR_INVALID_ARG;
    if (!workspace || workspace_bytes < chunked_ws_bytes(desc, true) || (reinterpret_cast<uintptr_t>(workspace) & 255u)) return SF_ERR_WORKSPACE;
    Args a{};
    a.q = q; a.k = k; a.v = v; a.g = g; a.S_in = S_in; a.dO = dO; a.dS_out = dS_out;
    a.dq = dq; a.dk = dk; a.dv = dv; a.dg = dg; a.dS_in = dS_in;
    a.ws = static_cast<float*>(workspace); a.st = reinterpret_cast<cudaStream_t>(stream);
    return run(desc, a);
}

}  // extern "C"

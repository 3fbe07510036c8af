// One (beam slot, head) of decode attention by four warps in fp32: the paper's per-beam formulation (Section 3.3)
// taken literally.  The per-beam kernel is made of it, and the wide kernel comes back to it for outputs that
// are not finite.
#pragma once

#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include "segkv_internal.h"

namespace segkv_impl {
namespace rowwise {

struct Args {
    const void* q;
    void* out;
    const float* slopes;
    const void *kp, *vp, *kr;
    const void* const* k_chunks;      // growing capacity: chunk base pointers, chunk_steps steps each
    long long vdelta;                 // elements from a response K row to its V row
    const int32_t *anc, *plens;
    PromptStrides ps;
    int prompt_len, steps, W, H, Hkv, group, chunk_steps, max_steps, rows;
};

inline Args make_args(const Dims& d, const SdpaArgs& a) {
    Args r;
    r.q = a.q; r.out = a.out; r.slopes = a.slopes;
    r.kp = a.kp; r.vp = a.vp; r.kr = a.kr; r.k_chunks = a.k_chunks; r.vdelta = a.vdelta / 2;
    r.anc = a.anc; r.plens = a.plens;
    r.ps = prompt_strides(d);
    r.prompt_len = a.prompt_len; r.steps = a.steps;
    r.W = d.beams; r.H = d.heads; r.Hkv = d.kv_heads; r.group = d.group;
    r.chunk_steps = d.chunk_steps; r.max_steps = d.max_steps; r.rows = d.rows;
    return r;
}

template <typename T> struct Cvt;
template <> struct Cvt<__half> {
    static __device__ __forceinline__ float2 up(uint32_t u) {
        return __half22float2(*reinterpret_cast<const __half2*>(&u));
    }
    static __device__ __forceinline__ __half down(float f) { return __float2half_rn(f); }
};
template <> struct Cvt<__nv_bfloat16> {
    static __device__ __forceinline__ float2 up(uint32_t u) {
        return __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&u));
    }
    static __device__ __forceinline__ __nv_bfloat16 down(float f) { return __float2bfloat16_rn(f); }
};

template <int E> struct Vec;                       // E 16-bit elements as 32-bit words
template <> struct Vec<2> { using type = uint32_t; };
template <> struct Vec<4> { using type = uint2; };
template <> struct Vec<8> { using type = uint4; };

template <typename T, int E>
__device__ __forceinline__ void load_row(const T* p, float (&f)[E]) {
    typename Vec<E>::type raw = __ldg(reinterpret_cast<const typename Vec<E>::type*>(p));   // (no launch writes what it reads here)
    const uint32_t* w = reinterpret_cast<const uint32_t*>(&raw);
#pragma unroll
    for (int i = 0; i < E / 2; ++i) {
        float2 t = Cvt<T>::up(w[i]);
        f[2 * i] = t.x;
        f[2 * i + 1] = t.y;
    }
}

constexpr int kWarps = 4;
template <int D> constexpr int kScratch = kWarps * (D + 2);       // floats of shared memory

// Row g, query head h.  `meet` is a barrier of the four warps; `s` may be used again behind the next one.
template <typename T, int D, typename Meet>
__device__ __forceinline__ void attend(const Args& a, int g, int h, int warp, int lane, float* s, Meet meet) {
    constexpr int E = D / 32;
    const int b = g / a.W, kvh = h / a.group;

    float qf[E];
    load_row<T, E>((const T*)a.q + ((size_t)g * a.H + h) * D + lane * E, qf);
    const float kLog2e = 1.4426950408889634f;
    const float scale2 = kLog2e / sqrtf((float)D);
    const float slope2 = a.slopes ? a.slopes[h] * kLog2e : 0.f;
    const int P = a.plens ? a.plens[b] : a.prompt_len;
    const int L = P + a.steps;
    const int qpos = L - 1;

    float m = -INFINITY, l = 0.f, acc[E];
#pragma unroll
    for (int e = 0; e < E; ++e) acc[e] = 0.f;

    for (int i = warp; i < L; i += kWarps) {
        const T* krow;
        const T* vrow;
        if (i < P) {
            const size_t off = (size_t)(b * a.ps.b + kvh * a.ps.h + i * a.ps.p);
            krow = (const T*)a.kp + off;
            vrow = (const T*)a.vp + off;
        } else {
            const int st = i - P;
            const int r = __ldg(a.anc + (size_t)g * a.max_steps + st);
            const size_t slab = (size_t)a.rows * a.Hkv * D;      // elements of one step
            const T* base = (const T*)a.kr + (size_t)st * slab;  // one array, or the chunk that holds the step
            if (a.chunk_steps) base = (const T*)a.k_chunks[st / a.chunk_steps] + (size_t)(st % a.chunk_steps) * slab;
            krow = base + ((size_t)r * a.Hkv + kvh) * D;
            vrow = krow + a.vdelta;                               // V rows sit a constant behind their K rows
        }
        float kf[E], vf[E];
        load_row<T, E>(krow + lane * E, kf);
        load_row<T, E>(vrow + lane * E, vf);
        float dot = 0.f;
#pragma unroll
        for (int e = 0; e < E; ++e) dot = fmaf(qf[e], kf[e], dot);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) dot += __shfl_xor_sync(0xffffffffu, dot, o);
        float s2 = dot * scale2 + slope2 * (float)(i - qpos);
        float mn = fmaxf(m, s2);
        float alpha = exp2f(m - mn);
        float p = exp2f(s2 - mn);
        l = l * alpha + p;
#pragma unroll
        for (int e = 0; e < E; ++e) acc[e] = acc[e] * alpha + p * vf[e];
        m = mn;
    }

    float *s_m = s + kWarps * D, *s_l = s_m + kWarps;
    if (lane == 0) { s_m[warp] = m; s_l[warp] = l; }
#pragma unroll
    for (int e = 0; e < E; ++e) s[warp * D + lane * E + e] = acc[e];
    meet();
    for (int d = warp * 32 + lane; d < D; d += kWarps * 32) {
        float mm = -INFINITY;
#pragma unroll
        for (int w = 0; w < kWarps; ++w) mm = fmaxf(mm, s_m[w]);
        float ll = 0.f, o = 0.f;
#pragma unroll
        for (int w = 0; w < kWarps; ++w) {
            float f = (s_m[w] == -INFINITY) ? 0.f : exp2f(s_m[w] - mm);
            ll += s_l[w] * f;
            o += s[w * D + d] * f;
        }
        ((T*)a.out)[((size_t)g * a.H + h) * D + d] = Cvt<T>::down(o / ll);
    }
}

}  // namespace rowwise
}  // namespace segkv_impl

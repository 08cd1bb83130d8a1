// Shared by the decode kernels: what a container's header says (checked on the device), the value of a symbol,
// and what happens to the finished sum of an element (stored, or applied to the parameters at once).
#pragma once
#include "nuq_common.cuh"

namespace nuq {

// `hdr`: the container (a level-table stream carries its s interior levels behind the 16 header words)
__device__ __forceinline__ float level_times_norm(float norm, uint32_t levelset, uint32_t s, uint32_t sym, const uint32_t* hdr) {
    // exponential: l_j = 2^(j-1-s) (exact scaling);  uniform: l_k = k / 2^s;  table: l_j as stored, l_{s+1} = 1
    float level;
    if (levelset == kLevelsExp) level = __uint_as_float((126u + sym - s) << 23);
    else if (levelset == kLevelsUniform) level = (float)sym * __uint_as_float((127u - s) << 23);
    else level = sym <= s ? __uint_as_float(hdr[kHeaderWords + sym - 1u]) : 1.0f;
    return __fmul_rn(norm, level);
}

// ---------------------------------------------------------------------------
// What happens to the finished sum G = sum_k DECODE(c_k) of an element: it is stored to acc (if there is
// one) and, when the call carries the aggregation step of Algorithm 1, applied to the parameters at once,
// so that the sum is not written out and read again by an optimizer kernel:
//     y = w - (alpha / K) G,   y^l = w - l (alpha / K) G,   w <- y + mu (y^l - y^l_prev)
// (Sec. 4, "NUQSGD with momentum"; mu = 0 is Algorithm 1's own line and leaves y^l alone).  fp32, each line
// one fused multiply-add.
// ---------------------------------------------------------------------------
__device__ __forceinline__ float step_value(const SumParams& P, float w, float G, float* yl) {
    const float y = __fmaf_rn(-P.step_c, G, w);
    if (P.mu == 0.0f) return y;
    const float yl_next = __fmaf_rn(-P.step_lc, G, w);
    const float w_next = __fmaf_rn(P.mu, __fsub_rn(yl_next, *yl), y);
    *yl = yl_next;
    return w_next;
}
// element e (a multiple of 4) and the three behind it, with the parameters and y^l as they were
__device__ __forceinline__ void step4(const SumParams& P, uint64_t e, float4 G, float4 w, float4 yl) {
    if (P.acc) *reinterpret_cast<float4*>(P.acc + e) = G;
    w.x = step_value(P, w.x, G.x, &yl.x);
    w.y = step_value(P, w.y, G.y, &yl.y);
    w.z = step_value(P, w.z, G.z, &yl.z);
    w.w = step_value(P, w.w, G.w, &yl.w);
    *reinterpret_cast<float4*>(P.w + e) = w;
    if (P.mu != 0.0f) *reinterpret_cast<float4*>(P.yl + e) = yl;
}
__device__ __forceinline__ void finish4(const SumParams& P, uint64_t e, float4 G) {
    if (!P.w) {
        *reinterpret_cast<float4*>(P.acc + e) = G;
        return;
    }
    float4 yl = make_float4(0.f, 0.f, 0.f, 0.f);
    const float4 w = *reinterpret_cast<const float4*>(P.w + e);
    if (P.mu != 0.0f) yl = *reinterpret_cast<const float4*>(P.yl + e);
    step4(P, e, G, w, yl);
}
__device__ __forceinline__ void finish1(const SumParams& P, uint64_t e, float G) {
    if (P.acc) P.acc[e] = G;
    if (P.w) {
        float yl = P.mu != 0.0f ? P.yl[e] : 0.0f;
        P.w[e] = step_value(P, P.w[e], G, &yl);
        if (P.mu != 0.0f) P.yl[e] = yl;
    }
}

// the first n < 4 elements from e on
__device__ __forceinline__ void finish_part(const SumParams& P, uint64_t e, float4 G, uint32_t n) {
    if (n > 0u) finish1(P, e, G.x);
    if (n > 1u) finish1(P, e + 1, G.y);
    if (n > 2u) finish1(P, e + 2, G.z);
}

// Per stream of the call: what its header says, checked once per CTA.
struct StreamHead {
    const uint32_t* hdr;
    uint64_t cwords;         // container words the header declares
    uint32_t ok, mode, levelset, nlev, width;
    uint32_t hwords;         // header words: 16, plus the level table of a level-table stream
};

// Levels of a level set (zero included) and the bits of a fixed-width field: sign and level index.
__device__ __forceinline__ uint32_t level_count(uint32_t levelset, uint32_t s) { return levelset == kLevelsUniform ? (1u << s) + 1u : s + 2u; }
__device__ __forceinline__ uint32_t field_width(uint32_t nlev) { return 1u + (32u - __clz(nlev - 1u)); }

// A container's header checked against the call's arguments.  Its words are loaded at once: the checks would otherwise
// wait for one word after the other.
__device__ __forceinline__ StreamHead read_head(const Geometry& G, const uint32_t* hdr) {
    const uint4 a = *reinterpret_cast<const uint4*>(hdr), b = *reinterpret_cast<const uint4*>(hdr + 4), c = *reinterpret_cast<const uint4*>(hdr + 8);
    const uint32_t flags = b.z;
    const uint32_t levelset = (flags >> 8) & 0xffu, mode = (flags >> 16) & 0xffu;
    const uint64_t hd = (uint64_t)a.z | ((uint64_t)a.w << 32);
    const uint64_t hnblk = (uint64_t)c.x | ((uint64_t)c.y << 32);
    const uint64_t cbits = (uint64_t)c.z | ((uint64_t)c.w << 32);
    bool ok = a.x == kMagic && a.y == kVersion && hd == G.d && b.x == G.bucket &&
              b.y == G.s && b.w == kSB && levelset <= 2u && mode <= 2u &&
              (flags & 0xffu) <= 1u && !(levelset == kLevelsUniform && G.s > 8u) && (cbits & 31u) == 0;
    const uint32_t nlev = level_count(levelset, G.s);
    const uint32_t hwords = kHeaderWords + (levelset == kLevelsTable ? ((G.s + 1u) & ~1u) : 0u) + (mode == kModeCoded ? 2u : 0u);
    if (ok && mode == kModeCoded) {                         // the lengths must be those of a prefix code of at most 7 bits
        ok = levelset != kLevelsUniform && G.s <= kMaxCodedS;
        uint32_t kraft = 0;
        for (uint32_t j = 0; ok && j <= G.s; ++j) {
            const uint32_t len = (hdr[hwords - 2u + (j >> 2)] >> (8u * (j & 3u))) & 0xffu;
            ok = len >= 1u && len <= kMaxCodedS;
            kraft += ok ? 1u << (kMaxCodedS - len) : 0u;
        }
        ok = ok && kraft <= (1u << kMaxCodedS);
    }
    if (ok && levelset == kLevelsTable) {                   // the levels must increase strictly inside (0, 1)
        float below = 0.0f;
        for (uint32_t j = 0; j < G.s; ++j) {
            const float l = __uint_as_float(hdr[kHeaderWords + j]);
            ok = ok && below < l;
            below = l;
        }
        ok = ok && below < 1.0f;
    }
    const uint32_t width = field_width(nlev);
    const uint64_t cwords = cbits >> 5;
    if (ok && mode != kModeFixed) {
        ok = hnblk == G.nblk && cwords > hwords + 2 * (G.nblk + 1);
    } else if (ok) {
        const uint32_t rec_words = 1u + (G.bucket * width + 31u) / 32u;
        const uint64_t last_len = G.d - (G.nb - 1) * G.bucket;
        ok = hnblk == G.nb &&
             cwords == hwords + (G.nb - 1) * (uint64_t)rec_words + 1 + (last_len * width + 31) / 32;
    }
    StreamHead h;
    h.hdr = hdr; h.cwords = cwords; h.ok = ok ? 1u : 0u; h.mode = mode; h.levelset = levelset;
    h.nlev = nlev; h.width = width; h.hwords = hwords;
    return h;
}

__device__ __forceinline__ uint64_t pack2(float a, float b) {
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ float2 unpack2(uint64_t v) {
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
    return r;
}
// two fp32 operations at once, each rounded like the single one
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
    uint64_t r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
// A rounded product that is added to something afterwards.  Not mul.rn.f32x2: with that and an add.rn.f32x2 behind it sums came
// out as if product and sum had been rounded once, in spite of the rounding modifiers (they differ from the oracle's then).
// A fused operation that adds -0 changes no product, and it cannot be fused again as long as the -0 is not known to be one.
__device__ __forceinline__ uint64_t product2(uint64_t a, uint64_t b, uint64_t minus_zero) { return fma2(a, b, minus_zero); }
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b) {
    uint64_t r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}

}  // namespace nuq

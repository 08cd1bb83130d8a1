// DECODE + aggregate for calls whose streams are all in the fixed-width mode: no chains to walk (token streams:
// nuq_decode_chains.cu), so a thread turns whole words of fields into values and adds them in stream order.
#include <type_traits>

#include "nuq_decode_common.cuh"
#include "nuq_launch.h"

namespace nuq {

// All streams in the fixed-width mode with the same field width W (sign bit + level index, MSB first):
// no tokens to walk, so a thread takes 32 consecutive elements (W words of every stream, never across a
// bucket: buckets are multiples of 256 elements), adds the K dequantized values of each element in
// stream order in registers and stores the 32 sums.  Same arithmetic and order as the general path.
template <uint32_t W, uint32_t LEVELSET>
__device__ __forceinline__ void decode_all_fixed(const DecodeParams& P, const StreamHead* heads) {
    const Geometry& G = P.geo;
    const uint64_t ngroups = (G.d + 31) / 32;
    const uint32_t nlev = heads[0].nlev;
    const uint32_t exp_bias = (126u - G.s) << 23;           // exponent field of 2^(-1-s)
    const float uni_scale = __uint_as_float((127u - G.s) << 23);
    uint32_t max_sym = 0;
    const uint32_t rec_words = 1u + G.bucket * W / 32u;
    const uint64_t last_len = G.d - (G.nb - 1) * G.bucket;
    constexpr uint32_t fmask = (1u << W) - 1u, smask = (1u << (W - 1u)) - 1u;
    for (uint64_t grp = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; grp < ngroups; grp += (uint64_t)gridDim.x * blockDim.x) {
        const uint64_t e0 = 32 * grp, b = e0 / G.bucket;
        const uint32_t eb = (uint32_t)(e0 - b * G.bucket);                         // first element within its bucket
        const uint32_t nel = G.d - e0 < 32 ? (uint32_t)(G.d - e0) : 32u;
        const uint32_t bucket_len = b == G.nb - 1 ? (uint32_t)last_len : G.bucket;
        const uint32_t avail = (bucket_len * W + 31u) / 32u - (eb / 32u) * W;      // field words of the record from here on
        float* dst = P.acc + e0;
        // branch free: a zero symbol adds +0 (the sums never are -0, so that changes nothing), the
        // largest symbol seen is checked once at the end; `whole`: all 32 elements exist
        auto body = [&](auto whole) {
#pragma unroll
            for (uint32_t half = 0; half < 2; ++half) {     // 16 elements at a time: the sums stay in few registers
                float acc[16];
#pragma unroll
                for (int i = 0; i < 16; ++i) acc[i] = 0.0f;
                for (uint32_t k = 0; k < P.K; ++k) {
                    const uint32_t* rec = heads[k].hdr + kHeaderWords + b * rec_words;
                    const float norm = __uint_as_float(__ldg(rec));
                    const uint32_t* fw = rec + 1u + (eb / 32u) * W;
                    // the words that hold fields 16 * half .. 16 * half + 15
                    constexpr uint32_t kHalfWords = (16u * W + 31u) / 32u + 1u;
                    const uint32_t w0 = (16u * half * W) >> 5;
                    uint32_t words[kHalfWords + 1];
#pragma unroll
                    for (uint32_t j = 0; j < kHalfWords; ++j) words[j] = w0 + j < avail ? __ldg(fw + w0 + j) : 0u;
                    words[kHalfWords] = 0;
#pragma unroll
                    for (uint32_t i = 0; i < 16; ++i) {
                        const uint32_t bit = (16u * half + i) * W - 32u * w0, a = bit >> 5, sh = bit & 31u;
                        const uint32_t field = sh + W <= 32u ? (words[a] >> (32u - sh - W)) & fmask
                                                             : __funnelshift_l(words[a + 1], words[a], sh) >> (32u - W);
                        const uint32_t sym = field & smask;
                        // exponential: l_j = 2^(j-1-s) (exact scaling);  uniform: l_k = k / 2^s
                        const float level = LEVELSET == kLevelsExp ? __uint_as_float((sym << 23) + exp_bias)
                                                                   : __fmul_rn((float)sym, uni_scale);
                        const float mag = sym ? __fmul_rn(norm, level) : 0.0f;
                        const float v = __uint_as_float(__float_as_uint(mag) ^ ((field << (32u - W)) & 0x80000000u));
                        if (decltype(whole)::value || 16u * half + i < nel) {
                            max_sym = max(max_sym, sym);
                            acc[i] += v;
                        }
                    }
                }
                if (decltype(whole)::value) {
#pragma unroll
                    for (int i = 0; i < 16; i += 4)
                        *reinterpret_cast<float4*>(dst + 16 * half + i) = make_float4(acc[i], acc[i + 1], acc[i + 2], acc[i + 3]);
                } else {
#pragma unroll
                    for (int i = 0; i < 16; ++i)
                        if (16u * half + (uint32_t)i < nel) dst[16 * half + i] = acc[i];
                }
            }
        };
        if (nel == 32u) body(std::true_type());
        else body(std::false_type());
    }
    if (max_sym >= nlev) latch_status(P.ws, kErrBadStream);
}

// The same for the 4-bit fields of the paper's "4-bit" variant (exponential levels with s = 3 .. 6; a
// sign bit and a 3-bit level index) and buckets that are multiples of 2048 elements, where almost all
// the work can be taken out of the inner loop: a CTA takes a tile of up to 8192 elements of one bucket
// by ticket, builds, per stream, the table of the 16 values a field can stand for (+-norm * level, the
// same multiplication as everywhere else, so the sums are bit-identical), and then every thread turns 8
// consecutive elements -- one word of every stream -- into table look-ups and adds, in stream order.
// Symbols that do not exist are found on whole words (a carry out of the index bits).
template <uint32_t LEVELSET>
__device__ __forceinline__ void decode_fixed4_tiles(const DecodeParams& P, const StreamHead* heads) {
    __shared__ float s_tab[kMaxK][16];
    __shared__ unsigned long long s_ticket;
    const Geometry& G = P.geo;
    const uint32_t K = P.K, tid = threadIdx.x;
    const uint32_t nlev = heads[0].nlev;                    // <= 8
    const uint32_t rec_words = 1u + G.bucket / 8u;
    const uint32_t tile_elems = G.bucket < kBLK ? G.bucket : kBLK;
    const uint32_t tiles_per_bucket = G.bucket / tile_elems;
    const uint64_t ntiles = G.nb * tiles_per_bucket;
    const uint64_t last_len = G.d - (G.nb - 1) * G.bucket;
    const uint32_t over = (8u - nlev) * 0x11111111u;        // added to the index bits, a missing symbol carries into bit 3
    uint32_t bad = 0;
    for (;;) {
        __syncthreads();                                    // the tables and the ticket of the previous tile are no longer read
        if (tid == 0) s_ticket = atomicAdd(reinterpret_cast<unsigned long long*>(&P.ws->dec_ticket[P.epoch & 1u]), 1ull);
        __syncthreads();
        const uint64_t tile = s_ticket;
        if (tile >= ntiles) break;
        const uint64_t b = tile / tiles_per_bucket;
        const uint32_t part = (uint32_t)(tile % tiles_per_bucket);
        const uint32_t bucket_len = b == G.nb - 1 ? (uint32_t)last_len : G.bucket;
        const uint32_t first = part * tile_elems;           // first element of the tile within its bucket
        if (first >= bucket_len) continue;
        const uint32_t tile_len = bucket_len - first < tile_elems ? bucket_len - first : tile_elems;
        for (uint32_t t = tid; t < 16u * K; t += blockDim.x) {
            const uint32_t k = t >> 4, f = t & 15u, sym = f & 7u;
            const float norm = __uint_as_float(__ldg(heads[k].hdr + kHeaderWords + b * rec_words));
            const float v = sym && sym < nlev ? level_times_norm(norm, LEVELSET, G.s, sym, heads[k].hdr) : 0.0f;
            s_tab[k][f] = (f & 8u) ? -v : v;
        }
        __syncthreads();
        float* const dst_tile = P.acc + b * G.bucket + first;
        const uint64_t word0 = kHeaderWords + b * rec_words + 1u + first / 8u;     // the tile's first field word in a container
        // Two groups of eight elements per thread and step (el and el + 8 * blockDim.x): the words of both are
        // asked for before either is used, which keeps twice as many loads in flight.
        const uint32_t stride = 8u * blockDim.x;
        for (uint32_t el = 8u * tid; el < tile_len; el += 2u * stride) {
            const bool second = el + stride < tile_len;
            float sum[2][8];
#pragma unroll
            for (int h = 0; h < 2; ++h)
#pragma unroll
                for (int i = 0; i < 8; ++i) sum[h][i] = 0.0f;
            for (uint32_t k0 = 0; k0 < K; k0 += 8u) {
                uint32_t wv[2][8];
#pragma unroll
                for (uint32_t j = 0; j < 8; ++j) {
                    const uint32_t* w = heads[k0 + j < K ? k0 + j : 0u].hdr + word0 + el / 8u;
                    wv[0][j] = k0 + j < K ? __ldg(w) : 0u;
                    wv[1][j] = k0 + j < K && second ? __ldg(w + blockDim.x) : 0u;
                }
#pragma unroll
                for (uint32_t j = 0; j < 8; ++j) {
                    if (k0 + j < K) {
                        const char* tab = reinterpret_cast<const char*>(s_tab[k0 + j]);
#pragma unroll
                        for (int h = 0; h < 2; ++h) {
                            const uint32_t x = wv[h][j];
                            bad |= ((x & 0x77777777u) + over) & 0x88888888u;
                            // the eight fields times four (byte offsets into the table), four to a register
                            const uint32_t a = (x >> 2) & 0x3C3C3C3Cu, c = (x << 2) & 0x3C3C3C3Cu;   // elements 0 2 4 6 / 1 3 5 7 from the top byte
                            sum[h][0] += *reinterpret_cast<const float*>(tab + __byte_perm(a, 0u, 0x4443));
                            sum[h][1] += *reinterpret_cast<const float*>(tab + __byte_perm(c, 0u, 0x4443));
                            sum[h][2] += *reinterpret_cast<const float*>(tab + __byte_perm(a, 0u, 0x4442));
                            sum[h][3] += *reinterpret_cast<const float*>(tab + __byte_perm(c, 0u, 0x4442));
                            sum[h][4] += *reinterpret_cast<const float*>(tab + __byte_perm(a, 0u, 0x4441));
                            sum[h][5] += *reinterpret_cast<const float*>(tab + __byte_perm(c, 0u, 0x4441));
                            sum[h][6] += *reinterpret_cast<const float*>(tab + __byte_perm(a, 0u, 0x4440));
                            sum[h][7] += *reinterpret_cast<const float*>(tab + __byte_perm(c, 0u, 0x4440));
                        }
                    }
                }
            }
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const uint32_t e0 = el + h * stride;
                if (h == 1 && !second) break;
                float* dst = dst_tile + e0;
                if (e0 + 8u <= tile_len) {
                    *reinterpret_cast<float4*>(dst) = make_float4(sum[h][0], sum[h][1], sum[h][2], sum[h][3]);
                    *reinterpret_cast<float4*>(dst + 4) = make_float4(sum[h][4], sum[h][5], sum[h][6], sum[h][7]);
                } else {
#pragma unroll
                    for (uint32_t i = 0; i < 8; ++i)
                        if (e0 + i < tile_len) dst[i] = sum[h][i];
                }
            }
        }
    }
    if (bad) latch_status(P.ws, kErrBadStream);
}

// The kernel of that path.  It is launched when the library believes that all streams are in the
// fixed-width mode (it wrote them itself) and the call wants the sums only (a call that carries the
// aggregation step takes the general kernel, which applies it); it checks the headers like the general kernel and, if they
// say otherwise, leaves everything to the general kernel, which is launched behind it in any case and
// returns at once when this one has done the work.
__global__ void __launch_bounds__(256) decode_fixed_kernel(const __grid_constant__ DecodeParams P) {
    __shared__ StreamHead heads[kMaxK];
    __shared__ uint32_t s_width;
    for (uint32_t k = threadIdx.x; k < P.K; k += blockDim.x) heads[k] = read_head(P.geo, P.streams[k]);
    __syncthreads();
    if (threadIdx.x == 0) {
        bool same = true;
        for (uint32_t k = 0; k < P.K; ++k)
            same = same && heads[k].ok && heads[k].mode == kModeFixed && heads[k].levelset == heads[0].levelset &&
                   heads[k].levelset != kLevelsTable;       // (streams with a level table take the general kernel)
        s_width = same ? heads[0].width : 0u;
        if (same && blockIdx.x == 0) *reinterpret_cast<volatile uint32_t*>(&P.ws->dec_done_epoch) = P.epoch;   // tell the general kernel
        if (blockIdx.x == 0) P.ws->dec_ticket[(P.epoch & 1u) ^ 1u] = 0;     // the next call's counter (nobody uses it during this call)
    }
    __syncthreads();
    if (heads[0].levelset == kLevelsExp) {                  // s <= 14: at most 16 levels, 5 bits
        switch (s_width) {
            case 3: decode_all_fixed<3, kLevelsExp>(P, heads); break;
            case 4:
                if (P.geo.bucket % 2048u == 0) decode_fixed4_tiles<kLevelsExp>(P, heads);
                else decode_all_fixed<4, kLevelsExp>(P, heads);
                break;
            case 5: decode_all_fixed<5, kLevelsExp>(P, heads); break;
            default: break;
        }
        return;
    }
    switch (s_width) {
        case 3: decode_all_fixed<3, kLevelsUniform>(P, heads); break;
        case 4: decode_all_fixed<4, kLevelsUniform>(P, heads); break;
        case 5: decode_all_fixed<5, kLevelsUniform>(P, heads); break;
        case 6: decode_all_fixed<6, kLevelsUniform>(P, heads); break;
        case 7: decode_all_fixed<7, kLevelsUniform>(P, heads); break;
        case 8: decode_all_fixed<8, kLevelsUniform>(P, heads); break;
        case 9: decode_all_fixed<9, kLevelsUniform>(P, heads); break;
        case 10: decode_all_fixed<10, kLevelsUniform>(P, heads); break;
        default: break;
    }
}

cudaError_t launch_decode(const DecodeParams& P, int sms, cudaStream_t stream) {
    if (P.after_fixed) {
        const uint64_t groups = (P.geo.d + 31) / 32, want_fixed = (groups + 255) / 256, cap_fixed = (uint64_t)sms * 4u;
        decode_fixed_kernel<<<(unsigned)(want_fixed < cap_fixed ? want_fixed : cap_fixed), 256, 0, stream>>>(P);
        if (cudaGetLastError() != cudaSuccess) return cudaErrorUnknown;
    }
    return launch_decode_chains(P, sms, stream);
}

}  // namespace nuq

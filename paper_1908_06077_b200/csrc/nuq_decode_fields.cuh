// DECODE + aggregate of calls whose streams are all in the fixed-width mode with the same field width and kind of levels:
// no chains to walk.  The kernels for it, and the way here from the kernels for token streams, are in nuq_decode_chains.cu.
//
// A warp takes units of up to four 256-element sub-blocks; a lane has eight consecutive elements of each, one word of
// every stream when fields have 4 bits.  A field, its sign bit included, is looked up in a table of level values in shared
// memory, multiplied by the bucket's norm and added in stream order: an element of a stream is one extraction, one look-up
// and one fused multiply-add.  No value depends on a unit, so nothing is built per
// unit and warps never meet.  An item, that is the fields of a unit in up to eight streams, is brought into the warp's
// shared memory by one bulk copy per stream, two items ahead, so that no address is computed per word and the bytes in
// flight do not depend on registers.  The copies are started in one place of the loop, which begins two rounds early: their
// code is there when the first item is.
// 25.6 x 10^6 elements, K = 8 (200 MB with 4 bits, 31 us at the memory's rate): 4-bit fields 51 us repeated and 56 us behind
// eight encode calls, level tables 57 us, 3 bits 56 us, 5 to 8 bits 72 to 85 us, 9 and 10 bits up to 107 us, buckets of 256 and 512
// 62 to 67 us; 65536 elements 4.8 us.  (A kernel of one thread per 32 elements: 104 to 117 us, level tables 547 us.)  What bounds
// it is the look-ups (one shared-memory word per element and stream, a wavefront per 32 of them) and, with four warps per
// scheduler, what the warps wait for.
#pragma once
#include <type_traits>

#include "nuq_async.cuh"
#include "nuq_decode_common.cuh"

namespace nuq {

constexpr uint32_t kFieldStreams = 8;                       // streams of an item
// words of a stream that hold a lane's eight fields (8 W bits from a byte boundary on)
__host__ __device__ constexpr uint32_t field_words(uint32_t w) { return w == 4u ? 1u : w == 7u || w > 8u ? 3u : 2u; }
// sub-blocks of a unit: two items fit the warp's shared memory
__host__ __device__ constexpr uint32_t field_slots(uint32_t w) { return w <= 5u ? 4u : 2u; }
// bytes of an item's part of a stream: the fields, norms between them, and what 16-byte alignment adds
__host__ __device__ constexpr uint32_t field_pitch(uint32_t w) { return 4u * ((field_slots(w) * (8u * w + 1u) + 6u + 3u) & ~3u); }
// a warp's shared memory: two items with their norms, two mbarriers
__host__ __device__ constexpr uint32_t field_warp_bytes(uint32_t w) { return 2u * kFieldStreams * field_pitch(w) + 256u + 16u; }

// Bytes between the tables of two streams (level-table streams have one each).
__host__ __device__ constexpr uint32_t field_table_stride(uint32_t w) { return w <= 6u ? 256u : 4u << w; }

// The level values by field; a symbol that does not exist stands for NaN, which the sums keep (and are checked for).
// `heads`: of the n streams whose own levels they are (level tables).
__device__ __noinline__ void build_field_tables(const Geometry& G, uint32_t levelset, const StreamHead* heads, uint32_t n, unsigned char* tables) {
    const uint32_t nlev = level_count(levelset, G.s), w = field_width(nlev), stride = field_table_stride(w);
    for (uint32_t i = threadIdx.x; i < n << w; i += blockDim.x) {
        const uint32_t k = i >> w, f = i & ((1u << w) - 1u), sym = f & ((1u << (w - 1u)) - 1u);
        float v = sym == 0u ? 0.0f : sym < nlev ? level_times_norm(1.0f, levelset, G.s, sym, levelset == kLevelsTable ? heads[k].hdr : nullptr)
                                                : __uint_as_float(0x7FC00000u);
        if (f >> (w - 1u)) v = -v;
        *reinterpret_cast<float*>(tables + k * stride + 4u * f) = v;
    }
}

__device__ __forceinline__ uint32_t field_word(uint32_t addr) {
    uint32_t v;
    asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(addr));
    return v;
}
// A table entry (tables do not change any more)
__device__ __forceinline__ float field_level(uint32_t addr) {
    float v;
    asm("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(addr));
    return v;
}

// The levels of a lane's eight fields.  `tab` is a multiple of 256 and of the table's size, so that it can be put together
// with a field's offset instead of added to it.
template <uint32_t W>
__device__ __forceinline__ void eight_levels(const uint32_t (&x)[field_words(W)], uint32_t shift, uint32_t tab, float (&l)[8]) {
    if (W == 4u) {
        // the fields times four, four to a register: elements 0 2 4 6 and 1 3 5 7 from the top byte
        const uint32_t a = (x[0] >> 2) & 0x3C3C3C3Cu, c = (x[0] << 2) & 0x3C3C3C3Cu;
        l[0] = field_level(__byte_perm(a, tab, 0x7653)); l[1] = field_level(__byte_perm(c, tab, 0x7653));
        l[2] = field_level(__byte_perm(a, tab, 0x7652)); l[3] = field_level(__byte_perm(c, tab, 0x7652));
        l[4] = field_level(__byte_perm(a, tab, 0x7651)); l[5] = field_level(__byte_perm(c, tab, 0x7651));
        l[6] = field_level(__byte_perm(a, tab, 0x7650)); l[7] = field_level(__byte_perm(c, tab, 0x7650));
        return;
    }
    constexpr uint32_t kWords = field_words(W);
    uint32_t y[4] = {0, 0, 0, 0};                           // the fields from bit 31 of y[0] on
#pragma unroll
    for (uint32_t i = 0; i < kWords; ++i) y[i] = __funnelshift_l(i + 1u < kWords ? x[i + 1u < kWords ? i + 1u : i] : 0u, x[i], shift);
#pragma unroll
    for (uint32_t i = 0; i < 8; ++i) {
        const uint32_t bit = i * W, at = bit >> 5, end = (bit & 31u) + W;          // in y[at], and in y[at + 1] if end > 32
        const uint32_t t = end <= 30u ? y[at] >> (30u - end) : end <= 32u ? y[at] << (end - 30u) : __funnelshift_r(y[at + 1u], y[at], 62u - end);
        l[i] = field_level((t & (((1u << W) - 1u) << 2)) | tab);
    }
}

// Four fields of a fixed-width stream, elements e .. e + 3 of the vector (e a multiple of 4), as values.  Returns
// false when a symbol does not exist.
__device__ __noinline__ bool four_fields(const Geometry& G, const StreamHead& hd, uint64_t e, float4* out) {
    const uint32_t wd = hd.width, smask = (1u << (wd - 1u)) - 1u;
    const uint64_t b = e / G.bucket;
    const uint32_t in_bucket = (uint32_t)(e - b * G.bucket), rec_words = 1u + (G.bucket * wd + 31u) / 32u;
    const uint64_t blen = G.d - b * G.bucket < G.bucket ? G.d - b * G.bucket : G.bucket;
    const uint32_t last = (uint32_t)((blen * wd + 31u) / 32u) - 1u, bit = in_bucket * wd, wi = bit >> 5;
    const uint32_t* const rec = hd.hdr + hd.hwords + b * rec_words;
    const float norm = __uint_as_float(rec[0]);
    const uint32_t x0 = rec[1u + min(wi, last)], x1 = rec[1u + min(wi + 1u, last)], x2 = rec[1u + min(wi + 2u, last)];
    const uint64_t win = ((uint64_t)__funnelshift_l(x1, x0, bit) << 32) | __funnelshift_l(x2, x1, bit);   // 64 bits from the first field on
    float v[4];
    bool ok = true;
#pragma unroll
    for (uint32_t c = 0; c < 4; ++c) {
        const uint32_t field = (uint32_t)(win >> (64u - (c + 1u) * wd)) & ((1u << wd) - 1u), sym = field & smask;
        v[c] = 0.0f;
        if (sym == 0u || e + c >= G.d) continue;
        if (sym >= hd.nlev) ok = false;
        else v[c] = level_times_norm(norm, hd.levelset, G.s, sym, hd.hdr);
        if (field >> (wd - 1u)) v[c] = -v[c];
    }
    *out = make_float4(v[0], v[1], v[2], v[3]);
    return ok;
}

// The rare parts are calls that need nothing of the loop's registers: inlined, their code lay between that of the common
// ones, and four warps per scheduler wait for instructions as much as for data (check_fields alone: 56.0 -> 52.3 us).

// A lane's elements (e0 + 256 q + 0 .. 7) of a unit with norms that are not all of ordinary size, from the containers.
__device__ __noinline__ void unit_slowly(const DecodeParams& P, const StreamHead* heads, uint64_t e0, uint32_t slots) {
    bool ok = true;
#pragma unroll 1
    for (uint32_t i = 0; i < 2u * slots; ++i) {
        const uint64_t e = e0 + kSB * (i / 2u) + 4u * (i & 1u);
        if (e >= P.geo.d) break;
        float4 sum = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 1
        for (uint32_t k = 0; k < P.K; ++k) {
            float4 v;
            ok = four_fields(P.geo, heads[k], e, &v) && ok;
            sum.x += v.x; sum.y += v.y; sum.z += v.z; sum.w += v.w;
        }
        if (e + 4u <= P.geo.d) finish4(P.sum, e, sum);
        else finish_part(P.sum, e, sum, (uint32_t)(P.geo.d - e));
    }
    if (!ok) latch_status(P.ws, kErrBadStream);
}

// Looks for symbols that do not exist among a lane's elements.
__device__ __noinline__ void check_fields(const DecodeParams& P, const StreamHead* heads, uint64_t e0, uint32_t slots) {
    bool ok = true;
    for (uint32_t i = 0; i < 2u * slots; ++i) {
        const uint64_t e = e0 + kSB * (i / 2u) + 4u * (i & 1u);
        for (uint32_t k = 0; k < P.K && e < P.geo.d; ++k) {
            float4 v;
            ok = four_fields(P.geo, heads[k], e, &v) && ok;
        }
    }
    if (!ok) latch_status(P.ws, kErrBadStream);
}

// The sums of a unit that reaches behind the vector's end.
template <uint32_t SLOTS>
__device__ __forceinline__ void finish_end(const SumParams& P, uint64_t d, uint64_t e0, uint32_t slots, const float (&sum)[SLOTS][8]) {
    float v[8u * SLOTS];                                    // (a copy that can be indexed)
#pragma unroll
    for (uint32_t i = 0; i < 8u * SLOTS; ++i) v[i] = sum[i / 8u][i % 8u];
#pragma unroll 1
    for (uint32_t i = 0; i < 2u * slots; ++i) {
        const uint64_t e = e0 + kSB * (i / 2u) + 4u * (i & 1u);
        if (e >= d) return;
        const float4 G = make_float4(v[4u * i], v[4u * i + 1u], v[4u * i + 2u], v[4u * i + 3u]);
        if (e + 4u <= d) finish4(P, e, G);
        else finish_part(P, e, G, (uint32_t)(d - e));
    }
}

// eight values to a multiple of 32 bytes: a whole sector per lane and instruction
__device__ __forceinline__ void store8(float* dst, const float (&v)[8]) {
    asm volatile("st.global.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(dst), "f"(v[0]), "f"(v[1]), "f"(v[2]), "f"(v[3]),
                 "f"(v[4]), "f"(v[5]), "f"(v[6]), "f"(v[7])
                 : "memory");
}

// EXACT: powers of two, whose product with a norm of ordinary size is exact, so that one fused operation gives the sum
// that two would; else product and sum are rounded one after the other.  Other norms (tiny ones; not finite ones, where an
// element without a symbol has no product) take the slow way.
// `mine`: the warp's shared memory (a multiple of 16).  `tables_ready`: the table of levels has been built, and all threads
// have met since.
template <uint32_t W, bool EXACT>
__device__ __forceinline__ void decode_fields(const DecodeParams& P, const StreamHead* heads, unsigned char* table_memory, bool tables_ready, uint32_t mine) {
    constexpr uint32_t kWords = field_words(W), kSlots = field_slots(W), kPitch = field_pitch(W), kItem = kFieldStreams * kPitch;
    const Geometry& G = P.geo;
    const uint32_t lane = lane_id(), K = P.K, spb = G.bucket / kSB, rec_words = 1u + G.bucket * W / 32u, hwords = heads[0].hwords;
    const uint32_t tab_stride = heads[0].levelset == kLevelsTable ? field_table_stride(W) : 0u;
    const uint32_t nsub = (uint32_t)((G.d + kSB - 1u) / kSB), nfull = (uint32_t)(G.d / kSB), nwarps = gridDim.x * (blockDim.x >> 5);
    const uint32_t S = min(max(nsub / nwarps, 1u), kSlots);                    // (a small call: one sub-block for every warp first)
    const uint32_t nunits = (nsub + S - 1u) / S;
    const uint32_t shift = W == 4u ? 0u : 8u * ((W * lane) & 3u);
    const uint32_t norms = mine + 2u * kItem, full = norms + 256u, tables = smem_u32(table_memory);

    struct Item {
        uint32_t unit, k0, b, in;                           // first stream; the first sub-block: the in-th of bucket b
    };
    const uint32_t stride_b = nwarps * S / spb, stride_in = nwarps * S - stride_b * spb;
    auto behind = [&](Item it) {
        it.k0 += kFieldStreams;
        if (it.k0 >= K) {
            it.k0 = 0;
            it.unit += nwarps;
            it.b += stride_b;
            it.in += stride_in;
            if (it.in >= spb) {
                it.in -= spb;
                it.b += 1u;
            }
        }
        return it;
    };
    auto norms_before = [&](const Item& it, uint32_t q) {   // bucket boundaries between the first sub-block and the q-th behind it
        return (it.in + q >= spb ? 1u : 0u) + (it.in + q >= 2u * spb ? 1u : 0u) + (it.in + q >= 3u * spb ? 1u : 0u);
    };
    // starts the copies of an item: lane j the fields of stream j, lane q * 8 + j the norm of slot q in stream j.  (No fence
    // in front of the bulk copies: the words they overwrite have been read, and the one place that writes such words has
    // its own.  A fence waits for the copies in flight.)
    auto start_copy = [&](const Item& it, uint32_t stage) {
        if (it.unit < nunits) {
            const uint32_t sub = it.unit * S, slots = min(S, nsub - sub), count = min(K - it.k0, kFieldStreams);
            const uint64_t rec = hwords + (uint64_t)it.b * rec_words;
            const uint32_t q = lane / kFieldStreams, j = lane % kFieldStreams;
            // where the fields start in every container, in words, and how many there are (with the norms between them)
            const uint64_t first = rec + 1u + it.in * (8u * W), from = first & ~(uint64_t)3u;
            const uint32_t words = (uint32_t)(first - from) + slots * 8u * W + norms_before(it, slots - 1u);
            const uint32_t dst = mine + stage * kItem, bar = full + 8u * stage;
            if (lane < kFieldStreams) {
                if (lane < count) {
                    const StreamHead& hd = heads[it.k0 + lane];
                    uint32_t n = (words + 3u) & ~3u;
                    if (__builtin_expect(hd.cwords - from < n, 0)) {    // the container ends here: its last words one by one
                        const uint32_t have = (uint32_t)(hd.cwords - from);
                        n = have & ~3u;
                        for (uint32_t i = n; i < have; ++i)
                            asm volatile("st.shared.u32 [%0], %1;" ::"r"(dst + lane * kPitch + 4u * i), "r"(hd.hdr[from + i]) : "memory");
                        for (uint32_t i = have; i < words; ++i)                 // and no symbols behind them
                            asm volatile("st.shared.u32 [%0], %1;" ::"r"(dst + lane * kPitch + 4u * i), "r"(0u) : "memory");
                        fence_async_proxy();                // (before a later item's copy to the same place)
                    }
                    if (n != 0u) bulk_load_unfenced(dst + lane * kPitch, hd.hdr + from, 4u * n, bar);
                    else mbar_arrive(bar);
                } else {
                    mbar_arrive(bar);
                }
            }
            if (q < slots && j < count)
                asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(norms + 128u * stage + 4u * lane), "l"(heads[it.k0 + j].hdr + rec + norms_before(it, q) * rec_words) : "memory");
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };

    if (lane == 0) {
        mbar_init(full, kFieldStreams);
        mbar_init(full + 8u, kFieldStreams);
    }
    fence_async_proxy();                                    // (rows may have been cleared here)
    __syncwarp();
    bool in_time = true;
    Item cur = {}, next = {}, after;                        // item n is copied two rounds before it is added up
    after.unit = (threadIdx.x >> 5) * gridDim.x + blockIdx.x;
    after.k0 = 0;
    after.b = after.unit * S / spb;
    after.in = after.unit * S - after.b * spb;
    const bool wide = (reinterpret_cast<uintptr_t>(P.sum.acc) & 31u) == 0;
    float sum[kSlots][8];
    bool ordinary = true;                                   // so far, all norms of the unit
    const uint32_t params = P.sum.w == nullptr ? 0u : P.sum.mu != 0.0f ? 2u : 1u;        // vectors of parameters
    auto clear = [&] {
#pragma unroll
        for (uint32_t i = 0; i < 8u * kSlots; ++i) sum[i / 8u][i % 8u] = 0.0f;
    };
    clear();
    for (uint32_t n = 0; n < 2u || cur.unit < nunits; ++n) {
        const uint32_t stage = n & 1u;
        const uint32_t sub = cur.unit * S, slots = min(S, nsub - sub), count = min(K - cur.k0, kFieldStreams);
        const uint64_t e0 = (uint64_t)sub * kSB + 8u * lane;
        if (n >= 2u) {
            if (cur.k0 == 0u && sub + slots <= nfull && lane < params)    // the parameters, for later
                asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"((lane == 0u ? P.sum.w : P.sum.yl) + (uint64_t)sub * kSB), "r"(4u * kSB * slots) : "memory");
            asm volatile("cp.async.wait_group 1;" ::: "memory");
            const float norm = lane / kFieldStreams < slots && lane % kFieldStreams < count ? __uint_as_float(field_word(norms + 128u * stage + 4u * lane)) : 0.0f;
            const bool fine = EXACT ? norm == 0.0f || (norm >= 0x1p-100f && norm < 0x1p126f) : fabsf(norm) <= 3.4028234e38f;
            const bool all_fine = __all_sync(0xffffffffu, fine);
            __syncwarp();                                   // the other lanes' norms are there
            in_time = mbar_wait(full + 8u * stage, ((n >> 1) & 1u) ^ 1u) && in_time;
            ordinary = ordinary && all_fine;
            if (__builtin_expect(ordinary, 1)) {
                // where the lane's fields of each slot start
                const uint32_t first = mine + stage * kItem + 4u * ((hwords + cur.b * rec_words + 1u + cur.in * (8u * W)) & 3u) + (W * lane & ~3u);
                auto add_item = [&](auto whole) {           // whole: all slots, within one bucket
                    uint32_t at = first, nrm = norms + 128u * stage, tab = tables + cur.k0 * tab_stride;
#pragma unroll 1
                    for (uint32_t j = 0; j < count; ++j) {
#pragma unroll
                        for (uint32_t q = 0; q < kSlots; ++q) {
                            if (!decltype(whole)::value && q >= slots) break;
                            const uint32_t from = decltype(whole)::value ? at : at + 4u * norms_before(cur, q);
                            uint32_t x[kWords];
                            float l[8];
#pragma unroll
                            for (uint32_t i = 0; i < kWords; ++i) x[i] = field_word(from + 32u * W * q + 4u * i);
                            const float nm = __uint_as_float(field_word(nrm + 4u * kFieldStreams * q));
                            eight_levels<W>(x, shift, tab, l);
#pragma unroll
                            for (int i = 0; i < 8; ++i) sum[q][i] = EXACT ? __fmaf_rn(l[i], nm, sum[q][i]) : __fadd_rn(sum[q][i], __fmul_rn(l[i], nm));
                        }
                        at += kPitch;
                        nrm += 4u;
                        tab += tab_stride;
                    }
                };
                if (slots == kSlots && cur.in + kSlots <= spb) add_item(std::true_type());
                else add_item(std::false_type());
            }
            __syncwarp();                                   // the item's words and norms have been read
        }
        start_copy(after, stage);
        if (n == 0u && !tables_ready) {                     // (every warp is here)
            build_field_tables(G, heads[0].levelset, heads, heads[0].levelset == kLevelsTable ? K : 1u, table_memory);
            __syncthreads();
        }
        if (n >= 2u && cur.k0 + kFieldStreams >= K) {       // the sums are complete
            const SumParams out = P.sum;
            float check = 0.0f;                             // NaN when a sum is not finite
#pragma unroll
            for (uint32_t i = 0; i < 8u * kSlots; ++i) check = __fmaf_rn(sum[i / 8u][i % 8u], 0.0f, check);
            auto value = [&](uint32_t q, uint32_t h) {
                return make_float4(sum[q][4u * h], sum[q][4u * h + 1u], sum[q][4u * h + 2u], sum[q][4u * h + 3u]);
            };
            if (__builtin_expect(!ordinary, 0)) {
                unit_slowly(P, heads, e0, slots);
            } else if (__builtin_expect(sub + slots > nfull, 0)) {
                finish_end<kSlots>(out, G.d, e0, slots, sum);
            } else if (out.w == nullptr) {
#pragma unroll
                for (uint32_t q = 0; q < kSlots; ++q) {
                    if (q >= slots) break;
                    float* const dst = out.acc + e0 + kSB * q;
                    if (wide) {
                        store8(dst, sum[q]);
                    } else {
                        *reinterpret_cast<float4*>(dst) = value(q, 0u);
                        *reinterpret_cast<float4*>(dst + 4) = value(q, 1u);
                    }
                }
            } else {
#pragma unroll
                for (uint32_t i0 = 0; i0 < 2u * kSlots; i0 += 4u) {            // the loads of two slots are on their way together
                    float4 w[4], yl[4];
#pragma unroll
                    for (uint32_t i = 0; i < 4; ++i) {
                        const uint64_t e = e0 + kSB * ((i0 + i) / 2u) + 4u * (i & 1u);
                        w[i] = yl[i] = make_float4(0.f, 0.f, 0.f, 0.f);
                        if ((i0 + i) / 2u < slots) {
                            w[i] = *reinterpret_cast<const float4*>(out.w + e);
                            if (out.mu != 0.0f) yl[i] = *reinterpret_cast<const float4*>(out.yl + e);
                        }
                    }
#pragma unroll
                    for (uint32_t i = 0; i < 4; ++i)
                        if ((i0 + i) / 2u < slots) step4(out, e0 + kSB * ((i0 + i) / 2u) + 4u * (i & 1u), value((i0 + i) / 2u, i & 1u), w[i], yl[i]);
                }
            }
            if (__builtin_expect(ordinary && !(check == 0.0f), 0)) check_fields(P, heads, e0, slots);   // a symbol that does not exist?
            ordinary = true;
            clear();
        }
        cur = next;
        next = after;
        after = behind(after);
    }
    if (__any_sync(0xffffffffu, !in_time) && lane == 0) latch_status(P.ws, kErrTimeout);
}

// The same as a function, for the kernels of token streams: inlined there, fields and tokens share registers and the
// instruction cache.  Kernel: a type of the calling kernel's own, so that each has a function for itself.  (In one that several
// kernels called, built by nvcc 12.9, store8 wrote its first element only, in all kernels but one.  The source has no reason for
// that: the same text is right where it is inlined and where one kernel calls it.)
template <uint32_t W, bool EXACT, class Kernel>
__device__ __noinline__ void decode_fields_call(const DecodeParams& P, const StreamHead* heads, unsigned char* table_memory, uint32_t mine) {
    decode_fields<W, EXACT>(P, heads, table_memory, false, mine);
}

}  // namespace nuq

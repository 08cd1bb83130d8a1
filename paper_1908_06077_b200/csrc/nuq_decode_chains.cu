// DECODE + aggregate (App. A decoding; Algorithm 1, aggregation line) of token streams: the K
// workers' containers are decoded and summed into one fp32 vector.
//
// A warp takes a unit of S consecutive 256-element sub-blocks in all K streams (up to 32 streams at a
// time), K S <= 32, and works in two passes:
//
//   walk   lane (j, q) walks the chain of tokens of stream j, sub-block q and writes the symbol of every
//          token, one byte, to its place in the chain's row of 256 positions in shared memory.  All
//          chains of a warp advance side by side; nothing is kept in lists, so the density of the
//          symbols does not matter.
//   add    the rows are read across: a lane takes four consecutive elements of all K streams, turns
//          their symbols into values and adds them up in ascending stream order, starting from +0, so
//          the sum equals ((0 + q_0) + q_1) + ... bit for bit.  It is stored (or applied to the
//          parameters) once, 512 contiguous bytes per warp and step.
//
// The walk is a chain of dependent steps.  What a step waits for is one table look-up and two shifts:
//
//   table   the next 13 bits of the chain give a whole token, or two that fit: the bits, the gap and the symbols.
//           A token that is longer than 13 bits is taken in two steps: the code of a gap ends with the
//           bit 0, which is itself the code of gap 1, so an entry that stands for the gap's code without
//           its last bit and for a gap one smaller, without a symbol, leaves an ordinary token of gap 1
//           behind.  What the table cannot resolve at all (gaps from 128 on, long level codes) takes
//           Algorithm 2's loop.
//   window  64 bits hi:lo, shifted by the token's length and refilled to at least 32 valid bits every
//           second step: a look-up needs the 13 top bits, so 32 last for two steps.  (Refilled at every
//           step the walk takes 3 of 18 instructions more: ResNet-50, K = 8 85.2 us, now 83.4.)
//   end     every lane has its own copy of its chain (cp.async, 112 bytes at a time) and puts ones
//           behind the chain's last bit: thirteen ones are no token, the table says "0 bits, no gap, no
//           symbol", and the lane stands still until all others have ended too.  So a step has no
//           branches; the lanes look up every four steps.
//
// The copy of the next unit's chains runs during the add pass, the block offsets of the one after that
// are on their way during the walk.  16 warps fit an SM (12 KB each: rows, chain copies).
#include <map>

#include "nuq_async.cuh"
#include "nuq_decode_common.cuh"
#include "nuq_decode_fields.cuh"
#include "nuq_launch.h"

namespace nuq {

constexpr uint32_t kTokBits = 13;                       // prefix bits the token table resolves
constexpr uint32_t kTokEntries = 1u << kTokBits;
constexpr uint32_t kChainMaxWarps = 16;                 // warps per CTA, one CTA per SM
constexpr uint32_t kChunkWords = 28;                    // words of its chain a lane holds at a time
constexpr uint32_t kChunkSlack = 3;                     // of these, words it needs behind the chain's last one
constexpr uint32_t kCodeBytes = 256;                    // per stream: level code by 7-bit prefix, or level by symbol
constexpr uint32_t kLevelBytes = 64;                    // per stream: level table
constexpr size_t kChainSmem = 227u * 1024u - 512u;      // (512 bytes: static)

// A row of symbols: 256 positions and a place for what a malformed chain would write behind them.  Rows of
// neighbouring lanes start in neighbouring banks.
template <class Sym>
struct Row {
    static constexpr uint32_t kPitch = kSB * sizeof(Sym) + 4u;
    static constexpr uint32_t kWarpBytes = 32u * kPitch + 128u + 32u * 4u * kChunkWords;   // rows, norms, chain copies
    static_assert(kWarpBytes >= field_warp_bytes(5) && kWarpBytes >= field_warp_bytes(10), "fixed-width streams use the same memory");
};

// Token table entries.  Bits 0-4: bits consumed (0: not resolved here); bits 8-15: gap; on top, from Symbol::kShift on, the symbol, signed
// (0: none, only a part of the gap).  Symbols: for exponential levels the upper byte of the level (with its sign) as
// an fp16 number, 2^(j-1-s) being one without mantissa bits; for uniform levels the signed index.
// With symbols of one byte an entry may stand for two tokens (pairs): the gap is then that of both together, bits 5-7 are the
// second one's (0: one token), bits 16-23 the first one's symbol.  Dense symbols take 5 bits a token and most look-ups give two;
// sparse ones (8 bits and more) one in four, and gain next to nothing (K = 8 ResNet-50 containers: largest-magnitude norms with uniform
// levels 193 -> 150 us, s = 4 in buckets of 512 149 -> 125, 8192 83.4 -> 81.1, s = 3 there 72.2 -> 72.6, s = 2 69.6 -> 70.5; with what came
// since 72.0 and 69.7; 33 streams of 6 x 10^6 elements with s = 3 are 1.2 % slower than without, 114.6 and 116.0).
constexpr uint32_t kLenMask = 31u, kGap2Shift = 5u, kMaxGap2 = 7u, kGapShift = 8u, kFirstShift = 16u;
template <class Sym>
constexpr bool kPairs = sizeof(Sym) == 1;
template <class Sym>
struct Symbol {
    static constexpr uint32_t kShift = sizeof(Sym) == 1 ? 24u : 22u;
    static __device__ __forceinline__ uint32_t exponential(uint32_t index, uint32_t negative, uint32_t s) {
        return ((negative ? 0x80u : 0u) | ((14u + index - s) << 2)) << kShift;
    }
    static __device__ __forceinline__ uint32_t uniform(uint32_t index, uint32_t negative) { return (negative ? 0u - index : index) << kShift; }
};

// Tables as kept in device memory: kTabErc and kTabGaps with one token to an entry, bits 22-30 the level index (1 .. 255), bit 31 its
// sign; and ERC tokens in pairs, in the format above but for the symbols, which are level indices (1 .. 31: longer codes do not fit) with the sign in bit 7.
constexpr uint32_t kTabPairs = 2u, kIndexShift = 22u;
__device__ uint32_t g_token_tables[3][kTokEntries];

// ERC^-1 of the nbits-bit prefix idx from bit `pos` on (Algorithm 2, decoding): false when the code does not end within it.
static bool erc_of_prefix(uint32_t idx, uint32_t nbits, uint32_t* pos, uint32_t* value) {
    uint32_t N = 1;
    for (;;) {
        if (*pos >= nbits) return false;
        if (!((idx >> (nbits - 1u - *pos)) & 1u)) {
            *pos += 1;
            *value = N;
            return true;
        }
        const uint32_t nb = N + 1u;
        if (*pos + nb > nbits) return false;
        N = (idx >> (nbits - *pos - nb)) & ((1u << nb) - 1u);
        *pos += nb;
    }
}

cudaError_t upload_token_tables() {
    static uint32_t tab[3][kTokEntries];
    for (uint32_t i = 0; i < kTokEntries; ++i) {
        uint32_t pos = 0, gap = 0;
        tab[kTabErc][i] = tab[kTabGaps][i] = 0;
        if (!erc_of_prefix(i, kTokBits, &pos, &gap) || gap >= kSB) continue;
        tab[kTabGaps][i] = pos | (gap << kGapShift);
        uint32_t at = pos + 1u, index = 0;                  // behind the sign bit
        if (at < kTokBits && erc_of_prefix(i, kTokBits, &at, &index) && index <= 255u)
            tab[kTabErc][i] = at | (gap << kGapShift) | (index << kIndexShift) | (((i >> (kTokBits - 1u - pos)) & 1u) << 31);
        else if (pos > 1u)
            tab[kTabErc][i] = (pos - 1u) | ((gap - 1u) << kGapShift);
    }
    for (uint32_t i = 0; i < kTokEntries; ++i) {
        auto symbol = [](uint32_t e) { return (e >> kIndexShift & 0x1ffu) | (e >> 31) << 7; };
        const uint32_t e = tab[kTabErc][i], then = tab[kTabErc][(i << (e & kLenMask)) & (kTokEntries - 1u)];
        const uint32_t len = (e & kLenMask) + (then & kLenMask), gap2 = (then >> kGapShift) & 0xffu;
        if (symbol(e) && symbol(then) && len <= kTokBits && gap2 <= kMaxGap2)
            tab[kTabPairs][i] = len | gap2 << kGap2Shift | ((e & 0xff00u) + (gap2 << kGapShift)) | symbol(e) << kFirstShift | symbol(then) << 24;
        else
            tab[kTabPairs][i] = (e & 0xffffu) | symbol(e) << 24;
    }
    const cudaError_t e = cudaMemcpyToSymbol(g_token_tables, tab, sizeof(tab));
    // (the copy goes by the default stream, whose end kernels of a non-blocking stream do not wait for)
    return e == cudaSuccess ? cudaStreamSynchronize(nullptr) : e;
}

__device__ __forceinline__ void copy_async16(uint32_t dst, const void* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void copy_async4(uint32_t dst, const void* src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ uint32_t lds_u32(uint32_t addr) {
    uint32_t v;
    asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(addr) : "memory");
    return v;
}

// One Elias-recursive integer from bit `at` of the 32-bit window on; false when it does not end within it.
__device__ __forceinline__ bool erc_in_window(uint32_t win, uint32_t* at, uint32_t* value) {
    uint32_t N = 1;
#pragma unroll 1
    for (int it = 0; it < 5; ++it) {
        const uint32_t w = win << *at;
        if (!(w >> 31)) {
            *at += 1;
            *value = N;
            return true;
        }
        const uint32_t nb = N + 1u;
        if (*at + nb > 31u) return false;
        N = w >> (32u - nb);
        *at += nb;
    }
    return false;
}

// A stream with coded level indices brings its own code, w0 and w1: the words' lengths, one byte each.  Canonical words: level
// indices by (length, index), the first word all zeros, each next one the previous plus one; so the word of index j (+ 1) counts, in
// units of its own length, the words before it.  Returned with its length << 16.
__device__ __forceinline__ uint32_t level_word(uint32_t w0, uint32_t w1, uint32_t s, uint32_t j) {
    auto len_of = [&](uint32_t j) { return ((j < 4u ? w0 : w1) >> (8u * (j & 3u))) & 0xffu; };
    const uint32_t lj = len_of(j);
    uint32_t word = 0;
    for (uint32_t k = 0; k <= s; ++k) {
        const uint32_t lk = len_of(k);
        if (lk < lj || (lk == lj && k < j)) word += 1u << (lj - lk);
    }
    return word | lj << 16;
}
// The level index and its word's length (<< 8) by the next 7 bits, 0 where no word starts (possible only with an incomplete code).
template <class WordOf>
__device__ __forceinline__ uint32_t coded_entry(WordOf word_of, uint32_t s, uint32_t prefix) {
    for (uint32_t j = 0; j <= s; ++j) {
        const uint32_t w = word_of(j);
        if ((prefix >> (kMaxCodedS - (w >> 16))) == (w & 0xffffu)) return (j + 1u) | (w >> 16 << 8);
    }
    return 0;
}

// A token the table does not resolve, by Algorithm 2's loop; a gap longer than 1 is taken on its own, as in the table.
// Returns the entry the table would hold, 0 when the bits are no token.
template <class Sym>
__device__ __noinline__ uint32_t long_token(uint32_t win, const StreamHead& hd, const uint16_t* code, bool gaps_only, uint32_t s) {
    uint32_t at = 0, gap = 0, index = 0;
    if (!erc_in_window(win, &at, &gap) || gap > kSB) return 0u;
    if (at > 1u) return (at - 1u) | ((gap - 1u) << kGapShift);
    at = 2u;
    if (hd.mode == kModeCoded) {
        if (!gaps_only) return 0u;                          // (such a token would be in the table)
        const uint32_t c = code[(win << 2) >> (32u - kMaxCodedS)];
        at += c >> 8;
        index = c & 0xffu;
    } else if (!erc_in_window(win, &at, &index)) {
        return 0u;
    }
    if (index == 0u || index >= hd.nlev) return 0u;
    const uint32_t negative = (win >> 30) & 1u;
    return at | (1u << kGapShift) | (hd.levelset == kLevelsUniform ? Symbol<Sym>::uniform(index, negative) : Symbol<Sym>::exponential(index, negative, s));
}

// What a lane knows of its chain.
struct Chain {
    const uint32_t* src;     // the 16-byte piece of the container that holds its first bit
    uint64_t left;           // words of the container from there on
    uint32_t bit, len;       // first bit behind src, bits (0: no chain here)
    float norm;
    bool good;               // what the container says about it makes sense
};

// One pass over the words a lane holds: walks `bits` bits from bit `from` of the copy on, or further up to the end of
// the token that crosses that point.  LONG: the copy ends before the chain does (in some lane); else every chain is
// followed by ones.  `row` is the address of the last position taken, and is moved on.
// GAPS: the table holds gaps alone; the level index comes from the stream's own table (by the 7 bits behind the sign).
template <class Sym, bool LONG, bool GAPS>
__device__ __forceinline__ uint32_t walk_body(uint32_t copy, uint32_t from, uint32_t bits, uint32_t tab, uint32_t& row, uint32_t row_end,
                                              const StreamHead& hd, const uint16_t* code, uint32_t s, bool& good) {
    const uint32_t sh = from & 31u, w0 = copy + 4u * (from >> 5);
    const uint32_t x0 = lds_u32(w0), x1 = lds_u32(w0 + 4u), x2 = lds_u32(w0 + 8u);
    uint32_t hi = __funnelshift_l(x1, x0, sh);
    uint32_t lo = sh ? x1 << sh : 0u, nxt = sh ? x2 : x1;
    uint32_t next = w0 + (sh ? 12u : 8u);                   // where the word behind nxt lies
    // q counts the bits down to c; its low five bits are those of the number of valid bits in hi:lo
    const uint32_t c = (0u - sh - bits) & 31u;
    uint32_t q = bits + c, q_was = q, e = 0, at = row;
    auto look_up = [&] {
        const uint32_t addr = tab + ((hi >> (32u - kTokBits)) << 2);
        if (LONG) asm("{\n\t.reg .pred p;\n\tsetp.gt.s32 p, %1, %2;\n\tmov.b32 %0, 0;\n\t@p ld.shared.u32 %0, [%3];\n\t}"
                      : "=r"(e) : "r"(q), "r"(c), "r"(addr));
        else asm("ld.shared.u32 %0, [%1];" : "=r"(e) : "r"(addr));
        if (GAPS) {
            const uint32_t behind = hi << (e & kLenMask), cw = code[(behind << 1) >> (32u - kMaxCodedS)];
            const uint32_t len = (e & kLenMask) + 1u + (cw >> 8), index = cw & 0xffu, negative = behind >> 31;
            const uint32_t sym = hd.levelset == kLevelsUniform ? Symbol<Sym>::uniform(index, negative) : Symbol<Sym>::exponential(index, negative, s);
            e = e != 0u && cw != 0u ? len | (e & (0xffu << kGapShift)) | sym : 0u;
        }
    };
    // brings the number of valid bits back to 32 at least, when it is below; fewer than 32 have been taken since it was done last
    auto refill = [&] {
        asm("{\n\t.reg .pred p;\n\t.reg .b32 t;\n\txor.b32 t, %4, %5;\n\tand.b32 t, t, 32;\n\tsetp.ne.u32 p, t, 0;\n\t"
            "shf.r.wrap.b32 t, %2, 0, %4;\n\t@p or.b32 %0, %0, t;\n\t@p shf.r.wrap.b32 %1, 0, %2, %4;\n\t"
            "@p ld.shared.u32 %2, [%3];\n\t@p add.u32 %3, %3, 4;\n\t}"
            : "+r"(hi), "+r"(lo), "+r"(nxt), "+r"(next) : "r"(q), "r"(q_was));
        q_was = q;
    };
    if (bits != 0u) {
        look_up();
        for (;;) {
            if (e == 0u) {
                if ((int32_t)(q - c) <= 0) break;
                e = long_token<Sym>(hi, hd, code, GAPS, s);
                if (e == 0u) {
                    good = false;
                    break;
                }
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                at += __byte_perm(e, 0u, 0x4441) * (uint32_t)sizeof(Sym);
                at = min(at, row_end);
                // (no symbol: a part of a gap, or a lane that stands still)
                if (sizeof(Sym) == 1)
                    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %1, 0;\n\t@p st.shared.u8 [%0], %1;\n\t}" ::"r"(at), "r"(e >> Symbol<Sym>::kShift) : "memory");
                else
                    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %1, 0;\n\t@p st.shared.u16 [%0], %1;\n\t}" ::"r"(at), "r"((int32_t)e >> Symbol<Sym>::kShift) : "memory");
                if (kPairs<Sym> && !GAPS) {
                    const uint32_t gap2 = (e >> kGap2Shift) & kMaxGap2;
                    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %1, 0;\n\t@p st.shared.u8 [%0], %2;\n\t}" ::"r"(at - gap2), "r"(gap2), "r"(e >> kFirstShift) : "memory");
                }
                hi = __funnelshift_l(lo, hi, e);
                lo = __funnelshift_l(0u, lo, e);
                q -= e & kLenMask;
                // A look-up needs 13 valid bits, so of 32 two tokens can be taken (18 bits at most by a long one, 13 by an entry of the table).
                // (With symbols of two bytes there are fewer warps and the look-ups' latency counts: each goes ahead of its refill.)
                if (!GAPS && sizeof(Sym) == 2) look_up();
                if (GAPS || sizeof(Sym) == 2 || (u & 1)) refill();
                if (GAPS || sizeof(Sym) == 1) look_up();
            }
        }
    }
    row = at;
    return bits + c - q;                                    // bits taken
}

// (the common walk is part of the kernel's loop, the others are calls)
template <class Sym, bool LONG, bool GAPS>
__device__ __noinline__ uint32_t walk_rare(uint32_t copy, uint32_t from, uint32_t bits, uint32_t tab, uint32_t& row, uint32_t row_end,
                                           const StreamHead& hd, const uint16_t* code, uint32_t s, bool& good) {
    return walk_body<Sym, LONG, GAPS>(copy, from, bits, tab, row, row_end, hd, code, s, good);
}

// two fp16 numbers given by their upper bytes, in the upper bytes of the halves
__device__ __forceinline__ uint64_t halves(uint32_t h) {
    uint64_t r;
    asm("{\n\t.reg .b16 a, b;\n\t.reg .f32 x, y;\n\tmov.b32 {a, b}, %1;\n\tcvt.f32.f16 x, a;\n\tcvt.f32.f16 y, b;\n\tmov.b64 %0, {x, y};\n\t}" : "=l"(r) : "r"(h));
    return r;
}

// Four symbols of one stream: powers of two (exponential levels, by way of fp16) ...
template <class Sym>
__device__ __forceinline__ void four_powers(uint32_t row, uint64_t* v01, uint64_t* v23) {
    const uint32_t x = lds_u32(row), y = sizeof(Sym) == 1 ? x : lds_u32(row + 4u);
    *v01 = halves(sizeof(Sym) == 1 ? __byte_perm(x, 0u, 0x1404) : __byte_perm(x, 0u, 0x2404));
    *v23 = halves(sizeof(Sym) == 1 ? __byte_perm(x, 0u, 0x3424) : __byte_perm(y, 0u, 0x2404));
}
// ... or signed level indices (uniform levels), put into the mantissa of 2^23: converting integers takes four times as long.
template <class Sym>
__device__ __forceinline__ void four_indices(uint32_t row, uint64_t* v01, uint64_t* v23) {
    constexpr bool kBytes = sizeof(Sym) == 1;
    const uint32_t flip = kBytes ? 0x80808080u : 0x80008000u, top = 0x4B000000u;
    const float bias = -(8388608.0f + (kBytes ? 128.0f : 32768.0f));
    const uint32_t x = lds_u32(row) ^ flip, y = kBytes ? x : lds_u32(row + 4u) ^ flip;
    const float m0 = __uint_as_float(__byte_perm(x, top, kBytes ? 0x7650 : 0x7610)), m1 = __uint_as_float(__byte_perm(x, top, kBytes ? 0x7651 : 0x7632)),
                m2 = __uint_as_float(__byte_perm(y, top, kBytes ? 0x7652 : 0x7610)), m3 = __uint_as_float(__byte_perm(y, top, kBytes ? 0x7653 : 0x7632));
    *v01 = add2(pack2(m0, m1), pack2(bias, bias));
    *v23 = add2(pack2(m2, m3), pack2(bias, bias));
}

// The add pass of a unit.
struct AddPass {
    const StreamHead* heads;           // of the group's streams
    const unsigned char* levels;       // their level tables, kLevelBytes each ...
    uint32_t by_symbol;                // ... and levels by symbol (alike == 3), kCodeBytes each: shared-memory address, a multiple of 256
    uint32_t rows, norms;              // shared-memory addresses
    uint32_t S, streams;
    uint32_t alike;                    // all streams are tokens of exponential (0), uniform (1) or table (3) levels; else 2
    bool last, carried;                // the last group of streams; sums of earlier groups are in `carry`
};

// NB sub-blocks from sub-block q0 of the unit on; e: the lane's first element, 128 more for each half of a sub-block.
template <class Sym, int NB, bool MANY>
__device__ __forceinline__ void add_block(const DecodeParams& P, const AddPass& A, uint32_t q0, uint64_t e, uint64_t (&carry)[4]) {
    const Geometry& G = P.geo;
    const uint32_t lane = lane_id(), s = G.s;
    uint64_t sum[4 * NB];                                   // two halves of each, four elements in two pairs
#pragma unroll
    for (int i = 0; i < 4 * NB; ++i) sum[i] = 0;
    if (MANY && NB == 1 && A.carried) {
#pragma unroll
        for (int i = 0; i < 4; ++i) sum[i] = carry[i];
    }
    uint32_t nrm = A.norms + 4u * q0, at = A.rows + q0 * Row<Sym>::kPitch + 4u * lane * (uint32_t)sizeof(Sym);
    const uint64_t minus_zero = pack2(P.minus_zero, P.minus_zero);
    const float step = __uint_as_float((127u - s) << 23);   // 2^-s
    auto add_rows = [&](auto value) {
#pragma unroll
        for (int b = 0; b < NB; ++b) {
            const float nm = __uint_as_float(lds_u32(nrm + 4u * b));
#pragma unroll
            for (int h = 2 * b; h < 2 * b + 2; ++h)
                value(at + b * Row<Sym>::kPitch + (h & 1) * 128u * (uint32_t)sizeof(Sym), nm, sum[2 * h], sum[2 * h + 1]);
        }
    };
    auto add_exp = [&](uint32_t row, float nm, uint64_t& s01, uint64_t& s23) {
        uint64_t a, b;
        four_powers<Sym>(row, &a, &b);
        s01 = fma2(a, pack2(nm, nm), s01);
        s23 = fma2(b, pack2(nm, nm), s23);
    };
    auto add_uniform = [&](uint32_t row, float nm, uint64_t& s01, uint64_t& s23) {
        uint64_t a, b;
        four_indices<Sym>(row, &a, &b);
        const float n = nm * step;                          // exact, like k 2^-s: either way one rounding of k nm 2^-s
        s01 = add2(s01, product2(a, pack2(n, n), minus_zero));
        s23 = add2(s23, product2(b, pack2(n, n), minus_zero));
    };
    if (A.alike == 0u) {
#pragma unroll 4 / NB
        for (uint32_t j = 0; j < A.streams; ++j, nrm += 4u * A.S, at += A.S * Row<Sym>::kPitch) add_rows(add_exp);
    } else if (A.alike == 1u) {
#pragma unroll 4 / NB
        for (uint32_t j = 0; j < A.streams; ++j, nrm += 4u * A.S, at += A.S * Row<Sym>::kPitch) add_rows(add_uniform);
    } else if (A.alike == 3u) {
        uint32_t by_symbol = A.by_symbol;
#pragma unroll 4 / NB
        for (uint32_t j = 0; j < A.streams; ++j, nrm += 4u * A.S, at += A.S * Row<Sym>::kPitch, by_symbol += kCodeBytes) {
            add_rows([&](uint32_t row, float nm, uint64_t& s01, uint64_t& s23) {
                const uint32_t x = lds_u32(row), y = sizeof(Sym) == 1 ? x : lds_u32(row + 4u);
                // a symbol's lower byte is the offset of its level
                const float l0 = field_level(__byte_perm(x, by_symbol, 0x7650)), l1 = field_level(__byte_perm(x, by_symbol, sizeof(Sym) == 1 ? 0x7651 : 0x7652)),
                            l2 = field_level(__byte_perm(y, by_symbol, sizeof(Sym) == 1 ? 0x7652 : 0x7650)), l3 = field_level(__byte_perm(y, by_symbol, sizeof(Sym) == 1 ? 0x7653 : 0x7652));
                s01 = add2(s01, product2(pack2(l0, l1), pack2(nm, nm), minus_zero));
                s23 = add2(s23, product2(pack2(l2, l3), pack2(nm, nm), minus_zero));
            });
        }
    } else {
#pragma unroll 1
        for (uint32_t j = 0; j < A.streams; ++j, nrm += 4u * A.S, at += A.S * Row<Sym>::kPitch) {
            const StreamHead& hd = A.heads[j];
            if (!hd.ok) continue;
            if (hd.mode == kModeFixed) {
                bool ok = true;
#pragma unroll
                for (int h = 0; h < 2 * NB; ++h) {
                    if (e + 128u * h < G.d) {
                        float4 v;
                        ok = four_fields(G, hd, e + 128u * h, &v) && ok;
                        sum[2 * h] = add2(sum[2 * h], pack2(v.x, v.y));
                        sum[2 * h + 1] = add2(sum[2 * h + 1], pack2(v.z, v.w));
                    }
                }
                if (!ok) latch_status(P.ws, kErrBadStream);
            } else {
                const float* const lv = reinterpret_cast<const float*>(A.levels + j * kLevelBytes);
                add_rows([&](uint32_t row, float nm, uint64_t& s01, uint64_t& s23) {
                    float v[4];
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        int32_t b;
                        if (sizeof(Sym) == 1) asm volatile("ld.shared.s8 %0, [%1];" : "=r"(b) : "r"(row + i) : "memory");
                        else asm volatile("ld.shared.s16 %0, [%1];" : "=r"(b) : "r"(row + 2u * i) : "memory");
                        float level = 0.0f;                 // (no product for an element without a symbol: the norm may not be finite)
                        if (b) {
                            const uint32_t field = ((uint32_t)b >> 2) & 31u;
                            level = hd.levelset == kLevelsUniform ? (float)b * __uint_as_float((127u - s) << 23)
                                    : hd.levelset == kLevelsTable ? lv[field + s - 15u] : __uint_as_float((field + 112u) << 23);
                            level = __fmul_rn(nm, level);
                            if (hd.levelset != kLevelsUniform && (b & 0x80)) level = -level;
                        }
                        v[i] = level;
                    }
                    s01 = add2(s01, pack2(v[0], v[1]));
                    s23 = add2(s23, pack2(v[2], v[3]));
                });
            }
        }
    }
    if (MANY && NB == 1 && !A.last) {
#pragma unroll
        for (int i = 0; i < 4; ++i) carry[i] = sum[i];
        return;
    }
    auto value = [&](int h) {
        const float2 a = unpack2(sum[2 * h]), b = unpack2(sum[2 * h + 1]);
        return make_float4(a.x, a.y, b.x, b.y);
    };
    if (e + 128u * (2 * NB - 1) + 4u <= G.d) {
        if (P.sum.w == nullptr) {
#pragma unroll
            for (int h = 0; h < 2 * NB; ++h) *reinterpret_cast<float4*>(P.sum.acc + e + 128 * h) = value(h);
        } else {
            constexpr int kAtOnce = NB == 1 ? 2 : 4;        // the loads of four steps are on their way together
#pragma unroll
            for (int h0 = 0; h0 < 2 * NB; h0 += kAtOnce) {
                float4 w[kAtOnce], yl[kAtOnce];
#pragma unroll
                for (int h = 0; h < kAtOnce; ++h) {
                    w[h] = *reinterpret_cast<const float4*>(P.sum.w + e + 128 * (h0 + h));
                    yl[h] = P.sum.mu != 0.0f ? *reinterpret_cast<const float4*>(P.sum.yl + e + 128 * (h0 + h)) : make_float4(0.f, 0.f, 0.f, 0.f);
                }
#pragma unroll
                for (int h = 0; h < kAtOnce; ++h) step4(P.sum, e + 128 * (h0 + h), value(h0 + h), w[h], yl[h]);
            }
        }
    } else {                                                // the end of the vector
#pragma unroll
        for (int h = 0; h < 2 * NB; ++h) {
            const uint64_t at_h = e + 128u * h;
            if (at_h + 4u <= G.d) finish4(P.sum, at_h, value(h));
            else if (at_h < G.d) finish_part(P.sum, at_h, value(h), (uint32_t)(G.d - at_h));
        }
    }
}

// Shared memory: the token table, the streams' tables and heads, then per warp its rows, norms and chain copies.
__host__ __device__ inline size_t chain_fixed_bytes(uint32_t K) {
    // (256: the codes start at a multiple of 256)
    return (4u * kTokEntries + 256u + (size_t)K * (kCodeBytes + kLevelBytes + sizeof(StreamHead)) + 15u) & ~(size_t)15u;
}

// Where things lie in it.
template <class Sym>
struct Layout {
    unsigned char* codes;
    unsigned char* levels;
    StreamHead* heads;
    unsigned char* field_tables;                            // fixed-width streams: where the token table would be, a multiple of 4096
    uint32_t rows;                                          // the warp's own
    __device__ __forceinline__ Layout(unsigned char* dsm, uint32_t K) {
        const uint32_t base = smem_u32(dsm);
        codes = dsm + 4u * kTokEntries + (0u - base & 255u);
        levels = codes + K * kCodeBytes;
        heads = reinterpret_cast<StreamHead*>(levels + K * kLevelBytes);
        field_tables = dsm + ((base + 4095u & ~4095u) - base);
        rows = base + (uint32_t)chain_fixed_bytes(K) + (threadIdx.x >> 5) * Row<Sym>::kWarpBytes;
    }
};

// An instance of the kernel for token streams.  Whatever makes instances differ is named here, and only here: the functions for
// fixed-width streams take the whole type as a template argument, so that no two kernels share one (decode_fields_call says why).
// MANY: more than 32 streams, in groups (the sums of a unit are kept in registers from group to group: an instance of its own,
// since these and the counters of groups cost the common one 2 % of its time in the walk).
// SHORT: blocks are of at most four sub-blocks, so that a unit's lengths are in a line of their own as a rule, which no unit before
// it has read; they are asked for a walk ahead (25 557 032 elements, buckets of 512: K = 8 123.6 -> 119.3 us, with the step 156 -> 148,
// K = 2 at 2^28 381 -> 362; buckets of 2048 and more gain nothing and lose up to 1 %: an instance of its own).
template <class SYMBOL, bool MANY_STREAMS, bool SHORT_BLOCKS>
struct Instance {
    using Sym = SYMBOL;
    static constexpr bool kMany = MANY_STREAMS, kShort = SHORT_BLOCKS;
};

// All streams in the fixed-width mode.  (16-bit symbols: s = 7 or 8, hence fields of 5 bits, or of 9 and 10 with uniform levels.)
template <class I>
__device__ __forceinline__ void fields_of_width(const DecodeParams& P, const StreamHead* heads, unsigned char* tables, uint32_t mine, uint32_t width) {
    constexpr bool kBytes = sizeof(typename I::Sym) == 1;
    if (heads[0].levelset == kLevelsExp) {
        if (width == 5u) return decode_fields_call<5, true, I>(P, heads, tables, mine);
        if (kBytes && width == 4u) return decode_fields_call<4, true, I>(P, heads, tables, mine);
        if (kBytes && width == 3u) return decode_fields_call<3, true, I>(P, heads, tables, mine);
    }
    if (width == 5u) return decode_fields_call<5, false, I>(P, heads, tables, mine);
    if (kBytes) {
        if (width == 3u) return decode_fields_call<3, false, I>(P, heads, tables, mine);
        if (width == 4u) return decode_fields_call<4, false, I>(P, heads, tables, mine);
        if (width == 6u) return decode_fields_call<6, false, I>(P, heads, tables, mine);
        if (width == 7u) return decode_fields_call<7, false, I>(P, heads, tables, mine);
        if (width == 8u) return decode_fields_call<8, false, I>(P, heads, tables, mine);
    } else {
        if (width == 9u) return decode_fields_call<9, false, I>(P, heads, tables, mine);
        if (width == 10u) return decode_fields_call<10, false, I>(P, heads, tables, mine);
    }
}

template <class Sym>
__device__ __forceinline__ void clear_rows(uint32_t rows) {
    for (uint32_t i = 16u * lane_id(); i < 32u * Row<Sym>::kPitch; i += 512u)
        asm volatile("st.shared.v4.u32 [%0], {%1, %1, %1, %1};" ::"r"(rows + i), "r"(0u) : "memory");
}

// The token table for ERC streams of one level set (kTabErc, kTabUniform), by all threads of the CTA.
template <class Sym>
__device__ __forceinline__ void build_erc_table(uint32_t* table, uint32_t kind, uint32_t s) {
    using Symbols = Symbol<Sym>;
    const uint4* src = reinterpret_cast<const uint4*>(g_token_tables[kPairs<Sym> ? kTabPairs : kTabErc]);
    const uint32_t top = kind == kTabUniform ? 1u << s : s + 1u;
    auto entry = [&](uint32_t e) {
        const uint32_t index = (e >> kIndexShift) & 0x1ffu, negative = e >> 31;
        if (index == 0u) return e;
        if (index > top) return 0u;
        return (e & 0xffffu) | (kind == kTabUniform ? Symbols::uniform(index, negative) : Symbols::exponential(index, negative, s));
    };
    // a ready-made pair with this call's symbols; 0 where there is no such index (long_token takes the first one then, if that exists)
    auto ready = [&](uint32_t e) {
        const uint32_t first = (e >> kFirstShift) & 31u, last = (e >> 24) & 31u;
        if (first > top || last > top) return 0u;
        if (last == 0u) return e;
        if (kind == kTabErc) return e + ((e & 0x1f1f0000u) * 3u) + ((14u - s) << 26) + (first ? (14u - s) << (kFirstShift + 2u) : 0u);
        const uint32_t f = e & 1u << 23 ? 0u - first : first, l = e >> 31 ? 0u - last : last;
        return (e & 0xffffu) | (f & 0xffu) << kFirstShift | l << 24;
    };
    // (rolled up: where the call comes behind other work its code has to be fetched, which takes longer than the loads: K = 4
    // ResNet-18 containers behind their encodes 38.9 us, 37.0 rolled up)
#pragma unroll 1
    for (uint32_t i = threadIdx.x; i < kTokEntries / 4u; i += blockDim.x) {
        uint4 e = __ldg(src + i);
        if (kPairs<Sym>) e = make_uint4(ready(e.x), ready(e.y), ready(e.z), ready(e.w));
        else e = make_uint4(entry(e.x), entry(e.y), entry(e.z), entry(e.w));
        reinterpret_cast<uint4*>(table)[i] = e;
    }
}

// Whatever table the streams need and the kernel has not prepared, with their level codes and level tables; all threads of the CTA.
// `words`: the level code of all streams (kTabCoded).  `several`: some warp has more than one unit.
template <class Sym>
__device__ __forceinline__ void prepare_tables(const DecodeParams& P, unsigned char* dsm, const uint32_t* words, uint32_t kind, uint32_t all_alike, bool several) {
    using Symbols = Symbol<Sym>;
    const Geometry& G = P.geo;
    const uint32_t K = P.K, tid = threadIdx.x;
    uint32_t* const table = reinterpret_cast<uint32_t*>(dsm);
    const Layout<Sym> at(dsm, K);
    unsigned char *const codes = at.codes, *const levels = at.levels;
    uint32_t first = K;                                     // the first token stream (all have the same code in the coded mode)
    for (uint32_t k = 0; k < K; ++k) {
        const StreamHead& hd = at.heads[k];
        if (!hd.ok || hd.mode == kModeFixed) continue;
        uint16_t* const code = reinterpret_cast<uint16_t*>(codes + k * kCodeBytes);
        if (kind == kTabGaps || (kind == kTabCoded && first == K)) {   // level index by the next 7 bits
            for (uint32_t i = tid; i < (1u << kMaxCodedS); i += blockDim.x) {
                uint32_t c = 0, at = 0, index = 0;
                if (kind == kTabCoded) c = coded_entry([&](uint32_t j) { return words[j]; }, G.s, i);     // (all streams have this code)
                else if (hd.mode == kModeCoded) c = coded_entry([&](uint32_t j) { return level_word(hd.hdr[hd.hwords - 2u], hd.hdr[hd.hwords - 1u], G.s, j); }, G.s, i);
                else if (erc_in_window(i << (32u - kMaxCodedS) | 0x01ffffffu, &at, &index) && at <= kMaxCodedS && index < hd.nlev) c = index | (at << 8);
                code[i] = (uint16_t)c;
            }
        }
        if (hd.levelset == kLevelsTable && tid <= G.s)
            reinterpret_cast<float*>(levels + k * kLevelBytes)[tid] = tid < G.s ? __uint_as_float(hd.hdr[kHeaderWords + tid]) : 1.0f;
        if (first == K) first = k;
    }
    if (kind == kTabCoded) __syncthreads();
    const uint16_t* const code = reinterpret_cast<const uint16_t*>(codes + (first == K ? 0u : first) * kCodeBytes);
    // the entry of the gap's code at prefix i joined with the streams' level code
    auto coded_token = [&](uint32_t e, uint32_t i) {
        const uint32_t at = e & kLenMask, low = e & 0xffffu;
        if (at == 0u) return 0u;
        const uint32_t rest = i << (32u - kTokBits + at), c = code[(rest << 1) >> (32u - kMaxCodedS)];
        const uint32_t len = at + 1u + (c >> 8);
        if (c != 0u && len <= kTokBits) return len | (low & (0xffu << kGapShift)) | Symbols::exponential(c & 0xffu, rest >> 31, G.s);
        return at > 1u ? (at - 1u) | ((low & (0xffu << kGapShift)) - (1u << kGapShift)) : 0u;
    };
    if (kPairs<Sym> && kind == kTabCoded && several) {
        // A level code's table in pairs, by way of the table of single tokens (kept where the rows will be): a token and the one behind it, if
        // that is a whole one and near enough.  (The bits behind the prefix are taken for zeros; they do not matter to a token that ends
        // within it.)  The entry behind prefix i is that of i moved up by a token's length, for neighbouring i a power of two
        // apart: entries are kept within 32 by the sum of their five-bit digits, which keeps them in different banks (2 us of 15
        // otherwise).  All this takes a microsecond more than single tokens: not where no warp has a second unit (65 536 elements 11.2 us
        // without, 12.6 with them; 8 x 10^6, K = 4: 27.3 and 26.0).
        uint32_t* const singles = reinterpret_cast<uint32_t*>(dsm + chain_fixed_bytes(K));
        auto place = [](uint32_t i) { return i ^ ((i >> 5 ^ i >> 10) & 31u); };
#pragma unroll 4
        for (uint32_t i = tid; i < kTokEntries; i += blockDim.x) singles[place(i)] = coded_token(__ldg(g_token_tables[kTabGaps] + i), i);
        __syncthreads();
#pragma unroll 4
        for (uint32_t i = tid; i < kTokEntries; i += blockDim.x) {
            const uint32_t e = singles[place(i)], then = singles[place((i << (e & kLenMask)) & (kTokEntries - 1u))];
            const uint32_t len = (e & kLenMask) + (then & kLenMask), gap2 = (then >> kGapShift) & 0xffu;
            const bool two = e >> 24 != 0u && then >> 24 != 0u && len <= kTokBits && gap2 <= kMaxGap2;
            table[i] = two ? len | gap2 << kGap2Shift | ((e & 0xff00u) + (gap2 << kGapShift)) | (e >> 24) << kFirstShift | (then & 0xff000000u) : e;
        }
        __syncthreads();
        clear_rows<Sym>(at.rows);
    } else if (kind == kTabCoded || kind == kTabGaps) {
        const uint4* const gaps = reinterpret_cast<const uint4*>(g_token_tables[kTabGaps]);
#pragma unroll 1
        for (uint32_t i = tid; i < kTokEntries / 4u; i += blockDim.x) {
            uint4 e = __ldg(gaps + i);
            if (kind == kTabCoded) e = make_uint4(coded_token(e.x, 4u * i), coded_token(e.y, 4u * i + 1u), coded_token(e.z, 4u * i + 2u), coded_token(e.w, 4u * i + 3u));
            reinterpret_cast<uint4*>(table)[i] = e;
        }
    } else if (kind != P.likely_table) {
        build_erc_table<Sym>(table, kind, G.s);
    }
    __syncthreads();
    if (all_alike == 3u) {                                  // levels by symbol, sign included (the codes are no longer needed)
        for (uint32_t i = tid; i < 64u * K; i += blockDim.x) {
            const uint32_t k = i >> 6, index = (i & 31u) + G.s - 14u;
            const float l = index >= 1u && index <= G.s + 1u ? reinterpret_cast<const float*>(levels + k * kLevelBytes)[index - 1u] : 0.0f;
            reinterpret_cast<float*>(codes + k * kCodeBytes)[i & 63u] = i & 32u ? -l : l;
        }
        __syncthreads();
    }
}

// Streams of any kind.
// CALLED: from a kernel for fixed-width streams, where those the call was made for are not; fields are then added one by one.
template <class I, bool CALLED>
__device__ __forceinline__ void decode_streams(const DecodeParams& P) {
    using Sym = typename I::Sym;
    constexpr bool MANY = I::kMany, SHORT = I::kShort;
    extern __shared__ __align__(128) unsigned char dsm[];
    __shared__ uint32_t s_kind, s_alike, s_fields, s_words[kMaxCodedS + 1];
    const Geometry& G = P.geo;
    const uint32_t K = P.K, tid = threadIdx.x, lane = tid & 31u, warp = tid >> 5;
    uint32_t* const table = reinterpret_cast<uint32_t*>(dsm);
    const Layout<Sym> at(dsm, K);
    unsigned char *const codes = at.codes, *const levels = at.levels;
    StreamHead* const heads = at.heads;
    const uint32_t rows = at.rows;
    const uint32_t norms = rows + 32u * Row<Sym>::kPitch;   // one per lane's chain
    const uint32_t copy = norms + 128u + lane * (4u * kChunkWords);   // this lane's words of its chain

    // The kernel is launched with programmatic stream serialization: its CTAs take the SMs as the kernel in front leaves
    // them, build the table that the call is likely to need and clear their rows, and wait here until that kernel has ended.
    // Nothing before the wait touches memory that another kernel writes.  The kernel behind is let in early only by calls
    // that give every warp several units: a small encode call let in early finds room only where CTAs of this kernel have
    // left and is packed onto a few SMs, four CTAs each (a step of 10^6 elements, K = 3: 66 -> 74 us).
    if (!CALLED) {
        if (P.let_next) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
        if (P.likely_table == kTabErc || P.likely_table == kTabUniform) build_erc_table<Sym>(table, P.likely_table, G.s);
        clear_rows<Sym>(rows);
        asm volatile("griddepcontrol.wait;" ::: "memory");
    }

    // ---- headers against the call's arguments, once per stream; then what kind of table serves all the token streams ----
    if (warp == 0) {
        enum : uint32_t { kCoded = 1, kErc = 2, kUniform = 4, kOther = 8, kTabled = 16, kOdd = 32, kNotFields = 64, kSeveralCodes = 128 };
        uint32_t found = 0;                                 // of these, among the streams
        uint32_t first0 = 0, first1 = 0;                    // the code lengths of the first coded stream
        uint32_t levels0 = 0, width0 = 0;                   // of the first stream
        for (uint32_t k0 = 0; k0 < K; k0 += 32u) {
            const uint32_t k = k0 + lane;
            StreamHead hd = {};
            if (k < K) {
                heads[k] = hd = read_head(G, P.streams[k]);
                if (!hd.ok) latch_status(P.ws, kErrBadStream);
            }
            if (k0 == 0u) {
                levels0 = __shfl_sync(0xffffffffu, hd.levelset, 0);
                width0 = __shfl_sync(0xffffffffu, hd.width, 0);
            }
            const bool tokens = hd.ok && hd.mode != kModeFixed, in_code = tokens && hd.mode == kModeCoded;
            uint32_t mine = 0;
            if (tokens) mine = (in_code ? kCoded : kErc) | (hd.levelset == kLevelsUniform ? kUniform : kOther) | (hd.levelset == kLevelsTable ? kTabled : 0u);
            if (k < K && (!tokens || hd.levelset != levels0)) mine |= kOdd;
            if (k < K && !(hd.ok && hd.mode == kModeFixed && hd.levelset == levels0)) mine |= kNotFields;
            const uint32_t had = found;
            found |= __reduce_or_sync(0xffffffffu, mine);
            if (found & kCoded) {
                uint32_t w0 = 0, w1 = 0;
                if (in_code) {
                    w0 = hd.hdr[hd.hwords - 2u];
                    w1 = hd.hdr[hd.hwords - 1u];
                }
                if (!(had & kCoded)) {
                    const int first = __ffs((int)__ballot_sync(0xffffffffu, in_code)) - 1;
                    first0 = __shfl_sync(0xffffffffu, w0, first);
                    first1 = __shfl_sync(0xffffffffu, w1, first);
                }
                if (__any_sync(0xffffffffu, in_code && (w0 != first0 || w1 != first1))) found |= kSeveralCodes;
            }
        }
        if ((found & kCoded) && lane <= min(G.s, kMaxCodedS)) s_words[lane] = level_word(first0, first1, G.s, lane);
        if (lane == 0) {
            s_kind = found & kCoded ? (found & (kErc | kSeveralCodes) ? kTabGaps : kTabCoded)
                     : found & kUniform ? (found & kOther ? kTabGaps : kTabUniform) : kTabErc;
            s_alike = found & kOdd ? 2u : found & kUniform ? 1u : found & kTabled ? 3u : 0u;
            s_fields = found & kNotFields ? 0u : width0;
        }
    }
    __syncthreads();
    if (!CALLED && s_fields != 0u) {                        // no tokens at all
        fields_of_width<I>(P, heads, at.field_tables, rows, s_fields);
        return;
    }
    if (CALLED) clear_rows<Sym>(rows);
    const uint32_t S = P.unit_subs;                         // sub-blocks of a unit
    const uint32_t nsub = (uint32_t)((G.d + kSB - 1u) / kSB), nunits = (uint32_t)(((uint64_t)nsub + S - 1u) / S), stride = gridDim.x * (blockDim.x >> 5);
    const uint32_t kind = s_kind, all_alike = s_alike == 3u && s_kind == kTabGaps ? 2u : s_alike;
    if (kind != P.likely_table || kind == kTabGaps || kind == kTabCoded || all_alike >= 2u)
        prepare_tables<Sym>(P, dsm, s_words, kind, all_alike, nunits > stride);
    // from here on warps run alone

    const uint32_t tab = smem_u32(table);
    const uint32_t spb = G.bucket <= kBLK ? G.sb_per_block : 32u;   // sub-blocks of a coding block
    const uint32_t lj = lane / S, lq = lane - lj * S;
    const uint32_t ngroups = MANY ? (K + 31u) / 32u : 1u;   // of up to 32 streams (S = 1 when there are several)

    // An item is a unit of a group of streams.  The block offsets of an item's chains ...
    struct Offsets {
        uint64_t from, to;
    };
    auto load_offsets = [&](uint32_t unit, uint32_t g0) {
        Offsets o;
        o.from = o.to = 0;
        const uint32_t sub = unit * S + lq, k = g0 + lj;    // (below 2^32 for units that exist: there are fewer sub-blocks)
        if (unit < nunits && sub < nsub && k < K && lj * S + lq < 32u && heads[k].ok && heads[k].mode != kModeFixed) {
            const uint64_t* at = reinterpret_cast<const uint64_t*>(heads[k].hdr + heads[k].hwords) + sub / spb;
            o.from = at[0];
            o.to = at[1];
        }
        return o;
    };
    // ... and, from them, where this lane's chain lies: the lengths of the sub-blocks before it in its block
    auto describe = [&](uint32_t unit, uint32_t g0, const Offsets& o) {
        Chain ch;
        ch.src = nullptr;
        ch.left = 0;
        ch.bit = ch.len = 0;
        ch.norm = 0.0f;
        ch.good = true;
        const uint32_t sub = unit * S + lq, k = g0 + lj;
        if (unit < nunits && sub < nsub && k < K && heads[k].ok && heads[k].mode != kModeFixed) {
            const StreamHead& hd = heads[k];
            const uint32_t blk = sub / spb, sbi = sub - blk * spb;
            const uint32_t nsb_blk = min(nsub - blk * spb, spb), head_words = 1u + (nsb_blk + 1u) / 2u;
            const uint64_t head = hd.hwords + 2 * (G.nblk + 1), words = (o.to - o.from) >> 5;
            ch.good = ((o.from | o.to) & 31u) == 0 && o.from < o.to && (o.to >> 5) <= hd.cwords - head &&
                      words >= head_words && words <= (1u << 20);
            if (ch.good) {
                const uint64_t rec = head + (o.from >> 5);
                const uint32_t* const lens = hd.hdr + rec + 1u;
                uint32_t start = 0;
                const uint32_t last = sbi >> 1, pair = lens[last];
#pragma unroll 4
                for (uint32_t w = 0; w < last; ++w) {
                    const uint32_t v = lens[w];
                    start += (v & 0xffffu) + (v >> 16);
                }
                ch.norm = __uint_as_float(lens[-1]);
                if (sbi & 1u) start += pair & 0xffffu;
                const uint32_t len = sbi & 1u ? pair >> 16 : pair & 0xffffu;
                ch.good = start + len <= 32u * ((uint32_t)words - head_words);
                if (ch.good) {
                    const uint64_t word = rec + head_words + (start >> 5), piece = word & ~(uint64_t)3u;
                    ch.src = hd.hdr + piece;
                    ch.left = hd.cwords - piece;
                    ch.bit = 32u * (uint32_t)(word - piece) + (start & 31u);
                    ch.len = len;
                }
            }
        }
        return ch;
    };
    // asks the lengths that describe() will read into the L1
    auto prefetch_lengths = [&](uint32_t g0, const Offsets& o) {
        if (o.from < o.to) {                                // (0 and 0 where there is no chain)
            const StreamHead& hd = heads[g0 + lj];
            const uint64_t head = hd.hwords + 2 * (G.nblk + 1);
            if ((o.to >> 5) <= hd.cwords - head) asm volatile("prefetch.global.L1 [%0];" ::"l"(hd.hdr + head + (o.from >> 5)));
        }
    };
    // starts the copy of the lane's next words: those with bits [bit, bit + len) of ch.src, as many as there is room for
    auto start_copy = [&](const Chain& ch) {
        if (ch.len != 0u) {
            const uint32_t n = min((ch.bit + ch.len + 31u) / 32u, kChunkWords);
#pragma unroll
            for (uint32_t i = 0; i < kChunkWords; i += 4u) {
                if (i >= n) break;
                if (i + 4u <= ch.left) copy_async16(copy + 4u * i, ch.src + i);
                else for (uint32_t j = i; j < ch.left; ++j) copy_async4(copy + 4u * j, ch.src + j);   // the container ends here
            }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    // the whole of the lane's chain is in its copy, with room for the ones behind it
    auto fits = [&](const Chain& ch) { return (ch.bit + ch.len + 31u) / 32u + kChunkSlack <= kChunkWords; };

    uint32_t unit = warp * gridDim.x + blockIdx.x, unit1 = unit;
    uint32_t group = 0, group1 = 0;
    auto advance = [&](uint32_t& u, uint32_t& g) {          // (behind the last unit u stays there: nunits + stride may pass 2^32)
        if (MANY && ++g != ngroups) return;
        g = 0;
        u = u < nunits && nunits - u > stride ? u + stride : nunits;
    };
    Chain ch = describe(unit, 0, load_offsets(unit, 0));
    start_copy(ch);
    advance(unit1, group1);
    Offsets next = load_offsets(unit1, 32u * group1);
    uint64_t carry[4] = {0, 0, 0, 0};                       // sums of the groups of streams before this one (S = 1)
    while (unit < nunits) {
        uint32_t unit2 = unit1, group2 = group1;
        advance(unit2, group2);
        const Offsets next2 = load_offsets(unit2, 32u * group2);
        const uint32_t g0 = 32u * group, gcount = min(K - g0, 32u);
        if (P.sum.w != nullptr && group == 0u) {                // the parameters the add pass will read and write
            const uint64_t first = (uint64_t)(unit * S) * kSB, left = G.d - first;
            const uint32_t bytes = 4u * ((left < S * kSB ? (uint32_t)left : S * kSB) & ~3u);
            if (bytes && lane < (P.sum.mu != 0.0f ? 2u : 1u))
                asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"((lane == 0u ? P.sum.w : P.sum.yl) + first), "r"(bytes) : "memory");
        }
        if (SHORT) prefetch_lengths(32u * group1, next);
        asm volatile("cp.async.wait_group 0;" ::: "memory");

        // ================= walk =================
        const StreamHead& my_head = heads[g0 + min(lj, gcount - 1u)];
        const uint16_t* const my_code = reinterpret_cast<const uint16_t*>(codes + (g0 + min(lj, gcount - 1u)) * kCodeBytes);
        const uint32_t row0 = rows + lane * Row<Sym>::kPitch - (uint32_t)sizeof(Sym), row_end = row0 + (kSB + 1u) * (uint32_t)sizeof(Sym);
        uint32_t row = row0;
        bool good = ch.good;
        const float norm = ch.len != 0u ? ch.norm : 0.0f;
        bool long_chain = __any_sync(0xffffffffu, !fits(ch));
        auto put_ones = [&] {                               // behind the chain's last bit
            if (ch.len != 0u) {
                const uint32_t end = ch.bit + ch.len, w = copy + 4u * (end >> 5);
                const uint32_t have = end & 31u ? lds_u32(w) : 0u;
                asm volatile("st.shared.u32 [%0], %1;" ::"r"(w), "r"(have | 0xFFFFFFFFu >> (end & 31u)) : "memory");
                asm volatile("st.shared.u32 [%0], %1;" ::"r"(w + 4u), "r"(0xFFFFFFFFu) : "memory");
            }
        };
        uint32_t left = ch.len;
        if (!long_chain) {
            put_ones();
            if (kind == kTabGaps) left -= walk_rare<Sym, false, true>(copy, ch.bit, left, tab, row, row_end, my_head, my_code, G.s, good);
            else left -= walk_body<Sym, false, false>(copy, ch.bit, left, tab, row, row_end, my_head, my_code, G.s, good);
        } else {
            // chains longer than a lane's copy: one copy after the other, each walked up to 96 bits before its end
            while (__any_sync(0xffffffffu, left != 0u)) {
                const uint32_t room = 32u * kChunkWords - ch.bit;
                const uint32_t bits = fits(ch) ? left : room - 96u;
                // (a pair of tokens must not reach into the chain behind: it may pass the point by 12 bits)
                if (kPairs<Sym> && ch.bit + ch.len <= 32u * (kChunkWords - 2u)) put_ones();
                uint32_t took;
                if (kind == kTabGaps) took = walk_rare<Sym, true, true>(copy, ch.bit, bits, tab, row, row_end, my_head, my_code, G.s, good);
                else took = walk_rare<Sym, true, false>(copy, ch.bit, bits, tab, row, row_end, my_head, my_code, G.s, good);
                if (!good || took > left) {
                    good = false;
                    took = left;
                }
                left -= took;
                ch.len = left;
                const uint32_t at = ch.bit + took, pieces = at / 128u;
                ch.src += 4u * pieces;
                ch.left -= 4u * pieces;
                ch.bit = at - 128u * pieces;
                start_copy(ch);
                asm volatile("cp.async.wait_group 0;" ::: "memory");
            }
        }
        // a well-formed chain ends exactly at its declared length, inside its sub-block
        const uint64_t my_sub = unit * S + lq;
        const uint32_t elems = (uint32_t)(G.d - min(G.d, my_sub * kSB) < kSB ? G.d - min(G.d, my_sub * kSB) : kSB);
        good = good && left == 0u && row <= row0 + elems * (uint32_t)sizeof(Sym);
        if (__any_sync(0xffffffffu, !good) && lane == 0) latch_status(P.ws, kErrBadStream);
        asm volatile("st.shared.f32 [%0], %1;" ::"r"(norms + 4u * lane), "f"(norm) : "memory");
        // norm times a power of two is exact for these norms (0 where there is no chain), so one fused operation does for two
        const bool exact = __all_sync(0xffffffffu, norm == 0.0f || (norm >= 0x1p-100f && norm < 0x1p126f));
        const Chain after = describe(unit1, 32u * group1, next);
        __syncwarp();
        start_copy(after);

        // ================= add =================
        const AddPass ap = {heads + g0, levels + g0 * kLevelBytes, smem_u32(codes) + g0 * kCodeBytes, rows, norms, S, gcount, exact ? all_alike : 2u,
                            !MANY || group + 1u == ngroups, MANY && group != 0u};
        const uint64_t e0 = (uint64_t)(unit * S) * kSB + 4u * lane;
        uint32_t q0 = 0;
#pragma unroll 1
        for (; q0 + 4u <= S; q0 += 4u) add_block<Sym, 4, MANY>(P, ap, q0, e0 + 256u * q0, carry);
#pragma unroll 1
        for (; q0 < S; ++q0) add_block<Sym, 1, MANY>(P, ap, q0, e0 + 256u * q0, carry);
        __syncwarp();
        clear_rows<Sym>(rows);
        __syncwarp();
        ch = after;
        next = next2;
        unit = unit1; group = group1;
        unit1 = unit2; group1 = group2;
    }
}

template <class I>
__global__ void __launch_bounds__(32 * kChainMaxWarps, 1) decode_chains_kernel(const __grid_constant__ DecodeParams P) {
    decode_streams<I, false>(P);
}

// (One function for all the kernels for fixed-width streams.  Its stores are of 16 bytes, not the wide ones that went wrong in a
// shared function; each kernel's way through it is tested.)
template <class Sym>
__device__ __noinline__ void decode_streams_call(const DecodeParams& P) {
    decode_streams<Instance<Sym, true, false>, true>(P);
}

// Calls whose streams are likely all in the fixed-width mode, with fields of W bits of one level set: a kernel of its own for
// each, so that neither its registers nor its code are shared with the walks of token streams.  25.6 x 10^6 elements, K = 8, 4
// bits, in one kernel with the walks: 67.6 us behind eight encode calls (where the code has to be fetched), 53.6 us repeated;
// here 56 and 51 us; as a function called by the kernel for token streams, which is what containers that were not encoded here
// take, 65.5 and 53 us.
template <uint32_t W, bool EXACT>
__global__ void __launch_bounds__(32 * kChainMaxWarps, 1) decode_fields_kernel(const __grid_constant__ DecodeParams P) {
    extern __shared__ __align__(128) unsigned char dsm[];
    __shared__ uint32_t s_likely;
    const uint32_t K = P.K, lane = lane_id();
    const bool wide_symbols = P.geo.s == 7u || P.geo.s == 8u;
    const Layout<int8_t> at(dsm, K);
    if (P.let_next) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const bool tables_ready = P.likely_levels != kLevelsTable;
    if (tables_ready) build_field_tables(P.geo, P.likely_levels, nullptr, 1u, at.field_tables);
    asm volatile("griddepcontrol.wait;" ::: "memory");
    if (threadIdx.x < 32u) {
        bool likely = true;
        for (uint32_t k = lane; k < K; k += 32u) {
            const StreamHead hd = read_head(P.geo, P.streams[k]);
            at.heads[k] = hd;
            likely = likely && hd.ok && hd.mode == kModeFixed && hd.levelset == P.likely_levels;
        }
        likely = __all_sync(0xffffffffu, likely);
        if (lane == 0) s_likely = likely;
    }
    __syncthreads();
    if (s_likely) {
        const uint32_t mine = wide_symbols ? Layout<int16_t>(dsm, K).rows : at.rows;
        decode_fields<W, EXACT>(P, at.heads, at.field_tables, tables_ready, mine);
    } else if (wide_symbols) {                              // another kind of streams after all
        decode_streams_call<int16_t>(P);
    } else {
        decode_streams_call<int8_t>(P);
    }
}

using DecodeKernel = void (*)(DecodeParams);
// (level tables and exponential levels: s + 2 of them; uniform levels: 2^s + 1, s <= 8)
static DecodeKernel fields_kernel(uint32_t s, uint32_t levelset) {
    if (levelset == kLevelsExp) return s <= 2u ? decode_fields_kernel<3, true> : s <= 6u ? decode_fields_kernel<4, true> : decode_fields_kernel<5, true>;
    const uint32_t width = levelset == kLevelsUniform ? s + 2u : s <= 2u ? 3u : s <= 6u ? 4u : 5u;
    static const DecodeKernel by_width[] = {decode_fields_kernel<3, false>, decode_fields_kernel<4, false>, decode_fields_kernel<5, false>, decode_fields_kernel<6, false>,
                                            decode_fields_kernel<7, false>, decode_fields_kernel<8, false>, decode_fields_kernel<9, false>, decode_fields_kernel<10, false>};
    return by_width[width - 3u];
}

template <class Sym>
static cudaError_t launch_chains(const DecodeParams& P, int sms, cudaStream_t stream) {
    const size_t fixed = chain_fixed_bytes(P.K);
    size_t warps = (kChainSmem - fixed) / Row<Sym>::kWarpBytes;
    if (warps > kChainMaxWarps) warps = kChainMaxWarps;
    const uint64_t nsub = (P.geo.d + kSB - 1u) / kSB;
    DecodeParams Q = P;
    // As many sub-blocks as give every lane a chain; in a small call no more than give every warp a unit (a walk
    // lasts as long for one lane as for 32).
    Q.unit_subs = P.K >= 32u ? 1u : 32u / P.K;
    const uint64_t share = (nsub + (uint64_t)sms * warps - 1u) / ((uint64_t)sms * warps);
    if (share < Q.unit_subs) Q.unit_subs = (uint32_t)share;
    const uint64_t units = (nsub + Q.unit_subs - 1u) / Q.unit_subs;
    Q.let_next = units > 2u * (uint64_t)sms * warps ? 1u : 0u;
    DecodeKernel kernel = P.K > 32u ? decode_chains_kernel<Instance<Sym, true, false>> : decode_chains_kernel<Instance<Sym, false, false>>;
    if constexpr (sizeof(Sym) == 1) {
        if (P.K <= 32u && P.geo.bucket <= 4u * kSB && Q.let_next) kernel = decode_chains_kernel<Instance<Sym, false, true>>;
    }
    if (P.likely_table == kTabFields) kernel = fields_kernel(P.geo.s, P.likely_levels);
    static std::map<DecodeKernel, OncePerDevice> prepared;
    const cudaError_t e = prepared[kernel]([=] { return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kChainSmem); });
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = cudaLaunchConfig_t{};
    cudaLaunchAttribute attr[1];
    cfg.gridDim = dim3((unsigned)(units < (uint64_t)sms ? units : (uint64_t)sms));
    cfg.blockDim = dim3(32u * (unsigned)warps);
    cfg.dynamicSmemBytes = fixed + warps * Row<Sym>::kWarpBytes;
    cfg.stream = stream;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    return cudaLaunchKernelEx(&cfg, kernel, Q);
}

cudaError_t launch_decode(const DecodeParams& P, int sms, cudaStream_t stream) {
    // With s = 7 or 8 the streams may have uniform levels, whose indices up to 256 do not fit a byte with their sign.
    return P.geo.s == 7u || P.geo.s == 8u ? launch_chains<int16_t>(P, sms, stream) : launch_chains<int8_t>(P, sms, stream);
}

}  // namespace nuq

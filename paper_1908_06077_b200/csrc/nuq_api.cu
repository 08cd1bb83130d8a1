// C ABI of the library (see include/nuq.h): argument validation, geometry,
// per-stream workspace, kernel launches.  No torch types, no CPU fallback: every
// step of the path runs in the kernels of nuq_encode.cu / nuq_decode_chains.cu.
#include <map>
#include <mutex>
#include <set>
#include <utility>

#include "../../include/nuq.h"
#include "nuq_common.cuh"
#include "nuq_launch.h"

namespace nuq {
namespace {

// Scratch of nuq_encode_static: lives in the library's device image, so every
// GPU that loads the library holds these bytes until the process exits.  In host
// code this name is only a handle for cudaGetSymbolAddress, never an address.
constexpr size_t kStaticScratchBytes = NUQ_STATIC_SCRATCH_BYTES;
static __device__ __align__(256) unsigned char g_static_scratch[kStaticScratchBytes];

struct WsEntry {
    Workspace* ptr = nullptr;
    size_t bytes = 0;
    // Something else than zeros may lie where an encode call keeps its scan state.  The allocation is zeroed and every
    // encode kernel leaves its scan state zeroed, so that is the case only after a launch that failed.
    bool dirty = false;
    // Bucket norms that are taken in a pass of their own (wide buckets with 4-bit fields, histograms): an allocation of its
    // own, so that no call (nor a replay of a captured one, of which the host knows nothing) leaves them where another
    // call's scan state lies.
    float* norms = nullptr;
    size_t norms_bytes = 0;
};

// One mutex guards the host-side bookkeeping below (maps, tables); it is held for the microseconds a
// call spends on the host, never across a wait for the device, except where a workspace has to grow.
std::mutex g_mu;
std::map<std::pair<int, cudaStream_t>, WsEntry> g_ws;
std::map<int, int> g_sms;                 // device -> SM count
std::set<int> g_lut_ready;                // devices whose constant LUT is uploaded ...
std::set<int> g_token_tables_ready;       // ... and those that hold the decoder's token tables
std::map<int, const float*> g_test_norms;   // device -> bucket norms of nuq_set_test_norms
float g_levels[kMaxTableS + 2], g_inv_width[kMaxTableS + 2];   // the level table of nuq_set_level_table ...
uint32_t g_levels_s = 0;                                       // ... and its number of interior levels (0: none set)
uint32_t g_level_code[kMaxCodedS + 1];                         // the code of nuq_set_level_code: word | length << 16 ...
uint32_t g_level_code_n = 0;                                   // ... and how many level indices it covers (0: none set)
std::map<int, Workspace*> g_static_ws;   // device -> address of g_static_scratch on that device
uint32_t g_erc_len[256];
bool g_erc_len_ready = false;

uint32_t erc_len(uint32_t n) {            // |ERC(n)|, 1 <= n <= 256
    if (!g_erc_len_ready) {
        uint32_t lut[256];
        build_erc_lut(lut);
        for (int i = 0; i < 256; ++i) g_erc_len[i] = lut[i] >> 16;
        g_erc_len_ready = true;
    }
    return g_erc_len[n - 1];
}

bool bucket_ok(uint32_t bucket) {
    if (bucket >= kSB && bucket <= kBLK) return bucket % kSB == 0;
    return bucket == 16384u || bucket == 32768u || bucket == 65536u;
}

bool make_geometry(uint64_t d, uint32_t bucket, uint32_t s, uint32_t flags, Geometry* G) {
    const uint32_t norm_kind = flags & 0xffu, levelset = (flags >> 8) & 0xffu, mode = (flags >> 16) & 0xffu;
    if (d == 0 || d >= (1ull << 40) || !bucket_ok(bucket) || s < 1) return false;
    if (norm_kind > 1 || levelset > 2 || mode > 2) return false;
    if (mode == kModeCoded && (levelset == kLevelsUniform || s > kMaxCodedS)) return false;
    if (s > (levelset == kLevelsUniform ? 8u : 14u)) return false;
    if (flags & ~(0x00ffffffu | NUQ_TEST_NORMS | NUQ_TEST_SHORT_PATIENCE)) return false;
    G->d = d;
    G->bucket = bucket;
    G->s = s;
    G->norm_kind = norm_kind;
    G->levelset = levelset;
    G->mode = mode;
    G->nb = (d + bucket - 1) / bucket;
    G->nlev = levelset == kLevelsUniform ? (1u << s) + 1u : s + 2u;
    G->header_words = kHeaderWords + (levelset == kLevelsTable ? ((s + 1u) & ~1u) : 0u) + (mode == kModeCoded ? 2u : 0u);
    G->pad = 0;
    uint32_t b = 0;
    while ((1u << b) < G->nlev) ++b;
    G->width = b + 1u;
    G->rec_words = 1u + (uint32_t)(((uint64_t)bucket * G->width + 31) / 32);
    const uint64_t last = d - (G->nb - 1) * bucket;
    if (bucket <= kBLK) {
        G->blocks_per_tile = kBLK / bucket;
        G->tile_elems = G->blocks_per_tile * bucket;
        G->sb_per_block = bucket / kSB;
        G->blk_per_bucket = 1;
        G->nblk = G->nb;
        G->ntiles = (G->nb + G->blocks_per_tile - 1) / G->blocks_per_tile;
    } else {
        G->blocks_per_tile = 1;
        G->tile_elems = kBLK;
        G->sb_per_block = 32;
        G->blk_per_bucket = bucket / kBLK;
        G->nblk = (G->nb - 1) * G->blk_per_bucket + (last + kBLK - 1) / kBLK;
        G->ntiles = G->nblk;
    }
    return true;
}

uint32_t max_level_code_bits(const Geometry& G) {
    if (G.mode == kModeCoded) return kMaxCodedS;            // whatever code is set
    uint32_t best = 0;
    for (uint32_t sym = 1; sym < G.nlev; ++sym) best = erc_len(sym) > best ? erc_len(sym) : best;
    return best;
}

// Most token bits that `elems` consecutive elements lying in at most `buckets` buckets can produce.
// Always true: a token has at most |ERC(1)| + 1 + L bits per position it consumes (L = longest
// level code), i.e. 2 + L bits per element.  With the Euclidean norm computed by the encoder
// itself a much smaller bound holds: a symbol above the lowest level needs r > 2^-s, and at most
// 4^s coordinates of a bucket can have that (the counting step of the paper's sparsity lemma,
// Lemma 10); all others cost at most |ERC(1)| + 1 + |ERC(1)| = 3 bits per consumed position.
// In the coded mode the same holds with the lengths of the code in use: a lowest-level token costs
// at most 2 + len(1) bits per consumed position (|ERC(gap)| + 1 + len(1) <= gap (2 + len(1))), the
// others at most the longest of the remaining words more.
uint32_t token_bits_bound(const Geometry& G, uint32_t elems, uint32_t buckets, bool norms_are_ours) {
    uint32_t L = max_level_code_bits(G), low = 1u, rest = L;    // longest code, code of index 1, longest of the others
    if (G.mode == kModeCoded) {
        L = rest = 0;
        low = g_level_code[0] >> 16;
        for (uint32_t j = 0; j <= G.s; ++j) {
            const uint32_t len = g_level_code[j] >> 16;
            L = len > L ? len : L;
            if (j >= 1) rest = len > rest ? len : rest;
        }
    }
    const uint32_t safe = elems * (2u + L);
    if (!norms_are_ours || G.norm_kind != kNormL2 || G.levelset != kLevelsExp || G.s > 7u) return safe;
    const uint64_t high = (uint64_t)buckets * ((1ull << (2u * G.s)) + 8u);      // + slack for the rounding of the norm
    const uint32_t nhigh = high < elems ? (uint32_t)high : elems;
    const uint32_t tight = (2u + low) * elems + nhigh * (rest > low ? rest - low : 0u);
    return tight < safe ? tight : safe;
}

// words of shared-memory staging the records of one ERC tile can need
uint32_t stage_words_for(const Geometry& G, bool norms_are_ours) {
    uint32_t head = 1u + (G.sb_per_block + 1u) / 2u + 1u;          // norm, lengths, padding
    return G.blocks_per_tile * head + (token_bits_bound(G, G.tile_elems, G.blocks_per_tile, norms_are_ours) + 31u) / 32u;
}

uint64_t bound_bytes(const Geometry& G) {
    if (G.mode == kModeFixed) return 4ull * (G.header_words + G.nb * G.rec_words);
    uint64_t head = 1u + (G.sb_per_block + 1u) / 2u + 1u;
    uint64_t token_words = (G.d * (2ull + max_level_code_bits(G)) + 31) / 32;
    return 4ull * (G.header_words + 2 * (G.nblk + 1) + G.nblk * head + token_words);
}

int device_sms(int dev) {
    auto it = g_sms.find(dev);
    if (it != g_sms.end()) return it->second;
    int sms = 0;
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms <= 0) sms = 148;
    g_sms[dev] = sms;
    return sms;
}

// Room for the scan state of `ntiles` tiles behind the control block: one look-back word per tile and per group of 32 tiles.
size_t scan_state_bytes(uint64_t ntiles) { return sizeof(Workspace) + 8 * (ntiles + (ntiles + 31) / 32); }

// The most tiles that an encode call of up to d elements has, whatever its buckets and its mode: tiles of more than kBLK / 2
// elements (whole buckets, as many as fit), or of more than kSmallTile / 2 in calls of up to one tile of kBLK per SM.  A stream's
// workspace is made for that number and not for the call's own, which small tiles and short buckets raise: a call with fewer
// elements than an earlier one must not make the workspace grow (it may be captured, and a graph may hold the workspace's address).
uint64_t most_tiles(uint64_t d, int sms) {
    const uint64_t whole = d / (kBLK / 2) + 2, few = (uint64_t)sms * kBLK, small = (d < few ? d : few) / (kSmallTile / 2) + 2;
    return whole > small ? whole : small;
}

// Workspace of (current device, stream), grown to `bytes`.  Growing synchronises the stream.
nuq_status get_workspace(cudaStream_t stream, size_t bytes, Workspace** out, int* dev_out) {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return NUQ_ERR_CUDA;
    *dev_out = dev;
    WsEntry& e = g_ws[std::make_pair(dev, stream)];
    if (e.bytes < bytes) {
        int carried = 0;
        if (e.ptr) {
            if (cudaStreamSynchronize(stream) != cudaSuccess) return NUQ_ERR_CUDA;
            if (cudaMemcpy(&carried, &e.ptr->status, sizeof(int), cudaMemcpyDeviceToHost) != cudaSuccess) return NUQ_ERR_CUDA;
            cudaFree(e.ptr);
            e.ptr = nullptr;
            e.bytes = 0;
        }
        size_t want = bytes + bytes / 2;
        void* p = nullptr;
        if (cudaMalloc(&p, want) != cudaSuccess) { cudaGetLastError(); return NUQ_ERR_CUDA; }
        // (in the call's own stream: a clearing pass on the default stream is not ordered before kernels of a
        // non-blocking stream, which would then run on a workspace that is still being cleared)
        if (cudaMemsetAsync(p, 0, want, stream) != cudaSuccess) return NUQ_ERR_CUDA;
        e.ptr = static_cast<Workspace*>(p);
        e.bytes = want;
        e.dirty = false;
        if (carried && (cudaMemcpyAsync(&e.ptr->status, &carried, sizeof(int), cudaMemcpyHostToDevice, stream) != cudaSuccess ||
                        cudaStreamSynchronize(stream) != cudaSuccess))
            return NUQ_ERR_CUDA;
    }
    *out = e.ptr;
    return NUQ_OK;
}

// Room for the bucket norms of a call of d elements in the stream's current device, for the shortest buckets there are: like the
// workspace it goes by d alone (a pass over wide buckets that is captured, a histogram over short ones behind it).  Growing
// synchronises the stream.
nuq_status get_norms(cudaStream_t stream, uint64_t d, WsEntry& e) {
    const size_t bytes = 4 * ((d + kSB - 1) / kSB);
    if (e.norms_bytes >= bytes) return NUQ_OK;
    if (e.norms) {
        if (cudaStreamSynchronize(stream) != cudaSuccess) return NUQ_ERR_CUDA;
        cudaFree(e.norms);
        e.norms = nullptr;
        e.norms_bytes = 0;
    }
    const size_t want = bytes + bytes / 2;
    void* p = nullptr;
    if (cudaMalloc(&p, want) != cudaSuccess) { cudaGetLastError(); return NUQ_ERR_CUDA; }
    e.norms = static_cast<float*>(p);
    e.norms_bytes = want;
    return NUQ_OK;
}

}  // namespace
}  // namespace nuq

using namespace nuq;

// Mode and level set of the containers this process has encoded, by device and address (see enqueue_encode): a hint
// for the decoder's choice of kernels, which go by the containers' headers.
// Guarded by g_mu.
static std::map<std::pair<int, const void*>, uint32_t> g_container_mode;   // mode | level set << 8

// What one encode call needs from its workspace and from shared memory.
struct EncodePlan {
    size_t state_bytes;      // control block + one look-back word per tile and per group of 32 tiles
    size_t norms_bytes;      // bucket norms that a pass of its own takes (0: none)
    uint32_t want_grid;      // CTAs that give every SM its full share
};

// What the runtime says about an encoder's occupancy depends on the kernel and its shared memory only; asking takes longer
// than the rest of a call's host work, so the answers are kept (guarded by g_mu; a few dozen entries at most, one per
// combination of level set, mode, bucket kind, number of levels and cluster size in use).
static int occupancy(const EncodeParams& P, int dev, bool clusters) {
    static std::map<uint64_t, int> known;
    const Geometry& G = P.geo;
    const uint64_t key = (uint64_t)encode_smem_bytes(P) | (uint64_t)G.levelset << 32 | (uint64_t)G.mode << 34 |
                         (uint64_t)(fixed4_applies(G) ? 1u + fixed4_variant(G) : 0u) << 36 |
                         (uint64_t)(P.warps >> 3) << 42 |
                         (uint64_t)(clusters ? P.cluster : 0) << 38 | (uint64_t)(uint32_t)dev << 44 | (uint64_t)(P.tile != kBLK) << 63;
    const auto it = known.find(key);
    if (it != known.end()) return it->second;
    const int n = clusters ? encode_max_clusters(P) : encode_blocks_per_sm(P);
    if (n > 0) known[key] = n;
    return n;
}

static EncodePlan plan_encode(EncodeParams& P, int dev, uint32_t flags) {
    const int sms = device_sms(dev);
    Geometry& G = P.geo;
    const bool norms_are_ours = (flags & NUQ_TEST_NORMS) == 0;
    EncodePlan pl;
    pl.norms_bytes = G.bucket > kBLK ? 4 * G.nb : 0;
    // a look-back wait polls this often (with a pause in between: tens of ms in all) before it gives up
    P.patience = (flags & NUQ_TEST_SHORT_PATIENCE) ? 2u : 1u << 16;
    P.window_words = 0;
    P.stage_words = 0;
    // Small calls: a tile's latency counts there, not the SM's throughput.  (The fixed-width encoders have no such variants.)
    // Twice the warps per tile, two such CTAs to an SM: up to 17/7 tiles per SM as a rule.  2.0 to 2.4 tiles of 8192 (2.4 to 2.9 x 10^6 elements)
    // take 18 to 20 us instead of 20 to 23; from 2.45 on some SM gets four tiles, and 20 us become 23 to 24 (s = 4 in buckets of 512:
    // 2.35 tiles 20.3 and 19.1, 2.43 20.3 and 19.5, 2.52 20.4 and 23.9; level tables 25.5 and 25.0, 25.6 and 25.1, 25.7 and 30.0).  Uniform
    // levels with many symbols (2.5 tiles 24.9 and 22.8, 2.95 25.9 and 24.9) and buckets in clusters of four and eight gain up to three tiles per
    // SM (buckets of 65536, 2.2 tiles 26.5 and 23.8, 2.9 27.8 and 25.6, level tables 37.9 and 34.6, 43.8 and 37.3; largest-magnitude norms and
    // uniform levels between 10 % less and 5 % more); clusters of two up to two tiles (2.3 tiles 24.0 and 23.8, but uniform levels with s = 2
    // 24.5 and 27.2, largest-magnitude norms 25.6 and 27.9).
    const bool tokens = G.mode != kModeFixed;
    const uint64_t sevenths = G.bucket == 2u * kBLK ? 14u : G.bucket > kBLK || (G.levelset == kLevelsUniform && G.s >= 4u) ? 21u : 17u;
    P.warps = tokens && 7u * G.ntiles <= sevenths * (uint64_t)sms ? kEncMaxWarps : kEncWarps;
    P.tile = kBLK;
    // A quarter of a tile, one sub-block per warp, four to an SM: with fewer whole tiles than SMs, as long as small ones (of whole
    // buckets too, so that there may be six for a whole one) are no more than 5.5 to an SM.  65 536 elements 10.2 us in whole tiles of 16 warps, 8.4 in
    // small ones (uniform levels 12.0 and 8.7), 10^6 elements 15.2 and 13.3, coded indices 15.4 and 12.5; 147 whole tiles, buckets of
    // 512 / 768 / 1536 (3.96, 4.95 and 4.95 small ones to an SM) 15.4 and 13.6, 15.2 and 14.7, 15.4 and 14.9; buckets of 1280 with 5.4
    // to an SM 15.9 and 15.1, 5.6 15.9 and 16.2.  Whole tiles for all 148 SMs 12.5 and 13.9 (no SM gets two, then).
    const uint32_t small_blocks = G.bucket <= kSmallTile ? kSmallTile / G.bucket : 1u;
    const uint64_t small_tiles = (G.nb + small_blocks - 1) / small_blocks;
    if (tokens && G.bucket <= kSmallTile && G.ntiles < (uint64_t)sms && 2u * small_tiles <= 11u * (uint64_t)sms) {
        P.tile = kSmallTile;
        P.warps = kEncWarps;
        G.blocks_per_tile = small_blocks;
        G.tile_elems = small_blocks * G.bucket;
        G.ntiles = small_tiles;
    }
    // (the tiles' number is what it will be from here on)
    pl.state_bytes = scan_state_bytes(G.ntiles);
    if (G.mode != kModeFixed) {
        P.stage_words = (stage_words_for(G, norms_are_ours) + 3u) & ~3u;
        // a warp's elements lie in at most this many buckets
        const uint32_t warp_elems = P.tile / P.warps;
        // (tiles start at bucket boundaries and a warp's part at a multiple of its size)
        const uint32_t warp_buckets = G.bucket >= warp_elems ? (G.bucket % warp_elems == 0 ? 1u : 2u)
                                                             : (warp_elems % G.bucket == 0 ? warp_elems / G.bucket : warp_elems / G.bucket + 1u);
        P.window_words = (token_bits_bound(G, warp_elems, warp_buckets, norms_are_ours) + 31u) / 32u + 4u;
    }
    int best = occupancy(P, dev, false);                    // resident CTAs per SM: what shared memory and registers allow
    if (best > kEncMaxBlocks) best = kEncMaxBlocks;
    const int per_sm = best < 1 ? 1 : best;
    const uint64_t cap = (uint64_t)sms * (uint64_t)per_sm;
    pl.want_grid = (uint32_t)(G.ntiles < cap ? G.ntiles : cap);
    // A bucket wider than a tile: a thread-block cluster of as many CTAs as the bucket has tiles encodes it and adds
    // up its norm through distributed shared memory, so there is no separate pass over the gradient for the norms.
    // (Not with norms supplied by the caller, and not in the 4-bit fixed-width encoder.)
    P.cluster = 0;
    P.overlap = 0;
    if (G.bucket > kBLK && norms_are_ours && !fixed4_applies(G)) {
        P.cluster = G.blk_per_bucket;
        int clusters = occupancy(P, dev, true);
        const int cap_clusters = sms * per_sm / (int)P.cluster;
        if (clusters > cap_clusters) clusters = cap_clusters;
        if (clusters >= 1) {
            pl.norms_bytes = 0;
            pl.want_grid = (uint32_t)(G.nb < (uint64_t)clusters ? G.nb : (uint64_t)clusters) * P.cluster;
        } else {
            P.cluster = 0;                                  // no room for a cluster: the separate norm pass
        }
    }
    return pl;
}

// Shared tail of the two encode entry points: clears the call's scan state in `ws` where needed and
// enqueues the kernels.  `ws` must hold pl.state_bytes, `norms` (if any) pl.norms_bytes.
static nuq_status enqueue_encode(EncodeParams& P, const EncodePlan& pl, const float* g, uint32_t norm_kind,
                                 uint64_t seed, uint64_t offset, void* out, uint64_t* out_bits, Workspace* ws, float* norms,
                                 WsEntry* entry, int dev, cudaStream_t stream) {
    Geometry& G = P.geo;
    const bool test_norms = (norm_kind & NUQ_TEST_NORMS) != 0;
    if (!g_lut_ready.count(dev)) {
        if (upload_erc_lut() != cudaSuccess) return NUQ_ERR_CUDA;
        g_lut_ready.insert(dev);
    }
    // The encode kernel leaves its scan state zeroed when it ends, so a clearing pass is needed only where
    // that cannot be relied on: entry == nullptr (the shared static array: always), or a launch failed (then all of
    // the workspace is cleared, not only what this call will use: a later, longer call keeps scan state further up).
    if (entry == nullptr || entry->dirty) {
        const size_t upto = entry ? entry->bytes : pl.state_bytes;
        if (cudaMemsetAsync(reinterpret_cast<char*>(ws) + kWorkspaceClearFrom, 0, upto - kWorkspaceClearFrom, stream) !=
            cudaSuccess)
            return NUQ_ERR_CUDA;
        if (entry) entry->dirty = false;
    }

    P.g = g;
    P.norms_in = nullptr;
    if (test_norms) {
        P.norms_in = g_test_norms[dev];
    } else if (pl.norms_bytes) {
        if (launch_bucket_norms(g, G.d, G.bucket, G.norm_kind, norms, G.nb, stream) != cudaSuccess) return NUQ_ERR_CUDA;
        P.norms_in = norms;
    }
    P.out = static_cast<uint32_t*>(out);
    P.out_bits = out_bits;
    P.ws = ws;
    // The kernel may be set up (its CTAs started, their tables built) while the kernel before it in the stream
    // ends; it touches global memory only when that kernel has ended.  Not on the static array, which is
    // cleared before every call, and not for calls with hundreds of tiles per CTA, which gain nothing from it
    // (the 2^30-element workload in clusters measured 2 % slower).
    P.overlap = entry && G.ntiles <= 32ull * P.grid ? 1u : 0u;
    // The kernel behind is let in early, except by a 4-bit fixed-width call that leaves SMs with room for more of its CTAs:
    // the next such call's CTAs would be packed there, four to an SM, instead of spread (10^6 elements 13.0 -> 8.05 us,
    // 3 x 10^6 13.4 -> 11.3 us).  The token encoders' small calls gain from it although those in small tiles are four to an SM too
    // (without / with: 65 536 elements 10.2 / 8.8 us, 6 x 10^5 13.2 / 11.0, 9 x 10^5 14.8 / 12.9, from 10^6 on the same; steps of four
    // workers with 65 536 and 6 x 10^5 elements 49.5 / 44.3 and 65.1 / 56.2).
    P.let_next = P.overlap && !(fixed4_applies(G) && P.grid <= 3u * (uint32_t)device_sms(dev)) ? 1u : 0u;
    P.seed = seed;
    P.offset = offset;
    for (uint32_t j = 0; j < kMaxTableS + 2u; ++j) {
        P.levels[j] = G.levelset == kLevelsTable ? g_levels[j] : 0.0f;
        P.inv_width[j] = G.levelset == kLevelsTable ? g_inv_width[j] : 0.0f;
    }
    for (uint32_t j = 0; j <= kMaxCodedS; ++j) P.level_code[j] = G.mode == kModeCoded ? g_level_code[j] : 0u;
    for (uint32_t r = 0; r < 10; ++r) {               // Philox key schedule (Weyl sequence)
        P.round_keys[2 * r] = (uint32_t)seed + r * 0x9E3779B9u;
        P.round_keys[2 * r + 1] = (uint32_t)(seed >> 32) + r * 0xBB67AE85u;
    }
    if (launch_encode(P, stream) != cudaSuccess) {
        if (entry) entry->dirty = true;                     // whatever state the failed launch left
        return NUQ_ERR_CUDA;
    }
    // what the container at this address is (a hint; the map is bounded)
    if (g_container_mode.size() > 4096) g_container_mode.clear();
    g_container_mode[std::make_pair(dev, static_cast<const void*>(out))] = G.mode | G.levelset << 8;
    return NUQ_OK;
}

static bool encode_args_ok(const float* g, uint64_t d, uint32_t bucket, uint32_t s, uint32_t norm_kind, void* out,
                           uint64_t* out_bits, Geometry* G) {
    if (!g || !out || !make_geometry(d, bucket, s, norm_kind, G)) return false;
    if ((reinterpret_cast<uintptr_t>(g) & 15u) || (reinterpret_cast<uintptr_t>(out) & 15u) ||
        (reinterpret_cast<uintptr_t>(out_bits) & 7u))
        return false;
    if (norm_kind & NUQ_TEST_NORMS) {
        int dev = 0;
        if (cudaGetDevice(&dev) != cudaSuccess || !g_test_norms.count(dev) || !g_test_norms[dev]) return false;
    }
    if (G->levelset == kLevelsTable && g_levels_s != s) return false;   // no level table of this length has been set
    if (G->mode == kModeCoded && g_level_code_n != s + 1) return false; // no code for s + 1 level indices has been set
    return true;
}

extern "C" {

uint64_t nuq_encode_bound(uint64_t d, uint32_t bucket, uint32_t s, uint32_t norm_kind) {
    std::lock_guard<std::mutex> lock(g_mu);
    Geometry G;
    if (!make_geometry(d, bucket, s, norm_kind, &G)) return 0;
    return (bound_bytes(G) + 15) & ~15ull;
}

nuq_status nuq_set_level_table(const float* interior_levels, uint32_t s) {
    std::lock_guard<std::mutex> lock(g_mu);
    if (!interior_levels || s < 1 || s > kMaxTableS) return NUQ_ERR_INVALID_ARG;
    float lv[kMaxTableS + 2], iw[kMaxTableS + 2];
    lv[0] = 0.0f;
    for (uint32_t j = 1; j <= s; ++j) lv[j] = interior_levels[j - 1];
    lv[s + 1] = 1.0f;
    for (uint32_t j = 0; j <= s; ++j) {
        if (!(lv[j] < lv[j + 1])) return NUQ_ERR_INVALID_ARG;              // strictly increasing inside (0, 1), no NaN
        iw[j] = 1.0f / (lv[j + 1] - lv[j]);                                 // one IEEE division per level
        if (!(iw[j] < __builtin_huge_valf())) return NUQ_ERR_INVALID_ARG;
    }
    iw[s + 1] = 0.0f;
    for (uint32_t j = 0; j < kMaxTableS + 2u; ++j) {
        g_levels[j] = j <= s + 1 ? lv[j] : 1.0f;
        g_inv_width[j] = j <= s + 1 ? iw[j] : 0.0f;
    }
    g_levels_s = s;
    return NUQ_OK;
}

// Canonical code words for the given lengths: level indices ordered by (length, index); the first
// word is all zeros, each next one is the previous plus one, extended with zeros to its length.
static bool canonical_code(const uint8_t* lengths, uint32_t n, uint32_t* code) {
    uint32_t kraft = 0;                                      // in units of 2^-7
    for (uint32_t j = 0; j < n; ++j) {
        if (lengths[j] < 1 || lengths[j] > kMaxCodedS) return false;
        kraft += 1u << (kMaxCodedS - lengths[j]);
    }
    if (kraft > (1u << kMaxCodedS)) return false;           // no prefix code has these lengths
    uint32_t word = 0, have = 0;
    for (uint32_t len = 1; len <= kMaxCodedS; ++len) {
        word <<= 1;
        for (uint32_t j = 0; j < n; ++j)
            if (lengths[j] == len) { code[j] = word | (len << 16); ++word; ++have; }
    }
    return have == n;
}

nuq_status nuq_set_level_code(const uint8_t* lengths, uint32_t s) {
    std::lock_guard<std::mutex> lock(g_mu);
    if (!lengths || s < 1 || s > kMaxCodedS) return NUQ_ERR_INVALID_ARG;
    uint32_t code[kMaxCodedS + 1] = {0};
    if (!canonical_code(lengths, s + 1, code)) return NUQ_ERR_INVALID_ARG;
    for (uint32_t j = 0; j <= kMaxCodedS; ++j) g_level_code[j] = j <= s ? code[j] : 0u;
    g_level_code_n = s + 1;
    return NUQ_OK;
}

nuq_status nuq_fit_level_code(const uint64_t* hist, uint32_t s, uint8_t* lengths) {
    if (!hist || !lengths || s < 1 || s > kMaxCodedS) return NUQ_ERR_INVALID_ARG;
    // Huffman's construction with two queues: the leaves sorted by (count, index) and the joined nodes in
    // the order they were made (their weights never decrease).  The lighter front is taken, a leaf
    // before a joined node of the same weight.
    const uint32_t n = s + 1;
    uint32_t order[kMaxCodedS + 1];
    for (uint32_t i = 0; i < n; ++i) order[i] = i;
    for (uint32_t i = 1; i < n; ++i)                        // insertion sort, stable: equal counts stay in index order
        for (uint32_t k = i; k > 0 && hist[1 + order[k]] < hist[1 + order[k - 1]]; --k) {
            const uint32_t t = order[k]; order[k] = order[k - 1]; order[k - 1] = t;
        }
    uint64_t weight[2 * (kMaxCodedS + 1)];
    int parent[2 * (kMaxCodedS + 1)];
    for (uint32_t i = 0; i < n; ++i) { weight[i] = hist[1 + i]; parent[i] = -1; }
    uint32_t leaf = 0, joined = n, made = n;                // fronts of the two queues, next node to make
    for (uint32_t step = 0; step + 1 < n; ++step) {
        int pick[2];
        for (int k = 0; k < 2; ++k) {
            const bool leaf_left = leaf < n, joined_left = joined < made;
            if (leaf_left && (!joined_left || weight[order[leaf]] <= weight[joined])) pick[k] = (int)order[leaf++];
            else pick[k] = (int)joined++;
        }
        weight[made] = weight[pick[0]] + weight[pick[1]];
        parent[made] = -1;
        parent[pick[0]] = parent[pick[1]] = (int)made;
        ++made;
    }
    for (uint32_t i = 0; i < n; ++i) {
        uint32_t depth = 0;
        for (int at = (int)i; parent[at] >= 0; at = parent[at]) ++depth;
        lengths[i] = (uint8_t)depth;
    }
    return NUQ_OK;
}

nuq_status nuq_level_histogram(const float* g, uint64_t d, uint32_t bucket, uint32_t s, uint32_t norm_kind, uint64_t seed,
                               uint64_t offset, uint64_t* hist, void* stream_) {
    std::lock_guard<std::mutex> lock(g_mu);
    cudaStream_t stream = static_cast<cudaStream_t>(stream_);
    EncodeParams P;
    Geometry& G = P.geo;
    if (!g || !hist || (reinterpret_cast<uintptr_t>(hist) & 7u) || (reinterpret_cast<uintptr_t>(g) & 15u)) return NUQ_ERR_INVALID_ARG;
    if ((norm_kind >> 16) & 0xffu) return NUQ_ERR_INVALID_ARG;                      // no mode: nothing is coded here
    if (!make_geometry(d, bucket, s, norm_kind, &G) || G.levelset == kLevelsUniform) return NUQ_ERR_INVALID_ARG;
    if (G.levelset == kLevelsTable && g_levels_s != s) return NUQ_ERR_INVALID_ARG;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return NUQ_ERR_CUDA;
    P.g = g;
    P.norms_in = nullptr;
    if (norm_kind & NUQ_TEST_NORMS) {
        if (!g_test_norms.count(dev) || !g_test_norms[dev]) return NUQ_ERR_INVALID_ARG;
        P.norms_in = g_test_norms[dev];
    } else {
        Workspace* ws = nullptr;
        WsEntry& e = g_ws[std::make_pair(dev, stream)];
        nuq_status st = get_workspace(stream, sizeof(Workspace), &ws, &dev);
        if (st == NUQ_OK) st = get_norms(stream, d, e);
        if (st != NUQ_OK) return st;
        if (launch_bucket_norms(g, G.d, G.bucket, G.norm_kind, e.norms, G.nb, stream) != cudaSuccess) return NUQ_ERR_CUDA;
        P.norms_in = e.norms;
    }
    P.out = nullptr; P.out_bits = nullptr; P.ws = nullptr;
    P.seed = seed;
    P.offset = offset;
    for (uint32_t j = 0; j < kMaxTableS + 2u; ++j) {
        P.levels[j] = G.levelset == kLevelsTable ? g_levels[j] : 0.0f;
        P.inv_width[j] = G.levelset == kLevelsTable ? g_inv_width[j] : 0.0f;
    }
    for (uint32_t j = 0; j <= kMaxCodedS; ++j) P.level_code[j] = 0;
    for (uint32_t r = 0; r < 10; ++r) {
        P.round_keys[2 * r] = (uint32_t)seed + r * 0x9E3779B9u;
        P.round_keys[2 * r + 1] = (uint32_t)(seed >> 32) + r * 0xBB67AE85u;
    }
    P.stage_words = P.window_words = P.patience = P.grid = P.cluster = P.overlap = P.let_next = P.warps = P.tile = 0;
    if (cudaMemsetAsync(hist, 0, 8 * (s + 2), stream) != cudaSuccess) return NUQ_ERR_CUDA;
    if (launch_level_histogram(P, hist, device_sms(dev), stream) != cudaSuccess) return NUQ_ERR_CUDA;
    return NUQ_OK;
}

nuq_status nuq_set_test_norms(const float* norms) {
    std::lock_guard<std::mutex> lock(g_mu);
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return NUQ_ERR_CUDA;
    g_test_norms[dev] = norms;
    return NUQ_OK;
}

nuq_status nuq_encode(const float* g, uint64_t d, uint32_t bucket, uint32_t s, uint32_t norm_kind, uint64_t seed,
                      uint64_t offset, void* out, uint64_t* out_bits, void* stream_) {
    std::lock_guard<std::mutex> lock(g_mu);
    cudaStream_t stream = static_cast<cudaStream_t>(stream_);
    EncodeParams P;
    Geometry& G = P.geo;
    if (!encode_args_ok(g, d, bucket, s, norm_kind, out, out_bits, &G)) return NUQ_ERR_INVALID_ARG;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return NUQ_ERR_CUDA;
    const EncodePlan pl = plan_encode(P, dev, norm_kind);
    P.grid = pl.want_grid;
    Workspace* ws = nullptr;
    WsEntry& e = g_ws[std::make_pair(dev, stream)];
    nuq_status st = get_workspace(stream, scan_state_bytes(most_tiles(d, device_sms(dev))), &ws, &dev);
    if (st == NUQ_OK && pl.norms_bytes && !(norm_kind & NUQ_TEST_NORMS)) st = get_norms(stream, d, e);
    if (st != NUQ_OK) return st;
    return enqueue_encode(P, pl, g, norm_kind, seed, offset, out, out_bits, ws, e.norms, &e, dev, stream);
}

nuq_status nuq_encode_static(const float* g, uint64_t d, uint32_t bucket, uint32_t s, uint32_t norm_kind,
                             uint64_t seed, uint64_t offset, void* out, uint64_t* out_bits, void* stream_) {
    std::lock_guard<std::mutex> lock(g_mu);
    cudaStream_t stream = static_cast<cudaStream_t>(stream_);
    EncodeParams P;
    Geometry& G = P.geo;
    if (!encode_args_ok(g, d, bucket, s, norm_kind, out, out_bits, &G)) return NUQ_ERR_INVALID_ARG;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return NUQ_ERR_CUDA;
    const EncodePlan pl = plan_encode(P, dev, norm_kind);
    if (pl.state_bytes + pl.norms_bytes > kStaticScratchBytes) return NUQ_ERR_CAPACITY;   // vector too long for the array
    P.grid = pl.want_grid;
    auto it = g_static_ws.find(dev);
    if (it == g_static_ws.end()) {
        // first call on this device: ask the runtime where this device keeps the array
        void* p = nullptr;
        if (cudaGetSymbolAddress(&p, g_static_scratch) != cudaSuccess || !p) {
            cudaGetLastError();
            return NUQ_ERR_CUDA;
        }
        it = g_static_ws.emplace(dev, static_cast<Workspace*>(p)).first;
    }
    // the array is shared by every stream of the device: it is cleared before every call
    float* const norms = reinterpret_cast<float*>(reinterpret_cast<char*>(it->second) + pl.state_bytes);
    return enqueue_encode(P, pl, g, norm_kind, seed, offset, out, out_bits, it->second, norms, nullptr, dev, stream);
}

// Shared by the two decode entry points.  `w` == nullptr: the sums only.
static nuq_status enqueue_decode(const void* const* streams, uint32_t K, uint64_t d, uint32_t bucket, uint32_t s, float* acc,
                                 float* w, float* yl, float alpha, float mu, float l, void* stream_) {
    std::lock_guard<std::mutex> lock(g_mu);
    cudaStream_t stream = static_cast<cudaStream_t>(stream_);
    DecodeParams P;
    if (!streams || K < 1 || K > kMaxK) return NUQ_ERR_INVALID_ARG;
    // (with one or two streams acc has to be given: a rule of the interface, which the kernels have no need of)
    if (!acc && (!w || K < 3)) return NUQ_ERR_INVALID_ARG;
    if (w && mu != 0.0f && !yl) return NUQ_ERR_INVALID_ARG;
    if (w && !(alpha == alpha && mu >= 0.0f && mu < 1.0f && l >= 0.0f && l <= 1.0f)) return NUQ_ERR_INVALID_ARG;
    if ((reinterpret_cast<uintptr_t>(acc) & 15u) || (reinterpret_cast<uintptr_t>(w) & 15u) ||
        (reinterpret_cast<uintptr_t>(yl) & 15u))
        return NUQ_ERR_INVALID_ARG;
    // the level set and mode come from each container's header; geometry only needs (d, bucket, s)
    if (!make_geometry(d, bucket, s, 0, &P.geo)) return NUQ_ERR_INVALID_ARG;
    for (uint32_t k = 0; k < K; ++k) {
        if (!streams[k] || (reinterpret_cast<uintptr_t>(streams[k]) & 15u)) return NUQ_ERR_INVALID_ARG;
        P.streams[k] = static_cast<const uint32_t*>(streams[k]);
    }
    for (uint32_t k = K; k < kMaxK; ++k) P.streams[k] = nullptr;
    P.K = K;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return NUQ_ERR_CUDA;
    if (!g_token_tables_ready.count(dev)) {
        if (upload_token_tables() != cudaSuccess) return NUQ_ERR_CUDA;
        g_token_tables_ready.insert(dev);
    }
    P.unit_subs = 0;                                    // (chosen at the launch)
    uint32_t fixed = 0, tokens = 0;                     // streams of each mode, as far as is known
    P.likely_levels = kLevelsExp;
    bool alike = true;
    for (uint32_t k = 0; k < K; ++k) {
        const auto it = g_container_mode.find(std::make_pair(dev, streams[k]));
        const uint32_t mode = it == g_container_mode.end() ? kModeErc : it->second & 0xffu;
        const uint32_t levels = it == g_container_mode.end() ? kLevelsExp : it->second >> 8;
        fixed += mode == kModeFixed;
        tokens += mode == kModeErc;
        if (k == 0) P.likely_levels = levels;
        alike = alike && levels == P.likely_levels;
    }
    // (what is known of an address may be out of date, also in s: tables are only prepared for level sets that exist)
    const bool exists = P.likely_levels != kLevelsUniform || s <= 8u;
    P.likely_table = kTabCoded;
    if (exists && fixed == K && alike) P.likely_table = kTabFields;
    else if (exists && tokens == K) P.likely_table = P.likely_levels == kLevelsUniform ? kTabUniform : kTabErc;
    P.sum.acc = acc;
    P.sum.w = w;
    P.sum.yl = w && mu != 0.0f ? yl : nullptr;
    P.sum.step_c = w ? (float)((double)alpha / (double)K) : 0.0f;          // one rounding each
    P.sum.step_lc = w ? (float)((double)l * (double)alpha / (double)K) : 0.0f;
    P.sum.mu = w ? mu : 0.0f;
    P.minus_zero = -0.0f;
    Workspace* ws = nullptr;
    nuq_status st = get_workspace(stream, sizeof(Workspace), &ws, &dev);
    if (st != NUQ_OK) return st;
    P.ws = ws;
    P.let_next = 0;                                     // (chosen at the launch, like unit_subs)
    if (launch_decode(P, device_sms(dev), stream) != cudaSuccess) return NUQ_ERR_CUDA;
    return NUQ_OK;
}

nuq_status nuq_decode_accumulate(const void* const* streams, uint32_t K, uint64_t d, uint32_t bucket, uint32_t s,
                                 float* acc, void* stream) {
    if (!acc) return NUQ_ERR_INVALID_ARG;
    return enqueue_decode(streams, K, d, bucket, s, acc, nullptr, nullptr, 0.0f, 0.0f, 0.0f, stream);
}

nuq_status nuq_decode_update(const void* const* streams, uint32_t K, uint64_t d, uint32_t bucket, uint32_t s, float* acc,
                             float* w, float* yl, float alpha, float mu, float l, void* stream) {
    if (!w) return NUQ_ERR_INVALID_ARG;
    return enqueue_decode(streams, K, d, bucket, s, acc, w, yl, alpha, mu, l, stream);
}

nuq_status nuq_last_status(void* stream_) {
    std::lock_guard<std::mutex> lock(g_mu);
    cudaStream_t stream = static_cast<cudaStream_t>(stream_);
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return NUQ_ERR_CUDA;
    if (cudaStreamSynchronize(stream) != cudaSuccess) return NUQ_ERR_CUDA;
    int status = 0;
    auto it = g_ws.find(std::make_pair(dev, stream));
    if (it != g_ws.end() && it->second.ptr) {
        if (cudaMemcpy(&status, &it->second.ptr->status, sizeof(int), cudaMemcpyDeviceToHost) != cudaSuccess) return NUQ_ERR_CUDA;
        // (cleared in the stream itself: its next kernels do not wait for the default stream)
        if (status != 0 && cudaMemsetAsync(&it->second.ptr->status, 0, sizeof(int), stream) != cudaSuccess) return NUQ_ERR_CUDA;
    }
    auto st = g_static_ws.find(dev);               // kernels of nuq_encode_static latch into the static scratch
    if (st != g_static_ws.end()) {
        int s2 = 0;
        if (cudaMemcpy(&s2, &st->second->status, sizeof(int), cudaMemcpyDeviceToHost) != cudaSuccess) return NUQ_ERR_CUDA;
        if (s2 != 0 && cudaMemsetAsync(&st->second->status, 0, sizeof(int), stream) != cudaSuccess) return NUQ_ERR_CUDA;
        if (s2 < 0 ? s2 < status : status == 0) status = s2;    // (a warning only where there is no error)
    }
    return status;
}

nuq_status nuq_stream_info(const void* out, nuq_info* host_out, void* stream_) {
    if (!out || !host_out) return NUQ_ERR_INVALID_ARG;
    cudaStream_t stream = static_cast<cudaStream_t>(stream_);
    uint32_t h[kHeaderWords];
    if (cudaMemcpyAsync(h, out, sizeof(h), cudaMemcpyDeviceToHost, stream) != cudaSuccess) return NUQ_ERR_CUDA;
    if (cudaStreamSynchronize(stream) != cudaSuccess) return NUQ_ERR_CUDA;
    if (h[0] != kMagic || h[1] != kVersion) return NUQ_ERR_BAD_STREAM;
    auto u64 = [&](int i) { return (uint64_t)h[i] | ((uint64_t)h[i + 1] << 32); };
    host_out->d = u64(2);
    host_out->bucket = h[4];
    host_out->s = h[5];
    host_out->flags = h[6];
    host_out->sub_block = h[7];
    host_out->nblk = u64(8);
    host_out->container_bits = u64(10);
    host_out->code_bits = u64(12);
    host_out->nnz = u64(14);
    return NUQ_OK;
}

void nuq_shutdown(void) {
    std::lock_guard<std::mutex> lock(g_mu);
    int cur = 0;
    cudaGetDevice(&cur);
    for (auto& kv : g_ws) {
        cudaSetDevice(kv.first.first);
        cudaFree(kv.second.ptr);
        cudaFree(kv.second.norms);
    }
    g_ws.clear();
    cudaSetDevice(cur);
}

const char* nuq_version(void) { return "nuq-b200 0.1 (sm_100a)"; }

}  // extern "C"

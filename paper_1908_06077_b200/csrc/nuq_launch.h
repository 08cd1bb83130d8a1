// Host-side entry points of the kernel translation units.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include <set>

#include "nuq_common.cuh"

namespace nuq {

// Runs what has to be done once per device (a kernel's attributes are kept per device) before the first launch there.
// Its callers hold the library's mutex.
class OncePerDevice {
    std::set<int> done_;

public:
    template <class F>
    cudaError_t operator()(F&& prepare) {
        int dev = 0;
        cudaError_t e = cudaGetDevice(&dev);
        if (e != cudaSuccess || done_.count(dev)) return e;
        e = prepare();
        if (e == cudaSuccess) done_.insert(dev);
        return e;
    }
};

void build_erc_lut(uint32_t* lut256);                 // ERC(N), N = 1..256: code | len << 16
cudaError_t upload_erc_lut();                         // the encoder's tables, into the current device's memory; returns when they are there
cudaError_t launch_bucket_norms(const float* g, uint64_t d, uint32_t bucket, uint32_t norm_kind, float* norms,
                                uint64_t nb, cudaStream_t stream);
size_t encode_smem_bytes(const EncodeParams& P);      // dynamic shared memory of one encoder CTA
int encode_blocks_per_sm(const EncodeParams& P);      // encoder CTAs one SM holds at once (0 on error)
int encode_max_clusters(const EncodeParams& P);       // clusters of P.cluster encoder CTAs the device holds at once (0 on error)
cudaError_t launch_encode(const EncodeParams& P, cudaStream_t stream);
bool fixed4_applies(const Geometry& G);               // the call is served by the 4-bit fixed-width encoder
uint32_t fixed4_variant(const Geometry& G);           // which instance of it (0 to 2)
int fixed4_blocks_per_sm(const EncodeParams& P);
cudaError_t launch_encode_fixed4(const EncodeParams& P, cudaStream_t stream);
cudaError_t launch_level_histogram(const EncodeParams& P, uint64_t* hist, int sms, cudaStream_t stream);   // hist: s + 2 zeroed counters
cudaError_t upload_token_tables();                    // the chain decoder's tables, likewise
cudaError_t launch_decode(const DecodeParams& P, int sms, cudaStream_t stream);

}  // namespace nuq

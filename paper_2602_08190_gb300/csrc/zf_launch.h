// zf_launch.h -- host-side launch descriptions of the decode kernels.
#pragma once
#include <cuda_runtime.h>

#include <cstring>

#include "zf_internal.h"

#ifdef __CUDACC__
#define ZF_HD __host__ __device__
#else
#define ZF_HD
#endif

namespace zf {

// Words of one decode stream's work queue: [0] next job, [1] CTAs done,
// [2, 2 + kAffinitySms) blocks taken from each SM's range (string-dictionary
// launches), zero between launches.
constexpr uint32_t kAffinitySms = 256;
constexpr uint32_t kQueueWords = 2 + kAffinitySms + 6;

// The chunk descriptors of a launch.  Up to kInlineChunks of them travel as
// the kernel's parameters; more are read from a device array that the caller
// has copied (a copy ahead of the first kernel costs a call 3 to 4 us: 22.6
// against 19.0 us for 1M resident rows of FOR, 41.3 against 38.7 us for their
// transfer).  A launch of any size carries the whole array: with room for 64,
// 128, 256 and 480 a call of one chunk takes 18.2, 18.5, 19.4 and 21.6 us; at
// 64 the calls of few chunks, which are the short ones, pay nothing for it.  A
// call of 65 chunks takes 24.5 us, one of 64 21.3.
constexpr uint32_t kInlineChunks = 64;
struct ChunkArgs {
    const ZfDevChunk* dev;   // device array, or null: the descriptors are in `inl`
    uint32_t n, pad;
    ZfDevChunk inl[kInlineChunks];
    // `host`: the descriptors on the host, used when `d` is null
    ChunkArgs(const ZfDevChunk* d, const ZfDevChunk* host, uint32_t count) : dev(d), n(count), pad(0) {
        if (!d) memcpy(inl, host, count * sizeof(ZfDevChunk));
    }
    ZF_HD const ZfDevChunk* list() const { return dev ? dev : inl; }
};

struct TileLaunch {
    const ZfDevChunk* chunks;   // device descriptors of this launch, or null
    const ZfDevChunk* host;     // the same on the host (read when chunks is null: nchunks <= kInlineChunks)
    uint32_t nchunks;
    uint32_t ntiles;            // warp jobs
    int scheme, dtype;          // -1, -1 for the batched work-queue kernel
    uint32_t tile_rows;         // rows per warp job
    uint32_t threads;
    uint32_t ctas_per_sm;       // 0 = occupancy limit
    uint32_t smem;              // dynamic shared memory: threads/32 slices of equal size
    int num_sms;
    uint32_t* err;
    uint32_t* queue;            // kQueueWords zeroed words owned by the launching stream
};

uint32_t warp_smem_bytes(int scheme, int dtype, uint32_t bmax);
cudaError_t launch_tiles(const TileLaunch& L, cudaStream_t s);
// LZ77 blocks, `runs` of them with ChunkInfo::lz_runs.
cudaError_t launch_lz(const ZfDevChunk* chunks, const ZfDevChunk* host, uint32_t n, uint32_t runs, uint32_t* err,
                      int num_sms, cudaStream_t s);
cudaError_t launch_lz_cta(const ChunkArgs& chunks, uint32_t* err, cudaStream_t s);
// String-dictionary chunks whose dictionaries take at most dict_bytes
// (ChunkInfo::dict_bytes, at most strdict_smem_limit()) of shared memory;
// descriptors carry tile0 and ntiles in 1024-token tiles.
uint32_t strdict_smem_limit();
cudaError_t launch_strdict(const ZfDevChunk* chunks, const ZfDevChunk* host, uint32_t nchunks, uint32_t ntiles,
                           uint32_t dict_bytes, uint32_t* err, int num_sms, cudaStream_t s);
// ANS chunks: njobs warp jobs of up to 32 streams (chunk descriptors carry tile0 in jobs).
cudaError_t launch_ans(const ZfDevChunk* chunks, const ZfDevChunk* host, uint32_t nchunks, uint32_t njobs, uint32_t* err,
                       cudaStream_t s);

}  // namespace zf

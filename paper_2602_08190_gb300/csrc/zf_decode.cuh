// zf_decode.cuh -- one warp job of any scheme and type, for the kernels that
// decode them (zf_kernels.cu, zf_noalloc.cu).
#pragma once
#include "zf_strdict.cuh"

namespace zfd {

// Decode rows [r0, r0 + nrows) of a chunk (string dictionary: tokens) by one
// warp.  MIXED: the kernel decodes every scheme.
template <int SCHEME, int DT, bool MIXED>
__device__ __forceinline__ void decode_one(const ZfDevChunk& c, const Hdr& h, uint32_t r0, uint32_t nrows,
                                           uint32_t* wsm, uint32_t* err) {
    if constexpr (DT == ZF_I32 || DT == ZF_I64) {
        using T = typename std::conditional<DT == ZF_I64, int64_t, int32_t>::type;
        if constexpr (SCHEME == ZF_FOR_BP || SCHEME == ZF_DICT_BP || SCHEME == ZF_RAW)
            fp_job<T, SCHEME>(c, h, r0, nrows, wsm, err);
        else if constexpr (SCHEME == ZF_DELTA_BP)
            delta_job<T>(c, h, r0, nrows, wsm, err, c.bmax);
        else if constexpr (SCHEME == ZF_RLE)
            rle_job<T, MIXED>(c, h, r0, nrows, wsm, err);
    } else if constexpr (DT == ZF_F64) {
        // doubles travel as their 64-bit patterns
        if constexpr (SCHEME == ZF_RAW || SCHEME == ZF_FLOAT2INT) fp_job<int64_t, SCHEME>(c, h, r0, nrows, wsm, err);
    } else if constexpr (DT == ZF_BYTES && SCHEME == ZF_STRDICT) {
        strdict_job(c, h, r0, nrows, wsm, err);   // r0, nrows count tokens
    } else if constexpr (DT == ZF_BYTES && SCHEME == ZF_RAW) {
        // raw bytes: 16-byte copies
        const uint32_t lane = threadIdx.x & 31;
        const uint8_t* src = c.blob + h.off[0] + r0;
        uint8_t* dst = c.dst + r0;
        for (uint32_t i0 = lane * 16; i0 < nrows; i0 += 512) {
            if (i0 + 16 <= nrows) reinterpret_cast<uint4*>(dst + i0)[0] = ldg16(src + i0);
            else
                for (uint32_t i = i0; i < nrows; i++) dst[i] = src[i];
        }
    }
}

}  // namespace zfd

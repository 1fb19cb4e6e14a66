// zf_device.cuh -- device-side decode of one warp job: up to K consecutive
// 1024-row warp tiles of one chunk, per scheme.
//
// A launch decodes a list of chunks (ZfDevChunk) cut into warp jobs.  Each
// warp decodes its job alone, in its own slice of shared memory, with no
// CTA-wide barrier.  Inside a job the warp fetches all block / directory
// metadata of its tiles at once and copies the next tile's compressed bytes
// into shared memory (cp.async, double-buffered) while it decodes the
// current tile, so DRAM latency overlaps the decode.  The decoders follow
// the parallel patterns of Section 3.1:
//   fp_job      Fully-Parallel: FOR / dictionary / Float2Int / raw.  Every
//               lane extracts C = 16/sizeof(T) consecutive values of the
//               staged bits with funnel shifts and writes them with one
//               16-byte store (coalesced).  Float2Int makes each integer
//               the double nearest d / 10^e with integer multiplies
//               (zf_f2i.h) and then patches the chunk's exceptions.
//   delta_job   Group-Parallel: one 1024-row block at a time, 128 values per
//               step: every lane extracts four differences, a warp shuffle
//               scan of their sums places them, and the values leave with one
//               coalesced vector store per lane.
//   rle_job     Group-Parallel: the tile's run lengths (the chunk's 1024-row
//               directory names the first run) are scanned into start rows,
//               four or eight per lane and one warp shuffle scan (the
//               presum of Section 3.2); every run but the first sets its start
//               row's bit in a 32-word bitmask, and a row's run is the number
//               of set bits at or before it.  Each tile writes exactly 1024
//               rows, so long and short runs balance.
//   strdict_job (zf_strdict.cuh) Group-Parallel: string-dictionary tokens
//               of a byte column, placed by one warp scan of their lengths.
// A failed check of the stream sets a bit in the launch's error word; the
// tile then writes in-bounds placeholder values.  Nothing traps.
#pragma once
#include <cuda_pipeline.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <type_traits>

#include "zf_f2i.h"
#include "zf_internal.h"

namespace zfd {

// Reciprocals of 5^e for the Float2Int value (zf_f2i.h); a warp job reads one
// row, the same for all its lanes.
static __constant__ zf::F2IRecip kF2IRecip[zf::kF2IMaxExp + 1] = {ZF_F2I_RECIP_ROWS};

constexpr uint32_t kWarpRows = 1024;

struct Hdr {
    uint32_t rows, n_aux, b, flags;
    uint64_t ref;
    uint32_t off[3], len[3];
};

__device__ __forceinline__ uint4 ldg16(const void* p) { return __ldg(reinterpret_cast<const uint4*>(p)); }

__device__ __forceinline__ void load_hdr(const uint8_t* blob, Hdr& h) {
    uint4 a = ldg16(blob), b = ldg16(blob + 16), c = ldg16(blob + 32);
    h.b = (a.y >> 16) & 0xFF;
    h.flags = a.y >> 24;
    h.rows = a.z;
    h.n_aux = a.w;
    h.ref = ((uint64_t)b.y << 32) | b.x;
    h.off[0] = b.z;
    h.off[1] = b.w;
    h.off[2] = c.x;
    h.len[0] = c.y;
    h.len[1] = c.z;
    h.len[2] = c.w;
}

__device__ __forceinline__ void report(uint32_t* err, uint32_t code, uint32_t chunk_id) {
    atomicOr(&err[0], 1u << code);
    atomicCAS(&err[1], 0xFFFFFFFFu, chunk_id);
}

// Bits [bitpos, bitpos + b) of a little-endian word stream in shared memory.
__device__ __forceinline__ uint64_t extract(const uint32_t* sm, uint32_t bitpos, uint32_t b) {
    uint32_t w = bitpos >> 5, sh = bitpos & 31;
    uint32_t w0 = sm[w], w1 = sm[w + 1];
    uint32_t lo = __funnelshift_r(w0, w1, sh);
    if (b <= 32) return b == 32 ? lo : (lo & ((1u << b) - 1u));
    uint32_t hi = __funnelshift_r(w1, sm[w + 2], sh);
    uint64_t v = ((uint64_t)hi << 32) | lo;
    return b == 64 ? v : (v & ((1ull << b) - 1ull));
}

// One 256-bit store of four 64-bit words to a 32-byte aligned global address:
// a lane writes a whole L2 sector at once.  st.global takes a global-space
// address, so the generic pointer is converted first.  The decoders that use
// it are inlined into their kernels (the batched kernel included): inside a
// function called out of line (through the ABI) the same store was seen to
// write only its first word on sm_103a, so no out-of-line function uses it
// (delta_block_wide).
__device__ __forceinline__ void store32(void* dst, unsigned long long a, unsigned long long b, unsigned long long c,
                                        unsigned long long d) {
    const size_t g = __cvta_generic_to_global(dst);
    asm volatile("st.global.v4.b64 [%0], {%1, %2, %3, %4};" ::"l"(g), "l"(a), "l"(b), "l"(c), "l"(d) : "memory");
}

// Store N consecutive values of type T with the widest aligned vector stores
// (the values are packed into 32-bit words in registers first).  32-byte rows
// use one 256-bit store when `al32` says the address is 32-byte aligned, so
// a lane writes a whole L2 sector at once.
template <class T, int N>
__device__ __forceinline__ void store_vec(T* dst, const T (&v)[N], bool al32 = false) {
    static_assert(sizeof(T) == 4 || sizeof(T) == 8, "int32 or int64 values");
    constexpr int W = N * (int)sizeof(T) / 4;
    uint32_t w[W];
#pragma unroll
    for (int k = 0; k < N; k++) {
        if constexpr (sizeof(T) == 8) {
            w[2 * k] = (uint32_t)(uint64_t)v[k];
            w[2 * k + 1] = (uint32_t)((uint64_t)v[k] >> 32);
        } else {
            w[k] = (uint32_t)v[k];
        }
    }
    if constexpr (W == 8) {
        if (al32) {
            store32(dst, ((unsigned long long)w[1] << 32) | w[0], ((unsigned long long)w[3] << 32) | w[2],
                    ((unsigned long long)w[5] << 32) | w[4], ((unsigned long long)w[7] << 32) | w[6]);
            return;
        }
    }
    if constexpr (W % 4 == 0) {
#pragma unroll
        for (int q = 0; q < W / 4; q++)
            reinterpret_cast<uint4*>(dst)[q] = make_uint4(w[4 * q], w[4 * q + 1], w[4 * q + 2], w[4 * q + 3]);
    } else if constexpr (W % 2 == 0) {
#pragma unroll
        for (int q = 0; q < W / 2; q++) reinterpret_cast<uint2*>(dst)[q] = make_uint2(w[2 * q], w[2 * q + 1]);
    } else {
#pragma unroll
        for (int q = 0; q < W; q++) reinterpret_cast<uint32_t*>(dst)[q] = w[q];
    }
}

template <class S>
__device__ __forceinline__ S warp_incl_sum(S x, uint32_t lane) {
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        S y = __shfl_up_sync(0xFFFFFFFFu, x, d);
        if (lane >= (uint32_t)d) x += y;
    }
    return x;
}

// ---------------------------------------------------------------- async staging
// Copy `nbytes` (rounded up to 16) from a 16-byte aligned global address into
// a warp's shared-memory buffer with cp.async, 16 bytes per lane per step.
// The caller commits the group.
__device__ __forceinline__ void stage_async(uint32_t* buf, const uint8_t* src, uint32_t nbytes, uint32_t lane) {
    const uint32_t nvec = (nbytes + 15) >> 4;
    for (uint32_t i = lane; i < nvec; i += 32) __pipeline_memcpy_async(buf + 4 * i, src + 16ull * i, 16);
}

// Four consecutive b-bit values starting at bit `bitpos`.  NARROW needs
// b <= 8 (4b + 31 <= 63: one 64-bit window of two words).
template <bool NARROW, class S>
__device__ __forceinline__ void extract4(const uint32_t* wsm, uint32_t bitpos, uint32_t b, S (&u)[4]) {
    if constexpr (NARROW) {
        const uint32_t w = bitpos >> 5, sh = bitpos & 31;
        const uint64_t x = ((((uint64_t)wsm[w + 1]) << 32) | wsm[w]) >> sh;
        const uint32_t m = (1u << b) - 1u;
#pragma unroll
        for (int k = 0; k < 4; k++) u[k] = (S)((uint32_t)(x >> (k * b)) & m);
    } else {
#pragma unroll
        for (int k = 0; k < 4; k++) u[k] = (S)extract(wsm, bitpos + k * b, b);
    }
}

// Bytes of one staging buffer of a warp for packed payloads of width bmax.
__host__ __device__ inline uint32_t stage_bytes_for(uint32_t bmax) { return ((kWarpRows * bmax / 8 + 15) & ~15u) + 32; }

// ---------------------------------------------------------------- Fully-Parallel
// Extract and store the rows of a staged FOR/dictionary/Float2Int warp tile;
// returns true if a dictionary code was out of range or a Float2Int integer
// was beyond 2^53.
// FLOAT2INT (T = int64 bits of the doubles): the integer d = reference + u
// becomes the double nearest d / 10^e, built with integer multiplies
// (zf::f2i_bits; `e` and its reciprocal row `rr` are the chunk's).
// WIN: 1 = NARROW (b <= 8, four int32 values from one two-word window),
// 0 = one extraction per value, 2 = Float2Int chunk whose integers all lie in
// [0, 2^32) with e >= 1 (32-bit extraction and zf::f2i_bits_u32, `kexp` the
// chunk's exponent constant).
template <class T, int SCHEME, int WIN>
__device__ __forceinline__ bool fp_rows(const ZfDevChunk& c, const Hdr& h, T* dst, const uint32_t* wsm, uint32_t nr,
                                        uint32_t b, uint32_t lane, uint32_t e = 0,
                                        const zf::F2IRecip& rr = zf::F2IRecip{0, 0, 0, 0}, bool chk = true,
                                        int32_t kexp = 0) {
    // Float2Int and dictionaries: four values (a 32-byte sector of 64-bit ones)
    // per lane per step.  Two gathers at a time of int64 values from a
    // dictionary of 1,000 or 20,000 took 139 and 232 us for 64M rows, four take
    // 134 and 212; FOR values, DRAM bound, measured the same with four.
    constexpr int V = SCHEME == ZF_FLOAT2INT || SCHEME == ZF_DICT_BP ? 4 : 16 / sizeof(T);
    const T* dict = reinterpret_cast<const T*>(c.blob + h.off[0]);
    const T ref = (T)h.ref;
    const bool al32 = (reinterpret_cast<uintptr_t>(dst) & 31) == 0;
    bool bad = false;
#pragma unroll 2
    for (uint32_t i0 = lane * V; i0 < nr; i0 += 32 * V) {
        if constexpr (WIN == 2) {
            const uint32_t m32 = b >= 32 ? 0xFFFFFFFFu : (1u << b) - 1u, ref32 = (uint32_t)h.ref;
            T v[V];
#pragma unroll
            for (int k = 0; k < V; k++) {
                const uint32_t pos = (i0 + k) * b, w = pos >> 5;
                const uint32_t u = __funnelshift_r(wsm[w], wsm[w + 1], pos & 31) & m32;
                v[k] = (T)zf::f2i_bits_u32(ref32 + u, e, rr, kexp);
            }
            if (i0 + V <= nr) {
                store_vec<T, V>(dst + i0, v, al32);
            } else {
#pragma unroll
                for (int k = 0; k < V; k++)
                    if (i0 + k < nr) dst[i0 + k] = v[k];
            }
            continue;
        }
        uint64_t u[V];
        if constexpr (WIN == 1 && V == 4) {
            uint32_t w4[4];
            extract4<true, uint32_t>(wsm, i0 * b, b, w4);
#pragma unroll
            for (int k = 0; k < V; k++) u[k] = w4[k];
        } else {
#pragma unroll
            for (int k = 0; k < V; k++) u[k] = extract(wsm, (i0 + k) * b, b);
        }
        T v[V];
#pragma unroll
        for (int k = 0; k < V; k++) {
            if constexpr (SCHEME == ZF_FOR_BP) {
                v[k] = (T)(ref + (T)u[k]);
            } else if constexpr (SCHEME == ZF_FLOAT2INT) {
                const int64_t d = (int64_t)(h.ref + u[k]);
                if (chk) bad |= i0 + k < nr && (d > zf::kF2IDMax || d < -zf::kF2IDMax);
                v[k] = (T)zf::f2i_bits(d, e, rr);
            } else {
                const bool in = i0 + k < nr;
                bad |= in && u[k] >= h.n_aux;
                v[k] = (in && u[k] < h.n_aux) ? __ldg(dict + u[k]) : (T)0;
            }
        }
        if (i0 + V <= nr) {
            store_vec<T, V>(dst + i0, v, al32);
        } else {
#pragma unroll
            for (int k = 0; k < V; k++)
                if (i0 + k < nr) dst[i0 + k] = v[k];
        }
    }
    return bad;
}

// Float2Int exceptions of rows [r0, r0 + nrows): their rows are ascending,
// so a 32-way search (one load per lane per round) finds the first at or
// after r0, and the warp writes the stored 64 bits over the decoded rows.
__device__ __forceinline__ void f2i_exceptions(const ZfDevChunk& c, const Hdr& h, unsigned long long* dst,
                                               uint32_t r0, uint32_t nrows, uint32_t lane) {
    const uint32_t n = h.n_aux;
    if (n == 0) return;
    const uint32_t* pos = reinterpret_cast<const uint32_t*>(c.blob + h.off[1]);
    const unsigned long long* val = reinterpret_cast<const unsigned long long*>(c.blob + h.off[2]);
    uint32_t lo = 0, hi = n;                      // rows at indices < lo are < r0; index hi counts as >= r0
    while (hi - lo > 32) {
        const uint32_t step = (hi - lo + 31) / 32, idx = lo + lane * step;
        const uint32_t ge = __ballot_sync(0xFFFFFFFFu, idx >= hi || __ldg(pos + idx) >= r0);
        if (ge & 1u) {
            hi = lo;
        } else {
            const uint32_t f = ge ? __ffs(ge) - 1 : 32;   // first sample at or after r0 (32: none)
            const uint32_t prev = lo + (f - 1) * step;
            hi = f < 32 ? min(hi, lo + f * step) : hi;
            lo = prev + 1;
        }
    }
    const uint32_t idx = lo + lane;
    const uint32_t ge = __ballot_sync(0xFFFFFFFFu, idx >= hi || __ldg(pos + idx) >= r0);
    uint32_t k0 = ge ? lo + __ffs(ge) - 1 : hi;
    __syncwarp();   // the decoded rows of this warp are written before they are replaced
    for (;; k0 += 32) {
        const uint32_t k = k0 + lane;
        const uint32_t r = k < n ? __ldg(pos + k) : 0xFFFFFFFFu;
        const bool in = r >= r0 && r - r0 < nrows;
        if (in) dst[r - r0] = __ldg(val + k);
        if (!__any_sync(0xFFFFFFFFu, in && k < n)) break;
    }
}

// SCHEME: ZF_FOR_BP, ZF_DICT_BP, ZF_FLOAT2INT or ZF_RAW.  Rows [r0, r0 + nrows)
// of the chunk (r0 a multiple of 1024).  The packed stream of consecutive
// tiles is contiguous, so tile i+1 is staged while tile i decodes.
template <class T, int SCHEME>
__device__ void fp_job(const ZfDevChunk& c, const Hdr& h, uint32_t r0, uint32_t nrows, uint32_t* wsm,
                       uint32_t* err) {
    constexpr int V = 16 / sizeof(T);
    const uint32_t lane = threadIdx.x & 31;
    T* dst = reinterpret_cast<T*>(c.dst) + r0;
    if constexpr (SCHEME == ZF_RAW) {
        const T* src = reinterpret_cast<const T*>(c.blob + h.off[0]) + r0;
        for (uint32_t i0 = lane * V; i0 < nrows; i0 += 32 * V) {
            if (i0 + V <= nrows) reinterpret_cast<uint4*>(dst + i0)[0] = ldg16(src + i0);
            else
                for (uint32_t i = i0; i < nrows; i++) dst[i] = src[i];
        }
    } else {
        const uint32_t b = h.b;
        uint32_t e = 0;
        zf::F2IRecip rr{0, 0, 0, 0};
        bool chk = true;   // Float2Int: whether an integer of the chunk can pass 2^53
        bool u32 = false;  // Float2Int: e >= 1 and every integer of the chunk in [0, 2^32)
        if constexpr (SCHEME == ZF_FLOAT2INT) {
            e = c.blob[48];
            if (e > (uint32_t)zf::kF2IMaxExp) {
                if (lane == 0) report(err, ZF_ECORRUPT, c.chunk_id);
                return;
            }
            rr = kF2IRecip[e];
            const int64_t ref = (int64_t)h.ref;
            if (b <= 54 && ref >= -zf::kF2IDMax && ref <= zf::kF2IDMax)
                chk = ref + (int64_t)((1ull << b) - 1) > zf::kF2IDMax;
            u32 = e >= 1 && b <= 32 && ref >= 0 && ref + (int64_t)((1ull << b) - 1) < ((int64_t)1 << 32);
        }
        if (b > 8 * sizeof(T) || (SCHEME == ZF_DICT_BP && b > 16)) {
            if (lane == 0) report(err, ZF_ECORRUPT, c.chunk_id);
            return;
        }
        const uint8_t* sec = c.blob + h.off[SCHEME == ZF_DICT_BP ? 1 : 0];
        const uint32_t sb = stage_bytes_for(b) / 4;          // words per staging buffer
        const uint32_t ntiles = (nrows + kWarpRows - 1) / kWarpRows;
        auto issue = [&](uint32_t i) {
            const uint32_t rr = r0 + i * kWarpRows, nr = min(kWarpRows, r0 + nrows - rr);
            stage_async(wsm + (i & 1) * sb, sec + ((uint64_t)rr * b >> 3), (nr * b + 7) >> 3, lane);
            __pipeline_commit();
        };
        issue(0);
        bool bad = false;
        for (uint32_t i = 0; i < ntiles; i++) {
            if (i + 1 < ntiles) {
                issue(i + 1);
                __pipeline_wait_prior(1);
            } else {
                __pipeline_wait_prior(0);
            }
            __syncwarp();
            const uint32_t nr = min(kWarpRows, nrows - i * kWarpRows);
            const uint32_t* buf = wsm + (i & 1) * sb;
            if (V == 4 && b <= 8) bad |= fp_rows<T, SCHEME, 1>(c, h, dst + i * kWarpRows, buf, nr, b, lane);
            else if (SCHEME == ZF_FLOAT2INT && u32)
                fp_rows<T, SCHEME, 2>(c, h, dst + i * kWarpRows, buf, nr, b, lane, e, rr, false,
                                      1052 - (int32_t)rr.s - (int32_t)e);
            else bad |= fp_rows<T, SCHEME, 0>(c, h, dst + i * kWarpRows, buf, nr, b, lane, e, rr, chk);
            __syncwarp();
        }
        if (bad) report(err, ZF_ECORRUPT, c.chunk_id);
        if constexpr (SCHEME == ZF_FLOAT2INT)
            f2i_exceptions(c, h, reinterpret_cast<unsigned long long*>(dst), r0, nrows, lane);
    }
}

// ---------------------------------------------------------------- delta (Group-Parallel)
// A block of differences of more than 21 bits: 64-bit sums.  Each lane owns 32
// consecutive values [32*lane, 32*lane + 32): it sums its differences, one warp
// scan gives every lane its offset, and the values are rebuilt from a second
// extraction, so no array of prefixes stays live in registers.
template <class T>
__device__ __forceinline__ void delta_block_lanes(T* dst, const uint32_t* wsm, uint32_t mk, uint32_t b, uint64_t base,
                                                  uint64_t min_d, uint32_t lane) {
    using U = typename std::conditional<sizeof(T) == 8, unsigned long long, unsigned int>::type;
    constexpr int PER = 32 / sizeof(T);           // values per 32-byte store
    const uint32_t j0 = lane * 32;
    const uint32_t nv = mk > j0 ? min(32u, mk - j0) : 0u;   // valid values of this lane
    // difference k of the lane (u_0 of the block and slots past the block count as 0)
    auto diff = [&](uint32_t k) -> unsigned long long {
        return k >= nv || (k == 0 && lane == 0) ? 0ull : extract(wsm, (j0 + k) * b, b);
    };
    unsigned long long total = 0;
#pragma unroll
    for (uint32_t k = 0; k < 32; k++) total += diff(k);
    const unsigned long long excl = warp_incl_sum<unsigned long long>(total, lane) - total;
    const U md = (U)min_d;
    // x_{j0+k} = base + (j0 + k) * min_d + (differences up to j0 + k): acc after
    // step k, where each step adds min_d + u_k
    U acc = (U)base + (U)j0 * md + (U)excl - md;
#pragma unroll
    for (int q = 0; q < 32 / PER; q++) {
        T v[PER];
#pragma unroll
        for (int e = 0; e < PER; e++) {
            acc += md + (U)diff(q * PER + e);
            v[e] = (T)acc;
        }
        if ((uint32_t)(q * PER + PER) <= nv) {
            store_vec<T, PER>(dst + j0 + q * PER, v);
        } else {
#pragma unroll
            for (int e = 0; e < PER; e++)
                if ((uint32_t)(q * PER + e) < nv) dst[j0 + q * PER + e] = v[e];
        }
    }
}

// Four consecutive differences of b bits from bit `pos` of the staged words.
// W = 1: b <= 8, all four in one window of two words; W = 2: b <= 16, two in
// each window; W = 4: one.
template <int W>
__device__ __forceinline__ void delta_diffs(const uint32_t* wsm, uint32_t pos, uint32_t b, uint32_t mask, uint32_t (&u)[4]) {
    constexpr int PER = 4 / W;
#pragma unroll
    for (int g = 0; g < W; g++) {
        const uint32_t p = pos + g * PER * b, w = p >> 5, sh = p & 31;
        const uint32_t w0 = wsm[w], w1 = wsm[w + 1];
        const uint32_t lo = __funnelshift_r(w0, w1, sh), hi = w1 >> sh;
#pragma unroll
        for (int k = 0; k < PER; k++) u[g * PER + k] = (k ? __funnelshift_r(lo, hi, k * b) : lo) & mask;   // k * b <= 24
    }
}

// A block of differences of at most 21 bits (32-bit sums: 1024 * (2^21 - 1) <
// 2^31), 128 values per step: lane l takes four consecutive differences, one
// warp scan of the lanes' sums places them, and the values leave with one
// coalesced 16- or 32-byte store per lane.  OFF32: base + j * min_d + sum fits
// 32 bits past the base (the caller has checked), so a 64-bit value is one
// 32-bit multiply-add and one 64-bit add.
// What bounds it: DRAM for int64 (64M rows, gaps of mean 4: 108 us per resident
// call, 6.0 TB/s over its kernel), the issue of 27 instructions a row and the
// scans' latency for int32 (77 us).  Lanes that owned 32 consecutive values,
// extracted them twice and turned them in shared memory took 39 instructions a
// row, 117 and 96 us.
template <class T, int W, bool OFF32>
__device__ __forceinline__ void delta_block(T* dst, const uint32_t* wsm, uint32_t mk, uint32_t b, uint64_t base,
                                            uint64_t min_d, uint32_t lane) {
    using U = typename std::conditional<sizeof(T) == 8, unsigned long long, unsigned int>::type;
    const uint32_t mask = (1u << b) - 1u;
    const bool al32 = (reinterpret_cast<uintptr_t>(dst) & 31) == 0;
    uint32_t carry = 0;                                    // differences of the steps before
#pragma unroll 2
    for (uint32_t j = 4 * lane; j - 4 * lane < mk; j += 128) {
        uint32_t u[4];
        delta_diffs<W>(wsm, j * b, b, mask, u);
        if (j == 0) u[0] = 0;                              // u_0 of the block counts as 0
        // values past the block (mk < 1024) take whatever the buffer holds after the payload: nothing is stored for them
        u[1] += u[0];
        u[2] += u[1];
        u[3] += u[2];
        const uint32_t incl = warp_incl_sum<uint32_t>(u[3], lane);
        const uint32_t before = carry + incl - u[3];
        carry += __shfl_sync(0xFFFFFFFFu, incl, 31);
        T v[4];
#pragma unroll
        for (int k = 0; k < 4; k++) {
            if constexpr (OFF32) v[k] = (T)((U)base + ((j + k) * (uint32_t)min_d + (before + u[k])));
            else v[k] = (T)((U)base + (U)(j + k) * (U)min_d + (U)(before + u[k]));
        }
        if (j + 4 <= mk) {
            store_vec<T, 4>(dst + j, v, al32);
        } else {
#pragma unroll
            for (int k = 0; k < 4; k++)
                if (j + k < mk) dst[j + k] = v[k];
        }
    }
}

template <class T, int W>
__device__ __forceinline__ void delta_block_of(T* dst, const uint32_t* wsm, uint32_t mk, uint32_t b, uint64_t base,
                                               uint64_t min_d, uint32_t lane) {
    // min_d < 2^21: 1024 * (min_d + 2^b) < 2^32; 32-bit values need 32 bits anyway
    if (sizeof(T) == 4 || min_d < (1u << 21)) delta_block<T, W, true>(dst, wsm, mk, b, base, min_d, lane);
    else delta_block<T, W, false>(dst, wsm, mk, b, base, min_d, lane);
}

// Out of line, these rare blocks do not add to the registers of the common
// path.  They keep 16-byte stores: in an out-of-line function a 256-bit store
// from inline PTX wrote only part of its data (seen on GB300; the same store
// inlined is exact).
template <class T>
__device__ __noinline__ void delta_block_wide(T* dst, const uint32_t* wsm, uint32_t mk, uint32_t b, uint64_t base,
                                              uint64_t min_d, uint32_t lane) {
    delta_block_lanes<T>(dst, wsm, mk, b, base, min_d, lane);
}

// Blocks of rows [r0, r0 + nrows) (r0 a multiple of 1024, at most 32 blocks).
// Lane j holds block j's 24-byte entry; block i+1's payload is staged while
// block i decodes.
template <class T>
__device__ void delta_job(const ZfDevChunk& c, const Hdr& h, uint32_t r0, uint32_t nrows, uint32_t* wsm,
                          uint32_t* err, uint32_t bmax) {
    using U = typename std::conditional<sizeof(T) == 8, unsigned long long, unsigned int>::type;
    const uint32_t lane = threadIdx.x & 31;
    const uint32_t blk0 = r0 / zf::kDeltaBlock;
    const uint32_t nblk = (nrows + zf::kDeltaBlock - 1) / zf::kDeltaBlock;
    uint64_t e_base = 0, e_md = 0;
    uint32_t e_poff = 0, e_b = 0;
    if (lane < nblk) {
        const uint8_t* e = c.blob + h.off[0] + (uint64_t)(blk0 + lane) * zf::kDeltaEntry;
        const uint2 e0 = __ldg(reinterpret_cast<const uint2*>(e));
        const uint2 e1 = __ldg(reinterpret_cast<const uint2*>(e + 8));
        const uint2 e2 = __ldg(reinterpret_cast<const uint2*>(e + 16));
        e_base = ((uint64_t)e0.y << 32) | e0.x;
        e_md = ((uint64_t)e1.y << 32) | e1.x;
        e_poff = e2.x;
        e_b = e2.y & 0xFF;
    }
    // a block whose entry is inconsistent is reported and skipped
    const uint32_t mk_lane = min(zf::kDeltaBlock, nrows - min(nrows, lane * zf::kDeltaBlock));
    const bool lane_ok = lane >= nblk || (e_b <= 8 * sizeof(T) && e_b <= bmax && !(e_poff & 15) &&
                                          (uint64_t)e_poff + ((mk_lane * e_b + 7) >> 3) <= h.len[1]);
    const uint32_t ok_mask = __ballot_sync(0xFFFFFFFFu, lane_ok);
    if (ok_mask != 0xFFFFFFFFu && lane == 0) report(err, ZF_ECORRUPT, c.chunk_id);
    const uint32_t sb = stage_bytes_for(bmax) / 4;
    const uint8_t* payload = c.blob + h.off[1];
    auto issue = [&](uint32_t i) {
        const uint32_t poff = __shfl_sync(0xFFFFFFFFu, e_poff, i);
        const uint32_t b = __shfl_sync(0xFFFFFFFFu, e_b, i);
        const uint32_t mk = min(zf::kDeltaBlock, nrows - i * zf::kDeltaBlock);
        if ((ok_mask >> i) & 1) stage_async(wsm + (i & 1) * sb, payload + poff, (mk * b + 7) >> 3, lane);
        __pipeline_commit();
    };
    issue(0);
    for (uint32_t i = 0; i < nblk; i++) {
        if (i + 1 < nblk) {
            issue(i + 1);
            __pipeline_wait_prior(1);
        } else {
            __pipeline_wait_prior(0);
        }
        __syncwarp();
        const uint64_t base = __shfl_sync(0xFFFFFFFFu, e_base, i);
        const uint64_t md = __shfl_sync(0xFFFFFFFFu, e_md, i);
        const uint32_t b = __shfl_sync(0xFFFFFFFFu, e_b, i);
        const uint32_t mk = min(zf::kDeltaBlock, nrows - i * zf::kDeltaBlock);
        if ((ok_mask >> i) & 1) {
            T* dst = reinterpret_cast<T*>(c.dst) + r0 + i * zf::kDeltaBlock;
            const uint32_t* buf = wsm + (i & 1) * sb;
            if (b <= 8) delta_block_of<T, 1>(dst, buf, mk, b, base, md, lane);
            else if (b <= 16) delta_block_of<T, 2>(dst, buf, mk, b, base, md, lane);
            else if (b <= 21) delta_block_of<T, 4>(dst, buf, mk, b, base, md, lane);
            else delta_block_wide<T>(dst, buf, mk, b, base, md, lane);
        }
        __syncwarp();
    }
}

// ---------------------------------------------------------------- RLE (Group-Parallel)
// Start bits of the runs whose lengths are entries [sft, sft + m) of lens_al,
// PER entries per lane and step: the prefix sums give each run its start row in
// the tile, and every run but the first (whose start is at or before row 0)
// sets its bit.  A length counts as at most kLong rows, the first without the
// `skip` rows before the tile: the lengths that decide anything are those that
// end inside the tile, so no sum comes near 2^32 whatever the stream holds.
// Returns whether a length is zero or longer than the chunk; `end` = the rows
// covered from the tile's first row on, `last_start` = the last run's start.
template <int PER>
__device__ __forceinline__ bool rle_starts(const uint32_t* lens_al, uint32_t sft, uint32_t m, uint32_t skip, uint32_t nr,
                                           uint32_t chunk_rows, uint32_t* bm, uint32_t lane, uint32_t& end,
                                           uint32_t& last_start) {
    constexpr uint32_t kLong = 2048;
    const uint32_t n = sft + m;   // entries from the aligned start
    bool bad = false;
    end = 0;
    uint32_t mine = 0;
    for (uint32_t g = 0; g < n; g += 32 * PER) {
        const uint32_t k0 = g + PER * lane;
        uint32_t L[PER];
#pragma unroll
        for (int q = 0; q < PER / 4; q++) {
            const uint4 x = k0 + 4 * q < n ? reinterpret_cast<const uint4*>(lens_al)[(k0 >> 2) + q] : make_uint4(0, 0, 0, 0);
            L[4 * q] = x.x;
            L[4 * q + 1] = x.y;
            L[4 * q + 2] = x.z;
            L[4 * q + 3] = x.w;
        }
        uint32_t sum = 0;
#pragma unroll
        for (int e = 0; e < PER; e++) {
            const bool valid = k0 + e - sft < m;
            bad |= valid && L[e] - 1u >= chunk_rows;
            if (e < 4 && k0 + e == sft) {                      // the first run: entry 0..3 of lane 0
                bad |= skip >= L[e];
                L[e] -= min(skip, L[e]);
            }
            L[e] = valid ? min(L[e], kLong) : 0u;
            sum += L[e];
        }
        const uint32_t incl = warp_incl_sum<uint32_t>(sum, lane);
        uint32_t st = end + incl - sum;                        // start of entry k0
        end += __shfl_sync(0xFFFFFFFFu, incl, 31);
#pragma unroll
        for (int e = 0; e < PER; e++) {
            // starts 1 .. nr - 1: the first run's is 0, entries past the last start at nr or later
            if (st - 1u < nr - 1u && k0 + e < n) atomicOr(&bm[st >> 5], 1u << (st & 31));
            if (k0 + e + 1 == n) mine = st;
            st += L[e];
        }
    }
    last_start = __shfl_sync(0xFFFFFFFFu, mine, ((n - 1) % (32 * PER)) / PER);
    return bad;
}

// Expansion of one 1024-row tile whose runs [rf, rf+m) have their lengths at
// `lens_al` + sft, lens_al 16-byte aligned and sft = rf mod 4 (staged in shared
// memory, or in global memory when the tile has more runs than a staging
// buffer holds), and their values at `vals`.  `bm` is the warp's 32-word
// bitmask of the tile's rows.
// TIGHT: four entries per lane and step only, for a kernel that decodes every
// scheme and would spill registers with eight.
// What bounds it: issue slots with short runs, DRAM from runs of 64 on.  64M
// int32 rows in runs of mean 2, 4, 8 and 64: 152, 117, 78 and 70 us per
// resident call; with saturating sums, four entries a step whatever the tile
// and start bits merged per word in registers 181, 130, 83 and 73.
template <class T, bool TIGHT>
__device__ __forceinline__ void rle_rows(const ZfDevChunk& c, const Hdr& h, T* dst, const uint32_t* lens_al,
                                         uint32_t sft, const T* vals, uint32_t* bm, uint32_t m, uint32_t skip,
                                         uint32_t nr, bool last_tile, uint32_t next_skip, uint32_t lane,
                                         uint32_t* err) {
    bm[lane] = 0;
    __syncwarp();
    uint32_t end, last_start;
    bool bad;
    if (TIGHT || sft + m <= 128) bad = rle_starts<4>(lens_al, sft, m, skip, nr, h.rows, bm, lane, end, last_start);
    else bad = rle_starts<8>(lens_al, sft, m, skip, nr, h.rows, bm, lane, end, last_start);
    // The runs cover exactly [0, nr): the last ends at nr or continues into the
    // next tile by the directory's amount (a single run started `skip` rows before).
    if (m == 1) last_start = 0u - skip;
    const bool ok = last_tile || next_skip == 0 ? end == nr : last_start + next_skip == nr && end > nr;
    const bool any_bad = __any_sync(0xFFFFFFFFu, bad);
    if (lane == 0 && (!ok || any_bad)) report(err, ZF_ECORRUPT, c.chunk_id);
    __syncwarp();
    // A row's run (relative to the tile's first) is the number of run starts
    // at or before it: lane l holds word l of the bitmask and the starts in
    // the words before it (one shuffle scan of the popcounts).  Expansion, 256
    // rows per step: lane l takes rows 8l..8l+7, a quarter of one word.  Each
    // run sets at most one bit and the first sets none, so a count never
    // passes m - 1.
    const uint32_t word = bm[lane];
    const uint32_t cnt = __popc(word);
    const uint32_t before = warp_incl_sum<uint32_t>(cnt, lane) - cnt;
    constexpr int V = 8;
    const bool al32 = (reinterpret_cast<uintptr_t>(dst) & 31) == 0;
    const uint32_t o = (lane & 3) * 8;
    for (uint32_t row = 0; row * 256 < nr; row++) {
        const uint32_t j = row * 256 + lane * V;
        const uint32_t w = row * 8 + (lane >> 2);
        const uint32_t ww = __shfl_sync(0xFFFFFFFFu, word, w);
        uint32_t idx = __shfl_sync(0xFFFFFFFFu, before, w) + __popc(ww & ((1u << o) - 1u));
        const uint32_t b8 = ww >> o;
        T v[V];
#pragma unroll
        for (int k = 0; k < V; k++) {
            idx += (b8 >> k) & 1u;
            v[k] = vals[idx];
        }
        if (j + V <= nr) {
            if constexpr (sizeof(T) == 4) {
                store_vec<T, V>(dst + j, v, al32);
            } else {
                const T a[4] = {v[0], v[1], v[2], v[3]}, z[4] = {v[4], v[5], v[6], v[7]};
                store_vec<T, 4>(dst + j, a, al32);
                store_vec<T, 4>(dst + j + 4, z, al32);
            }
        } else {
#pragma unroll
            for (int k = 0; k < V; k++)
                if (j + k < nr) dst[j + k] = v[k];
        }
    }
    __syncwarp();
}

constexpr uint32_t kRleStageRuns = 256;   // runs per staging buffer
constexpr uint32_t kRleStages = 2;        // staging buffers per warp: tile i+1 loads while tile i expands

// Shared memory of one RLE staging buffer: lengths then values, each with
// room for the 16-byte aligned copy that starts up to 3 entries early.
__host__ __device__ inline uint32_t rle_buf_bytes(uint32_t value_bytes) {
    return (kRleStageRuns + 4) * 4 + (((kRleStageRuns + 4) * value_bytes + 15) & ~15u);
}

// Tiles of rows [r0, r0 + nrows) (r0 a multiple of 1024, at most 31 tiles).
// Lane j holds the directory entry of tile j (and of the tile after the
// last); the next tile's lengths and values are staged while a tile expands.
template <class T, bool TIGHT>
__device__ void rle_job(const ZfDevChunk& c, const Hdr& h, uint32_t r0, uint32_t nrows, uint32_t* wsm,
                        uint32_t* err) {
    const uint32_t lane = threadIdx.x & 31;
    if (h.rows > (1u << 30)) {   // chunks hold at most 2^30 rows
        if (lane == 0) report(err, ZF_ECORRUPT, c.chunk_id);
        return;
    }
    const T* vals = reinterpret_cast<const T*>(c.blob + h.off[0]);
    const uint32_t* lens = reinterpret_cast<const uint32_t*>(c.blob + h.off[1]);
    const uint2* dir = reinterpret_cast<const uint2*>(c.blob + h.off[2]);
    const uint32_t R = h.n_aux;
    const uint32_t t0 = r0 / zf::kRleDirRows;
    const uint32_t nt = (nrows + zf::kRleDirRows - 1) / zf::kRleDirRows;
    const uint32_t tiles_in_chunk = (h.rows + zf::kRleDirRows - 1) / zf::kRleDirRows;
    uint2 d = make_uint2(0, 0);
    if (lane <= nt && t0 + lane < tiles_in_chunk) d = __ldg(dir + t0 + lane);
    uint32_t* bm = wsm;
    uint8_t* bufs = reinterpret_cast<uint8_t*>(wsm) + 128;
    const uint32_t bb = rle_buf_bytes(sizeof(T));
    constexpr uint32_t VPER = 16 / sizeof(T);   // values per 16-byte copy
    // run range [rf, rf + m) of tile i, or m = 0 if its directory entries are inconsistent
    auto runs = [&](uint32_t i, uint32_t& rf, uint32_t& skip, uint32_t& m, uint32_t& next_skip, bool& last) {
        rf = __shfl_sync(0xFFFFFFFFu, d.x, i);
        skip = __shfl_sync(0xFFFFFFFFu, d.y, i);
        const uint32_t nx = __shfl_sync(0xFFFFFFFFu, d.x, i + 1);
        next_skip = __shfl_sync(0xFFFFFFFFu, d.y, i + 1);
        const uint32_t rr = r0 + i * zf::kRleDirRows, nr = min(zf::kRleDirRows, r0 + nrows - rr);
        last = rr + nr >= h.rows;
        uint32_t rl = R - 1;
        bool bad = (rr == 0 && (rf != 0 || skip != 0)) || R == 0 || skip >= h.rows;
        if (!last) {
            bad |= next_skip == 0 && nx == 0;
            rl = next_skip > 0 ? nx : nx - 1;
        } else {
            next_skip = 0;
        }
        bad |= rf > rl || rl >= R || rl - rf + 1 > nr + 1;
        m = bad ? 0 : rl - rf + 1;
    };
    auto issue = [&](uint32_t i) {
        uint32_t rf, skip, m, ns;
        bool last;
        runs(i, rf, skip, m, ns, last);
        if (m && m <= kRleStageRuns) {
            // 16-byte copies from the aligned entries at or before rf (the
            // sections are 16-byte aligned and padded, so they stay inside)
            uint8_t* b = bufs + (i % kRleStages) * bb;
            const uint32_t l0 = rf & ~3u, nl = (rf + m - l0 + 3) / 4;
            const uint32_t v0 = rf & ~(VPER - 1), nv = (rf + m - v0 + VPER - 1) / VPER;
            for (uint32_t k = lane; k < nl; k += 32)
                __pipeline_memcpy_async(b + 16 * k, lens + l0 + 4 * k, 16);
            for (uint32_t k = lane; k < nv; k += 32)
                __pipeline_memcpy_async(b + (kRleStageRuns + 4) * 4 + 16 * k, vals + v0 + VPER * k, 16);
        }
        __pipeline_commit();
    };
    // The next kRleStages - 1 tiles are staged while a tile expands (one
    // commit group per tile, empty ones included).  Deeper staging (four
    // buffers) measured slower on GB300: it costs occupancy.
    for (uint32_t i = 0; i + 1 < kRleStages && i < nt; i++) issue(i);
    for (uint32_t i = 0; i < nt; i++) {
        if (i + kRleStages - 1 < nt) issue(i + kRleStages - 1);
        switch (min(nt - 1, i + kRleStages - 1) - i) {   // groups committed after tile i's
        case 0: __pipeline_wait_prior(0); break;
        case 1: __pipeline_wait_prior(1); break;
        case 2: __pipeline_wait_prior(2); break;
        default: __pipeline_wait_prior(3); break;
        }
        __syncwarp();
        uint32_t rf, skip, m, ns;
        bool last;
        runs(i, rf, skip, m, ns, last);
        const uint32_t rr = r0 + i * zf::kRleDirRows, nr = min(zf::kRleDirRows, r0 + nrows - rr);
        if (!m) {
            if (lane == 0) report(err, ZF_ECORRUPT, c.chunk_id);
        } else {
            T* dst = reinterpret_cast<T*>(c.dst) + rr;
            if (m <= kRleStageRuns) {
                const uint8_t* b = bufs + (i % kRleStages) * bb;
                rle_rows<T, TIGHT>(c, h, dst, reinterpret_cast<const uint32_t*>(b), rf & 3u,
                                reinterpret_cast<const T*>(b + (kRleStageRuns + 4) * 4) + (rf & (VPER - 1)), bm, m,
                                skip, nr, last, ns, lane, err);
            } else {
                rle_rows<T, TIGHT>(c, h, dst, lens + (rf & ~3u), rf & 3u, vals + rf, bm, m, skip, nr, last, ns, lane,
                                err);
            }
        }
        __syncwarp();
    }
}

// ---------------------------------------------------------------- string dictionary sizes
// (the decoder is in zf_strdict.cuh)
constexpr uint32_t kStrCodeBuf = (1024u * 16u / 8u) + 32u;   // one tile of codes at b <= 16, plus the reader's overrun
constexpr uint32_t kStrWin = 16u * zf::kStrTokenMax + 32u;    // 16 tokens of at most 64 bytes, at the output's alignment

// Shared memory (bytes) one warp needs for a scheme, given the value size and
// the widest bit width of the chunks it decodes (two staging buffers).
__host__ __device__ inline uint32_t warp_smem(int scheme, uint32_t value_bytes, uint32_t bmax) {
    switch (scheme) {
    case ZF_FOR_BP: case ZF_DICT_BP: case ZF_FLOAT2INT: case ZF_DELTA_BP: return 2 * stage_bytes_for(bmax);
    case ZF_RLE: return 128 + kRleStages * rle_buf_bytes(value_bytes);   // row bitmask + staging buffers
    case ZF_STRDICT: return kStrCodeBuf + kStrWin;                      // one tile of codes + the output window
    }
    return 0;
}

}  // namespace zfd

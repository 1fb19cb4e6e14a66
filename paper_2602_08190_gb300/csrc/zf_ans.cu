// zf_ans.cu -- dictionary + range ANS decode.  Section 2.1 lists ANS among
// the entropy-based algorithms and Section 3.1 takes its decode as the
// Non-Parallel example: each decode state follows from the one before, so
// the parallelism comes from decoding many independent streams at once.  A
// chunk's rows are cut into streams of 2^k rows (header byte 48; the chunk
// size Section 5.2.3 varies); one warp job takes up to 32 streams of one
// chunk, one per lane, and the four warps of a CTA take consecutive jobs of
// the same chunk (every chunk's jobs are padded to a multiple of four).  The
// rANS coder is Duda's range variant with byte-wise renormalization; the
// layout is described with the container format in zf.h.
#include <cuda_runtime.h>

#include "zf_device.cuh"
#include "zf_launch.h"

namespace {

constexpr uint32_t kWarps = zf::kAnsJobsPerCta;   // warps (jobs) per CTA, all of one chunk

constexpr uint32_t kRing = 4;                     // 16-byte words of a lane's stream in shared memory

// The CTA's tables for its chunk.  A slot's entry holds its symbol, the
// symbol's frequency f and the slot's offset in the symbol's range [c, c + f),
// so a decode step takes one shared load for the state and one for the value.
// Up to 128 symbols: f << 19 | symbol << 12 | (slot - c), where a shift gives
// f; more (WIDE): symbol << 24 | (f - 1) << 12 | (slot - c).
struct AnsSmem {
    uint32_t slot[zf::kAnsM];
    unsigned long long val[zf::kAnsMaxSymbols];   // the symbols' values (64-bit patterns)
    uint32_t cum[zf::kAnsMaxSymbols + 1];         // cumulative frequencies, cum[nd] = M
    uint32_t wsum[kWarps];
    uint4 ring[kWarps * 32][kRing + 1];           // per lane: 16-byte word c of s2 at c mod kRing (one more: spreads the banks)
};

template <bool WIDE>
__device__ __forceinline__ uint32_t ans_entry(uint32_t sym, uint32_t f, uint32_t d) {
    return WIDE ? (sym << 24) | ((f - 1u) << 12) | d : (f << 19) | (sym << 12) | d;
}

// Stream k of the chunk, rows [k L, k L + n), decoded by one lane.  The
// stream's bytes [a0, a1) of s2 pass through a window of two 32-bit words,
// first byte on top.  Per row: the slot entry of x mod M gives the value and
// x = f (x >> 12) + (slot - c); then zero, one or two bytes enter while x < L
// (after a step x >= 2^11): one shift of the window brings its next 16 bits to
// the top, a funnel shift moves them into x.  A row takes at most two bytes, so
// the window moves up by a word after every second row at the most, by every
// lane at once (no lane waits on another's refill).  The words come from a
// ring of 64 bytes per lane that cp.async keeps ahead: eight rows take at most
// 16 bytes and the window reaches 15 further, so before every eight rows the
// third 16-byte word from the current one is asked for and the one asked for
// eight rows earlier is there.  (A refill from global memory holds up the
// whole warp: 93 us for 0.3M rows, where this takes 46.)  Only words that
// hold stream bytes are asked for (s2 starts on a 16-byte boundary of the blob,
// so they lie inside it); what the ring holds past the stream may enter the
// window, a valid stream never takes it.
// Eight int32 or four int64 rows leave as one 32-byte sector.  Returns true
// if the stream is malformed: it must use exactly its bytes and end at x = L.
// What bounds it: the latency of a row's dependent chain (slot lookup among
// bank conflicts, multiply-add, renormalization), with the 27 warps per SM that
// the streams of 64M rows give and more so with fewer; about 30 instructions a
// row.  Symbols of up to four values found by compares in registers, with a
// 64-bit byte buffer topped up every four rows, took 41 instructions and
// bound the ALU pipe; larger alphabets took a lookup and the same buffer.
// Resident calls of 64M int32 rows in 512-row streams, before and now: 3
// values 157 and 108 us (2.6 TB/s), 16 values 206 and 114, 200 values 231 and
// 137; 4M rows of 3 values 61 and 46.  A window refilled without a branch (the
// ring is then read by every lane) added 5 us.
template <class T, bool WIDE>
__device__ __forceinline__ bool ans_stream(AnsSmem& sm, const uint8_t* s2, uint32_t a0, uint32_t a1, T* dst,
                                           uint32_t n) {
    uint4* ring = sm.ring[threadIdx.x];
    const uint32_t* ring32 = reinterpret_cast<const uint32_t*>(ring);
    const uint32_t end = ((a1 - 1) >> 4) + 1;             // 16-byte words [a0 >> 4, end) hold stream bytes (a1 > a0)
    const uint32_t first = a0 >> 2;
    uint32_t asked = (a0 >> 4) + kRing;                   // 16-byte words asked for (the first by ans_ask)
    __pipeline_wait_prior(0);
    auto load = [&](uint32_t i) { return ring32[i % (4 * kRing)]; };
    uint32_t hi = __byte_perm(load(first), 0, 0x0123), lo = __byte_perm(load(first + 1), 0, 0x0123);
    uint32_t next = first + 2, ahead = load(next);        // the word after the window
    uint32_t used = 8u * (a0 & 3u);                       // bits of the window that have been taken
    auto refill = [&]() {                                 // used < 64 -> used < 32
        if (used >= 32u) {
            hi = lo;
            lo = __byte_perm(ahead, 0, 0x0123);
            next++;
            ahead = load(next);
        }
        used &= 31u;
    };
    // before eight rows: the window's first byte lies in 16-byte word (next - 2) / 4
    auto keep_ahead = [&]() {
        if (asked < ((next - 2u) >> 2) + kRing) {
            if (asked < end) __pipeline_memcpy_async(ring + asked % kRing, s2 + 16ull * asked, 16);
            asked++;
        }
        __pipeline_commit();
        __pipeline_wait_prior(1);
    };
    // the state: the first four bytes, little-endian
    uint32_t x = __byte_perm(__funnelshift_l(lo, hi, used), 0, 0x0123);
    used += 32;
    refill();
    const uint32_t* val32 = reinterpret_cast<const uint32_t*>(sm.val);
    auto step = [&]() -> T {
        const uint32_t t = sm.slot[x & (zf::kAnsM - 1u)], xh = x >> zf::kAnsScale;
        const uint32_t sym = WIDE ? t >> 24 : (t >> 12) & 0x7Fu;
        T v;
        if constexpr (sizeof(T) == 4) v = (T)val32[2 * sym];   // the low word of the 64-bit pattern
        else v = (T)sm.val[sym];
        x = WIDE ? ((t >> 12) & 0xFFFu) * xh + (xh + (t & 0xFFFu)) : (t >> 19) * xh + (t & 0xFFFu);
        const uint32_t s = x < (zf::kAnsL >> 8) ? 16u : x < zf::kAnsL ? 8u : 0u;
        x = __funnelshift_l((uint32_t)(((((uint64_t)hi << 32) | lo) << used) >> 32), x, s);   // used < 48: its next 16 bits
        used += s;
        return v;
    };
    constexpr uint32_t G = 8, V = 32 / sizeof(T);   // rows per step of the ring, rows per store
    const bool al32 = (reinterpret_cast<uintptr_t>(dst) & 31) == 0;
    uint32_t i0 = 0;
    for (; i0 + G <= n; i0 += G) {
        keep_ahead();
#pragma unroll
        for (uint32_t g = 0; g < G; g += V) {
            T v[V];
#pragma unroll
            for (uint32_t e = 0; e < V; e += 2) {
                v[e] = step();
                v[e + 1] = step();
                refill();
            }
            if (al32) {
                if constexpr (sizeof(T) == 4)
                    zfd::store32(dst + i0 + g, ((unsigned long long)(uint32_t)v[1] << 32) | (uint32_t)v[0],
                                 ((unsigned long long)(uint32_t)v[3] << 32) | (uint32_t)v[2],
                                 ((unsigned long long)(uint32_t)v[5] << 32) | (uint32_t)v[4],
                                 ((unsigned long long)(uint32_t)v[7] << 32) | (uint32_t)v[6]);
                else
                    zfd::store32(dst + i0 + g, (uint64_t)v[0], (uint64_t)v[1], (uint64_t)v[2], (uint64_t)v[3]);
            } else {
                zfd::store_vec<T, V>(dst + i0 + g, v);
            }
        }
    }
    keep_ahead();
    for (; i0 < n; i0++) {
        dst[i0] = step();
        refill();
    }
    __pipeline_wait_prior(0);
    const uint32_t taken = 4u * (next - 2u - first) + used / 8u - (a0 & 3u);   // bytes the state and the rows took
    return taken != a1 - a0 || x != zf::kAnsL;
}

// Ask for the first 16-byte words of a lane's stream.
__device__ __forceinline__ void ans_ask(AnsSmem& sm, const uint8_t* s2, uint32_t a0, uint32_t a1) {
    const uint32_t w = a0 >> 4, end = ((a1 - 1) >> 4) + 1;
    for (uint32_t i = w; i < w + kRing; i++)
        if (i < end) __pipeline_memcpy_async(sm.ring[threadIdx.x] + i % kRing, s2 + 16ull * i, 16);
    __pipeline_commit();
}

// Slot entries: warp w fills the ranges of symbols w, w + kWarps, ... (lane l has
// every 32nd of them): a range of up to kShort slots by its lane, a longer one by
// the whole warp, its slots side by side over the lanes.  (A contiguous 32 slots
// per thread, each thread walking its symbols, took 4 to 8 us more of a call of
// few symbols; all ranges by whole warps 4 us more of one of 256.)
template <bool WIDE>
__device__ __forceinline__ void ans_table(AnsSmem& sm, uint32_t nd, uint32_t lane, uint32_t warp) {
    constexpr uint32_t kShort = 16;
    for (uint32_t s0 = warp; s0 < nd; s0 += 32 * kWarps) {
        const uint32_t s = s0 + lane * kWarps;
        const uint32_t c = s < nd ? sm.cum[s] : 0u, f = s < nd ? sm.cum[s + 1] - c : 0u;
        if (f <= kShort)
            for (uint32_t d = 0; d < f; d++) sm.slot[c + d] = ans_entry<WIDE>(s, f, d);
        for (uint32_t m = __ballot_sync(0xFFFFFFFFu, f > kShort); m; m &= m - 1) {
            const uint32_t l = __ffs(m) - 1;
            const uint32_t ck = __shfl_sync(0xFFFFFFFFu, c, l), fk = __shfl_sync(0xFFFFFFFFu, f, l);
            for (uint32_t d = lane; d < fk; d += 32) sm.slot[ck + d] = ans_entry<WIDE>(s0 + l * kWarps, fk, d);
        }
    }
}

// The CTA builds its chunk's tables, then warp w decodes job blockIdx.x *
// kWarps + w: lane i takes the job's stream i.
__global__ void __launch_bounds__(kWarps * 32) ans_kernel(const __grid_constant__ zf::ChunkArgs args, uint32_t njobs,
                                                           uint32_t* err) {
    __shared__ AnsSmem sm;
    const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t job0 = blockIdx.x * kWarps;
    if (job0 >= njobs) return;
    const ZfDevChunk* chunks = args.list();
    uint32_t a = 0, z = args.n;
    while (z - a > 1) {
        const uint32_t mid = (a + z) >> 1;
        if (chunks[mid].tile0 <= job0) a = mid;
        else z = mid;
    }
    const ZfDevChunk c = chunks[a];
    zfd::Hdr h;
    zfd::load_hdr(c.blob, h);
    const uint32_t sz = c.dtype == ZF_I64 ? 8u : 4u;
    const uint32_t lg = c.blob[48], nd = h.n_aux;
    const uint32_t L = 1u << (lg & 31u);
    const uint32_t K = (lg >= zf::kAnsLogMin && lg <= zf::kAnsLogMax) ? (h.rows + L - 1) / L : 0u;
    const uint32_t fb = (2u * nd + 3u) & ~3u;
    // header and section bounds (checked on the host too; the device does not rely on it)
    bool ok = h.rows == c.rows && (uint64_t)c.rows * sz <= c.dst_cap && (c.dtype == ZF_I32 || c.dtype == ZF_I64) &&
              h.b == zf::kAnsScale && nd > 0 && nd <= zf::kAnsMaxSymbols && K > 0 && h.ref == K &&
              h.len[0] == nd * sz && h.len[1] == fb + 4u * (K + 1u);
    for (int s = 0; s < 3; s++)
        ok = ok && h.off[s] >= 64 && !(h.off[s] & 15) && (uint64_t)h.off[s] + h.len[s] <= c.blob_bytes;
    if (!ok) {
        if (tid == 0) zfd::report(err, ZF_ECORRUPT, c.chunk_id);
        return;   // uniform over the CTA
    }
    // one stream per lane; its first bytes are on their way while the tables are built
    const uint32_t job = job0 + warp;
    const uint32_t k = (job - c.tile0) * zf::kAnsStreamsPerJob + lane;
    const uint8_t* s2 = c.blob + h.off[2];
    uint32_t a0 = 0, a1 = 0;
    bool bad = false;
    if (k < K) {
        const uint32_t* starts = reinterpret_cast<const uint32_t*>(c.blob + h.off[1] + fb);
        a0 = __ldg(starts + k);
        a1 = __ldg(starts + k + 1);
        bad = a1 < a0 || a1 - a0 < 4u || a1 > h.len[2];
        if (!bad) ans_ask(sm, s2, a0, a1);
    }
    // frequencies, two per thread, and their exclusive scan over the CTA
    const uint16_t* fq = reinterpret_cast<const uint16_t*>(c.blob + h.off[1]);
    const uint32_t i0 = 2 * tid;
    const uint32_t f0 = i0 < nd ? (uint32_t)__ldg(fq + i0) : 0u, f1 = i0 + 1 < nd ? (uint32_t)__ldg(fq + i0 + 1) : 0u;
    const bool fbad = (i0 < nd && f0 == 0) || (i0 + 1 < nd && f1 == 0);
    const uint32_t pair = f0 + f1;
    const uint32_t incl = zfd::warp_incl_sum<uint32_t>(pair, lane);
    if (lane == 31) sm.wsum[warp] = incl;
    __syncthreads();
    uint32_t before = 0, total = 0;
#pragma unroll
    for (uint32_t q = 0; q < kWarps; q++) {
        before += q < warp ? sm.wsum[q] : 0u;
        total += sm.wsum[q];
    }
    if (__syncthreads_or(fbad) || total != zf::kAnsM) {
        __pipeline_wait_prior(0);
        if (tid == 0) zfd::report(err, ZF_ECORRUPT, c.chunk_id);
        return;
    }
    const uint32_t c0 = before + incl - pair;
    if (i0 < nd) sm.cum[i0] = c0;
    if (i0 + 1 < nd) sm.cum[i0 + 1] = c0 + f0;
    if (tid == 0) sm.cum[nd] = zf::kAnsM;
    for (uint32_t k = tid; k < nd; k += kWarps * 32)
        sm.val[k] = sz == 8 ? (unsigned long long)__ldg(reinterpret_cast<const int64_t*>(c.blob + h.off[0]) + k)
                            : (unsigned long long)(uint32_t)__ldg(reinterpret_cast<const int32_t*>(c.blob + h.off[0]) + k);
    __syncthreads();
    if (nd > 128) ans_table<true>(sm, nd, lane, warp);
    else ans_table<false>(sm, nd, lane, warp);
    __syncthreads();
    if (k < K && !bad) {
        const uint32_t r0 = k * L, n = min(L, h.rows - r0);
        int32_t* d4 = reinterpret_cast<int32_t*>(c.dst) + r0;
        int64_t* d8 = reinterpret_cast<int64_t*>(c.dst) + r0;
        if (sz == 8) bad = nd > 128 ? ans_stream<int64_t, true>(sm, s2, a0, a1, d8, n) : ans_stream<int64_t, false>(sm, s2, a0, a1, d8, n);
        else bad = nd > 128 ? ans_stream<int32_t, true>(sm, s2, a0, a1, d4, n) : ans_stream<int32_t, false>(sm, s2, a0, a1, d4, n);
    }
    if (bad) zfd::report(err, ZF_ECORRUPT, c.chunk_id);
}

}  // namespace

namespace zf {

// njobs is a multiple of kAnsJobsPerCta: every chunk's jobs are padded to it.
cudaError_t launch_ans(const ZfDevChunk* chunks, const ZfDevChunk* host, uint32_t nchunks, uint32_t njobs, uint32_t* err,
                       cudaStream_t s) {
    if (njobs == 0) return cudaSuccess;
    ans_kernel<<<(njobs + kWarps - 1) / kWarps, kWarps * 32, 0, s>>>(ChunkArgs(chunks, host, nchunks), njobs, err);
    return cudaGetLastError();
}

}  // namespace zf

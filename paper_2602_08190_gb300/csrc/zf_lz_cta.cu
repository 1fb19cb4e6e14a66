// zf_lz_cta.cu -- LZ77 decode of launches with few blocks: the 512 threads of
// a CTA share one 64 KiB block, so its decode takes a seventh of the time that
// one warp takes for it (zf_lz.cu, which says where the line lies).
#include <cuda_runtime.h>

#include "zf_device.cuh"
#include "zf_launch.h"
#include "zf_once.h"

namespace {

// One CTA decodes one block, 512 tokens at a time (thread i holds token t0+i),
// into a copy of the block's output in shared memory, so every back-reference
// is a shared-memory read.
//   Lengths: 2,048 bytes of the LEB128 stream per step, four per thread; a CTA
//   scan of the counts of bytes without a continuation bit places the values
//   in a ring in shared memory.
//   Positions: a CTA scan of the lengths gives every token its literal range
//   in s2 and its output range; the whole batch is validated before a byte
//   is written.
//   Segments: the batch's output goes through segments of at most kLzSeg
//   bytes.  Each token sets the bit of its first byte in a mask of the segment,
//   and leaves its index with every 32-byte word of the mask that starts inside
//   it, so a byte finds its token by one popcount.
//   Shortcuts: a match whose source lies inside one earlier match of the
//   segment copies that match's source instead (the offsets add up), again
//   until its source is no match or lies before the segment, a few times at
//   the most: a word's earlier
//   occurrences form chains of 11 copies for the longest of 128 bytes of text,
//   3 after this.
//   Bytes: thread i takes the segment's aligned 4-byte words i, i + 512, ...: a
//   byte is a literal, a byte of the output before the segment (final), or a
//   byte of this segment.  The first two are states with the byte's value, the
//   last a state with the position it copies (a match that overlaps its own
//   output points into its first period).  After one barrier every byte follows
//   its positions until it meets a value: positions only decrease, nothing
//   waits on another thread, and a byte that is done leaves its value for the
//   others.
//   Literals: the next kLzLit bytes of s2 are kept in a ring in shared memory
//   (cp.async, refilled after every batch); a batch with more reads them from
//   global memory.
// What bounds it: the latency of a batch's chain of barriers, scans and
// shared-memory lookups (14 batches of text per block).  Among thousands of
// blocks it is bound by issue slots (64% busy), 229,000 warp instructions per
// block of text: 40% of them to parse, place and store tokens, the rest in
// about equal parts shortcuts with lookups of bytes.  Measured on GB300: 21
// blocks of text (1.3 MB) 82 us per call with its host part, 548 us with one
// warp per block; 1,024 blocks 327 and 652 us.  Shortcuts whose steps were not
// left for other tokens cost 27 us more of them.
constexpr uint32_t kLzThreads = 512;
constexpr uint32_t kLzWarps = kLzThreads / 32;
constexpr uint32_t kLzRing = 4096;             // parsed lengths: at most 1,023 left over and 2,048 more
constexpr uint32_t kLzStep = 4 * kLzThreads;   // bytes of the lengths stream parsed per step
constexpr uint32_t kLzSeg = 8192;              // output bytes of a segment, from its first aligned word
constexpr uint32_t kLzLit = 8192;              // ring of literal bytes
// Shortcut steps of a token.  A match that overlaps its own output (a run) is
// left period by period: without a bound, 512 random bytes and 512 zeros in turn
// took 655 us a block, where the bytes' own way into the run's first period is
// one step.  120 MB of text: 554 us with 4, 579 with 8, 16 or no bound.
constexpr uint32_t kLzShortcuts = 4;
constexpr uint32_t kFull = 0xFFFFFFFFu;
constexpr uint32_t kDone = 0x8000u;            // state of a byte: kDone | value, or the position it copies

struct LzSmem {
    uint2 st[kLzSeg / 4];                 // states of the segment's bytes, four 16-bit states per word
    uint8_t out[zf::kLzBlock];            // the block's output (a lookup may read three bytes on either side)
    uint8_t lit[kLzLit + 16];             // literal byte i of s2 at i mod kLzLit; the first 16 again at the end
    uint2 tok[kLzThreads];                // x = last byte before the match | offset << 16,
                                          // y = output minus literal position | last byte << 16
    uint2 starts[kLzSeg / 32];            // x = token starts in 32 bytes, y = tokens of the batch that start before them
    uint16_t lens[kLzRing];
    uint32_t wl[kLzWarps], wo[kLzWarps], wc[kLzWarps];   // per-warp totals: literals, output, lengths
};

// Sum over the warps before this one, and over all of them, of per-warp totals.
__device__ __forceinline__ void warp_totals(const uint32_t* w, uint32_t lane, uint32_t warp, uint32_t& before,
                                            uint32_t& total) {
    const uint32_t x = lane < kLzWarps ? w[lane] : 0;
    before = __reduce_add_sync(kFull, lane < warp ? x : 0u);
    total = __reduce_add_sync(kFull, x);
}

__device__ __forceinline__ void prefetch_l2(const void* p) {
    asm volatile("prefetch.global.L2 [%0];" ::"l"(p));
}

// Copy n bytes between 16-byte aligned global addresses.
__device__ __forceinline__ void lz_copy(uint8_t* dst, const uint8_t* src, uint32_t n) {
    for (uint32_t i = threadIdx.x; i < (n >> 4); i += kLzThreads)
        reinterpret_cast<uint4*>(dst)[i] = zfd::ldg16(src + 16 * i);
    for (uint32_t i = (n & ~15u) + threadIdx.x; i < n; i += kLzThreads) dst[i] = __ldg(src + i);
}

// Token number + 1 of the byte at `bit` bits into word m of the start mask.
__device__ __forceinline__ uint32_t lz_token(uint2 m, uint32_t bit) { return m.y + __popc(m.x & ((2u << bit) - 1u)); }

// States of the four bytes of word w of the segment (base = output position
// of state 0; only bytes in [s0, s1) belong to the segment).  RING: the
// batch's literals are all in the ring; `lit` is s2 otherwise.
template <bool RING>
__device__ __forceinline__ uint2 lz_lookup(const LzSmem& sm, const uint8_t* __restrict__ lit, uint32_t w,
                                           uint32_t base, uint32_t s0, uint32_t s1) {
    const uint2 m = sm.starts[w >> 3];
    const uint32_t bit = (w & 7u) * 4u, j0 = base + 4 * w;
    // the token of byte 0; a token has at least four bytes (the block's last
    // one apart), so one more at most starts in bytes 1..3
    const uint32_t n = lz_token(m, bit);
    const uint32_t nib = (m.x >> bit) & 0xEu;
    const uint32_t pb = nib ? __ffs(nib) - 1 : 4u;
    const uint2 ta = sm.tok[n ? n - 1 : 0];
    const uint2 tb = nib ? sm.tok[n] : ta;
    uint32_t v[4];
    if constexpr (RING) {
        // per token: the byte 0 of the word as a literal and as a copy, one address each
        constexpr uint32_t OUT = offsetof(LzSmem, out), LIT = offsetof(LzSmem, lit);
        const uint8_t* smb = reinterpret_cast<const uint8_t*>(&sm);
        const uint32_t la = ta.x & 0xFFFFu, lb = tb.x & 0xFFFFu, oa = ta.x >> 16, ob = tb.x >> 16;
        const int ma = (int)(j0 - oa), mb = (int)(j0 - ob);   // -3 or more where a byte of the segment copies from them
        const uint32_t ka = LIT + ((j0 - (ta.y & 0xFFFFu)) & (kLzLit - 1)), kb = LIT + ((j0 - (tb.y & 0xFFFFu)) & (kLzLit - 1));
        bool over = false;   // a byte that copies its own match's output
#pragma unroll
        for (uint32_t b = 0; b < 4; b++) {
            const bool second = b >= pb;
            const uint32_t last = second ? lb : la, k = second ? kb : ka;
            const int m = second ? mb : ma;
            const bool is_lit = j0 + b <= last, here = !is_lit && m + (int)b >= (int)s0;
            over |= !is_lit && m + (int)b > (int)last;
            const uint32_t x = smb[(is_lit ? k : OUT + (uint32_t)max(m, -3)) + b];
            v[b] = here ? (uint32_t)m + b - base : kDone | x;
        }
        if (over) {
            uint32_t rem = j0 > la ? (j0 - la - 1) % oa : 0u;   // byte 0's place in the match's period; the next ones' follow
#pragma unroll
            for (uint32_t b = 0; b < 4; b++) {
                const bool second = b >= pb;
                const uint32_t last = second ? lb : la, off = second ? ob : oa, j = j0 + b;
                if (b == pb) rem = 0;
                if (j <= last) continue;
                const uint32_t src = last + 1 - off + rem;
                rem = rem + 1 == off ? 0 : rem + 1;
                if (j >= s0 && j < s1) v[b] = src >= s0 ? src - base : kDone | sm.out[src];
            }
        }
        if (j0 < s0 || j0 + 4 > s1) {   // bytes outside the segment: nothing copies them
#pragma unroll
            for (uint32_t b = 0; b < 4; b++)
                if (j0 + b < s0 || j0 + b >= s1) v[b] = kDone;
        }
    } else {
#pragma unroll
        for (uint32_t b = 0; b < 4; b++) {
            const uint32_t j = j0 + b;
            const uint2 t = b >= pb ? tb : ta;
            const uint32_t last = t.x & 0xFFFFu, off = t.x >> 16;
            v[b] = kDone;
            if (j < s0 || j >= s1) continue;
            if (j <= last) {
                v[b] = kDone | __ldg(lit + (j - (t.y & 0xFFFFu)));
            } else {
                uint32_t src = j - off;
                if (src > last) src = last + 1 - off + (j - last - 1) % off;
                v[b] = src >= s0 ? src - base : kDone | sm.out[src];
            }
        }
    }
    return make_uint2(v[0] | (v[1] << 16), v[2] | (v[3] << 16));
}

// Keep literals [from, from + kLzLit) of the l2 bytes at `lit` in the ring:
// asks for the 16-byte words from `have` on and returns the new `have`.
__device__ __forceinline__ uint32_t lz_fill(LzSmem& sm, const uint8_t* lit, uint32_t l2, uint32_t from, uint32_t have) {
    const uint32_t to = min((l2 + 15) & ~15u, (from & ~15u) + kLzLit);
    for (uint32_t i = have + 16 * threadIdx.x; i < to; i += 16 * kLzThreads) {
        __pipeline_memcpy_async(sm.lit + (i & (kLzLit - 1)), lit + i, 16);
        if ((i & (kLzLit - 1)) == 0) __pipeline_memcpy_async(sm.lit + kLzLit, lit + i, 16);
    }
    __pipeline_commit();
    return max(have, to);
}

__device__ void lz_block(const ZfDevChunk& c, LzSmem& sm, uint32_t* err) {
    const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    zfd::Hdr h;
    zfd::load_hdr(c.blob, h);
    uint8_t* dst = c.dst;
    if (h.rows != c.rows || h.rows > zf::kLzBlock || h.rows > c.dst_cap) {
        if (tid == 0) zfd::report(err, ZF_ECORRUPT, c.chunk_id);
        return;
    }
    const uint8_t* s0p = c.blob + h.off[0];
    if (h.flags & 1) {  // stored raw
        lz_copy(dst, s0p, h.rows);
        return;
    }
    const uint16_t* offs = reinterpret_cast<const uint16_t*>(c.blob + h.off[1]);
    const uint8_t* lit = c.blob + h.off[2];
    const uint32_t T = h.n_aux, l0 = h.len[0], l2 = h.len[2], rows = h.rows;
    bool ok = T > 0 && h.len[1] == 2 * (T - 1) && l0 > 0;
    if (ok) ok = !(__ldg(s0p + l0 - 1) & 0x80u);             // no varint is left open
    if (ok && T == 1) {
        // literals alone: the one length is the only one that may be 2^16 (the ring holds 16 bits)
        uint32_t v = 0;
        ok = l0 <= 3;
        for (uint32_t i = 0; ok && i < l0; i++) {
            const uint32_t b = __ldg(s0p + i);
            ok = i + 1 == l0 || (b & 0x80u);                 // one varint
            v |= (b & 0x7Fu) << (7 * i);
        }
        ok = ok && v == rows && l2 == rows;
        if (ok) {
            lz_copy(dst, lit, rows);
            return;
        }
    }
    if (!ok) {
        if (tid == 0) zfd::report(err, ZF_ECORRUPT, c.chunk_id);
        return;
    }
    const uint32_t nlen = 2 * T - 1;                         // lengths in the stream
    // the streams are read once, front to back: start them towards L2
    for (uint32_t i = 128 * tid; i < l0; i += 128 * kLzThreads) prefetch_l2(s0p + i);
    for (uint32_t i = 128 * tid; i < h.len[1]; i += 128 * kLzThreads) prefetch_l2(c.blob + h.off[1] + i);
    for (uint32_t i = 128 * tid; i < l2; i += 128 * kLzThreads) prefetch_l2(lit + i);
    uint32_t have = lz_fill(sm, lit, l2, 0, 0);              // literals asked for
    if (tid < kLzSeg / 32) sm.starts[tid].x = 0;
    uint32_t vp = 0, parsed = 0;                             // lengths stream: bytes taken, lengths parsed
    uint32_t lp = 0, op = 0;                                 // literal and output bytes done
    bool bad = false;                                        // a varint of more than three bytes, an offset out of range
    const uint32_t* w0 = reinterpret_cast<const uint32_t*>(s0p);
    uint32_t word = 4 * tid < l0 ? __ldg(w0 + tid) : 0;      // the next step's bytes, loaded a step ahead
    uint32_t prev = tid && 4 * tid < l0 ? __ldg(w0 + tid - 1) : 0;
    uint32_t off_next = tid + 1 < T ? __ldg(offs + tid) : 0; // offsets are loaded a batch ahead
    for (uint32_t t0 = 0; t0 < T; t0 += kLzThreads) {
        const uint32_t need = min(nlen, 2 * (t0 + kLzThreads));
        while (parsed < need && vp < l0) {
            const uint32_t pos = vp + 4 * tid;
            const uint32_t nv = pos < l0 ? min(4u, l0 - pos) : 0u;
            const uint32_t ends = ~word & 0x80808080u & (nv == 4 ? kFull : (1u << (8 * nv)) - 1u);
            const uint32_t cnt = __popc(ends);
            const uint32_t incl = zfd::warp_incl_sum<uint32_t>(cnt, lane);
            if (lane == 31) sm.wc[warp] = incl;
            __syncthreads();
            uint32_t before, total;
            warp_totals(sm.wc, lane, warp, before, total);
            uint32_t i = parsed + before + incl - cnt;
#pragma unroll
            for (uint32_t e = 0; e < 4; e++) {
                if ((ends >> (8 * e + 7)) & 1u) {
                    // the end byte on top, the three bytes before it below
                    const uint32_t x = e == 3 ? word : __funnelshift_r(prev, word, 8 * (e + 1));
                    const uint32_t b0 = x >> 24, b1 = (x >> 16) & 0x7Fu, b2 = (x >> 8) & 0x7Fu;
                    const bool c1 = (x >> 23) & 1u, c2 = c1 && ((x >> 15) & 1u);
                    const uint32_t v = c2 ? b2 | (b1 << 7) | (b0 << 14) : c1 ? b1 | (b0 << 7) : b0;
                    bad |= c2 && ((x >> 7) & 1u);
                    sm.lens[i & (kLzRing - 1)] = (uint16_t)min(v, 0xFFFFu);   // 2^16 - 1 fits no block of two tokens
                    i++;
                }
            }
            parsed += total;
            vp += kLzStep;
            word = vp + 4 * tid < l0 ? __ldg(w0 + (vp >> 2) + tid) : 0;
            prev = vp + 4 * tid < l0 ? __ldg(w0 + (vp >> 2) + tid - 1) : 0;
            __syncthreads();
        }
        if (parsed < need) { ok = false; break; }
        // token t0 + tid: lengths, literal and output positions
        const uint32_t t = t0 + tid;
        const bool in = t < T, has_m = t + 1 < T;
        const uint32_t pair = in ? *reinterpret_cast<const uint32_t*>(&sm.lens[(2 * t) & (kLzRing - 1)]) : 0;
        const uint32_t ll = pair & 0xFFFFu, ml = has_m ? (pair >> 16) + zf::kLzMinMatch : 0;
        const uint32_t off = has_m ? off_next : 0;
        off_next = t + kLzThreads + 1 < T ? __ldg(offs + t + kLzThreads) : 0;
        uint32_t lend, oend;                                 // inclusive sums over the lanes
        if (!__any_sync(kFull, ll + ml >= 2048u)) {          // both below 2^16: one scan
            const uint32_t both = zfd::warp_incl_sum<uint32_t>(ll | ((ll + ml) << 16), lane);
            lend = both & 0xFFFFu;
            oend = both >> 16;
        } else {                                             // at most 512 * 2^17 over the CTA: no sum wraps
            lend = zfd::warp_incl_sum<uint32_t>(ll, lane);
            oend = zfd::warp_incl_sum<uint32_t>(ll + ml, lane);
        }
        if (lane == 31) {
            sm.wl[warp] = lend;
            sm.wo[warp] = oend;
        }
        __syncthreads();
        uint32_t lbefore, lb, obefore, ob;
        warp_totals(sm.wl, lane, warp, lbefore, lb);
        warp_totals(sm.wo, lane, warp, obefore, ob);
        if (lp + lb > l2 || op + ob > rows) { ok = false; break; }
        lend += lp + lbefore;
        oend += op + obefore;
        const uint32_t ostart = oend - ml - ll, mpos = oend - ml, op_end = op + ob;
        bad |= has_m && (off == 0 || off > mpos);
        const uint32_t tx = has_m ? (mpos - 1) | (off << 16) : 0xFFFFu;
        if (in) sm.tok[tid] = make_uint2(tx, (ostart - (lend - ll)) | ((oend - 1) << 16));
        const bool ring = lp + lb <= have;
        for (uint32_t s0 = op;;) {
            const uint32_t base = s0 & ~3u, s1 = min(op_end, base + kLzSeg);
            const uint32_t nm = (s1 - base + 31) >> 5;       // words of the start mask
            if (in) {
                if (ostart >= s0 && ostart < s1) atomicOr(&sm.starts[(ostart - base) >> 5].x, 1u << ((ostart - base) & 31u));
                // mask words that start after this token does and no later than the next one
                uint32_t q = ostart >= base ? ((ostart - base) >> 5) + 1 : 0;
                const uint32_t q1 = oend >= base ? min(((oend - base) >> 5) + 1, nm) : 0;
                for (; q < q1; q++) sm.starts[q].y = tid + 1;
                if (tid == 0 && ostart >= base) sm.starts[0].y = 0;
            }
            if (__syncthreads_or(bad)) { ok = false; break; }
            if (has_m && mpos < s1 && oend > s0) {
                // the source lies inside one match of this segment: copy what that match copies; every step is
                // left for the tokens that look here, so a chain of n matches takes about log2 n steps, and what is
                // left of it the bytes follow by themselves
                uint32_t o = off;
#pragma unroll 1
                for (uint32_t step = 0; step < kLzShortcuts; step++) {
                    const uint32_t src = mpos - o;
                    if (src < s0 || o < ml) break;
                    const uint32_t n = lz_token(sm.starts[(src - base) >> 5], (src - base) & 31u);
                    const uint2* u = &sm.tok[n ? n - 1 : 0];
                    const uint32_t ux = *const_cast<const volatile uint32_t*>(&u->x);   // its owner may shorten it meanwhile
                    if (src <= (ux & 0xFFFFu) || src + ml - 1 > (u->y >> 16)) break;
                    o += ux >> 16;
                    *reinterpret_cast<volatile uint32_t*>(&sm.tok[tid].x) = (mpos - 1) | (o << 16);
                }
            }
            __pipeline_wait_prior(0);
            __syncthreads();
            const uint32_t nw = (s1 - base + 3) >> 2;
            if (ring) {
#pragma unroll 2
                for (uint32_t w = tid; w < nw; w += kLzThreads) sm.st[w] = lz_lookup<true>(sm, lit, w, base, s0, s1);
            } else {
                for (uint32_t w = tid; w < nw; w += kLzThreads) sm.st[w] = lz_lookup<false>(sm, lit, w, base, s0, s1);
            }
            __syncthreads();
            for (uint32_t w = tid; w < nw; w += kLzThreads) {
                uint2 s = sm.st[w];
                if ((s.x & s.y & 0x80008000u) != 0x80008000u) {
                    const volatile uint16_t* st = reinterpret_cast<const volatile uint16_t*>(sm.st);
                    uint32_t v0 = s.x & 0xFFFFu, v1 = s.x >> 16, v2 = s.y & 0xFFFFu, v3 = s.y >> 16;
                    do {
                        if (!(v0 & kDone)) v0 = st[v0];
                        if (!(v1 & kDone)) v1 = st[v1];
                        if (!(v2 & kDone)) v2 = st[v2];
                        if (!(v3 & kDone)) v3 = st[v3];
                    } while (!(v0 & v1 & v2 & v3 & kDone));
                    s = make_uint2(v0 | (v1 << 16), v2 | (v3 << 16));
                    *reinterpret_cast<volatile uint32_t*>(&sm.st[w].x) = s.x;
                    *reinterpret_cast<volatile uint32_t*>(&sm.st[w].y) = s.y;
                }
                const uint32_t x = __byte_perm(s.x, s.y, 0x6420), j = base + 4 * w;
                if (j >= s0 && j + 4 <= s1) {
                    *reinterpret_cast<uint32_t*>(sm.out + j) = x;
                } else {
#pragma unroll
                    for (uint32_t b = 0; b < 4; b++)
                        if (j + b >= s0 && j + b < s1) sm.out[j + b] = (uint8_t)(x >> (8 * b));
                }
            }
            if (tid < kLzSeg / 32) sm.starts[tid].x = 0;
            __syncthreads();
            // the output's whole 16-byte words that are now final
            const uint32_t f1 = (s1 == rows ? s1 + 15 : s1) >> 4;
            for (uint32_t q = (s0 >> 4) + tid; q < f1; q += kLzThreads) {
                if (16 * q + 16 <= rows) {
                    reinterpret_cast<uint4*>(dst)[q] = *reinterpret_cast<const uint4*>(sm.out + 16 * q);
                } else {
                    for (uint32_t i = 16 * q; i < rows; i++) dst[i] = sm.out[i];
                }
            }
            s0 = s1;
            if (s0 >= op_end) break;
        }
        if (!ok) break;
        lp += lb;
        op = op_end;
        have = lz_fill(sm, lit, l2, lp, max(have, lp & ~15u));
    }
    // every length used, every literal and output byte accounted for
    ok = ok && parsed == nlen && vp >= l0 && op == rows && lp == l2;
    if (__syncthreads_or(bad || !ok) && tid == 0) zfd::report(err, ZF_ECORRUPT, c.chunk_id);
}

__global__ void __launch_bounds__(kLzThreads, 2) lz_cta_kernel(const __grid_constant__ zf::ChunkArgs chunks,
                                                               uint32_t* err) {
    extern __shared__ uint4 smem4[];
    const ZfDevChunk c = chunks.list()[blockIdx.x];
    lz_block(c, *reinterpret_cast<LzSmem*>(smem4), err);
}

zf::OncePerDevice g_smem_allowed;

}  // namespace

namespace zf {

cudaError_t launch_lz_cta(const ChunkArgs& chunks, uint32_t* err, cudaStream_t s) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    e = g_smem_allowed(dev, (const void*)lz_cta_kernel, [] {
        return cudaFuncSetAttribute(lz_cta_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(LzSmem));
    });
    if (e != cudaSuccess) return e;
    lz_cta_kernel<<<chunks.n, kLzThreads, sizeof(LzSmem), s>>>(chunks, err);
    return cudaGetLastError();
}

}  // namespace zf

// zf_strdict_sm.cu -- string-dictionary decode with the chunk's dictionary in
// shared memory (zf_strdict.cuh reads dictionaries that do not fit there).
//
// One CTA of 32 warps per SM takes a contiguous range of the launch's
// 1024-token tiles.  For every chunk in its range the CTA lays the dictionary
// out anew: each entry starts at a word boundary and is padded with zeros to
// whole words, and a table word per entry holds its first word and its length.
// A warp then decodes a tile 64 tokens at a time, two adjacent tokens per lane:
// the codes (loaded a batch ahead) give two table words, one scan of the
// lengths places the tokens, and every entry is ORed into a zeroed window of
// the output, a word at a time: the padding is zero, so a destination word is
// one funnel shift of two entry words, with no mask and no second offset.  The
// window's whole 16-byte blocks are stored and zeroed behind.
// What bounds it: issue slots (71% busy) and shared-memory accesses.  Measured
// on GB300, resident calls of text from a 5,000-word vocabulary in 8 MB chunks
// (the int32 row offsets included), with the dictionary read through L1 and
// now: 256 MB 374 and 222 us (1.5 TB/s), 64 MB 146 and 104, 8 MB 86 and 54.
#include <cuda_runtime.h>

#include "zf_decode.cuh"
#include "zf_launch.h"
#include "zf_once.h"

namespace {

constexpr uint32_t kThreads = 1024, kWarps = kThreads / 32;
constexpr uint32_t kWin = zfd::kStrWin / 4;    // words of a warp's output window
constexpr uint32_t kFull = 0xFFFFFFFFu;

struct Args {
    zf::ChunkArgs chunks;   // tile0, ntiles: tiles of 1024 tokens
    uint32_t ntiles;        // of the launch
    uint32_t dict_bytes;    // shared memory for a chunk's table and entries
    uint32_t* err;
};

// OR an entry of `len` bytes, word-aligned and zero-padded at `e`, into byte w0 of the window.
__device__ __forceinline__ void put(uint32_t* win, const uint32_t* e, uint32_t len, uint32_t w0) {
    const uint32_t sh = 8u * (w0 & 3u), ns = (len + 3) >> 2;       // words of the entry
    const uint32_t nd = ((w0 & 3u) + len + 3) >> 2;                // words it touches, ns or ns + 1 (0 for no entry)
    uint32_t* q = win + (w0 >> 2);
    uint32_t prev = 0;
    for (uint32_t j0 = 0; j0 < nd; j0 += 4) {
        uint32_t s[4];
#pragma unroll
        for (uint32_t j = 0; j < 4; j++) s[j] = j0 + j < ns ? e[j0 + j] : 0u;
#pragma unroll
        for (uint32_t j = 0; j < 4; j++) {
            if (j0 + j < nd) atomicOr(q + j0 + j, __funnelshift_l(prev, s[j], sh));
            prev = s[j];
        }
    }
}

// Lay the chunk's dictionary out in shared memory: table[k] = first word |
// length << 16 (length 0: not a valid entry), entries from `ent` on.  False
// if it does not fit `bytes`.  Ends with the CTA's threads in step.
__device__ bool load_dictionary(const ZfDevChunk& c, const zfd::Hdr& h, uint32_t* table, uint32_t bytes,
                                uint32_t* s_sum) {
    const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t nd = h.n_aux, dlen = h.len[1];
    const uint32_t* doff = reinterpret_cast<const uint32_t*>(c.blob + h.off[0]);
    const uint32_t* dw = reinterpret_cast<const uint32_t*>(c.blob + h.off[1]);
    const uint32_t per = (nd + kThreads - 1) / kThreads, k0 = min(nd, tid * per), k1 = min(nd, k0 + per);
    auto length = [&](uint32_t a, uint32_t z) { return z - a - 1u < zf::kStrTokenMax && z <= dlen ? z - a : 0u; };
    uint32_t words = 0;
    for (uint32_t k = k0, a = __ldg(doff + k0); k < k1; k++) {
        const uint32_t z = __ldg(doff + k + 1);
        words += (length(a, z) + 3) >> 2;
        a = z;
    }
    const uint32_t incl = zfd::warp_incl_sum<uint32_t>(words, lane);
    if (lane == 31) s_sum[warp] = incl;
    __syncthreads();
    const uint32_t ws = s_sum[lane], wi = zfd::warp_incl_sum<uint32_t>(ws, lane);
    const uint32_t before = __shfl_sync(kFull, wi - ws, warp), total = __shfl_sync(kFull, wi, 31);
    if (4ull * nd + 4ull * total > bytes || total > 0xFFFFu) return false;
    uint32_t* ent = table + nd;
    uint32_t at = before + incl - words;
    const uint32_t last = (dlen - 1) >> 2;
    for (uint32_t k = k0, a = __ldg(doff + k0); k < k1; k++) {
        const uint32_t z = __ldg(doff + k + 1), len = length(a, z), ns = (len + 3) >> 2, sh = 8u * (a & 3u);
        table[k] = at | (len << 16);
        uint32_t lo = ns ? __ldg(dw + (a >> 2)) : 0u;
        for (uint32_t j = 0; j < ns; j++) {
            const uint32_t hi = __ldg(dw + min((a >> 2) + j + 1, last));
            uint32_t x = __funnelshift_r(lo, hi, sh);
            if (j + 1 == ns) x &= 0xFFFFFFFFu >> (8u * (4u * ns - len));
            ent[at + j] = x;
            lo = hi;
        }
        at += ns;
        a = z;
    }
    __syncthreads();
    return true;
}

// One tile of up to 1024 tokens by one warp; false if the stream is malformed.
__device__ __forceinline__ bool tile_tokens(const ZfDevChunk& c, const zfd::Hdr& h, const uint32_t* table, uint32_t tile,
                                            uint32_t ntiles, uint32_t* win) {
    const uint32_t lane = threadIdx.x & 31;
    const uint32_t nd = h.n_aux, b = h.b, cmask = (1u << b) - 1u;   // b <= 16
    const uint32_t nt = (uint32_t)min((unsigned long long)zf::kStrTile, (unsigned long long)(h.ref - (uint64_t)tile * zf::kStrTile));
    const uint32_t* ent = table + nd;
    const uint32_t* tstart = reinterpret_cast<const uint32_t*>(c.blob + h.off[0]) + nd + 1;
    // the tile's codes start at bit tile * 1024 * b, a word boundary
    const uint32_t* cw = reinterpret_cast<const uint32_t*>(c.blob + h.off[2]) + (uint64_t)tile * 32u * b;
    const uint32_t last_w = b ? (nt * b + 31) / 32 - 1 : 0;
    const uint8_t* winb = reinterpret_cast<const uint8_t*>(win);
    __syncwarp();   // the warp's tile before may still be reading its last block there
    for (uint32_t w = lane; w < kWin; w += 32) win[w] = 0;
    uint32_t op = __ldg(tstart + tile);
    const uint32_t o1 = tile + 1 < ntiles ? __ldg(tstart + tile + 1) : h.rows;
    if (op > o1 || o1 > h.rows) return false;
    uint32_t a = op & 15u, head = a;           // window byte a holds output byte op; bytes before it are not this tile's
    uint8_t* base = c.dst + (op - a);          // output address of window byte 0 (16-byte aligned)
    __syncwarp();
    // the two code words of the lane's tokens k and k + 1
    auto codes = [&](uint32_t k, uint32_t& w0, uint32_t& w1) {
        const uint32_t w = (k * b) >> 5;
        w0 = k < nt && b ? __ldg(cw + w) : 0u;
        w1 = k < nt && b ? __ldg(cw + min(w + 1, last_w)) : 0u;
    };
    uint32_t n0, n1;
    codes(2 * lane, n0, n1);
    for (uint32_t t = 0; t < nt; t += 64) {
        const uint32_t k = t + 2 * lane;
        const uint32_t pair = __funnelshift_r(n0, n1, (k * b) & 31u);
        codes(k + 64, n0, n1);
        const uint32_t c0 = pair & cmask, c1 = (pair >> b) & cmask;
        const uint32_t e0 = k < nt && c0 < nd ? table[c0] : 0u, e1 = k + 1 < nt && c1 < nd ? table[c1] : 0u;
        const uint32_t len0 = e0 >> 16, len1 = e1 >> 16, s2 = len0 + len1;
        const bool lbad = (k < nt && !len0) || (k + 1 < nt && !len1);
        const uint32_t incl = zfd::warp_incl_sum<uint32_t>(s2, lane);
        const uint32_t total = __shfl_sync(kFull, incl, 31), start = incl - s2;
        if (__any_sync(kFull, lbad) || total > o1 - op) return false;
        // the batch's bytes go through the window in one round, or, when they
        // would not fit, in two or four rounds of consecutive lanes (a round
        // of eight lanes, 16 tokens of at most 64 bytes, always fits)
        const uint32_t half = __shfl_sync(kFull, incl, 15);
        const uint32_t R = a + total + 16u <= zfd::kStrWin ? 1u : max(half, total - half) + 31u <= zfd::kStrWin ? 2u : 4u;
        const uint32_t per = 32u / R;
        for (uint32_t r = 0; r < R; r++) {
            const uint32_t l0 = r * per;
            const uint32_t before = l0 ? __shfl_sync(kFull, incl, l0 - 1) : 0u;
            const uint32_t rtot = __shfl_sync(kFull, incl, l0 + per - 1) - before;
            if (lane - l0 < per) {
                put(win, ent + (e0 & 0xFFFFu), len0, a + start - before);
                put(win, ent + (e1 & 0xFFFFu), len1, a + start - before + len0);
            }
            __syncwarp();
            // whole blocks out (zeroed behind), block 0 keeping its leading bytes that are not this tile's
            const uint32_t e = a + rtot, x1 = e & ~15u;
            if (x1) {
                if (head) {
                    if (lane >= head && lane < 16) base[lane] = winb[lane];
                    __syncwarp();
                    if (lane < 4) win[lane] = 0;
                }
                uint4* wv = reinterpret_cast<uint4*>(win);
                for (uint32_t q = (head ? 1u : 0u) + lane; q < (x1 >> 4); q += 32) {
                    reinterpret_cast<uint4*>(base)[q] = wv[q];
                    wv[q] = make_uint4(0, 0, 0, 0);
                }
                head = 0;
                __syncwarp();
                // the partial block [x1, e) becomes block 0 (its old place is zeroed)
                if (x1 < e && lane < 4) {
                    win[lane] = win[(x1 >> 2) + lane];
                    win[(x1 >> 2) + lane] = 0;
                }
                __syncwarp();
            }
            base += x1;
            a = e - x1;
        }
        op += total;
    }
    if (op != o1) return false;
    // the tile's last partial block, byte by byte
    if (lane >= head && lane < a) base[lane] = winb[lane];
    return true;
}

__global__ void __launch_bounds__(kThreads, 1) strdict_kernel(const __grid_constant__ Args args) {
    extern __shared__ uint4 smem4[];
    __shared__ uint32_t s_sum[kWarps];
    const uint32_t warp = threadIdx.x >> 5;
    uint32_t* win = reinterpret_cast<uint32_t*>(smem4) + warp * kWin;
    uint32_t* table = reinterpret_cast<uint32_t*>(smem4) + kWarps * kWin;
    const ZfDevChunk* chunks = args.chunks.list();
    uint32_t t = (uint32_t)((uint64_t)args.ntiles * blockIdx.x / gridDim.x);
    const uint32_t end = (uint32_t)((uint64_t)args.ntiles * (blockIdx.x + 1) / gridDim.x);
    uint32_t k = 0, z = args.chunks.n;   // the chunk holding tile t
    while (z - k > 1) {
        const uint32_t mid = (k + z) >> 1;
        if (chunks[mid].tile0 <= t) k = mid;
        else z = mid;
    }
    for (; t < end; k++) {
        const ZfDevChunk c = chunks[k];
        zfd::Hdr h;
        zfd::load_hdr(c.blob, h);
        const uint32_t stop = min(end, c.tile0 + c.ntiles);
        const uint64_t T = h.ref;
        const uint32_t ntiles = (uint32_t)((T + zf::kStrTile - 1) / zf::kStrTile);
        bool ok = h.rows == c.rows && (uint64_t)c.rows <= c.dst_cap && h.n_aux && h.n_aux <= zf::kStrDictMax && h.b <= 16 &&
                  T <= h.rows && ntiles == c.ntiles && (uint64_t)h.len[0] >= 4ull * (h.n_aux + 1 + (uint64_t)ntiles) &&
                  h.len[1];
        ok = ok && load_dictionary(c, h, table, args.dict_bytes, s_sum);
        if (ok) {
            for (uint32_t i = t + warp; i < stop; i += kWarps)
                if (!tile_tokens(c, h, table, i - c.tile0, ntiles, win) && (threadIdx.x & 31) == 0)
                    zfd::report(args.err, ZF_ECORRUPT, c.chunk_id);
        } else if (threadIdx.x == 0) {
            zfd::report(args.err, ZF_ECORRUPT, c.chunk_id);
        }
        __syncthreads();   // the next chunk's dictionary takes this one's place
        t = stop;
    }
}

zf::OncePerDevice g_smem_allowed;

}  // namespace

namespace zf {

uint32_t strdict_smem_limit() { return 227u * 1024u - 1024u - kWarps * kWin * 4u; }

cudaError_t launch_strdict(const ZfDevChunk* chunks, const ZfDevChunk* host, uint32_t nchunks, uint32_t ntiles,
                           uint32_t dict_bytes, uint32_t* err, int num_sms, cudaStream_t s) {
    if (ntiles == 0) return cudaSuccess;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    e = g_smem_allowed(dev, (const void*)strdict_kernel, [] {
        return cudaFuncSetAttribute(strdict_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    (int)(kWarps * kWin * 4u + strdict_smem_limit()));
    });
    if (e != cudaSuccess) return e;
    const uint32_t grid = ntiles < (uint32_t)num_sms ? ntiles : (uint32_t)num_sms;
    strdict_kernel<<<grid, kThreads, kWarps * kWin * 4u + ((dict_bytes + 15u) & ~15u), s>>>(
        Args{ChunkArgs(chunks, host, nchunks), ntiles, (dict_bytes + 15u) & ~15u, err});
    return cudaGetLastError();
}

}  // namespace zf

// zf_noalloc.cu -- zf_decompress_device_noalloc: decode a compressed integer
// or float64 column that is already in device memory without allocating
// anything.
//
// Who needs it: code that must not call cudaMalloc (or any allocator) after
// start-up -- for example a query engine that reserved all device memory up
// front, a process whose memory budget is fixed by another runtime, or code
// running inside a library call that may not grow the device heap.  Such a
// caller passes its own input and output buffers; the only other memory the
// decode needs (the result words the host reads) lives in the fixed-size
// device array below, which every GPU that loads the library holds until the
// process exits.
//
// Calls are numbered; call n uses result word n mod kSlots and writes it only
// to report an error, as its number and the status.  Nothing is cleared
// between calls: a word that names another call says nothing about this one,
// whatever that call did, so calls may overlap (kSlots of them, before two
// that fail could share a word).
//
// Two launches, one wait by the host: noalloc_check looks the whole column
// over, noalloc_decode decodes it if nothing was found.  In both every warp
// reads the column header and finds its chunk by division (all chunks but the
// last have chunk_rows rows).  A header read by the host, a set-up kernel of
// one CTA for the chunk descriptors (whose threads each walked a chunk's
// delta entries) and a persistent decode launch took 46.3 us for 3M rows of
// RLE and 220 us for 1M rows of delta in one chunk; this takes 28 us for
// either, most of it the host's wait.  (One launch, in which a warp checked
// only what it was about to decode, took 27 and 26.5 us, but had decoded
// other chunks when one was found malformed.)  33M rows of Float2Int in
// 65,536-row chunks took 317 us and take 102 us: about 25 us of launches and
// wait, as for the smallest column, then 4.7 TB/s.
#include <cuda_runtime.h>

#include <algorithm>
#include <mutex>

#include "zf_decode.cuh"

namespace {

constexpr uint32_t kNoallocMaxChunks = 4096;
constexpr uint32_t kWarps = 4;                // warps per CTA
// Seven CTAs fit an SM beside one another (29 KB of shared memory each); the
// eighth of a full grid starts as one of them ends.  A grid of seven (33M wide
// differences 3% faster, 33M narrow FOR 4% slower) and eight of 27,632 bytes
// that do fit (the wide differences 5% slower) measured the same elsewhere.
constexpr uint32_t kCtasPerSm = 8;
constexpr uint32_t kSmem = 28 * 1024;         // a CTA's staging memory: four warps of up to 7 KB, fewer at a time of more
constexpr uint32_t kJobTiles = 4;             // 1024-row tiles of a job at most
constexpr int kMaxDevices = 64;
constexpr uint32_t kSlots = 64;
constexpr uint32_t kRefused = 0x80;           // beside the status in a result word: nothing is decoded
constexpr uint32_t kCheckTiles = 32;          // 1024-row tiles of a checking job: an entry of a delta block per lane

// Result words: number << 8 | status of the last call that failed with it.
static __device__ unsigned long long g_noalloc_slots[kSlots];

std::mutex g_mu;
struct Device {
    unsigned long long* slots = nullptr;   // device address of g_noalloc_slots (set once)
    int sms = 0;
    uint64_t calls = 0;                    // so far
} g_dev[kMaxDevices];

struct Column {
    uint32_t scheme, dtype, nch, chunk_rows, size;   // size: bytes of a value
    uint64_t n_rows, total;
};

// The column header's fields and what the call returns for them.
__device__ zf_status read_column(const uint8_t* col, uint64_t col_bytes, uint64_t out_bytes, Column& c) {
    const uint4 a = zfd::ldg16(col), b = zfd::ldg16(col + 16);
    const uint2 t = __ldg(reinterpret_cast<const uint2*>(col + 32));
    c.scheme = (a.y >> 16) & 0xFFu;
    c.dtype = a.y >> 24;
    c.nch = a.z;
    c.chunk_rows = a.w;
    c.n_rows = ((uint64_t)b.y << 32) | b.x;
    c.total = ((uint64_t)t.y << 32) | t.x;
    c.size = c.dtype == ZF_I32 ? 4 : 8;
    if (a.x != zf::kColMagic || (a.y & 0xFFFFu) != 1) return ZF_ECORRUPT;
    if (c.dtype != ZF_I32 && c.dtype != ZF_I64 && c.dtype != ZF_F64) return ZF_EUNSUPPORTED;
    if (c.scheme == ZF_ANS) return ZF_EUNSUPPORTED;   // decoded by its own kernel on the regular paths
    const bool scheme_ok = c.dtype == ZF_F64 ? (c.scheme == ZF_RAW || c.scheme == ZF_FLOAT2INT) : c.scheme <= ZF_RLE;
    if (!scheme_ok || c.chunk_rows == 0 || c.chunk_rows % 1024 || c.chunk_rows > (1u << 30) || c.n_rows > (1ull << 48))
        return ZF_ECORRUPT;
    if (c.nch > kNoallocMaxChunks) return ZF_EINVAL;
    if ((uint64_t)c.nch != (c.n_rows + c.chunk_rows - 1) / c.chunk_rows || c.total > col_bytes ||
        64 + 32ull * c.nch > c.total)
        return ZF_ECORRUPT;
    return c.n_rows * c.size > out_bytes ? ZF_EINVAL : ZF_OK;
}

// The warp jobs of a column, each of at most `rows` rows of one chunk.
struct Jobs {
    uint32_t rows, per, n;   // rows of a job, jobs of a chunk, jobs of the column
};
__device__ Jobs cut(const Column& c, uint32_t tiles) {
    const uint32_t rows = 1024u * tiles, per = (c.chunk_rows + rows - 1) / rows;
    const uint32_t last = (uint32_t)(c.n_rows - (uint64_t)(c.nch - 1) * c.chunk_rows);
    return {rows, per, (c.nch - 1) * per + (last + rows - 1) / rows};   // a column of 2^32 jobs has 2^42 rows
}

__device__ __forceinline__ void post(unsigned long long* slot, uint64_t call, uint32_t status) {
    atomicMax(slot, (call << 8) | status);
}

// Structural checks of chunk k (the host path makes the same checks before a
// column is accepted) and its descriptor; false if it is malformed.  The
// entries of delta blocks and Float2Int exceptions are left to job_ok.
__device__ bool chunk_ok(const uint8_t* col, const Column& c, uint32_t k, uint8_t* out, uint64_t out_bytes,
                         ZfDevChunk& dc, zfd::Hdr& h) {
    const uint8_t* d = col + 64 + 32ull * k;
    const ulonglong2 e = *reinterpret_cast<const ulonglong2*>(d);        // offset, bytes
    const ulonglong2 r = *reinterpret_cast<const ulonglong2*>(d + 16);   // first row, rows
    const uint64_t off = e.x, len = e.y;
    // chunks follow each other: each starts where the previous one ends
    uint64_t start = 64 + 32ull * c.nch;
    if (k) {
        const ulonglong2 p = *reinterpret_cast<const ulonglong2*>(d - 32);
        start = p.x + p.y;
    }
    const uint64_t row0 = (uint64_t)k * c.chunk_rows;
    const uint32_t rows = (uint32_t)min((unsigned long long)c.chunk_rows, (unsigned long long)(c.n_rows - row0));
    if (off != start || off < 64 + 32ull * c.nch || off > c.total || len > c.total - off || r.x != row0 ||
        (uint32_t)r.y != rows || len < 64 || (len & 15) || (off & 15))
        return false;
    const uint8_t* blob = col + off;
    dc.blob = blob;
    dc.dst = out + row0 * c.size;
    dc.dst_cap = out_bytes - row0 * c.size;
    dc.rows = rows;
    dc.blob_bytes = (uint32_t)len;
    dc.chunk_id = k;
    dc.scheme = (uint8_t)c.scheme;
    dc.dtype = (uint8_t)c.dtype;
    zfd::load_hdr(blob, h);
    const uint2 m = __ldg(reinterpret_cast<const uint2*>(blob));
    if (m.x != zf::kChunkMagic || (m.y & 0xFFu) != c.scheme || ((m.y >> 8) & 0xFFu) != c.dtype || h.rows != rows)
        return false;
    const int nsec = (c.scheme == ZF_RLE || c.scheme == ZF_FLOAT2INT) ? 3
                     : (c.scheme == ZF_DICT_BP || c.scheme == ZF_DELTA_BP) ? 2 : 1;
    for (int s = 0; s < 3; s++)
        if (s < nsec && (h.off[s] < 64 || (h.off[s] & 15) || (uint64_t)h.off[s] + h.len[s] > len)) return false;
    const uint32_t sz = c.size, wd = 8 * sz, b = h.b, n_aux = h.n_aux;
    const uint64_t packed = ((uint64_t)rows * b + 7) / 8;
    switch (c.scheme) {
    case ZF_RAW: return h.len[0] == (uint64_t)rows * sz;
    case ZF_FOR_BP: return b <= wd && h.len[0] == packed;
    case ZF_DICT_BP:
        return n_aux <= zf::kMaxDict && n_aux && h.len[0] == (uint64_t)n_aux * sz && b == 32u - __clz(n_aux - 1) &&
               h.len[1] == packed;
    case ZF_DELTA_BP: {
        const uint32_t nb = (rows + zf::kDeltaBlock - 1) / zf::kDeltaBlock;
        return n_aux == nb && h.len[0] == (uint64_t)nb * zf::kDeltaEntry;
    }
    case ZF_RLE:
        return n_aux <= rows && n_aux && h.len[0] == (uint64_t)n_aux * sz && h.len[1] == 4ull * n_aux &&
               h.len[2] == 8ull * ((rows + zf::kRleDirRows - 1) / zf::kRleDirRows);
    case ZF_FLOAT2INT:
        return b <= 64 && blob[48] <= zf::kF2IMaxExp && n_aux <= rows && h.len[0] == packed &&
               h.len[1] == 4ull * n_aux && h.len[2] == 8ull * n_aux;
    }
    return false;
}

// Delta block entries of rows [r0, r0 + nrows) (32 blocks at most): true if
// they lie inside the chunk; `widest` = the widest of them.
__device__ bool delta_entries(const zfd::Hdr& h, uint32_t r0, uint32_t nrows, const ZfDevChunk& dc, uint32_t& widest) {
    const uint32_t lane = threadIdx.x & 31;
    uint32_t b = 0;
    bool ok = true;
    if (lane * zf::kDeltaBlock < nrows) {
        const uint8_t* e = dc.blob + h.off[0] + (uint64_t)(r0 / zf::kDeltaBlock + lane) * zf::kDeltaEntry;
        const uint2 w = __ldg(reinterpret_cast<const uint2*>(e + 16));
        const uint32_t mk = min(zf::kDeltaBlock, nrows - lane * zf::kDeltaBlock);
        b = w.y & 0xFFu;
        ok = b <= (dc.dtype == ZF_I32 ? 32u : 64u) && !(w.x & 15) &&
             (uint64_t)w.x + ((((uint64_t)mk * b + 7) / 8 + 15) & ~15ull) <= h.len[1];
    }
    widest = __reduce_max_sync(0xFFFFFFFFu, b);
    return __all_sync(0xFFFFFFFFu, ok);
}

// The rest of a chunk's checks, shared by its jobs: delta block entries of
// the job's rows and the job's share of a Float2Int chunk's exception rows,
// which must be strictly increasing and inside the chunk.
__device__ bool job_ok(const zfd::Hdr& h, uint32_t r0, uint32_t nrows, uint32_t job_rows, const ZfDevChunk& dc) {
    uint32_t widest;
    if (dc.scheme == ZF_DELTA_BP) return delta_entries(h, r0, nrows, dc, widest);
    bool ok = true;
    if (dc.scheme == ZF_FLOAT2INT) {
        const uint64_t jobs = (dc.rows + job_rows - 1) / job_rows, j = r0 / job_rows;
        const uint32_t z = (uint32_t)((j + 1) * h.n_aux / jobs);
        const uint32_t* er = reinterpret_cast<const uint32_t*>(dc.blob + h.off[1]);
        for (uint32_t i = (uint32_t)(j * h.n_aux / jobs) + (threadIdx.x & 31); i < z; i += 32) {
            const uint32_t x = __ldg(er + i);
            ok &= x < dc.rows && (i == 0 || x > __ldg(er + i - 1));
        }
    }
    return __all_sync(0xFFFFFFFFu, ok);
}

// Checks every chunk of the column; what it finds is in the call's result word
// before noalloc_decode starts.  What bounds it: the latency of a chain of four
// reads (column header, directory entry, chunk header, block entries).
__global__ void __launch_bounds__(kWarps * 32) noalloc_check(const uint8_t* col, uint64_t col_bytes, uint8_t* out,
                                                             uint64_t out_bytes, unsigned long long* slot,
                                                             uint64_t call) {
    __shared__ Column s_col;
    __shared__ Jobs s_jobs;
    if (threadIdx.x == 0) {
        Column c;
        const zf_status st = read_column(col, col_bytes, out_bytes, c);
        if (blockIdx.x == 0 && st != ZF_OK) post(slot, call, kRefused | (uint32_t)st);
        s_jobs = st == ZF_OK && c.n_rows ? cut(c, kCheckTiles) : Jobs{1, 1, 0};
        s_col = c;
    }
    __syncthreads();
    for (uint32_t job = blockIdx.x * kWarps + (threadIdx.x >> 5); job < s_jobs.n; job += gridDim.x * kWarps) {
        ZfDevChunk dc{};
        zfd::Hdr h{};
        const uint32_t r0 = (job % s_jobs.per) * s_jobs.rows;
        if (!chunk_ok(col, s_col, job / s_jobs.per, out, out_bytes, dc, h) ||
            !job_ok(h, r0, min(s_jobs.rows, dc.rows - r0), s_jobs.rows, dc)) {
            if ((threadIdx.x & 31) == 0) post(slot, call, kRefused | ZF_ECORRUPT);
        }
    }
}

__device__ __forceinline__ void decode(const ZfDevChunk& c, const zfd::Hdr& h, uint32_t r0, uint32_t nr, uint32_t* wsm,
                                       uint32_t* err) {
    switch (c.scheme * 4 + c.dtype) {
#define ZF_CASE(S, D) \
    case S * 4 + D: zfd::decode_one<S, D, true>(c, h, r0, nr, wsm, err); break;
        ZF_CASE(ZF_RAW, ZF_I32) ZF_CASE(ZF_RAW, ZF_I64) ZF_CASE(ZF_RAW, ZF_F64)
        ZF_CASE(ZF_FOR_BP, ZF_I32) ZF_CASE(ZF_FOR_BP, ZF_I64)
        ZF_CASE(ZF_DICT_BP, ZF_I32) ZF_CASE(ZF_DICT_BP, ZF_I64)
        ZF_CASE(ZF_DELTA_BP, ZF_I32) ZF_CASE(ZF_DELTA_BP, ZF_I64)
        ZF_CASE(ZF_RLE, ZF_I32) ZF_CASE(ZF_RLE, ZF_I64) ZF_CASE(ZF_FLOAT2INT, ZF_F64)
#undef ZF_CASE
    }
}

// A CTA's warps take consecutive jobs, then the jobs gridDim CTAs further.
// The jobs of a CTA share kSmem bytes: when the widest of them does not fit
// four times, fewer warps decode at a time.
__global__ void __launch_bounds__(kWarps * 32, kCtasPerSm) noalloc_decode(const uint8_t* col, uint64_t col_bytes,
                                                                          uint8_t* out, uint64_t out_bytes,
                                                                          unsigned long long* slot, uint64_t call) {
    __shared__ uint4 smem4[kSmem / 16];
    __shared__ uint32_t s_need[kWarps];
    __shared__ Column s_col;
    __shared__ ZfDevChunk s_dc[kWarps];   // the warps' chunks, here and not in registers: 64 a thread are few
    __shared__ zfd::Hdr s_h[kWarps];      // for a kernel that decodes every scheme
    __shared__ Jobs s_jobs;
    __shared__ uint32_t err[2];           // error bits of the CTA's jobs and a chunk that failed
    const uint32_t warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        Column c;
        const zf_status st = read_column(col, col_bytes, out_bytes, c);
        const unsigned long long found = __ldcg(slot);
        err[0] = 0;
        err[1] = 0xFFFFFFFFu;
        s_jobs = Jobs{1, 1, 0};
        if (st == ZF_OK && c.n_rows && !(found >> 8 == call && (found & kRefused))) {
            const uint64_t tiles = (c.n_rows + 1023) / 1024, warps = (uint64_t)gridDim.x * kWarps;
            s_jobs = cut(c, (uint32_t)min((unsigned long long)kJobTiles, (unsigned long long)((tiles + warps - 1) / warps)));
        }
        s_col = c;
    }
    __syncthreads();
    for (uint32_t base = blockIdx.x * kWarps; base < s_jobs.n; base += gridDim.x * kWarps) {
        const uint32_t job = base + warp;
        uint32_t need = 0, r0 = 0, nr = 0;
        ZfDevChunk dc{};
        zfd::Hdr h{};
        if (job < s_jobs.n) {
            const uint32_t k = job / s_jobs.per;
            r0 = (job % s_jobs.per) * s_jobs.rows;
            if (chunk_ok(col, s_col, k, out, out_bytes, dc, h)) {   // as noalloc_check found it
                nr = min(s_jobs.rows, dc.rows - r0);
                uint32_t widest = h.b;
                if (s_col.scheme == ZF_DELTA_BP) delta_entries(h, r0, nr, dc, widest);
                dc.bmax = (uint8_t)widest;
                need = max(16u, (zfd::warp_smem((int)s_col.scheme, s_col.size, dc.bmax) + 15u) & ~15u);
            }
            __syncwarp();   // lanes may still be reading the job before's chunk there
            if (lane == 0) {
                s_dc[warp] = dc;
                s_h[warp] = h;
            }
        }
        __syncthreads();
        if (lane == 0) s_need[warp] = need;
        __syncthreads();
        uint32_t most = 16;
#pragma unroll
        for (uint32_t w = 0; w < kWarps; w++) most = max(most, s_need[w]);
        const uint32_t at_once = min(kWarps, kSmem / most);
        for (uint32_t g = 0; g < kWarps; g += at_once) {
            if (need && warp >= g && warp < g + at_once)
                decode(s_dc[warp], s_h[warp], r0, nr, reinterpret_cast<uint32_t*>(smem4) + (warp - g) * (most / 4), err);
            if (at_once < kWarps) __syncthreads();
        }
    }
    __syncthreads();
    if (threadIdx.x == 0 && err[0])
        post(slot, call, err[0] & (1u << ZF_ECORRUPT) ? ZF_ECORRUPT : ZF_EINVAL);
}

}  // namespace

extern "C" zf_status zf_decompress_device_noalloc(const void* d_column, uint64_t column_bytes, void* d_out,
                                                  uint64_t out_bytes, void* stream) {
    if (!d_column || column_bytes < 64 || ((uintptr_t)d_column & 15) || ((uintptr_t)d_out & 15))
        return ZF_EINVAL;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return ZF_ECUDA;
    Device d;   // with this call's number
    {
        // first call on this device: look up the array's device address (the
        // host-side name of the array is not a device address)
        std::lock_guard<std::mutex> g(g_mu);
        if (!g_dev[dev].slots) {
            if (cudaGetSymbolAddress((void**)&d.slots, g_noalloc_slots) != cudaSuccess || !d.slots ||
                cudaDeviceGetAttribute(&d.sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || d.sms < 1) {
                cudaGetLastError();
                return ZF_ECUDA;
            }
            g_dev[dev] = d;
        }
        g_dev[dev].calls++;
        d = g_dev[dev];
    }
    cudaStream_t s = (cudaStream_t)stream;
    // a column has at most out_bytes / 4 rows, or the kernels refuse it
    const uint64_t ctas = (out_bytes / 4096 + kWarps) / kWarps, sms = (uint64_t)d.sms;
    const uint8_t* col = (const uint8_t*)d_column;
    uint8_t* out = (uint8_t*)d_out;
    unsigned long long* slot = d.slots + d.calls % kSlots;
    noalloc_check<<<(unsigned)std::min(ctas, 2 * sms), kWarps * 32, 0, s>>>(col, column_bytes, out, out_bytes, slot, d.calls);
    noalloc_decode<<<(unsigned)std::min(ctas, kCtasPerSm * sms), kWarps * 32, 0, s>>>(col, column_bytes, out, out_bytes, slot,
                                                                                      d.calls);
    if (cudaGetLastError() != cudaSuccess) return ZF_ECUDA;
    unsigned long long r = 0;
    if (cudaMemcpyAsync(&r, slot, sizeof(r), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
        cudaStreamSynchronize(s) != cudaSuccess)
        return ZF_ECUDA;
    return r >> 8 == d.calls ? (zf_status)(r & 0xFFu & ~kRefused) : ZF_OK;
}

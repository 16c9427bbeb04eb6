// Device code of the paged tensor store: the batched page-table scatter
// (put), gather (get), gather with a fused fp32 -> bf16 round-to-nearest-even
// cast, and live-page moves (compaction, pulls). A launch carries its
// descriptors in its own parameter space (up to ~31 KiB): no host->device
// descriptor copy.
//
// Work split: every segment of a launch is cut into tiles, and a tile is
// copied in one round by one CTA (16 KiB, tile_copy) or one warp (4 KiB,
// warp_tile): all its loads, then all its stores. No counters, no shared
// memory, no barriers; the hardware block scheduler balances the SMs.
//
// HBM-bound by construction (2 bytes of traffic per payload byte, 1.5 for the
// cast): every global access but the first and last bytes of an unaligned
// buffer is one coalesced 16-byte vector, and programmatic dependent launch
// lets the next launch's set-up, and an L2 prefetch of each tile's source,
// overlap the end of this one. Default caching (streaming hints lost ~1.5%).
#pragma once

#include <cstdint>

namespace t2i {

// Loads and stores (T2I_TUNE_* macros can be overridden at compile time, for
// tuning sweeps).
#ifndef T2I_TUNE_CACHE
#define T2I_TUNE_CACHE 1  // 0: streaming (.cs) loads and stores; 1: default caching; 2: loads bypass L1
#endif

// Every source byte of the launch is device memory: a tile may ask L2 for its
// source lines before the previous grid on the stream has completed. A CTA
// of the next launch becomes resident as soon as one of the draining launch
// exits, so its first HBM reads overlap that drain. A prefetch is only a
// cache hint: it changes no value that a load returns (L2 serves every SM's
// loads), so a source that the previous grid is still writing is read
// correctly after the wait.
constexpr uint32_t kPrefetchSources = 1u;
#ifndef T2I_TUNE_PREFETCH
#define T2I_TUNE_PREFETCH 1
#endif
constexpr bool kPrefetch = T2I_TUNE_PREFETCH != 0;

// Parameter-space tiers: a launch copies only its tier's bytes of parameters,
// and smaller parameters launch faster: the launch call alone takes 1.35 us
// with 256 bytes, 1.5 with 1 KiB, 1.75 with 8 KiB, 1.85 with 16 KiB and 2.1
// with 31 KiB (a get of 646 small tensors, 15.5 KiB of descriptors, 19.9 us in
// the largest tier, 18.8 in its own).
constexpr int kBlobTiny = 256;
constexpr int kBlobSmall = 1024;
constexpr int kBlobMid = 8192;
constexpr int kBlobHalf = 16384;
constexpr int kBlobLarge = 31 * 1024;  // header + blob stays below the 32,764-byte parameter limit

// ---- tiled launches (see tile_copy): the segments cut into 16 KiB tiles,
// one CTA each. 512 threads x 2 vectors, from a sweep on GB300 over threads x
// vectors (us a pass; put + get of B=4 requests of 45 MB on one stream / of 16
// B=8 requests of 92 MB on four / get of 2.7 GB / put, compaction and get of
// 1 GiB). Tiles of 16 KiB: 512 x 2 94.1 / 810 / 755 / 895; 256 x 4 96.7 / 815 /
// 760 / 904. Of 32 KiB: 1024 x 2 94.6 / 810 / 765 / 901; 512 x 4 98.2 / 814 / 759 /
// 904. Of 8 KiB: 256 x 2 95.1 / 812 / 757 / 900; 128 x 4 93.9 / 815 / 760 / 904.
// 512 x 2 without the L2 prefetch: 102.0 / 811 / 757 / 902.
constexpr uint32_t kTileShift = 14;
constexpr uint32_t kTileBytes = 1u << kTileShift;
#ifndef T2I_TUNE_TILE_THREADS
#define T2I_TUNE_TILE_THREADS 512
#endif
constexpr unsigned kTileThreads = T2I_TUNE_TILE_THREADS;
#ifndef T2I_TUNE_TILE_MIN_BYTES
#define T2I_TUNE_TILE_MIN_BYTES (4ull << 20)
#endif
// Threads of a launch whose tiles fit the SMs at once, by tiles per SM: as many
// as leave an SM room for just these CTAs (2,048 threads). With room to
// spare, the next grid's CTAs fill some SMs early and others late, and its
// slowest SM decides: eight B=1 requests on one stream (11.5 MB, 705 tiles a
// call) took 62.4 us a pass in 512 threads, 58.0 in 384; of 14 MB (870) 74.7,
// 70.0 in 320; a launch of over 8 tiles an SM takes 512. (kTileMinBytes makes
// two tiles an SM or more on 152 SMs: the first two entries serve larger chips.)
#ifndef T2I_TUNE_TILE_BALANCE
#define T2I_TUNE_TILE_BALANCE 1
#endif
constexpr unsigned kTileWaveThreads[] = {1024, 1024, 1024, 672, 512, 384, 320, 288, 256};
constexpr unsigned kTileMaxPerSm = T2I_TUNE_TILE_BALANCE ? 8 : 0;
// Threads of a launch beside other streams' launches. Those hide each other's
// ramps; what counts then is bytes in flight against latency (longer in
// scattered pages), and six CTAs an SM hold 96 KiB, the four of 512 threads 64.
// In 512 / 384 / 320 / 256 threads on four streams: handoffs of 58 MB a call in
// scattered 64 KiB pages 195.5 / 191.0 / 190.0 / 190.3 us a pass, of 29 MB 132.4
// / 128.6 / 127.0 / 126.9, of 14 MB in 2 MiB pages 98.6 / 96.7 / 94.9 / 94.8, of
// 92 MB 814.8 / 813.7 / 813.7 / 814.9; adapter gets of 98 MB 6.83 / 7.06 / 7.11 /
// 7.14 TB/s; pulls of 92 MB 7.06 / 7.15 / 7.16 / 7.15.
constexpr unsigned kTileOverlapThreads = 320;
// Such launches of fewer bytes run as warp tiles: of 11.5 MB on four streams,
// issued from C, 6.82 TB/s, against 6.85 / 6.70 / 6.66 / 6.55 in CTA tiles of 512
// / 384 / 320 / 256 threads. In warp tiles and in CTA tiles of 320 threads (us a
// pass): sixteen handoffs on four streams, in scattered 64 KiB pages, of 14 MiB
// 158.6 and 162.5, of 16 172.1 and 175.3, of 17 175.8 and 176.0, of 19 191.6 and
// 190.1; in 2 MiB pages of 14 139.0 and 139.9, of 16 164.7 and 158.2, of 18 176.3
// and 176.2. Eight requests put on one stream and got on another, each get
// waiting for its put, of 14 MiB 124.7 and 117.2, of 16 130.7 and 125.7, of 18
// 149.2 and 132.8 (there a warp CTA of 31 warps takes an SM's registers; the
// kernels before the tiles took 132.1, 134.0 and 140.0).
constexpr uint64_t kTileOverlapMinBytes = 16ull << 20;
// Vectors per thread, and the most threads of a kernel of V vectors.
constexpr int tile_vec(unsigned threads) { return threads >= 512 ? 2 : 4; }
template <int V>
constexpr unsigned kTileMaxThreads = V == 2 ? 1024 : 384;
// A CTA's threads copy a whole tile in one round, within their kernel's bound.
constexpr bool tile_threads_ok(unsigned threads) {
    const int v = tile_vec(threads);
    return threads % 32 == 0 && threads * unsigned(v) * 16 >= kTileBytes &&
           threads <= (v == 2 ? kTileMaxThreads<2> : kTileMaxThreads<4>);
}
constexpr bool tile_wave_threads_ok() {
    for (unsigned t : kTileWaveThreads)
        if (!tile_threads_ok(t)) return false;
    return kTileMaxPerSm < sizeof(kTileWaveThreads) / sizeof(kTileWaveThreads[0]);
}
static_assert(tile_threads_ok(kTileThreads), "T2I_TUNE_TILE_THREADS does not cover a tile");
static_assert(tile_threads_ok(kTileOverlapThreads), "kTileOverlapThreads does not cover a tile");
static_assert(tile_wave_threads_ok(), "kTileWaveThreads: an entry does not cover a tile, or one is missing");
// Aligned launches of at least this many bytes run as CTA tiles, others as
// warp tiles. On one stream eight B=1 requests took (us a pass) 47.1 in CTA
// tiles and 59.7 in warp tiles at 7 MB a call, 58.0 and 59.3 at 11.5 MB, four
// of 39 MB 94.1 and 95.3. Below the line the host issues a call in the time
// that either kernel takes (4 MB: 42.9 and 43.5), and calls of many small
// segments are the usual ones.
constexpr uint64_t kTileMinBytes = T2I_TUNE_TILE_MIN_BYTES;

// Warp tiles (see warp_tile): 4 KiB each, one warp each, any alignment. A
// launch that fits runs one CTA an SM, of as many warps (up to 32) as share its
// tiles out evenly; a larger one CTAs of 4 warps. With 4 warps a CTA, eight B=1
// requests in warp tiles took 68.2 us a pass, evenly shared 59.3 (11.5 MB a
// call); 14 MB 75.8 and 69.5.
#ifndef T2I_TUNE_WARP_BALANCE
#define T2I_TUNE_WARP_BALANCE 1
#endif
constexpr unsigned kWarpThreads = 128;
constexpr unsigned kWarpMaxPerSm = T2I_TUNE_WARP_BALANCE ? 32 : 0;  // warps of one CTA
constexpr int kWarpVec = 8;  // 16-byte source vectors per lane
constexpr uint32_t kWarpTileShift = 12;
constexpr uint32_t kWarpTileBytes = 1u << kWarpTileShift;
static_assert(kWarpTileBytes == 32 * kWarpVec * 16, "one round of a warp's loads per tile");

struct TileSeg {
    uint64_t user;
    uint32_t nbytes;  // 1 .. 1 GiB: longer segments are split at page boundaries
    uint32_t tile0;   // first tile of the segment in the launch
    uint32_t page;    // its page number (kTileOnePage), else its first entry in the page array
    uint32_t flags;
};
static_assert(sizeof(TileSeg) == 24, "TileSeg layout");
constexpr uint32_t kTileCast = 1u;     // fp32 -> bf16 (get only)
constexpr uint32_t kTileOnePage = 2u;  // one page, or a run of consecutive ones from `page` on
constexpr uint64_t kTileMaxSegBytes = uint64_t(1) << 30;

struct TileHeader {
    uint64_t pool;
    uint32_t n_seg;
    uint32_t page_shift;
    uint32_t n_tiles;
    uint32_t flags;  // kPrefetchSources, kTileTable
    uint32_t table_at;     // byte offset of the segment table in blob (kTileTable)
    uint32_t table_shift;  // tiles per entry, as a power of two
};
static_assert(sizeof(TileHeader) == 32, "TileHeader layout");
// The launch carries a table of segments: uint16 entry e is the segment of tile
// e << table_shift, so a tile's segment lies between two entries. Searching
// 256 descriptors takes 8 dependent loads of parameters, which miss the
// constant cache in turn; with the table it takes one or two. A 40 MB get of
// 256 adapter tensors took 12.2 us without it and 11.8 with it, such gets on
// four streams ran at 6.13 TB/s and 6.90. The table costs the host about a
// nanosecond a segment, so it comes with segments of many tiles only; and a
// long launch alone on the GPU gains nothing from CTAs that start sooner (a
// 2.7 GB get took 753 us without and 757 with it, compaction of 1 GiB in calls
// of up to 512 MiB 891 and 899), so it has none.
constexpr uint32_t kTileTable = 2u;
#ifndef T2I_TUNE_TABLE_MIN_SEGS
#define T2I_TUNE_TABLE_MIN_SEGS 5
#endif
constexpr uint32_t kTableMinSegs = T2I_TUNE_TABLE_MIN_SEGS;
constexpr uint32_t kTableMinTilesPerSeg = 8;
#ifndef T2I_TUNE_TABLE_MAX_BYTES
#define T2I_TUNE_TABLE_MAX_BYTES (256u << 20)
#endif
constexpr uint32_t kTableMaxBytes = T2I_TUNE_TABLE_MAX_BYTES;

template <int BLOB>
struct TileParams {
    TileHeader h;
    alignas(8) unsigned char blob[BLOB];  // TileSeg[n_seg], then uint32 pages[], then the uint16 table
};

enum class Mode { Put, Get, Move };

#ifdef __CUDACC__

// ---------------------------------------------------------------- loads/stores
#if T2I_TUNE_CACHE == 0
__device__ __forceinline__ uint4 ld_stream(const uint4* p) { return __ldcs(p); }
__device__ __forceinline__ void st_stream(uint4* p, const uint4& v) { __stcs(p, v); }
#elif T2I_TUNE_CACHE == 1
__device__ __forceinline__ uint4 ld_stream(const uint4* p) { return *p; }
__device__ __forceinline__ void st_stream(uint4* p, const uint4& v) { *p = v; }
#else
__device__ __forceinline__ uint4 ld_stream(const uint4* p) {
    uint4 v;
    asm volatile("ld.global.nc.L1::no_allocate.v4.u32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
                 : "l"(p));
    return v;
}
__device__ __forceinline__ void st_stream(uint4* p, const uint4& v) { __stcs(p, v); }
#endif

// fp32 -> bf16, round to nearest even, on bit patterns: add just under half
// an ulp of bf16, plus one when the kept part is odd, and drop 16 bits (the
// classic bias-and-truncate method); NaN (exponent all ones, mantissa not
// zero) becomes a quiet NaN with its sign.
__device__ __forceinline__ uint32_t bf16_rne_bits(uint32_t u) {
    const bool nan = (u & 0x7FFFFFFFu) > 0x7F800000u;
    const uint32_t r = (u + 0x7FFFu + ((u >> 16) & 1u)) >> 16;
    return nan ? (0x7FC0u | ((u >> 16) & 0x8000u)) : r;
}

// Two of them packed (a in the low half). By default the hardware's
// round-to-nearest-even conversion (cvt.rn.bf16x2.f32, which keeps
// subnormals and rounds overflow to infinity like the bit arithmetic above),
// with NaN results replaced by the quiet NaN with the input's sign; a sweep
// on GB300 over 1 GiB of fp32: casts into 2-byte-aligned destinations 5.83 ->
// 6.50 TB/s (the shuffle cast was bound by its arithmetic), into aligned ones
// 6.45 -> 6.67; handoff gets unchanged. T2I_TUNE_CVT=0 packs two
// bf16_rne_bits instead. Both are compared with the oracle over all 2^32
// inputs by the GPU tests.
#ifndef T2I_TUNE_CVT
#define T2I_TUNE_CVT 1
#endif
__device__ __forceinline__ uint32_t pack_bf16x2(uint32_t a, uint32_t b) {
#if T2I_TUNE_CVT
    uint32_t r;
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(__uint_as_float(b)), "f"(__uint_as_float(a)));
    if ((a & 0x7FFFFFFFu) > 0x7F800000u) r = (r & 0xFFFF0000u) | 0x7FC0u | ((a >> 16) & 0x8000u);
    if ((b & 0x7FFFFFFFu) > 0x7F800000u) r = (r & 0x0000FFFFu) | ((0x7FC0u | ((b >> 16) & 0x8000u)) << 16);
    return r;
#else
    return bf16_rne_bits(a) | (bf16_rne_bits(b) << 16);
#endif
}

// The copy of one tile by the CTA's threads (len <= kTileBytes <= blockDim.x *
// V vectors, both sides 16-byte aligned).
template <int V>
__device__ __forceinline__ void tile_copy_bytes(unsigned char* __restrict__ dst, const unsigned char* __restrict__ src,
                                                uint32_t len) {
    const uint32_t nvec = len >> 4;
    const uint4* s = reinterpret_cast<const uint4*>(src);
    uint4* d = reinterpret_cast<uint4*>(dst);
    uint4 r[V];
#pragma unroll
    for (int j = 0; j < V; ++j) {
        const uint32_t v = j * blockDim.x + threadIdx.x;
        if (v < nvec) r[j] = ld_stream(s + v);
    }
#pragma unroll
    for (int j = 0; j < V; ++j) {
        const uint32_t v = j * blockDim.x + threadIdx.x;
        if (v < nvec) st_stream(d + v, r[j]);
    }
    const uint32_t at = (nvec << 4) + threadIdx.x;
    if (at < len) dst[at] = src[at];
}

// The same with the cast: len source bytes, a multiple of 4. Blocks of 8
// floats (two 16-byte loads, one 16-byte store), the last < 8 one by one.
template <int V>
__device__ __forceinline__ void tile_cast(unsigned char* __restrict__ dst, const unsigned char* __restrict__ src,
                                          uint32_t len) {
    static_assert(V % 2 == 0, "a block is two vectors");
    const uint32_t n8 = len >> 5;
    const uint4* s = reinterpret_cast<const uint4*>(src);
    uint4* d = reinterpret_cast<uint4*>(dst);
    uint4 a[V / 2], b[V / 2];
#pragma unroll
    for (int j = 0; j < V / 2; ++j) {
        const uint32_t v = j * blockDim.x + threadIdx.x;
        if (v < n8) {
            a[j] = ld_stream(s + 2 * v);
            b[j] = ld_stream(s + 2 * v + 1);
        }
    }
#pragma unroll
    for (int j = 0; j < V / 2; ++j) {
        const uint32_t v = j * blockDim.x + threadIdx.x;
        if (v < n8) {
            uint4 o;
            o.x = pack_bf16x2(a[j].x, a[j].y);
            o.y = pack_bf16x2(a[j].z, a[j].w);
            o.z = pack_bf16x2(b[j].x, b[j].y);
            o.w = pack_bf16x2(b[j].z, b[j].w);
            st_stream(d + v, o);
        }
    }
    const uint32_t at = (n8 << 3) + threadIdx.x;
    if (at < len >> 2)
        reinterpret_cast<uint16_t*>(dst)[at] = (uint16_t)bf16_rne_bits(reinterpret_cast<const uint32_t*>(src)[at]);
}

// Programmatic dependent launch: wait until the previous grid in the stream
// has completed and its memory is visible (returns at once when this launch
// has no such dependency), then let the next launch begin its set-up.
__device__ __forceinline__ void pdl_wait_then_release() {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// The last segment that starts at or before this tile.
template <int BLOB>
__device__ __forceinline__ uint32_t find_tile(const TileParams<BLOB>& p, uint32_t tile) {
    const TileSeg* segs = reinterpret_cast<const TileSeg*>(p.blob);
    uint32_t lo = 0, hi = p.h.n_seg - 1;
    if (p.h.flags & kTileTable) {
        const uint16_t* table = reinterpret_cast<const uint16_t*>(p.blob + p.h.table_at) + (tile >> p.h.table_shift);
        lo = table[0];
        hi = table[1];
    }
    while (lo < hi) {
        const uint32_t mid = (lo + hi + 1) >> 1;
        if (segs[mid].tile0 <= tile)
            lo = mid;
        else
            hi = mid - 1;
    }
    return lo;
}

// ------------------------------------------------------------- tiled launches
// One CTA per tile: the 16 KiB (or the rest) of one segment at a multiple of
// 16 KiB, in one page or one run of pages, both sides 16-byte aligned. Bound
// by HBM; between launches on one stream by the drain of one grid and the
// ramp-up of the next. So a CTA lives for one round of straight-line code:
// its tile is worked out, and its source lines asked of L2, before the wait
// for the previous grid; then come its loads, then its stores. CTAs of the
// next grid take over an SM 16 KiB at a time as this one drains, and the
// hardware block scheduler balances the SMs without a counter or a barrier.
// Against CTAs that walk 64 KiB shares in 32 KiB rounds (us a pass, the cases
// of the sweep above): 109.9 / 818 / 766 / 921; requests pulled between
// stores (92 MB a launch) 54.7 -> 51.8.
template <Mode M, int V, int BLOB>
__device__ __forceinline__ void tile_copy(const TileParams<BLOB>& p) {
    constexpr bool kToUser = M == Mode::Get;
    const TileSeg* segs = reinterpret_cast<const TileSeg*>(p.blob);
    const uint32_t lo = find_tile(p, blockIdx.x);
    const uint32_t off = (blockIdx.x - segs[lo].tile0) << kTileShift;
    const uint32_t len = umin(kTileBytes, segs[lo].nbytes - off);
    const uint32_t flags = segs[lo].flags;
    const bool cast = kToUser && (flags & kTileCast);
    uint32_t page = segs[lo].page, in_page = off;
    if (!(flags & kTileOnePage)) {
        page = reinterpret_cast<const uint32_t*>(segs + p.h.n_seg)[page + (off >> p.h.page_shift)];
        in_page = off & ((1u << p.h.page_shift) - 1);
    }
    unsigned char* pa = reinterpret_cast<unsigned char*>(p.h.pool) + (uint64_t(page) << p.h.page_shift) + in_page;
    unsigned char* ua = reinterpret_cast<unsigned char*>(segs[lo].user) + (cast ? off >> 1 : off);
    const unsigned char* src = kToUser ? pa : ua;
    unsigned char* dst = kToUser ? ua : pa;
    if (kPrefetch && (p.h.flags & kPrefetchSources) && threadIdx.x * 128u < len)
        asm volatile("prefetch.global.L2 [%0];" ::"l"(src + threadIdx.x * 128u));
    pdl_wait_then_release();
    if (cast)
        tile_cast<V>(dst, src, len);
    else
        tile_copy_bytes<V>(dst, src, len);
}

// ---------------------------------------------------------------- warp tiles
// Bytes [n, n + 16) of lo|hi, n in 0..15.
__device__ __forceinline__ uint4 bytes_from(uint4 lo, uint4 hi, uint32_t n) {
    const bool by8 = n & 8u, by4 = n & 4u;
    const uint32_t a0 = by8 ? lo.z : lo.x, a1 = by8 ? lo.w : lo.y, a2 = by8 ? hi.x : lo.z, a3 = by8 ? hi.y : lo.w,
                   a4 = by8 ? hi.z : hi.x, a5 = by8 ? hi.w : hi.y;
    const uint32_t b0 = by4 ? a1 : a0, b1 = by4 ? a2 : a1, b2 = by4 ? a3 : a2, b3 = by4 ? a4 : a3, b4 = by4 ? a5 : a4;
    const uint32_t r = 8u * (n & 3u);
    return make_uint4(__funnelshift_r(b0, b1, r), __funnelshift_r(b1, b2, r), __funnelshift_r(b2, b3, r),
                      __funnelshift_r(b3, b4, r));
}

__device__ __forceinline__ uint4 shfl4(uint4 v, uint32_t from) {
    return make_uint4(__shfl_sync(0xFFFFFFFFu, v.x, from), __shfl_sync(0xFFFFFFFFu, v.y, from),
                      __shfl_sync(0xFFFFFFFFu, v.z, from), __shfl_sync(0xFFFFFFFFu, v.w, from));
}

// Stores output vectors d[first .. nv): d[k] = bytes [n, n + 16) of w[k]|w[k + 1].
// Lane l holds w[32 j + l] in r[j], lane 31 also w[32 V] in last.
template <int V>
__device__ __forceinline__ void store_shifted(uint4* d, const uint4 (&r)[V], uint4 last, uint32_t n, uint32_t first,
                                              uint32_t nv) {
    const uint32_t lane = threadIdx.x & 31u;
#pragma unroll
    for (int j = 0; j < V; ++j) {
        // the next vector: lane + 1's, or for lane 31 lane 0's of the next 32
        uint4 next = shfl4(j + 1 < V && lane == 0 ? r[j + 1 < V ? j + 1 : j] : r[j], (lane + 1) & 31u);
        if (j + 1 == V && lane == 31) next = last;
        const uint32_t k = j * 32 + lane;
        if (k >= first && k < nv) st_stream(d + k, bytes_from(r[j], next, n));
    }
}

// One warp per tile: 4 KiB of one segment's source, at any alignment of the
// user's address, pages of any size. No shared memory, no barrier: a warp
// finds its tile, asks L2 for its source lines and then waits for the
// previous grid; every global access but a segment's first and last bytes
// is one aligned 16-byte vector. Where the two sides are misaligned to each
// other, each output vector is cut out of two source vectors, the second
// one taken from the next lane (a shuffle). Tiles are cut at 16-byte
// boundaries of the side that is written, so that only a segment's first
// and last vectors are partial.
// Bound by latency in small launches: a warp holds 4 KiB of one segment, so
// that many small segments run side by side instead of one after another in
// a CTA's share, and a call with any mix of alignments is one launch instead
// of two. Bound by HBM in large ones, which come here for their alignment or
// their small pages. Before (CTAs walking shares, pieces realigned in shared
// memory) and after, kernel times of one launch on an idle GPU: 646 tensors of
// 256 B to 36 KiB got in 10.6 -> 5.0 us, 40 ragged objects put in 14.5 (two
// launches) -> 4.9, got in 10.4 -> 4.9. Ten launches back to back: 1 GiB puts from
// unaligned sources 7.13 -> 7.21 TB/s, gets into unaligned destinations 7.08 ->
// 7.13, casts into 2-byte aligned ones 6.92 -> 7.18 (timed alone, such a put
// 331 -> 327 us, a get 329 -> 322); 64 MiB in scattered 8 KiB pages put
// 4.97 -> 7.25, got 4.81 -> 6.50, cast 3.24 -> 6.53. Tiles of 1 or 2 KiB in small
// launches (fewer vectors a lane, more warps) changed no pass.
template <Mode M, int BLOB>
__device__ __forceinline__ void warp_tile(const TileParams<BLOB>& p) {
    constexpr bool kToUser = M == Mode::Get;
    const uint32_t lane = threadIdx.x & 31u;
    const uint32_t tile = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (tile >= p.h.n_tiles) {
        pdl_wait_then_release();
        return;
    }
    const TileSeg* segs = reinterpret_cast<const TileSeg*>(p.blob);
    const TileSeg& s = segs[find_tile(p, tile)];
    const uint32_t* pages = reinterpret_cast<const uint32_t*>(segs + p.h.n_seg);
    unsigned char* pool = reinterpret_cast<unsigned char*>(p.h.pool);
    unsigned char* user = reinterpret_cast<unsigned char*>(s.user);
    const uint32_t nbytes = s.nbytes, flags = s.flags, page = s.page, pshift = p.h.page_shift;
    const uint32_t at = (tile - s.tile0) << kWarpTileShift;  // source bytes before this tile (less the phase)
    const uint32_t phase = uint32_t(s.user) & 15u;           // of the user's side; pages are 16-byte aligned
    // pool address of byte o of the segment
    auto paged = [&](uint32_t o) -> unsigned char* {
        if (flags & kTileOnePage) return pool + (uint64_t(page) << pshift) + o;
        return pool + (uint64_t(pages[page + (o >> pshift)]) << pshift) + (o & ((1u << pshift) - 1));
    };
    // the same for bytes of this tile, whose page (or run) is looked up once
    const bool one_page = (flags & kTileOnePage) || pshift >= kWarpTileShift;
    unsigned char* const base = one_page && at < nbytes ? paged(at) : pool;
    auto in_tile = [&](uint32_t o) -> unsigned char* { return one_page ? base + (o - at) : paged(o); };

    if (kPrefetch && (p.h.flags & kPrefetchSources) && at + lane * 128u < nbytes)
        asm volatile("prefetch.global.L2 [%0];" ::"l"(kToUser ? in_tile(at + lane * 128u) : user + at + lane * 128u));
    pdl_wait_then_release();

    if (kToUser && (flags & kTileCast)) {
        // fp32 -> bf16: blocks of 8 floats (32 bytes) make one output vector.
        // With q counting output bytes from the 16-byte boundary at or before
        // `user`, the tile is q in [at / 2, at / 2 + 2048) and its vector k
        // holds the last phase bytes of block at / 32 + k - 1 and the first of
        // block at / 32 + k.
        constexpr int kBlocks = kWarpVec / 2;
        const uint32_t nq = umin((nbytes >> 1) + phase - (at >> 1), kWarpTileBytes / 2);
        const uint32_t nv = nq >> 4;
        uint16_t* d16 = reinterpret_cast<uint16_t*>(user - phase + (at >> 1));
        const uint32_t back = phase ? 32u : 0u;  // w[0] is the block before the tile's
        const uint32_t need = phase ? nv + 1 : nv;
        const uint4 zero = make_uint4(0u, 0u, 0u, 0u);
        auto load = [&](uint32_t k, uint4* a, uint4* b) {  // the two vectors of w[k]; those without a source byte are zero
            const uint32_t o = at + 32u * k - back;
            *a = *b = zero;
            if (k >= need || int32_t(o) < 0 || o >= nbytes) return;
            const unsigned char* src = o < at ? paged(o) : in_tile(o);
            *a = ld_stream(reinterpret_cast<const uint4*>(src));
            if (o + 16u < nbytes) *b = ld_stream(reinterpret_cast<const uint4*>(src) + 1);
        };
        auto bf16 = [](const uint4& a, const uint4& b) {
            return make_uint4(pack_bf16x2(a.x, a.y), pack_bf16x2(a.z, a.w), pack_bf16x2(b.x, b.y), pack_bf16x2(b.z, b.w));
        };
        uint4 a[kBlocks], b[kBlocks], la = zero, lb = zero;
#pragma unroll
        for (int j = 0; j < kBlocks; ++j) load(j * 32 + lane, &a[j], &b[j]);
        if (phase && lane == 31) load(kBlocks * 32, &la, &lb);
        // the elements before the first whole vector and after the last one
        const bool head = phase && at == 0;
        const uint32_t n_head = head ? umin((16u - phase) >> 1, nbytes >> 2) : 0u;
        const uint32_t n_tail = head && nv == 0 ? 0u : (nq & 15u) >> 1;
        const uint32_t e_head = phase >> 1, e_tail = nv << 3;
        uint16_t x_head = 0, x_tail = 0;
        if (lane < n_head) x_head = (uint16_t)bf16_rne_bits(*reinterpret_cast<const uint32_t*>(paged(4u * lane)));
        if (lane < n_tail)
            x_tail = (uint16_t)bf16_rne_bits(*reinterpret_cast<const uint32_t*>(paged(at + 4u * (e_tail + lane - e_head))));
        uint4* d = reinterpret_cast<uint4*>(d16);
        uint4 r[kBlocks];
#pragma unroll
        for (int j = 0; j < kBlocks; ++j) r[j] = bf16(a[j], b[j]);
        if (phase) {
            store_shifted<kBlocks>(d, r, bf16(la, lb), 16u - phase, head ? 1u : 0u, nv);
        } else {
#pragma unroll
            for (int j = 0; j < kBlocks; ++j)
                if (j * 32 + lane < nv) st_stream(d + j * 32 + lane, r[j]);
        }
        if (lane < n_head) d16[e_head + lane] = x_head;
        if (lane < n_tail) d16[e_tail + lane] = x_tail;
        return;
    }

    // A copy. With q counting bytes from the 16-byte boundary at or before
    // the first byte written (q = byte + skip), the tile is q in
    // [at, at + 4096). Output vector k is bytes [n, n + 16) of w[k]|w[k + 1]:
    // get: w[k] = the object's vector at / 16 + k - 1, n = 16 - phase;
    // put: w[k] = the user's aligned vector at / 16 + k, n = phase.
    const uint32_t skip = kToUser ? phase : 0u;
    const uint32_t nq = umin(nbytes + skip - at, kWarpTileBytes);
    const uint32_t nv = nq >> 4;
    unsigned char* const out = kToUser ? user - phase + at : nullptr;
    const unsigned char* const in = kToUser ? nullptr : user - phase + at;
    auto w = [&](uint32_t k) -> uint4 {
        const unsigned char* a;
        if (kToUser) {
            const uint32_t o = at + 16u * k - (phase ? 16u : 0u);
            if (int32_t(o) < 0 || o >= nbytes) return make_uint4(0u, 0u, 0u, 0u);
            a = o < at ? paged(o) : in_tile(o);
        } else {
            a = in + 16u * k;
        }
        return ld_stream(reinterpret_cast<const uint4*>(a));
    };
    const uint32_t need = phase ? nv + 1 : nv;
    uint4 r[kWarpVec], last = make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
    for (int j = 0; j < kWarpVec; ++j) r[j] = (nv && j * 32 + lane < need) ? w(j * 32 + lane) : last;
    if (phase && lane == 31 && need > kWarpVec * 32) last = w(kWarpVec * 32);
    const bool head = skip && at == 0;
    const uint32_t n_head = head ? umin(16u - phase, nbytes) : 0u;
    const uint32_t n_tail = head && nv == 0 ? 0u : nq & 15u;
    const uint32_t o_tail = at + (nv << 4) - skip;  // first byte after the last whole vector
    unsigned char x_head = 0, x_tail = 0;
    if (kToUser && lane < n_head) x_head = *paged(lane);
    if (lane < n_tail) x_tail = kToUser ? *paged(o_tail + lane) : user[o_tail + lane];
    const uint32_t first = head ? 1u : 0u, n = kToUser ? 16u - phase : phase;
    if (kToUser || one_page) {
        uint4* d = reinterpret_cast<uint4*>(kToUser ? out : base);
        if (phase) {
            store_shifted<kWarpVec>(d, r, last, n, first, nv);
        } else {
#pragma unroll
            for (int j = 0; j < kWarpVec; ++j)
                if (j * 32 + lane < nv) st_stream(d + j * 32 + lane, r[j]);
        }
    } else {  // pages smaller than a tile: each vector finds its own
#pragma unroll
        for (int j = 0; j < kWarpVec; ++j) {
            uint4 v = r[j];
            if (phase) {
                uint4 next = shfl4(j + 1 < kWarpVec && lane == 0 ? r[j + 1 < kWarpVec ? j + 1 : j] : r[j], (lane + 1) & 31u);
                if (j + 1 == kWarpVec && lane == 31) next = last;
                v = bytes_from(v, next, n);
            }
            const uint32_t k = j * 32 + lane;
            if (k < nv) st_stream(reinterpret_cast<uint4*>(paged(at + 16u * k)), v);
        }
    }
    if (kToUser && lane < n_head) user[lane] = x_head;
    if (lane < n_tail) {
        if (kToUser)
            user[o_tail + lane] = x_tail;
        else
            *paged(o_tail + lane) = x_tail;
    }
}

// Entry points (one per operation and kind of tile, so that profiles name
// them). A move's source and destination are both pool pages; as warp tiles
// it is a put.
template <int V, int BLOB>
__global__ void __launch_bounds__(kTileMaxThreads<V>, 2048 / kTileMaxThreads<V>)
    scatter_put_kernel(const __grid_constant__ TileParams<BLOB> p) {
    tile_copy<Mode::Put, V, BLOB>(p);
}
template <int V, int BLOB>
__global__ void __launch_bounds__(kTileMaxThreads<V>, 2048 / kTileMaxThreads<V>)
    gather_get_kernel(const __grid_constant__ TileParams<BLOB> p) {
    tile_copy<Mode::Get, V, BLOB>(p);
}
template <int V, int BLOB>
__global__ void __launch_bounds__(kTileMaxThreads<V>, 2048 / kTileMaxThreads<V>)
    compact_move_kernel(const __grid_constant__ TileParams<BLOB> p) {
    tile_copy<Mode::Move, V, BLOB>(p);
}
template <int BLOB>
__global__ void __launch_bounds__(1024, 1)
    scatter_put_warp_kernel(const __grid_constant__ TileParams<BLOB> p) {
    warp_tile<Mode::Put, BLOB>(p);
}
template <int BLOB>
__global__ void __launch_bounds__(1024, 1)
    gather_get_warp_kernel(const __grid_constant__ TileParams<BLOB> p) {
    warp_tile<Mode::Get, BLOB>(p);
}

#endif  // __CUDACC__

}  // namespace t2i

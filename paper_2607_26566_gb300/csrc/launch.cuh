// Launch packing of the store's kernels (part of store.cu). A batch's segments
// are packed into as few launches as their descriptors allow (each launch
// carries up to ~31 KiB of descriptors and page numbers in its parameters),
// as CTA tiles or as warp tiles, and launched with programmatic dependent
// launch. Together with kernels.cuh this decides what a launch does, so
// profiles are keyed to a hash of both files. Included by store.cu inside
// namespace t2i.
#pragma once

// One object (or page) of a batch, on its way to a launch.
struct Seg {
    uint64_t user;          // device-visible address of the user's side
    uint64_t nbytes_flags;  // bytes in the pool, kCastFlag (and kRunFlag, set by the launcher)
    const uint32_t* pages;
    uint32_t n_pages;
};
constexpr uint64_t kCastFlag = uint64_t(1) << 63;
constexpr uint64_t kRunFlag = uint64_t(1) << 62;  // one page, or consecutive ones
constexpr uint64_t kSegBytesMask = ~(kCastFlag | kRunFlag);

// Whether the pages are consecutive. Scattered pages mostly show at the last
// one; a run is then read in one pass without branches.
inline bool pages_are_run(const Seg& s) {
    const uint32_t first = s.pages[0], n = s.n_pages;
    if (s.pages[n - 1] != first + (n - 1)) return false;
    uint32_t off = 0;
    for (uint32_t k = 0; k < n; ++k) off |= s.pages[k] ^ (first + k);
    return off == 0;
}

// The kernel of a mode, a kind of tile (V = 0: warp tiles, else CTA tiles of V
// vectors per thread) and a tier of parameters.
template <Mode M, int V, int BLOB>
const void* tile_kernel() {
    if constexpr (V == 0)
        return M == Mode::Get ? reinterpret_cast<const void*>(gather_get_warp_kernel<BLOB>)
                              : reinterpret_cast<const void*>(scatter_put_warp_kernel<BLOB>);
    else
        return M == Mode::Put   ? reinterpret_cast<const void*>(scatter_put_kernel<V, BLOB>)
               : M == Mode::Get ? reinterpret_cast<const void*>(gather_get_kernel<V, BLOB>)
                                : reinterpret_cast<const void*>(compact_move_kernel<V, BLOB>);
}

// Loads every kernel on the current device, once per device (the driver loads
// a kernel, allocating device memory for it, when it is first named): calls
// then allocate nothing and can be captured.
template <int... BLOB>
cudaError_t load_tier_kernels() {
    const void* fns[] = {tile_kernel<Mode::Get, 0, BLOB>()...,  tile_kernel<Mode::Put, 0, BLOB>()...,
                         tile_kernel<Mode::Get, 2, BLOB>()...,  tile_kernel<Mode::Get, 4, BLOB>()...,
                         tile_kernel<Mode::Put, 2, BLOB>()...,  tile_kernel<Mode::Put, 4, BLOB>()...,
                         tile_kernel<Mode::Move, 2, BLOB>()..., tile_kernel<Mode::Move, 4, BLOB>()...};
    cudaFuncAttributes a;
    cudaError_t e = cudaSuccess;
    for (const void* fn : fns)
        if (e == cudaSuccess) e = cudaFuncGetAttributes(&a, fn);
    return e;
}
inline cudaError_t load_kernels(int device) {
    static std::mutex mu;
    static std::vector<bool> loaded;
    std::lock_guard<std::mutex> lock(mu);
    if (loaded.size() <= size_t(device)) loaded.resize(size_t(device) + 1, false);
    if (loaded[device]) return cudaSuccess;
    const cudaError_t e = load_tier_kernels<kBlobTiny, kBlobSmall, kBlobMid, kBlobHalf, kBlobLarge>();
    if (e == cudaSuccess) loaded[device] = true;
    return e;
}

// Packs and launches the segments of one pool.
class TileLauncher {
  public:
    // launches (nullable) counts the kernels launched
    TileLauncher(uint64_t pool, uint32_t page_shift, int device, uint64_t* launches)
        : pool_(pool), page_shift_(page_shift), launches_(launches) {
        int n = 0;
        if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, device) == cudaSuccess) sms_ = unsigned(n);
    }

    // kPrefetchSources, or 0 when a source is (or may be) other than device memory
    uint32_t flags = kPrefetchSources;
    bool overlapped = false;      // launches of other streams are likely to run beside these
    uint32_t fail_countdown = 0;  // > 0: that many launches from now, report a failure (testing)
    std::string error;

    template <Mode M>
    t2i_status launch(std::vector<Seg>& segs, cudaStream_t stream);

  private:
    template <Mode M, bool WARP>
    t2i_status launch_tiles(const std::vector<Seg>& segs, cudaStream_t stream);
    void add_table(TileHeader* h, unsigned char* blob, size_t blob_bytes);
    template <Mode M, bool WARP, int BLOB>
    t2i_status launch_one(uint32_t n_seg, uint32_t n_tiles, cudaStream_t stream);

    uint64_t pool_;
    uint32_t page_shift_;
    unsigned sms_ = 0;
    uint64_t* launches_;
    std::vector<uint32_t> lp_;  // page lists of the launch being packed
    alignas(16) unsigned char param_buf_[sizeof(TileParams<kBlobLarge>)];
};

// One launch of the n_seg descriptors in param_buf_ and the pages in lp_.
template <Mode M, bool WARP, int BLOB>
t2i_status TileLauncher::launch_one(uint32_t n_seg, uint32_t n_tiles, cudaStream_t stream) {
    if (fail_countdown && --fail_countdown == 0) {
        error = "kernel launch failed: injected failure (t2i_inject_launch_failure)";
        return T2I_ERR_CUDA;
    }
    auto* p = reinterpret_cast<TileParams<BLOB>*>(param_buf_);
    p->h.pool = pool_;
    p->h.n_seg = n_seg;
    p->h.page_shift = page_shift_;
    p->h.n_tiles = n_tiles;
    p->h.flags = flags;
    std::memcpy(p->blob + n_seg * sizeof(TileSeg), lp_.data(), lp_.size() * sizeof(uint32_t));
    if (n_seg >= kTableMinSegs && n_tiles / n_seg >= kTableMinTilesPerSeg &&
        (overlapped || n_tiles < kTableMaxBytes / (WARP ? kWarpTileBytes : kTileBytes)))
        add_table(&p->h, p->blob, BLOB);
    const void* fn;
    unsigned grid = n_tiles, threads = kTileThreads;
    if constexpr (WARP) {
        fn = tile_kernel<M, 0, BLOB>();
        unsigned warps = kWarpThreads / 32;
        if (n_tiles <= kWarpMaxPerSm * sms_) warps = (n_tiles + sms_ - 1) / sms_;
        threads = 32 * warps;
        grid = (n_tiles + warps - 1) / warps;
    } else {
        if (overlapped)
            threads = kTileOverlapThreads;
        else if (n_tiles <= kTileMaxPerSm * sms_)
            threads = kTileWaveThreads[(n_tiles + sms_ - 1) / sms_];
        fn = tile_vec(threads) == 2 ? tile_kernel<M, 2, BLOB>() : tile_kernel<M, 4, BLOB>();
    }
    void* args[] = {param_buf_};
    cudaLaunchConfig_t lc = {};
    lc.gridDim = dim3(grid);
    lc.blockDim = dim3(threads);
    lc.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    lc.attrs = attr;
    lc.numAttrs = 1;
    const cudaError_t e = cudaLaunchKernelExC(&lc, fn, args);
    if (e != cudaSuccess) {
        error = std::string("kernel launch failed: ") + cudaGetErrorString(e);
        return T2I_ERR_CUDA;
    }
    if (launches_) ++*launches_;
    return T2I_OK;
}

// Puts the segment table behind the page lists, with up to two entries a
// segment, as far as the tier has room (it is not worth a larger tier).
inline void TileLauncher::add_table(TileHeader* h, unsigned char* blob, size_t blob_bytes) {
    const TileSeg* segs = reinterpret_cast<const TileSeg*>(blob);
    const size_t at = h->n_seg * sizeof(TileSeg) + lp_.size() * sizeof(uint32_t);
    const size_t room = std::min<size_t>(2 * h->n_seg, (blob_bytes - at) / sizeof(uint16_t));
    if (room < 3) return;
    uint32_t shift = 0;  // entries 0 .. ((n_tiles - 1) >> shift) + 1
    while (((h->n_tiles - 1) >> shift) + 2 > room) ++shift;
    const uint32_t n = ((h->n_tiles - 1) >> shift) + 2;
    uint16_t* table = reinterpret_cast<uint16_t*>(blob + at);
    uint32_t e = 0;
    for (uint32_t i = 0; i < h->n_seg; ++i) {
        const uint64_t end = i + 1 < h->n_seg ? segs[i + 1].tile0 : uint64_t(n) << shift;
        for (; e < n && (uint64_t(e) << shift) < end; ++e) table[e] = static_cast<uint16_t>(i);
    }
    h->table_at = static_cast<uint32_t>(at);
    h->table_shift = shift;
    h->flags |= kTileTable;
}

// The segments as tiles, in as few launches as their descriptors allow.
// Descriptors are written where the launch reads them; page lists follow.
// WARP = false: every user address is 16-byte aligned, and every tile lies in
// one page or run.
template <Mode M, bool WARP>
t2i_status TileLauncher::launch_tiles(const std::vector<Seg>& segs, cudaStream_t stream) {
    constexpr uint64_t kTile = WARP ? kWarpTileBytes : kTileBytes;
    static_assert(offsetof(TileParams<kBlobLarge>, blob) == sizeof(TileHeader), "the same place in every tier");
    TileSeg* const out = reinterpret_cast<TileSeg*>(param_buf_ + sizeof(TileHeader));
    uint32_t n_seg = 0, tiles = 0;
    lp_.clear();
    auto flush = [&]() -> t2i_status {
        const size_t bytes = n_seg * sizeof(TileSeg) + lp_.size() * sizeof(uint32_t);
        const t2i_status st = n_seg == 0                    ? T2I_OK
                              : bytes <= size_t(kBlobTiny)  ? launch_one<M, WARP, kBlobTiny>(n_seg, tiles, stream)
                              : bytes <= size_t(kBlobSmall) ? launch_one<M, WARP, kBlobSmall>(n_seg, tiles, stream)
                              : bytes <= size_t(kBlobMid)   ? launch_one<M, WARP, kBlobMid>(n_seg, tiles, stream)
                              : bytes <= size_t(kBlobHalf)  ? launch_one<M, WARP, kBlobHalf>(n_seg, tiles, stream)
                                                            : launch_one<M, WARP, kBlobLarge>(n_seg, tiles, stream);
        n_seg = tiles = 0;
        lp_.clear();
        return st;
    };
    const uint64_t P = uint64_t(1) << page_shift_;
    const uint64_t seg_pages = kTileMaxSegBytes / P;
    const uint64_t list_pages = std::min<uint64_t>(seg_pages, (kBlobLarge - sizeof(TileSeg)) / sizeof(uint32_t));
    for (const Seg& s : segs) {
        const uint64_t nbytes = s.nbytes_flags & kSegBytesMask;
        const uint32_t cast = (s.nbytes_flags & kCastFlag) != 0;
        const bool run = (s.nbytes_flags & kRunFlag) != 0;
        const uint64_t step = run ? seg_pages : list_pages;
        for (uint64_t p0 = 0; p0 < s.n_pages; p0 += step) {
            const uint64_t np = std::min<uint64_t>(step, s.n_pages - p0);
            const bool one = run || np == 1;
            const uint64_t off = p0 * P;
            TileSeg d;
            d.user = s.user + (off >> cast);
            d.nbytes = static_cast<uint32_t>(std::min<uint64_t>(nbytes - off, np * P));
            // a get's warp tiles start at 16-byte boundaries of the destination
            const uint64_t phase = WARP && M == Mode::Get ? (d.user & 15u) << cast : 0;
            const uint32_t n = static_cast<uint32_t>((d.nbytes + phase + kTile - 1) / kTile);
            if ((n_seg + 1) * sizeof(TileSeg) + (lp_.size() + (one ? 0 : np)) * sizeof(uint32_t) > size_t(kBlobLarge) ||
                uint64_t(tiles) + n > 0x7FFFFFFFull) {
                const t2i_status st = flush();
                if (st != T2I_OK) return st;
            }
            d.tile0 = tiles;
            d.page = one ? s.pages[p0] : static_cast<uint32_t>(lp_.size());
            d.flags = (cast ? kTileCast : 0) | (one ? kTileOnePage : 0);
            out[n_seg++] = d;
            if (!one) lp_.insert(lp_.end(), s.pages + p0, s.pages + p0 + np);
            tiles += n;
        }
    }
    return flush();
}

// A call whose segments are all aligned and fit CTA tiles runs as those, any
// other call as warp tiles. (A call of aligned and other segments is not
// split: 200 ragged objects, 26 MB, took 33.7 us a put and get with their
// aligned ones as CTA tiles, 32.4 as one launch.)
template <Mode M>
t2i_status TileLauncher::launch(std::vector<Seg>& segs, cudaStream_t stream) {
    uint64_t bytes = 0, tiles = 0;
    bool aligned = true;
    bool runs = true;  // every segment is one page or one run of pages
    for (Seg& s : segs) {
        const uint64_t n = s.nbytes_flags & kSegBytesMask;
        bytes += n;
        tiles += (n + kTileBytes - 1) / kTileBytes;
        aligned = aligned && (s.user & 15u) == 0;
        const bool run = s.n_pages == 1 || pages_are_run(s);
        if (run) s.nbytes_flags |= kRunFlag;
        runs = runs && run;
    }
    // CTA tiles: each in one page or run; the call large enough; its tiles filled
    // well enough (a half-empty one costs as much as a full one)
    const bool fit = aligned && (runs || page_shift_ >= kTileShift) &&
                     bytes >= (overlapped ? kTileOverlapMinBytes : kTileMinBytes) &&
                     tiles * kTileBytes <= bytes + bytes / 4;
    return fit ? launch_tiles<M, false>(segs, stream) : launch_tiles<M, true>(segs, stream);
}

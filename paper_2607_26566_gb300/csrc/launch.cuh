// Launch packing of the store's kernels (part of store.cu; included after
// the Store class). A batch's segments are packed into as few launches as
// their descriptors allow (each launch carries up to ~31 KiB of descriptors
// and page numbers in its parameters), as CTA tiles or as warp tiles, and
// launched with programmatic dependent launch. Together with kernels.cuh
// this decides what a launch does, so profiles are keyed to a hash of both
// files. Included by store.cu inside namespace t2i.
#pragma once

// One kernel launch of the parameters in param_buf_.
inline t2i_status Store::launch_kernel(const void* fn, unsigned grid, unsigned threads, cudaStream_t stream) {
    void* args[] = {param_buf_};
    if (fail_countdown_ && --fail_countdown_ == 0) {
        err_ = "kernel launch failed: injected failure (t2i_inject_launch_failure)";
        return T2I_ERR_CUDA;
    }
    cudaLaunchConfig_t lc = {};
    lc.gridDim = dim3(grid);
    lc.blockDim = dim3(threads);
    lc.dynamicSmemBytes = 0;
    lc.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    lc.attrs = attr;
    lc.numAttrs = 1;
    cudaError_t e = cudaLaunchKernelExC(&lc, fn, args);
    if (e != cudaSuccess) {
        err_ = std::string("kernel launch failed: ") + cudaGetErrorString(e);
        return T2I_ERR_CUDA;
    }
    ctl_.counters().launches++;
    return T2I_OK;
}

template <Mode M, bool WARP, int BLOB>
t2i_status Store::launch_tiles_one(uint32_t n_seg, uint32_t n_tiles, cudaStream_t stream) {
    auto* p = reinterpret_cast<TileParams<BLOB>*>(param_buf_);
    p->h.pool = pool_;
    p->h.n_seg = n_seg;
    p->h.page_shift = page_shift_;
    p->h.n_tiles = n_tiles;
    p->h.flags = launch_flags_;
    std::memcpy(p->blob + n_seg * sizeof(TileSeg), lp_.data(), lp_.size() * sizeof(uint32_t));
    const void* fn = WARP ? (M == Mode::Get ? reinterpret_cast<const void*>(get_warp_kernel<BLOB>)
                                            : reinterpret_cast<const void*>(put_warp_kernel<BLOB>))
                          : (M == Mode::Put   ? reinterpret_cast<const void*>(put_tile_kernel<BLOB>)
                             : M == Mode::Get ? reinterpret_cast<const void*>(get_tile_kernel<BLOB>)
                                              : reinterpret_cast<const void*>(move_tile_kernel<BLOB>));
    constexpr uint32_t kPerCta = WARP ? kWarpThreads / 32 : 1;
    return launch_kernel(fn, (n_tiles + kPerCta - 1) / kPerCta, WARP ? kWarpThreads : kTileThreads, stream);
}

// The segments as tiles, in as few launches as their descriptors allow.
// Descriptors are written where the launch reads them; page lists follow.
// WARP = false: every user address is 16-byte aligned, and tiles_fit.
template <Mode M, bool WARP>
t2i_status Store::launch_tiles(const std::vector<Seg>& segs, cudaStream_t stream) {
    constexpr uint64_t kTile = WARP ? kWarpTileBytes : kTileBytes;
    TileSeg* const out = reinterpret_cast<TileSeg*>(param_buf_ + sizeof(TileHeader));
    uint32_t n_seg = 0, tiles = 0;
    lp_.clear();
    auto flush = [&]() -> t2i_status {
        const size_t bytes = n_seg * sizeof(TileSeg) + lp_.size() * sizeof(uint32_t);
        const t2i_status st = n_seg == 0                    ? T2I_OK
                              : bytes <= size_t(kBlobTiny)  ? launch_tiles_one<M, WARP, kBlobTiny>(n_seg, tiles, stream)
                              : bytes <= size_t(kBlobSmall) ? launch_tiles_one<M, WARP, kBlobSmall>(n_seg, tiles, stream)
                              : bytes <= size_t(kBlobMid)   ? launch_tiles_one<M, WARP, kBlobMid>(n_seg, tiles, stream)
                                                            : launch_tiles_one<M, WARP, kBlobLarge>(n_seg, tiles, stream);
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
        const bool run = pages_are_run(s);
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

// Aligned segments that fit CTA tiles run as those; the rest of the call, or
// all of it, is one launch of warp tiles.
template <Mode M>
t2i_status Store::launch_segments(const std::vector<Seg>& segs, cudaStream_t stream) {
    uint64_t bytes = 0, tiles = 0;
    uint32_t n_other = 0;
    bool fit = true;  // every aligned segment's tiles lie in one page or run
    for (const Seg& s : segs) {
        if (s.user & 15u) {
            ++n_other;
            continue;
        }
        const uint64_t n = s.nbytes_flags & kSegBytesMask;
        bytes += n;
        tiles += (n + kTileBytes - 1) / kTileBytes;
        if (page_shift_ < kTileShift && fit) fit = pages_are_run(s);
    }
    // large enough, and the tiles filled well enough: a half-empty one costs as much as a full one
    if (!fit || bytes < kTileMinBytes || tiles * kTileBytes > bytes + bytes / 4) return launch_tiles<M, true>(segs, stream);
    if (n_other == 0) return launch_tiles<M, false>(segs, stream);
    aligned_.clear();
    general_.clear();
    for (const Seg& s : segs) ((s.user & 15u) == 0 ? aligned_ : general_).push_back(s);
    const t2i_status st = launch_tiles<M, false>(aligned_, stream);
    return st != T2I_OK ? st : launch_tiles<M, true>(general_, stream);
}

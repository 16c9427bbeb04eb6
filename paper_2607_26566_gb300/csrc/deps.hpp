// Stream-ordered page dependencies of a store.
//
// The store's pages are its only shared resource, so its calls are ordered
// by their data dependencies instead of by the order they were made in:
//   - a get (and a compaction, for the pages it moves out) waits for the
//     call that last wrote each page it reads (read after write);
//   - a put (and a compaction, for the pages it moves into) waits for the
//     calls that last wrote or read each page it reuses (write after read,
//     write after write: pages of freed or evicted objects).
// Waiting happens on the GPU (cudaStreamWaitEvent) and only across streams:
// work on one stream is already ordered. Per-call events are recorded only
// once a second stream has used the store, so that single-stream use keeps
// consecutive launches adjacent (programmatic dependent launch). Calls made
// before that have no event of their own; a dependency on one of them waits
// for everything its stream has been given so far.
//
// Streams given to a store must stay valid until the store is destroyed.
#pragma once

#include <cuda_runtime.h>

#include <cstdint>
#include <vector>

namespace t2i {

class StreamDeps {
  public:
    struct Dep {
        uint32_t seq = 0;        // 0 = none; else the call's number on its stream
        uint16_t stream = 0;
    };
    struct PageDeps {
        Dep writer;
        Dep readers[2];
        uint8_t more_readers = 0;  // > 2 reading streams since the last write
        uint16_t viewer = 0;       // stream + 1 that was given a view since (kViewers: several)
    };
    static constexpr uint16_t kViewers = 0xFFFF;
    static constexpr uint32_t kRing = 64;
    // a view's reads are not calls of the store: later writers wait for
    // everything its stream has been given by then
    static constexpr uint32_t kOpen = 0xFFFFFFFFu;

    ~StreamDeps() { release(); }

    void resize_pages(uint64_t n) { pages_.assign(n, PageDeps{}); }

    // Index of `s`, registering it on first use. -1 if an event that the call
    // will need cannot be created. (Events are created when they are first
    // recorded: a stream used alone needs none.)
    int stream_index(cudaStream_t s) {
        size_t i = 0;
        while (i < streams_.size() && streams_[i].s != s) ++i;
        if (i == streams_.size()) {
            if (streams_.size() >= 0xFFFF) return -1;
            streams_.emplace_back();
            streams_.back().s = s;
        }
        if (streams_.size() > 1 && ensure(&streams_[i].ring[(streams_[i].seq + 1) % kRing]) != cudaSuccess) return -1;
        return static_cast<int>(i);
    }

    // Whether a call may depend on another stream's. While one stream alone has
    // used the store, reads() and writes() find nothing to wait for and need
    // not be called; the marks are kept for streams to come.
    bool several() const { return streams_.size() > 1; }

    // Whether the current call and those before it came on several streams in
    // turn (a change of stream within the last kInterleave calls), so that
    // their work is likely to overlap. A hint for the shape of a launch only.
    static constexpr uint32_t kInterleave = 16;
    bool interleaved() const { return since_change_ < kInterleave; }

    // --- one call on stream index `si`
    void begin(int si) {
        since_change_ = si != cur_ ? 0 : since_change_ < kInterleave ? since_change_ + 1 : kInterleave;
        cur_ = si;
        need_.assign(streams_.size(), 0);
        wait_all_ = wait_views_ = false;
    }
    void reads(uint32_t page) { note(pages_[page].writer); }
    void writes(uint32_t page) {
        const PageDeps& d = pages_[page];
        note(d.writer);
        note(d.readers[0]);
        note(d.readers[1]);
        if (d.more_readers) wait_all_ = true;
        if (d.viewer == kViewers)
            wait_views_ = true;
        else if (d.viewer)
            note({kOpen, static_cast<uint16_t>(d.viewer - 1)});
    }
    // Makes the call's stream wait for what it depends on.
    cudaError_t wait() {
        cudaStream_t s = streams_[cur_].s;
        for (size_t j = 0; j < streams_.size(); ++j) {
            uint32_t q = need_[j];
            if (wait_all_ && q < streams_[j].seq) q = streams_[j].seq;
            if (wait_views_ && streams_[j].viewed) q = kOpen;
            if (int(j) == cur_ || q == 0) continue;
            cudaError_t e = wait_for(static_cast<int>(j), q, s);
            if (e != cudaSuccess) return e;
        }
        return cudaSuccess;
    }
    // After the call's work is enqueued: its number (and event, once more than
    // one stream has used the store).
    cudaError_t end(uint32_t* seq_out) {
        State& st = streams_[cur_];
        const uint32_t q = ++st.seq;
        *seq_out = q;
        if (streams_.size() > 1) {
            const uint32_t k = q % kRing;
            cudaError_t e = ensure(&st.ring[k]);
            if (e == cudaSuccess) e = cudaEventRecord(st.ring[k], st.s);
            if (e != cudaSuccess) return e;
            st.ring_seq[k] = q;
        }
        return cudaSuccess;
    }
    void mark_write(uint32_t page, uint32_t seq) {
        PageDeps& d = pages_[page];
        d.writer = {seq, static_cast<uint16_t>(cur_)};
        d.readers[0] = d.readers[1] = Dep{};
        d.more_readers = 0;
        d.viewer = 0;
    }
    void mark_read(uint32_t page, uint32_t seq) {
        PageDeps& d = pages_[page];
        const Dep me{seq, static_cast<uint16_t>(cur_)};
        for (Dep& r : d.readers) {
            if (r.seq == 0 || r.stream == me.stream) {
                r = me;
                return;
            }
        }
        d.more_readers = 1;
    }
    // A view lasts until the page is written: calls made meanwhile, on its
    // stream or on others, do not end its reads.
    void mark_view(uint32_t page) {
        PageDeps& d = pages_[page];
        const uint16_t me = static_cast<uint16_t>(cur_ + 1);
        d.viewer = d.viewer == 0 || d.viewer == me ? me : kViewers;
        streams_[cur_].viewed = true;
    }

    // Waits on the host for everything every known stream has been given.
    void synchronize_all() {
        for (State& st : streams_) {
            if (st.seq == 0 && !st.viewed) continue;
            if (ensure(&st.lazy) == cudaSuccess && cudaEventRecord(st.lazy, st.s) == cudaSuccess)
                cudaEventSynchronize(st.lazy);
        }
    }

    void release() {
        for (State& st : streams_) {
            if (st.lazy) cudaEventDestroy(st.lazy);
            for (cudaEvent_t e : st.ring)
                if (e) cudaEventDestroy(e);
        }
        streams_.clear();
    }


  private:
    struct State {
        cudaStream_t s = nullptr;
        uint32_t seq = 0;           // calls enqueued on this stream
        cudaEvent_t ring[kRing] = {};   // call q's event lives in ring[q % kRing]
        uint32_t ring_seq[kRing] = {};  // the call each ring event was last recorded for
        cudaEvent_t lazy = nullptr; // "everything so far" on this stream
        uint32_t lazy_seq = 0;
        bool viewed = false;        // a view was given to it: reads beyond its calls
    };

    static cudaError_t ensure(cudaEvent_t* e) {
        return *e ? cudaSuccess : cudaEventCreateWithFlags(e, cudaEventDisableTiming);
    }
    void note(const Dep& d) {
        if (d.seq == 0 || d.stream == cur_) return;
        if (need_[d.stream] < d.seq) need_[d.stream] = d.seq;
    }

    // Stream `s` waits until call q of stream j has run: on q's own event if
    // it has one (or on a later call's, which is later on the same stream),
    // else on an event recorded now after everything stream j was given.
    cudaError_t wait_for(int j, uint32_t q, cudaStream_t s) {
        State& st = streams_[j];
        const uint32_t k = q % kRing;
        if (st.ring_seq[k] >= q) return cudaStreamWaitEvent(s, st.ring[k], 0);
        if (st.lazy_seq < q) {
            cudaError_t e = ensure(&st.lazy);
            if (e == cudaSuccess) e = cudaEventRecord(st.lazy, st.s);
            if (e != cudaSuccess) return e;
            st.lazy_seq = st.seq;
        }
        return cudaStreamWaitEvent(s, st.lazy, 0);
    }

    std::vector<State> streams_;
    std::vector<PageDeps> pages_;
    std::vector<uint32_t> need_;
    int cur_ = 0;
    uint32_t since_change_ = kInterleave;  // calls since the last change of stream
    bool wait_all_ = false;    // the call overwrites a page with more_readers
    bool wait_views_ = false;  // ... or with views on several streams
};

}  // namespace t2i

"""Ordering across streams (csrc/deps.hpp) on the CPU, against a recording CUDA
runtime: a stream is a count of the work it was given, an event the count at
its record, a wait raises what the waiting stream has seen of the other. Each
scenario says which of a stream's work a later call has to wait for."""
import os
import subprocess

import pytest

from paper_2607_26566_gb300 import build as b

FAKE_RUNTIME = r"""
#pragma once
#include <algorithm>
#include <map>
typedef int cudaError_t;
enum { cudaSuccess = 0, cudaEventDisableTiming = 2 };
struct FakeStream { int work = 0; std::map<FakeStream*, int> seen; };
struct FakeEvent { FakeStream* s = nullptr; int at = 0; };
typedef FakeStream* cudaStream_t;
typedef FakeEvent* cudaEvent_t;
inline std::map<FakeStream*, int> host_seen;
inline cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { *e = new FakeEvent; return 0; }
inline cudaError_t cudaEventDestroy(cudaEvent_t e) { delete e; return 0; }
inline cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t s) { *e = {s, s->work}; return 0; }
inline cudaError_t cudaStreamWaitEvent(cudaStream_t s, cudaEvent_t e, unsigned) {
    if (e->s) s->seen[e->s] = std::max(s->seen[e->s], e->at);
    return 0;
}
inline cudaError_t cudaEventSynchronize(cudaEvent_t e) { if (e->s) host_seen[e->s] = e->at; return 0; }
"""

# Commands: "<verb><stream>", verbs v(iew), g(et), p(ut) of page 0 and k: work
# the caller gives the stream itself; x: the store is destroyed. Output: the
# work of A, B and C that the last command's stream (x: the host) has waited for.
DRIVER = r"""
#include <cstdio>
#include <string>
#include "deps.hpp"
int main(int argc, char** argv) {
    t2i::StreamDeps d;
    d.resize_pages(1);
    FakeStream s[4];
    auto call = [&](char verb, FakeStream* st) {
        d.begin(d.stream_index(st));
        if (verb == 'p') d.writes(0); else d.reads(0);
        d.wait();
        if (verb == 'v') { d.mark_view(0); return; }
        st->work++;
        uint32_t q = 0;
        d.end(&q);
        if (verb == 'p') d.mark_write(0, q); else d.mark_read(0, q);
    };
    for (int i = 1; i < argc; ++i) {
        const char verb = argv[i][0];
        if (verb == 'x') {
            d.synchronize_all();
            for (int k = 0; k < 3; ++k) std::printf("%d ", host_seen[&s[k]]);
            return 0;
        }
        FakeStream* st = &s[argv[i][1] - 'A'];
        if (verb == 'k') st->work++;
        else call(verb, st);
        if (i + 1 == argc) for (int k = 0; k < 3; ++k) std::printf("%d ", st->seen[&s[k]]);
    }
}
"""


@pytest.fixture(scope="module")
def driver(tmp_path_factory):
    d = tmp_path_factory.mktemp("deps")
    (d / "cuda_runtime.h").write_text(FAKE_RUNTIME)
    (d / "main.cpp").write_text(DRIVER)
    subprocess.run([os.environ.get("CXX", "g++"), "-std=c++17", "-Wall", "-I", str(d), "-I", b.CSRC, str(d / "main.cpp"),
                    "-o", str(d / "deps")], check=True)
    return str(d / "deps")


def waited(driver, calls):
    out = subprocess.run([driver, *calls.split()], capture_output=True, text=True, check=True).stdout
    return [int(x) for x in out.split()]


@pytest.mark.parametrize("calls,want", [
    ("vA kA pB", [1, 0, 0]),                    # a view, a late read in place, the pages reused
    ("vA gA kA pB", [2, 0, 0]),                 # a get on the view's stream ends no view
    ("gA vA kA pB", [2, 0, 0]),
    ("vA gB gA kA pB", [2, 0, 0]),
    ("vA kA vB kB kB vC kC pD", [1, 2, 1]),     # more viewing streams than a page has entries
    ("vA gB gC kA pD", [1, 1, 1]),              # the view in an entry, more readers than entries
    ("gA gB vC kC kC pD", [1, 1, 2]),           # the view beyond the entries
    ("vA gB gC kA gA kA pD", [3, 1, 1]),
    ("vA vB vA kA kB kB pB", [1, 0, 0]),        # views on two streams, one of them the writer's
    ("vA vB kA kB kB pA vC kC pB", [2, 0, 1]),  # a write ends them all
    ("gD gA gB gC kA kB kC pD", [1, 1, 1]),     # without a view: the calls, not the work after them
    ("vA kA pA gB pB kA gB gC gA gD kA pD", [4, 3, 1]),  # a write ends the views before it
])
def test_a_put_waits_for_the_readers_of_the_pages_it_reuses(driver, calls, want):
    got = waited(driver, calls)
    if calls.split()[-1] == "pB":
        got[1] = 0  # its own stream
    assert got == want


@pytest.mark.parametrize("calls,want", [("gA kA gB x", [2, 1, 0]), ("vA kA x", [1, 0, 0]), ("gA vB kB x", [1, 1, 0])])
def test_destroy_waits_for_every_stream(driver, calls, want):
    assert waited(driver, calls) == want

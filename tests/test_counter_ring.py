"""The ring of request counters (csrc/nls_ring.h), compiled with the host
compiler and run against a model of streams: every entry that a flush takes
must have been zeroed since its last use, by a memset that the flush's stream
is ordered after."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

HARNESS = r"""
#include <algorithm>
#include <array>
#include <cstdio>
#include <cstdlib>
#include <random>
#include <vector>

#include "nls_ring.h"

// An operation is its stream and its number there (0: none); a clock holds the
// number of each stream's last operation that something is ordered after.
struct Op { int st = 0, no = 0; };
using Clock = std::array<int, 2>;

struct Model {
    std::array<Clock, 2> known{};
    Clock event{}, host{};
    std::vector<Op> zeroed_by, used_by; // per entry: the last memset, the last use
    std::vector<bool> zero;             // as the device memory holds it in submission order
    int memsets = 0;
    explicit Model(int size) : zeroed_by(size), used_by(size), zero(size, false) {}

    static void join(Clock &a, const Clock &b) { for (int i = 0; i < 2; ++i) a[i] = std::max(a[i], b[i]); }
    bool after(int st, Op o) const { return known[st][o.st] >= o.no; }
    Op issue(int st)
    {
        join(known[st], host);
        return Op{st, ++known[st][st]};
    }
    // the CounterRing's operations
    int release(int i) // the host has waited for the entry's last use
    {
        host[used_by[i].st] = std::max(host[used_by[i].st], used_by[i].no);
        return 0;
    }
    int zero_range(int first, int end, int st)
    {
        const Op op = issue(st);
        for (int i = first; i < end; ++i) {
            if (!after(st, used_by[i])) { std::puts("a memset races with a use"); std::exit(1); }
            zeroed_by[i] = op;
            zero[i] = true;
        }
        event = known[st];
        ++memsets;
        return 0;
    }
    int after_zero(int st)
    {
        join(known[st], event);
        return 0;
    }
    // a flush on `st` uses the entries (recorded by a capture: after a memset of its own)
    void use(int first, int count, int st, bool recorded = false)
    {
        issue(st); // picks up what the host is ordered after
        for (int i = first; i < first + count; ++i) {
            if (recorded) continue;
            if (!zero[i]) { std::printf("entry %d is handed out dirty\n", i); std::exit(1); }
            if (!after(st, zeroed_by[i])) { std::printf("entry %d: not ordered after its memset\n", i); std::exit(1); }
        }
        const Op op = issue(st);
        for (int i = first; i < first + count; ++i) {
            zero[i] = false;
            used_by[i] = op;
        }
    }
};
struct Ops {
    Model *m;
    int release(int i) { return m->release(i); }
    int zero(int a, int b, int st) { return m->zero_range(a, b, st); }
    int after_zero(int st) { return m->after_zero(st); }
};

int main(int argc, char **argv)
{
    const int kind = std::atoi(argv[1]), size = std::atoi(argv[2]), block = std::atoi(argv[3]);
    Model m(size);
    nls::CounterRing<int> ring(size, block);
    int s = -1;
    auto flush = [&](int count, int st) {
        if (ring.take(count, st, false, Ops{&m}, &s)) std::exit(2);
        if (s < 0 || s + count > size) { std::puts("out of the ring"); std::exit(1); }
        m.use(s, count, st);
    };
    if (kind == 0) { // the second stream crosses into a block, then a flush of the first takes its rest and more
        for (int i = 0; i < block / 2 - 1; ++i) flush(2, 0);
        flush(2, 0);
        flush(2, 1);
        flush(block + 104, 0);
        std::printf("%d\n", m.memsets);
    } else if (kind == 1) { // one stream: one memset per block
        for (int i = 0; i < 3 * size / 2; ++i) flush(2, 0);
        std::printf("%d\n", m.memsets);
    } else if (kind == 1000) { // one stream, with flushes that a capture recorded, replayed at any time
        std::mt19937 rng(block);
        std::vector<std::pair<int, int>> recorded;
        for (int i = 0; i < 4000; ++i) {
            const int count = 2 * (1 + rng() % 4);
            if (i > 100 && recorded.size() < 3 && rng() % 8 == 0) {
                if (ring.take(count, 0, true, Ops{&m}, &s)) std::exit(2);
                recorded.push_back({s, count});
            } else if (!recorded.empty() && rng() % 3 == 0) {
                const auto r = recorded[rng() % recorded.size()];
                m.use(r.first, r.second, 0, true);
            } else {
                flush(count, 0);
            }
        }
    } else { // any order of streams and sizes over many laps
        std::mt19937 rng(kind);
        for (int i = 0; i < 4000; ++i) {
            const int most = rng() % 8 ? 8 : size / (1 + rng() % 4);
            flush(2 * (1 + rng() % (most / 2)), rng() % 2);
        }
    }
    return 0;
}
"""


@pytest.fixture(scope="module")
def harness(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("no C++ compiler")
    d = tmp_path_factory.mktemp("ring")
    (d / "ring.cpp").write_text(HARNESS)
    subprocess.run([cxx, "-std=c++17", "-O1", "-Wall", "-Werror", "-I",
                    os.path.join(ROOT, "paper_2403_16341_gb300", "csrc"), "-o", str(d / "ring"), str(d / "ring.cpp")],
                   check=True)
    return str(d / "ring")


def run(harness, *args):
    r = subprocess.run([harness, *map(str, args)], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout
    return r.stdout


def test_rest_of_a_block_zeroed_on_another_stream(harness):
    run(harness, 0, 1 << 16, 1 << 12)


def test_one_memset_per_block(harness):
    assert int(run(harness, 1, 1 << 12, 1 << 8)) == 3 * (1 << 12) // (1 << 8)


@pytest.mark.parametrize("seed", range(2, 10))
@pytest.mark.parametrize("size,block", [(64, 16), (256, 64), (1024, 64)])
def test_any_order_of_streams(harness, seed, size, block):
    run(harness, seed, size, block)


@pytest.mark.parametrize("block", [16, 64, 256])
def test_replays_of_a_captured_flush(harness, block):
    run(harness, 1000, 1024, block)

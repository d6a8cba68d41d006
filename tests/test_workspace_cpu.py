"""How a context's memory for the checkerboard phases grows (csrc/workspace.h),
against an allocator that counts, remembers what is alive, never hands out an
address twice and has a limit: no pointer of a call is given back before the
call's work is enqueued, a buffer that fits stays, and a device without room
for the windows costs a call nothing."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2104_06165_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <map>
#include <vector>
#include "workspace.h"
struct Fake {
    size_t room;
    std::map<void*, size_t> live;
    uintptr_t next = 4096;
    int gets = 0, fails = 0, puts = 0;
    bool failed = false;
    size_t used() const { size_t s = 0; for (auto& e : live) s += e.second; return s; }
    void* get(size_t b) {
        gets++;
        failed = used() + b > room;
        if (failed) { fails++; return nullptr; }
        void* p = (void*)next;
        next += b + 256;
        live[p] = b;
        return p;
    }
    bool full() const { return failed; }
    size_t hidden = 0;                  // free bytes that cannot be had in one piece
    bool captures = false;
    bool capturing() const { return captures; }
    size_t available() const { return room - used() + hidden; }
    void put(void* p) { puts++; if (!live.erase(p)) { std::puts("put of a dead pointer"); std::exit(2); } }
};
// arguments: room, limit, then "draws windows" per call; draws < 0: that much
// for something else of the context (-1: free bytes that cannot be had, -2:
// whether the calls are captured, -3: a map of 2 x windows bytes in four buffers)
int main(int argc, char** argv) {
    Fake a{(size_t)std::atoll(argv[1])};
    PhaseWorkspace w;
    w.limit = (size_t)std::atoll(argv[2]);
    for (int i = 3; i + 1 < argc; i += 2) {
        const long long d = std::atoll(argv[i]);
        const size_t draws = d < 0 ? 0 : d, windows = std::atoll(argv[i + 1]);
        bool stored = false;
        if (d < 0) {
            if (d == -1) a.hidden = windows;
            if (d == -2) a.captures = windows != 0;
            bool got = d >= -2 || (d != -3 && ws_get(w, -d, a) != nullptr);
            if (d == -3) {
                const size_t b[4] = {windows, windows / 4, windows / 2, windows / 4};
                void* p[4];
                got = ws_get_all(w, b, p, 4, a);
            }
            std::printf("%d 0 1 %d %d %d %zu %zu %zu\n", (int)got, a.gets, a.fails, a.puts, (size_t)w.draws.p,
                        (size_t)w.windows.p, a.used());
            continue;
        }
        const bool ok = ws_reserve(w, draws, windows, &stored, a);
        const bool fits = ok && a.live.count(w.draws.p) && a.live[w.draws.p] >= draws &&
                          (!stored || (a.live.count(w.windows.p) && a.live[w.windows.p] >= windows));
        std::printf("%d %d %d %d %d %d %zu %zu %zu\n", (int)ok, (int)stored, (int)fits, a.gets, a.fails, a.puts,
                    (size_t)w.draws.p, (size_t)w.windows.p, a.used());
    }
}
"""


@pytest.fixture(scope="module")
def workspace(tmp_path_factory):
    d = tmp_path_factory.mktemp("ws")
    src, exe = d / "t.cc", d / "t"
    src.write_text(PROGRAM)
    subprocess.check_call(["g++", "-std=c++17", "-Wall", "-Werror", "-I", CSRC, str(src), "-o", str(exe)])

    def run(room, limit, *calls):
        """Per call: ok, stored, buffers alive and large enough, allocations,
        failed ones, frees, the two pointers, bytes held."""
        out = subprocess.check_output([str(exe), str(room), str(limit), *[str(v) for c in calls for v in c]], text=True)
        return [tuple(int(v) for v in line.split()) for line in out.splitlines()]
    return run


def test_a_call_that_fits_changes_nothing(workspace):
    r = workspace(10000, 1 << 40, (20, 1000), (20, 1000), (10, 500), (20, 0))
    assert [c[:3] for c in r] == [(1, 1, 1)] * 3 + [(1, 0, 1)]
    assert all(c[3:] == r[0][3:] for c in r) and r[0][3:6] == (2, 0, 0)


def test_windows_without_room_cost_nothing(workspace):
    """Views of one call share one choice, and calls after the first allocate
    and free nothing: the perturbations stay where the captured graph has them."""
    r = workspace(900, 1 << 40, (20, 1000), (20, 1000), (10, 2000), (20, 1000))
    assert [c[:3] for c in r] == [(1, 0, 1)] * 4
    assert all(c[3:] == r[0][3:] for c in r) and r[0][4:6] == (0, 0)
    # smaller windows that fit are stored all the same
    r = workspace(900, 1 << 40, (20, 1000), (20, 400), (20, 1000), (20, 400))
    assert [c[1] for c in r] == [0, 1, 0, 1] and r[3][6:] == r[1][6:]
    # free memory that turns out not to be there is asked for once
    r = workspace(900, 1 << 40, (-1, 5000), (20, 1000), (20, 1000), (20, 2000), (20, 800))
    assert [c[1] for c in r] == [0, 0, 0, 0, 1] and [c[4] for c in r] == [0, 1, 1, 1, 1]


def test_the_larger_buffer_is_there_before_the_smaller_one_goes(workspace):
    r = workspace(10000, 1 << 40, (20, 1000), (40, 3000))
    assert r[1][:3] == (1, 1, 1) and r[1][5] == 2 and r[1][8] == 3040
    # no room for a larger one: the smaller windows stay for the smaller views
    r = workspace(1500, 1 << 40, (20, 700), (20, 1400), (20, 700))
    assert [c[1] for c in r] == [1, 0, 1] and r[2][7] == r[0][7] and r[2][5] == 0


def test_windows_take_half_of_what_is_free_and_give_way(workspace):
    r = workspace(2020, 1 << 40, (20, 1001), (20, 1000))
    assert [c[1] for c in r] == [0, 1]
    # something else of the context needs more than is left
    r = workspace(2020, 1 << 40, (20, 1000), (-1500, 0), (20, 1000), (20, 250))
    assert [c[0] for c in r] == [1, 1, 1, 1] and [c[1] for c in r] == [1, 0, 0, 1]
    assert r[1][7] == 0 and r[1][8] == 1520
    # also the perturbations of a larger view
    r = workspace(2020, 1 << 40, (20, 1000), (1200, 0))
    assert r[1][0] == 1 and r[1][7] == 0
    # more than there is: refused, and what was there stays usable
    r = workspace(2020, 1 << 40, (20, 0), (-5000, 0), (20, 0))
    assert [c[0] for c in r] == [1, 0, 1] and r[2][6] == r[0][6]


def test_what_a_captured_call_uses_stays(workspace):
    # captured, then a larger call: new buffers, and nothing goes back
    r = workspace(9000, 1 << 40, (20, 1000), (-2, 1), (20, 1000), (-2, 0), (40, 2000), (40, 3000))
    assert r[2][:3] == (1, 1, 1) and r[2][6:8] == r[0][6:8]
    assert r[4][5] == 0 and r[4][8] == 20 + 1000 + 40 + 2000
    assert r[5][5] == 1 and r[5][8] == 20 + 1000 + 40 + 3000     # the later ones were not captured
    # nothing is allocated during a capture: without room for the windows they are rebuilt
    r = workspace(9000, 1 << 40, (20, 0), (-2, 1), (20, 1000), (20, 1000))
    assert [c[1] for c in r] == [0, 0, 0, 0] and r[3][3] == r[0][3]
    # windows of a captured call give way to nothing
    r = workspace(2020, 1 << 40, (20, 0), (20, 900), (-2, 1), (20, 900), (-2, 0), (-1500, 0))
    assert [c[0] for c in r] == [1, 1, 1, 1, 1, 0] and r[5][7] == r[1][7]


def test_a_map_is_there_whole_or_not_at_all(workspace):
    r = workspace(1900, 1 << 40, (-3, 1000), (-3, 800))
    assert [c[0] for c in r] == [0, 1] and [c[8] for c in r] == [0, 1600]
    # windows give way to it
    r = workspace(2000, 1 << 40, (20, 900), (-3, 800))
    assert [c[0] for c in r] == [1, 1] and r[1][8] == 1620


def test_limit_and_no_room_at_all(workspace):
    r = workspace(10000, 999, (20, 1000), (20, 999))
    assert [c[1] for c in r] == [0, 1] and r[0][3] == 1
    r = workspace(10, 1 << 40, (20, 1000), (5, 0))
    assert [c[0] for c in r] == [0, 1] and r[0][8] == 0

"""The stream kernel's byte ring, run on the host: tiles in flight never share
bytes, and a wait that gives up leaves its tile among those that the producer
still waits for before it leaves (their copies may be on their way)."""
import os
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1409_8608_gb300", "csrc")

PROGRAM = r"""
#include "tc_ring.h"
#include <cstdio>
#include <cstdlib>
#include <vector>
constexpr int kBytes = 1000, kSlots = 5;
#define CHECK(x) do { if (!(x)) { std::printf("line %d: %s\n", __LINE__, #x); return 1; } } while (0)
int main() {
    for (int seed = 1; seed <= 200; ++seed) {
        std::srand(seed);
        tc::ByteRing<kBytes, kSlots> ring;
        struct Tile { int at, size, slot; unsigned ph; };
        std::vector<Tile> flight;          // oldest first: what the copies and their readers hold
        int held[kSlots] = {};
        unsigned phase[kSlots] = {};
        const int fail_at = std::rand() % 60;
        int waits = 0;
        bool gave_up = false;
        for (int t = 0; t < 100 && !gave_up; ++t) {
            const int size = 1 + std::rand() % 400;
            int skip = -1;
            gave_up = !ring.make_room(
                size, skip,
                [&](int s, uint32_t ph) {
                    if (flight.empty() || flight[0].slot != s || flight[0].ph != ph) std::exit(2);
                    if (waits++ == fail_at) return false;   // the limit ran out: not released
                    flight.erase(flight.begin());
                    return true;
                },
                [&](int s) { return held[s]; });
            if (gave_up) break;
            const int slot = ring.slot, at = ring.take(size, skip);
            CHECK(at >= 0 && at + size <= kBytes);
            for (const Tile &x : flight) CHECK((at + size <= x.at || x.at + x.size <= at) && x.slot != slot);
            held[slot] = size + skip;
            flight.push_back({at, size, slot, phase[slot]});
            phase[slot] ^= 1u;
        }
        CHECK(gave_up);
        std::vector<Tile> waited;
        ring.drain([&](int s, uint32_t ph) { waited.push_back({0, 0, s, ph}); });
        CHECK(waited.size() == flight.size() && !flight.empty());
        for (size_t i = 0; i < flight.size(); ++i)
            CHECK(waited[i].slot == flight[i].slot && waited[i].ph == flight[i].ph);
        CHECK(ring.busy == 0);
    }
    // the fillings of a ring's slots that a producer waits for at the end: each
    // slot's last one, with the parity of the phase that it completes
    for (int slots = 1; slots <= 8; ++slots)
        for (int filled = 0; filled < 40; ++filled) {
            std::vector<int> last(slots, -1);
            for (int q = 0; q < filled; ++q) last[q % slots] = q;
            int n = 0, ok = 0;
            tc::last_filled(filled, slots, [&](int s, unsigned parity) {
                ++n;
                ok += last[s] >= 0 && parity == (unsigned)(last[s] / slots % 2);
                last[s] = -1;
            });
            CHECK(n == (filled < slots ? filled : slots) && ok == n);
        }
    return 0;
}
"""


def test_ring_keeps_what_is_in_flight(tmp_path):
    src, exe = tmp_path / "ring.cpp", tmp_path / "ring"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout

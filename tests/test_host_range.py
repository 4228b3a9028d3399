"""Which host arrays a call that asked for nothing reads in place: only those in
one page-locked allocation or registration, mapped without a break.  Decided on
the host (sr_hostrange.h), against every layout of registrations over a small
address range."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include <cstdio>
#include <vector>
#include "sr_hostrange.h"
using namespace sr;
struct Reg { uintptr_t start; size_t size; uintptr_t device; bool mapped; };

int main() {
    const std::vector<std::vector<Reg>> layouts = {
        {},
        {{100, 50, 100, true}},
        {{100, 50, 9100, true}},                           // another device address
        {{100, 20, 100, true}, {140, 20, 140, true}},      // ordinary memory between two registrations
        {{100, 20, 100, true}, {120, 20, 120, true}},      // side by side
        {{100, 20, 100, true}, {120, 20, 500, true}},      // side by side, mapped apart
        {{100, 50, 0, false}},                             // not mapped for the device
    };
    long in = 0;
    for (const auto& regs : layouts) {
        auto query = [&](uintptr_t at) {
            HostRange h;
            for (const Reg& r : regs)
                if (at >= r.start && at - r.start < r.size)
                    h = HostRange{r.mapped, r.start, r.size, r.device + (at - r.start)};
            return h;
        };
        for (uintptr_t x = 90; x < 170; ++x)
            for (size_t n = 1; n <= 80; ++n) {
                bool want = false;
                for (const Reg& r : regs) want = want || (r.mapped && x >= r.start && x + n <= r.start + r.size);
                const bool got = one_page_locked_range(x, n, query);
                if (got != want) { std::printf("x %lu n %lu: %d, want %d\n", (unsigned long)x, (unsigned long)n, got, want); return 1; }
                in += got;
            }
    }
    // the top of the address space does not wrap around
    auto top = [](uintptr_t at) { return HostRange{true, UINTPTR_MAX - 9, 10, at}; };
    if (one_page_locked_range(UINTPTR_MAX - 4, 6, top) || !one_page_locked_range(UINTPTR_MAX - 4, 5, top)) return 2;
    std::printf("ok %ld\n", in);
}
"""


def test_only_one_registration_is_read_in_place(tmp_path):
    src, exe = tmp_path / "range.cpp", tmp_path / "range"
    src.write_text(PROGRAM)
    csrc = os.path.join(ROOT, "paper_2004_05371_gb300", "csrc")
    subprocess.run(["g++", "-std=c++17", "-Wall", "-I", csrc, str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
    assert int(r.stdout.split()[1]) > 0

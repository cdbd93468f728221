"""Which host buffers nkv_compress_host lets the device read where they lie: the decision alone, with the driver's answers made
up, compiled for the host (no device, no kernel)."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include "nkv_hostrange.h"
#include <stdio.h>
using nkv::HostRange;
struct Entry { uintptr_t start; size_t size; bool mapped; };
static const Entry kTable[] = {{0x10000, 0x4000, true}, {0x14000, 0x1000, true},   // two that touch
                               {0x20000, 0x1000, true}, {0x22000, 0x1000, true},   // two with a page between them
                               {0x30000, 0x8000, false}};                          // pinned, but not mapped
static bool driver(const void* p, HostRange* r) {
    const uintptr_t at = (uintptr_t)p;
    for (const Entry& e : kTable)
        if (at >= e.start && at - e.start < e.size) {
            *r = {e.mapped ? (const unsigned char*)p : nullptr, e.start, e.size};
            return true;
        }
    return false;
}
static int bad = 0;
static void check(uintptr_t p, size_t bytes, bool want) {
    const void* got = nkv::readable_in_place((const void*)p, bytes, driver);
    if ((got != nullptr) != want || (got && got != (const void*)p)) {
        printf("%#zx + %#zx: %p\n", (size_t)p, bytes, got);
        ++bad;
    }
}
int main() {
    check(0x10000, 0x4000, true);     // all of one
    check(0x11000, 0x3000, true);     // its end
    check(0x11000, 0x3001, false);    // one byte more, though another one follows
    check(0x10000, 0x5000, false);
    check(0x20000, 0x3000, false);    // first and last byte pinned, a page between them not
    check(0x20000, 0x1000, true);
    check(0x22800, 0x900, false);     // runs out of the last one
    check(0x30000, 0x100, false);     // no device address
    check(0x50000, 0x100, false);     // pageable
    check(0x10000, 0, false);
    check(0x10000, (size_t)-1, false);
    check(0, 16, false);
    // an allocation that the device sees at another address
    const void* got = nkv::readable_in_place((const void*)0x70010, 0xff0, [](const void*, HostRange* r) {
        *r = {(const unsigned char*)0x90010, 0x90000, 0x1000};
        return true;
    });
    if (got != (const void*)0x90010) ++bad;
    return bad;
}
"""


def test_only_one_allocation_or_registration_is_read_in_place(tmp_path):
    src, exe = tmp_path / "range.cpp", tmp_path / "range"
    src.write_text(PROGRAM)
    subprocess.check_call(["g++", "-std=c++17", "-Wall", "-I", os.path.join(ROOT, "paper_2605_26678_b200", "csrc"), str(src), "-o", str(exe)])
    done = subprocess.run([str(exe)], capture_output=True, text=True)
    assert done.returncode == 0, done.stdout

"""The device-pointer checks of a batch call on the CPU: csrc/pc_pointers.h
compiled with a made-up driver.  Whatever was asked before, a pointer is
accepted exactly when the driver calls it device memory -- host memory after
device memory, the ends of an allocation, more allocations than are held, an
allocation whose range is unknown, too long or empty."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SOURCE = r"""
#include <cstdio>
#include <random>
#include "pc_pointers.h"
struct Block { uintptr_t base; size_t size; bool device, ranged; size_t told; };
// sixteen device blocks, host blocks between them and beside them
static Block blocks[32];
static long queries;
static const Block* find(uintptr_t a) {
    for (const Block& b : blocks) if (a >= b.base && a - b.base < b.size) return &b;
    return nullptr;
}
struct Driver {
    static bool is_device(const void* p) { queries++; const Block* b = find((uintptr_t)p); return b && b->device; }
    static bool range(const void* p, uintptr_t* base, size_t* size) {
        const Block* b = find((uintptr_t)p);
        if (!b || !b->ranged) return false;
        *base = b->base; *size = b->told;
        return true;
    }
};
int main() {
    uintptr_t a = 0x10000;
    for (int i = 0; i < 32; i++) {
        const bool device = i % 2 == 0;
        blocks[i] = Block{a, (size_t)256 * (i + 1), device, i != 6, (size_t)256 * (i + 1)};
        a += blocks[i].size + (i % 3 == 0 ? 512 : 0);   // some blocks adjoin the next, some leave a gap
    }
    blocks[8].told += 64;    // said to reach into the host block beside it
    blocks[10].told = 0;
    std::mt19937 rng(1);
    for (int call = 0; call < 2000; call++) {
        pcurv::DevicePointers<Driver> ok;
        for (int k = 0; k < 60; k++) {
            const Block& b = blocks[rng() % 32];
            const uintptr_t at[] = {b.base, b.base + b.size - 1, b.base + b.size, b.base + b.size + 100, b.base - 1, b.base + rng() % b.size};
            const uintptr_t p = at[rng() % 6];
            const Block* in = find(p);
            if (ok((const void*)p) != (in && in->device)) { printf("call %d: %llx\n", call, (unsigned long long)p); return 1; }
        }
    }
    pcurv::DevicePointers<Driver> ok;   // four pointers of each of 256 frames in one allocation: two queries
    queries = 0;
    for (int i = 0; i < 1024; i++) if (!ok((const void*)(blocks[30].base + 4 * i % blocks[30].size))) return 2;
    if (queries != 2) { printf("%ld queries\n", queries); return 3; }
    if (ok((const void*)nullptr)) return 4;
    printf("ok\n");
    return 0;
}
"""


def test_accepts_what_the_driver_calls_device_memory(tmp_path):
    if not shutil.which("g++"):
        pytest.skip("needs g++")
    src = tmp_path / "pointers.cpp"
    src.write_text(SOURCE)
    exe = tmp_path / "pointers"
    subprocess.run(["g++", "-std=c++17", "-O2", "-I" + os.path.join(ROOT, "paper_1707_00385_gb300", "csrc"), str(src),
                    "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0 and r.stdout.strip() == "ok", (r.returncode, r.stdout)

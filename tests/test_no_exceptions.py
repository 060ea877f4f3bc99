"""Nothing is thrown across the C interface when host memory runs out: a small C++ program whose operator new fails on the
i-th allocation of a call, for every i that the call makes."""
import os
import subprocess

from paper_2110_14871_b200 import build as gbuild

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include <stdint.h>
#include <stdio.h>
#include <stdlib.h>
#include <new>
#include "gdws.h"

static long left = -1;          // allocations until one fails, -1: none does
static bool spent;
static void *get(size_t n)
{
    if (left == 0) { left = -1; spent = true; return nullptr; }
    if (left > 0) --left;
    return malloc(n ? n : 1);
}
void *operator new(size_t n) { void *p = get(n); if (!p) throw std::bad_alloc(); return p; }
void *operator new(size_t n, const std::nothrow_t &) noexcept { return get(n); }
void operator delete(void *p) noexcept { free(p); }
void operator delete(void *p, size_t) noexcept { free(p); }

int main()
{
    int32_t g[64];
    for (int &v : g) v = 5;
    for (int call = 0; call < 2; ++call)
        for (int i = 0; i < 200; ++i) {
            gdws_plan_t *plan = nullptr;
            int form = 0;
            gdws_status_t st = GDWS_OK;
            if (call == 1 && gdws_plan(64, 64, 3, 1, 1, g, &plan) != GDWS_OK) return 2;
            left = i;
            spent = false;
            try {
                st = call == 0 ? gdws_plan(64, 64, 3, 1, 1, g, &plan) : gdws_plan_form(plan, 512, 32, 32, &form);
            } catch (...) {
                printf("call %d, allocation %d: thrown\n", call, i);
                return 1;
            }
            const bool failed = spent;
            left = -1;
            if (st != GDWS_OK && st != GDWS_ERR_ALLOC) return 3;
            if (call == 1 && st == GDWS_OK && form != 3) return 4;
            if (!failed && st != GDWS_OK) return 5;
            gdws_destroy(plan);
            if (!failed) break;       // the call makes no more allocations
        }
    puts("ok");
    return 0;
}
"""


def test_out_of_host_memory_is_a_status(tmp_path):
    lib = gbuild.build_library()
    src, exe = tmp_path / "p.cpp", tmp_path / "p"
    src.write_text(PROGRAM)
    subprocess.check_call(["g++", "-std=c++17", "-rdynamic", "-I", os.path.join(ROOT, "include"), str(src), "-o", str(exe), lib,
                           "-Wl,-rpath," + os.path.dirname(lib)])
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0 and r.stdout == "ok\n", (r.returncode, r.stdout, r.stderr)

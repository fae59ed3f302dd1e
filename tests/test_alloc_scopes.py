"""The library's allocator against a device of 3 GiB that exists only on the
host (its runtime calls replaced at link time): memory that a set-up call of one
thread has released but still holds must be there for another thread's
allocation, memory that one thread is giving back for another that fails at the same
time, and no block may be freed that queued work could still use."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1806_11558_gb300", "csrc")

RUNTIME = r"""
#include <cstdio>
#include <cstdlib>
#include <map>
#include <mutex>
#include <unistd.h>
typedef unsigned long size_type;
std::mutex mu;
std::map<void *, size_type> live;
size_type in_use = 0, total = size_type(3) << 30;
int frees = 0, syncs = 0;
extern "C" {
int cudaMalloc(void **p, size_type n) {
    std::lock_guard<std::mutex> lk(mu);
    if (in_use + n > total) return 2;  // cudaErrorMemoryAllocation
    *p = malloc(16);
    live[*p] = n;
    in_use += n;
    return 0;
}
int cudaFree(void *p) {
    usleep(2000);
    std::lock_guard<std::mutex> lk(mu);
    if (!live.count(p)) { printf("freed twice\n"); exit(3); }
    in_use -= live[p];
    live.erase(p);  // the address is not given back: a second free would be seen
    ++frees;
    return 0;
}
int cudaMemGetInfo(size_type *f, size_type *t) { *f = total - in_use; *t = total; return 0; }
int cudaGetDevice(int *d) { *d = 0; return 0; }
int cudaSetDevice(int) { return 0; }
int cudaDeviceSynchronize() { std::lock_guard<std::mutex> lk(mu); ++syncs; return 0; }
int cudaGetLastError() { return 0; }
const char *cudaGetErrorString(int) { return "error"; }
void **__cudaRegisterFatBinary(void *) { static void *h = nullptr; return &h; }
void __cudaRegisterFatBinaryEnd(void **) {}
void __cudaUnregisterFatBinary(void **) {}
void __cudaRegisterFunction(void **, const char *, char *, const char *, int, void *, void *, void *, void *, int *) {}
void __cudaRegisterVar(void **, char *, char *, const char *, int, size_type, int, int) {}
}
"""

MAIN = r"""
#include <cstdio>
#include <future>
#include <thread>
#include "hm_internal.cuh"
extern size_t in_use;
extern int frees, syncs;
using namespace hm;
#define CHECK(c) do { if (!(c)) { printf("line %d: %s\n", __LINE__, #c); return 1; } } while (0)
constexpr size_t MiB = size_t(1) << 20;
int main() {
    std::promise<void> held, tried;
    bool again = false;
    std::thread setup([&] {
        AllocScope scope;
        {
            DBuf a, b;
            a.alloc(600 * MiB);
            b.alloc(300 * MiB);
        }  // released, kept by the scope
        held.set_value();
        tried.get_future().wait();
        DBuf c;
        c.alloc(200 * MiB);  // nothing of the list is left to take
        again = c.p != nullptr;
    });
    held.get_future().wait();
    CHECK(in_use == 900 * MiB);
    bool ok = true;
    const int s0 = syncs;
    {
        DBuf d;
        try { d.alloc(2500 * MiB); }
        catch (...) { ok = false; }
        if (ok && (in_use != 2500 * MiB || frees != 2 || syncs == s0)) ok = false;
        tried.set_value();
        setup.join();
    }
    CHECK(ok);
    CHECK(again);
    cache_trim();
    CHECK(in_use == 0);
    // two threads that need the cached memory at once
    for (int k = 0; k < 20; ++k) {
        DBuf fixed;
        fixed.alloc(1660 * MiB);
        {
            AllocScope scope;
            DBuf b[7];
            for (auto &x : b) x.alloc(109 * MiB);
        }
        CHECK(in_use == (1660 + 763) * MiB);
        bool had[2] = {false, false};
        std::promise<void> done[2];
        auto ask = [&](int i) {
            DBuf a;
            try { a.alloc(700 * MiB); had[i] = true; }
            catch (...) {}
            done[i].set_value();
            done[1 - i].get_future().wait();
        };
        std::thread one(ask, 0), two(ask, 1);
        one.join();
        two.join();
        CHECK(had[0] && had[1]);
        fixed.release();
        cache_trim();
    }
    CHECK(in_use == 0);
    // an allocation that cannot be had fails and leaves the scope usable
    {
        AllocScope scope;
        bool failed = false;
        { DBuf a; a.alloc(100 * MiB); }
        DBuf big;
        try { big.alloc(4000 * MiB); }
        catch (...) { failed = true; }
        CHECK(failed && in_use == 0);
        { DBuf a; a.alloc(100 * MiB); }
        DBuf b;
        b.alloc(100 * MiB);
        CHECK(in_use == 100 * MiB);  // the list's block
    }
    cache_trim();
    CHECK(in_use == 0);
    printf("ok\n");
    return 0;
}
"""


def test_released_memory_of_a_set_up_reaches_other_threads(tmp_path):
    nvcc = next((c for c in ("/usr/local/cuda/bin/nvcc", shutil.which("nvcc")) if c and os.path.exists(c)), None)
    if nvcc is None or shutil.which("g++") is None:
        pytest.skip("no nvcc")
    (tmp_path / "main.cu").write_text(MAIN)
    (tmp_path / "runtime.cpp").write_text(RUNTIME)
    cc = [nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-O1", "-std=c++17", "-I", CSRC, "-c"]
    jobs = [subprocess.Popen(cc + [src, "-o", str(tmp_path / out)]) for src, out in
            ((os.path.join(CSRC, "prims.cu"), "prims.o"), (str(tmp_path / "main.cu"), "main.o"))]
    jobs.append(subprocess.Popen(["g++", "-O1", "-c", str(tmp_path / "runtime.cpp"), "-o", str(tmp_path / "runtime.o")]))
    assert [j.wait() for j in jobs] == [0, 0, 0]
    exe = str(tmp_path / "scopes")
    subprocess.check_call(["g++", "-no-pie", str(tmp_path / "main.o"), str(tmp_path / "prims.o"),
                           str(tmp_path / "runtime.o"), "-o", exe, "-lpthread", "-Wl,--unresolved-symbols=ignore-all"])
    p = subprocess.run([exe], capture_output=True, text=True, timeout=60)
    assert p.returncode == 0 and p.stdout.strip() == "ok", (p.returncode, p.stdout, p.stderr)

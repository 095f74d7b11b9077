"""The opt-in to large shared memory holds per device and for the largest need,
whichever thread asks first (a fake of the two CUDA runtime calls, host only)."""
import glob
import os
import re
import subprocess

from paper_2601_00761_gb300 import build

FAKE = r"""
#include "smem_optin.cuh"
#include <cstdio>
#include <map>
#include <thread>
#include <vector>
static thread_local int device = 0;
static std::mutex mu;
static std::map<std::pair<const void *, int>, int> limit;      // what a launch could use
static int calls = 0;
cudaError_t cudaGetDevice(int *d) { *d = device; return cudaSuccess; }
cudaError_t cudaFuncSetAttribute(const void *k, cudaFuncAttribute, int v) {
    std::lock_guard<std::mutex> lk(mu);
    ++calls;
    if (v > 232448) return cudaErrorInvalidValue;
    limit[{k, device}] = v;
    return cudaSuccess;
}
#define EXPECT(c) if (!(c)) { printf("line %d: " #c "\n", __LINE__); return 1; }
int main() {
    static int kernel, many;
    static sre::SmemOptIn a;
    EXPECT(a.allow(&kernel, 70000) == cudaSuccess && limit[std::make_pair((const void *)&kernel, 0)] == 70000);
    EXPECT(a.allow(&kernel, 60000) == cudaSuccess && calls == 1);
    device = 1;                                                // a second device asks for itself
    EXPECT(a.allow(&kernel, 60000) == cudaSuccess && limit[std::make_pair((const void *)&kernel, 1)] == 60000);
    EXPECT(a.allow(&kernel, 90000) == cudaSuccess && limit[std::make_pair((const void *)&kernel, 1)] == 90000);
    EXPECT(limit[std::make_pair((const void *)&kernel, 0)] == 70000 && calls == 3);
    EXPECT(a.allow(&kernel, 300000) == cudaErrorInvalidValue);   // a refusal is reported and forgotten
    EXPECT(a.allow(&kernel, 90000) == cudaSuccess && calls == 4);
    device = 100;                                              // past the table: asked each time
    EXPECT(a.allow(&kernel, 50000) == cudaSuccess && limit[std::make_pair((const void *)&kernel, 100)] == 50000);
    for (int rep = 0; rep < 200; ++rep) {                      // different needs at once: the largest stays
        sre::SmemOptIn b;
        limit.clear();
        std::vector<std::thread> ts;
        bool bad[8] = {};
        for (int i = 0; i < 8; ++i)
            ts.emplace_back([&b, &bad, i] {
                device = 0;
                b.allow(&many, 50000 + 1000 * i);
                std::lock_guard<std::mutex> lk(mu);
                bad[i] = limit[std::make_pair((const void *)&many, 0)] < 50000 + 1000 * i;
            });
        for (auto &t : ts) t.join();
        for (bool x : bad) EXPECT(!x);
        EXPECT(limit[std::make_pair((const void *)&many, 0)] == 57000);
    }
    return 0;
}
"""


def test_per_device_and_largest(tmp_path):
    src, exe = tmp_path / "optin.cpp", tmp_path / "optin"
    src.write_text(FAKE)
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(build.nvcc()))), "include")
    r = subprocess.run(["g++", "-std=c++17", "-O1", "-pthread", "-I", build.CSRC, "-I", cuda, str(src), "-o", str(exe)],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-2000:]
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout


def test_every_launch_site_uses_it():
    """No other file asks for the attribute, and no launch remembers it in a plain static."""
    for f in glob.glob(os.path.join(build.CSRC, "*.cu*")):
        text = open(f).read()
        if os.path.basename(f) != "smem_optin.cuh":
            assert "cudaFuncSetAttribute" not in text, f
            assert not re.search(r"static (bool|size_t) (attr|done)", text), f

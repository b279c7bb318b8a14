"""CPU test of the batch's device lists (csrc/lbm_lists.h) against a fake of the CUDA calls: when an
allocation fails, every list keeps the memory and the contents that the launch counts belong to (a list
freed before its successor was there would leave the next step a null pointer), and nothing leaks."""
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1409_5929_gb300", "csrc")

FAKE = r"""
#pragma once
#include <stdlib.h>
#include <string.h>
typedef int cudaError_t;
typedef void* cudaStream_t;
enum { cudaSuccess = 0, cudaErrorInvalidValue = 1, cudaErrorMemoryAllocation = 2 };
enum { cudaMemcpyHostToDevice = 1 };
static int fake_allocs, fake_fail_at = -1, fake_live;
static cudaError_t cudaMalloc(void** p, size_t n) {
    if (fake_allocs++ == fake_fail_at) return cudaErrorMemoryAllocation;
    *p = malloc(n);
    ++fake_live;
    return cudaSuccess;
}
static cudaError_t cudaFree(void* p) { if (p) --fake_live; free(p); return cudaSuccess; }
static cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, int, cudaStream_t) { memcpy(d, s, n); return cudaSuccess; }
static cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
static cudaError_t cudaGetLastError(void) { return cudaSuccess; }
"""

PROGRAM = r"""
#include <stdio.h>
#include <vector>
#include "lbm_lists.h"
using namespace lbm;
static int check(bool ok, const char* what) { if (!ok) printf("%s\n", what); return ok ? 0 : 1; }
int main() {
    int bad = 0;
    for (int fail = 0; fail < 4; ++fail) {
        DeviceList l[3];
        std::vector<int> a(5, 1), b(7, 2), c, a2(50, 3), b2(3, 4), c2(60, 5);
        const ListUpload first[] = {{&l[0], a.data(), a.size() * 4}, {&l[1], b.data(), b.size() * 4}, {&l[2], c.data(), 0}};
        bad += check(upload_lists(first, 3, nullptr) == cudaSuccess && fake_live == 2 && !l[2].dev, "first");
        void* const dev[] = {l[0].dev, l[1].dev};
        fake_allocs = 0;
        fake_fail_at = fail < 2 ? fail : -1;   // the first or second list that has to grow, or none
        const ListUpload next[] = {{&l[0], a2.data(), 200}, {&l[1], b2.data(), 12}, {&l[2], c2.data(), 240}};
        const cudaError_t e = upload_lists(next, 3, nullptr);
        if (fail < 2) {
            bad += check(e == cudaErrorMemoryAllocation && fake_live == 2, "failure, nothing leaks");
            bad += check(l[0].dev == dev[0] && l[1].dev == dev[1] && !l[2].dev, "memory kept");
            bad += check(l[0].cap == 20 && l[1].cap == 28 && l[2].cap == 0, "capacities kept");
            bad += check(!memcmp(l[0].dev, a.data(), 20) && !memcmp(l[1].dev, b.data(), 28), "contents kept");
            fake_fail_at = -1;
            bad += check(upload_lists(next, 3, nullptr) == cudaSuccess, "later success");
        } else {
            bad += check(e == cudaSuccess, "success");
        }
        bad += check(l[0].cap == 200 && l[1].cap == 28 && l[2].cap == 240 && l[1].dev == dev[1] && fake_live == 3, "grown");
        bad += check(!memcmp(l[0].dev, a2.data(), 200) && !memcmp(l[1].dev, b2.data(), 12) && !memcmp(l[2].dev, c2.data(), 240),
                     "contents");
        for (auto& x : l) cudaFree(x.dev);
        bad += check(fake_live == 0, "freed");
    }
    return bad;
}
"""


def test_lists_survive_a_failed_allocation(tmp_path):
    (tmp_path / "cuda_runtime.h").write_text(FAKE)
    (tmp_path / "main.cpp").write_text(PROGRAM)
    exe = str(tmp_path / "lists")
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", str(tmp_path), "-I", CSRC, "-o", exe, str(tmp_path / "main.cpp")],
                   check=True)
    r = subprocess.run([exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout


def test_batch_replaces_its_lists_together():
    """lbm.cu allocates none of those lists elsewhere, and sets its counts after the upload."""
    src = open(os.path.join(CSRC, "lbm.cu")).read()
    body = src[src.index("static int batch_rebuild"):]
    body = body[:body.index("\n}\n")]
    assert body.count("upload_lists(") == 1 and "cudaMalloc" not in body and "cudaFree" not in body
    assert min(body.index(f"b->{n} =") for n in ("ntiles", "nstiles", "step16", "nactive")) > body.index("upload_lists(")

"""Copies of results into the caller's memory, compiled from the engine's header
against a stand-in for the CUDA calls: no GPU."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC, INCLUDE = os.path.join(ROOT, "paper_2207_05535_gb300", "csrc"), os.path.join(ROOT, "include")

FAKE = r"""
#pragma once
#include <cstddef>
#include <cstring>
#define __host__
#define __device__
enum cudaError_t { cudaSuccess = 0, cudaErrorInvalidValue = 1, cudaErrorUnknown = 999 };
enum cudaMemoryType { cudaMemoryTypeUnregistered = 0, cudaMemoryTypeHost = 1, cudaMemoryTypeManaged = 3 };
enum cudaMemcpyKind { cudaMemcpyDeviceToHost = 2 };
struct cudaPointerAttributes { cudaMemoryType type; };
typedef void *cudaStream_t;
static cudaError_t fake_attr = cudaSuccess, fake_last = cudaSuccess, fake_copy = cudaSuccess;
static cudaMemoryType fake_type = cudaMemoryTypeUnregistered;
static size_t fake_copied = 0;
static cudaError_t cudaPointerGetAttributes(cudaPointerAttributes *a, const void *)
{
    a->type = fake_type;
    if (fake_attr) fake_last = fake_attr;
    return fake_attr;
}
static cudaError_t cudaGetLastError()
{
    const cudaError_t e = fake_last;
    fake_last = cudaSuccess;
    return e;
}
static cudaError_t cudaMemcpyAsync(void *, const void *, size_t n, cudaMemcpyKind, cudaStream_t)
{
    fake_copied += n;
    return fake_copy;
}
"""

MAIN = r"""
#include <cstdio>
#include <vector>
#include <sys/mman.h>
#include <cuda_runtime.h>
#include "pa_internal.cuh"
static size_t resident(void *p, size_t n)
{
    const size_t page = (size_t)sysconf(_SC_PAGESIZE);
    std::vector<unsigned char> v(n / page);
    if (mincore(p, n, v.data())) return (size_t)-1;
    size_t k = 0;
    for (unsigned char c : v) k += c & 1;
    return k;
}
static char *map(size_t n, int prot)
{
    return static_cast<char *>(mmap(nullptr, n, prot, MAP_PRIVATE | MAP_ANONYMOUS, -1, 0));
}
#define CHECK(x) if (!(x)) { std::printf("line %d: %s\n", __LINE__, #x); return 1; }
int main()
{
    const size_t n = 4u << 20, page = (size_t)sysconf(_SC_PAGESIZE);
    @
    return 0;
}
"""

CASES = {
    # a buffer the host cannot write, and one shorter than stated: the copy's to refuse, not a fault here
    "read_only": """char *p = map(n, PROT_READ);
    CHECK(pa::copy_out(p, nullptr, n, nullptr) == cudaSuccess && fake_copied == n);""",
    "none": """char *p = map(n, PROT_NONE); fake_copy = cudaErrorInvalidValue;
    CHECK(pa::copy_out(p, nullptr, n, nullptr) == cudaErrorInvalidValue);""",
    "short": """char *p = map(2 * n, PROT_READ | PROT_WRITE);
    munmap(p + n / 2, 2 * n - n / 2);
    CHECK(pa::copy_out(p, nullptr, n, nullptr) == cudaSuccess && fake_copied == n);""",
    # what the buffer holds stays until the copy overwrites it
    "kept": """char *p = map(n, PROT_READ | PROT_WRITE); std::memset(p, 7, n);
    pa::copy_out(p + 3, nullptr, n - 9, nullptr);
    for (size_t k = 0; k < n; ++k) CHECK(p[k] == 7);""",
    # fresh pages are there before the copy, at both ends of an unaligned range
    "fresh": """char *p = map(n, PROT_READ | PROT_WRITE);
    CHECK(resident(p, n) == 0);
    pa::copy_out(p + page - 1, nullptr, n - 2 * page + 2, nullptr);
    CHECK(resident(p, n) == n / page);""",
    "pinned": """char *p = map(n, PROT_READ | PROT_WRITE); fake_type = cudaMemoryTypeHost;
    pa::copy_out(p, nullptr, n, nullptr);
    CHECK(resident(p, n) == 0 && fake_copied == n);""",
    # a query that fails leaves no error behind for the next check of unrelated work
    "query_fails": """char *p = map(n, PROT_READ | PROT_WRITE); fake_attr = cudaErrorUnknown;
    CHECK(pa::copy_out(p, nullptr, n, nullptr) == cudaSuccess && fake_copied == n && resident(p, n) == 0);
    CHECK(cudaGetLastError() == cudaSuccess);""",
    "small": """char *p = map(n, PROT_READ | PROT_WRITE);
    pa::copy_out(p, nullptr, (1u << 20) - 1, nullptr);
    CHECK(resident(p, n) == 0);""",
}


def _run(tmp_path, body):
    (tmp_path / "cuda_runtime.h").write_text(FAKE)
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(MAIN.replace("@", body))
    subprocess.run(["g++", "-std=c++17", "-I", str(tmp_path), "-I", CSRC, "-I", INCLUDE, str(src), "-o", str(exe)], check=True)
    res = subprocess.run([str(exe)], capture_output=True, text=True)
    assert res.returncode == 0, (res.returncode, res.stdout)


@pytest.mark.parametrize("case", sorted(CASES))
def test_pages_of_results(tmp_path, case):
    _run(tmp_path, CASES[case])

"""A device copy that fails half way leaves nothing behind (host code of pc_digits.h with the
runtime's allocation and copy replaced): a later call would take the pointer for the copy."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CUDA = "/usr/local/cuda/include"

SOURCE = r"""
#include <cuda_runtime.h>
#include <cstdlib>
static int live = 0, malloc_fails = 0, copy_fails = 0;
static cudaError_t fake_malloc(void **p, size_t n) {
  if (malloc_fails) return cudaErrorMemoryAllocation;
  *p = std::malloc(n);
  live++;
  return cudaSuccess;
}
static cudaError_t fake_copy(void *d, const void *s, size_t n, cudaMemcpyKind) {
  if (copy_fails) return cudaErrorInvalidValue;
  __builtin_memcpy(d, s, n);
  return cudaSuccess;
}
static cudaError_t fake_free(void *p) {
  if (p) live--;
  std::free(p);
  return cudaSuccess;
}
#define cudaMalloc fake_malloc
#define cudaMemcpy fake_copy
#define cudaFree fake_free
#include "pc_digits.h"
int main() {
  const std::vector<int> v{1, 2, 3};
  int *d = nullptr;
  malloc_fails = 1;
  if (pcx::upload(&d, v) != cudaErrorMemoryAllocation || d || live) return 1;
  malloc_fails = 0;
  copy_fails = 1;
  if (pcx::upload(&d, v) != cudaErrorInvalidValue || d || live) return 2;
  copy_fails = 0;
  if (pcx::upload(&d, v) != cudaSuccess || !d || d[2] != 3 || live != 1) return 3;
  return 0;
}
"""


def test_failed_upload_leaves_no_pointer(tmp_path):
    if not shutil.which("g++") or not os.path.exists(os.path.join(CUDA, "cuda_runtime.h")):
        pytest.skip("needs g++ and the CUDA headers")
    src, exe = tmp_path / "upload.cpp", tmp_path / "upload"
    src.write_text(SOURCE)
    r = subprocess.run(["g++", "-std=c++17", "-I", CUDA, "-I", os.path.join(ROOT, "include"), "-I",
                        os.path.join(ROOT, "paper_2301_03989_gb300", "csrc"), str(src), "-o", str(exe)],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    assert subprocess.run([str(exe)]).returncode == 0

"""A bounded wait that nothing ends gives up, leaves the context usable, and is
reported as an error by the handle's next product.  The program below includes
the library's own wait and handle definitions."""

import os
import subprocess

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SOURCE = r"""
#include <chrono>
#include <cstdio>
#include <cstring>
#include <vector>
#include "bounded_wait.cuh"
#include "internal.cuh"

__global__ void wait_once(int arrive, int *fault, int *got) {
  __shared__ __align__(8) unsigned long long bar;
  const unsigned bar32 = static_cast<unsigned>(__cvta_generic_to_shared(&bar));
  if (threadIdx.x == 0) asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(bar32) : "memory");
  __syncthreads();
  if (arrive && threadIdx.x == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar32) : "memory");
  got[blockIdx.x * blockDim.x + threadIdx.x] = sphynx::bounded_wait_or_fault(bar32, fault) ? 1 : 0;
}

#define CHECK(c) do { if (!(c)) { printf("line %d: %s (%s)\n", __LINE__, #c, sphynx_last_error()); return 1; } } while (0)

int main() {
  const int n = 40, ld = 4;
  std::vector<int64_t> rp{0};
  std::vector<int32_t> col;
  for (int i = 0; i < n; ++i) {
    if (i > 0) col.push_back(i - 1);
    if (i + 1 < n) col.push_back(i + 1);
    rp.push_back(static_cast<int64_t>(col.size()));
  }
  sphynx_handle g = nullptr;
  CHECK(sphynx_create(rp.data(), col.data(), nullptr, nullptr, n, rp[n], SPHYNX_HOST_PTRS, nullptr, &g) == SPHYNX_OK);
  int *got;
  float *x, *y;
  CHECK(cudaMalloc(&got, 128 * sizeof(int)) == cudaSuccess);
  CHECK(cudaMalloc(&x, n * ld * sizeof(float)) == cudaSuccess);
  CHECK(cudaMalloc(&y, n * ld * sizeof(float)) == cudaSuccess);
  std::vector<float> ones(n * ld, 1.f);
  CHECK(cudaMemcpy(x, ones.data(), ones.size() * 4, cudaMemcpyHostToDevice) == cudaSuccess);
  std::vector<int> h(128);
  // an arrival in time: no fault
  wait_once<<<2, 64>>>(1, g->fault(), got);
  CHECK(cudaMemcpy(h.data(), got, 128 * 4, cudaMemcpyDeviceToHost) == cudaSuccess);
  for (int v : h) CHECK(v == 1);
  CHECK(*g->fault() == 0);
  // none: both waits run out
  const auto t0 = std::chrono::steady_clock::now();
  wait_once<<<2, 64>>>(0, g->fault(), got);
  CHECK(cudaMemcpy(h.data(), got, 128 * 4, cudaMemcpyDeviceToHost) == cudaSuccess);
  const double s = std::chrono::duration<double>(std::chrono::steady_clock::now() - t0).count();
  for (int v : h) CHECK(v == 0);
  CHECK(*g->fault() == 1);
  // reported once, by the next product; the one after it works
  CHECK(sphynx_laplacian_apply(g, SPHYNX_COMBINATORIAL, SPHYNX_DT_F32, x, ld, y, ld, ld) == SPHYNX_ERR_CUDA);
  CHECK(strstr(sphynx_last_error(), "did not arrive") != nullptr);
  CHECK(sphynx_laplacian_apply(g, SPHYNX_COMBINATORIAL, SPHYNX_DT_F32, x, ld, y, ld, ld) == SPHYNX_OK);
  std::vector<float> out(n * ld, 7.f);
  CHECK(cudaMemcpy(out.data(), y, out.size() * 4, cudaMemcpyDeviceToHost) == cudaSuccess);
  for (float v : out) CHECK(v == 0.f);
  sphynx_destroy(g);
  printf("ok %.2f\n", s);
  return 0;
}
"""


def test_a_wait_that_nothing_ends_is_reported(tmp_path):
    from paper_2105_00578_gb300 import build as B
    src, exe = tmp_path / "wait.cu", tmp_path / "wait"
    src.write_text(SOURCE)
    subprocess.run([B.nvcc(), *B.ARCH, *B.NVCC_FLAGS, "-I", B.CSRC, str(src), "-o", str(exe), "-L", B.OUT_DIR,
                    "-lsphynx", "-Xlinker", "-rpath=" + B.OUT_DIR], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout + r.stderr
    # two waits of about a second each, the blocks at the same time
    assert r.stdout.startswith("ok") and float(r.stdout.split()[1]) < 20.0, r.stdout

"""What sw_align_pair makes of the status word its kernel leaves (no GPU): the
host code of pair.cu, compiled against a stand-in of the CUDA runtime whose
kernel writes a score and a status.  Only status 0 may return the score."""

import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2412_08308_gb300", "csrc")
CUDA_INCLUDE = "/usr/local/cuda/include"

STAND_IN = r"""
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include "internal.h"
#include "host_pool.h"
#include "../../include/swgb.h"

static int32_t g_status = 0;

namespace swgb {
int set_last_error(int code, const char *) { return code; }
void clear_last_error() {}
cudaError_t pool_alloc(void **p, size_t bytes, cudaStream_t) { *p = calloc(bytes, 1); return cudaSuccess; }
int pair_max_warps() { return 8; }
int pair_slot_bytes(int R) { return (R + 3) / 4 * 4; }
size_t pair_smem_bytes(int pbuf_bytes, int warps) { return (size_t)warps * (pbuf_bytes + 1280); }
int pair_max_ctas_per_sm(int, int, int, size_t) { return 1; }
cudaError_t launch_build_profiles(const uint8_t *, const QDesc *, int, const int8_t *, int32_t, uint8_t *, cudaStream_t) {
  return cudaSuccess;
}
cudaError_t launch_pair(const PairBandArgs &a, int, int, int, size_t, cudaStream_t) {
  *a.best = 77;
  *a.status = g_status;
  return cudaSuccess;
}
}  // namespace swgb

extern "C" {
const char *cudaGetErrorString(cudaError_t) { return ""; }
cudaError_t cudaGetDevice(int *d) { *d = 0; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr, int) { *v = 152; return cudaSuccess; }
cudaError_t cudaMemGetInfo(size_t *f, size_t *t) { *f = *t = (size_t)1 << 40; return cudaSuccess; }
cudaError_t cudaMemcpyAsync(void *d, const void *s, size_t n, cudaMemcpyKind, cudaStream_t) {
  memcpy(d, s, n);
  return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void *d, int v, size_t n, cudaStream_t) { memset(d, v, n); return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaFreeAsync(void *p, cudaStream_t) { free(p); return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t *e) { *e = nullptr; return cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float *ms, cudaEvent_t, cudaEvent_t) { *ms = 0.f; return cudaSuccess; }
}

int main(int, char **argv) {
  g_status = atoi(argv[1]);
  const uint8_t q[40] = {}, t[50] = {};
  const int8_t sub[400] = {1};
  int32_t score = -1;
  const int rc = sw_align_pair(q, 40, t, 50, sub, 5, 2, nullptr, &score, nullptr, nullptr);
  printf("%d %d\n", rc, score);
  return 0;
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    d = tmp_path_factory.mktemp("pair")
    src, exe = str(d / "stand_in.cpp"), str(d / "pair_status")
    with open(src, "w") as f:
        f.write(STAND_IN.replace('"../../include/swgb.h"', '"swgb.h"'))
    subprocess.run(["g++", "-std=c++17", "-w", "-I", CSRC, "-I", os.path.join(ROOT, "include"), "-I", CUDA_INCLUDE,
                    "-x", "c++", os.path.join(CSRC, "pair.cu"), src, "-o", exe], check=True)
    return exe


@pytest.mark.parametrize("status,code,score", [(0, 0, 77), (4, 4, 0), (100, 3, 0), (101, 3, 0)])
def test_status_word(program, status, code, score):
    out = subprocess.run([program, str(status)], check=True, capture_output=True, text=True).stdout.split()
    assert [int(x) for x in out] == [code, score]

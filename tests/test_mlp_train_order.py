"""Host side of cr_mlp_train against a stand-in for the CUDA runtime whose stream
runs nothing before it has to: every copy reads its host memory as late as the
runtime may (at the next wait for it).  The sample orders and bias corrections that
the epochs then see must be those of the seed.  It also sees the kernel's shared
memory limit and each launch's need.
"""
import json
import os
import subprocess
import sys

import numpy as np
import pytest

from tests.test_gpu_mlp_train import _orders

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

FAKE = r"""
#include <cuda_runtime.h>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <deque>
#include <functional>
static std::deque<std::pair<std::function<void()>, void*>> queue_;   // work of the stream, and the event behind it
static void drain(void* until) {
  bool in = until == nullptr;
  for (auto& q : queue_) in = in || q.second == until;
  if (!in) return;
  while (!queue_.empty()) {
    auto q = queue_.front();
    queue_.pop_front();
    if (q.first) q.first();
    if (until && q.second == until) return;
  }
}
extern "C" {
cudaError_t cudaMalloc(void** p, size_t n) { *p = malloc(n); return cudaSuccess; }
cudaError_t cudaFree(void* p) { drain(nullptr); free(p); return cudaSuccess; }
cudaError_t cudaMemsetAsync(void* p, int v, size_t n, cudaStream_t) {
  queue_.push_back({[=] { memset(p, v, n); }, nullptr});
  return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind, cudaStream_t) {
  queue_.push_back({[=] { memcpy(d, s, n); }, nullptr});
  return cudaSuccess;
}
cudaError_t cudaStreamSynchronize(cudaStream_t) { drain(nullptr); return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { *e = (cudaEvent_t)malloc(8); return cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t e) { free(e); return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t) { queue_.push_back({nullptr, (void*)e}); return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t e) { drain((void*)e); return cudaSuccess; }
cudaError_t cudaFuncSetAttribute(const void*, cudaFuncAttribute, int v) {
  printf("{\"limit\": %d}\n", v);
  return cudaSuccess;
}
// the epoch kernel: (prm, mom, var, X, T, idx, n, batch, corr, lr, loss)
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void*, void** a) {
  const int* idx = *(const int**)a[5];
  const int n = *(int*)a[6], batch = *(int*)a[7];
  const float2* corr = *(const float2**)a[8];
  float* loss = *(float**)a[10];
  const size_t smem = c->dynamicSmemBytes;
  queue_.push_back({[=] {
    printf("{\"smem\": %zu, \"order\": [", smem);
    for (int i = 0; i < n; ++i) printf("%s%d", i ? "," : "", idx[i]);
    printf("], \"corr\": [");
    for (int k = 0; k * (long long)batch < n; ++k) printf("%s%.9g", k ? "," : "", corr[k].x);
    printf("]}\n");
    *loss = 0.0f;
  }, nullptr});
  return cudaSuccess;
}
}
"""

CALL = r"""
import ctypes, sys
lib, n, batch, epochs, seed = ctypes.CDLL(sys.argv[1]), *(int(a) for a in sys.argv[2:])
f = lib.cr_mlp_train
f.argtypes = [ctypes.c_int] + [ctypes.c_void_p] * 3 + [ctypes.c_int] * 3 + [ctypes.c_float, ctypes.c_ulonglong,
                                                                           ctypes.c_void_p, ctypes.c_void_p]
mem = (ctypes.c_float * 4096)()
assert f(16, mem, mem, mem, n, batch, epochs, 1e-3, seed, None, None) == 0
"""


@pytest.fixture(scope="module")
def call(tmp_path_factory):
    from paper_2502_07517_gb300 import build
    d = tmp_path_factory.mktemp("fake")
    src, fake = d / "fake.cpp", d / "libfake.so"
    src.write_text(FAKE)
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    subprocess.run(["g++", "-O1", "-std=c++17", "-shared", "-fPIC", "-I", os.path.join(cuda, "include"), str(src), "-o",
                    str(fake)], check=True)
    lib = build.build()

    def run(*args):
        out = subprocess.run([sys.executable, "-c", CALL, lib] + [str(a) for a in args], capture_output=True, text=True,
                             env=dict(os.environ, LD_PRELOAD=str(fake)))
        assert out.returncode == 0, out.stderr
        return [json.loads(line) for line in out.stdout.splitlines()]
    return run


@pytest.mark.parametrize("n,batch,epochs", [(700, 64, 1), (700, 64, 2), (700, 64, 3), (700, 2000, 6), (129, 1, 5)])
def test_every_epoch_sees_its_own_order(call, n, batch, epochs):
    seen = [e for e in call(n, batch, epochs, 11) if "order" in e]
    assert len(seen) == epochs
    step = 0
    for e, perm in zip(seen, _orders(n, epochs, 11)):
        np.testing.assert_array_equal(e["order"], perm)
        want = [1.0 - 0.9 ** (step + 1 + k) for k in range(len(e["corr"]))]
        np.testing.assert_allclose(e["corr"], want, rtol=1e-5)
        step += len(want)


def test_shared_memory_limit_is_the_same_for_every_call(call):
    """The limit is a property of the kernel: a call that set a lower one between
    another thread's limit and launch would make that launch fail."""
    limits, needs = set(), []
    for n, batch in ((10, 1), (700, 64), (700, 700), (3072, 3072)):
        out = call(n, batch, 1, 3)
        limits |= {e["limit"] for e in out if "limit" in e}
        needs += [e["smem"] for e in out if "smem" in e]
    assert len(limits) == 1 and max(needs) <= min(limits)

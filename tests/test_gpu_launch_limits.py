"""Calls of different sizes from two host threads.

The shared-memory limit of a kernel is process-wide.  A launcher that set it to
each call's own size could have it lowered by another thread between setting it
and launching, and the launch would be refused.  Two native threads (Python's
would take turns) call one entry point at its smallest and at a large size, all
on one stream; every call has to be accepted."""
import ctypes
import os
import subprocess

import pytest
import torch

from gpu_common import api

pytestmark = pytest.mark.gpu

CALLS = 4000

SOURCE = r"""
#include <thread>
#include "soma_api.h"

struct Args {
  float *params, *m, *v, *coef, *losses;
  const unsigned char* bytes;
  void* ws;
  unsigned long long ws_bytes;
  int E, H, n, B;
};

static int call(int kind, const Args& a) {
  const soma_dims d = {256, a.E, a.H};
  if (kind == 0) return soma_spsa_update(a.params, 1, d, a.n, 1e-6f, 3, 0, a.coef, nullptr);
  if (kind == 1) {
    const uint64_t step = 0;
    const soma_adam_config c = {1e-6f, 0.9f, 0.999f, 1e-8f, 0.f, 1};
    return soma_adam_update(a.params, a.m, a.v, 1, d, a.n, SOMA_PROBE_SPARSE, 3, &step, 1, a.coef, c,
                            nullptr);
  }
  return soma_spsa_estimate(a.params, 1, d, a.n, SOMA_PROBE_DENSE, 1e-3f, 3, 0, a.bytes, a.B, 1,
                            a.losses, a.coef, a.ws, a.ws_bytes, nullptr);
}

// calls refused by either thread
extern "C" int hammer(int kind, int calls, const Args* args) {
  int refused[2] = {0, 0};
  auto loop = [&](int j) {
    for (int k = 0; k < calls; ++k) {
      refused[j] += call(kind, args[j]) != SOMA_OK;
      if (k % 256 == 255) soma_get_status(nullptr);  // waits for the stream
    }
  };
  std::thread t(loop, 1);
  loop(0);
  t.join();
  soma_get_status(nullptr);
  return refused[0] + refused[1];
}
"""


class Args(ctypes.Structure):
    _fields_ = [(k, ctypes.c_void_p) for k in ("params", "m", "v", "coef", "losses", "bytes", "ws")]
    _fields_ += [("ws_bytes", ctypes.c_ulonglong)]
    _fields_ += [(k, ctypes.c_int) for k in ("E", "H", "n", "B")]


@pytest.fixture(scope="module")
def hammer(tmp_path_factory):
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    lib = api().LIB_PATH
    d = tmp_path_factory.mktemp("hammer")
    (d / "hammer.cpp").write_text(SOURCE)
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-pthread",
                    f"-I{root}/include", str(d / "hammer.cpp"), lib,
                    f"-Wl,-rpath,{os.path.dirname(lib)}", "-o", str(d / "hammer.so")], check=True)
    return ctypes.CDLL(str(d / "hammer.so")).hammer


@pytest.mark.parametrize("kind,small,large", [
    (0, (1, 1, 8, 1), (1, 1, 12 * 1024, 1)),
    (1, (1, 1, 8, 1), (1, 1, 12 * 1024, 1)),
    (2, (1, 1, 1, 1), (32, 64, 1, 16)),     # the resident kernel
    (2, (1, 65, 1, 1), (1, 65, 1, 32)),     # the persistent kernel
])
def test_sizes_from_two_threads(hammer, kind, small, large):
    a = api()
    keep, args = [], (Args * 2)()
    for j, (E, H, n, B) in enumerate((small, large)):
        P = a.param_count(E, H)
        t = dict(params=torch.zeros(P), m=torch.zeros(P), v=torch.zeros(P),
                 coef=torch.full((n,), 1e-6), losses=torch.zeros(2 * n),
                 bytes=torch.zeros(B, 2, dtype=torch.uint8),
                 ws=torch.zeros(a.workspace_bytes(E, H, 1, n, B, 1), dtype=torch.uint8))
        t = {k: x.cuda() for k, x in t.items()}
        keep.append(t)
        args[j] = Args(**{k: x.data_ptr() for k, x in t.items()}, ws_bytes=t["ws"].numel(),
                       E=E, H=H, n=n, B=B)
    torch.cuda.synchronize()
    assert hammer(kind, CALLS, args) == 0
    assert a.get_status() == 0

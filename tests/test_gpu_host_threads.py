"""Calls of one entry point from two host threads, each on its own stream, with shapes whose
kernels need different amounts of shared memory: every call succeeds and the results are those
of the same calls made alone.  (The threads are native ones: interpreter threads hand over
too seldom for two calls to meet.)"""
import ctypes as C

import numpy as np
import pytest
import torch

from host_probe import compile_probe
from paper_2102_02440_gb300 import compass as K
from paper_2102_02440_gb300 import pipeline as P
from test_gpu_enumerate import _connected, _graph

pytestmark = pytest.mark.gpu

CALLS = 20_000

SOURCE = r"""
#include <atomic>
#include <thread>
#include "compass.h"

// Two threads make `calls` calls each, at once; the number that failed.
template <typename F>
static int both(int calls, F&& call) {
  std::atomic<int> failed{0}, ready{0};
  auto work = [&](int k) {
    cudaStream_t st;
    if (cudaStreamCreate(&st) != cudaSuccess) {
      failed += calls;
      ready++;
      return;
    }
    ready++;
    while (ready < 2) std::this_thread::yield();
    for (int i = 0; i < calls; i++) {
      if (call(k, st) != CMP_OK) failed++;
      if (i % 256 == 255) cudaStreamSynchronize(st);
    }
    cudaStreamSynchronize(st);
    cudaStreamDestroy(st);
  };
  std::thread a(work, 0), b(work, 1);
  a.join();
  b.join();
  return failed;
}

struct Presort { const int32_t* c; int64_t rows; int32_t w; uint32_t* abs; int32_t* perm; };
struct Enumerate {
  const void *plan, *plan_dev;
  const double* est;
  cmp_enum_cfg cfg;
  void* ws;
  size_t ws_bytes;
  int32_t* order;
  double* cost;
  int64_t* stats;
  int32_t* status;
};
extern "C" int presorts(decltype(&cmp_presort) f, const Presort* j, int calls) {
  return both(calls, [&](int k, cudaStream_t st) { return f(j[k].c, j[k].rows, j[k].w, j[k].abs, j[k].perm, nullptr, 0, st); });
}
extern "C" int enumerations(decltype(&cmp_enumerate) f, const Enumerate* j, int calls) {
  return both(calls, [&](int k, cudaStream_t st) {
    const Enumerate& e = j[k];
    return f(e.plan, e.plan_dev, e.est, &e.cfg, e.ws, e.ws_bytes, e.order, e.cost, e.stats, e.status, st);
  });
}
"""


class Presort(C.Structure):
    _fields_ = [("c", C.c_void_p), ("rows", C.c_int64), ("w", C.c_int32), ("abs", C.c_void_p), ("perm", C.c_void_p)]


class Enumerate(C.Structure):
    _fields_ = [("plan", C.c_void_p), ("plan_dev", C.c_void_p), ("est", C.c_void_p), ("cfg", K.cmp_enum_cfg),
                ("ws", C.c_void_p), ("ws_bytes", C.c_size_t), ("order", C.c_void_p), ("cost", C.c_void_p),
                ("stats", C.c_void_p), ("status", C.c_void_p)]


@pytest.fixture(scope="module")
def probe(tmp_path_factory):
    return compile_probe(tmp_path_factory.mktemp("probe"), SOURCE)


def test_presort_widths_side_by_side(probe):
    rng = np.random.default_rng(1)
    args, jobs = (Presort * 2)(), []
    for k, w in enumerate((64, 8192)):  # 2 KB and 70 KB, of one kernel
        c = torch.from_numpy(rng.integers(-50, 50, (3, w)).astype(np.int32)).cuda()
        a, p = torch.empty_like(c), torch.empty_like(c)
        K.cmp_presort(c.data_ptr(), 3, w, a.data_ptr(), p.data_ptr(), 0, 0, K.stream_handle())
        torch.cuda.synchronize()
        jobs.append((c, a, p, a.clone(), p.clone()))
        a.zero_()
        p.zero_()
        args[k] = Presort(c.data_ptr(), 3, w, a.data_ptr(), p.data_ptr())
    torch.cuda.synchronize()
    failed = probe.presorts(C.cast(K.lib().cmp_presort, C.c_void_p), args, CALLS)
    assert failed == 0, failed
    torch.cuda.synchronize()
    for _, a, p, ra, rp in jobs:
        assert torch.equal(a, ra) and torch.equal(p, rp)


def test_enumerations_of_small_and_large_graphs_side_by_side(probe):
    rng = np.random.default_rng(2)
    args, jobs = (Enumerate * 2)(), []
    for k, n in enumerate((4, 40)):
        eu, ev = list(range(n - 1)), list(range(1, n))
        masks = _connected(n, eu, ev) if n < 16 else [((1 << m) - 1) << i for m in range(2, n + 1) for i in range(n - m + 1)]
        est = torch.tensor([float(bin(m).count("1") * 100 + rng.integers(0, 3)) for m in masks], dtype=torch.float64,
                           device="cuda")
        cfg = K.cmp_enum_cfg.make(max_plans=1, max_nodes=200)
        en = P.Enumerator([_graph(n, eu, ev, [int(x) for x in rng.integers(1, 1000, n)])], [0] * len(masks), masks, cfg=cfg)
        en.run(est)
        torch.cuda.synchronize()
        jobs.append((en, est, en.plans()))
        en.cost.zero_()
        args[k] = Enumerate(en.plan_host.ctypes.data, en.plan_dev.data_ptr(), est.data_ptr(), cfg, en.ws.data_ptr(),
                            en.ws.numel(), en.order.data_ptr(), en.cost.data_ptr(), en.stats.data_ptr(),
                            en.status.data_ptr())
    torch.cuda.synchronize()
    failed = probe.enumerations(C.cast(K.lib().cmp_enumerate, C.c_void_p), args, CALLS)
    assert failed == 0, failed
    torch.cuda.synchronize()
    for en, _, ref in jobs:
        assert en.plans() == ref

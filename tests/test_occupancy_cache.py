"""The cache of resident blocks per SM (csrc/pa_occ_cache.cuh, plain C++) compiled
on the host: many more shapes than a process usually sees are each asked for once,
each kernel is prepared once per device, failures are passed on and not kept, and
several threads agree."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SOURCE = r"""
#include "pa_occ_cache.cuh"
#include <atomic>
#include <cstdio>
#include <thread>
#include <vector>
#define CHECK(x) do { if (!(x)) { std::printf("failed: %s\n", #x); return 1; } } while (0)
int main() {
  static char fns[200];
  pa::OccCache c;
  std::atomic<int> prepared{0}, queried{0};
  auto ask = [&](int f, int dev, int threads, size_t smem) {
    int v = -1;
    int e = c.get({fns + f, dev, threads, smem}, &v, [&] { ++prepared; return 0; },
                  [&](int* p) { ++queried; *p = (int)(f + 3 * dev + threads + smem) % 97; return 0; });
    return e == 0 && v == (int)(f + 3 * dev + threads + smem) % 97;
  };
  for (int rep = 0; rep < 3; ++rep)
    for (int f = 0; f < 200; ++f)
      for (int dev = 0; dev < 2; ++dev)
        for (int t = 32; t <= 128; t += 32)
          for (size_t s = 0; s < 4; ++s) CHECK(ask(f, dev, t, 1000 * s + 16));
  CHECK(queried == 200 * 2 * 4 * 4);
  CHECK(prepared == 200 * 2);
  // failures: passed on, asked again
  int v = 5, tries = 0;
  for (int rep = 0; rep < 2; ++rep)
    CHECK(c.get({&tries, 0, 1, 1}, &v, [&] { ++tries; return 7; }, [&](int*) { return 0; }) == 7);
  CHECK(tries == 2);
  for (int rep = 0; rep < 2; ++rep)
    CHECK(c.get({&tries, 0, 1, 1}, &v, [&] { ++tries; return 0; }, [&](int*) { ++tries; return 9; }) == 9);
  CHECK(tries == 5);
  std::vector<std::thread> ts;
  std::atomic<int> bad{0};
  for (int k = 0; k < 8; ++k)
    ts.emplace_back([&] {
      for (int s = 0; s < 2000; ++s)
        if (!ask(s % 200, 0, 256, (size_t)s)) ++bad;
    });
  for (auto& t : ts) t.join();
  CHECK(bad == 0 && queried == 200 * 2 * 4 * 4 + 2000);
  std::printf("ok\n");
}
"""


def test_every_shape_is_asked_for_once(tmp_path):
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(SOURCE)
    subprocess.run(["g++", "-std=c++17", "-O1", "-pthread", "-I",
                    os.path.join(ROOT, "paper_2511_20511_gb300", "csrc"), str(src), "-o", str(exe)],
                   check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0 and r.stdout.strip() == "ok", r.stdout


@pytest.mark.gpu
def test_many_shapes_on_the_gpu():
    """More than 256 shapes through the small and the large calls' kernels of one
    process: their values do not depend on what was asked before."""
    import numpy as np

    from paper_2511_20511_gb300 import binding as B
    from paper_2511_20511_gb300 import build, inputs

    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    build.build()
    first = {}
    for rep in range(2):
        for L in range(2, 49, 2):
            for K in range(2, 14):
                rng = np.random.default_rng(64 * L + K)
                beta = np.exp(rng.normal(-20.0, 1.0, size=(L, L, K)))
                with B.Context(B.pa_config_default(L, K, N=32), beta) as ctx:
                    pop = inputs.random_population_torch(40, L, K, K, "cuda")
                    fit = ctx.eval_population(pop).cpu()
                if rep == 0:
                    first[L, K] = fit
                else:
                    assert torch.equal(fit, first[L, K])

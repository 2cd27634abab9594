"""The shared-memory rule of the plane pass: which items one launch takes, for every side and every pair
of sphere spans (CPU), and batches of items whose spans differ (GPU).

One launch runs with one size of shared memory, sized by the largest m1 span and the largest m2 span of
its items.  They may come from different items, so items that fit alone need not fit together."""
import os
import subprocess

import numpy as np
import pytest

from paper_1406_7803_gb300 import build

# Every (side, side) the context accepts: all pairs of spans as two items of a batch, then longer random
# lists.  A list must be cut into launches that hold its items in order and whose combined spans fit; a
# cut is wanted only before an item that would not fit with the launch so far, or when it is full.
PROGRAM = r"""
#include <cstdio>
#include <vector>
#include "hpsi2_p.cuh"
using namespace fde;
static long lists = 0, cuts = 0;
template <typename T> static int check(const GridDims& g, const std::vector<HpsiItemDesc<T>>& it) {
  const int n = (int)it.size();
  ++lists;
  for (int i0 = 0, k = 0; i0 < n; i0 += k) {
    k = plane_group<T>(g, it.data() + i0, n - i0, kBatchMax);
    if (k < 1 || k > kBatchMax || i0 + k > n) return 1;
    int s1 = 0, s2 = 0;
    for (int j = i0; j < i0 + k; ++j) {
      s1 = std::max(s1, it[j].sp.span1);
      s2 = std::max(s2, it[j].sp.span2);
    }
    if (plane_fit<T>(g, s1, s2).smem > kCtaSmemMax) return 2;
    if (i0 + k < n && k < kBatchMax) {
      ++cuts;
      s1 = std::max(s1, it[i0 + k].sp.span1);
      s2 = std::max(s2, it[i0 + k].sp.span2);
      if (plane_fit<T>(g, s1, s2).smem <= kCtaSmemMax) return 3;
    }
  }
  return 0;
}
template <typename T> static int sides(const std::vector<int>& ns) {
  unsigned rnd = 12345;
  for (int n1 : ns)
    for (int n2 : ns) {
      if ((size_t)n1 * (n2 + 1) * sizeof(cplx<T>) > 227 * 1024) continue;
      const GridDims g{n1, n2, 24};
      std::vector<SphereDev> ok;
      for (int a = 1; a <= n1; a += n1 == n2 ? 1 : 3)
        for (int b = std::max(1, a * n2 / n1 - 6); b <= std::min(n2, a * n2 / n1 + 6); ++b) {
          SphereDev sp{};
          sp.span1 = a;
          sp.span2 = b;
          if (two_step_grid<T>(g, sp)) ok.push_back(sp);
        }
      std::vector<HpsiItemDesc<T>> it;
      const auto put = [&](const SphereDev& sp) {
        HpsiItemDesc<T> d{};
        d.sp = sp;
        it.push_back(d);
      };
      for (size_t x = 0; x < ok.size(); ++x)
        for (size_t y = 0; y < ok.size(); y += n1 == n2 ? 1 : 7) {
          it.clear();
          put(ok[x]);
          put(ok[y]);
          if (int e = check<T>(g, it)) return printf("%d x %d, %d bytes: pair, error %d\n", n1, n2, (int)sizeof(T), e), 1;
        }
      for (int t = 0; t < 20; ++t) {
        it.clear();
        for (int k = 0; k < 60; ++k) put(ok[(rnd = rnd * 1664525u + 1013904223u) / 65536 % ok.size()]);
        if (int e = check<T>(g, it)) return printf("%d x %d, %d bytes: list, error %d\n", n1, n2, (int)sizeof(T), e), 1;
      }
    }
  return 0;
}
// Spheres as wide as the plane, which the compiled-side kernels have always served.
template <typename T> static int widest(const std::vector<int>& ns, size_t most) {
  for (int n : ns)
    for (int a = 1; a <= n; ++a)
      for (int b = 1; b <= n; ++b) {
        SphereDev sp{};
        sp.span1 = a;
        sp.span2 = b;
        if ((size_t)n * n * sizeof(cplx<T>) <= most && !two_step_grid<T>(GridDims{n, n, 24}, sp))
          return printf("%d x %d, %d bytes: spans %d, %d refused\n", n, n, (int)sizeof(T), a, b), 1;
      }
  return 0;
}
// The thread rule of a side: whole batches of items, one a thread, in a CTA that can run.
template <typename T> static bool shape_ok(int n, int r1, int r2) {
  const PlaneShape s = plane_shape<T>(n);
  const int lb = plane_lb<T>(n, n);
  const int runs = plane_has_runs<T>(n) ? plane_runs_lb<T>(n) * r1 : 0;
  return s.nt >= 128 && s.nt <= 512 && s.nt % 32 == 0 && s.minb >= 1 && s.minb * s.nt <= 1024 && r1 >= r2 && lb >= 1 &&
         lb * r1 <= s.nt && runs <= 512;
}
int main() {
#define SHAPE(N, A, B) \
  if (!shape_ok<float>(N, A, B) || !shape_ok<double>(N, A, B)) return printf("shape of %d\n", N), 1;
  FDE_PLANE_SIDES(SHAPE)
  const std::vector<int> ns = {
#define ONE(N, A, B) N,
      FDE_PLANE_SIDES(ONE)
  };
  if (sides<float>(ns) || sides<double>(ns)) return 1;
  if (widest<float>(ns, 227 * 1024) || widest<double>(ns, 190 * 1024)) return 1;
  printf("%ld lists, %ld cuts\n", lists, cuts);
  return 0;
}
"""


def run(tmp_path, text):
    src, exe = tmp_path / "fit.cu", tmp_path / "fit"
    src.write_text(text)
    cmd = [build.nvcc()] + build.ARCH + ["-std=c++17", "-O1", "-I", build.CSRC, "-I",
                                         os.path.join(build.ROOT, "include"), str(src), "-o", str(exe)]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
    return r.stdout


def test_launches_fit_shared_memory_for_every_side_and_pair_of_spans(tmp_path):
    assert int(run(tmp_path, PROGRAM).split()[2]) > 0, "no list needed a cut: the test would not see a missing rule"


# A launch of no blocks is refused before anything runs, with or without a GPU: the program sees what the
# host side does around it.
ATTRIBUTE = r"""
#include <cstdio>
#include <vector>
#include <cuda_runtime.h>
static std::vector<int> limits;
template <typename K> static cudaError_t record(K, cudaFuncAttribute a, int v) {
  if (a == cudaFuncAttributeMaxDynamicSharedMemorySize) limits.push_back(v);
  return cudaSuccess;
}
#define cudaFuncSetAttribute record
#include "hpsi2_p.cuh"
namespace fde { thread_local Profiler* tl_prof = nullptr; }
using namespace fde;
int main() {
  HpsiBatch<float> B{};
  FftPlans<float> fp{};
  for (size_t bytes : {100000u, 200000u, 60000u}) plane_square<float, 9, 8>(0, B, 24, fp, 0, PlaneFit{1, false, bytes}, 0);
  for (int v : limits)
    if (v != (int)kCtaSmemMax) return printf("limit set to %d\n", v), 1;
  return limits.size() == 3 ? 0 : 1;
}
"""


# The same launches' own status, and the limit's when that is what fails.
STATUS = ATTRIBUTE[:ATTRIBUTE.index("int main")].replace("return cudaSuccess;", "return answer;").replace(
    "template <typename K>", "static cudaError_t answer = cudaSuccess;\ntemplate <typename K>", 1) + r"""
int main() {
  HpsiBatch<float> B{};
  FftPlans<float> fp{};
  SphereDev sp{};
  const PlaneFit f{1, false, 60000};
  if (plane_square<float, 9, 8>(0, B, 24, fp, 0, f, 0) == cudaSuccess) return printf("plane pass\n"), 1;
  if (rho_square<float, 9, 8>(dim3(0), nullptr, sp, 1, nullptr, nullptr, 24, fp, 0, f, 0) == cudaSuccess)
    return printf("density\n"), 1;
  answer = cudaErrorInvalidValue;
  return plane_square<float, 9, 8>(0, B, 24, fp, 0, f, 0) == answer ? 0 : 1;
}
"""


def test_no_launch_lowers_the_shared_memory_limit_of_its_kernel(tmp_path):
    """Threads share the limit: one that a launch lowers to its own bytes makes another thread's launch of
    the same kernel, with more, fail."""
    run(tmp_path, ATTRIBUTE)


def test_a_refused_launch_is_reported(tmp_path):
    run(tmp_path, STATUS)


gpu = pytest.mark.gpu


@gpu
@pytest.mark.parametrize("prec,grid,lengths,ecut,kpts,spans,tol", [
    ("fp64", (96, 96, 24), (24.0, 24.36, 6.0), 55.4, ((0, 0, 0), (0.5, 0.5, 0)), ((81, 81), (80, 82)), 1e-13),
    ("mixed", (144, 144, 24), (38.92, 40.53, 7.45), 40.0, ((0, 0, 0), (0.5, 0.5, 0)), ((111, 115), (110, 116)), 2e-6),
    # sides that differ: the kernel with runtime sides
    ("fp64", (96, 90, 24), (24.0, 21.0, 6.0), 63.4, ((0, 0, 0), (0.5, 0.5, 0)), ((87, 75), (86, 76)), 1e-13),
])
def test_batches_of_items_with_unequal_spans(prec, grid, lengths, ecut, kpts, spans, tol):
    """H psi of two k-points that fit shared memory one by one, as one hot step (eager and replayed) and as
    one block at a time: the same kernels on the same potential, so equal up to the rounding of a plane
    whose columns come in other groups."""
    torch = pytest.importorskip("torch")
    from paper_1406_7803_gb300 import fde
    build.build()
    if not torch.cuda.is_available():
        pytest.fail("GPU tests need a CUDA device")
    k = np.array(kpts, dtype=float)
    for kf, want in zip(k, spans):
        m = fde.host_sphere(np.array(lengths), kf, ecut)[0]
        assert tuple(int(np.ptp(m[:, j])) + 1 for j in range(2)) == want
    rng = np.random.default_rng(grid[0])
    stream = torch.cuda.Stream()  # a graph is captured on a stream of its own
    ctx = fde.Context(np.diag(lengths), grid, ecut, 0, 0, prec=prec, stream=stream.cuda_stream)
    nb = 2
    ctx.add_subsystem(np.array([[1.0, 2.0, 3.0]]), np.ones(1), 0.5, nb, k, np.full(2, 0.5), 2.0, 0.01)
    ctx.set_density(0, 0.01 + 0.01 * rng.random(grid))
    want = []
    ctx.build_vemb()
    for q in range(2):
        npw = len(ctx.basis(0, q))
        c = rng.standard_normal((nb, npw)) + 1j * rng.standard_normal((nb, npw))
        c /= np.linalg.norm(c, axis=1)[:, None]
        c = torch.from_numpy(c).cuda()
        if prec == "mixed":
            c = c.to(torch.complex64)
        c64, h = c.to(torch.complex128), torch.zeros_like(c)
        torch.cuda.synchronize()  # filled on torch's stream, read on the context's
        ctx.set_orbitals(0, q, c64)
        ctx.apply_h(0, q, c, h, nb)
        ctx.sync()
        want.append(h.to(torch.complex128).cpu().numpy())
    for graph in (False, True, True):
        ctx.hot_step(graph)
        ctx.sync()
        for q in range(2):
            out = torch.zeros(want[q].shape, dtype=torch.complex128, device="cuda")
            torch.cuda.synchronize()
            ctx.get_hpsi(0, q, out)
            err = np.abs(out.cpu().numpy() - want[q]).max() / np.abs(want[q]).max()
            assert err < tol, (graph, q, err)

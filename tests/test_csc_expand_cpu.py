"""csc_expand at the top of the edge counts hg_build_csr accepts: one warp of the kernel's own source, on the host.

The kernel's text is compiled with g++, a thread per lane and the shuffles over a barrier, and given the last
1024 positions of about 2^31 edges through pointers moved by the positions before them.  A position that wraps
stores gigabytes away from the arrays and ends the child process."""
import os
import re
import subprocess

import pytest

import paper_2608_02168_gb300

GRAPH_CU = os.path.join(os.path.dirname(paper_2608_02168_gb300.__file__), "csrc", "graph.cu")

HARNESS = r"""
#include <barrier>
#include <cstdint>
#include <cstdio>
#include <cstdlib>
#include <thread>
#include <vector>
#define __global__
#define __launch_bounds__(...)
#define __restrict__
struct Dim { unsigned x; };
static Dim blockIdx, gridDim, blockDim{256};
static thread_local Dim threadIdx;
static std::barrier<> bar(32);
static uint64_t lanes[32];
template <typename T> T __shfl_sync(unsigned, T v, int src) {
  T out;
  __builtin_memcpy(&lanes[threadIdx.x & 31], &v, sizeof(T));
  bar.arrive_and_wait();
  __builtin_memcpy(&out, &lanes[src], sizeof(T));
  bar.arrive_and_wait();
  return out;
}
template <typename T> T __ldg(const T* p) { return *p; }
static int64_t min(int64_t a, int64_t b) { return a < b ? a : b; }
static void pdl_begin() {}
@KERNEL@
int main(int, char** argv) {
  const int64_t nv = atoll(argv[1]), single = atoll(argv[2]);  // a run of all edges but the last `single`, which are runs of one
  const int64_t w = (nv - 1) / kExpand, p0 = w * kExpand, cnt = nv - p0, U = single + 1;
  std::vector<int32_t> qpos(U + 1), qstart(U), eid(kExpand), col(kExpand + 256, -7), out(kExpand + 256, -7);
  std::vector<uint32_t> qdst(U);
  std::vector<float> qcoef(U), coef(kExpand + 256, -7.f);
  qpos[U] = (int32_t)nv;
  for (int64_t q = 0; q < U; ++q) {
    qpos[q] = q == 0 ? 0 : (int32_t)(nv - single + q - 1);
    qstart[q] = q == 0 ? 0 : (int32_t)(kOneEdge | (uint32_t)(5000 + q));
    qdst[q] = (uint32_t)(100 + q);
    qcoef[q] = 1.f + q;
  }
  for (int k = 0; k < kExpand; ++k) eid[k] = 100000 + k;
  const int32_t n_dev = (int32_t)U;
  blockIdx.x = (unsigned)(w / 8);
  gridDim.x = 1u << 24;  // this warp takes one stretch
  std::vector<std::thread> t;
  for (int lane = 0; lane < 32; ++lane)
    t.emplace_back([&, lane] {
      threadIdx.x = (unsigned)(w % 8 * 32 + lane);
      csc_expand(qpos.data(), qstart.data(), qcoef.data(), qdst.data(), &n_dev, eid.data() - p0, col.data() - p0,
                 out.data() - p0, coef.data() - p0);
    });
  for (auto& x : t) x.join();
  for (int64_t k = 0; k < kExpand + 256; ++k) {
    const int64_t p = p0 + k, q = p < nv - single ? 0 : p - (nv - single) + 1;
    const bool in = k < cnt;
    const int32_t e = !in ? -7 : q == 0 ? 100000 + (int32_t)k : 5000 + (int32_t)q;
    if (out[k] != e || col[k] != (in ? 100 + (int32_t)q : -7) || coef[k] != (in ? 1.f + q : -7.f)) {
      printf("position %lld of %lld: edge %d, destination %d\n", (long long)p, (long long)nv, out[k], col[k]);
      return 1;
    }
  }
  return 0;
}
"""


@pytest.fixture(scope="module")
def binary(tmp_path_factory):
    src = open(GRAPH_CU).read()
    one = re.search(r"constexpr uint32_t kOneEdge = [^;]*;", src).group(0)
    kernel = re.search(r"constexpr int kExpand = .*?\n}\n", src, re.S).group(0)
    assert "csc_expand" in kernel
    d = tmp_path_factory.mktemp("expand")
    (d / "t.cpp").write_text(HARNESS.replace("@KERNEL@", one + "\n" + kernel))
    subprocess.run(["g++", "-std=c++20", "-O1", "-fwrapv", "-pthread", "-w", "t.cpp", "-o", "t"], cwd=d, check=True)
    return str(d / "t")


@pytest.mark.parametrize("nv", [5000, 2**31 - 129, 2**31 - 128, 2**31 - 127, 2**31 - 31, 2**31 - 1])
@pytest.mark.parametrize("single", [0, 1, 500])
def test_last_positions(binary, nv, single):
    r = subprocess.run([binary, str(nv), str(single)], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, (r.returncode, r.stdout)

"""What the launchers remember is kept by device (csrc/sq_device_state.h), compiled for the host against a
counterfeit CUDA runtime with several devices: no box here has more than one."""
import os
import re
import shutil
import subprocess

import pytest

from paper_2404_04793_b200 import build

PROGRAM = r"""
#include <cstdio>
#include <map>
#include <utility>
#include "sq_device_state.h"
static int g_dev = 0, g_fail = 0;
static std::map<std::pair<int, const void*>, int> g_limit;   // (device, kernel) -> bytes
static int g_sets = 0, g_asked = 0;
static int g_room = 0;                                        // CTAs of the largest cluster that fits
extern "C" {
cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaOccupancyMaxActiveClusters(int* n, const void*, const cudaLaunchConfig_t* c) {
  ++g_asked;
  if (c->numAttrs != 1 || c->attrs[0].id != cudaLaunchAttributeClusterDimension || c->gridDim.x != c->attrs[0].val.clusterDim.x)
    return cudaErrorInvalidValue;
  *n = (int)c->attrs[0].val.clusterDim.x <= g_room ? 3 : 0;
  return cudaSuccess;
}
cudaError_t cudaGetDevice(int* d) { *d = g_dev; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int d) { *v = 100 + d; return cudaSuccess; }
cudaError_t cudaFuncSetAttribute(const void* f, cudaFuncAttribute, int v) {
  if (g_fail) return cudaErrorInvalidValue;
  ++g_sets;
  g_limit[{g_dev, f}] = v;
  return cudaSuccess;
}
}
static void kern_a(int) {}
static void kern_b(float) {}
#define CHECK(x) do { if (!(x)) { std::printf("line %d: %s\n", __LINE__, #x); return 1; } } while (0)
int main() {
  static sq::PerDevice state, other;
  for (int round = 0; round < 3; ++round)
    for (int d : {0, 3, 1, 63, 200}) {
      g_dev = d;
      CHECK(sq::allow_smem(state, 70000, kern_a, kern_b) == cudaSuccess);
      CHECK((g_limit[{d, (const void*)kern_a}]) == 70000 && (g_limit[{d, (const void*)kern_b}]) == 70000);
      CHECK(sq::sm_count() == 100 + d);
    }
  CHECK(g_sets == 2 * (4 + 3));   // once on each device that is remembered, every time on the one beyond
  g_dev = 2;
  g_fail = 1;
  CHECK(sq::allow_smem(other, 5, kern_a) == cudaErrorInvalidValue);
  g_fail = 0;
  CHECK(sq::allow_smem(other, 5, kern_a) == cudaSuccess);   // a failure is not remembered as done
  CHECK((g_limit[{2, (const void*)kern_a}]) == 5);
  static sq::ClusterFit fit;
  const void* k = (const void*)kern_a;
  for (int round = 0; round < 2; ++round) {
    g_dev = 0, g_room = 16;
    CHECK(fit.fits(k, 16, 128, 1000));
    g_dev = 1, g_room = 8;
    CHECK(!fit.fits(k, 16, 128, 1000));
  }
  CHECK(g_asked == 2);
  // a launch that asks for 16 and finds no room is made with 8, once; other results are passed on
  for (int d : {0, 1}) {
    g_dev = d;
    int made = 0, calls = 0;
    auto launch = [&](int limit) {
      ++calls;
      if (limit > 8 && !fit.fits(k, 16, 128, 1000)) return cudaErrorNotSupported;
      made = limit;
      return cudaSuccess;
    };
    CHECK(sq::with_portable_clusters(16, launch) == cudaSuccess && made == (d == 0 ? 16 : 8) && calls == 1 + d);
  }
  int calls = 0;
  CHECK(sq::with_portable_clusters(8, [&](int) { ++calls; return cudaErrorNotSupported; }) == cudaErrorNotSupported && calls == 1);
  CHECK(sq::with_portable_clusters(16, [&](int) { ++calls; return cudaErrorInvalidValue; }) == cudaErrorInvalidValue && calls == 2);
  std::puts("ok");
}
"""


def cuda_include():
    return os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(build._nvcc()))), "include")


def run_host_program(tmp_path, source):
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(source)
    subprocess.run(["g++", "-std=c++17", "-I", build.CSRC, "-I", build.INCLUDE, "-I", cuda_include(), str(src), "-o", str(exe)], check=True)
    return subprocess.run([str(exe)], capture_output=True, text=True, timeout=60).stdout.strip()


PIECES = r"""
#include <cstdio>
#include "sq_device_state.h"
int main() {
  // room of a device by cluster size: as many CTAs as there are slots, none of more than `largest`
  int slots = 264, largest = 16;
  auto room = [&](int ctas) { return ctas <= largest ? slots / ctas : 0; };
  bool ok = sq::most_ctas(14, 1, room) == 14 && sq::most_ctas(14, 33, room) == 8 && sq::most_ctas(14, 132, room) == 2 &&
            sq::most_ctas(14, 133, room) == 0 && sq::most_ctas(1, 1, room) == 0 && sq::most_ctas(3, 1, room) == 3;
  largest = 8;   // a device without the larger sizes: the portable ones are still taken
  ok = ok && sq::most_ctas(14, 1, room) == 8 && sq::most_ctas(14, 33, room) == 8 && sq::most_ctas(14, 60, room) == 4;
  largest = 0;
  ok = ok && sq::most_ctas(14, 1, room) == 0;
  std::puts(ok ? "ok" : "wrong");
}
"""


@pytest.mark.skipif(shutil.which("g++") is None, reason="no host compiler")
def test_pieces_of_a_unit_shrink_to_the_clusters_that_a_device_holds(tmp_path):
    assert run_host_program(tmp_path, PIECES) == "ok"


@pytest.mark.skipif(shutil.which("g++") is None, reason="no host compiler")
def test_set_up_clusters_and_sm_count_are_kept_by_device(tmp_path):
    assert run_host_program(tmp_path, PROGRAM) == "ok"


def test_no_launcher_keeps_a_flag_of_its_own():
    """Attributes are set through PerDevice alone."""
    for path in build.sources():
        text = open(path).read()
        assert not re.search(r"static\s+(bool|size_t|int)\s+(configured|n_sm)", text), path
        for call in re.finditer(r"cudaFuncSetAttribute", text):
            assert ".once(" in text[max(0, call.start() - 400):call.start()], path

"""The conditioning cache's check, compiled for the host: 32 threads run the
device function on arrays that end at an unreadable page, so that a read or
write past any of them ends the program."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2609_34170_gb300", "csrc")

HARNESS = r"""
#include <cuda_runtime.h>
#include <pthread.h>
#include <string.h>
#include <sys/mman.h>
#include <unistd.h>

#include <cstdio>
#include <cstdlib>
#include <thread>
#include <vector>

struct Idx { unsigned x; };
static thread_local Idx threadIdx;
static const Idx blockDim = {32};
static pthread_barrier_t bar;
static void __syncthreads() { pthread_barrier_wait(&bar); }
static unsigned atomicOr(unsigned* p, unsigned v) { return __atomic_fetch_or(p, v, __ATOMIC_SEQ_CST); }
#undef __shared__
#undef __device__
#define __shared__ static
#define __device__
#include "cond_cache.cuh"

using namespace ravel;

// n elements that end where an unreadable page begins
template <typename T>
T* guarded(size_t n) {
  const size_t page = sysconf(_SC_PAGESIZE), bytes = (n * sizeof(T) + page - 1) / page * page;
  char* m = (char*)mmap(nullptr, bytes + page, PROT_READ | PROT_WRITE, MAP_PRIVATE | MAP_ANONYMOUS, -1, 0);
  mprotect(m + bytes, page, PROT_NONE);
  return (T*)(m + bytes - n * sizeof(T));
}

int main(int argc, char** argv) {
  const int slots = atoi(argv[1]), B = atoi(argv[2]), per_robot = atoi(argv[3]), Bmax = B;
  const int H = per_robot ? B * slots : slots;
  float *t = guarded<float>(H), *key = guarded<float>(slots), *delta = guarded<float>(B);
  int *drow = guarded<int>(B), *commit = guarded<int>(2 * B);
  CondCache* cc = guarded<CondCache>(1);
  memset(cc, 0, sizeof *cc);
  memset(key, 0, slots * sizeof(float));
  for (int j = 0; j < H; ++j) t[j] = (j + 1) / (float)H;
  for (int b = 0; b < B; ++b) delta[b] = 0.02f * (b % 3);
  CondArgs a{cc, key, drow, commit, t, delta, H, B, Bmax, nullptr, 0, per_robot ? 0 : 1};
  pthread_barrier_init(&bar, nullptr, 32);
  for (int step = 0; step < 3; ++step) {   // a first step, the same again, other slot times
    if (step == 2) t[slots - 1] = 0.5f;
    std::vector<std::thread> ts;
    for (unsigned i = 0; i < 32; ++i)
      ts.emplace_back([&, i] {
        threadIdx.x = i;
        cond_check(a);
      });
    for (auto& th : ts) th.join();
    printf("%d", cc->skip);
    for (int b = 0; b < B; ++b) printf(" %d", drow[b]);
    printf("\n");
  }
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    include = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include")
    if not shutil.which("g++") or not os.path.exists(os.path.join(include, "cuda_runtime.h")):
        pytest.skip("needs g++ and the CUDA headers")
    d = tmp_path_factory.mktemp("cond")
    (d / "main.cpp").write_text(HARNESS)
    subprocess.run(["g++", "-std=c++17", "-O1", "-w", "-pthread", "-I", CSRC, "-I", os.path.join(ROOT, "include"),
                    "-I", include, str(d / "main.cpp"), "-o", str(d / "main")], check=True)
    return str(d / "main")


@pytest.mark.parametrize("slots,B", [(1, 1), (10, 3), (50, 16)])
@pytest.mark.parametrize("per_robot", [0, 1])
def test_cond_check_stays_in_its_arrays(program, slots, B, per_robot):
    out = subprocess.run([program, str(slots), str(B), str(per_robot)], capture_output=True, text=True)
    assert out.returncode == 0, out
    steps = [[int(x) for x in line.split()] for line in out.stdout.splitlines()]
    H = B * slots if per_robot else slots
    # with a schedule per robot nothing is cached and every robot has its fresh row
    assert [s[0] for s in steps] == ([0, 0, 0] if per_robot else [0, 1, 0])
    want = [H + b for b in range(B)] if per_robot else [H + B + b % 3 for b in range(B)]
    assert all(s[1:] == want for s in steps)

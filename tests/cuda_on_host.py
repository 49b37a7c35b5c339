"""Runs kernels of csrc/ on the CPU, from their source: the definitions asked for are taken out of
the .cu files by name, compiled by g++ with the address sanitizer beside a main() of the test's, and
executed block by block, one host thread per CUDA thread. For kernels that use indexes, shared
memory and __syncthreads only; what they read and write out of bounds ends the program."""
import os
import re
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1310_7202_gb300", "csrc")

SHIM = r"""
#include <algorithm>
#include <barrier>
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <limits>
#include <thread>
#include <type_traits>
#include <vector>
#define __global__
#define __device__
#define __host__
#define __forceinline__ inline
#define __shared__ static
#define __launch_bounds__(...)
using std::isfinite;
struct dim3 {
  unsigned x = 1, y = 1, z = 1;
  dim3(unsigned a = 1, unsigned b = 1, unsigned c = 1) : x(a), y(b), z(c) {}
};
struct float2 { float x, y; };
inline float2 make_float2(float x, float y) { return {x, y}; }
inline float __uint_as_float(uint32_t v) { float f; std::memcpy(&f, &v, 4); return f; }
inline uint32_t __float_as_uint(float f) { uint32_t v; std::memcpy(&v, &f, 4); return v; }
inline float __fadd_rn(float a, float b) { return a + b; }
inline float __fsub_rn(float a, float b) { return a - b; }
thread_local dim3 threadIdx, blockIdx;
dim3 blockDim, gridDim;
std::barrier<>* the_barrier;
inline void __syncthreads() { the_barrier->arrive_and_wait(); }
template <typename F> void launch(dim3 grid, dim3 block, F kernel) {
  gridDim = grid;
  blockDim = block;
  const unsigned nt = block.x * block.y;
  for (unsigned by = 0; by < grid.y; ++by)
    for (unsigned bx = 0; bx < grid.x; ++bx) {
      std::barrier<> bar(nt);
      the_barrier = &bar;
      std::vector<std::thread> ts;
      for (unsigned t = 0; t < nt; ++t)
        ts.emplace_back([&, t] {
          threadIdx = dim3(t % block.x, t / block.x);
          blockIdx = dim3(bx, by);
          kernel();
          bar.arrive_and_drop();
        });
      for (auto& t : ts) t.join();
    }
}
#define CHECK(x) do { if (!(x)) { std::printf("failed: %s (line %d)\n", #x, __LINE__); std::exit(1); } } while (0)
"""


def definition(file, name):
    """The text of every definition of `name` in csrc/file, each with its template line."""
    src = open(os.path.join(CSRC, file)).read()
    found = []
    for m in re.finditer(r"(?:^template <[^\n]*>\n)?^[^\n/#]*\b" + name + r"\(", src, re.M):
        depth, at = 0, m.end() - 1
        while True:  # the argument list, then the body
            depth += {"(": 1, ")": -1}.get(src[at], 0)
            at += 1
            if depth == 0:
                break
        rest = re.match(r"\s*\{", src[at:])
        if not rest:
            continue  # a declaration or a call
        at += rest.end()
        depth = 1
        while depth:
            depth += {"{": 1, "}": -1}.get(src[at], 0)
            at += 1
        found.append(src[m.start():at])
    assert found, (file, name)
    return "\n".join(found)


def run(tmp_path, parts, main):
    """Compiles the shim, the definitions `parts` ((file, name) pairs) and main, and runs it."""
    cu, exe = os.path.join(tmp_path, "k.cpp"), os.path.join(tmp_path, "k")
    with open(cu, "w") as f:
        f.write(SHIM + "\n".join(definition(*p) for p in parts) + "\n" + main)
    subprocess.run(["g++", "-std=c++20", "-O1", "-g", "-ffp-contract=off", "-fsanitize=address",
                    "-Wno-unknown-pragmas", "-pthread", cu, "-o", exe], check=True)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=300,
                       env=dict(os.environ, ASAN_OPTIONS="detect_leaks=0"))
    assert r.returncode == 0, (r.stdout + r.stderr)[-3000:]

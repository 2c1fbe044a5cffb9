"""Host check of the complex128 line transforms: fft_line_fx and the FP64 stages of
csrc/qfd_kernels.cuh compiled for the host (device builtins replaced by their
definitions, the threads of a line by host threads) and compared with an
extended-precision DFT.

The bound is the FP64 transform itself: over the lines of a class the rms error of the
fixed-point transform is no larger than that of the FP64 butterflies on the same lines,
with 15% allowed for the few lines of a class (a line's error depends on where its largest
component lies between two powers of two, by up to a factor of two).  The classes are the lines a solve meets: one site,
narrow and broad states and their spectra, a few modes, slow tails, a peak on a
floor of noise, and noise.  Lines of the largest growth check that no sum leaves 64 bits.
"""
import os
import shutil
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2006_16935_gb300", "csrc")
CUDA_INC = "/usr/local/cuda/include"
SIZES = (8, 16, 32, 64, 96, 128, 192, 256, 512, 1024)

HARNESS = r"""
#include <cuda_runtime.h>
#include <algorithm>
#include <barrier>
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <thread>
#include <vector>
#undef __launch_bounds__
#define __launch_bounds__(...)
#ifndef __noinline__
#define __noinline__ __attribute__((noinline))
#endif
using std::max;
using std::min;
static uint3 threadIdx, blockIdx;
static dim3 blockDim, gridDim;
template <class T> inline T __ldg(const T* p) { return *p; }
inline int64_t bits_of(double d) { int64_t b; std::memcpy(&b, &d, 8); return b; }
inline int __double2hiint(double d) { return (int)(bits_of(d) >> 32); }
inline int __double2loint(double d) { return (int)bits_of(d); }
inline double __hiloint2double(int h, int l) {
  const uint64_t b = ((uint64_t)(uint32_t)h << 32) | (uint32_t)l;
  double d;
  std::memcpy(&d, &b, 8);
  return d;
}
inline double __ll2double_rn(long long v) { return (double)v; }
inline int __clz(int m) { return m ? __builtin_clz(m) : 32; }
// named by code that this program does not run
inline float __fadd_rn(float a, float b) { return a + b; }
inline float __fsub_rn(float a, float b) { return a - b; }
inline float __fmul_rn(float a, float b) { return a * b; }
inline float __fdiv_rn(float a, float b) { return a / b; }
inline float __frcp_rn(float a) { return 1 / a; }
inline float __fmaf_rn(float a, float b, float c) { return fmaf(a, b, c); }
inline float __double2float_rn(double a) { return (float)a; }
inline float rsqrtf(float a) { return 1 / sqrtf(a); }
inline void sincospif(float, float*, float*) {}
inline void __syncthreads() {}
inline void __syncwarp(unsigned = 0) {}
inline bool __syncthreads_or(int a) { return a; }
inline int __any_sync(unsigned, int a) { return a; }
inline unsigned __activemask() { return 0; }
template <class T> inline T __shfl_xor_sync(unsigned, T a, int) { return a; }
template <class T> inline T __shfl_down_sync(unsigned, T a, int) { return a; }
inline int __reduce_max_sync(unsigned, int a) { return a; }
#include "qfd_kernels.cuh"
#include "qfd_launch.h"
using namespace qfd;

struct Line {  // what the threads of a line share
  std::barrier<> bar;
  std::vector<int> mx;
  explicit Line(int t) : bar(t), mx(t) {}
};
template <class C> struct HostAcc {
  void* buf;
  Line* ln;
  int t;
  C& at(int p) { return static_cast<C*>(buf)[p]; }
  int key(int b) const { return b; }
  C& at(int k, int c) { return at(k + c); }
  void sync() { ln->bar.arrive_and_wait(); }
  template <class D> HostAcc<D> as() const { return {buf, ln, t}; }
  template <class... X> bool line_max(int& mx, X...) {
    ln->mx[t] = mx;
    sync();
    for (int v : ln->mx) mx = max(mx, v);
    sync();
    return false;  // the lines of this program stay inside the fixed-point range
  }
};
template <int N, int DIR, bool FP64> void run(std::vector<double2>& x, const double2* tw) {
  using PL = FftPlan<N>;
  const size_t lines = x.size() / N;
  std::vector<double2> buf(N);
  Line ln(PL::T);
  std::vector<std::thread> th;
  for (int t = 0; t < PL::T; ++t)
    th.emplace_back([&, t] {
      for (size_t l = 0; l < lines; ++l) {
        double2* p = x.data() + l * N;
        double2 v[PL::E];
        for (int m = 0; m < PL::E; ++m) v[m] = p[t + m * PL::T];
        HostAcc<double2> acc{buf.data(), &ln, t};
        if constexpr (FP64) fft_stages<F64, N, 0, DIR, 0, false>(v, t, tw, acc);
        else fft_line_fx<N, DIR>(v, t, tw, acc);
        for (int m = 0; m < PL::E; ++m) p[t + m * PL::T] = v[m];
        ln.bar.arrive_and_wait();
      }
    });
  for (auto& t : th) t.join();
}
template <int N> void all(std::vector<double2>& x, bool fp64, int dir) {
  std::vector<double2> tw(4 * N);
  for (int e = 0; e < N; ++e) {
    const long double a = 2.0L * 3.14159265358979323846264338327950288L * e / N;
    tw[e] = double2{(double)cosl(a), (double)-sinl(a)};
  }
  scaled_twiddle_table(N, tw.data(), tw.data() + N);
  fixed_twiddle_table(N, tw.data() + 3 * N);
  if (fp64) dir < 0 ? run<N, -1, true>(x, tw.data()) : run<N, 1, true>(x, tw.data());
  else dir < 0 ? run<N, -1, false>(x, tw.data()) : run<N, 1, false>(x, tw.data());
}
int main(int, char** argv) {
  const int n = std::atoi(argv[1]), dir = std::atoi(argv[3]);
  const bool f = std::atoi(argv[2]);
  std::vector<double2> x;
  double2 v;
  while (std::fread(&v, sizeof(v), 1, stdin) == 1) x.push_back(v);
  dispatch_n(n, [&](auto t) {
    all<decltype(t)::value>(x, f, dir);
    return cudaSuccess;
  });
  std::fwrite(x.data(), sizeof(v), x.size(), stdout);
  return 0;
}
"""


@pytest.fixture(scope="module")
def transform(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx or not os.path.isdir(CUDA_INC):
        pytest.skip("needs a host C++ compiler and the CUDA headers")
    if np.finfo(np.longdouble).eps > 1e-18:
        pytest.skip("needs an extended-precision long double")
    d = tmp_path_factory.mktemp("lines")
    src, exe = d / "h.cpp", d / "h"
    src.write_text(HARNESS)
    subprocess.run([cxx, "-std=c++20", "-O1", "-w", "-pthread", "-ffp-contract=off", "-I" + CUDA_INC, "-I" + CSRC,
                    str(src), "-o", str(exe)], check=True)

    def go(x, fp64, direction):
        out = subprocess.run([str(exe), str(x.shape[1]), str(int(fp64)), str(direction)],
                             input=np.ascontiguousarray(x).tobytes(), check=True, capture_output=True).stdout
        return np.frombuffer(out, dtype=np.complex128).reshape(x.shape)

    return go


def dft(x, direction):
    """Real and imaginary parts of the DFT of every row, in extended precision."""
    n = x.shape[1]
    e = np.arange(n)
    a = 2 * np.longdouble("3.14159265358979323846264338327950288") * e.astype(np.longdouble) / n
    k = np.outer(e, e) % n
    c, s = np.cos(a)[k], direction * np.sin(a)[k]
    xr, xi = x.real.astype(np.longdouble), x.imag.astype(np.longdouble)
    return xr @ c - xi @ s, xr @ s + xi @ c


def errors(x, direction, got):
    r, i = dft(x, direction)
    d = (got.real - r) ** 2 + (got.imag - i) ** 2
    return np.sqrt((d.sum(1) / (r * r + i * i).sum(1)).astype(float))


def line_classes(n, rng):
    j = np.arange(n) - n // 2
    out = {}

    def g(w):
        return np.exp(-j ** 2 / (2.0 * w * w))

    def noise():
        return rng.uniform(-1, 1, n) + 1j * rng.uniform(-1, 1, n)

    out["site"] = np.eye(n)[n // 3]
    out["broad"] = g(n / 10)
    out["broad spectrum"] = np.fft.fft(np.fft.ifftshift(g(n / 10)))
    out["narrow spectrum"] = np.fft.fft(np.fft.ifftshift(g(3)))
    out["modes"] = np.where((j == 3) | (j == -4), 1.0, 0.0) + 0.3j * (j == 2)
    out["exponential"] = np.exp(-abs(j) / 2.0)
    out["tail"] = 1 / (1.0 + j ** 2)
    out["site on a floor"] = out["site"] + 1e-6 * noise()
    out["narrow on a floor"] = g(1.5) + 1e-6 * noise()
    out["spectrum on a floor"] = out["broad spectrum"] + 1e-6 * noise()
    out["noise"] = noise()
    return {k: v * np.exp(2j * np.pi * rng.random()) * rng.uniform(0.5, 1) for k, v in out.items()}


@pytest.mark.parametrize("n", SIZES)
def test_fixed_point_lines_are_no_less_exact_than_fp64(transform, n):
    rng = np.random.default_rng(n)
    sets = [line_classes(n, rng) for _ in range(8)]
    names = list(sets[0])
    x = np.array([s[k] for s in sets for k in names])
    rms = {f: np.mean([errors(x, d, transform(x, f, d)).reshape(len(sets), -1) ** 2 for d in (-1, 1)], axis=(0, 1)) ** 0.5
           for f in (False, True)}
    worse = {k: (a, b) for k, a, b in zip(names, rms[False], rms[True]) if a > 1.15 * b}
    assert not worse, worse


@pytest.mark.parametrize("n", SIZES)
def test_lines_of_the_largest_growth_stay_inside_64_bits(transform, n):
    # both components just below a power of two, all of it in one output (times sqrt 2 N)
    j = np.arange(n)
    big = (1 - 2.0 ** -53) * (1 + 1j)
    x = np.array([big * 1j ** (k * j % 4) for k in range(4)] + [big.conjugate() * 1j ** (k * j % 4) for k in range(4)])
    for d in (-1, 1):
        assert np.max(errors(x, d, transform(x, False, d))) < 2.0 ** -52

"""The fused slab kernel of csrc/slab.cuh on the CPU: each thread of a CTA a host thread, barriers and
shuffles as thread barriers, the staged bulk copy done where it is issued; under the compiler's
race detector, which orders accesses by those barriers alone. Every warp count tried leaves
lane groups without columns or rows in some round, and every length lanes outside a group: they
may read shared memory only where no other warp writes in the same phase.

The values are compared with the same operations in numpy: 1e-5 of the largest output (FP32, four
transforms of up to 225 points, about 1e-6)."""
import os
import shutil
import subprocess

import numpy as np
import pytest

from test_ffloat_host import CSRC, SHIM

SHIM_EXTRA = r"""
#include <algorithm>
#include <barrier>
#include <cstdint>
#include <cstring>
#include <vector>
struct float2 { float x, y; };
inline float2 make_float2(float x, float y) { return float2{x, y}; }
struct HostDim { unsigned x, y, z; };
inline thread_local HostDim threadIdx{0, 0, 0};
inline HostDim blockDim{1, 1, 1}, blockIdx{0, 0, 0}, gridDim{1, 1, 1};
struct Cta {
  std::barrier<> all;
  std::vector<std::barrier<>*> warp;
  float xch[32][32];
  int votes[2] = {0, 0};
  unsigned char* smem;
  explicit Cta(int n) : all(n) {}
};
inline Cta* g_cta = nullptr;
inline void __syncthreads() { g_cta->all.arrive_and_wait(); }
inline int __syncthreads_and(int v) { __syncthreads(); return v; }   // the staged copy has always come
inline void __syncwarp() { g_cta->warp[threadIdx.x >> 5]->arrive_and_wait(); }
inline float __shfl_sync(unsigned, float v, int src) {
  float* x = g_cta->xch[threadIdx.x >> 5];
  x[threadIdx.x & 31] = v;
  __syncwarp();
  const float r = x[src];
  __syncwarp();
  return r;
}
inline double __shfl_down_sync(unsigned, double v, int) { return v; }
inline unsigned __umulhi(unsigned a, unsigned b) { return (unsigned)(((unsigned long long)a * b) >> 32); }
inline float __ldg(const float* p) { return *p; }
inline int atomicExch(int* p, int v) { const int o = *p; *p = v; return o; }
inline size_t __cvta_generic_to_shared(const void*) { return 0; }
inline float2 __fadd2_rn(float2 a, float2 b) { return float2{a.x + b.x, a.y + b.y}; }
inline float2 __fmul2_rn(float2 a, float2 b) { return float2{a.x * b.x, a.y * b.y}; }
inline float2 __ffma2_rn(float2 a, float2 b, float2 c) { return float2{std::fmaf(a.x, b.x, c.x), std::fmaf(a.y, b.y, c.y)}; }
using std::min;
#define __global__
#define __launch_bounds__(...)
"""

DRIVER = r"""
#include <cstdio>
#include <cstdlib>
#include <thread>
#include "common.cuh"
#include "fpair.cuh"
namespace homb {
#include "slab.inc"
}
using namespace homb;
template <int R, bool ZB> static void run(SlabArgs a, int warps) {
  Cta cta(warps * 32);
  std::vector<unsigned char> smem(slab_smem_bytes(R, ZB, a.Ny, a.Nh, warps) + 32);
  cta.smem = (unsigned char*)(((uintptr_t)smem.data() + 15) & ~(uintptr_t)15);
  std::vector<std::thread> t;
  for (int w = 0; w < warps; ++w) cta.warp.push_back(new std::barrier<>(32));
  g_cta = &cta;
  blockDim.x = warps * 32;
  for (int i = 0; i < warps * 32; ++i)
    t.emplace_back([=] {
      threadIdx.x = (unsigned)i;
      k_slab<R, ZB>(a);
    });
  for (auto& x : t) x.join();
  for (auto* b : cta.warp) delete b;
}
template <typename T> static std::vector<T> load(const char* f) {
  FILE* h = std::fopen(f, "rb");
  std::fseek(h, 0, SEEK_END);
  std::vector<T> v(std::ftell(h) / sizeof(T));
  std::rewind(h);
  if (std::fread(v.data(), sizeof(T), v.size(), h) != v.size()) std::exit(3);
  std::fclose(h);
  return v;
}
// M N nrc Mz warps in coef twiddles out; or M N asked: the warps of a launch
int main(int argc, char** argv) {
  if (argc == 4) {
    const int M = std::atoi(argv[1]), N = std::atoi(argv[2]);
    std::printf("%d\n", slab_warps_asked<float>(M, N, (N + 1) / 2, std::atoi(argv[3])));
    return 0;
  }
  const int M = std::atoi(argv[1]), N = std::atoi(argv[2]), nrc = std::atoi(argv[3]), Mz = std::atoi(argv[4]);
  int warps = std::atoi(argv[5]);
  std::vector<float2> x = load<float2>(argv[6]), W = load<float2>(argv[8]);
  std::vector<float> c = load<float>(argv[7]);
  CgScalars cg{};
  cg.active[0] = cg.active[2] = 1;   // right-hand side 1 has converged: its slabs are skipped
  SlabArgs a{};
  a.in = x.data(); a.out = x.data(); a.coef = c.data(); a.W = W.data(); a.cg = &cg;
  a.nrc = nrc; a.C = 1; a.Mz = Mz; a.M = M; a.Ny = N; a.Nh = (N + 1) / 2;
  a.scale = 1.0 / ((double)M * M);
  if (warps == 0) warps = slab_warps<float>(M, N, a.Nh);
  const bool zb = slab_band_free(M, N, a.Nh);
  switch (M) {
    case 9: zb ? run<3, true>(a, warps) : run<3, false>(a, warps); break;
    case 25: zb ? run<5, true>(a, warps) : run<5, false>(a, warps); break;
    case 81: zb ? run<9, true>(a, warps) : run<9, false>(a, warps); break;
    default: run<15, true>(a, warps);   // a slab of M = N = 225 does not fit in shared memory
  }
  FILE* h = std::fopen(argv[9], "wb");
  std::fwrite(x.data(), sizeof(float2), x.size(), h);
  std::fclose(h);
  return 0;
}
"""


def _statement(src, i):
    """End of the statement (closing parenthesis and semicolon) that starts at src[i]."""
    depth, quoted = 0, False
    for k in range(i, len(src)):
        c = src[k]
        if c == '"' and src[k - 1] != "\\":
            quoted = not quoted
        elif not quoted and c == "(":
            depth += 1
        elif not quoted and c == ")":
            depth -= 1
        elif not quoted and c == ";" and depth == 0:
            return k + 1
    raise ValueError("unterminated statement")


def host_slab_source():
    """The kernel, its layout and its size rules, with the PTX statements taken out (the bulk copy: a
    plain one)."""
    src = open(os.path.join(CSRC, "slab.cuh")).read()
    kern = src[src.index("constexpr int kSlabMaxThreads"):src.index("template <int R, bool ZB, int NT> cudaError_t launch_slab_nt")]
    rules = src[src.index("inline bool slab_band_free"):src.index("template <int R> cudaError_t launch_slab_r")]
    rules += src[src.index("template <typename T> int slab_warps"):src.index("template <typename T> cudaError_t launch_slab(")]
    wait = kern.index("__device__ __forceinline__ bool slab_wait")
    after = kern.index("\n}\n", wait) + 3
    kern = kern[:wait] + "inline bool slab_wait(uint32_t, uint32_t) { return true; }\n" + kern[after:]
    while "asm volatile(" in kern:
        i = kern.index("asm volatile(")
        j = _statement(kern, i)
        copy = "cp.async.bulk.shared" in kern[i:j]
        kern = kern[:i] + ("std::memcpy(stage + st.head, src + st.head, st.body);" if copy else ";") + kern[j:]
    decl = "extern __shared__ __align__(16) unsigned char smem[];"
    assert decl in kern
    kern = kern.replace(decl, "unsigned char* smem = g_cta->smem;")
    hdr = open(os.path.join(CSRC, "kernels.cuh")).read()
    i = hdr.index("struct SlabArgs {")
    return hdr[i:hdr.index("};", i) + 2] + "\n" + kern + rules


@pytest.fixture(scope="module")
def exe(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    d = tmp_path_factory.mktemp("slab")
    (d / "probe.cpp").write_text("#include <barrier>\nint main() { std::barrier<> b(1); b.arrive_and_wait(); }\n")
    flags = ["-std=c++20", "-O1", "-g", "-fsanitize=thread", "-pthread", "-I", str(d), "-I", CSRC]
    if subprocess.run([cxx, *flags, str(d / "probe.cpp"), "-o", str(d / "probe")], capture_output=True).returncode or \
            subprocess.run([str(d / "probe")], capture_output=True).returncode:
        pytest.skip("no C++20 barrier or no race detector")
    (d / "cuda_runtime.h").write_text(SHIM + SHIM_EXTRA)
    (d / "slab.inc").write_text(host_slab_source())
    (d / "main.cpp").write_text(DRIVER)
    out = d / "slabcheck"
    r = subprocess.run([cxx, *flags, "-Wno-tsan", "-ffp-contract=off", str(d / "main.cpp"), "-o", str(out)],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return out


def reference(x, coef, M, N):
    """One slab [N, Nh] in float64: pad, inverse y, real x rows, coefficient / M^2, forward, truncate."""
    Nh, half = (N + 1) // 2, (N - 1) // 2
    at = np.where(np.arange(N) <= half, np.arange(N), np.arange(N) - N + M)
    full = np.zeros((M, Nh), complex)
    full[at] = x
    cols = np.fft.ifft(full, axis=0) * M
    spec = np.zeros((M, M), complex)
    spec[:, :Nh] = cols
    spec[:, 0] = spec[:, 0].real
    spec[:, M - np.arange(1, Nh)] = cols[:, 1:].conj()
    rows = (np.fft.ifft(spec, axis=1) * M).real * coef / M ** 2
    return np.fft.fft(np.fft.fft(rows, axis=1)[:, :Nh], axis=0)[at]


@pytest.mark.parametrize("M,N,warps", [(9, 5, 0), (9, 9, 2), (25, 13, 0), (25, 13, 3), (25, 25, 4), (81, 41, 0), (81, 41, 8),
                                       (81, 81, 0), (225, 113, 0), (225, 113, 8), (225, 111, 4)])
def test_slab_kernel(exe, tmp_path, M, N, warps):
    rng = np.random.default_rng([M, N, warps])
    nrc, Mz, Nh = 3, 1, (N + 1) // 2
    x = (rng.normal(size=(nrc, Mz, N, Nh)) + 1j * rng.normal(size=(nrc, Mz, N, Nh))).astype(np.complex64)
    coef = rng.uniform(1.0, 10.0, size=(Mz, M, M)).astype(np.float32)
    tw = np.exp(-2j * np.pi * np.arange(M) / M).astype(np.complex64)
    for name, v in (("x", x), ("c", coef), ("w", tw)):
        v.tofile(tmp_path / name)
    r = subprocess.run([str(exe), str(M), str(N), str(nrc), str(Mz), str(warps)] +
                       [str(tmp_path / f) for f in ("x", "c", "w", "y")], capture_output=True, text=True,
                       env={**os.environ, "TSAN_OPTIONS": "halt_on_error=1 exitcode=66"})
    assert r.returncode == 0, r.stderr[:4000]
    y = np.fromfile(tmp_path / "y", np.complex64).reshape(x.shape)
    assert (y[1] == x[1]).all()
    for rc in (0, 2):
        ref = reference(x[rc, 0].astype(complex), coef[0].astype(float), M, N)
        assert np.abs(y[rc, 0] - ref).max() <= 1e-5 * np.abs(ref).max()


def warps_of(exe, M, N, asked):
    return int(subprocess.run([str(exe), str(M), str(N), str(asked)], check=True, capture_output=True, text=True).stdout)


@pytest.mark.parametrize("M,N", [(9, 5), (25, 13), (81, 41), (225, 113), (9, 9), (25, 25), (81, 81)])
def test_asked_warps_are_taken_where_they_fit(exe, M, N):
    auto = warps_of(exe, M, N, 0)
    assert auto > 0
    for asked in (4, 8, 12, 16, 20):
        assert warps_of(exe, M, N, asked) == (auto if (M, asked) == (225, 20) else asked)


@pytest.mark.parametrize("M,N,warps", [(225, 113, 15), (81, 41, 7), (25, 13, 1), (9, 5, 1), (81, 81, 9), (25, 25, 2), (9, 9, 1)])
def test_automatic_warps(exe, M, N, warps):
    """The counts that the rule's comment names."""
    assert warps_of(exe, M, N, 0) == warps

"""Device functions of the tracers and dust kernels on the CPU: their source
is taken from the .cu / .cuh files as it stands, compiled with g++ over
cuda_on_host.h (lanes of a warp as threads) and run."""
import os
import re
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_1206_3710_gb300", "csrc")


def _source(name):
    with open(os.path.join(CSRC, name)) as f:
        return f.read()


def _take(name, start):
    """The definition that begins at the regular expression `start`, up to its
    closing brace (and the semicolon of a struct)."""
    text = _source(name)
    m = re.search(start, text, re.M)
    assert m, f"{name}: {start}"
    i = text.index("{", m.end() - 1 if text[m.end() - 1] == "{" else m.end())
    depth, j = 0, i
    while True:
        depth += {"{": 1, "}": -1}.get(text[j], 0)
        j += 1
        if depth == 0:
            break
    return text[m.start():j] + (";" if text[j:j + 1] == ";" else "") + "\n"


def _run(tmp_path, body, *args):
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text('#include "cuda_on_host.h"\n' + body)
    r = subprocess.run(["g++", "-std=c++17", "-O1", "-pthread", "-ffp-contract=off", "-w", "-I" + HERE, "-I" + CSRC,
                        str(src), "-o", str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-4000:]
    r = subprocess.run([str(exe), *map(str, args)], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, (r.returncode, r.stdout[-2000:], r.stderr[-2000:])
    return r.stdout


@pytest.mark.parametrize("n", [0, 1, 31, 33, 128, 129, 1000])
def test_work_items_are_given_out_once(tmp_path, n):
    """next_work: the warps of a grid take every item exactly once when a
    lane's store to the warp's state reaches the other lanes no sooner than
    the memory model promises it (at a __syncwarp)."""
    body = _take("rt_trace.cu", r"^__device__ __forceinline__ long long next_work\(") + r"""
int main(int argc, char** argv) {
  const long long n = atoll(argv[1]);
  gridDim.x = 2;
  blockDim.x = 64;
  unsigned long long counter = 0;
  std::vector<std::atomic<int>> given((size_t)n);
  for (auto& g : given) g = 0;
  for (unsigned b = 0; b < gridDim.x; ++b)
    for (unsigned w = 0; w < blockDim.x / 32; ++w) {
      on_lanes(32, [&](int lane) {
        threadIdx.x = 32 * w + (unsigned)lane;
        blockIdx.x = b;
        int state = 0;  // this lane's view of the warp's shared variable
        warp_state->view[lane] = &state;
        unsigned dead = 0xFFFFFFFFu, done = 0u, rnd = 12345u + 7u * b + w;
        while (done != 0xFFFFFFFFu) {
          const bool mine = dead >> lane & 1u;
          const long long i = next_work(&counter, n, dead, __ffs(dead) - 1, lane, state);
          if (mine && i >= 0 && i < n) given[(size_t)i].fetch_add(1);
          // lanes without an item are done, some of the others die (all lanes
          // agree on the masks, as by a ballot)
          warp_state->slot[lane] = mine && i >= n;
          meet(0xFFFFFFFFu);
          for (int l = 0; l < 32; ++l)
            if (warp_state->slot[l]) done |= 1u << l;
          rnd = rnd * 1664525u + 1013904223u;
          dead = (rnd >> 3 | rnd << 7) & ~done;
          if (dead == 0u) dead = ~done;
          meet(0xFFFFFFFFu);
        }
      });
    }
  for (long long i = 0; i < n; ++i)
    if (given[(size_t)i] != 1) {
      printf("item %lld given %d times\n", i, given[(size_t)i].load());
      return 1;
    }
  return 0;
}
"""
    _run(tmp_path, body, n)


def _num(kind):
    """The number traits, without the accessors of the device tables."""
    t = _take("rt_device.cuh", r"^template <>\nstruct Num<%s> \{" % kind)
    return "template <typename R>\nstruct Num;\n" + re.sub(r"^.*\b(BinDev|ItemDev|JobDev)\b.*\}\n", "", t, flags=re.M)


@pytest.mark.parametrize("kind", ["float", "double"])
def test_finite_distance(tmp_path, kind):
    """Num::finite tells an exit distance (not negative) from the infinity and
    the NaNs, of either sign, that a zero direction component gives."""
    body = "#include <cmath>\n#include <float.h>\n" + _num(kind) + r"""
typedef KIND R;
int main() {
  const R big = sizeof(R) == 4 ? (R)FLT_MAX : (R)DBL_MAX, tiny = sizeof(R) == 4 ? (R)1e-45f : (R)4.9e-324;
  const R yes[] = {R(0), tiny, R(0.5), R(1.7320508), big};
  const R nan = (R)NAN, no[] = {(R)INFINITY, nan, -nan, R(0) * (R)INFINITY};
  int bad = 0;
  for (R v : yes)
    if (!Num<R>::finite(v)) printf("%g is not finite\n", (double)v), bad = 1;
  for (R v : no)
    if (Num<R>::finite(v)) printf("%s%g is finite\n", std::signbit(v) ? "-" : "+", (double)fabs(v)), bad = 1;
  return bad;
}
""".replace("KIND", kind)
    _run(tmp_path, body)


def test_face_ahead_of_tiny_components(tmp_path):
    """Num<float>::ahead is exactly 0 or 1 for every direction component whose
    reciprocal is finite: a fraction there would put the face ahead inside the
    cell, at distance zero for a package that sits on it.  Every float from
    the smallest to twice the smallest with a finite reciprocal, and its
    negative, then powers of two up to 1."""
    body = _num("float") + _take("rt_device.cuh", r"^template <typename R>\n__device__ __forceinline__ R inv_abs\(") + r"""
int main() {
  long long bad = 0;
  auto look = [&](float d) {
    const float s = Num<float>::ahead(d), i = inv_abs(d);
    const bool ok = d > 0.0f ? (s == 1.0f || i == INFINITY) && s >= 0.0f && s <= 1.0f : s == 0.0f;
    if (!ok && bad++ < 3) printf("d = %g (1/d = %g): ahead %.9g\n", d, i, s);
  };
  look(0.0f);
  look(-0.0f);
  for (unsigned u = 1; u <= 1u << 22; ++u) {
    look(__uint_as_float(u));
    look(-__uint_as_float(u));
  }
  for (float d = 1.0f; d > 1e-38f; d *= 0.5f) {
    look(d);
    look(-d);
  }
  return bad != 0;
}
"""
    _run(tmp_path, body)


def test_occupancy_is_the_launched_tracers(tmp_path):
    """A launch's grid is sized by the occupancy of the tracer that it starts:
    for both precisions, with and without peel-off, untiled and tiled, and
    every number of stored path levels, the kernel, block size and dynamic
    shared memory that the occupancy is asked for are the launch's."""
    text = _source("rt_trace.cu")
    form = re.search(r"^enum \{ PATH_NONE.*?^\}\n", text, re.M | re.S).group(0)
    host = text[text.index("template <typename K>\nstatic cudaError_t path_smem("):]
    host = host[:host.index("template <typename R, bool PEEL, int EST, bool HITS, bool LEVELS = false>\nstatic")]
    occ = text[text.rindex("template <", 0, text.index("static cudaError_t occ_t(")):]
    occ = occ[:occ.index("cudaError_t launch_walk(")]
    code = re.sub(r"(\w+)<<<(.*?)>>>\(", r"launch_of(\1, \2)(", form + host + occ, flags=re.S)
    depth = int(re.search(r"#define RT_ANC_MAX (\d+)", _source("rt_internal.cuh")).group(1))
    body = r"""
enum cudaError_t { cudaSuccess, cudaErrorOther };
enum { cudaFuncAttributeMaxDynamicSharedMemorySize };
typedef void* cudaStream_t;
enum { RT_EST_CONTINUOUS = 0, RT_EST_ANALOG = 1 };
struct JobDev; struct ItemDev;
struct PeelQueue {}; struct TileRun {};
struct LaunchCfg { int block = 256, blocks = 1, refill = 8, blocks_tiled = 1, ev_batch = 12, anc = 0; };
struct Use { const void* k = nullptr; int block = 0; size_t dyn = 0; };
static Use launched, asked;
template <typename R, int MODE> struct MaxThreads { static constexpr int value = sizeof(R) == 4 && MODE == 2 ? 224 : 256; };
template <typename R, bool PEEL, int EST, bool HITS, int MODE, bool LEVELS = false, bool SPLIT = false, int PATH = 0>
void trace_kernel() { static volatile int one; one = PATH; }
template <typename K> cudaError_t cudaFuncSetAttribute(K, int, int) { return cudaSuccess; }
static cudaError_t cudaGetLastError() { return cudaSuccess; }
template <typename K> cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessor(int* n, K k, int block, size_t dyn) {
  asked.k = (const void*)k; asked.block = block; asked.dyn = dyn; *n = 1;
  return cudaSuccess;
}
template <typename K> auto launch_of(K k, int, int block, size_t dyn, cudaStream_t) {
  launched.k = (const void*)k; launched.block = block; launched.dyn = dyn;
  return [](auto&&...) {};
}
""" + code + r"""
template <typename R, bool PEEL, int MODE>
static int look(int block, int anc) {
  LaunchCfg cfg;
  cfg.block = block;
  cfg.anc = anc;
  int n = 0;
  launch_mode<R, PEEL, RT_EST_CONTINUOUS, false, MODE, false, false>(nullptr, nullptr, 0, nullptr, 0, cfg, PeelQueue(),
                                                                    nullptr, TileRun());
  trace_occupancy(8 * sizeof(R), PEEL, block, &n, MODE, anc);
  if (launched.k == asked.k && launched.block == asked.block && launched.dyn == asked.dyn) return 0;
  printf("FP%d peel %d mode %d block %d levels %d: kernel %s, block %d / %d, shared %zu / %zu\n", (int)(8 * sizeof(R)),
         PEEL, MODE, block, anc, launched.k == asked.k ? "same" : "another", launched.block, asked.block, launched.dyn,
         asked.dyn);
  return 1;
}
int main() {
  int bad = 0;
  for (int block : {32, 256})
    for (int anc = 0; anc <= DEPTH; ++anc) {
      bad += look<float, false, 0>(block, anc) + look<float, true, 0>(block, anc);
      bad += look<float, false, 2>(block, anc) + look<float, true, 2>(block, anc);
      bad += look<double, false, 0>(block, anc) + look<double, true, 0>(block, anc);
      bad += look<double, false, 2>(block, anc) + look<double, true, 2>(block, anc);
    }
  return bad != 0;
}
""".replace("DEPTH", str(depth))
    _run(tmp_path, body)


def test_ali_temperatures(tmp_path):
    """temperature_weighted_kernel against bisection in long double, 40 cells:
    each cell's T within 1e-13 of the root of sum_b w_b E_b(T) = rhs / (rho V)
    whatever its start (rounding of the sum and of x = h nu / k T, eps each,
    moves T by a few eps; 1e-13 leaves room for weights near 1e-3), T_min and
    T_max where the target lies outside, zero density and cells not in use
    left out.  Then, where Newton's factor is largest (one bin, x near 690),
    500 cells that start just under 1e-9 from the root: their mean error is
    below 1e-16.  A step of 0.99e-9 that ends the iteration leaves x / 2 times
    its square, 3.4e-16, on the same side in every cell; rounding (2 eps of
    either sign) averages to 2e-17."""
    names = [r"^struct EmitBin \{", r"^__device__ __forceinline__ void planck_and_deriv\(",
             r"^__device__ __forceinline__ double leaf_mass\(", r"^__device__ __forceinline__ void emit_setup\(",
             r"^__device__ __forceinline__ double emit_term\(", r"^__device__ __forceinline__ double weighted_emission\("]
    consts = "".join(re.findall(r"^#define (?:\w+_CGS|FOUR_PI) .*\n", _source("rt_dust.cu"), re.M))
    body = r"""
#include "rt_planck.cuh"
static inline void __syncthreads() { meet(0xFFu); }
namespace rtk {
alignas(16) unsigned char smem[1 << 15];
""" + consts + "".join(_take("rt_dust.cu", n) for n in names) + \
        _take("rt_dust.cu", r"^__global__ void __launch_bounds__\(128\) temperature_weighted_kernel\(") + r"""
}
using namespace rtk;
typedef long double LD;
static LD emission(const std::vector<double>& lam, const std::vector<double>& kabs, const std::vector<double>& dnu,
                   const double* w, long long n, long long c, LD T) {
  LD s = 0;
  for (size_t b = 0; b < lam.size(); ++b) {
    // (the bin's frequency and h nu are rounded once, for all cells)
    const double nud = C_CGS / (lam[b] * 1e-4), hnu = H_CGS * nud;
    const LD nu = nud;
    s += (LD)w[b * n + c] * 4 * (LD)M_PIl * (LD)kabs[b] * (LD)dnu[b] * 2 * (LD)H_CGS * nu * nu * nu /
         ((LD)C_CGS * (LD)C_CGS) / expm1l((LD)hnu / ((LD)K_CGS * T));
  }
  return s;
}
static std::vector<double> solve(const std::vector<double>& lam, const std::vector<double>& kabs,
                                 const std::vector<double>& dnu, const std::vector<double>& w,
                                 const std::vector<double>& rhs, const std::vector<double>& rho,
                                 const std::vector<uint8_t>& use, std::vector<double> T, double Tmin, double Tmax) {
  const long long n = (long long)rhs.size();
  std::vector<uint32_t> child(n, 0u);
  std::vector<uint8_t> level(n, 1);
  gridDim.x = 1;
  blockDim.x = 8;
  on_lanes(8, [&](int) {
    temperature_weighted_kernel(rhs.data(), w.data(), use.data(), n, child.data(), rho.data(), level.data(), 2.0,
                                lam.data(), kabs.data(), dnu.data(), (int)lam.size(), Tmin, Tmax, T.data());
  });
  return T;
}
int main() {
  int bad = 0;
  unsigned rnd = 1u;
  auto uni = [&] { return (rnd = rnd * 1664525u + 1013904223u) * 2.3283064365386963e-10; };
  {
    const int nl = 12;
    const long long n = 40;
    std::vector<double> lam, kabs, dnu, w(nl * n), rhs(n), rho(n), T0(n), Tt(n);
    for (int b = 0; b < nl; ++b) {
      lam.push_back(0.3 * pow(10.0, 0.35 * b));
      kabs.push_back(300.0 * pow(lam[b] / 0.55, -1.8));
      dnu.push_back(0.8 * C_CGS / (lam[b] * 1e-4));
    }
    std::vector<uint8_t> use(n, 1);
    for (long long c = 0; c < n; ++c) {
      for (int b = 0; b < nl; ++b) w[b * n + c] = 1.0 - 0.999 * uni();
      rho[c] = 1e-19 * (1 + uni());  // V = 1 at level 1 of h0 = 2
      Tt[c] = 4.0 * pow(500.0, uni());
      if (c == 0) Tt[c] = 2.0;     // below T_min
      if (c == 1) Tt[c] = 5000.0;  // above T_max
      rhs[c] = (double)((LD)rho[c] * emission(lam, kabs, dnu, w.data(), n, c, Tt[c]));
      T0[c] = c % 4 == 0 ? 0.0 : c % 4 == 1 ? 2.7 : c % 4 == 2 ? 3000.0 : Tt[c] * 1.3;
    }
    rho[2] = 0.0;
    use[3] = 0;
    const std::vector<double> T = solve(lam, kabs, dnu, w, rhs, rho, use, T0, 2.7, 3000.0);
    for (long long c = 0; c < n; ++c) {
      LD lo = 2.7L, hi = 3000.0L;
      const LD target = c == 2 ? 0 : (LD)rhs[c] / (LD)rho[c];
      if (c != 2)
        while (hi - lo > 1e-17L * lo) {
          const LD mid = (lo + hi) / 2;
          if (mid == lo || mid == hi) break;
          (emission(lam, kabs, dnu, w.data(), n, c, mid) < target ? lo : hi) = mid;
        }
      const LD want = c == 0 || c == 2 ? 2.7L : c == 1 ? 3000.0L : c == 3 ? (LD)T0[3] : lo;
      if (fabsl((LD)T[c] - want) > 1e-13L * want) {
        printf("cell %lld: T %.17g, not %.17Lg\n", c, T[c], want);
        bad = 1;
      }
    }
  }
  {
    const long long n = 500;
    const std::vector<double> lam{1.0}, kabs{100.0}, dnu{1e14};
    std::vector<double> w(n, 1.0), rhs(n), rho(n, 1.0), T0(n), Tt(n);
    for (long long c = 0; c < n; ++c) {
      Tt[c] = H_CGS * C_CGS / 1e-4 / (K_CGS * (680.0 + 20.0 * uni()));
      rhs[c] = (double)emission(lam, kabs, dnu, w.data(), n, c, (LD)Tt[c]);
      T0[c] = Tt[c] * (1.0 + (c & 1 ? 0.99e-9 : -0.99e-9));
    }
    const std::vector<double> T = solve(lam, kabs, dnu, w, rhs, rho, std::vector<uint8_t>(n, 1), T0, 2.7, 3000.0);
    LD mean = 0;
    for (long long c = 0; c < n; ++c) mean += ((LD)T[c] - (LD)Tt[c]) / (LD)Tt[c] / n;
    printf("mean error %.3Lg\n", mean);
    if (fabsl(mean) > 1e-16L) bad = 1;
  }
  return bad;
}
"""
    _run(tmp_path, body)


@pytest.mark.parametrize("hx,short_form", [(8.6e-4, True), (1.09e-3, True), (1.11e-3, False), (1.7e-3, False)])
def test_wide_temperature_tables(tmp_path, hx, short_form):
    """dust_temperature on tables of log E = 5 log T (E = T^5, an exactly
    linear interpolant) of spacing hx: the short form of the inversion serves
    every cell inside the table to 1e-14 where its series holds, and is not
    begun where it does not."""
    body = r"""
struct double2 { double x, y; };
enum cudaError_t { cudaSuccess };
typedef void* cudaStream_t;
static cudaError_t cudaGetLastError() { return cudaSuccess; }
#define __log2f(x) log2f(x)
static inline void __syncthreads() {}
#include "rt_planck.cuh"
namespace rtk {
alignas(16) float lg[8192];
static long long quotients, general;
static double quotient(double a, double b) { ++quotients; return a / b; }
static double solve_by_table(double A, double mass, const double*, const double*, const double*, int, double, double,
                             const double*, int) { ++general; return pow(A / mass, 0.2); }
""" + _take("rt_dust.cu", r"^struct InvNode \{") + \
        _take("rt_dust.cu", r"^__device__ __forceinline__ double leaf_mass\(") + \
        _take("rt_dust.cu", r"^__global__ void __launch_bounds__\(256, 4\) temperature_kernel\(") + \
        re.sub(r"<<<.*?>>>", "", _take("rt_dust.cu", r"^cudaError_t dust_temperature\("), flags=re.S) + r"""
}
using namespace rtk;
int main(int argc, char** argv) {
  const int nt = 8192, n = 2000;
  const double hx = atof(argv[1]);
  std::vector<double> table(12 * nt + 2), rho(n, 1.0), A(n), T(n), want(n);
  double* tab = (double*)(((uintptr_t)table.data() + 15) / 16 * 16);
  for (int i = 0; i < nt; ++i) {
    InvNode N{};
    N.T = 2.7 * exp(i * hx);
    N.inv_e = 1.0 / pow(N.T, 5.0);
    N.c1 = 5.0 * hx;
    N.hx = hx;
    ((InvNode*)(tab + 3 * nt))[i] = N;
    ((float*)(tab + 11 * nt))[i] = (float)(5.0 * log2(N.T));
  }
  std::vector<uint32_t> child(n, 0u);
  std::vector<uint8_t> level(n, 0);
  for (int c = 0; c < n; ++c) {
    want[c] = 2.7 * exp(hx * (2.0 + (nt - 6.0) * (c + 0.37) / n));
    A[c] = pow(want[c], 5.0);
  }
  gridDim.x = 1;
  blockDim.x = 1;
  dust_temperature(A.data(), 1, n, child.data(), rho.data(), level.data(), 1.0, nullptr, nullptr, nullptr, 1, 2.7,
                   2.7 * exp((nt - 1) * hx), tab, nt, T.data(), 1, nullptr);
  double far = 0.0;
  for (int c = 0; c < n; ++c) far = std::max(far, fabs(T[c] / want[c] - 1.0));
  printf("%lld quotients, %lld general, error %.2g\n", quotients, general, far);
  const bool ok = atoi(argv[2]) ? quotients == n && general == 0 : quotients == 0 && general == n;
  return !(ok && far < 1e-14);
}
"""
    _run(tmp_path, body, hx, int(short_form))

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

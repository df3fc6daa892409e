"""The bounds-checked build's test of a triangle edge (tri_edge_broken in
csrc/kcommon.cuh, the code its kernels run before they use an edge's partner
points), compiled for the host: whole edges pass, and for every other word the
edge is refused, so that the points read after it lie within one edge."""
import os
import subprocess


ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SRC = r"""
#include <cstdio>
#include <vector>
#include "kcommon.cuh"
template <int N>
int run() {
  constexpr int E = 2, NF = 3 * N, n = E * NF;
  std::vector<int32_t> f(n);
  for (int g = 0; g < n; ++g) f[g] = g << 1 | 1;
  for (int k = 0; k < N; ++k) {  // edge 1 of element 0 (L side) meets edge 0 of element 1
    f[N + k] = (NF + N - 1 - k) << 1 | 1;
    f[NF + N - 1 - k] = (N + k) << 1;
  }
  int bad = 0;
  for (int own = 0; own < n; own += N) bad += frp::tri_edge_broken<N>(f.data(), n, own) != -1;
  // every other value of every word near the range, and far outside it
  for (int own = 0; own < n; own += N)
    for (int k = 0; k < N; ++k) {
      const int32_t keep = f[own + k];
      for (int32_t w = -9; w < 2 * n + 9; ++w)
        for (int32_t v : {w, w ^ (1 << 29), w ^ (1 << 30), (int32_t)(w ^ (1u << 31))}) {
          if (v == keep) continue;
          f[own + k] = v;
          if (frp::tri_edge_broken<N>(f.data(), n, own) < 0) {
            ++bad;
            std::printf("N %d own %d k %d word %d accepted\n", N, own, k, v);
          }
        }
      f[own + k] = keep;
    }
  return bad;
}
int main() { return run<2>() + run<3>() + run<4>() + run<5>(); }
"""


def test_broken_triangle_edges_are_refused(tmp_path):
    (tmp_path / "edge.cu").write_text(SRC)
    csrc = os.path.join(ROOT, "paper_2006_10967_gb300", "csrc")
    exe = str(tmp_path / "edge")
    r = subprocess.run(["nvcc", "-std=c++17", "-gencode", "arch=compute_103a,code=sm_103a", "-I", csrc, "-o", exe,
                        str(tmp_path / "edge.cu")], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([exe], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout

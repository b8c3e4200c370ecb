"""The z-march length of the fused 3D sweeps (host code of a header): the search stops early, and
gives what trying every length gives, at every shape."""
import subprocess

import pytest

SOURCE = """
#include <cstdio>
#include "ep_internal.cuh"
int main() {
  const int planes[] = {1, 2, 3, 7, 25, 64, 128, 200, 384, 512, 2001, 20001, 60001};
  const int edges[] = {2, 29, 41, 64, 128, 300, 384, 512, 1024};
  int bad = 0;
  for (int pz : planes)
    for (int px : edges)
      for (int py : edges)
        for (int ty : {8, 12, 20}) {
          ep::Geo g{};
          g.px = px; g.py = py; g.pz = pz;
          long long cost = 0, best = -1;
          const int kz = ep::fused3d_kz(g, 28, ty, 0, 1, &cost);
          const long long cols = (long long)((px + 27) / 28) * ((py + ty - 1) / ty);
          // one of the two SM counts the search can have asked for
          int want = 0;
          bool ok = false;
          for (long long sms : {148ll, 152ll}) {
            best = -1;
            for (int k = 1; k <= pz; ++k) {
              const long long c = (cols * ((pz + k - 1) / k) + sms - 1) / sms * (k + 4);
              if (best < 0 || c < best) { best = c; want = k; }
            }
            ok = ok || (want == kz && best == cost);
          }
          bad += !ok;
        }
  std::printf("%d\\n", bad);
  return bad != 0;
}
"""


def test_early_end_of_the_search_changes_nothing(tmp_path):
    from paper_2305_01701_gb300 import build as B
    try:
        cc = B.nvcc()
    except RuntimeError:
        pytest.skip("nvcc not found")
    src, exe = str(tmp_path / "kz.cu"), str(tmp_path / "kz")
    with open(src, "w") as f:
        f.write(SOURCE)
    subprocess.run([cc, *B.ARCH, "-O2", "-std=c++17", "--expt-relaxed-constexpr", "-I", B.CSRC, "-I", B.INCLUDE, src,
                    "-o", exe], check=True)
    r = subprocess.run([exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout

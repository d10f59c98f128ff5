"""The longest run of packed blocks that one warp of the flat plan folds
(csrc/attn.cu, compiled for the host): an fp32 accumulator's error grows with
the blocks it takes, so the weight of the fp16 windows, which lengthens every
block range, stays at no more than four blocks' time for 32 tokens."""

import shutil
import subprocess

import pytest

from test_flat_plan import HARNESS, _plan_source

MAIN = r"""
int main() {
  for (int it = 0; it < 4000; ++it) {
    const int hkv = 1 + (int)(next() %% 8), batch = 1 + (int)(next() %% 24);
    const long long top = 300 + (long long)(next() %% 70000);
    WorkSums w = {0, 0, 0, 0};
    long long chunks = 0;
    for (int b = 0; b < batch; ++b) {
      const int L = (int)(top / 4 + (long long)(next() %% (unsigned long long)(3 * top / 4)));
      const PairShape s = pair_shape(L, 128);
      w.nb += (long long)hkv * s.nb;
      w.nr += (long long)hkv * s.nr;
      w.np += hkv;
      chunks += (long long)hkv * ((L - s.Lq + 31) / 32);
    }
    const FlatGrid g = flat_grid(w, 152);
    if (g.k.cw != 2) continue;  // lighter weights: little work
    // the range of a plan in which 32 window tokens cost four blocks
    const long long range = (w.nb + 4 * chunks + g.k.sc * w.np + g.n_v - 1) / g.n_v;
    CHECK((g.N + g.n_v - 1) / g.n_v <= range);
  }
  printf("ok\n");
  return 0;
}
"""


def test_windows_do_not_lengthen_the_block_ranges(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no host C++ compiler")
    src = tmp_path / "ranges.cc"
    src.write_text((HARNESS[:HARNESS.index("int main()")] + MAIN) % _plan_source())
    exe = tmp_path / "ranges"
    subprocess.run([cxx, "-O2", "-std=c++17", str(src), "-o", str(exe)], check=True,
                   capture_output=True, text=True)
    out = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert out.returncode == 0, out.stdout + out.stderr

"""Which entries of the correction index are read as words: the words of every
block lie inside the index, at both alignments, and the blocks' words and the
entries read alone are all entries, once (csrc/tq_ew_pairs.cuh compiled for
the host)."""
import subprocess

PROGRAM = r"""
#include <cstdio>
#include <vector>

#include "tq_ew_pairs.cuh"

int main() {
  using namespace tq::ew;
  for (int odd = 0; odd < 2; ++odd)
    for (int total = 0; total <= 24; ++total)
      for (int m0 = 0; m0 <= total; ++m0)
        for (int m1 = m0; m1 <= total; ++m1) {
          std::vector<int> seen(total, 0);
          bool ok = true;
          const int end = pairs_end(odd, total), off[4] = {0, m0, m1, total};  // three blocks
          for (int b = 0; b < 3; ++b) {
            const int e = pairs_clamp(off[b], odd, end), e1 = pairs_clamp(off[b + 1], odd, end);
            if (e >= e1) continue;
            for (int w = (e + odd) / 2; w < (e1 + odd + 1) / 2; ++w) ok = ok && 2 * w - odd >= 0 && 2 * w + 1 - odd < total;
            for (int i = e; i < e1; ++i) ok = ok && i >= off[b] && i < off[b + 1] && !seen[i]++;
          }
          if (read_alone(false, odd, total)) ok = ok && !seen[0]++;
          if (read_alone(true, odd, total)) ok = ok && !seen[total - 1]++;
          for (int i = 0; i < total; ++i) ok = ok && seen[i];
          if (!ok) return printf("odd %d total %d blocks at %d, %d\n", odd, total, m0, m1), 1;
        }
  return 0;
}
"""


def test_words_of_every_block_stay_inside_the_index(tmp_path):
    from paper_2609_09240_gb300 import build
    (tmp_path / "pairs.cu").write_text(PROGRAM)
    exe = str(tmp_path / "pairs")
    subprocess.run([build.nvcc(), "-std=c++17", "-I", build.CSRC, str(tmp_path / "pairs.cu"), "-o", exe], check=True)
    r = subprocess.run([exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout

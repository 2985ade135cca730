"""CPU check of which words of a packed sequence the kernels load
(csrc/genasm_words.h, compiled for the host): each holds a base of the sequence,
and every base of the window lies in one. A sequence without bases at the window's
place, an empty one above all, has none loaded, whatever its address."""
import shutil
import subprocess
from pathlib import Path

import pytest

CSRC = Path(__file__).resolve().parent.parent / "paper_2203_15561_gb300" / "csrc"

PROGRAM = r"""
#include <cstdio>
#include <initializer_list>
#include "genasm_words.h"
int main() {
  for (uint32_t most : {32u, 64u, 80u, 96u, 128u, 144u})  // a window's bases, and the staged ones
    for (uint32_t byte = 0; byte < 4; ++byte)             // the sequence's first byte in its word
      for (uint32_t len = 0; len <= 300; ++len)
        for (uint32_t pos = 0; pos <= len + 3; ++pos) {
          const uint32_t o = 8u * ((byte + (pos >> 2)) & 3u) + 2u * (pos & 3u);
          const uint32_t end = ga::bases_end(o, len, pos, most);
          const uint32_t bases = pos < len ? (len - pos < most ? len - pos : most) : 0u;
          // The bases are bits o .. o + 2 bases - 1, in words 0 .. want - 1.
          const uint32_t want = bases ? (o + 2u * bases + 31u) / 32u : 0u;
          for (uint32_t k = 0; k < 12; ++k)
            if (ga::holds_base(k, o, end) != (k < want)) {
              std::printf("most %u byte %u len %u pos %u: word %u of %u\n", most, byte, len, pos, k, want);
              return 1;
            }
        }
  return 0;
}
"""


@pytest.mark.skipif(shutil.which("g++") is None, reason="needs g++")
def test_words_loaded_hold_a_base(tmp_path):
    (tmp_path / "words.cpp").write_text(PROGRAM)
    exe = tmp_path / "words"
    subprocess.run(["g++", "-std=c++17", "-O1", f"-I{CSRC}", str(tmp_path / "words.cpp"), "-o", str(exe)],
                   check=True, capture_output=True, text=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout

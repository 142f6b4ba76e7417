"""hac_dendrogram touches the pages of the caller's buffer before the copy: nothing in it
may change by that (the copy may still fail).  The routine is compiled here as
host code, straight from the library's source."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CORE = os.path.join(os.path.dirname(HERE), "paper_2106_04727_gb300", "csrc", "hac_core.cu")
CXX = shutil.which("g++") or shutil.which("c++")

MAIN = r"""
int main() {
  for (size_t bytes : {(size_t)0, (size_t)100, (size_t)1 << 20, ((size_t)1 << 20) + 4097,
                       ((size_t)9 << 20) + 33, (size_t)200 << 20})
    for (size_t shift : {(size_t)0, (size_t)8, (size_t)4095}) {
      std::vector<unsigned char> v(bytes + 8192);
      for (size_t i = 0; i < v.size(); ++i) v[i] = (unsigned char)(i * 131 + 17);
      touch_pages(v.data() + shift, bytes);
      for (size_t i = 0; i < v.size(); ++i)
        if (v[i] != (unsigned char)(i * 131 + 17)) {
          printf("byte %zu of %zu (shift %zu) changed\n", i, bytes, shift);
          return 1;
        }
    }
  return 0;
}
"""


@pytest.mark.skipif(CXX is None, reason="no host compiler")
def test_touching_changes_nothing(tmp_path):
    text = open(CORE).read()
    a = text.index("static void touch_pages(")
    body = text[a:text.index("\n}\n", a) + 3]
    src = tmp_path / "touch.cpp"
    src.write_text("#include <errno.h>\n#include <sys/mman.h>\n#include <unistd.h>\n"
                   "#include <algorithm>\n#include <cstddef>\n#include <cstdint>\n"
                   "#include <cstdio>\n#include <thread>\n#include <vector>\n" + body + MAIN)
    exe = tmp_path / "touch"
    r = subprocess.run([CXX, "-O2", "-std=c++17", "-pthread", str(src), "-o", str(exe)],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-2000:]
    out = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert out.returncode == 0, out.stdout

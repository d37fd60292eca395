"""Scratch of the radix sort, on the CPU: sized for n rows it holds a sort of
any fewer rows too, on either side of every change of the tile."""
import subprocess

import pytest

from paper_2106_06889_gb300 import _build

MAIN = """
#include <cstddef>
#include <cstdint>
#include <cstdio>
#include <cstdlib>
namespace gt { size_t radix_scratch_bytes(int64_t, bool, int); }
int main(int argc, char** argv) {
  for (int i = 1; i < argc; ++i) std::printf("%zu\\n", gt::radix_scratch_bytes(atoll(argv[i]), true, 4));
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    """The engine's objects and a main that calls the size function (internal: the library does not export it)."""
    objs = [_build.BUILD / (s.stem + ".o") for s in _build.gtadoc_sources()]
    _build.build_gtadoc(force=not all(o.exists() for o in objs))
    d = tmp_path_factory.mktemp("scratch")
    (d / "main.cpp").write_text(MAIN)
    subprocess.run([_build._nvcc(), *_build.ARCH, str(d / "main.cpp"), *map(str, objs), "-o", str(d / "main"), "-lcudart"],
                   check=True)
    return d / "main"


def test_scratch_never_shrinks(program):
    edges = [1, 2048, 6144, 8192, 400_000, 1 << 20, 171 * 6144, 1 << 22, 1 << 30, 1 << 32]
    ns = sorted({max(1, e + k) for e in edges for k in (-1, 0, 1)})
    out = subprocess.run([str(program), *map(str, ns)], check=True, capture_output=True, text=True).stdout
    sizes = [int(x) for x in out.split()]
    assert len(sizes) == len(ns) and all(a <= b for a, b in zip(sizes, sizes[1:])), list(zip(ns, sizes))

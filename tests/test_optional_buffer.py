"""The buffer that a distance query can do without (csrc/optional_buffer.h, compiled
as C++) against an allocator that refuses large requests: a refused size costs one
attempt, not one per call, and what is held stays in place."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2203_14362_gb300", "csrc")
DRIVER = r"""
#include "optional_buffer.h"
#include <cstdio>
#include <cstdlib>
using spx::OptionalBuffer;
#define CHECK(x) do { if (!(x)) { std::printf("line %d: %s\n", __LINE__, #x); return 1; } } while (0)
int main()
{
    size_t limit = 1000;
    int tries = 0, freed = 0;
    auto alloc = [&](void **p, size_t n) { ++tries; if (n > limit) return false; *p = std::malloc(n); return true; };
    auto release = [&](void *p) { ++freed; std::free(p); };
    OptionalBuffer b;
    CHECK(b.want(0, alloc, release) == nullptr && tries == 0);
    void *first = b.want(400, alloc, release);
    CHECK(first && tries == 1 && b.bytes == 400);
    CHECK(b.want(400, alloc, release) == first && b.want(1, alloc, release) == first && tries == 1);
    for (int i = 0; i < 100; ++i) // refused once, then not asked for; the smaller one stays
        CHECK(b.want(5000, alloc, release) == nullptr);
    CHECK(tries == 2 && freed == 0 && b.p == first && b.want(300, alloc, release) == first);
    CHECK(b.want(6000, alloc, release) == nullptr && tries == 2); // larger than a refused one
    void *second = b.want(900, alloc, release); // smaller than it
    CHECK(second && tries == 3 && freed == 1 && b.bytes == 900);
    CHECK(b.want(5000, alloc, release) == nullptr && tries == 4); // memory moved: asked once more
    limit = 10000;
    b.retry(); // memory was freed
    CHECK(b.want(5000, alloc, release) && tries == 5 && freed == 2 && b.bytes == 5000);
    limit = 0;
    CHECK(b.want(8000, alloc, release) == nullptr && tries == 6);
    limit = 10000;
    int calls = 0;
    while (!b.want(8000, alloc, release)) // others may have freed memory: asked again after a while
        CHECK(++calls < 1000);
    CHECK(calls + 1 == (int)OptionalBuffer::kSkip && tries == 7);
    std::free(b.p);
    return 0;
}
"""


def test_optional_buffer(tmp_path):
    if not shutil.which("g++"):
        pytest.skip("no g++")
    (tmp_path / "t.cpp").write_text(DRIVER)
    subprocess.run(["g++", "-O1", "-std=c++17", "-Wall", "-Werror", "-I", CSRC, "-o", str(tmp_path / "t"), str(tmp_path / "t.cpp")],
                   check=True)
    r = subprocess.run([str(tmp_path / "t")], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout

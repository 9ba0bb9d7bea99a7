"""The grid barrier's wait ends at its own generation or any later one (no GPU: the
predicate's own source is compiled by itself).  A CTA that leaves after a barrier
the others go on from may look at the word only after it has moved on."""
import ctypes
import os
import re
import subprocess

import pytest

from paper_1412_1127_gb300 import build

MASK = 0x7fffffff


@pytest.fixture(scope="module")
def reached(tmp_path_factory):
    src = open(os.path.join(build.CSRC, "patterns.cu")).read()
    body = re.search(r"__host__ __device__ __forceinline__ bool generation_reached.*?\n\}\n", src, re.S).group(0)
    wait = re.search(r"int grid_barrier_or\(.*?\n\}\n", src, re.S).group(0)
    assert "(v >> 1) == my" not in wait and "(v >> 1) != my" not in wait  # waits go through the predicate
    assert wait.count("generation_reached(v, my)") == 2
    d = tmp_path_factory.mktemp("barrier")
    cpp, lib = os.path.join(d, "b.cpp"), os.path.join(d, "b.so")
    with open(cpp, "w") as f:
        f.write("#define __host__\n#define __device__\n#define __forceinline__ inline\n" + body +
                'extern "C" int run(unsigned w, unsigned g) { return generation_reached(w, g); }\n')
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", cpp, "-o", lib], check=True)
    L = ctypes.CDLL(lib)
    L.run.argtypes = [ctypes.c_uint, ctypes.c_uint]
    return lambda gen_seen, flag, gen: bool(L.run(((gen_seen & MASK) << 1) | flag, gen & MASK))


@pytest.mark.parametrize("gen", [1, 2, 1000, MASK - 1, MASK, 0])  # the last ones wrap
@pytest.mark.parametrize("flag", [0, 1])
def test_own_and_later_generations_end_the_wait(reached, gen, flag):
    for ahead in (0, 1, 2, 50, 100000):
        assert reached(gen + ahead, flag, gen)
    for behind in (1, 2, 100000):
        assert not reached(gen - behind, flag, gen)

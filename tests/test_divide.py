"""The kernels' division by a number that the host knows (csrc/lossy_divide.h), compiled for the host: floor(x m / 2^64) with m = 2^64 / d
rounded up, in the two products that are taken of it, is x / d for every 32-bit x and d."""
import ctypes as C
import os
import random
import subprocess

from paper_2507_07114_b200 import build

SOURCE = """
#include "lossy_divide.h"
extern "C" uint32_t quotient(uint32_t x, uint32_t d) { return lossy::divide_by(x, d, lossy::magic_of(d)); }
extern "C" uint64_t wrong(uint32_t d, uint32_t from, uint64_t count) {   // quotients of `count` numbers from `from` on that differ from x / d
  uint64_t n = 0;
  const uint64_t magic = lossy::magic_of(d);
  for (uint64_t x = from; x < from + count && x <= 0xFFFFFFFFull; ++x) n += lossy::divide_by((uint32_t)x, d, magic) != (uint32_t)x / d;
  return n;
}
"""


def test_division_by_multiplication(tmp_path):
    src, lib = tmp_path / "divide.cpp", tmp_path / "divide.so"
    src.write_text(SOURCE)
    subprocess.run([os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-fPIC", "-shared", "-D__host__=", "-D__device__=", "-D__forceinline__=inline",
                    "-I", build.CSRC, str(src), "-o", str(lib)], check=True, capture_output=True)
    f = C.CDLL(str(lib))
    f.quotient.argtypes, f.quotient.restype = [C.c_uint32, C.c_uint32], C.c_uint32
    f.wrong.argtypes, f.wrong.restype = [C.c_uint32, C.c_uint32, C.c_uint64], C.c_uint64
    rng, top = random.Random(3), 2 ** 32 - 1
    for d in [1, 2, 3, 7, 64, 641, 2 ** 16 - 1, 2 ** 16 + 1, 2 ** 31, top] + [rng.randrange(1, 2 ** rng.randrange(2, 33)) for _ in range(2000)]:
        for x in (0, 1, d - 1, d, top, top // d * d, top // d * d - 1, rng.randrange(top + 1)):
            assert f.quotient(x, d) == x // d, (x, d)
        for at in (0, top // d * d - 500, rng.randrange(top)):       # on both sides of a multiple, low and high
            assert f.wrong(d, max(at, 0), 1000) == 0, d

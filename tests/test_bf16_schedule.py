"""The choice of column tiles of a BF16 launch (host code of its launcher), compiled for the host: the estimate against a walk of
every tile, the search against all schedules, and what a new shape costs."""
import ctypes
import os
import random
import subprocess

import pytest

from conftest import ROOT

SOURCE = """
#include "bf16_schedule.h"
using namespace nvfp4;
static void walks(const int* p, int n, Bf16Walk* w, int base = 4096) {
  for (int i = 0; i < n; ++i) w[i] = bf16_walk(p[5 * i], p[5 * i + 1], p[5 * i + 2], base, p[5 * i + 3], base, p[5 * i + 4]);
}
extern "C" int on_sector(unsigned long long base, long long ld) { return bf16_on_sector(base, ld); }
extern "C" long long estimate(const int* p, int n, int pairs, int w0, int w1, int lower) {
  Bf16Walk w[2];
  walks(p, n, w);
  const Bf16Estimate e(w, n, pairs);
  return lower ? e.least(Bf16Wide{{w0, w1}}) : e.until_the_last(Bf16Wide{{w0, w1}});
}
extern "C" int choose(const int* p, int n, int pairs, int remember, int base, int* wide) {
  Bf16Walk w[2];
  walks(p, n, w, base);
  int walked = 0;
  const Bf16Wide v = remember ? bf16_wide_tiles(w, n, pairs, &walked) : bf16_wide_search(w, n, pairs, &walked);
  wide[0] = v.n[0];
  wide[1] = v.n[1];
  return walked;
}
"""


@pytest.fixture()
def lib(tmp_path):
    src, so = tmp_path / "schedule.cpp", tmp_path / "libschedule.so"
    src.write_text(SOURCE)
    subprocess.run(["g++", "-std=c++17", "-O1", "-fPIC", "-shared", "-pthread", "-o", str(so), str(src),
                    "-I" + os.path.join(ROOT, "paper_2509_25149_b200", "csrc")], check=True)
    lib = ctypes.CDLL(str(so))
    lib.estimate.restype = ctypes.c_longlong
    return lib


def forward(M, N, K):
    return [(M, N, K, K, K)]  # M, N, K, leading dimensions


def backward(M, N, K):
    products = [(M, K, N, N, K), (N, K, M, N, K)]  # dX and dW of a layer, the longer contraction first
    return products if N >= M else products[::-1]


def _flat(products):
    return (ctypes.c_int * 10)(*[v for p in products for v in p])


def choose(lib, products, pairs=74, remember=False, base=4096):
    wide = (ctypes.c_int * 2)()
    walked = lib.choose(_flat(products), len(products), pairs, int(remember), base, wide)
    return (wide[0], wide[1]), walked


def walk_every_tile(products, pairs, wide):
    """Cycles until the last pair is done, one tile after the other."""
    tiles = []
    for halves in (2, 1):
        for (M, N, K, lda, ldb), w in zip(products, wide):
            def bytes_(ld):
                return 16384.0 * (1.75 - 0.375 * (1 if ld % 16 else 2))
            k_block = max(halves * 530.0, (bytes_(lda) + halves * bytes_(ldb)) / 63.0)
            cols = w if halves == 2 else -(-N // 256) - 2 * w
            if halves == 1 and sum(wide) and len(products) == 2:
                k_block *= 1.04  # 256-wide tiles beside wide ones in a launch of two products
            tiles += [(k_block * -(-K // 64) + (3000 if halves == 2 else 500), halves)] * (-(-M // 256) * cols)
    load, last = [0.0] * pairs, [0] * pairs
    for i, (cost, halves) in enumerate(tiles):
        p = i % pairs
        if sum(wide) and (i // pairs) & 1:
            p = pairs - 1 - p
        load[p] += cost
        last[p] = 3000 if halves == 2 else 0
    return max(a + b for a, b in zip(load, last)), len(tiles)


def test_the_estimate_is_a_walk_of_every_tile(lib):
    rng = random.Random(3)
    for _ in range(400):
        M, N, K = (8 * rng.randint(1, hi) for hi in (600, 600, 300))
        products = rng.choice([forward, backward])(M, N, K)
        pairs = rng.choice([1, 2, 7, 66, 74])
        wide = [rng.randint(0, -(-p[1] // 256) // 2) for p in products]
        want, tiles = walk_every_tile(products, pairs, wide)
        args = _flat(products), len(products), pairs, *(wide + [0])[:2]
        got, least = lib.estimate(*args, 0), lib.estimate(*args, 1)
        assert abs(got - want) <= tiles, (products, pairs, wide)  # (a tile's cycles are whole numbers there)
        assert least <= got + 1 or not sum(wide)


def test_rows_that_begin_on_32_bytes(lib):
    """Operands need 16-byte alignment only: a slice whose rows are a multiple of 32 bytes apart may begin beside one."""
    lib.on_sector.argtypes = [ctypes.c_ulonglong, ctypes.c_longlong]
    for base in range(4096, 4096 + 128, 16):
        for ld in (8, 16, 24, 32, 40, 48, 64, 96, 1024, 5120, 5128, 5136, 5152):
            assert lib.on_sector(base, ld) == sum((base + 2 * ld * r) % 32 == 0 for r in range(2)), (base, ld)
    aligned, beside = (choose(lib, [(1536, 4608, 1024, 1056, 1056)], base=b, remember=True)[0] for b in (4096, 4112))
    assert aligned == (0, 0) and beside[0] > 0


def test_no_schedule_is_estimated_shorter_than_the_chosen_one(lib):
    for products in (forward(4088, 5128, 5112), forward(2048, 7168, 2056), forward(1040, 3664, 904), forward(4096, 4096, 4096),
                     backward(1544, 1680, 1912), backward(3000, 3000, 1000), backward(4096, 2048, 1024)):
        args = _flat(products), len(products), 74
        narrow = lib.estimate(*args, 0, 0, 0)
        most = [-(-p[1] // 256) // 2 if p[2] > 832 else 0 for p in products] + [0]
        all_ = min(lib.estimate(*args, i, j, 0) for i in range(most[0] + 1) for j in range(most[1] + 1) if i + j)
        wide, _ = choose(lib, products)
        assert lib.estimate(*args, *wide, 0) == (all_ if all_ < int(0.97 * narrow) else narrow)


def test_launches_of_both_widths(lib):
    """What 74 pairs get for the shapes that the GPU tests name for their tiles of both widths: column tiles 512 wide of each product."""
    for shape, want in {(1608, 2600, 968): 1, (1056, 3960, 1032): 2, (2056, 7176, 1064): 13}.items():
        assert choose(lib, forward(*shape))[0] == (want, 0), shape
    for shape, want in {(1040, 3664, 904): (0, 1), (1112, 1144, 2344): (1, 5), (1224, 1192, 2328): (1, 5)}.items():
        assert choose(lib, backward(*shape))[0] == want, shape


def test_what_a_new_shape_costs(lib):
    """A call searches where its shape is new: schedules that cannot be the shortest are not walked through, and token counts that
    differ within a tile are one shape."""
    rng = random.Random(5)
    walked = []
    for _ in range(500):
        M, N, K = (8 * rng.randint(64, 2560) for _ in range(3))
        walked.append(choose(lib, backward(M, N, K))[1])
    assert max(walked) <= 289 and sum(walked) <= 80 * len(walked)
    assert choose(lib, backward(4096, 4096, 4096))[1] <= 40 and choose(lib, backward(16384, 20480, 5120))[1] <= 40
    for i in range(1000):
        M = 4096 - 8 * (i % 32)
        first = choose(lib, backward(M, 5128, 5112), remember=True)
        assert first[0] == choose(lib, backward(-(-M // 64) * 64, 5128, 5112))[0]
        assert (first[1] > 0) == (i % 32 in (0, 8, 16, 24) and i < 32), i  # (every 64 tokens there is a k-block less in dW)

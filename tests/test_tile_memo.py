"""The table of remembered tile choices (host code of the GEMM launchers), compiled for the host: any number of shapes, one answer
per device."""
import ctypes
import os
import subprocess

import pytest

from conftest import ROOT

SOURCE = """
#include "tile_memo.h"
static nvfp4::TileMemo memo;
extern "C" int find(const int* key) {
  int k[nvfp4::TileMemo::kKey], tile = -1;
  std::copy(key, key + nvfp4::TileMemo::kKey, k);
  return memo.find(k, &tile) ? tile : -1;
}
extern "C" void put(const int* key, int tile) {
  int k[nvfp4::TileMemo::kKey];
  std::copy(key, key + nvfp4::TileMemo::kKey, k);
  memo.put(k, tile);
}
"""


@pytest.fixture()
def memo(tmp_path):
    src, so = tmp_path / "memo.cpp", tmp_path / "libmemo.so"
    src.write_text(SOURCE)
    subprocess.run(["g++", "-std=c++17", "-O1", "-fPIC", "-shared", "-pthread", "-o", str(so), str(src),
                    "-I" + os.path.join(ROOT, "paper_2509_25149_b200", "csrc")], check=True)
    return ctypes.CDLL(str(so))


def _key(m, device=0):
    return (ctypes.c_int * 8)(m, 512, 1024, 0, 0, 0, 1, device)


def test_the_newest_shapes_are_remembered(memo):
    for i in range(1000):
        assert memo.find(_key(i)) == -1
        memo.put(_key(i), i)
        assert memo.find(_key(i)) == i  # also when the table is full
        assert memo.find(_key(max(0, i - 255))) == max(0, i - 255)
    assert memo.find(_key(1000 - 257)) == -1 and memo.find(_key(999)) == 999


def test_a_choice_belongs_to_a_device(memo):
    memo.put(_key(256, device=0), 642)
    assert memo.find(_key(256, device=1)) == -1
    memo.put(_key(256, device=1), 640)
    assert memo.find(_key(256, device=0)) == 642 and memo.find(_key(256, device=1)) == 640

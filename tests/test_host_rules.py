"""The host-side rules that need no GPU (csrc/host_rules.h), compiled by themselves."""
import ctypes
import os
import subprocess

import pytest

from paper_2601_13143_b200 import build

SOURCE = """
#include "host_rules.h"
extern "C" int inside(unsigned long long at, unsigned long long bytes, unsigned long long start, unsigned long long size) {
  return fastav::inside_range(at, bytes, start, size);
}
extern "C" int blocks(int batch, int max_seqlen, int slice, int limit) { return fastav::cluster_blocks(batch, max_seqlen, slice, limit); }
"""


@pytest.fixture(scope="module")
def rules(tmp_path_factory):
    where = tmp_path_factory.mktemp("rules")
    source, lib = where / "rules.cpp", where / "rules.so"
    source.write_text(SOURCE)
    subprocess.run([os.environ.get("CXX", "g++"), "-std=c++17", "-Wall", "-Werror", "-shared", "-fPIC", f"-I{build.CSRC}", "-o", str(lib), str(source)], check=True)
    return ctypes.CDLL(str(lib))


@pytest.mark.parametrize("at,bytes_,start,size,inside", [
    (100, 50, 100, 50, True), (100, 51, 100, 50, False), (99, 10, 100, 50, False), (149, 1, 100, 50, True), (150, 0, 100, 50, True),
    (120, 40, 100, 50, False), (0, 1 << 40, 1 << 39, 1 << 41, False), ((1 << 64) - 16, 16, (1 << 64) - 32, 32, True),
    ((1 << 64) - 16, 32, (1 << 64) - 32, 32, False), (100, (1 << 64) - 50, 100, 50, False),
])
def test_an_array_is_inside_one_range_or_not(rules, at, bytes_, start, size, inside):
    """Two registrations with a gap between them are two ranges: the first byte's range has to hold the last byte too."""
    u64 = ctypes.c_uint64
    assert rules.inside(u64(at), u64(bytes_), u64(start), u64(size)) == inside


@pytest.mark.parametrize("batch,tokens,slice_,sixteen,eight", [
    (1, 2048, 32, 16, 8), (1, 512, 32, 16, 8), (1, 257, 32, 16, 8), (1, 256, 32, 8, 8), (7, 2048, 32, 16, 8), (8, 2048, 32, 8, 8), (16, 2048, 32, 4, 4),
    (1, 2048, 256, 8, 8), (75, 2048, 32, 1, 1), (149, 100, 32, 1, 1), (1, 0, 32, 1, 1),
])
def test_blocks_per_sequence_keep_within_what_can_be_placed(rules, batch, tokens, slice_, sixteen, eight):
    assert rules.blocks(batch, tokens, slice_, 16) == sixteen
    assert rules.blocks(batch, tokens, slice_, 8) == eight

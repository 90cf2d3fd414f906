"""The store of captured launch chains (csrc/chain_store.h, plain C++): what is captured, kept and given up for what."""
import os
import subprocess

import pytest

from conftest import ROOT

DRIVER = r"""
#include <cstdio>
#include "chain_store.h"
// reads keys, one per line; prints r (replayed), c (captured) or b (launched bare) for each
int main() {
    rp::ChainStore s{};
    unsigned long long k;
    while (std::scanf("%llu", &k) == 1) {
        int slot = s.find(k);
        if (slot >= 0) { std::putchar('r'); continue; }
        slot = s.place(k);
        if (slot >= 0) s.put(slot, k);
        std::putchar(slot >= 0 ? 'c' : 'b');
    }
    return 0;
}
"""


@pytest.fixture(scope="module")
def store(tmp_path_factory):
    d = tmp_path_factory.mktemp("chain_store")
    (d / "driver.cpp").write_text(DRIVER)
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-Wall", "-Werror", "-I", os.path.join(ROOT, "paper_2601_12347_b200", "csrc"),
                           str(d / "driver.cpp"), "-o", str(d / "driver")])
    return lambda keys: subprocess.run([str(d / "driver")], input="\n".join(map(str, keys)), capture_output=True, text=True, check=True).stdout


def test_a_geometry_is_captured_when_it_comes_back(store):
    assert store([7, 8, 7, 7, 8, 9, 8]) == "bbcrcbr"


def test_a_round_of_more_geometries_than_slots_is_not_captured_over_and_over(store):
    out = store(list(range(1, 21)) * 50)
    assert out.count("c") == 16
    assert out[40:].count("r") == 16 * 48        # the sixteen that fit are replayed from then on


def test_a_chain_gives_way_once_the_stream_has_moved_on(store):
    first, then = list(range(1, 17)), list(range(101, 117))
    out = store(first * 3 + then * 3)
    assert out[48:] == "b" * 16 + "c" * 16 + "r" * 16
    # ... the least recently used one first, and a chain still in use stays
    out = store(first * 3 + [1, 50] * 3 + [1])
    assert out[48:] == "rbrcrrr"
    assert store(first * 3 + [1, 50] * 3 + [2, 2, 2])[-3:] == "bcr"     # the one that gave way starts over


def test_geometries_seen_long_ago_are_forgotten(store):
    assert store([5] + list(range(100, 140)) + [5, 5, 5])[-3:] == "bcr"

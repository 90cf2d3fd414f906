"""When a hop is swept instead of pushed (csrc/sweep_rule.h, plain C++): the rule of the device and that of the host."""
import os
import subprocess

import pytest

from conftest import ROOT

DRIVER = r"""
#include <cstdio>
#include "sweep_rule.h"
// reads lines of: messages, senders, edges, vertices, width; prints for each 0/1 whether the device sweeps, whether the
// host has both forms in the chain of the batch after one that carried as much, and whether a sweep that the caller wants
// reads every list; "stream" in the arguments: one stream of batches, what the host has in the chain lasts from line to line
int main(int argc, char**) {
    double m, s, e, v;
    int w;
    bool armed = false;
    while (std::scanf("%lf %lf %lf %lf %d", &m, &s, &e, &v, &w) == 5) {
        const bool may = rp::sweep_may_pay(true, argc > 1 && armed, m, s, e, v, w);
        std::printf("%d%d%d\n", (int)rp::sweep_pays(m, s, e, v, w), (int)may, (int)rp::sweep_reads_all(m, e));
        armed = may;
    }
    return 0;
}
"""


@pytest.fixture(scope="module")
def rule(tmp_path_factory):
    d = tmp_path_factory.mktemp("sweep_rule")
    (d / "driver.cpp").write_text(DRIVER)
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-Wall", "-Werror", "-I", os.path.join(ROOT, "paper_2601_12347_b200", "csrc"),
                           str(d / "driver.cpp"), "-o", str(d / "driver")])

    def ask(hops, *args):
        out = subprocess.run([str(d / "driver"), *args], input="\n".join(" ".join(map(str, h)) for h in hops), capture_output=True, text=True, check=True)
        return [tuple(c == "1" for c in line) for line in out.stdout.split()]
    return ask


DENSE = (123_718_280, 2_449_029)


def test_the_measured_hops_fall_on_their_side(rule):
    swept = [(990_000, 80_000, 1_166_243, 169_343, 256), (1_100_000, 80_000, 1_166_243, 169_343, 40),
             (20_000_000, 9_000, *DENSE, 256)]
    pushed = [(26_000_000, 9_000, *DENSE, 48), (2_068, 3, *DENSE, 256), (1_500_000, 300, *DENSE, 256), (8_000, 200, *DENSE, 104)]
    assert [r[0] for r in rule(swept)] == [True] * 3
    assert [r[0] for r in rule(pushed)] == [False] * 4


def test_what_the_device_may_sweep_is_in_the_chain(rule):
    """A hop that is swept was in the chain if the batch before carried at least half as much, at every size."""
    hops = [(m, m / k, e, v, w) for m in (1e4, 1e5, 1e6, 1e7, 1e8) for k in (10, 300, 10_000) for e, v in ((1.2e6, 1.7e5), DENSE)
            for w in (16, 48, 104, 256, 1024) if m <= e]
    half = [(m / 2, s / 2, e, v, w) for m, s, e, v, w in hops]
    device = [r[0] for r in rule(hops)]
    assert any(device) and not all(device)
    for sweeps, before in zip(device, rule(half)):
        assert not sweeps or before[1]


def test_a_small_hop_does_not_read_the_whole_graph(rule):
    small = [(m, 10, *DENSE, w) for m in (0, 9, 22_000, 2_300_000) for w in (48, 256)]
    large = [(m, 10_000, *DENSE, w) for m in (20_000_000, 122_000_000) for w in (48, 256)]
    assert not any(r[2] for r in rule(small)) and all(r[2] for r in rule(large))


@pytest.mark.parametrize("width, edges, vertices, senders", [(256, *DENSE, 5_000), (128, 1_166_243, 169_343, 20_000), (40, 1_166_243, 169_343, 10_000)])
def test_a_stream_near_the_line_keeps_its_chain(rule, width, edges, vertices, senders):
    """Batches that carry between 0.75 and 1.3 times what a hop needs to bring the sweep into the chain."""
    lo, hi = 1.0, float(edges)
    for _ in range(60):     # the least number of messages after which both forms are in the chain
        mid = (lo * hi) ** 0.5
        lo, hi = (lo, mid) if rule([(mid, senders, edges, vertices, width)])[0][1] else (mid, hi)
    assert 1.0 < hi < edges
    sizes = [0.8, 1.3, 0.75, 1.1, 0.9, 1.25] * 8
    chain = [r[1] for r in rule([(f * hi, f * senders, edges, vertices, width) for f in sizes], "stream")]
    assert sum(a != b for a, b in zip(chain, chain[1:])) <= 1
    gone = [r[1] for r in rule([(f * hi, f * senders, edges, vertices, width) for f in (1.3, 0.8, 0.2, 0.2)], "stream")]
    assert gone == [True, True, False, False]     # and leaves it when the stream has become small

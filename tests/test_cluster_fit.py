"""The cluster-size rule (csrc/cluster_fit.h), compiled on the host with a fake
of the runtime's queries: what is asked, how often, and that an error which
waits to be reported is never cleared.
"""
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2606_04292_gb300", "csrc")

# arguments: consent (0/1), pending (0/1), held per size (5 numbers, negative:
# the query fails), then pairs "blocks clusters"; prints one line per pair:
# blocks taken, queries, consents and clears so far
HARNESS = r"""
#include <cstdio>
#include <cstdlib>
#include "cluster_fit.h"
struct Fake {
  int consent_, pending_, held_[5], asked = 0, consents = 0, clears = 0;
  bool pending() { return pending_; }
  bool consent() { ++consents; return consent_; }
  int held(int blocks) { ++asked; int k = 0; while ((1 << k) < blocks) ++k; return held_[k]; }
  void clear() { ++clears; }
};
int main(int, char** v) {
  Fake f{};
  f.consent_ = atoi(v[1]);
  f.pending_ = atoi(v[2]);
  for (int k = 0; k < 5; ++k) f.held_[k] = atoi(v[3 + k]);
  rich::ClusterFit fit;
  for (int a = 8; v[a]; a += 2) {
    const int b = rich::fit_blocks(fit, atoi(v[a]), atoi(v[a + 1]), f);
    printf("%d %d %d %d\n", b, f.asked, f.consents, f.clears);
  }
}
"""


@pytest.fixture(scope="module")
def rule(tmp_path_factory):
    d = tmp_path_factory.mktemp("fit")
    src, exe = d / "fit.cpp", d / "fit"
    src.write_text(HARNESS)
    subprocess.run(["g++", "-std=c++17", "-Wall", "-Werror", "-I", CSRC, str(src), "-o", str(exe)], check=True)

    def run(consent, pending, held, *pairs):
        args = [str(x) for x in (consent, pending, *held, *[y for p in pairs for y in p])]
        out = subprocess.run([str(exe)] + args, check=True, capture_output=True, text=True).stdout
        return [tuple(int(x) for x in line.split()) for line in out.splitlines()]
    return run


HELD = (152, 76, 36, 15, 7)


def test_asked_once(rule):
    got = rule(1, 0, HELD, (16, 1), (16, 1), (8, 1), (8, 1), (16, 1))
    assert [g[0] for g in got] == [16, 16, 8, 8, 16]
    assert got[0][1:] == (1, 1, 0) and got[1][1:] == (1, 1, 0) and got[-1][1:] == (2, 1, 0)


def test_next_smaller_size(rule):
    assert [g[0] for g in rule(1, 0, (152, 76, 36, 15, 0), (16, 1), (16, 1))] == [8, 8]
    assert [g[0] for g in rule(1, 0, (152, 4, 0, 0, 0), (16, 1), (2, 1), (1, 1))] == [2, 2, 1]


def test_as_many_clusters_as_are_wanted(rule):
    pairs = [(16, n) for n in (1, 7, 8, 15, 16, 36, 37, 76, 77, 1000)] + [(4, 1), (4, 37), (2, 15)]
    assert [g[0] for g in rule(1, 0, HELD, *pairs)] == [16, 16, 8, 8, 4, 4, 2, 2, 1, 1, 4, 2, 2]


def test_a_pending_error_is_left_alone(rule):
    got = rule(1, 1, HELD, (16, 1), (8, 1))
    assert [g[0] for g in got] == [8, 8]
    assert got[-1][1:] == (0, 0, 0)


def test_failed_queries_take_back_their_own_error(rule):
    assert rule(1, 0, (-1,) * 5, (8, 1)) == [(8, 1, 0, 1)]
    assert rule(0, 0, HELD, (16, 1), (16, 1)) == [(8, 1, 1, 1), (8, 1, 2, 2)]

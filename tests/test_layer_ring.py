"""The ring of K blocks of the fused-epilogue GEMM (no GPU).

The kernel's rule -- stages per tile width, which gather warp writes which block -- is compiled from its
header, and a model of the ring runs it under random schedules.  As in the kernel, the weights' producer
and the block's gather warp each wait until the stage is empty, write their half and arrive; the consumer
waits until it is full, reads it and frees it.  A wait sees one parity bit: it passes as soon as the
barrier's current phase has the other parity.  A block may only be written over one that has been read, and
the consumer must find both halves of the block it is at."""
import random
import shutil
import subprocess

import pytest

from tests.conftest import ROOT

N_BLOCKS = 40


@pytest.fixture(scope="module")
def rule(tmp_path_factory):
    """(stages, owners of blocks 0 .. N_BLOCKS - 1) of the gathering form, per tile width."""
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("no host compiler")
    d = tmp_path_factory.mktemp("ring")
    (d / "ring.cc").write_text("""
#include <cstdio>
#include "layer_ring.h"
using namespace bcrown::lt;
int main() {
  for (int np = 16; np <= 256; np += 16) {
    const int ns = lt_stages(false, np);
    std::printf("%%d %%d %%d", np, ns, NS_GATHER);
    for (int s = 0; s < %d; ++s) std::printf(" %%d", lt_gather_warp(s %% ns));
    std::printf("\\n");
  }
}
""" % N_BLOCKS)
    subprocess.run([cxx, "-std=c++17", "-I", ROOT + "/paper_2103_06624_gb300/csrc", "-o", str(d / "ring"), str(d / "ring.cc")],
                   check=True)
    rows = [list(map(int, ln.split())) for ln in subprocess.run([str(d / "ring")], capture_output=True, text=True,
                                                                check=True).stdout.splitlines()]
    return {r[0]: (r[1], r[2], r[3:]) for r in rows}


class _Barrier:
    def __init__(self, count):
        self.count, self.left, self.phase = count, count, 0

    def passes(self, parity):
        return (self.phase & 1) != parity

    def arrive(self):
        self.left -= 1
        if self.left == 0:
            self.left, self.phase = self.count, self.phase + 1


def _run(ns, warps, owner, seed):
    """One schedule: None, or what went wrong."""
    rng = random.Random(seed)
    full, empty = [_Barrier(2) for _ in range(ns)], [_Barrier(1) for _ in range(ns)]
    held = [[None, None] for _ in range(ns)]   # per stage: the block whose A and B it holds, unread
    error = []

    def writer(half, blocks):
        for s in blocks:
            st = s % ns
            while not empty[st].passes(((s // ns) & 1) ^ 1):
                yield False
            if held[st][half] is not None:
                error.append("block %d written over block %d" % (s, held[st][half]))
            held[st][half] = s
            yield True
            full[st].arrive()
            yield True

    def reader():
        for s in range(N_BLOCKS):
            st = s % ns
            while not full[st].passes((s // ns) & 1):
                yield False
            if held[st] != [s, s]:
                error.append("block %d read as %s" % (s, held[st]))
            held[st] = [None, None]
            yield True
            empty[st].arrive()
            yield True

    agents = [writer(1, range(N_BLOCKS)), reader()]
    agents += [writer(0, [s for s in range(N_BLOCKS) if owner[s] == w]) for w in range(warps)]
    slow = [rng.choice([1, 1, 10, 100]) for _ in agents]
    idle = 0
    while agents and not error and idle < 20000:
        i = rng.choices(range(len(agents)), [1 / x for x in slow])[0]
        try:
            idle = 0 if next(agents[i]) else idle + 1
        except StopIteration:
            del agents[i], slow[i]
    return error[0] if error else ("stuck" if agents else None)


def test_every_tile_width_keeps_its_blocks_apart(rule):
    for np, (ns, warps, owner) in rule.items():
        assert max(owner) < warps
        for seed in range(60):
            assert _run(ns, warps, owner, seed) is None, (np, ns, seed)


def test_the_model_sees_a_warp_that_writes_several_stages():
    """Four warps that take turns over three stages: a warp's next wait can be two rounds ahead."""
    assert any(_run(3, 4, [s % 4 for s in range(N_BLOCKS)], seed) for seed in range(60))
    assert all(_run(4, 4, [s % 4 for s in range(N_BLOCKS)], seed) is None for seed in range(60))

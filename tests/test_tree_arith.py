"""The tree work's index arithmetic and the bounded wait, compiled for the host with the sanitizer for undefined behaviour."""
import os
import subprocess

import numpy as np
import pytest

from conftest import ROOT


@pytest.fixture(scope="module")
def probe(tmp_path_factory):
    exe = str(tmp_path_factory.mktemp("arith") / "tree_arith_probe")
    subprocess.check_call(["g++", "-O1", "-std=c++17", "-fsanitize=undefined", "-fno-sanitize-recover=all",
                           "-I", os.path.join(ROOT, "paper_2311_09445_b200", "csrc"), "-o", exe,
                           os.path.join(ROOT, "tests", "tree_arith_probe.cpp")])
    return lambda lines: subprocess.run([exe], input="".join(ln + "\n" for ln in lines), capture_output=True, text=True, check=True).stdout.split()


def test_nodes_of_every_level(probe):
    # capacities up to the largest a handle takes (2^30), about every power of the fanout; every level
    ask = []
    for lg in (1, 2, 3, 4, 5):
        for cap in sorted({min(max(1, (1 << e) + d), 1 << 30) for e in range(0, 31) for d in (-1, 0, 1)}):
            depth = 1
            while (1 << (lg * depth)) < cap:
                depth += 1
            ask += [(cap, lg * up) for up in range(depth + 1)]
    got = probe("nodes %d %d" % q for q in ask)
    assert [int(g) for g in got] == [-((-cap) >> sh) for cap, sh in ask]
    assert max(sh for _, sh in ask) >= 32


def test_no_stride_of_indices_meets_in_one_line_of_probes(probe):
    # full tables of the tree kernel (twice as many places as entries), linear probing: a random batch of 1024 needs some
    # tens of probes at worst, so 64 is the line; one place for all would need 1024
    rng = np.random.default_rng(0)
    for bits in (11, 12):
        n = 1 << (bits - 1)
        batches = [(np.arange(n, dtype=np.int64) << k) & ((1 << 30) - 1) for k in range(0, 21)]
        batches += [(np.arange(n) * step) % (1 << 30) for step in (3, 84, 1000, 4097, 999_983)] + [rng.integers(0, 1 << 30, n)]
        for keys in batches:
            keys = np.unique(keys)
            at = [int(x) for x in probe("place %d %d" % (i, 32 - bits) for i in keys)]
            assert max(at) < 1 << bits
            taken, worst = set(), 0
            for h in at:
                probes = 1
                while h in taken:
                    h, probes = (h + 1) % (1 << bits), probes + 1
                taken.add(h)
                worst = max(worst, probes)
            assert worst <= 64, (bits, keys[:3], worst)


def test_a_wait_that_runs_out_is_reported_and_goes_on_for_what_is_in_flight(probe):
    # limit 5: in time up to poll 5, late (reported, but waited for) up to poll 10, never beyond
    got = probe("wait %d 5" % ready for ready in (1, 5, 6, 10, 11, 1000))
    assert got == ["0:1", "0:5", "1:6", "1:10", "2:10", "2:10"]

"""The cluster of prb_step.cu over trees so deep that several steps of groups lie below its staged levels: the iteration with its descent over
those steps in L2, the tree work alone with a min-tree or with frames, batches that go in rounds, insertions beyond what the
cluster takes -- against the oracle.

Steps of groups, by the kernel's own cut: two from 2^20 + 1 slots on for fanouts 2, 4 and 16 (batches of more than 256: 2^21 + 1), from 2^19 + 1 for 8, from
2^21 + 1 (2^22 + 1) for 32; three for fanout 8 from 2^22 + 1; with a min-tree earlier by a factor of two or more.  Fewer CTAs, which a small batch gets, stage
less."""
import numpy as np
import pytest

from prb_harness import Pair

pytestmark = pytest.mark.gpu
OBS, ACT, CHUNK = 10, 4, 1 << 20


def _filled(oracle_mod, N, K, obs=OBS, store=False, **kw):
    rng = np.random.default_rng(K + N)
    pr = Pair(oracle_mod, N, K, obs, ACT, CHUNK, oracle_store=store, **kw)
    at, goal = 0, N - N // 7                                                  # (part of the ring stays unwritten)
    while at < goal:
        n = min(CHUNK, goal - at)
        pr.insert(_new(rng, n, pr, 0.0))
        at += n
    return pr, rng


def _new(rng, n, pr, bad=0.03):
    prio = np.exp(rng.standard_normal(n)).astype(np.float32)
    prio[rng.random(n) < bad] = np.nan
    b = dict(prio=prio)
    if pr.ora.frame_stack:
        b["done"] = (rng.random(n) < 0.01).astype(np.uint8) * 2
    elif pr.oracle_store:
        b.update(obs=rng.integers(0, 256, size=(n, OBS), dtype=np.uint8), next_obs=rng.integers(0, 256, size=(n, OBS), dtype=np.uint8),
                 act=rng.integers(0, 256, size=(n, ACT), dtype=np.uint8), rew=rng.standard_normal(n).astype(np.float32),
                 done=rng.integers(0, 2, size=n, dtype=np.uint8))
    return b


def _check(pr, min_tree=False):
    pr.compare_tree()
    if min_tree:
        pr.compare_min_tree()
    pr.compare_status()
    pr.compare_state()


def _indices(rng, fill, B, span):
    idx = rng.integers(-1, fill + 1, size=B) if span == 0 else fill // 3 + rng.integers(0, span, size=B)
    return idx.astype(np.int32)


@pytest.mark.parametrize("K,N", [(2, 2_100_003), (2, 1 << 22), (4, 2_100_003), (8, 1_300_001), (8, 1 << 21), (8, 4_300_000), (16, 2_100_003), (32, 4_300_000)])
def test_step_over_several_steps_of_groups(oracle_mod, K, N):
    pr, rng = _filled(oracle_mod, N, K)
    for B_upd, n, B, span in [(1, 1, 5, 0), (256, 256, 256, 0), (100, 30, 1500, 40), (1000, 777, 1536, 0), (1024, 1000, 64, 300), (1024, 1024, 64, 9000)]:
        idx, td = _indices(rng, pr.gpu.info()[0], B_upd, span), rng.standard_normal(B_upd).astype(np.float32)
        if B_upd == 1000:
            td[rng.random(B_upd) < 0.05] = np.inf
        before = pr.gpu.kernel_launches()
        pr.step(idx, td, 0.6, 1e-6, _new(rng, n, pr), B, 0.4, 7)
        assert pr.gpu.kernel_launches() - before == 1
        _check(pr)
    pr.close()


@pytest.mark.parametrize("K,N", [(2, 1 << 21), (4, 1_100_000), (8, 600_000), (8, 4_300_000), (16, 1_100_000), (32, 2_100_003)])
def test_tree_work_with_a_min_tree(oracle_mod, K, N):
    pr, rng = _filled(oracle_mod, N, K, min_tree=True)
    _check(pr, True)
    for B, n, span in [(1, 0, 0), (256, 256, 0), (200, 30, 40), (1000, 777, 0), (1024, 1000, 300), (1024, 1024, 9000), (0, 400, 0)]:
        new = _new(rng, n, pr) if n else None
        if B == 0:
            pr.insert(new)
        else:
            idx, td = _indices(rng, pr.gpu.info()[0], B, span), rng.standard_normal(B).astype(np.float32)
            td[rng.random(B) < 0.02] = np.nan
            if n:
                pr.update_insert(idx, td, 0.6, 1e-6, new)
            else:
                pr.update(idx, td, 0.6, 1e-6)
        _check(pr, True)
    pr.close()


@pytest.mark.parametrize("min_tree", [False, True])
@pytest.mark.parametrize("K,N", [(2, 70_001), (4, 2_100_003), (8, 300_007), (8, 1 << 21), (16, 70_001), (16, 2_100_003), (32, 100_000)])
def test_frames_in_trees_with_staged_levels(oracle_mod, K, N, min_tree):
    # (a slot's leaf, and the leaves of the four slots behind the cursor, through staged levels and several steps; up to 1024 inserted leaves)
    pr, rng = _filled(oracle_mod, N, K, obs=32, store=True, frame_stack=4, min_tree=min_tree)
    fill = pr.gpu.info()[0]
    for B, n, span in [(32, 16, 0), (256, 252, 0), (300, 500, 0), (1000, 1020, 700)]:
        idx, td = _indices(rng, fill, B, span), rng.standard_normal(B).astype(np.float32)
        pr.update_insert(idx, td, 0.6, 1e-6, _new(rng, n, pr))
        _check(pr, min_tree)
    pr.close()


@pytest.mark.parametrize("K", [2, 4, 8, 16, 32])
def test_insertions_beyond_the_cluster_of_the_iteration(oracle_mod, K):
    # 1025 to 4096 insertions with priorities behind an update: the other tree kernel's cluster
    pr, rng = _filled(oracle_mod, 70_001, K, store=True)
    for B, n in [(300, 1025), (1024, 2000), (31, 4096)]:
        idx, td = _indices(rng, pr.gpu.info()[0], B, 0), rng.standard_normal(B).astype(np.float32)
        pr.update_insert(idx, td, 0.6, 1e-6, _new(rng, n, pr))
        _check(pr)
    pr.compare_rows(np.arange(0, pr.gpu.info()[0], 3, dtype=np.int32))
    pr.close()


@pytest.mark.parametrize("K,N,kw", [(2, 4096, {}), (2, 1_000_003, {}), (4, 1000, {}), (4, 2_100_003, {}), (8, 100, {}), (8, 1 << 20, {}), (8, 1 << 21, {}), (16, 5000, {}),
                                    (16, 1 << 20, {}), (32, 40_000, {}), (32, 1_100_000, {}), (2, 1 << 18, dict(min_tree=True)), (16, 1 << 20, dict(min_tree=True)),
                                    (32, 1 << 20, dict(min_tree=True)), (4, 33_000, dict(min_tree=True)), (8, 300_007, dict(frame_stack=4, obs=32, store=True)),
                                    (16, 1 << 20, dict(frame_stack=4, obs=32, store=True, min_tree=True))])
def test_few_entries(oracle_mod, K, N, kw):
    # around the lines at which a small batch gets fewer CTAs, and at which insertions alone go to the other kernel; with the same entries in one CTA's part
    pr, rng = _filled(oracle_mod, N, K, **kw)
    for B, n in [(1, 0), (31, 0), (32, 0), (33, 0), (64, 0), (65, 0), (32, 1), (64, 60), (64, 64), (65, 10), (10, 65),
                 (0, 1), (0, 60), (0, 64), (0, 65), (0, 252), (0, 256), (0, 257), (0, 512), (0, 513)]:
        if n > N // 2:
            continue
        new = _new(rng, n, pr) if n else None
        fill = pr.gpu.info()[0]
        for span in (0, min(5, fill // 2)) if B else (0,):
            idx, td = _indices(rng, fill, B, span), rng.standard_normal(B).astype(np.float32)
            if B and n:
                pr.update_insert(idx, td, 0.6, 1e-6, new)
            elif B:
                pr.update(idx, td, 0.6, 1e-6)
            else:
                pr.insert(new)
        if B in (1, 33, 64) or n in (65, 257, 513):
            _check(pr, kw.get("min_tree", False))
        if "frame_stack" not in kw and not kw.get("min_tree") and B and B <= 64 and n:
            pr.step(_indices(rng, fill, B, 0), td, 0.6, 1e-6, _new(rng, n, pr), 64, 0.4, 3)
    _check(pr, kw.get("min_tree", False))
    pr.close()

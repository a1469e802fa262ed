"""The tree kernel (update, insertion, both) at the sizes where its form changes: one CTA, clusters, the grid; several
levels per pass (fanouts 2 and 4), trees too shallow for that, levels that end inside a group; batches that fall to one
subtree; insertions that wrap; and what an update and an insertion both write."""
import numpy as np
import pytest
import torch

from prb_harness import Pair

pytestmark = pytest.mark.gpu


def _batch(rng, n, obs_bytes, act_bytes):
    prio = np.exp(rng.standard_normal(n)).astype(np.float32)
    prio[rng.random(n) < 0.05] = np.nan
    return dict(obs=rng.integers(0, 256, size=(n, obs_bytes), dtype=np.uint8), act=rng.integers(0, 256, size=(n, act_bytes), dtype=np.uint8),
                rew=rng.standard_normal(n).astype(np.float32), next_obs=rng.integers(0, 256, size=(n, obs_bytes), dtype=np.uint8),
                done=rng.integers(0, 2, size=n, dtype=np.uint8), prio=prio)


def _check(pr, min_tree):
    pr.compare_tree()
    if min_tree:
        pr.compare_min_tree()
    pr.compare_status()
    pr.compare_state()


@pytest.mark.parametrize("min_tree", [False, True])
@pytest.mark.parametrize("K,N", [(2, 3), (2, 33), (2, 70), (2, 40_001), (4, 17), (4, 30_000), (8, 9000), (16, 70_001), (32, 31), (32, 40_000)])
def test_forms(oracle_mod, K, N, min_tree):
    rng = np.random.default_rng(K * 100 + N)
    pr = Pair(oracle_mod, N, K, 12, 4, 70_000, min_tree=min_tree)
    pr.insert(_batch(rng, N - N // 4, 12, 4))                                 # (a quarter of the ring stays unwritten)
    _check(pr, min_tree)
    for B, n in [(1, 1), (33, 5), (64, 64), (65, 300), (257, 0), (512, 777), (1000, 31), (1024, 4097), (1025, 1), (4099, 100), (20_000, 17)]:
        n = min(n, N)
        fill = pr.gpu.info()[0]
        idx = rng.integers(-1, fill + 1, size=B).astype(np.int32)             # (some out of range)
        if B > 40:
            idx[B // 2:] = np.where(rng.random(B - B // 2) < 0.5, idx[:B - B // 2], idx[B // 2:])     # repeats, the later one wins
        td = rng.standard_normal(B).astype(np.float32)
        td[rng.random(B) < 0.02] = np.inf
        if n:
            pr.update_insert(idx, td, 0.6, 1e-6, _batch(rng, n, 12, 4))
        else:
            pr.update(idx, td, 0.6, 1e-6)
        _check(pr, min_tree)
    pr.compare_rows(np.arange(pr.gpu.info()[0], dtype=np.int32))
    pr.close()


@pytest.mark.parametrize("K,N", [(2, 1 << 16), (4, 1 << 18), (32, 1 << 19)])
def test_batch_in_one_subtree(oracle_mod, K, N):
    # all entries fall to the leaves of one CTA: more than its list holds at a time, worked off in batch order
    rng = np.random.default_rng(K)
    pr = Pair(oracle_mod, N, K, 0, 0, 30_000)
    for at in range(0, N, 30_000):
        pr.insert(dict(prio=np.exp(rng.standard_normal(min(30_000, N - at))).astype(np.float32)))
    for span in (1, 30, 5000):
        for B in (1500, 9000, 30_000):
            idx = (N // 2 + rng.integers(0, span, size=B)).astype(np.int32)
            pr.update_priorities(idx, np.exp(rng.standard_normal(B)).astype(np.float32))
            pr.compare_tree()
    pr.compare_status()
    pr.close()


@pytest.mark.parametrize("K,n", [(16, 1), (16, 300), (2, 777), (32, 1500)])
def test_rows_of_many_insertions_in_a_row(oracle_mod, K, n):
    # every insertion's copying CTAs read the row cursor that the last of the insertion before moved; rows of several
    # CTAs' worth, a ring that wraps every few calls, nothing waited for in between
    rng = np.random.default_rng(n)
    N = 2 * n + 3
    pr = Pair(oracle_mod, N, K, 40, 4, 1500)
    batches = [_batch(rng, n, 40, 4) for _ in range(3)]
    dev = [{k: torch.from_numpy(v).to(pr.dev) for k, v in b.items()} for b in batches]
    for i in range(100):
        pr.insert(batches[i % 3], dev_batch=dev[i % 3])
    _check(pr, False)
    pr.compare_rows(np.arange(N, dtype=np.int32))
    pr.close()


@pytest.mark.parametrize("K,N", [(2, 5000), (4, 30_000), (16, 70_001), (32, 40_000)])
def test_default_priorities_with_an_update(oracle_mod, K, N):
    # new transitions without priorities take the running maximum, the very update's writes included, whichever CTA
    # made them: one launch up to 2048 update entries (one CTA, a cluster, the grid), two beyond
    rng = np.random.default_rng(K)
    pr = Pair(oracle_mod, N, K, 12, 4, 5000)
    for at in range(0, N, 4000):
        pr.insert(_batch(rng, min(4000, N - at), 12, 4))
    for step, (B, n) in enumerate([(1, 1), (40, 3), (64, 64), (256, 256), (1000, 777), (1024, 4096), (300, 4097), (1025, 20), (2048, 300), (2049, 300), (4000, 4900)]):
        idx = rng.integers(-1, N + 1, size=B).astype(np.int32)
        td = (rng.standard_normal(B) * 3.0 ** step).astype(np.float32)        # (the largest so far, somewhere in the batch)
        td[rng.random(B) < 0.05] = np.nan
        b = _batch(rng, n, 12, 4)
        assert pr.ora.update(idx, td, 0.6, 1e-6) == 0
        assert pr.ora.insert(b["obs"], b["act"], b["rew"], b["next_obs"], b["done"], None, n=n) == 0
        d = {k: torch.from_numpy(v).to(pr.dev) for k, v in b.items()}
        before = pr.gpu.kernel_launches()
        pr.gpu.update_insert(torch.from_numpy(idx).to(pr.dev), torch.from_numpy(td).to(pr.dev), 0.6, 1e-6, d["obs"], d["act"], d["rew"],
                             d["next_obs"], d["done"], None, n=n)
        assert pr.gpu.kernel_launches() - before == (1 if B <= 2048 else 2)
        _check(pr, False)
    pr.close()


@pytest.mark.parametrize("min_tree", [False, True])
@pytest.mark.parametrize("K,N,B", [(2, 90_001, 32_769), (2, 200_000, 100_000), (4, 70_000, 24_577), (8, 40_000, 33_000), (16, 100_001, 16_385), (32, 60_000, 50_000)])
def test_very_large_updates(oracle_mod, K, N, B, min_tree):
    # beyond the line where the batch is shared out over co-resident CTAs: repeats (the last valid entry wins), refused
    # entries, leaves of -0.0; alone, after an insertion, and with one (one launch, or two beyond three times the line)
    rng = np.random.default_rng(K + B)
    pr = Pair(oracle_mod, N, K, 4, 4, 100_000, min_tree=min_tree)
    for at in range(0, N - N // 8, 50_000):
        b = _batch(rng, min(50_000, N - N // 8 - at), 4, 4)
        b["prio"][rng.random(b["prio"].size) < 0.05] = -0.0
        pr.insert(b)
    fill = pr.gpu.info()[0]
    for call in range(3):
        idx = rng.integers(-1, fill + 1, size=B).astype(np.int32)
        if call:
            idx = np.sort(idx)
        td = rng.standard_normal(B).astype(np.float32)
        td[rng.random(B) < 0.02] = np.inf
        if call == 0:
            pr.update(idx, td, 0.6, 1e-6)
        elif call == 1:
            pr.update_after_insert(idx, td, 0.6, 1e-6, 100)
        else:
            pr.update_insert(idx, td, 0.6, 1e-6, _batch(rng, 1000, 4, 4))
        _check(pr, min_tree)
    pr.close()

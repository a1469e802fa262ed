"""The iteration in one launch (prb_step.cu): trees of every depth it takes (with and without staged levels, one and several steps of
groups below them), batches of one entry and of several per thread, batches that fall to one CTA, refused entries, insertions
that wrap or fill the ring, sampled slots that the same call inserts, fields left out -- against the oracle's update, insertion and sample."""
import numpy as np
import pytest
import torch

from prb_harness import Pair

pytestmark = pytest.mark.gpu
OBS, ACT = 10, 4


def _batch(rng, n, bad=0.03):
    prio = np.exp(rng.standard_normal(n)).astype(np.float32)
    prio[rng.random(n) < bad] = np.nan
    return dict(obs=rng.integers(0, 256, size=(n, OBS), dtype=np.uint8), act=rng.integers(0, 256, size=(n, ACT), dtype=np.uint8),
                rew=rng.standard_normal(n).astype(np.float32), next_obs=rng.integers(0, 256, size=(n, OBS), dtype=np.uint8),
                done=rng.integers(0, 2, size=n, dtype=np.uint8), prio=prio)


def _check(pr):
    pr.compare_tree()
    pr.compare_status()
    pr.compare_state()


def _step(pr, *args):
    before = pr.gpu.kernel_launches()
    pr.step(*args)
    return pr.gpu.kernel_launches() - before


@pytest.mark.parametrize("K,N", [(2, 300), (2, 4096), (2, 5000), (2, 70_001), (2, 131_072), (4, 1000), (4, 16_384), (4, 100_003), (8, 100), (8, 40_000),
                                 (8, 300_007), (16, 1030), (16, 70_001), (16, 1 << 20), (32, 2000), (32, 40_000), (32, 1_100_000)])
def test_step_in_one(oracle_mod, K, N):
    rng = np.random.default_rng(K * 1000 + N)
    pr = Pair(oracle_mod, N, K, OBS, ACT, 65_536)
    goal, at = N - N // 5, 0                                                  # (part of the ring stays unwritten)
    while at < goal:
        k = min(65_536, goal - at)
        pr.insert(_batch(rng, k))
        at += k
    _check(pr)
    for B_upd, n, B in [(1, 1, 1), (32, 5, 33), (64, 64, 64), (256, 256, 256), (255, 1, 1000), (257, 3, 16), (1000, 777, 1536), (1024, 1024, 40), (96, 300, 96)]:
        n = min(n, N)
        fill = pr.gpu.info()[0]
        idx = rng.integers(-1, fill + 1, size=B_upd).astype(np.int32)         # (some out of range)
        if B_upd > 40:
            idx[B_upd // 2:] = np.where(rng.random(B_upd - B_upd // 2) < 0.5, idx[:B_upd - B_upd // 2], idx[B_upd // 2:])      # repeats
        td = rng.standard_normal(B_upd).astype(np.float32)
        if B_upd not in (64, 1000):
            td[rng.random(B_upd) < 0.05] = np.inf
        launches = _step(pr, idx, td, 0.6, 1e-6, _batch(rng, n), B, 0.4, 7)
        assert launches == 1
        _check(pr)
    pr.compare_rows(np.arange(0, pr.gpu.info()[0], max(1, N // 20_000), dtype=np.int32))
    pr.close()


@pytest.mark.parametrize("K,N", [(2, 1 << 16), (4, 1 << 16), (8, 1 << 18), (16, 1 << 20), (32, 1 << 20)])
@pytest.mark.parametrize("span", [8, 300, 4000])
def test_step_in_one_subtree(oracle_mod, K, N, span):
    # every entry falls to one CTA, or to a few: more groups than it holds at a time
    rng = np.random.default_rng(K + span)
    pr = Pair(oracle_mod, N, K, OBS, ACT, 65_536, oracle_store=False)
    for at in range(0, N, 65_536):
        pr.insert(dict(prio=np.exp(rng.standard_normal(min(65_536, N - at))).astype(np.float32)))
    for B, n in [(200, 250), (1024, 1000)]:
        idx = (N // 3 + rng.integers(0, span, size=B)).astype(np.int32)
        assert _step(pr, idx, rng.standard_normal(B).astype(np.float32), 0.6, 1e-6,
                     dict(prio=np.exp(rng.standard_normal(n)).astype(np.float32)), 64, 0.5, 3) == 1
        _check(pr)
    pr.close()


@pytest.mark.parametrize("K", [2, 8, 16])
def test_sampled_slots_that_are_inserted(oracle_mod, K):
    # a ring hardly larger than what is inserted, and inserted priorities that draw nearly every stratum; the insertions wrap
    rng = np.random.default_rng(K)
    pr = Pair(oracle_mod, 1100, K, OBS, ACT, 1024)
    pr.insert(_batch(rng, 1024, 0.0))
    pr.insert(_batch(rng, 76, 0.0))
    for i, n in enumerate((500, 1, 1024, 900, 255)):
        b = _batch(rng, n, 0.0)
        b["prio"] *= np.float32(1e4 ** (i + 1))
        idx = rng.integers(0, 1100, size=100).astype(np.int32)
        _, g = pr.step(idx, rng.standard_normal(100).astype(np.float32), 0.6, 1e-6, b, 300, 0.4, 5)
        if n > 1:
            first = (pr.gpu.info()[1] - n) % 1100
            assert ((g["idx"] - first) % 1100 < n).mean() > 0.9
        _check(pr)
    pr.compare_rows(np.arange(1100, dtype=np.int32))
    # rows that the insertion does not carry stay what they were, sampled or not
    b = _batch(rng, 700, 0.0)
    b["obs"], b["rew"] = None, None
    pr.step(np.arange(10, dtype=np.int32), np.ones(10, np.float32), 0.6, 1e-6, b, 300, 0.4, 5)
    _check(pr)
    pr.compare_rows(np.arange(1100, dtype=np.int32))
    pr.close()


def test_step_without_insertion_or_mass(oracle_mod):
    rng = np.random.default_rng(4)
    pr = Pair(oracle_mod, 5000, 16, OBS, ACT, 1024)
    for _ in range(5):
        pr.insert(_batch(rng, 1000, 0.0))
    idx, td = rng.integers(0, 5000, size=300).astype(np.int32), rng.standard_normal(300).astype(np.float32)
    assert pr.ora.update(idx, td, 0.6, 1e-6) == 0
    o = pr.ora.sample(64, 0.4, 9)
    t = {"idx": torch.zeros(64, dtype=torch.int32, device=pr.dev), "w": torch.zeros(64, device=pr.dev)}
    pr.gpu.step(torch.from_numpy(idx).to(pr.dev), torch.from_numpy(td).to(pr.dev), 0.6, 1e-6, None, None, None, None, None, None,
                64, 0.4, 9, t["idx"], t["w"], n=0)
    torch.cuda.synchronize()
    assert np.array_equal(t["idx"].cpu().numpy(), o["idx"])
    np.testing.assert_allclose(t["w"].cpu().numpy(), o["w"], rtol=1e-5)
    _check(pr)
    pr.close()
    # nothing with a priority above zero: EMPTY, and the outputs are left alone
    pr = Pair(oracle_mod, 4096, 2, OBS, ACT, 1024)
    pr.insert(dict(_batch(rng, 100, 0.0), prio=np.zeros(100, np.float32)))
    o, g = pr.step(np.arange(20, dtype=np.int32), np.zeros(20, np.float32), 0.6, 0.0, dict(_batch(rng, 50, 0.0), prio=np.zeros(50, np.float32)), 32, 0.4, 1, False)
    assert (g["idx"] == -1).all() and (g["w"] == 0).all()
    _check(pr)
    pr.close()


def test_overlapping_arrays_take_the_other_route(oracle_mod):
    # the update's indices may be the array that the sampled ones go to; rows that are read and written take two launches, same results
    rng = np.random.default_rng(11)
    pr = Pair(oracle_mod, 3000, 16, OBS, ACT, 1024)
    pr.insert(_batch(rng, 1024, 0.0))
    B, dev = 128, pr.dev
    t = {"idx": torch.from_numpy(rng.integers(0, 1024, size=B).astype(np.int32)).to(dev), "w": torch.zeros(B, device=dev),
         "obs": torch.zeros((B, OBS), dtype=torch.uint8, device=dev)}
    for shared in (False, True):
        b = _batch(rng, B, 0.0)
        td = rng.standard_normal(B).astype(np.float32)
        assert pr.ora.update(t["idx"].cpu().numpy(), td, 0.6, 1e-6) == 0
        assert pr.ora.insert(b["obs"], b["act"], b["rew"], b["next_obs"], b["done"], b["prio"]) == 0
        o = pr.ora.sample(B, 0.4, 2)
        d = {k: torch.from_numpy(v).to(dev) for k, v in b.items()}
        out = d["obs"] if shared else t["obs"]
        before = pr.gpu.kernel_launches()
        pr.gpu.step(t["idx"], torch.from_numpy(td).to(dev), 0.6, 1e-6, d["obs"], d["act"], d["rew"], d["next_obs"], d["done"], d["prio"],
                    B, 0.4, 2, t["idx"], t["w"], out)
        torch.cuda.synchronize()
        assert pr.gpu.kernel_launches() - before == (2 if shared else 1)
        assert np.array_equal(t["idx"].cpu().numpy(), o["idx"])
        assert np.array_equal(out.cpu().numpy(), np.asarray(o["obs"]).view(np.uint8).reshape(B, OBS))
        _check(pr)
    pr.close()


@pytest.mark.parametrize("captured", [False, True])
def test_long_rows_left_out(oracle_mod, captured):
    # a buffer of long rows whose iteration leaves them out goes in one launch, between iterations that copy them on the handle's streams
    rng = np.random.default_rng(5)
    N, E, B, n = 1800, 16_384, 64, 48                                          # (the ring is full: every row that is compared has been written)
    stream = torch.cuda.Stream()
    from paper_2311_09445_b200 import PrioritizedReplay
    gpu = PrioritizedReplay(N, 16, E, 4, 1024, stream=stream)
    ora = oracle_mod.OraclePRB(N, 16, E, 4)

    def batch(k):
        return dict(obs=rng.integers(0, 256, size=(k, E), dtype=np.uint8), act=rng.integers(0, 256, size=(k, 4), dtype=np.uint8),
                    rew=rng.standard_normal(k).astype(np.float32), next_obs=rng.integers(0, 256, size=(k, E), dtype=np.uint8),
                    done=rng.integers(0, 2, size=k, dtype=np.uint8), prio=np.exp(rng.standard_normal(k)).astype(np.float32))
    def up(b):
        return {k: torch.from_numpy(v).cuda() for k, v in b.items()}
    for _ in range(2):
        b = batch(900)
        d = up(b)
        torch.cuda.synchronize()
        gpu.insert(d["obs"], d["act"], d["rew"], d["next_obs"], d["done"], d["prio"])
        assert ora.insert(b["obs"], b["act"], b["rew"], b["next_obs"], b["done"], b["prio"]) == 0
        torch.cuda.synchronize()
    full = (True, False, True, False, False, True)
    host = [batch(n) for _ in full]
    for b, whole in zip(host, full):
        if not whole:
            b["obs"] = b["next_obs"] = None
    new = [up({k: v for k, v in b.items() if v is not None}) for b in host]
    idx = [rng.integers(0, 1800, size=B).astype(np.int32) for _ in full]
    td = [rng.standard_normal(B).astype(np.float32) for _ in full]
    d_idx, d_td = [torch.from_numpy(x).cuda() for x in idx], [torch.from_numpy(x).cuda() for x in td]
    z = lambda *s: torch.zeros(s, dtype=torch.uint8, device="cuda")
    out = [dict(idx=torch.zeros(B, dtype=torch.int32, device="cuda"), w=torch.zeros(B, device="cuda"), obs=z(B, E) if whole else None, act=z(B, 4),
                rew=torch.zeros(B, device="cuda"), next_obs=z(B, E) if whole else None, done=z(B)) for whole in full]

    def iterations():
        for i in range(len(full)):
            r, o = new[i], out[i]
            gpu.step(d_idx[i], d_td[i], 0.6, 1e-6, r.get("obs"), r["act"], r["rew"], r.get("next_obs"), r["done"], r["prio"], B, 0.4, 7,
                     o["idx"], o["w"], o["obs"], o["act"], o["rew"], o["next_obs"], o["done"])
    torch.cuda.synchronize()
    graph = None
    if captured:
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            iterations()
    for _ in range(3):
        with torch.cuda.stream(stream):
            if graph is not None:
                graph.replay()
            else:
                iterations()
        torch.cuda.synchronize()
        for i, whole in enumerate(full):
            b = host[i]
            assert ora.update(idx[i], td[i], 0.6, 1e-6) == 0
            assert ora.insert(b["obs"], b["act"], b["rew"], b["next_obs"], b["done"], b["prio"]) == 0
            o = ora.sample(B, 0.4, 7)
            assert np.array_equal(out[i]["idx"].cpu().numpy(), o["idx"])
            np.testing.assert_allclose(out[i]["w"].cpu().numpy(), o["w"], rtol=1e-5)
            for f in ("obs", "act", "rew", "next_obs", "done"):
                if out[i][f] is not None:
                    assert np.array_equal(out[i][f].cpu().numpy().view(np.uint8).reshape(-1), np.ascontiguousarray(o[f]).view(np.uint8).reshape(-1)), (i, f)
    assert gpu.info() == ora.info() and gpu.sync() == ora.status()
    keep = np.arange(0, 1800, 7, dtype=np.int32)
    a, g = ora.read_rows(keep), gpu.read_rows(keep)
    for f in ("obs", "act", "rew", "next_obs", "done"):
        assert np.array_equal(np.ascontiguousarray(a[f]).view(np.uint8).reshape(-1), np.ascontiguousarray(g[f]).view(np.uint8).reshape(-1)), f
    gpu.close()
    ora.close()

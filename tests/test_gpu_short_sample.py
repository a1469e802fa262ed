"""The short-row sample at the sizes where its two shapes (one cluster, a grid) and its copy of rows
change: batches around a warp, a CTA's share and the line between the shapes; rows of 1-, 2- and 4-byte words, shorter
than half a warp's words and longer than a CTA's; and its weights against binary64."""
import numpy as np
import pytest
import torch

from prb_harness import Pair

pytestmark = pytest.mark.gpu


def _fill(pr, rng, N, obs_bytes, act_bytes, chunk):
    for at in range(0, N, chunk):
        n = min(chunk, N - at)
        prio = np.exp(rng.standard_normal(n)).astype(np.float32)
        prio[rng.random(n) < 0.1] = 0.0
        pr.insert(dict(obs=rng.integers(0, 256, size=(n, obs_bytes), dtype=np.uint8),
                       act=rng.integers(0, 256, size=(n, act_bytes), dtype=np.uint8),
                       rew=rng.standard_normal(n).astype(np.float32),
                       next_obs=rng.integers(0, 256, size=(n, obs_bytes), dtype=np.uint8),
                       done=rng.integers(0, 2, size=n, dtype=np.uint8), prio=prio))


@pytest.mark.parametrize("K,N", [(2, 5000), (2, 40_001), (4, 20_000), (8, 4097), (16, 70_000), (32, 33_000)])
@pytest.mark.parametrize("obs_bytes,act_bytes", [(3, 1), (12, 4), (242, 6), (2052, 24)])
def test_batch_sizes(oracle_mod, K, N, obs_bytes, act_bytes):
    rng = np.random.default_rng(N + obs_bytes)
    pr = Pair(oracle_mod, N, K, obs_bytes, act_bytes, 4096)
    _fill(pr, rng, N, obs_bytes, act_bytes, 4096)
    for call, B in enumerate([1, 4, 5, 31, 33, 64, 65, 511, 1025, 1536, 1537, 4000]):
        pr.sample(B, 0.4 if call % 2 else 1.0, 7 + call)
        pr.compare_state()
    assert pr.compare_status() in (0, 8)
    pr.close()


@pytest.mark.parametrize("K", [2, 16, 32])
@pytest.mark.parametrize("obs_bytes,act_bytes", [(128, 4), (132, 4), (1024, 16), (4104, 4), (7056, 8), (8190, 4), (9001, 3)])
def test_longer_rows(oracle_mod, K, obs_bytes, act_bytes):
    # rows on either side of the line between words and larger granules (16, 8, 4, 2 and 1 bytes), inserted in batches that
    # end inside a tile and wrap, sampled by each of the three kernels: the cluster (few, or little to copy), the lane
    # groups (medium rows), the grid
    rng = np.random.default_rng(obs_bytes + K)
    N = 701
    pr = Pair(oracle_mod, N, K, obs_bytes, act_bytes, 1600)
    _fill(pr, rng, N, obs_bytes, act_bytes, 333)
    for n in (1, 2, 17, 256, 700):
        _fill(pr, rng, n, obs_bytes, act_bytes, n)
    pr.compare_rows(np.arange(N, dtype=np.int32))
    for call, B in enumerate([1, 31, 33, 64, 65, 300, 1000, 1600]):
        pr.sample(B, 0.4, 7 + call)
        pr.compare_state()
    assert pr.compare_status() in (0, 8)
    pr.close()


@pytest.mark.parametrize("B", [48, 3000, 200_000])
def test_weights_against_binary64(oracle_mod, B):
    # (p / p_min)^-beta is formed in binary64 and rounded once to binary32: half a unit in the last place, 2^-24
    # relative, and nothing else that shows (1e-9 allowed for the two logarithms and the exponential)
    rng = np.random.default_rng(B)
    N, K = 200_000, 16
    pr = Pair(oracle_mod, N, K, 4, 4, 200_000)
    prio = np.exp(6 * rng.standard_normal(N)).astype(np.float32)
    pr.insert(dict(obs=np.zeros((N, 4), np.uint8), act=np.zeros((N, 4), np.uint8), rew=np.zeros(N, np.float32),
                   next_obs=np.zeros((N, 4), np.uint8), done=np.zeros(N, np.uint8), prio=prio))
    dev = pr.dev
    idx, w = torch.zeros(B, dtype=torch.int32, device=dev), torch.zeros(B, device=dev)
    for beta in (0.4, 1.0, 3.7, 0.0):
        for norm in ("batch", "buffer"):
            (pr.gpu.sample if norm == "batch" else pr.gpu.sample_buffer_norm)(B, beta, 3, idx, w)
            p = prio[idx.cpu().numpy()].astype(np.float64)
            # (the exponent crosses the C ABI as a binary32)
            want = (p / (p.min() if norm == "batch" else prio[prio > 0].min().astype(np.float64))) ** -float(np.float32(beta))
            got = w.cpu().numpy().astype(np.float64)
            normal = want > 2.0 ** -125                                 # below: binary32's subnormals
            assert np.all(np.abs(got - want)[normal] <= want[normal] * (2.0 ** -24 + 1e-9))
            assert np.all(np.abs(got - want)[~normal] <= 2.0 ** -149)
    pr.close()


@pytest.mark.parametrize("K", [2, 4, 8, 16, 32])
def test_negative_zero_priorities(oracle_mod, K):
    # -0.0 is a valid priority (p >= 0), stored as it is; a node whose leaves are all -0.0 sums to -0.0.  As the first
    # child of its group it is passed by every target, and what is subtracted is still the prefix before the child
    # entered, not the -0.0.  First by insertion, then by an update; the cluster's and the grid's form.
    rng = np.random.default_rng(K)
    N = K ** 3 if K > 4 else 512
    pr = Pair(oracle_mod, N, K, 4, 4, 4096)
    rows = lambda n: dict(obs=rng.integers(0, 256, size=(n, 4), dtype=np.uint8), act=rng.integers(0, 256, size=(n, 4), dtype=np.uint8),
                          rew=rng.standard_normal(n).astype(np.float32), next_obs=rng.integers(0, 256, size=(n, 4), dtype=np.uint8),
                          done=rng.integers(0, 2, size=n, dtype=np.uint8))
    prio = np.exp(rng.standard_normal(N)).astype(np.float32)
    for a in range(0, N, K * K):
        prio[a:a + K] = -0.0                                   # the first leaf group under a node two levels up
    prio[5 * K * K:5 * K * K + K * K] = -0.0                   # a whole node's leaves
    prio[rng.random(N) < 0.1] = -0.0
    for at in range(0, N, 4096):
        b = rows(min(4096, N - at))
        pr.insert(dict(b, prio=prio[at:at + 4096]))
    for B in (64, 1500, 1537, 4000):
        pr.sample(B, 0.7, 11 + B)
    idx = np.arange(3 * K * K, min(N, 3 * K * K + 1000), dtype=np.int32)
    pr.update_priorities(idx, np.where(rng.random(idx.size) < 0.7, -0.0, 2.5).astype(np.float32))
    pr.compare_tree()
    for B in (64, 1500, 1537, 4000):
        pr.sample(B, 0.7, 17 + B)
    pr.compare_state()
    assert pr.compare_status() in (0, 8)
    pr.close()


@pytest.mark.parametrize("K,B", [(4, 20_000), (16, 4096)])
def test_large_batch_beside_other_work(oracle_mod, K, B):
    # the grid's CTAs get their SMs one by one while another stream holds most of them: no CTA may count on the others being there
    rng = np.random.default_rng(B)
    pr = Pair(oracle_mod, 1 << 18, K, 68, 24, 65_536, oracle_store=False)
    for _ in range(4):
        pr.insert(dict(prio=np.exp(rng.standard_normal(65_536)).astype(np.float32)))
    side = torch.cuda.Stream()
    a = torch.randn(8192, 8192, device=pr.dev, dtype=torch.bfloat16)
    torch.cuda.synchronize()
    for i in range(6):
        with torch.cuda.stream(side):
            for _ in range(3):
                a @ a
        pr.sample(B, 0.4, i)
    pr.compare_state()
    pr.compare_status()
    pr.close()


@pytest.mark.parametrize("K,B", [(2, 1537), (8, 5000), (16, 160_000)])
def test_weights_left_to_the_last_cta(oracle_mod, K, B):
    # the checked library looks at no other CTA's progress: all CTAs but one leave their priorities behind, of one pass of strata or of
    # several (160000: more than 512 strata a CTA)
    rng = np.random.default_rng(B)
    pr = Pair(oracle_mod, 1 << 18, K, 68, 24, 160_000, oracle_store=False)
    for n in (160_000, 102_144):
        pr.insert(dict(prio=np.exp(rng.standard_normal(n)).astype(np.float32)))
    for i in range(8):
        pr.sample(B, 0.4, i)
    pr.compare_state()
    pr.compare_status()
    pr.close()

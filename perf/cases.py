"""The replay buffer's work that is timed: one case is one or several iterations of a training loop.

An iteration is the one of the training protocol: the priority update for the batch the learner has
finished with, the insertion of the transitions the actors have collected meanwhile, the sample of the
next batch (indices, importance-sampling weights, gathered rows).  A loop written in PyTorch calls the
library once per iteration (`captured` = 0); a loop that is launch-bound captures several iterations in a
CUDA graph and replays it (`captured` = the iterations of the graph); a loop whose learner lives in host
memory goes through the host-buffer call (`host`).

Fields of a case
  capacity, fanout   geometry of the buffer
  fill               part of the ring that holds transitions when the loop starts
  obs, act           bytes of one observation and of one action
  stack              0: both observations are stored; s > 0: one frame per slot, s frames an observation
  batch, insert      transitions sampled and updated, and inserted, per iteration (insert 0: none)
  captured, host     see above
  norm               "batch": weights divided by the batch's largest; "buffer": by the whole buffer's
  min_tree           the buffer keeps a min-tree (for norm "buffer")
  order              "sampled": the update names what the sample before it drew, in that order;
                     "mixed": an index batch in random order with 5 % of its entries naming another's
                     transition (minibatches shuffled by the learner, several learners' batches in one)
"""
import math

import torch

from paper_2311_09445_b200 import PrioritizedReplay
from paper_2311_09445_b200 import workloads as wk

ALPHA, BETA, EPS = 0.6, 0.4, 1e-6
FILL_BYTES = 64 << 20          # rows handed to one insertion while a ring is filled


def case(name, capacity, fanout, obs, act, batch, insert, captured=0, stack=0, norm="batch", min_tree=False, host=False,
         order="sampled", fill=1.0):
    return {"name": name, "capacity": capacity, "fanout": fanout, "fill": fill, "obs": obs, "act": act, "stack": stack,
            "batch": batch, "insert": insert, "captured": captured, "host": host, "norm": norm, "min_tree": min_tree,
            "order": order}


def listed():
    w = wk.WORKLOADS

    def of(wl, name, **kw):
        return case(name, wl.capacity, wl.fanout, wl.obs_bytes, wl.act_bytes, wl.batch, wl.n_insert, stack=wl.frame_stack, **kw)

    return [
        # a control task's replay in its smallest form: launches and host code are the whole cost
        of(w["tiny"], "tiny_step"),
        # the classic-control loop of the benchmark, one call per iteration
        of(w["cartpole_dqn"], "cartpole_step"),
        # the continuous-control loop as a captured graph; the learner hands the batch back shuffled
        of(w["mujoco_ddpg"], "mujoco_steps", captured=8, order="mixed"),
        # the same loop with its learner in host memory
        of(w["mujoco_ddpg"], "mujoco_host_step", host=True),
        # weights normalised over the whole buffer, as the prioritized-replay paper writes them
        case("buffer_norm_steps", 1 << 20, 16, 68, 24, 256, 256, captured=8, norm="buffer", min_tree=True),
        # a binary tree (the form most implementations use) of a capacity that is no power of anything
        case("binary_tree_steps", 1_000_003, 2, 104, 24, 1000, 777, captured=8),
        # many environments stepped at once: large insertions, a large batch for each of them
        case("vector_env_step", 2_000_000, 16, 240, 32, 4096, 16384),
        # large-batch learners: two cells of the benchmark's sweep
        case("large_batch_step", 1 << 22, 32, 68, 24, 4096, 1024),
        case("largest_batch_step", 1 << 24, 4, 68, 24, 65536, 1024),
        # image observations: a single learner's small batch every few environment steps
        case("atari_small_step", 1 << 17, 32, 28224, 4, 32, 4),
        # ... the benchmark's headline loop
        of(w["atari_dqn"], "atari_steps", captured=8),
        # ... and the same with one frame stored per transition
        of(w["atari_dqn_frames"], "frames_steps", captured=8),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["short"] * 7 + ["host", "rows", "frames"])
    fanout = rng.choice([2, 4, 8, 16, 32])
    fill = rng.choice([1.0, 1.0, 1.0, round(rng.uniform(0.2, 0.9), 2)])
    order = rng.choice(["sampled", "sampled", "mixed"])
    norm = rng.choice(["batch", "batch", "batch", "buffer"])
    d = dict(fill=fill, order=order, norm=norm, min_tree=norm == "buffer" and rng.random() < 0.5)
    if kind in ("rows", "frames"):
        fanout = rng.choice([8, 16, 32])
        batch = _log(rng, 24, 512)
        n = rng.choice([0, 4, 16, batch, _log(rng, 16, 512)])
        if kind == "rows":
            obs = rng.choice([12288, 28224, 28224, 36864])
            if obs > 28224:
                batch, n = min(batch, 384), min(n, 384)
            return case("", _log(rng, 1 << 14, 1 << 17), fanout, obs, 4, batch, n, captured=rng.choice([0, 4]), **d)
        frame = rng.choice([7056, 7056, 4096, 9216])
        return case("", _log(rng, 1 << 15, 1 << 19), fanout, 4 * frame, 4, min(batch, 384), n, captured=rng.choice([0, 4]), stack=4, **d)
    obs, act = 4 * _log(rng, 3, 64), 4 * rng.choice([1, 1, 2, 3, 6, 8])
    if kind == "host":
        batch = _log(rng, 16, 2048)
        return case("", _log(rng, 1 << 13, 1 << 21), fanout, obs, act, batch, rng.choice([0, batch, _log(rng, 16, 1024)]), host=True,
                    order=order, fill=fill)
    capacity = _log(rng, 1 << 12, 1 << 24)
    batch = min(_log(rng, 16, 49152), capacity // 4)
    n = min(rng.choice([0, batch, _log(rng, 16, 16384), _log(rng, 16, 16384)]), 16384, capacity // 4)
    captured = rng.choice([0, 4]) if batch <= 2048 and n <= 2048 else 0
    return case("", capacity, fanout, obs, act, batch, n, captured=captured, **d)


def _rows(c, gen, n, first, episode):
    """n transitions as the actors hand them over (frames: every `episode`-th slot begins an episode)."""
    dev = gen.device
    width = c["obs"] // c["stack"] if c["stack"] else c["obs"]
    r = {"obs": torch.randint(0, 256, (n, width), dtype=torch.uint8, device=dev, generator=gen)}
    r["next_obs"] = None if c["stack"] else torch.randint(0, 256, (n, width), dtype=torch.uint8, device=dev, generator=gen)
    r["act"] = torch.randint(0, 256, (n, c["act"]), dtype=torch.uint8, device=dev, generator=gen)
    r["rew"] = torch.randn(n, device=dev, generator=gen)
    r["done"] = (torch.rand(n, device=dev, generator=gen) < 0.01).to(torch.uint8)
    if c["stack"]:
        start = (torch.arange(first, first + n, device=dev) % episode) == 0
        r["done"] = torch.where(start, torch.full_like(r["done"], 2), r["done"])
    r["prio"] = ((_td(gen, n).double().abs() + EPS) ** ALPHA).float()
    return r


def _td(gen, n):
    """TD errors: mostly small, some large (log-normal, the benchmark's heavier tail halved)."""
    return torch.exp(torch.randn(n, device=gen.device, generator=gen))


def prepare(c, seed):
    dev = torch.device("cuda:%d" % torch.cuda.current_device())
    gen = torch.Generator(device=dev)
    gen.manual_seed(seed)
    B, n, N = c["batch"], c["insert"], c["capacity"]
    stored = 2 * c["obs"] + c["act"] + 5 if not c["stack"] else c["obs"] // c["stack"] + c["act"] + 5
    chunk = max(1, min(N, 65536, FILL_BYTES // stored))
    steps = max(1, c["captured"])
    current = torch.cuda.current_stream(dev)
    stream = torch.cuda.Stream(dev) if c["captured"] else current      # (the default stream cannot be captured)
    stream.wait_stream(current)
    with torch.cuda.stream(stream):
        prb = PrioritizedReplay(N, c["fanout"], c["obs"], c["act"], max(B, n, chunk), device=dev, stream=stream,
                                frame_stack=c["stack"], min_tree=c["min_tree"])
        # fill the ring through the insertion call: fresh priorities throughout, rows from one chunk
        rows, at, goal = _rows(c, gen, chunk, 0, 197), 0, max(B, int(N * c["fill"]))
        while at < goal:
            k = min(chunk, goal - at)
            prio = ((_td(gen, k).double().abs() + EPS) ** ALPHA).float()
            prb.insert(rows["obs"][:k], rows["act"][:k], rows["rew"][:k], None if c["stack"] else rows["next_obs"][:k],
                       rows["done"][:k], prio)
            at += k
        del rows
        new = [_rows(c, gen, n, at + i * n, 197) if n else None for i in range(steps)]
        td = [_td(gen, B) for _ in range(steps)]
        host = dict(device="cpu", pin_memory=True) if c["host"] else dict(device=dev)
        out = [{"idx": torch.zeros(B, dtype=torch.int32, **host), "w": torch.zeros(B, **host),
                "obs": torch.zeros((B, c["obs"]), dtype=torch.uint8, **host),
                "act": torch.zeros((B, c["act"]), dtype=torch.uint8, **host), "rew": torch.zeros(B, **host),
                "next_obs": torch.zeros((B, c["obs"]), dtype=torch.uint8, **host),
                "done": torch.zeros(B, dtype=torch.uint8, **host)} for _ in range(steps)]
        # the batch that the loop's first update is for
        first = torch.zeros(B, dtype=torch.int32, device=dev)
        prb.sample(B, BETA, seed, first)
        s = {"case": c, "prb": prb, "seed": seed, "td": td, "new": new, "out": out, "graph": None, "stream": stream}
        if c["order"] == "mixed":
            mixed = first[torch.randperm(B, device=dev, generator=gen)]
            k = max(1, B // 20)
            mixed[torch.randperm(B, device=dev, generator=gen)[:k]] = mixed[torch.randint(0, B, (k,), device=dev, generator=gen)]
            s["upd"] = [mixed.contiguous()] * steps
        else:
            out[-1]["idx"].copy_(first)
            s["upd"] = [out[i - 1]["idx"] for i in range(steps)]
        if c["host"]:
            s["new"] = [{k: None if v is None else v.cpu().pin_memory() for k, v in r.items()} if r else None for r in new]
            s["td"] = [t.cpu().pin_memory() for t in td]
            s["upd"] = [u if not u.is_cuda else u.cpu().pin_memory() for u in s["upd"]]
            torch.cuda.synchronize(dev)
    if c["captured"]:
        torch.cuda.synchronize(dev)
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            for i in range(steps):
                _iteration(s, i)
        s["graph"] = graph
    current.wait_stream(stream)
    return s


def _iteration(s, i):
    c, prb, td, upd, r, o = s["case"], s["prb"], s["td"][i], s["upd"][i], s["new"][i], s["out"][i]
    sampled = (o["idx"], o["w"], o["obs"], o["act"], o["rew"], o["next_obs"], o["done"])
    if r is None:
        fresh = (None,) * 6
    else:
        fresh = (r["obs"], r["act"], r["rew"], r["next_obs"], r["done"], r["prio"])
    if c["host"]:
        prb.step_host(upd, td, ALPHA, EPS, *fresh, c["batch"], BETA, s["seed"], *sampled, n=c["insert"])
    elif c["norm"] == "batch":
        prb.step(upd, td, ALPHA, EPS, *fresh, c["batch"], BETA, s["seed"], *sampled, n=c["insert"])
    else:
        if r is None:
            prb.update(upd, td, ALPHA, EPS)
        else:
            prb.update_insert(upd, td, ALPHA, EPS, *fresh)
        prb.sample_buffer_norm(c["batch"], BETA, s["seed"], *sampled)


def run(s):
    if s["graph"] is not None:
        s["graph"].replay()
    else:
        _iteration(s, 0)
    return s["out"]


def work(c):
    B, n, K = c["batch"], c["insert"], c["fanout"]
    small = c["act"] + 5
    if c["stack"]:
        frame = c["obs"] // c["stack"]
        read, written, stored = (c["stack"] + 1) * frame + small, 2 * c["obs"] + small, frame + small
    else:
        read = written = stored = 2 * c["obs"] + small
    # the sampled rows, the new rows in and out, indices, TD errors, weights and priorities
    nbytes = B * (read + written + 8) + 2 * n * stored + B * 8 + n * 4
    # the tree: the child groups on the paths of the sampled, updated and inserted leaves (each node of a
    # level at most once), read, and one node per group written
    level, groups = c["capacity"], 0
    while level > 1:
        groups += min((level + K - 1) // K, 2 * B + (n + K - 1) // K)
        level = (level + K - 1) // K
    nbytes += groups * (K + 1) * 4
    flops = groups * 2 * K + B * 160
    steps = max(1, c["captured"])
    return {"bytes": steps * nbytes, "flops": steps * flops}


def tolerance(c):
    # Indices and rows are whole numbers and do not differ.  A weight is formed in binary64 and rounded once to
    # binary32.  Against the same weights formed in binary64 from the stored priorities the listed cases show
    # 2.5e-8 .. 2.9e-8 (2-norm) and 7e-8 at most (a rounding is half a unit in the last place, 6e-8): four
    # times that.
    return {"rel": 1.2e-7, "max": 3e-7, "differ": 0.0}

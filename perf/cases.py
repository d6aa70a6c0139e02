"""What the library is asked to do in earnest, as cases that can be timed: training steps from the smallest to the largest
configuration, evaluation, steps from host buffers, and the model snapshot -- each through the public entry points of
`paper_2010_11305_b200.binding`, the way a training program calls them.

A case is a dict of plain values:
  mode     "train"     `steps` consecutive training steps (forward, backward) on as many batches
           "eval"      the forward pass alone over `steps` batches (validation)
           "static"    the allocation-free evaluation forward over `steps` small batches (serving beside other work)
           "host"      `steps` training steps from pinned host buffers, submitted back to back, then one wait
           "snapshot"  flush the caches and read every table back to the host (a checkpoint)
  ahead    train: the next batch is handed to prepare() while the current step runs (the loop the C header documents)
  tables, rows_lo, rows_hi   number of tables and their row counts, spread over the logarithm of the range
  dim, bits, cache, ways, lfu, adagrad   as in Mpe(...)
  batch, bag, mean, cap      samples per batch; bag lengths "fixed" (mean), "poisson" or "poisson_cap" (at most cap)
  zipf_lo, zipf_hi           per-table exponent of the row ids, spread over the range; 0 and 0 = uniform ids
  steps    steps or batches of one pass
"""
import math
import random

import numpy as np
import torch

from paper_2010_11305_b200 import binding as mpe
from paper_2010_11305_b200 import workloads as wl

WARM_STEPS = 4          # training steps on other batches before the timed ones: caches, counters and time stamps are in use


def _case(name, mode, tables, rows, dim, bits, cache, ways, lfu, adagrad, batch, bag, mean, zipf, steps, ahead=False, cap=100):
    return {"name": name, "mode": mode, "tables": tables, "rows_lo": rows[0], "rows_hi": rows[1], "dim": dim, "bits": bits,
            "cache": cache, "ways": ways, "lfu": lfu, "adagrad": adagrad, "batch": batch, "bag": bag, "mean": mean, "cap": cap,
            "zipf_lo": zipf[0], "zipf_hi": zipf[1], "steps": steps, "ahead": ahead}


def listed():
    return [
        # configuration 1: the smallest model, where a step is a handful of short launches
        _case("train_tiny", "train", 1, (10_000, 10_000), 16, 8, 0.05, 8, False, False, 128, "fixed", 4, (1.05, 1.05), 4),
        # configuration 2: 26 tables of very different sizes, one index per table and sample (Criteo-Kaggle's shape)
        _case("train_criteo", "train", 26, (3, 10_000_000), 16, 8, 0.05, 32, True, False, 2048, "fixed", 1, (1.1, 1.1), 4),
        # an odd batch over uneven FP16 tables (the paper's FP16 + LRU setting at a ragged size)
        _case("train_fp16_ragged", "train", 13, (11, 2_000_000), 32, 16, 0.01, 32, False, False, 3001, "poisson_cap", 11, (0.9, 1.3), 4,
              cap=50),
        # configuration 5: two corners of the policy / skew sweep
        _case("train_sweep_int8_lru", "train", 4, (10_000_000, 10_000_000), 64, 8, 0.01, 32, False, False, 8192, "fixed", 10,
              (1.05, 1.05), 4, ahead=True),
        _case("train_sweep_int4_lfu_uniform", "train", 4, (10_000_000, 10_000_000), 64, 4, 0.05, 32, True, False, 8192, "fixed", 10,
              (0, 0), 4),
        # configuration 3: multi-hot bags, packed INT4, row-wise Adagrad
        _case("train_int4_adagrad", "train", 8, (20_000_000, 20_000_000), 64, 4, 0.01, 16, False, True, 4096, "poisson", 20,
              (1.2, 1.2), 4, ahead=True),
        # between configurations 3 and 4: many mid-sized tables, INT8
        _case("train_mid_int8", "train", 32, (300_000, 3_000_000), 64, 8, 0.05, 32, True, True, 8192, "poisson_cap", 25, (1.0, 1.3), 3,
              ahead=True),
        # configuration 4: the largest model, 31 million indices per step
        _case("train_largest", "train", 64, (5_000_000, 5_000_000), 128, 4, 0.01, 32, True, False, 16384, "poisson_cap", 30,
              (1.0, 1.3), 3, ahead=True),
        # a small request answered without allocating, beside other work on the GPU
        _case("eval_static_small", "static", 26, (1_000, 1_000_000), 32, 8, 0.05, 32, False, False, 257, "poisson_cap", 3, (1.05, 1.05), 4,
              cap=12),
        # validation: forward only, large bags, wide rows
        _case("eval_large", "eval", 16, (5_000_000, 5_000_000), 128, 8, 0.01, 32, True, False, 16384, "poisson_cap", 30, (1.0, 1.3), 2),
        # a training program whose batches arrive in pinned host memory
        _case("host_steps", "host", 4, (10_000_000, 10_000_000), 64, 8, 0.01, 32, False, False, 8192, "fixed", 10, (1.05, 1.05), 6),
        # checkpoint: every cached row written back, every table read to the host
        _case("snapshot", "snapshot", 6, (20_000, 500_000), 64, 8, 0.05, 32, True, False, 4096, "fixed", 4, (1.05, 1.05), 1),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng: random.Random):
    mode = rng.choices(["train", "eval", "static", "host", "snapshot"], [65, 12, 8, 9, 6])[0]
    dim, bits = rng.choice([16, 32, 64, 128]), rng.choices([8, 4, 16, 2], [5, 4, 2, 1])[0]
    while True:
        tables = _log_int(rng, 1, {"static": 40, "snapshot": 10}.get(mode, 64))
        rows_hi = _log_int(rng, 1_000, {"static": 1_000_000, "snapshot": 400_000}.get(mode, 10_000_000))
        rows_lo = max(3, int(rows_hi * rng.choice([1, 1, 0.1, 0.001])))
        batch = _log_int(rng, 100, {"static": 1024, "host": 8192, "snapshot": 4096}.get(mode, 16384))
        bag = rng.choice(["fixed", "poisson", "poisson_cap"])
        mean = _log_int(rng, 1, {"static": 8, "snapshot": 8}.get(mode, 40))
        total = tables * batch * mean
        if total > {"static": 28_000, "host": 3_000_000, "snapshot": 500_000}.get(mode, 28_000_000) or total < 400:
            continue
        if mode == "static" and tables * batch > 32_768:
            continue
        if tables * rows_hi * (dim * bits // 8 + 12) > 16e9 or tables * rows_hi * dim > 4e10:
            continue
        if batch * tables * dim > (8_000_000 if mode == "host" else 120_000_000):
            continue
        break
    uniform = rng.random() < 0.15
    z = sorted(rng.uniform(0.8, 1.4) for _ in range(2))
    c = _case("", mode, tables, (rows_lo, rows_hi), dim, bits, rng.choice([0.005, 0.01, 0.05, 0.1]), rng.choices([32, 16, 8, 4, 1], [6, 3, 2, 1, 1])[0],
              rng.random() < 0.5, rng.random() < 0.35, batch, bag, mean, (0, 0) if uniform else (round(z[0], 3), round(z[1], 3)),
              {"snapshot": 1, "eval": 2}.get(mode, 2 if total > 4_000_000 else 4), ahead=mode == "train" and rng.random() < 0.5,
              cap=max(2, 3 * mean))
    del c["name"]
    return c


def _spread(lo, hi, n, log):
    if n == 1 or lo == hi:
        return [hi] * n
    if log:
        return [int(round(math.exp(math.log(lo) + (math.log(hi) - math.log(lo)) * i / (n - 1)))) for i in range(n)]
    return [lo + (hi - lo) * i / (n - 1) for i in range(n)]


def _rows(case):
    return _spread(case["rows_lo"], case["rows_hi"], case["tables"], True)


def _zipf(case):
    """Exponents in an order of their own, so that skew and table size are not tied to each other."""
    z = _spread(case["zipf_lo"], case["zipf_hi"], case["tables"], False)
    random.Random(case["tables"]).shuffle(z)
    return [float(a) if a > 0 else None for a in z]


def _config(case, seed):
    bag = (case["bag"], case["mean"]) + ((case["cap"],) if case["bag"] == "poisson_cap" else ())
    return wl.Config("case", _rows(case), case["dim"], case["bits"], case["cache"], case["ways"], wl.LFU if case["lfu"] else wl.LRU,
                     wl.ROWWISE_ADAGRAD if case["adagrad"] else wl.SGD, 0.05, case["batch"], bag, _zipf(case), case["steps"], seed=seed)


class _State:
    """What a program holds: the handle, its batches, its output buffers, its streams and the step number."""


def prepare(case, seed):
    s = _State()
    cfg = s.cfg = _config(case, int(seed) % 1_000_003)
    s.mode, s.B, s.ahead = case["mode"], cfg.batch, case["ahead"]
    dev = torch.device("cuda", 0)
    s.h = mpe.Mpe(cfg.num_rows, cfg.dim, cfg.bits, cfg.cache_fraction, cfg.ways, cfg.policy, cfg.optimizer, cfg.eps, cfg.init_lo,
                  cfg.init_hi, cfg.seed, 0)
    data = wl.Stream(cfg, dev)
    batches = [data.batch(k) for k in range(1, WARM_STEPS + cfg.steps + 1)]
    s.h.reserve(cfg.batch, max(b[0].numel() for b in batches))
    s.stream = torch.cuda.current_stream(dev).cuda_stream
    s.side = torch.cuda.Stream(dev)                     # the next batch is prepared here
    s.step = 0
    s.outs = [torch.empty(cfg.batch, cfg.num_tables * cfg.dim, dtype=torch.float32, device=dev) for _ in range(cfg.steps)]
    s.batches = batches[:WARM_STEPS]
    _train(s, s.outs[:1] * WARM_STEPS)
    s.batches = batches[WARM_STEPS:]
    if s.mode == "host":
        s.batches = [tuple(x.cpu().pin_memory() for x in b) for b in s.batches]
        s.outs = [torch.empty(cfg.batch, cfg.num_tables * cfg.dim, dtype=torch.float32).pin_memory() for _ in range(cfg.steps)]
    if s.mode == "snapshot":
        s.all_rows = [np.arange(n, dtype=np.int64) for n in cfg.num_rows]
    return s


def _train(s, outs):
    """The training loop of the C header: forward(k); prepare(k+1, other stream); backward(k)."""
    for k, (indices, offsets, grad) in enumerate(s.batches):
        s.step += 1
        s.h.forward(indices, offsets, s.B, outs[k], s.stream)
        if s.ahead and k + 1 < len(s.batches):
            s.h.prepare(s.batches[k + 1][0], s.batches[k + 1][1], s.B, s.side.cuda_stream)
        s.h.backward(grad, s.cfg.lr, s.step)


def run(s):
    """Pooled vectors of every batch; from the second batch on they show the rows that the steps before it have updated."""
    if s.mode == "train":
        _train(s, s.outs)
    elif s.mode == "eval":
        for k, (indices, offsets, _) in enumerate(s.batches):
            s.h.forward(indices, offsets, s.B, s.outs[k], s.stream)
    elif s.mode == "static":
        for k, (indices, offsets, _) in enumerate(s.batches):
            s.h.forward_static(indices, offsets, s.B, s.outs[k], s.stream)
    elif s.mode == "host":
        for k, (indices, offsets, grad) in enumerate(s.batches):
            s.step += 1
            s.h.step_host_submit(indices, offsets, s.B, grad, s.outs[k], s.cfg.lr, s.step)
        s.h.step_host_wait()
    else:
        s.h.flush()
        return [a for t, rows in enumerate(s.all_rows) for a in s.h.export_rows(t, rows) + s.h.export_aux(t, rows)]
    return s.outs


def _distinct(n_rows, zipf, draws, slots):
    """Expected number of distinct rows among `draws` ids, and how many of them are among the `slots` likeliest rows."""
    edges = np.unique(np.round(np.geomspace(1, n_rows + 1, 2000)).astype(np.int64))
    edges = np.unique(np.concatenate([edges, [1, min(slots, n_rows) + 1, n_rows + 1]]))
    mid, width = (edges[:-1] + edges[1:] - 1) / 2.0, np.diff(edges).astype(np.float64)
    p = mid ** -(zipf or 0.0)
    p /= float((p * width).sum())
    seen = -np.expm1(-draws * p) * width
    return float(seen.sum()), float(seen[edges[:-1] <= slots].sum())


def work(case):
    """Bytes: every index, offset, pooled value and gradient once; per distinct row of a batch one read and (in training) one
    write of the row where it lives -- FP32 in the cache, codes with scale and bias in the table -- and its tag, priority value
    and optimizer state."""
    d, bits, T, B = case["dim"], case["bits"], case["tables"], case["batch"]
    rb, fb = d * bits // 8 + (0 if bits == 16 else 8), 4 * d
    rows = _rows(case)
    slots = [max(1, int(case["cache"] * n) // case["ways"]) * case["ways"] for n in rows]
    if case["mode"] == "snapshot":
        aux = 4 * (int(case["lfu"]) + int(case["adagrad"]))
        return {"bytes": 2.0 * sum(rows) * (rb + aux) + sum(min(n, s) for n, s in zip(rows, slots)) * (fb + rb), "flops": 0.0}
    per_table = float(B * case["mean"])
    L = per_table * T
    seen = [_distinct(n, z, per_table, s) for n, z, s in zip(rows, _zipf(case), slots)]
    U, hits = sum(a for a, _ in seen), sum(b for _, b in seen)
    train = case["mode"] in ("train", "host")
    nbytes = 4 * L + 4 * (T * B + 1) + 4.0 * B * T * d + 4 * U + (2 if train else 1) * (hits * fb + (U - hits) * rb)
    flops = L * d
    if train:
        nbytes += 4.0 * B * T * d + (8 * U if case["lfu"] else 4 * hits) + (8 * U if case["adagrad"] else 0)
        flops += L * d + 10 * U * d
    return {"bytes": case["steps"] * nbytes, "flops": case["steps"] * flops}


def tolerance(case):
    """Codes, scales, biases and counters are defined bit for bit; pooled vectors are FP32 sums of FP32 terms."""
    return "exact" if case["mode"] == "snapshot" else {"rel": 1e-5}

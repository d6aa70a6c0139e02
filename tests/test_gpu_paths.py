"""Each kernel variant at the sizes where it begins, ends or has a remainder, against the CPU oracle.

The library chooses by sizes: a thread-block cluster per table sorts a batch (4096 or 12288 elements per block; a table with
more than its cluster holds goes through global memory) until the tables average over 150000 indices or one of them is larger than
that in the batches seen so far, then, and as long as none has been seen, grid-wide kernels do; up
to 131072 indices one launch updates every row; a row's gradient is summed by its group of lanes, by a warp's list of mid rows (from
16 occurrences) or by whole blocks (from 64 or 256); a cache set finds its candidates in a bucket until that overflows."""
import numpy as np
import pytest
import torch

from paper_2010_11305_b200 import workloads as wl

pytestmark = pytest.mark.gpu


def _cfg(num_rows, batch, **kw):
    base = dict(name="paths", num_rows=num_rows, dim=4, bits=8, cache_fraction=0.05, ways=8, policy=wl.LFU, optimizer=wl.SGD, lr=0.05,
                batch=batch, bag=("fixed", 1), zipf=[None] * len(num_rows), steps=2, seed=3)
    base.update(kw)
    return wl.Config(**base)


def _batch(rng, ids, batch, dim):
    """One batch from a list of ids per table, the ids cut into `batch` bags at random places."""
    lens = []
    for x in ids:
        cuts = np.sort(rng.integers(0, len(x) + 1, batch - 1))
        lens.append(np.diff(np.concatenate([[0], cuts, [len(x)]])))
    off = np.concatenate([[0], np.cumsum(np.concatenate(lens))]).astype(np.int32)
    grad = rng.uniform(-1, 1, (batch, len(ids) * dim)).astype(np.float32)
    return np.concatenate(ids).astype(np.int32), off, grad


def _check(cfg, make_ids, steps=2):
    from parity_util import compare_state, make_pair
    h, o = make_pair(cfg)
    rng = np.random.default_rng(cfg.seed)
    for step in range(1, steps + 1):
        idx, off, grad = _batch(rng, make_ids(rng), cfg.batch, cfg.dim)
        out = torch.empty(cfg.batch, cfg.num_tables * cfg.dim, device="cuda")
        h.forward(torch.from_numpy(idx).cuda(), torch.from_numpy(off).cuda(), cfg.batch, out)
        ref = o.forward(idx, off, cfg.batch)
        assert np.array_equal(out.cpu().numpy(), ref), f"step {step}"
        h.backward(torch.from_numpy(grad).cuda(), cfg.lr, step)
        o.backward(grad, cfg.lr, step)
    assert h.last_error() == (0, 0)
    compare_state(h, o, cfg, range(cfg.num_tables), rng)
    h.close()


def _skewed(rng, n_rows, count):
    return np.minimum((n_rows * rng.random(count) ** 3).astype(np.int64), n_rows - 1)


@pytest.mark.parametrize("counts", [
    (0, 1, 31, 33, 1023, 1025, 3000),           # one block per table, tables without indices among them
    (3641,), (3642,), (4097,),                  # the last size of one block, the first of two
    (8000, 10, 0),                              # four blocks, for one table that is larger than the average
    (7281,), (7283, 7290), (57000,),            # two, four and sixteen blocks
    (60000, 5, 5),                              # sixteen
    (5000,) * 99 + (12289,),                    # one table beyond 12288 elements per block, which all have: grid-wide
    (100003,), (199000, 900),                   # sixteen large blocks: within; one table beyond: grid-wide
    (150000,), (150001,),                       # the last average of the cluster kernel, the first of the grid-wide ones
    (320000, 7, 0), (1048576 + 9,),             # grid-wide: a few tiles and none, large tiles
])
def test_index_work_at_its_boundaries(counts):
    """The host has waited for the forward when it chooses the kernels of the backward, so it goes by this batch's largest table."""
    num_rows = [max(3, c // 3) for c in counts]
    num_rows[0] = 70001                         # keys of three digits
    _check(_cfg(num_rows, 16), lambda rng: [_skewed(rng, n, c) for n, c in zip(num_rows, counts)])


@pytest.mark.parametrize("total", [131072, 131073])
def test_one_launch_update_at_its_last_size(total):
    counts = [total // 36 + (t < total % 36) for t in range(36)]
    _check(_cfg([9000] * 36, 64, dim=8), lambda rng: [_skewed(rng, 9000, c) for c in counts])


@pytest.mark.parametrize("dim,bits,rest,tables", [(4, 8, 300, 1), (64, 4, 400, 3), (128, 16, 300, 1), (4, 8, 140000, 1), (64, 4, 140000, 1),
                                                  (128, 16, 140000, 1), (4, 8, 1 << 20, 1)])
def test_rows_with_few_and_many_occurrences(dim, bits, rest, tables):
    """Multiplicities around every limit of the gradient sums, beside rows that occur once or twice."""
    times = [1, 2, 15, 16, 17, 31, 32, 33, 63, 64, 65, 255, 256, 257, 1023, 1024, 1025, 2100]
    hot = np.repeat(np.arange(len(times)), times)
    cfg = _cfg([900000] * tables, 512, dim=dim, bits=bits, cache_fraction=0.001, optimizer=wl.ROWWISE_ADAGRAD)
    _check(cfg, lambda rng: [rng.permutation(np.concatenate([hot, rng.integers(100, 900000, rest)])) for _ in range(tables)])


@pytest.mark.parametrize("ways", [1, 2, 4, 8, 16, 32])
@pytest.mark.parametrize("policy", [wl.LRU, wl.LFU])
@pytest.mark.parametrize("count", [3000, 9000])
def test_sets_with_few_and_with_too_many_candidates(ways, policy, count):
    """Per set about half as many candidates as ways, one and a half times, and five times as many; one block per table (which
    admits by itself) and several."""
    sizes = [40000, 8000, 2500]
    cfg = _cfg(sizes, 128, ways=ways, policy=policy, cache_fraction=0.2, dim=8, bits=4)
    _check(cfg, lambda rng: [_skewed(rng, n, count) for n in sizes], steps=4)


@pytest.mark.parametrize("dim,bits,n", [(64, 8, 400001), (4, 2, 5000003)])
def test_exports_of_many_pieces(dim, bits, n):
    """More rows than one staging slot takes, in any order and more than once; rows that are whole words, and of one byte."""
    from parity_util import make_pair
    cfg = _cfg([300000], 16, dim=dim, bits=bits)
    h, o = make_pair(cfg)
    rows = np.random.default_rng(1).integers(0, 300000, n)
    every = np.arange(300000, dtype=np.int64)
    for got, ref in zip(h.export_rows(0, rows), o.rows(0, every)):
        assert np.array_equal(got, ref[rows])
    h.close()


def _ahead(cfg, counts, stream, busy):
    """The loop forward(k); prepare(k + 1); backward(k) with no wait of the host between them, against the oracle; counts[k] indices
    per table in step k, the workspace reserved when it grows.  `busy`: clock cycles of other work in front of every forward, so
    that all that follows is queued behind it."""
    from parity_util import compare_state, make_pair
    h, o = make_pair(cfg)
    rng = np.random.default_rng(cfg.seed)
    T, steps = cfg.num_tables, len(counts)
    batches = [_batch(rng, [_skewed(rng, r, c) for r in cfg.num_rows], cfg.batch, cfg.dim) for c in counts]
    dev = [tuple(torch.from_numpy(x).cuda() for x in b) for b in batches]
    outs = [torch.empty(cfg.batch, T * cfg.dim, device="cuda") for _ in range(steps)]
    side = torch.cuda.Stream()
    torch.cuda.synchronize()
    with torch.cuda.stream(stream):
        for k, (idx, off, grad) in enumerate(dev):
            h.reserve(cfg.batch, T * counts[k])
            if busy:
                torch.cuda._sleep(busy)
            h.forward(idx, off, cfg.batch, outs[k], stream.cuda_stream)
            if k + 1 < steps:
                h.prepare(dev[k + 1][0], dev[k + 1][1], cfg.batch, side.cuda_stream)
            h.backward(grad, cfg.lr, k + 1)
    assert h.last_error() == (0, 0)
    for k, (idx, off, grad) in enumerate(batches):
        assert np.array_equal(outs[k].cpu().numpy(), o.forward(idx, off, cfg.batch)), f"step {k + 1}"
        o.backward(grad, cfg.lr, k + 1)
    compare_state(h, o, cfg, range(T), rng)
    h.close()


@pytest.mark.parametrize("count", [300, 155000])
def test_first_prepared_batch_of_a_handle_whose_memory_was_used_before(count):
    """The second workspace is allocated by the first prepare, in memory that an earlier handle has left full, while the default
    stream is busy with the forward: its counters have to be zero before the sort on the other stream begins."""
    for seed in (3, 4, 5):
        _ahead(_cfg([70001, 900], 64, seed=seed), [count] * 3, torch.cuda.default_stream(), 20_000_000)


@pytest.mark.parametrize("count", [300, 155000])
def test_step_on_a_non_blocking_stream_straight_after_reserve(count):
    """The workspace grows between two steps of a stream that does not wait for the default one."""
    for seed in (6, 7):
        _ahead(_cfg([70001, 900], 64, seed=seed), [count // 3, count, count, 2 * count, 2 * count], torch.cuda.Stream(), 0)


class _OneStepMore:
    """A handle that has counted a step which the oracle never saw."""
    def __init__(self, h):
        self._h = h

    def __getattr__(self, name):
        return getattr(self._h, name)

    def stats(self, t):
        s = np.array(self._h.stats(t))
        s[7] -= 1
        return s


def _abandon(cfg, counts, abandoned):
    """Three steps; before the second one the look-backs of the next sort are made to give up."""
    from paper_2010_11305_b200 import binding as mpe
    from parity_util import compare_state, make_pair
    h, o = make_pair(cfg)
    rng = np.random.default_rng(cfg.seed)
    every = range(cfg.num_tables)
    for step in (1, 2, 3):
        idx, off, grad = _batch(rng, [_skewed(rng, r, c) for r, c in zip(cfg.num_rows, counts)], cfg.batch, cfg.dim)
        if step == 2:
            h.selftest(mpe.SELFTEST_ABANDON_NEXT_SORT)
        out = torch.empty(cfg.batch, cfg.num_tables * cfg.dim, device="cuda")
        h.forward(torch.from_numpy(idx).cuda(), torch.from_numpy(off).cuda(), cfg.batch, out)
        assert np.array_equal(out.cpu().numpy(), o.forward(idx, off, cfg.batch)), f"step {step}"
        h.backward(torch.from_numpy(grad).cuda(), cfg.lr, step)
        code, detail = h.last_error()
        if step == 2 and abandoned:
            assert code == mpe.ERR_TIMEOUT and detail > 0
        else:
            assert (code, detail) == (0, 0)
            o.backward(grad, cfg.lr, step)
        compare_state(_OneStepMore(h) if abandoned and step >= 2 else h, o, cfg, every, rng)
    h.close()


@pytest.mark.parametrize("policy,optimizer", [(wl.LFU, wl.ROWWISE_ADAGRAD), (wl.LRU, wl.SGD)])
@pytest.mark.parametrize("counts", [(3000, 900, 0, 31), (8000, 7000), (20000, 90000)])
def test_steps_sorted_inside_clusters_have_no_wait_that_could_abandon_them(counts, policy, optimizer):
    """No table waits for another one, so a step cannot be left with some tables' priorities and caches changed and others' not."""
    _abandon(_cfg([9000] * len(counts), 64, policy=policy, optimizer=optimizer), counts, abandoned=False)


@pytest.mark.parametrize("policy,optimizer", [(wl.LFU, wl.ROWWISE_ADAGRAD), (wl.LRU, wl.SGD)])
def test_a_step_whose_sort_is_abandoned_changes_nothing(policy, optimizer):
    """Tables, caches, counters, accumulators and statistics stay as they were, and the next step goes on from there."""
    _abandon(_cfg([90000, 900], 64, policy=policy, optimizer=optimizer), (302000, 500), abandoned=True)


def _planned(num_rows, seen, counts, busy, **kw):
    """A step with `counts` indices per table after a step with `seen` (None: it is the handle's first).  `busy`: the GPU has other work
    while the host chooses the kernels of the step, so that it knows of the earlier batches only.  Returns the kernels it chose."""
    from parity_util import compare_state, make_pair
    cfg = _cfg(num_rows, 16, **kw)
    h, o = make_pair(cfg)
    rng = np.random.default_rng(cfg.seed)
    batches = [_batch(rng, [_skewed(rng, r, c) for r, c in zip(num_rows, cs)], cfg.batch, cfg.dim) for cs in (seen, counts) if cs]
    dev = [tuple(torch.from_numpy(x).cuda() for x in b) for b in batches]
    h.reserve(cfg.batch, max(b[0].size for b in batches))
    for step, ((idx, off, grad), (d_idx, d_off, d_grad)) in enumerate(zip(batches, dev), start=1):
        out = torch.empty(cfg.batch, cfg.num_tables * cfg.dim, device="cuda")
        last = step == len(batches)
        h.profile(last)
        torch.cuda.synchronize()
        if busy and last:
            torch.cuda._sleep(40_000_000)
        h.forward(d_idx, d_off, cfg.batch, out)
        if not (busy and last):
            torch.cuda.synchronize()
        h.backward(d_grad, cfg.lr, step)
        assert np.array_equal(out.cpu().numpy(), o.forward(idx, off, cfg.batch)), f"step {step}"
        o.backward(grad, cfg.lr, step)
    chosen = set(h.profile_read())
    assert h.last_error() == (0, 0)
    compare_state(h, o, cfg, range(cfg.num_tables), rng)
    h.close()
    return chosen


@pytest.mark.parametrize("counts,kernel", [
    ((3000,) * 5, "table"), ((3641, 3641, 10), "table"),            # one block per table
    ((7000, 7000, 3000), "table_sort"),                             # several
    ((20000, 10000) + (2000,) * 18, "table_sort"),                  # a larger one among small ones: all clusters grow with it
    ((51200,) + (512,) * 25, "sort_scatter"),                       # one that would take more than the GPU has for each
    ((512,) * 25 + (151000,), "sort_scatter"),                      # one that fits no cluster
])
def test_kernels_follow_the_largest_table_not_only_the_average(counts, kernel):
    chosen = _planned([max(3, c // 3) for c in counts], counts, counts, busy=False)
    assert kernel in chosen and len(chosen & {"table", "table_sort", "sort_scatter"}) == 1, chosen


@pytest.mark.parametrize("counts", [(8000, 10, 0), (60000, 5, 5), (5000,) * 99 + (12289,), (199000, 900)])
def test_a_table_larger_than_the_batches_before_let_expect(counts):
    """Its cluster sorts it through global memory: one block, sixteen small ones, one large one, sixteen large ones."""
    even = [max(1, sum(counts) // len(counts) - 100)] * len(counts)
    num_rows = [max(3, c // 3) for c in counts]
    num_rows[0] = 70001
    assert _planned(num_rows, even, counts, busy=True) & {"table", "table_sort"}


@pytest.mark.parametrize("counts", [(1,), (0, 0), (0, 1, 31, 33, 1023, 1025, 3000), (2048, 2049, 0), (4097,) * 30, (57000,)])
def test_first_step_of_a_handle_has_no_earlier_batch_to_go_by(counts):
    num_rows = [max(3, c // 3) for c in counts]
    num_rows[0] = 70001
    assert "sort_scatter" in _planned(num_rows, None, counts, busy=True)


@pytest.mark.parametrize("count,rows,steps,ahead", [(700, 3000, 150, False), (30000, 40000, 60, True), (160000, 60000, 30, True)])
def test_forward_behind_a_backward_reads_what_that_one_wrote(count, rows, steps, ahead):
    """The forward's blocks may be on the GPU before the last kernel of the step before has finished.  A second forward of the same
    batch, behind a wait, must give the same values to the bit."""
    from paper_2010_11305_b200 import binding as mpe
    T, dim, B = 3, 32, 64
    rng = np.random.default_rng(count)
    h = mpe.Mpe([rows] * T, dim, 4, 0.05, 4, mpe.LFU, seed=5)
    batches = [tuple(torch.from_numpy(x).cuda() for x in _batch(rng, [_skewed(rng, rows, count) for _ in range(T)], B, dim)) for _ in range(4)]
    h.reserve(B, T * count)
    outs = torch.zeros(2, B, T * dim, device="cuda")
    wrong = torch.zeros(1, dtype=torch.int64, device="cuda")
    side = torch.cuda.Stream()
    torch.cuda.synchronize()
    for step in range(1, steps + 1):
        idx, off, grad = batches[step % 4]
        h.forward(idx, off, B, outs[0])
        if ahead:
            side.wait_stream(torch.cuda.current_stream())
            h.prepare(batches[(step + 1) % 4][0], batches[(step + 1) % 4][1], B, side.cuda_stream)
        h.backward(grad, 0.5, step)
        if step % 5 == 0:                             # the next batch once more: behind the backward, then behind a wait
            nxt = batches[(step + 1) % 4]
            h.forward(nxt[0], nxt[1], B, outs[0])
            torch.cuda.synchronize()
            h.forward(nxt[0], nxt[1], B, outs[1])
            wrong += (outs[0] != outs[1]).sum()
    assert int(wrong) == 0 and h.last_error() == (0, 0)
    h.close()


@pytest.mark.parametrize("what", ["event", "copy"])
def test_forward_waits_for_what_the_caller_put_in_front_of_it(what):
    """Between a backward, whose last kernel lets the next one be set up early, and the next forward the caller makes the stream wait
    for another one that writes the batch, or copies the batch in."""
    from parity_util import make_pair
    cfg = _cfg([3000, 500], 64, dim=16)
    h, o = make_pair(cfg)
    rng = np.random.default_rng(1)
    batches = [_batch(rng, [_skewed(rng, n, 400) for n in cfg.num_rows], cfg.batch, cfg.dim) for _ in range(12)]
    pinned = [tuple(torch.from_numpy(x).pin_memory() for x in b) for b in batches]
    dev = [tuple(torch.from_numpy(x).cuda() for x in b) for b in batches]
    idx, off, grad = (torch.zeros_like(x) for x in dev[0])
    big, big_host = torch.empty(1 << 23, device="cuda"), torch.empty(1 << 23).pin_memory()
    outs = [torch.empty(cfg.batch, cfg.num_tables * cfg.dim, device="cuda") for _ in batches]
    own, other = torch.cuda.Stream(), torch.cuda.Stream()
    torch.cuda.synchronize()
    with torch.cuda.stream(own):
        for k in range(len(batches)):
            if what == "event":
                other.wait_stream(own)
                with torch.cuda.stream(other):
                    torch.cuda._sleep(500_000)
                    for to, frm in zip((idx, off, grad), dev[k]):
                        to.copy_(frm)
                own.wait_stream(other)
            else:
                big.copy_(big_host, non_blocking=True)
                for to, frm in zip((idx, off, grad), pinned[k]):
                    to.copy_(frm, non_blocking=True)
            h.forward(idx, off, cfg.batch, outs[k], own.cuda_stream)
            h.backward(grad, cfg.lr, k + 1)
    torch.cuda.synchronize()
    assert h.last_error() == (0, 0)
    for k, b in enumerate(batches):
        assert np.array_equal(outs[k].cpu().numpy(), o.forward(b[0], b[1], cfg.batch)), f"step {k + 1}"
        o.backward(b[2], cfg.lr, k + 1)
    h.close()


@pytest.mark.parametrize("counts", [(3000, 900), (8000, 7000), (160000, 150100)])
def test_step_info_is_the_same_before_and_after_backward(counts):
    from paper_2010_11305_b200 import binding as mpe
    rng = np.random.default_rng(2)
    ids = [np.concatenate([_skewed(rng, 5000, c - 700), np.full(400, 7), np.full(300, 9000 + t)]) for t, c in enumerate(counts)]
    idx, off, grad = (torch.from_numpy(x).cuda() for x in _batch(rng, [rng.permutation(x) for x in ids], 16, 4))
    h = mpe.Mpe([5000] * len(counts), 4, 8, 0.05, 8, mpe.LFU)
    out = torch.empty(16, 4 * len(counts), device="cuda")
    ref = np.array([0] * 6, np.int64)
    threshold = 64 if sum(counts) <= 1 << 20 else 256
    for x in ids:
        n = np.bincount(x[x < 5000])
        ref += [int(n.sum()), int((n > 0).sum()), 300, int((n > threshold).sum()), int(n[n > threshold].sum()), 0]
    for step in (1, 2):
        h.forward(idx, off, 16, out)
        torch.cuda.synchronize()
        before = np.array(h.step_info())
        h.backward(grad, 0.1, step)
        after = np.array(h.step_info())
        assert np.array_equal(before[:5], ref[:5]) and np.array_equal(after[:5], ref[:5]) and ref[3] > 0, (before, after, ref)
    h.close()


def test_many_handles_at_once():
    """Handles share a page of host words: 70 are more than it holds, and a word is as good as new for its next handle."""
    from paper_2010_11305_b200 import binding as mpe
    idx, off, grad = (torch.from_numpy(x).cuda() for x in _batch(np.random.default_rng(3), [np.arange(300) % 90], 8, 4))
    outs = []

    def use(h):
        out = torch.empty(8, 4, device="cuda")
        for step in (1, 2):
            h.forward(idx, off, 8, out)
            torch.cuda.synchronize()
            h.backward(grad, 0.1, step)
        h.forward(idx, off, 8, out)
        assert h.last_error() == (0, 0)
        outs.append(out.cpu())

    def make(n):
        return [mpe.Mpe([100], 4, 8, 0.1, 2, mpe.LRU, seed=9) for _ in range(n)]

    first = make(70)
    for h in first[::7] + first[-2:]:
        use(h)
    for h in first[1::2]:
        h.close()
    second = make(40)
    for h in second[::9]:
        use(h)
    for h in first[::2] + second:
        h.close()
    for h in make(2):
        use(h)
        h.close()
    assert all(torch.equal(outs[0], o) for o in outs)

"""GPU parity of the online n-gram cache (insertion of unseen n-grams, LRU / LFU trim,
access stamping by od_map_proposals) against the dictionary oracle: table contents,
access clocks and frequencies are integers and must match exactly."""
import numpy as np
import pytest
import torch

from oracle import cache_policy as cp
from paper_2507_02659_b200 import binding as od

pytestmark = pytest.mark.gpu


def _universe(rng, n, v_q):
    lens = rng.integers(2, 5, size=n).astype(np.int32)
    runs = rng.integers(0, v_q, size=(n, 4)).astype(np.int32)
    return runs, lens


def _compare(ctx, ref):
    got = ctx.cache_dump()
    want = {k: (v[0], v[1], v[2]) for k, v in ref.entries.items()}
    assert len(got) == len(want)
    assert got == want


@pytest.mark.parametrize("policy", [cp.LRU, cp.LFU])
def test_insert_access_trim_match_the_oracle(cuda_device, policy):
    rng = np.random.default_rng(20 + policy)
    v_q, v_p, B, K = 60, 300, 16, 6
    vocab_map = np.where(rng.random(v_q) < 0.7, rng.permutation(v_p)[:v_q], -1).astype(np.int32)
    ctx = od.Context(cuda_device, v_q, v_p, B, K)
    ctx.set_vocab_map(vocab_map)
    ctx.cache_configure(40, policy, 64)
    ref = cp.DynamicCache(40, policy, v_q, v_p)
    uruns, ulens = _universe(rng, 120, v_q)
    utgt = rng.integers(0, v_p, size=120).astype(np.int32)
    dev = cuda_device
    for tick in range(1, 25):
        ctx.cache_set_clock(tick); ref.set_clock(tick)
        # a batch of proposals, most of them carrying a run of the universe
        d = rng.integers(0, v_q, size=(B, K)).astype(np.int32)
        klen = rng.integers(0, K + 1, size=B).astype(np.int32)
        for b in range(B):
            e = int(rng.integers(0, 120)); L = int(ulens[e])
            if L <= klen[b] and rng.random() < 0.8:
                o = int(rng.integers(0, klen[b] - L + 1)); d[b, o:o + L] = uruns[e, :L]
        q = rng.random((B, K)).astype(np.float32)
        mp = od.od_map_proposals(ctx, torch.from_numpy(d).to(dev), torch.from_numpy(klen).to(dev),
                                 torch.from_numpy(q).to(dev))
        torch.cuda.synchronize()
        for b in range(B):
            tgt, qp, ss, sl, m, stop = ref.map_sequence(vocab_map, d[b, :klen[b]], q[b])
            assert int(mp.m[b]) == m and bool(mp.tail_kind[b]) == stop
            assert mp.tgt_ids[b, :m].tolist() == tgt and mp.span_len[b, :m].tolist() == sl
            np.testing.assert_allclose(mp.q_prime[b, :m].cpu().numpy(), qp, rtol=1e-6)
        _compare(ctx, ref)
        # what "reverse translation" found this step: duplicates inside the batch (the
        # first wins), runs already cached, malformed candidates
        n = 20
        pick = rng.integers(0, 120, size=n)
        runs, lens, tg = uruns[pick].copy(), ulens[pick].copy(), utgt[pick].copy()
        tg[n // 2:] = rng.integers(0, v_p, size=n - n // 2)       # same run, another target: must lose
        lens[3] = 5; runs[5, 0] = v_q + 1; tg[7] = v_p              # malformed
        ctx.cache_insert(torch.from_numpy(runs).to(dev), torch.from_numpy(lens).to(dev),
                         torch.from_numpy(tg).to(dev))
        ref.insert_batch(runs, lens, tg)
        _compare(ctx, ref)
        if tick % 2 == 0:
            ctx.cache_trim(); ref.trim()
            assert len(ref) <= 40
            _compare(ctx, ref)
    ctx.close()


@pytest.mark.parametrize("policy", [cp.LRU, cp.LFU])
def test_large_batches_and_many_ties(cuda_device, policy):
    """Thousands of candidates per batch, most scores tied: the radix select has to
    resolve the order down to the run keys."""
    rng = np.random.default_rng(30 + policy)
    v_q, v_p = 32000, 128256
    ctx = od.Context(cuda_device, v_q, v_p, 4, 4)
    ctx.set_vocab_map(np.full(v_q, -1, np.int32))
    ctx.cache_configure(5000, policy, 4096)
    ref = cp.DynamicCache(5000, policy, v_q, v_p)
    uruns, ulens = _universe(rng, 20000, v_q)
    utgt = rng.integers(0, v_p, size=20000).astype(np.int32)
    dev = cuda_device
    evicted = 0
    for tick in range(1, 9):
        ctx.cache_set_clock(tick); ref.set_clock(tick)
        pick = np.where(rng.random(4096) < 0.5, (rng.zipf(1.3, size=4096) - 1) % 20000,
                        rng.integers(0, 20000, size=4096))
        runs, lens, tg = uruns[pick].copy(), ulens[pick].copy(), utgt[pick].copy()
        ctx.cache_insert(torch.from_numpy(runs).to(dev), torch.from_numpy(lens).to(dev),
                         torch.from_numpy(tg).to(dev))
        ref.insert_batch(runs, lens, tg)
        if tick % 3 == 0 or tick == 8:
            ctx.cache_trim(); evicted += ref.trim()
        _compare(ctx, ref)
    assert len(ref) == 5000 and evicted > 1000
    ctx.close()


def test_full_size_cache_fills_and_trims_to_its_bound(cuda_device):
    """262144 entries (the largest cache of the workloads): 20 batches of 16384 fresh
    candidates overfill it, the trim brings it back to exactly the bound."""
    rng = np.random.default_rng(40)
    v_q, v_p, cap = 32000, 128256, 262144
    ctx = od.Context(cuda_device, v_q, v_p, 4, 4)
    ctx.set_vocab_map(np.full(v_q, -1, np.int32))
    ctx.cache_configure(cap, cp.LRU, 16384)
    ref = cp.DynamicCache(cap, cp.LRU, v_q, v_p)
    dev = cuda_device
    for tick in range(1, 21):
        ctx.cache_set_clock(tick); ref.set_clock(tick)
        lens = rng.integers(2, 5, size=16384).astype(np.int32)
        runs = rng.integers(0, v_q, size=(16384, 4)).astype(np.int32)
        tg = rng.integers(0, v_p, size=16384).astype(np.int32)
        ctx.cache_insert(torch.from_numpy(runs).to(dev), torch.from_numpy(lens).to(dev),
                         torch.from_numpy(tg).to(dev))
        ref.insert_batch(runs, lens, tg)
    assert len(ref) > cap
    ctx.cache_trim(); ref.trim()
    assert len(ref) == cap
    _compare(ctx, ref)
    ctx.close()


# a table of a few entries (blocks of the select without any), ties that overflow the select's shared
# memory because the trim comes late, ties that fill it, and a table too large for one cluster
@pytest.mark.parametrize("bound, batch, batches", [(5, 8, 2), (1000, 512, 5), (20000, 8000, 2), (400000, 65536, 8)])
@pytest.mark.parametrize("policy", [cp.LRU, cp.LFU])
def test_trim_over_ties(cuda_device, policy, bound, batch, batches):
    """All scores equal but for the last batch's: the run keys decide."""
    rng = np.random.default_rng(50)
    v_q, v_p, dev = 32000, 128256, cuda_device
    ctx = od.Context(cuda_device, v_q, v_p, 4, 4)
    ctx.set_vocab_map(np.full(v_q, -1, np.int32))
    ctx.cache_configure(bound, policy, batch)
    ref = cp.DynamicCache(bound, policy, v_q, v_p)
    for turn in range(2):
        for i in range(batches):
            clock = 10 * turn + (2 if i == batches - 1 else 1)
            ctx.cache_set_clock(clock); ref.set_clock(clock)
            runs, lens = _universe(rng, batch, v_q)
            tg = rng.integers(0, v_p, size=batch).astype(np.int32)
            ctx.cache_insert(torch.from_numpy(runs).to(dev), torch.from_numpy(lens).to(dev), torch.from_numpy(tg).to(dev))
            ref.insert_batch(runs, lens, tg)
        ctx.cache_trim(); ref.trim()
        assert len(ref) <= bound and ctx.cache_stats()[0] == len(ref)
        _compare(ctx, ref)
        if bound == 400000:
            break
    ctx.cache_trim()                                        # nothing to drop
    _compare(ctx, ref)
    ctx.close()


# scores whose varying bits lie apart (more than two runs of them, more than eight bits) and whole-word clocks; runs
# of one length, of leading ids from 0 to the last, and the bound inside and at the ends of a group of equal scores
@pytest.mark.parametrize("clocks", [(1, 2, 3), (0x80000001, 0x7FFFFFFF, 5), (1, 0x4000, 0x10002, 0x1010101, 0xFFFFFFF0)])
@pytest.mark.parametrize("length", [2, 3, 4, 0])
@pytest.mark.parametrize("bound", [1, 299, 300, 301, 555])
def test_trim_over_scores_with_bits_apart(cuda_device, clocks, length, bound):
    rng = np.random.default_rng(70 + length)
    v_q, v_p, dev = 65535, 1000, cuda_device
    ctx = od.Context(cuda_device, v_q, v_p, 4, 4)
    ctx.set_vocab_map(np.full(v_q, -1, np.int32))
    ctx.cache_configure(bound, cp.LRU, 300)
    ref = cp.DynamicCache(bound, cp.LRU, v_q, v_p)
    for clock in clocks:
        ctx.cache_set_clock(clock); ref.set_clock(clock)
        n = min(300, bound)
        lens = np.full(n, length, np.int32) if length else rng.integers(2, 5, size=n).astype(np.int32)
        runs = rng.choice([0, 1, 1022, 1023, 1024, 32767, 65534, 7, 511, 512], size=(n, 4)).astype(np.int32)
        runs[:, 1] = rng.integers(0, v_q, size=n)
        tg = rng.integers(0, v_p, size=n).astype(np.int32)
        for _ in range(2 if bound < 300 else 1):
            ctx.cache_insert(torch.from_numpy(runs).to(dev), torch.from_numpy(lens).to(dev), torch.from_numpy(tg).to(dev))
            ref.insert_batch(runs, lens, tg)
        if clock == clocks[-1] or bound < 400:
            ctx.cache_trim(); ref.trim()
            assert len(ref) <= bound
            _compare(ctx, ref)
    ctx.close()


# the select in one launch, and the chain of launches for a table too large for it
@pytest.mark.parametrize("bound", [100, 400000])
@pytest.mark.parametrize("trims", [1, 2])
def test_a_trim_replayed_from_a_graph(cuda_device, bound, trims):
    """A captured trim leaves nothing behind that its next replay adds to: the same entries every
    time. (One trim per graph reads the same table at every replay; two end on the one they began with.)"""
    rng = np.random.default_rng(60)
    v_q, v_p, dev = 32000, 128256, cuda_device
    ctx = od.Context(dev, v_q, v_p, 4, 4)
    ctx.set_vocab_map(np.full(v_q, -1, np.int32))
    ctx.cache_configure(bound, cp.LRU, 64)
    ctx.cache_set_clock(1)
    runs, lens = _universe(rng, 50, v_q)
    insert = lambda: ctx.cache_insert(*(torch.from_numpy(a).to(dev) for a in (runs, lens, np.arange(50, dtype=np.int32))))
    insert()
    ctx.cache_trim()
    want = ctx.cache_dump()
    assert len(want) == 50
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        for _ in range(trims):
            ctx.cache_trim()
    for _ in range(8):
        graph.replay()
        assert ctx.cache_dump() == want
    insert()                                                # the same runs: nothing new
    ctx.cache_trim()
    assert ctx.cache_dump() == want and ctx.cache_stats()[0] == 50
    ctx.close()


def test_online_cache_argument_checks(cuda_device):
    ctx = od.Context(cuda_device, 100, 100, 4, 4)
    with pytest.raises(od.OdError) as e:
        ctx.cache_trim()                                  # no online cache yet
    assert e.value.status == -8
    with pytest.raises(od.OdError):
        ctx.cache_configure(10, 2, 8)                     # unknown policy
    ctx.cache_configure(10, cp.LFU, 8)
    z = torch.zeros(9, 4, dtype=torch.int32, device=cuda_device)
    with pytest.raises(od.OdError):                       # batch beyond max_insert
        ctx.cache_insert(z, torch.zeros(9, dtype=torch.int32, device=cuda_device),
                         torch.zeros(9, dtype=torch.int32, device=cuda_device))
    big = od.Context(cuda_device, 70000, 70000, 1, 2)
    with pytest.raises(od.OdError) as e:
        big.cache_configure(10, 0, 8)                     # ids do not fit 16 bits
    assert e.value.status == -5
    big.close(); ctx.close()


def test_translation_directly_behind_cache_writers_with_early_inputs(cuda_device):
    """With "early_inputs" the translation kernel reads the proposal before it waits for the launch
    in front of it, never the table. Nothing is synchronised between an insertion or a trim and
    the translations behind it: they must see the table those leave."""
    rng = np.random.default_rng(77)
    v_q, v_p, B, K = 60, 300, 32, 6
    vocab_map = np.where(rng.random(v_q) < 0.7, rng.permutation(v_p)[:v_q], -1).astype(np.int32)
    ctx = od.Context(cuda_device, v_q, v_p, B, K)
    ctx.set_vocab_map(vocab_map)
    ctx.cache_configure(40, cp.LRU, 64)
    ctx.set_option("early_inputs", 1)
    ref = cp.DynamicCache(40, cp.LRU, v_q, v_p)
    uruns, ulens = _universe(rng, 120, v_q)
    utgt = rng.integers(0, v_p, size=120).astype(np.int32)
    dev = cuda_device
    for tick in range(1, 13):
        ctx.cache_set_clock(tick); ref.set_clock(tick)
        props = []
        for _ in range(3):
            d = rng.integers(0, v_q, size=(B, K)).astype(np.int32)
            klen = rng.integers(0, K + 1, size=B).astype(np.int32)
            for b in range(B):
                e = int(rng.integers(0, 120)); L = int(ulens[e])
                if L <= klen[b] and rng.random() < 0.9:
                    o = int(rng.integers(0, klen[b] - L + 1)); d[b, o:o + L] = uruns[e, :L]
            q = rng.random((B, K)).astype(np.float32)
            props.append((d, klen, q, torch.from_numpy(d).to(dev), torch.from_numpy(klen).to(dev),
                          torch.from_numpy(q).to(dev)))
        pick = rng.integers(0, 120, size=30)
        runs, lens, tg = uruns[pick].copy(), ulens[pick].copy(), utgt[pick].copy()
        d_runs, d_lens, d_tg = (torch.from_numpy(x).to(dev) for x in (runs, lens, tg))
        torch.cuda.synchronize()                              # every input is resident from here on
        ctx.cache_insert(d_runs, d_lens, d_tg)
        mp0 = od.od_map_proposals(ctx, *props[0][3:])        # directly behind the insertion
        mp1 = od.od_map_proposals(ctx, *props[1][3:])        # behind another translation
        ctx.cache_trim()
        mp2 = od.od_map_proposals(ctx, *props[2][3:])        # directly behind the trim
        torch.cuda.synchronize()
        ref.insert_batch(runs, lens, tg)
        for i, mp in enumerate((mp0, mp1, mp2)):
            if i == 2:
                ref.trim()
            d, klen, q = props[i][:3]
            for b in range(B):
                tgt, qp, ss, sl, m, stop = ref.map_sequence(vocab_map, d[b, :klen[b]], q[b])
                assert int(mp.m[b]) == m and bool(mp.tail_kind[b]) == stop, (tick, i, b)
                assert mp.tgt_ids[b, :m].tolist() == tgt and mp.span_len[b, :m].tolist() == sl
        _compare(ctx, ref)
    ctx.close()


@pytest.mark.parametrize("B,grid", [(2, 0), (2, 100), (20, 0)])
def test_steps_directly_behind_cache_writers_with_early_inputs(cuda_device, B, grid):
    """The same for od_step: in one launch, which reads all its inputs and the table before its wait unless a writer of the
    table may be at work, and in three."""
    rng = np.random.default_rng(78)
    v_q, v_p, K, dev = 60, 8000, 6, cuda_device
    vocab_map = np.where(rng.random(v_q) < 0.7, rng.permutation(v_p)[:v_q], -1).astype(np.int32)
    ctx = od.Context(dev, v_q, v_p, B, K)
    ctx.set_vocab_map(vocab_map)
    ctx.cache_configure(40, cp.LRU, 64)
    ctx.set_option("early_inputs", 1)
    ctx.set_option("verify_grid", grid)
    ref = cp.DynamicCache(40, cp.LRU, v_q, v_p)
    uruns, ulens = _universe(rng, 120, v_q)
    utgt = rng.integers(0, v_p, size=120).astype(np.int32)
    g = torch.Generator(device=dev).manual_seed(3)
    logits = torch.randn(B, K + 1, v_p, generator=g, device=dev).bfloat16()
    q_rows = torch.softmax(torch.randn(B, K, v_q, generator=g, device=dev), -1)
    T, seed = torch.ones(B, device=dev), torch.arange(B, device=dev)
    for tick in range(1, 13):
        ctx.cache_set_clock(tick); ref.set_clock(tick)
        props = []
        for _ in range(4):
            d = rng.integers(0, v_q, size=(B, K)).astype(np.int32)
            klen = rng.integers(0, K + 1, size=B).astype(np.int32)
            for b in range(B):
                e = int(rng.integers(0, 120)); L = int(ulens[e])
                if L <= klen[b] and rng.random() < 0.9:
                    o = int(rng.integers(0, klen[b] - L + 1)); d[b, o:o + L] = uruns[e, :L]
            q = rng.random((B, K)).astype(np.float32)
            props.append((d, klen, q, torch.from_numpy(d).to(dev), torch.from_numpy(klen).to(dev), torch.from_numpy(q).to(dev)))
        pick = rng.integers(0, 120, size=30)
        runs, lens, tg = uruns[pick].copy(), ulens[pick].copy(), utgt[pick].copy()
        d_runs, d_lens, d_tg = (torch.from_numpy(x).to(dev) for x in (runs, lens, tg))
        torch.cuda.synchronize()                              # every input is resident from here on
        step = lambda i: od.od_step(ctx, *props[i][3:], q_rows, logits, T, seed, tick)[0]
        ctx.cache_insert(d_runs, d_lens, d_tg)
        got = [step(0), step(1)]                              # directly behind the insertion, behind another step
        ctx.cache_trim()
        got += [step(2), step(3)]
        torch.cuda.synchronize()
        if B == 2:
            assert (ctx.last_launch_info(0) == ctx.last_launch_info(2)) == (grid == 0)
        ref.insert_batch(runs, lens, tg)
        for i, mp in enumerate(got):
            if i == 2:
                ref.trim()
            d, klen, q = props[i][:3]
            for b in range(B):
                tgt, qp, ss, sl, m, stop = ref.map_sequence(vocab_map, d[b, :klen[b]], q[b])
                assert int(mp.m[b]) == m and bool(mp.tail_kind[b]) == stop, (tick, i, b)
                assert mp.tgt_ids[b, :m].tolist() == tgt and mp.span_len[b, :m].tolist() == sl
        _compare(ctx, ref)
    ctx.close()


def test_a_full_table_counts_what_it_loses(cuda_device):
    """Insertions without a trim until the table (64 slots for a bound of 8 + 8) is full: every
    candidate is either in the cache or counted as lost, and malformed ones are counted too."""
    rng = np.random.default_rng(5)
    v_q, v_p = 200, 300
    ctx = od.Context(cuda_device, v_q, v_p, 4, 4)
    ctx.set_vocab_map(np.full(v_q, -1, np.int32))
    ctx.cache_configure(8, cp.LRU, 8)
    seen = set()
    bad = 0
    for tick in range(1, 16):
        ctx.cache_set_clock(tick)
        runs = np.full((8, 4), -1, np.int32); lens = np.full(8, 2, np.int32)
        for i in range(8):
            while True:
                r = tuple(int(x) for x in rng.integers(0, v_q, size=2))
                if r not in seen:
                    break
            seen.add(r); runs[i, :2] = r
        tg = rng.integers(0, v_p, size=8).astype(np.int32)
        if tick == 3:
            lens[0] = 7; seen.discard(tuple(int(x) for x in runs[0, :2])); bad += 1
        ctx.cache_insert(torch.from_numpy(runs).to(cuda_device), torch.from_numpy(lens).to(cuda_device),
                         torch.from_numpy(tg).to(cuda_device))
    entries, invalid, dropped = ctx.cache_stats()
    held = ctx.cache_dump()
    assert invalid == bad
    assert entries == len(held) == 64                 # every slot taken
    assert dropped == len(seen) - 64 and dropped > 0
    assert set(held) <= seen
    ctx.close()



@pytest.mark.parametrize("policy", [cp.LRU, cp.LFU])
@pytest.mark.parametrize("bound, batch", [(100, 28), (8, 24), (2000, 48), (60000, 30000)])
def test_trim_of_a_table_filled_to_the_brim(cuda_device, policy, bound, batch):
    """Insertions without a trim until almost every slot is taken: entries stand in groups that their run does not hash
    to, and groups beyond their first sixteen slots; clocks far enough apart for bins of many scores."""
    rng = np.random.default_rng(90 + bound)
    v_q, v_p, dev = 60, 300, cuda_device
    cap = 64
    while cap < 2 * (bound + batch):
        cap *= 2
    ctx = od.Context(dev, v_q, v_p, 64, 4)
    ctx.set_vocab_map(np.full(v_q, -1, np.int32))
    ctx.cache_configure(bound, policy, batch)
    ref = cp.DynamicCache(bound, policy, v_q, v_p)
    clock = 1
    for turn in range(3):
        while len(ref) + batch <= cap * 31 // 32:
            clock += int(rng.choice([1, 3, 40, 200, 5000]))
            ctx.cache_set_clock(clock); ref.set_clock(clock)
            runs, lens = _universe(rng, batch, v_q)
            tg = rng.integers(0, v_p, size=batch).astype(np.int32)
            ctx.cache_insert(torch.from_numpy(runs).to(dev), torch.from_numpy(lens).to(dev), torch.from_numpy(tg).to(dev))
            ref.insert_batch(runs, lens, tg)
            # accesses: a few runs often, up to 150 times a batch
            d = np.zeros((64, 4), np.int32)
            klen = np.zeros(64, np.int32)
            for b in range(64):
                i = int(rng.integers(0, batch)) if b < 60 else 0
                klen[b] = lens[i]; d[b] = runs[i]
            for _ in range(int(rng.choice([1, 1, 30]))):
                od.od_map_proposals(ctx, torch.from_numpy(d).to(dev), torch.from_numpy(klen).to(dev), torch.rand(64, 4, device=dev))
                for b in range(64):
                    ref.map_sequence(np.full(v_q, -1, np.int32), d[b, :klen[b]], np.ones(4, np.float32))
        _compare(ctx, ref)
        ctx.cache_trim(); ref.trim()
        assert len(ref) == bound and ctx.cache_stats() == (bound, 0, 0)
        _compare(ctx, ref)
    ctx.close()


# lists of one clock's entries from more than a cluster of the select holds down to none, over every number of its blocks
@pytest.mark.parametrize("policy", [cp.LRU, cp.LFU])
@pytest.mark.parametrize("bound, batch, tick", [(500, 90, 1), (3000, 170, 1), (3000, 170, 1000), (20000, 1100, 1)])
def test_trims_while_the_entries_of_one_clock_run_out(cuda_device, policy, bound, batch, tick):
    rng = np.random.default_rng(70)
    v_q, v_p, dev = 32000, 128256, cuda_device
    ctx = od.Context(cuda_device, v_q, v_p, 4, 4)
    ctx.set_vocab_map(np.full(v_q, -1, np.int32))
    ctx.cache_configure(bound, policy, batch)
    ref = cp.DynamicCache(bound, policy, v_q, v_p)
    clock = 5
    while True:
        ctx.cache_set_clock(clock); ref.set_clock(clock)
        runs, lens = _universe(rng, batch, v_q)
        tg = rng.integers(0, v_p, size=batch).astype(np.int32)
        ctx.cache_insert(torch.from_numpy(runs).to(dev), torch.from_numpy(lens).to(dev), torch.from_numpy(tg).to(dev))
        ref.insert_batch(runs, lens, tg)
        if clock == 5 and len(ref) < bound:
            continue                                        # the first clock's entries, without a trim between
        ctx.cache_trim(); ref.trim()
        _compare(ctx, ref)
        assert ctx.cache_stats()[0] == len(ref)
        if clock > 5 + tick * (bound // batch + 2):
            break
        clock += tick
    ctx.close()


def _clocks(kind, n):
    if kind == "steps of 1000":
        return [4000 + 1000 * i for i in range(n)]
    if kind == "any":
        return list(np.cumsum(np.random.default_rng(3).choice([1, 2, 130, 5000, 70000000], size=n)))
    if kind == "set back":                                  # and on from there, and behind the end of 32 bits
        return [100000 + 10 * i for i in range(n // 3)] + [50 + i for i in range(n // 3)] + [0xFFFFFFF0 + i for i in range(15)]
    return [7 + i // 4 for i in range(n)]                   # four insertions to a tick


# the bins by clock begin where the last trim left off, which says nothing about entries that the caller dates back
@pytest.mark.parametrize("kind, bound, batch", [(kind, *size) for kind in ("steps of 1000", "any", "set back", "four a tick")
                                                for size in ((200, 30), (2048, 256), (5000, 900))] + [("steps of 1000", 400000, 50000)])
def test_trims_by_clocks_of_any_step(cuda_device, kind, bound, batch):
    rng = np.random.default_rng(77)
    v_q, v_p, dev = 3000, 30000, cuda_device
    ctx = od.Context(cuda_device, v_q, v_p, 64, 4)
    ctx.set_vocab_map(np.full(v_q, -1, np.int32))
    ctx.cache_configure(bound, cp.LRU, batch)
    ref = cp.DynamicCache(bound, cp.LRU, v_q, v_p)
    for clock in _clocks(kind, bound // batch + (4 if bound > 100000 else 30)):
        ctx.cache_set_clock(int(clock)); ref.set_clock(int(clock))
        runs, lens = _universe(rng, batch, v_q)
        tg = rng.integers(0, v_p, size=batch).astype(np.int32)
        ctx.cache_insert(torch.from_numpy(runs).to(dev), torch.from_numpy(lens).to(dev), torch.from_numpy(tg).to(dev))
        ref.insert_batch(runs, lens, tg)
        # some of the entries are accessed
        held = list(ref.entries)
        picked = [held[i] for i in rng.integers(0, len(held), size=64)]
        d, klen = np.zeros((64, 4), np.int32), np.zeros(64, np.int32)
        for b, run in enumerate(picked):
            klen[b] = len(run); d[b, :len(run)] = run
        od.od_map_proposals(ctx, torch.from_numpy(d).to(dev), torch.from_numpy(klen).to(dev), torch.ones(64, 4, device=dev))
        for b in range(64):
            ref.map_sequence(np.full(v_q, -1, np.int32), d[b, :klen[b]], np.ones(4, np.float32))
        ctx.cache_trim(); ref.trim()
        assert ctx.cache_stats()[0] == len(ref)
    _compare(ctx, ref)
    ctx.close()

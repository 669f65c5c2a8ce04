"""Calls whose inputs are written by a launch that is still at work when the library's kernels become resident: a producer
that releases its dependents first and writes half a millisecond later (tests/helpers/early_producer.cu)."""
import ctypes as C

import numpy as np
import pytest
import torch

import helpers
from paper_2507_02659_b200 import binding as od
from paper_2507_02659_b200 import synth, vshard

import parity

pytestmark = pytest.mark.gpu
LATE = 1000000                                              # cycles from the producer's release to its stores


def _workload(**kw):
    base = dict(B=48, steps=4, k_max=4, k_min=2, v_q=3000, v_p=40000, logit_dtype="bf16", map_kind="random", mapped_frac=0.7,
                cache_entries=400, hit_prob=0.95, logit_kind="zipf", targets_on_prefix=0.4, plant_boost=8.0, rho=0.95,
                temperatures=(1.0, 0.5, 0.7), per_seq_seed=True, gen_seed=0xBEEFA1, unmapped_shift=2.0, sigma=2.0)
    base.update(kw)
    return synth.Workload("order", **base)


def _produce(dst, src):
    """Writes src over dst, late, as the launch directly in front of the next one."""
    n = src.numel() * src.element_size()
    assert n % 16 == 0 and dst.is_contiguous() and src.is_contiguous()
    stream = torch.cuda.current_stream(src.device).cuda_stream
    assert helpers.early_producer_lib().early_producer(dst.data_ptr(), src.data_ptr(), n, LATE, stream) == 0


@pytest.mark.parametrize("shards", [0, 2])
def test_the_drafters_rows_may_be_written_directly_in_front_of_the_draw(cuda_device, shards):
    """The draw is the first call that reads them; at a cached run it reads the probability of the run's first token first."""
    w = _workload()
    st = synth.make_static(w)
    ctx = parity.make_context(w, st, cuda_device)
    s = synth.make_step(w, st, 0, device=cuda_device)
    mp = od.od_map_proposals(ctx, s.draft_ids, s.draft_len, s.q_sel)
    vo = od.od_verify(ctx, s.logits, mp, s.temperature, s.seed, s.step)
    bounds = [vshard.split_vocab(w.v_p, r, shards) for r in range(shards)]
    late = torch.full_like(s.q_rows, float("nan"))

    def draw(q_rows):
        if not shards:
            so = od.od_sample_residual(ctx, s.logits, vo, q_rows, s.draft_ids, mp, s.temperature, s.seed, s.step)
            return [so.out_token, so.resid_mass, so.flags]
        return [od.od_sample_shard_mass(ctx, lo, s.logits[:, :, lo:hi], vo, q_rows, s.draft_ids, mp, s.temperature) for lo, hi in bounds]
    want = draw(s.q_rows)
    torch.cuda.synchronize()
    j = vo.n_accepted.long()
    merged = (j < mp.m) & (torch.gather(mp.span_len, 1, j[:, None].clamp(max=w.k_max - 1))[:, 0] >= 2)
    assert int(merged.sum()) >= 10                          # draws that need that probability
    for _ in range(4):
        late.fill_(float("nan"))
        torch.cuda.synchronize()
        od.od_verify(ctx, s.logits, mp, s.temperature, s.seed, s.step, out=vo)      # (behind it a draw reads ahead)
        _produce(late, s.q_rows)
        got = draw(late)
        torch.cuda.synchronize()
        for a, b in zip(want, got):
            assert torch.equal(a, b)
    ctx.close()


def test_the_seeds_may_be_written_directly_in_front_of_the_shards_decisions(cuda_device):
    """od_verify_shard_finish is the first call of a sharded step that reads them."""
    w = _workload(B=24)
    st = synth.make_static(w)
    ctx = parity.make_context(w, st, cuda_device)
    s = synth.make_step(w, st, 0, device=cuda_device)
    mp = od.od_map_proposals(ctx, s.draft_ids, s.draft_len, s.q_sel)
    stats = od.od_verify_shard_stats(ctx, 0, s.logits, mp, s.temperature)[None]
    # acceptances that the uniforms decide: a ratio of a half everywhere
    mp.q_prime.copy_(2 * od.od_verify(ctx, s.logits, mp, s.temperature, s.seed, s.step).p_sel)
    finish = lambda seed: od.od_verify_shard_finish(ctx, stats, mp, s.temperature, seed, s.step)
    want, other = finish(s.seed), finish(s.seed + 1)
    torch.cuda.synchronize()
    assert not torch.equal(want.flags, other.flags) or not torch.equal(want.n_accepted, other.n_accepted)
    late = torch.empty_like(s.seed)
    for _ in range(4):
        late.copy_(s.seed + 1)
        torch.cuda.synchronize()
        _produce(late, s.seed)
        got = finish(late)
        torch.cuda.synchronize()
        assert torch.equal(got.n_accepted, want.n_accepted) and torch.equal(got.flags, want.flags)
    ctx.close()


@pytest.mark.parametrize("late", ["logits", "draft_ids", "q_rows"])
@pytest.mark.parametrize("between", [1, 3])
def test_inputs_written_two_launches_back_are_complete(cuda_device, late, between):
    """Under early_inputs a step reads its inputs while the launch in front of it runs: that launch must not have let it
    start before the producer in front of itself was done."""
    w = _workload(B=2, k_max=3)
    st = synth.make_static(w)
    ctx = parity.make_context(w, st, cuda_device)
    first, s = (synth.make_step(w, st, i, device=cuda_device) for i in range(2))

    def step(x, **kw):
        return od.od_step(ctx, *(kw.get(n, getattr(x, n)) for n in ("draft_ids", "draft_len", "q_sel", "q_rows", "logits", "temperature", "seed")), x.step)
    flat = lambda out: [t.clone() for o, names in zip(out, (("m", "tail_kind"), ("n_accepted", "n_draft_accepted", "flags"), ("out_token", "resid_mass", "flags")))
                        for t in (getattr(o, n) for n in names)]
    src = getattr(s, late)
    n = src.numel() + -src.numel() % 8                      # (whole 16-byte pieces)
    padded, dst = torch.zeros(n, dtype=src.dtype, device=cuda_device), torch.zeros(n, dtype=src.dtype, device=cuda_device)
    padded[:src.numel()] = src.flatten()
    view = dst[:src.numel()].view(src.shape)
    want = flat(step(s))
    ctx.set_option("early_inputs", 1)
    for _ in range(4):
        dst.fill_(1 if late == "draft_ids" else float("nan"))
        torch.cuda.synchronize()
        _produce(dst, padded)
        for _ in range(between):
            step(first)
        got = flat(step(s, **{late: view}))
        torch.cuda.synchronize()
        for a, b in zip(want, got):
            assert torch.equal(a, b)
    ctx.close()


@pytest.mark.parametrize("call", ["map", "verify", "noalloc", "sample", "stats", "finish", "mass", "pick", "distill", "exit", "insert", "trim"])
def test_no_call_lets_the_next_one_start_before_its_own_wait(cuda_device, call):
    """The same with each other call in between: a translation behind it reads its proposal early."""
    w = _workload(B=2, k_max=3)
    st = synth.make_static(w)
    ctx = parity.make_context(w, st, cuda_device)
    ctx.cache_configure(1000, 0, len(st.runs))              # nothing is evicted
    dev = lambda x: torch.as_tensor(np.ascontiguousarray(x), dtype=torch.int32, device=cuda_device)
    cached = [dev(x) for x in (st.runs, st.run_len, st.run_target)]
    ctx.cache_set_clock(1)
    ctx.cache_insert(*cached)
    a, s = (synth.make_step(w, st, i, device=cuda_device) for i in range(2))
    mp = od.od_map_proposals(ctx, a.draft_ids, a.draft_len, a.q_sel)
    vo = od.od_verify(ctx, a.logits, mp, a.temperature, a.seed, 0)
    shard = (0, a.logits)
    stats = od.od_verify_shard_stats(ctx, *shard, mp, a.temperature)[None]
    mass = od.od_sample_shard_mass(ctx, *shard, vo, a.q_rows, a.draft_ids, mp, a.temperature)[None]
    vo2 = od.alloc_verify_out(ctx, w.B, w.k_max)
    head = torch.zeros(w.B, w.k_max, device=cuda_device)
    calls = {
        "map": lambda: od.od_map_proposals(ctx, a.draft_ids, a.draft_len, a.q_sel),
        "verify": lambda: od.od_verify(ctx, a.logits, mp, a.temperature, a.seed, 0, out=vo2),
        "noalloc": lambda: od.od_verify_noalloc(w.v_p, a.logits, mp, a.temperature, a.seed, 0, vo2),
        "sample": lambda: od.od_sample_residual(ctx, a.logits, vo, a.q_rows, a.draft_ids, mp, a.temperature, a.seed, 0),
        "stats": lambda: od.od_verify_shard_stats(ctx, *shard, mp, a.temperature),
        "finish": lambda: od.od_verify_shard_finish(ctx, stats, mp, a.temperature, a.seed, 0),
        "mass": lambda: od.od_sample_shard_mass(ctx, *shard, vo, a.q_rows, a.draft_ids, mp, a.temperature),
        "pick": lambda: od.od_sample_shard_pick(ctx, 0, 0, mass, a.logits, vo, a.q_rows, a.draft_ids, mp, a.temperature, a.seed, 0),
        "distill": lambda: od.od_distill_loss(ctx, a.q_rows, a.draft_ids, mp, a.logits, vo, a.temperature, 0.2, 0),
        "exit": lambda: od.od_exit_rule(ctx, head, None, 0.5),
        "insert": lambda: ctx.cache_insert(*cached),
        "trim": lambda: ctx.cache_trim(),
    }
    want = od.od_map_proposals(ctx, s.draft_ids, s.draft_len, s.q_sel)
    source = torch.zeros(s.draft_ids.numel() + -s.draft_ids.numel() % 4, dtype=torch.int32, device=cuda_device)
    late = torch.zeros_like(source)
    source[:s.draft_ids.numel()] = s.draft_ids.flatten()
    ctx.set_option("early_inputs", 1)
    for _ in range(3):
        late.fill_(1)
        torch.cuda.synchronize()
        _produce(late, source)
        calls[call]()
        got = od.od_map_proposals(ctx, late[:s.draft_ids.numel()].view(s.draft_ids.shape), s.draft_len, s.q_sel)
        torch.cuda.synchronize()
        assert torch.equal(got.m, want.m) and torch.equal(got.tail_kind, want.tail_kind)
        for b, m in enumerate(want.m.tolist()):
            assert torch.equal(got.tgt_ids[b, :m], want.tgt_ids[b, :m]) and torch.equal(got.span_len[b, :m], want.span_len[b, :m])
    ctx.close()


def test_the_driver_says_which_host_buffers_the_device_can_read(cuda_device):
    """od_step_host fetches rows from page-locked memory and copies from other; both give the same results, so this asks
    the rule itself, with the driver's answers: all of a range, and one byte more than is left of it."""
    lib = C.CDLL(od.lib()._name)
    readable = lib._Z21od_host_rows_readablePKvmS0_mPPKcS3_
    readable.restype = C.c_bool
    pinned = torch.empty(1 << 20, dtype=torch.uint8, pin_memory=True)
    other = torch.empty(1 << 20, dtype=torch.uint8)
    on_device = torch.empty(1 << 20, dtype=torch.uint8, device=cuda_device)
    a, b = C.c_void_p(), C.c_void_p()

    def ask(t, at, n):
        return readable(C.c_void_p(t.data_ptr() + at), C.c_size_t(n), C.c_void_p(pinned.data_ptr()), C.c_size_t(16), C.byref(a), C.byref(b))
    assert ask(pinned, 0, 1 << 20) and a.value == pinned.data_ptr() and b.value == pinned.data_ptr()
    assert ask(pinned, 4096, (1 << 20) - 4096)
    assert not ask(pinned, 8, 64)                           # not 16-byte aligned
    assert not ask(pinned, 0, 1 << 40)                      # beyond any page-locked range
    assert not ask(other, 0, 64) and not ask(on_device, 0, 64)


# The tests of the order in three launches that are elsewhere take whichever path the chip's resident clusters give at
# their sizes; the same here with the streaming pass for certain.
@pytest.mark.parametrize("early", [0, 1])
def test_three_launches_equal_the_three_calls(cuda_device, early):
    w = _workload(B=40, v_p=30011, cache_entries=800)
    st = synth.make_static(w)
    ctx = parity.make_context(w, st, cuda_device)
    ctx.set_option("verify_grid", 148)
    s = synth.make_step(w, st, 3, device=cuda_device)
    lg = parity.pad_rows(s.logits)
    want = parity.gpu_step(ctx, s, logits=lg)
    ctx.set_option("early_inputs", early)
    torch.cuda.synchronize()
    runs = [od.od_step(ctx, s.draft_ids, s.draft_len, s.q_sel, s.q_rows, lg, s.temperature, s.seed, s.step) for _ in range(4)]
    torch.cuda.synchronize()
    rows = torch.arange(w.k_max + 1, device=cuda_device)[None, :] <= want[0].m[:, None]
    pos = rows[:, 1:]
    for got in runs:
        for o, names, where in ((0, ("tgt_ids", "q_prime"), pos), (1, ("row_max", "row_sum"), rows), (1, ("p_sel", "ratio"), pos),
                                (0, ("m", "tail_kind"), ...), (1, ("n_accepted", "n_draft_accepted", "flags"), ...),
                                (2, ("out_token", "resid_mass", "flags"), ...)):
            for n in names:
                assert torch.equal(getattr(got[o], n)[where], getattr(want[o], n)[where]), n
    ctx.close()


@pytest.mark.parametrize("grid", [0, 148])
@pytest.mark.parametrize("B", [2, 48])
@pytest.mark.parametrize("call", ["step", "verify"])
def test_logits_may_be_written_directly_in_front(cuda_device, grid, B, call):
    w = _workload(B=B)
    st = synth.make_static(w)
    ctx = parity.make_context(w, st, cuda_device)
    ctx.set_option("verify_grid", grid)
    s = synth.make_step(w, st, 0, device=cuda_device)
    mp = od.od_map_proposals(ctx, s.draft_ids, s.draft_len, s.q_sel)
    late = torch.empty_like(s.logits)

    def run(lg):
        if call == "verify":
            vo = od.od_verify(ctx, lg, mp, s.temperature, s.seed, s.step)
            return [vo.n_accepted, vo.flags]
        _, vo, so = od.od_step(ctx, s.draft_ids, s.draft_len, s.q_sel, s.q_rows, lg, s.temperature, s.seed, s.step)
        return [vo.n_accepted, vo.flags, so.out_token, so.resid_mass, so.flags]
    want = run(s.logits)
    for _ in range(4):
        late.fill_(float("nan"))
        torch.cuda.synchronize()
        _produce(late, s.logits)
        got = run(late)
        torch.cuda.synchronize()
        for a, b in zip(want, got):
            assert torch.equal(a, b)
    ctx.close()

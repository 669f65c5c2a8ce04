"""The whole step in one launch (small batches): every number of blocks per sequence, both sources of the
drafter's probabilities and the inverse map, against the oracle and against the same step in three launches; and
the page-locked form of the step on host buffers."""
import dataclasses

import numpy as np
import pytest
import torch

import oracle
from paper_2507_02659_b200 import binding as od
from paper_2507_02659_b200 import synth

import parity

pytestmark = pytest.mark.gpu


def _workload(**kw):
    base = dict(B=1, steps=4, k_max=4, k_min=1, v_q=3000, v_p=40000, logit_dtype="bf16", map_kind="random",
                mapped_frac=0.7, cache_entries=600, hit_prob=0.6, logit_kind="corr", rho=0.9,
                temperatures=(1.0, 0.5, 0.7), per_seq_seed=True, gen_seed=0x0E51A0, unmapped_shift=2.0, sigma=2.0)
    base.update(kw)
    return synth.Workload("onelaunch", **base)


def _step(ctx, s, logits):
    out = od.od_step(ctx, s.draft_ids, s.draft_len, s.q_sel, s.q_rows, logits, s.temperature, s.seed, s.step)
    torch.cuda.synchronize()
    return out


# batches at which the number of blocks changes; row ends inside a unit, a tile and a vector; a part without tiles
# (33 tiles in 16 parts of 3); the longest proposals; more mapped ids in a part than are staged
@pytest.mark.parametrize("kw", [dict(B=B) for B in (1, 7, 8, 15, 16, 22, 23, 30, 36, 40)] +
                         [dict(B=1, v_q=600, v_p=1003), dict(B=40, v_q=600, v_p=4096, logit_dtype="f32"), dict(B=120, v_q=64, v_p=300),
                          dict(B=3, v_p=8449, logit_dtype="f32"), dict(B=4, v_p=50001, k_max=16), dict(B=2, v_p=50003, k_max=16, logit_dtype="f32"),
                          dict(B=5, v_q=5003, v_p=5003, map_kind="identity", cache_entries=0),
                          dict(B=18, v_q=4096, v_p=4096, map_kind="identity", cache_entries=0, logit_dtype="f32"),
                          dict(B=1, v_q=60000, v_p=900_000, k_max=1, cache_entries=0)])
def test_one_launch_against_the_oracle_and_three_launches(cuda_device, kw):
    w = _workload(**kw)
    st = synth.make_static(w)
    if w.v_p >= 900_000:
        st.vocab_map = np.arange(w.v_q, dtype=np.int32) + 1
    ctx = parity.make_context(w, st, cuda_device)
    cache = oracle.Cache(st.runs, st.run_len, st.run_target)
    for step in range(2):
        s = synth.make_step(w, st, step, device=cuda_device)
        lg = parity.pad_rows(s.logits)
        mp, vo, so = _step(ctx, s, lg)
        if w.B <= 14 and w.v_p < 900_000:                                   # (how many larger clusters are resident differs from chip to chip)
            assert ctx.last_launch_info(0) == ctx.last_launch_info(2)      # one grid
        sel = sorted({0, w.B // 3, w.B // 2, w.B - 1})
        ref = parity.oracle_step(cache, st, w, dataclasses.replace(
            s.to("cpu"), **{k: getattr(s, k).cpu()[sel] for k in ("draft_ids", "draft_len", "q_sel", "q_rows", "logits", "temperature", "seed")}),
            probe=so.out_token.cpu().numpy()[sel])
        stats = parity.compare(mp, vo, so, ref, s.draft_len.cpu().numpy()[sel], step, s.seed.cpu().numpy().astype(np.uint64)[sel],
                               bf16=w.logit_dtype == "bf16", sel=np.asarray(sel))
        assert stats.sequences == len(sel)
        ctx.set_option("verify_grid", 100)                                  # three launches
        mp3, vo3, so3 = _step(ctx, s, lg)
        ctx.set_option("verify_grid", 0)
        for name in ("m", "tail_kind", "counters"):
            assert torch.equal(getattr(mp, name), getattr(mp3, name)), name
        pos = torch.arange(w.k_max, device=cuda_device)[None, :] < mp.m[:, None]
        for name in ("tgt_ids", "q_prime", "span_start", "span_len"):
            assert torch.equal(getattr(mp, name)[pos], getattr(mp3, name)[pos]), name
        rows = torch.arange(w.k_max + 1, device=cuda_device)[None, :] <= mp.m[:, None]
        assert torch.equal(vo.row_max[rows], vo3.row_max[rows])
        # two sums of up to 9e5 positive fp32 terms, each within 2e-5 / 2 of exact (the parity bound)
        torch.testing.assert_close(vo.row_sum[rows], vo3.row_sum[rows], rtol=2e-5, atol=0)
        settled = ((vo.flags | vo3.flags) == 0) & ((so.flags | so3.flags) & od.OD_SF_BOUNDARY == 0)
        assert torch.equal(vo.n_accepted[settled], vo3.n_accepted[settled])
        assert torch.equal(vo.n_draft_accepted[settled], vo3.n_draft_accepted[settled])
        assert torch.equal(so.out_token[settled], so3.out_token[settled])
    ctx.close()


def test_one_launch_with_nothing_to_translate_and_bad_temperatures(cuda_device):
    """Empty proposals, ids outside the vocabulary, a temperature of zero: flags and outputs as in three launches."""
    w = _workload(B=6, k_max=3)
    st = synth.make_static(w)
    ctx = parity.make_context(w, st, cuda_device)
    s = synth.make_step(w, st, 0, device=cuda_device)
    s.draft_len[:3] = torch.tensor([0, -5, 99], dtype=torch.int32)
    s.draft_ids[3, 0] = w.v_q + 7
    s.temperature[4] = 0.0
    lg = parity.pad_rows(s.logits)
    one = _step(ctx, s, lg)
    ctx.set_option("verify_grid", 100)
    three = _step(ctx, s, lg)
    for a, b in zip(one, three):
        for name in ("m", "tail_kind", "counters", "n_accepted", "n_draft_accepted", "flags", "out_token"):
            if hasattr(a, name):
                assert torch.equal(getattr(a, name), getattr(b, name)), name
    assert int(one[0].counters[od.OD_CNT_INVALID_IDS]) >= 1
    assert int(one[2].out_token[4]) == -1
    ctx.close()


def test_one_launch_stamps_the_online_cache_once(cuda_device):
    """Several blocks look a run up; its access counts once."""
    freq = []
    for grid in (0, 100):
        w = _workload(B=4, k_max=4, cache_entries=64, hit_prob=1.0)
        st = synth.make_static(w)
        ctx = parity.make_context(w, st, cuda_device)
        ctx.cache_configure(256, 1, 64)
        dev = lambda x: torch.as_tensor(np.ascontiguousarray(x), dtype=torch.int32, device=cuda_device)
        ctx.cache_set_clock(1)
        ctx.cache_insert(dev(st.runs), dev(st.run_len), dev(st.run_target))
        ctx.set_option("verify_grid", grid)
        for step in range(3):
            s = synth.make_step(w, st, step, device=cuda_device)
            ctx.cache_set_clock(2 + step)
            _step(ctx, s, parity.pad_rows(s.logits))
        freq.append(ctx.cache_dump())
        ctx.close()
    assert freq[0] == freq[1] and max(f for _, _, f in freq[0].values()) > 1


# page-locked buffers, which the device fetches itself (drafter rows of whole vectors, and not), parts of a larger
# page-locked block, a base off 16 bytes and pageable memory, which are copied
@pytest.mark.parametrize("v_q", [2000, 2001])
@pytest.mark.parametrize("where", ["pinned", "inside", "offset", "pageable"])
def test_host_buffers(cuda_device, v_q, where):
    w = _workload(B=9, v_q=v_q, v_p=30000, k_max=5)
    st = synth.make_static(w)
    ctx = parity.make_context(w, st, cuda_device)
    ctx.host_step_reserve(od.OD_BF16)
    for step in range(2):
        s = synth.make_step(w, st, step, device=cuda_device)
        mp, vo, so = parity.gpu_step(ctx, s)
        h = s.to("cpu")

        def put(t):
            if where == "pageable":
                return t.contiguous()
            pad = {"pinned": 0, "inside": 64, "offset": 2}[where] if t.dtype in (torch.bfloat16, torch.float32) else 0
            big = torch.empty(t.numel() + 2 * pad, dtype=t.dtype, pin_memory=True)
            return big[pad:pad + t.numel()].view(t.shape).copy_(t)
        out = od.od_step_host(ctx, put(h.draft_ids), put(h.draft_len), put(h.q_sel), put(h.q_rows), put(h.logits),
                              put(h.temperature), put(h.seed), s.step)
        for name, ref in (("n_accepted", vo.n_accepted), ("n_draft_accepted", vo.n_draft_accepted), ("out_token", so.out_token),
                          ("m", mp.m), ("verify_flags", vo.flags), ("sample_flags", so.flags)):
            assert torch.equal(getattr(out, name), ref.cpu()), name
    ctx.close()


def test_the_step_takes_every_number_of_blocks_per_sequence(cuda_device):
    """Which of the batches above were one launch, and of how many blocks, differs from chip to chip; all of them occur."""
    w = _workload(B=50, k_max=2)
    st = synth.make_static(w)
    ctx = parity.make_context(w, st, cuda_device)
    s = synth.make_step(w, st, 0, device=cuda_device)
    parts = set()
    for B in range(1, 51):
        cut = dataclasses.replace(s, **{k: getattr(s, k)[:B].contiguous() for k in ("draft_ids", "draft_len", "q_sel", "q_rows", "logits", "temperature", "seed")})
        _step(ctx, cut, parity.pad_rows(cut.logits))
        if ctx.last_launch_info(0) == ctx.last_launch_info(2):             # one grid
            parts.add(ctx.last_launch_info(0) // B)
    assert parts >= {16, 8, 6, 5, 4, 3}, parts
    ctx.close()


# Each of a sum's terms is within 2^-22, its partial sums within 2^-24 of themselves, errors of both signs: 600 sums of
# thousands of terms come to 1e-7 or less on average, and to a mean error that says what is on one side. 2^-25 is six times
# what the merge has and half of what it had with ex2.approx (-4.5e-8 to -5.6e-8).
@pytest.mark.parametrize("B,V,K", [(15, 50001, 4), (60, 8000, 4)])
@pytest.mark.parametrize("dtype", ["bf16", "f32"])
def test_row_sums_are_not_off_to_one_side(cuda_device, B, V, K, dtype):
    dev, dt, per = cuda_device, torch.bfloat16 if dtype == "bf16" else torch.float32, 8 if dtype == "bf16" else 4
    g = torch.Generator(device=dev).manual_seed(1)
    ctx = od.Context(dev, 1000, V, B, K)
    ctx.set_vocab_map(np.arange(1000, dtype=np.int32) + 1)
    T = torch.tensor([0.5, 0.7, 1.0], device=dev).repeat(B)[:B].contiguous()
    seed, ln = torch.arange(B, device=dev), torch.full((B,), K, dtype=torch.int32, device=dev)
    err = {"step": [], "verify": [], "shard": []}
    for step in range(600 // (B * (K + 1))):
        lg = torch.zeros(B, K + 1, -(-V // per) * per, dtype=dt, device=dev)[:, :, :V]
        lg.copy_(torch.randn(B, K + 1, V, generator=g, device=dev) * 3)
        ids = torch.randint(0, 1000, (B, K), generator=g, device=dev, dtype=torch.int32)
        q = torch.full((B, K, 1000), 1e-3, device=dev)
        x = lg.double()
        want = torch.exp((x - x.amax(-1, keepdim=True)) / T.double()[:, None, None]).sum(-1)
        mp, vo, _ = od.od_step(ctx, ids, ln, q[:, :, 0].contiguous(), q, lg, T, seed, step)
        assert ctx.last_launch_info(0) == ctx.last_launch_info(2)          # one grid
        err["step"].append(vo.row_sum / want - 1)
        err["verify"].append(od.od_verify(ctx, lg, mp, T, seed, step).row_sum / want - 1)
        stats = od.od_verify_shard_stats(ctx, 0, lg, mp, T)[None]
        err["shard"].append(od.od_verify_shard_finish(ctx, stats, mp, T, seed, step).row_sum / want - 1)
    for name, e in err.items():
        e = torch.cat(e)
        assert e.abs().max() <= 2.0 ** -20 and e.pow(2).mean().sqrt() <= 2.0 ** -23, name
        assert abs(float(e.mean())) <= 2.0 ** -25, name
    ctx.close()


@pytest.mark.parametrize("late", [False, True])
def test_a_draw_behind_a_step_in_one_launch_waits_for_its_outputs(cuda_device, late):
    """od_sample_residual on the outputs of the od_step directly in front, over garbage; `late`: that step itself waits
    half a millisecond for its logits."""
    import helpers
    w = _workload(B=4, v_p=40000)
    st = synth.make_static(w)
    ctx = parity.make_context(w, st, cuda_device)
    s = synth.make_step(w, st, 0, device=cuda_device)
    _, _, want = _step(ctx, s, s.logits)
    mp, vo, so = od.alloc_map_out(ctx, w.B, w.k_max), od.alloc_verify_out(ctx, w.B, w.k_max), od.alloc_sample_out(ctx, w.B)
    logits = s.logits.clone()
    stream = torch.cuda.current_stream(cuda_device).cuda_stream
    for _ in range(4):
        for t in (mp.tgt_ids, mp.span_start, mp.span_len, mp.m, vo.n_accepted):
            t.fill_(-1)
        vo.row_sum.fill_(float("nan"))
        if late:
            logits.fill_(float("nan"))
        torch.cuda.synchronize()
        if late:
            assert helpers.early_producer_lib().early_producer(logits.data_ptr(), s.logits.data_ptr(), logits.numel() * 2, 1000000, stream) == 0
        od.od_step(ctx, s.draft_ids, s.draft_len, s.q_sel, s.q_rows, logits, s.temperature, s.seed, s.step, mp=mp, vo=vo, so=so)
        assert ctx.last_launch_info(0) == ctx.last_launch_info(2)
        again = od.od_sample_residual(ctx, logits, vo, s.q_rows, s.draft_ids, mp, s.temperature, s.seed, s.step)
        torch.cuda.synchronize()
        for got in (so, again):
            assert torch.equal(got.out_token, want.out_token) and torch.equal(got.flags, want.flags)
            torch.testing.assert_close(got.resid_mass, want.resid_mass, rtol=2.0 ** -22, atol=0)   # (other cuts: fp64 sums, one rounding)
    ctx.close()

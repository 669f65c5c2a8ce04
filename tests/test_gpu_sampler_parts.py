"""The sampler's cuts of a row (1 to 16 blocks per sequence) and its sources of the drafter's
probabilities (staged in target order, the row itself, the inverse map) against the oracle."""
import dataclasses

import numpy as np
import pytest
import torch

import oracle
from paper_2507_02659_b200 import binding as od
from paper_2507_02659_b200 import synth, vshard

import parity

pytestmark = pytest.mark.gpu


def _workload(**kw):
    base = dict(B=5, steps=4, k_max=4, k_min=1, v_q=600, v_p=1003, logit_dtype="bf16", map_kind="random",
                mapped_frac=0.7, cache_entries=150, hit_prob=0.6, logit_kind="corr", rho=0.9,
                temperatures=(1.0, 0.5, 0.7), per_seq_seed=True, gen_seed=0xFACE10, unmapped_shift=2.0, sigma=2.0)
    base.update(kw)
    return synth.Workload("parts", **base)


def _check(w, st, device, tiles, steps):
    ctx = parity.make_context(w, st, device)
    ctx.set_option("sample_tiles_per_warp", tiles)
    cache = oracle.Cache(st.runs, st.run_len, st.run_target)
    blocks = set()
    for step in range(steps):
        s = synth.make_step(w, st, step, device=device)
        logits = parity.pad_rows(s.logits)
        parity.check_step(ctx, cache, st, w, s, logits=logits)
        blocks.add(ctx.last_launch_info(2) // w.B)
        mp, vo, so = parity.gpu_step(ctx, s, logits=logits)
        _, _, one = od.od_step(ctx, s.draft_ids, s.draft_len, s.q_sel, s.q_rows, logits, s.temperature, s.seed, step)
        torch.cuda.synchronize()
        for name, t in vars(one).items():
            assert torch.equal(t, vars(so)[name]), name
    ctx.close()
    return blocks


# vocabularies of less than a tile per warp, ragged last tiles and octets, parts without tiles, target
# ids beyond the drafter's where ids are shared, gaps in the map
@pytest.mark.parametrize("shape", [dict(), dict(v_q=599, v_p=4099, logit_dtype="f32"),
                                   dict(v_q=512, v_p=5003, map_kind="identity", cache_entries=0),
                                   dict(v_q=4096, v_p=4096, map_kind="identity", cache_entries=0, logit_dtype="f32"),
                                   dict(v_q=333, v_p=1000, map_kind="identity", cache_entries=0),
                                   dict(v_q=33, v_p=70001, cache_entries=0), dict(v_q=9000, v_p=9001, mapped_frac=1.0, cache_entries=0)])
def test_every_number_of_parts(cuda_device, shape):
    w = _workload(**shape)
    st = synth.make_static(w)
    seen = set()
    for tiles in (0, 1, 3, 5, 9, 1000):
        seen |= _check(w, st, cuda_device, tiles, 2)
    assert 1 in seen
    if w.v_p > 60000:
        assert seen >= {1, 2, 4, 8, 16}


def test_more_mapped_ids_in_a_part_than_are_staged(cuda_device):
    """60000 draft ids on neighbouring target ids: the probabilities come through the inverse map."""
    w = _workload(B=2, k_max=2, v_q=60000, v_p=1_000_000, cache_entries=0)
    st = synth.make_static(w)
    st.vocab_map = np.arange(w.v_q, dtype=np.int32) + 1
    _check(w, st, cuda_device, 0, 2)


# where ids are shared: an odd vocabulary, and rows that begin off a 16-byte boundary; a few sequences, and
# more than are resident at a time; vocabularies that staged would fill a block's shared memory or not fit it
@pytest.mark.parametrize("v_q, v_p, B, offset", [(333, 1000, 5, 0), (512, 1003, 5, 1), (50001, 50001, 4, 0), (50001, 50001, 300, 0),
                                                 (60001, 60100, 300, 0), (4096, 4096, 300, 3)])
def test_shared_ids_off_the_vector_width(cuda_device, v_q, v_p, B, offset):
    w = _workload(B=B, k_max=2, v_q=v_q, v_p=v_p, map_kind="identity", cache_entries=0)
    st = synth.make_static(w)
    ctx = parity.make_context(w, st, cuda_device)
    cache = oracle.Cache(st.runs, st.run_len, st.run_target)
    s = synth.make_step(w, st, 0, device=cuda_device)
    rows = torch.empty(s.q_rows.numel() + offset, device=cuda_device)[offset:].view(s.q_rows.shape).copy_(s.q_rows)
    s = dataclasses.replace(s, q_rows=rows)
    assert rows.data_ptr() % 16 == 4 * offset
    logits = parity.pad_rows(s.logits)
    stats = parity.check_step(ctx, cache, st, w, s, logits=logits, sel=list(range(min(B, 12))))
    assert stats.sample_compared > 0
    mp, vo, so = parity.gpu_step(ctx, s, logits=logits)
    _, _, one = od.od_step(ctx, s.draft_ids, s.draft_len, s.q_sel, s.q_rows, logits, s.temperature, s.seed, 0)
    _, sh, _ = vshard.emulate_step(ctx, logits, 2, mp, s.q_rows, s.draft_ids, s.temperature, s.seed, 0)
    torch.cuda.synchronize()
    for name, t in vars(one).items():
        assert torch.equal(t, vars(so)[name]), name
    settled = ((so.flags | sh.flags) & od.OD_SF_BOUNDARY) == 0
    assert settled.any() and torch.equal(sh.out_token[settled], so.out_token[settled])
    ctx.close()


def test_parts_between_the_powers_of_two(cuda_device):
    """From one sequence to more than fill the chip: every number of parts that the batch can choose."""
    seen = set()
    for B in (1, 13, 24, 30, 37, 48, 60, 73, 90, 148, 300):
        w = _workload(B=B, k_max=2, v_q=1500, v_p=70001, cache_entries=0, mapped_frac=0.9, gen_seed=0xFACE50 + B)
        st = synth.make_static(w)
        ctx = parity.make_context(w, st, cuda_device)
        cache = oracle.Cache(st.runs, st.run_len, st.run_target)
        s = synth.make_step(w, st, 0, device=cuda_device)
        logits = parity.pad_rows(s.logits)
        stats = parity.check_step(ctx, cache, st, w, s, logits=logits, sel=sorted({0, B // 2, B - 1}))
        seen.add(ctx.last_launch_info(2) // B)
        mp, vo, so = parity.gpu_step(ctx, s, logits=logits)
        _, _, one = od.od_step(ctx, s.draft_ids, s.draft_len, s.q_sel, s.q_rows, logits, s.temperature, s.seed, 0)
        torch.cuda.synchronize()
        for name, t in vars(one).items():
            assert torch.equal(t, vars(so)[name]), name
        ctx.close()
    assert seen == {1, 2, 3, 4, 6, 8, 16}, seen


def test_a_smaller_context_made_after_a_larger_one(cuda_device):
    """The limit of dynamic shared memory belongs to the kernels, not to a context: a shard of the larger one
    keeps the tile values of its rows (8 bytes per 256 ids, over 48 KB in both) as before."""
    w = _workload(B=1, k_max=1, v_q=300, v_p=4_000_000, cache_entries=0)
    st = synth.make_static(w)
    ctx = parity.make_context(w, st, cuda_device)
    other = od.Context(cuda_device, 300, 2_000_000, 1, 1)
    s = synth.make_step(w, st, 0, device=cuda_device)
    cache = oracle.Cache(st.runs, st.run_len, st.run_target)
    parity.check_step(ctx, cache, st, w, s)
    mp, vo, so = parity.gpu_step(ctx, s)
    _, sh, _ = vshard.emulate_step(ctx, s.logits, 2, mp, s.q_rows, s.draft_ids, s.temperature, s.seed, 0)
    torch.cuda.synchronize()
    assert int((so.flags | sh.flags)[0]) & od.OD_SF_BOUNDARY or torch.equal(sh.out_token, so.out_token)
    other.close()
    ctx.close()


@pytest.mark.parametrize("dtype", ["bf16", "f32"])
def test_staged_ids_beyond_one_page_of_draft_ids(cuda_device, dtype):
    """Over 65536 draft ids: the groups of the staging lists have bases of their own."""
    w = _workload(B=5, k_max=3, v_q=70001, v_p=90001, mapped_frac=0.6, cache_entries=0, logit_dtype=dtype)
    st = synth.make_static(w)
    assert {2, 16} <= {b for tiles in (0, 3, 1000) for b in _check(w, st, cuda_device, tiles, 2)}


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("v_p", [4096, 70001])
def test_residual_that_is_small_beside_the_n_gram_token(cuda_device, dtype, v_p):
    """Eq. (2) takes the n-gram's token, which has all but 1e-17 of the target's mass, off the residual: what is left
    is e^-50 for every other id, and it is drawn as any other mass, the ids around that token too. Bounds: an exponent
    of 72 is off by half an ulp (4e-6), a term by ln 2 of that, the fp32 sums by less; 1e-5 of up to 70000 ids moves a
    draw by less than one id, so a draw near an id's end may be its neighbour."""
    v_q, B, gram = 64, 256, 300
    ctx = od.Context(cuda_device, v_q, v_p, B, 2)
    vmap = np.full(v_q, -1, np.int32)
    vmap[3:40] = 1000 + 7 * np.arange(37)
    ctx.set_vocab_map(vmap)
    ctx.cache_build(np.array([[1, 2, -1, -1]], np.int32), np.array([2], np.int32), np.array([gram], np.int32))
    ids = torch.tensor([[1, 2]], dtype=torch.int32, device=cuda_device).repeat(B, 1)
    q_sel, q_rows = torch.ones(B, 2, device=cuda_device), torch.zeros(B, 2, v_q, device=cuda_device)
    q_rows[:, 0, 1] = q_rows[:, 1, 2] = 1.0
    logits = parity.pad_rows(torch.full((B, 3, v_p), -50.0, dtype=dtype, device=cuda_device))
    logits[:, :, gram] = 0.0
    T = torch.ones(B, device=cuda_device)
    seed = torch.arange(B, device=cuda_device)
    mp = od.od_map_proposals(ctx, ids, torch.full((B,), 2, dtype=torch.int32, device=cuda_device), q_sel)
    vo = od.od_verify(ctx, logits, mp, T, seed, 0)
    assert (mp.m == 1).all() and (mp.tgt_ids[:, 0] == gram).all()
    vo.n_accepted.zero_()                                   # (p = q' = 1: a verification accepts it)
    so = od.od_sample_residual(ctx, logits, vo, q_rows, ids, mp, T, seed, 0)
    assert (so.flags & ~od.OD_SF_BOUNDARY == 0).all()
    want = (v_p - 1) * np.exp(-50.0)
    np.testing.assert_allclose(so.resid_mass.cpu().numpy(), want, rtol=1e-5)
    at = np.array([oracle.uniform(b, 0, 0, 1) for b in range(B)]) * (v_p - 1)
    token = so.out_token.cpu().numpy()
    index = token - (token > gram)
    assert (token != gram).all() and (np.abs(index - np.floor(at)) <= (np.abs(at - np.round(at)) < 1e-5 * at + 1e-3)).all()
    assert (at < 4000).sum() > 4                            # ids around the n-gram's token are drawn
    ctx.close()

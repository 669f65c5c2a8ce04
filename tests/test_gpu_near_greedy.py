"""Temperatures that all but make the draw greedy, large logits, and masked ids (logits of -inf)
against the oracle: the whole step from each source of the drafter's probabilities, and shards."""
import dataclasses

import pytest
import torch

import oracle
from paper_2507_02659_b200 import binding as od
from paper_2507_02659_b200 import synth
from paper_2507_02659_b200 import vshard

import parity

pytestmark = pytest.mark.gpu

SHAPES = {"staged": dict(), "row": dict(v_q=512, v_p=1003, map_kind="identity", cache_entries=0)}


def _workload(dtype, **kw):
    base = dict(B=12, steps=1, k_max=4, k_min=1, v_q=600, v_p=1003, logit_dtype=dtype, map_kind="random", mapped_frac=0.7,
                cache_entries=150, hit_prob=0.6, logit_kind="corr", rho=0.9, temperatures=(1.0, 0.5), per_seq_seed=True,
                gen_seed=0xFACE30, unmapped_shift=2.0, sigma=2.0)
    base.update(kw)
    return synth.Workload("near_greedy", **base)


def _check(w, st, s, logits, device):
    """The three calls against the oracle, od_step with the same bits, and two shards with the same tokens."""
    ctx = parity.make_context(w, st, device)
    s = dataclasses.replace(s, logits=logits)
    rows = parity.pad_rows(logits)
    cache = oracle.Cache(st.runs, st.run_len, st.run_target)
    stats = parity.check_step(ctx, cache, st, w, s, logits=rows)
    mp, vo, so = parity.gpu_step(ctx, s, logits=rows)
    _, _, one = od.od_step(ctx, s.draft_ids, s.draft_len, s.q_sel, s.q_rows, rows, s.temperature, s.seed, s.step)
    _, sh, _ = vshard.emulate_step(ctx, rows, 2, mp, s.q_rows, s.draft_ids, s.temperature, s.seed, s.step)
    torch.cuda.synchronize()
    for name, t in vars(one).items():
        assert torch.equal(t, vars(so)[name]), name
    settled = ((so.flags | sh.flags) & od.OD_SF_BOUNDARY) == 0
    assert torch.equal(sh.out_token[settled], so.out_token[settled]) and (so.out_token >= 0).all()
    ctx.close()
    return stats


# |M| * log2(e) / T from 2.9e7 (where a float's ulp is 2) to 1.4e9 (128, below what exp2 can hold)
@pytest.mark.parametrize("dtype", ["bf16", "f32"])
@pytest.mark.parametrize("source", sorted(SHAPES))
@pytest.mark.parametrize("M,T", [(20.0, 1e-6), (100.0, 1e-6), (20.0, 1e-7), (-37.0, 1e-7), (100.0, 1e-7), (0.0, 1e-7)])
def test_near_greedy(cuda_device, M, T, source, dtype):
    w = _workload(dtype, **SHAPES[source])
    st = synth.make_static(w)
    s = synth.make_step(w, st, 0, device=cuda_device)
    x = s.logits.float()
    logits = (x - x.amax(2, keepdim=True) + M).to(s.logits.dtype)
    stats = _check(w, st, dataclasses.replace(s, temperature=torch.full_like(s.temperature, T)), logits, cuda_device)
    assert stats.sample_compared > 0


# half of the ids masked; some whole tiles (256 ids), others in part; the mapped ones among them keep their q'
@pytest.mark.parametrize("dtype", ["bf16", "f32"])
@pytest.mark.parametrize("source", sorted(SHAPES))
def test_masked_ids(cuda_device, source, dtype):
    w = _workload(dtype, **SHAPES[source])
    st = synth.make_static(w)
    s = synth.make_step(w, st, 0, device=cuda_device)
    logits = s.logits.clone()
    logits[:, :, 256:512] = float("-inf")
    logits[:, :, 600:900:2] = float("-inf")
    assert _check(w, st, s, logits, cuda_device).sample_compared > 0

"""Calls whose inputs are written by a launch that is still at work when the library's kernels become resident: a producer
that releases its dependents first and writes half a millisecond later (tests/helpers/early_producer.cu)."""
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

"""The native marshalling of the binding: the same calls with the same results as the checks in
Python, and the same errors."""
import pytest
import torch

from paper_2507_02659_b200 import binding as od
from paper_2507_02659_b200 import synth
from paper_2507_02659_b200 import vshard

import parity

pytestmark = pytest.mark.gpu


class _Nothing:
    """A stand-in for _marshal that takes no call."""

    def __getattr__(self, name):
        return lambda *a: None


def _inputs(device, dtype):
    w = synth.Workload("marshal", B=5, steps=1, k_max=4, k_min=1, v_q=600, v_p=1024, logit_dtype=dtype, map_kind="random",
                       mapped_frac=0.7, cache_entries=100, hit_prob=0.5, logit_kind="corr", rho=0.9, temperatures=(1.0, 0.5),
                       per_seq_seed=True, gen_seed=0xFACE20, unmapped_shift=2.0, sigma=2.0)
    st = synth.make_static(w)
    s = synth.make_step(w, st, 0, device=device)
    return w, parity.make_context(w, st, device), s, parity.pad_rows(s.logits)


def _run(w, ctx, s, logits):
    """Every call that has a native form; their outputs in one list."""
    a = (s.draft_ids, s.draft_len, s.q_sel)
    out = [vars(v) for v in od.od_step(ctx, *a, s.q_rows, logits, s.temperature, s.seed, 7)]
    mp, vo, so = od.od_map_proposals(ctx, *a), None, None
    vo = od.od_verify(ctx, logits, mp, s.temperature, s.seed, 7)
    so = od.od_sample_residual(ctx, logits, vo, s.q_rows, s.draft_ids, mp, s.temperature, s.seed, 7)
    out += [vars(mp), vars(vo), vars(so)]
    loss, grad = od.od_distill_loss(ctx, s.q_rows, s.draft_ids, mp, logits, vo, s.temperature, 0.2)
    out.append(dict(loss=loss, grad=grad, lone=od.od_distill_loss(ctx, s.q_rows, s.draft_ids, mp, logits, vo, s.temperature,
                                                                   0.2, 1, want_grad=False)[0]))
    head = torch.linspace(2, -2, w.B * w.k_max, device=ctx.device).view(w.B, w.k_max)
    out.append(dict(enumerate(od.od_exit_rule(ctx, head, None, 0.6))))
    out.append(dict(enumerate(od.od_exit_rule(ctx, head, s.draft_len, 0.6))))
    shards = vshard.emulate_step(ctx, logits, 2, mp, s.q_rows, s.draft_ids, s.temperature, s.seed, 7)
    out += [vars(v) for v in shards if hasattr(v, "__dict__")]
    ctx.cache_configure(64, 0, 32)
    ctx.cache_set_clock(3)
    runs = torch.arange(128, dtype=torch.int32, device=ctx.device).view(32, 4)
    ctx.cache_insert(runs, torch.full((32,), 3, dtype=torch.int32, device=ctx.device), runs[:, 0].contiguous())
    ctx.cache_trim()
    out.append(dict(n=torch.tensor(ctx.cache_stats())))
    return out


@pytest.mark.parametrize("dtype", ["bf16", "f32"])
def test_the_same_results_as_the_checks_in_python(cuda_device, dtype, monkeypatch):
    w, ctx, s, logits = _inputs(cuda_device, dtype)
    native = _run(w, ctx, s, logits)
    ctx.close()
    w, ctx, s, logits = _inputs(cuda_device, dtype)
    monkeypatch.setattr(od, "_native", _Nothing())
    plain = _run(w, ctx, s, logits)
    ctx.close()
    assert len(native) == len(plain) >= 10
    for x, y in zip(native, plain):
        assert x.keys() == y.keys()
        for k in x:
            assert torch.equal(x[k], y[k]), k


def test_the_same_errors(cuda_device):
    w, ctx, s, logits = _inputs(cuda_device, "bf16")
    call = lambda **kw: od.od_step(ctx, *({"ids": s.draft_ids, "len": s.draft_len, "q": s.q_sel, "rows": s.q_rows,
                                           "logits": logits, "T": s.temperature, "seed": s.seed, "step": 0} | kw).values())
    call()
    with pytest.raises(TypeError):
        call(ids=s.draft_ids.long())
    with pytest.raises(ValueError):
        call(T=s.temperature.cpu())
    with pytest.raises(ValueError):
        call(q=s.q_sel.t().contiguous().t())
    with pytest.raises(ValueError):
        call(rows=s.q_rows[:, :, :-1].contiguous())
    with pytest.raises(ValueError):
        call(logits=logits[:, :-1])
    with pytest.raises(TypeError):
        call(logits=logits.half())
    with pytest.raises(od.OdError):
        call(logits=torch.empty(w.B, w.k_max + 1, w.v_p + 1, dtype=torch.bfloat16, device=cuda_device)[:, :, :w.v_p])
    call(step=2 ** 64 + 3)
    ctx.close()


class _Recorder:
    """Passes calls on to _marshal and keeps what each returned."""

    def __init__(self, native):
        self.native, self.calls = native, []

    def __getattr__(self, name):
        def call(*a):
            status = getattr(self.native, name)(*a)
            self.calls.append((name, status))
            return status
        return call


def test_every_well_formed_call_is_made_natively(cuda_device, monkeypatch):
    w, ctx, s, logits = _inputs(cuda_device, "bf16")
    assert not isinstance(od._native, od._InPython)
    rec = _Recorder(od._native)
    monkeypatch.setattr(od, "_native", rec)
    _run(w, ctx, s, logits)
    assert {n for n, _ in rec.calls} == {"map_proposals", "verify", "sample_residual", "step", "exit_rule", "distill_loss",
                                         "verify_shard_stats", "verify_shard_finish", "sample_shard_mass", "sample_shard_pick",
                                         "cache_insert", "cache_trim"}
    assert all(status == 0 for _, status in rec.calls), rec.calls
    # and one that does not take its arguments as they stand is not
    del rec.calls[:]
    with pytest.raises(TypeError):
        od.od_map_proposals(ctx, s.draft_ids.long(), s.draft_len, s.q_sel)
    assert rec.calls == [("map_proposals", None)]
    ctx.close()

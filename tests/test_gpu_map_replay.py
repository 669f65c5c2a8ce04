"""A CUDA graph captured under one vocabulary map and replayed under another computes with the
map of its replay, as kernels that look every id up would."""
import numpy as np
import pytest
import torch

from paper_2507_02659_b200 import binding as od
from paper_2507_02659_b200 import synth

pytestmark = pytest.mark.gpu

V_Q, V_P = 2000, 9001


def _map(kind, seed):
    if kind == "identity":
        return np.arange(V_Q, dtype=np.int32)
    rng = np.random.default_rng(seed)
    m = np.full(V_Q, -1, np.int32)
    if kind == "sparse":
        d = rng.permutation(V_Q)[:300]
        m[d] = rng.permutation(V_P)[:300]
    else:                                                   # every id, all of them in one part of a row
        m[:] = V_P - V_Q + rng.permutation(V_Q)
    return m


def _passes(ctx, s, logits, out):
    """The step, a two-shard step's first shard, the loss with and without a gradient."""
    mp, vo, so = od.od_step(ctx, s.draft_ids, s.draft_len, s.q_sel, s.q_rows, logits, s.temperature, s.seed, 0,
                            mp=out["mp"], vo=out["vo"], so=out["so"])
    od.od_sample_shard_mass(ctx, 0, logits, vo, s.q_rows, s.draft_ids, mp, s.temperature, out=out["mass"])
    od.od_distill_loss(ctx, s.q_rows, s.draft_ids, mp, logits, vo, s.temperature, 0.2, loss=out["loss"], grad=out["grad"])
    od.od_distill_loss(ctx, s.q_rows, s.draft_ids, mp, logits, vo, s.temperature, 0.2, want_grad=False, loss=out["lone"])


def _buffers(ctx, B, K, dev):
    return dict(mp=od.alloc_map_out(ctx, B, K), vo=od.alloc_verify_out(ctx, B, K), so=od.alloc_sample_out(ctx, B),
                mass=torch.zeros(B, 2, dtype=torch.float64, device=dev), loss=torch.zeros(B, K, device=dev),
                grad=torch.zeros(B, K, V_Q, device=dev), lone=torch.zeros(B, K, device=dev))


# few sequences (16 blocks each) and many (one); sums in another order differ by fp32 rounding: the
# residual mass and the loss by some 2e-7 of the summed terms
@pytest.mark.parametrize("dtype", ["bf16", "f32"])
@pytest.mark.parametrize("B", [3, 330])
@pytest.mark.parametrize("before, after", [("sparse", "dense"), ("dense", "sparse"), ("identity", "dense"), ("dense", "identity"),
                                           ("identity", "sparse"), ("sparse", "identity")])
def test_replay_under_another_map(cuda_device, before, after, B, dtype):
    w = synth.Workload("replay", B=B, steps=1, k_max=3, k_min=1, v_q=V_Q, v_p=V_P, logit_dtype=dtype, map_kind="random",
                       mapped_frac=0.5, cache_entries=0, hit_prob=0.0, logit_kind="corr", rho=0.9, temperatures=(1.0, 0.5),
                       per_seq_seed=True, gen_seed=0xFACE40, unmapped_shift=0.0, sigma=2.0)
    s = synth.make_step(w, synth.Static(_map(after, 1), *(np.zeros(n, np.int32) for n in ((0, 4), 0, 0))), 0, device=cuda_device)
    per = 16 // s.logits.element_size()
    store = torch.zeros(B, w.k_max + 1, -(-V_P // per) * per, dtype=s.logits.dtype, device=cuda_device)
    store[:, :, :V_P] = s.logits
    logits = store[:, :, :V_P]
    ctx = od.Context(cuda_device, V_Q, V_P, B, w.k_max)
    ctx.set_vocab_map(_map(before, 2))
    got, want = _buffers(ctx, B, w.k_max, cuda_device), _buffers(ctx, B, w.k_max, cuda_device)
    _passes(ctx, s, logits, got)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        _passes(ctx, s, logits, got)
    ctx.set_vocab_map(_map(after, 1))
    _passes(ctx, s, logits, want)
    for part in (got["mp"], got["vo"]):                     # (entries behind a sequence's m are not written)
        for t in vars(part).values():
            t.zero_()
    want["mp"].counters.zero_()
    graph.replay()
    torch.cuda.synchronize()
    for name in ("tgt_ids", "m", "tail_kind", "span_len"):
        assert torch.equal(getattr(got["mp"], name), getattr(want["mp"], name)), name
    for name, t in vars(got["vo"]).items():
        assert torch.equal(t, getattr(want["vo"], name)), name
    g, x = got["so"], want["so"]
    settled = ((g.flags | x.flags) & od.OD_SF_BOUNDARY) == 0
    assert settled.any() and torch.equal(g.out_token[settled], x.out_token[settled])
    torch.testing.assert_close(g.resid_mass, x.resid_mass, rtol=2e-6, atol=2e-6)
    torch.testing.assert_close(got["mass"], want["mass"], rtol=2e-6, atol=2e-6)
    for name in ("loss", "lone", "grad"):
        torch.testing.assert_close(got[name], want[name], rtol=2e-5, atol=2e-6)
    assert B < 100 or (want["loss"] != 0).any()
    ctx.close()

"""The exit rule's sixteen lanes per sequence: every proposal length, the first and last sequence of a warp and of
a block, thresholds that never and always fire, against the oracle."""
import numpy as np
import pytest
import torch

from oracle import exit_rule as er
from paper_2507_02659_b200 import binding as od

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("K", [1, 2, 15, 16])
@pytest.mark.parametrize("B", [1, 2, 7, 8, 9, 257])
def test_exit_rule_at_the_edges_of_its_lanes(cuda_device, B, K):
    rng = np.random.default_rng(100 * B + K)
    f = rng.normal(2.5, 1.5, size=(B, K)).astype(np.float32)
    avail = rng.integers(-1, K + 2, size=B).astype(np.int32)
    ctx = od.Context(cuda_device, 100, 100, 4, K)
    for gamma in (0.0, 0.37, 1.0):
        for a in (avail, None):
            got = od.od_exit_rule(ctx, torch.from_numpy(f).to(cuda_device), None if a is None else torch.from_numpy(a).to(cuda_device), gamma)
            torch.cuda.synchronize()
            length, reject, flags = (t.cpu().numpy() for t in got)
            n = np.full(B, K, np.int32) if a is None else np.clip(a, 0, K)
            want_len, want_rej = er.exit_rule(f, n.astype(np.int32), gamma)
            # a product of at most 16 fp32 sigmoids: 16 * 2^-23 and each sigmoid's own few units in the last place
            np.testing.assert_allclose(reject, want_rej, rtol=0, atol=3e-6)
            assert (flags[length != want_len] != 0).all()
            assert (flags >> np.maximum(length, 1) == 0).all()
    ctx.close()

"""A binary64 launch that starts with enough warps for the integer pipes' software
arithmetic leaves it, warp by warp, as the others end: the whole warp at once, and
the rows keep the bits of launches that never use it (at most two warps per
sub-partition)."""
import numpy as np
import pytest
import torch

import aeb_inputs as ai

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def aeb():
    import paper_2604_27193_gb300 as m
    m.build()
    return m


@pytest.mark.parametrize("n", [45_000, 98_311])  # 2.3 warps a sub-partition; more than fit at once
def test_rows_alike_whatever_the_tail_runs_on(aeb, n):
    rng = np.random.default_rng(2)
    m = ai.single_model(4e-3)
    p = ai.draw_params(m, ai.single_scenario(), n, 7)
    p["v0"][rng.random(n) < 0.9] *= 0.3  # few long rollouts among short ones: a long tail
    P = {k: torch.from_numpy(np.ascontiguousarray(v)).cuda() for k, v in p.items()}
    out, ref = aeb.alloc_outputs(n), aeb.alloc_outputs(n)
    aeb.aeb_rollout(m, P, n, aeb.FP64_PLAIN, out)
    for lo in range(0, n, 16_384):
        hi = min(n, lo + 16_384)
        aeb.aeb_rollout(m, {k: v[lo:hi].contiguous() for k, v in P.items()}, hi - lo,
                        aeb.FP64_PLAIN, {k: v[lo:hi] for k, v in ref.items()})
    torch.cuda.synchronize()
    for k in out:
        assert out[k].cpu().numpy().tobytes() == ref[k].cpu().numpy().tobytes(), k

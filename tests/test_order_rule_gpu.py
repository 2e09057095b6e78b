"""The rule that orders a binary32 launch: few steps, or few samples times steps, stay
in index order, where the order costs more than it saves.  A plan shows which way it
went by the device memory it holds (6 B per sample more when ordered); around the
lines, both ways give the bits of a captured launch, which takes index order."""
import numpy as np
import pytest
import torch

import aeb_inputs as ai

pytestmark = pytest.mark.gpu

ONE, TTC = ai.single_model(), ai.ttc_model(2.0)
READ = ai.replace(TTC, perc_sigma=1.0, perc_drop=0.2, perc_latency=0.05, perc_seed=3)


@pytest.fixture(scope="module")
def aeb():
    import paper_2604_27193_gb300 as m
    m.build()
    return m


def _steps(m, n, dt=1e-3):
    return ai.replace(m, dt=dt, t_max=n * dt)


def _columns(m, n):
    k = min(n, 50_000)
    p = ai.draw_params(m, ai.single_scenario(), k, 3)
    return {f: torch.from_numpy(np.ascontiguousarray(p[f])).cuda().repeat(-(-n // k))[:n].contiguous()
            for f in ai.FIELDS}


def _plan(aeb, m, P, n, out):
    st = torch.empty(aeb.JOB_STATS_BYTES, dtype=torch.uint8, device="cuda")
    return aeb.BatchPlan(m, [(0, 0, n, m.ttc_thr)], P, aeb.FP32_COMP, out, st), st


@pytest.mark.parametrize("m,ordered", [
    (_steps(ONE, 999), False), (_steps(ONE, 1000), True), (ai.single_model(2e-2), False),
    (ai.single_model(1e-2), True), (_steps(TTC, 2999), False), (_steps(TTC, 3000), True),
    (_steps(READ, 2999), False), (_steps(READ, 3000), True),
    (_steps(ai.replace(ONE, lead=0), 1499), False), (_steps(ai.replace(ONE, lead=0), 1500), True)])
def test_which_plans_hold_an_order(aeb, m, ordered):
    n = 4_000_000
    P, out = _columns(m, n), aeb.alloc_outputs(n, which=("status", "x_ref", "v_imp", "n_steps"))
    warm, _keep = _plan(aeb, m, P, 32, out)  # the kernels are loaded
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    plan, _keep2 = _plan(aeb, m, P, n, out)
    held = free - torch.cuda.mem_get_info()[0]
    plan.close()
    warm.close()
    assert (held > 5 * n) == ordered, held  # (its tables take 0.5 B per sample)


@pytest.mark.parametrize("m,n", [(_steps(ONE, 999), 100_001), (_steps(ONE, 1000), 100_001),
                                 (_steps(ONE, 2499), 40_001), (_steps(ONE, 2500), 40_001),
                                 (_steps(TTC, 1999), 530_001), (_steps(TTC, 2000), 530_001),
                                 (_steps(READ, 2000), 99_999), (_steps(READ, 2000), 100_001)])
def test_both_sides_of_the_lines_same_bits(aeb, m, n):
    P, a, b = _columns(m, n), aeb.alloc_outputs(n), aeb.alloc_outputs(n)
    plan, _keep = _plan(aeb, m, P, n, a)
    plan.run()
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        aeb.aeb_rollout(m, P, 1, aeb.FP32_COMP, b)  # the stream's fixed scratch
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        aeb.aeb_rollout(m, P, n, aeb.FP32_COMP, b)
    g.replay()
    torch.cuda.synchronize()
    for k in a:
        assert a[k].cpu().numpy().tobytes() == b[k].cpu().numpy().tobytes(), k
    plan.close()

"""The processing order of a rollout launch changes no result: the same bits
as in natural order (which a launch under stream capture takes, since its
order's scratch must not be allocated there), at the sizes around the rule
that orders a launch, for every trigger, lead and cap kind, in both precisions,
over more than one piece, and in a table of ragged jobs."""
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


def _device(p):
    return {k: torch.from_numpy(np.ascontiguousarray(v)).cuda() for k, v in p.items()}


def _bits(out):
    return {k: v.cpu().numpy().tobytes() for k, v in out.items()}


def _both(aeb, m, p, n, precision, which):
    a, b = aeb.alloc_outputs(n, which=which), aeb.alloc_outputs(n, which=which)
    aeb.aeb_rollout(m, p, n, precision, a)
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        aeb.aeb_rollout(m, p, 1, precision, b)  # the stream's fixed scratch
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        aeb.aeb_rollout(m, p, n, precision, b)
    g.replay()
    torch.cuda.synchronize()
    return _bits(a), _bits(b)


def _models():
    lead = ai.lead_braking_model(dt=5e-3)
    return {
        "single": (ai.single_model(5e-3), ai.single_scenario()),
        "paper": (ai.replace(ai.paper_model(), dt=5e-3), ai.paper_scenario()),
        "icy lumped": (ai.replace(ai.single_model(5e-3), cap_mode=ai.CAP_LUMPED),
                       ai.scenario_from_means(25.0, 0.1, 0.25, 60.0, 1, 1)),
        "lead": (lead, ai.lead_braking_scenario()),
        "ttc": (ai.ttc_model(2.0, 5e-3), ai.single_scenario()),
        "ttc lead readings": (ai.replace(lead, trigger=ai.TRIGGER_TTC, ttc_thr=2.0, perc_sigma=1.0,
                                         perc_drop=0.2, perc_latency=0.05, perc_seed=3),
                              ai.lead_braking_scenario()),
        "no braking": (ai.replace(ai.single_model(5e-3), a_cmd=1.0), ai.single_scenario()),
    }


@pytest.mark.parametrize("kind", list(_models()))
@pytest.mark.parametrize("n", [19456, 19457, 40961])
def test_ordered_rollouts_same_bits_fp32(aeb, kind, n):
    m, sc = _models()[kind]
    edge = ai.edge_params(m)
    p = ai.concat_params([ai.draw_params(m, sc, n - len(edge["v0"]), 5), edge])
    a, b = _both(aeb, m, _device(p), n, aeb.FP32_COMP, aeb.OUTPUTS)
    assert a == b


@pytest.mark.parametrize("kind", list(_models()))
def test_ordered_rollouts_same_bits_fp64(aeb, kind):
    m, sc = _models()[kind]
    edge = ai.edge_params(m)
    p = ai.concat_params([ai.draw_params(m, sc, 20480, 6), edge])
    a, b = _both(aeb, m, _device(p), len(p["v0"]), aeb.FP64_PLAIN, aeb.OUTPUTS)
    assert a == b


@pytest.mark.parametrize("a_cmd", [-6.0, 1.0])
@pytest.mark.parametrize("dt,t_max", [(1e-3, 1.2), (5e-3, 3.0), (2e-2, 10.0)])
def test_fp32_lone_and_full_launches_same_bits(aeb, a_cmd, dt, t_max):
    """A launch of at most one warp per sub-partition takes no flat windows (and
    so keeps every lane's actuator state); one that fills the GPU does.  Roads and
    actuators around the flat condition (saturated, no grip, instantaneous, dt / tau
    past 1.6), ended by the horizon as well as by stops and contacts."""
    rng = np.random.default_rng(12)
    m = ai.replace(ai.single_model(dt), t_max=t_max, a_cmd=a_cmd)
    n, few = 40_960, 2048
    p = ai.draw_params(m, ai.scenario_from_means(25.0, 0.05, 0.7, 70.0, 3, 0), n, 9)
    p["tau"] = rng.choice([0.0, dt / 3, dt / 1.7, dt / 1.5, dt, 0.1, 0.3], n)
    p["mu"][::29] = 0.0
    p["mu"][3::31] = 6.0  # mu h / L above 1: a falling line
    P = _device(p)
    full, lone = aeb.alloc_outputs(n), aeb.alloc_outputs(few)
    aeb.aeb_rollout(m, P, n, aeb.FP32_COMP, full)
    aeb.aeb_rollout(m, {k: v[:few].contiguous() for k, v in P.items()}, few, aeb.FP32_COMP, lone)
    torch.cuda.synchronize()
    assert _bits({k: v[:few] for k, v in full.items()}) == _bits(lone)


def test_order_in_pieces(aeb):
    """2^24 positions are ordered at a time: a launch of 33 more takes two pieces."""
    n = (1 << 24) + 33
    m = ai.single_model(2e-2)
    base = _device(ai.draw_params(m, ai.single_scenario(), 1 << 16, 7))
    p = {k: v.repeat(257)[:n].contiguous() for k, v in base.items()}
    a, b = _both(aeb, m, p, n, aeb.FP32_COMP, ("status", "x_ref", "n_steps"))
    assert a == b


def test_ordered_table(aeb):
    """Jobs of ragged sizes (empty, one sample, one short of a tile, ...) in one ordered plan:
    each row as in a flat launch of its job's rows."""
    m = ai.single_model(5e-3)
    sizes = [0, 1, 31, 32, 33, 9000, 64, 14001, 7, 0, 12345]
    n = sum(sizes)
    p = _device(ai.draw_params(m, ai.single_scenario(), n, 8))
    out = aeb.alloc_outputs(n)
    first = np.concatenate([[0], np.cumsum(sizes)])
    st = torch.empty(aeb.JOB_STATS_BYTES * len(sizes), dtype=torch.uint8, device="cuda")
    plan = aeb.BatchPlan(m, [(int(o), int(o), k, 0.0) for o, k in zip(first, sizes)], p,
                         aeb.FP32_COMP, out, st)
    plan.run()
    ref = aeb.alloc_outputs(n)
    for o, k in zip(first, sizes):
        if k:
            aeb.aeb_rollout(m, {f: c[int(o):int(o) + k] for f, c in p.items()}, k, aeb.FP32_COMP,
                            {f: c[int(o):int(o) + k] for f, c in ref.items()})
    torch.cuda.synchronize()
    assert _bits(out) == _bits(ref)
    plan.close()

"""Ordered launches against index order where it is certain that one arm is ordered: a
plan, whose order's scratch is part of its own allocation, at sizes and steps at which
the rule orders every kind of launch; the other arm is a captured launch, which takes
index order.  Both precisions, more than one piece, a table of ragged jobs."""
import numpy as np
import pytest
import torch

import aeb_inputs as ai

pytestmark = pytest.mark.gpu

REDUCED = ("status", "x_ref", "v_imp", "n_steps")


@pytest.fixture(scope="module")
def aeb():
    import paper_2604_27193_gb300 as m
    m.build()
    return m


def _kinds(dt):
    lead = ai.lead_braking_model(dt=dt)
    one, near = ai.single_scenario(), ai.lead_braking_scenario()
    readings = dict(perc_sigma=1.0, perc_drop=0.2, perc_latency=0.05, perc_seed=3)
    return {
        "single": (ai.single_model(dt), one),
        "paper": (ai.replace(ai.paper_model(), dt=dt), ai.paper_scenario()),
        "icy lumped": (ai.replace(ai.single_model(dt), cap_mode=ai.CAP_LUMPED),
                       ai.scenario_from_means(25.0, 0.1, 0.25, 60.0, 1, 1)),
        "lead": (lead, near),
        "ttc": (ai.ttc_model(2.0, dt), one),
        "ttc below zero": (ai.replace(ai.ttc_model(-1.0, dt), lead=0), one),
        "ttc lead readings": (ai.replace(lead, trigger=ai.TRIGGER_TTC, ttc_thr=2.0, **readings), near),
        "no braking": (ai.replace(ai.single_model(dt), a_cmd=1.0), one),
    }


def _device(p, n=None):
    P = {k: torch.from_numpy(np.ascontiguousarray(v)).cuda() for k, v in p.items()}
    return P if n is None else {k: v.repeat(-(-n // len(v)))[:n].contiguous() for k, v in P.items()}


def _bits(out):
    return {k: v.cpu().numpy().tobytes() for k, v in out.items()}


def _ordered(aeb, m, P, n, precision, which):
    out = aeb.alloc_outputs(n, which=which)
    st = torch.empty(aeb.JOB_STATS_BYTES, dtype=torch.uint8, device="cuda")
    plan = aeb.BatchPlan(m, [(0, 0, n, m.ttc_thr)], P, precision, out, st)
    plan.run()
    torch.cuda.synchronize()
    plan.close()
    return _bits(out)


def _index_order(aeb, m, P, n, precision, which):
    out = aeb.alloc_outputs(n, which=which)
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        aeb.aeb_rollout(m, P, 1, precision, out)  # the stream's fixed scratch
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        aeb.aeb_rollout(m, P, n, precision, out)
    g.replay()
    torch.cuda.synchronize()
    return _bits(out)


@pytest.mark.parametrize("n", [20_001, 60_013])
@pytest.mark.parametrize("kind", list(_kinds(1e-3)))
def test_fp32_same_bits(aeb, kind, n):
    m, sc = _kinds(1e-3)[kind]  # 10,000 steps: every kind is ordered from 20,000 samples on
    edge = ai.edge_params(m)
    P = _device(ai.concat_params([ai.draw_params(m, sc, n - len(edge["v0"]), 5), edge]))
    want = _index_order(aeb, m, P, n, aeb.FP32_COMP, aeb.OUTPUTS)
    assert _ordered(aeb, m, P, n, aeb.FP32_COMP, aeb.OUTPUTS) == want


@pytest.mark.parametrize("n", [33, 20_500])
@pytest.mark.parametrize("kind", list(_kinds(5e-3)))
def test_fp64_same_bits(aeb, kind, n):
    m, sc = _kinds(5e-3)[kind]
    edge = ai.edge_params(m)
    P = _device(ai.concat_params([ai.draw_params(m, sc, n - len(edge["v0"]), 6), edge]))
    want = _index_order(aeb, m, P, n, aeb.FP64_PLAIN, aeb.OUTPUTS)
    assert _ordered(aeb, m, P, n, aeb.FP64_PLAIN, aeb.OUTPUTS) == want


def test_more_than_one_piece(aeb):
    """2^24 positions are ordered at a time; 33 more take a second piece, in a plan and in a
    launch of its own (which has its order's scratch from the pool)."""
    n, m = (1 << 24) + 33, ai.single_model(1e-2)
    P = _device(ai.draw_params(m, ai.single_scenario(), 1 << 16, 7), n)
    want = _index_order(aeb, m, P, n, aeb.FP32_COMP, REDUCED)
    assert _ordered(aeb, m, P, n, aeb.FP32_COMP, REDUCED) == want
    out = aeb.alloc_outputs(n, which=REDUCED)
    aeb.aeb_rollout(m, P, n, aeb.FP32_COMP, out)
    assert _bits(out) == want


@pytest.mark.parametrize("precision,dt", [("FP32_COMP", 1e-3), ("FP64_PLAIN", 5e-3)])
def test_ragged_jobs(aeb, precision, dt):
    m, prec = ai.single_model(dt), getattr(aeb, precision)
    sizes = [0, 1, 31, 32, 33, 9000, 64, 14_001, 7, 0, 12_345]
    first = np.concatenate([[0], np.cumsum(sizes)])
    n = int(first[-1])
    P = _device(ai.draw_params(m, ai.single_scenario(), n, 8))
    out = aeb.alloc_outputs(n)
    st = torch.empty(aeb.JOB_STATS_BYTES * len(sizes), dtype=torch.uint8, device="cuda")
    plan = aeb.BatchPlan(m, [(int(o), int(o), k, 0.0) for o, k in zip(first, sizes)], P, prec, out, st)
    plan.run()
    torch.cuda.synchronize()
    plan.close()
    ref = _index_order(aeb, m, P, n, prec, aeb.OUTPUTS)
    assert _bits(out) == ref

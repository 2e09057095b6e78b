"""Trigger tests that the kernels skip may never hide a trigger, and steps that run
without a contact test may never hide a contact, also where the margin (gap + noise)
- thr (v - v_L) falls because the car slows (a negative threshold: uphill, drag) or
because drag drives it (a negative air density).  Most samples of every model trigger;
binary64 gives the oracle's bits, binary32 stays within its bounds of it (no drag that
drives: binary32 scales by the drag coefficient's root)."""
import numpy as np
import pytest

import aeb_inputs as ai
from fp32_bounds import fp32_report, resolve_onset_ties, with_gap

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

N = 1200


@pytest.fixture(scope="module")
def aeb():
    import paper_2604_27193_gb300 as m
    m.build()
    return m


def _free(thr, dt=2e-3, **kw):  # no lead: the gap to d0 closes and turns negative
    return ai.replace(ai.ttc_model(thr, dt), lead=0, **kw)


def _lead(thr, v, b, dt=2e-3, **kw):
    return ai.replace(ai.lead_braking_model(lead_v0=v, lead_decel=b, dt=dt),
                      trigger=ai.TRIGGER_TTC, ttc_thr=thr, **kw)


# (model, the noise as a share of -d0, mean speed)
CASES = {
    "-1 s": (_free(-1.0), 0.0, 25.0),
    "-2 s": (_free(-2.0), 0.0, 25.0),
    "-5 s": (_free(-5.0), 0.5, 20.0),
    "-2 s 10 ms": (_free(-2.0, 1e-2), 0.0, 25.0),
    "-3 s standing lead": (ai.ttc_model(-3.0, 4e-3), 1.6, 12.0),
    "-2 s moving lead": (_lead(-2.0, 8.0, 0.0), 1.7, 18.0),
    "-2 s braking lead": (_lead(-2.0, 8.0, 3.0), 1.7, 18.0),
    "-2 s readings": (_free(-2.0, perc_sigma=1.0, perc_drop=0.2, perc_latency=0.05,
                            perc_seed=5), 0.0, 25.0),
}
DRIVEN = {
    "driven 2 s": (_free(2.0, rho=-20.0), 0.0, 20.0),
    "driven -2 s": (_free(-2.0, rho=-20.0), 0.0, 20.0),
    "driven moving lead": (_lead(2.0, 8.0, 0.0, rho=-20.0), 0.0, 20.0),
    "driven braking lead": (ai.replace(ai.lead_braking_model(dt=2e-3), rho=-20.0), 0.0, 20.0),
}


def _params(case, seed):
    m, share, v = case
    rng = np.random.default_rng(seed)
    p = ai.draw_params(m, ai.scenario_from_means(v, 0.3, 0.95, 45.0, seed, 0), N)
    grade = rng.uniform(-0.1, 0.2, N)
    p["gs"], p["gc"] = m.g * np.sin(grade), m.g * np.cos(grade)
    p["cd"] = rng.choice([0.0, 0.3, 1.0], N)
    p["noise"] = p["noise"] - share * p["d0"]
    return p


@pytest.mark.parametrize("copies", [1, 45])  # 54,000 rollouts: software arithmetic too
@pytest.mark.parametrize("kind", list(CASES) + list(DRIVEN))
def test_fp64_triggers_as_the_oracle(aeb, oracle_mod, kind, copies):
    case = {**CASES, **DRIVEN}[kind]
    m = case[0]
    if m.perc_sigma > 0 and copies > 1:
        pytest.skip("a copy's readings are keyed by its own row")
    p = _params(case, 3)
    exp = oracle_mod.rollout(m, p, threads=8)
    assert np.mean(exp["n_onset"] >= 0) > 0.5
    exp = {k: np.tile(v, copies) for k, v in exp.items()}
    P = {f: torch.from_numpy(np.tile(p[f], copies)).cuda() for f in ai.FIELDS}
    out = aeb.alloc_outputs(N * copies)
    aeb.aeb_rollout(m, P, N * copies, aeb.FP64_PLAIN, out)
    torch.cuda.synchronize()
    for k, v in out.items():
        got, want = v.cpu().numpy(), exp[k]
        if got.dtype == np.float64:
            got, want = got.view(np.uint64), want.view(np.uint64)
        bad = np.nonzero(got != want)[0]
        assert len(bad) == 0, (k, len(bad), bad[:5])


@pytest.mark.parametrize("kind", list(CASES))
def test_fp32_triggers_within_bounds(aeb, oracle_mod, kind):
    m = CASES[kind][0]
    p = _params(CASES[kind], 4)
    exp = oracle_mod.rollout(m, p, threads=8)
    assert np.mean(exp["n_onset"] >= 0) > 0.5
    P = {f: torch.from_numpy(np.ascontiguousarray(p[f])).cuda() for f in ai.FIELDS}
    out = aeb.alloc_outputs(N)
    aeb.aeb_rollout(m, P, N, aeb.FP32_COMP, out)
    torch.cuda.synchronize()
    got = {k: v.cpu().numpy() for k, v in out.items()}
    exp, ties = resolve_onset_ties(oracle_mod, m, p, np.arange(N), got, exp)
    fp32_report(m, with_gap(got, p, m), with_gap(exp, p, m), ties)
    assert ties[0] <= 3, ties

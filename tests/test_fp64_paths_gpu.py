"""The binary64 kernel's ways through a step -- r(D) held, one piece, the full
minimum -- give the oracle's bits where they meet: instantaneous and slow
actuators, dt / tau from well below 1 to past 2, saturated and unsaturated
roads, no grip, commands that brake hard, hardly, not at all or backwards,
trigger tests that are skipped and readings inside and outside the noise band,
and states beyond the range of the fused forms; in launches that leave the
integer pipes alone and in launches that use them."""
import numpy as np
import pytest

import aeb_inputs as ai

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def aeb():
    import paper_2604_27193_gb300 as m
    m.build()
    return m


MODELS = {
    "single": ai.single_model(4e-3),
    "lumped no lead": ai.replace(ai.paper_model(), dt=4e-3),
    "gentle command": ai.replace(ai.single_model(4e-3), a_cmd=-0.5),
    "hard command": ai.replace(ai.single_model(4e-3), a_cmd=-30.0),
    "no command": ai.replace(ai.single_model(4e-3), a_cmd=0.0),
    "forward command": ai.replace(ai.single_model(4e-3), a_cmd=2.0),
    "ttc": ai.ttc_model(2.0, 4e-3),
    "ttc negative threshold": ai.ttc_model(-0.5, 4e-3),
    "ttc readings": ai.replace(ai.ttc_model(1.5, 4e-3), perc_sigma=2.0, perc_drop=0.3,
                               perc_latency=0.1, perc_seed=5),
    "ttc moving lead": ai.replace(ai.lead_braking_model(dt=4e-3), trigger=ai.TRIGGER_TTC,
                                  ttc_thr=2.5),
    "coarse 0.5 s": ai.single_model(0.5),
}


def _params(m, seed):
    """Ordinary samples whose fields are stretched over the edges of the paths."""
    n = 1500
    rng = np.random.default_rng(seed)
    p = ai.draw_params(m, ai.scenario_from_means(25.0, 0.05, 0.95, 70.0, seed, 0), n)
    p["tau"] = rng.choice([0.0, 1e-3, 2e-3, 4e-3, 8e-3, 0.05, 0.2, 1.0, 30.0], n)
    p["t_delay"] = rng.choice([0.0, 0.004, 0.1, 0.5, 20.0], n)
    p["mu"][::37] = 0.0
    p["cd"][::41] = 0.0
    # 1 - mu h / L near, at and below zero
    p["mu"][5::53] = 1.0 / (m.h_cg / m.wheelbase)
    p["mu"][6::53] *= 9.0
    # beyond the fused forms: speed, drag, grade
    p["v0"][7::59] = rng.uniform(9e4, 2e5, len(p["v0"][7::59]))
    p["cd"][8::61] = 5e3
    p["gs"][9::67] = rng.uniform(-3e5, 3e5, len(p["gs"][9::67]))
    return p


@pytest.mark.parametrize("copies", [1, 45])  # 67,500 rollouts: software arithmetic too
@pytest.mark.parametrize("kind", list(MODELS))
def test_fp64_paths_bit_exact(aeb, oracle_mod, kind, copies):
    m = MODELS[kind]
    p = _params(m, 31)
    if kind == "ttc readings" and copies > 1:
        pytest.skip("a copy's readings are keyed by its own row")
    exp = {k: np.tile(v, copies) for k, v in oracle_mod.rollout(m, p).items()}
    p = {k: np.tile(v, copies) for k, v in p.items()}
    P = {f: torch.from_numpy(np.ascontiguousarray(p[f])).cuda() for f in ai.FIELDS}
    out = aeb.alloc_outputs(len(p["v0"]))
    aeb.aeb_rollout(m, P, len(p["v0"]), aeb.FP64_PLAIN, out)
    torch.cuda.synchronize()
    for k, v in out.items():
        got, want = v.cpu().numpy(), exp[k]
        if got.dtype == np.float64:  # a NaN is a NaN (an overflowed sample)
            nan = np.isnan(want)
            assert np.array_equal(nan, np.isnan(got)), k
            got, want = got[~nan].view(np.uint64), want[~nan].view(np.uint64)
        bad = np.nonzero(got != want)[0]
        assert len(bad) == 0, (k, len(bad), bad[:5])

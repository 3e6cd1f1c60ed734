"""Launches of a context that fsmp_autotune has tuned: it tunes the shape of a launch with a warp (or
half a warp) per chain, keeps the rule that gives a chain a team of four warps, and reports the
launch that the tuned batch then is."""
import numpy as np
import pytest

from paper_2403_03156_gb300 import fsmp, workloads
from tests import gpu_util

pytestmark = pytest.mark.gpu

UNEVEN, MIX, PILEUP = "batched_uneven_100k", "mcp_uneven_20k", "highpileup_20k_1024"


def _params(workload, **kw):
    return dict(workloads.CONFIGS[workload]["params"], **{**dict(precision=fsmp.FP32_REFRESH, refresh_every=16, pe_lanes=32,
                                                                 n_max=1024, n_streams=1), **kw})


def _device(workload, lam, seed=17):
    import torch
    cfg, lam = workloads.CONFIGS[workload], np.asarray(lam, float)
    rng = np.random.Generator(np.random.PCG64(seed))
    rule = ["trimmed"] if cfg["window"] == "trimmed" else ["uniform", 900, 1024]
    b = workloads.simulate(cfg["params"], lam, rng.uniform(30, 40, len(lam)), rng, *rule)[0]
    dev = torch.device("cuda", 0)
    d = {k: torch.from_numpy(np.ascontiguousarray(b[k])).to(dev) for k in ("samples", "offsets", "lambda0", "t_origin_ns")}
    d["out"] = torch.zeros(len(lam) * fsmp.SUMMARY_DTYPE.itemsize, dtype=torch.uint8, device=dev)
    return d


def _run(ctx, d, steps):
    import torch
    d["out"].zero_()
    ctx.run_device(d, n_steps=steps, burn_in=10, seed=9, n_max_hint=1024)
    torch.cuda.synchronize()
    return d["out"].cpu().numpy(), ctx.last_launch()


@pytest.mark.parametrize("workload,tuned_on,sample,launches", [
    # tuned on a bulk batch, on the heaviest few of one, and in steps that are too few for teams
    (UNEVEN, np.geomspace(50, 0.5, 6000), 6000, [((60, 40, 400), 400, 1), ((100, 0.5, 1300), 400, 1), ((8, 8, 1300), 200, 0)]),
    (UNEVEN, np.geomspace(50, 0.5, 6000), 300, [((60, 40, 400), 400, 1), ((8, 8, 1300), 200, 0), ((2, 0.5, 6000), 200, 0)]),
    (MIX, np.geomspace(50, 0.5, 5000), 500, [((100, 0.5, 1300), 400, 1), ((15, 5, 1300), 200, 0), ((15, 5, 5000), 200, 0)]),
    (PILEUP, np.geomspace(200, 100, 1300), 1300, [((200, 100, 1300), 600, 1), ((5, 0.5, 1300), 200, 0)])])
def test_a_tuned_context_keeps_the_rule_for_teams(workload, tuned_on, sample, launches):
    """The form of each later launch, whatever its size, is the one an untuned context takes, and so
    are its bits."""
    pytest.importorskip("torch")
    p = _params(workload, n_cap=384 if workload == PILEUP else 128)
    with gpu_util.context(p) as ctx, gpu_util.context(p) as plain:
        tune = ctx.autotune(_device(workload, tuned_on), sample=sample, trial_steps=128, seed=9, n_max_hint=1024)
        print("tuned:", tune)
        assert tune["default_steps_per_s"] > 0 and tune["best_steps_per_s"] >= tune["default_steps_per_s"]
        for lam, steps, team in launches:
            d = _device(workload, np.geomspace(*lam))
            a, la = _run(ctx, d, steps)
            b, lb = _run(plain, d, steps)
            assert la["team"] == lb["team"] == team, (lam, la, lb)
            np.testing.assert_array_equal(a, b)


@pytest.mark.parametrize("workload,lam,kw", [
    (UNEVEN, (30, 0.5, 900), dict(precision=fsmp.FP64)),      # no team: FP64,
    (UNEVEN, (10, 0.5, 900), dict(n_cap=24)),                 # a small capacity,
    (UNEVEN, (60, 0.5, 500), dict(threads_per_chain=64)),     # a given shape
    (UNEVEN, (60, 0.5, 500), dict(pe_ctas_per_sm=2)),
    (UNEVEN, (20, 0.5, 6000), dict()),                        # a bulk batch
    (UNEVEN, (60, 30, 500), dict()),                          # a batch in teams
    (UNEVEN, (60, 30, 500), dict(pe_lanes=0)),
    (MIX, (15, 5, 7000), dict()),
    (PILEUP, (200, 100, 700), dict(n_cap=384))])
def test_the_report_is_the_launch(workload, lam, kw):
    pytest.importorskip("torch")
    d = _device(workload, np.geomspace(*lam))
    with gpu_util.context(_params(workload, **{**dict(n_cap=128), **kw})) as ctx:
        tune = ctx.autotune(d, sample=300, trial_steps=300, seed=9, n_max_hint=1024)
        _, l = _run(ctx, d, 300)
    print("tuned:", tune, "launched:", l)
    assert {k: tune[k] for k in ("lanes_per_chain", "chains_per_cta", "pe_tile")} == \
        {k: l[k] for k in ("lanes_per_chain", "chains_per_cta", "pe_tile")}
    if kw and "n_cap" not in kw and "pe_lanes" not in kw or kw.get("n_cap") == 24:
        assert l["team"] == 0


def test_a_default_shape_that_has_to_shrink_is_timed():
    """Windows at which four chains of the default tile do not fit an SM's shared memory: the default
    launch takes a smaller shape, which the report rates."""
    pytest.importorskip("torch")
    p = _params(PILEUP, precision=fsmp.FP64, n_cap=384, grid_ns=1.0, n_max=3000)
    d = _device(PILEUP, np.geomspace(5, 0.5, 200))
    with gpu_util.context(p) as ctx:
        hint = 3000
        while hint > 1024:  # the longest window that is taken, to 64 samples
            try:
                ctx.run_device(d, n_steps=2, burn_in=1, seed=9, n_max_hint=hint)
                break
            except fsmp.FsmpError:
                hint -= 64
        l = ctx.last_launch()
        assert (l["pe_tile"], l["chains_per_cta"]) != (40, 4)
        tune = ctx.autotune(d, sample=200, trial_steps=30, seed=9, n_max_hint=hint)
    print("hint:", hint, "launched:", l, "tuned:", tune)
    assert tune["default_steps_per_s"] > 0 and tune["n_tried"] >= 2


def test_a_captured_launch_chooses_its_form_at_each_replay():
    """1300 chains, beyond those that are all resident as teams: the form is chosen on the device, so
    a graph captured on light chains runs in teams once its lambda0 are heavy, and the other way round."""
    torch = pytest.importorskip("torch")
    p = _params(UNEVEN, n_cap=128)
    heavy, light = np.geomspace(100, 0.5, 1300), np.full(1300, 2.0)
    d = _device(UNEVEN, heavy)
    with gpu_util.context(p) as ctx:
        want = {}
        for lam, team in ((heavy, 1), (light, 0)):
            d["lambda0"].copy_(torch.from_numpy(lam))
            want[team], launch = _run(ctx, d, 400)
            assert launch["team"] == team
        side, graph = torch.cuda.Stream(), torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=side):
            ctx.run_device(d, n_steps=400, burn_in=10, seed=9, n_max_hint=1024, stream=side)
        for lam, team in ((light, 0), (heavy, 1), (light, 0)):
            d["lambda0"].copy_(torch.from_numpy(lam))
            d["out"].zero_()
            graph.replay()
            torch.cuda.synchronize()
            assert ctx.last_launch()["team"] == team
            np.testing.assert_array_equal(d["out"].cpu().numpy(), want[team])

"""The forms of a PE-space launch -- a warp per chain, or a team of four warps per chain -- and which
of them ran (fsmp_last_launch). A form keeps every operation and the order of every sum, so all
outputs are equal bit for bit."""
import numpy as np
import pytest

from paper_2403_03156_gb300 import fsmp, workloads
from tests import gpu_util

pytestmark = pytest.mark.gpu

ONE_WARP = dict(threads_per_chain=128)


def _simulate(workload, lam, seed=17):
    cfg = workloads.CONFIGS[workload]
    rng = np.random.Generator(np.random.PCG64(seed))
    W = len(lam)
    rule = ["trimmed"] if cfg["window"] == "trimmed" else ["uniform", 900, 1024]
    return workloads.simulate(cfg["params"], np.asarray(lam, float), rng.uniform(30, 40, W), rng, *rule)[0]


def _run(params, b, steps, burn=10, lucy=False, trace=False, z=None):
    import torch
    dev, W = torch.device("cuda", 0), len(b["lambda0"])
    d = {k: torch.from_numpy(np.ascontiguousarray(b[k])).to(dev) for k in ("samples", "offsets", "lambda0", "t_origin_ns")}
    d["out"] = torch.zeros(W * fsmp.SUMMARY_DTYPE.itemsize, dtype=torch.uint8, device=dev)
    d["pe_hist"] = torch.zeros((W, 256), dtype=torch.int32, device=dev)
    if trace:
        d["trace"] = torch.zeros(W * steps * fsmp.TRACE_DTYPE.itemsize, dtype=torch.uint8, device=dev)
    if z is not None:
        d.update(z_init=torch.from_numpy(z).to(dev), n_init=torch.full((W,), z.shape[1], dtype=torch.int32, device=dev))
    with gpu_util.context(params) as ctx:
        if lucy:
            s = ctx.lucyddm(d, n_iter=300, n_max_hint=params["n_max"])
            d.update({k: s[k] for k in ("T_lo", "T_hi", "t0_init", "z_init", "n_init")})
        ctx.run_device(d, n_steps=steps, burn_in=burn, seed=9, n_max_hint=params["n_max"])
        torch.cuda.synchronize(dev)
        launch = ctx.last_launch()
    out = [d[k].cpu().numpy() for k in ("out", "pe_hist", "trace") if k in d]
    return out, launch


@pytest.mark.parametrize("lam", [[75.0], list(np.linspace(45.0, 75.0, 37))])
@pytest.mark.parametrize("lucy", [False, True])
@pytest.mark.parametrize("workload,n_cap,steps", [("batched_uneven_100k", 128, 700), ("mcp_uneven_20k", 128, 700),
                                                  ("batched_uneven_100k", 64, 500), ("highpileup_20k_1024", 384, 500)])
def test_a_team_runs_and_gives_the_bits_of_one_warp(workload, n_cap, steps, lucy, lam):
    """Chains beyond 32 PEs (where a team's passes start) and 40 (where C^-1 leaves shared memory)."""
    pytest.importorskip("torch")
    p = dict(workloads.CONFIGS[workload]["params"], n_cap=n_cap, precision=fsmp.FP32_REFRESH, refresh_every=8, pe_lanes=32,
             n_max=1024, n_streams=1)
    b = _simulate(workload, lam)
    team, l_team = _run(p, b, steps, lucy=lucy, trace=True)
    warp, l_warp = _run(dict(p, **ONE_WARP), b, steps, lucy=lucy, trace=True)
    assert (l_team["team"], l_team["chains_per_cta"]) == (1, 1)
    assert (l_warp["team"], l_warp["chains_per_cta"]) == (0, 4)
    N = fsmp.traces_from_bytes(team[2], len(lam))["N"].max(1)
    assert np.all(N > 32) and N.max() > 40, N
    for a, c in zip(team, warp):
        np.testing.assert_array_equal(a, c)


@pytest.mark.parametrize("workload,n_cap", [("batched_uneven_100k", 128), ("mcp_uneven_20k", 128),
                                            ("highpileup_20k_1024", 384)])
def test_a_rebuild_that_fails_in_a_team(workload, n_cap):
    """An initial state of 40 PEs at one grid point and next to no noise: C has rank one to FP64
    rounding, the rebuild's inversion meets a pivot that is not positive, every warp of the team
    leaves it, and the chain starts empty with the status that one warp reports."""
    pytest.importorskip("torch")
    p = dict(workloads.CONFIGS[workload]["params"], n_cap=n_cap, precision=fsmp.FP32_REFRESH, refresh_every=1,
             sigma_noise=1e-9, n_max=1024, n_streams=1)
    b = _simulate(workload, [3.0, 20.0, 60.0])
    z = np.full((3, 40), 160, np.int32)
    team, l_team = _run(p, b, 40, z=z)
    warp, l_warp = _run(dict(p, **ONE_WARP), b, 40, z=z)
    assert l_team["team"] == 1 and l_warp["team"] == 0
    assert np.all(team[0].view(fsmp.SUMMARY_DTYPE)["status"] & fsmp.ST_BADDET)
    for a, c in zip(team, warp):
        np.testing.assert_array_equal(a, c)


def test_no_launch_yet():
    with gpu_util.context(dict(workloads.CONFIGS["plain_fp64_256x128"]["params"], n_max=128, n_streams=1)) as ctx:
        with pytest.raises(fsmp.FsmpError) as e:
            ctx.last_launch()
    assert e.value.code == fsmp.ERR_INVALID


@pytest.mark.parametrize("workload,n_cap,lam,steps,team", [
    ("batched_uneven_100k", 128, (8.0, 8.0), 200, 0),     # light: a warp per chain
    ("batched_uneven_100k", 128, (0.2, 2.0), 200, 0),
    ("batched_uneven_100k", 64, (0.2, 2.0), 200, 0),
    ("batched_uneven_100k", 128, (0.5, 100.0), 400, 1),   # a tail of heavy chains: teams
    ("mcp_uneven_20k", 128, (5.0, 15.0), 200, 0),
    ("mcp_uneven_20k", 128, (0.5, 100.0), 400, 1),
    ("highpileup_20k_1024", 384, (0.5, 5.0), 200, 0),
    ("highpileup_20k_1024", 384, (100.0, 200.0), 600, 1)])
def test_the_form_follows_the_chains(workload, n_cap, lam, steps, team):
    """1300 chains, more than the GPU holds as teams: the form follows their lambda0 and steps, on the
    device-resident path and from host memory alike; a lambda0 that is not a number spoils its own
    chain only; and the outputs are those of one warp per chain."""
    pytest.importorskip("torch")
    W = 1300
    p = dict(workloads.CONFIGS[workload]["params"], n_cap=n_cap, precision=fsmp.FP32_REFRESH, refresh_every=16, pe_lanes=32,
             n_max=1024, n_streams=1)
    b = _simulate(workload, np.geomspace(lam[1], lam[0], W))
    b["lambda0"][7] = np.nan
    got, launch = _run(p, b, steps)
    ref, _ = _run(dict(p, **ONE_WARP), b, steps)
    assert launch["team"] == team and launch["chains_per_cta"] == (1 if team else 4)
    assert np.array_equal(np.nonzero(got[0].view(fsmp.SUMMARY_DTYPE)["status"] & fsmp.ST_INVALID)[0], [7])
    for a, c in zip(got, ref):
        np.testing.assert_array_equal(a, c)
    host = dict(b, lambda0=np.where(np.isnan(b["lambda0"]), lam[0], b["lambda0"]), n_steps=steps, burn_in=10, seed=9, index_base=0)
    for k in ("T_lo", "T_hi", "wf_ids"):
        host.pop(k, None)
    with gpu_util.context(p) as ctx:
        s, _ = ctx.run(host)
        assert ctx.last_launch()["team"] == team
    others = np.arange(W) != 7
    assert s[others].tobytes() == got[0].view(fsmp.SUMMARY_DTYPE)[others].tobytes()


def test_short_chains_take_no_team():
    """A chain of 100 steps does not get far beyond 20 PEs, whatever its lambda0."""
    pytest.importorskip("torch")
    for workload, n_cap in (("batched_uneven_100k", 128), ("highpileup_20k_1024", 384)):
        p = dict(workloads.CONFIGS[workload]["params"], n_cap=n_cap, precision=fsmp.FP32_REFRESH, n_max=1024, n_streams=1)
        assert _run(p, _simulate(workload, np.full(1300, 60.0)), 100)[1]["team"] == 0

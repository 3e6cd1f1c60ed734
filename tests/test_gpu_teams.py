"""Chains run by a team of four warps (the default for launches of few chains) against the same
chains on one warp each: the team splits passes over C^-1 and the FP64 rebuild, and keeps every
operation and the order of every sum, so the summaries are equal bit for bit. Chains here grow
through 32 PEs (where the team starts) and 40 (where C^-1 leaves shared memory) and shrink again,
start empty or from a given state, and are rebuilt often."""
import numpy as np
import pytest

from paper_2403_03156_gb300 import fsmp, workloads
from tests import gpu_util

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_waveforms", [1, 37])
@pytest.mark.parametrize("start", ["empty", "lucyddm"])
@pytest.mark.parametrize("workload,lam,n_cap,steps", [("batched_uneven_100k", (25.0, 75.0), 128, 700),
                                                      ("mcp_uneven_20k", (25.0, 75.0), 128, 700),
                                                      ("batched_uneven_100k", (31.0, 36.0), 64, 400),
                                                      ("highpileup_20k_1024", (60.0, 200.0), 384, 500)])
def test_a_team_gives_the_bits_of_one_warp(workload, lam, n_cap, steps, start, n_waveforms):
    torch = pytest.importorskip("torch")
    dev = torch.device("cuda", 0)
    cfg = workloads.CONFIGS[workload]
    p = dict(cfg["params"], n_cap=n_cap, precision=fsmp.FP32_REFRESH, refresh_every=8, pe_lanes=32, n_max=1024, n_streams=1)
    rng = np.random.Generator(np.random.PCG64(17))
    W = n_waveforms
    kind = "trimmed" if cfg["window"] == "trimmed" else "uniform"
    b, _ = workloads.simulate(p, np.linspace(lam[0], lam[1], W), rng.uniform(30, 40, W), rng, kind, *([] if kind == "trimmed" else [900, 1024]))
    got = []
    for shape in (dict(), dict(threads_per_chain=128)):
        d = {k: torch.from_numpy(np.ascontiguousarray(b[k])).to(dev) for k in ("samples", "offsets", "lambda0", "t_origin_ns")}
        d["out"] = torch.zeros(W * fsmp.SUMMARY_DTYPE.itemsize, dtype=torch.uint8, device=dev)
        d["pe_hist"] = torch.zeros((W, 256), dtype=torch.int32, device=dev)
        with gpu_util.context(dict(p, **shape)) as ctx:
            if start == "lucyddm":
                s = ctx.lucyddm(d, n_iter=300, n_max_hint=1024)
                d.update({k: s[k] for k in ("T_lo", "T_hi", "t0_init", "z_init", "n_init")})
            ctx.run_device(d, n_steps=steps, burn_in=10, seed=9, n_max_hint=1024)
            torch.cuda.synchronize(dev)
        got.append((d["out"].cpu().numpy(), d["pe_hist"].cpu().numpy()))
    top = got[0][0].view(fsmp.SUMMARY_DTYPE)["N_final"].max()
    assert top > (20 if W > 1 and steps >= 500 else 0)  # a team had work to do
    np.testing.assert_array_equal(got[0][0], got[1][0])
    np.testing.assert_array_equal(got[0][1], got[1][1])

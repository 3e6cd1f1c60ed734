"""The default launch shape holds as many chains on an SM as the smaller tile of C^-1 (32 PEs)
allows: a larger tile is for contexts where it takes no chain's place."""
import numpy as np
import pytest

from paper_2403_03156_gb300 import fsmp, workloads
from tests import gpu_util

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("workload,n_cap,n_max,precision", [
    ("highpileup_20k_1024", 384, 1024, fsmp.FP32_REFRESH), ("highpileup_20k_1024", 384, 1024, fsmp.FP64),
    ("batched_uneven_100k", 64, 2000, fsmp.FP32_REFRESH), ("batched_uneven_100k", 128, 400, fsmp.FP64),
    ("batched_uneven_100k", 64, 1024, fsmp.FP64), ("mcp_uneven_20k", 128, 1024, fsmp.FP32_REFRESH),
    ("batched_uneven_100k", 36, 512, fsmp.FP32_REFRESH)])
def test_the_default_tile_keeps_no_chain_out(workload, n_cap, n_max, precision):
    p = dict(workloads.CONFIGS[workload]["params"], n_cap=n_cap, n_max=n_max, precision=precision, n_streams=1)
    with gpu_util.context(p) as free, gpu_util.context(dict(p, pe_tile=32)) as small:
        assert free.info()["ctas_per_sm"] >= small.info()["ctas_per_sm"] >= 1


@pytest.mark.parametrize("n_cap,n_waveforms,per_sm", [(128, 7000, 3), (48, 2000, 3), (128, 3500, 2)])
def test_mixture_chains_per_sm(n_cap, n_waveforms, per_sm):
    """Three CTAs of mixture chains on an SM where the launch fills the SMs many times over or n_cap is
    small, else two; their outputs are the same bit for bit."""
    torch = pytest.importorskip("torch")
    dev = torch.device("cuda", 0)
    cfg = workloads.CONFIGS["mcp_uneven_20k"]
    p = dict(cfg["params"], n_cap=n_cap, n_max=512, precision=fsmp.FP32_REFRESH, refresh_every=16, pe_lanes=32, n_streams=1)
    rng = np.random.Generator(np.random.PCG64(23))
    b, _ = workloads.simulate(p, np.geomspace(50.0 if n_cap > 100 else 20.0, 0.5, n_waveforms), rng.uniform(30, 40, n_waveforms), rng, "trimmed")
    got = []
    for shape in (dict(threads_per_chain=128), dict(pe_ctas_per_sm=2), dict(pe_ctas_per_sm=3)):
        d = {k: torch.from_numpy(np.ascontiguousarray(b[k])).to(dev) for k in ("samples", "offsets", "lambda0", "t_origin_ns")}
        d["out"] = torch.zeros(n_waveforms * fsmp.SUMMARY_DTYPE.itemsize, dtype=torch.uint8, device=dev)
        with gpu_util.context(dict(p, **shape)) as ctx:
            ctx.run_device(d, n_steps=120, burn_in=20, seed=9, n_max_hint=512)
            torch.cuda.synchronize(dev)
            ctas = ctx.last_launch()["ctas"]
            assert ctas == ctx.info()["sm_count"] * shape.get("pe_ctas_per_sm", per_sm)
        got.append(d["out"].cpu().numpy())
    for other in got[1:]:
        np.testing.assert_array_equal(got[0], other)


@pytest.mark.parametrize("n_waveforms,tile", [(2600, 40), (4000, 32)])
def test_the_smaller_tile_is_for_launches_of_many_chains(n_waveforms, tile):
    """16 lanes per chain and n_cap 128: an SM holds one CTA (8 chains) with the tile of 40, two with 32,
    which a launch takes from 2.5 chains per resident one on (3040 on 152 SMs). The outputs are the
    same bit for bit."""
    torch = pytest.importorskip("torch")
    dev = torch.device("cuda", 0)
    cfg = workloads.CONFIGS["batched_uneven_100k"]
    p = dict(cfg["params"], n_cap=128, n_max=512, precision=fsmp.FP32_REFRESH, refresh_every=16, pe_lanes=16, n_streams=1)
    rng = np.random.Generator(np.random.PCG64(29))
    b, _ = workloads.simulate(p, np.geomspace(45.0, 0.5, n_waveforms), rng.uniform(30, 40, n_waveforms), rng, "trimmed")
    got = []
    for shape in (dict(), dict(pe_tile=32), dict(pe_tile=40)):
        d = {k: torch.from_numpy(np.ascontiguousarray(b[k])).to(dev) for k in ("samples", "offsets", "lambda0", "t_origin_ns")}
        d["out"] = torch.zeros(n_waveforms * fsmp.SUMMARY_DTYPE.itemsize, dtype=torch.uint8, device=dev)
        with gpu_util.context(dict(p, **shape)) as ctx:
            ctx.run_device(d, n_steps=250, burn_in=20, seed=9, n_max_hint=512)
            torch.cuda.synchronize(dev)
            assert ctx.last_launch()["pe_tile"] == shape.get("pe_tile", tile)
        got.append(d["out"].cpu().numpy())
    for other in got[1:]:
        np.testing.assert_array_equal(got[0], other)

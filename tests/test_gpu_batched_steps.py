"""The PE-space kernel's batches of steps scored ahead of their turn, where they can go wrong: chains
that cross the batch's limit of 32 PEs, that sit at a small capacity or at N = 0, chains of a few
steps, lists of steps cut by the end of the chain or of a draw block -- step by step against the
oracle in FP64 mode (log acceptance ratios to 1e-9, as the other lockstep tests). And the launch
shapes: the default one and given ones run the same arithmetic, so their summaries are equal bit
for bit."""
import numpy as np
import pytest

from paper_2403_03156_gb300 import fsmp, workloads
from tests import gpu_util

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lib():
    from paper_2403_03156_gb300 import build
    build.build()
    return fsmp.load()


@pytest.fixture(scope="module")
def orc():
    from oracle import oracle
    oracle.build()
    return oracle


@pytest.mark.parametrize("lanes", [32, 16])
@pytest.mark.parametrize("lam,n_cap,steps", [(34.0, 128, 420), (3.0, 4, 200), (0.05, 24, 67), (2.0, 24, 1), (2.0, 24, 3),
                                             (6.0, 33, 34)])
def test_batches_in_lockstep_with_the_oracle(lib, orc, lam, n_cap, steps, lanes):
    cfg = workloads.CONFIGS["batched_uneven_100k"]
    params = dict(cfg["params"], n_cap=n_cap, precision=fsmp.FP64, pe_lanes=lanes, n_max=512)
    rng = np.random.Generator(np.random.PCG64(61))
    W = 6
    batch, _ = workloads.simulate(params, np.full(W, lam), rng.uniform(30, 40, W), rng, "trimmed")
    batch.update(seed=5, index_base=0, n_steps=steps, burn_in=steps // 4)
    with gpu_util.context(params) as ctx:
        s_gpu, t_gpu = ctx.run(batch, record_trace=True)
    s_orc, t_orc = orc.run_batch(params, batch, orc.MODE_DEFINITION, n_threads=6, trace=True)
    gpu_util.compare_traces(t_gpu, t_orc)
    for f in ("acc", "prop", "acc_t0", "prop_t0", "N_final", "k0_final", "status"):
        np.testing.assert_array_equal(s_gpu[f], s_orc[f], err_msg=f)
    for f in ("mean_N", "var_N", "mean_t0", "mean_wt"):
        np.testing.assert_allclose(s_gpu[f], s_orc[f], rtol=1e-9, atol=1e-9, err_msg=f)


@pytest.mark.parametrize("n_waveforms", [1, 153, 700])
@pytest.mark.parametrize("workload,lanes", [("batched_uneven_100k", 32), ("lowocc_bulk_1m", 16), ("mcp_uneven_20k", 32),
                                            ("highpileup_20k_1024", 32)])
def test_launch_shapes_give_the_same_bits(lib, workload, lanes, n_waveforms):
    torch = pytest.importorskip("torch")
    steps = 60 if workload == "highpileup_20k_1024" else 120
    wl = workloads.make_workload(workload, n_waveforms=n_waveforms, seed=4)
    b, dev = wl["batch"], torch.device("cuda", 0)
    got = []
    for shape in (dict(), dict(threads_per_chain=128), dict(pe_tile=8, threads_per_chain=32),
                  dict(pe_ctas_per_sm=1, pe_tile=24)):
        params = dict(wl["params"], precision=fsmp.FP32_REFRESH, refresh_every=16, pe_lanes=lanes,
                      n_max=int(np.diff(b["offsets"]).max()), n_streams=1, **shape)
        d = {k: torch.from_numpy(np.ascontiguousarray(b[k])).to(dev)
             for k in ("samples", "offsets", "lambda0", "t_origin_ns", "T_lo", "T_hi") if k in b}
        d["out"] = torch.zeros(n_waveforms * fsmp.SUMMARY_DTYPE.itemsize, dtype=torch.uint8, device=dev)
        with gpu_util.context(params) as ctx:
            ctx.run_device(d, n_steps=steps, burn_in=10, seed=9)
            torch.cuda.synchronize(dev)
        got.append(d["out"].cpu().numpy())
    for other in got[1:]:
        np.testing.assert_array_equal(got[0], other)

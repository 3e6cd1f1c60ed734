"""The longest window a PE-space context takes is set when it is created: tuning on short windows
does not change what is refused, and a window at the limit runs in the tuned context in a shape that
fits, with the bits of an explicit small one."""
import numpy as np
import pytest

from paper_2403_03156_gb300 import fsmp, workloads
from tests import gpu_util

pytestmark = pytest.mark.gpu


def _batch(params, W, samples, seed):
    rng = np.random.Generator(np.random.PCG64(seed))
    return workloads.simulate(params, np.geomspace(2.0, 0.2, W), rng.uniform(30, 40, W), rng, "fixed", fixed_window=samples)[0]


def _device(b):
    import torch
    dev = torch.device("cuda", 0)
    d = {k: torch.from_numpy(np.ascontiguousarray(b[k])).to(dev) for k in ("samples", "offsets", "lambda0", "t_origin_ns")}
    d["out"] = torch.zeros(len(b["lambda0"]) * fsmp.SUMMARY_DTYPE.itemsize, dtype=torch.uint8, device=dev)
    return d


def _run(ctx, d, hint):
    import torch
    ctx.run_device(d, n_steps=60, burn_in=10, seed=3, n_max_hint=hint)
    torch.cuda.synchronize()
    return d["out"].cpu().numpy()


def _accepts(ctx, d, hint):
    try:
        _run(ctx, d, hint)
        return True
    except fsmp.FsmpError as e:
        assert e.code == fsmp.ERR_INVALID
        return False


def _longest(p):
    """The parameters with the largest n_max, to 64 samples, that fsmp_create takes."""
    for n_max in range(8192, 0, -64):
        try:
            gpu_util.context(dict(p, n_max=n_max)).close()
            return dict(p, n_max=n_max)
        except fsmp.FsmpError:
            pass


@pytest.mark.parametrize("precision,n_cap", [(fsmp.FP32_REFRESH, 192), (fsmp.FP64, 24), (fsmp.FP64, 192)])
def test_tuning_leaves_the_window_limit(precision, n_cap):
    pytest.importorskip("torch")
    p = _longest(dict(workloads.CONFIGS["lowocc_bulk_1m"]["params"], grid_ns=1.0, precision=precision, n_cap=n_cap,
                      refresh_every=16, n_streams=1))
    few, many = _device(_batch(p, 5, 128, 1)), _device(_batch(p, 20000, 128, 2))
    with gpu_util.context(p) as ctx:
        lo, hi = 128, p["n_max"] + 1  # lo is taken, hi is not
        while hi - lo > 1:
            mid = (lo + hi) // 2
            lo, hi = (mid, hi) if _accepts(ctx, few, mid) else (lo, mid)
        tune = ctx.autotune(many, sample=20000, trial_steps=200, seed=3, n_max_hint=128)
        print("tuned:", tune, "longest window:", lo, "n_max:", p["n_max"])
        at_limit = _device(_batch(p, 5, lo, 4))
        assert lo == p["n_max"] or not _accepts(ctx, few, lo + 1)
        got = _run(ctx, at_limit, lo)
    assert not np.any(got.view(fsmp.SUMMARY_DTYPE)["status"] & (fsmp.ST_INVALID | fsmp.ST_BADDET | fsmp.ST_NONFINITE))
    with gpu_util.context(dict(p, pe_lanes=tune["lanes_per_chain"], threads_per_chain=32, pe_tile=8)) as ctx:
        np.testing.assert_array_equal(got, _run(ctx, at_limit, lo))


def test_windows_that_no_launch_takes_are_not_tuned_on():
    pytest.importorskip("torch")
    p = dict(workloads.CONFIGS["highpileup_20k_1024"]["params"], grid_ns=1.0, precision=fsmp.FP64, n_max=3000, n_streams=1)
    few = _device(_batch(p, 5, 128, 1))
    with gpu_util.context(p) as ctx:
        assert not _accepts(ctx, few, 3000)
        before = _run(ctx, few, 128), ctx.last_launch()
        tune = ctx.autotune(few, sample=5, trial_steps=20, seed=3, n_max_hint=3000)
        assert (tune["n_tried"], tune["best_steps_per_s"], tune["default_steps_per_s"]) == (0, -1.0, -1.0)
        after = _run(ctx, few, 128), ctx.last_launch()
    np.testing.assert_array_equal(before[0], after[0])
    assert before[1] == after[1]

"""The default launch shape holds as many chains on an SM as the smaller tile of C^-1 (32 PEs)
allows: a larger tile is for contexts where it takes no chain's place."""
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

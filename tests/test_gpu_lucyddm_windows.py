"""The LucyDDM kernel over window lengths and responses that take each of its splits (4 to 8 outputs
a lane in one or more passes, whole and remaining blocks of taps): q-hat after three iterations
against the same iterations in FP64. All terms are positive, so a correlation of L_V terms is off by
at most (L_V + 2) u relative (u = 2^-24); q-hat takes its own error and the ratio's, which is w^r's:
e <- 2 e + 2 (L_V + 2) u, 14 (L_V + 2) u after three iterations from an exact start to one rounding."""
import numpy as np
import pytest

from paper_2403_03156_gb300 import fsmp
from tests import gpu_util

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ser", [dict(), dict(ser_sigma=0.4, ser_tau=1.0), dict(ser_sigma=2.0, ser_tau=9.5)])
@pytest.mark.parametrize("lengths", [range(1, 40, 3), range(60, 200, 9), (255, 256, 257, 320, 447, 448, 511, 512),
                                     (700, 1024, 2000)])
def test_q_hat_of_every_split(ser, lengths):
    torch = pytest.importorskip("torch")
    lengths = np.array(list(lengths))
    rng = np.random.default_rng(17)
    off = np.concatenate([[0], np.cumsum(lengths)]).astype(np.int32)
    samples = np.abs(rng.normal(0.0, 0.3, int(off[-1]))).astype(np.float32)
    samples[rng.random(len(samples)) < 0.2] = -0.1
    dev = torch.device("cuda", 0)
    with gpu_util.context(dict(n_max=int(lengths.max()), precision=fsmp.FP32_REFRESH, n_streams=1, **ser)) as ctx:
        V = ctx.tables()[0][::ctx.info()["R"]]
        got = ctx.lucyddm({"samples": torch.from_numpy(samples).to(dev), "offsets": torch.from_numpy(off).to(dev)},
                          n_iter=3, with_q=True)["q"].cpu().numpy().astype(np.float64)
    S, LV = V.sum(), len(V)
    tol = 14 * (LV + 2) * 2.0 ** -24
    for i, n in enumerate(lengths):
        d = np.maximum(samples[off[i]:off[i + 1]].astype(np.float64), 0.0) / S
        q = np.full(n + LV - 1, d.sum() / (n + LV - 1))
        for _ in range(3):
            wr = np.convolve(q, V / S)[LV - 1:LV - 1 + n]
            r = np.where(wr > 0, d / np.where(wr > 0, wr, 1.0), 0.0)
            q = q * np.convolve(r, (V / S)[::-1])
        at = off[i] + i * (LV - 1)
        np.testing.assert_allclose(got[at:at + n + LV - 1], q, rtol=tol, atol=1e-30, err_msg="n = %d" % n)

"""The stored run-time model describes the present kernels: predicted against
measured census times of graphs that it was not fitted to."""
import numpy as np
import pytest

import graphgen as gg
from paper_1610_09411_gb300 import predict as pr

pytestmark = pytest.mark.gpu


def test_predictions_follow_the_kernels():
    """Held out, the fit is off by a fifth in the median; half as much again on
    other graphs and an idle machine still tells it from kernels of twice the speed."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    torch.cuda.set_device(0)
    graphs = [gg.erdos_renyi(3000, 0.006, 71), gg.erdos_renyi(1200, 0.25, 72), gg.barabasi_albert(60000, 5, 73),
              gg.chung_lu(90000, 2.1, 14, 8192, 74), gg.chung_lu(200000, 2.3, 12, 8192, 75),
              gg.chung_lu(40000, 2.1, 18, 8192, 76), gg.config_rmat(15, 77), gg.config_rmat(17, 78)]
    p = pr.Predictor()
    off = [p.seconds(s) / s["seconds"] - 1 for s in pr.measure(graphs)]
    print([round(x, 2) for x in off])
    assert np.median(np.abs(off)) <= 0.35

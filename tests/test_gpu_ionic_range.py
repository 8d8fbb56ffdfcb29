"""Bueno-Orovio gates far from the smoothed steps, with long time constants and
steep steps: the rates stay those of the model (a rate behind a step that is fully
off is 1/tau). Where time constants of very different size cancel to 0/0 in the
model's formula, the oracle has no value and none is compared. Tolerance: a few
roundings per rate."""
import numpy as np
import pytest

from oracle import monodomain as omd
from paper_2602_16312_gb300 import workloads as W

from gpu_util import rel

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("tau2p,tau2pp", [(0.06, 0.015), (3e4, 1e4), (1e5, 3e5), (1e250, 1e5)])
@pytest.mark.parametrize("k", [1.0, 65.0, 4000.0])
def test_gate_rates_far_from_the_steps(tau2p, tau2pp, k):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2602_16312_gb300 import aggmg, build
    build.build()
    p = dict(W.BUENO_OROVIO, tau2p=tau2p, tau2pp=tau2pp, k2=k, k3=k)
    n = 2001
    u = np.linspace(-90.0, 40.0, n)
    w = np.random.default_rng(3).uniform(0.0, 1.0, (3, n))
    dt = 0.25 * min(tau2p, tau2pp)
    wd = torch.tensor(w.reshape(-1), device="cuda")
    aggmg.ionic_update(p, dt, torch.tensor(u, device="cuda"), wd)
    torch.cuda.synchronize()
    got = wd.cpu().numpy().reshape(3, n)
    with np.errstate(invalid="ignore", divide="ignore"):
        _, H = omd.ionic(p, u, w)
    for g in range(3):
        ref = w[g] + dt * H[g]
        has = np.isfinite(ref)
        assert has.sum() > n // 2 and rel(got[g][has], ref[has]) <= 1e-13, g

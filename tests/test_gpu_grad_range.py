"""The gradient is linear in dL/dE over magnitudes far from 1, at angles whose
rounds carry a large scale."""
import numpy as np
import pytest
import torch

from oracle import oracle as orc
from paper_2603_02804_gb300 import build as qbuild
from paper_2603_02804_gb300 import workloads
from paper_2603_02804_gb300.torch_api import Simulator

pytestmark = pytest.mark.gpu
PI = np.pi
SCALES = [1.0, -1e-12, 1e-24, -1e-28, 1e-100, 1e25]  # one per sample, in turn


@pytest.fixture(scope="module", autouse=True)
def built():
    qbuild.build()
    orc.build()


# threads per tile 8 to 256, one and two per column, several tiles per CTA; several tiles per sample; passes that seed
# from other tiles; RX items
@pytest.mark.parametrize("near", [PI - 0.009, PI - 0.1, None])
@pytest.mark.parametrize("n,d,B,obs,ansatz", [(7, 3, 6, "ZX", "hea"), (7, 3, 2500, "ZX", "hea"), (8, 3, 1300, "Z", "xyz"),
                                              (9, 3, 660, "ZX", "hea"), (11, 2, 162, "Z", "hea"), (12, 3, 6, "ZX", "hea"),
                                              (12, 2, 160, "Z", "xyz"), (13, 3, 6, "ZX", "hea"), (13, 3, 6, "X" * 13, "xyz")])
def test_gradient_is_linear_in_dLdE(n, d, B, obs, ansatz, near):
    """Per sample, the gradient over dL/dE against the oracle's at dL/dE = 1: the
    parity tests' 1e-5, as a power-of-two scale changes no digit."""
    rng = np.random.default_rng(n + B)
    P = 3 * n * d
    theta = rng.uniform(0, 2 * PI, P) if near is None else near + rng.uniform(-1e-4, 1e-4, P)
    theta = theta.astype(np.float32)
    x = rng.uniform(0, PI, (B, n)).astype(np.float32)
    if ansatz == "hea":
        sim, circ = Simulator(n, d, B, obs=obs), orc.hea(n, d)
    else:
        rows = workloads.xyz_ring_gates(n, d)
        sim, circ = Simulator(n, 0, B, gates=rows, n_params=P, obs=obs), orc.Circuit(n=n, gates=np.array(rows, np.int32), n_params=P)
    dl = np.array([SCALES[b % len(SCALES)] for b in range(B)])
    th, xd = torch.from_numpy(theta).cuda(), torch.from_numpy(x).cuda()
    sim.forward(th, xd)
    g = sim.backward(th, xd, torch.from_numpy(dl), per_sample=True).cpu().numpy() / dl[:, None]
    gr, _ = orc.gradient(circ, theta.astype(np.float64), x.astype(np.float64), obs, per_sample=True)
    assert np.max(np.abs(g - gr)) < 1e-5


def test_zero_infinite_and_nan_dLdE():
    """They reach their own samples' gradients only, as 0, infinity or NaN."""
    n, d, B = 8, 2, 5
    sim = Simulator(n, d, B)
    theta, x = torch.rand(3 * n * d, device="cuda") * 6, torch.rand(B, n, device="cuda") * 3
    dl = torch.tensor([1.0, 0.0, float("inf"), float("nan"), 5e-324], dtype=torch.float64)
    sim.forward(theta, x)
    g = sim.backward(theta, x, dl, per_sample=True)
    one = sim.backward(theta, x, torch.ones(B, dtype=torch.float64), per_sample=True)
    assert torch.equal(g[0], one[0]) and (g[1] == 0).all()
    assert not torch.isfinite(g[2]).any() and torch.isnan(g[3]).all() and torch.isfinite(g[4]).all()

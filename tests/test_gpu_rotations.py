"""Round programs at the angles where a rotation's reduced form changes: the
wrap to [-pi, pi], a tangent of 1 and its poles (steep rounds)."""
import numpy as np
import pytest
import torch

from oracle import oracle as orc
from paper_2603_02804_gb300 import build as qbuild
from paper_2603_02804_gb300 import workloads
from paper_2603_02804_gb300.torch_api import Simulator

pytestmark = pytest.mark.gpu
PI = np.pi
EDGES = [0.0, PI / 2, -PI / 2, PI, -PI, 3 * PI / 2, 2 * PI, -2 * PI, 3 * PI, 5 * PI / 2, 1e-7, PI + 1e-6, PI / 2 + 3e-7,
         PI / 2 - 3e-7, 100.0, -37.5, 0.3, 2.0]


@pytest.fixture(scope="module", autouse=True)
def built():
    qbuild.build()
    orc.build()


@pytest.mark.parametrize("ansatz", ["hea", "xyz"])
@pytest.mark.parametrize("n,d", [(7, 3), (9, 4), (12, 3), (13, 3)])
def test_edge_angles(n, d, ansatz):
    """Every angle from the edge list (exact float32 multiples of pi / 2 among
    them), per-sample gradients against the oracle. Tolerance: the 1e-5 bar of
    the parity tests (float32 states, about 100 gates)."""
    rng = np.random.default_rng(n + d)
    B, P = 3, 3 * n * d
    theta = rng.choice(EDGES, size=P).astype(np.float32)
    x = rng.uniform(0, PI, (B, n)).astype(np.float32)
    obs = "ZXY"
    if ansatz == "hea":
        sim, circ = Simulator(n, d, B, obs=obs, entangler="ring"), orc.hea(n, d, "ring")
    else:
        rows = workloads.xyz_ring_gates(n, d)
        sim, circ = Simulator(n, 0, B, gates=rows, n_params=P, obs=obs), orc.Circuit(n=n, gates=np.array(rows, np.int32), n_params=P)
    th, xd = torch.from_numpy(theta).cuda(), torch.from_numpy(x).cuda()
    E = sim.forward(th, xd)
    g = sim.backward(th, xd, torch.ones(B, dtype=torch.float64), per_sample=True)
    gr, Er = orc.gradient(circ, theta.astype(np.float64), x.astype(np.float64), obs, per_sample=True)
    assert np.max(np.abs(E.cpu().numpy() - Er)) < 1e-5
    assert np.max(np.abs(g.cpu().numpy() - gr)) < 1e-5

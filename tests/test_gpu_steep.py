"""Rounds of steep rotations (angles at or near pi), whose rotations run twice
in complex64: values in every launch shape that has code of its own, and the
time they cost."""
import numpy as np
import pytest
import torch

from oracle import oracle as orc
from paper_2603_02804_gb300 import build as qbuild
from paper_2603_02804_gb300 import workloads
from paper_2603_02804_gb300.torch_api import Batch, Simulator

pytestmark = pytest.mark.gpu
PI = np.pi
EDGES = [0.0, PI / 2, PI, -PI, 3 * PI / 2, 3 * PI, 1e-7, PI + 1e-6, PI / 2 - 3e-7, PI - 1e-3, PI + 0.01, 0.3, 2.0]


@pytest.fixture(scope="module", autouse=True)
def built():
    qbuild.build()
    orc.build()


def circuit(ansatz, n, d):
    if ansatz == "hea":
        return dict(n=n, d=d, entangler="ring"), orc.hea(n, d, "ring")
    rows = workloads.xyz_ring_gates(n, d)
    return (dict(n=n, d=0, gates=rows, n_params=3 * n * d),
            orc.Circuit(n=n, gates=np.array(rows, np.int32), n_params=3 * n * d))


def angles(rng, P, real):
    """Mostly edge angles; a run of exact pi, so that some rounds have four."""
    theta = rng.choice(EDGES, size=P)
    theta[P // 3:2 * P // 3] = PI
    return theta.astype(real)


def check(ansatz, n, d, B, precision):
    rng = np.random.default_rng(1000 * n + B)
    real, tol = (np.float64, 1e-11) if precision == "complex128" else (np.float32, 1e-5)
    kw, circ = circuit(ansatz, n, d)
    sim = Simulator(batch=B, obs="ZXY", precision=precision, **kw)
    theta = angles(rng, 3 * n * d, real)
    x = rng.uniform(0, PI, (B, n)).astype(real)
    th, xd = torch.from_numpy(theta).cuda(), torch.from_numpy(x).cuda()
    E = sim.forward(th, xd)
    g = sim.backward(th, xd, torch.ones(B, dtype=torch.float64), per_sample=True)
    gr, Er = orc.gradient(circ, theta.astype(np.float64), x.astype(np.float64), "ZXY", per_sample=True)
    assert np.max(np.abs(E.cpu().numpy() - Er)) < tol
    assert np.max(np.abs(g.cpu().numpy() - gr)) < tol


# the parity tests' bars: 1e-5 complex64, 1e-11 complex128. Batches on a GPU of about 150 SMs: two threads per column
# (B = 3 of fewer than 12 qubits), one thread (128 threads per SM and more), 12-qubit tiles on one CTA per SM, two, three
@pytest.mark.parametrize("ansatz", ["hea", "xyz"])
@pytest.mark.parametrize("n,d,B", [(7, 3, 3), (7, 3, 2500), (8, 3, 1300), (9, 3, 650), (10, 3, 330), (11, 3, 3), (11, 3, 160),
                                   (12, 3, 3), (12, 2, 200), (12, 2, 320), (13, 3, 3), (7, 2, 10000)])
def test_edge_angles(n, d, B, ansatz):
    check(ansatz, n, d, B, "complex64")


@pytest.mark.parametrize("ansatz", ["hea", "xyz"])
@pytest.mark.parametrize("n,d,B", [(7, 3, 3), (9, 3, 3), (9, 3, 700), (12, 3, 3), (12, 2, 80), (13, 2, 3)])
def test_edge_angles_complex128(n, d, B, ansatz):
    """Whole tiles and tiles of two CTAs (12 qubits, 3 samples)."""
    check(ansatz, n, d, B, "complex128")


def test_edge_angles_in_a_batch():
    specs = [(7, 3, 40), (8, 3, 20), (12, 3, 5), (13, 3, 3), (14, 2, 2)]
    rng = np.random.default_rng(5)
    th = [angles(rng, 3 * n * d, np.float32) for n, d, _ in specs]
    xs = [rng.uniform(0, PI, (B, n)).astype(np.float32) for n, _, B in specs]
    cat = lambda v: torch.from_numpy(np.concatenate([a.reshape(-1) for a in v])).cuda()
    bt = Batch(specs)
    _, E, g = bt.train_step(cat(th), cat(xs))
    E, g = E.cpu().numpy(), g.cpu().numpy()
    for i, (n, d, B) in enumerate(specs):
        gr, Er = orc.gradient(orc.hea(n, d), th[i].astype(np.float64), xs[i].astype(np.float64), "Z")
        assert np.max(np.abs(E[bt.sample_off[i]:bt.sample_off[i + 1]] - Er)) < 1e-5, (n, d, B)
        assert np.max(np.abs(g[bt.theta_off[i]:bt.theta_off[i + 1]] - gr)) < 1e-5 * B, (n, d, B)


def step_time(sim, theta, x, out):
    """Least of 15 times of four steps, device clock."""
    for _ in range(3):
        sim.train_step(theta, x, out=out)
    best = float("inf")
    for _ in range(15):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        for _ in range(4):
            sim.train_step(theta, x, out=out)
        b.record()
        b.synchronize()
        best = min(best, a.elapsed_time(b))
    return best


@pytest.mark.parametrize("ansatz,n,d,B,precision,most", [("hea", 12, 20, 256, "complex64", 1.4),
                                                         ("xyz", 12, 10, 256, "complex64", 1.4),
                                                         ("hea", 8, 20, 4096, "complex64", 1.4),
                                                         ("hea", 12, 10, 64, "complex128", 1.1),
                                                         ("xyz", 12, 5, 64, "complex128", 1.1)])
def test_steep_rounds_repeat_their_rotations_only(ansatz, n, d, B, precision, most):
    """A step at exactly pi against one at uniform angles. complex64: the
    rotations are at most a third of a round's instructions (adjoint: 128 of
    650 for RY, 256 of 780 for RX), so running them twice is below 1.34 times a
    whole step; the bound leaves 5 % for the clock. complex128 runs every round
    once."""
    kw, _ = circuit(ansatz, n, d)
    sim = Simulator(batch=B, precision=precision, **kw)
    g = torch.Generator(device="cuda").manual_seed(3)
    rand = lambda *s: torch.rand(*s, generator=g, device="cuda", dtype=sim.real)
    x, out = rand(B, n) * PI, sim.device_outputs()
    t = [step_time(sim, theta, x, out) for theta in (rand(3 * n * d) * 2 * PI, torch.full_like(rand(3 * n * d), PI))]
    assert t[1] < most * t[0], t

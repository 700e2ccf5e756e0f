"""Launch shapes that depend on the number of tiles: CTAs of 32 to 256 threads
for small tiles, and two CTAs per 12-qubit complex128 tile."""
import numpy as np
import pytest
import torch

from oracle import oracle as orc
from paper_2603_02804_gb300 import build as qbuild, workloads
from paper_2603_02804_gb300.torch_api import Batch, Simulator

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    qbuild.build()
    orc.build()


def check(sim, circ, n, P, B, obs, real, tol, seed):
    rng = np.random.default_rng(seed)
    theta = rng.uniform(0, 2 * np.pi, P).astype(real)
    x = rng.uniform(0, np.pi, (B, n)).astype(real)
    y = (2 * rng.integers(0, 2, B) - 1).astype(real)
    loss, E, g = sim.train_step(*(torch.from_numpy(v).cuda() for v in (theta, x, y)), loss="mse")
    t64, x64 = theta.astype(np.float64), x.astype(np.float64)
    Er = orc.expectation(circ, t64, x64, obs)
    gr, _ = orc.gradient(circ, t64, x64, obs, dLdE=orc.mse_dLdE(Er, y))
    assert np.max(np.abs(E.cpu().numpy() - Er)) < tol
    assert np.max(np.abs(g.cpu().numpy() - gr)) < tol
    assert abs(loss.item() - orc.mse_loss(Er, y)) < tol * 4


# batches around the sizes where the CTA shrinks to 128, 64 and 32 threads on a GPU of about 150 SMs, ragged
# tails of a CTA's tiles among them; the parity tests' tolerances (1e-5 complex64, 1e-11 complex128)
@pytest.mark.parametrize("n,B", [(4, 3), (5, 700), (7, 1), (7, 37), (7, 1400), (8, 600), (8, 1300), (9, 330),
                                 (10, 75), (10, 310), (11, 151), (11, 153)])
def test_small_tiles(n, B):
    check(Simulator(n, 2, B, obs="ZX"), orc.hea(n, 2), n, 6 * n, B, "ZX", np.float32, 1e-5, n * B)


def generic_rows(n, d):
    rows = []
    for layer in range(d):
        for q in range(n):
            rows += [(1, q, -1, (layer * n + q) * 2), (2, q, -1, (layer * n + q) * 2 + 1)]
        rows += [(4, q, q + 1, -1) for q in range(n - 1)]
    return rows


@pytest.mark.parametrize("program", ["rounds", "cnot"])
@pytest.mark.parametrize("n,B", [(7, 3), (11, 5), (12, 1), (12, 76), (12, 80), (13, 3)])
def test_complex128_shapes(n, B, program):
    """Whole and shared tiles; X and Y on the bits that a shared tile splits."""
    obs = "Z" + "I" * (n - 2) + "Y" if n <= 12 else "ZX"
    if program == "rounds":
        sim, circ, P = Simulator(n, 2, B, obs=obs, precision="complex128"), orc.hea(n, 2), 6 * n
    else:
        rows, P = generic_rows(n, 2), 4 * n
        sim = Simulator(n, 0, B, gates=rows, n_params=P, obs=obs, precision="complex128")
        circ = orc.Circuit(n=n, gates=np.array(rows, np.int32), n_params=P)
    check(sim, circ, n, P, B, obs, np.float64, 1e-11, n + B)


@pytest.mark.parametrize("K,specs", [(8, [(9, 2, 5), (10, 2, 3), (13, 2, 2)]), (9, [(10, 2, 9), (12, 2, 3), (14, 1, 2)]),
                                     (12, [(13, 2, 9), (15, 2, 3), (16, 1, 2), (17, 1, 1), (12, 2, 5), (8, 3, 40)])])
def test_batch_tiles_dealt_to_a_cluster(K, specs):
    """Persistent batches whose samples span 2 to 32 tiles, of every tile width
    class (several samples per CTA, one tile per CTA, several per CTA)."""
    rng = np.random.default_rng(K)
    th = [rng.uniform(0, 2 * np.pi, 3 * n * d).astype(np.float32) for n, d, _ in specs]
    xs = [rng.uniform(0, np.pi, (B, n)).astype(np.float32) for n, _, B in specs]
    cat = lambda v: torch.from_numpy(np.concatenate([a.reshape(-1) for a in v])).cuda()
    bt = Batch(specs, tile_bits=K)
    _, E, g = bt.train_step(cat(th), cat(xs))
    E, g = E.cpu().numpy(), g.cpu().numpy()
    for i, (n, d, B) in enumerate(specs):
        c, t64, x64 = orc.hea(n, d), th[i].astype(np.float64), xs[i].astype(np.float64)
        gr, Er = orc.gradient(c, t64, x64, "Z")
        assert np.max(np.abs(E[bt.sample_off[i]:bt.sample_off[i + 1]] - Er)) < 1e-5, (n, d, B)
        assert np.max(np.abs(g[bt.theta_off[i]:bt.theta_off[i + 1]] - gr)) < 1e-5 * B, (n, d, B)


@pytest.mark.parametrize("n,B", [(4, 9), (6, 5), (7, 3), (8, 33), (9, 2), (12, 3), (13, 2)])
def test_generic_terms_are_reduced_by_eights(n, B):
    """CNOT circuits (generic steps): 1 to 32 lanes per tile, term counts per
    step that are no multiple of 8, RX gates among them."""
    rows, P = [], 0
    for layer in range(3):
        for q in range(n):
            for kind in ((1, 2), (0, 1, 2), (1,))[(layer + q) % 3]:
                rows.append((kind, q, -1, P))
                P += 1
        rows += [(4, q, q + 1, -1) for q in range(layer % 2, n - 1, 2)] + [(3, 0, n - 1, -1)]
    sim = Simulator(n, 0, B, gates=rows, n_params=P, obs="ZX")
    check(sim, orc.Circuit(n=n, gates=np.array(rows, np.int32), n_params=P), n, P, B, "ZX", np.float32, 1e-5, n)


@pytest.mark.parametrize("n,kw,obs", [(9, dict(tile_bits=5), "XIIIIIYIZ"), (10, dict(tile_bits=8), "YZIIIIIIIX"),
                                      (13, {}, "X" * 13), (13, dict(ckpt_mode=1, ckpt_layers=1), "ZYIIIIXIIIIIX"),
                                      (14, {}, "IXYZIXYZIXYZIX")])
def test_observables_beyond_the_tile(n, kw, obs):
    """The adjoint seeded from another tile's amplitudes (X or Y on qubits
    outside the last pass's tile, on bit 0 and not), and E over half the state."""
    check(Simulator(n, 3, 3, obs=obs, **kw), orc.hea(n, 3), n, 9 * n, 3, obs, np.float32, 1e-5, n)


@pytest.mark.parametrize("precision,real,tol", [("complex64", np.float32, 1e-5), ("complex128", np.float64, 1e-11)])
@pytest.mark.parametrize("n", [1, 2, 3, 4, 5, 6])
def test_few_qubits_on_seven(n, precision, real, tol):
    """Chains of fewer than 7 qubits run as round programs on 7, up to the batch
    where the larger state costs more, and up to a bounded workspace; observables
    on the last qubits, given states and rings (whose closing link has no
    neighbours there) keep their results."""
    obs = "YX"[:n] if n < 3 else "I" * (n - 3) + "ZYX"
    most = 2048 if precision == "complex128" else 4096
    for B in (5, most, most + 1):
        sim = Simulator(n, 2, B, obs=obs, precision=precision)
        padded = B <= most and (precision == "complex64" or n >= 4)
        assert sim.info()["n_eff"] == (7 if padded else max(n, 4))
        check(sim, orc.hea(n, 2), n, 6 * n, B, obs, real, tol, 40 + n + B)
    assert Simulator(n, 2000, 512, precision=precision).info()["n_eff"] == max(n, 4)  # 200 stored states
    if n >= 3:
        rows = workloads.xyz_ring_gates(n, 2)
        sim = Simulator(n, 0, 5, gates=rows, n_params=6 * n, obs=obs, precision=precision)
        assert sim.info()["n_eff"] == max(n, 4)
        check(sim, orc.Circuit(n=n, gates=np.array(rows, np.int32), n_params=6 * n), n, 6 * n, 5, obs, real, tol, n)
    if precision == "complex64":
        rows = [r for r in workloads.xyz_ring_gates(n, 2) if r[0] != 3 or r[2] == r[1] + 1]
        rng = np.random.default_rng(n)
        psi = rng.normal(size=(3, 2 ** n, 2))
        psi = np.ascontiguousarray((psi / np.linalg.norm(psi, axis=(1, 2), keepdims=True)).astype(np.float32))
        states = torch.view_as_complex(torch.from_numpy(psi)).cuda()
        theta = torch.from_numpy(rng.uniform(0, 2 * np.pi, 6 * n).astype(np.float32)).cuda()
        out = []
        for program in (0, 1):
            sim = Simulator(n, 0, 3, gates=rows, n_params=6 * n, obs=obs, encoding="state", program=program)
            assert sim.info()["n_eff"] == (7 if program == 0 else max(n, 4))
            out.append([v.double().cpu().numpy() for v in sim.train_step(theta, states)])
        for a, b in zip(*out):
            assert np.max(np.abs(a - b)) < tol

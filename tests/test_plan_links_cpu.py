"""Where round programs apply their pending CZ signs (the flush bit of a step),
on the exported plans. The interpreter of the plan tests applies every link at
its round and does not look at the bit."""
import numpy as np
import pytest

from oracle import oracle as orc
from paper_2603_02804_gb300 import build as qbuild
from paper_2603_02804_gb300 import qfuse, workloads
from tests import plan_interp as pi

FLUSH = 1 << 24
# (words of a round, links, links between register bits, links that leave the group), forward and adjoint
WORDS = [(pi.FWD_ROUND_WORDS, 4, 5, 7), (pi.BWD_ROUND_WORDS, 8, 9, 11)]


@pytest.fixture(scope="module", autouse=True)
def lib():
    qbuild.build()


def parity(links, x, n):
    return sum((x >> q) & (x >> ((q + 1) % n)) & 1 for q in range(n) if (links >> q) & 1) & 1


def check_linear(pend, regs, n, rng):
    """The pending signs are affine in the register index for every thread: they
    meet a rotation as a sign of its angle."""
    own = sum(1 << q for q in regs)
    for _ in range(6):
        base = int(rng.integers(1 << n)) & ~own
        f = [parity(pend, base | sum(1 << regs[r] for r in range(4) if (j >> r) & 1), n) for j in range(16)]
        for j in range(16):
            want = f[0]
            for r in range(4):
                if (j >> r) & 1:
                    want ^= f[0] ^ f[1 << r]
            assert f[j] == want, (hex(pend), regs, j)


def check_plan(h):
    """Returns how many steps carry links on without applying them."""
    rng = np.random.default_rng(0)
    n = qfuse.qf_plan_info(h)["n_eff"]
    carried = 0
    for direction, (words, at_links, at_inner, at_out) in enumerate(WORDS):
        prog = pi.parse(qfuse.qf_plan_export(h, direction))
        assert prog.rounds_mode
        for pd in prog.passes:
            pend = 0
            for w0, w1 in prog.ops[pd["op_begin"]:pd["op_end"]]:
                if w0 & 15 != pi.OP_STEP:
                    assert pend == 0, "a checkpoint is stored or read with signs pending"
                    continue
                group = pd["groups"][(w0 >> 4) & 3]
                # the kernels' constant offsets: four consecutive local bits from one of these
                assert group[0] in ((0, 4, 8) if pd["K"] == 12 else (0, 3, 4, 5, 6, 7))
                assert group == [group[0] + r for r in range(4)] and group[3] < pd["K"]
                regs = [pd["gmap"][q] for q in group]
                check_linear(pend, regs, n, rng)
                for k in range((w0 >> 8) & 0xFFFF):
                    rec = prog.round_words[(w1 + k) * words:(w1 + k + 1) * words]
                    out = pi._links_rest(rec[at_links] & 0xFFFFFFFF, rec[at_inner], regs)
                    assert rec[at_out] & 0xFFFFFFFF == out
                    pend ^= out
                    check_linear(pend, regs, n, rng)  # the step's next rounds meet them too
                if w0 & FLUSH:
                    pend = 0
                carried += pend != 0
            assert pend == 0, "the pass ends with signs pending"
    return carried


@pytest.mark.parametrize("ring", [False, True])
@pytest.mark.parametrize("n,d,K,ck", [(7, 5, 0, 1), (8, 4, 0, 2), (9, 6, 0, 10), (10, 4, 7, 2), (11, 6, 0, 2), (12, 20, 0, 10),
                                      (13, 8, 0, 2), (13, 5, 8, 1), (14, 6, 9, 3), (16, 10, 0, 4), (17, 6, 0, 3), (20, 8, 0, 4)])
@pytest.mark.parametrize("catch_up", [1, 2])
def test_pending_links_are_applied_in_time(n, d, K, ck, ring, catch_up):
    h = qfuse.qf_hea_create(n, d, qfuse.QF_ENT_RING if ring else qfuse.QF_ENT_CHAIN)
    try:
        qfuse.qf_plan(h, 1, tile_bits=K, ckpt_layers=ck, host_only=True, catch_up=catch_up)
        carried = check_plan(h)
        assert carried > 0 or n < 8  # (7 qubits: two groups that share one)
    finally:
        qfuse.qf_circuit_destroy(h)


@pytest.mark.parametrize("n,d", [(4, 3), (7, 3), (12, 3), (15, 3), (20, 2)])
def test_pending_links_with_rx_and_padding(n, d):
    """XYZ rings, and (4 qubits, a chain) a circuit simulated on 7."""
    rows = workloads.xyz_ring_gates(n, d)
    if n < 7:
        rows = [r for r in rows if r[0] != orc.CZ or r[2] == r[1] + 1]
    h = qfuse.qf_circuit_create(n, rows, 3 * n * d)
    try:
        qfuse.qf_plan(h, 1, ckpt_layers=1, host_only=True)
        carried = check_plan(h)
        assert carried > 0 or n < 8
    finally:
        qfuse.qf_circuit_destroy(h)


@pytest.mark.parametrize("seed", range(6))
def test_pending_links_of_random_lists(seed):
    """Uneven gate lists: links that stay pending over several steps."""
    rng = np.random.default_rng(seed)
    n = int(rng.integers(7, 13))
    rows = []
    for _ in range(30 * n):
        q = int(rng.integers(n))
        if rng.random() < 0.4:
            rows.append((orc.CZ, min(q, n - 2), min(q, n - 2) + 1, -1))
        else:
            rows.append((int(rng.choice([orc.RX, orc.RY, orc.RZ])), q, -1, int(rng.integers(5))))
    h = qfuse.qf_circuit_create(n, rows, 5)
    try:
        qfuse.qf_plan(h, 1, ckpt_layers=3, host_only=True)
        check_plan(h)
    finally:
        qfuse.qf_circuit_destroy(h)

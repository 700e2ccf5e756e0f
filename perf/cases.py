"""Performance cases: training steps, inference and batched training of the simulator, each through the
entry point a program calls (Simulator, HEA, Batch), from one small circuit to a batch of 20-qubit states.

A case names a circuit (``ansatz``, ``n`` qubits, ``d`` layers), a batch of ``B`` samples and the call
(``kind``). The ansatz layers:

- ``hea_chain`` / ``hea_ring``: RZ, RY, RZ on every qubit, then CZ(q, q+1) (a ring adds CZ(n-1, 0));
- ``xyz_ring``: RX, RY, RZ on every qubit, then the CZ ring, on given initial states, observable IXYZ...;
- ``cnot_chain``: RY, RZ on every qubit, then CNOT(q, q+1): a user gate list.

Results of a complex64 plan carry float32 accuracy in float64 containers; a float32 training program takes
them as float32 before it updates float32 parameters, and so do the passes here. complex128 plans return
their float64 results as they are.
"""
import math

import torch

from paper_2603_02804_gb300 import qfuse, workloads
from paper_2603_02804_gb300.torch_api import HEA, Batch, Simulator

_TWO_PI = 2.0 * math.pi


def listed():
    step = dict(kind="step", ansatz="hea_chain", precision="complex64", ckpt=0, mode=0)
    return [
        # the smallest circuit in use: latency of one training step (launches, tables, reductions)
        {**step, "name": "step_n4", "n": 4, "d": 2, "B": 8},
        # a small classifier, the usual size of a first model: 8 qubits, one mini-batch of 64
        {**step, "name": "step_n8", "n": 8, "d": 20, "B": 64},
        # a hybrid model: the circuit as a torch module inside autograd, forward and backward apart
        {"name": "module_n10", "kind": "module", "ansatz": "hea_ring", "n": 10, "d": 10, "B": 100},
        # a user circuit with CNOTs (the efficient-SU2 form many papers train)
        {**step, "name": "step_cnot_n10", "ansatz": "cnot_chain", "n": 10, "d": 6, "B": 100},
        # the 12-qubit training workload: a whole state per thread block
        {**step, "name": "step_n12", "n": 12, "d": 20, "B": 256},
        # odd sizes: 13 qubits, a ring, an odd depth and a ragged batch
        {**step, "name": "step_n13_ring", "ansatz": "hea_ring", "n": 13, "d": 31, "B": 37},
        # the 16-qubit, 100-layer training workload (checkpoints every 10 layers), a micro-batch of it
        {**step, "name": "step_n16", "n": 16, "d": 100, "B": 64, "ckpt": 10},
        # inference: expectations of a whole test set, no gradients
        {"name": "forward_n16", "kind": "forward", "ansatz": "hea_chain", "n": 16, "d": 20, "B": 500},
        # the 20-qubit workload's plan (checkpoints every 4 layers) over part of its depth and micro-batch
        {**step, "name": "step_n20", "n": 20, "d": 24, "B": 64, "ckpt": 4},
        # the throughput setting: given 20-qubit states, one layer, an observable on every qubit
        {**step, "name": "step_states_n20", "ansatz": "xyz_ring", "n": 20, "d": 1, "B": 100},
        # double precision, for gradients that have to be exact
        {**step, "name": "step_c128_n12", "n": 12, "d": 20, "B": 64, "precision": "complex128"},
        # many uneven circuits trained in one persistent launch
        {"name": "mixed_32", "kind": "mixed", "circuits": 32, "structure": 104, "n_hi": 16, "d_hi": 60, "b_hi": 64},
    ]


# qubits and the layers x samples a drawn case may have at that width stay below the largest listed one
_MOST = 24 * 64 * 20 << 20


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi + 0.49)))))))


def _fit(n, d, B, most):
    """Fewer samples, then layers, until layers x samples x qubits x 2^n is within `most`."""
    B = max(1, min(B, most // ((n * d) << n)))
    return max(1, min(d, most // ((n * B) << n))), B


def draw(rng):
    what = rng.choice(["step", "step", "step", "module", "cnot", "forward", "states", "c128", "modeA", "mixed"])
    step = dict(kind="step", ansatz=rng.choice(["hea_chain", "hea_ring"]), precision="complex64",
                ckpt=0, mode=0)
    if what == "mixed":
        return {"kind": "mixed", "circuits": rng.randint(8, 40), "structure": rng.randint(1, 10 ** 6),
                "n_hi": rng.randint(10, 16), "d_hi": rng.randint(20, 60), "b_hi": rng.randint(8, 64)}
    if what == "module":
        n, d, B = rng.randint(4, 14), _log_int(rng, 2, 40), _log_int(rng, 8, 512)
        d, B = _fit(n, d, B, _MOST // 4)
        return {"kind": "module", "ansatz": step["ansatz"], "n": n, "d": d, "B": B}
    if what == "cnot":
        n, d, B = rng.randint(4, 14), _log_int(rng, 1, 12), _log_int(rng, 8, 256)
        return {**step, "ansatz": "cnot_chain", "n": n, "d": d, "B": B}
    if what == "forward":
        n, d, B = rng.randint(6, 18), _log_int(rng, 2, 60), _log_int(rng, 32, 2048)
        d, B = _fit(n, d, B, _MOST)
        return {"kind": "forward", "ansatz": step["ansatz"], "n": n, "d": d, "B": B}
    if what == "states":
        n = rng.randint(12, 20)
        B = max(2, min(_log_int(rng, 8, 256), 100 << 20 >> n))
        return {**step, "ansatz": "xyz_ring", "n": n, "d": rng.randint(1, 3), "B": B}
    if what == "c128":
        n, d, B = rng.randint(4, 14), _log_int(rng, 2, 30), _log_int(rng, 8, 128)
        d, B = _fit(n, d, B, (20 * 64 * 12) << 12)
        return {**step, "n": n, "d": d, "B": B, "precision": "complex128"}
    if what == "modeA":
        n, d, B = rng.randint(13, 19), _log_int(rng, 8, 48), _log_int(rng, 4, 64)
        d, B = _fit(n, d, B, _MOST // 2)
        return {**step, "n": n, "d": d, "B": B, "ckpt": rng.randint(3, 8), "mode": 1}
    n, d, B = rng.randint(4, 20), _log_int(rng, 2, 100), _log_int(rng, 8, 512)
    d, B = _fit(n, min(d, 30 if n > 16 else 100), B, _MOST)
    return {**step, "n": n, "d": d, "B": B, "ckpt": rng.choice([0, 4, 10])}


# ---- the circuits as rows (kind, q0, q1, parameter), for user gate lists and for the reference below ------------
_RX, _RY, _RZ = 0, 1, 2
_ROTATIONS = {"hea_chain": (_RZ, _RY, _RZ), "hea_ring": (_RZ, _RY, _RZ), "xyz_ring": (_RX, _RY, _RZ),
              "cnot_chain": (_RY, _RZ)}


def _n_params(case):
    return len(_ROTATIONS[case["ansatz"]]) * case["n"] * case["d"]


def _pairs(ansatz, n):
    p = [(q, q + 1) for q in range(n - 1)]
    return p + [(n - 1, 0)] if ansatz.endswith("ring") and n > 2 else p


def _rows(case):
    n, kinds = case["n"], _ROTATIONS[case["ansatz"]]
    ent = qfuse.QF_GATE_CNOT if case["ansatz"] == "cnot_chain" else qfuse.QF_GATE_CZ
    rows = []
    for layer in range(case["d"]):
        for q in range(n):
            rows += [(k, q, -1, (layer * n + q) * len(kinds) + g) for g, k in enumerate(kinds)]
        rows += [(ent, a, b, -1) for a, b in _pairs(case["ansatz"], n)]
    return rows


def _observable(case):
    return workloads.ixyz(case["n"]) if case["ansatz"] == "xyz_ring" else "Z"


def _specs(case):
    return [(c.n, c.d, c.B) for c in workloads.mixed_circuits(case["circuits"], case["structure"], (8, case["n_hi"]),
                                                              (10, case["d_hi"]), (1, case["b_hi"]),
                                                              with_values=False)]


def _angles(n, d, u):
    """Rotation angles from u ~ U[0, 1): the whole circle, and near the identity for deep circuits, which is how those
    are started (random deep circuits sit on a barren plateau: expectations and gradients vanish, nothing trains)."""
    return u * _TWO_PI if d <= 24 else (2 * u - 1) * (1.2 / math.sqrt(d))


def _inputs(case, seed):
    """Parameters (_angles), encoding angles x ~ U[0, pi] or random normalised states, labels -1 / +1."""
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    g = torch.Generator(device=dev).manual_seed(int(seed))
    f64 = case.get("precision") == "complex128"
    real, cplx = (torch.float64, torch.complex128) if f64 else (torch.float32, torch.complex64)
    if case["kind"] == "mixed":  # concatenated over the circuits
        specs = _specs(case)
        P, X, B = sum(3 * n * d for n, d, _ in specs), sum(n * B for n, _, B in specs), sum(B for _, _, B in specs)
        u = torch.rand(P, generator=g, device=dev)
        u = [_angles(n, d, v) for (n, d, _), v in zip(specs, u.split([3 * n * d for n, d, _ in specs]))]
        return (torch.cat(u), torch.rand(X, generator=g, device=dev) * math.pi,
                (torch.randint(0, 2, (B,), generator=g, device=dev) * 2 - 1).to(real))
    n, B = case["n"], case["B"]
    theta = _angles(n, case["d"], torch.rand(_n_params(case), generator=g, device=dev, dtype=real))
    if case["ansatz"] == "xyz_ring":
        x = torch.randn(B, 1 << n, 2, generator=g, device=dev, dtype=real)
        x /= x.square().sum(dim=(1, 2), keepdim=True).sqrt()
        x = torch.view_as_complex(x).to(cplx)
    else:
        x = torch.rand(B, n, generator=g, device=dev, dtype=real) * math.pi
    y = (torch.randint(0, 2, (B,), generator=g, device=dev) * 2 - 1).to(real)
    return theta, x, y


def prepare(case, seed):
    theta, x, y = _inputs(case, seed)
    s = {"case": case, "theta": theta, "x": x, "y": y}
    if case["kind"] == "mixed":
        s["batch"] = Batch(_specs(case), loss="mse")
        s["buf"], s["out"] = _result_buffers(s["batch"].n_samples, s["batch"].n_params, theta.device)
        return s
    ent = "ring" if case["ansatz"].endswith("ring") else "chain"
    if case["kind"] == "module":
        s["model"] = HEA(case["n"], case["d"], case["B"], entangler=ent, init=theta)
        return s
    kw = dict(obs=_observable(case), ckpt_layers=case.get("ckpt", 0), ckpt_mode=case.get("mode", 0),
              precision=case.get("precision", "complex64"))
    if case["ansatz"] in ("xyz_ring", "cnot_chain"):
        kw.update(gates=_rows(case), n_params=_n_params(case), host_staging=False,
                  encoding="state" if case["ansatz"] == "xyz_ring" else "angles")
        s["sim"] = Simulator(case["n"], 0, case["B"], **kw)
    else:
        s["sim"] = Simulator(case["n"], case["d"], case["B"], entangler=ent, **kw)
    if case["kind"] == "step":
        s["buf"], s["out"] = _result_buffers(case["B"], _n_params(case), theta.device)
    return s


def _result_buffers(B, P, device):
    """One float64 buffer for (loss [1], E [B], grad [P]), so that one conversion reads a step's results."""
    buf = torch.empty(1 + B + P, dtype=torch.float64, device=device)
    return buf, (buf[:1], buf[1:1 + B], buf[1 + B:])


def _named(buf, B):
    return {"loss": buf[:1], "E": buf[1:1 + B], "grad": buf[1 + B:]}


def run(state):
    case = state["case"]
    theta, x, y = state["theta"], state["x"], state["y"]
    if case["kind"] == "mixed":
        state["batch"].train_step(theta, x, y, out=state["out"])
        return _named(state["buf"].float(), state["batch"].n_samples)
    if case["kind"] == "module":
        model = state["model"]
        model.zero_grad(set_to_none=True)
        pred = model(x).float()
        loss = torch.nn.functional.mse_loss(pred, y)
        loss.backward()
        return {"loss": loss.detach().reshape(1), "E": pred.detach(), "grad": model.theta.grad}
    if case["kind"] == "forward":
        return {"E": state["sim"].forward(theta, x).float()}
    state["sim"].train_step(theta, x, y, loss="mse", out=state["out"])
    buf = state["buf"] if case["precision"] == "complex128" else state["buf"].float()
    return _named(buf, case["B"])


def work(case):
    """Input and output bytes, and the arithmetic: per pair of amplitudes a real 2x2 on (re, im) is 12 flops, a phase
    per amplitude 6 (merged over a register group's four qubits: 3 a pair and qubit); the adjoint does both to psi and
    lambda and takes one inner product per rotation (8 flops a pair, half of that for the merged diagonal ones)."""
    if case["kind"] == "mixed":
        parts = [work({"kind": "step", "ansatz": "hea_chain", "n": n, "d": d, "B": B}) for n, d, B in _specs(case)]
        return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}
    n, d, B = case["n"], case["d"], case["B"]
    pairs = B * (n * d) << (n - 1)
    fwd, bwd = (15, 40) if case["ansatz"] != "xyz_ring" else (27, 72)
    w = 8 if case.get("precision") == "complex128" else 4
    P = _n_params(case)
    x = B * 2 * w << n if case["ansatz"] == "xyz_ring" else B * n * w
    out = 4 * B if case["kind"] == "forward" else w * (P + B + 1)
    return {"bytes": P * w + x + out, "flops": pairs * (fwd if case["kind"] == "forward" else fwd + bwd)}


# ---- the same results in 64 bits, gate by gate with plain torch ---------------------------------------------------
_I2 = torch.eye(2, dtype=torch.complex128)
_PAULI = torch.tensor([[[0, 1], [1, 0]], [[0, -1j], [1j, 0]], [[1, 0], [0, -1]]], dtype=torch.complex128)


def _rot(kind, angle):
    return math.cos(angle / 2) * _I2 - 1j * math.sin(angle / 2) * _PAULI[kind]


def _apply(s, q, u):
    """A 2x2 on qubit q (bit q of the index) of states [B, 2^n]."""
    v = s.view(s.shape[0], -1, 2, 1 << q)
    a, b = v[:, :, 0], v[:, :, 1]
    r = torch.empty_like(v)
    (u00, u01), (u10, u11) = u.tolist()
    torch.add(a * u00, b, alpha=u01, out=r[:, :, 0])
    torch.add(a * u10, b, alpha=u11, out=r[:, :, 1])
    return r.view(s.shape)


class _Exact:
    """Forward and adjoint of one circuit for states [B, 2^n] in complex128."""

    def __init__(self, case, theta):
        self.n, self.d, self.kinds = case["n"], case["d"], _ROTATIONS[case["ansatz"]]
        self.dev, self.theta, self.obs = theta.device, theta.double().cpu().tolist(), _observable(case)
        idx = torch.arange(1 << self.n, device=self.dev)
        pairs = _pairs(case["ansatz"], self.n)
        self.sign = self.perm = None
        if case["ansatz"] == "cnot_chain":
            self.perm = idx  # new state [i] = old state [perm[i]]; CNOT(a, b) is its own inverse
            for a, b in pairs:
                self.perm = self.perm[idx ^ (((idx >> a) & 1) << b)]
            self.inv = torch.argsort(self.perm)
        else:
            par = torch.zeros_like(idx)
            for a, b in pairs:
                par ^= (idx >> a) & (idx >> b) & 1
            self.sign = (1 - 2 * par).double()

    def angles(self, layer, q):
        k = len(self.kinds)
        at = (layer * self.n + q) * k
        return [(kind, at + g, self.theta[at + g]) for g, kind in enumerate(self.kinds)]

    def entangle(self, s, back=False):
        if self.sign is not None:
            return s.mul_(self.sign)
        return s[:, self.inv if back else self.perm]

    def fused(self, layer, q):
        u = _I2
        for kind, _, t in self.angles(layer, q):
            u = _rot(kind, t) @ u
        return u

    def forward(self, s):
        for layer in range(self.d):
            for q in range(self.n):
                s = _apply(s, q, self.fused(layer, q))
            s = self.entangle(s)
        return s

    def observe(self, s):
        for q, c in enumerate(self.obs):
            if c != "I":
                s = _apply(s, q, _PAULI["XYZ".index(c)])
        return s

    def gradient(self, s, lam):
        grad = torch.zeros(len(self.theta), dtype=torch.float64)
        for layer in reversed(range(self.d)):
            s, lam = self.entangle(s, True), self.entangle(lam, True)
            sums = []
            for q in range(self.n):
                p, l = (v.view(v.shape[0], -1, 2, 1 << q) for v in (s, lam))
                sums.append(torch.stack([(l[:, :, a].conj() * p[:, :, b]).sum() for a in (0, 1) for b in (0, 1)]))
                u = self.fused(layer, q).conj().T
                s, lam = _apply(s, q, u), _apply(lam, q, u)
            # T[a, b] = sum conj(lambda_a) psi_b after the layer's rotations; the gradient of a rotation
            # exp(-i t P / 2) is Im <lambda| P |psi> right after it
            for q, T in enumerate(torch.stack(sums).cpu().reshape(self.n, 2, 2)):
                for kind, at, t in reversed(self.angles(layer, q)):
                    grad[at] = (_PAULI[kind] * T).sum().imag
                    v = _rot(kind, t).conj().T
                    T = v.conj() @ T @ v.T
        return grad


def _exact_one(case, theta, x, y):
    c = _Exact(case, theta)
    x = x.to(torch.complex128 if x.is_complex() else torch.float64)
    if x.is_complex():
        s = x.clone()
    else:
        s = torch.ones(x.shape[0], 1, dtype=torch.complex128, device=x.device)
        for q in range(c.n):  # RY(x_q) |0> on every qubit, qubit q as bit q
            s = torch.cat([s * torch.cos(x[:, q:q + 1] / 2), s * torch.sin(x[:, q:q + 1] / 2)], dim=1)
    s = c.forward(s)
    lam = c.observe(s)
    E = (s.conj() * lam).sum(dim=1).real
    if case["kind"] == "forward":
        return {"E": E}
    r = E - y.double()  # mean squared error
    loss, dE = r.square().mean().reshape(1), 2 * r / len(E)
    # lambda = (dL/dE) O psi, so that the gradient of E = <psi|O|psi> is 2 Re <lambda| d psi>
    return {"loss": loss, "E": E, "grad": c.gradient(s, lam * dE[:, None])}


def exact(case, seed):
    theta, x, y = _inputs(case, seed)
    if case["kind"] != "mixed":
        return _exact_one(case, theta, x, y)
    out = {"loss": 0.0, "E": [], "grad": []}
    at = bt = ct = 0
    for n, d, B in _specs(case):
        one = {"kind": "step", "ansatz": "hea_chain", "n": n, "d": d, "B": B}
        r = _exact_one(one, theta[at:at + 3 * n * d], x[bt:bt + n * B].view(B, n), y[ct:ct + B])
        at, bt, ct = at + 3 * n * d, bt + n * B, ct + B
        out["loss"] = out["loss"] + r["loss"]
        out["E"].append(r["E"])
        out["grad"].append(r["grad"])
    return {"loss": out["loss"], "E": torch.cat(out["E"]), "grad": torch.cat(out["grad"])}

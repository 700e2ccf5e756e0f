"""Order of a batch's steps over streams and threads."""
import threading

import numpy as np
import pytest
import torch

from paper_2603_02804_gb300 import build as qbuild, qfuse
from paper_2603_02804_gb300.torch_api import Batch

pytestmark = pytest.mark.gpu
SPECS = [(13, 6, 8), (12, 6, 16), (8, 10, 40)]
PER_THREAD = 2  # the CUDA runtime's handle of the calling thread's own stream


@pytest.fixture(scope="module")
def batch():
    qbuild.build()
    rng = np.random.default_rng(21)
    bt = Batch(SPECS, loss="mse")
    dev = lambda k, hi: torch.from_numpy(rng.uniform(0, hi, k).astype(np.float32)).cuda()
    theta, x = dev(bt.n_params, 2 * np.pi), dev(sum(n * B for n, _, B in SPECS), np.pi)
    y = dev(bt.n_samples, 1.0)
    ref = [t.clone() for t in bt.train_step(theta, x, y)]
    torch.cuda.synchronize()
    return bt, (theta, x, y), ref


def step(bt, inputs, out, ws, stream):
    qfuse.qf_batch_train_step(bt.handle, *inputs, *out, ws, bt.ws_bytes, stream)


def test_threads_on_their_own_per_thread_stream(batch):
    """Two threads use one handle value for two streams: the steps share the
    workspace and give the same bits as alone."""
    bt, inputs, ref = batch
    outs = [bt.outputs(), bt.outputs()]
    torch.cuda.synchronize()

    def run(out):
        for _ in range(10):
            step(bt, inputs, out, bt.ws, PER_THREAD)

    threads = [threading.Thread(target=run, args=(o,)) for o in outs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    for out in outs:
        assert all(torch.equal(a, b) for a, b in zip(out, ref))


def test_steps_with_workspaces_of_their_own_overlap(batch):
    """A step on another stream and workspace does not wait for one that is
    still queued behind 0.5 s of other work."""
    bt, inputs, ref = batch
    ws2 = torch.empty_like(bt.ws)
    outs = [bt.outputs(), bt.outputs()]
    s1, s2 = torch.cuda.Stream(), torch.cuda.Stream()
    step(bt, inputs, outs[1], ws2, s2)
    torch.cuda.synchronize()
    with torch.cuda.stream(s1):
        torch.cuda._sleep(1_000_000_000)  # cycles
    step(bt, inputs, outs[0], bt.ws, s1)
    step(bt, inputs, outs[1], ws2, s2)
    s2.synchronize()
    assert not s1.query()
    torch.cuda.synchronize()
    for out in outs:
        assert all(torch.equal(a, b) for a, b in zip(out, ref))


def test_more_workspaces_than_the_order_remembers(batch):
    """Seven workspaces in turn on three streams, each used again later on
    another stream behind other work, one of them reached by overlapping ranges."""
    bt, inputs, ref = batch
    size = bt.ws.numel() + 256
    spaces = [torch.empty(size, dtype=torch.uint8, device="cuda") for _ in range(7)]
    streams = [torch.cuda.Stream() for _ in range(3)]
    outs = [bt.outputs() for _ in range(21)]
    torch.cuda.synchronize()
    for k, out in enumerate(outs):
        s = streams[k % 3]
        if k % 4 == 0:
            with torch.cuda.stream(s):
                torch.cuda._sleep(2_000_000)
        w = spaces[(k * 5) % 7]
        step(bt, inputs, out, w[256:] if k % 2 else w, s)
    torch.cuda.synchronize()
    for out in outs:
        assert all(torch.equal(a, b) for a, b in zip(out, ref))

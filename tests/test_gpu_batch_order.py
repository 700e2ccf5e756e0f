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

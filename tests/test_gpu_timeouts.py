"""What a layer is after a device-side wait ran out: every path on which one can is made to run out
without a copy left in flight (a first wait that gives up without polling), and afterwards the
cached rows, the window state and the next token must be the oracle's."""
import numpy as np
import pytest
import torch

from paper_2312_11514_b200 import binding as B
from paper_2312_11514_b200 import workloads as W

import parity_util as P

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
POLLS = 1 << 22          # LIF_TUNE_WAIT_POLLS as a layer is created


def _layer(S=1, steps=3, d=1032, F=4096, **kw):
    """A layer a few tokens into a sequence, its oracle, the inputs, an output and two streams."""
    cfg = W.LifConfig("timeouts", 1, d, F, 32, 3, S, 8, 0.10, 1.0, 0.8, 0.6, 91)
    gpu, ora = P.make_layer_pair(cfg, 0, b_down=True, **kw)
    X = W.make_inputs(cfg, device=DEV)
    y = torch.empty(S, d, dtype=torch.float32, device=DEV)
    streams = torch.cuda.Stream(), torch.cuda.Stream()
    torch.cuda.synchronize()
    for t in range(steps):
        B.lif_decode_step(gpu.handle, X[t], y, *streams)
        P.check_decode_step(gpu, ora, X[t].cpu().numpy(), y)
    return gpu, ora, X, y, streams


def test_a_timeout_is_recorded_over_another_condition():
    gpu, ora, X, y, streams = _layer()
    bad = torch.tensor([gpu.capacity], dtype=torch.int32, device=DEV)       # no such row
    B.lif_sparse_ffn(gpu.handle, X[0], bad, torch.ones(1, dtype=torch.int32, device=DEV), y)
    assert B.lif_get_stats(gpu.handle).status == B.LIF_ERR_INVALID_ARG
    B.lif_set_tuning(gpu.handle, B.TUNE_WAIT_POLLS, 0)
    B.lif_decode_step(gpu.handle, X[3], y, *streams)
    B.lif_set_tuning(gpu.handle, B.TUNE_WAIT_POLLS, POLLS)
    before = gpu.lists()
    assert before["status"] == B.LIF_ERR_TIMEOUT
    B.lif_decode_step(gpu.handle, X[4], y, *streams)                        # so this one is refused
    after = gpu.lists()
    assert after["status"] == B.LIF_ERR_TIMEOUT and after["step"] == before["step"]
    np.testing.assert_array_equal(after["pointers"], before["pointers"])
    gpu.close()

"""The low-rank predictor in one launch: its scores bit for bit in the stated order of additions, at the
edges of its launch shapes, and what a call is in which a value of z does not come."""
import numpy as np
import pytest
import torch

from paper_2312_11514_b200 import binding as B
from paper_2312_11514_b200 import workloads as W

import parity_util as P

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _scores_in_order(x, A, Bm, c):
    """Rows of A in parts of consecutive ones (about 32); a part in 256 / (rank / 8) interleaved runs; runs,
    then parts in order; rows of B in 16 interleaved runs, then those in order.  Products of fp16 values are
    exact in fp32; a product of z and B plus a sum is exact in 64 bits but for the last rounding."""
    S, d, (r, F) = x.shape[0], x.shape[1], Bm.shape
    rows = max(32, ((d + 31) // 32 + 31) // 32 * 32)
    lanes = 256 // (r // 8)
    x32, A32, B32 = x.astype(np.float32), A.astype(np.float32), Bm.astype(np.longdouble)
    out = np.empty((S, F), np.float32)
    for s in range(S):
        z = np.zeros(r, np.float32)
        for m0 in range(0, d, rows):
            part = np.zeros((lanes, r), np.float32)
            end = min(d, m0 + rows)
            for m in range(m0, end, lanes):
                n = min(lanes, end - m)
                part[:n] += x32[s, m:m + n, None] * A32[m:m + n]
            total = np.zeros(r, np.float32)
            for lane in range(lanes):
                total += part[lane]
            z += total
        runs = np.zeros((16, F), np.float32)
        for j in range(r):
            runs[j % 16] = (runs[j % 16].astype(np.longdouble) + z[j].astype(np.longdouble) * B32[j]).astype(np.float32)
        v = np.zeros(F, np.float32)
        for k in range(16):
            v += runs[k]
        out[s] = v + c
    return out


@pytest.mark.parametrize("S,d,F,r", [
    (1, 8, 8, 8),            # one run with a row
    (1, 8192, 136, 8),       # by parts: one column group, most lanes
    (1, 6128, 136, 136),     # ... a column group that is too long
    (5, 2568, 136, 48),      # by columns; a last part of 72 rows
    (2, 2568, 136, 56),      # by parts, two streams; a number of words that 256 threads do not divide
    (4, 4104, 136, 16),      # ... four, which would be 4 columns at a time
    (8, 5120, 136, 16),      # ... eight, which would be 2
    (1, 1024, 136, 64),      # ... the largest small rank
    (8, 4104, 136, 40),      # by columns at a small rank: many runs, few columns at a time
    (1, 4104, 264, 120),     # a last part of 8 rows
    (1, 1000, 520, 248),     # runs of different lengths, rank not a multiple of 16
    (1, 8192, 128, 1024),    # few long runs
    (2, 264, 136, 136),
    (3, 1544, 392, 72),
    (5, 4096, 136, 128),
    (8, 7168, 264, 256),     # two streams per CTA
    (7, 520, 136, 1024),     # four, the last CTA three
    (8, 8000, 136, 264),     # two: four streams' x and sums, 230 KB, would not fit
    (8, 8192, 136, 520),     # four of the widest
])
def test_scores_are_those_of_the_stated_order_of_additions(S, d, F, r):
    cfg = W.LifConfig("scores", 1, d, F, r, 2, S, 2, 0.10, 1.0, 0.7, 0.7, 75)
    gpu, _ = P.make_layer_pair(cfg, 0, capacity=F)
    X = W.make_inputs(cfg, device=DEV)
    logits = torch.empty(S, F, dtype=torch.float32, device=DEV)
    act, n = torch.empty(F, dtype=torch.int32, device=DEV), torch.zeros(1, dtype=torch.int32, device=DEV)
    A, Bm, c = (gpu.keep[k].cpu().numpy() for k in ("pred_A", "pred_B", "pred_c"))
    for t in range(2):
        B.lif_predict(gpu.handle, X[t], logits, act, n)
        got = logits.cpu().numpy()
        want = _scores_in_order(X[t].cpu().numpy(), A, Bm, c)
        np.testing.assert_array_equal(got, want)
        np.testing.assert_array_equal(act[:int(n)].cpu().numpy(), np.nonzero((want > 0).any(axis=0))[0])
    gpu.close()


@pytest.mark.parametrize("S,d,F,r", [
    (1, 8, 64, 8),
    (1, 8192, 136, 8),       # by parts
    (5, 2568, 136, 48),
    (2, 2568, 136, 48),      # by parts, several streams
    (8, 5120, 136, 16),
    (8, 4104, 136, 40),      # few columns at a time
    (1, 1000, 520, 248),
    (3, 1544, 392, 72),
    (8, 7168, 264, 256),     # two streams per CTA
    (7, 520, 136, 1024),     # four
])
def test_later_layers_of_a_graph_equal_steps_by_themselves(S, d, F, r):
    # the first stage of a graph's later layers runs once ahead of its wait, that of a step by itself does not
    cfg = W.LifConfig("passes", 3, d, F, r, 2, S, 4, 0.10, 1.0, 0.7, 0.7, 77)
    gpus = [P.make_layer_pair(cfg, l, capacity=F, append_first=1)[0] for l in range(cfg.n_layers)]
    X = W.make_inputs(cfg, device=DEV)
    x = torch.empty(S, d, dtype=torch.float16, device=DEV)
    y = torch.empty(2, cfg.steps, cfg.n_layers, S, d, dtype=torch.float32, device=DEV)
    out = torch.empty(cfg.n_layers, S, d, dtype=torch.float32, device=DEV)
    sc, sf = torch.cuda.Stream(), torch.cuda.Stream()
    torch.cuda.synchronize()
    graph = B.lif_graph_capture([gpu.handle for gpu in gpus], x, out, sc, sf)
    with torch.cuda.stream(sc):
        for t in range(cfg.steps):
            x.copy_(X[t])
            B.lif_graph_launch(graph, sc)
            y[0, t].copy_(out)
    torch.cuda.synchronize()
    state = [gpu.lists() for gpu in gpus]
    for gpu in gpus:
        B.lif_reset(gpu.handle)
    torch.cuda.synchronize()
    for t in range(cfg.steps):
        for l, gpu in enumerate(gpus):
            B.lif_decode_step(gpu.handle, X[t], y[1, t, l], sc, sf)
    torch.cuda.synchronize()
    assert torch.equal(y[0], y[1])
    for gpu, one in zip(gpus, state):
        other = gpu.lists()
        assert one["status"] == other["status"] == B.LIF_OK and one["step"] == other["step"] == cfg.steps
        for key in ("pointers", "slot_of", "last_active"):
            np.testing.assert_array_equal(one[key], other[key])
    B.lif_graph_destroy(graph)
    for gpu in gpus:
        gpu.close()


@pytest.mark.parametrize("S", [1, 3])
def test_a_score_that_lacks_z_is_not_active_and_the_call_says_so(S):
    cfg = W.LifConfig("lost z", 1, 4096, 2048, 128, 3, S, 5, 0.08, 1.0, 0.8, 0.6, 76)
    gpu, ora = P.make_layer_pair(cfg, 0, b_down=True, append_first=1)
    X = W.make_inputs(cfg, device=DEV)
    y = torch.empty(S, cfg.d_model, dtype=torch.float32, device=DEV)
    for t in range(5):
        lost = t == 2
        if lost:
            B.lif_set_tuning(gpu.handle, B.TUNE_PREDICTOR_POLLS, 0)
        B.lif_decode_step(gpu.handle, X[t], y)
        if lost:
            B.lif_set_tuning(gpu.handle, B.TUNE_PREDICTOR_POLLS, 1 << 20)
            g = gpu.lists()
            assert g["status"] == B.LIF_ERR_TIMEOUT
            if g["step"] == t + 1:                       # (refused where the window CTA saw the status)
                ora.cache.insert(ora.cache.window_update(g["active_idx"]), ora.bundles, ora.bias_up)
            np.testing.assert_array_equal(g["pointers"], ora.cache.pointers)
            B.lif_clear_status(gpu.handle)
        else:
            P.check_decode_step(gpu, ora, X[t].cpu().numpy(), y)
        P.compare_cache_rows(gpu, ora)
    with pytest.raises(B.LifError):
        B.lif_set_tuning(gpu.handle, B.TUNE_PREDICTOR_POLLS, -1)
    gpu.close()

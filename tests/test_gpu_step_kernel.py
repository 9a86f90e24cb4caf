"""The decode step at the edges of its single-launch form (one stream, or several whose sums fit a
CTA's registers), of the kernels beyond them, and of the multi-stream predictor: widths and stream
counts on both sides of each limit, ranks around the two forms of the first predictor stage, fewer new
neurons than fetch CTAs, more than a ring holds, refused updates."""
import copy

import numpy as np
import pytest
import torch

from paper_2312_11514_b200 import binding as B
from paper_2312_11514_b200 import workloads as W

import parity_util as P

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _steps(cfg, **kw):
    gpu, ora = P.make_layer_pair(cfg, 0, b_down=True, **kw)
    X = W.make_inputs(cfg, device=DEV)
    y = torch.empty(cfg.n_streams, cfg.d_model, dtype=torch.float32, device=DEV)
    sc, sf = torch.cuda.Stream(), torch.cuda.Stream()
    torch.cuda.synchronize()
    loads = []
    for t in range(cfg.steps):
        B.lif_decode_step(gpu.handle, X[t], y, sc, sf)
        loads.append(len(P.check_decode_step(gpu, ora, X[t].cpu().numpy(), y)["load_ids"]))
        P.compare_cache_rows(gpu, ora)
    gpu.close()
    return loads


@pytest.mark.parametrize("append_first", [0, 1])
@pytest.mark.parametrize("S,d,F,r,fire,gate_mode", [
    (1, 8, 64, 8, 0.20, 0),            # one 16-byte piece per vector
    (1, 4104, 1032, 120, 0.10, 0),     # a thread's second piece begins; tail of the entries
    (1, 8192, 520, 16, 0.10, 1),       # widest rows, three vectors: the smallest ring
    (1, 520, 32768, 136, 0.02, 0),     # most neurons, most cache CTAs (grouped partials)
    (1, 520, 32768, 8, 0.0005, 2),     # fewer new neurons than fetch CTAs, some steps none
    (2, 8192, 520, 128, 0.10, 0),      # two streams: any width
    (3, 1032, 2056, 248, 0.10, 0),     # three in the four-stream form, rank not a multiple of 16
    (4, 8192, 264, 24, 0.10, 0),
    (5, 4096, 1032, 128, 0.06, 0),     # widest row of the eight-stream form
    (5, 4112, 1032, 128, 0.06, 0),     # beyond it: tensor cores, cached rows beside the fetch
    (7, 1040, 4104, 2048, 0.03, 0),    # largest rank
    (8, 4096, 2056, 120, 0.05, 0),
    (8, 7168, 1032, 256, 0.05, 0),
    (4, 1040, 2056, 40, 0.08, 2),      # resident gate, several streams
])
def test_decode_step_at_the_edges(S, d, F, r, fire, gate_mode, append_first):
    act, thr = (B.ACT_FATRELU, 0.05) if gate_mode else (B.ACT_RELU, 0.0)
    cfg = W.LifConfig("edges", 1, d, F, r, 2, S, 7, fire, 1.0, 0.7, 0.7, 71)
    loads = _steps(cfg, capacity=F if F <= 2056 else None, append_first=append_first,
                   gate_mode=gate_mode, activation=act, act_threshold=thr)
    assert sum(loads) > 0


@pytest.mark.parametrize("S,d", [(1, 1032), (3, 1032), (2, 4096)])       # (the last: rows handed over)
def test_a_refused_update_brings_nothing_in_and_the_next_step_follows_the_oracle(S, d):
    cfg = W.LifConfig("refused", 1, d, 4096, 32, 3, S, 8, 0.04, 1.0, 0.8, 0.6, 72)
    gpu, ora = P.make_layer_pair(cfg, 0, b_down=True, append_first=1, capacity=1500)
    X = W.make_inputs(cfg, device=DEV)
    y = torch.empty(S, cfg.d_model, dtype=torch.float32, device=DEV)
    sc, sf = torch.cuda.Stream(), torch.cuda.Stream()
    torch.cuda.synchronize()
    for t in range(cfg.steps):
        B.lif_decode_step(gpu.handle, X[t], y, sc, sf)
        P.check_decode_step(gpu, ora, X[t].cpu().numpy(), y)
        before = gpu.lists()
        B.lif_decode_step(gpu.handle, (X[t] * 30).half(), y, sc, sf)   # about half of all neurons
        after = gpu.lists()
        assert after["status"] == B.LIF_ERR_CAPACITY and len(after["load_ids"]) == 0
        for key in ("pointers", "slot_of", "last_active", "num_used", "step"):
            np.testing.assert_array_equal(after[key], before[key])
        P.compare_cache_rows(gpu, ora)
        want = np.tile(gpu.keep["bias_down"].float().cpu().numpy(), (S, 1))
        np.testing.assert_array_equal(y.cpu().numpy(), want)
        B.lif_clear_status(gpu.handle)
    gpu.close()


def test_steps_of_more_layers_than_the_chip_holds_at_a_time():
    # Eight layers on streams of their own and of several priorities: their steps together have more CTAs
    # than there are SMs, and rows of 16 KB leave room for one CTA on an SM.  Every CTA of a step must get by
    # without those that have not started yet; outputs and state are those of the layers run one by one.
    cfg = W.LifConfig("together", 8, 4096, 2048, 32, 3, 1, 10, 0.08, 1.0, 0.8, 0.6, 73)
    pairs = [P.make_layer_pair(cfg, l, b_down=True, append_first=l % 2) for l in range(cfg.n_layers)]
    X = W.make_inputs(cfg, device=DEV)
    greatest = torch.cuda.Stream.priority_range()[1]
    streams = [torch.cuda.Stream(priority=max(greatest, -(l % 4))) for l in range(cfg.n_layers)]
    y = torch.empty(2, cfg.steps, cfg.n_layers, cfg.d_model, dtype=torch.float32, device=DEV)
    state = []
    for together in (0, 1):
        torch.cuda.synchronize()
        for t in range(cfg.steps):
            for l, (gpu, _) in enumerate(pairs):
                B.lif_decode_step(gpu.handle, X[t], y[together, t, l], streams[l if together else 0], None)
        torch.cuda.synchronize()
        state.append([gpu.lists() for gpu, _ in pairs])
        for gpu, _ in pairs:
            B.lif_reset(gpu.handle)
    assert torch.equal(y[0], y[1])
    for one, other in zip(*state):
        assert one["status"] == other["status"] == B.LIF_OK and one["step"] == cfg.steps
        for key in ("pointers", "slot_of", "last_active"):
            np.testing.assert_array_equal(one[key], other[key])
    for gpu, _ in pairs:
        gpu.close()


@pytest.mark.parametrize("S,gate_mode,append_first", [(1, 0, 0), (1, 2, 1), (3, 0, 1)])
def test_other_tokens_after_a_restore_do_not_meet_words_of_runs_of_the_same_number(S, gate_mode, append_first):
    # the rows and gate values that the predictor stores beside its entries carry its run's number, which a
    # restore puts back: with other tokens the same numbers belong to other rows
    act, thr = (B.ACT_FATRELU, 0.05) if gate_mode else (B.ACT_RELU, 0.0)
    cfg = W.LifConfig("again", 1, 520, 4096, 32, 3, S, 9, 0.08, 1.0, 0.3, 0.95, 74)
    gpu, ora = P.make_layer_pair(cfg, 0, b_down=True, append_first=append_first, gate_mode=gate_mode,
                                 activation=act, act_threshold=thr)
    X = W.make_inputs(cfg, device=DEV)
    y = torch.empty(S, cfg.d_model, dtype=torch.float32, device=DEV)
    torch.cuda.synchronize()

    def run(tokens):
        for t in tokens:
            B.lif_decode_step(gpu.handle, X[t], y)
            P.check_decode_step(gpu, ora, X[t].cpu().numpy(), y)
            P.compare_cache_rows(gpu, ora)

    run(range(3))
    snap, cache = B.lif_snapshot(gpu.handle), copy.deepcopy(ora.cache)
    run(range(3, 6))
    B.lif_restore(gpu.handle, snap)
    ora.cache = cache
    run(range(6, 9))
    gpu.close()


@pytest.mark.parametrize("S,d,fire", [
    (2, 4096, 0.003),     # every new neuron is its fetch CTA's only one: its row is handed over
    (2, 4096, 0.04),      # several rows a CTA, the last one handed over
    (4, 2048, 0.01),
    (3, 1032, 0.01),      # not handed over
])
def test_a_down_column_is_not_read_by_a_stream_in_which_its_neuron_is_off(S, d, fire):
    # infinities in the down columns of neurons that are off in stream 0: its output stays, bit for bit,
    # wherever in the load list the neuron is
    cfg = W.LifConfig("off", 1, d, 2048, 32, 3, S, 2, fire, 1.0, 0.8, 0.6, 78)
    gpu, ora = P.make_layer_pair(cfg, 0, b_down=True, capacity=cfg.d_ff, append_first=1)
    X = W.make_inputs(cfg, device=DEV)
    y = torch.empty(2, S, d, dtype=torch.float32, device=DEV)
    gpu.keep["bias_up"].zero_()                    # on in about every second stream
    ora.bias_up[:] = 0
    torch.cuda.synchronize()
    B.lif_decode_step(gpu.handle, X[0], y[0])
    lists = P.check_decode_step(gpu, ora, X[0].cpu().numpy(), y[0])
    x = X[0].cpu().numpy().astype(np.float64)
    pre = x @ ora.bundles[lists["load_ids"], :d].astype(np.float64).T
    off = lists["load_ids"][(pre[0] < -1e-3) & (pre[1:] > 1e-3).any(axis=0)]
    assert len(off) > 0
    gpu.keep["host_bundles"][torch.from_numpy(off.astype(np.int64)), d:] = float("inf")
    B.lif_reset(gpu.handle)
    torch.cuda.synchronize()
    B.lif_decode_step(gpu.handle, X[0], y[1])
    torch.cuda.synchronize()
    assert torch.equal(y[0, 0], y[1, 0])
    assert torch.isinf(y[1, 1:]).any()
    gpu.close()


@pytest.mark.parametrize("F,cap,one", [
    (16384, 16384, True),     # a row for every neuron
    (18176, 18176, True),
    (32768, 11999, True),     # the largest caches: 4 * d_ff + 8 * capacity bytes in a CTA's shared memory
    (32768, 12100, False),    # beyond them
])
def test_layers_with_large_caches_are_one_launch(F, cap, one):
    # only the single launch has CTAs that wait for one another, so with no polls its steps end in a timeout
    cfg = W.LifConfig("large", 1, 8, F, 8, 4, 1, 7, 0.05, 1.0, 0.5, 0.8, 79)
    gpu, ora = P.make_layer_pair(cfg, 0, b_down=True, capacity=cap, append_first=1)
    X = W.make_inputs(cfg, device=DEV)
    y = torch.empty(1, cfg.d_model, dtype=torch.float32, device=DEV)
    for t in range(cfg.steps):
        none = t == 4
        if none:
            B.lif_set_tuning(gpu.handle, B.TUNE_STEP_POLLS, 0)
        B.lif_decode_step(gpu.handle, X[t], y)
        if none:
            B.lif_set_tuning(gpu.handle, B.TUNE_STEP_POLLS, 1 << 20)
            assert (gpu.lists()["status"] == B.LIF_ERR_TIMEOUT) == one
        if none and one:
            lists = ora.cache.window_update(gpu.lists()["active_idx"])
            ora.cache.insert(lists, ora.bundles, ora.bias_up)
            B.lif_clear_status(gpu.handle)
        else:
            lists = P.check_decode_step(gpu, ora, X[t].cpu().numpy(), y)
        assert len(lists["load_ids"]) > 0 and (t < 4 or len(lists["evict_ids"]) > 0)
        torch.cuda.synchronize()
        P.compare_cache_rows(gpu, ora)
    gpu.close()

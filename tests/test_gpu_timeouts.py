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


def _rows_after_the_step(gpu, ora):
    """The window state and every cached row are the oracle's after a step that timed out."""
    g = gpu.lists()
    assert g["status"] == B.LIF_ERR_TIMEOUT
    lists = ora.cache.window_update(g["active_idx"])
    ora.cache.insert(lists, ora.bundles, ora.bias_up)
    for key in P.LIST_KEYS:
        np.testing.assert_array_equal(g[key], lists[key], err_msg=key)
    np.testing.assert_array_equal(g["pointers"], ora.cache.pointers)
    np.testing.assert_array_equal(g["slot_of"], ora.cache.slot_of)
    P.compare_cache_rows(gpu, ora)
    return lists


@pytest.mark.parametrize("d,n_new", [(264, "many"), (8192, "few")])
def test_bundles_whose_copies_are_given_up_are_fetched_all_the_same(d, n_new):
    # a cold start, so that a CTA has more rows than its ring holds, or wide rows: two in flight
    cfg = W.LifConfig("fetch", 1, d, 4096 if n_new == "many" else 512, 16, 3, 1, 4, 0.15, 1.0, 0.8, 0.6, 92)
    gpu, ora = P.make_layer_pair(cfg, 0, b_down=True, capacity=cfg.d_ff)
    X, bufs = W.make_inputs(cfg, device=DEV), P.make_bufs(gpu)
    B.lif_predict(gpu.handle, X[0], None, bufs["act"], bufs["n_act"])
    B.lif_window_update(gpu.handle, bufs["act"], bufs["n_act"])
    B.lif_set_tuning(gpu.handle, B.TUNE_WAIT_POLLS, 0)
    B.lif_fetch_bundles(gpu.handle)
    B.lif_set_tuning(gpu.handle, B.TUNE_WAIT_POLLS, POLLS)
    assert len(_rows_after_the_step(gpu, ora)["load_ids"]) > (16 * 14 if n_new == "many" else 16)
    B.lif_clear_status(gpu.handle)
    P.staged_step(gpu, ora, X[1], bufs)
    gpu.close()


@pytest.mark.parametrize("append_first", [0, 1])
def test_early_copies_given_up_beyond_the_single_launch(append_first):
    # three streams with a resident gate: the fetch is a kernel of its own and starts early
    gpu, ora, X, y, streams = _layer(S=3, gate_mode=B.GATE_RESIDENT, activation=B.ACT_FATRELU,
                                     act_threshold=0.05, append_first=append_first)
    B.lif_set_tuning(gpu.handle, B.TUNE_WAIT_POLLS, 0)
    B.lif_decode_step(gpu.handle, X[3], y, *streams)
    B.lif_set_tuning(gpu.handle, B.TUNE_WAIT_POLLS, POLLS)
    _rows_after_the_step(gpu, ora)
    B.lif_clear_status(gpu.handle, streams[0])
    B.lif_decode_step(gpu.handle, X[4], y, *streams)
    P.check_decode_step(gpu, ora, X[4].cpu().numpy(), y)
    gpu.close()


def test_staged_bundles_of_a_file_store_whose_copies_are_given_up(tmp_path):
    cfg = W.LifConfig("file", 1, 264, 1000, 16, 3, 1, 6, 0.15, 1.0, 0.8, 0.6, 93)
    path = str(tmp_path / "bundles.bin")
    gpu, ora = P.make_layer_pair(cfg, 0, b_down=True, store_file=path)
    store = B.lif_store_open(path, cfg.d_ff, 4 * cfg.d_model, n_threads=4, direct_io=False)
    X = W.make_inputs(cfg, device=DEV)
    y = torch.empty(1, cfg.d_model, dtype=torch.float32, device=DEV)
    B.lif_set_tuning(gpu.handle, B.TUNE_WAIT_POLLS, 0)
    B.lif_decode_step_store(gpu.handle, store, X[0], y)
    B.lif_set_tuning(gpu.handle, B.TUNE_WAIT_POLLS, POLLS)
    _rows_after_the_step(gpu, ora)
    B.lif_clear_status(gpu.handle)
    B.lif_decode_step_store(gpu.handle, store, X[1], y)
    P.check_decode_step(gpu, ora, X[1].cpu().numpy(), y)
    P.compare_cache_rows(gpu, ora)
    B.lif_store_close(store)
    gpu.close()


@pytest.mark.parametrize("append_first", [0, 1])
@pytest.mark.parametrize("S,d,F,gate_mode", [
    (1, 264, 4096, B.GATE_NONE),     # a ring of 16 stages
    (1, 8192, 1024, B.GATE_BUNDLED),   # two stages of 48 KB
    (1, 1032, 4096, B.GATE_RESIDENT),
    (5, 1032, 4096, B.GATE_NONE),
    (5, 2056, 4096, B.GATE_NONE),    # last rows handed over, never reached
    (4, 2056, 128, B.GATE_NONE),     # ... the only row of its fetch CTA
])
def test_the_single_launch_fills_rows_whose_copies_it_gave_up(S, d, F, gate_mode, append_first):
    act, thr = (B.ACT_FATRELU, 0.05) if gate_mode else (B.ACT_RELU, 0.0)
    gpu, ora, X, y, streams = _layer(S=S, steps=0, d=d, F=F, gate_mode=gate_mode,
                                     activation=act, act_threshold=thr, append_first=append_first)
    for t in range(6):               # cold (more rows than a ring) and warm (rows of others move) in turn
        lost = t % 2 == 0
        B.lif_set_tuning(gpu.handle, B.TUNE_WAIT_POLLS, 0 if lost else POLLS)
        B.lif_decode_step(gpu.handle, X[t], y, *streams)
        if lost:
            _rows_after_the_step(gpu, ora)
            B.lif_clear_status(gpu.handle, streams[0])
        else:
            P.check_decode_step(gpu, ora, X[t].cpu().numpy(), y)
            P.compare_cache_rows(gpu, ora)
    gpu.close()


def test_cached_rows_whose_copies_were_given_up_leave_the_layer_usable():
    # every neuron active: 1024 cached rows of 32 KB, three rounds of a cache CTA's ring
    cfg = W.LifConfig("rounds", 1, 8192, 1024, 16, 3, 1, 3, 0.3, 0.3, 0.5, 0.6, 94)
    gpu, ora = P.make_layer_pair(cfg, 0, capacity=cfg.d_ff, theta=-1e30, b_down=True)
    X = W.make_inputs(cfg, device=DEV)
    y = torch.empty(1, cfg.d_model, dtype=torch.float32, device=DEV)
    B.lif_decode_step(gpu.handle, X[0], y)
    P.check_decode_step(gpu, ora, X[0].cpu().numpy(), y)
    B.lif_set_tuning(gpu.handle, B.TUNE_WAIT_POLLS, 0)
    B.lif_decode_step(gpu.handle, X[1], y)
    B.lif_set_tuning(gpu.handle, B.TUNE_WAIT_POLLS, POLLS)
    assert len(_rows_after_the_step(gpu, ora)["hit_slots"]) == cfg.d_ff
    want = gpu.keep["bias_down"].float().cpu().numpy()[None]     # no CTA went past its first round
    np.testing.assert_array_equal(y.cpu().numpy(), want)
    B.lif_clear_status(gpu.handle)
    B.lif_decode_step(gpu.handle, X[2], y)
    P.check_decode_step(gpu, ora, X[2].cpu().numpy(), y)
    gpu.close()


@pytest.mark.parametrize("S,d,gate_mode,ffn_mode,append_first", [
    (1, 1032, B.GATE_NONE, 0, 0), (1, 1032, B.GATE_NONE, 0, 1), (1, 1032, B.GATE_NONE, 1, 0),
    (1, 1032, B.GATE_BUNDLED, 0, 0), (1, 1032, B.GATE_BUNDLED, 0, 1), (4, 1032, B.GATE_NONE, 0, 0),
    (4, 1032, B.GATE_NONE, 0, 1),
    (4, 2056, B.GATE_NONE, 0, 0), (4, 2056, B.GATE_NONE, 0, 1)])     # last rows handed over
def test_rows_named_by_a_step_whose_parts_gave_up_are_read_again_when_the_status_is_cleared(
        S, d, gate_mode, ffn_mode, append_first):
    # Every wait of a CTA for another gives up at once: the window CTA commits the plan, no row of it is
    # moved or brought in.  No copy is left behind: those asked for ahead of the plan are waited for.
    gpu, ora, X, y, streams = _layer(S=S, steps=0 if ffn_mode else 4, d=d, gate_mode=gate_mode, ffn_mode=ffn_mode,
                                     append_first=append_first)
    for t in range(4 if ffn_mode else 0):
        B.lif_decode_step(gpu.handle, X[t], y, *streams)
        lists = ora.cache.window_update(gpu.lists()["active_idx"])
        ora.cache.insert(lists, ora.bundles, ora.bias_up)
    P.compare_cache_rows(gpu, ora)
    B.lif_set_tuning(gpu.handle, B.TUNE_STEP_POLLS, 0)
    B.lif_decode_step(gpu.handle, X[4], y, *streams)
    B.lif_set_tuning(gpu.handle, B.TUNE_STEP_POLLS, 1 << 20)
    g = gpu.lists()
    assert g["status"] == B.LIF_ERR_TIMEOUT
    lists = ora.cache.window_update(g["active_idx"])
    ora.cache.insert(lists, ora.bundles, ora.bias_up)
    for key in P.LIST_KEYS:
        np.testing.assert_array_equal(g[key], lists[key], err_msg=key)
    assert len(lists["load_ids"]) > 0 and (append_first or len(lists["move_src"]) > 0)
    rows = gpu.cache[torch.tensor(lists["load_slots"], device=DEV).long()].cpu().numpy()
    assert not np.array_equal(rows, ora.bundles[lists["load_ids"]])          # nothing has come in
    B.lif_decode_step(gpu.handle, X[5], y, *streams)                         # refused
    after = gpu.lists()
    assert after["status"] == B.LIF_ERR_TIMEOUT and after["step"] == g["step"]
    np.testing.assert_array_equal(after["pointers"], g["pointers"])
    B.lif_clear_status(gpu.handle, streams[0])
    torch.cuda.synchronize()
    P.compare_cache_rows(gpu, ora)
    B.lif_decode_step(gpu.handle, X[5], y, *streams)
    g = gpu.lists()
    assert g["status"] == B.LIF_OK
    if ffn_mode == 0:
        P.check_decode_step(gpu, ora, X[5].cpu().numpy(), y)
    else:                                                                    # FFN over every cached row
        lists = ora.cache.window_update(g["active_idx"])
        ora.cache.insert(lists, ora.bundles, ora.bias_up)
        ref, flips = P.ffn_reference(ora, np.arange(ora.cache.num_used), X[5].cpu().numpy())
        P.assert_y_close(y.cpu().numpy().astype(np.float64), ref, flips)
    P.compare_cache_rows(gpu, ora)
    with pytest.raises(B.LifError):
        B.lif_set_tuning(gpu.handle, B.TUNE_STEP_POLLS, -1)
    gpu.close()


def test_clearing_another_status_leaves_the_cached_rows_alone():
    gpu, ora, X, y, streams = _layer()
    marked = torch.full_like(gpu.cache[0], 7.0)
    gpu.cache[0].copy_(marked)
    bad = torch.tensor([-1], dtype=torch.int32, device=DEV)
    B.lif_sparse_ffn(gpu.handle, X[0], bad, torch.ones(1, dtype=torch.int32, device=DEV), y)
    assert B.lif_get_stats(gpu.handle).status == B.LIF_ERR_INVALID_ARG
    B.lif_clear_status(gpu.handle)
    assert B.lif_get_stats(gpu.handle).status == B.LIF_OK
    assert torch.equal(gpu.cache[0], marked)
    gpu.close()

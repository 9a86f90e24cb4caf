"""The work that is measured: one decoded token through a stack of FFN layers, by every route a
user's program has for it, over the range of shapes and options the library takes.

A case names the shape of a layer (`d_model`, `d_ff`, `rank`), the stack (`layers`), the window
(`window_k`, `streams`, and for speculative decoding the kept tokens `keep`), the workload (`fire`:
mean share of active neurons per stream, `sigma`: spread of the neurons' popularity, `rho`:
correlation of consecutive tokens), the options of the layer description, and the `route`:

  graph   the token's input is put into the graph's input buffer, then lif_graph_launch
  host    lif_graph_launch_host: pinned input in, all layers' outputs back, synchronised
  steps   lif_decode_step layer by layer, as a program does that has attention in between
  staged  lif_predict, lif_window_update, lif_fetch_bundles and lif_sparse_ffn, one by one

A state is a stack in the middle of a sequence: its window is full before the first pass, and every
pass decodes the sequence's next token (back and forth over the prepared inputs, so that two
consecutive passes always see neighbouring tokens)."""
import math

import numpy as np
import torch

from paper_2312_11514_b200 import binding as B
from paper_2312_11514_b200 import runtime as R
from paper_2312_11514_b200 import workloads as W

TOKENS = 32            # prepared inputs per state

PLAIN = dict(route="graph", layers=4, d_model=4096, d_ff=16384, rank=128, window_k=5, streams=1,
             keep=0, fire=0.03, sigma=1.0, rho=0.9, gate=B.GATE_NONE, activation=B.ACT_RELU,
             threshold=0.0, whole_cache=0, budget=0.0, append_first=1)


def _case(name, **kw):
    assert set(kw) <= set(PLAIN), kw
    return dict(PLAIN, name=name, **kw)


def _config(name, **kw):
    """A case with the shape and workload of one of the named configurations."""
    c = W.CONFIGS[name]
    return dict(d_model=c.d_model, d_ff=c.d_ff, rank=c.rank, window_k=c.window_k,
                streams=c.n_streams, fire=c.mean_fire, sigma=c.sigma_pop, rho=c.rho, **kw)


def listed():
    return [
        # the smallest stack there is: latency and launches
        _case("tiny_graph", **_config("tiny", layers=2)),
        # a small model driven layer by layer from the host
        _case("small_steps", route="steps", d_model=768, d_ff=3072, rank=64, fire=0.05),
        # the headline: a token of the OPT-6.7B-shaped stack as one graph
        _case("opt6p7b_graph", **_config("opt6p7b", layers=8)),
        # the same layers end to end from host buffers, as the paper writes them: cache operations
        # in its order, FFN over every cached row, squared ReLU, memory-budgeted window
        _case("opt6p7b_host_budget", **_config(
            "opt6p7b", route="host", activation=B.ACT_RELU_SQUARED, whole_cache=1, budget=0.7,
            append_first=0)),
        # the four calls of the method one by one on one stream
        _case("opt6p7b_staged", **_config("opt6p7b", route="staged")),
        # speculative decoding: five tokens in one pass, three of them kept
        _case("opt6p7b_speculative", **dict(_config("opt6p7b", layers=2, keep=3), streams=5)),
        # a width that is no power of two, heavier-tailed popularity
        _case("falcon7b_graph", **_config("falcon7b")),
        # dense activations and little reuse, layer by layer (attention in between)
        _case("phi2_steps", **_config("phi2", route="steps")),
        # gated FFN, the gate row in the bundle
        _case("llama2_7b_gate_bundled", **_config("llama2_7b", gate=B.GATE_BUNDLED)),
        # gated FFN, the gate projection resident and used as the predictor
        _case("llama2_7b_gate_resident", **_config(
            "llama2_7b", gate=B.GATE_RESIDENT, activation=B.ACT_FATRELU, threshold=0.1)),
        # several sequences with a ragged width (not a multiple of 16)
        _case("ragged_streams_steps", route="steps", d_model=1544, d_ff=6168, rank=72, window_k=3,
              streams=3, fire=0.06, rho=0.8),
        # the largest: eight sequences
        _case("batched8_graph", **_config("batched8", layers=2)),
    ]


def draw(rng):
    """Another case of the same ranges: every route, gate form and option; widths 256 to 8192,
    one to eight streams; sizes are multiples of 8 spread over their logarithm."""
    def spread(lo, hi, step=8):
        return step * max(1, round(math.exp(rng.uniform(math.log(lo), math.log(hi))) / step))

    largest = work(next(c for c in listed() if c["name"] == "batched8_graph"))["bytes"]
    while True:
        d = spread(256, 8192)
        c = dict(PLAIN, route=rng.choice(["graph", "graph", "steps", "staged", "host"]),
                 layers=rng.randint(1, 6), d_model=d,
                 d_ff=min(32768, 8 * round(d * rng.uniform(2.5, 4.5) / 8)), rank=spread(16, 256),
                 window_k=rng.randint(1, 8), fire=round(math.exp(rng.uniform(math.log(0.02), math.log(0.1))), 4),
                 sigma=rng.choice([1.0, 1.5]), rho=round(rng.uniform(0.7, 0.95), 3))
        kind = rng.choice(["plain", "plain", "bundled", "resident", "streams", "streams", "speculative",
                           "whole"])
        if kind == "bundled":
            c.update(gate=B.GATE_BUNDLED)
        elif kind == "resident":
            c.update(gate=B.GATE_RESIDENT, activation=B.ACT_FATRELU, threshold=0.1)
        elif kind == "streams":
            c.update(streams=rng.randint(2, 8))
        elif kind == "speculative":
            c.update(streams=rng.randint(2, 6))
            c.update(keep=rng.randint(1, c["streams"]))
        elif kind == "whole":
            c.update(whole_cache=1, append_first=0, activation=rng.choice([B.ACT_RELU, B.ACT_RELU_SQUARED]))
            if c["window_k"] >= 4:
                c.update(budget=rng.choice([0.0, 0.7]))
        if kind in ("plain", "streams"):
            c.update(append_first=rng.choice([0, 1, 1]))
        store = c["layers"] * c["d_ff"] * _bundle_bytes(c)
        if store <= (2 << 30) and work(c)["bytes"] <= largest:
            return c


def _bundle_bytes(case):
    return 2 * case["d_model"] * (3 if case["gate"] == B.GATE_BUNDLED else 2)


def _lif_config(case, seed):
    return W.LifConfig("case", case["layers"], case["d_model"], case["d_ff"], case["rank"],
                       case["window_k"], case["streams"], TOKENS, case["fire"], case["sigma"],
                       case["rho"], math.sqrt(1.0 - case["rho"] ** 2), seed)


def _capacity(case):
    """Rows of every layer's cache: a function of the shape, so that all seeds have the same; the
    margin is twice the usual one because the seeds' popularities differ."""
    cfg = _lif_config(case, 0)
    return W.window_capacity(cfg, W.popularity(cfg, 0), margin_sigmas=16.0)


_streams = {}


def _stream(name):
    """The program's two streams: one for everything, one for what overlaps the fetch."""
    if name not in _streams:
        _streams[name] = torch.cuda.Stream()
    return _streams[name]


class Program:
    """What a decoding program keeps: the layers, their inputs and outputs, the graph."""

    def __init__(self, case, seed):
        cfg = _lif_config(case, seed)
        S, d, L = cfg.n_streams, cfg.d_model, cfg.n_layers
        self.route, self.gate = case["route"], case["gate"]
        self.compute, self.fetch = _stream("compute"), _stream("fetch")
        self.graph = None
        self.layers = []
        cap = _capacity(case)
        for l in range(L):
            store = R.pinned_store(cfg.d_ff, d, _bundle_bytes(case) // (2 * d))
            w = W.make_layer(cfg, l, device="cuda", bundles_out=store, gate_mode=case["gate"],
                             act_threshold=case["threshold"])
            self.layers.append(R.Layer(
                d_model=d, d_ff=cfg.d_ff, rank=cfg.rank, window_k=cfg.window_k, capacity=cap,
                host_bundles=store, bias_up=w["bias_up"], pred_A=w["A"], pred_B=w["B"],
                pred_c=w["c"], n_streams=S, ffn_mode=case["whole_cache"],
                activation=case["activation"], activation_threshold=case["threshold"],
                budget_rows=int(cap * case["budget"]), spec_keep=case["keep"],
                gate_mode=case["gate"], gate=w.get("gate"), append_first=case["append_first"]))
        if case["keep"]:     # consecutive tokens of one sequence, `keep` of them new each pass
            seq = W.make_inputs(cfg.scaled(n_streams=1, steps=TOKENS * case["keep"] + S), device="cuda")
            xs = torch.stack([seq[t * case["keep"]:t * case["keep"] + S, 0] for t in range(TOKENS)])
        else:
            xs = W.make_inputs(cfg, device="cuda")
        if self.route == "host":
            pinned = torch.empty(xs.shape, dtype=xs.dtype, pin_memory=True)
            xs = pinned.copy_(xs)
        self.order = list(xs.unbind(0)) + list(xs.unbind(0))[-2:0:-1]
        self.x = torch.empty(S, d, dtype=torch.float16, device="cuda")
        self.y = torch.empty(L, S, d, dtype=torch.float32, device="cuda")
        self.y_of = list(self.y.unbind(0))
        self.host_y = torch.empty(L, S, d, dtype=torch.float32, pin_memory=True) if self.route == "host" else None
        self.active = torch.empty(cfg.d_ff, dtype=torch.int32, device="cuda")
        self.n_active = torch.zeros(1, dtype=torch.int32, device="cuda")
        self.lists = [B.lif_get_lists(layer.handle) for layer in self.layers]
        self.at = 0
        torch.cuda.synchronize()
        if self.route in ("graph", "host"):
            self.graph = B.lif_graph_capture([layer.handle for layer in self.layers], self.x, self.y,
                                             self.compute, self.fetch)
        self.outputs = {"y": self.y if self.host_y is None else self.host_y}
        for l, layer in enumerate(self.layers):
            self.outputs[f"layer{l}"] = {
                "pointers": self._int32(l, "pointers", layer.capacity),
                "slot_of": self._int32(l, "slot_of", cfg.d_ff),
                "last_active": self._int32(l, "last_active", cfg.d_ff),
                "cache": layer.cache}
        for _ in range(case["window_k"] + 3):        # the window fills
            self.token()
        for layer in self.layers:
            status = B.lif_get_stats(layer.handle).status
            if status != B.LIF_OK:
                raise RuntimeError("a layer reports: " + B.status_str(status))

    def _int32(self, l, name, n):
        ws = self.layers[l].workspace
        off = getattr(self.lists[l], name) - ws.data_ptr()
        return ws[off:off + 4 * n].view(torch.int32)

    def token(self):
        x = self.order[self.at]
        self.at = (self.at + 1) % len(self.order)
        if self.route == "graph":
            with torch.cuda.stream(self.compute):
                self.x.copy_(x)
            B.lif_graph_launch(self.graph, self.compute)
        elif self.route == "host":
            B.lif_graph_launch_host(self.graph, x, self.host_y, self.compute)
        elif self.route == "steps":
            for layer, y in zip(self.layers, self.y_of):
                B.lif_decode_step(layer.handle, x, y, self.compute, self.fetch)
        else:
            s = self.compute
            for layer, lists, y in zip(self.layers, self.lists, self.y_of):
                B.lif_predict(layer.handle, x, None, self.active, self.n_active, s)
                B.lif_window_update(layer.handle, self.active, self.n_active, s)
                B.lif_fetch_bundles(layer.handle, s)
                B.lif_sparse_ffn(layer.handle, x, lists.active_slots,
                                 lists.counts + 4 * B.CNT_N_ACTIVE, y, s)
        return self.outputs

    def __del__(self):
        if getattr(self, "graph", None):
            torch.cuda.synchronize()
            B.lif_graph_destroy(self.graph)
            self.graph = None


def prepare(case, seed):
    return Program(case, seed)


def run(state):
    return state.token()


def _expected_rows(case):
    """Rows per layer and pass in the steady state: (used by the FFN, of these brought in), from a
    simulation of the workload's marginals (unit normal scores, AR(1) in time, a threshold per
    neuron that gives its popularity)."""
    n, k, S, keep = 4096, case["window_k"], case["streams"], case["keep"]
    rng = np.random.default_rng(0)
    p = np.exp(case["sigma"] * rng.standard_normal(n))
    p = np.minimum(0.95, p * case["fire"] / p.mean())
    theta = -torch.special.ndtri(torch.from_numpy(p)).numpy()[:, None]
    chains = 1 if keep else S
    rho, noise = case["rho"], math.sqrt(1.0 - case["rho"] ** 2)
    score = rng.standard_normal((n, chains))
    tokens = []
    passes = k + 6
    for _ in range(passes * keep + S if keep else passes):
        tokens.append((score > theta).any(axis=1))
        score = rho * score + noise * rng.standard_normal((n, chains))
    used = new = union = count = 0
    cached = np.zeros(n, bool)
    for t in range(passes):
        if keep:
            active = np.any(tokens[t * keep:t * keep + S], axis=0)
            window = np.any(tokens[max(0, t * keep + keep - k):t * keep + keep], axis=0)
        else:
            active = tokens[t]
            window = np.any(tokens[max(0, t - k + 1):t + 1], axis=0)
        if t >= k:
            used, new, count = used + active.sum(), new + (active & ~cached).sum(), count + 1
            union += (window | active).sum()
        cached = window | active
    scale = case["d_ff"] / n / count
    rows = (union if case["whole_cache"] else used) * scale
    if case["budget"]:
        rows = min(rows, case["budget"] * _capacity(case))
    return rows, new * scale


def work(case):
    """Per layer: the predictor's factors (or the gate projection), the rows that come in (read
    from the host store, written to the cache), the other rows of the FFN (read from the cache),
    the input and the output, each once."""
    d, F, r, S, row = case["d_model"], case["d_ff"], case["rank"], case["streams"], _bundle_bytes(case)
    rows, new = _expected_rows(case)
    if case["gate"] == B.GATE_RESIDENT:
        factors, mults = 2 * d * F + 2 * F, S * d * F
    else:
        factors, mults = 2 * d * r + 2 * r * F + 4 * F, S * (d * r + r * F)
    per_layer = factors + 2 * new * row + (rows - new) * row + S * d * 4
    flops = 2 * mults + 2 * S * rows * (row // 2)
    return {"bytes": case["layers"] * per_layer + 2 * S * d, "flops": case["layers"] * flops}


def tolerance(case):
    """Outputs are fp32 sums of products of fp16 values; everything else is whole numbers (the
    window's bookkeeping) or copies (the cached rows) and stays exactly the same."""
    return {"rel": 1e-5, "differ": 0.0}

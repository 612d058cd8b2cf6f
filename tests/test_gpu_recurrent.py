"""The recurrent family on the GPU (the paper's RNN models, Sec. 5.3 / Table 1):
embedding + two LSTM layers (the first returning every step) + dense.  A mutant of an
embedding channel changes that channel at every step (its delta is the table entry of
the step's id); a mutant of an LSTM unit changes the whole layer from the first step on
(the recurrence), so the layer is recomputed for the mutant's rows with the unit's rows
rewritten.  Every operator on every layer against the oracle (logits within the fp32
rule, kill bits exact outside near ties), memoized == vanilla bit for bit, the
unchanged-row elimination exact, identity mutants never killed; the IMDB-sized model of
Table 1 (vocabulary 20,000, width 128, 64 units, 80 steps) on a sample; an id outside the
table is refused."""
import ctypes

import numpy as np
import pytest

from parity_util import compare_kills, logits_close
from paper_2607_18582_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def M():
    from paper_2607_18582_gb300 import build
    build.build()
    from paper_2607_18582_gb300 import mure
    return mure


@pytest.fixture(scope="module")
def ctx(M):
    return M.mure_create(0)


def small_rnn(seed=0):
    return wl.rnn(seed, n_classes=2, vocab=50, dim=8, units=(6, 5), steps=12, name="rnn_small")


def every_operator(model, per_layer, seed):
    subs = []
    for l in range(model.n_layers()):
        ops = tuple(wl.OPS[(l + i) % 6] for i in range(per_layer))
        subs.append(wl.mutants(model, per_layer, seed=seed + l, ratios=(0.3,), ops=ops, layers=[l]))
    return wl.concat(subs)


@pytest.mark.parametrize("size", ["small", "imdb", "reuters"])
def test_recurrent_network_matches_oracle(M, ctx, oracle_mod, size):
    if size == "small":
        model, n_in, per_layer = small_rnn(), 160, 12
    elif size == "imdb":
        model, n_in, per_layer = wl.rnn(), 64, 6
    else:
        # 90 classes: the 96-accumulator output layer and 96-label score sets
        model, n_in, per_layer = wl.rnn_reuters(), 64, 6
    X = wl.inputs(model, n_in, 1)
    table = every_operator(model, per_layer, 70)
    ora = oracle_mod.vanilla(model, X, table)
    m = M.mure_model_load(ctx, model, precision="tf32x3")
    assert [m.layer_kernel(l)[0] for l in range(model.n_layers())][-1] == "output"
    cache = M.mure_build_prefix_cache(m, X)
    lg0, _ = M.mure_cache_outputs(cache)
    ok, worst = logits_close(lg0, ora["orig_logits"])
    assert ok, worst
    r = M.mure_eval_mutants(cache, table, logits=True)
    ok, worst = logits_close(r["logits"], ora["logits"])
    assert ok, worst
    bad, _ = compare_kills(r["kill_bits"], ora["kill_bits"], ora["orig_logits"], ora["logits"], n_in)
    assert bad == 0
    assert r["kill_bits"].any()          # the table kills something
    v = M.mure_eval_vanilla(m, X, table, logits=True)
    assert np.array_equal(v["kill_bits"], r["kill_bits"])
    assert np.array_equal(v["logits"].view(np.uint32), r["logits"].view(np.uint32))
    u = M.mure_eval_mutants(cache, table, logits=True, skip_unchanged=True)
    assert np.array_equal(u["logits"].view(np.uint32), r["logits"].view(np.uint32))
    assert np.array_equal(u["kill_bits"], r["kill_bits"])


@pytest.mark.parametrize("n_in,per_layer", [(1, 4), (65, 7), (200, 40), (1500, 12)])
def test_lstm_split_over_batches(M, ctx, oracle_mod, n_in, per_layer):
    """The LSTM's rows per block, the waves of blocks and the sharing of the input sums follow the
    batch: the same bits from one large batch, many small ones and vanilla; widths that are no
    multiple of 4 and the 64-unit limit; logits against the oracle."""
    model = wl.rnn(3, n_classes=5, vocab=40, dim=13, units=(64, 33), steps=5, name="rnn_odd")
    X = wl.inputs(model, n_in, 2)
    table = every_operator(model, per_layer, 90)
    m = M.mure_model_load(ctx, model)
    cache = M.mure_build_prefix_cache(m, X)
    r = M.mure_eval_mutants(cache, table, logits=True)
    for other in (M.mure_eval_mutants(cache, table, logits=True, workspace_bytes=1 << 20),
                  M.mure_eval_mutants(cache, table, logits=True, skip_unchanged=True),
                  M.mure_eval_vanilla(m, X, table, logits=True)):
        assert np.array_equal(other["logits"].view(np.uint32), r["logits"].view(np.uint32))
        assert np.array_equal(other["kill_bits"], r["kill_bits"])
    some = np.unique(np.linspace(0, n_in - 1, 8).round().astype(np.int64))
    ora = oracle_mod.vanilla(model, X[some], table)
    ok, worst = logits_close(r["logits"][:, some], ora["logits"])
    assert ok, worst


@pytest.mark.parametrize("n_in,vocab", [(1, 2), (70, 129), (300, 129), (300, 700), (70, 4000)])
def test_lstm_sums_by_token(M, ctx, n_in, vocab):
    """The first LSTM's input sums per distinct token (few tokens) or per position (many, or a
    small tile of inputs): the bits of vanilla, which always takes the positions; token counts
    at the edges of a product's 128 rows, every operator on the embedding and the first LSTM."""
    model = wl.rnn(4, n_classes=3, vocab=vocab, dim=13, units=(9, 6), steps=5, name="rnn_tokens")
    X = wl.inputs(model, n_in, 5)
    table = wl.concat([wl.mutants(model, 12, seed=30 + l, ratios=(0.3,), ops=wl.OPS, layers=[l]) for l in (0, 1)])
    m = M.mure_model_load(ctx, model)
    cache = M.mure_build_prefix_cache(m, X)
    v = M.mure_eval_vanilla(m, X, table, logits=True)
    for r in (M.mure_eval_mutants(cache, table, logits=True),
              M.mure_eval_mutants(cache, table, logits=True, workspace_bytes=1 << 19)):
        assert np.array_equal(v["logits"].view(np.uint32), r["logits"].view(np.uint32))
        assert np.array_equal(v["kill_bits"], r["kill_bits"])


def test_recurrent_identity_mutants_and_bad_ids(M, ctx):
    model = small_rnn()
    X = wl.inputs(model, 64, 1)
    rows = []
    for l in range(model.n_layers()):
        rows.append((l, "IDENTITY", [], 0.0, 0))
        rows.append((l, "GF", [0, 1], 0.0, 3))
    m = M.mure_model_load(ctx, model)
    cache = M.mure_build_prefix_cache(m, X)
    lg0, _ = M.mure_cache_outputs(cache)
    r = M.mure_eval_mutants(cache, wl.table_from_rows(rows), logits=True)
    assert not r["kill_bits"].any()
    for i in range(len(rows)):
        assert np.array_equal(r["logits"][i].view(np.uint32), lg0.view(np.uint32))
    bad = X.copy()
    bad[3, 0, 5, 0] = 50.0                 # one id past the table
    with pytest.raises(M.MureError) as ei:
        M.mure_build_prefix_cache(m, bad)
    assert ei.value.status == 1
    # the context stays usable
    again = M.mure_eval_mutants(M.mure_build_prefix_cache(m, X), wl.table_from_rows(rows), logits=True)
    assert np.array_equal(again["logits"].view(np.uint32), r["logits"].view(np.uint32))


def cell_outputs(M, ctx, x):
    """h of one LSTM step on the scalars x, [len(x)][units], one unit per form (biases +-100
    saturate a gate to 1 or 0):
      0: sigmoid(x) tanh(1)   1: tanh(tanh(x))   2: tanh(sigmoid(x))   3, 4, 5: the same with 3e38 x"""
    H, on = 6, 100.0
    W, b = np.zeros((H, 4, 1 + H), np.float32), np.full((H, 4), on, np.float32)
    for u in range(H):
        gate = (3, 2, 0)[u % 3]   # the gates are i, f, g, o
        W[u, gate, 0] = 1.0 if u < 3 else 3e38
        b[u, gate] = 0.0
    net = wl.Model("cell", (1, 1, 1), H)
    net.nodes.append(wl.Node("lstm", (-1,), "none", 0, 1, 1, 0, 1, H, W, b))
    net.nodes.append(wl.Node("dense", (0,), "none", 1, 1, 1, 0, H, H, np.eye(H, dtype=np.float32), np.zeros(H, np.float32)))
    X = np.asarray(x, np.float32).reshape(-1, 1, 1, 1)
    return M.mure_cache_outputs(M.mure_build_prefix_cache(M.mure_model_load(ctx, net), X))[0]


def test_cell_functions(M, ctx):
    """The cell's sigmoid and tanh against 64 bits, over [-100, 100] densely and around 0, the change
    of form at 0.6 (in either place of tanh(tanh(x))) and the clamps.  Bounds: the worst relative
    error that the kernel's comment states, 1.6e-7 each (the inner tanh's arrives damped), and 2^-24
    per product.  The mean matters more than the spread, since a recurrence adds it up."""
    near = lambda v: np.float32(v) * (1 + np.arange(-40, 41, dtype=np.float32) * np.float32(2.0 ** -23))  # noqa: E731
    x = np.concatenate([np.linspace(-100, 100, 200001), np.linspace(-1, 1, 50001)] +
                       [s * near(v) for s in (1, -1) for v in (0.6, np.arctanh(0.6), 40.0, 87.0, 1e-30, 1e-6, 20.0)]).astype(np.float32)
    h = cell_outputs(M, ctx, x).astype(np.float64)
    x64 = x.astype(np.float64)
    u = 2.0 ** -24
    sig, tanh = 1 / (1 + np.exp(-x64)), np.tanh(x64)
    live = x64 >= -87                       # below, sigmoid is 0 (it would be a subnormal number)
    assert not h[~live, 0].any() and not h[~live, 2].any()
    one = cell_outputs(M, ctx, [100.0])[0, 0].astype(np.float64)   # tanh(1), the gate at 1
    assert abs(one / np.tanh(1.0) - 1) <= 2 * 1.6e-7 + 2 * u
    e = h[live, 0] / (one * sig[live]) - 1
    assert np.abs(e).max() <= 1.6e-7 + 2 * u, np.abs(e).max()
    dense = np.abs(x64[live]) <= 20
    assert abs(e[dense].mean()) <= 1e-8 and e[dense].std() <= 6e-8, (e[dense].mean(), e[dense].std())
    with np.errstate(divide="ignore", invalid="ignore"):
        e = np.where(x64 == 0, h[:, 1], h[:, 1] / np.tanh(tanh) - 1)
    assert np.abs(e).max() <= 2 * 1.6e-7 + 2 * u, np.abs(e).max()
    e = h[live, 2] / np.tanh(sig[live]) - 1
    assert np.abs(e).max() <= 2 * 1.6e-7 + 2 * u, np.abs(e).max()


def test_cell_functions_at_the_ends(M, ctx):
    """Signs, zeros, subnormal numbers, infinities and NaN."""
    x = np.array([0.0, -0.0, 1e-40, -1e-40, 1e-45, 200.0, -200.0, 3e38, -3e38], np.float32)
    h = cell_outputs(M, ctx, x)
    tanh1 = cell_outputs(M, ctx, [100.0])[0, 0]
    half = np.float32(0.5) * tanh1
    assert np.abs(h[:5, 0] - half).max() <= 2.0 ** -24 and np.abs(h[:5, 2] - np.tanh(0.5)).max() <= 2.0 ** -23
    # an argument below the normal numbers may come back as 0 of either sign, no more
    assert np.abs(h[:5, 1]).max() <= 1e-40
    assert np.array_equal(h[5:, 0], np.float32([tanh1, 0, tanh1, 0]))
    assert np.allclose(h[5:, 1], np.tanh(1.0) * np.float32([1, -1, 1, -1]), rtol=5e-7, atol=0)
    # 3e38 x: infinite from |x| >= 2 on
    inf = cell_outputs(M, ctx, np.array([10.0, -10.0], np.float32))
    assert np.array_equal(inf[:, 3], np.float32([tanh1, 0]))
    assert np.allclose(inf[:, 4], np.tanh(1.0) * np.float32([1, -1]), rtol=5e-7, atol=0)
    assert np.allclose(inf[:, 5], np.float32([np.tanh(1.0), 0]), rtol=5e-7, atol=0)
    assert np.isnan(cell_outputs(M, ctx, np.array([np.nan], np.float32))).all()


class CountedMemory:
    """A context whose device memory is counted: `live` and `peak` bytes."""

    def __init__(self, M):
        import torch
        self.live = self.peak = 0
        self.size = {}

        def alloc(n, stream, user):
            p = torch.cuda.caching_allocator_alloc(int(n), 0, int(stream or 0))
            self.size[p] = n
            self.live += n
            self.peak = max(self.peak, self.live)
            return p

        def free(p, stream, user):
            self.live -= self.size.pop(p)
            torch.cuda.caching_allocator_delete(p)

        self.keep = M._Allocator(M._ALLOC_FN(alloc), M._FREE_FN(free), None)
        h = ctypes.c_void_p()
        assert M.lib().mure_create(0, torch.cuda.current_stream().cuda_stream, ctypes.byref(self.keep), ctypes.byref(h)) == 0
        self.ctx = M.Context(h.value, [self.keep])

    def peak_of(self, call):
        """(the call's result, the most bytes it held beyond those held before it)."""
        before = self.peak = self.live
        r = call()
        return r, self.peak - before


@pytest.mark.parametrize("layer", [0, 1, 2, 3])
def test_scratch_within_the_workspace(M, layer):
    """The scratch of a call stays within workspace_bytes (and 4 MiB for the table and the results),
    whichever layers run: with output-layer mutants no LSTM does, so none of its sums (80 KiB a row here)
    are allocated.  Memoized and vanilla give the same bits."""
    model = wl.rnn(3, n_classes=3, vocab=60, dim=8, units=(64, 64), steps=80, name="rnn_scratch")
    X = wl.inputs(model, 256, 2)
    table = wl.mutants(model, 64, seed=5, ratios=(0.02,), ops=("GF", "NAI", "NEB"), layers=[layer])
    mem = CountedMemory(M)
    m = M.mure_model_load(mem.ctx, model)
    cache = M.mure_build_prefix_cache(m, X)
    cap = 32 << 20
    r, peak = mem.peak_of(lambda: M.mure_eval_mutants(cache, table, logits=True, workspace_bytes=cap))
    assert peak <= cap + (4 << 20), peak
    v = M.mure_eval_vanilla(m, X, table, logits=True, workspace_bytes=cap)
    assert np.array_equal(v["logits"].view(np.uint32), r["logits"].view(np.uint32))


@pytest.mark.parametrize("vocab", [60, 1500000])
def test_cache_build_in_parts(M, vocab):
    """Building a cache holds at most 1 GiB of an LSTM's input sums (80 KiB a row here; and 32 MiB for
    the tokens' tables) beside the cache itself: the layer runs in parts.  The logits of inputs in
    every part are those of a cache of these inputs alone; with few tokens, and with more than the
    scratch has sums for."""
    model = wl.rnn(3, n_classes=3, vocab=vocab, dim=4, units=(64, 64), steps=80, name="rnn_parts")
    X = wl.inputs(model, 20000, 2)
    mem = CountedMemory(M)
    m = M.mure_model_load(mem.ctx, model)
    held = mem.live
    cache, peak = mem.peak_of(lambda: M.mure_build_prefix_cache(m, X))
    scratch = peak - (mem.live - held)
    assert scratch <= (1 << 30) + (32 << 20), scratch
    logits, pred = M.mure_cache_outputs(cache)
    cache.free()
    some = np.r_[0:70, 13070:13140, 19940:20000]
    lg, pr = M.mure_cache_outputs(M.mure_build_prefix_cache(m, X[some]))
    assert np.array_equal(lg.view(np.uint32), logits[some].view(np.uint32)) and np.array_equal(pr, pred[some])

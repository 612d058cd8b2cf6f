"""The 1 x 1 convolution kernel of few channels (fp32 on the CUDA cores, from the tensor-core modes the
layers where it is faster):
the same bits as the implicit-GEMM kernel over channel counts, map sizes, residual adds, pooling
tails, the first suffix layer's patch and compacted batches; logits against the oracle."""
import numpy as np
import pytest

from parity_util import logits_close
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


@pytest.mark.parametrize("h,w,ic,oc", [(8, 8, 16, 64), (16, 8, 4, 4), (16, 16, 24, 96), (8, 24, 96, 24), (32, 32, 64, 16),
                                       (8, 16, 128, 32), (16, 16, 36, 100), (8, 8, 20, 12), (12, 12, 16, 32), (16, 8, 64, 128)])
def test_conv1x1_equals_the_generic_kernel(M, ctx, oracle_mod, monkeypatch, h, w, ic, oc):
    b = wl._Builder("conv1x1", (h, w, 3), 6, 21)
    x = b.conv(-1, ic, 3, pad=1)
    y = b.conv(x, oc, 1)                                   # the patch of layer 0 arrives here
    y = b.add(b.conv(y, ic, 1, act="none"), x, act="relu")  # a residual add; skip of layer 0
    y = b.gap(b.conv(y, oc, 1, act="relu6"))
    b.dense(y, 6, act="none")
    X = wl.inputs(b.m, 66, 3)
    table = wl.concat([wl.mutants(b.m, 5, seed=40 + l, ratios=(0.1,), ops=("GF", "NS", "NAI", "WS", "NEB"), layers=[l])
                       for l in range(b.m.n_layers())])
    ora = oracle_mod.vanilla(b.m, X, table)
    m = M.mure_model_load(ctx, b.m, precision="fp32")
    monkeypatch.setenv("MURE_FORCE_GENERIC", "1")
    generic = M.mure_model_load(ctx, b.m, precision="fp32")
    monkeypatch.delenv("MURE_FORCE_GENERIC")
    cache = M.mure_build_prefix_cache(m, X)
    r = M.mure_eval_mutants(cache, table, logits=True)
    ok, worst = logits_close(r["logits"], ora["logits"])
    assert ok, worst
    for other in (M.mure_eval_mutants(M.mure_build_prefix_cache(generic, X), table, logits=True),
                  M.mure_eval_mutants(cache, table, logits=True, skip_unchanged=True),
                  M.mure_eval_mutants(cache, table, logits=True, workspace_bytes=1 << 21),
                  M.mure_eval_vanilla(m, X, table, logits=True)):
        assert np.array_equal(other["logits"].view(np.uint32), r["logits"].view(np.uint32))
    # a tensor-core mode: these layers in fp32 or on the tensor cores, memoized == vanilla bit for bit
    t = M.mure_model_load(ctx, b.m, precision="tf32x3")
    a = M.mure_eval_mutants(M.mure_build_prefix_cache(t, X), table, logits=True)
    ok, worst = logits_close(a["logits"], ora["logits"])
    assert ok, worst
    assert np.array_equal(a["logits"].view(np.uint32),
                          M.mure_eval_vanilla(t, X, table, logits=True)["logits"].view(np.uint32))


@pytest.mark.parametrize("prec", ["tf32x3", "tf32"])
@pytest.mark.parametrize("size,ic,oc,fp32", [
    (8, 16, 64, True), (16, 32, 128, True), (16, 36, 80, True), (16, 40, 80, False), (16, 48, 64, True), (16, 52, 64, False),
    (16, 64, 32, True), (16, 64, 40, False), (16, 64, 64, False), (8, 64, 64, True), (8, 64, 68, False), (16, 80, 32, True),
    (16, 96, 24, True), (16, 96, 32, False), (8, 128, 32, False), (16, 128, 16, False), (16, 64, 12, True)])
def test_which_layers_leave_the_tensor_cores(M, ctx, prec, size, ic, oc, fp32):
    """The line between the two kernels, on both sides; in fp32 it holds for all of them up to 4,096
    products; the bits of vanilla."""
    b = wl._Builder("line", (size, size, 3), 6, 5)
    b.dense(b.gap(b.conv(b.conv(-1, ic, 3, pad=1), oc, 1)), 6, act="none")
    m = M.mure_model_load(ctx, b.m, precision=prec)
    assert (m.layer_kernel(1)[0] == "simt_gemm") == fp32
    X = wl.inputs(b.m, 66, 3)
    table = wl.mutants(b.m, 8, seed=4, ratios=(0.05,), layers=[0])
    r = M.mure_eval_mutants(M.mure_build_prefix_cache(m, X), table, logits=True)
    v = M.mure_eval_vanilla(m, X, table, logits=True)
    assert np.array_equal(v["logits"].view(np.uint32), r["logits"].view(np.uint32))

"""Two host threads with a context each, as the header allows: the launches of one do not depend on
what the other launches.  The amount of dynamic shared memory a kernel may be given is state of the
process, so each pair of calls here needs different amounts for the same kernels."""
import threading

import numpy as np
import pytest

from paper_2607_18582_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def M():
    from paper_2607_18582_gb300 import build
    build.build()
    from paper_2607_18582_gb300 import mure
    return mure


def conv1x1(ic, oc):
    b = wl._Builder("c11", (16, 8, 4), 5, 21)
    b.dense(b.gap(b.conv(b.conv(b.conv(-1, ic, 1), oc, 1), ic, 1)), 5, act="none")
    return b.m


# (network, precision, operators) of either thread
PAIRS = {
    "shuffle": ((wl.mlp(1, (20000, 3, 2)), "fp32", ("WS",)), (wl.mlp(1, (900, 3, 2)), "fp32", ("WS",))),
    "conv1x1": ((conv1x1(128, 32), "fp32", ("NEB",)), (conv1x1(16, 16), "fp32", ("NEB",))),
    "lstm": ((wl.rnn(3, 2, 20, 8, (64, 8), 3), "fp32", ("NEB",)), (wl.rnn(3, 2, 20, 8, (8, 8), 3), "fp32", ("GF",))),
    "output": ((wl.mlp(1, (8, 1000, 10)), "fp32", ("NEB",)), (wl.mlp(1, (8, 64, 10)), "fp32", ("NEB",))),
    "tensor cores": ((wl.mlp(1, (512, 128, 112, 40)), "tf32x3", ("NEB",)), (wl.mlp(1, (16, 16, 16, 40)), "tf32x3", ("NEB",))),
}


@pytest.mark.parametrize("pair", list(PAIRS))
def test_contexts_side_by_side(M, pair):
    import torch
    errors = []
    start = threading.Barrier(2)

    def work(net, prec, ops, n_in):
        try:
            ctx = M.mure_create(0, stream=torch.cuda.Stream(), torch_allocator=False)
            m = M.mure_model_load(ctx, net, precision=prec)
            cache = None if pair == "shuffle" else M.mure_build_prefix_cache(m, wl.inputs(net, n_in, 3))
            table = wl.mutants(net, 4, seed=4, ratios=(0.3,), ops=ops, layers=[0])
            start.wait()
            first = None
            for _ in range(1500 if pair == "shuffle" else 12):
                # (the smallest workspace: a hundred batches of 64 rows in a call)
                r = (M.mure_expand_patches(m, table)[0] if pair == "shuffle" else
                     M.mure_eval_mutants(cache, table, logits=True, workspace_bytes=1)["logits"])
                first = r if first is None else first
                assert np.array_equal(r.view(np.uint32), first.view(np.uint32))
        except BaseException as e:   # noqa: BLE001 - reported by the main thread
            errors.append(e)
            start.abort()

    threads = [threading.Thread(target=work, args=(*how, 3000 if pair == "output" else 9000)) for how in PAIRS[pair]]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors

"""A mixed-precision model that only runs in batches holds no pool of walks of
its own (the batch has one); its first run by itself takes one, and results
are the same bits either way."""
import ctypes as C

import numpy as np
import pytest

from paper_1401_5469_gb300 import synth

pytestmark = pytest.mark.gpu


def test_models_of_a_batch_hold_no_pool():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    from paper_1401_5469_gb300 import mc
    held = {}

    def alloc(nbytes, ctx):
        t = torch.empty(max(int(nbytes), 1), dtype=torch.uint8, device="cuda")
        held[t.data_ptr()] = t
        return t.data_ptr()

    def free(ptr, ctx):
        held.pop(ptr)

    a, f = mc.ALLOC_FN(alloc), mc.FREE_FN(free)
    own = mc.mc_allocator(alloc=a, free=f, ctx=None)
    spec = synth.downbranch_model(n_lines=20_000, n_shells=8, n_packets=20_000)
    n = spec.n_packets
    m = mc.Model(spec, precision=mc.MC_PRECISION_MIXED)  # the descriptors
    h = m.h
    m.h = mc.mc_model_create(m.geom, m.lines, m.atomic, m.run, own, m.stream)
    mc.mc_model_destroy(h)
    m.set_plasma()
    used = lambda: sum(t.numel() for t in held.values())  # noqa: E731
    created = used()
    b = mc.Batch([m])
    b.run_iteration([3], 0, [n], [spec.t_inner], update=False)
    b.synchronize()
    batched, sums = used(), [x.copy() for x in m.estimators(j_blue=True)[:3]]
    b.close()
    m.run_iteration(3, 0, n, spec.t_inner)
    alone, again = used(), m.estimators(j_blue=True)[:3]
    m.run_iteration(3, 1, n, spec.t_inner)
    m.synchronize()
    assert batched == created and alone == used()
    assert 0 < alone - batched <= 152 * 12 * 2 * 128 + 256
    for x, y in zip(sums, again):
        assert np.array_equal(x, y)
    m.close()
    torch.cuda.synchronize()
    assert not held

"""Batches on both sides of the model count from which blocks of 128 threads
take the build without lone walks: every model's estimators are the same bits
as with blocks of 256 threads, which always take that build."""
import numpy as np
import pytest

from paper_1401_5469_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mc():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_1401_5469_gb300 import mc
    return mc


@pytest.mark.parametrize("n_models", [96, 97])
def test_same_bits_with_and_without_lone_walks(mc, n_models):
    specs = [synth.downbranch_model(n_lines=1000 + 37 * (k % 9), n_shells=5 + k % 7, n_packets=200 + 11 * k)
             for k in range(n_models)]
    sums = []
    for block in (128, 256):
        models = [mc.Model(s, precision=mc.MC_PRECISION_MIXED) for s in specs]
        for m in models:
            m.set_plasma()
        batch = mc.Batch(models)
        batch.set_launch(block=block)
        batch.run_iteration([7 + k for k in range(n_models)], 0, [s.n_packets for s in specs],
                            [s.t_inner for s in specs], update=False)
        batch.synchronize()
        sums.append([np.concatenate(m.estimators()[:2]) for m in models])
        batch.close()
        for m in models:
            m.close()
    for a, b in zip(*sums):
        assert np.array_equal(a, b)

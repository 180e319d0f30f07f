"""Walks that end soon gain nothing from running one after the other: a launch
of many walks cut at 300 segments takes no longer in the build with lone walks
and the pool than side by side in the build without (blocks of 256 threads);
batches of short line lists take that build with either block size, and the
two give the same bits on both sides of the line count between them."""
import numpy as np
import pytest

from paper_1401_5469_gb300 import synth

pytestmark = pytest.mark.gpu


def test_many_short_walks_stay_side_by_side():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    from paper_1401_5469_gb300 import mc
    spec = synth.downbranch_model(n_lines=50_000, n_packets=100_000)
    ms = {}
    for block in (128, 256):
        m = mc.Model(spec, precision=mc.MC_PRECISION_MIXED, max_segments=300)
        m.set_plasma()
        b = mc.Batch([m])
        b.set_launch(block=block)
        times = []
        for k in range(10):
            b.run_iteration([k % 2], 0, [spec.n_packets], [spec.t_inner], update=False)
            b.synchronize()
            times.append(b.transport_ms())
        ms[block] = min(times[2:])
        b.close()
        m.close()
    assert ms[128] < 1.3 * ms[256], ms


def _batch(mc, specs, block, reps):
    models = [mc.Model(s, precision=mc.MC_PRECISION_MIXED) for s in specs]
    for m in models:
        m.set_plasma()
    b = mc.Batch(models)
    b.set_launch(block=block)
    times = []
    for _ in range(reps):
        b.run_iteration([7 + k for k in range(len(specs))], 0, [s.n_packets for s in specs],
                        [s.t_inner for s in specs], update=False)
        b.synchronize()
        times.append(b.transport_ms())
    sums = [np.concatenate(m.estimators()[:2]) for m in models]
    b.close()
    for m in models:
        m.close()
    return min(times), sums


def test_batches_of_short_lists_run_side_by_side():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    from paper_1401_5469_gb300 import mc
    specs = [synth.downbranch_model(n_lines=3000 + k, n_shells=12, n_packets=100_000, seed=k) for k in range(8)]
    (t128, s128), (t256, s256) = (_batch(mc, specs, block, 8) for block in (128, 256))
    assert t128 < 1.1 * t256, (t128, t256)  # 4.90 and 4.01 ms in the two builds
    for a, b in zip(s128, s256):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("n_lines", [9_999, 10_000])
def test_same_bits_on_both_sides_of_the_line_count(n_lines):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    from paper_1401_5469_gb300 import mc
    specs = [synth.downbranch_model(n_lines=n, n_shells=9, n_packets=3001, seed=n) for n in (2000, n_lines, 900)]
    for a, b in zip(*(_batch(mc, specs, block, 1)[1] for block in (128, 256))):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("n_models", [96, 97])
def test_same_bits_on_both_sides_of_the_model_count(n_models):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    from paper_1401_5469_gb300 import mc
    specs = [synth.downbranch_model(n_lines=12_000 if k == 5 else 1000 + 37 * (k % 9), n_shells=5 + k % 7,
                                    n_packets=200 + 11 * k) for k in range(n_models)]
    for a, b in zip(*(_batch(mc, specs, block, 1)[1] for block in (128, 256))):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("line_mode,n_lines", [(1, 2000), (1, 5_999), (1, 6_000), (2, 5_999), (2, 6_000)])
def test_single_models_of_short_lists_run_side_by_side(line_mode, n_lines):
    """A model by itself against blocks of 256 threads: the same bits on both
    sides of its own line count, and with a short list (0.87 and 0.69 ms in the
    two builds) about the same time."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    from paper_1401_5469_gb300 import mc
    make = synth.downbranch_model if line_mode == 1 else synth.macroatom_model
    spec = make(n_lines=n_lines, n_shells=20, n_packets=20_000)
    m = mc.Model(spec, precision=mc.MC_PRECISION_MIXED, record_packets=True)
    m.set_plasma()
    times = []
    for _ in range(10):
        m.run_iteration(7, 0, spec.n_packets, spec.t_inner)
        m.synchronize()
        times.append(sum(m.phases()[:2]))
    runs = [(*m.packets(0, spec.n_packets), *m.estimators()[:2])]
    b = mc.Batch([m])
    b.set_launch(block=256)
    batch_times = []
    for _ in range(10):
        b.run_iteration([7], 0, [spec.n_packets], [spec.t_inner], update=False)
        b.synchronize()
        batch_times.append(b.transport_ms())
    runs.append((*m.packets(0, spec.n_packets), *m.estimators()[:2]))
    b.close()
    m.close()
    for x, y in zip(*runs):
        assert np.array_equal(x, y)
    if n_lines == 2000:
        assert min(times) < 1.12 * min(batch_times), (min(times), min(batch_times))

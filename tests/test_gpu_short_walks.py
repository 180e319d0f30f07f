"""Walks that end soon gain nothing from running one after the other: a launch
of many walks cut at 300 segments takes no longer in the build with lone walks
and the pool than side by side in the build without (blocks of 256 threads)."""
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

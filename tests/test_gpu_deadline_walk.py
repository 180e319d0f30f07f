"""A deadline and a long walk alone in its warp: one that does not expire costs
the walk next to nothing (16.58 and 16.62 ms, mixed 25.88 and 26.04), and one
that expires ends it within a fraction of a millisecond."""
import numpy as np
import pytest

from paper_1401_5469_gb300 import synth

pytestmark = pytest.mark.gpu


def _walk_ms(m, pid, n, t_inner):
    ms = []
    for _ in range(6):
        m.run_iteration_range(5469, 0, pid, 1, n, t_inner)
        m.synchronize()
        ms.append(sum(m.phases()[:2]))
    return min(ms)


@pytest.mark.parametrize("precision", [0, 1])
def test_deadline_leaves_a_lone_walk_its_speed_and_ends_it(precision):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    from paper_1401_5469_gb300 import mc
    spec = synth.downbranch_model(n_lines=50_000, n_packets=30_000)
    n = spec.n_packets
    m = mc.Model(spec, precision=precision, record_packets=True)
    m.set_plasma()
    m.run_iteration(5469, 0, n, spec.t_inner)
    pid = int(np.argmax(m.packets(0, n)[3][:, 0]))
    free = _walk_ms(m, pid, n, spec.t_inner)
    m.close()
    assert free > 6.0  # long enough for the deadline below
    m = mc.Model(spec, precision=precision, timeout_ns=60_000_000_000)
    m.set_plasma()
    timed = _walk_ms(m, pid, n, spec.t_inner)
    m.close()
    assert timed < 1.25 * free, (timed, free)
    m = mc.Model(spec, precision=precision, timeout_ns=2_000_000)
    m.set_plasma()
    m.run_iteration_range(5469, 0, pid, 1, n, spec.t_inner)
    with pytest.raises(mc.MCError) as ei:
        m.estimators()
    assert ei.value.code == mc.MC_ERR_TIMEOUT
    assert 2.0 <= sum(m.phases()[:2]) < 4.0
    m.close()

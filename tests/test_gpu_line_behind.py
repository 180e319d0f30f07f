"""Mixed precision: a line behind the packet.

After an electron scattering or a shell crossing the comoving frequency comes
from binary32 positions, so that the next line can lie up to 2^-24 above it:
its path length is negative, and kappa' D of it, which counts in the optical
depth left at the line, is not negligible.  A walk alone in its warp must
decide such a line as a lane of a full warp does.  The model makes the case
common: kappa' = 1e5, lines of depth 0.7 at 1e-5 of each other.  16 x 1200 walks, each alone in its warp (a launch of few packets; a batch with
lone walks), against blocks of 256 threads, which never run a walk alone.
"""
import numpy as np
import pytest

from paper_1401_5469_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("line_mode", [1, 2])
def test_a_walk_alone_decides_lines_behind_it_like_a_full_warp(line_mode):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    from paper_1401_5469_gb300 import mc
    make = synth.downbranch_model if line_mode == 1 else synth.macroatom_model
    spec = make(n_lines=100_000, n_shells=3, n_packets=1200)
    spec.nu = 1.0e15 * np.exp(-1e-5 * np.arange(spec.n_lines))
    spec.n_e = np.full(spec.n_shells, 4.5e12)
    n, seeds, runs = spec.n_packets, range(16), []
    for block in (0, 128, 256):
        m = mc.Model(spec, precision=mc.MC_PRECISION_MIXED, record_packets=True, max_segments=20_000)
        m.set_plasma(tau=np.full((spec.n_shells, spec.n_lines), 0.7))
        b = mc.Batch([m]) if block else None
        if b:
            b.set_launch(block=block)
        out = []
        for seed in seeds:
            if b:
                b.run_iteration([seed], 0, [n], [spec.t_inner], update=False)
                b.synchronize()
            else:
                m.run_iteration(seed, 0, n, spec.t_inner)
            out.append((*m.packets(0, n), *m.estimators()[:2]))
        if b:
            b.close()
        m.close()
        runs.append(out)
    counts = sum(r[3].sum(0) for r in runs[2])
    assert min(counts[3:5]) > 1_000_000  # line events, electron scatterings
    for alone in runs[:2]:
        for r, want in zip(alone, runs[2]):
            for a, b in zip(r, want):
                assert np.array_equal(a, b)


def test_a_batch_that_uses_the_pool_equals_the_build_without_lone_walks():
    """Every packet of 4e5, whose longest walks change warps through the pool."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    from paper_1401_5469_gb300 import mc
    specs = [synth.downbranch_model(n_lines=60_000 + 20_000 * k, n_shells=10 + 3 * k, n_packets=70_000 + 42_000 * k,
                                    seed=40 + k) for k in range(3)]
    packets = [s.n_packets for s in specs]
    models = [mc.Model(s, precision=mc.MC_PRECISION_MIXED, record_packets=True) for s in specs]
    for m in models:
        m.set_plasma()
    runs = []
    for block in (128, 256):
        b = mc.Batch(models)
        b.set_launch(block=block)
        for seed in (11, 12):
            b.run_iteration([seed] * 3, 0, packets, [s.t_inner for s in specs], update=False)
            b.synchronize()
            runs.append([(*m.packets(0, n), *m.estimators(j_blue=True)[:3]) for m, n in zip(models, packets)])
        b.close()
    for m in models:
        m.close()
    for alone, want in zip(runs[:2], runs[2:]):
        for r, w in zip(alone, want):
            for a, b in zip(r, w):
                assert np.array_equal(a, b)

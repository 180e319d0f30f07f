"""v-packets flown by whole warps from their queued launches (Sect. 2.9): the
v-spectrum equals the oracle's where a warp's 32 launches times n_virtual leave
remainders (1, 7, 33 v-packets a launch), with few packets (every walk runs
alone) and with full warps, with and without the cut."""
import numpy as np
import pytest

import oracle
from paper_1401_5469_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_virtual,n_packets,cut", [(1, 37, 0.0), (7, 700, 0.0), (33, 300, 4.0), (2, 60_000, 10.0)])
def test_virtual_spectrum_equals_the_oracle(n_virtual, n_packets, cut):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    from paper_1401_5469_gb300 import mc
    spec = synth.scatter_model(n_lines=1501, n_shells=7, n_packets=n_packets, seed=n_virtual)
    m = mc.Model(spec)
    m.set_plasma(tau=spec.tau)
    m.set_virtual_packets(n_virtual, cut)
    m.run_iteration(3, 1, n_packets, spec.t_inner)
    got, r_got = m.virtual_spectrum(), m.spectrum()[0]
    m.close()
    om = oracle.OracleModel(spec, tau=spec.tau)
    om.set_virtual(n_virtual, cut)
    r = oracle.run_iteration(om, 3, 1, n_packets, spec.t_inner, threads=8, record=False)
    # the sums' own rounding: 1e-9 of a bin, as for the r-packet spectrum
    for a, b in ((got, r.spectrum_v), (r_got, r.spectrum)):
        assert np.all(np.abs(a - b) <= 1e-9 * np.abs(b) + 1e-12 * np.abs(b).max())

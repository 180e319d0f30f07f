"""v-packets of a packet that has just been injected leave in directions mu in
(0, 1] exactly (x_in / x is 1 there), whatever the inner velocity: the
v-spectrum equals the oracle's for inner velocities of which x_in times its
rounded reciprocal is 1 and of which it is not."""
import numpy as np
import pytest

import oracle
from paper_1401_5469_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("v_in", [1.0, 7000.0, 9100.0, 9500.0, 10_300.0, 11_000.0, 12_345.0, 13_700.0, 15_000.0])
def test_virtual_spectrum_for_any_inner_velocity(v_in):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    from paper_1401_5469_gb300 import mc
    spec = synth.scatter_model(n_lines=300, n_shells=4, n_packets=4000, v_in_kms=v_in, v_out_kms=1.7 * v_in)
    m = mc.Model(spec)
    m.set_plasma(tau=spec.tau)
    m.set_virtual_packets(3)
    m.run_iteration(3, 1, spec.n_packets, spec.t_inner)
    got = m.virtual_spectrum()
    m.close()
    om = oracle.OracleModel(spec, tau=spec.tau)
    om.set_virtual(3, 0.0)
    want = oracle.run_iteration(om, 3, 1, spec.n_packets, spec.t_inner, threads=8, record=False).spectrum_v
    # sums of positive terms, each known to 1e-12: 1e-9 of a bin as for the other spectra
    assert np.all(np.abs(got - want) <= 1e-9 * want)

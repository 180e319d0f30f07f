"""v-packets through lines deeper than the fixed-point sum of their depths
holds (512 at a time): the v-spectrum equals the oracle's without a cut, with
cuts above and below the depths, with neighbouring deep lines, and where
negative depths bring a deep sum back."""
import numpy as np
import pytest

import oracle
from paper_1401_5469_gb300 import synth

pytestmark = pytest.mark.gpu


def _deep(spec, negative):
    tau = spec.tau.copy()
    if negative:  # + 560 - 550, from the 10th line of 40 on
        tau[:, 10::40] = 560.0
        tau[:, 11::40] = -550.0
    tau[:, 20::40] = 2000.0
    tau[:, 21::40] = 3000.0
    tau[:, 22::40] = 1.0e5
    tau[:, 30::40] = 400.0  # the fixed-point sum reaches its limit by two of these
    tau[:, 31::40] = 400.0
    return tau


@pytest.mark.parametrize("kind,cut", [("deep", 0.0), ("deep", 700.0), ("deep", 2000.0), ("deep", 1.0e7),
                                      ("negative", 0.0), ("negative", 30.0), ("negative", 1500.0),
                                      ("downbranch", 0.0), ("downbranch", 2000.0)])
def test_virtual_spectrum_with_deep_lines_equals_the_oracle(kind, cut):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    from paper_1401_5469_gb300 import mc
    if kind == "downbranch":
        spec = synth.downbranch_model(n_lines=30_000, n_shells=10, n_packets=1500)
        tau = oracle.plasma_tau(spec, np.full(spec.n_shells, 1.0e4), oracle.geometric_dilution(spec))
        assert np.sum((tau[:, 1:] > 1024) & (tau[:, :-1] > 1024)) > 100
    else:
        spec = synth.scatter_model(n_lines=1501, n_shells=7, n_packets=3000, seed=2)
        tau = _deep(spec, kind == "negative")
    n = spec.n_packets
    m = mc.Model(spec)
    m.set_plasma(tau=tau)
    m.set_virtual_packets(3, cut)
    m.run_iteration(3, 1, n, spec.t_inner)
    got = m.virtual_spectrum()
    m.close()
    om = oracle.OracleModel(spec, tau=tau)
    om.set_virtual(3, cut)
    want = oracle.run_iteration(om, 3, 1, n, spec.t_inner, threads=8, record=False).spectrum_v
    assert np.all(np.isfinite(want)) and np.all(np.isfinite(got)) and np.count_nonzero(want) > 100
    # sums of positive terms; a depth of 1e3 in binary64 is known to 1e-13, and so is its
    # exponential, down to e^-708 (times below 1e42 erg/s a bin), from where the oracle's is 0
    assert want.max() < 1e42 or kind == "negative"
    assert np.all(np.abs(got - want) <= 1e-9 * want + np.exp(-708.0) * 1e42)

"""Caller-owned buffers: a line of depth 0 absorbs nothing, so that its row
number is not looked up -- lines marked with row -1 give what the same lines
give with their own rows (walks alone in their warps, and full warps)."""
import numpy as np
import pytest

from paper_1401_5469_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [300, 20_000])
def test_lines_that_cannot_absorb_need_no_row(n):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    from paper_1401_5469_gb300 import mc
    spec = synth.downbranch_model(n_lines=20_000, n_packets=n)
    S, L, B = spec.n_shells, spec.n_lines, spec.spec_bins
    rng = np.random.default_rng(6)
    none = rng.random(L) < 0.3
    tau = np.exp(-2 + 2 * rng.standard_normal((S, L)))
    tau[:, none] = 0.0
    row = spec.ion.astype(np.int64) * spec.n_levels + spec.upper
    out = []
    for rows in (row, np.where(none, -1, row)):
        def dev(a, t):
            return torch.as_tensor(np.ascontiguousarray(a, dtype=t), device="cuda")
        k = dict(v_inner=dev(spec.v_inner, np.float64), v_outer=dev(spec.v_outer, np.float64),
                 n_e=dev(spec.n_e, np.float64), nu=dev(spec.nu, np.float64), tau=dev(tau, np.float64),
                 line_row=dev(rows, np.int32), dbr_offset=dev(spec.dbr_offset, np.int32),
                 dbr_line=dev(spec.dbr_line, np.int32), dbr_cdf=dev(spec.dbr_cdf, np.float64),
                 j_est=dev(np.zeros(S), np.float64), nu_bar=dev(np.zeros(S), np.float64),
                 spectrum=dev(np.zeros(B + 2), np.float64), stats=dev(np.zeros(9), np.int64))
        args = mc.mc_noalloc_args(
            n_shells=S, v_inner_0=float(spec.v_inner[0]), t_exp=float(spec.t_exp), n_lines=L,
            line_mode=int(spec.line_mode), seed=3, iteration=0, n_packets=n, t_inner=float(spec.t_inner),
            max_segments=0, delta_t=1.0, spec_bins=B, spec_nu_lo=float(spec.spec_nu_lo),
            spec_nu_hi=float(spec.spec_nu_hi), **{name: t.data_ptr() for name, t in k.items()})
        mc.mc_transport_noalloc(args, torch.cuda.current_stream().cuda_stream)
        torch.cuda.synchronize()
        out.append([k[name].cpu().numpy() for name in ("stats", "j_est", "nu_bar", "spectrum")])
    assert np.array_equal(out[0][0], out[1][0]) and out[0][0][6] > n
    for a, b in zip(out[0][1:], out[1][1:]):  # the sums' order
        assert np.allclose(a, b, rtol=1e-9, atol=0.0)

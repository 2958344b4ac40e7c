"""Expected emission in thin plasmas and at tiny ionization, where the Debye length
grows to 1e11 reduced Compton lengths (and far beyond, where the nodes run in
FP64): non-relativistic samples keep their rate, power and gradient; against the
oracle, with the operator's tolerances."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

RTOL, GTOL = 2e-5, 1e-4     # FP32 nodes and compensated sums (forward; gradient on the scale of its sensitivity)


@pytest.mark.parametrize("Z,n_i,T_e,Zs", [
    (29, 1e17, 1e4, 5.0), (29, 7e16, 1e4, 5.0), (29, 1e16, 1e4, 5.0), (1, 1e14, 1e3, 1.0), (29, 1e12, 1e5, 29.0),
    (79, 1e13, 1e6, 3.0), (29, 8.5e28, 1e4, 1e-12), (29, 8.5e28, 1e4, 1e-9), (13, 1e24, 1e3, 1e-13), (29, 1e-6, 1e4, 5.0)])
def test_thin_plasma_against_the_oracle(orc, Z, n_i, T_e, Zs):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1907_02814_gb300 import build, pcc
    build.build()
    rng = np.random.default_rng(7)
    n = 70
    params = np.array([[n_i, T_e, Zs, 1.0, 1.0]], np.float32)
    gamma = rng.uniform(1.05, 1.999, (1, n)).astype(np.float32)
    w = rng.uniform(0.5, 2.0, (1, n)).astype(np.float32)
    gout = np.array([[1.0, 0.5, -0.7]], np.float32)
    ctx = pcc.Context(0)
    t = lambda v: torch.as_tensor(v, device="cuda")
    out = pcc.expected_emission_fwd(ctx, Z, t(params), t(gamma), t(w)).cpu().numpy()[0]
    grad = pcc.expected_emission_bwd(ctx, Z, t(params), t(gamma), t(w), t(gout)).cpu().numpy()[0]
    status, _ = ctx.read_status()
    ctx.close()
    p = [float(v) for v in params[0]]
    mat = orc.material(Z, p[2], p[0], p[1], p[3], p[4])
    g, ww, go = gamma[0].astype(np.float64), w[0].astype(np.float64), gout[0].astype(np.float64)
    ref = np.asarray(orc.expected_emission(mat, g, ww))
    assert status == 0 and ref[0] > 0 and ref[2] > 0
    np.testing.assert_allclose(out, ref, rtol=RTOL)
    gr = np.asarray(orc.expected_emission_grad_analytic(mat, g, ww, go))
    th = np.asarray(p)
    assert np.all(np.abs(th * (grad - gr)) <= GTOL * (np.abs(go * ref).sum() + np.abs(th * gr))), (grad, gr)

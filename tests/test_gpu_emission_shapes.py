"""The expected-emission kernels where their work is cut differently: sample
counts on both sides of a warp and of a block's batch, node counts from two to
the largest, all samples in one energy regime, samples without weight or at
rest among them, every charge's Elwert factor, cells whose Debye length is near
the Thomas-Fermi one (FP64 nodes) and empty cells; against the oracle, with the
operator's tolerances."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

RTOL, GTOL = 2e-5, 1e-4     # FP32 nodes and compensated sums (forward; gradient on the scale of its sensitivity)


@pytest.mark.parametrize("samples,nodes,kind,Z", [
    (1, 64, "mixed", 29), (31, 64, "mixed", 29), (33, 7, "mixed", 29), (257, 16, "mixed", 79), (300, 128, "mixed", 6),
    (64, 2, "rel", 29), (40, 48, "rel", 92), (40, 48, "nr", 29), (70, 33, "nr", 1), (0, 64, "rel", 29)])
def test_shapes_against_the_oracle(orc, samples, nodes, kind, Z):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1907_02814_gb300 import build, pcc
    build.build()
    rng = np.random.default_rng(samples + nodes + Z)
    n = 5
    params = np.stack([10.0 ** rng.uniform(26, 29, n), 10.0 ** rng.uniform(1, 4, n), rng.uniform(0.2, 1.0, n) * Z,
                       rng.uniform(0.7, 1.4, n), rng.uniform(0.7, 1.4, n)], 1)
    scr = orc.screening(orc.material(Z, *[float(v) for v in params[1, [2, 0, 1]]])).as_dict()
    params[1, 3], params[1, 4] = 1.0, scr["LTF"] / scr["LD"] * 1.01          # lengths 1 % apart
    params = params.astype(np.float32)
    T = {"mixed": rng.exponential(2.0, (n, samples)), "rel": 10.0 ** rng.uniform(0.05, 3, (n, samples)),
         "nr": rng.uniform(0.01, 0.99, (n, samples))}[kind]
    gamma = (1.0 + T).astype(np.float32)
    w = rng.uniform(0.5, 2.0, (n, samples)).astype(np.float32)
    if samples > 8:
        w[:, 3], gamma[:, 5] = 0.0, 1.0
    gout = rng.normal(size=(n, 3)).astype(np.float32)
    ctx = pcc.Context(0)
    t = lambda v: torch.as_tensor(v, device="cuda")
    out = pcc.expected_emission_fwd(ctx, Z, t(params), t(gamma), t(w), n_quad=nodes).cpu().numpy()
    grad = pcc.expected_emission_bwd(ctx, Z, t(params), t(gamma), t(w), t(gout), n_quad=nodes).cpu().numpy()
    again = pcc.expected_emission_bwd(ctx, Z, t(params), t(gamma), t(w), t(gout), n_quad=nodes).cpu().numpy()
    assert np.array_equal(grad, again)
    ctx.close()
    for c in range(n):
        p = [float(v) for v in params[c]]
        mat = orc.material(Z, p[2], p[0], p[1], p[3], p[4])
        live = (w[c] != 0) & (gamma[c] > 1)
        g, ww = gamma[c][live].astype(np.float64), w[c][live].astype(np.float64)
        ref = np.asarray(orc.expected_emission(mat, g, ww, n_quad=nodes))
        np.testing.assert_allclose(out[c], ref, rtol=RTOL)
        go = gout[c].astype(np.float64)
        gr = np.asarray(orc.expected_emission_grad_analytic(mat, g, ww, go, n_quad=nodes))
        th = np.asarray(p)
        assert np.all(np.abs(th * (grad[c] - gr)) <= GTOL * (np.abs(go * ref).sum() + np.abs(th * gr))), (c, grad[c], gr)

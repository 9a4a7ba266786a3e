"""Column transforms of run-time lengths (k_colfft and the z stage of three passes around it): G and
the weighted densities against the oracle at the lengths where they can go wrong.

Lengths: one radix stage (4, 14, 15), every composite radix and prime stage (11..31; two of them in
one length, so that the second takes twiddles), three stages (343 = 7^3), 256 rows (one TMA box) and
more (two boxes, of an odd length the second partly past the axis), column counts that leave a tile
partly empty, short axes whose tiles take several planes (133 of them, the last tile partly past the
end).  Along z the columns of a plane are cut together: as chunks that divide it (100 x 36 x 70), as one
row with a partly empty last tile (120 x 75 x 84; two boxes: 275 x 7 x 20; compile-time length: 96 x 75 x
33), or per ky (10 x 133 x 100).  Along y the last tile of 33 columns holds one (20 x 128 x 64).  FP32 is held to 1e-5 and FP64 to 1e-10 per field, the library's stated bounds
(about 30 transform passes of log2(N) roundings each are 4e-7 in FP32).
"""
import numpy as np
import pytest

from oracle import functional as F
from oracle import picard as P
from paper_0910_1531_gb300 import workloads

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

TOL = {"fp32": 1e-5, "fp64": 1e-10}
FIELDS = [[0], [1], [2], [3], [4, 5, 6], [7, 8, 9]]
SPECIES = ([0.095, 0.099, 0.181], [1.0, 2.0, -1.0], [0.1, 0.01, 0.12])


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_0910_1531_gb300 import build
    build.build()


def relerr(a, b):
    scale = np.max(np.abs(b))
    return float(np.max(np.abs(np.asarray(a) - b)) / (scale if scale > 0 else 1.0))


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("shape", [
    (4, 5, 6), (14, 15, 16), (9, 10, 4), (7, 512, 6), (261, 6, 8), (323, 8, 4), (6, 343, 5), (289, 4, 34), (22, 26, 12),
    (38, 46, 10), (58, 62, 36), (256, 20, 6), (12, 275, 8), (160, 9, 33), (100, 36, 70), (17, 23, 130), (10, 133, 100), (133, 10, 60),
    (120, 75, 84), (275, 7, 20), (96, 75, 33), (20, 128, 64)])
def test_runtime_lengths_match_the_oracle(shape, precision):
    from paper_0910_1531_gb300 import binding
    prob = F.Problem(shape, (0.11, 0.1, 0.09), *SPECIES)
    rho = workloads.random_density(shape, 3, prob.bath.rho, 0.3, seed=61)
    V = np.zeros_like(rho)
    V[1, : shape[0] // 3] = np.inf
    rho[1, : shape[0] // 3] = 0.0
    plan = binding.Plan(shape, prob.h, *SPECIES, precision=precision)
    dev = lambda x: torch.tensor(np.ascontiguousarray(x), dtype=plan.dtype, device="cuda")
    n, n_ref = plan.weighted_densities(dev(rho)).double().cpu().numpy(), F.weighted_densities(prob, rho)
    for f in FIELDS:
        assert relerr(n[f], n_ref[f]) < TOL[precision], (f, plan.tuning())
    g, _ = plan.picard_map(dev(rho), dev(V))
    g_ref = F.picard_map(prob, rho, V)
    assert relerr(g.double().cpu().numpy(), g_ref) < TOL[precision], plan.tuning()
    plan.set_variants(x=1, z=2)                       # the first half's z stage as three passes
    g, _ = plan.picard_map(dev(rho), dev(V))
    assert relerr(g.double().cpu().numpy(), g_ref) < TOL[precision], plan.tuning()
    plan.close()


FIVE = ([0.095, 0.099, 0.181, 0.14, 0.12], [1.0, 2.0, -1.0, -0.5, 0.0], [0.1, 0.01, 0.1, 0.04, 0.3])


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("shape,species", [((32, 12, 20), SPECIES), ((18, 32, 21), SPECIES), ((32, 12, 20), FIVE)])
def test_plans_without_a_k_table_match_the_oracle(shape, species, precision, monkeypatch):
    # a non-cubic box's |k| table holds one record per octant point (weights 2 S, kernels S (S + 1) / 2, each rounded
    # up to 16 bytes, and no Gamma derivatives before dft_grad asks for them); a plan that cannot have it evaluates
    # the factors per point, in the weighted densities, G, the line search's paired samples and the gradients
    from paper_0910_1531_gb300 import binding
    prob = F.Problem(shape, (0.11, 0.1, 0.09), *species)
    S = len(species[0])
    v = 4 if precision == "fp32" else 2
    up = lambda n: (n + v - 1) // v * v
    size = (shape[2] // 2 + 1) * (shape[1] // 2 + 1) * (shape[0] // 2 + 1) * (up(2 * S) + up(S * (S + 1) // 2)) * 16 // v
    rho = workloads.random_density(shape, S, prob.bath.rho, 0.3, seed=67)
    V = np.zeros_like(rho)
    V[0, : shape[0] // 3] = np.inf
    rho[0, : shape[0] // 3] = 0.0
    g_ref, om_ref = F.picard_map(prob, rho, V), F.grand_potential(prob, rho, V)
    d_ref = F.grad_omega_rho(prob, rho, V)
    b_ref = F.grad_omega_bulk(shape, prob.h, *species, rho, V)
    step_ref, _ = P.picard_step(prob, rho, V, g0=g_ref)
    for limit, table in ((size, True), (size - 1, False)):
        monkeypatch.setenv("DFT_KTAB_BYTES", str(limit))
        plan = binding.Plan(shape, prob.h, *species, precision=precision)
        assert ("table per octant point" in plan.tuning()) == table, plan.tuning()
        dev = lambda x: torch.tensor(np.ascontiguousarray(x), dtype=plan.dtype, device="cuda")
        n, n_ref = plan.weighted_densities(dev(rho)).double().cpu().numpy(), F.weighted_densities(prob, rho)
        for f in FIELDS:
            assert relerr(n[f], n_ref[f]) < TOL[precision], (f, table)
        g, _ = plan.picard_map(dev(rho), dev(V))
        assert relerr(g.double().cpu().numpy(), g_ref) < TOL[precision], table
        om, d_rho, _, d_bulk = plan.grad(dev(rho), dev(V))
        assert om == pytest.approx(om_ref, rel=TOL[precision])
        assert relerr(d_rho.double().cpu().numpy(), d_ref) < TOL[precision], table
        # bath derivatives: central differences of the oracle
        assert np.allclose(d_bulk, b_ref, rtol=2e-3 if precision == "fp32" else 1e-6, atol=0), table
        r = dev(rho)
        plan.picard_step(r, dev(V), -1.0)
        assert relerr(r.double().cpu().numpy(), step_ref) < TOL[precision], table
        plan.close()

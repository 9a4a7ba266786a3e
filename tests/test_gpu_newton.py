"""Newton-Krylov solver (dft_solve_newton): converges to the fixed point the oracle defines,
including where the Picard line search stalls (the pore with confined fixed-number O)."""
import numpy as np
import pytest

from oracle import functional as F
from oracle import picard as P
from paper_0910_1531_gb300 import workloads

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_0910_1531_gb300 import build
    build.build()


def relerr(a, b):
    b = np.asarray(b)
    return float(np.max(np.abs(np.asarray(a) - b)) / np.max(np.abs(b)))


def _plan(w, precision):
    from paper_0910_1531_gb300 import binding
    plan = binding.Plan(w.shape, w.h, w.radius, w.z, w.bulk_molar, precision=precision, n_fixed=w.n_fixed)
    dev = lambda x: torch.tensor(np.ascontiguousarray(x), dtype=plan.dtype, device="cuda")
    return plan, dev


def test_newton_matches_oracle_picard_fp64():
    w = workloads.centred_sphere(n=16, h=0.1, molar=1.0, sphere_radius=0.3)
    prob = F.Problem(w.shape, w.h, w.radius, w.z, w.bulk_molar)
    rho0 = w.initial_rho_nm3(prob.bath.rho)
    ref, _, r_ref = P.solve(prob, rho0.copy(), w.V, tol=1e-11, max_it=500)
    assert r_ref < 1e-11
    plan, dev = _plan(w, "fp64")
    rho = dev(rho0)
    its, gevals, r, ok = plan.solve_newton(rho, dev(w.V), tol=1e-11, max_newton=30, krylov_dim=30)
    assert ok and r < 1e-11, (its, gevals, r)
    assert its <= 15
    assert relerr(rho.cpu().numpy(), ref) < 1e-9
    plan.close()


def test_newton_converges_where_the_line_search_stalls_fp64():
    # 0.1 nm grid of the pore: Picard with the line search stays at r = 0.245 (oracle and GPU);
    # Newton-Krylov reaches the fixed point, and the oracle's own map confirms it
    w = workloads.pore_slab_4species(n=32, h=0.1)
    prob = F.Problem(w.shape, w.h, w.radius, w.z, w.bulk_molar, n_fixed=w.n_fixed)
    plan, dev = _plan(w, "fp64")
    rho = dev(w.initial_rho_nm3(prob.bath.rho))
    its, gevals, r, ok = plan.solve_newton(rho, dev(w.V), tol=1e-8, max_newton=40, krylov_dim=30)
    assert ok, (its, gevals, r)
    got = rho.cpu().numpy()
    g = F.picard_map(prob, got, w.V)
    assert np.sqrt(P.residual_sq(prob, got, g)) < 1e-7
    assert np.sum(got[3]) * prob.dv == pytest.approx(8.0, rel=1e-10)
    plan.close()


def test_newton_fp32_reaches_the_fp32_floor():
    w = workloads.obstacles_3species(n=32, h=0.2, n_obstacles=4, seed=3)
    prob = F.Problem(w.shape, w.h, w.radius, w.z, w.bulk_molar)
    plan, dev = _plan(w, "fp32")
    rho = dev(w.initial_rho_nm3(prob.bath.rho))
    its, gevals, r, ok = plan.solve_newton(rho, dev(w.V), tol=1e-6, max_newton=30, krylov_dim=30)
    assert ok, (its, gevals, r)
    got = rho.cpu().numpy().astype(np.float64)
    g = F.picard_map(prob, got, w.V)
    assert np.sqrt(P.residual_sq(prob, got, g)) < 1e-5
    plan.close()


@pytest.mark.parametrize("shape,krylov_dim", [((4, 4, 4), 30), ((5, 6, 7), 3), ((48, 10, 33), 30), ((48, 33, 35), 30)])
def test_newton_orthogonalisation_sizes_fp64(shape, krylov_dim):
    # fields smaller than one block of the orthogonalisation, of an odd length, of one element per thread for part of
    # its grid, and larger than its grid (two blocks of 256 threads per SM: 77824 threads on 152 SMs; 110880
    # elements); a restart at the largest basis.  r < 1e-11 on the GPU leaves the oracle's residual at the maps'
    # difference, 1e-10 per point
    prob = F.Problem(shape, 0.1, [0.095, 0.181], [1.0, -1.0], [1.0, 1.0])
    V = np.stack([z * 2.0 * np.sin(2 * np.pi * np.arange(shape[0]) / shape[0])[:, None, None] * np.ones(shape)
                  for z in (1.0, -1.0)])
    V[:, 0, 0, 0] = np.inf
    rho0 = np.where(np.isinf(V), 0.0, prob.bath.rho[:, None, None, None])
    from paper_0910_1531_gb300 import binding
    plan = binding.Plan(shape, 0.1, [0.095, 0.181], [1.0, -1.0], [1.0, 1.0], precision="fp64")
    rho = torch.tensor(rho0, dtype=torch.float64, device="cuda")
    its, gevals, r, ok = plan.solve_newton(rho, torch.tensor(V, device="cuda"), tol=1e-11, max_newton=40,
                                           krylov_dim=krylov_dim)
    assert ok and r < 1e-11, (its, gevals, r)
    got = rho.cpu().numpy()
    assert np.sqrt(P.residual_sq(prob, got, F.picard_map(prob, got, V))) < 2e-10
    plan.close()

"""The one-launch stage solves against the oracle's sparse LU through a primal step, its tangent and
its adjoint, where the kernel can go wrong: fewer kept elements than CTAs, meshes that are not
two-colourable (an odd count around the airfoil), the largest system of the cluster variant and the
first one of the grid variant (2560 kept rows), cycles of one and three steps (restarts), and each
block size.  Bar: the repository's FP64 parity bar, the solves running to 1e-13."""
import numpy as np
import pytest

from gpu_common import PARITY_TOL, TIGHT, make, perturbed_state, rel_err, to_dev, to_host
from oracle import periodic as OP
from oracle.dg import DG
from pp_inputs import KIN_HEAVE_PITCH, MU_C0, ogrid

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("n_theta,n_r,p,restart", [
    (3, 1, 1, 40),     # 6 elements, not two-colourable
    (7, 2, 2, 3),      # 28 elements, odd, restarts
    (8, 2, 1, 1),      # restart after every step
    (32, 2, 3, 40),    # 64 kept elements x 40 = 2560 rows: the last cluster case
    (43, 1, 4, 60),    # 43 or more kept elements x 60 > 2560 rows: grid, odd
])
def test_stage_solves_against_oracle(n_theta, n_r, p, restart):
    mesh = ogrid(n_theta, n_r, seed=2)
    T = 0.05
    mu = MU_C0 * np.array([0.01, 0.01, 1.0])
    dg = DG(mesh, p, T=T)
    u0 = perturbed_state(dg.Ne, p, seed=60 + p, amp=1e-3)
    cfg = dict(TIGHT, newton_tol=1e-14, lin_rtol=1e-13, gmres_restart=restart, gmres_maxit=4000, T=T)
    A, ctx, m = make(p, KIN_HEAVE_PITCH, mesh, **cfg)
    try:
        tr = OP.primal_sweep(dg, mu, u0, 1, newton_tol=1e-14)
        uN = torch.zeros(dg.Nu, dtype=torch.float64, device="cuda")
        A.pp_primal_period(ctx, m, mu, to_dev(u0), 1, u_final=uN)
        assert rel_err(to_host(uN), tr.u[-1]) <= PARITY_TOL
        v = np.random.default_rng(p).standard_normal(dg.Nu)
        out = torch.zeros_like(uN)
        A.pp_tangent_matvec(ctx, to_dev(v), out)
        assert rel_err(to_host(out), v - OP.tangent_sweep(dg, tr, v)) <= PARITY_TOL
        g = A.pp_adjoint_sweep(ctx, to_dev(v), out, weights=[1.0, 0.5], n_mu=3)
        lam, grad = OP.adjoint_sweep(dg, tr, v, np.array([1.0, 0.5]))
        assert rel_err(to_host(out), lam) <= PARITY_TOL
        assert rel_err(g, grad) <= PARITY_TOL
    finally:
        A.pp_mesh_destroy(m)
        A.pp_destroy(ctx)


def test_cap_reached_is_reported_and_cleared():
    """A linear solve that hits gmres_maxit fails its sweep with PP_ENOCONV; the next sweep is clean."""
    mesh = ogrid(8, 2, seed=2)
    dt = dict(T=0.5)
    A, ctx, m = make(1, KIN_HEAVE_PITCH, mesh, lin_rtol=1e-13, gmres_maxit=2, newton_maxit=60, gmres_rtol=1e-1, **dt)
    try:
        u0 = to_dev(perturbed_state(mesh.nt, 1, seed=3))
        A.pp_primal_period(ctx, m, MU_C0, u0, 2)
        v = torch.ones_like(u0)
        out = torch.zeros_like(u0)
        for _ in range(2):
            with pytest.raises(A.PPError) as ei:
                A.pp_tangent_matvec(ctx, v, out)
            assert ei.value.code == A.PP_ENOCONV
            assert float(out.abs().max()) == 0.0
        A.pp_primal_period(ctx, m, MU_C0, u0, 2)
    finally:
        A.pp_mesh_destroy(m)
        A.pp_destroy(ctx)

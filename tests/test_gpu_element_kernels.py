"""The element kernels where their work is split: residuals of meshes with full, partial and single
groups of elements per block (more elements than fit the resident blocks at once, remainders, odd
counts), the block Jacobian at every degree on wall, far-field and interior elements of the same
meshes, and the motion-seed terms of dF/dmu (kappa . dr/ds) on a mesh with several elements per
group.  Reference: the oracle; bar: the repository's FP64 parity bar."""
import numpy as np
import pytest

from gpu_common import PARITY_TOL, TIGHT, make, perturbed_state, rel_err, to_dev, to_host
from oracle import periodic as OP
from oracle.dg import DG
from pp_inputs import KIN_HEAVE_PITCH, MU_C0, ogrid

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("n_theta,n_r,p", [(3, 1, 1), (131, 37, 1), (61, 13, 2), (67, 17, 3), (59, 29, 4)])
def test_residual_and_jacobian_rows(n_theta, n_r, p):
    mesh = ogrid(n_theta, n_r, seed=5)
    A, ctx, m = make(p, KIN_HEAVE_PITCH, mesh)
    try:
        dg = DG(mesh, p)
        u = perturbed_state(dg.Ne, p, seed=70 + p, amp=3e-2)
        r = torch.zeros(dg.Nu, dtype=torch.float64, device="cuda")
        A.pp_residual(ctx, m, MU_C0, 0.7, to_dev(u), r)
        assert rel_err(to_host(r), dg.residual(u, MU_C0, 0.7)) <= PARITY_TOL
        nb = dg.nb
        blk = torch.zeros(dg.Ne * 4 * nb * nb, dtype=torch.float64, device="cuda")
        A.pp_jacobian_blocks(ctx, m, MU_C0, 0.7, to_dev(u), blk)
        pick = [np.nonzero(np.any(dg.tag == t, 1))[0][:3] for t in (1, 2)] + [[0, dg.Ne // 2, dg.Ne - 1]]
        elems = np.unique(np.concatenate(pick)).astype(int)
        gpu = to_host(blk).reshape(dg.Ne, 4, nb, nb)[elems].transpose(0, 1, 3, 2)
        assert rel_err(gpu, dg.jac_blocks_subset(u, MU_C0, 0.7, elems)) <= PARITY_TOL
    finally:
        A.pp_mesh_destroy(m)
        A.pp_destroy(ctx)


@pytest.mark.parametrize("n_theta,n_r,p", [(41, 9, 1), (31, 7, 2)])
def test_gradient_terms_of_grouped_elements(n_theta, n_r, p):
    mesh = ogrid(n_theta, n_r, seed=6)
    T = 0.05
    mu = MU_C0 * np.array([0.01, 0.01, 1.0])
    dg = DG(mesh, p, T=T)
    u0 = perturbed_state(dg.Ne, p, seed=80 + p, amp=1e-3)
    A, ctx, m = make(p, KIN_HEAVE_PITCH, mesh, **dict(TIGHT, newton_tol=1e-14, gmres_maxit=4000, T=T))
    try:
        tr = OP.primal_sweep(dg, mu, u0, 1, newton_tol=1e-14)
        A.pp_primal_period(ctx, m, mu, to_dev(u0), 1)
        lam = np.random.default_rng(p).standard_normal(dg.Nu)
        out = torch.zeros(dg.Nu, dtype=torch.float64, device="cuda")
        g = A.pp_adjoint_sweep(ctx, to_dev(lam), out, weights=[1.0, 0.5], n_mu=3)
        _, ref = OP.adjoint_sweep(dg, tr, lam, np.array([1.0, 0.5]))
        assert rel_err(g, ref) <= PARITY_TOL
    finally:
        A.pp_mesh_destroy(m)
        A.pp_destroy(ctx)

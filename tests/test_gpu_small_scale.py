"""The sweeps are linear in their direction, down to directions whose squared norm is just a normal FP64 number
(2^-500: squares near 1e-301).  Scaling by a power of two is exact, so the bar is the FP64 parity bar."""
import numpy as np
import pytest

from gpu_common import PARITY_TOL, TIGHT, make, perturbed_state, rel_err, to_dev, to_host
from pp_inputs import KIN_HEAVE_PITCH, MU_C0, ogrid

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("n_theta,n_r,p", [(8, 2, 1), (16, 3, 3), (43, 6, 1)])  # one CTA, a cluster, all SMs
def test_tiny_directions(n_theta, n_r, p):
    mesh = ogrid(n_theta, n_r, seed=2)
    A, ctx, m = make(p, KIN_HEAVE_PITCH, mesh, **dict(TIGHT, T=0.02))
    try:
        u0 = to_dev(perturbed_state(mesh.nt, p, seed=3, amp=1e-4))
        A.pp_primal_period(ctx, m, MU_C0 * np.array([0.004, 0.004, 1.0]), u0, 1)
        v = to_dev(np.random.default_rng(8).standard_normal(u0.numel()))
        out = torch.zeros_like(u0)
        for sweep in (A.pp_tangent_matvec, A.pp_adjoint_sweep):
            sweep(ctx, v, out)
            ref = to_host(out).copy()
            sweep(ctx, v * 2.0 ** -500, out)
            assert rel_err(to_host(out) * 2.0 ** 500, ref) <= PARITY_TOL
    finally:
        A.pp_mesh_destroy(m)
        A.pp_destroy(ctx)

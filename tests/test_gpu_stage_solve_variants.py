"""The one-launch stage solves in both precisions through each way they are launched, for each block size:
one CTA, one cluster, all SMs with the basis in shared memory, and all SMs with the basis in global memory
and the longer ring of block columns (the last four meshes: at 60 basis vectors the own slices of a CTA
and the short ring need more than the 227 KB of an SM in FP32, and so in FP64).

Mixed precision runs FP32 solves under an FP64 outer iteration, which hides a wrong inner operator as extra
iterations; so the steps are bounded.  With inner_rtol = 1e-5 an outer iteration gains five digits, so 1e-13
takes three, four with one to spare; an inner solve to 1e-5 takes no more steps than the FP64 solve to 1e-13;
hence for the three solves of a step mixed <= 4 (FP64 + 3).  An inner operator that is wrong in
a part of its columns gains less than a digit per outer iteration and needs more than ten of them.
Values: the two precisions, and FP64 with the basis in shared memory (8 vectors), solve the same systems to
1e-13: the repository's FP64 parity bar."""
import numpy as np
import pytest

from gpu_common import PARITY_TOL, TIGHT, make, perturbed_state, rel_err, to_dev, to_host
from pp_inputs import KIN_HEAVE_PITCH, MU_C0, ogrid

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("p,n_theta,n_r,T", [
    (1, 8, 2, 0.05),       # one CTA: 16 kept elements
    (2, 6, 2, 0.05),       # one CTA: 12
    (1, 32, 4, 0.02),      # a cluster of 8: 1536 kept rows
    (2, 15, 6, 0.02),      # 2160
    (3, 16, 3, 0.02),      # 1920
    (4, 9, 4, 0.02),       # 2160
    (1, 43, 6, 0.01),      # all SMs, basis in shared memory
    (3, 25, 8, 0.01),
    (4, 21, 8, 0.01),
    (1, 128, 68, 0.002),   # all SMs, basis in global memory
    (2, 96, 48, 0.002),
    (3, 64, 34, 0.002),
    (4, 48, 28, 0.002),
])
def test_launch_variants_agree(p, n_theta, n_r, T):
    mesh = ogrid(n_theta, n_r, seed=3)
    mu = MU_C0 * np.array([T / 5.0, T / 5.0, 1.0])
    u0 = to_dev(perturbed_state(mesh.nt, p, seed=70 + p, amp=1e-4))
    rng = np.random.default_rng(p)
    v, w = (to_dev(rng.standard_normal(u0.numel())) for _ in range(2))
    tight = dict(TIGHT, newton_tol=1e-13, newton_maxit=60, lin_rtol=1e-13, gmres_maxit=4000, T=T)
    got = {}
    for name, cfg in {"fp64": dict(gmres_restart=60), "short": dict(gmres_restart=8),
                      "mixed": dict(gmres_restart=60, precision=1, inner_maxit=60, inner_rtol=1e-5)}.items():
        A, ctx, m = make(p, KIN_HEAVE_PITCH, mesh, **dict(tight, **cfg))
        try:
            uN, tv, aw = (torch.zeros_like(u0) for _ in range(3))
            A.pp_primal_period(ctx, m, mu, u0, 1, u_final=uN)
            A.pp_tangent_matvec(ctx, v, tv)
            A.pp_adjoint_sweep(ctx, w, aw)
            got[name] = (to_host(uN), to_host(tv), to_host(aw), A.pp_sweep_counts(ctx))
        finally:
            A.pp_mesh_destroy(m)
            A.pp_destroy(ctx)
    counts = {name: g[3] for name, g in got.items()}
    print(f"p={p} {mesh.nt} triangles: {counts}")
    for name in ("short", "mixed"):
        for a, b in zip(got["fp64"][:3], got[name][:3]):
            assert rel_err(b, a) <= PARITY_TOL
    for k in ("gmres_tangent", "gmres_adjoint"):
        assert counts["mixed"][k] <= 4 * (counts["fp64"][k] + 3)

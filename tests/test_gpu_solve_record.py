"""A sweep that fails leaves nothing behind: a direction with a NaN or of infinities is refused with PP_ENAN, and
the next call on the same context gives what a fresh context gives, with the same step counts, in both
precisions."""
import numpy as np
import pytest

from gpu_common import PARITY_TOL, TIGHT, make, perturbed_state, rel_err, to_dev, to_host
from pp_inputs import KIN_HEAVE_PITCH, MU_C0, ogrid

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _calls(A, ctx, m, u0, v):
    out = torch.zeros_like(u0)
    A.pp_tangent_matvec(ctx, v, out)
    tangent = to_host(out).copy()
    A.pp_adjoint_sweep(ctx, v, out)
    adjoint = to_host(out).copy()
    A.pp_primal_period(ctx, m, MU_C0, u0, 2, u_final=out)
    return tangent, adjoint, to_host(out).copy(), A.pp_sweep_counts(ctx)


@pytest.mark.parametrize("stride", [0, 1])
@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("sweep", ["tangent", "adjoint"])
@pytest.mark.parametrize("what", ["nan", "inf"])
def test_bad_direction_leaves_nothing_behind(what, sweep, precision, stride):
    mesh = ogrid(8, 2, seed=2)
    cfg = dict(TIGHT, precision=precision, T=0.5, checkpoint_stride=stride)
    u0 = to_dev(perturbed_state(mesh.nt, 1, seed=3))
    v = to_dev(np.random.default_rng(5).standard_normal(u0.numel()))
    bad = v * float("inf")
    if what == "nan":
        bad = v.clone()
        bad[7] = float("nan")
    got = []
    for fail in (False, True):
        A, ctx, m = make(1, KIN_HEAVE_PITCH, mesh, **cfg)
        try:
            A.pp_primal_period(ctx, m, MU_C0, u0, 2)
            if fail:
                with pytest.raises(A.PPError) as ei:
                    if sweep == "tangent":
                        A.pp_tangent_matvec(ctx, bad, torch.zeros_like(bad))
                    else:
                        A.pp_adjoint_sweep(ctx, bad, torch.zeros_like(bad))
                assert ei.value.code == A.PP_ENAN
            got.append(_calls(A, ctx, m, u0, v))
        finally:
            A.pp_mesh_destroy(m)
            A.pp_destroy(ctx)
    for fresh, after in zip(got[0][:3], got[1][:3]):
        assert rel_err(after, fresh) <= PARITY_TOL
    assert got[0][3] == got[1][3]

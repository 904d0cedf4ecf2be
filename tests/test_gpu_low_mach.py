"""Precision of the folded stage operator where the four variables differ in scale: the energy is 1 / M^2 of
the others.

Rows of (I + B) x = (M - cJ) D^-1 x and of its transpose against 80-bit products of the stored factors, for
directions that have the variables' scales and live on every other element, in the rows of the elements between
(where x itself is zero, so the row is B's alone), each within the bound of FP64 chains: nb + 4 roundings of an
entry of B (4: c, -1, the entry itself, M - cJ as it is read back) and 3 nb + 2 of a row, so (4 nb + 6) 2^-53
times the sum of |p| |q| |x|.  Sweeps variable by variable against the oracle's sparse LU: the
solves stop at 1e-14 of the whole right-hand side and the stage Newton at 1e-15 of the whole state, of which the
energy is up to 714 times the rest at M = 0.05 (1e-11 and 1e-12 of the other variables), so the parity bar of
1e-10 leaves a factor of ten for the three stages."""
import numpy as np
import pytest

from gpu_common import PARITY_TOL, TIGHT, make, rel_err, to_dev, to_host
from oracle import periodic as OP
from oracle.dg import DG
from pp_inputs import KIN_HEAVE_PITCH, MU_C0, free_stream_state, ogrid

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _state(mesh, p, mach, seed):
    u = free_stream_state(mesh.nt, p, mach=mach)
    return (u * (1.0 + 1e-5 * np.random.default_rng(seed).uniform(-1.0, 1.0, u.shape))).reshape(-1)


def _setup(p, mach, **more):
    mesh = ogrid(8, 2, seed=2)
    T = 0.05 * mach      # the same acoustic Courant number at every Mach number
    mu = MU_C0 * np.array([T / 5.0, T / 5.0, 1.0])
    A, ctx, m = make(p, KIN_HEAVE_PITCH, mesh, **dict(TIGHT, Mach=mach, T=T, newton_maxit=60, gmres_maxit=4000, **more))
    return mesh, T, mu, A, ctx, m


def _scale(mach):
    return np.array([1.0, 1.0, 1.0, 1.0 / (1.4 * 0.4 * mach ** 2) + 0.5])[None, :, None]


@pytest.mark.parametrize("p", [1, 2])
@pytest.mark.parametrize("mach", [0.2, 0.05, 0.01])
def test_folded_rows(p, mach):
    mesh, _, mu, A, ctx, m = _setup(p, mach)
    try:
        u0 = to_dev(_state(mesh, p, mach, 3))
        A.pp_primal_period(ctx, m, mu, u0, 1)
        n, nb = u0.numel(), u0.numel() // mesh.nt
        x, y = torch.zeros_like(u0), torch.zeros_like(u0)

        def dense(kind, trans):
            out = np.zeros((n, n))
            for j in range(n):
                x.zero_()
                x[j] = 1.0
                A.pp_stage_apply(ctx, 0, 1, kind, x, y, trans=trans)
                out[:, j] = to_host(y)
            return out.reshape(mesh.nt, nb, mesh.nt, nb)

        d = np.random.default_rng(9).standard_normal((mesh.nt, 4, nb // 4))
        for trans in (False, True):
            S, D = (dense(kind, trans) for kind in range(2))
            nbr = [[e2 for e2 in range(mesh.nt) if e2 != e and S[e, :, e2].any()] for e in range(mesh.nt)]
            colour, queue = {0: 0}, [0]
            for e in queue:
                for e2 in nbr[e]:
                    if e2 not in colour:
                        colour[e2] = 1 - colour[e]
                        queue.append(e2)
            for on in range(2):
                v = (d / _scale(mach) if trans else d * _scale(mach)).reshape(mesh.nt, nb).copy()
                rows = [e for e in range(mesh.nt) if colour[e] != on]
                v[rows] = 0.0
                A.pp_stage_apply(ctx, 0, 1, 2, to_dev(v), y, trans=trans)
                got, worst = to_host(y).reshape(mesh.nt, nb), 0.0
                for e in rows:
                    ref, size = np.zeros(nb, dtype=np.longdouble), np.zeros(nb, dtype=np.longdouble)
                    for e2 in nbr[e]:
                        P, Q = S[e, :, e2].astype(np.longdouble), D[e2, :, e2].astype(np.longdouble)
                        ref += P @ (Q @ v[e2])
                        size += np.abs(P) @ (np.abs(Q) @ np.abs(v[e2]))
                    bound = (4 * nb + 6) * 2.0 ** -53 * size
                    worst = max(worst, float(np.max(np.abs(got[e] - ref) / np.where(bound > 0, bound, 1))))
                    assert np.all(np.abs(got[e] - ref) <= bound), worst
                print(f"p={p} M={mach} trans={trans}: {worst:.3f} of the bound")
    finally:
        A.pp_mesh_destroy(m)
        A.pp_destroy(ctx)


@pytest.mark.parametrize("mach", [0.2, 0.05])
def test_sweeps_variable_by_variable(mach):
    p = 2
    mesh, T, mu, A, ctx, m = _setup(p, mach, lin_rtol=1e-14, newton_tol=1e-15)
    try:
        dg = DG(mesh, p, Mach=mach, T=T)
        u0 = _state(mesh, p, mach, 4)
        tr = OP.primal_sweep(dg, mu, u0, 1, newton_tol=1e-15)
        A.pp_primal_period(ctx, m, mu, to_dev(u0), 1)
        scale = _scale(mach)
        d = np.random.default_rng(6).standard_normal((mesh.nt, 4, dg.nb // 4))
        out = torch.zeros(dg.Nu, dtype=torch.float64, device="cuda")
        v, w = (d * scale).reshape(-1), (d / scale).reshape(-1)
        A.pp_tangent_matvec(ctx, to_dev(v), out)
        pairs = [(to_host(out).copy(), v - OP.tangent_sweep(dg, tr, v))]
        A.pp_adjoint_sweep(ctx, to_dev(w), out)
        pairs.append((to_host(out), OP.adjoint_sweep(dg, tr, w)[0]))
        for got, ref in pairs:
            for a in range(4):
                assert rel_err(got.reshape(d.shape)[:, a], ref.reshape(d.shape)[:, a]) <= PARITY_TOL
    finally:
        A.pp_mesh_destroy(m)
        A.pp_destroy(ctx)

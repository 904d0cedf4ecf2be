"""The stage solves on meshes whose dual graph is not two-colourable.  (The O-grids and boxes of the other
tests are all two-colourable, with classes of equal size: every ring of triangles crosses two per quad.)  A
flipped diagonal changes the number of triangles around four vertices by one, so kept elements become
neighbours, the block B_RR of the reduced system is not zero, and the classes differ in size.  Checked against
the oracle's sparse LU through a primal step, its tangent and its adjoint, in each way a solve is launched,
at the repository's FP64 parity bar (the solves run to 1e-13)."""
import numpy as np
import pytest

from gpu_common import PARITY_TOL, TIGHT, make, perturbed_state, rel_err, to_dev, to_host
from oracle import periodic as OP
from oracle.dg import DG
from pp_inputs import KIN_HEAVE_PITCH, MU_C0, ogrid
from pp_inputs.mesh import Mesh

torch = pytest.importorskip("torch")


def _area(P):
    (a, b, c) = P
    return (b[0] - a[0]) * (c[1] - a[1]) - (b[1] - a[1]) * (c[0] - a[0])


def flipped(mesh, count, seed):
    """The mesh with up to `count` interior diagonals flipped, no triangle touched twice and the four outer
    edges of each pair interior."""
    tris, verts, ftag = mesh.tris.copy(), mesh.verts, mesh.ftag
    at = {(int(t[f]), int(t[(f + 1) % 3])): (e, f) for e, t in enumerate(tris) for f in range(3)}
    done, used = 0, set()
    for (a, b) in np.random.default_rng(seed).permutation(sorted(k for k in at if k[0] < k[1])):
        a, b = int(a), int(b)
        if (b, a) not in at or done == count:
            continue
        (e1, f1), (e2, f2) = at[a, b], at[b, a]
        if e1 in used or e2 in used or ftag[e1].any() or ftag[e2].any():
            continue
        c, d = int(mesh.tris[e1][(f1 + 2) % 3]), int(mesh.tris[e2][(f2 + 2) % 3])
        old = min(_area(verts[mesh.tris[e]]) for e in (e1, e2))
        new = [(c, a, d), (d, b, c)]
        if min(_area(verts[list(t)]) for t in new) < 0.3 * old:
            continue
        tris[e1], tris[e2] = new
        used |= {e1, e2}
        done += 1
    assert done == count
    return Mesh(verts, tris, ftag, name=f"{mesh.name}f{count}")


def odd_edges(mesh):
    """Edges of the dual graph whose ends get the same colour breadth first."""
    face, pairs = {}, []
    for e, t in enumerate(mesh.tris):
        for f in range(3):
            k = frozenset((int(t[f]), int(t[(f + 1) % 3])))
            if k in face:
                pairs.append((face[k], e))
            face[k] = e
    nbr = [[] for _ in mesh.tris]
    for a, b in pairs:
        nbr[a].append(b)
        nbr[b].append(a)
    colour, queue = {0: 0}, [0]
    for e in queue:
        for n in nbr[e]:
            if n not in colour:
                colour[n] = 1 - colour[e]
                queue.append(n)
    return sum(colour[a] == colour[b] for a, b in pairs)


MESHES = [(8, 3, 1), (16, 6, 12), (43, 6, 40)]   # (around, across, flips): one CTA, a cluster and all SMs at p = 1


@pytest.mark.parametrize("n_theta,n_r,flips", MESHES)
def test_these_meshes_are_not_two_colourable(n_theta, n_r, flips):
    mesh = ogrid(n_theta, n_r, seed=2)
    assert odd_edges(mesh) == 0
    assert odd_edges(flipped(mesh, flips, seed=1)) > 0


@pytest.mark.gpu
@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("n_theta,n_r,flips,p", [(*m, 1) for m in MESHES] + [(8, 3, 3, 2), (9, 4, 5, 3), (8, 3, 4, 4)])
def test_sweeps_on_odd_meshes(n_theta, n_r, flips, p, precision):
    mesh = flipped(ogrid(n_theta, n_r, seed=2), flips, seed=1)
    T = 0.02
    mu = MU_C0 * np.array([T / 5.0, T / 5.0, 1.0])
    dg = DG(mesh, p, T=T)
    u0 = perturbed_state(dg.Ne, p, seed=80 + p, amp=1e-4)
    cfg = dict(TIGHT, newton_tol=1e-14, newton_maxit=60, gmres_maxit=4000, T=T, precision=precision, inner_rtol=1e-4)
    A, ctx, m = make(p, KIN_HEAVE_PITCH, mesh, **cfg)
    try:
        tr = OP.primal_sweep(dg, mu, u0, 1, newton_tol=1e-14)
        out = torch.zeros(dg.Nu, dtype=torch.float64, device="cuda")
        A.pp_primal_period(ctx, m, mu, to_dev(u0), 1, u_final=out)
        assert rel_err(to_host(out), tr.u[-1]) <= PARITY_TOL
        v = np.random.default_rng(p).standard_normal(dg.Nu)
        A.pp_tangent_matvec(ctx, to_dev(v), out)
        assert rel_err(to_host(out), v - OP.tangent_sweep(dg, tr, v)) <= PARITY_TOL
        A.pp_adjoint_sweep(ctx, to_dev(v), out)
        assert rel_err(to_host(out), OP.adjoint_sweep(dg, tr, v)[0]) <= PARITY_TOL
    finally:
        A.pp_mesh_destroy(m)
        A.pp_destroy(ctx)

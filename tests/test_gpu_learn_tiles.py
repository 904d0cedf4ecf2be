"""The 32 x 32 product tiles at their edges: one row or column, one more or less than a tile, depths that
are not a multiple of a tile, both transpositions; and the network's one-call passes on such sizes.
Reference: the same in FP64.  Bar: a sum of k FP32 products is off by at most k eps of the sum of their
magnitudes (eps = 2^-24; FP64: 2^-53), doubled for the accumulation's own rounding."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("dtype,eps", [("float32", 2.0 ** -24), ("float64", 2.0 ** -53)])
@pytest.mark.parametrize("m,n,k", [(1, 1, 1), (33, 31, 65), (32, 64, 32), (7, 257, 100)])
def test_gemm_tiles(dtype, eps, m, n, k):
    from paper_1512_00616_gb300 import api as A
    rng = np.random.default_rng(m + n + k)
    dev = lambda x: torch.tensor(x, dtype=getattr(torch, dtype), device="cuda")  # noqa: E731
    for ta in (False, True):
        for tb in (False, True):
            a = rng.standard_normal((k, m) if ta else (m, k)).astype(dtype)
            b = rng.standard_normal((n, k) if tb else (k, n)).astype(dtype)
            c = rng.standard_normal((m, n)).astype(dtype)
            out = dev(c)
            A.pp_gemm(dev(a), dev(b), out, ta=ta, tb=tb, alpha=0.5, beta=2.0)
            x, y = (a.T if ta else a).astype(np.longdouble), (b.T if tb else b).astype(np.longdouble)
            ref = 0.5 * (x @ y) + 2.0 * c
            bound = 2 * (k + 3) * eps * (0.5 * np.abs(x) @ np.abs(y) + 2.0 * np.abs(c))
            assert np.all(np.abs(out.cpu().numpy().astype(np.longdouble) - ref) <= bound)


@pytest.mark.parametrize("rows,widths", [(1, [3, 33, 1]), (31, [6, 32, 64, 7]), (33, [8, 31, 65, 2]), (65, [5, 9])])
def test_network_passes(rows, widths):
    from paper_1512_00616_gb300.warmstart import MLP
    rng = np.random.default_rng(rows)
    net = MLP(widths, seed=rows)
    for _, b in net.params:
        b.copy_(torch.tensor(rng.standard_normal(b.numel()), dtype=torch.float32))
    X = torch.tensor(rng.standard_normal((rows, widths[0])), dtype=torch.float32, device="cuda")
    T = torch.tensor(rng.standard_normal((rows, widths[-1])), dtype=torch.float32, device="cuda")
    loss, grads = net.loss_and_grads(X, T)
    par = [[x.double().requires_grad_() for x in layer] for layer in net.params]
    H = X.double()
    for l, (W, b) in enumerate(par):
        Z = H @ W + b
        H = torch.nn.functional.gelu(Z) if l < len(par) - 1 else Z
    ref = ((H - T.double()) ** 2).mean()
    g = torch.autograd.grad(ref, [x for layer in par for x in layer])
    # rounding of up to four chained layers of at most max(rows, widths) terms, relative to the largest entry
    tol = 4 * 2 * (max(rows, *widths) + 3) * 2.0 ** -24 * 8
    assert abs(float(loss) - float(ref)) <= tol * abs(float(ref))
    for got, want in zip([x for layer in grads for x in layer], g):
        assert got.shape == want.shape
        assert float((got.double() - want).abs().max()) <= tol * float(want.abs().max())

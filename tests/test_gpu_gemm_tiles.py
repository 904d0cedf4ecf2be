"""Both product tiles where the choice between them and their edges lie: 16 x 16 (FP64, and FP32 with B
transposed up to 240 large tiles, 112 with both transposed) at one less and one more than a tile in each
direction, and the large tile with B transposed above that.  Reference and bar as for the other tile tests: the products in 80 bits, and a sum
of k products off by at most 2 (k + 3) eps of the sum of their magnitudes."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("dtype,eps", [("float32", 2.0 ** -24), ("float64", 2.0 ** -53)])
@pytest.mark.parametrize("m,n,k", [(16, 16, 16), (15, 17, 1), (17, 15, 33), (48, 47, 1000), (1, 300, 64), (300, 1, 17),
                                   (320, 350, 20), (352, 353, 20), (512, 480, 20), (511, 481, 20)])
def test_gemm_small_tiles(dtype, eps, m, n, k):
    from paper_1512_00616_gb300 import api as A
    rng = np.random.default_rng(m + n + k)
    dev = lambda x: torch.tensor(x, dtype=getattr(torch, dtype), device="cuda")  # noqa: E731
    for ta in (False, True):
        for tb in (False, True):
            a = rng.standard_normal((k, m) if ta else (m, k)).astype(dtype)
            b = rng.standard_normal((n, k) if tb else (k, n)).astype(dtype)
            x, y = (a.T if ta else a).astype(np.longdouble), (b.T if tb else b).astype(np.longdouble)
            for beta in (0.0, -1.5):
                c = rng.standard_normal((m, n)).astype(dtype)
                if beta == 0.0:
                    c[:] = np.nan     # not read
                out = dev(c)
                A.pp_gemm(dev(a), dev(b), out, ta=ta, tb=tb, alpha=0.5, beta=beta)
                c = np.nan_to_num(c)
                bound = 2 * (k + 3) * eps * (0.5 * np.abs(x) @ np.abs(y) + abs(beta) * np.abs(c))
                assert np.all(np.abs(out.cpu().numpy().astype(np.longdouble) - (0.5 * (x @ y) + beta * c)) <= bound)

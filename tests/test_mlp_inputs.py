"""The network's passes take their sizes from the layers they have now and refuse what the kernels would read
as something else: checked on the CPU, with the library's calls recorded instead of made."""
import types

import numpy as np
import pytest

torch = pytest.importorskip("torch")
api = pytest.importorskip("paper_1512_00616_gb300.api")
from paper_1512_00616_gb300 import warmstart  # noqa: E402
from paper_1512_00616_gb300.warmstart import MLP  # noqa: E402


@pytest.fixture
def calls(monkeypatch):
    got = []
    call = lambda name: lambda n, rows, sizes, *a: got.append((name, list(sizes), rows)) or 0  # noqa: E731
    monkeypatch.setattr(api, "_lib", types.SimpleNamespace(pp_mlp_forward_f32=call("forward"), pp_mlp_backward_f32=call("backward")))
    monkeypatch.setattr(api, "_stream", lambda: None)
    monkeypatch.setattr(warmstart, "_on_gpu", lambda x: True)
    return got


def test_a_replaced_layer_counts(calls):
    net = MLP([6, 8, 4], device="cpu")
    net.params[-1] = [torch.zeros(8, 2), torch.zeros(2)]
    Y = net.forward(torch.zeros(5, 6))
    grads = net.backward(torch.zeros(5, 2))
    assert Y.shape == (5, 2)
    assert [tuple(g.shape) for layer in grads for g in layer] == [(6, 8), (8,), (8, 2), (2,)]
    assert calls == [("forward", [6, 8, 2], 5), ("backward", [6, 8, 2], 5)]


@pytest.mark.parametrize("X", [torch.zeros(6), torch.zeros(5, 5), torch.zeros(5, 7), torch.zeros(2, 5, 6),
                               torch.zeros(5, 6, dtype=torch.float64), torch.zeros(5, 6, dtype=torch.int32)])
def test_inputs_of_another_shape_or_type_are_refused(calls, X):
    net = MLP([6, 8, 4], device="cpu")
    with pytest.raises(ValueError):
        net.forward(X)
    assert not calls


@pytest.mark.parametrize("dY", [torch.zeros(4), torch.zeros(5, 3), torch.zeros(4, 4), torch.zeros(6, 4),
                                torch.zeros(5, 4, dtype=torch.float64)])
def test_gradients_of_another_shape_or_type_are_refused(calls, dY):
    net = MLP([6, 8, 4], device="cpu")
    net.forward(torch.zeros(5, 6))
    with pytest.raises(ValueError):
        net.backward(dY)
    assert [c[0] for c in calls] == ["forward"]


@pytest.mark.parametrize("layer", [[torch.zeros(7, 4), torch.zeros(4)], [torch.zeros(8, 4), torch.zeros(3)],
                                   [torch.zeros(8), torch.zeros(4)], [torch.zeros(8, 4).double(), torch.zeros(4)]])
def test_layers_that_do_not_fit_are_refused(calls, layer):
    net = MLP([6, 8, 4], device="cpu")
    net.params[-1] = layer
    with pytest.raises(ValueError):
        net.forward(torch.zeros(5, 6))
    assert not calls


def test_layers_changed_between_the_passes_are_refused(calls):
    net = MLP([6, 8, 4], device="cpu")
    net.forward(torch.zeros(5, 6))
    net.params[0] = [torch.zeros(6, 9), torch.zeros(9)]
    with pytest.raises(ValueError):
        net.backward(torch.zeros(5, 4))


def test_inputs_on_the_cpu_are_refused(calls, monkeypatch):
    net = MLP([6, 8, 4], device="cpu")
    monkeypatch.setattr(warmstart, "_on_gpu", lambda x: x.is_cuda)
    with pytest.raises(ValueError):
        net.forward(torch.zeros(5, 6))
    assert not calls


def test_the_calls_check_their_tensors():
    """The API's own calls, on CPU tensors of the right sizes, refuse them before anything is launched."""
    X, W, b, Z = torch.zeros(5, 6), [torch.zeros(6, 4)], [torch.zeros(4)], [torch.zeros(5, 4)]
    with pytest.raises(ValueError):
        api.pp_mlp_forward_f32([6, 4], 5, X, W, b, Z, Z)
    with pytest.raises(ValueError):
        api.pp_mlp_forward_f32([6, 4, 2], 5, X, W, b, Z, Z)
    with pytest.raises(ValueError):
        api.pp_mlp_backward_f32([6, 4], 5, X, W, Z, Z, Z[0], [], W, b)


@pytest.mark.gpu
def test_a_replaced_layer_gives_its_own_result():
    net = MLP([6, 8, 4], seed=1)
    g = torch.Generator().manual_seed(2)
    W, b, X = (torch.randn(s, generator=g).cuda() for s in ((8, 2), (2,), (5, 6)))
    net.params[-1] = [W.t().contiguous().t(), b]   # another width, and not contiguous
    Y = net.forward(X)
    H = torch.nn.functional.gelu(X.double() @ net.params[0][0].double() + net.params[0][1].double())
    ref = H @ W.double() + b.double()
    # two layers of at most eight FP32 terms, relative to the largest entry
    assert np.max(np.abs((Y.double() - ref).cpu().numpy())) <= 2 * 2 * 11 * 2.0 ** -24 * 8 * float(ref.abs().max())

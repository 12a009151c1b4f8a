"""The network's convolution kernels at the edges of their tiles: batches that do not fill a
tile of images, and gradients that must not depend on how images share a tile."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
from paper_2407_20469_gb300 import apic, learn  # noqa: E402

pytestmark = pytest.mark.gpu


def _net(max_batch):
    net = apic.Net(max_batch)
    p = apic.unpack_params(learn.init_params(3))
    rng = np.random.default_rng(4)
    for l in range(6):
        p[f"b{l}"] = 0.05 * rng.standard_normal(p[f"b{l}"].shape)
    net.set_params(apic.pack_params(p))
    return net


def _inputs(B):
    g = torch.Generator(device="cuda").manual_seed(B)
    feat = torch.randn((B, 64, 64, 8), device="cuda", generator=g) - 4.0
    uv = torch.rand((B, 2), device="cuda", generator=g)
    target = torch.randn((B, 15), device="cuda", generator=g)
    return feat, uv, target


def _step(net, feat, uv, target):
    B = feat.shape[0]
    out = torch.empty((B, 15), device="cuda")
    net.forward(B, feat, uv, out)
    net.backward(target)
    return out, net.get_grads()


@pytest.mark.parametrize("B", [1, 2, 3, 7, 65])
def test_images_of_a_batch_are_independent(B):
    """Each image's outputs are those of a batch of its own, bit for bit."""
    feat, uv, target = _inputs(B)
    net = _net(B)
    out, _ = _step(net, feat, uv, target)
    one = torch.empty((1, 15), device="cuda")
    for b in {0, B // 2, B - 1}:
        net.forward(1, feat[b:b + 1], uv[b:b + 1].contiguous(), one)
        assert torch.equal(out[b], one[0]), b


@pytest.mark.parametrize("B", [1, 2, 3, 8, 33])
def test_gradients_are_the_mean_over_the_images(B):
    """The batch's gradients against the mean of its images' own. The pre-activation
    gradients are rounded to BF16 (2^-9 relative), once scaled by 1 / B and once not: exact
    where B is a power of two, independent roundings below 1 % in sum where not."""
    feat, uv, target = _inputs(B)
    net = _net(B)
    _, g = _step(net, feat, uv, target)
    acc = np.zeros(len(g))
    for b in range(B):
        acc += _step(net, feat[b:b + 1].contiguous(), uv[b:b + 1].contiguous(), target[b:b + 1].contiguous())[1]
    acc /= B
    tol = 1e-5 if B & (B - 1) == 0 else 1e-2
    assert np.linalg.norm(g - acc) <= tol * np.linalg.norm(acc)


@pytest.mark.parametrize("B", [1, 31, 32, 33, 64, 130])
def test_dense_layers_at_the_edges_of_their_tiles(B):
    """Both dense layers and their weight gradients from the stored activations, in float64 with
    the operands rounded to BF16 as the kernel rounds them. FP32 sums of at most 258 products are
    within 258 2^-24 of the sum of their magnitudes; the hidden layer's gradient is rounded to
    BF16 after such a sum, where a rare other rounding (2^-9 of an element) adds to the error."""
    def b16(x):
        return torch.as_tensor(np.asarray(x, np.float32)).bfloat16().double().numpy()

    feat, uv, target = _inputs(B)
    net = _net(B)
    out, g = _step(net, feat, uv, target)
    p, d = apic.unpack_params(net.get_params()), apic.unpack_params(g)
    x, h = net.activation(4, B).astype(np.float64), net.activation(5, B).astype(np.float64)
    W4, W5 = b16(p["w4"]), b16(p["w5"])
    eps = 258 * 2.0 ** -24
    pre = b16(x) @ W4.T + p["b4"]
    assert (np.abs(h - np.maximum(pre, 0)) <= eps * (np.abs(b16(x)) @ np.abs(W4).T + np.abs(p["b4"])) + 1e-30).all()
    y = b16(h) @ W5.T + p["b5"]
    got = out.cpu().numpy().astype(np.float64)[:, 3:]
    assert (np.abs(got - y) <= eps * (np.abs(b16(h)) @ np.abs(W5).T + np.abs(p["b5"]))).all()
    gy = b16((2 * (out[:, 3:] - target[:, 3:]) / torch.tensor(12.0 * B)).cpu().numpy())
    gh = b16((gy @ W5) * (h > 0))
    for name, ref, tol in (("w5", gy.T @ b16(h), 1e-4), ("b5", gy.sum(0), 1e-4),
                           ("w4", gh.T @ b16(x), 1e-3), ("b4", gh.sum(0), 1e-3)):
        assert np.linalg.norm(d[name].reshape(ref.shape) - ref) <= tol * np.linalg.norm(ref), name

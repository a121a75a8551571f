"""The warm-start network's passes around its convolutions: the fused ReLU mask
and bias gradient, and the one-call forward pass, against the single torch
operations of the same layers.

Tolerances: masked gradients and pooled or copied activations are exact; a bias
gradient is a sum of n BF16 values held in FP32 on both sides, so it may differ
from the FP64 sum by a few units of 2^-24 of sum |g|; the forward pass differs
from the layer-by-layer one in the order of the head's 16-term FP32 sum only.
"""

import copy

import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mods():
    from paper_2609_30166_gb300 import _build, ctrex, unet

    _build.build_library()
    return ctrex, unet


@pytest.mark.parametrize("shape", [(1, 1, 1, 1, 8), (1, 3, 5, 7, 16), (2, 9, 8, 33, 32), (1, 4, 4, 4, 128),
                                   (1, 1, 1, 2, 2048), (2, 64, 64, 40, 16)])
@pytest.mark.parametrize("relu", [True, False])
def test_bias_grad(mods, shape, relu):
    ctrex, _ = mods
    g = torch.Generator(device="cuda").manual_seed(1)
    dy = torch.randn(shape, generator=g, device="cuda").to(torch.bfloat16)
    y = torch.randn(shape, generator=g, device="cuda").relu().to(torch.bfloat16) if relu else None
    want = dy * (y > 0).to(dy.dtype) if relu else dy
    got, db = ctrex.conv3d_bias_grad(dy, y)
    assert torch.equal(got, want)
    ref = want.double().reshape(-1, shape[-1])
    assert bool(((db.double() - ref.sum(0)).abs() <= 8 * 2.0 ** -24 * ref.abs().sum(0) + 1e-30).all())


def test_bias_grad_of_other_channel_counts_is_left_alone(mods):
    ctrex, _ = mods
    for c in (4, 24, 40):
        assert ctrex.conv3d_bias_grad(torch.zeros((1, 2, 2, 2, c), dtype=torch.bfloat16, device="cuda")) is None


@pytest.mark.parametrize("shape,base", [((1, 8, 8, 8), 16), ((2, 16, 24, 8), 16), ((1, 40, 32, 48), 16),
                                        ((1, 16, 16, 16), 8), ((1, 16, 8, 16), 32)])
def test_one_call_forward(mods, shape, base):
    ctrex, unet = mods
    net = unet.UNet3D(base=base, seed=3)
    with torch.no_grad():
        net.head_w.normal_()
        net.head_b.fill_(0.3)
        for layer in net._layers():
            layer.b.normal_(std=0.1)
    net = net.cuda()
    x = torch.rand(shape, generator=torch.Generator(device="cuda").manual_seed(2), device="cuda")
    want = net(x).detach()  # parameters require gradients: layer by layer
    with torch.no_grad():
        assert net._one_call(x) is not None
        got = net(x)
        assert torch.allclose(got, want, rtol=0, atol=1e-5 * float((want - x).abs().max()) + 1e-6)
        # whatever has to see single operations keeps the layers
        hooked = copy.deepcopy(net)
        seen = []
        hooked.d1[1].register_forward_hook(lambda *a: seen.append(1))
        assert torch.equal(hooked(x), want) and seen
        assert net._one_call(x.transpose(1, 2)) is None and net._one_call(x.double()) is None
    assert net._one_call(x) is None
    ctrex.conv_status_check()


def _net(unet):
    return unet.UNet3D(base=8, seed=3).cuda(), torch.rand((1, 8, 8, 8), device="cuda")


def test_forward_mode_is_refused(mods):
    """The layers have no forward-mode derivative: a dual input or parameter
    raises, as it does with gradients enabled, and is never taken for a
    constant."""
    _, unet = mods
    import torch.autograd.forward_ad as fwd

    net, x = _net(unet)
    with torch.no_grad(), fwd.dual_level():
        for name, grad in ((None, False), ("e1.0.w", False), ("head_b", False)):
            if name is None:
                with pytest.raises(NotImplementedError):
                    net(fwd.make_dual(x, torch.ones_like(x)))
            else:
                p = dict(net.named_parameters())[name]
                dual = fwd.make_dual(p.detach(), torch.ones_like(p))
                if name == "head_b":  # the head alone is made of differentiable operations
                    y = torch.func.functional_call(net, {name: dual}, (x,))
                    assert fwd.unpack_dual(y).tangent is not None
                else:
                    with pytest.raises(NotImplementedError):
                        torch.func.functional_call(net, {name: dual}, (x,))


def test_replaced_layers_are_called(mods):
    """Offloading and instrumentation replace a layer's forward on the
    instance, or override a part of the network in a subclass."""
    _, unet = mods
    net, x = _net(unet)
    seen = []
    layer = net.e1[0]
    plain = layer.forward

    def wrapped(v):
        seen.append("forward")
        return plain(v)

    class Sub(unet.UNet3D):
        @staticmethod
        def _block(convs, v):
            seen.append("subclass")
            return unet.UNet3D._block(convs, v)

    def block(convs, v):
        seen.append("block")
        return unet.UNet3D._block(convs, v)

    with torch.no_grad():
        layer.forward = wrapped
        net(x)
        assert seen == ["forward"]
        del layer.forward, seen[:]
        sub = Sub(base=8, seed=3).cuda()
        sub(x)
        assert seen == ["subclass"] * 7
        del seen[:]
        net._block = block
        net(x)
        assert seen == ["block"] * 7


@pytest.mark.parametrize("where,name", [("_functorch", "peek_interpreter_stack"), (None, "_len_torch_dispatch_stack"),
                                        (None, "_len_torch_function_stack")])
def test_inference_without_private_names(mods, monkeypatch, where, name):
    """A torch that does not tell what is active keeps the layers."""
    _, unet = mods
    net, x = _net(unet)
    with torch.no_grad():
        want = net(x)
        monkeypatch.delattr(getattr(torch._C, where) if where else torch._C, name)
        assert net._one_call(x) is None
        got = net(x)
    monkeypatch.undo()
    assert torch.allclose(got, want, rtol=0, atol=1e-5)


@pytest.mark.parametrize("relu", [True, False])
def test_second_derivative_through_the_bias_gradient(mods, relu):
    """With create_graph the bias gradient is a function of the output's
    gradient: sum over the voxels of dy (where the ReLU passes)."""
    _, unet = mods
    layer = unet.Conv3(16, 16, relu=relu, gen=torch.Generator().manual_seed(2)).cuda()
    x = torch.randn((1, 4, 6, 8, 16), device="cuda").to(torch.bfloat16)
    y = layer(x)
    dy = torch.randn(y.shape, device="cuda").to(torch.bfloat16).requires_grad_(True)
    (db,) = torch.autograd.grad(y, layer.b, grad_outputs=dy, create_graph=True)
    assert db.requires_grad
    k = torch.arange(1.0, 17.0, device="cuda")
    (g,) = torch.autograd.grad((db * k).sum(), dy)
    mask = (y > 0) if relu else torch.ones_like(y)
    assert torch.equal(g, (mask * k).to(g.dtype))


@pytest.mark.parametrize("relu", [True, False])
def test_batched_bias_gradient(mods, relu):
    """Several output gradients at once (vmap over the backward pass), where
    only the bias asks for a gradient."""
    _, unet = mods
    layer = unet.Conv3(16, 16, relu=relu, gen=torch.Generator().manual_seed(2)).cuda()
    layer.w.requires_grad_(False)
    y = layer(torch.randn((1, 4, 6, 8, 16), device="cuda").to(torch.bfloat16))
    dy = torch.randn((3,) + y.shape, device="cuda").to(torch.bfloat16)
    (db,) = torch.autograd.grad(y, layer.b, grad_outputs=dy, is_grads_batched=True, retain_graph=True)
    for k in range(3):
        (want,) = torch.autograd.grad(y, layer.b, grad_outputs=dy[k], retain_graph=True)
        assert torch.allclose(db[k], want, rtol=0, atol=8 * 2.0 ** -24 * float(dy[k].float().abs().sum()))


def test_bias_grad_of_long_sums(mods):
    """103 terms a thread, of one sign: the bound of test_bias_grad."""
    ctrex, _ = mods
    g = torch.Generator(device="cuda").manual_seed(4)
    dy = (torch.randn((2, 200, 200, 200, 16), generator=g, device="cuda") + 1.0).to(torch.bfloat16)
    _, db = ctrex.conv3d_bias_grad(dy)
    flat = dy.reshape(-1, 16)
    want = sum(part.double().sum(0) for part in flat.split(1 << 21))
    size = sum(part.double().abs().sum(0) for part in flat.split(1 << 21))
    assert bool(((db.double() - want).abs() <= 8 * 2.0 ** -24 * size).all())

"""The training kernel over batches around its 32-sample blocks and 64-sample
pairs, and over more pairs of blocks than the device holds at once: against the
FP32-activation kernels and as a sum over parts of the batch."""
import pytest
import torch

import paper_2108_11775_gb300 as pdmp

pytestmark = pytest.mark.gpu


def setup(B, seed=2):
    assert torch.cuda.is_available()
    g = torch.Generator(device="cuda").manual_seed(1000 * seed + B)
    net = pdmp.Surrogate([0.0] * 3, [5.0] * 3, [0.05, 0.07, 0.03], seed=seed)
    net.b.copy_(0.1 * torch.randn(pdmp.MLP_NB, generator=g, device="cuda"))
    x = torch.rand(B, 3, generator=g, device="cuda") * 5.0
    return net, x, x + 0.05 * torch.randn(B, 3, generator=g, device="cuda")


def layers(gW, gb):
    H, E = pdmp.MLP_H, pdmp.MLP_ENC
    return list(torch.split(gW, [H * E, H * H, H * H, 3 * H])) + list(torch.split(gb, [H, H, H, 3]))


@pytest.mark.parametrize("B", [31, 32, 33, 63, 64, 65, 96, 129, 9000, 20001])
def test_gradient_matches_the_fp32_activation_kernels(B):
    net, x, y = setup(B)
    l0, w0, b0 = net.gradient(x, y, fp32_act=True)
    l1, w1, b1 = net.gradient(x, y)
    assert abs(float(l1) - float(l0)) <= 2e-2 * float(l0)     # BF16 activations
    for q, r in zip(layers(w1, b1), layers(w0, b0)):
        assert float((q - r).norm()) <= 2e-2 * float(r.norm())


@pytest.mark.parametrize("parts", [(1, 31), (32, 1), (33, 64, 65), (127, 9000, 1)])
def test_gradient_is_the_mean_over_parts_of_the_batch(parts):
    """The same BF16 operands in other places; FP32 sums and dY's scale round differently (2^-9 of a BF16 dY)."""
    B = sum(parts)
    net, x, y = setup(B, seed=5)
    _, w, b = net.gradient(x, y)
    sw, sb, o = torch.zeros_like(w), torch.zeros_like(b), 0
    for n in parts:
        _, pw, pb = net.gradient(x[o:o + n].clone(), y[o:o + n].clone())
        sw += pw * (n / B)
        sb += pb * (n / B)
        o += n
    for q, r in zip(layers(sw, sb), layers(w, b)):
        assert float((q - r).norm()) <= 2.0 ** -7 * float(r.norm())


def test_the_step_takes_the_gradient():
    net, x, y = setup(200)
    _, w, b = net.gradient(x, y)
    net.train_step(x, y)
    # the first step's first moment is (1 - beta1) of the gradient
    torch.testing.assert_close(net.adam[:pdmp.MLP_NW], (1.0 - 0.9) * w, rtol=1e-6, atol=0.0)
    torch.testing.assert_close(net.adam[2 * pdmp.MLP_NW:2 * pdmp.MLP_NW + pdmp.MLP_NB], (1.0 - 0.9) * b, rtol=1e-6,
                               atol=0.0)
    copies = (net.W_bf16.clone(), net.Wt_bf16.clone())
    net.refresh()
    assert torch.equal(copies[0], net.W_bf16) and torch.equal(copies[1], net.Wt_bf16)

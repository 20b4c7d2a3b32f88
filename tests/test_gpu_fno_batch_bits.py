"""Training batches of four samples and more mix modes and transform back along y in
kernels of their own; a rounding that differs there from the other kernels' turns over
a BF16 value now and then, and all gradients with it.  Both are held to the same bits:
the forward pass trained on is the one that mm_fno_forward returns (a loss of exactly
zero against it), and a batch of four whose other samples have a zero loss gives half
the spectral gradients of such a batch of two (a power of two: exact; at width 64 the
transforms along y split alike for both)."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def network(H, W, C, m, L):
    """A network with weights at its initial scale, its parameters, and inputs of four samples."""
    from paper_1406_7459_gb300 import mm
    gen = torch.Generator(device="cuda").manual_seed(H * W)

    def normal(shape, scale):
        return scale * torch.randn(shape, generator=gen, device="cuda")

    flat = torch.cat([v.reshape(-1) for v in (
        normal((C, 5), 5 ** -0.5), normal((C,), 0.05), normal((2, L, C, C, 2 * m, m), 1 / C),
        normal((L, C, C), C ** -0.5), normal((L, C), 0.05), normal((3, C), C ** -0.5), normal((3,), 0.05))])
    net = mm.mm_fno_create(H, W, C, m, L, max_batch=4)
    mm.mm_fno_set_params(net, flat)
    x, t = normal((4, 3, H, W), 1.0), normal((1, 3, H, W), 1.0)
    return mm, net, flat, x, mm.mm_fno_forward(net, x, torch.empty_like(x)), t


# (H, W, width, modes, layers)
CASES = [(62, 86, 16, 16, 4), (64, 96, 16, 16, 4), (62, 86, 16, 4, 4), (128, 128, 32, 16, 2), (33, 49, 8, 8, 4),
         (101, 133, 32, 12, 2)]


@pytest.mark.parametrize("case", CASES, ids=["x".join(map(str, c)) for c in CASES])
def test_forward_of_a_training_batch(case):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    mm, net, flat, x, y, _ = network(*case)
    g = torch.empty_like(flat)
    assert mm.mm_fno_grad(net, x, y, g) == 0.0
    assert not g.any()


@pytest.mark.parametrize("case", [(62, 86, 64, 16, 3), (128, 96, 64, 8, 3)], ids=["62x86", "128x96"])
def test_spectral_gradients_of_a_training_batch(case):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    mm, net, flat, x, y, t = network(*case)
    _, _, C, m, L = case
    four, two = torch.empty_like(flat), torch.empty_like(flat)
    t = torch.cat([t, y[1:]])
    mm.mm_fno_grad(net, x, t, four)
    mm.mm_fno_grad(net, x[:2].contiguous(), t[:2].contiguous(), two)
    r = slice(6 * C, 6 * C + 4 * L * C * C * m * m)
    assert two[r].any() and torch.equal(2 * four[r], two[r])

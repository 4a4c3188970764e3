"""Gradients of weighted BP are summed over the shots in FP64: sums whose parts
cancel, lie above the float range on the way, or are not finite."""
import math

import pytest

import bpdc_inputs as bi

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def case():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2510_08695_gb300 as pkg
    from paper_2510_08695_gb300 import wbp
    g = pkg.Graph.from_problem(bi.bb_problem("bb72", 0.06), pkg.Options(variant=1, max_iter=2))
    syn, _, _ = g.sample(64, 11, 0)
    gen = torch.Generator(device="cuda").manual_seed(5)
    W = 1 + 0.1 * torch.randn((2, 2, g.E), generator=gen, device="cuda")
    up = torch.randn((64, 2, g.N), generator=gen, device="cuda")

    def grad(shots, upstream):
        w = W.clone().requires_grad_(True)
        wbp.weighted_bp(w, g, syn[shots].contiguous(), 20.0, 1).backward(upstream)
        return w.grad

    return torch, up, grad


@pytest.mark.parametrize("B", [7, 9, 33, 1217, 2001])
def test_partial_sums_above_the_float_range(case, B):
    """One shot B times, (B + 1) / 2 times with its upstream gradient and then as
    often but once with the opposite: half the sum is up to 2^137, the sum is the
    gradient of one shot.  Every partial sum has at most 24 + 11 bits, so FP64
    gives it exactly in any order."""
    torch, up, grad = case
    one = grad([3], up[3:4])
    k = 126 - math.floor(math.log2(float(one.abs().max())))
    big = up[3:4] * 2.0 ** (k // 2) * 2.0 ** (k - k // 2)
    ref = grad([3], big)
    assert bool(ref.isfinite().all()) and 2.0 ** 126 <= float(ref.abs().max()) < 2.0 ** 127
    sign = torch.ones(B, 1, 1, device="cuda")
    sign[(B + 1) // 2:] = -1
    assert torch.equal(grad([3] * B, sign * big), ref)


@pytest.mark.parametrize("B", [4, 13, 500, 1300])
def test_cancelling_sums(case, B):
    """Large gradients and their opposites around small ones, against the FP64 sum
    of the shots' own gradients: two sums of B terms in some order, each within
    B 2^-53 of the sum of the magnitudes, and the result rounded to 24 bits."""
    torch, up, grad = case
    gen = torch.Generator().manual_seed(B)
    shot = torch.randint(0, 64, (B,), generator=gen)
    scale = 2.0 ** torch.randint(0, 30, (B,), generator=gen).double()
    half = B // 2
    order = torch.randperm(half, generator=gen)
    shot[half:2 * half], scale[half:2 * half] = shot[:half][order], -scale[:half][order]
    scale[order[0]] += 1   # what is left in the end
    shot, u = shot.tolist(), up[shot.cuda()] * scale.float().cuda()[:, None, None]
    parts = torch.stack([grad([s], u[i:i + 1]).double() for i, s in enumerate(shot)])
    got = grad(shot, u).double()
    want = parts.sum(0)
    bound = 2 * B * 2.0 ** -53 * parts.abs().sum(0) + 2.0 ** -24 * want.abs() + 1e-37
    assert ((got - want).abs() <= bound).all()


@pytest.mark.parametrize("B", [3, 40, 1300])
@pytest.mark.parametrize("value", [math.inf, math.nan])
def test_infinities_and_nans(case, B, value):
    torch, up, grad = case
    shots = [i % 64 for i in range(B)]
    u = up[shots].clone()
    u[B // 2, 1] = value
    alone = torch.stack([grad([s], u[i:i + 1]).double() for i, s in enumerate(shots[:3])] +
                        [grad([shots[B // 2]], u[B // 2:B // 2 + 1]).double()])
    got = grad(shots, u)
    bad = ~alone[-1].isfinite()
    assert bool(bad.any())
    assert torch.equal(~got.isfinite(), bad)
    assert torch.equal(got[bad].isnan(), alone[-1][bad].isnan())

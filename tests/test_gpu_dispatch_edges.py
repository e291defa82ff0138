"""GPU parity at the places where a kernel or a dispatch rule changes over: remainders, the edges of
tiles, one more layer than fits a launch.  Float64 references on the host; bf16 inputs are exact on
both sides, so only fp32 accumulation order (norms) and one bf16 rounding of R_i * g (sums) differ."""
import numpy as np
import pytest
import torch

from paper_2609_40335_b200 import binding as dp

pytestmark = pytest.mark.gpu


def bf16(shape, std, seed, ld=None):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    t = torch.full(shape[:-1] + (ld or shape[-1],), float("nan"), dtype=torch.bfloat16, device="cuda")
    t[..., :shape[-1]] = torch.randn(shape, generator=g, device="cuda") * std
    return t


def f64(t, cols):
    return t[..., :cols].double().cpu().numpy()


@pytest.mark.parametrize("n_layers", [102, 103, 112, 113])
def test_as_many_layers_as_one_launch_holds_and_one_more(n_layers):
    """The clipped sums take 102 layers per launch and the Gram kernels 112."""
    B, T, d, p = 2, 20, 64, 72
    layers = [dp.Linear(bf16((B, T, d), 1.0, 3 * k), bf16((B, T, p), 0.1, 3 * k + 1), d=d, p=p)
              for k in range(n_layers)]
    sq = torch.zeros(B, device="cuda")
    dp.dp_ghost_norms(layers, B, T, sq)
    clip = torch.tensor([0.5, 0.25], device="cuda")
    outs = [torch.full((p, d), float("nan"), device="cuda") for _ in layers]
    dp.dp_clip_accumulate_grouped(layers, B, T, None, 1.0, outs, clip=clip)
    want_sq = np.zeros(B)
    for l, o in zip(layers, outs):
        per = np.einsum("btp,btd->bpd", f64(l.G, p), f64(l.A, d))
        want_sq += (per ** 2).sum((1, 2))
        # powers of two: R_i * g is exact in bf16, what is left is fp32 accumulation of 40 terms
        want = np.einsum("b,bpd->pd", clip.double().cpu().numpy(), per)
        assert np.linalg.norm(o.double().cpu().numpy() - want) < 1e-5 * np.linalg.norm(want)
    assert (np.abs(sq.double().cpu().numpy() / want_sq - 1) < 1e-5).all()

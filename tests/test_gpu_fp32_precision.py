"""fp32 inputs on the tensor cores: the error of long sums against 64 bits.  Operands are two bf16 terms (4.5e-6 of a
product's size, random); an MMA adds 16 products to a sum and rounds it towards zero, by 2^-24 of it on average."""
import pytest
import torch

from paper_2609_40335_b200 import binding as dp

pytestmark = pytest.mark.gpu


def normal(*shape, std=1.0, seed=0):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return torch.empty(*shape, device="cuda").normal_(0.0, std, generator=g)


# 150 layers of one output tile share the tensors: tiles enough that K is not split; of one layer by itself it is
@pytest.mark.parametrize("n_layers", [150, 1])
def test_clipped_sums_over_many_tokens(n_layers):
    B, T, d, p = 64, 256, 64, 72
    A, G = normal(B, T, d, seed=1), normal(B, T, p, std=1e-2, seed=2)
    clip = 1e-3 * torch.rand(B, generator=torch.Generator(device="cuda").manual_seed(3), device="cuda")
    layers = [dp.Linear(A, G, d=d, p=p) for _ in range(n_layers)]
    outs = [torch.empty(p, d, device="cuda") for _ in layers]
    ws = torch.empty(n_layers * 4 * B * T * (d + p) + (1 << 28), dtype=torch.uint8, device="cuda")
    dp.dp_clip_accumulate_grouped(layers, B, T, None, 1.0, outs, clip=clip, ws=ws)
    want = torch.einsum("btp,btd->pd", G.double() * clip.double()[:, None, None], A.double())
    # 1024 MMAs of full size; the sum grows as the root of their number: 2/3 * 1024 * 2^-24 if all errors add up
    bound = 4.5e-6 + 2 / 3 * 1024 * 2.0 ** -24
    for o in (outs[0], outs[-1]):
        assert float((o.double() - want).norm() / want.norm()) < bound


# many examples: work items enough without cutting wide operands
@pytest.mark.parametrize("B,T", [(64, 256), (128, 64)])
@pytest.mark.parametrize("shapes", [[(768, 2304), (768, 768), (768, 3072), (3072, 768)], [(66, 2000)], [(128, 5000), (64, 2304)]])
def test_norms_of_many_examples(shapes, B, T):
    layers = [dp.Linear(normal(B, T, d, seed=k), normal(B, T, p, std=1e-2, seed=50 + k), d=d, p=p, mode=dp.DP_NORM_GHOST)
              for k, (d, p) in enumerate(shapes)]
    sq = torch.zeros(B, device="cuda")
    ws = torch.empty(1 << 32, dtype=torch.uint8, device="cuda")
    dp.dp_ghost_norms(layers, B, T, sq, ws=ws)
    want = 0
    for l in layers:
        a, g = l.A.double(), l.G.double()
        want = want + (torch.bmm(a, a.transpose(1, 2)) * torch.bmm(g, g.transpose(1, 2))).sum((1, 2))
    # A Gram entry's diagonal is a sum of positive terms: an MMA of full size, four per 64 columns, takes 2^-24 of its
    # final size from it (measured: 0.7 of that).  Narrow and wide part of an item are 60 steps together.  lo lo' is left
    # out: |lo| <= 2^-8 of a value's power of two, 2.6e-6 of the sum of squares, for either operand.
    assert float(((sq.double() - want) / want).norm() / B ** 0.5) < 60 * 4 * 2.0 ** -24 + 2 * 2.6e-6

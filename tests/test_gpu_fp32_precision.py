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

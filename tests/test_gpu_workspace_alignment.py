"""Workspaces on a 4-byte boundary: the same results where that will do, a status where it will not."""
import pytest
import torch

from paper_2609_40335_b200 import binding as dp

pytestmark = pytest.mark.gpu


def ws_at(nbytes, offset):
    return torch.empty(int(nbytes) + 16, dtype=torch.uint8, device="cuda")[offset:offset + int(nbytes)]


# one block, chunks with one and with several blocks in the scan
@pytest.mark.parametrize("n,V", [(300, 700), (5000, 1000), (5000, 5003), (40000, 9000)])
@pytest.mark.parametrize("offset", [4, 8])
def test_token_sort_and_row_sums(n, V, offset):
    g = torch.Generator(device="cuda")
    g.manual_seed(n)
    ids = torch.randint(0, V, (4, n // 4), generator=g, device="cuda", dtype=torch.int32)
    G = torch.randn(4, n // 4, 40, generator=g, device="cuda")
    clip = torch.rand(4, generator=g, device="cuda")
    lib, got = dp.load(), []
    for off in (0, offset):
        perm, seg = torch.empty(n, dtype=torch.int32, device="cuda"), torch.empty(V + 1, dtype=torch.int32, device="cuda")
        out = torch.empty(V, 40, device="cuda")
        sq = torch.zeros(4, device="cuda")
        dp.dp_embed_sort(ids, V, perm, seg, ws=ws_at(lib.dp_embed_sort_ws_bytes(4, n // 4, V), off))
        dp.dp_clip_accumulate_embed(ids, G, V, None, 1.0, out, d=40, clip=clip,
                                    ws=ws_at(lib.dp_clip_accumulate_embed_ws_bytes(4, n // 4, 40, V), off))
        if n // 4 <= 4096:
            dp.dp_embed_norms(ids, G, V, sq, ws=ws_at(lib.dp_embed_norms_ws_bytes(4, n // 4, 40), off))
        got.append((perm, seg, out, sq))
    torch.cuda.synchronize()
    for a, b in zip(*got):
        assert torch.equal(a, b)


@pytest.mark.parametrize("offset", [4, 8])
def test_k_split_planes(offset):
    B, T, d, p = 16, 64, 72, 136                     # few tiles: K is split
    g = torch.Generator(device="cuda")
    g.manual_seed(1)
    layer = [dp.Linear(torch.randn(B, T, d, generator=g, device="cuda").bfloat16(),
                       torch.randn(B, T, p, generator=g, device="cuda").bfloat16(), d=d, p=p)]
    clip = torch.rand(B, generator=g, device="cuda")
    need, got = dp.dp_clip_accumulate_grouped_ws_bytes(layer, B, T), []
    assert need > 4 * d * p
    for off in (0, offset):
        out = torch.empty(p, d, device="cuda")
        dp.dp_clip_accumulate_grouped(layer, B, T, None, 1.0, [out], clip=clip, ws=ws_at(need, off))
        got.append(out)
    assert torch.equal(*got)


@pytest.mark.parametrize("dtype,d,p", [(torch.float32, 64, 128), (torch.bfloat16, 64, 4096)])
def test_operands_for_tma_are_refused_a_misaligned_workspace(dtype, d, p):
    B, T = 2, 64
    layer = [dp.Linear(torch.zeros(B, T, d, dtype=dtype, device="cuda"), torch.zeros(B, T, p, dtype=dtype, device="cuda"), d=d, p=p)]
    out, clip = torch.full((p, d), 7.0, device="cuda"), torch.ones(B, device="cuda")
    launched = dp.dp_kernel_launches()
    with pytest.raises(dp.DpGhostError) as e:
        dp.dp_clip_accumulate_grouped(layer, B, T, None, 1.0, [out], clip=clip,
                                      ws=ws_at(dp.dp_clip_accumulate_grouped_ws_bytes(layer, B, T), 4))
    assert e.value.status == 3 and dp.dp_kernel_launches() == launched
    torch.cuda.synchronize()
    assert (out == 7.0).all()

"""GPU parity at the places where a kernel or a dispatch rule changes over: remainders, the edges of
tiles, one more layer than fits a launch.  Float64 references on the host; bf16 inputs are exact on
both sides, so only fp32 accumulation order (norms) and one bf16 rounding of R_i * g (sums) differ."""
import numpy as np
import pytest
import torch

from paper_2609_40335_b200 import binding as dp, pipeline

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


def reference_sort(ids, V):
    flat = ids.cpu().numpy().reshape(-1)
    ok = np.flatnonzero((flat >= 0) & (flat < V))
    perm = ok[np.argsort(flat[ok], kind="stable")]
    return perm, np.concatenate([[0], np.cumsum(np.bincount(flat[ok], minlength=V))])


# one block or chunks of 1024 tokens, of 4096 beyond 32768 tokens
@pytest.mark.parametrize("B,T,V", [(1, 1, 1), (1, 31, 5), (2, 2048, 8192), (1, 4097, 100), (3, 1365, 8193),
                                   (8, 4096, 300), (1, 32769, 70000), (3, 13107, 9)])
def test_token_sort_at_the_edges_of_its_variants(B, T, V):
    g = torch.Generator(device="cuda")
    g.manual_seed(B * T)
    ids = torch.randint(-1, V + 1, (B, T), generator=g, device="cuda", dtype=torch.int32)   # -1, V: out of range
    if T > 100:
        ids[:, 50:T // 2] = min(2, V - 1)                # one id far more frequent than the others
    perm = torch.full((B * T,), -7, dtype=torch.int32, device="cuda")
    seg = torch.empty(V + 1, dtype=torch.int32, device="cuda")
    dp.dp_embed_sort(ids, V, perm, seg)
    want_perm, want_seg = reference_sort(ids, V)
    assert np.array_equal(seg.cpu().numpy(), want_seg)
    got = perm.cpu().numpy()
    assert np.array_equal(got[:len(want_perm)], want_perm)
    assert (got[len(want_perm):] == -7).all()


# one block up to 2048 tokens and 8192 ids; counts of up to 8 chunks are added up token by token, of more once for
# all; tokens per 1024 ids are counted in shared memory up to 262144 ids
@pytest.mark.parametrize("B,T,V", [(1, 2048, 8192), (1, 2049, 8192), (1, 64, 8193), (2, 4096, 6000),
                                   (1, 8193, 6000), (9, 4096, 1025), (8, 4097, 262144), (2, 4096, 262145), (300, 2048, 5000)])
def test_token_sort_at_the_lines_of_its_rules(B, T, V):
    test_token_sort_at_the_edges_of_its_variants(B, T, V)


# 48 rows of one id are summed by one warp, 49 by eight; rows are cut into parts of at least 64
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("T,frequent", [(48, 48), (49, 49), (64, 48), (65, 49), (129, 80), (1000, 500), (4096, 2100)])
def test_embedding_norm_with_frequent_tokens(dtype, T, frequent):
    B, d, V = 2, 264, 5000
    g = torch.Generator(device="cuda")
    g.manual_seed(T)
    ids = torch.randint(0, V, (B, T), generator=g, device="cuda", dtype=torch.int32)
    for i in range(B):
        ids[i, torch.randperm(T, generator=g, device="cuda")[:frequent]] = 3 + i
    G = torch.randn(B, T, d, generator=g, device="cuda").to(torch.float32 if dtype == "f32" else torch.bfloat16)
    sq = torch.zeros(B, device="cuda")
    first = torch.empty(B, T, dtype=torch.int32, device="cuda")
    dp.dp_embed_norms(ids, G, V, sq, first_occ=first)
    for i in range(B):
        row = ids[i].cpu().numpy()
        table = np.zeros((V, d))
        np.add.at(table, row, G[i].double().cpu().numpy())
        want = (table ** 2).sum()
        assert abs(float(sq[i]) / want - 1) < 1e-5       # fp32 sums of at most 2100 terms
        uniq, where = np.unique(row, return_index=True)
        assert np.array_equal(first[i].cpu().numpy(), where[np.searchsorted(uniq, row)])


# fp32 layers share the workspace in groups: all at once, one at a time (the reported size holds the
# largest with little to spare), and mixed with layers that stay on the FMA kernels
@pytest.mark.parametrize("extra", [0, 1 << 26])
@pytest.mark.parametrize("T", [32, 128, 129, 260])
def test_fp32_layers_in_groups(extra, T):
    B = 2
    shapes = [(64, 64), (136, 72), (64, 300), (40, 64), (520, 256), (65, 131)]
    g = torch.Generator(device="cuda")
    g.manual_seed(T)
    layers = [dp.Linear(torch.randn(B, T, d, generator=g, device="cuda"),
                        0.1 * torch.randn(B, T, p, generator=g, device="cuda"), d=d, p=p) for d, p in shapes]
    layers[1].mode = dp.DP_NORM_DIRECT

    def ws(need):
        return torch.empty(max(need, 256) + extra, dtype=torch.uint8, device="cuda")

    sq = torch.zeros(B, device="cuda")
    dp.dp_ghost_norms(layers, B, T, sq, ws=ws(dp.dp_ghost_norms_ws_bytes(layers, B, T)))
    clip = torch.tensor([0.3, 1.0], device="cuda")
    outs = [torch.ones(p, d, device="cuda") for d, p in shapes]
    dp.dp_clip_accumulate_grouped(layers, B, T, None, 1.0, outs, beta=1.0, clip=clip,
                                  ws=ws(dp.dp_clip_accumulate_grouped_ws_bytes(layers, B, T)))
    want_sq = np.zeros(B)
    for l, o in zip(layers, outs):
        per = np.einsum("btp,btd->bpd", f64(l.G, l.p), f64(l.A, l.d))
        want_sq += (per ** 2).sum((1, 2))
        want = 1.0 + np.einsum("b,bpd->pd", clip.double().cpu().numpy(), per)
        assert np.linalg.norm(o.double().cpu().numpy() - want) < 2e-5 * np.linalg.norm(want)   # two bf16 terms
    assert (np.abs(sq.double().cpu().numpy() / want_sq - 1) < 2e-5).all()


# one reduction for the K-split planes of all layers: widths that are and are not multiples of 4
@pytest.mark.parametrize("shapes", [[(64, 64), (256, 300)], [(50, 70), (33, 41), (3, 5)], [(512, 592)], [(512, 591), (4, 1)]])
@pytest.mark.parametrize("noise", [False, True])
def test_k_split_planes_of_several_layers(shapes, noise):
    B, T = 16, 64
    layers = [dp.Linear(bf16((B, T, d), 1.0, k, ld=(d + 7) // 8 * 8), bf16((B, T, p), 0.1, 50 + k, ld=(p + 7) // 8 * 8),
                        d=d, p=p) for k, (d, p) in enumerate(shapes)]
    clip = torch.full((B,), 0.5, device="cuda")
    start = [torch.randn(p, d, device="cuda") for d, p in shapes]
    plain, outs = [t.clone() for t in start], [t.clone() for t in start]
    dp.dp_clip_accumulate_grouped(layers, B, T, None, 1.0, plain, beta=1.0, clip=clip)
    if noise:
        ids = list(range(5, 5 + len(shapes)))
        dp.dp_clip_accumulate_noise_grouped(layers, B, T, None, 1.0, outs, 0.7, 0.5, 11, ids, 2, beta=1.0, clip=clip)
        for t, i in zip(plain, ids):
            dp.dp_add_noise(t, 0.7, 1.0, 0.5, 11, i, 2)
        for a, b in zip(plain, outs):
            assert torch.equal(a, b)
    else:
        for l, o, s in zip(layers, plain, start):
            want = s.double().cpu().numpy() + 0.5 * np.einsum("btp,btd->pd", f64(l.G, l.p), f64(l.A, l.d))
            assert np.linalg.norm(o.double().cpu().numpy() - want) < 1e-5 * np.linalg.norm(want)


# two-tile items: both orientations, leftover lines of tiles paired along their length, a last corner tile,
# items converted to single tiles in a last wave, partial tiles, widths that are no multiple of 4 or 8
BIG_SHAPES = [[(257, 19001)], [(19000, 250)], [(700, 13000), (100, 3000), (64, 64)], [(511, 6500), (2600, 1281), (768, 768)],
              [(768, 14300)]]


@pytest.mark.parametrize("shapes", BIG_SHAPES)
@pytest.mark.parametrize("beta,noise,B,T", [(0.0, False, 3, 50), (1.0, True, 3, 50), (0.0, True, 1, 7), (0.0, True, 15, 64),
                                            (0.0, True, 16, 64)])
def test_two_tile_items(shapes, beta, noise, B, T):
    layers = [dp.Linear(bf16((B, T, d), 1.0, k, ld=(d + 7) // 8 * 8), bf16((B, T, p), 0.1, 50 + k, ld=(p + 7) // 8 * 8),
                        d=d, p=p) for k, (d, p) in enumerate(shapes)]
    clip = torch.tensor([2.0 ** -(i % 3) for i in range(B)], device="cuda")
    start = [torch.randn(p, d, device="cuda") for d, p in shapes]
    outs, st = [t.clone() for t in start], torch.zeros(1, dtype=torch.int32, device="cuda")
    dp.dp_clip_accumulate_grouped(layers, B, T, None, 1.0, outs, beta=beta, clip=clip, dev_status=st)
    for l, o, s in zip(layers, outs, start):
        g = l.G[..., :l.p].double().cpu() * clip.double().cpu()[:, None, None]
        want = g.reshape(-1, l.p).T @ l.A[..., :l.d].double().cpu().reshape(-1, l.d) + beta * s.double().cpu()
        # powers of two: R_i * x is exact in bf16, what is left is fp32 accumulation
        assert float((o.double().cpu() - want).norm() / want.norm()) < 1e-5
    if noise:
        again = [t.clone() for t in start]
        ids = list(range(3, 3 + len(shapes)))
        dp.dp_clip_accumulate_noise_grouped(layers, B, T, None, 1.0, again, 0.9, 0.5, 7, ids, 1, beta=beta, clip=clip,
                                            dev_status=st)
        for a, o, i in zip(again, outs, ids):
            dp.dp_add_noise(o, 0.9, 1.0, 0.5, 7, i, 1)
            assert torch.equal(a, o)
    assert int(st.item()) == 0


# straight code for noise at scale 1 onto aligned outputs, a few odd columns beside it (chunks of 32 columns, words of
# eight, widths whose noise is drawn later), the general code from one odd output in eight on, and for scales, beta and alignments of its own
@pytest.mark.parametrize("widths", [(768,), (800,), (776, 1284), (772, 130), (288, 40, 36, 33), (40,)])
@pytest.mark.parametrize("scale,beta,pad,offset", [(1.0, 0.0, 0, 0), (0.25, 0.0, 0, 0), (1.0, 1.0, 0, 0), (1.0, 0.0, 8, 0), (1.0, 0.0, 4, 0),
                                                   (1.0, 0.0, 0, 4), (1.0, 0.0, 1, 3)])
def test_noise_onto_outputs_of_every_kind(widths, scale, beta, pad, offset):
    B, T, p = 2, 40, 40000
    layers = [dp.Linear(bf16((B, T, d), 1.0, k, ld=(d + 7) // 8 * 8), bf16((B, T, p), 0.1, 50 + k), d=d, p=p) for k, d in enumerate(widths)]
    clip, ids = torch.tensor([0.5, 1.0], device="cuda"), list(range(3, 3 + len(widths)))

    def outs(d_all):
        return [torch.full((p * (d + pad) + offset,), 0.5, device="cuda")[offset:].view(p, d + pad)[:, :d] for d in d_all]

    got, want = outs(widths), [torch.full((p, d), 0.5, device="cuda") for d in widths]
    dp.dp_clip_accumulate_noise_grouped(layers, B, T, None, 1.0, got, 0.9, scale, 7, ids, 1, beta=beta, clip=clip)
    dp.dp_clip_accumulate_grouped(layers, B, T, None, 1.0, want, beta=beta, clip=clip)
    for g, w, i in zip(got, want, ids):
        dp.dp_add_noise(w, 0.9, 1.0, scale, 7, i, 1)
        assert torch.equal(g, w)


# K steps run over the rows of the whole batch: one example or many per 64 rows, a step that begins and ends inside
# one, the last step short; the one-tile kernel (K split and not), the two-tile one, either operand scaled
@pytest.mark.parametrize("B,T", [(1, 1), (70, 1), (37, 3), (9, 16), (5, 63), (5, 65), (3, 100), (4, 203), (2, 320)])
@pytest.mark.parametrize("d,p", [(64, 72), (768, 14300), (14300, 768)])
def test_every_row_gets_its_own_clip_factor(B, T, d, p):
    layer = dp.Linear(bf16((B, T, d), 1.0, T, ld=(d + 7) // 8 * 8), bf16((B, T, p), 0.1, B, ld=(p + 7) // 8 * 8), d=d, p=p)
    clip = torch.tensor([2.0 ** -(i % 5) for i in range(B)], device="cuda")
    out, st = torch.empty(p, d, device="cuda"), torch.zeros(1, dtype=torch.int32, device="cuda")
    dp.dp_clip_accumulate_grouped([layer], B, T, None, 1.0, [out], clip=clip, dev_status=st)
    g = layer.G[..., :p].double() * clip.double()[:, None, None]
    want = g.reshape(-1, p).T @ layer.A[..., :d].double().reshape(-1, d)
    # powers of two: R_i * x is exact in bf16, what is left is fp32 accumulation
    assert float((out.double() - want).norm() / want.norm()) < 1e-5
    assert int(st.item()) == 0


@pytest.mark.parametrize("B,T", [(37, 3), (9, 16), (3, 100), (4, 203), (6, 64)])
@pytest.mark.parametrize("d,p", [(64, 72), (768, 14300), (14300, 768)])
def test_factors_of_any_value_are_applied_in_two_parts(B, T, d, p):
    """R_i x is the correctly rounded bf16 product, for rows of one K step with factors of their own too: 1.4e-4 from rounding it once
    (one element in 1400 is rounded up instead of down or the other way); with R_i's upper half alone 2.7e-3."""
    layer = dp.Linear(bf16((B, T, d), 1.0, T, ld=(d + 7) // 8 * 8), bf16((B, T, p), 0.1, B, ld=(p + 7) // 8 * 8), d=d, p=p)
    g = torch.Generator(device="cuda")
    g.manual_seed(B + T)
    clip = torch.rand(B, generator=g, device="cuda") * 0.9 + 0.05
    out = torch.empty(p, d, device="cuda")
    dp.dp_clip_accumulate_grouped([layer], B, T, None, 1.0, [out], clip=clip)
    G, A, R = layer.G[..., :p].double(), layer.A[..., :d].double(), clip.double()[:, None, None]
    rounded = lambda x: (R * x).to(torch.bfloat16).double()
    errors, size = [], 0.0
    for r0 in range(0, p, 256):                          # which operand is scaled is each output tile's own
        both = [torch.einsum("btp,btd->pd", g_[..., r0:r0 + 256], a_) for g_, a_ in ((rounded(G), A), (G, rounded(A)))]
        for c0 in range(0, d, 256):
            got = out[r0:r0 + 256, c0:c0 + 256].double()
            errors.append(min(float((got - w[:, c0:c0 + 256]).norm()) ** 2 for w in both))
        size += float(both[0].norm()) ** 2
    assert (sum(errors) / size) ** 0.5 < 5e-4


def test_two_tile_items_give_up_cleanly():
    """A wait limit of zero: the kernel flags DP_DEV_TIMEOUT and returns; the same call then succeeds."""
    B, T, d, p = 32, 128, 512, 19000               # long enough a contraction that some wait is not over at once
    layer = [dp.Linear(bf16((B, T, d), 1.0, 1), bf16((B, T, p), 0.1, 2), d=d, p=p)]
    clip = torch.full((B,), 0.3, device="cuda")
    lib = dp.load()

    def run():
        out, st = torch.zeros(p, d, device="cuda"), torch.zeros(1, dtype=torch.int32, device="cuda")
        dp.dp_clip_accumulate_grouped(layer, B, T, None, 1.0, [out], clip=clip, dev_status=st)
        torch.cuda.synchronize()
        return out, int(st.item())

    good, flag = run()
    assert flag == 0
    prev = lib.dp_debug_set_wait_limit(0)
    try:
        assert run()[1] & dp.DP_DEV_TIMEOUT
    finally:
        lib.dp_debug_set_wait_limit(prev)
    again, flag = run()
    assert flag == 0 and torch.equal(good, again)


# the fill kernel writes whole counters of an aligned tensor, its last one element by element; a launch of it
# covers 148 * 16 * 128 counters per pass
@pytest.mark.parametrize("n", [1, 3, 4, 5, 511, 512, 513, 4 * 148 * 16 * 128 + 6])
def test_noise_fill_equals_noise_on_zeros(n):
    filled = torch.full((n + 4,), 7.0, device="cuda")
    added = torch.zeros(n, device="cuda")
    dp.dp_fill_noise(filled, 0.7, 1.5, 0.5, 11, 3, 9, n=n)
    dp.dp_add_noise(added, 0.7, 1.5, 0.5, 11, 3, 9)
    assert torch.equal(filled[:n], added)                # the same stream, bit for bit
    assert (filled[n:] == 7.0).all()


# row sums: four columns per lane, 128 per block, a warp per quarter of a chunk of 32 sorted positions;
# segments of up to 32 rows belong to one warp, longer ones to all blocks they meet
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("d,ldo,ldg", [(1, 1, 1), (3, 4, 6), (127, 131, 128), (128, 128, 128), (129, 132, 132), (264, 264, 266)])
def test_row_sums_at_the_edges(dtype, d, ldo, ldg):
    B, T, V = 2, 210, 40
    lengths = [1, 7, 8, 9, 31, 32, 33, 64, 2, 1, 30, 1, 32, 100, 3, 66]
    assert sum(lengths) == B * T
    ids = torch.repeat_interleave(torch.arange(len(lengths)), torch.tensor(lengths))
    g = torch.Generator()
    g.manual_seed(d)
    ids = ids[torch.randperm(B * T, generator=g)].to(torch.int32).view(B, T).cuda()
    G = torch.randn(B, T, ldg, generator=g).to(torch.float32 if dtype == "f32" else torch.bfloat16).cuda()
    clip = torch.rand(B, generator=g).cuda()
    out = torch.full((V, ldo), 5.0, device="cuda")
    dp.dp_clip_accumulate_embed(ids, G, V, None, 1.0, out, d=d, clip=clip)
    want = torch.zeros(V, d, dtype=torch.float64, device="cuda")
    rows = (G[..., :d].double() * clip.double()[:, None, None]).reshape(B * T, d)
    want.index_add_(0, ids.flatten().long(), rows)
    # fp32 sums of at most 100 terms of size |R g|: n eps times their sum of magnitudes
    size = torch.zeros_like(want).index_add_(0, ids.flatten().long(), rows.abs())
    assert ((out[:, :d].double() - want).abs() <= 110 * 2.0 ** -24 * size).all()
    if ldo > d:
        assert (out[:, d:] == 5.0).all()


# up to 32 rows no segment is long, and there is no second pass; a single window of tokens is grouped by one warp
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("T", [1, 2, 31, 32, 33, 34])
@pytest.mark.parametrize("kind", ["same", "distinct", "mixed", "out"])
def test_embedding_of_few_tokens(dtype, T, kind):
    d, V = 70, 50
    ids = {"same": torch.full((T,), 7), "distinct": torch.arange(T), "mixed": torch.arange(T) * 7 % 5,
           "out": torch.arange(T) % 3 * 30 - 1}[kind].to(torch.int32).view(1, T).cuda()      # -1, 29, 59
    G = torch.randn(1, T, d, generator=torch.Generator().manual_seed(T)).to(torch.float32 if dtype == "f32" else torch.bfloat16).cuda()
    sq, out, st = torch.zeros(1, device="cuda"), torch.empty(V, d, device="cuda"), torch.zeros(1, dtype=torch.int32, device="cuda")
    first = torch.empty(1, T, dtype=torch.int32, device="cuda")
    dp.dp_embed_norms(ids, G, V, sq, first_occ=first, dev_status=st)
    dp.dp_clip_accumulate_embed(ids, G, V, None, 1.0, out, d=d, clip=torch.full((1,), 0.5, device="cuda"), dev_status=st)
    rows, inside = ids.flatten().long(), (ids.flatten() >= 0) & (ids.flatten() < V)
    table = torch.zeros(V, d, dtype=torch.float64, device="cuda").index_add_(0, rows[inside], G[0].double()[inside])
    assert abs(float(sq) - float((table ** 2).sum())) <= 1e-5 * float((table ** 2).sum())
    assert float((out.double() - 0.5 * table).norm()) <= 1e-6 * float(table.norm())
    assert int(st.item()) == (0 if bool(inside.all()) else dp.DP_DEV_BAD_ID)
    for t in range(T):                                     # a token out of range is a group of its own
        want = t if not inside[t] else int((rows == rows[t]).nonzero()[0])
        assert int(first[0, t]) == want


# layers that stay on the fp32 kernels: tiles of 32 or 64 outputs (64 from 148 of them on), noise inside the
# kernel where d is a multiple of 4; sums and noise are the same bits as in two calls
@pytest.mark.parametrize("d,p,B,T", [(64, 64, 4, 16), (32, 33, 1, 1), (4, 7, 3, 5), (30, 40, 2, 31), (62, 70, 1, 33),
                                     (768, 800, 2, 9), (770, 769, 2, 9)])
def test_fp32_kernels_with_noise(d, p, B, T):
    g = torch.Generator(device="cuda")
    g.manual_seed(d + p)
    A = torch.randn(B, T, d, generator=g, device="cuda")
    G = torch.randn(B, T, p, generator=g, device="cuda")
    clip = torch.rand(B, generator=g, device="cuda")
    layers = [dp.Linear(A, G, d=d, p=p)]
    out, noisy = torch.full((p, d), 3.0, device="cuda"), torch.full((p, d), 3.0, device="cuda")
    before = dp.dp_debug_force_fma(True)
    try:
        dp.dp_clip_accumulate_grouped(layers, B, T, None, 1.0, [out], beta=1.0, clip=clip)
        dp.dp_clip_accumulate_noise_grouped(layers, B, T, None, 1.0, [noisy], 0.7, 0.5, 5, [2], 3, beta=1.0, clip=clip)
        sq = torch.zeros(B, device="cuda")
        dp.dp_ghost_norms(layers, B, T, sq)
    finally:
        dp.dp_debug_force_fma(before)
    G64, A64 = (G * clip[:, None, None]).double(), A.double()
    want = 3.0 + torch.einsum("btp,btd->pd", G64, A64)
    size = 3.0 + torch.einsum("btp,btd->pd", G64.abs(), A64.abs())
    assert ((out.double() - want).abs() <= (B * T + 2) * 2.0 ** -24 * size).all()
    dp.dp_add_noise(out, 0.7, 1.0, 0.5, 5, 2, 3)
    assert torch.equal(out, noisy)
    grads = torch.einsum("btp,btd->bpd", G.double(), A64)
    norms = (grads ** 2).sum((1, 2))
    # sums of at most T^2 products of dots of max(d, p) terms; their magnitudes add up to |A|^2 |G|^2
    size = (A64 ** 2).sum((1, 2)) * (G.double() ** 2).sum((1, 2))
    assert ((sq.double() - norms).abs() <= 2.0 ** -24 * (64 + T * T / 32) * size).all()


# fp32 step: split operands kept from the norms for the sums (ample workspace), layers in groups (the least
# workspace), one layer on the FMA kernels among them; against the same step call by call
@pytest.mark.parametrize("ample", [False, True])
@pytest.mark.parametrize("kind", ["plain", "tied", "vectors", "fma", "direct"])
def test_fp32_step_with_kept_operands(ample, kind):
    B, T, V, d = 3, 40, 700, 72
    g = torch.Generator(device="cuda")
    g.manual_seed(5)

    def normal(cols, std):
        return torch.empty(B, T, cols, device="cuda").normal_(0.0, std, generator=g)

    shapes = [(d, 3 * d), (3 * d, d), (d, d)] + ([(d, 8)] if kind == "fma" else [])
    linears = [dp.Linear(normal(i, 1.0), normal(o, 0.05), d=i, p=o) for i, o in shapes]
    if kind == "direct":
        linears[1].mode = dp.DP_NORM_DIRECT
    ids = torch.randint(0, V, (B, T), generator=g, device="cuda", dtype=torch.int32)
    vec = dict(dtype=torch.float32, device="cuda")
    ds = pipeline.DeviceStep(
        B=B, T=T, V=V, C=1.0, sigma=0.8, tied=kind == "tied", positions=False, linears=linears,
        lm=dp.Linear(normal(d, 1.0), normal(V, 0.02), d=d, p=V), ids=ids, pos_ids=None, G_emb=normal(d, 0.05), d_model=d,
        sq=torch.zeros(B, **vec), clip=torch.zeros(B, **vec), norms=torch.zeros(B, **vec),
        cross=torch.zeros(B, **vec) if kind == "tied" else None,
        dev_status=torch.zeros(1, dtype=torch.int32, device="cuda"))
    if kind == "vectors":
        ds.vectors = [dp.Vector(normal(d, 0.05), normal(d, 1.0), p=d), dp.Vector(linears[0].G, None, p=3 * d)]
    pipeline.allocate(ds)
    full = ds.ws.numel()
    if not ample:
        every = ds.linears + [ds.lm]
        least = max(dp.dp_ghost_norms_ws_bytes(every, B, T), dp.dp_clip_accumulate_grouped_ws_bytes(every, B, T),
                    int(dp.load().dp_clip_accumulate_embed_ws_bytes(B, T, d, V)))
        assert least < full
        ds.ws = torch.empty(least, dtype=torch.uint8, device="cuda")
    pipeline.dp_step(ds, noise=False, overlap=False)
    want = {n: t.clone() for n, t in ds.outs.items()}
    want_sq = ds.sq.clone()
    for t in ds.outs.values():
        t.fill_(9.0)
    pipeline.dp_step(ds, noise=False)
    assert torch.allclose(ds.sq, want_sq, rtol=1e-5)     # the same products, summed in groups of another size
    for n, t in ds.outs.items():
        assert float((t - want[n]).norm()) <= 1e-5 * float(want[n].norm()), n
    assert int(ds.dev_status.item()) == 0


# fp32 norms that split their operands on the way, for the sums to use: every height of a tile, several examples in one,
# widths that end inside a step of 64 columns or a word of 8, layers cut into chunks; one whose rows TMA cannot read among them
@pytest.mark.parametrize("B,T", [(3, 32), (8, 32), (5, 33), (7, 42), (3, 64), (2, 65), (3, 77), (2, 96), (1, 100), (3, 127), (2, 128), (3, 129)])
def test_fp32_norms_split_on_the_way(B, T):
    g = torch.Generator(device="cuda")
    g.manual_seed(B * T)

    def normal(cols, std, ld=None):
        t = torch.full((B, T, ld or cols), float("nan"), device="cuda")
        t[..., :cols] = torch.randn(B, T, cols, generator=g, device="cuda") * std
        return t

    shapes = [(64, 64, None), (72, 300, None), (132, 68, 140), (68, 9000, None), (5000, 64, None), (67, 130, 133)]
    linears = [dp.Linear(normal(i, 1.0, ld), normal(o, 0.05, ld), d=i, p=o) for i, o, ld in shapes]
    linears[4].mode = dp.DP_NORM_DIRECT
    vec = dict(dtype=torch.float32, device="cuda")
    ds = pipeline.DeviceStep(
        B=B, T=T, V=50, C=1.0, sigma=0.8, tied=False, positions=False, linears=linears, lm=None,
        ids=torch.zeros(B, T, dtype=torch.int32, device="cuda"), pos_ids=None, G_emb=normal(64, 0.05), d_model=64,
        sq=torch.zeros(B, **vec), clip=torch.zeros(B, **vec), norms=torch.zeros(B, **vec), cross=None,
        dev_status=torch.zeros(1, dtype=torch.int32, device="cuda"))
    pipeline.allocate(ds)
    for _ in range(2):                                     # the second step finds the first one's workspace
        ds.ws.fill_(255)
        pipeline.dp_step(ds, noise=False)
    want = (ds.G_emb.double().sum(1) ** 2).sum(1)
    for l in linears:
        want += (torch.einsum("btp,btd->bpd", l.G[..., :l.p].double(), l.A[..., :l.d].double()) ** 2).sum((1, 2))
    assert ((ds.sq.double() / want - 1).abs() < 4e-5).all()          # two bf16 terms: 2^-16 of a product at most
    R = ds.clip.double()[:, None, None]
    for k, l in enumerate(linears):
        ref = torch.einsum("btp,btd->pd", R * l.G[..., :l.p].double(), l.A[..., :l.d].double())
        assert float((ds.outs[f"linear{k}"].double() - ref).norm() / ref.norm()) < 2e-5, k
    assert int(ds.dev_status.item()) == 0


# the same where the pass over fp32 operands pays: two SMs, which it fills
@pytest.mark.parametrize("B,T", [(3, 32), (8, 32), (5, 33), (7, 42), (3, 64), (2, 65), (3, 77), (2, 96), (1, 100), (3, 127), (2, 128)])
def test_fp32_norms_split_on_the_way_on_two_sms(B, T):
    before = dp.dp_set_reserved_sms(146)
    try:
        test_fp32_norms_split_on_the_way(B, T)
    finally:
        dp.dp_set_reserved_sms(before)


# one pass where it is short or fills the chip, split first where it would wait for a few SMs or has few rows per tile
@pytest.mark.parametrize("shapes,B,T,launches", [([(256, 768), (256, 256)], 1, 64, 2), ([(256, 768), (256, 256)], 1, 128, 3),
                                                 ([(768, 2304)], 8, 128, 3), ([(768, 2304)] * 12, 16, 128, 2), ([(768, 2304)] * 12, 8, 32, 3)])
def test_fp32_norms_take_the_way_that_pays(shapes, B, T, launches):
    layers = [dp.Linear(torch.randn(B, T, d, device="cuda"), torch.randn(B, T, p, device="cuda") * 0.05, d=d, p=p) for d, p in shapes]
    ws = torch.empty(max(dp.dp_ghost_norms_ws_bytes(layers, B, T), dp.dp_step_ws_bytes(layers, B, T)), dtype=torch.uint8, device="cuda")
    sq = torch.zeros(B, device="cuda")
    n0 = dp.dp_kernel_launches()
    dp.dp_ghost_norms(layers, B, T, sq, ws=ws)
    assert dp.dp_kernel_launches() - n0 == launches
    want = sum((torch.einsum("btp,btd->bpd", l.G.double(), l.A.double()) ** 2).sum((1, 2)) for l in layers)
    assert ((sq.double() / want - 1).abs() < 4e-5).all()             # two bf16 terms: 2^-16 of a product at most


# layers that fit the workspace together go together, although the first few of them alone would be split along K into more planes
# than it holds; 64-token blocks 2, 3 and 5
@pytest.mark.parametrize("B,T", [(1, 77), (1, 128), (3, 64), (4, 77)])
def test_fp32_sums_of_layers_that_fit_go_together(B, T):
    shapes = [(576, 1728), (576, 576), (576, 2304), (2304, 576)]
    layers = [dp.Linear(torch.randn(B, T, d, device="cuda"), torch.randn(B, T, p, device="cuda") * 0.1, d=d, p=p) for d, p in shapes]
    outs, clip = [torch.empty(p, d, device="cuda") for d, p in shapes], torch.rand(B, device="cuda")
    need = max(dp.dp_step_ws_bytes(layers, B, T), dp.dp_clip_accumulate_grouped_ws_bytes(layers, B, T))
    ws = torch.empty(need, dtype=torch.uint8, device="cuda")
    n0 = dp.dp_kernel_launches()
    dp.dp_clip_accumulate_grouped(layers, B, T, None, 1.0, outs, clip=clip, ws=ws)
    assert dp.dp_kernel_launches() - n0 == 2                 # the split, the sums
    for l, o in zip(layers, outs):
        want = torch.einsum("btp,btd->pd", l.G.double() * clip.double()[:, None, None], l.A.double())
        assert float((o.double() - want).norm() / want.norm()) < 2e-5         # two bf16 terms


def test_fp32_norms_alone_store_no_split_operands():
    """Nobody reads them there: only the partial sums behind them are written."""
    B, T = 3, 40
    layers = [dp.Linear(torch.randn(B, T, d, device="cuda"), torch.randn(B, T, p, device="cuda"), d=d, p=p) for d, p in [(72, 304), (304, 72), (64, 64)]]
    ws = torch.full((dp.dp_ghost_norms_ws_bytes(layers, B, T),), 255, dtype=torch.uint8, device="cuda")
    sq = torch.zeros(B, device="cuda")
    dp.dp_ghost_norms(layers[:2], B, T, sq, ws=ws)
    planes = 2 * B * T * 2 * (72 + 304) * 2                # of two layers, every one a multiple of 256 bytes
    assert bool((ws[:planes] == 255).all()) and not bool((ws[planes:] == 255).all())


# tiles of 128 tokens x 32 positions, several per block from 2 x 148 tiles on
@pytest.mark.parametrize("B,T,d,V", [(1, 1, 64, 40), (2, 31, 72, 300), (3, 33, 64, 300), (2, 129, 136, 1000), (75, 128, 64, 100),
                                     (130, 97, 64, 64)])
def test_cross_term_tiles(B, T, d, V):
    G_emb, A_lm = bf16((B, T, d), 0.1, 1), bf16((B, T, d), 1.0, 2)
    G_lm = bf16((B, T, V), 0.1, 3, ld=(V + 7) // 8 * 8)
    g = torch.Generator(device="cuda")
    g.manual_seed(B + T)
    ids = torch.randint(0, V, (B, T), generator=g, device="cuda", dtype=torch.int32)
    sq, cross = torch.ones(B, device="cuda"), torch.zeros(B, device="cuda")
    dp.dp_tied_cross_term(ids, G_emb, A_lm, G_lm, V, sq=sq, cross=cross, d=d)
    M = torch.einsum("btd,bsd->bts", G_emb.double(), A_lm.double())
    W = torch.gather(G_lm[..., :V].double().transpose(1, 2), 1, ids.long()[:, :, None].expand(B, T, T))   # [b, t, s]
    want, size = (M * W).sum((1, 2)), (M * W).abs().sum((1, 2))
    # fp32 sums: d terms per entry of M (sizes |g||a|), then T*T entries in chains of 32
    entry = torch.einsum("btd,bsd->bts", G_emb.double().abs(), A_lm.double().abs())
    bound = 2.0 ** -24 * ((d + 8) * (entry * W.abs()).sum((1, 2)) + 64 * size)
    assert ((cross.double() - want).abs() <= bound).all()
    assert ((sq.double() - 1.0 - 2.0 * want).abs() <= 2.0 * bound + 2.0 ** -22 * (1.0 + size)).all()


# ghost norms on the fp32 kernels: tiles of 32 tokens, steps of 32 columns, chunks of 2048 of the wider operand,
# 64 layers per launch; without a workspace for the partial sums a launch per layer
@pytest.mark.parametrize("shapes,T", [([(31, 33)], 1), ([(32, 64), (5, 2048), (2049, 7)], 31), ([(40, 60)] * 65, 32),
                                      ([(33, 4100)], 33), ([(100, 50), (64, 64)], 65)])
@pytest.mark.parametrize("room", [True, False])
def test_fp32_gram_norms(shapes, T, room):
    B = 2
    g = torch.Generator(device="cuda")
    g.manual_seed(T)
    layers = [dp.Linear(torch.randn(B, T, d, generator=g, device="cuda"), torch.randn(B, T, p, generator=g, device="cuda"),
                        d=d, p=p, mode=dp.DP_NORM_GHOST) for d, p in shapes]
    sq = torch.zeros(B, device="cuda")
    before = dp.dp_debug_force_fma(True)
    try:
        ws = torch.empty(dp.dp_step_ws_bytes(layers, B, T) if room else 16, dtype=torch.uint8, device="cuda")
        n0 = dp.dp_kernel_launches()
        dp.dp_ghost_norms(layers, B, T, sq, ws=ws)
        assert dp.dp_kernel_launches() - n0 == (-(-len(shapes) // 64) + 1 if room else len(shapes))
    finally:
        dp.dp_debug_force_fma(before)
    want, size = 0, 0
    for l in layers:
        want = want + (torch.einsum("btp,btd->bpd", l.G.double(), l.A.double()) ** 2).sum((1, 2))
        size = size + (l.A.double() ** 2).sum((1, 2)) * (l.G.double() ** 2).sum((1, 2))
    # dots in chains of at most 32 + p / 32 terms, then sums over pairs: against |A|^2 |G|^2
    assert ((sq.double() - want).abs() <= 2.0 ** -24 * 256 * size).all()


# very short sequences: a warp per pair of tokens, up to 12 tokens, or 24 where some operand has 512 columns
@pytest.mark.parametrize("T", [1, 2, 11, 12, 13, 24, 25])
@pytest.mark.parametrize("shapes", [[(32, 511), (5, 70)], [(32, 512), (5, 70)], [(40, 60)] * 65, [(33, 4100), (2049, 2048)],
                                    [(33, 4100)]])     # 4100: three chunks
def test_fp32_gram_norms_of_very_short_sequences(shapes, T):
    test_fp32_gram_norms(shapes, T, True)


@pytest.mark.parametrize("d,p,T", [(511, 30, 31), (512, 30, 31), (700, 2048, 1), (700, 2049, 1), (64, 600, 33)])
def test_fp32_gram_norm_of_one_layer(d, p, T):
    """A layer of 512 columns or more by itself: one kernel, if its partial sums are one per example."""
    g = torch.Generator(device="cuda")
    g.manual_seed(T)
    layer = dp.Linear(torch.randn(2, T, d, generator=g, device="cuda"), torch.randn(2, T, p, generator=g, device="cuda"), d=d, p=p)
    sq = torch.ones(2, device="cuda")
    before = dp.dp_debug_force_fma(True)
    try:
        n0 = dp.dp_kernel_launches()
        dp.dp_ghost_norms([layer], 2, T, sq, ws=torch.empty(dp.dp_step_ws_bytes([layer], 2, T), dtype=torch.uint8, device="cuda"))
        assert dp.dp_kernel_launches() - n0 == (1 if max(d, p) >= 512 and p <= 2048 and T <= 32 else 2)
    finally:
        dp.dp_debug_force_fma(before)
    want = (torch.einsum("btp,btd->bpd", layer.G.double(), layer.A.double()) ** 2).sum((1, 2))
    size = (layer.A.double() ** 2).sum((1, 2)) * (layer.G.double() ** 2).sum((1, 2))
    assert ((sq.double() - 1.0 - want).abs() <= 2.0 ** -24 * 256 * size).all()


# Gram tiles as tall as the sequence, rounded up to 16 tokens, up to 64 tokens: rings of up to 32 stages of two
# or four column tiles; bf16 and split fp32
@pytest.mark.parametrize("T", [1, 15, 16, 17, 31, 32, 33, 48, 49, 64, 65, 77, 127, 128, 129])
@pytest.mark.parametrize("dtype", ["bf16", "f32"])
def test_gram_tiles_of_short_sequences(T, dtype):
    B, shapes = 3, [(64, 72), (300, 64), (136, 2500)]
    layers = [dp.Linear(bf16((B, T, d), 1.0, k, ld=(d + 7) // 8 * 8), bf16((B, T, p), 0.1, 50 + k, ld=(p + 7) // 8 * 8),
                        d=d, p=p, mode=dp.DP_NORM_GHOST) for k, (d, p) in enumerate(shapes)]
    if dtype == "f32":
        layers = [dp.Linear(l.A[..., :l.d].float().contiguous(), l.G[..., :l.p].float().contiguous(), d=l.d, p=l.p,
                            mode=dp.DP_NORM_GHOST) for l in layers]
    st = torch.zeros(1, dtype=torch.int32, device="cuda")
    for _ in range(2):                                     # the second call finds the first one's shared memory
        sq = torch.zeros(B, device="cuda")
        dp.dp_ghost_norms(layers, B, T, sq, dev_status=st)
    want = np.zeros(B)
    for l in layers:
        want += (np.einsum("btp,btd->bpd", f64(l.G, l.p), f64(l.A, l.d)) ** 2).sum((1, 2))
    # exact products, fp32 sums of at most 2500 terms
    assert (np.abs(sq.double().cpu().numpy() / want - 1) < 1e-5).all()
    assert int(st.item()) == 0


# several examples per Gram tile up to 64 tokens: as many as fit and one more or less, tiles of every multiple of 16 rows,
# examples across the quarters of a tile; one example that is not a number leaves the others alone
@pytest.mark.parametrize("B,T", [(300, 1), (127, 1), (2, 7), (40, 3), (8, 16), (9, 16), (7, 17), (15, 17), (33, 31), (4, 32), (5, 32), (4, 33),
                                 (7, 42), (2, 43), (5, 57), (1, 64), (4, 64)])
@pytest.mark.parametrize("dtype", ["bf16", "f32"])
def test_gram_tiles_of_several_examples(B, T, dtype):
    shapes = [(64, 72), (300, 64), (136, 2500)]
    layers = [dp.Linear(bf16((B, T, d), 1.0, k, ld=(d + 7) // 8 * 8), bf16((B, T, p), 0.1, 50 + k, ld=(p + 7) // 8 * 8),
                        d=d, p=p, mode=dp.DP_NORM_GHOST) for k, (d, p) in enumerate(shapes)]
    if B > 2:
        layers[1].A[1, T - 1, 5] = float("nan")
    if dtype == "f32":
        layers = [dp.Linear(l.A[..., :l.d].float().contiguous(), l.G[..., :l.p].float().contiguous(), d=l.d, p=l.p,
                            mode=dp.DP_NORM_GHOST) for l in layers]
    st = torch.zeros(1, dtype=torch.int32, device="cuda")
    before = dp.dp_set_reserved_sms(146)                   # with two SMs left, tiles are filled however few the items
    try:
        for _ in range(2):                                 # the second call finds the first one's shared memory
            sq = torch.zeros(B, device="cuda")
            dp.dp_ghost_norms(layers + layers, B, T, sq, dev_status=st)
    finally:
        dp.dp_set_reserved_sms(before)
    got, want = sq.double().cpu().numpy(), np.zeros(B)
    for l in layers + layers:
        want += (np.einsum("btp,btd->bpd", f64(l.G, l.p), f64(l.A, l.d)) ** 2).sum((1, 2))
    keep = np.arange(B) != 1 if B > 2 else np.ones(B, bool)
    assert keep.all() or np.isnan(got[1])
    # exact products (f32: the inputs are bf16 numbers), fp32 sums of at most 2500 terms
    assert (np.abs(got[keep] / want[keep] - 1) < 1e-5).all()
    assert int(st.item()) == 0


# row blocks of equal height in steps of 32 rows: one, two and three blocks of every height, an odd number of column steps
@pytest.mark.parametrize("T", [129, 160, 161, 192, 200, 224, 225, 256, 257, 300, 330, 384, 390, 430, 448, 512, 513, 600, 768])
def test_gram_blocks_of_longer_sequences(T):
    B, shapes = 2, [(64, 72), (300, 64), (136, 2500)]
    layers = [dp.Linear(bf16((B, T, d), 1.0, k, ld=(d + 7) // 8 * 8), bf16((B, T, p), 0.1, 50 + k, ld=(p + 7) // 8 * 8),
                        d=d, p=p, mode=dp.DP_NORM_GHOST) for k, (d, p) in enumerate(shapes)]
    st = torch.zeros(1, dtype=torch.int32, device="cuda")
    for _ in range(2):                                     # the second call finds the first one's shared memory
        sq = torch.zeros(B, device="cuda")
        dp.dp_ghost_norms(layers, B, T, sq, dev_status=st)
    want = np.zeros(B)
    for l in layers:
        want += (np.einsum("btp,btd->bpd", f64(l.G, l.p), f64(l.A, l.d)) ** 2).sum((1, 2))
    # exact products, fp32 sums of at most 2500 terms
    assert (np.abs(sq.double().cpu().numpy() / want - 1) < 1e-5).all()
    assert int(st.item()) == 0

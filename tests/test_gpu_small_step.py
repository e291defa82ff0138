"""Steps that are short of work take two launches (csrc/small_step.cu): against float64, in every form that is accepted,
and the forms that are not, which go the general way."""
import pytest
import torch

from paper_2609_40335_b200 import binding as dp, pipeline

pytestmark = pytest.mark.gpu

F32, BF16 = torch.float32, torch.bfloat16
SIGMA = 0.8


def make(layers, embed, B, T, d, shapes, V, *, pad=8, bad_ids=False, out_pad=0, offset=0, mode=dp.DP_NORM_AUTO, seed=1):
    """pad: pitches are multiples of it; out_pad, offset: outputs with a pitch and a base of their own."""
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)

    def rows(cols, std, dtype):
        t = torch.full((B, T, (cols + pad - 1) // pad * pad), float("nan"), dtype=dtype, device="cuda")
        t[..., :cols] = torch.randn(B, T, cols, generator=g, device="cuda") * std
        return t

    def out(r, c):
        flat = torch.full((r * (c + out_pad) + offset,), 7.0, device="cuda")
        return flat[offset:].view(r, c + out_pad)[:, :c]

    linears = [dp.Linear(rows(i, 1.0, layers), rows(o, 0.05, layers), d=i, p=o, mode=mode) for i, o in shapes]
    lo, hi = (-1, V + 1) if bad_ids else (0, V)
    ids = torch.randint(lo, hi, (B, T), generator=g, device="cuda", dtype=torch.int32)
    ids[torch.rand(B, T, generator=g, device="cuda") < 0.3] = V // 2          # a frequent token
    per = dict(dtype=F32, device="cuda")
    ds = pipeline.DeviceStep(
        B=B, T=T, V=V, C=1.0, sigma=SIGMA, tied=False, positions=False, linears=linears, lm=None, ids=ids, pos_ids=None,
        G_emb=rows(d, 0.05, embed), d_model=d, sq=torch.zeros(B, **per), clip=torch.zeros(B, **per),
        norms=torch.zeros(B, **per), cross=None, dev_status=torch.zeros(1, dtype=torch.int32, device="cuda"))
    pipeline.allocate(ds)
    for k, (i, o) in enumerate(shapes):
        ds.outs[f"linear{k}"] = out(o, i)
    ds.outs["wte"] = out(V, d)
    return ds


def check(ds, seed, step, noise, counter=0):
    """Everything against float64; an fp32 sum of n terms is off by at most n 2^-24 of the terms' magnitudes."""
    B, T, V, d = ds.B, ds.T, ds.V, ds.d_model
    eps, tid = 2.0 ** -24, pipeline.tensor_ids(ds)
    want = torch.zeros(B, dtype=torch.float64, device="cuda")
    size = torch.zeros_like(want)
    per = []
    for l in ds.linears:
        A, G = l.A[..., :l.d].double(), l.G[..., :l.p].double()
        per.append(torch.einsum("btp,btd->bpd", G, A))
        want += (per[-1] ** 2).sum((1, 2))
        # entries of two Gram matrices: dots of at most 256 terms, at most T^2 products
        size += (A ** 2).sum((1, 2)) * (G ** 2).sum((1, 2))
    hot = torch.zeros(B, T, V, dtype=torch.float64, device="cuda")
    ok = (ds.ids >= 0) & (ds.ids < V)
    hot.scatter_(2, ds.ids.clamp(0, V - 1).long().unsqueeze(2), ok.double().unsqueeze(2))
    G = ds.G_emb[..., :d].double()
    emb = torch.einsum("btv,btd->bvd", hot, G)
    want += (emb ** 2).sum((1, 2))
    size += T * (G ** 2).sum((1, 2))
    assert ((ds.sq.double() - want).abs() <= eps * (256 + T) * size).all()
    assert torch.allclose(ds.norms.double(), want.sqrt(), rtol=1e-4)
    assert torch.allclose(ds.clip.double(), (1.0 / want.sqrt()).clamp(max=1.0), rtol=1e-4)
    R = ds.clip.double()
    for name, grads, mag in [(f"linear{k}", per[k], torch.einsum("btp,btd->bpd", l.G[..., :l.p].double().abs(), l.A[..., :l.d].double().abs()))
                             for k, l in enumerate(ds.linears)] + [("wte", emb, torch.einsum("btv,btd->bvd", hot, G.abs()))]:
        z = torch.zeros(grads.shape[1], grads.shape[2], device="cuda")
        if noise:
            dp.dp_fill_noise(z, SIGMA, 1.0, 1.0, seed, tid[name], step + counter)
        ref = torch.einsum("b,bpd->pd", R, grads) + z.double()
        bound = eps * ((B * T + 4) * torch.einsum("b,bpd->pd", R, mag) + 2 * z.double().abs()) + 1e-30
        assert ((ds.outs[name].double() - ref).abs() <= bound).all(), name
    assert int(ds.dev_status.item()) == (0 if bool(ok.all()) else dp.DP_DEV_BAD_ID)


def launches(ds, **kw):
    n0 = dp.dp_kernel_launches()
    pipeline.dp_step(ds, **kw)
    return dp.dp_kernel_launches() - n0


# the smallest, edges of the 32-token and 32 x 32 tiles, of the 128-row stages and the 64-column items; the most tokens,
# layers, columns, examples and table rows
SIZES = [(4, 16, 64, [(64, 64)], 1000), (1, 1, 4, [(4, 8)], 3), (8, 64, 192, [(192, 192)], 5000), (64, 8, 36, [(36, 100), (256, 4)], 300),
         (5, 33, 200, [(200, 256)] * 2, 2600), (4, 24, 64, [(64, 128)] * 8, 100), (7, 63, 256, [], 4096), (2, 32, 12, [(60, 68)], 9472), (3, 43, 68, [(68, 132), (96, 96)], 295),
         (1, 31, 128, [(32, 160)], 297)]


@pytest.mark.parametrize("layers,embed", [(F32, F32), (BF16, BF16), (F32, BF16), (BF16, F32)])
@pytest.mark.parametrize("B,T,d,shapes,V", SIZES)
def test_small_step_against_float64(layers, embed, B, T, d, shapes, V):
    for noise in (False, True):
        ds = make(layers, embed, B, T, d, shapes, V)
        assert launches(ds, seed=9, step=4, noise=noise) == 2
        check(ds, 9, 4, noise)


@pytest.mark.parametrize("kw", [dict(bad_ids=True), dict(out_pad=4), dict(out_pad=3), dict(offset=1), dict(out_pad=5, offset=3)])
def test_ids_out_of_range_and_outputs_of_any_alignment(kw):
    ds = make(F32, F32, 4, 40, 64, [(64, 96)], 700, **kw)
    assert launches(ds, seed=2, step=1) == 2
    check(ds, 2, 1, True)


# what the two kernels do not take goes the general way, with the same results: widths that are no multiple of four, layers
# with a DIRECT norm (forced, and by the rule), one token, column or layer too many, a larger table
@pytest.mark.parametrize("B,T,d,shapes,V,kw", [
    (3, 17, 62, [(62, 70)], 300, {}), (3, 17, 64, [(64, 70)], 300, {}), (3, 17, 64, [(64, 64)], 300, dict(mode=dp.DP_NORM_DIRECT)),
    (3, 40, 32, [(32, 32)], 300, {}), (3, 65, 64, [(64, 96)], 300, {}), (9, 57, 64, [(64, 96)], 300, {}),
    (3, 17, 64, [(260, 64)], 300, {}), (3, 17, 64, [(256, 256)] * 5, 300, {}), (13, 33, 64, [(64, 64)] * 8, 300, {}), (3, 17, 64, [(64, 64)] * 9, 300, {}), (3, 17, 8, [(64, 64)], 9473, {}),
    (65, 4, 8, [(64, 64)], 100, {})])
def test_what_is_not_taken_goes_the_general_way(B, T, d, shapes, V, kw):
    ds = make(F32, F32, B, T, d, shapes, V, pad=1, **kw)
    assert launches(ds, seed=2, step=1, noise=False) > 2
    want = {n: t.clone() for n, t in ds.outs.items()}
    sq = ds.sq.clone()
    pipeline.dp_step(ds, seed=2, step=1, noise=False, overlap=False)
    assert torch.allclose(ds.sq, sq, rtol=1e-5)
    for n, t in ds.outs.items():
        assert float((t - want[n]).norm()) <= 2e-5 * float(t.norm()), n


def test_small_step_graph_draws_the_noise_of_its_step():
    ds = make(F32, F32, 4, 16, 64, [(64, 64)], 1000)
    graph = pipeline.StepGraph(ds, seed=5, first_step=3)
    assert graph.kernels_per_replay == 2
    for k in range(3):
        for t in ds.outs.values():
            t.fill_(9.0)
        graph.replay()
        check(ds, 5, 3, True, counter=k)


def test_small_step_comes_after_the_side_stream():
    """A fill of the table that nobody waited for is over before the step writes it."""
    ds = make(F32, F32, 8, 64, 128, [(128, 128)], 8192)
    for k in range(20):
        pipeline.prefill_embedding_noise(ds, seed=77, step=k)
        pipeline.dp_step(ds, seed=5, step=k)
    torch.cuda.synchronize()
    check(ds, 5, 19, True)


@pytest.mark.parametrize("captured", [False, True])
def test_side_stream_comes_after_the_small_step(captured):
    """Work put on the side stream after the step finds the table as the step wrote it, also inside a capture."""
    ds = make(F32, F32, 8, 64, 128, [(128, 128)], 8192)
    pipeline.dp_step(ds, seed=5, step=0)                 # makes the side stream
    got = torch.empty_like(ds.outs["wte"])
    torch.cuda.synchronize()

    def step_and_read():
        torch.cuda._sleep(20_000_000)                    # some 10 ms: the step has not begun when the copy is enqueued
        n0 = dp.dp_kernel_launches()
        pipeline.dp_step(ds, seed=5, step=4)
        assert dp.dp_kernel_launches() - n0 == 2
        with torch.cuda.stream(ds.side_stream):
            got.copy_(ds.outs["wte"])
        torch.cuda.current_stream().wait_stream(ds.side_stream)

    if captured:
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            step_and_read()
        for t in ds.outs.values():
            t.fill_(9.0)
        graph.replay()
    else:
        step_and_read()
    torch.cuda.synchronize()
    check(ds, 5, 4, True)
    assert torch.equal(got, ds.outs["wte"])


# bf16 layers whose norms would fill an SM's shared memory go the general way; fp32 ones, fewer table columns or layers do not
@pytest.mark.parametrize("layers,d,n,taken", [(BF16, 256, 2, False), (F32, 256, 2, True), (BF16, 64, 2, True), (BF16, 256, 1, True)])
def test_bf16_steps_of_many_wide_blocks(layers, d, n, taken):
    ds = make(layers, layers, 64, 8, d, [(256, 256)] * n, 300)
    assert (launches(ds, seed=2, step=1, noise=False) == 2) == taken
    want, sq = {n: t.clone() for n, t in ds.outs.items()}, ds.sq.clone()
    pipeline.dp_step(ds, seed=2, step=1, noise=False, overlap=False)
    assert torch.allclose(ds.sq, sq, rtol=1e-5)
    for n, t in ds.outs.items():
        # bf16 tensor cores round R_i * g once, by 2^-9 at most
        assert float((t - want[n]).norm()) <= (2e-5 if layers == F32 else 2.0 ** -8) * float(t.norm()), n

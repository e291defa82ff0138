"""The one-call step (pipeline.dp_step, dp_step_enqueue) against the same step call by call."""
import pytest
import torch

from paper_2609_40335_b200 import binding as dp, pipeline

pytestmark = pytest.mark.gpu

F32, BF16 = torch.float32, torch.bfloat16


def make_step(layers=BF16, vectors=BF16, embed=BF16, *, B=3, T=40, V=700, d=64, tied=False, lm=True, positions=False,
              pos_ids=None, seed=5):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)

    def normal(cols, std, dtype, ld=None):
        return torch.empty(B, T, ld or cols, dtype=dtype, device="cuda").normal_(0.0, std, generator=g)

    linears = [dp.Linear(normal(i, 1.0, layers), normal(o, 0.05, layers), d=i, p=o) for i, o in [(d, 3 * d), (3 * d, d), (d, 72)]]
    head = dp.Linear(normal(d, 1.0, layers), normal(V, 0.02, layers, ld=(V + 7) // 8 * 8), d=d, p=V) if lm else None
    per = dict(dtype=F32, device="cuda")
    if positions and pos_ids is None:
        pos_ids = torch.arange(T, dtype=torch.int32, device="cuda").repeat(B, 1).contiguous()
    ds = pipeline.DeviceStep(
        B=B, T=T, V=V, C=1.0, sigma=0.8, tied=tied, positions=positions, linears=linears, lm=head,
        ids=torch.randint(0, V, (B, T), generator=g, device="cuda", dtype=torch.int32), pos_ids=pos_ids,
        G_emb=normal(d, 0.05, embed), d_model=d, sq=torch.zeros(B, **per), clip=torch.zeros(B, **per),
        norms=torch.zeros(B, **per), cross=torch.zeros(B, **per) if tied else None,
        dev_status=torch.zeros(1, dtype=torch.int32, device="cuda"))
    ds.vectors = [dp.Vector(normal(d, 0.05, vectors), normal(d, 1.0, vectors), p=d), dp.Vector(normal(3 * d, 0.05, vectors), None, p=3 * d)]
    pipeline.allocate(ds)
    return ds


def state(ds):
    torch.cuda.synchronize()
    return dict({n: t.clone() for n, t in ds.outs.items()}, sq=ds.sq.clone(), clip=ds.clip.clone())


def wipe(ds):
    for t in ds.outs.values():
        t.fill_(9.0)
    ds.sq.fill_(-1.0)
    ds.clip.fill_(-1.0)


def assert_same(got, want, rel=5e-5):
    """The same products in fp32, summed in another order: 1e-5.  A clip factor that differs by 2^-24 flips the bf16
    rounding of 2^-16 of the R_i * x, by 2^-8 each: 2^-16 = 1.5e-5 more."""
    for n, t in want.items():
        assert float((got[n] - t).norm()) <= rel * float(t.norm()), n


@pytest.mark.parametrize("noise", [False, True])
@pytest.mark.parametrize("layers,vectors,embed", [(BF16, F32, BF16), (F32, BF16, BF16), (BF16, BF16, F32), (BF16, F32, F32),
                                                  (F32, BF16, F32), (F32, F32, BF16)])
def test_step_of_mixed_dtypes(layers, vectors, embed, noise):
    ds = make_step(layers, vectors, embed, positions=True)
    pipeline.dp_step(ds, seed=3, step=2, noise=noise, overlap=False)
    want = state(ds)
    wipe(ds)
    pipeline.dp_step(ds, seed=3, step=2, noise=noise)
    assert_same(state(ds), want)
    assert int(ds.dev_status.item()) == 0


def test_unsupported_and_clashing_dtypes_are_refused():
    for change in ("half_vector", "mixed_vector", "mixed_layer", "ids", "out", "tied"):
        ds = make_step(tied=change == "tied")
        if change == "half_vector":
            ds.vectors[1].G = ds.vectors[1].G.half()
        elif change == "mixed_vector":
            ds.vectors[0].X = ds.vectors[0].X.float()
        elif change == "mixed_layer":
            ds.linears[1].G = ds.linears[1].G.float()
        elif change == "ids":
            ds.ids = ds.ids.long()
        elif change == "out":
            ds.outs["linear1"] = ds.outs["linear1"].bfloat16()
        else:
            ds.G_emb = ds.G_emb.float()
        with pytest.raises(dp.DpGhostError) as e:
            pipeline.dp_step(ds)
        assert e.value.status == 1
        torch.cuda.synchronize()


@pytest.mark.parametrize("overlap", [False, True])
def test_positions_beyond_the_sequence_length_count_in_the_norm(overlap):
    """Offset (packed, left-padded) positions: rows of the table that the sum receives belong to the norm as well."""
    B, T, d = 3, 40, 64
    first = torch.tensor([0, 100, 1024 - T], dtype=torch.int32, device="cuda")
    pos = (first[:, None] + torch.arange(T, dtype=torch.int32, device="cuda")).contiguous()
    ds = make_step(B=B, T=T, d=d, positions=True, pos_ids=pos)
    plain = make_step(B=B, T=T, d=d)                  # the same inputs without the position table
    pipeline.dp_step(plain, noise=False, overlap=False)
    pipeline.dp_step(ds, noise=False, overlap=overlap)
    torch.cuda.synchronize()
    assert int(ds.dev_status.item()) == 0
    rows = ds.G_emb.double()                          # every position is its own row: the norm of its gradient
    want = plain.sq.double() + (rows ** 2).sum((1, 2))
    assert ((ds.sq.double() / want - 1).abs() < 1e-5).all()
    table = torch.zeros(1024, d, dtype=torch.float64, device="cuda")
    table.index_add_(0, pos.flatten().long(), (rows * ds.clip.double()[:, None, None]).reshape(-1, d))
    assert float((ds.outs["wpe"].double() - table).norm() / table.norm()) < 1e-6


def test_position_outside_the_table_is_flagged_and_skipped_by_both():
    pos = torch.arange(40, dtype=torch.int32, device="cuda").repeat(3, 1).contiguous()
    pos[1, 7], pos[2, 0] = 1024, -1
    ds = make_step(positions=True, pos_ids=pos)
    plain = make_step()
    pipeline.dp_step(plain, noise=False)
    pipeline.dp_step(ds, noise=False)
    torch.cuda.synchronize()
    assert int(ds.dev_status.item()) == dp.DP_DEV_BAD_ID
    rows = ds.G_emb.double()
    inside = ((pos >= 0) & (pos < 1024)).double()
    want = plain.sq.double() + (rows ** 2 * inside[:, :, None]).sum((1, 2))
    assert ((ds.sq.double() / want - 1).abs() < 1e-5).all()


def test_copy_on_write_outputs_are_written_apart():
    """A lazy clone shares memory until it is written to; the library's writes count."""
    ds = make_step()
    pipeline.dp_step(ds, noise=False)
    want = state(ds)
    wipe(ds)
    kept = {n: ds.outs[n] for n in ("linear0", "wte", "vector0")}
    for n, t in kept.items():
        ds.outs[n] = torch._lazy_clone(t)
    pipeline.dp_step(ds, noise=False)
    assert_same(state(ds), want)
    for n, t in kept.items():
        assert (t == 9.0).all(), n
    for n, t in kept.items():
        ds.outs[n] = torch._lazy_clone(t)
    pipeline.dp_step(ds, noise=False, overlap=False)      # call by call: lists of outputs
    assert_same(state(ds), want)
    for n, t in kept.items():
        assert (t == 9.0).all(), n


def test_clip_factors_changed_between_the_phases_reach_the_row_sums():
    """Work on the caller's stream between the norms and the sums is ordered before all sums, those of the side stream
    too: here the factors change 50 ms later."""
    ds = make_step(positions=True)
    step = dict(seed=3, step=2)
    pipeline.clip_after_prefill(ds, **step, filled=pipeline.overlapped_norms(ds, **step))     # a kernel's first launch waits
    filled = pipeline.overlapped_norms(ds, **step)
    torch.cuda._sleep(100_000_000)
    ds.clip.fill_(0.25)
    pipeline.clip_after_prefill(ds, **step, filled=filled)
    torch.cuda.synchronize()
    for name, ids in (("wte", ds.ids), ("wpe", ds.pos_ids)):
        noise = torch.empty_like(ds.outs[name])
        dp.dp_fill_noise(noise, ds.sigma, ds.C, 1.0, 3, pipeline.tensor_ids(ds)[name], 2)
        want = noise.double().index_add_(0, ids.flatten().long(), 0.25 * ds.G_emb.double().reshape(-1, ds.d_model))
        assert float((ds.outs[name].double() - want).norm() / want.norm()) < 1e-6, name


def test_event_of_the_overlapped_norms_orders_the_tables_and_sorts():
    """A third stream that waits for it sees the table's noise and the sort, not what was there before."""
    ds = make_step(V=200000, d=768, B=4, lm=False)        # the fill outlasts the norms
    step = dict(seed=3, step=2)
    pipeline.clip_after_prefill(ds, **step, filled=pipeline.overlapped_norms(ds, **step))
    want = state(ds)
    noise = torch.empty_like(ds.outs["wte"])
    dp.dp_fill_noise(noise, ds.sigma, ds.C, 1.0, 3, pipeline.tensor_ids(ds)["wte"], 2)
    parts = [ds.side["perm"], ds.side["seg"], ds.outs["wte"][-20000:]]       # the fill's last rows
    expected = [parts[0].cpu(), parts[1].cpu(), noise[-20000:].cpu()]
    seen = [torch.empty(p.shape, dtype=p.dtype, pin_memory=True) for p in parts]
    other = torch.cuda.Stream()
    for _ in range(5):
        wipe(ds)
        for p in parts[:2]:
            p.fill_(-1)
        torch.cuda.synchronize()
        filled = pipeline.overlapped_norms(ds, **step)
        other.wait_event(filled)
        with torch.cuda.stream(other):
            for s, p in zip(reversed(seen), reversed(parts)):    # the copy engine's work: no kernel, which would have to
                s.copy_(p, non_blocking=True)                    # wait until the fill leaves it room
        torch.cuda.current_stream().wait_stream(other)
        pipeline.clip_after_prefill(ds, **step, filled=filled)
        torch.cuda.synchronize()
        for s, e in zip(seen, expected):
            assert torch.equal(s, e)
        assert_same(state(ds), want)


@pytest.mark.parametrize("tied", [False, True])
def test_prefill_and_scale_of_the_overlapped_step(tied):
    """Tables filled at a scale of the caller's; layers and vectors scaled by clip_after_prefill."""
    step, scale = dict(seed=3, step=2), 0.25
    ds = make_step(tied=tied, positions=True)
    tid = pipeline.tensor_ids(ds)
    pipeline.dp_step(ds, **step, noise=False)
    sums = state(ds)
    rows = torch.zeros_like(ds.outs["wte"])
    dp.dp_clip_accumulate_embed(ds.ids, ds.G_emb, ds.V, None, ds.C, rows, d=ds.d_model, clip=ds.clip)
    wipe(ds)
    pipeline.overlapped_norms(ds, **step)
    filled = pipeline.prefill_embedding_noise(ds, **step, scale=scale)
    pipeline.clip_after_prefill(ds, **step, filled=filled, scale=scale)
    got = state(ds)
    for name in ds.outs:
        want = torch.zeros_like(got[name])
        if name in ("wte", "wpe") and not (tied and name == "wte"):
            dp.dp_fill_noise(want, ds.sigma, ds.C, scale, 3, tid[name], 2)
            want += sums[name]
        elif name == "wte":                              # head's sum and noise, scaled; the rows as they are
            want = sums[name] - rows
            dp.dp_add_noise(want, ds.sigma, ds.C, scale, 3, tid[name], 2)
            want += rows
        else:
            want = sums[name].clone()
            dp.dp_add_noise(want, ds.sigma, ds.C, scale, 3, tid[name], 2)
        assert float((got[name] - want).norm()) < 1e-5 * float(want.norm()), name


def test_tied_step_without_a_place_for_the_cross_term():
    ds = make_step(tied=True)
    pipeline.dp_step(ds, noise=False)
    want = state(ds)
    ds.cross = ds.norms = None
    wipe(ds)
    pipeline.dp_step(ds, noise=False)
    got = state(ds)
    for n, t in want.items():
        assert torch.equal(got[n], t), n


@pytest.mark.parametrize("dtype", [BF16, F32])
def test_step_without_a_workspace_of_its_own(dtype):
    """A DeviceStep whose user gave it outputs but no workspace."""
    ds = make_step(dtype, dtype, dtype, tied=True, positions=True)
    pipeline.dp_step(ds, seed=3, step=2)
    want = state(ds)
    ds.ws = None
    for by_phases in (False, True):
        wipe(ds)
        if by_phases:
            pipeline.clip_after_prefill(ds, seed=3, step=2, filled=pipeline.overlapped_norms(ds, seed=3, step=2))
        else:
            pipeline.dp_step(ds, seed=3, step=2)
        assert_same(state(ds), want)
        assert ds.ws is None


def test_fp32_step_in_the_least_memory(monkeypatch):
    """By request, and where the large workspace does not fit."""
    ds = make_step(F32, F32, F32)
    pipeline.dp_step(ds, noise=False)
    want, large = state(ds), ds.ws.numel()
    every = ds.linears + [ds.lm]
    pipeline.allocate(ds, split_once=False)
    small = ds.ws.numel()
    lib = dp.load()
    assert small == max(dp.dp_ghost_norms_ws_bytes(every, ds.B, ds.T), dp.dp_clip_accumulate_grouped_ws_bytes(every, ds.B, ds.T),
                        int(lib.dp_clip_accumulate_embed_ws_bytes(ds.B, ds.T, ds.d_model, ds.V))) < large
    pipeline.dp_step(ds, noise=False)
    assert_same(state(ds), want)
    empty = torch.empty

    def full(*size, **kw):
        if kw.get("dtype") == torch.uint8 and size[0] > small:
            raise torch.cuda.OutOfMemoryError("no room")
        return empty(*size, **kw)

    monkeypatch.setattr(torch, "empty", full)
    pipeline.allocate(ds)
    assert ds.ws.numel() == small


# vectors read once (row sums kept from the norms) or twice; widths around a slab of 256 columns and a Philox counter of
# four, one more vector than a launch holds, fewer tokens than pay
@pytest.mark.parametrize("dtype", [BF16, F32])
@pytest.mark.parametrize("B,T,widths", [(3, 40, [1, 3, 4, 255, 256, 257, 700]), (9, 8, [64] * 97), (2, 7, [64, 70]), (1, 9, [513])])
def test_vectors_read_once_and_twice(dtype, B, T, widths):
    ds = make_step(vectors=dtype, B=B, T=T)
    g = torch.Generator(device="cuda")
    g.manual_seed(T)
    rand = lambda p, std: torch.empty(B, T, p, dtype=dtype, device="cuda").normal_(0.0, std, generator=g)
    ds.vectors = [dp.Vector(rand(p, 0.05), rand(p, 1.0) if k % 2 else None, p=p) for k, p in enumerate(widths)]
    pipeline.allocate(ds)
    keep = dp.dp_step_vectors_ws_bytes(ds.vectors, B, T)
    assert (keep == 0) == (T < 8)
    results, launches = [], []
    for ws in (ds.ws, ds.ws[:ds.ws.numel() - max(keep, 256)], ds.ws[4:]):      # with room, with less, off the boundary
        ds.ws = ws
        for noise in (True, False):
            wipe(ds)
            n0 = dp.dp_kernel_launches()
            pipeline.dp_step(ds, seed=3, step=2, noise=noise)
            launches.append(dp.dp_kernel_launches() - n0)
            results.append(state(ds))
    groups = (len(widths) + 95) // 96
    assert launches[4] - launches[0] == (groups if T >= 8 else 0) and launches[2] in (launches[0], launches[4])
    for got, want in ((0, 2), (1, 3), (4, 2), (5, 3)):
        # at most 360 products in fp32, added up in another order
        assert_same(results[got], results[want], rel=360 * 2.0 ** -24)
    assert int(ds.dev_status.item()) == 0


# finite gradients of one example that overflow when they are summed over its tokens: no finite norm, factor 0, and the
# example leaves every sum; a term that is itself infinite or not a number shows in its column.  With and without kept sums
@pytest.mark.parametrize("dtype", [BF16, F32])
def test_vector_sums_that_overflow_drop_out(dtype):
    ds = make_step(vectors=dtype, B=5, T=24)
    big = torch.finfo(dtype).max
    gain, bias = ds.vectors
    bias.G[1, :, 3] = big                         # +inf, and with the second pair of signs inf - inf between two warps' rows
    bias.G[1, ::2, 4], bias.G[1, 1::2, 4] = big, -big
    gain.G[1, :, 5], gain.X[1, :, 5] = 1e25, 1e10
    gain.G[2, 7, 6], gain.X[2, 7, 6] = 1e25, 1e25            # the term itself is infinite
    bias.G[3, 9, 7] = float("nan")
    results = []
    for ws in (ds.ws, ds.ws[:ds.ws.numel() - dp.dp_step_vectors_ws_bytes(ds.vectors, ds.B, ds.T)]):
        ds.ws = ws
        wipe(ds)
        pipeline.dp_step(ds, noise=False)
        results.append(state(ds))
    kept, read_again = results
    assert kept["clip"].tolist()[1:4] == [0.0, 0.0, 0.0] and bool((kept["clip"][[0, 4]] > 0).all())
    for k, (v, bad) in enumerate([(gain, 6), (bias, 7)]):
        terms = v.G.double() * (v.X.double() if v.X is not None else 1.0)
        want = (kept["clip"][[0, 4]].double()[:, None] * terms[[0, 4]].sum(1)).sum(0)
        for got in (kept[f"vector{k}"], read_again[f"vector{k}"]):
            fine = torch.arange(v.p, device="cuda") != bad
            assert bool(got[bad].isnan())
            # at most 48 products in fp32
            assert float((got.double() - want)[fine].norm()) <= 48 * 2.0 ** -24 * float(want[fine].norm())


# kept sums of fewer examples than a block has parts, of as many as it walks by itself, one more, a short part, parts of more than 128 rows
@pytest.mark.parametrize("B", [7, 9, 448, 449, 1030, 16400])
def test_kept_sums_of_large_batches(B):
    ds = make_step(vectors=F32, B=B, T=8, V=100, lm=False)
    g = torch.Generator(device="cuda")
    g.manual_seed(B)
    ds.vectors = [dp.Vector(torch.randn(B, 8, p, generator=g, device="cuda") * 0.05, None, p=p) for p in (3, 64, 300)]
    pipeline.allocate(ds)
    wipe(ds)
    n0 = dp.dp_kernel_launches()
    pipeline.dp_step(ds, seed=3, step=2)
    with_room = dp.dp_kernel_launches() - n0
    got = state(ds)
    tid = pipeline.tensor_ids(ds)
    for k, v in enumerate(ds.vectors):
        z = torch.zeros((v.p + 3) // 4 * 4, device="cuda")
        dp.dp_fill_noise(z, ds.sigma, 1.0, 1.0, 3, tid[f"vector{k}"], 2)
        terms = v.G.double() * got["clip"].double()[:, None, None]
        # at most 8 B products in fp32, and the noise's own rounding
        bound = 2.0 ** -24 * (8 * B * terms.abs().sum((0, 1)) / B + 4 * z[:v.p].double().abs() + terms.abs().sum((0, 1)))
        assert ((got[f"vector{k}"].double() - terms.sum((0, 1)) - z[:v.p].double()).abs() <= bound).all(), k
    ds.ws = ds.ws[:ds.ws.numel() - dp.dp_step_vectors_ws_bytes(ds.vectors, B, 8)]
    n0 = dp.dp_kernel_launches()
    pipeline.dp_step(ds, seed=3, step=2)
    assert dp.dp_kernel_launches() - n0 - with_room == (1 if B <= 448 else 0)
    assert_same(state(ds), got, rel=8 * 64 * 2.0 ** -24)

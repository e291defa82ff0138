"""dp_step_enqueue finds what is wrong with its arguments before it enqueues anything.  No GPU: a call that got as
far as the CUDA runtime would return DP_ERR_CUDA here."""
import ctypes as C

import pytest
import torch

from paper_2609_40335_b200 import binding, build

if torch.cuda.is_available():                     # made-up addresses: only where nothing can run
    pytest.skip("for machines without a GPU", allow_module_level=True)

OK, INVALID, UNSUPPORTED, ALIGNMENT, WORKSPACE, CUDA = 0, 1, 2, 3, 4, 5
vp, i64, i32, u32, f32 = C.c_void_p, C.c_int64, C.c_int32, C.c_uint32, C.c_float


class StepDesc(C.Structure):
    _fields_ = ([("layers", C.POINTER(binding._LinearDesc)), ("outs", C.POINTER(vp)), ("ldos", C.POINTER(i64)),
                 ("tensor_ids", C.POINTER(u32)), ("vectors", C.POINTER(binding._VectorDesc)), ("vector_outs", C.POINTER(vp)),
                 ("vector_ids", C.POINTER(u32)), ("ids", vp), ("G_emb", vp), ("ldge", i64), ("pos_ids", vp), ("wte", vp),
                 ("ld_wte", i64), ("wpe", vp), ("ld_wpe", i64)] +
                [(n, vp) for n in "sq clip norms cross side_sq perm seg pos_perm pos_seg ws".split()] +
                [("ws_bytes", C.c_size_t), ("side_ws", vp), ("side_ws_bytes", C.c_size_t), ("dev_status", vp), ("stream", vp),
                 ("side_stream", vp), ("events", vp * 4), ("seed", C.c_uint64)] +
                [(n, i32) for n in "n_layers n_vectors layer_dtype vector_dtype embed_dtype B T V d pos_rows tied with_noise".split()] +
                [("C", f32), ("sigma", f32), ("step", u32), ("wte_id", u32), ("wpe_id", u32)])


@pytest.fixture(scope="module")
def lib():
    build.build()
    L = binding.load()
    L.dp_step_enqueue.argtypes = [vp, i32]
    return L


def desc(dtype=1, T=40, V=2000, tied=False):
    """A step that only lacks a GPU: addresses nobody reads, on 4 KiB boundaries."""
    at = iter(range(1 << 20, 1 << 30, 1 << 12))
    B, d, shapes = 3, 64, [(64, 192), (192, 64), (64, V)]
    S = StepDesc()
    S.keep = [(binding._LinearDesc * 3)(), (vp * 3)(), (i64 * 3)(), (u32 * 3)(1, 2, 3), (binding._VectorDesc * 2)(), (vp * 2)(),
              (u32 * 2)(4, 5)]
    layers, outs, ldos, tids, vecs, vouts, vids = S.keep
    for k, (i, o) in enumerate(shapes):
        layers[k].A, layers[k].lda, layers[k].d = next(at), i, i
        layers[k].G, layers[k].ldg, layers[k].p = next(at), (o + 7) // 8 * 8, o
        outs[k], ldos[k] = next(at), i
    for k in range(2):
        vecs[k].G, vecs[k].ldg, vecs[k].p, vouts[k] = next(at), 64, 64, next(at)
    S.layers, S.outs, S.ldos, S.tensor_ids = layers, outs, ldos, tids
    S.vectors, S.vector_outs, S.vector_ids = vecs, vouts, vids
    for n in "ids G_emb wte sq clip norms cross side_sq perm seg pos_perm pos_seg ws side_ws dev_status wpe pos_ids".split():
        setattr(S, n, next(at))
    S.events = (vp * 4)(*[next(at) for _ in range(4)])
    S.ldge = S.ld_wte = S.ld_wpe = d
    S.ws_bytes = S.side_ws_bytes = 1 << 34
    S.n_layers, S.n_vectors, S.layer_dtype, S.vector_dtype, S.embed_dtype = 3, 2, dtype, dtype, dtype
    S.B, S.T, S.V, S.d, S.pos_rows, S.tied, S.with_noise, S.C, S.sigma = B, T, V, d, 1024, int(tied), 1, 1.0, 0.8
    return S


def call(lib, S, phases=7):
    return lib.dp_step_enqueue(C.byref(S), phases)


def test_a_sound_step_reaches_the_runtime(lib):
    for dtype in (0, 1):
        for tied in (False, True):
            assert call(lib, desc(dtype, tied=tied)) == CUDA


def test_what_may_be_left_out(lib):
    S = desc(tied=True)
    S.norms = S.cross = S.dev_status = S.pos_ids = S.wpe = S.pos_perm = S.pos_seg = None
    S.n_vectors, S.vectors, S.vector_outs, S.vector_ids = 0, None, None, None
    S.with_noise, S.tensor_ids = 0, None
    assert call(lib, S) == CUDA


def spoil(S, what):
    if what == "T":
        S.T = 4097
    elif what == "C":
        S.C = 0.0
    elif what == "C, no noise":
        S.C, S.with_noise = -1.0, 0
    elif what == "sigma":
        S.sigma = float("nan")
    elif what == "ldge":
        S.ldge = 63
    elif what == "ld_wte":
        S.ld_wte = 63
    elif what == "ld_wpe":
        S.ld_wpe = 63
    elif what == "vector ld":
        S.vectors[1].ldg = 63
    elif what == "vector out":
        S.vector_outs[1] = None
    elif what == "vector ids":
        S.vector_ids = None
    elif what == "no vectors":
        S.vectors = None
    elif what == "layer out":
        S.outs[2] = None
    elif what == "layer ldo":
        S.ldos[1] = 191
    elif what == "layer ld":
        S.layers[0].ldg = 191
    elif what == "layer mode":
        S.layers[0].mode = 7
    elif what == "dtype":
        S.vector_dtype = 2
    elif what == "layer address":
        S.layers[1].A += 8
    elif what == "embedding address":
        S.tied, S.G_emb = 1, S.G_emb + 8
    elif what == "ws":
        S.ws_bytes = 255
    elif what == "no ws":
        S.ws = None
    elif what == "side ws":
        S.side_ws_bytes = 255
    elif what == "no side ws":
        S.side_ws = None
    elif what == "clash of dtypes":
        S.tied, S.embed_dtype = 1, 1 - S.layer_dtype
    else:
        raise ValueError(what)


@pytest.mark.parametrize("what,status", [
    ("T", UNSUPPORTED), ("C", INVALID), ("C, no noise", INVALID), ("sigma", INVALID), ("ldge", INVALID), ("ld_wte", INVALID),
    ("ld_wpe", INVALID), ("vector ld", INVALID), ("vector out", INVALID), ("vector ids", INVALID), ("no vectors", INVALID),
    ("layer out", INVALID), ("layer ldo", INVALID), ("layer ld", INVALID), ("layer mode", INVALID), ("dtype", INVALID),
    ("layer address", ALIGNMENT), ("embedding address", ALIGNMENT), ("ws", WORKSPACE), ("no ws", WORKSPACE),
    ("side ws", WORKSPACE), ("no side ws", WORKSPACE), ("clash of dtypes", INVALID)])
def test_errors_are_found_before_anything_is_enqueued(lib, what, status):
    S = desc()
    spoil(S, what)
    assert call(lib, S) == status


@pytest.mark.parametrize("dtype", [0, 1])
@pytest.mark.parametrize("tied", [False, True])
def test_least_workspaces(lib, dtype, tied):
    """What the calls that a step stands for ask for is enough, and a byte less is not."""
    S = desc(dtype, tied=tied)
    B, T, V, d, n = S.B, S.T, S.V, S.d, S.n_layers
    ws = [lib.dp_ghost_norms_ws_bytes(S.layers, n, dtype, B, T), lib.dp_clip_accumulate_grouped_ws_bytes(S.layers, n, dtype, B, T),
          lib.dp_vector_norms_ws_bytes(S.vectors, 2, B, T), lib.dp_clip_accumulate_vectors_ws_bytes(S.vectors, 2, B, T)]
    side = [lib.dp_embed_norms_ws_bytes(B, T, d)] + [lib.dp_embed_sort_ws_bytes(B, T, v) for v in (V, 1024)]
    side.append(lib.dp_clip_accumulate_embed_ws_bytes(B, T, d, 1024))
    (ws if tied else side).append(lib.dp_clip_accumulate_embed_ws_bytes(B, T, d, V))
    if tied:
        ws.append(lib.dp_tied_cross_term_ws_bytes(B, T, d, V))
    S.ws_bytes, S.side_ws_bytes = max(ws), max(side)
    assert call(lib, S) == CUDA
    S.ws_bytes -= 1
    assert call(lib, S) == WORKSPACE
    S.ws_bytes, S.side_ws_bytes = max(ws), max(side) - 1
    assert call(lib, S) == WORKSPACE


@pytest.mark.parametrize("phase", [1, 2, 4])
def test_a_phase_asks_for_what_it_uses(lib, phase):
    S = desc()
    assert call(lib, S, phase) == CUDA
    S.ws_bytes = S.side_ws_bytes = 255
    assert call(lib, S, phase) == WORKSPACE
